// field.cuh -- prime-field arithmetic on 8 x 32-bit limbs for sm_103a.
//
// Elements are 256-bit little-endian limb vectors in Montgomery form
// (X = x * 2^256 mod r), as the paper describes field elements: word-sized
// limbs (Section II).  mul, add and sub give results in [0, r); the operations of a
// transform (the _loose ones and mul_factor) keep residues in [0, 2r), or below 4r for
// a difference that only feeds a product, and its last pass brings the outputs below r.
//
// * mul: Montgomery product X * Y * 2^-256 mod r, coarsely integrated operand
//   scanning (CIOS): for each limb b_i, t += a * b_i, then m = t_0 * r' and
//   t = (t + m * r) / 2^32.  The paper finds FF_mul to be the dominant cost of
//   the NTT (Section IV-B: FF_mul + FF_sqr are 93.8% of NTT time) and the
//   32-bit multiply-add (IMAD) the dominant instruction (Section IV-B-2).  Every
//   carry chain is a single asm statement, so the carry flag never has to
//   survive between statements.
// * add / sub: the paper measures the conditional-reduction branches as 70.5%
//   of FF_add latency (Section IV-B-1) and 52-56% branch efficiency (Section
//   IV-C).  Here both candidates are computed and one is selected with a mask
//   from the borrow -- no branch.
//
// The reduction rows use the low limbs of the moduli (row_reduce).
#pragma once
#include <cstdint>

namespace zkntt {

struct FrBLS12_381 {
    static constexpr uint32_t P0 = 0x00000001u, P1 = 0xffffffffu, P2 = 0xfffe5bfeu, P3 = 0x53bda402u,
                              P4 = 0x09a1d805u, P5 = 0x3339d808u, P6 = 0x299d7d48u, P7 = 0x73eda753u;
    static constexpr uint32_t RP = 0xffffffffu;  // -r^-1 mod 2^32
    static constexpr int ID = 0;
};

struct FrBN254 {
    static constexpr uint32_t P0 = 0xf0000001u, P1 = 0x43e1f593u, P2 = 0x79b97091u, P3 = 0x2833e848u,
                              P4 = 0x8181585du, P5 = 0xb85045b6u, P6 = 0xe131a029u, P7 = 0x30644e72u;
    static constexpr uint32_t RP = 0xefffffffu;
    static constexpr int ID = 1;
};

// BLS12-377 F_r (253 bits; r = 1 mod 2^32 as for BLS12-381, so m = -t_0)
struct FrBLS12_377 {
    static constexpr uint32_t P0 = 0x00000001u, P1 = 0x0a118000u, P2 = 0xd0000001u, P3 = 0x59aa76feu,
                              P4 = 0x5c37b001u, P5 = 0x60b44d1eu, P6 = 0x9a2ca556u, P7 = 0x12ab655eu;
    static constexpr uint32_t RP = 0xffffffffu;
    static constexpr int ID = 2;
};

// ---------------------------------------------------------------------------
// conditional subtraction of r: x in [0, 2r) -> [0, r), branch-free
template <class F>
__device__ __forceinline__ void reduce_once(uint32_t x[8]) {
    uint32_t u[8], mask;
    asm("sub.cc.u32  %0, %9, %17;\n\t"
        "subc.cc.u32 %1, %10, %18;\n\t"
        "subc.cc.u32 %2, %11, %19;\n\t"
        "subc.cc.u32 %3, %12, %20;\n\t"
        "subc.cc.u32 %4, %13, %21;\n\t"
        "subc.cc.u32 %5, %14, %22;\n\t"
        "subc.cc.u32 %6, %15, %23;\n\t"
        "subc.cc.u32 %7, %16, %24;\n\t"
        "subc.u32    %8, 0, 0;"
        : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]),
          "=r"(u[7]), "=r"(mask)
        : "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3]), "r"(x[4]), "r"(x[5]), "r"(x[6]), "r"(x[7]),
          "n"(F::P0), "n"(F::P1), "n"(F::P2), "n"(F::P3), "n"(F::P4), "n"(F::P5), "n"(F::P6),
          "n"(F::P7));
    // mask = all ones when x < r (borrow): keep x, else take x - r
#pragma unroll
    for (int i = 0; i < 8; i++) x[i] = u[i] ^ ((x[i] ^ u[i]) & mask);
}

// r = a + b mod p, inputs canonical
template <class F>
__device__ __forceinline__ void add(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) {
    asm("add.cc.u32  %0, %8, %16;\n\t"
        "addc.cc.u32 %1, %9, %17;\n\t"
        "addc.cc.u32 %2, %10, %18;\n\t"
        "addc.cc.u32 %3, %11, %19;\n\t"
        "addc.cc.u32 %4, %12, %20;\n\t"
        "addc.cc.u32 %5, %13, %21;\n\t"
        "addc.cc.u32 %6, %14, %22;\n\t"
        "addc.u32    %7, %15, %23;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]),
          "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]));
    reduce_once<F>(r);  // a + b < 2r < 2^256: no carry out of limb 7
}

// r = a - b mod p, inputs canonical
template <class F>
__device__ __forceinline__ void sub(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) {
    uint32_t mask;
    asm("sub.cc.u32  %0, %9, %17;\n\t"
        "subc.cc.u32 %1, %10, %18;\n\t"
        "subc.cc.u32 %2, %11, %19;\n\t"
        "subc.cc.u32 %3, %12, %20;\n\t"
        "subc.cc.u32 %4, %13, %21;\n\t"
        "subc.cc.u32 %5, %14, %22;\n\t"
        "subc.cc.u32 %6, %15, %23;\n\t"
        "subc.cc.u32 %7, %16, %24;\n\t"
        "subc.u32    %8, 0, 0;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(mask)
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]),
          "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]));
    // on borrow add r back (mask selects the modulus limbs)
    asm("add.cc.u32  %0, %0, %8;\n\t"
        "addc.cc.u32 %1, %1, %9;\n\t"
        "addc.cc.u32 %2, %2, %10;\n\t"
        "addc.cc.u32 %3, %3, %11;\n\t"
        "addc.cc.u32 %4, %4, %12;\n\t"
        "addc.cc.u32 %5, %5, %13;\n\t"
        "addc.cc.u32 %6, %6, %14;\n\t"
        "addc.u32    %7, %7, %15;"
        : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
          "+r"(r[7])
        : "r"(F::P0 & mask), "r"(F::P1 & mask), "r"(F::P2 & mask), "r"(F::P3 & mask),
          "r"(F::P4 & mask), "r"(F::P5 & mask), "r"(F::P6 & mask), "r"(F::P7 & mask));
}

// ---------------------------------------------------------------------------
// Residues in [0, 2r) ("loose"): inside a transform no value is brought below r;
// the last pass does that once per output.  2r < 2^256 for the three fields; 4r
// is too for BN254 and BLS12-377, not for BLS12-381.
template <class F>
struct Twice {
    static constexpr uint32_t D0 = F::P0 << 1, D1 = (F::P1 << 1) | (F::P0 >> 31),
                              D2 = (F::P2 << 1) | (F::P1 >> 31), D3 = (F::P3 << 1) | (F::P2 >> 31),
                              D4 = (F::P4 << 1) | (F::P3 >> 31), D5 = (F::P5 << 1) | (F::P4 >> 31),
                              D6 = (F::P6 << 1) | (F::P5 >> 31), D7 = (F::P7 << 1) | (F::P6 >> 31);
    static constexpr bool SUM_FITS = F::P7 < 0x40000000u;  // 4r < 2^256
};

// r = a + b, less 2p unless below it: loose from loose
template <class F>
__device__ __forceinline__ void add_loose(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) {
    using D = Twice<F>;
    uint32_t s[8], u[8], mask, c = 0;
    if constexpr (D::SUM_FITS)
        asm("add.cc.u32  %0, %8, %16;\n\t"
            "addc.cc.u32 %1, %9, %17;\n\t"
            "addc.cc.u32 %2, %10, %18;\n\t"
            "addc.cc.u32 %3, %11, %19;\n\t"
            "addc.cc.u32 %4, %12, %20;\n\t"
            "addc.cc.u32 %5, %13, %21;\n\t"
            "addc.cc.u32 %6, %14, %22;\n\t"
            "addc.u32    %7, %15, %23;"
            : "=r"(s[0]), "=r"(s[1]), "=r"(s[2]), "=r"(s[3]), "=r"(s[4]), "=r"(s[5]), "=r"(s[6]),
              "=r"(s[7])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]),
              "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]),
              "r"(b[7]));
    else
        asm("add.cc.u32  %0, %9, %17;\n\t"
            "addc.cc.u32 %1, %10, %18;\n\t"
            "addc.cc.u32 %2, %11, %19;\n\t"
            "addc.cc.u32 %3, %12, %20;\n\t"
            "addc.cc.u32 %4, %13, %21;\n\t"
            "addc.cc.u32 %5, %14, %22;\n\t"
            "addc.cc.u32 %6, %15, %23;\n\t"
            "addc.cc.u32 %7, %16, %24;\n\t"
            "addc.u32    %8, 0, 0;"
            : "=r"(s[0]), "=r"(s[1]), "=r"(s[2]), "=r"(s[3]), "=r"(s[4]), "=r"(s[5]), "=r"(s[6]),
              "=r"(s[7]), "=r"(c)
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]),
              "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]),
              "r"(b[7]));
    // mask = c - borrow: all ones when the sum is below 2p (c = 0 and a borrow;
    // a carry out always comes with a borrow, since a + b - 2p < 2^256)
    asm("sub.cc.u32  %0, %9, %17;\n\t"
        "subc.cc.u32 %1, %10, %18;\n\t"
        "subc.cc.u32 %2, %11, %19;\n\t"
        "subc.cc.u32 %3, %12, %20;\n\t"
        "subc.cc.u32 %4, %13, %21;\n\t"
        "subc.cc.u32 %5, %14, %22;\n\t"
        "subc.cc.u32 %6, %15, %23;\n\t"
        "subc.cc.u32 %7, %16, %24;\n\t"
        "subc.u32    %8, %25, 0;"
        : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]),
          "=r"(u[7]), "=r"(mask)
        : "r"(s[0]), "r"(s[1]), "r"(s[2]), "r"(s[3]), "r"(s[4]), "r"(s[5]), "r"(s[6]), "r"(s[7]),
          "n"(D::D0), "n"(D::D1), "n"(D::D2), "n"(D::D3), "n"(D::D4), "n"(D::D5), "n"(D::D6),
          "n"(D::D7), "r"(c));
#pragma unroll
    for (int i = 0; i < 8; i++) r[i] = u[i] ^ ((s[i] ^ u[i]) & mask);
}

// r = a - b, plus 2p if negative: loose from loose
template <class F>
__device__ __forceinline__ void sub_loose(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) {
    using D = Twice<F>;
    asm("{\n\t.reg .pred p;\n\t.reg .u32 m;\n\t"
        "sub.cc.u32  %0, %8, %16;\n\t"
        "subc.cc.u32 %1, %9, %17;\n\t"
        "subc.cc.u32 %2, %10, %18;\n\t"
        "subc.cc.u32 %3, %11, %19;\n\t"
        "subc.cc.u32 %4, %12, %20;\n\t"
        "subc.cc.u32 %5, %13, %21;\n\t"
        "subc.cc.u32 %6, %14, %22;\n\t"
        "subc.cc.u32 %7, %15, %23;\n\t"
        "subc.u32    m, 0, 0;\n\t"
        "setp.ne.u32 p, m, 0;\n\t"
        "@p add.cc.u32  %0, %0, %24;\n\t"
        "@p addc.cc.u32 %1, %1, %25;\n\t"
        "@p addc.cc.u32 %2, %2, %26;\n\t"
        "@p addc.cc.u32 %3, %3, %27;\n\t"
        "@p addc.cc.u32 %4, %4, %28;\n\t"
        "@p addc.cc.u32 %5, %5, %29;\n\t"
        "@p addc.cc.u32 %6, %6, %30;\n\t"
        "@p addc.u32    %7, %7, %31;\n\t}"
        : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]), "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]),
          "=&r"(r[7])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]),
          "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]),
          "n"(D::D0), "n"(D::D1), "n"(D::D2), "n"(D::D3), "n"(D::D4), "n"(D::D5), "n"(D::D6),
          "n"(D::D7));
}

// r congruent to a - b for loose a, b, only to be multiplied by a factor: where
// 4p < 2^256, a + 2p - b in (0, 4p) without a correction
template <class F>
__device__ __forceinline__ void diff_loose(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) {
    using D = Twice<F>;
    if constexpr (!D::SUM_FITS) {
        sub_loose<F>(r, a, b);
    } else {
        uint32_t u[8];
        asm("add.cc.u32  %0, %8, %16;\n\t"
            "addc.cc.u32 %1, %9, %17;\n\t"
            "addc.cc.u32 %2, %10, %18;\n\t"
            "addc.cc.u32 %3, %11, %19;\n\t"
            "addc.cc.u32 %4, %12, %20;\n\t"
            "addc.cc.u32 %5, %13, %21;\n\t"
            "addc.cc.u32 %6, %14, %22;\n\t"
            "addc.u32    %7, %15, %23;"
            : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]),
              "=r"(u[7])
            : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]),
              "n"(D::D0), "n"(D::D1), "n"(D::D2), "n"(D::D3), "n"(D::D4), "n"(D::D5), "n"(D::D6),
              "n"(D::D7));
        asm("sub.cc.u32  %0, %8, %16;\n\t"
            "subc.cc.u32 %1, %9, %17;\n\t"
            "subc.cc.u32 %2, %10, %18;\n\t"
            "subc.cc.u32 %3, %11, %19;\n\t"
            "subc.cc.u32 %4, %12, %20;\n\t"
            "subc.cc.u32 %5, %13, %21;\n\t"
            "subc.cc.u32 %6, %14, %22;\n\t"
            "subc.u32    %7, %15, %23;"
            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
              "=r"(r[7])
            : "r"(u[0]), "r"(u[1]), "r"(u[2]), "r"(u[3]), "r"(u[4]), "r"(u[5]), "r"(u[6]), "r"(u[7]),
              "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]),
              "r"(b[7]));
    }
}

// r = a + p - b, in (0, 2p) and congruent to a - b, for canonical a, b: no
// conditional correction (the G-point block transforms).  Only for values that feed mul as its second
// (limb-scanned) operand, which may be any value below 2^256.
template <class F>
__device__ __forceinline__ void sub_lazy(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) {
    // r = a + p into fresh registers (a stays live for the caller: no copy),
    // then r -= b in place
    asm("add.cc.u32  %0, %8, %16;\n\t"
        "addc.cc.u32 %1, %9, %17;\n\t"
        "addc.cc.u32 %2, %10, %18;\n\t"
        "addc.cc.u32 %3, %11, %19;\n\t"
        "addc.cc.u32 %4, %12, %20;\n\t"
        "addc.cc.u32 %5, %13, %21;\n\t"
        "addc.cc.u32 %6, %14, %22;\n\t"
        "addc.u32    %7, %15, %23;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]),
          "n"(F::P0), "n"(F::P1), "n"(F::P2), "n"(F::P3), "n"(F::P4), "n"(F::P5), "n"(F::P6),
          "n"(F::P7));
    asm("sub.cc.u32  %0, %0, %8;\n\t"
        "subc.cc.u32 %1, %1, %9;\n\t"
        "subc.cc.u32 %2, %2, %10;\n\t"
        "subc.cc.u32 %3, %3, %11;\n\t"
        "subc.cc.u32 %4, %4, %12;\n\t"
        "subc.cc.u32 %5, %5, %13;\n\t"
        "subc.cc.u32 %6, %6, %14;\n\t"
        "subc.u32    %7, %7, %15;"
        : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
          "+r"(r[7])
        : "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]), "r"(b[7]));
}

// ---------------------------------------------------------------------------
// Montgomery product, CIOS on two accumulators of wide multiply-adds.
//
// The running value is t = sum E_k 2^(32 k) + sum O_k 2^(32 (k + 1)): E takes
// the partial products whose low word falls on an even limb, O the others
// (the even/odd split of Emmart, Luitjens, Weems and Woolley, "Optimizing
// modular multiplication for NVIDIA's Maxwell GPUs", ARITH 2016).  Within one
// accumulator the 64-bit partial products of a row lie end to end, so a row is
// a single carry chain of mad.lo.cc / madc.hi.cc pairs whose two words are one
// register pair: the assembler makes each pair one wide multiply-add with
// carry in and carry out, and no add instruction merges partial products.
// Outer step i adds a b_i, then m r with m = t_0 r' mod 2^32; that clears E_0,
// and dividing by 2^32 makes O the even accumulator and E, moved by two limbs
// (a renaming), the odd one; the left-over E_1 enters at the head of the next
// row's chain.  With r < 2^255 t < 2r after every step, so O_7 never overflows.
//
// What bounds it: the heavy FMA datapath, which a wide multiply(-add) holds
// for four cycles a warp.  This form issues 112 (BLS12-381) or 120 wide
// multiplies and about 80 other instructions, where the previous one (wide
// products merged by add-with-carry chains on the ALU pipe) issued 112 to 120
// and about 300, among them 82 register moves on the heavy datapath for the
// zero-extended 64-bit addends.  Measured in isolation on GB300, G products/s
// (four blocks of 256 threads an SM, one chain a thread): BLS12-381 56.9 ->
// 80.3, BN254 58.0 -> 73.8, BLS12-377 56.9 -> 79.4; with one block an SM
// still 70 to 76.

// t += a b (row i > 0).  E: the even accumulator; O: the odd one, limbs 0..5
// of it (limbs 6 and 7 are zero); e1: the limb left over at position 0.
__device__ __forceinline__ void row_product(uint32_t E[8], uint32_t O[8], uint32_t e1,
                                            const uint32_t a[8], uint32_t b) {
    asm("add.cc.u32      %0, %0, %16;\n\t"
        "madc.lo.cc.u32  %8, %18, %25, %8;\n\t"
        "madc.hi.cc.u32  %9, %18, %25, %9;\n\t"
        "madc.lo.cc.u32 %10, %20, %25, %10;\n\t"
        "madc.hi.cc.u32 %11, %20, %25, %11;\n\t"
        "madc.lo.cc.u32 %12, %22, %25, %12;\n\t"
        "madc.hi.cc.u32 %13, %22, %25, %13;\n\t"
        "madc.lo.cc.u32 %14, %24, %25, 0;\n\t"
        "madc.hi.u32    %15, %24, %25, 0;\n\t"
        "mad.lo.cc.u32   %0, %17, %25, %0;\n\t"
        "madc.hi.cc.u32  %1, %17, %25, %1;\n\t"
        "madc.lo.cc.u32  %2, %19, %25, %2;\n\t"
        "madc.hi.cc.u32  %3, %19, %25, %3;\n\t"
        "madc.lo.cc.u32  %4, %21, %25, %4;\n\t"
        "madc.hi.cc.u32  %5, %21, %25, %5;\n\t"
        "madc.lo.cc.u32  %6, %23, %25, %6;\n\t"
        "madc.hi.cc.u32  %7, %23, %25, %7;\n\t"
        "addc.u32       %15, %15, 0;"
        : "+r"(E[0]), "+r"(E[1]), "+r"(E[2]), "+r"(E[3]), "+r"(E[4]), "+r"(E[5]), "+r"(E[6]),
          "+r"(E[7]), "+r"(O[0]), "+r"(O[1]), "+r"(O[2]), "+r"(O[3]), "+r"(O[4]), "+r"(O[5]),
          "=&r"(O[6]), "=&r"(O[7])
        : "r"(e1), "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]),
          "r"(a[7]), "r"(b));
}

// t += m r with m chosen so that limb 0 of the sum is zero.  E_0 is left as it
// was (the caller drops it); its carry, 1 unless it was zero, is in.
//   r_0 = 1:                 m = -E_0, and m r_0 + E_0 only carries.
//   r_0 = 1, r_1 = 2^32 - 1: also m r_1 + carry = m 2^32 - m + carry, its words
//                            E_0 (= -m) and m - carry plus the carry itself: one
//                            wide multiply fewer (80.3 against 79.4 G/s).
//   r_0 = 2^32 - 2^28 + 1 (r' = 2^32 - 2^28 - 1): m and the high word
//                            m - (m >> 4) of m r_0 come from shifts and adds.
//   any other r_0:           m = E_0 r' and both words of m r_0 by multiplies.
// m = -E_0 is written as sub.cc: as a plain negation the assembler folds it
// into the multiplies' operands, which splits every wide multiply-add in two
// (232 instead of 182 instructions a product).
template <class F>
__device__ __forceinline__ void row_reduce(uint32_t E[8], uint32_t O[8]) {
    if constexpr (F::P0 == 1u && F::P1 == 0xffffffffu) {
        uint32_t m, h, z;
        asm("sub.cc.u32 %0, 0, %2;\n\t"
            "subc.u32   %1, %0, 0;"
            : "=&r"(m), "=r"(h)
            : "r"(E[0]));
        asm("add.cc.u32     %14, %15, 0xffffffff;\n\t"
            "addc.cc.u32     %0, %0, %15;\n\t"
            "addc.cc.u32     %1, %1, %17;\n\t"
            "madc.lo.cc.u32  %2, %16, %18, %2;\n\t"
            "madc.hi.cc.u32  %3, %16, %18, %3;\n\t"
            "madc.lo.cc.u32  %4, %16, %19, %4;\n\t"
            "madc.hi.cc.u32  %5, %16, %19, %5;\n\t"
            "madc.lo.cc.u32  %6, %16, %20, %6;\n\t"
            "madc.hi.u32     %7, %16, %20, %7;\n\t"
            "mad.lo.cc.u32   %8, %16, %21, %8;\n\t"
            "madc.hi.cc.u32  %9, %16, %21, %9;\n\t"
            "madc.lo.cc.u32 %10, %16, %22, %10;\n\t"
            "madc.hi.cc.u32 %11, %16, %22, %11;\n\t"
            "madc.lo.cc.u32 %12, %16, %23, %12;\n\t"
            "madc.hi.cc.u32 %13, %16, %23, %13;\n\t"
            "addc.u32        %7, %7, 0;"
            : "+r"(O[0]), "+r"(O[1]), "+r"(O[2]), "+r"(O[3]), "+r"(O[4]), "+r"(O[5]), "+r"(O[6]),
              "+r"(O[7]), "+r"(E[2]), "+r"(E[3]), "+r"(E[4]), "+r"(E[5]), "+r"(E[6]), "+r"(E[7]),
              "=&r"(z)
            : "r"(E[0]), "r"(m), "r"(h), "n"(F::P3), "n"(F::P5), "n"(F::P7), "n"(F::P2),
              "n"(F::P4), "n"(F::P6));
    } else if constexpr (F::P0 == 1u) {
        uint32_t m, z;
        asm("sub.cc.u32 %0, 0, %1;" : "=r"(m) : "r"(E[0]));
        asm("mad.lo.cc.u32   %8, %16, %21, %8;\n\t"
            "madc.hi.cc.u32  %9, %16, %21, %9;\n\t"
            "madc.lo.cc.u32 %10, %16, %22, %10;\n\t"
            "madc.hi.cc.u32 %11, %16, %22, %11;\n\t"
            "madc.lo.cc.u32 %12, %16, %23, %12;\n\t"
            "madc.hi.cc.u32 %13, %16, %23, %13;\n\t"
            "addc.u32        %7, %7, 0;\n\t"
            "add.cc.u32     %14, %15, 0xffffffff;\n\t"
            "madc.lo.cc.u32  %0, %16, %17, %0;\n\t"
            "madc.hi.cc.u32  %1, %16, %17, %1;\n\t"
            "madc.lo.cc.u32  %2, %16, %18, %2;\n\t"
            "madc.hi.cc.u32  %3, %16, %18, %3;\n\t"
            "madc.lo.cc.u32  %4, %16, %19, %4;\n\t"
            "madc.hi.cc.u32  %5, %16, %19, %5;\n\t"
            "madc.lo.cc.u32  %6, %16, %20, %6;\n\t"
            "madc.hi.u32     %7, %16, %20, %7;"
            : "+r"(O[0]), "+r"(O[1]), "+r"(O[2]), "+r"(O[3]), "+r"(O[4]), "+r"(O[5]), "+r"(O[6]),
              "+r"(O[7]), "+r"(E[2]), "+r"(E[3]), "+r"(E[4]), "+r"(E[5]), "+r"(E[6]), "+r"(E[7]),
              "=&r"(z)
            : "r"(E[0]), "r"(m), "n"(F::P1), "n"(F::P3), "n"(F::P5), "n"(F::P7), "n"(F::P2),
              "n"(F::P4), "n"(F::P6));
    } else {
        constexpr bool SHIFTS = F::P0 == 0xf0000001u;
        const uint32_t m = SHIFTS ? 0u - E[0] - (E[0] << 28) : E[0] * F::RP;
        // high word of m r_0, by shifts without the carry of its low word
        const uint32_t h = SHIFTS ? m - (m >> 4) : __umulhi(m, F::P0);
        const uint32_t l = SHIFTS ? m : m * F::P0;
        uint32_t z;
        asm("add.cc.u32     %14, %16, %26;\n\t"
            "addc.cc.u32    %15, %15, %18;\n\t"
            "madc.lo.cc.u32  %8, %17, %23, %8;\n\t"
            "madc.hi.cc.u32  %9, %17, %23, %9;\n\t"
            "madc.lo.cc.u32 %10, %17, %24, %10;\n\t"
            "madc.hi.cc.u32 %11, %17, %24, %11;\n\t"
            "madc.lo.cc.u32 %12, %17, %25, %12;\n\t"
            "madc.hi.cc.u32 %13, %17, %25, %13;\n\t"
            "addc.u32        %7, %7, 0;\n\t"
            "mad.lo.cc.u32   %0, %17, %19, %0;\n\t"
            "madc.hi.cc.u32  %1, %17, %19, %1;\n\t"
            "madc.lo.cc.u32  %2, %17, %20, %2;\n\t"
            "madc.hi.cc.u32  %3, %17, %20, %3;\n\t"
            "madc.lo.cc.u32  %4, %17, %21, %4;\n\t"
            "madc.hi.cc.u32  %5, %17, %21, %5;\n\t"
            "madc.lo.cc.u32  %6, %17, %22, %6;\n\t"
            "madc.hi.u32     %7, %17, %22, %7;"
            : "+r"(O[0]), "+r"(O[1]), "+r"(O[2]), "+r"(O[3]), "+r"(O[4]), "+r"(O[5]), "+r"(O[6]),
              "+r"(O[7]), "+r"(E[2]), "+r"(E[3]), "+r"(E[4]), "+r"(E[5]), "+r"(E[6]), "+r"(E[7]),
              "=&r"(z), "+r"(E[1])
            : "r"(E[0]), "r"(m), "r"(h), "n"(F::P1), "n"(F::P3), "n"(F::P5), "n"(F::P7),
              "n"(F::P2), "n"(F::P4), "n"(F::P6), "r"(l));
    }
}

// r = a * b * 2^-256 mod p, canonical.  a must be canonical; b may be any
// value below 2^256: with t <= 2r - 1, a <= r - 1 and b_i, m <= 2^32 - 1 an
// outer step gives (t + a b_i + m r) / 2^32 <= 2r - 1 whatever b is, and the
// final value is below r b / 2^256 + r < 2r, so one conditional subtraction
// canonicalises it.  r may alias a or b.
template <class F>
__device__ __forceinline__ void mul(uint32_t r[8], const uint32_t a[8], const uint32_t b[8]) {
    uint32_t X[8], Y[8];  // step i: the even accumulator is X for even i, Y for odd i
#pragma unroll
    for (int k = 0; k < 4; k++) {
        const uint64_t e = uint64_t(a[2 * k]) * b[0], o = uint64_t(a[2 * k + 1]) * b[0];
        X[2 * k] = uint32_t(e);
        X[2 * k + 1] = uint32_t(e >> 32);
        Y[2 * k] = uint32_t(o);
        Y[2 * k + 1] = uint32_t(o >> 32);
    }
    row_reduce<F>(X, Y);
#pragma unroll
    for (int i = 1; i < 8; i++) {
        uint32_t *E = (i & 1) ? Y : X, *O = (i & 1) ? X : Y;
        const uint32_t e1 = O[1];
#pragma unroll
        for (int k = 0; k < 6; k++) O[k] = O[k + 2];
        row_product(E, O, e1, a, b[i]);
        row_reduce<F>(E, O);
    }
    uint32_t t[8];  // X + Y / 2^32 (the low limb of Y is zero modulo 2^32)
    asm("add.cc.u32  %0, %8, %16;\n\t"
        "addc.cc.u32 %1, %9, %17;\n\t"
        "addc.cc.u32 %2, %10, %18;\n\t"
        "addc.cc.u32 %3, %11, %19;\n\t"
        "addc.cc.u32 %4, %12, %20;\n\t"
        "addc.cc.u32 %5, %13, %21;\n\t"
        "addc.cc.u32 %6, %14, %22;\n\t"
        "addc.u32    %7, %15, 0;"
        : "=r"(t[0]), "=r"(t[1]), "=r"(t[2]), "=r"(t[3]), "=r"(t[4]), "=r"(t[5]), "=r"(t[6]),
          "=r"(t[7])
        : "r"(X[0]), "r"(X[1]), "r"(X[2]), "r"(X[3]), "r"(X[4]), "r"(X[5]), "r"(X[6]), "r"(X[7]),
          "r"(Y[1]), "r"(Y[2]), "r"(Y[3]), "r"(Y[4]), "r"(Y[5]), "r"(Y[6]), "r"(Y[7]));
    reduce_once<F>(t);
#pragma unroll
    for (int i = 0; i < 8; i++) r[i] = t[i];
}

// ---------------------------------------------------------------------------
// Product with a constant known in advance (a twiddle): Shoup's method with a
// precomputed quotient (V. Shoup's NTL; D. Harvey, "Faster arithmetic for
// number-theoretic transforms", J. Symb. Comp. 2014), on eight limbs.
//
// The constant w is kept as the plain integer w in [0, r) together with
// w' = floor(w 2^256 / r).  With q about floor(x w' / 2^256), x w - q r is
// x w mod r up to a small multiple of r, and since it is known to lie in
// [0, 2r) only its low 256 bits are formed:
//     q  = columns 6..14 of x w' (column c: partial products x_i w'_j, i + j = c)
//     t  = low 256 bits of x w + q (2^256 - r)
// Bounds: w' loses less than 1, so x w'/2^256 loses less than x/2^256 < 1; the
// dropped columns 0..5 are below 7 * 2^224, so they cost q less than 2^-29; the
// floor costs less than 1.  Hence 0 <= x w - q r < (x/2^256 + 1 + 2^-29) r, below
// 2r for every x <= 2^256 - 2^228, in particular for loose x and differences
// of them (2r, and where it is below 2^256 4r, stay under 2^256 - 2^251).  If x is
// a value in Montgomery form, so is the result: w itself is not in it.
//
// Work on the heavy FMA datapath: 43 + 28 wide multiply-adds and 8 narrow ones for q
// and x w, and 15 and 6 (BLS12-381: r_1 = 2^32 - 1) or 21 and 7 (BLS12-377, BN254)
// for q (2^256 - r), whose lowest limb is 2^32 - 1 (r_0 = 1) or 2^28 - 1 (BN254) and
// takes shifts and a subtraction; against 112 to 120 wide ones of the Montgomery
// product.  About 135 instructions.  Measured in isolation as above: BLS12-381 80.8
// -> 95.9 G products/s, BN254 73.7 -> 90, BLS12-377 79.3 -> 95.  A wide multiply-add
// is issued every 4.5 cycles at best (the datapath holds it for 4), and every other
// instruction costs about 0.75 cycles beside it.  The price is 64 bytes a twiddle.
//
// The chains below are written on named registers: e_c and o_c hold the words
// of columns of even and odd index, a wide multiply-add's two words side by
// side, so that each pair becomes one instruction (see the Montgomery product).
// ZK_MUL starts a pair of words, ZK_MAD heads a carry chain, ZK_MADC continues
// it; a trailing LH: the pair is new, its addend only the carry in; L: only the
// low word of the product, into the last column.  ZK_CARRY stores a carry out.
#define ZK_MUL(l, h, a, b) "mul.wide.u32 t, " #a ", " #b ";\n\tmov.b64 {" #l ", " #h "}, t;\n\t"
#define ZK_MAD2_(c, l, h, a, b, x, y)                                     \
    "mad" c ".lo.cc.u32 " #l ", " #a ", " #b ", " x ";\n\t"              \
    "madc.hi.cc.u32 " #h ", " #a ", " #b ", " y ";\n\t"
#define ZK_MAD(l, h, a, b) ZK_MAD2_("", l, h, a, b, #l, #h)
#define ZK_MADC(l, h, a, b) ZK_MAD2_("c", l, h, a, b, #l, #h)
#define ZK_MADCLH(l, h, a, b) ZK_MAD2_("c", l, h, a, b, "0", "0")
#define ZK_MULL(l, a, b) "mul.lo.u32 " #l ", " #a ", " #b ";\n\t"
#define ZK_MADL(l, a, b) "mad.lo.u32 " #l ", " #a ", " #b ", " #l ";\n\t"
// (the carry by an add of its own: a narrow multiply-add with carry in holds the
// heavy datapath for four cycles, without it for two)
#define ZK_MADCL(l, a, b) "addc.u32 " #l ", " #l ", 0;\n\t" ZK_MADL(l, a, b)
#define ZK_CARRY(l) "addc.u32 " #l ", 0, 0;\n\t"
#define ZK_NAME8(n, a, b, c, d, e, f, g, h)                                              \
    ".reg .u32 " #n "<8>;\n\t"                                                           \
    "mov.u32 " #n "0, " a "; mov.u32 " #n "1, " b "; mov.u32 " #n "2, " c "; mov.u32 " #n "3, " d ";\n\t" \
    "mov.u32 " #n "4, " e "; mov.u32 " #n "5, " f "; mov.u32 " #n "6, " g "; mov.u32 " #n "7, " h ";\n\t"

// columns 6..14 of x y.  A row's carries out are single bits.  That of the odd
// columns is kept as the low word of the next row's top pair; that of the even
// columns (rows 2, 4, 6) as the high word of the same row's odd top pair, which
// is otherwise new: x_i y_7 < 2^64 - 2^33 + 2 leaves room for both.
#define ZK_ROWS_HIGH                                                                                   \
    ZK_MUL(e6, e7, x0, y6) ZK_MUL(o7, o8, x0, y7)                                                      \
    ZK_MAD(e6, e7, x1, y5) ZK_MADCLH(e8, e9, x1, y7) ZK_MAD(o7, o8, x1, y6) ZK_CARRY(o9)               \
    ZK_MAD(e6, e7, x2, y4) ZK_MADC(e8, e9, x2, y6) ZK_CARRY(o10)                                       \
    ZK_MAD(o7, o8, x2, y5) ZK_MADC(o9, o10, x2, y7)                                                    \
    ZK_MAD(e6, e7, x3, y3) ZK_MADC(e8, e9, x3, y5) ZK_MADCLH(e10, e11, x3, y7)                         \
    ZK_MAD(o7, o8, x3, y4) ZK_MADC(o9, o10, x3, y6) ZK_CARRY(o11)                                      \
    ZK_MAD(e6, e7, x4, y2) ZK_MADC(e8, e9, x4, y4) ZK_MADC(e10, e11, x4, y6) ZK_CARRY(o12)             \
    ZK_MAD(o7, o8, x4, y3) ZK_MADC(o9, o10, x4, y5) ZK_MADC(o11, o12, x4, y7)                          \
    ZK_MAD(e6, e7, x5, y1) ZK_MADC(e8, e9, x5, y3) ZK_MADC(e10, e11, x5, y5) ZK_MADCLH(e12, e13, x5, y7)\
    ZK_MAD(o7, o8, x5, y2) ZK_MADC(o9, o10, x5, y4) ZK_MADC(o11, o12, x5, y6) ZK_CARRY(o13)            \
    ZK_MAD(e6, e7, x6, y0) ZK_MADC(e8, e9, x6, y2) ZK_MADC(e10, e11, x6, y4) ZK_MADC(e12, e13, x6, y6) \
    ZK_CARRY(o14) ZK_MAD(o7, o8, x6, y1) ZK_MADC(o9, o10, x6, y3) ZK_MADC(o11, o12, x6, y5)            \
    ZK_MADC(o13, o14, x6, y7)                                                                          \
    ZK_MAD(e8, e9, x7, y1) ZK_MADC(e10, e11, x7, y3) ZK_MADC(e12, e13, x7, y5) ZK_MADCLH(e14, e15, x7, y7)\
    ZK_MAD(o7, o8, x7, y0) ZK_MADC(o9, o10, x7, y2) ZK_MADC(o11, o12, x7, y4) ZK_MADC(o13, o14, x7, y6)\
    ZK_CARRY(o15)
// columns 0..7 of x w: the first row's even columns, new or added to e, and the rest
#define ZK_ROW_LOW_NEW                                                                              \
    ZK_MUL(e0, e1, x0, w0) ZK_MUL(e2, e3, x0, w2) ZK_MUL(e4, e5, x0, w4) ZK_MUL(e6, e7, x0, w6)
#define ZK_ROW_LOW_ADD                                                                              \
    ZK_MAD(e0, e1, x0, w0) ZK_MADC(e2, e3, x0, w2) ZK_MADC(e4, e5, x0, w4) ZK_MADC(e6, e7, x0, w6)
#define ZK_ROWS_LOW                                                                                \
    ZK_MUL(o1, o2, x0, w1) ZK_MUL(o3, o4, x0, w3) ZK_MUL(o5, o6, x0, w5) ZK_MULL(o7, x0, w7)       \
    ZK_MAD(e2, e3, x1, w1) ZK_MADC(e4, e5, x1, w3) ZK_MADC(e6, e7, x1, w5)                         \
    ZK_MAD(o1, o2, x1, w0) ZK_MADC(o3, o4, x1, w2) ZK_MADC(o5, o6, x1, w4) ZK_MADCL(o7, x1, w6)    \
    ZK_MAD(e2, e3, x2, w0) ZK_MADC(e4, e5, x2, w2) ZK_MADC(e6, e7, x2, w4)                         \
    ZK_MAD(o3, o4, x2, w1) ZK_MADC(o5, o6, x2, w3) ZK_MADCL(o7, x2, w5)                            \
    ZK_MAD(e4, e5, x3, w1) ZK_MADC(e6, e7, x3, w3) ZK_MAD(o3, o4, x3, w0)                          \
    ZK_MADC(o5, o6, x3, w2) ZK_MADCL(o7, x3, w4)                                                   \
    ZK_MAD(e4, e5, x4, w0) ZK_MADC(e6, e7, x4, w2) ZK_MAD(o5, o6, x4, w1) ZK_MADCL(o7, x4, w3)     \
    ZK_MAD(e6, e7, x5, w1) ZK_MAD(o5, o6, x5, w0) ZK_MADCL(o7, x5, w2)                             \
    ZK_MAD(e6, e7, x6, w0) ZK_MADL(o7, x6, w1)                                                     \
    ZK_MADL(o7, x7, w0)
// columns 0..7 of q n added, n = n_j 2^(32 j) + ... + n_7 2^224 (j = 2, 1)
#define ZK_ROWS_N2                                                                                 \
    ZK_MAD(e2, e3, q0, n2) ZK_MADC(e4, e5, q0, n4) ZK_MADC(e6, e7, q0, n6)                         \
    ZK_MAD(o3, o4, q0, n3) ZK_MADC(o5, o6, q0, n5) ZK_MADCL(o7, q0, n7)                            \
    ZK_MAD(e4, e5, q1, n3) ZK_MADC(e6, e7, q1, n5) ZK_MAD(o3, o4, q1, n2)                          \
    ZK_MADC(o5, o6, q1, n4) ZK_MADCL(o7, q1, n6)                                                   \
    ZK_MAD(e4, e5, q2, n2) ZK_MADC(e6, e7, q2, n4) ZK_MAD(o5, o6, q2, n3) ZK_MADCL(o7, q2, n5)     \
    ZK_MAD(e6, e7, q3, n3) ZK_MAD(o5, o6, q3, n2) ZK_MADCL(o7, q3, n4)                             \
    ZK_MAD(e6, e7, q4, n2) ZK_MADL(o7, q4, n3)                                                     \
    ZK_MADL(o7, q5, n2)
#define ZK_ROWS_N1                                                                                 \
    ZK_MAD(e2, e3, q0, n2) ZK_MADC(e4, e5, q0, n4) ZK_MADC(e6, e7, q0, n6)                         \
    ZK_MAD(o1, o2, q0, n1) ZK_MADC(o3, o4, q0, n3) ZK_MADC(o5, o6, q0, n5) ZK_MADCL(o7, q0, n7)    \
    ZK_MAD(e2, e3, q1, n1) ZK_MADC(e4, e5, q1, n3) ZK_MADC(e6, e7, q1, n5)                         \
    ZK_MAD(o3, o4, q1, n2) ZK_MADC(o5, o6, q1, n4) ZK_MADCL(o7, q1, n6)                            \
    ZK_MAD(e4, e5, q2, n2) ZK_MADC(e6, e7, q2, n4) ZK_MAD(o3, o4, q2, n1)                          \
    ZK_MADC(o5, o6, q2, n3) ZK_MADCL(o7, q2, n5)                                                   \
    ZK_MAD(e4, e5, q3, n1) ZK_MADC(e6, e7, q3, n3) ZK_MAD(o5, o6, q3, n2) ZK_MADCL(o7, q3, n4)     \
    ZK_MAD(e6, e7, q4, n2) ZK_MAD(o5, o6, q4, n1) ZK_MADCL(o7, q4, n3)                             \
    ZK_MAD(e6, e7, q5, n1) ZK_MADL(o7, q5, n2)                                                     \
    ZK_MADL(o7, q6, n1)

// q = floor(x y / 2^256), less at most 1 (bound above)
__device__ __forceinline__ void mul_high(uint32_t q[8], const uint32_t x[8], const uint32_t y[8]) {
    asm("{\n\t.reg .u32 e<16>, o<16>;\n\t.reg .u64 t;\n\t"
        ZK_NAME8(x, "%8", "%9", "%10", "%11", "%12", "%13", "%14", "%15")
        ZK_NAME8(y, "%16", "%17", "%18", "%19", "%20", "%21", "%22", "%23")
        ZK_ROWS_HIGH
        "add.cc.u32 o7, o7, e7;\n\t"
        "addc.cc.u32 %0, o8, e8;\n\t"
        "addc.cc.u32 %1, o9, e9;\n\t"
        "addc.cc.u32 %2, o10, e10;\n\t"
        "addc.cc.u32 %3, o11, e11;\n\t"
        "addc.cc.u32 %4, o12, e12;\n\t"
        "addc.cc.u32 %5, o13, e13;\n\t"
        "addc.cc.u32 %6, o14, e14;\n\t"
        "addc.u32 %7, o15, e15;\n\t"
        "}"
        : "=&r"(q[0]), "=&r"(q[1]), "=&r"(q[2]), "=&r"(q[3]), "=&r"(q[4]),
          "=&r"(q[5]), "=&r"(q[6]), "=&r"(q[7])
        : "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3]), "r"(x[4]), "r"(x[5]), "r"(x[6]), "r"(x[7]),
          "r"(y[0]), "r"(y[1]), "r"(y[2]), "r"(y[3]), "r"(y[4]), "r"(y[5]), "r"(y[6]), "r"(y[7]));
}

// low 256 bits of x w
__device__ __forceinline__ void mul_low(uint32_t t[8], const uint32_t x[8], const uint32_t w[8]) {
    asm("{\n\t.reg .u32 e<16>, o<16>;\n\t.reg .u64 t;\n\t"
        ZK_NAME8(x, "%8", "%9", "%10", "%11", "%12", "%13", "%14", "%15")
        ZK_NAME8(w, "%16", "%17", "%18", "%19", "%20", "%21", "%22", "%23")
        ZK_ROW_LOW_NEW ZK_ROWS_LOW
        "mov.u32 %0, e0;\n\t"
        "add.cc.u32 %1, e1, o1;\n\taddc.cc.u32 %2, e2, o2;\n\t"
        "addc.cc.u32 %3, e3, o3;\n\taddc.cc.u32 %4, e4, o4;\n\t"
        "addc.cc.u32 %5, e5, o5;\n\taddc.cc.u32 %6, e6, o6;\n\taddc.u32 %7, e7, o7;\n\t}"
        : "=&r"(t[0]), "=&r"(t[1]), "=&r"(t[2]), "=&r"(t[3]), "=&r"(t[4]), "=&r"(t[5]),
          "=&r"(t[6]), "=&r"(t[7])
        : "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3]), "r"(x[4]), "r"(x[5]), "r"(x[6]), "r"(x[7]),
          "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]));
}

// t = x w + q (2^256 - r) mod 2^256
template <class F>
__device__ __forceinline__ void mul_low_fold(uint32_t t[8], const uint32_t x[8], const uint32_t w[8],
                                             const uint32_t q[8]) {
#define ZK_LOW_HEAD                                                                \
    "{\n\t.reg .u32 e<16>, o<16>;\n\t.reg .u64 t;\n\t"                           \
    ZK_NAME8(x, "%8", "%9", "%10", "%11", "%12", "%13", "%14", "%15")              \
    ZK_NAME8(w, "%16", "%17", "%18", "%19", "%20", "%21", "%22", "%23")            \
    ZK_NAME8(q, "%24", "%25", "%26", "%27", "%28", "%29", "%30", "%31")            \
    ZK_NAME8(n, "%32", "%33", "%34", "%35", "%36", "%37", "%38", "%39")
#define ZK_LOW_Q  /* q (2^32 - 1) = (q << 32) - q */                               \
    "sub.cc.u32 e0, 0, q0;\n\tsubc.cc.u32 e1, q0, q1;\n\t"                       \
    "subc.cc.u32 e2, q1, q2;\n\tsubc.cc.u32 e3, q2, q3;\n\t"                     \
    "subc.cc.u32 e4, q3, q4;\n\tsubc.cc.u32 e5, q4, q5;\n\t"                     \
    "subc.cc.u32 e6, q5, q6;\n\tsubc.u32 e7, q6, q7;\n\t"
#define ZK_LOW_Q28  /* q (2^28 - 1) = (q << 28) - q */                              \
    ".reg .u32 s<8>;\n\t"                                                          \
    "shl.b32 s0, q0, 28;\n\tshf.l.wrap.b32 s1, q0, q1, 28;\n\t"                   \
    "shf.l.wrap.b32 s2, q1, q2, 28;\n\tshf.l.wrap.b32 s3, q2, q3, 28;\n\t"        \
    "shf.l.wrap.b32 s4, q3, q4, 28;\n\tshf.l.wrap.b32 s5, q4, q5, 28;\n\t"        \
    "shf.l.wrap.b32 s6, q5, q6, 28;\n\tshf.l.wrap.b32 s7, q6, q7, 28;\n\t"        \
    "sub.cc.u32 e0, s0, q0;\n\tsubc.cc.u32 e1, s1, q1;\n\t"                      \
    "subc.cc.u32 e2, s2, q2;\n\tsubc.cc.u32 e3, s3, q3;\n\t"                     \
    "subc.cc.u32 e4, s4, q4;\n\tsubc.cc.u32 e5, s5, q5;\n\t"                     \
    "subc.cc.u32 e6, s6, q6;\n\tsubc.u32 e7, s7, q7;\n\t"
#define ZK_LOW_TAIL                                                                \
    "mov.u32 %0, e0;\n\t"                                                          \
    "add.cc.u32 %1, e1, o1;\n\taddc.cc.u32 %2, e2, o2;\n\t"                      \
    "addc.cc.u32 %3, e3, o3;\n\taddc.cc.u32 %4, e4, o4;\n\t"                     \
    "addc.cc.u32 %5, e5, o5;\n\taddc.cc.u32 %6, e6, o6;\n\taddc.u32 %7, e7, o7;\n\t}"
#define ZK_LOW_OPERANDS(n0, n1)                                                                 \
    : "=&r"(t[0]), "=&r"(t[1]), "=&r"(t[2]), "=&r"(t[3]), "=&r"(t[4]), "=&r"(t[5]), "=&r"(t[6]), "=&r"(t[7])            \
    : "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3]), "r"(x[4]), "r"(x[5]), "r"(x[6]), "r"(x[7]),                \
      "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]),                \
      "r"(q[0]), "r"(q[1]), "r"(q[2]), "r"(q[3]), "r"(q[4]), "r"(q[5]), "r"(q[6]), "r"(q[7]),                \
      "n"(n0), "n"(n1), "n"(~F::P2), "n"(~F::P3), "n"(~F::P4), "n"(~F::P5), "n"(~F::P6), "n"(~F::P7)
    if constexpr (F::P0 == 1u && F::P1 == 0xffffffffu) {
        asm(ZK_LOW_HEAD ZK_LOW_Q ZK_ROW_LOW_ADD ZK_ROWS_LOW ZK_ROWS_N2 ZK_LOW_TAIL
            ZK_LOW_OPERANDS(0, 0));
    } else if constexpr (F::P0 == 1u) {
        asm(ZK_LOW_HEAD ZK_LOW_Q ZK_ROW_LOW_ADD ZK_ROWS_LOW ZK_ROWS_N1 ZK_LOW_TAIL
            ZK_LOW_OPERANDS(0, ~F::P1));
    } else if constexpr (F::P0 == 0xf0000001u) {
        asm(ZK_LOW_HEAD ZK_LOW_Q28 ZK_ROW_LOW_ADD ZK_ROWS_LOW ZK_ROWS_N1 ZK_LOW_TAIL
            ZK_LOW_OPERANDS(0, ~F::P1));
    } else {  // any other lowest limb
        const uint32_t n[8] = {0u - F::P0, ~F::P1, ~F::P2, ~F::P3, ~F::P4, ~F::P5, ~F::P6, ~F::P7};
        uint32_t a[8], b[8];
        mul_low(a, x, w);
        mul_low(b, q, n);
        uint64_t c = 0;
#pragma unroll
        for (int i = 0; i < 8; i++) {
            c += uint64_t(a[i]) + b[i];
            t[i] = uint32_t(c);
            c >>= 32;
        }
    }
#undef ZK_LOW_HEAD
#undef ZK_LOW_Q
#undef ZK_LOW_Q28
#undef ZK_LOW_TAIL
#undef ZK_LOW_OPERANDS
}

// A constant factor and its quotient (both 256-bit integers), as the twiddle
// tables hold them: 64 bytes.
struct Factor {
    uint32_t w[8], wq[8];
};

// r = x f mod p, loose (in [0, 2p)), for any x <= 2^256 - 2^228
template <class F>
__device__ __forceinline__ void mul_factor(uint32_t r[8], const uint32_t x[8], const Factor &f) {
    uint32_t q[8], t[8];
    mul_high(q, x, f.wq);
    mul_low_fold<F>(t, x, f.w, q);
#pragma unroll
    for (int i = 0; i < 8; i++) r[i] = t[i];
}

// The factor of a constant given in Montgomery form, m = w R mod r, R = 2^256:
// w R = floor(w R / r) r + m, so the quotient is -m r^-1 mod R (ninv = -r^-1
// mod R), and w is m without its R.
template <class F>
__device__ __forceinline__ void make_factor(Factor &f, const uint32_t m[8], const uint32_t ninv[8]) {
    const uint32_t one[8] = {1, 0, 0, 0, 0, 0, 0, 0};
    mul<F>(f.w, m, one);
    mul_low(f.wq, m, ninv);
}

// ---------------------------------------------------------------------------
// element load/store: 32 bytes as two 16-byte vectors
__device__ __forceinline__ void ldg_elem(uint32_t x[8], const uint4 *p) {
    uint4 lo = __ldg(p), hi = __ldg(p + 1);
    x[0] = lo.x; x[1] = lo.y; x[2] = lo.z; x[3] = lo.w;
    x[4] = hi.x; x[5] = hi.y; x[6] = hi.z; x[7] = hi.w;
}

// one 32-byte load a lane: a whole sector in one request
#define ZK_LD8(hint, x, p)                                                                      \
    asm("ld.global.nc" hint ".v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"                   \
        : "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]), "=r"(x[5]), "=r"(x[6]),   \
          "=r"(x[7])                                                                            \
        : "l"(p))

// a factor of a small table, which L1 keeps
__device__ __forceinline__ void ldg_factor(Factor &f, const uint4 *p) {
    ZK_LD8("", f.w, p);
    ZK_LD8("", f.wq, p + 2);
}

// a factor that is read once
__device__ __forceinline__ void ldg_factor_stream(Factor &f, const uint4 *p) {
    ZK_LD8(".L1::no_allocate", f.w, p);
    ZK_LD8(".L1::no_allocate", f.wq, p + 2);
}

// L2-coherent load (bypasses L1) for data another block wrote in this launch
__device__ __forceinline__ void ld_elem_cg(uint32_t x[8], const uint4 *p) {
    uint4 lo = __ldcg(p), hi = __ldcg(p + 1);
    x[0] = lo.x; x[1] = lo.y; x[2] = lo.z; x[3] = lo.w;
    x[4] = hi.x; x[5] = hi.y; x[6] = hi.z; x[7] = hi.w;
}

__device__ __forceinline__ void st_elem(uint4 *p, const uint32_t x[8]) {
    p[0] = make_uint4(x[0], x[1], x[2], x[3]);
    p[1] = make_uint4(x[4], x[5], x[6], x[7]);
}

// one 32-byte store a lane: a whole sector in one request
__device__ __forceinline__ void st_elem8(uint4 *p, const uint32_t x[8]) {
    asm volatile("st.global.v8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};" ::"r"(x[0]), "r"(x[1]),
                 "r"(x[2]), "r"(x[3]), "r"(x[4]), "r"(x[5]), "r"(x[6]), "r"(x[7]), "l"(p)
                 : "memory");
}

__device__ __forceinline__ void st_factor(uint4 *p, const Factor &f) {
    st_elem(p, f.w);
    st_elem(p + 2, f.wq);
}

}  // namespace zkntt
