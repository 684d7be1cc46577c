// ntt_pass.cuh -- one pass of the multi-pass NTT for sm_103a.
//
// Decomposition (the four-step identity applied recursively; Section II-B of
// the paper notes that a block NTT is bounded by shared memory and that groups
// of stages may be run together):
//   n = 2^L is split into digits k_1 + ... + k_p = L (top digit first).  Pass i
//   treats the vector as columns: for fixed (hi, lo) the N = 2^K elements at
//       q = (hi * N + d) * 2^lo_bits + lo,   d = 0..N-1
//   form one sub-transform.  It is computed by decimation-in-frequency stages
//   (output position d then holds frequency rev(d)) and, for every pass but the
//   last, multiplied by the inter-pass twiddle w_{n_i}^(lo * rev(d)),
//   n_i = N * 2^lo_bits.  After the last pass the value at position q is
//   output bitrev_L(q); the last pass writes it there directly, so the result
//   is in natural order without a permutation pass.
//
// Inside a thread block: a tile of C columns x N rows (C consecutive lo values,
// or for the last pass C blocks whose bit-reversed indices are consecutive, so
// the scattered writes form C*32-byte runs) is copied into shared memory with
// cp.async.  Two stages at a time then run as radix-4 steps: a thread loads the
// four rows of a group, takes their four butterflies (x, y) -> (x + y, (x - y) w)
// in registers and writes them back (a radix-2 step comes first when K is odd).
// The last step, rows d0..d0+3 with one product by w_4, is followed by the
// element's output factor and the store to global memory.  Tiles with more than
// one thread per four elements (small transforms, where warps in flight count)
// take the stages one by one, one butterfly a thread.
// A difference that only feeds a product is formed as x + 2r - y, below 4r, without a
// correction where 4r < 2^256 (BN254, BLS12-377), else corrected by 2r (BLS12-381): the
// product takes any x up to 2^256 - 2^228.
// Digits of 5 to 10 bits in the usual tile width have kernels compiled for them;
// every other digit and width is served by kernels whose sizes are runtime values.
//
// What bounds it: the heavy FMA datapath and the issue of everything beside it.  A
// pass of 8 bits makes 3.25 products an element in its stages and one for the output
// factor, 133 instructions each, 86 of them wide multiply-adds that hold the datapath
// for four cycles.  At 2^24 (three passes of 8 bits, 2590 us on GB300; 4537 with
// Montgomery products and radix-2 steps) the datapath is busy 67 to 72% of the
// cycles.  Memory costs little: with neither vectors nor inter-pass factors read, the
// first pass takes 926 us instead of 985.
//
// Values are residues in [0, 2r) throughout; the last pass brings its outputs
// below r.
//
// Shared memory holds elements in groups of eight: eight low 16-byte halves,
// then the eight high ones.  The slot of (column c, row d) is c*N + (d ^ s), with
// s in the low three bits a linear function of bits 3 and 4 of d and of c
// (smem_unit), chosen so that the eight lanes of an access fall into different
// bank groups in every pattern: copies with columns or rows fastest, steps at
// distance 4 and above, and the last step on rows 4 g + i with columns fastest.
//
// Per-element factors (one product each, only when present), all held as
// (w, quotient) pairs of 64 bytes for mul_factor:
//   pre[d]          first pass, on input row d (coset forward shift powers)
//   pw_b, pw_c      first pass, x <- x * pw_b[q] - pw_c[q] (Groth16 pointwise;
//                   these are vectors of elements)
//   tw[d][lo]       inter-pass twiddles, precomputed, or applied on the fly as
//                   the factors w_hi, w_lo of the split exponent and optional
//                   per-column (fl) and per-row (fd) ones
//   post[d]         last pass, on output position d (inverse / coset scales)
#pragma once
#include <cstdint>

#include "field.cuh"

namespace zkntt {

struct PassArgs {
    const uint4 *in;
    uint4 *out;
    const uint4 *w_stage; // the factors w_N^e, e < N/2, as they lie in shared memory (tab_slot)
    const uint4 *tw;      // precomputed inter-pass factors [N][2^lo_bits] (row-major by d)
    const uint4 *w_hi;    // on-the-fly: w^((e >> split_bits) << split_bits)
    const uint4 *w_lo;    // on-the-fly: w^(e & (2^split_bits - 1)) (times any folded scalar)
    const uint4 *fl;      // on-the-fly: per-column factor (may be null)
    const uint4 *fd;      // on-the-fly: per-row factor (may be null)
    const uint4 *pre;     // first pass input scale by row (may be null)
    const uint4 *post;    // last pass output scale by position (may be null)
    const uint4 *pw_b;    // fused Groth16 pointwise: x <- x * pw_b[q] - pw_c[q] on load
    const uint4 *pw_c;    //   (first pass only; both null otherwise)
    uint32_t K;           // log2 of the sub-transform size N
    uint32_t lo_bits;     // log2 of this digit's stride
    uint32_t hi_bits;     // bits above this digit
    uint32_t tw_bits;     // on-the-fly: log2 n_i (exponents are taken mod n_i)
    uint32_t split_bits;  // on-the-fly: width of the low exponent table
    uint32_t log_cols;    // log2 C
    uint32_t last;        // 1: last pass (bit-reversed scatter to natural order)
    uint32_t otf;         // 1: inter-pass twiddles on the fly
    uint32_t num_tiles;   // tiles in this pass
};

// The vectors of a launch: up to three of one plan, whose tiles follow each other
// (three independent transforms fill the GPU where one does not).
constexpr int PASS_VECTORS = 3;
struct PassVectors {
    const uint4 *in[PASS_VECTORS];
    uint4 *out[PASS_VECTORS];
    uint32_t tiles;  // tiles of one vector
};

// the tile within its vector v
__device__ __forceinline__ uint32_t vector_tile(const PassVectors &vec, uint32_t tile, uint32_t &v) {
    for (v = 0; tile >= vec.tiles; v++) tile -= vec.tiles;
    return tile;
}

__device__ __forceinline__ uint32_t brev_bits(uint32_t x, uint32_t bits) {
    return bits == 0 ? 0u : (__brev(x) >> (32 - bits));
}

// Place of slot s among the 16-byte units of shared memory: the low half, and
// the high one HALF units on.
constexpr uint32_t HALF = 8;
__host__ __device__ __forceinline__ uint32_t slot_unit(uint32_t s) {
    return ((s & ~7u) << 1) | (s & 7u);
}

// units of a tile of CN elements
__host__ __device__ constexpr uint32_t tile_units(uint32_t CN) { return CN < 8 ? 16u : 2 * CN; }

// Row part of an element's unit (K >= 3): d with its low three bits xor 5 for
// bit 3 and xor 6 for bit 4 (0, 5, 6, 3 by the two bits).  Linear over xor, so
// the rows of a group at distances that are powers of two have units at xor
// distances.
__device__ __forceinline__ uint32_t row_unit(uint32_t d) {
    return slot_unit(d ^ ((0x3650u >> ((d >> 1) & 12u)) & 7u));
}

// column part of an element's unit, to be xor-ed to the row's
__device__ __forceinline__ uint32_t col_unit(uint32_t c, uint32_t K, uint32_t lc) {
    if (K < 3) return slot_unit(c << K);
    const uint32_t s = lc == 3 ? c : lc == 2 ? ((c & 1u) << 1) ^ ((c >> 1) * 5u) : c * 6u;
    return (c << (K + 1)) | s;
}

// unit of element (column c, row d)
__device__ __forceinline__ uint32_t smem_unit(uint32_t c, uint32_t d, uint32_t K, uint32_t lc) {
    return K < 3 ? slot_unit((c << K) + d) : col_unit(c, K, lc) ^ row_unit(d);
}

__device__ __forceinline__ void cp_async16(void *smem_dst, const void *gmem_src) {
    uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(smem_dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem_src) : "memory");
}

// the same with the shared-memory destination as a 32-bit shared address
__device__ __forceinline__ void cp_async16_sa(uint32_t s, const void *gmem_src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(gmem_src) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
}

__device__ __forceinline__ void lds_elem(uint32_t x[8], const uint4 *buf, uint32_t unit) {
    const uint4 v0 = buf[unit], v1 = buf[unit + HALF];
    x[0] = v0.x; x[1] = v0.y; x[2] = v0.z; x[3] = v0.w;
    x[4] = v1.x; x[5] = v1.y; x[6] = v1.z; x[7] = v1.w;
}

__device__ __forceinline__ void sts_elem(uint4 *buf, uint32_t unit, const uint32_t x[8]) {
    buf[unit] = make_uint4(x[0], x[1], x[2], x[3]);
    buf[unit + HALF] = make_uint4(x[4], x[5], x[6], x[7]);
}

// Global index of tile element (row d, column cc) before (src) and after (dst)
// the pass.
__device__ __forceinline__ size_t tile_src(const PassArgs &a, uint32_t tile, uint32_t d,
                                           uint32_t cc) {
    if (!a.last) {
        const uint32_t lo_tiles_bits = a.lo_bits - a.log_cols;
        const size_t hi = tile >> lo_tiles_bits;
        const size_t lo0 = size_t(tile & ((1u << lo_tiles_bits) - 1u)) << a.log_cols;
        return ((hi << a.K | d) << a.lo_bits) + lo0 + cc;
    }
    const uint32_t b = (tile << a.log_cols) + cc;
    return (size_t(brev_bits(b, a.hi_bits)) << a.K) + d;
}

// The factors of row position d in column cc on the way out, formed on the fly:
// a null p[k] ends the list.
__device__ __forceinline__ void otf_factors(const uint4 *p[4], const PassArgs &a, uint32_t tile,
                                            uint32_t d, uint32_t cc) {
    const uint32_t lo_tiles_bits = a.lo_bits - a.log_cols;
    const uint32_t lo = ((tile & ((1u << lo_tiles_bits) - 1u)) << a.log_cols) + cc;
    // lo < 2^lo_bits and rev(d) < 2^K, so e < 2^tw_bits = n_i: no reduction
    // (and no overflow: tw_bits <= 32)
    const uint32_t e = lo * brev_bits(d, a.K);
    p[0] = a.w_hi + 4 * size_t(e >> a.split_bits);
    p[1] = a.w_lo + 4 * size_t(e & ((1u << a.split_bits) - 1u));
    p[2] = p[3] = nullptr;
    if (a.fl) p[2] = a.fl + 4 * size_t(lo);
    if (a.fd) (a.fl ? p[3] : p[2]) = a.fd + 4 * size_t(d);
}

// Where a thread's rows d0 .. d0 + R - 1 of column cc go (R = 4, or 2 when
// N = 2; d0 a multiple of R), and their factors: row d0 + i, in order of i in a
// strided pass, of rev(i) in the last, is `step` elements on from the one before;
// its factor (null: none, or on the fly) is `fstep` units on in order of i.
struct OutRows {
    uint4 *out;
    size_t step, fstep;
    const uint4 *f;
};
template <int R>
__device__ __forceinline__ OutRows out_rows(const PassArgs &a, uint32_t tile, uint32_t d0,
                                            uint32_t cc) {
    OutRows o;
    if (a.last) {
        o.out = a.out + 2 * ((size_t(brev_bits(d0, a.K)) << a.hi_bits) +
                             (size_t(tile) << a.log_cols) + cc);
        o.step = size_t(1) << (a.K - (R == 4 ? 2 : 1) + a.hi_bits);
        o.f = a.post ? a.post + 4 * size_t(d0) : nullptr;
        o.fstep = 4;
    } else {
        const uint32_t lo_tiles_bits = a.lo_bits - a.log_cols;
        const uint32_t lo = ((tile & ((1u << lo_tiles_bits) - 1u)) << a.log_cols) + cc;
        const size_t hi = tile >> lo_tiles_bits;
        o.out = a.out + 2 * (((hi << a.K | d0) << a.lo_bits) + lo);
        o.step = size_t(1) << a.lo_bits;
        o.f = a.otf ? nullptr : a.tw + 4 * ((size_t(d0) << a.lo_bits) + lo);
        o.fstep = 4 * o.step;
    }
    return o;
}

// x times the factors of row d in column cc formed on the fly
template <class F>
__device__ __forceinline__ void otf_scale(uint32_t x[8], const PassArgs &a, uint32_t tile, uint32_t d,
                                          uint32_t cc) {
    const uint4 *p[4];
    otf_factors(p, a, tile, d, cc);
#pragma unroll 1
    while (p[0]) {
        Factor v;
        ldg_factor(v, p[0]);
        mul_factor<F>(x, x, v);
        p[0] = p[1];
        p[1] = p[2];
        p[2] = p[3];
        p[3] = nullptr;
    }
}

// the factor at f of the output's table (an entry of the big one is read once: it
// takes no place in L1)
__device__ __forceinline__ void ldg_out_factor(Factor &v, const PassArgs &a, const uint4 *f) {
    if (a.last) ldg_factor(v, f);
    else ldg_factor_stream(v, f);
}

// The rows at units u0 ^ i, times their output factors, to global memory: a
// loop with one product in the code (unrolled, the kernels outgrow the
// instruction cache).  The table's factor of the next row is read into the
// registers of the present one as soon as the product is done with them: its
// quotient during the second half of the product, its value during the store and
// the first half of the next.  AHEAD: factors on the fly too (the batch kernel, with
// 80 registers, reads those when it needs them).
template <class F, int R, bool AHEAD>
__device__ __forceinline__ void scale_and_store(const PassArgs &a, const uint4 *buf, uint32_t u0,
                                                const OutRows &o, uint32_t tile, uint32_t d0,
                                                uint32_t cc) {
    if (o.f) {
        Factor v;
        ldg_out_factor(v, a, o.f);
        const uint4 *f = o.f;
#pragma unroll 1
        for (uint32_t i = 0; i < R; i++) {
            uint32_t x[8], q[8];
            lds_elem(x, buf, u0 ^ i);
            mul_high(q, x, v.wq);
            if (i + 1 < R) f += o.fstep;
            if (a.last) ZK_LD8("", v.wq, f + 2);
            else ZK_LD8(".L1::no_allocate", v.wq, f + 2);
            mul_low_fold<F>(x, x, v.w, q);
            if (a.last) ZK_LD8("", v.w, f);
            else ZK_LD8(".L1::no_allocate", v.w, f);
            uint32_t r = i;
            if (a.last) {
                reduce_once<F>(x);
                if (R == 4) r = ((i & 1u) << 1) | (i >> 1);
            }
            st_elem8(o.out + 2 * r * o.step, x);
        }
        return;
    }
    if (!AHEAD) {
#pragma unroll 1
        for (uint32_t i = 0; i < R; i++) {
            uint32_t x[8];
            lds_elem(x, buf, u0 ^ i);
            otf_scale<F>(x, a, tile, d0 + i, cc);
            st_elem8(o.out + 2 * i * o.step, x);
        }
        return;
    }
    // on the fly: the two to four factors of each row one after the other, read ahead
    // in the same way (2^22, BN254: 783 -> 758 us)
    const uint32_t lo_tiles_bits = a.lo_bits - a.log_cols;
    const uint32_t lo = ((tile & ((1u << lo_tiles_bits) - 1u)) << a.log_cols) + cc;
    // lo < 2^lo_bits and rev(d) < 2^K, so the exponent is below 2^tw_bits = n_i: no
    // reduction (and no overflow: tw_bits <= 32); row i adds rev(i) parts of it
    const uint32_t e0 = lo * brev_bits(d0, a.K), part = lo << (a.K - (R == 4 ? 2 : 1));
    const uint32_t factors = 2 + (a.fl != nullptr) + (a.fd != nullptr);
    auto factor = [&](uint32_t i, uint32_t j) -> const uint4 * {
        const uint32_t e = e0 + part * (R == 4 ? ((i & 1u) << 1) | (i >> 1) : i);
        if (j == 0) return a.w_hi + 4 * size_t(e >> a.split_bits);
        if (j == 1) return a.w_lo + 4 * size_t(e & ((1u << a.split_bits) - 1u));
        return j == 2 && a.fl ? a.fl + 4 * size_t(lo) : a.fd + 4 * size_t(d0 + i);
    };
    Factor v;
    ldg_factor(v, factor(0, 0));
    uint32_t x[8], q[8];
    lds_elem(x, buf, u0);
#pragma unroll 1
    for (uint32_t i = 0, j = 0;;) {
        mul_high(q, x, v.wq);
        const bool row_done = j + 1 == factors, done = row_done && i + 1 == R;
        const uint4 *f = done ? a.w_hi : row_done ? factor(i + 1, 0) : factor(i, j + 1);
        ZK_LD8("", v.wq, f + 2);
        mul_low_fold<F>(x, x, v.w, q);
        ZK_LD8("", v.w, f);
        j++;
        if (!row_done) continue;
        st_elem8(o.out + 2 * i * o.step, x);
        if (done) break;
        i++;
        j = 0;
        lds_elem(x, buf, u0 ^ i);
    }
}

// Issue (without waiting) the 16-byte copies of one tile into shared memory:
// 8 lanes copy the low halves of 8 elements, the next 8 lanes their high
// halves (tiles under 8 elements: element-major); columns fastest for strided
// passes, rows fastest for the last.
__device__ __forceinline__ void issue_tile_load(const PassArgs &a, uint4 *buf, uint32_t tile,
                                                uint32_t nthreads) {
    const uint32_t K = a.K, lc = a.log_cols;
    const uint32_t N = 1u << K, C = 1u << lc, CN = C << K;
    const uint32_t tid = threadIdx.x;
    if (tid >= nthreads) return;
    if (CN >= 64 && (nthreads & 15u) == 0 && (nthreads & (nthreads - 1u)) == 0 && nthreads <= 2 * CN) {
        // Every thread makes 2 C N / nthreads copies of one half (the lane's
        // bit 3) of elements e0, e0 + E, e0 + 2E, ... (E = nthreads / 2): rows
        // at a power-of-two step in one column, so the source steps by a fixed
        // stride and the units lie at xor distances (the same for all threads).
        const uint32_t half = (tid >> 3) & 1u;
        const uint32_t e0 = (tid & 7u) | ((tid >> 4) << 3);
        // (four copies at a time: one per four elements makes eight or more)
        const uint32_t E = nthreads >> 1, iters = (2 * CN) / nthreads;
        const uint32_t sbase = static_cast<uint32_t>(__cvta_generic_to_shared(buf + half * HALF));
        if (!a.last && iters >= 4) {
            const uint32_t cc = e0 & (C - 1), dstep = E >> lc, d = e0 >> lc;
            const uint4 *src = a.in + 2 * tile_src(a, tile, d, cc) + half;
            const size_t sstep = size_t(2 * dstep) << a.lo_bits;
            const uint32_t u1 = row_unit(dstep), u2 = row_unit(2 * dstep);
            const uint32_t u = smem_unit(cc, d, K, lc);
#pragma unroll 1
            for (uint32_t k = 0; k < iters; k += 4, src += 4 * sstep) {
                const uint32_t v = u ^ row_unit(k * dstep);
                cp_async16_sa(sbase + 16u * v, src);
                cp_async16_sa(sbase + 16u * (v ^ u1), src + sstep);
                cp_async16_sa(sbase + 16u * (v ^ u2), src + 2 * sstep);
                cp_async16_sa(sbase + 16u * (v ^ u1 ^ u2), src + 3 * sstep);
            }
        } else if (a.last && 4 * E <= N) {
            // last pass, rows fastest: N / E copies in one column (rows e0,
            // e0 + E, ...; e0 < E), then the next column
            const uint32_t per = N / E;
            const uint32_t u1 = row_unit(E), u2 = row_unit(2 * E);
#pragma unroll 1
            for (uint32_t cc = 0; cc < C; cc++) {
                const uint4 *src = a.in + 2 * tile_src(a, tile, e0, cc) + half;
                const uint32_t u = smem_unit(cc, e0, K, lc);
#pragma unroll 1
                for (uint32_t j = 0; j < per; j += 4, src += 8 * E) {
                    const uint32_t v = u ^ row_unit(j * E);
                    cp_async16_sa(sbase + 16u * v, src);
                    cp_async16_sa(sbase + 16u * (v ^ u1), src + 2 * E);
                    cp_async16_sa(sbase + 16u * (v ^ u2), src + 4 * E);
                    cp_async16_sa(sbase + 16u * (v ^ u1 ^ u2), src + 6 * E);
                }
            }
        } else {
            uint32_t e = e0;
#pragma unroll 1
            for (uint32_t k = 0; k < iters; k++, e += E) {
                const uint32_t d = e & (N - 1), cc = e >> K;
                cp_async16_sa(sbase + 16u * smem_unit(cc, d, K, lc),
                              a.in + 2 * tile_src(a, tile, d, cc) + half);
            }
        }
        return;
    }
    const bool grouped = CN >= 8;
#pragma unroll 1
    for (uint32_t u = tid; u < 2 * CN; u += nthreads) {
        const uint32_t e = grouped ? ((u & 7u) | ((u >> 4) << 3)) : (u >> 1);
        const uint32_t half = grouped ? ((u >> 3) & 1u) : (u & 1u);
        uint32_t d, cc;
        if (a.last) { d = e & (N - 1); cc = e >> K; }
        else        { cc = e & (C - 1); d = e >> lc; }
        const size_t g = tile_src(a, tile, d, cc);
        cp_async16(buf + smem_unit(cc, d, K, lc) + half * HALF, a.in + 2 * g + half);
    }
}

// The sub-transform's twiddles in shared memory: the N/2 factors w_N^e in groups
// of eight, each group as four rows of eight 16-byte quarters.  Entry e's slot
// is e with its low three bits xor its higher ones in threes, so eight entries at
// any power-of-two stride lie in different bank groups.  (Read from global
// memory instead, they missed L1 half the time and were two thirds of the
// load/store wavefronts.)  tab_unit is linear over xor.
__host__ __device__ __forceinline__ uint32_t tab_unit(uint32_t e) {
    return ((e & ~7u) << 2) | ((e ^ (e >> 3) ^ (e >> 6) ^ (e >> 9)) & 7u);
}

// entries of the table of a 2^K-point sub-transform (at least one group)
__host__ __device__ constexpr uint32_t tab_entries(uint32_t K) { return K > 3 ? 1u << (K - 1) : 8u; }

// issue (without waiting) the copies of the table, which is laid out in global
// memory as in shared memory
__device__ __forceinline__ void issue_table_load(const PassArgs &a, uint4 *tab, uint32_t nthreads) {
    const uint32_t units = 4 * tab_entries(a.K);
#pragma unroll 1
    for (uint32_t u = threadIdx.x; u < units; u += nthreads) cp_async16(tab + u, a.w_stage + u);
}

// the factor at unit u of the table
__device__ __forceinline__ void lds_factor(Factor &f, const uint4 *tab, uint32_t u) {
    lds_elem(f.w, tab, u);
    lds_elem(f.wq, tab, u + 16);
}

// How a tile's stages run: two at a time, four elements a thread (radix 4), or
// one by one, one butterfly a thread (radix 2); or either by the thread count.
enum Steps { RADIX4 = 1, RADIX2 = 2, EITHER = 3 };

// x <- x + y, t = x - y (for the product): a butterfly but for its product
template <class F>
__device__ __forceinline__ void sum_diff(uint32_t x[8], uint32_t t[8], const uint32_t y[8]) {
    diff_loose<F>(t, x, y);
    add_loose<F>(x, x, y);
}

// x <- x + y, y <- x - y: a butterfly with twiddle 1
template <class F>
__device__ __forceinline__ void sum_sub(uint32_t x[8], uint32_t y[8]) {
    uint32_t t[8];
    sub_loose<F>(t, x, y);
    add_loose<F>(x, x, y);
#pragma unroll
    for (int k = 0; k < 8; k++) y[k] = t[k];
}

// two products side by side
template <class F>
__device__ __forceinline__ void mul_factor2(uint32_t r[8], const uint32_t x[8], const Factor &f,
                                            uint32_t s[8], const uint32_t y[8], const Factor &g) {
    uint32_t p[8], q[8];
    mul_high(p, x, f.wq);
    mul_high(q, y, g.wq);
    mul_low_fold<F>(r, x, f.w, p);
    mul_low_fold<F>(s, y, g.w, q);
}

// One stage, pairs at distance h, one butterfly after the other.
template <class F>
__device__ __forceinline__ void radix2_stage(uint4 *buf, const uint4 *tab, uint32_t h,
                                             uint32_t K, uint32_t lc, uint32_t tid,
                                             uint32_t nthreads) {
    const uint32_t N = 1u << K, CN = N << lc, step = row_unit(h);
    const uint32_t shift = K - 1 - (31 - __clz(h));  // entry j 2^stage
    for (uint32_t bk = tid; tid < nthreads && bk < (CN >> 1); bk += nthreads) {
        const uint32_t cc = bk >> (K - 1), b = bk & ((N >> 1) - 1), j = b & (h - 1);
        const uint32_t s0 = smem_unit(cc, ((b ^ j) << 1) | j, K, lc), s1 = s0 ^ step;
        uint32_t x[8], y[8], t[8];
        Factor w;
        lds_elem(x, buf, s0);
        lds_elem(y, buf, s1);
        lds_factor(w, tab, tab_unit(j << shift));
        sum_diff<F>(x, t, y);
        mul_factor<F>(t, t, w);
        sts_elem(buf, s0, x);
        sts_elem(buf, s1, t);
    }
}

// The stages of a tile one by one, one butterfly a thread and stage, and its
// output: for transforms with few warps in flight, whose time is the chain of
// products of one thread.  A digit of K bits is a chain of K - 1 products and two
// independent ones for the output factors, where the radix-4 steps make up to
// 2 K + 1 (2^12, digits 6 and 6: 14.3 -> 10.5 us, 2^14 16.4 -> 13.6, 2^15, 7 and 8,
// 16.5 -> 12.8, 2^16, 7 and 9, 18.4 -> 16.7; 2^17, with two warps for every scheduler
// of the GPU, 24.9 -> 31.0).  EARLY: read the output factors before the stages (32
// registers held across them).
template <class F, bool EARLY>
__device__ __forceinline__ void run_stages(const PassArgs &a, const uint4 *tab, uint4 *buf,
                                           uint32_t tile, uint32_t nthreads) {
    const uint32_t K = a.K, lc = a.log_cols, tid = threadIdx.x;
    const uint32_t half = 1u << (K + lc - 1);  // pairs in the tile
    Factor v0, v1;
    if (EARLY && tid < nthreads) {
        const OutRows o = out_rows<2>(a, tile, (tid >> lc) << 1, tid & ((1u << lc) - 1u));
        if (o.f) {
            ldg_out_factor(v0, a, o.f);
            ldg_out_factor(v1, a, o.f + o.fstep);
        }
    }
    for (uint32_t h = 1u << (K - 1); h >= 2; h >>= 1) {
        radix2_stage<F>(buf, tab, h, K, lc, tid, nthreads);
        // at h <= 32 a warp's pairs, 32 consecutive ones, are made of rows of its
        // own, at this stage and the next; the last (columns fastest) reads others',
        // but of one column
        if (h > 32 || (h == 2 && lc > 0)) __syncthreads();
        else __syncwarp();
    }
#pragma unroll 1
    for (uint32_t g = tid; tid < nthreads && g < half; g += nthreads) {
        const uint32_t cc = g & ((1u << lc) - 1u), d0 = (g >> lc) << 1;
        const uint32_t u0 = smem_unit(cc, d0, K, lc);
        const OutRows o = out_rows<2>(a, tile, d0, cc);
        uint32_t x0[8], x1[8];
        lds_elem(x0, buf, u0);
        lds_elem(x1, buf, u0 ^ 1u);
        sum_sub<F>(x0, x1);
        if (o.f) {
            if (!EARLY) ldg_out_factor(v0, a, o.f);
            mul_factor<F>(x0, x0, v0);
            if (!EARLY) ldg_out_factor(v1, a, o.f + o.fstep);
            mul_factor<F>(x1, x1, v1);
        } else if (!a.last) {
            otf_scale<F>(x0, a, tile, d0, cc);
            otf_scale<F>(x1, a, tile, d0 + 1, cc);
        }
        if (a.last) {
            reduce_once<F>(x0);
            reduce_once<F>(x1);
        }
        st_elem8(o.out, x0);
        st_elem8(o.out + 2 * o.step, x1);
    }
}

// Process one tile, copied to `buf` with the table in `tab` (the block has
// synchronised since), with `nthreads` threads of the block (threads at or
// beyond nthreads only take part in the barriers).  The block does not
// synchronise at the end: `buf` may be written again after a barrier.
// COMPILED: the sizes are constants and all threads of the block have one group
// (radix 4) or pair (radix 2) in each step.
template <class F, Steps STEPS, bool COMPILED = false>
__device__ __forceinline__ void run_tile(const PassArgs &a, const uint4 *tab, uint4 *buf,
                                         uint32_t tile, uint32_t nthreads) {
    const uint32_t K = a.K, lc = a.log_cols;
    const uint32_t N = 1u << K;
    const uint32_t C = 1u << lc;
    const uint32_t CN = C << K;
    const uint32_t tid = threadIdx.x;
    const bool active = tid < nthreads;

    // ---- input factors.  Each is read into the registers of the one before it as
    // soon as that has been used (not in the batch kernel, with 80 registers and
    // without the pointwise step).
    auto place = [&](uint32_t e, uint32_t &d, uint32_t &cc) {
        if (a.last) { d = e & (N - 1); cc = e >> K; }
        else        { cc = e & (C - 1); d = e >> lc; }
    };
    if (STEPS == EITHER && a.pre) {
#pragma unroll 1
        for (uint32_t e = tid; active && e < CN; e += nthreads) {
            uint32_t d, cc, x[8];
            place(e, d, cc);
            const uint32_t u = smem_unit(cc, d, K, lc);
            Factor f;
            ldg_factor(f, a.pre + 4 * size_t(d));
            lds_elem(x, buf, u);
            mul_factor<F>(x, x, f);
            sts_elem(buf, u, x);
        }
        __syncthreads();
    }
    if (STEPS != EITHER && (a.pre || a.pw_b)) {
        uint32_t d, cc, b[8], c[8];
        Factor f;
        place(active ? tid : 0, d, cc);
        size_t g = tile_src(a, tile, d, cc);
        if (a.pw_b) {
            ld_elem_cg(b, a.pw_b + 2 * g);
            ld_elem_cg(c, a.pw_c + 2 * g);
        }
        if (a.pre) ldg_factor(f, a.pre + 4 * size_t(d));
#pragma unroll 1
        for (uint32_t e = tid; active && e < CN; e += nthreads) {
            const uint32_t u = smem_unit(cc, d, K, lc);
            uint32_t x[8], q[8];
            lds_elem(x, buf, u);
            if (e + nthreads < CN) place(e + nthreads, d, cc);
            g = tile_src(a, tile, d, cc);
            if (a.pw_b) {
                mul<F>(x, b, x);
                ld_elem_cg(b, a.pw_b + 2 * g);
                sub<F>(x, x, c);
                ld_elem_cg(c, a.pw_c + 2 * g);
            }
            if (a.pre) {
                mul_high(q, x, f.wq);
                ZK_LD8("", f.wq, a.pre + 4 * size_t(d) + 2);
                mul_low_fold<F>(x, x, f.w, q);
                ZK_LD8("", f.w, a.pre + 4 * size_t(d));
            }
            sts_elem(buf, u, x);
        }
        __syncthreads();
    }

    if (STEPS == RADIX2 || (STEPS == EITHER && nthreads > (CN >> 2))) {
        run_stages<F, COMPILED>(a, tab, buf, tile, nthreads);
        return;
    }

    // With 10 bits and more two blocks fit an SM, too few to wait for the entries of
    // the big table that the last step wants: into L2 (2^20, digits 10 and 10: 157 ->
    // 148 us; no gain for smaller digits).
    if (K >= 10 && !a.last && !a.otf && active && tid < (CN >> 2)) {
        const OutRows o = out_rows<4>(a, tile, (tid >> lc) << 2, tid & (C - 1));
#pragma unroll
        for (int i = 0; i < 4; i++)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(o.f + i * o.fstep));
    }

    // ---- stages 0 .. K-3
    if (K > 2) {
        uint32_t q = N >> 2;  // distance of a radix-4 step's rows
        // the thread's group, and its column's part of the units
        const uint32_t g0 = tid & ((N >> 2) - 1), c0 = col_unit(tid >> (K - 2), K, lc);
        // After a step at distance q that the step at q/4 or q/8 follows: at q <= 32 a
        // warp's groups, 32 consecutive ones, are made of rows of its own, at this
        // step and the next; a column's threads exchange rows otherwise.  The last
        // step (columns fastest) reads every column.
        auto sync = [&](uint32_t q, bool to_last) {
            if (to_last && (lc > 0 || q > 32)) __syncthreads();
            else if (q <= 32) __syncwarp();
            else if (COMPILED && lc > 0)
                asm volatile("bar.sync %0, %1;" ::"r"(1 + (tid >> (K - 2))), "r"(N >> 2) : "memory");
            else __syncthreads();
        };
        if (K & 1u) {
            // the first stage alone, on the rows of a step at distance N/4
            const uint32_t x1 = row_unit(q), x2 = row_unit(2 * q), xt = tab_unit(q);
            uint32_t g = tid, b = g0, c = c0;
            while (active && g < (CN >> 2)) {
                const uint32_t u0 = c ^ row_unit(b), ta = tab_unit(b);
                uint32_t v0[8], v1[8], v2[8], v3[8], t[8], u[8];
                Factor w, z;
                lds_elem(v0, buf, u0);
                lds_elem(v2, buf, u0 ^ x2);
                lds_factor(w, tab, ta);
                lds_elem(v1, buf, u0 ^ x1);
                lds_elem(v3, buf, u0 ^ x1 ^ x2);
                lds_factor(z, tab, ta ^ xt);
                sum_diff<F>(v0, t, v2);
                sts_elem(buf, u0, v0);
                sum_diff<F>(v1, u, v3);
                sts_elem(buf, u0 ^ x1, v1);
                mul_factor2<F>(v2, t, w, v3, u, z);
                sts_elem(buf, u0 ^ x2, v2);
                sts_elem(buf, u0 ^ x1 ^ x2, v3);
                g += nthreads;
                b = g & ((N >> 2) - 1);
                c = col_unit(g >> (K - 2), K, lc);
            }
            sync(q, K == 3);
            q >>= 1;
        }
        uint32_t shift = K & 1u;  // the step's first stage: entries j 2^shift and (j + q) 2^shift
#pragma unroll
        for (; q > 1; q >>= 2, shift += 2) {
            // rows i0 + {0, q, 2q, 3q}: the stage of distance 2q, then of distance q
            const uint32_t x1 = row_unit(q), x2 = row_unit(2 * q), xt = tab_unit(q << shift);
            uint32_t g = tid, b = g0, c = c0;
            while (active && g < (CN >> 2)) {
                const uint32_t j = b & (q - 1);
                const uint32_t u0 = c ^ row_unit(4 * b - 3 * j);
                const uint32_t ta = tab_unit(j << shift), tb = tab_unit(j << (shift + 1));
                uint32_t v0[8], v1[8], v2[8], v3[8], t[8], u[8];
                Factor w, z;
                lds_elem(v0, buf, u0);
                lds_elem(v2, buf, u0 ^ x2);
                lds_factor(w, tab, ta);
                lds_elem(v1, buf, u0 ^ x1);
                lds_elem(v3, buf, u0 ^ x1 ^ x2);
                lds_factor(z, tab, ta ^ xt);
                sum_diff<F>(v0, t, v2);
                sum_diff<F>(v1, u, v3);
                mul_factor2<F>(v2, t, w, v3, u, z);
                lds_factor(w, tab, tb);
                sum_diff<F>(v0, t, v1);
                sum_diff<F>(v2, u, v3);
                sts_elem(buf, u0, v0);
                sts_elem(buf, u0 ^ x2, v2);
                mul_factor2<F>(v1, t, w, v3, u, w);
                sts_elem(buf, u0 ^ x1, v1);
                sts_elem(buf, u0 ^ x1 ^ x2, v3);
                g += nthreads;
                b = g & ((N >> 2) - 1);
                c = col_unit(g >> (K - 2), K, lc);
            }
            sync(q, q == 4);
        }
    }

    // ---- last two stages as radix-4 on rows d0..d0+3, factors and store
    // (columns fastest: C-element runs in global memory)
    if (K >= 2) {
        Factor w4;
        lds_factor(w4, tab, tab_unit(N >> 2));  // w_N^(N/4) = w_4
        for (uint32_t qd = tid; active && qd < (CN >> 2); qd += nthreads) {
            const uint32_t cc = qd & (C - 1);
            const uint32_t d0 = (qd >> lc) << 2;
            uint32_t x0[8], x1[8], x2[8], x3[8], t[8];
            // rows d0 + i (d0 a multiple of 4) share the swizzle term: their
            // units are the first one's with i in the low two bits
            const uint32_t u0 = smem_unit(cc, d0, K, lc);
            lds_elem(x1, buf, u0 ^ 1u);
            lds_elem(x3, buf, u0 ^ 3u);
            lds_elem(x0, buf, u0);
            lds_elem(x2, buf, u0 ^ 2u);
            // stage K-2: pairs (0,2) with twiddle 1, (1,3) with w_4
            sum_diff<F>(x1, t, x3);
            mul_factor<F>(x3, t, w4);
            sum_sub<F>(x0, x2);
            // stage K-1: pairs (0,1), (2,3), twiddle 1
            sum_sub<F>(x0, x1);
            sum_sub<F>(x2, x3);
            const OutRows o = out_rows<4>(a, tile, d0, cc);
            if (a.last && !o.f) {
                // no factor: below r, and out (rows in bit-reversed order)
                reduce_once<F>(x0);
                st_elem8(o.out, x0);
                reduce_once<F>(x1);
                st_elem8(o.out + 4 * o.step, x1);
                reduce_once<F>(x2);
                st_elem8(o.out + 2 * o.step, x2);
                reduce_once<F>(x3);
                st_elem8(o.out + 6 * o.step, x3);
            } else {
                // through the thread's own slots into a loop over the rows
                sts_elem(buf, u0, x0);
                sts_elem(buf, u0 ^ 1u, x1);
                sts_elem(buf, u0 ^ 2u, x2);
                sts_elem(buf, u0 ^ 3u, x3);
                scale_and_store<F, 4, STEPS != EITHER>(a, buf, u0, o, tile, d0, cc);
            }
        }
    } else {
        // N = 2: one radix-2 butterfly per column
        for (uint32_t cc = tid; active && cc < C; cc += nthreads) {
            uint32_t x0[8], x1[8];
            const uint32_t u0 = smem_unit(cc, 0, K, lc);
            lds_elem(x0, buf, u0);
            lds_elem(x1, buf, u0 ^ 1u);
            sum_sub<F>(x0, x1);
            const OutRows o = out_rows<2>(a, tile, 0, cc);
            if (a.last && !o.f) {
                reduce_once<F>(x0);
                st_elem8(o.out, x0);
                reduce_once<F>(x1);
                st_elem8(o.out + 2 * o.step, x1);
            } else {
                sts_elem(buf, u0, x0);
                sts_elem(buf, u0 ^ 1u, x1);
                scale_and_store<F, 2, STEPS != EITHER>(a, buf, u0, o, tile, 0, cc);
            }
        }
    }
}

// threads per block of schedule variant v for a tile of C x 2^K elements: one
// per four elements (variant 5: two, one butterfly a thread and stage), at most
// 256
__host__ __device__ constexpr uint32_t pass_threads_for(uint32_t K, uint32_t lc, int v) {
    const uint32_t t = K >= 2 ? 1u << (K + lc - (v == 5 ? 1 : 2)) : 1u << lc;
    return t < 256u ? t : 256u;
}

// What a pass kernel is compiled for.  ANY: every argument is a runtime value.
// The others: a digit of K bits in tiles of fixed_cols columns; a strided pass
// with precomputed twiddles, its input without factors (STRIDED) or with
// (STRIDED_PRE: input scales or the pointwise step), or with twiddles on the fly
// (STRIDED_OTF); the last pass without output factors (LAST) or with (LAST_POST).  With these fixed the index
// arithmetic of a tile shrinks: 803 -> 692 instructions an element in the last
// pass of 2^22, which was 691 us and is 642 (BLS12-381, digits 8, 7, 7).  (With
// the digit alone fixed and the factors left to the arguments 2^22 took 648, 2^12
// to 2^16 a tenth longer.)
enum Kind { ANY, STRIDED, STRIDED_PRE, STRIDED_OTF, LAST, LAST_POST, NUM_KINDS };

// log2 of the columns of the tiles of the compiled digits: two, so that global
// memory is read and written in 64-byte pieces; one where two make a tile and
// table of which only one would fit an SM, and for one butterfly a thread, where
// twice the blocks matter more (2^12 12.6 -> 10.5 us, 2^15 16.4 -> 12.8).  (Four or eight columns for digits of 6
// and 7 bits: 2^24 2591 -> 2705 us, 2^26 11417 -> 11641.)
__host__ __device__ constexpr int fixed_cols(int K, Steps steps = RADIX4) {
    return K < 10 && steps == RADIX4 ? 1 : 0;
}

template <int K, Kind KIND, Steps STEPS>
__device__ __forceinline__ void fix_args(PassArgs &a) {
    if (KIND == ANY) return;
    a.K = K;
    a.log_cols = fixed_cols(K, STEPS);
    a.last = KIND == LAST || KIND == LAST_POST;
    a.otf = KIND == STRIDED_OTF;
    if (KIND != STRIDED_PRE) a.pre = a.pw_b = a.pw_c = nullptr;
    if (KIND != LAST_POST) a.post = nullptr;
}

// One pass over the vectors' tiles (args: num_tiles of them in all; its own `in`
// and `out` are not used).  The register budget is for BLOCKS blocks of THREADS
// threads an SM.
template <class F, int THREADS, int BLOCKS, Steps STEPS, int K, Kind KIND>
__global__ void __launch_bounds__(THREADS, BLOCKS)
    ntt_pass_kernel(const PassArgs args, const __grid_constant__ PassVectors vec) {
    extern __shared__ uint4 smem[];
    PassArgs a = args;
    fix_args<K, KIND, STEPS>(a);
    const uint32_t nthreads = KIND == ANY ? blockDim.x : THREADS;
    const uint32_t units = tile_units(1u << (a.K + a.log_cols));
    uint4 *tab = smem, *buf = smem + 4 * tab_entries(a.K);
    issue_table_load(a, tab, nthreads);  // (a plan's table: no pass writes it)
    // Passes after the first are launched as programmatic dependents of the
    // pass before, and wait here until that pass has completed and its writes
    // are visible (launched without that attribute, the wait returns at once).
    // A block lets the next pass launch when it starts its last tile, so the
    // next pass's blocks take SM places only as this grid winds down.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    uint32_t tile = a.num_tiles;  // the tile to compute (none yet)
    // Two tile buffers when the block has more than one tile: the copies of its
    // next tile are in flight while the current one is computed.
    uint4 *cur = buf + units, *other = buf;
#pragma unroll 1
    for (uint32_t fetch = blockIdx.x;; fetch += gridDim.x) {
        uint32_t v;
        if (fetch < a.num_tiles) {
            const uint32_t t = vector_tile(vec, fetch, v);
            a.in = vec.in[v];
            issue_tile_load(a, other, t, nthreads);
        } else {
            asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        }
        if (tile < a.num_tiles) {
            const uint32_t t = vector_tile(vec, tile, v);
            a.out = vec.out[v];
            run_tile<F, STEPS, KIND != ANY>(a, tab, cur, t, nthreads);
        }
        if (fetch >= a.num_tiles) break;
        cp_async_wait_all();
        // the fetched tile is there, and every thread is done with the other one
        __syncthreads();
        tile = fetch;
        uint4 *const t = cur;
        cur = other;
        other = t;
    }
}

}  // namespace zkntt
