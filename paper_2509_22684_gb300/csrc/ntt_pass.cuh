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
// The difference x - y is formed as x + r - y with no conditional correction:
// it only feeds the product, which takes any x below 2r.
// All sizes (K, C, the stride) are runtime values: one kernel per field serves
// every digit size.
//
// Shared memory holds each element as two 16-byte halves in separate arrays.
// The slot of (column c, row d) is c*N + (d ^ s), with s in the low three bits
// a linear function of bits 3 and 4 of d and of c (smem_slot), chosen so that
// the eight lanes of an access fall into different bank groups in every
// pattern: copies with columns or rows fastest, steps at distance 4 and above,
// and the last step on rows 4 g + i with columns fastest.
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

__device__ __forceinline__ uint32_t brev_bits(uint32_t x, uint32_t bits) {
    return bits == 0 ? 0u : (__brev(x) >> (32 - bits));
}

// Row part of the shared-memory slot (K >= 3): d with its low three bits
// xor 5 for bit 3 and xor 6 for bit 4.  Linear over xor, so the rows of a group
// at distances that are powers of two have slots at xor distances.
__device__ __forceinline__ uint32_t row_slot(uint32_t d) {
    return d ^ (((d >> 3) & 1u) * 5u) ^ (((d >> 4) & 1u) * 6u);
}

// shared-memory slot of element (column c, row d)
__device__ __forceinline__ uint32_t smem_slot(uint32_t c, uint32_t d, uint32_t K, uint32_t lc) {
    if (K < 3) return (c << K) + d;
    const uint32_t s = lc == 3 ? c : lc == 2 ? ((c & 1u) << 1) ^ ((c >> 1) * 5u) : c * 6u;
    return (c << K) + (row_slot(d) ^ s);
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

__device__ __forceinline__ void lds_elem(uint32_t x[8], const uint4 *s_lo, const uint4 *s_hi,
                                         uint32_t slot) {
    uint4 v0 = s_lo[slot], v1 = s_hi[slot];
    x[0] = v0.x; x[1] = v0.y; x[2] = v0.z; x[3] = v0.w;
    x[4] = v1.x; x[5] = v1.y; x[6] = v1.z; x[7] = v1.w;
}

__device__ __forceinline__ void sts_elem(uint4 *s_lo, uint4 *s_hi, uint32_t slot,
                                         const uint32_t x[8]) {
    s_lo[slot] = make_uint4(x[0], x[1], x[2], x[3]);
    s_hi[slot] = make_uint4(x[4], x[5], x[6], x[7]);
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

__device__ __forceinline__ size_t tile_dst(const PassArgs &a, uint32_t tile, uint32_t d,
                                           uint32_t cc) {
    if (!a.last) return tile_src(a, tile, d, cc);
    return (size_t(brev_bits(d, a.K)) << a.hi_bits) + (size_t(tile) << a.log_cols) + cc;
}

// The factors of row position d in column cc on the way out: the inter-pass
// twiddle (precomputed, or up to four factors on the fly) or the last pass's
// post scale.  A null p[0]: none; a null p[k] ends the list.
__device__ __forceinline__ void out_factors(const uint4 *p[4], const PassArgs &a, uint32_t tile,
                                            uint32_t d, uint32_t cc) {
    p[0] = p[1] = p[2] = p[3] = nullptr;
    if (a.last) {
        if (a.post) p[0] = a.post + 4 * size_t(d);
        return;
    }
    const uint32_t lo_tiles_bits = a.lo_bits - a.log_cols;
    const uint32_t lo = ((tile & ((1u << lo_tiles_bits) - 1u)) << a.log_cols) + cc;
    if (!a.otf) {
        p[0] = a.tw + 4 * ((size_t(d) << a.lo_bits) + lo);
        return;
    }
    // lo < 2^lo_bits and rev(d) < 2^K, so e < 2^tw_bits = n_i: no reduction
    // (and no overflow: tw_bits <= 32)
    const uint32_t e = lo * brev_bits(d, a.K);
    p[0] = a.w_hi + 4 * size_t(e >> a.split_bits);
    p[1] = a.w_lo + 4 * size_t(e & ((1u << a.split_bits) - 1u));
    if (a.fl) p[2] = a.fl + 4 * size_t(lo);
    if (a.fd) (a.fl ? p[3] : p[2]) = a.fd + 4 * size_t(d);
}

// x times its output factors, to its place in global memory.  One product in
// the code, in a loop over the factors: unrolled, the kernels outgrow the
// instruction cache.
template <class F>
__device__ __forceinline__ void scale_and_store(uint32_t x[8], const PassArgs &a, uint32_t tile,
                                                uint32_t d, uint32_t cc) {
    const uint4 *p[4];
    out_factors(p, a, tile, d, cc);
    // an entry of the big table is read once: it takes no place in L1
    const bool stream = !a.last && !a.otf;
#pragma unroll 1
    while (p[0]) {
        Factor f;
        if (stream) ldg_factor_stream(f, p[0]);
        else ldg_factor(f, p[0]);
        mul_factor<F>(x, x, f);
        p[0] = p[1];
        p[1] = p[2];
        p[2] = p[3];
        p[3] = nullptr;
    }
    st_elem(a.out + 2 * tile_dst(a, tile, d, cc), x);
}

// Issue (without waiting) the 16-byte copies of one tile into shared memory:
// 8 lanes copy the low halves of 8 elements, the next 8 lanes their high
// halves (tiles under 8 elements: element-major); columns fastest for strided
// passes, rows fastest for the last.
__device__ __forceinline__ void issue_tile_load(const PassArgs &a, uint4 *smem, uint32_t tile,
                                                uint32_t nthreads) {
    const uint32_t K = a.K, lc = a.log_cols;
    const uint32_t N = 1u << K, C = 1u << lc, CN = C << K;
    uint4 *s_lo = smem, *s_hi = smem + CN;
    const uint32_t tid = threadIdx.x;
    if (tid >= nthreads) return;
    if (CN >= 64 && (nthreads & 15u) == 0 && (nthreads & (nthreads - 1u)) == 0 && nthreads <= 2 * CN) {
        // Every thread makes 2 C N / nthreads copies of one half (the lane's
        // bit 3) of elements e0, e0 + E, e0 + 2E, ... (E = nthreads / 2); in
        // a strided pass they share a column and step by a fixed row count,
        // so the source address steps by a fixed stride and only the shared
        // slot is formed per copy.
        const uint32_t half = (tid >> 3) & 1u;
        const uint32_t e0 = (tid & 7u) | ((tid >> 4) << 3);
        const uint32_t E = nthreads >> 1, iters = (2 * CN) / nthreads;
        const uint32_t sbase =
            static_cast<uint32_t>(__cvta_generic_to_shared(half ? s_hi : s_lo));
        if (!a.last) {
            const uint32_t cc = e0 & (C - 1), dstep = E >> lc;
            uint32_t d = e0 >> lc;
            const uint4 *src = a.in + 2 * tile_src(a, tile, d, cc) + half;
            const size_t sstep = size_t(2 * dstep) << a.lo_bits;
            if ((dstep & 31u) == 0) {
                // rows d, d + dstep, ... agree in their low five bits, so they
                // share the swizzle term and their slots step by dstep too
                uint32_t sa = sbase + 16u * smem_slot(cc, d, K, lc);
                for (uint32_t k = 0; k < iters; k++, sa += 16u * dstep, src += sstep)
                    cp_async16_sa(sa, src);
            } else {
                for (uint32_t k = 0; k < iters; k++, d += dstep, src += sstep)
                    cp_async16_sa(sbase + 16u * smem_slot(cc, d, K, lc), src);
            }
        } else if (E < N) {
            // last pass, rows fastest: N / E copies in one column (rows e0,
            // e0 + E, ...; e0 < E), then the next column
            const uint32_t per = N / E;
            for (uint32_t cc = 0; cc < C; cc++) {
                const uint4 *row = a.in + 2 * tile_src(a, tile, 0, cc) + half;
                for (uint32_t j = 0, d = e0; j < per; j++, d += E)
                    cp_async16_sa(sbase + 16u * smem_slot(cc, d, K, lc), row + 2 * d);
            }
        } else {
            uint32_t e = e0;
            for (uint32_t k = 0; k < iters; k++, e += E) {
                const uint32_t d = e & (N - 1), cc = e >> K;
                cp_async16_sa(sbase + 16u * smem_slot(cc, d, K, lc),
                              a.in + 2 * tile_src(a, tile, d, cc) + half);
            }
        }
        return;
    }
    const bool grouped = CN >= 8;
    for (uint32_t u = tid; u < 2 * CN; u += nthreads) {
        const uint32_t e = grouped ? ((u & 7u) | ((u >> 4) << 3)) : (u >> 1);
        const uint32_t half = grouped ? ((u >> 3) & 1u) : (u & 1u);
        uint32_t d, cc;
        if (a.last) { d = e & (N - 1); cc = e >> K; }
        else        { cc = e & (C - 1); d = e >> lc; }
        const size_t g = tile_src(a, tile, d, cc);
        cp_async16((half ? s_hi : s_lo) + smem_slot(cc, d, K, lc), a.in + 2 * g + half);
    }
}

// The sub-transform's twiddles in shared memory: the N/2 factors w_N^e in four
// planes of N/2 16-byte quarters, entry e at slot tab_slot(e).  The slot's low
// three bits fold in the higher ones, so eight entries at any power-of-two
// stride lie in different bank groups.  (Read from global memory instead, they
// missed L1 half the time and were two thirds of the load/store wavefronts.)
__host__ __device__ __forceinline__ uint32_t tab_slot(uint32_t e) {
    return e ^ (((e >> 3) ^ (e >> 6) ^ (e >> 9)) & 7u);
}

// entries of the table of a 2^K-point sub-transform
__host__ __device__ constexpr uint32_t tab_entries(uint32_t K) { return K > 1 ? 1u << (K - 1) : 1u; }

// issue (without waiting) the copies of the table, which is laid out in global
// memory as in shared memory
__device__ __forceinline__ void issue_table_load(const PassArgs &a, uint4 *tab) {
    const uint32_t units = 4 * tab_entries(a.K);
    for (uint32_t u = threadIdx.x; u < units; u += blockDim.x) cp_async16(tab + u, a.w_stage + u);
}

// the factor at table slot s (h = entries)
__device__ __forceinline__ void lds_factor(Factor &f, const uint4 *tab, uint32_t h, uint32_t s) {
    lds_elem(f.w, tab, tab + h, s);
    lds_elem(f.wq, tab + 2 * h, tab + 3 * h, s);
}

// How a tile's stages run: two at a time, four elements a thread (radix 4), or
// one by one, one butterfly a thread (radix 2); or either by the thread count.
enum Steps { RADIX4 = 1, RADIX2 = 2, EITHER = 3 };

// x <- x + y, t = x - y + r (for the product): the sum and lazy difference of
// a butterfly
template <class F>
__device__ __forceinline__ void sum_diff(uint32_t x[8], uint32_t t[8], const uint32_t y[8]) {
    sub_lazy<F>(t, x, y);
    add<F>(x, x, y);
}

// One stage, pairs at distance h, one butterfly after the other.
template <class F>
__device__ __forceinline__ void radix2_stage(uint4 *s_lo, uint4 *s_hi, const uint4 *tab, uint32_t h,
                                             uint32_t K, uint32_t lc, uint32_t tid,
                                             uint32_t nthreads) {
    const uint32_t N = 1u << K, CN = N << lc, step = row_slot(h);
    const uint32_t shift = K - 1 - (31 - __clz(h));  // entry j 2^stage
    for (uint32_t bk = tid; tid < nthreads && bk < (CN >> 1); bk += nthreads) {
        const uint32_t cc = bk >> (K - 1), b = bk & ((N >> 1) - 1), j = b & (h - 1);
        const uint32_t s0 = smem_slot(cc, ((b ^ j) << 1) | j, K, lc), s1 = s0 ^ step;
        uint32_t x[8], y[8], t[8];
        Factor w;
        lds_elem(x, s_lo, s_hi, s0);
        lds_elem(y, s_lo, s_hi, s1);
        lds_factor(w, tab, N >> 1, tab_slot(j << shift));
        sum_diff<F>(x, t, y);
        mul_factor<F>(t, t, w);
        sts_elem(s_lo, s_hi, s0, x);
        sts_elem(s_lo, s_hi, s1, t);
    }
}

// Process one tile, copied to `buf` with the table in `tab` (the block has
// synchronised since), with `nthreads` threads of the block (threads at or
// beyond nthreads only take part in the barriers).  The block does not
// synchronise at the end: `buf` may be written again after a barrier.
template <class F, Steps STEPS>
__device__ __forceinline__ void run_tile(const PassArgs &a, const uint4 *tab, uint4 *buf,
                                         uint32_t tile, uint32_t nthreads) {
    const uint32_t K = a.K, lc = a.log_cols;
    const uint32_t N = 1u << K;
    const uint32_t C = 1u << lc;
    const uint32_t CN = C << K;
    uint4 *s_lo = buf;
    uint4 *s_hi = buf + CN;
    const uint32_t tid = threadIdx.x;
    const bool active = tid < nthreads;

    // ---- input factors
    if (a.pre || a.pw_b) {
#pragma unroll 1
        for (uint32_t e = tid; active && e < CN; e += nthreads) {
            uint32_t d, cc;
            if (a.last) { d = e & (N - 1); cc = e >> K; }
            else        { cc = e & (C - 1); d = e >> lc; }
            const uint32_t s = smem_slot(cc, d, K, lc);
            uint32_t x[8];
            lds_elem(x, s_lo, s_hi, s);
            if (a.pw_b) {
                const size_t g = tile_src(a, tile, d, cc);
                uint32_t v[8], u[8];
                ld_elem_cg(v, a.pw_b + 2 * g);
                ld_elem_cg(u, a.pw_c + 2 * g);
                mul<F>(x, x, v);
                sub<F>(x, x, u);
            }
            if (a.pre) {
                Factor f;
                ldg_factor(f, a.pre + 4 * size_t(d));
                mul_factor<F>(x, x, f);
            }
            sts_elem(s_lo, s_hi, s, x);
        }
        __syncthreads();
    }

    // ---- stages 0 .. K-3
    if (STEPS == RADIX2 || (STEPS == EITHER && nthreads > (CN >> 2))) {
        for (uint32_t h = N >> 1; h >= 4; h >>= 1) {
            radix2_stage<F>(s_lo, s_hi, tab, h, K, lc, tid, nthreads);
            __syncthreads();
        }
    } else if (K > 2) {
        uint32_t q = N >> 2;  // distance of a radix-4 step's rows
        if (K & 1u) {
            radix2_stage<F>(s_lo, s_hi, tab, N >> 1, K, lc, tid, nthreads);
            __syncthreads();
            q >>= 1;
        }
        uint32_t shift = K & 1u;  // the step's first stage: entries j 2^shift and (j + q) 2^shift
        for (; q > 1; q >>= 2, shift += 2) {
            // rows i0 + {0, q, 2q, 3q}: the stage of distance 2q, then of distance q
            const uint32_t x1 = row_slot(q), x2 = row_slot(2 * q), xt = tab_slot(q << shift);
            for (uint32_t g = tid; active && g < (CN >> 2); g += nthreads) {
                const uint32_t cc = g >> (K - 2), b = g & ((N >> 2) - 1), j = b & (q - 1);
                const uint32_t s0 = smem_slot(cc, ((b ^ j) << 2) | j, K, lc);
                const uint32_t ta = tab_slot(j << shift), tb = tab_slot(j << (shift + 1));
                uint32_t v0[8], v1[8], v2[8], v3[8], t[8];
                Factor w;
                lds_elem(v0, s_lo, s_hi, s0);
                lds_elem(v2, s_lo, s_hi, s0 ^ x2);
                lds_factor(w, tab, N >> 1, ta);
                sum_diff<F>(v0, t, v2);
                mul_factor<F>(v2, t, w);
                lds_elem(v1, s_lo, s_hi, s0 ^ x1);
                lds_elem(v3, s_lo, s_hi, s0 ^ x1 ^ x2);
                lds_factor(w, tab, N >> 1, ta ^ xt);
                sum_diff<F>(v1, t, v3);
                mul_factor<F>(v3, t, w);
                lds_factor(w, tab, N >> 1, tb);
                sum_diff<F>(v0, t, v1);
                sts_elem(s_lo, s_hi, s0, v0);
                mul_factor<F>(v1, t, w);
                sts_elem(s_lo, s_hi, s0 ^ x1, v1);
                sum_diff<F>(v2, t, v3);
                sts_elem(s_lo, s_hi, s0 ^ x2, v2);
                mul_factor<F>(v3, t, w);
                sts_elem(s_lo, s_hi, s0 ^ x1 ^ x2, v3);
            }
            // at q <= 32 a warp's groups, 32 consecutive ones, are made of rows
            // of its own, at this step and the next: only the last step (columns
            // fastest) reads another warp's
            if (q > 32 || q == 4) __syncthreads();
            else __syncwarp();
        }
    }

    // ---- last two stages as radix-4 on rows d0..d0+3, factors and store
    // (columns fastest: C-element runs in global memory)
    const bool scaled = a.last ? a.post != nullptr : true;
    if (K >= 2) {
        Factor w4;
        lds_factor(w4, tab, N >> 1, tab_slot(N >> 2));  // w_N^(N/4) = w_4
        for (uint32_t qd = tid; active && qd < (CN >> 2); qd += nthreads) {
            const uint32_t cc = qd & (C - 1);
            const uint32_t d0 = (qd >> lc) << 2;
            uint32_t x0[8], x1[8], x2[8], x3[8], t[8];
            // rows d0 + i (d0 a multiple of 4) share the swizzle term: their
            // slots are the first one's with i in the low two bits
            const uint32_t s0 = smem_slot(cc, d0, K, lc), s1 = s0 ^ 1u, s2 = s0 ^ 2u, s3 = s0 ^ 3u;
            lds_elem(x0, s_lo, s_hi, s0);
            lds_elem(x1, s_lo, s_hi, s1);
            lds_elem(x2, s_lo, s_hi, s2);
            lds_elem(x3, s_lo, s_hi, s3);
            // stage K-2: pairs (0,2) with twiddle 1, (1,3) with w_4
            sub<F>(t, x0, x2);
            add<F>(x0, x0, x2);
#pragma unroll
            for (int k = 0; k < 8; k++) x2[k] = t[k];
            sum_diff<F>(x1, t, x3);
            mul_factor<F>(x3, t, w4);
            // stage K-1: pairs (0,1), (2,3), twiddle 1
            sub<F>(t, x0, x1);
            add<F>(x0, x0, x1);
            if (!scaled) {
                st_elem(a.out + 2 * tile_dst(a, tile, d0, cc), x0);
                st_elem(a.out + 2 * tile_dst(a, tile, d0 + 1, cc), t);
                sub<F>(t, x2, x3);
                add<F>(x2, x2, x3);
                st_elem(a.out + 2 * tile_dst(a, tile, d0 + 2, cc), x2);
                st_elem(a.out + 2 * tile_dst(a, tile, d0 + 3, cc), t);
                continue;
            }
            // through the thread's own slots into a loop with one product
            sts_elem(s_lo, s_hi, s0, x0);
            sts_elem(s_lo, s_hi, s1, t);
            sub<F>(t, x2, x3);
            add<F>(x2, x2, x3);
            sts_elem(s_lo, s_hi, s2, x2);
            sts_elem(s_lo, s_hi, s3, t);
#pragma unroll 1
            for (uint32_t i = 0; i < 4; i++) {
                uint32_t x[8];
                lds_elem(x, s_lo, s_hi, s0 ^ i);
                scale_and_store<F>(x, a, tile, d0 + i, cc);
            }
        }
    } else {
        // N = 2: one radix-2 butterfly per column
        for (uint32_t cc = tid; active && cc < C; cc += nthreads) {
            uint32_t x0[8], x1[8], t[8];
            const uint32_t s0 = smem_slot(cc, 0, K, lc), s1 = smem_slot(cc, 1, K, lc);
            lds_elem(x0, s_lo, s_hi, s0);
            lds_elem(x1, s_lo, s_hi, s1);
            sub<F>(t, x0, x1);
            add<F>(x0, x0, x1);
            sts_elem(s_lo, s_hi, s0, x0);
            sts_elem(s_lo, s_hi, s1, t);
#pragma unroll 1
            for (uint32_t i = 0; i < 2; i++) {
                uint32_t x[8];
                lds_elem(x, s_lo, s_hi, s0 + i);
                scale_and_store<F>(x, a, tile, i, cc);
            }
        }
    }
}

// threads per block for a tile of C x 2^K elements: one per radix-4 group,
// at most 256
__host__ __device__ constexpr uint32_t pass_threads(uint32_t K, uint32_t lc) {
    return ((K >= 2 ? (1u << (K + lc - 2)) : (1u << lc)) < 256u)
               ? (K >= 2 ? (1u << (K + lc - 2)) : (1u << lc))
               : 256u;
}

// threads per block for schedule variant v: variant 5 doubles the count (one
// butterfly per thread per stage), still at most 256
__host__ __device__ constexpr uint32_t pass_threads_for(uint32_t K, uint32_t lc, int v) {
    return v == 5 && K >= 2 && pass_threads(K, lc) < 256u ? 2u * pass_threads(K, lc)
                                                           : pass_threads(K, lc);
}

// One pass.  MIN_BLOCKS: blocks of 256 threads an SM the register budget is
// for (2: 128 registers, 3: 80, 4: 64).
template <class F, int MIN_BLOCKS, Steps STEPS>
__global__ void __launch_bounds__(256, MIN_BLOCKS) ntt_pass_kernel(const PassArgs a) {
    extern __shared__ uint4 smem[];
    // Two tile buffers when the block has more than one tile: the copies of its
    // next tile are in flight while the current one is computed.
    const uint32_t CN = 1u << (a.K + a.log_cols);
    uint4 *tab = smem, *buf = smem + 4 * tab_entries(a.K);
    uint32_t tile = blockIdx.x;
    issue_table_load(a, tab);  // (a plan's table: no pass writes it)
    // Passes after the first are launched as programmatic dependents of the
    // pass before, and wait here until that pass has completed and its writes
    // are visible (launched without that attribute, the wait returns at once).
    // A block lets the next pass launch when it starts its last tile, so the
    // next pass's blocks take SM places only as this grid winds down.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (tile < a.num_tiles) issue_tile_load(a, buf, tile, blockDim.x);
    for (uint32_t cur = 0; tile < a.num_tiles; tile += gridDim.x, cur ^= 2 * CN) {
        cp_async_wait_all();
        // the tile is there, and every thread is done with the other buffer
        __syncthreads();
        const uint32_t next = tile + gridDim.x;
        if (next < a.num_tiles) issue_tile_load(a, buf + (cur ^ (2 * CN)), next, blockDim.x);
        else asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        run_tile<F, STEPS>(a, tab, buf + cur, tile, blockDim.x);
    }
}

}  // namespace zkntt
