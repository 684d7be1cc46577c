// field_kernels.cuh -- the kernel table of one field (included by the
// field-specific translation units).
#pragma once
#include "aux_kernels.cuh"
#include "kernels.h"
#include "ntt_pass.cuh"

namespace zkntt {

static_assert(NUM_KINDS == PASS_KINDS, "the kernel tables have a place for every kind");

// the pass kernels compiled for a digit of K bits: one thread per four elements
// of a tile, 128 registers (2^24: 2594 us, with 96 2606, with 80 2702)
template <class F, int K, Kind KIND>
const void *fixed_kernel() {
    constexpr int T = 1 << (K + fixed_cols(K) - 2);
    constexpr int B = T >= 32 ? 512 / T : 16;
    return (const void *)&ntt_pass_kernel<F, T, B, RADIX4, K, KIND>;
}

// the same one butterfly a thread and stage, in tiles of one column, for small
// transforms: 128 registers
template <class F, int K, Kind KIND>
const void *wide_kernel() {
    constexpr int T = 1 << (K + fixed_cols(K, RADIX2) - 1);
    return (const void *)&ntt_pass_kernel<F, T, T >= 32 ? 512 / T : 16, RADIX2, K, KIND>;
}

template <class F, int K>
void set_wide(FieldKernels &k) {
    k.wide[K][STRIDED] = wide_kernel<F, K, STRIDED>();
    k.wide[K][STRIDED_PRE] = wide_kernel<F, K, STRIDED_PRE>();
    k.wide[K][LAST] = wide_kernel<F, K, LAST>();
    k.wide[K][LAST_POST] = wide_kernel<F, K, LAST_POST>();
}

template <class F, int K>
void set_fixed(FieldKernels &k) {
    k.fixed[K][STRIDED] = fixed_kernel<F, K, STRIDED>();
    k.fixed[K][STRIDED_PRE] = fixed_kernel<F, K, STRIDED_PRE>();
    k.fixed[K][STRIDED_OTF] = fixed_kernel<F, K, STRIDED_OTF>();
    k.fixed[K][LAST] = fixed_kernel<F, K, LAST>();
    k.fixed[K][LAST_POST] = fixed_kernel<F, K, LAST_POST>();
}

template <class F>
FieldKernels make_field_kernels() {
    FieldKernels k = {};
    k.any4 = (const void *)&ntt_pass_kernel<F, 256, 2, RADIX4, 0, ANY>;
    k.any2 = (const void *)&ntt_pass_kernel<F, 256, 2, RADIX2, 0, ANY>;
    set_wide<F, 5>(k);
    set_wide<F, 6>(k);
    set_wide<F, 7>(k);
    set_wide<F, 8>(k);
    set_wide<F, 9>(k);
    set_fixed<F, 5>(k);
    set_fixed<F, 6>(k);
    set_fixed<F, 7>(k);
    set_fixed<F, 8>(k);
    set_fixed<F, 9>(k);
    set_fixed<F, 10>(k);
    k.gen_powers = (const void *)&gen_powers_kernel<F>;
    k.gen_twiddle = (const void *)&gen_twiddle_kernel<F>;
    k.field_op = (const void *)&field_op_kernel<F>;
    k.pointwise = (const void *)&pointwise_kernel<F>;
    k.mulbench = (const void *)&mulbench_kernel<F>;
    k.scale_powers = (const void *)&scale_powers_kernel<F>;
    k.block_dft[1] = (const void *)&block_dft_kernel<F, 2>;
    k.block_dft[2] = (const void *)&block_dft_kernel<F, 4>;
    k.block_dft[3] = (const void *)&block_dft_kernel<F, 8>;
    return k;
}

}  // namespace zkntt
