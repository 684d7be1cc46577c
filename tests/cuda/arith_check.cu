// arith_check.cu -- the field arithmetic of field.cuh, one operation on every element
// of host arrays, for the tests.  Besides the three scalar fields it instantiates two
// moduli whose lowest limb has no shortcut: the general rows of the products.
#include <cuda_runtime.h>

#include "field.cuh"

using namespace zkntt;

// 2^252 + 27742317777372353535851937790883648493: 4r < 2^256
struct General252 {
    static constexpr uint32_t P0 = 0x5cf5d3edu, P1 = 0x5812631au, P2 = 0xa2f79cd6u, P3 = 0x14def9deu,
                              P4 = 0, P5 = 0, P6 = 0, P7 = 0x10000000u;
    static constexpr uint32_t RP = 0x12547e1bu;
};

// 2^255 - 19: 4r > 2^256
struct General255 {
    static constexpr uint32_t P0 = 0xffffffedu, P1 = 0xffffffffu, P2 = 0xffffffffu, P3 = 0xffffffffu,
                              P4 = 0xffffffffu, P5 = 0xffffffffu, P6 = 0xffffffffu,
                              P7 = 0x7fffffffu;
    static constexpr uint32_t RP = 0x286bca1bu;
};

template <class F>
__global__ void check_kernel(int op, const uint4 *a, const uint4 *b, const uint4 *c, uint4 *out,
                             uint4 *out2, size_t n) {
    const size_t i = size_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t x[8], y[8], z[8], r[8] = {0}, s[8] = {0};
    ldg_elem(x, a + 2 * i);
    ldg_elem(y, b + 2 * i);
    ldg_elem(z, c + 2 * i);
    Factor f;
    for (int k = 0; k < 8; k++) {
        f.w[k] = y[k];
        f.wq[k] = z[k];
    }
    switch (op) {
        case 0: mul<F>(r, x, y); break;
        case 1: add_loose<F>(r, x, y); break;
        case 2: sub_loose<F>(r, x, y); break;
        case 3: diff_loose<F>(r, x, y); break;
        case 4: mul_factor<F>(r, x, f); break;
        case 5: mul_high(r, x, y); break;
        case 6: mul_low(r, x, y); break;
        case 7: mul_low_fold<F>(r, x, y, z); break;
        case 8:
            make_factor<F>(f, x, y);
            for (int k = 0; k < 8; k++) {
                r[k] = f.w[k];
                s[k] = f.wq[k];
            }
            break;
        case 9:
            for (int k = 0; k < 8; k++) r[k] = x[k];
            reduce_once<F>(r);
            break;
    }
    st_elem(out + 2 * i, r);
    st_elem(out2 + 2 * i, s);
}

// host arrays of n elements of 32 bytes each; returns a CUDA error code
extern "C" int arith_check(int field, int op, const void *a, const void *b, const void *c, void *out,
                           void *out2, size_t n) {
    const void *k = field == 0   ? (const void *)&check_kernel<FrBLS12_381>
                    : field == 1 ? (const void *)&check_kernel<FrBN254>
                    : field == 2 ? (const void *)&check_kernel<FrBLS12_377>
                    : field == 3 ? (const void *)&check_kernel<General252>
                                 : (const void *)&check_kernel<General255>;
    if (field < 0 || field > 4 || op < 0 || op > 9 || n == 0 || n > (size_t(1) << 24)) return -1;
    const size_t bytes = 32 * n;
    char *d = nullptr;
    cudaError_t e = cudaMalloc(&d, 5 * bytes);
    if (e != cudaSuccess) return int(e);
    const void *in[3] = {a, b, c};
    for (int j = 0; j < 3 && e == cudaSuccess; j++)
        e = cudaMemcpy(d + j * bytes, in[j], bytes, cudaMemcpyHostToDevice);
    char *p[5];
    for (int j = 0; j < 5; j++) p[j] = d + j * bytes;
    void *args[] = {&op, &p[0], &p[1], &p[2], &p[3], &p[4], &n};
    if (e == cudaSuccess)
        e = cudaLaunchKernel(k, dim3(unsigned((n + 127) / 128)), dim3(128), args, 0, nullptr);
    if (e == cudaSuccess) e = cudaMemcpy(out, p[3], bytes, cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(out2, p[4], bytes, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return int(e);
}
