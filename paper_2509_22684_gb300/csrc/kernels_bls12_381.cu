// kernels_bls12_381.cu -- kernel instantiations for the bls12_381 scalar field.
#include "field_kernels.cuh"

namespace zkntt {

const FieldKernels &kernels_bls12_381() {
    static const FieldKernels k = make_field_kernels<FrBLS12_381>();
    return k;
}

}  // namespace zkntt
