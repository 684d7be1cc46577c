// kernels_bls12_377.cu -- kernel instantiations for the bls12_377 scalar field.
#include "field_kernels.cuh"

namespace zkntt {

const FieldKernels &kernels_bls12_377() {
    static const FieldKernels k = make_field_kernels<FrBLS12_377>();
    return k;
}

}  // namespace zkntt
