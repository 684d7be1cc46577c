// kernels_bn254.cu -- kernel instantiations for the bn254 scalar field.
#include "field_kernels.cuh"

namespace zkntt {

const FieldKernels &kernels_bn254() {
    static const FieldKernels k = make_field_kernels<FrBN254>();
    return k;
}

}  // namespace zkntt
