// FP32 line-engine kernels of compiled lengths (one of four units, built side by side).
#include "line_kernels.cuh"

namespace mm {

const void* line_ct_kernel1(LineKind kind, int L) {
    switch (L) {
        case 256: return line_ct_pick<256>(kind);
        case 512: return line_ct_pick<512>(kind);
        case 1024: return line_ct_pick<1024>(kind);
        default: return nullptr;
    }
}

}  // namespace mm
