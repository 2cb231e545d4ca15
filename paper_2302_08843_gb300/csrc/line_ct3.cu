// FP32 line-engine kernels of compiled lengths (one of four units, built side by side).
#include "line_kernels.cuh"

namespace mm {

const void* line_ct_kernel3(LineKind kind, int L) {
    switch (L) {
        case 384: return line_ct_pick<384>(kind);
        case 400: return line_ct_pick<400>(kind);
        case 448: return line_ct_pick<448>(kind);
        case 768: return line_ct_pick<768>(kind);
        case 800: return line_ct_pick<800>(kind);
        case 896: return line_ct_pick<896>(kind);
        default: return nullptr;
    }
}

}  // namespace mm
