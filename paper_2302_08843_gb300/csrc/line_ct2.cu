// FP32 line-engine kernels of compiled lengths (one of four units, built side by side).
#include "line_kernels.cuh"

namespace mm {

const void* line_ct_kernel2(LineKind kind, int L) {
    switch (L) {
        case 96: return line_ct_pick<96>(kind);
        case 100: return line_ct_pick<100>(kind);
        case 112: return line_ct_pick<112>(kind);
        case 192: return line_ct_pick<192>(kind);
        case 200: return line_ct_pick<200>(kind);
        case 224: return line_ct_pick<224>(kind);
        default: return nullptr;
    }
}

}  // namespace mm
