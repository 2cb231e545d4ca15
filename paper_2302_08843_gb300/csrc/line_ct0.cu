// FP32 line-engine kernels of compiled lengths (one of four units, built side by side).
#include "line_kernels.cuh"

namespace mm {

const void* line_ct_kernel0(LineKind kind, int L) {
    switch (L) {
        case 16: return line_ct_pick<16>(kind);
        case 32: return line_ct_pick<32>(kind);
        case 64: return line_ct_pick<64>(kind);
        case 128: return line_ct_pick<128>(kind);
        default: return nullptr;
    }
}

}  // namespace mm
