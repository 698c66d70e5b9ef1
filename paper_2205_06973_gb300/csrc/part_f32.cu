// Part interpreter kernels for complex64 states.
#include "part_kernel.cuh"

namespace hisv {

cudaError_t launch_part_f32(int t, int R, void *sv, const PartLaunch &L, const void *stream,
                            const IWindow *windows, uint64_t n_tiles, cudaStream_t st) {
    if (R == 3) {
        if (t == 10) return launch_part_t<float, 10, 3>(sv, L, stream, windows, n_tiles, st);   // small states
    } else if (R == 4) {
        switch (t) {
        case 10: return launch_part_t<float, 10, 4>(sv, L, stream, windows, n_tiles, st);
        case 11: return launch_part_t<float, 11, 4>(sv, L, stream, windows, n_tiles, st);
        case 12: return launch_part_t<float, 12, 4>(sv, L, stream, windows, n_tiles, st);
        case 13: return launch_part_t<float, 13, 4>(sv, L, stream, windows, n_tiles, st);
        }
    } else if (R == 5) {   // multi-level plans: a second-level part may need five register qubits
        switch (t) {
        case 10: return launch_part_t<float, 10, 5>(sv, L, stream, windows, n_tiles, st);
        case 11: return launch_part_t<float, 11, 5>(sv, L, stream, windows, n_tiles, st);
        case 12: return launch_part_t<float, 12, 5>(sv, L, stream, windows, n_tiles, st);
        case 13: return launch_part_t<float, 13, 5>(sv, L, stream, windows, n_tiles, st);
        }
    }
    return cudaErrorInvalidValue;
}

}  // namespace hisv
