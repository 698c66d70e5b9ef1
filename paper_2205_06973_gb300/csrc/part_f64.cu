// Part interpreter kernels for complex128 states.
#include "part_kernel.cuh"

namespace hisv {

cudaError_t launch_part_f64(int t, int R, void *sv, const PartLaunch &L, const void *stream,
                            const IWindow *windows, uint64_t n_tiles, cudaStream_t st) {
    if (R == 3) {
        switch (t) {
        case 8: return launch_part_t<double, 8, 3>(sv, L, stream, windows, n_tiles, st);
        case 9: return launch_part_t<double, 9, 3>(sv, L, stream, windows, n_tiles, st);
        case 10: return launch_part_t<double, 10, 3>(sv, L, stream, windows, n_tiles, st);
        case 11: return launch_part_t<double, 11, 3>(sv, L, stream, windows, n_tiles, st);
        case 12: return launch_part_t<double, 12, 3>(sv, L, stream, windows, n_tiles, st);
        }
    } else if (R == 4) {   // multi-level plans: a second-level part may need four register qubits
        switch (t) {
        case 10: return launch_part_t<double, 10, 4>(sv, L, stream, windows, n_tiles, st);
        case 11: return launch_part_t<double, 11, 4>(sv, L, stream, windows, n_tiles, st);
        case 12: return launch_part_t<double, 12, 4>(sv, L, stream, windows, n_tiles, st);
        }
    }
    return cudaErrorInvalidValue;
}

}  // namespace hisv
