// Instantiation of the fused stream-and-collide kernels for f64 population storage.
#include "launchers.cuh"

namespace nomrt {
const Launchers &launchers_f64() {
    static const Launchers L = make_launchers<double>();
    return L;
}
}  // namespace nomrt
