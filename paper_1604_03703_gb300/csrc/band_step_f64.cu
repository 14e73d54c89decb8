// band_step_f64.cu -- the FP64 instances of the band step kernel (band_step.cuh).
#include "band_step.cuh"

namespace sev {

int launch_band_step(sev_ctx *hd, int n, double *AB, int ldab, int b, int h, void *ws, size_t ws_bytes) {
    if (!step_shape_ok(b, h)) return SEV_ERR_UNSUPPORTED;
    const int rt = step_rt(b), q = step_q(h);
    // Always a CTA per role: a step's products take tens of thousands of cycles
    // of one SM's FP64 pipes even at b = 32.
    if (rt == 1 && q == 2) return launch_step<double, 1, 2, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    if (rt == 1 && q == 4) return launch_step<double, 1, 4, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    if (rt == 2 && q == 2) return launch_step<double, 2, 2, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    if (rt == 2 && q == 4) return launch_step<double, 2, 4, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    if (rt == 2 && q == 8) return launch_step<double, 2, 8, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    if (rt == 4 && q == 2) return launch_step<double, 4, 2, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    if (rt == 4 && q == 4) return launch_step<double, 4, 4, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    if (rt == 4 && q == 8) return launch_step<double, 4, 8, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    return SEV_ERR_UNSUPPORTED;
}

}  // namespace sev
