// band_step_f32.cu -- the FP32 instances of the band step kernel (band_step.cuh).
#include "band_step.cuh"

namespace sev {

int launch_band_step(sev_ctx *hd, int n, float *AB, int ldab, int b, int h, void *ws, size_t ws_bytes) {
    if (!step_shape_ok(b, h)) return SEV_ERR_UNSUPPORTED;
    const int rt = step_rt(b), q = step_q(h);
    // One CTA a sweep for narrow bands: 32 -> 16 at n = 8191 11.5 ms against
    // 14.4 ms on four CTAs (a step's products are short, the exchange through
    // global memory is not); 64 -> 16 at n = 8192 16.7 against 13.9 ms.
    if (b < hd->chase_x3_min_b) {
        if (rt == 1 && q == 2) return launch_step<float, 1, 2, false>(hd, n, AB, ldab, b, h, ws, ws_bytes);
        if (rt == 1 && q == 4) return launch_step<float, 1, 4, false>(hd, n, AB, ldab, b, h, ws, ws_bytes);
        if (rt == 2 && q == 2) return launch_step<float, 2, 2, false>(hd, n, AB, ldab, b, h, ws, ws_bytes);
        if (rt == 2 && q == 4) return launch_step<float, 2, 4, false>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    }
    if (rt == 1 && q == 2) return launch_step<float, 1, 2, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    if (rt == 1 && q == 4) return launch_step<float, 1, 4, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    if (rt == 2 && q == 2) return launch_step<float, 2, 2, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    if (rt == 2 && q == 4) return launch_step<float, 2, 4, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    if (rt == 2 && q == 8) return launch_step<float, 2, 8, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    if (rt == 4 && q == 2) return launch_step<float, 4, 2, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    if (rt == 4 && q == 4) return launch_step<float, 4, 4, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    if (rt == 4 && q == 8) return launch_step<float, 4, 8, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    if (rt == 4 && q == 16) return launch_step<float, 4, 16, true>(hd, n, AB, ldab, b, h, ws, ws_bytes);
    return SEV_ERR_UNSUPPORTED;
}

size_t band_step_workspace(int n, int b, int h) { return step_workspace(n, b, h); }

}  // namespace sev
