// Host build of the oriented-box fit of the patches above the buckets (obb.cuh),
// by a team of one, for the CPU tests.
#include <math.h>
#include <string.h>
#include <vector>

#include "../paper_2007_07627_gb300/csrc/obb.cuh"

extern "C" {

// pts: cnt float4 (x, y, z, unused); out: 16 floats.
void h_obb_fit_patch(const float *pts, int cnt, float *out) {
    std::vector<float4> p(cnt);
    memcpy(p.data(), pts, sizeof(float4) * (size_t)cnt);
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY}, c[3];
    for (const float4 &q : p) {
        const float v[3] = {q.x, q.y, q.z};
        for (int a = 0; a < 3; ++a) {
            lo[a] = fminf(lo[a], v[a]);
            hi[a] = fmaxf(hi[a], v[a]);
        }
    }
    for (int a = 0; a < 3; ++a) c[a] = 0.5f * lo[a] + 0.5f * hi[a];
    float4 box[4];
    fricp::obb_fit_patch(p.data(), cnt, c, 0, 1, [](float *, int, bool) {}, box);
    memcpy(out, box, sizeof(box));
}

// Squared distances of n points x = xh + xl to the box.
void h_obb_d2(const float *box, const float *xh, const float *xl, int n, float *d2) {
    float4 b[4];
    memcpy(b, box, sizeof(b));
    for (int i = 0; i < n; ++i) d2[i] = fricp::obb_eval(b[0], b[1], b[2], b[3], xh + 3 * i, xl + 3 * i);
}

}
