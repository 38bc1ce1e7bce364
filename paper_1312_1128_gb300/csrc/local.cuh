// local.cuh -- local expansions of a ray group's far field (FP32 trees).
//
// A source whose distance from the group is several times the group's own
// size has a smooth field over the group: instead of evaluating it for every
// ray, one lane adds its Taylor coefficients about the centre of the group's
// box, and the sum of all such sources is evaluated once per ray.  With zeta =
// (ray - centre) / d, d the half diagonal of the box, and A = conj(alpha)
// (Sec. 3.2; gamma = conj(dA/dz), kappa = dA/dz*):
//   point mass, far cell:  A = M/w + Q2/w^3, w = w0 + d zeta, so with u = 1/w0
//     the coefficient of zeta^k is (-d u)^k u (M + (k+1)(k+2)/2 Q2 u^2);
// So the field of all sources is one complex polynomial h(zeta) of degree
// kLocP.  A source is expanded if d/|w0| <= 0.18; the first omitted term, at
// the corners of the box (the worst rays), is then at most 0.18^12 = 1.2e-9 of
// the source's own alpha and 13 times that of its gamma: below the rounding of
// one FP32 evaluation.  (One order more costs every expanded source 10
// operations; one fewer leaves 1.4 times as many sources to be evaluated ray
// by ray, at 18 operations each.)
//
// Point masses and NFW trees only.  A listed Gaussian's correction can be
// expanded too (the same h with masses that depend on the order, and a real
// polynomial for kappa), and halved the instructions of the 1e6-particle map;
// but at one lane per source its code is 600 instructions executed a few times
// per flush, which held the kernel in instruction fetch (2.7 of 7 stall cycles;
// walk 21.7 against 22.4 ms at 2048^2 rays, slower at 1024^2), and kappa in the
// sparse outskirts, where one particle's tail is all there is, lost digits.
#pragma once

#include "profiles.cuh"

namespace lens {

constexpr int kLocP = 11;
constexpr int kLocH = 2 * (kLocP + 1);                      // 24 reals of h
constexpr float kLocRho2 = 0.18f * 0.18f;                     // (d/|w0|)^2

// A warp's running coefficients (Neumaier sums), spread over the lanes:
// slots 0 (reals 0..15 of h, one per two lanes) and 1 (reals 16..23, one per
// four).
struct LocalSum {
    float s[2][32], c[2][32];
};

// The finished coefficients of a group.
struct LocalFields {
    float h[kLocH];
};

// Sum v[i] over the warp for N = 2^m values at once: each exchange halves the
// values a lane carries.  Lane l returns the total of value l / (32 / N).
template <int N> LENS_DEV float lane_totals(float (&v)[N])
{
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int n = N / 2; n >= 1; n >>= 1, o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < n; ++i) {
            const float give = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    float t = v[0];
    for (; o >= 1; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    return t;
}

LENS_DEV void local_zero(LocalSum& L)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int q = 0; q < 2; ++q) L.s[q][lane] = L.c[q][lane] = 0.0f;
}

LENS_DEV void local_add(LocalSum& L, int q, float v)
{
    const int lane = threadIdx.x & 31;
    float s = L.s[q][lane], c = L.c[q][lane];
    Comp5<float>::add1(s, c, v);
    L.s[q][lane] = s;
    L.c[q][lane] = c;
}

// Every ray of the group is at least this fraction of |w0| away from an
// expanded source (squared).
constexpr float kLocNear2 = (1.0f - 0.18f) * (1.0f - 0.18f) * 0.9999f;

// Half diagonal of the group's box (no underflow for the smallest boxes).
LENS_DEV float box_radius(float hx, float hy)
{
    const float a = fmaxf(hx, hy), b = fminf(hx, hy) / a;
    return a * sqrtf(fmaf(b, b, 1.0f));
}

// Scale d of a group's expansion: its half diagonal, but at least an FP32
// rounding (2^-24) of the root's r_cm.  A group of one ray
// has a half diagonal of 1e-30; the coefficient of zeta is then d m / w^2, below
// the normal numbers for m / w^2 < 1e-8, and its quotient by d, gamma, is lost.
// Sources nearer than d / 0.18 are evaluated ray by ray, so a larger d only
// makes the expansion's remainder smaller.
LENS_DEV float local_scale(float hx, float hy, float root_rcm)
{
    return fmaxf(box_radius(hx, hy), 5.9604645e-8f * root_rcm);
}

// A lane's share of h.
struct LocalH {
    float v[kLocH];
    LENS_DEV void zero()
    {
#pragma unroll
        for (int i = 0; i < kLocH; ++i) v[i] = 0.0f;
    }
    // a far cell at separation w0 (inv = 1/|w0|^2)
    LENS_DEV void cell(float wx, float wy, float inv, float d, float M, float qr, float qi)
    {
        const float ux = wx * inv, uy = -wy * inv;
        const float sx = -d * ux, sy = -d * uy;  // ratio of successive orders
        const float u2x = fmaf(ux, ux, -uy * uy), u2y = (ux + ux) * uy;
        const float ax = fmaf(qr, u2x, -qi * u2y), ay = fmaf(qr, u2y, qi * u2x);
        float px = ux, py = uy;
#pragma unroll
        for (int k = 0; k <= kLocP; ++k) {
            const float b = 0.5f * (k + 1) * (k + 2);
            const float cx = fmaf(b, ax, M), cy = b * ay;
            v[2 * k] = fmaf(px, cx, fmaf(-py, cy, v[2 * k]));
            v[2 * k + 1] = fmaf(px, cy, fmaf(py, cx, v[2 * k + 1]));
            const float t = px;
            px = fmaf(px, sx, -py * sy);
            py = fmaf(t, sy, py * sx);
        }
    }
    LENS_DEV void point(float wx, float wy, float inv, float d, float m)
    {
        const float ux = wx * inv, uy = -wy * inv;
        const float sx = -d * ux, sy = -d * uy;
        float px = m * ux, py = m * uy;
#pragma unroll
        for (int k = 0; k <= kLocP; ++k) {
            v[2 * k] += px;
            v[2 * k + 1] += py;
            const float t = px;
            px = fmaf(px, sx, -py * sy);
            py = fmaf(t, sy, py * sx);
        }
    }
};

// The finished coefficients of a group, by all lanes of its warp.
LENS_DEV void local_finish(const LocalSum& L, LocalFields& F)
{
    const int lane = threadIdx.x & 31;
    __syncwarp();
    const float t0 = L.s[0][lane] + L.c[0][lane], t1 = L.s[1][lane] + L.c[1][lane];
    if ((lane & 1) == 0) F.h[lane >> 1] = t0;
    if ((lane & 3) == 0) F.h[16 + (lane >> 2)] = t1;
    __syncwarp();
}

// The expansion at offset (x, y) = (ray - centre) / d: alpha, and gamma
// unless AO.  id = 1/d.
template <bool AO> LENS_DEV void local_eval(const LocalFields& F, float x, float y, float id, Acc5<float>& acc)
{
    // h and its derivative
    float ax = F.h[2 * kLocP], ay = F.h[2 * kLocP + 1], bx = 0.0f, by = 0.0f;
#pragma unroll
    for (int k = kLocP - 1; k >= 0; --k) {
        if (!AO) {
            const float t = bx;
            bx = fmaf(bx, x, fmaf(-by, y, ax));
            by = fmaf(t, y, fmaf(by, x, ay));
        }
        const float t = ax;
        ax = fmaf(ax, x, fmaf(-ay, y, F.h[2 * k]));
        ay = fmaf(t, y, fmaf(ay, x, F.h[2 * k + 1]));
    }
    acc.a1 += ax;
    acc.a2 -= ay;
    if (!AO) {
        acc.g1 = fmaf(bx, id, acc.g1);
        acc.g2 = fmaf(-by, id, acc.g2);
    }
}

}  // namespace lens
