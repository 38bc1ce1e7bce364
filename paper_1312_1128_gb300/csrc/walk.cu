// walk.cu -- ray grouping and the warp-cooperative tree walk (Sec. 3.2 tree
// walk, Sec. 3.3 ray-parallel evaluation), plus the direct sum (Sec. 5.1,
// theta_force = 0) and the analytic components evaluated for every ray.
//
// One warp owns a group of up to 32*R spatially sorted rays and walks the tree
// once for the whole group:
//   - up to 32 candidate boxes are taken from the warp's stack at a time, one
//     per lane, and the MAC |x - x_cm| > r_cut is applied to the group's
//     bounding box (accepting a box only if every ray of the group would);
//   - accepted boxes go to a far buffer (monopole + quadrupole), opened leaves
//     to a near buffer of particle records, opened internal boxes push their
//     children; the big list of every visited box is scanned and the
//     particles whose support reaches the group's box go to a big buffer;
//   - full buffers are evaluated by all lanes, each lane for its own rays,
//     with the records broadcast from shared memory; partial sums are folded
//     into Neumaier-compensated totals after every buffer.
// Big-particle semantics (Sec. 3.2): every box's moments include all its
// particles as point masses.  A listed particle counts inside leaves as a
// point mass softened within r0 = min(s, r_cm(leaf)(1/theta - 1)), which is
// exactly the point mass wherever a cell containing it can be accepted, and
// its box's list adds (full profile - softened point) for rays inside its
// support s.  The softening removes the cancellation of a huge point term
// against its correction when a ray passes close to a listed particle.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "profiles.cuh"
#include "sort.cuh"
#include "walk_shared.cuh"
#include "walk_dev.cuh"

namespace lens {

// ------------------------------------------------------------ grouping

__global__ void k_ray_bbox(const int64_t* boff, int nb, const double* borig, const void* dx,
                           const void* dy, int dtype, int64_t n, unsigned long long* bbox)
{
    __shared__ unsigned long long red[4][8];
    __shared__ int bsame;
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool valid = i < n;
    int b = valid ? batch_of(boff, nb, i) : -1;
    double px = 0, py = 0;
    if (valid) {
        px = borig[2 * b] + ray_offset(dx, dtype, i);
        py = borig[2 * b + 1] + ray_offset(dy, dtype, i);
    }
    // whole block in one batch (the common case): reduce in the block, then
    // four atomics per block
    int64_t first = (int64_t)blockIdx.x * blockDim.x;
    int64_t last = first + blockDim.x - 1 < n - 1 ? first + blockDim.x - 1 : n - 1;
    if (threadIdx.x == 0) bsame = batch_of(boff, nb, first) == batch_of(boff, nb, last);
    __syncthreads();
    const unsigned full = 0xffffffffu;
    unsigned long long x0 = valid ? dbl_to_ordered(px) : ~0ull, x1 = valid ? dbl_to_ordered(px) : 0ull;
    unsigned long long y0 = valid ? dbl_to_ordered(py) : ~0ull, y1 = valid ? dbl_to_ordered(py) : 0ull;
    if (bsame) {
        for (int o = 16; o; o >>= 1) {
            x0 = min(x0, __shfl_xor_sync(full, x0, o));
            x1 = max(x1, __shfl_xor_sync(full, x1, o));
            y0 = min(y0, __shfl_xor_sync(full, y0, o));
            y1 = max(y1, __shfl_xor_sync(full, y1, o));
        }
        int w = threadIdx.x >> 5;
        if ((threadIdx.x & 31) == 0) {
            red[0][w] = x0; red[1][w] = x1; red[2][w] = y0; red[3][w] = y1;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int bb = batch_of(boff, nb, first);
            for (int k = 1; k < (int)(blockDim.x >> 5); ++k) {
                red[0][0] = min(red[0][0], red[0][k]);
                red[1][0] = max(red[1][0], red[1][k]);
                red[2][0] = min(red[2][0], red[2][k]);
                red[3][0] = max(red[3][0], red[3][k]);
            }
            atomicMin(&bbox[4 * bb + 0], red[0][0]);
            atomicMax(&bbox[4 * bb + 1], red[1][0]);
            atomicMin(&bbox[4 * bb + 2], red[2][0]);
            atomicMax(&bbox[4 * bb + 3], red[3][0]);
        }
        return;
    }
    if (!valid) return;
    atomicMin(&bbox[4 * b + 0], x0);
    atomicMax(&bbox[4 * b + 1], x1);
    atomicMin(&bbox[4 * b + 2], y0);
    atomicMax(&bbox[4 * b + 3], y1);
}

__global__ void k_bbox_init(unsigned long long* bbox, int64_t nb)
{
    int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nb) return;
    bbox[4 * b] = ~0ull;
    bbox[4 * b + 1] = 0ull;
    bbox[4 * b + 2] = ~0ull;
    bbox[4 * b + 3] = 0ull;
}

// Order-preserving map of a float to uint32.
__device__ __forceinline__ uint32_t flt_to_ordered(float f)
{
    uint32_t u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float ordered_to_flt(uint32_t u)
{
    u = (u & 0x80000000u) ? (u & 0x7fffffffu) : ~u;
    return __uint_as_float(u);
}

__device__ __forceinline__ uint32_t spread16(uint32_t x)
{
    x &= 0xffffu;
    x = (x | (x << 8)) & 0x00ff00ffu;
    x = (x | (x << 4)) & 0x0f0f0f0fu;
    x = (x | (x << 2)) & 0x33333333u;
    x = (x | (x << 1)) & 0x55555555u;
    return x;
}

__global__ void k_ray_keys(const int64_t* boff, int nb, const double* borig, const void* dx,
                           const void* dy, int dtype, int64_t n, const unsigned long long* bbox,
                           uint64_t* keys, uint32_t* vals)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int b = batch_of(boff, nb, i);
    double px = borig[2 * b] + ray_offset(dx, dtype, i);
    double py = borig[2 * b + 1] + ray_offset(dy, dtype, i);
    double x0 = ordered_to_dbl(bbox[4 * b]), x1 = ordered_to_dbl(bbox[4 * b + 1]);
    double y0 = ordered_to_dbl(bbox[4 * b + 2]), y1 = ordered_to_dbl(bbox[4 * b + 3]);
    double ext = fmax(x1 - x0, y1 - y0);
    double inv = ext > 0 ? 65535.99 / ext : 0.0;
    uint32_t qx = (uint32_t)fmin(fmax((px - x0) * inv, 0.0), 65535.0);
    uint32_t qy = (uint32_t)fmin(fmax((py - y0) * inv, 0.0), 65535.0);
    keys[i] = ((uint64_t)b << 32) | (uint64_t)(spread16(qx) | (spread16(qy) << 1));
    vals[i] = (uint32_t)i;
}

// Mark group g if its box is stretched (kStretch): ex, ey = half sides of an
// even share of its batch.
template <typename T>
__device__ __forceinline__ void mark_stretched(int64_t g, T hx, T hy, T ex, T ey, uint8_t* gflag, uint32_t* sub)
{
    const bool st = (hx > T(kStretch) * ex && hx > T(1e-25)) || (hy > T(kStretch) * ey && hy > T(1e-25));
    gflag[g] = st ? 1 : 0;
    if (st) sub[16 + atomicAdd(sub, 1u)] = (uint32_t)g;
}

template <typename T, int R>
__global__ void k_groups(int64_t n_groups, const int64_t* boff, const uint32_t* gfirst, int nb,
                         const double* borig, const void* dx, const void* dy, int dtype,
                         const uint32_t* svals, v2_t<T>* gH, vec4_t<T>* gbox, uint2* grange,
                         v2_t<T>* ray_l, uint32_t* ray_idx, const unsigned long long* bbox, const uint32_t* bb32,
                         uint8_t* gflag, uint32_t* sub)
{
    const unsigned full = 0xffffffffu;
    int lane = threadIdx.x & 31;
    int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (g >= n_groups) return;
    int lo = 0, hi = nb;
    while (hi - lo > 1) {
        int mid = (lo + hi) >> 1;
        if ((int64_t)gfirst[mid] <= g) lo = mid;
        else hi = mid;
    }
    const int b = lo;
    const int GR = 32 * R;
    int64_t first = boff[b] + (g - (int64_t)gfirst[b]) * GR;
    int64_t cnt64 = boff[b + 1] - first;
    int count = (int)(cnt64 < GR ? cnt64 : GR);
    double px[R], py[R];
    uint32_t idx[R];
    bool v[R];
    double xmin = INFINITY, xmax = -INFINITY, ymin = INFINITY, ymax = -INFINITY;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        int k = r * 32 + lane;
        v[r] = k < count;
        idx[r] = 0;
        px[r] = py[r] = 0.0;
        if (v[r]) {
            idx[r] = svals[first + k];
            px[r] = borig[2 * b] + ray_offset(dx, dtype, idx[r]);
            py[r] = borig[2 * b + 1] + ray_offset(dy, dtype, idx[r]);
            xmin = fmin(xmin, px[r]); xmax = fmax(xmax, px[r]);
            ymin = fmin(ymin, py[r]); ymax = fmax(ymax, py[r]);
        }
    }
    for (int o = 16; o; o >>= 1) {
        xmin = fmin(xmin, __shfl_xor_sync(full, xmin, o));
        xmax = fmax(xmax, __shfl_xor_sync(full, xmax, o));
        ymin = fmin(ymin, __shfl_xor_sync(full, ymin, o));
        ymax = fmax(ymax, __shfl_xor_sync(full, ymax, o));
    }
    // Anchor: if every ray of the group is exactly representable in T (for
    // example FP32 rays with origin 0), H = 0 keeps each separation a single
    // rounding of (ray - particle); otherwise H is the T value nearest the
    // group centre, so that far from the coordinate zero the small offsets
    // l = ray - H keep their resolution.
    bool exact = true;
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (v[r]) exact = exact && (double)(T)px[r] == px[r] && (double)(T)py[r] == py[r];
    exact = __all_sync(full, exact);
    T Hx = exact ? T(0) : (T)(0.5 * (xmin + xmax)), Hy = exact ? T(0) : (T)(0.5 * (ymin + ymax));
    T lxmin = (T)INFINITY, lxmax = (T)-INFINITY, lymin = (T)INFINITY, lymax = (T)-INFINITY;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        if (!v[r]) continue;
        T lx = (T)(px[r] - (double)Hx), ly = (T)(py[r] - (double)Hy);
        lxmin = fmin(lxmin, lx); lxmax = fmax(lxmax, lx);
        lymin = fmin(lymin, ly); lymax = fmax(lymax, ly);
        v2_t<T> l;
        l.x = lx;
        l.y = ly;
        ray_l[first + r * 32 + lane] = l;
        ray_idx[first + r * 32 + lane] = idx[r];
    }
    for (int o = 16; o; o >>= 1) {
        lxmin = fmin(lxmin, __shfl_xor_sync(full, lxmin, o));
        lxmax = fmax(lxmax, __shfl_xor_sync(full, lxmax, o));
        lymin = fmin(lymin, __shfl_xor_sync(full, lymin, o));
        lymax = fmax(lymax, __shfl_xor_sync(full, lymax, o));
    }
    if (lane == 0) {
        T cx = T(0.5) * (lxmin + lxmax), cy = T(0.5) * (lymin + lymax);
        T hx = fmax(lxmax - cx, cx - lxmin), hy = fmax(lymax - cy, cy - lymin);
        // inflate so that every ray is inside after rounding
        hx = hx * T(1.0 + 1e-5) + T(1e-30);
        hy = hy * T(1.0 + 1e-5) + T(1e-30);
        v2_t<T> H;
        H.x = Hx;
        H.y = Hy;
        gH[g] = H;
        vec4_t<T> bx;
        bx.x = cx; bx.y = cy; bx.z = hx; bx.w = hy;
        gbox[g] = bx;
        grange[g] = make_uint2((uint32_t)first, (uint32_t)count);
        const float share = 0.5f * sqrtf((float)GR / (float)(boff[b + 1] - boff[b]));
        float wx, wy;
        if (bb32) {
            wx = ordered_to_flt(bb32[2]) - ordered_to_flt(bb32[0]);
            wy = ordered_to_flt(bb32[3]) - ordered_to_flt(bb32[1]);
        } else {
            wx = (float)(ordered_to_dbl(bbox[4 * b + 1]) - ordered_to_dbl(bbox[4 * b]));
            wy = (float)(ordered_to_dbl(bbox[4 * b + 3]) - ordered_to_dbl(bbox[4 * b + 2]));
        }
        mark_stretched<T>(g, hx, hy, (T)(wx * share), (T)(wy * share), gflag, sub);
    }
}

// One batch of FP32 offsets (the common case) needs no FP64 on the grouping
// path (FP64 runs at 1/64 of the FP32 rate here): the offsets' bounding box
// from order-preserving uint32 images of the floats, 32-bit Morton keys of
// the offsets (relative positions do not depend on the origin), and, when
// the origin is zero, groups anchored at H = 0 with l = the offsets
// themselves -- what the FP64 path computes in that case.
// bb = {min x, min y, max x, max y} as ordered images; the caller sets the
// minima to 0xffffffff and the maxima to 0 first.
__global__ void __launch_bounds__(256) k_ray_bbox32(const float* dx, const float* dy, int64_t n, uint32_t* bb)
{
    __shared__ uint32_t red[4][8];
    const unsigned full = 0xffffffffu;
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint32_t v[4] = {~0u, ~0u, 0u, 0u};
    if (i < n) {
        v[0] = v[2] = flt_to_ordered(dx[i]);
        v[1] = v[3] = flt_to_ordered(dy[i]);
    }
    for (int o = 16; o; o >>= 1) {
        v[0] = min(v[0], __shfl_xor_sync(full, v[0], o));
        v[1] = min(v[1], __shfl_xor_sync(full, v[1], o));
        v[2] = max(v[2], __shfl_xor_sync(full, v[2], o));
        v[3] = max(v[3], __shfl_xor_sync(full, v[3], o));
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0)
        for (int q = 0; q < 4; ++q) red[q][w] = v[q];
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) {
            v[0] = min(v[0], red[0][k]);
            v[1] = min(v[1], red[1][k]);
            v[2] = max(v[2], red[2][k]);
            v[3] = max(v[3], red[3][k]);
        }
        atomicMin(&bb[0], v[0]);
        atomicMin(&bb[1], v[1]);
        atomicMax(&bb[2], v[2]);
        atomicMax(&bb[3], v[3]);
    }
}

__global__ void k_ray_keys32(const float* dx, const float* dy, int64_t n, const uint32_t* bb, uint32_t* keys,
                             uint32_t* vals)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float x0 = ordered_to_flt(bb[0]), y0 = ordered_to_flt(bb[1]);
    const float ext = fmaxf(ordered_to_flt(bb[2]) - x0, ordered_to_flt(bb[3]) - y0);
    const float inv = ext > 0.f ? 65535.99f / ext : 0.f;
    const uint32_t qx = (uint32_t)fminf(fmaxf((dx[i] - x0) * inv, 0.f), 65535.f);
    const uint32_t qy = (uint32_t)fminf(fmaxf((dy[i] - y0) * inv, 0.f), 65535.f);
    keys[i] = spread16(qx) | (spread16(qy) << 1);
    vals[i] = (uint32_t)i;
}

// Groups of one batch of FP32 offsets at origin zero: every ray is exact in
// T, so H = 0 and l = the offset (as k_groups then has it).
template <typename T, int R>
__global__ void k_groups32(int64_t n_groups, int64_t n, const float* dx, const float* dy, const uint32_t* svals,
                           v2_t<T>* gH, vec4_t<T>* gbox, uint2* grange, v2_t<T>* ray_l, uint32_t* ray_idx,
                           const uint32_t* bb32, uint8_t* gflag, uint32_t* sub)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (g >= n_groups) return;
    const int64_t first = g * (32 * R);
    const int count = (int)(n - first < 32 * R ? n - first : 32 * R);
    T lxmin = (T)INFINITY, lxmax = (T)-INFINITY, lymin = (T)INFINITY, lymax = (T)-INFINITY;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int k = r * 32 + lane;
        if (k >= count) continue;
        const uint32_t idx = svals[first + k];
        v2_t<T> l;
        l.x = (T)dx[idx];
        l.y = (T)dy[idx];
        lxmin = fmin(lxmin, l.x); lxmax = fmax(lxmax, l.x);
        lymin = fmin(lymin, l.y); lymax = fmax(lymax, l.y);
        ray_l[first + k] = l;
        ray_idx[first + k] = idx;
    }
    for (int o = 16; o; o >>= 1) {
        lxmin = fmin(lxmin, __shfl_xor_sync(full, lxmin, o));
        lxmax = fmax(lxmax, __shfl_xor_sync(full, lxmax, o));
        lymin = fmin(lymin, __shfl_xor_sync(full, lymin, o));
        lymax = fmax(lymax, __shfl_xor_sync(full, lymax, o));
    }
    if (lane == 0) {
        T cx = T(0.5) * (lxmin + lxmax), cy = T(0.5) * (lymin + lymax);
        T hx = fmax(lxmax - cx, cx - lxmin), hy = fmax(lymax - cy, cy - lymin);
        hx = hx * T(1.0 + 1e-5) + T(1e-30);
        hy = hy * T(1.0 + 1e-5) + T(1e-30);
        v2_t<T> H;
        H.x = T(0);
        H.y = T(0);
        gH[g] = H;
        vec4_t<T> bx;
        bx.x = cx; bx.y = cy; bx.z = hx; bx.w = hy;
        gbox[g] = bx;
        grange[g] = make_uint2((uint32_t)first, (uint32_t)count);
        const float share = 0.5f * sqrtf((float)(32 * R) / (float)n);
        mark_stretched<T>(g, hx, hy, (T)((ordered_to_flt(bb32[2]) - ordered_to_flt(bb32[0])) * share),
                          (T)((ordered_to_flt(bb32[3]) - ordered_to_flt(bb32[1])) * share), gflag, sub);
    }
}

// ---------------------------------------------------------------- walk

// LOC: with local expansions (local.cuh).  FP32 NFW trees, and point masses
// where the groups are many enough for supergroups (launch_super).
template <int KIND, typename T, int R, bool AO, bool DIRECT, int TILE, bool LOC>
__global__ void __launch_bounds__(kWalkWarps * 32, sizeof(T) == 4 ? (LOC || R == 4 ? 4 : (R == 2 ? 4 : 5)) : 2)
walk_kernel(const __grid_constant__ WalkParams<T> P)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const unsigned full = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    using WS = WalkShared<KIND, T, TILE, tot_rays<R>()>;
    WS& S = reinterpret_cast<WS*>(smem_raw)[warp];
    int* stack = P.stack + ((int64_t)blockIdx.x * kWalkWarps + warp) * kStackCap;
    using Ctx = WalkCtx<KIND, T, R, AO, TILE, LOC>;
    Ctx C(P, S);

    const int NS = DIRECT && P.n_slices > 1 ? P.n_slices : 1;
    for (;;) {
        uint32_t slice = 0, g = 0;
        if constexpr (DIRECT) {
            uint32_t item = 0;
            if (lane == 0) item = atomicAdd(P.counter, 1u);
            item = __shfl_sync(full, item, 0);
            if ((int64_t)item >= P.n_groups * NS) break;
            slice = item % (uint32_t)NS;
            g = item / (uint32_t)NS;
        } else {
            if (!next_item<R>(P, stack, S.cut)) break;
            g = S.cut.g;
        }
        // the group's first (or only) item
        const bool head = DIRECT ? slice == 0 : S.cut.item == kNoItem;
        C.load_group(g);
        if constexpr (DIRECT) {
            C.start();
            if (KIND >= 0 && P.n_part > 0) {
                // every particle of this item's slice with its full profile
                const int64_t p0 = P.n_part * slice / NS, p1 = P.n_part * (slice + 1) / NS;
                for (int64_t base = p0; base < p1; base += 0x40000000) {
                    int64_t rem = p1 - base;
                    int c = (int)(rem < 0x40000000 ? rem : 0x40000000);
                    append_ranges(C, lane == 0 ? c : 0, (int)base, P.leaf0, P.leaf1);
                }
                C.flush_near();
            }
            if (P.n_halos > 0 && head) Ctx::Flush::finish(P.halos, P.n_halos, nullptr, float4{});
        } else {
            C.rec = P.list_ids ? P.list_ids + (int64_t)g * P.list_K : nullptr;
            C.rec_shared = head ? nullptr : P.list_n + g;
            C.rec_n = 0;
            C.rec_cap = P.list_K;
            do {  // (once, or once for each part of a cut whose pool was full)
                C.start();
                const bool whole = traverse(C, stack, S.cut.sp);
                if (C.rec && lane == 0) {
                    // (above the room, whatever parts add to it: the lists did not fit)
                    if (head) P.list_n[g] = whole && C.rec_n <= C.rec_cap && (S.cut.seg == 0 || P.list_n[g] != kListTooLong)
                                                ? (uint32_t)C.rec_n : kListTooLong;
                    else if (!whole) atomicOr(P.list_n + g, kListTooLong);
                }
                C.flush_far();
                C.flush_near();
                C.flush_big();
                const bool first = head && S.cut.seg == 0;
                const SuperRec* sr = nullptr;
                float4 delta = make_float4(0.f, 0.f, 0.f, 0.f);
                if constexpr (LOC) {
                    if (P.super && first && P.super[g / kSuperGroups].ok == 1) {
                        sr = P.super + g / kSuperGroups;
                        delta = P.sdelta[g];
                    }
                }
                Ctx::Flush::finish(P.halos, first ? P.n_halos : 0, sr, delta);
                // (a part's cut counts from its own start)
                count_item(C, g, first);
                C.c_vis = C.c_acc = C.c_near = C.c_bigs = C.c_bigk = 0;
            } while (S.cut.local && local_next_part<R, AO ? 2 : 5>(P.cut, S.cut, stack,
                                                                   [&](int r, int q) { return C.total(r, q); }));
        }
        __syncwarp();
        const uint2 rg = P.grange[g];
        if constexpr (DIRECT) count_item(C, g, head);

        T* tot = DIRECT ? nullptr : item_totals<R>(P.cut, S.cut);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int k = r * 32 + lane;
            const bool ray = k < (int)rg.y;
            if (!ray && !tot) continue;
            const uint32_t i = ray ? P.ray_idx[rg.x + k] : 0u;
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                if (AO && q >= 2) break;
                T val = C.total(r, q);
                if (!DIRECT && S.cut.local) val = local_total<R>(P.cut, r, q);
                if (NS > 1) {
                    P.split[((int64_t)slice * 5 + q) * P.split_n + i] = val;
                    continue;
                }
                if (tot) {
                    tot[(q * R + r) * 32 + lane] = val;
                    continue;
                }
                if (P.accumulate) val += P.out[q][i];
                P.out[q][i] = val;
            }
        }
        __syncwarp();
    }
}

// The plain tree walk: whole groups, without expansions, fewer registers than
// the cut form; with P.skip all but the stretched ones.  CUTS: heavy groups
// (cut_limit) hand the rest of their walk to parts (FP32 point masses only: the
// code cost Gaussian trees 4 to 8 % on calls that cut nothing).
template <int KIND, typename T, int R, bool AO, int TILE, bool CUTS>
__global__ void __launch_bounds__(kWalkWarps * 32, sizeof(T) == 4 ? (R == 4 ? 4 : (R == 2 ? 5 : 6)) : 2)
walk_plain(const __grid_constant__ WalkParams<T> P)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const unsigned full = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    PlainShared<KIND, T, TILE, tot_rays<R>()>& S = reinterpret_cast<PlainShared<KIND, T, TILE, tot_rays<R>()>*>(smem_raw)[warp];
    int* stack = P.stack + ((int64_t)blockIdx.x * kWalkWarps + warp) * kStackCap;
    PlainCtx<KIND, T, R, AO, TILE, CUTS> C(P, &S.buf, &S.tot, &S.rng, &S.cut);
    if (P.super && P.super[0].ok != 3) return;  // the supergroups' walk has run
    // the rays' indices are read again after the walk where they cost it spills
    constexpr bool kAgain = CUTS || KIND != LENS_POINT;
    uint32_t ridx[R];
    bool rv[R];
    for (;;) {
        uint32_t item = 0;
        if (lane == 0) item = atomicAdd(P.counter, 1u);
        item = __shfl_sync(full, item, 0);
        if ((int64_t)item >= P.n_groups) break;
        const uint32_t g = P.order ? P.order[item] : item;
        if (!CUTS && P.skip && P.gflag[g]) continue;
        whole_group(P, S.cut, g, stack);
        C.H = P.gH[g];
        C.box = P.gbox[g];
        uint2 rg = P.grange[g];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int k = r * 32 + lane;
            rv[r] = k < (int)rg.y;
            if (rv[r]) {
                const v2_t<T> l = P.ray_l[rg.x + k];
                C.lx[r] = l.x;
                C.ly[r] = l.y;
                ridx[r] = P.ray_idx[rg.x + k];
            } else {
                C.lx[r] = C.box.x;
                C.ly[r] = C.box.y;
                ridx[r] = 0;
            }
            C.part[r].zero();
        }
        C.tot_zero();
        C.c_vis = C.c_acc = C.c_near = C.c_bigs = C.c_bigk = 0;
        C.nf = C.nn = C.nb = 0;
        C.rec = P.list_ids ? P.list_ids + (int64_t)g * P.list_K : nullptr;
        C.rec_n = 0;
        C.rec_cap = P.list_K;
        const bool whole = traverse(C, stack, 1);
        if (C.rec && lane == 0)
            P.list_n[kAgain ? S.cut.g : g] = whole && C.rec_n <= C.rec_cap ? (uint32_t)C.rec_n : kListTooLong;
        C.flush_far();
        C.flush_near();
        if constexpr (KIND != LENS_POINT) C.flush_big();
        if (P.n_halos > 0) C.halos(P.halos, P.n_halos);
        if constexpr (kAgain) {
            rg = P.grange[S.cut.g];
#pragma unroll
            for (int r = 0; r < R; ++r) {
                rv[r] = r * 32 + lane < (int)rg.y;
                ridx[r] = rv[r] ? P.ray_idx[rg.x + r * 32 + lane] : 0u;
            }
        }
        count_item(C, kAgain ? S.cut.g : g, true);
        if (CUTS && S.cut.sp > 0) cut_now<R, false>(P.cut, S.cut, stack, S.cut.sp);
        __syncwarp();
        T* tot = CUTS ? item_totals<R>(P.cut, S.cut) : nullptr;
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (!rv[r] && !tot) continue;
            const uint32_t i = ridx[r];
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                if (AO && q >= 2) break;
                T val = C.tot_get(r, q);
                if (tot) {
                    tot[(q * R + r) * 32 + lane] = val;
                    continue;
                }
                if (P.accumulate) val += P.out[q][i];
                P.out[q][i] = val;
            }
        }
        __syncwarp();
    }
}

template <int KIND, typename T, int R, bool AO, int TILE, bool CUTS> static int plain_blocks_per_sm()
{
    constexpr size_t smem = kWalkWarps * sizeof(PlainShared<KIND, T, TILE, tot_rays<R>()>);
    constexpr auto kernel = walk_plain<KIND, T, R, AO, TILE, CUTS>;
    static const int bps = [] {
        if (smem > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        int nb = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, kWalkWarps * 32, smem);
        // (stacks are allocated for 16 blocks per SM; where cuts lie behind them: walk_blocks)
        return std::min(std::max(nb, 1), CUTS ? walk_blocks<T, R>() : 16);
    }();
    return bps;
}

template <int KIND, typename T, int R, bool AO, int TILE, bool CUTS = false>
static void launch_plain(const WalkParams<T>& P, int num_sms, cudaStream_t s)
{
    constexpr size_t smem = kWalkWarps * sizeof(PlainShared<KIND, T, TILE, tot_rays<R>()>);
    const int bps = plain_blocks_per_sm<KIND, T, R, AO, TILE, CUTS>();
    walk_plain<KIND, T, R, AO, TILE, CUTS><<<num_sms * bps, kWalkWarps * 32, smem, s>>>(P);
    note_launch();
}

// The common part of the walk of kSuperGroups consecutive groups of a point-
// mass tree (SuperRec), one warp each, one group per lane.
//
// The warp walks the tree as the first group's own walk does: the same tests,
// the same order, the same buffers, evaluated at the groups' centres.  Beside
// the first group's test every box gets two bounds: it is accepted for all if
// the supergroup's box is beyond r_cut, opened for all if the box's farthest
// point is within (a margin of 1e-5 covers the rounding of the groups' own
// tests).  Accepted for all and far from the supergroup, or a leaf opened for
// all and far: its sources go to the expansion.  Any other box that is not
// opened for all is left to the groups; what the first group's walk finds
// inside it (kLeftBit) is evaluated in its place and taken off again at the
// end.  More boxes left than a record holds: the groups start at the root.
// (A walk of more than kSuperWork boxes and entries is that of a stretched
// group: not worth one warp's time.)
constexpr uint32_t kSuperWork = 16384;
// Most boxes left to the groups (200,000 stars, 70,312 groups, 0.2 of the lens,
// theta 0.3: 64 boxes 1.45 ms, 128 1.11, 256 1.11; 0.06 of it, theta 0.1: 3.49,
// 1.84, 1.66).
constexpr int kSuperLeft = 128, kTinyLeft = 8;
// When expansions are taken (one batch; r: the root's r_cm):
//   Over a patch narrower than kNarrow r the sums of all rays are nearly one
//     sum, and a component that cancels to 1e-3 of the sum of |terms| is FP32
//     noise in its fourth digit.  Expanded or not, its error against 64 bits is
//     the same (rms 3e-8 to 9e-8 of the sum of |terms| from 1e-6 to 0.1 wide),
//     but the digits are others: up to 2e-4 of alpha2 for 3e6 stars, theta 0.3.
//     Such patches go to the plain kernel and keep their digits.
//   Where a group's side is below kTiny r, an eighth of the rounding of a
//     distance r, all its rays round alike and the correction at the group's
//     centre (sdelta) gives the plain kernel's digits back (2e-6 to 4e-5 of
//     alpha2); 4096^2 rays, 1e7 stars over 1e-6: 78 -> 7.7 ms.
//   Over a wide field nothing is far from a supergroup.  near: the stars in the
//     zone (of radius d / 0.18) that its expansion cannot stand for, in the mean.
//     They are evaluated for every ray of 32 R, where the plain kernel evaluates
//     some number for theta; times of start and supergroups, theta 0.3: R = 1,
//     near 282: 2.02 -> 1.56 ms, 704: 0.47 -> 0.67; R = 2, 1,131: 1.06 -> 1.03,
//     2,034: 2.65 -> 2.73; R = 4, 3,973: 4.62 -> 3.89, 7,430: 2.02 -> 2.22.
//     theta 0.1: R = 1, 990: 2.41 -> 2.14, 7,044: 2.73 -> 2.78, R = 2 and 4
//     always faster.  Hence 400 R^2 (0.3 / theta)^3 for R = 1 and 2; R = 4 (at
//     worst 0.91 times as fast, and 1.2 times where groups are stretched): none.
// Several batches: only the last, for each supergroup by its own d.
constexpr float kNarrow = 0.01f, kTiny = 7.4505806e-9f;
constexpr float kNearMax = 400.0f;
static_assert(kSuperLeft <= kCutNodes, "room in the record");
constexpr int kLeftBit = 1 << 30;  // (a tree has fewer boxes)

__global__ void __launch_bounds__(kWalkWarps * 32, 4)
k_super(const __grid_constant__ WalkParams<float> P, const float* rcm, const unsigned long long* bbox,
        const uint32_t* bb32, float near_max, SuperRec* rec, float4* sdelta)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    using Flush = WalkFlush<LENS_POINT, float, 1, false, 0, true>;
    using WS = Flush::WS;
    const unsigned full = 0xffffffffu;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    WS& S = reinterpret_cast<WS*>(smem_raw)[warp];
    uint8_t* far_left = S.loc.idx;             // of the far buffer's cells and the
    uint8_t* near_left = S.loc.idx + kBigCap;  // near buffer's particles: left to the groups
    int* stack = P.stack + ((int64_t)blockIdx.x * kWalkWarps + warp) * kStackCap;
    const int64_t n_super = (P.n_groups + kSuperGroups - 1) / kSuperGroups;
    float wx = INFINITY, wy = INFINITY;
    if (bb32) {
        wx = ordered_to_flt(bb32[2]) - ordered_to_flt(bb32[0]);
        wy = ordered_to_flt(bb32[3]) - ordered_to_flt(bb32[1]);
    } else if (bbox) {
        wx = (float)(ordered_to_dbl(bbox[1]) - ordered_to_dbl(bbox[0]));
        wy = (float)(ordered_to_dbl(bbox[3]) - ordered_to_dbl(bbox[2]));
    }
    const float ext = fmaxf(wx, wy), ng = (float)P.n_groups;
    const float per_d2 = (float)P.n_part / (kLocRho2 * rcm[0] * rcm[0]);  // stars near, over d^2
    const bool narrow = ext < kNarrow * rcm[0], tiny = ext * rsqrtf(ng) < kTiny * rcm[0];
    const bool dense = (bb32 || bbox) && wx * wy * (0.5f * kSuperGroups) * per_d2 > near_max * ng;
    const int most_left = narrow ? (tiny ? kTinyLeft : -1) : dense ? -1 : kSuperLeft;
    for (;;) {
        uint32_t sg = 0;
        if (lane == 0) sg = atomicAdd(P.counter, 1u);
        sg = __shfl_sync(full, sg, 0);
        if ((int64_t)sg >= n_super) break;
        SuperRec& Q = rec[sg];
        const int64_t g = (int64_t)sg * kSuperGroups + lane;
        const bool have = g < P.n_groups;
        const float2 Hg = P.gH[have ? g : (int64_t)sg * kSuperGroups];
        const float4 bg = P.gbox[have ? g : (int64_t)sg * kSuperGroups];
        const float Hx = __shfl_sync(full, Hg.x, 0), Hy = __shfl_sync(full, Hg.y, 0);
        const float4 b0 = make_float4(__shfl_sync(full, bg.x, 0), __shfl_sync(full, bg.y, 0),
                                      __shfl_sync(full, bg.z, 0), __shfl_sync(full, bg.w, 0));
        const float gx = (Hg.x - Hx) + bg.x, gy = (Hg.y - Hy) + bg.y;  // this group's centre
        float x0 = gx - bg.z, x1 = gx + bg.z, y0 = gy - bg.w, y1 = gy + bg.w;
        for (int o = 16; o; o >>= 1) {
            x0 = fminf(x0, __shfl_xor_sync(full, x0, o));
            x1 = fmaxf(x1, __shfl_xor_sync(full, x1, o));
            y0 = fminf(y0, __shfl_xor_sync(full, y0, o));
            y1 = fmaxf(y1, __shfl_xor_sync(full, y1, o));
        }
        const float cx = 0.5f * (x0 + x1), cy = 0.5f * (y0 + y1);
        const float hx = fmaxf(x1 - cx, cx - x0) * 1.00001f, hy = fmaxf(y1 - cy, cy - y0) * 1.00001f;
        const float d = local_scale(hx, hy, rcm[0]), far2 = d * d * (1.0f / kLocRho2);
        if (lane == 0) stack[0] = 0;
        local_zero(S.loc.sum);
        __syncwarp();
        LocalH L;
        L.zero();
        // alpha at this group's centre, and of it what is left to the groups;
        // gamma without what is left (a star at the centre would drown it)
        Comp5<float> all, own;
        all.zero();
        own.zero();
        float top2 = 0.0f;  // largest |alpha|^2 of one star left to the groups
        int sp = 1, left = 0, nf = 0, nn = 0;
        uint32_t work = 0;
        bool ok = d < 1e30f && d * d * per_d2 <= 4.0f * near_max;
        // The buffers hold positions as the tree has them: the sums at the
        // centres subtract each group's own anchor, as its own walk does (the
        // subtraction is rounded: the anchor is part of the result's last digits).
        auto flush_far = [&]() {
            Acc5<float> a, f;
            a.zero();
            f.zero();
            for (int b = 0; b < nf; b += 32) {
                const unsigned m = __ballot_sync(full, b + lane < nf && far_left[b + lane]);
                const int e = nf - b < 32 ? nf - b : 32;
                for (int j = 0; j < e; ++j) {
                    const int i = b + j;
                    const float wx = bg.x - (S.buf.fdx[i] - Hg.x), wy = bg.y - (S.buf.fdy[i] - Hg.y);
                    if (m >> j & 1u) {
                        cell_terms<float, true>(f, wx, wy, S.buf.fM[i], S.buf.fqr[i], S.buf.fqi[i]);
                        cell_terms<float, true>(a, wx, wy, S.buf.fM[i], S.buf.fqr[i], S.buf.fqi[i]);
                    } else {
                        cell_terms<float, false>(f, wx, wy, S.buf.fM[i], S.buf.fqr[i], S.buf.fqi[i]);
                    }
                }
            }
            all.add(f);
            own.add(a);
            for (int i = lane; i < nf; i += 32) {
                if (far_left[i]) continue;
                const float wx = cx - (S.buf.fdx[i] - Hx), wy = cy - (S.buf.fdy[i] - Hy);
                L.cell(wx, wy, rcp(fmaf(wx, wx, wy * wy)), d, S.buf.fM[i], S.buf.fqr[i], S.buf.fqi[i]);
            }
            __syncwarp();
            nf = 0;
        };
        auto flush_near = [&]() {
            Acc5<float> a, f;
            a.zero();
            f.zero();
            for (int b = 0; b < nn; b += 32) {
                const unsigned m = __ballot_sync(full, b + lane < nn && near_left[b + lane]);
                const int e = nn - b < 32 ? nn - b : 32;
                for (int j = 0; j < e; ++j) {
                    const float4 q = S.buf.n0[b + j];
                    const float wx = bg.x - (q.x - Hg.x), wy = bg.y - (q.y - Hg.y);
                    float kb, Dp;
                    point_terms(q.z, fmaf(wx, wx, wy * wy), kb, Dp);
                    if (m >> j & 1u) {
                        f.radial<true>(wx, wy, kb, 0.0f, Dp);
                        a.radial<true>(wx, wy, kb, 0.0f, Dp);
                        top2 = fmaxf(top2, kb * kb * fmaf(wx, wx, wy * wy));
                    } else {
                        f.radial<false>(wx, wy, kb, 0.0f, Dp);
                    }
                }
            }
            all.add(f);
            own.add(a);
            for (int i = lane; i < nn; i += 32) {
                if (near_left[i]) continue;
                const float4 q = S.buf.n0[i];
                const float wx = cx - (q.x - Hx), wy = cy - (q.y - Hy);
                L.point(wx, wy, rcp(fmaf(wx, wx, wy * wy)), d, q.z);
            }
            __syncwarp();
            nn = 0;
        };
        while (sp > 0 && ok) {
            const int k = sp < 32 ? sp : 32;
            sp -= k;
            const int e = lane < k ? stack[sp + lane] : -1;
            __syncwarp();
            const int v = e & (kLeftBit - 1);
            bool acc = false, leaf = false, open = false, is_left = false, keep = false;
            float4 A = make_float4(0.f, 0.f, 0.f, 0.f);
            int4 Lk = make_int4(0, 0, 0, 0);
            float dx = 0.f, dy = 0.f;
            if (e >= 0) {
                A = P.nodeA[v];
                Lk = P.link[v];
                dx = A.x - Hx;
                dy = A.y - Hy;
                // the first group's test
                const float ex = fmaxf(fabsf(dx - b0.x) - b0.z, 0.0f), ey = fmaxf(fabsf(dy - b0.y) - b0.w, 0.0f);
                acc = fmaf(ex, ex, ey * ey) > A.w;
                leaf = !acc && (Lk.y & kLeafBit);
                open = !acc && !leaf;
                is_left = (e & kLeftBit) != 0;
                if (!is_left) {
                    const float ux = fabsf(dx - cx), uy = fabsf(dy - cy);
                    const float lx = fmaxf(ux - hx, 0.0f), ly = fmaxf(uy - hy, 0.0f);
                    const float fx = ux + hx, fy = uy + hy;
                    const float w2 = fmaf(ux, ux, uy * uy);
                    const bool all_acc = fmaf(lx, lx, ly * ly) > A.w * 1.00001f;
                    const bool all_opn = fmaf(fx, fx, fy * fy) * 1.00001f < A.w;
                    // every particle of a leaf is within r_cm of its centre of mass
                    const float m = sqrtf(w2) - rcm[v] * 1.00001f;
                    keep = acc ? !(all_acc && w2 >= far2) : leaf ? !(all_opn && m > 0.0f && m * m >= far2) : !all_opn;
                    is_left = keep;
                }
            }
            const unsigned lt = (1u << lane) - 1u;
            unsigned ball = __ballot_sync(full, acc);
            if (acc) {
                const int pos = nf + __popc(ball & lt);
                const float2 Qm = P.nodeB[v];
                S.buf.fdx[pos] = A.x;
                S.buf.fdy[pos] = A.y;
                S.buf.fM[pos] = A.z;
                S.buf.fqr[pos] = Qm.x;
                S.buf.fqi[pos] = Qm.y;
                far_left[pos] = is_left ? 1 : 0;
            }
            nf += __popc(ball);
            work += (uint32_t)(k + __popc(ball));
            ball = __ballot_sync(full, keep);
            if (left + __popc(ball) > most_left) {
                ok = false;
                break;
            }
            if (keep) Q.nodes[left + __popc(ball & lt)] = v;
            left += __popc(ball);
            const int nc = open ? Lk.y : 0;
            int totc;
            const int offc = warp_exclusive_scan(nc, &totc);
            if (sp + totc > kStackCap) {
                if (lane == 0) atomicOr(P.err, DERR_STACK_OVERFLOW);
                ok = false;
                break;
            }
            for (int c = 0; c < nc; ++c) stack[sp + offc + c] = (Lk.x + c) | (is_left ? kLeftBit : 0);
            sp += totc;
            // leaf particles, in order, as append_ranges takes them
            const int cnt = leaf ? (Lk.y & kCountMask) : 0;
            int tot;
            const int off = warp_exclusive_scan(cnt, &tot);
            work += (uint32_t)tot;
            for (int b = 0; b < tot; b += 32) {
                if (nn + 32 > kNearCap) flush_near();
                for (int c = 0; c < cnt; ++c) {
                    const int i = off + c - b;
                    if (i < 0 || i >= 32) continue;
                    S.buf.n0[nn + i] = P.leaf0[Lk.x + c];
                    near_left[nn + i] = is_left ? 1 : 0;
                }
                nn += tot - b < 32 ? tot - b : 32;
                __syncwarp();
            }
            __syncwarp();
            if (nf >= 32) flush_far();
            ok = work < kSuperWork;
        }
        if (ok) {
            flush_far();
            flush_near();
            Flush::add_h(L);
            LocalFields& F = *reinterpret_cast<LocalFields*>(S.buf.n0);
            local_finish(S.loc.sum, F);
            const float id = 1.0f / d;
            Acc5<float> a;
            a.zero();
            local_eval<false>(F, (gx - cx) * id, (gy - cy) * id, id, a);
            if (have) {
                const float e[5] = {a.a1, a.a2, 0.0f, a.g1, a.g2};
                float v[5];
#pragma unroll
                for (int q = 0; q < 5; ++q)
                    v[q] = ((all.s[q] - own.s[q]) - e[q]) + (all.c[q] - own.c[q]);
                // where one star outweighs the rest (it lies at the centre), the
                // difference of alpha is that star's rounding
                if (sqrtf(top2) > 0.5f * (fabsf(all.s[0]) + fabsf(all.s[1]))) v[0] = v[1] = 0.0f;
                const float4 dl = make_float4(v[0], v[1], v[3], v[4]);
                sdelta[g] = dl;
                if (P.gcost) atomicAdd(P.gcost + g, work);
            }
            if (lane < kLocH) Q.h[lane] = F.h[lane];
            if (lane == 0) {
                Q.hx = Hx;
                Q.hy = Hy;
                Q.cx = cx;
                Q.cy = cy;
                Q.id = id;
                Q.n = left;
            }
        }
        if (lane == 0) Q.ok = ok ? 1 : most_left < 0 ? 3 : narrow ? 2 : 0;
        __syncwarp();
    }
}

// Supergroups' records for the walk of a point-mass tree (null: not worth it).
static const SuperRec* launch_super(WalkParams<float>& P, const SpeciesTree& st, char* base, const Layout& L,
                                    uint32_t* counter, int64_t nb, int dtype, float near_max, int num_sms,
                                    cudaStream_t s)
{
    constexpr size_t smem = kWalkWarps * sizeof(WalkShared<LENS_POINT, float, 0, 2>);
    static const int bps = [] {
        if (smem > 48 * 1024)
            cudaFuncSetAttribute(k_super, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        int nb = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_super, kWalkWarps * 32, smem);
        return std::min(std::max(nb, 1), 16);
    }();
    SuperRec* rec = (SuperRec*)(base + L.super);
    P.sdelta = (const float4*)(base + L.sdelta);
    P.counter = counter;
    const int64_t ns = (P.n_groups + kSuperGroups - 1) / kSuperGroups;
    const int64_t blocks = std::min<int64_t>((ns + kWalkWarps - 1) / kWalkWarps, (int64_t)num_sms * bps);
    const void* box = base + L.bbox;  // of a single batch: ordered uint32 or FP64 images (enqueue_groups)
    k_super<<<(unsigned)blocks, kWalkWarps * 32, smem, s>>>(P, st.node_rcm, nb == 1 && dtype != LENS_F32 ? (const unsigned long long*)box : nullptr,
                                                            nb == 1 && dtype == LENS_F32 ? (const uint32_t*)box : nullptr, near_max, rec, (float4*)(base + L.sdelta));
    note_launch();
    return rec;
}

// The slices of a split direct sum, added per ray in slice order with
// Neumaier compensation (deterministic), into the outputs.
template <typename T>
__global__ void k_split_sum(int64_t n, int S, int nq, const T* split, T* o0, T* o1, T* o2, T* o3, T* o4,
                            int accumulate)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    T* out[5] = {o0, o1, o2, o3, o4};
    for (int q = 0; q < nq; ++q) {
        T s = T(0), c = T(0);
        for (int k = 0; k < S; ++k) Comp5<T>::add1(s, c, split[((int64_t)k * 5 + q) * n + i]);
        T v = s + c;
        if (accumulate) v += out[q][i];
        out[q][i] = v;
    }
}

// Particle slices for a direct sum of ng ray groups over n_part particles:
// enough work items (group x slice) for about 16 warps per SM when the rays
// alone give fewer, each slice at least 128 particles, the partial sums
// within the scratch of the split region.
static int split_slices(const lens_tree* t, int64_t ng, int64_t n_rays, int64_t n_part)
{
    const int64_t target = (int64_t)t->num_sms * 16;
    if (ng <= 0 || ng >= target) return 1;
    int64_t S = (target + ng - 1) / ng;
    S = std::min<int64_t>(S, std::max<int64_t>(1, n_part / 128));
    S = std::min<int64_t>(S, 64);
    S = std::min<int64_t>(S, (int64_t)split_values(max_slots(const_cast<lens_tree*>(t))) / std::max<int64_t>(1, n_rays));
    return S < 2 ? 1 : (int)S;
}

// ------------------------------------------------------------- host side

template <int KIND, typename T, int R, bool AO, bool DIRECT, int TILE, bool LOC>
static int walk_blocks_per_sm()
{
    static int cached = -1;
    if (cached < 0) {
        size_t smem = kWalkWarps * sizeof(WalkShared<KIND, T, TILE, tot_rays<R>()>);
        if (smem > 48 * 1024)
            cudaFuncSetAttribute(walk_kernel<KIND, T, R, AO, DIRECT, TILE, LOC>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        // the walk keeps its working set in shared memory and registers:
        // prefer the largest shared-memory carveout
        cudaFuncSetAttribute(walk_kernel<KIND, T, R, AO, DIRECT, TILE, LOC>,
                             cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        int nb = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, walk_kernel<KIND, T, R, AO, DIRECT, TILE, LOC>,
                                                      kWalkWarps * 32, smem);
        cached = std::min(std::max(nb, 1), DIRECT ? 16 : walk_blocks<T, R>());  // (room for stacks and cuts)
    }
    return cached;
}

void free_graphs(lens_tree* t);

lens_status reserve_rays(lens_tree* t, int64_t n, int64_t nb, cudaStream_t s)
{
    if (n <= t->ray_cap && nb <= t->batch_cap && t->ray_scratch.ptr) return LENS_OK;
    int64_t nn = std::max(n, t->ray_cap), bb = std::max(nb, t->batch_cap);
    Layout L = make_layout(nn, bb, max_slots(t));
    free_graphs(t);  // captured graphs point into the old scratch
    t->cost_n = -1;  // so does the work record
    t->grp_n = -1;   // and the groups
    if (t->ray_scratch.ptr) cudaFreeAsync(t->ray_scratch.ptr, s);
    t->ray_scratch.ptr = nullptr;
    t->ray_cap = t->batch_cap = 0;
    cudaError_t e = lens_malloc_async(&t->ray_scratch.ptr, L.total, s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return lens_set_error(LENS_ERR_OOM, "cannot allocate %zu bytes of ray scratch", L.total);
    }
    t->ray_scratch.bytes = L.total;
    t->ray_cap = nn;
    t->batch_cap = bb;
    return LENS_OK;
}

template <int KIND, typename T, int R, bool AO, bool DIRECT, int TILE, bool LOC>
static void launch_one(const WalkParams<T>& P, int num_sms, cudaStream_t s)
{
    size_t smem = kWalkWarps * sizeof(WalkShared<KIND, T, TILE, tot_rays<R>()>);
    int bps = walk_blocks_per_sm<KIND, T, R, AO, DIRECT, TILE, LOC>();
    int grid = num_sms * bps;
    { walk_kernel<KIND, T, R, AO, DIRECT, TILE, LOC><<<grid, kWalkWarps * 32, smem, s>>>(P); note_launch(); }
}

template <typename T, int R, bool AO>
static void launch_kind(int kind, const WalkParams<T>& P, int num_sms, cudaStream_t s)
{
    if (kind == LENS_POINT) launch_one<LENS_POINT, T, R, AO, true, 0, false>(P, num_sms, s);
    else if (kind == LENS_GAUSS) launch_one<LENS_GAUSS, T, R, AO, true, 0, false>(P, num_sms, s);
    else launch_one<LENS_NFW, T, R, AO, true, 0, false>(P, num_sms, s);
}

template <typename T, int R>
static void launch_direct(int kind, bool ao, const WalkParams<T>& P, int num_sms, cudaStream_t s)
{
    if (ao) launch_kind<T, R, true>(kind, P, num_sms, s);
    else launch_kind<T, R, false>(kind, P, num_sms, s);
}

// The one-warp tree walk of all groups.
//   FP32 NFW trees (expansions) and, where all groups are cut (few_groups), all
//     but FP32 point masses: the cut form.
//   FP32 point masses: the plain kernel with cuts; up to 32 groups per SM (about
//     as many warps as it holds) the cut form, whose steps are shorter (504
//     groups of 67,587 stars 1.22 and 1.11 ms; 2,793 of 2e6 2.01, 1.83; 4,278
//     over a wide field of 1e6 1.12, 1.14; 14,964 1.33, 1.38).
//     With supergroups the cut form with expansions or, as only the device
//     knows, the plain kernel: the other of the two launches finds no work.
//   The others: from kPlainGroups groups on the stretched groups by the cut
//     form and the rest by the plain kernel, whose 80 to 96 registers the cut
//     form's 96 to 128 cost 5 to 10 %; below, all by the cut form, which cuts
//     heavy groups too (1e5 and 1e6 particles, 4,300 to 22,000 groups: 1.3 to 5
//     times as fast as the plain kernel), unless the tree has fewer than
//     kPlainParticles (20,000: no group is heavy, 1.03 to 1.08).
constexpr int64_t kPlainGroups = 24576, kPlainParticles = 24576;
template <int KIND, typename T, int R, bool AO, int TILE>
static void walk_tree_kind(WalkParams<T> P, lens_tree* t, int nq, char* base, const Layout& L, cudaStream_t s)
{
    constexpr bool kF32 = sizeof(T) == 4, kNfw = KIND == LENS_NFW && kF32, kPoint = KIND == LENS_POINT && kF32;
    const int sms = t->num_sms;
    const int64_t ng = P.n_groups;
    uint32_t* counter = P.counter;
    auto cut = [&](const WalkParams<T>& Q) {
        if constexpr (kPoint) {
            if (Q.super) {
                launch_one<KIND, T, R, AO, false, TILE, true>(Q, sms, s);
                return;
            }
        }
        launch_one<KIND, T, R, AO, false, TILE, kNfw>(Q, sms, s);
    };
    const int cut_warps = kWalkWarps * sms * (P.super ? walk_blocks_per_sm<KIND, T, R, AO, false, TILE, kPoint || kNfw>()
                                                      : walk_blocks_per_sm<KIND, T, R, AO, false, TILE, kNfw>());
    const CutPlan plan{ng <= few_groups(KIND, kF32, P.n_part) && !kPoint, kPoint, false};
    if constexpr (kNfw) {
        if (never_cut(t, ng, P.n_rays, P.n_part, plan)) cut(P);
        else walk_rounds<T, R>(P, plan, nq, base, L, counter, cut, cut, cut_warps, cut_warps, s);
    } else if constexpr (kPoint) {
        const int warps = std::max(cut_warps, kWalkWarps * sms * plain_blocks_per_sm<KIND, T, R, AO, TILE, true>());
        const bool fit = cuts_fit<T, R>(ng, L, warps, cut_warps);
        auto groups = [&](const WalkParams<T>& Q) {
            const bool whole = fit && ng > 32 * sms;
            if (Q.super || !whole) cut(Q);
            if (!Q.super && !whole) return;
            WalkParams<T> W = Q;
            if (Q.super) W.counter = counter + 6;
            if (fit) launch_plain<KIND, T, R, AO, TILE, true>(W, sms, s);
            else launch_plain<KIND, T, R, AO, TILE>(W, sms, s);
        };
        if (never_cut(t, ng, P.n_rays, P.n_part, plan)) {
            WalkParams<T> W = P;
            if (P.super) {
                cut(P);
                W.counter = counter + 6;
            }
            launch_plain<KIND, T, R, AO, TILE>(W, sms, s);
        } else {
            walk_rounds<T, R>(P, plan, nq, base, L, counter, groups, cut, warps, cut_warps, s);
        }
    } else {
        if (plan.few && never_cut(t, ng, P.n_rays, P.n_part, plan)) {
            launch_plain<KIND, T, R, AO, TILE>(P, sms, s);
            return;
        }
        if (plan.few || (ng < kPlainGroups && !(kF32 && P.n_part < kPlainParticles))) {
            walk_rounds<T, R>(P, plan, nq, base, L, counter, cut, cut, cut_warps, cut_warps, s);
            return;
        }
        if (P.n_part > 4 * ng) {
            // (fewer particles: even a group that meets all of them is done
            // before the others; lens fit, 1e5 particles, 31,250 groups)
            const uint32_t* sub = (const uint32_t*)(base + L.sub);
            WalkParams<T> Q = P;
            Q.sub = sub + 16;
            Q.sub_n = sub;
            walk_rounds<T, R>(Q, CutPlan{false, false, true}, nq, base, L, counter, cut, cut, cut_warps, cut_warps, s);
            P.gflag = (const uint8_t*)(base + L.gflag);
            P.skip = 1;
            cudaMemsetAsync(counter, 0, sizeof(uint32_t), s);
            P.counter = counter;
        }
        launch_plain<KIND, T, R, AO, TILE>(P, sms, s);
    }
}

template <typename T, int R>
static void walk_tree(int kind, bool ao, const WalkParams<T>& P, lens_tree* t, int nq, char* base, const Layout& L,
                      cudaStream_t s)
{
    auto go = [&](auto tile) {
        constexpr int TILE = decltype(tile)::value;
        if (kind == LENS_POINT) {
            if (ao) walk_tree_kind<LENS_POINT, T, R, true, TILE>(P, t, nq, base, L, s);
            else walk_tree_kind<LENS_POINT, T, R, false, TILE>(P, t, nq, base, L, s);
        } else if (kind == LENS_GAUSS) {
            if (ao) walk_tree_kind<LENS_GAUSS, T, R, true, TILE>(P, t, nq, base, L, s);
            else walk_tree_kind<LENS_GAUSS, T, R, false, TILE>(P, t, nq, base, L, s);
        } else {
            if (ao) walk_tree_kind<LENS_NFW, T, R, true, TILE>(P, t, nq, base, L, s);
            else walk_tree_kind<LENS_NFW, T, R, false, TILE>(P, t, nq, base, L, s);
        }
    };
    // (the larger near-field tile is built for FP32 trees, 128-ray groups
    // likewise)
    if constexpr (sizeof(T) == 8 && R == 4) {
        return;
    } else if constexpr (sizeof(T) == 4) {
        if (t->tile == 1) go(std::integral_constant<int, 1>{});
        else go(std::integral_constant<int, 0>{});
    } else {
        go(std::integral_constant<int, 0>{});
    }
}

static int rays_per_lane(const lens_tree* t, int max_r)
{
    const int r = (t->precision == LENS_PREC_FP64 || t->group_rays <= 32) ? 1 : t->group_rays >= 128 ? 4 : 2;
    return r < max_r ? r : max_r;
}

// 128-ray groups only for the one-warp tree walk of an FP32 tree.
int shoot_max_r(const lens_tree* t, int flags)
{
    const bool ws = t->walk_mode == LENS_WALK_PAIRS || t->walk_mode == LENS_WALK_TRIOS;
    return (flags & LENS_DIRECT) || ws || t->precision != LENS_PREC_FP32 ? 2 : 4;
}

// Copy the batch table to the device (stream ordered) and size the groups.
lens_status upload_batches(lens_tree* t, int64_t nb, const int64_t* h_off, const double* h_orig,
                           cudaStream_t s, ShootPlan* plan, int max_r)
{
    const int64_t n = h_off[nb];
    const int R = rays_per_lane(t, max_r);
    const int GR = 32 * R;
    LENS_TRY(reserve_rays(t, n, nb, s));
    Layout L = make_layout(t->ray_cap, t->batch_cap, max_slots(t));
    char* base = (char*)t->ray_scratch.ptr;
    // pageable host copies: the CUDA driver stages them before returning
    std::vector<uint32_t> gf(nb + 1);
    uint64_t ng = 0;
    for (int64_t b = 0; b < nb; ++b) {
        gf[b] = (uint32_t)ng;
        ng += (uint64_t)((h_off[b + 1] - h_off[b] + GR - 1) / GR);
    }
    gf[nb] = (uint32_t)ng;
    LENS_CUDA(cudaMemcpyAsync(base + L.boff, h_off, (nb + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, s));
    LENS_CUDA(cudaMemcpyAsync(base + L.borig, h_orig, nb * 2 * sizeof(double), cudaMemcpyHostToDevice, s));
    LENS_CUDA(cudaMemcpyAsync(base + L.gfirst, gf.data(), (nb + 1) * sizeof(uint32_t),
                              cudaMemcpyHostToDevice, s));
    plan->n = n;
    plan->nb = nb;
    plan->ng = ng;
    plan->R = R;
    plan->ox = nb == 1 ? h_orig[0] : 0.0;
    plan->oy = nb == 1 ? h_orig[1] : 0.0;
    return LENS_OK;
}

template <typename T>
lens_status enqueue_groups(lens_tree* t, const ShootPlan& plan, const void* dx, const void* dy, int dtype,
                           cudaStream_t s)
{
    t->grp_n = -1;  // (set again below once these rays are grouped)
    using T4 = vec4_t<T>;
    using T2 = v2_t<T>;
    const int64_t n = plan.n, nb = plan.nb;
    const uint64_t ng = plan.ng;
    const int R = plan.R;
    Layout L = make_layout(t->ray_cap, t->batch_cap, max_slots(t));
    char* base = (char*)t->ray_scratch.ptr;
    int64_t* d_boff = (int64_t*)(base + L.boff);
    double* d_borig = (double*)(base + L.borig);
    uint32_t* d_gfirst = (uint32_t*)(base + L.gfirst);
    unsigned long long* d_bbox = (unsigned long long*)(base + L.bbox);
    T2* ray_l = (T2*)(base + L.rl);
    uint32_t* ray_idx = (uint32_t*)(base + L.ridx);
    T2* gH = (T2*)(base + L.gH);
    T4* gbox = (T4*)(base + L.gbox);
    uint2* grange = (uint2*)(base + L.grange);
    uint8_t* gflag = (uint8_t*)(base + L.gflag);
    uint32_t* sub = (uint32_t*)(base + L.sub);
    LENS_CUDA(cudaMemsetAsync(sub, 0, sizeof(uint32_t), s));
    if (nb == 1 && dtype == LENS_F32) {
        const int TB = 256;
        const float* fx = (const float*)dx;
        const float* fy = (const float*)dy;
        uint32_t* bb = (uint32_t*)d_bbox;
        uint32_t* k0 = (uint32_t*)(base + L.k0);
        uint32_t* k1 = (uint32_t*)(base + L.k1);
        uint32_t* v0 = (uint32_t*)(base + L.v0);
        uint32_t* v1 = (uint32_t*)(base + L.v1);
        LENS_CUDA(cudaMemsetAsync(bb, 0xff, 2 * sizeof(uint32_t), s));
        LENS_CUDA(cudaMemsetAsync(bb + 2, 0, 2 * sizeof(uint32_t), s));
        { k_ray_bbox32<<<grid_for(n, TB), TB, 0, s>>>(fx, fy, n, bb); note_launch(); }
        { k_ray_keys32<<<grid_for(n, TB), TB, 0, s>>>(fx, fy, n, bb, k0, v0); note_launch(); }
        uint32_t *sk, *sv;
        radix_sort_pairs<uint32_t>(k0, v0, k1, v1, n, 0, 32, base + L.tmp, s, &sk, &sv, t->d_err);
        unsigned gg = grid_for((int64_t)ng * 32, TB);
        if (plan.ox == 0.0 && plan.oy == 0.0) {
            if (R == 1)
                { k_groups32<T, 1><<<gg, TB, 0, s>>>((int64_t)ng, n, fx, fy, sv, gH, gbox, grange, ray_l, ray_idx, bb,
                                                gflag, sub);
                  note_launch(); }
            else if (R == 2)
                { k_groups32<T, 2><<<gg, TB, 0, s>>>((int64_t)ng, n, fx, fy, sv, gH, gbox, grange, ray_l, ray_idx, bb,
                                                gflag, sub);
                  note_launch(); }
            else
                { k_groups32<T, 4><<<gg, TB, 0, s>>>((int64_t)ng, n, fx, fy, sv, gH, gbox, grange, ray_l, ray_idx, bb,
                                                gflag, sub);
                  note_launch(); }
        } else if (R == 1) {
            { k_groups<T, 1><<<gg, TB, 0, s>>>((int64_t)ng, d_boff, d_gfirst, (int)nb, d_borig, dx, dy, dtype,
                                             sv, gH, gbox, grange, ray_l, ray_idx, nullptr, bb, gflag, sub); note_launch(); }
        } else if (R == 2) {
            { k_groups<T, 2><<<gg, TB, 0, s>>>((int64_t)ng, d_boff, d_gfirst, (int)nb, d_borig, dx, dy, dtype,
                                             sv, gH, gbox, grange, ray_l, ray_idx, nullptr, bb, gflag, sub); note_launch(); }
        } else {
            { k_groups<T, 4><<<gg, TB, 0, s>>>((int64_t)ng, d_boff, d_gfirst, (int)nb, d_borig, dx, dy, dtype,
                                             sv, gH, gbox, grange, ray_l, ray_idx, nullptr, bb, gflag, sub); note_launch(); }
        }
    } else {
        const int TB = 256;
        { k_bbox_init<<<grid_for(nb, 128), 128, 0, s>>>(d_bbox, nb); note_launch(); }
        { k_ray_bbox<<<grid_for(n, TB), TB, 0, s>>>(d_boff, (int)nb, d_borig, dx, dy, dtype, n, d_bbox); note_launch(); }
        uint64_t* k0 = (uint64_t*)(base + L.k0);
        uint64_t* k1 = (uint64_t*)(base + L.k1);
        uint32_t* v0 = (uint32_t*)(base + L.v0);
        uint32_t* v1 = (uint32_t*)(base + L.v1);
        { k_ray_keys<<<grid_for(n, TB), TB, 0, s>>>(d_boff, (int)nb, d_borig, dx, dy, dtype, n, d_bbox, k0, v0); note_launch(); }
        int bbits = 0;
        while ((1ll << bbits) < nb) ++bbits;
        int end_bit = (32 + bbits + 7) & ~7;
        uint64_t* sk;
        uint32_t* sv;
        radix_sort_pairs<uint64_t>(k0, v0, k1, v1, n, 0, end_bit, base + L.tmp, s, &sk, &sv, t->d_err);
        unsigned gg = grid_for((int64_t)ng * 32, TB);
        if (R == 1)
            { k_groups<T, 1><<<gg, TB, 0, s>>>((int64_t)ng, d_boff, d_gfirst, (int)nb, d_borig, dx, dy, dtype,
                                             sv, gH, gbox, grange, ray_l, ray_idx, d_bbox, nullptr, gflag, sub); note_launch(); }
        else if (R == 2)
            { k_groups<T, 2><<<gg, TB, 0, s>>>((int64_t)ng, d_boff, d_gfirst, (int)nb, d_borig, dx, dy, dtype,
                                             sv, gH, gbox, grange, ray_l, ray_idx, d_bbox, nullptr, gflag, sub); note_launch(); }
        else
            { k_groups<T, 4><<<gg, TB, 0, s>>>((int64_t)ng, d_boff, d_gfirst, (int)nb, d_borig, dx, dy, dtype,
                                             sv, gH, gbox, grange, ray_l, ray_idx, d_bbox, nullptr, gflag, sub); note_launch(); }
    }

    if (nb == 1) {
        t->grp_dx = dx;
        t->grp_dy = dy;
        t->grp_n = n;
        t->grp_dtype = dtype;
        t->grp_R = R;
        t->grp_ox = plan.ox;
        t->grp_oy = plan.oy;
    }
    return LENS_OK;
}
template lens_status enqueue_groups<float>(lens_tree*, const ShootPlan&, const void*, const void*, int, cudaStream_t);
template lens_status enqueue_groups<double>(lens_tree*, const ShootPlan&, const void*, const void*, int, cudaStream_t);

void set_cost_key(lens_tree* t, const RayKey& k);

// Enqueue the kernels of one shoot call (no allocation, no host sync: safe
// to capture into a CUDA graph).
template <typename T>
static lens_status enqueue_typed(lens_tree* t, const ShootPlan& plan, const void* dx, const void* dy,
                                 int dtype, void* const out[5], int flags, cudaStream_t s)
{
    using T4 = vec4_t<T>;
    using T2 = v2_t<T>;
    const int64_t n = plan.n, nb = plan.nb;
    const uint64_t ng = plan.ng;
    const int R = plan.R;
    Layout L = make_layout(t->ray_cap, t->batch_cap, max_slots(t));
    char* base = (char*)t->ray_scratch.ptr;
    int64_t* d_boff = (int64_t*)(base + L.boff);
    double* d_borig = (double*)(base + L.borig);
    uint32_t* d_gfirst = (uint32_t*)(base + L.gfirst);
    unsigned long long* d_bbox = (unsigned long long*)(base + L.bbox);
    T2* ray_l = (T2*)(base + L.rl);
    uint32_t* ray_idx = (uint32_t*)(base + L.ridx);
    T2* gH = (T2*)(base + L.gH);
    T4* gbox = (T4*)(base + L.gbox);
    uint2* grange = (uint2*)(base + L.grange);
    uint32_t* counter = (uint32_t*)(base + L.counter);
    int* stack = (int*)(base + L.stack);
    const bool timing = (flags & LENS_TIMING) != 0;
    if (timing) {
        for (int i = 0; i < 4; ++i)
            if (!t->ev[i]) LENS_CUDA(cudaEventCreate(&t->ev[i]));
        LENS_CUDA(cudaEventRecord(t->ev[0], s));
    }
    if (n > 0) LENS_TRY(enqueue_groups<T>(t, plan, dx, dy, dtype, s));
    // a tree walk of one batch records its groups' work, and takes them
    // heaviest first when these rays were walked before on this tree
    RayKey key;
    key.dx = dx; key.dy = dy; key.n = n; key.dtype = dtype; key.R = R; key.ox = plan.ox; key.oy = plan.oy;
    const bool record = n > 0 && nb == 1 && !(flags & LENS_DIRECT);
    const uint32_t* order = record ? heavy_first_order<T>(t, plan, key, 0, s).order : nullptr;
    uint32_t* gcost = record ? (uint32_t*)(base + L.gcost) : nullptr;
    if (gcost) LENS_CUDA(cudaMemsetAsync(gcost, 0, ng * sizeof(uint32_t), s));
    // interaction lists for the adjoint (room made by the caller, shoot())
    const bool keep = record && (flags & LENS_KEEP_LISTS) && t->list_ids && t->list_groups >= (int64_t)ng;
    if (keep) LENS_CUDA(cudaMemsetAsync(t->list_n, 0xff, ng * sizeof(uint32_t), s));  // kListOverflow

    if (timing) LENS_CUDA(cudaEventRecord(t->ev[1], s));
    // the grouping above reads only the rays: it may overlap the end of a
    // build on another stream; the walk reads the tree
    LENS_TRY(wait_built(t, s));
    if (timing) LENS_CUDA(cudaEventRecord(t->ev[2], s));
    WalkParams<T> P{};
    P.stats = (flags & LENS_COUNT) ? t->d_stats : nullptr;
    P.gH = gH; P.gbox = gbox; P.grange = grange; P.ray_l = ray_l; P.ray_idx = ray_idx;
    P.n_groups = (int64_t)ng;
    P.n_rays = n;
    P.stack = stack;
    P.err = t->d_err;
    P.wait_cycles = t->wait_cycles;
    P.order = order;
    P.gcost = gcost;
    P.list_ids = keep ? t->list_ids : nullptr;
    P.list_n = keep ? t->list_n : nullptr;
    P.list_K = keep ? t->list_K : 0;
    for (int q = 0; q < 5; ++q) P.out[q] = (T*)out[q];
    const bool ao = (flags & LENS_ALPHA_ONLY) != 0;
    const bool direct = (flags & LENS_DIRECT) != 0;
    bool first_launch = true;
    int launches = 0;
    for (size_t si = 0; si < t->sp.size(); ++si) {
        const SpeciesTree& st = t->sp[si];
        if (st.n == 0) continue;
        P.nodeA = (const T4*)st.nodeA;
        P.nodeB = (const T2*)st.nodeB;
        P.link = st.link;
        P.node_rcm = st.node_rcm;
        P.leaf0 = (const T4*)((direct || st.kind == LENS_POINT) ? st.exact0 : st.leaf0);
        P.leaf1 = (const T4*)st.exact1;
        P.big0 = (const T4*)st.big0;
        P.big1 = (const T4*)st.big1;
        P.big_chunk = (const T4*)st.big_chunk;
        P.node_bigbox = (const T4*)st.node_bigbox;
        P.n_part = st.n;
        P.Uq = (T)st.Uq;
        P.invNq = (T)st.invNq;
        P.Uq2 = (T)(st.Uq * 1.4426950408889634074);
        P.Nq = (T)(st.invNq > 0 ? 1.0 / st.invNq : 0.0);
        P.eU = (T)std::exp(-st.Uq);
        P.halos = t->halos;
        P.n_halos = first_launch ? (int)t->n_halos : 0;
        P.accumulate = first_launch ? ((flags & LENS_ACCUMULATE) ? 1 : 0) : 1;
        P.counter = counter + 8 * launches;
        LENS_CUDA(cudaMemsetAsync(P.counter, 0, 8 * sizeof(uint32_t), s));
        // few ray groups in a direct sum: split the particles over slices too
        P.n_slices = direct ? split_slices(t, (int64_t)ng, n, st.n) : 1;
        P.split_n = n;
        P.split = (T*)(base + L.split);
        if (n > 0) {
            bool done = false;
            if (!direct && (t->walk_mode == LENS_WALK_PAIRS || t->walk_mode == LENS_WALK_TRIOS)) {
                const int consumers = t->walk_mode == LENS_WALK_TRIOS ? 2 : 1;
                if (R <= 2)
                    done = R == 1 ? launch_ws<T, 1>(st.kind, ao, P, t->num_sms, s, consumers)
                                  : launch_ws<T, 2>(st.kind, ao, P, t->num_sms, s, consumers);
            }
            if (!done && direct) {
                if (R == 1) launch_direct<T, 1>(st.kind, ao, P, t->num_sms, s);
                else if (R == 2) launch_direct<T, 2>(st.kind, ao, P, t->num_sms, s);
                else return lens_set_error(LENS_ERR_INTERNAL, "128-ray groups in a direct sum");
            } else if (!done) {
                const int nq = ao ? 2 : 5;
                // supergroups from 16,384 groups (512 warps of k_super), where
                // the caller keeps no lists and counts nothing
                if constexpr (sizeof(T) == 4) {
                    P.super = nullptr;
                    if (st.kind == LENS_POINT && ng >= 16384 && !keep && !P.stats) {
                        const double th = 0.3 / t->theta;
                        P.super = launch_super(P, st, base, L, counter + 8 * launches + 3, nb, dtype,
                                               R == 4 ? INFINITY : (float)(kNearMax * R * R * th * th * th), t->num_sms, s);
                    }
                }
                P.counter = counter + 8 * launches;
                if (R == 1) walk_tree<T, 1>(st.kind, ao, P, t, nq, base, L, s);
                else if (R == 2) walk_tree<T, 2>(st.kind, ao, P, t, nq, base, L, s);
                else walk_tree<T, 4>(st.kind, ao, P, t, nq, base, L, s);
            }
            if (P.n_slices > 1) {
                k_split_sum<T><<<grid_for(n, 256), 256, 0, s>>>(n, P.n_slices, ao ? 2 : 5, P.split, P.out[0], P.out[1],
                                                              P.out[2], P.out[3], P.out[4], P.accumulate);
                note_launch();
            }
        }
        first_launch = false;
        ++launches;
    }
    if (first_launch && n > 0) {
        // no particles at all: analytic components only
        P.n_part = 0;
        P.halos = t->halos;
        P.n_halos = (int)t->n_halos;
        P.accumulate = (flags & LENS_ACCUMULATE) ? 1 : 0;
        P.counter = counter;
        LENS_CUDA(cudaMemsetAsync(P.counter, 0, sizeof(uint32_t), s));
        if (R == 1) launch_direct<T, 1>(LENS_POINT, ao, P, t->num_sms, s);
        else if (R == 2) launch_direct<T, 2>(LENS_POINT, ao, P, t->num_sms, s);
        else return lens_set_error(LENS_ERR_INTERNAL, "128-ray groups without particles");
    }
    if (timing) {
        LENS_CUDA(cudaEventRecord(t->ev[3], s));
        t->timed = true;
    }
    if (record) set_cost_key(t, key);
    if (keep) {
        t->list_dx = key.dx;
        t->list_dy = key.dy;
        t->list_rays = key.n;
        t->list_dtype = key.dtype;
        t->list_R = key.R;
        t->list_ox = key.ox;
        t->list_oy = key.oy;
    }
    LENS_CUDA(cudaGetLastError());
    return LENS_OK;
}

lens_status enqueue_shoot(lens_tree* t, const ShootPlan& plan, const void* dx, const void* dy, int dtype,
                          void* const out[5], int flags, cudaStream_t s)
{
    if (t->precision == LENS_PREC_FP64) return enqueue_typed<double>(t, plan, dx, dy, dtype, out, flags, s);
    return enqueue_typed<float>(t, plan, dx, dy, dtype, out, flags, s);
}

// Room for the interaction lists of ng groups of R * 32 rays (512 entries
// per 32 rays).  The old lists are dropped.
static lens_status reserve_lists(lens_tree* t, int64_t ng, int R, cudaStream_t s)
{
    const int K = 512 * R;
    t->list_rays = -1;  // whatever is kept belongs to no rays until the walk records
    if (t->list_ids && t->list_groups >= ng && t->list_K == K) return LENS_OK;
    if (t->list_ids || t->list_n) {
        LENS_CUDA(cudaStreamSynchronize(s));  // the old lists may still be read
        if (t->list_ids) cudaFreeAsync(t->list_ids, s);
        if (t->list_n) cudaFreeAsync(t->list_n, s);
    }
    t->list_ids = t->list_n = nullptr;
    t->list_groups = 0;
    // from the stream-ordered pool: a new tree's first kept lists cost no
    // device allocation call
    LENS_CUDA(lens_malloc_async((void**)&t->list_ids, (size_t)ng * K * sizeof(uint32_t), s));
    cudaError_t e = lens_malloc_async((void**)&t->list_n, (size_t)ng * sizeof(uint32_t), s);
    if (e != cudaSuccess) {
        cudaFreeAsync(t->list_ids, s);
        t->list_ids = nullptr;
        return lens_cuda_check(e, "cudaMallocAsync(lists)");
    }
    t->list_groups = ng;
    t->list_K = K;
    return LENS_OK;
}

lens_status shoot(lens_tree* t, int64_t nb, const int64_t* h_off, const double* h_orig, const void* dx,
                  const void* dy, int dtype, void* const out[5], int flags, cudaStream_t s)
{
    ShootPlan plan;
    LENS_TRY(upload_batches(t, nb, h_off, h_orig, s, &plan, shoot_max_r(t, flags)));
    // kept lists hold box indices in 29 bits
    bool small_tree = true;
    for (const auto& st : t->sp) small_tree = small_tree && st.n_nodes < (int64_t)kListIdMask;
    // (the adjoint groups at most 64 rays: lists of 128-ray groups would not be its)
    if ((flags & LENS_KEEP_LISTS) && !(flags & LENS_DIRECT) && nb == 1 && plan.n > 0 && small_tree && plan.R <= 2)
        LENS_TRY(reserve_lists(t, (int64_t)plan.ng, plan.R, s));
    else
        flags &= ~LENS_KEEP_LISTS;
    return enqueue_shoot(t, plan, dx, dy, dtype, out, flags, s);
}

bool groups_hold(const lens_tree* t, const RayKey& k)
{
    return t->grp_n >= 0 && t->grp_dx == k.dx && t->grp_dy == k.dy && t->grp_n == k.n &&
           t->grp_dtype == k.dtype && t->grp_R == k.R && t->grp_ox == k.ox && t->grp_oy == k.oy;
}

// The kept interaction lists if they belong to these rays, else null.
const uint32_t* kept_lists(const lens_tree* t, const RayKey& k)
{
    if (!t->list_ids || t->list_rays < 0) return nullptr;
    const bool same = t->list_dx == k.dx && t->list_dy == k.dy && t->list_rays == k.n && t->list_dtype == k.dtype &&
                      t->list_R == k.R && t->list_ox == k.ox && t->list_oy == k.oy;
    return same ? t->list_ids : nullptr;
}

// Scratch views shared with the backward walk.
void* scratch_base(lens_tree* t) { return t->ray_scratch.ptr; }

__global__ void k_cost_keys(uint32_t ng, const uint32_t* gcost, uint32_t* keys, uint32_t* vals,
                            unsigned long long* total)
{
    const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t c = g < ng ? gcost[g] : 0u;
    if (g < ng) {
        keys[g] = ~c;  // ascending sort of the complement: heaviest first, ties in group order
        vals[g] = g;
    }
    unsigned long long w = c;
    for (int o = 16; o; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
    if ((threadIdx.x & 31) == 0 && w) atomicAdd(total, w);
}

// Slices of the heaviest groups (one block of kHeavyGroups threads; thread
// i owns the group at position i of the order).  The slice counts are
// non-increasing along the order, so the split groups are its first Kc.
__global__ void __launch_bounds__(kHeavyGroups) k_heavy_plan(uint32_t ng, const uint32_t* sorted_keys,
                                                             unsigned long long n_warps, uint32_t* hdr,
                                                             uint32_t* table)
{
    __shared__ uint32_t wsum[kHeavyGroups / 32];
    const uint32_t i = threadIdx.x, lane = i & 31, warp = i >> 5;
    const unsigned long long total = *(const unsigned long long*)(hdr + 8);
    unsigned long long cap = total / (4ull * n_warps);  // a quarter of one warp's share
    if (cap < 1) cap = 1;
    uint32_t v = 0;  // slices of a split group, 0 for a whole one
    if (i < ng) {
        unsigned long long q = ((unsigned long long)(~sorted_keys[i]) + cap - 1) / cap;
        if (q > 1) v = q > 32 ? 32u : (uint32_t)q;
    }
    uint32_t x = v;  // inclusive scan over the block
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= (uint32_t)o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    const int kc = __syncthreads_count(v > 0);
    if (warp == 0) {
        uint32_t w = wsum[lane];
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= (uint32_t)o) w += y;
        }
        wsum[lane] = w;
    }
    __syncthreads();
    const uint32_t first = x - v + (warp ? wsum[warp - 1] : 0u);
    for (uint32_t k = 0; k < v; ++k) table[first + k] = (i << 10) | (k << 5) | (v - 1);
    if (i == 0) {
        hdr[0] = (uint32_t)kc;
        hdr[1] = wsum[kHeavyGroups / 32 - 1];
    }
}

static bool cost_key_matches(const lens_tree* t, const RayKey& k)
{
    return t->cost_dx == k.dx && t->cost_dy == k.dy && t->cost_n == k.n && t->cost_dtype == k.dtype &&
           t->cost_R == k.R && t->cost_ox == k.ox && t->cost_oy == k.oy;
}

void set_cost_key(lens_tree* t, const RayKey& k)
{
    t->cost_dx = k.dx;
    t->cost_dy = k.dy;
    t->cost_n = k.n;
    t->cost_dtype = k.dtype;
    t->cost_R = k.R;
    t->cost_ox = k.ox;
    t->cost_oy = k.oy;
}

template <typename T>
HeavyPlan heavy_first_order(lens_tree* t, const ShootPlan& plan, const RayKey& key, int64_t n_warps,
                            cudaStream_t s)
{
    HeavyPlan hp;
    if (plan.nb != 1 || plan.ng < 2 || !cost_key_matches(t, key)) return hp;
    Layout L = make_layout(t->ray_cap, t->batch_cap, max_slots(t));
    char* base = (char*)t->ray_scratch.ptr;
    uint32_t* k0 = (uint32_t*)(base + L.k0);
    uint32_t* k1 = (uint32_t*)(base + L.k1);
    uint32_t* v0 = (uint32_t*)(base + L.v0);
    uint32_t* v1 = (uint32_t*)(base + L.v1);
    uint32_t* hdr = (uint32_t*)(base + L.heavy);
    uint32_t* table = hdr + 16;
    const uint32_t ng = (uint32_t)plan.ng;
    if (cudaMemsetAsync(hdr, 0, 64, s) != cudaSuccess) return hp;
    {
        k_cost_keys<<<grid_for(ng, 256), 256, 0, s>>>(ng, (const uint32_t*)(base + L.gcost), k0, v0,
                                                       (unsigned long long*)(hdr + 8));
        note_launch();
    }
    uint32_t *sk, *sv;
    radix_sort_pairs<uint32_t>(k0, v0, k1, v1, ng, 0, 32, base + L.tmp, s, &sk, &sv, t->d_err);
    hp.order = sv;
    if (n_warps > 0) {
        { k_heavy_plan<<<1, kHeavyGroups, 0, s>>>(ng, sk, (unsigned long long)n_warps, hdr, table); note_launch(); }
        hp.hdr = hdr;
        hp.table = table;
    }
    return hp;
}
template HeavyPlan heavy_first_order<float>(lens_tree*, const ShootPlan&, const RayKey&, int64_t, cudaStream_t);
template HeavyPlan heavy_first_order<double>(lens_tree*, const ShootPlan&, const RayKey&, int64_t, cudaStream_t);

}  // namespace lens

// ===================================================== allocation-free shoot
//
// lens_shoot_rays_direct_noalloc: the direct sum over every particle of a
// built tree, for callers that must not allocate device memory while they
// shoot rays.  Its ray-group scratch (work counters, per-group anchors and
// boxes, per-ray offsets and indices) lives in one file-scope device array of
// fixed size instead of the tree's on-demand buffers; rays are grouped in
// their input order, 32 per group, so no sort buffers are needed.

namespace lens {

constexpr int64_t kNoAllocMaxRays = 262144;
constexpr size_t kNoAllocGroups = (size_t)(kNoAllocMaxRays / 32 + 1);
constexpr size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }
// byte offsets of the pieces (every piece 256-byte aligned; sizes for FP64)
constexpr size_t kNaCounters = 0;  // one work counter per launch (64 launches)
constexpr size_t kNaRayL = kNaCounters + 256;
constexpr size_t kNaRayIdx = kNaRayL + al256((size_t)kNoAllocMaxRays * 2 * sizeof(double));
constexpr size_t kNaGH = kNaRayIdx + al256((size_t)kNoAllocMaxRays * sizeof(uint32_t));
constexpr size_t kNaGBox = kNaGH + al256(kNoAllocGroups * 2 * sizeof(double));
constexpr size_t kNaGRange = kNaGBox + al256(kNoAllocGroups * 4 * sizeof(double));
constexpr size_t kNoAllocBytes = kNaGRange + al256(kNoAllocGroups * sizeof(uint2));

// One copy per device that loads the library, held until the process exits.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

template <typename T>
__global__ void k_groups_inorder(int64_t n, double ox, double oy, const void* dx, const void* dy, int dtype,
                                 int64_t n_groups, v2_t<T>* gH, vec4_t<T>* gbox, uint2* grange,
                                 v2_t<T>* ray_l, uint32_t* ray_idx)
{
    const unsigned full = 0xffffffffu;
    int lane = threadIdx.x & 31;
    int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (g >= n_groups) return;
    int64_t i = 32 * g + lane;
    bool v = i < n;
    double px = v ? ox + ray_offset(dx, dtype, i) : 0.0, py = v ? oy + ray_offset(dy, dtype, i) : 0.0;
    double xmin = v ? px : INFINITY, xmax = v ? px : -INFINITY, ymin = v ? py : INFINITY, ymax = v ? py : -INFINITY;
    for (int o = 16; o; o >>= 1) {
        xmin = fmin(xmin, __shfl_xor_sync(full, xmin, o));
        xmax = fmax(xmax, __shfl_xor_sync(full, xmax, o));
        ymin = fmin(ymin, __shfl_xor_sync(full, ymin, o));
        ymax = fmax(ymax, __shfl_xor_sync(full, ymax, o));
    }
    bool exact = !v || ((double)(T)px == px && (double)(T)py == py);
    exact = __all_sync(full, exact);
    T Hx = exact ? T(0) : (T)(0.5 * (xmin + xmax)), Hy = exact ? T(0) : (T)(0.5 * (ymin + ymax));
    T lx = v ? (T)(px - (double)Hx) : T(0), ly = v ? (T)(py - (double)Hy) : T(0);
    T lxmin = v ? lx : (T)INFINITY, lxmax = v ? lx : (T)-INFINITY, lymin = v ? ly : (T)INFINITY,
      lymax = v ? ly : (T)-INFINITY;
    for (int o = 16; o; o >>= 1) {
        lxmin = fmin(lxmin, __shfl_xor_sync(full, lxmin, o));
        lxmax = fmax(lxmax, __shfl_xor_sync(full, lxmax, o));
        lymin = fmin(lymin, __shfl_xor_sync(full, lymin, o));
        lymax = fmax(lymax, __shfl_xor_sync(full, lymax, o));
    }
    if (v) {
        v2_t<T> l;
        l.x = lx;
        l.y = ly;
        ray_l[i] = l;
        ray_idx[i] = (uint32_t)i;
    }
    if (lane == 0) {
        T cx = T(0.5) * (lxmin + lxmax), cy = T(0.5) * (lymin + lymax);
        T hx = fmax(lxmax - cx, cx - lxmin) * T(1.0 + 1e-5) + T(1e-30);
        T hy = fmax(lymax - cy, cy - lymin) * T(1.0 + 1e-5) + T(1e-30);
        v2_t<T> H;
        H.x = Hx;
        H.y = Hy;
        gH[g] = H;
        vec4_t<T> bx;
        bx.x = cx; bx.y = cy; bx.z = hx; bx.w = hy;
        gbox[g] = bx;
        int64_t cnt = n - 32 * g;
        grange[g] = make_uint2((uint32_t)(32 * g), (uint32_t)(cnt < 32 ? cnt : 32));
    }
}

// Device address of the scratch array on the current device (the host-side
// name of a __device__ array is only a handle, not a device address).
// lens_build_tree looks it up with the tree's device current and keeps it in
// the tree, so the allocation-free call itself makes no runtime lookup, and a
// tree built after a device reset holds the new address.
lens_status noalloc_scratch_address(void** out)
{
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) {
        *out = nullptr;
        return lens_cuda_check(e == cudaSuccess ? cudaErrorInvalidSymbol : e, "cudaGetSymbolAddress(no-alloc scratch)");
    }
    *out = p;
    return LENS_OK;
}

template <typename T>
static lens_status noalloc_typed(lens_tree* t, double ox, double oy, const void* dx, const void* dy,
                                 int dtype, int64_t n, void* const out[5], int flags, cudaStream_t s)
{
    using T4 = vec4_t<T>;
    using T2 = v2_t<T>;
    unsigned char* base = (unsigned char*)t->noalloc_scratch;
    if (!base) return lens_set_error(LENS_ERR_INTERNAL, "tree holds no address of the no-alloc scratch");
    uint32_t* counters = (uint32_t*)(base + kNaCounters);
    T2* ray_l = (T2*)(base + kNaRayL);
    uint32_t* ray_idx = (uint32_t*)(base + kNaRayIdx);
    T2* gH = (T2*)(base + kNaGH);
    T4* gbox = (T4*)(base + kNaGBox);
    uint2* grange = (uint2*)(base + kNaGRange);
    const int64_t ng = (n + 31) / 32;
    // the work counters must start at zero: the array keeps the last call's values
    LENS_CUDA(cudaMemsetAsync(counters, 0, 256, s));
    { k_groups_inorder<T><<<grid_for(ng * 32, 256), 256, 0, s>>>(n, ox, oy, dx, dy, dtype, ng, gH, gbox, grange,
                                                                 ray_l, ray_idx); note_launch(); }
    WalkParams<T> P{};
    P.gH = gH; P.gbox = gbox; P.grange = grange; P.ray_l = ray_l; P.ray_idx = ray_idx;
    P.n_groups = ng;
    P.stack = (int*)base;  // the direct sum never touches a stack
    P.err = t->d_err;
    for (int q = 0; q < 5; ++q) P.out[q] = (T*)out[q];
    const bool ao = (flags & LENS_ALPHA_ONLY) != 0;
    int launches = 0;
    bool first_launch = true;
    for (size_t si = 0; si < t->sp.size(); ++si) {
        const SpeciesTree& sp = t->sp[si];
        if (sp.n == 0) continue;
        P.leaf0 = (const T4*)sp.exact0;
        P.leaf1 = (const T4*)sp.exact1;
        P.n_part = sp.n;
        P.Uq = (T)sp.Uq;
        P.invNq = (T)sp.invNq;
        P.halos = t->halos;
        P.n_halos = first_launch ? (int)t->n_halos : 0;
        P.accumulate = first_launch ? ((flags & LENS_ACCUMULATE) ? 1 : 0) : 1;
        P.counter = counters + launches;
        launch_direct<T, 1>(sp.kind, ao, P, t->num_sms, s);
        first_launch = false;
        ++launches;
    }
    if (first_launch) {
        P.n_part = 0;
        P.halos = t->halos;
        P.n_halos = (int)t->n_halos;
        P.accumulate = (flags & LENS_ACCUMULATE) ? 1 : 0;
        P.counter = counters;
        launch_direct<T, 1>(LENS_POINT, ao, P, t->num_sms, s);
    }
    LENS_CUDA(cudaGetLastError());
    return LENS_OK;
}

}  // namespace lens

extern "C" lens_status lens_shoot_rays_direct_noalloc(lens_tree* tree, double origin_x, double origin_y,
                                                      const void* ray_dx, const void* ray_dy,
                                                      int32_t ray_dtype, int64_t n, void* alpha1,
                                                      void* alpha2, void* kappa, void* gamma1, void* gamma2,
                                                      int32_t flags, void* stream)
{
    using namespace lens;
    if (!tree) return lens_set_error(LENS_ERR_INVALID_ARG, "tree is NULL");
    if (flags & ~(LENS_ALPHA_ONLY | LENS_ACCUMULATE))
        return lens_set_error(LENS_ERR_INVALID_ARG, "only LENS_ALPHA_ONLY and LENS_ACCUMULATE apply here");
    if (n < 0) return lens_set_error(LENS_ERR_INVALID_ARG, "n must be >= 0");
    if (n > kNoAllocMaxRays)
        return lens_set_error(LENS_ERR_INVALID_ARG,
                              "lens_shoot_rays_direct_noalloc takes at most %lld rays per call (got %lld)",
                              (long long)kNoAllocMaxRays, (long long)n);
    if (ray_dtype != LENS_F32 && ray_dtype != LENS_F64) return lens_set_error(LENS_ERR_INVALID_ARG, "bad ray dtype");
    if (!std::isfinite(origin_x) || !std::isfinite(origin_y))
        return lens_set_error(LENS_ERR_INVALID_ARG, "origin must be finite");
    if (n == 0) return LENS_OK;
    if (!ray_dx || !ray_dy || !alpha1 || !alpha2) return lens_set_error(LENS_ERR_INVALID_ARG, "NULL array");
    if (!(flags & LENS_ALPHA_ONLY) && (!kappa || !gamma1 || !gamma2))
        return lens_set_error(LENS_ERR_INVALID_ARG, "kappa/gamma outputs are NULL without LENS_ALPHA_ONLY");
    int dev = -1;
    LENS_CUDA(cudaGetDevice(&dev));
    if (dev != tree->device) return lens_set_error(LENS_ERR_INVALID_ARG, "tree was built on another device");
    void* out[5] = {alpha1, alpha2, kappa, gamma1, gamma2};
    cudaStream_t s = (cudaStream_t)stream;
    LENS_TRY(wait_built(tree, s));
    if (tree->precision == LENS_PREC_FP64)
        return noalloc_typed<double>(tree, origin_x, origin_y, ray_dx, ray_dy, ray_dtype, n, out, flags, s);
    return noalloc_typed<float>(tree, origin_x, origin_y, ray_dx, ray_dy, ray_dtype, n, out, flags, s);
}
