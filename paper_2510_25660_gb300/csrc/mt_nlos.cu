// mt_nlos.cu -- relay-wall NLOS impulse responses (arXiv 2510.25660 Sec. 4.5).
//
// Third-bounce transport laser -> x_l -> y -> x_s -> sensor with y drawn
// uniformly by area on the hidden triangles; the clock is the relay-wall
// clock |x_l - y| + |y - x_s|.  With unit laser power at x_l and Lambertian
// wall (albedo rho_w) and hidden surface (rho_h):
//   H = (rho_w/pi) cos_l (rho_h/pi) cos_y1 cos_y2 (rho_w/pi) cos_s
//       / (|x_l - y|^2 |y - x_s|^2) * A_hidden * V(x_l, y) V(y, x_s)
// per sample.  All scan pairs are one persistent launch.  The default forms add
// to the film in L2: k_nlos_scan takes a scan point per CTA and its samples in
// the order of the hidden surface, k_nlos_pairs takes 32 sensors of a laser per
// warp.  k_nlos (small exhaustive grids and those of few sensors, a launch
// configuration that privatises bins, aggregates or sets a tile, and the dump)
// pulls tiles of consecutive film rows and keeps the rows' time histograms in
// shared memory.  In the exhaustive grid the hidden
// samples of a laser are drawn once (visibility x_l -> y included) by
// k_nlos_ysample and shared by all its sensors.
#include "mt_common.cuh"
#include "mt_internal.h"
#include "mt_launch.h"
#include "mt_trace.cuh"

namespace {

// CTAs per SM the default kernels leave room for.  64x64 scan points, 1024 samples: 1.42 / 1.31 / 1.26 / 1.27 ms at 4 /
// 5 / 6 / 8 (the traversal waits on gathers and on the CTA's last warp); 16x16 x 32x32 pairs, 1024 samples: 10.97 /
// 11.05 / 11.09 / 11.03 ms.
#ifndef MT_NLOS_SCAN_MINB
#define MT_NLOS_SCAN_MINB 6
#endif
#ifndef MT_NLOS_PAIRS_MINB
#define MT_NLOS_PAIRS_MINB 4
#endif

// smallest i with key < hcdf[i] (the last index if none); the guide table only
// narrows the bracket the same search runs in, so the pick is unchanged
__device__ __forceinline__ int pick_hidden(const NlosParams &p, uint32_t u) {
    int lo = 0, hi = p.hidden_n - 1;
    const uint32_t key = u >> 8;
    if (p.hguide) {
        const uint32_t g = key >> 12;
        lo = min((int)__ldg(&p.hguide[g]), p.hidden_n - 1);
        hi = min((int)__ldg(&p.hguide[g + 1]), p.hidden_n - 1);
    }
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (key < __ldg(&p.hcdf[mid])) hi = mid;
        else lo = mid + 1;
    }
    return p.hidden_first + lo;
}

// The arithmetic of a connection is spelled out, once for all kernels of this file: which product of a sum of
// products is fused is the compiler's choice at each place a function is inlined, and a path length that differs in
// its last bit moves a connection across a bin edge (about 75 of the 67 M that reach the film of 16x16 x 32x32 pairs,
// T = 4096, 1024 samples: 3e-4 to 4e-3 of the film's norm, while each kernel repeats its own film to 1e-8).  Each sum
// has one order; dot_xyz and dot_yxz name the order in which the products enter.
__device__ __forceinline__ float dot_xyz(float3 a, float3 b) {
    return fmaf(a.z, b.z, fmaf(a.y, b.y, __fmul_rn(a.x, b.x)));
}
__device__ __forceinline__ float dot_yxz(float3 a, float3 b) {
    return fmaf(a.z, b.z, fmaf(a.x, b.x, __fmul_rn(a.y, b.y)));
}

// uniform point on a triangle (tri_point)
__device__ __forceinline__ float3 hidden_point(float3 v0, float3 v1, float3 v2, float u1, float u2) {
    const float su = sqrtf(u1);
    const float b0 = 1.0f - su, b1 = __fmul_rn(u2, su), b2 = __fsub_rn(1.0f - b0, b1);
    auto mix = [&](float x0, float x1, float x2) { return fmaf(x2, b2, fmaf(x0, b0, __fmul_rn(x1, b1))); };
    return f3(mix(v0.x, v1.x, v2.x), mix(v0.y, v1.y, v2.y), mix(v0.z, v1.z, v2.z));
}

__device__ __forceinline__ float3 hidden_normal(float3 v0, float3 v1, float3 v2) {
    const float3 a = v1 - v0, b = v2 - v0;
    auto minor = [](float x, float y, float z, float w) { return fmaf(x, y, -__fmul_rn(z, w)); };
    const float3 c = f3(minor(a.y, b.z, a.z, b.y), minor(a.z, b.x, a.x, b.z), minor(a.x, b.y, a.y, b.x));
    return c * (1.0f / sqrtf(dot_yxz(c, c)));
}

// p moved off its surface along the unit normal n
__device__ __forceinline__ float3 lift(float3 p, float3 n) {
    const float e = eps_of(p);
    return f3(fmaf(n.x, e, p.x), fmaf(n.y, e, p.y), fmaf(n.z, e, p.z));
}

struct HiddenSample {
    float3 y, ny;
    float d1, partial;  // partial = fw cos_l fh cos_y1 / d1^2 * A (0 if invalid or occluded)
    float cl, cy1;
    int tri;
};

// hidden sample (l, smp) on triangle `tri`, leaf index k; R = its random words
template <bool CNT>
__device__ __forceinline__ HiddenSample sample_on(const DevScene &s, const NlosParams &p, const uint4 R, int tri, int k,
                                                  float3 xl, TraceCnt &tc, uint32_t &rays) {
    HiddenSample h;
    float3 v0, v1, v2;
    tri_vertices(s, k, v0, v1, v2);
    h.tri = tri;
    h.y = hidden_point(v0, v1, v2, u24(R.y), u24(R.z));
    h.partial = 0.f;
    h.cl = h.cy1 = 0.f;
    const float3 ng = hidden_normal(v0, v1, v2);
    const float3 d1v = h.y - xl;
    h.d1 = sqrtf(dot_yxz(d1v, d1v));
    if (!(h.d1 > 0.f)) return h;
    const float3 w1 = d1v * (1.0f / h.d1);
    h.ny = dot_yxz(ng, -w1) >= 0.f ? ng : -ng;
    const float cl = dot_yxz(p.nw, w1), cy1 = -dot_yxz(h.ny, w1);
    h.cl = cl;
    h.cy1 = cy1;
    if (!(cl > 0.f && cy1 > 0.f)) return h;
    const float3 xlo = lift(xl, p.nw);
    const float3 r1 = h.y - xlo;
    const float l1 = sqrtf(dot_yxz(r1, r1));
    rays++;
    const RayT ray = make_ray(s, xlo, r1 * (1.0f / l1));
    if (trace_any<CNT>(s, ray, l1 - eps_of(h.y), tc)) return h;
    const float4 m = __ldg(&s.mats[tri]);
    const float fh = (m.x + m.y + m.z) * (1.0f / 3.0f) * (1.0f / MT_PI);
    const float area = p.hidden_area_dev ? __ldg(p.hidden_area_dev) : p.hidden_area;
    h.partial = p.fw * cl * fh * cy1 / (h.d1 * h.d1) * area;
    return h;
}

// confocal connection of a visible hidden sample (x_s = x_l, the same segment both ways)
__device__ __forceinline__ float confocal_value(const NlosParams &p, const HiddenSample &h) {
    return h.partial * h.cy1 * h.cl * p.fw / (h.d1 * h.d1);
}

// connection of a hidden sample of its laser (ya = y, d1; yb = normal, partial) with the sensor at xs: its value (0:
// none) and its path length
template <bool CNT>
__device__ __forceinline__ float sensor_value(const DevScene &s, const NlosParams &p, float4 ya, float4 yb, float3 xs,
                                              float &opl, TraceCnt &tc, uint32_t &rays) {
    if (!(yb.w > 0.f)) return 0.f;
    const float3 y = xyz(ya), ny = xyz(yb);
    const float3 d2v = xs - y;
    const float d2 = sqrtf(dot_xyz(d2v, d2v));
    if (!(d2 > 0.f)) return 0.f;
    const float3 w2 = d2v * (1.0f / d2);
    const float cs = -dot_yxz(p.nw, w2), cy2 = dot_yxz(ny, w2);
    if (!(cs > 0.f && cy2 > 0.f)) return 0.f;
    const float3 yo = lift(y, ny);
    const float3 r2 = xs - yo;
    const float l2 = sqrtf(dot_xyz(r2, r2));
    rays++;
    const RayT ray = make_ray(s, yo, r2 * (1.0f / l2));
    if (trace_any<CNT>(s, ray, l2 - eps_of(xs), tc)) return 0.f;
    opl = ya.w + d2;
    return yb.w * cy2 * cs * p.fw / (d2 * d2);
}

__device__ __forceinline__ uint4 hidden_words(const NlosParams &p, int l, uint32_t smp) {
    return philox4x32_10(make_uint4((uint32_t)l, smp, 0u, 0u), p.k0, p.k1);
}

template <bool CNT>
__device__ __forceinline__ HiddenSample sample_hidden(const DevScene &s, const NlosParams &p, int l, uint32_t smp,
                                                      float3 xl, TraceCnt &tc, uint32_t &rays) {
    const uint4 R = hidden_words(p, l, smp);
    const int tri = pick_hidden(p, R.x);
    return sample_on<CNT>(s, p, R, tri, __ldg(&s.leaf_of[tri]), xl, tc, rays);
}

// Samples j0 .. j0 + n of laser l, n <= MT_NLOS_BATCH, in the order of the
// hidden surface: a counting sort of their triangles' leaf indices (the
// depth-first order of the tree, so neighbours in space) into 256 buckets.
// Warps that take the samples in this order trace rays toward one patch of the
// surface instead of all over it (10.6 active lanes per instruction against
// 5.4, half the warp instructions).  o.at receives the order, o.tri the
// triangle of each sample (indices relative to j0).
#define MT_NLOS_BATCH 1024
struct SampleOrder {
    uint32_t cnt[256];
    uint32_t key[MT_NLOS_BATCH];  // bucket << 16 | rank in the bucket
    int tri[MT_NLOS_BATCH];
    uint16_t at[MT_NLOS_BATCH];
};
__device__ __forceinline__ void order_samples(const DevScene &s, const NlosParams &p, int l, int j0, int n,
                                              SampleOrder &o) {
    for (int b = threadIdx.x; b < 256; b += blockDim.x) o.cnt[b] = 0u;
    __syncthreads();
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const int tri = pick_hidden(p, hidden_words(p, l, p.sample_offset + (uint32_t)(j0 + j)).x);
        const uint32_t k = (uint32_t)__ldg(&s.leaf_of[tri]);
        const uint32_t b = (uint32_t)((unsigned long long)k * 256u / (uint32_t)s.n_tris);
        o.tri[j] = tri;
        o.key[j] = (b << 16) | atomicAdd(&o.cnt[b], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 32) {  // exclusive scan of the 256 counts, eight per lane
        uint32_t c[8], sum = 0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            c[q] = sum;
            sum += o.cnt[threadIdx.x * 8 + q];
        }
        uint32_t x = sum;
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
            if ((int)threadIdx.x >= d) x += y;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) o.cnt[threadIdx.x * 8 + q] = x - sum + c[q];
    }
    __syncthreads();
    for (int j = threadIdx.x; j < n; j += blockDim.x)
        o.at[o.cnt[o.key[j] >> 16] + (o.key[j] & 0xFFFFu)] = (uint16_t)j;
    __syncthreads();
}

__device__ __forceinline__ void add_counters(const DevScene &s, uint32_t conns, uint32_t contribs, uint32_t rays,
                                             const TraceCnt &tc) {
    unsigned long long v[5] = {conns, contribs, rays, tc.nodes, tc.tris};
    const int c_idx[5] = {1, 2, 3, 4, 5};
    for (int c = 0; c < 5; ++c) {
        unsigned long long x = v[c];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if ((threadIdx.x & 31) == 0 && x) atomicAdd(&s.counters[c_idx[c]], x);
    }
}

// a connection of value H at opl into film row `row`
__device__ __forceinline__ void nlos_splat(const NlosParams &p, long long row, float opl, float v) {
    const float x = (opl - p.start) / p.width;
    if (x >= 0.f && x < (float)p.T) atomicAdd(&p.film[(size_t)row * p.T + (int)x], v);
}

// scan points: a CTA takes one film row at a time, its samples in the order of the hidden surface
template <bool CNT>
__global__ void __launch_bounds__(256, MT_NLOS_SCAN_MINB) k_nlos_scan(const DevScene s, const NlosParams p) {
    __shared__ SampleOrder so;
    __shared__ float s_steady;
    __shared__ int s_row;
    uint32_t conns = 0, contribs = 0, rays = 0;
    TraceCnt tc{0, 0};
    for (;;) {
        if (threadIdx.x == 0) {
            s_row = atomicAdd(p.tile_counter, 1);
            s_steady = 0.f;
        }
        __syncthreads();
        const int row = s_row;
        if (row >= p.n_l) break;
        const float3 xl = f3(p.lasers[3 * row], p.lasers[3 * row + 1], p.lasers[3 * row + 2]);
        float steady = 0.f;
        for (int j0 = 0; j0 < p.spp; j0 += MT_NLOS_BATCH) {
            const int n = min(MT_NLOS_BATCH, p.spp - j0);
            order_samples(s, p, row, j0, n, so);
            for (int i = threadIdx.x; i < n; i += blockDim.x) {
                const int j = so.at[i], tri = so.tri[j];
                conns++;
                const uint4 R = hidden_words(p, row, p.sample_offset + (uint32_t)(j0 + j));
                const HiddenSample h = sample_on<CNT>(s, p, R, tri, __ldg(&s.leaf_of[tri]), xl, tc, rays);
                if (h.partial > 0.f) {
                    const float H = confocal_value(p, h);
                    if (H > 0.f) {
                        contribs++;
                        const float v = H * p.scale;
                        nlos_splat(p, row, 2.0f * h.d1, v);
                        steady += v;
                    }
                }
            }
            __syncthreads();
        }
        for (int o = 16; o > 0; o >>= 1) steady += __shfl_xor_sync(0xffffffffu, steady, o);
        if ((threadIdx.x & 31) == 0) atomicAdd(&s_steady, steady);
        __syncthreads();
        if (threadIdx.x == 0 && p.steady) p.steady[row] = (p.flags & MT_ACCUMULATE) ? p.steady[row] + s_steady : s_steady;
    }
    add_counters(s, conns, contribs, rays, tc);
}

// exhaustive pass 1: hidden samples of every laser, shared by its sensors
template <bool CNT>
__global__ void __launch_bounds__(256) k_nlos_ysample(const DevScene s, const NlosParams p) {
    uint32_t rays = 0;
    TraceCnt tc{0, 0};
    const long long total = (long long)p.n_l * p.spp;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
         i += (long long)gridDim.x * blockDim.x) {
        const int l = (int)(i / p.spp);
        const uint32_t smp = p.sample_offset + (uint32_t)(i - (long long)l * p.spp);
        const float3 xl = f3(p.lasers[3 * l], p.lasers[3 * l + 1], p.lasers[3 * l + 2]);
        const HiddenSample h = sample_hidden<CNT>(s, p, l, smp, xl, tc, rays);
        p.ysamp[2 * i] = make_float4(h.y.x, h.y.y, h.y.z, h.d1);
        p.ysamp[2 * i + 1] = make_float4(h.ny.x, h.ny.y, h.ny.z, h.partial);
        p.ysamp_tri[i] = h.tri;
    }
    add_counters(s, 0u, 0u, rays, tc);
}

// the same for k_nlos_pairs: a CTA per (laser, batch of samples), written in the order of the hidden surface within
// the batch (only the sum over samples is formed, so their order is free)
template <bool CNT>
__global__ void __launch_bounds__(256) k_nlos_ysample_ordered(const DevScene s, const NlosParams p) {
    __shared__ SampleOrder so;
    uint32_t rays = 0;
    TraceCnt tc{0, 0};
    const int batches = (p.spp + MT_NLOS_BATCH - 1) / MT_NLOS_BATCH;
    for (long long b = blockIdx.x; b < (long long)p.n_l * batches; b += gridDim.x) {
        const int l = (int)(b / batches), j0 = (int)(b - (long long)l * batches) * MT_NLOS_BATCH;
        const int n = min(MT_NLOS_BATCH, p.spp - j0);
        const float3 xl = f3(p.lasers[3 * l], p.lasers[3 * l + 1], p.lasers[3 * l + 2]);
        order_samples(s, p, l, j0, n, so);
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const int j = so.at[i], tri = so.tri[j];
            const uint4 R = hidden_words(p, l, p.sample_offset + (uint32_t)(j0 + j));
            const HiddenSample h = sample_on<CNT>(s, p, R, tri, __ldg(&s.leaf_of[tri]), xl, tc, rays);
            const size_t o = (size_t)l * p.spp + j0 + i;
            p.ysamp[2 * o] = make_float4(h.y.x, h.y.y, h.y.z, h.d1);
            p.ysamp[2 * o + 1] = make_float4(h.ny.x, h.ny.y, h.ny.z, h.partial);
        }
        __syncthreads();
    }
    add_counters(s, 0u, 0u, rays, tc);
}

// Sensor order of k_nlos_pairs: by the Morton code of their position on the wall (32 x 32 cells over the points'
// extent along two axes across the wall normal), so that the 32 rays of a warp go from one point y to a patch of the
// wall instead of a line across it (16x16 x 32x32 pairs, 1024 samples: 14.8 -> 10.97 ms).  One CTA; the order within
// a cell is free.  A sensor's cell is computed once and kept behind the order (order holds 2 n_s entries): counted and
// placed from one value, the order is a permutation of the sensors whatever the rounding of the cell, NaN included.
__global__ void __launch_bounds__(1024) k_nlos_sensor_order(const NlosParams p, int32_t *order) {
    __shared__ int s_box[4];  // ordered ints: lower t, b; upper t, b
    __shared__ uint32_t s_cnt[1024], s_warp[32];
    auto f2o = [](float f) {
        const int i = __float_as_int(f);
        return i >= 0 ? i : i ^ 0x7FFFFFFF;
    };
    auto o2f = [](int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7FFFFFFF); };
    float3 tb, bb;
    onb(p.nw, tb, bb);
    s_cnt[threadIdx.x] = 0u;
    if (threadIdx.x < 4) s_box[threadIdx.x] = threadIdx.x < 2 ? 0x7FFFFFFF : (int)0x80000000;
    __syncthreads();
    for (int i = threadIdx.x; i < p.n_s; i += blockDim.x) {
        const float3 x = f3(p.sensors[3 * i], p.sensors[3 * i + 1], p.sensors[3 * i + 2]);
        const int u = f2o(dot(x, tb)), v = f2o(dot(x, bb));
        atomicMin(&s_box[0], u);
        atomicMin(&s_box[1], v);
        atomicMax(&s_box[2], u);
        atomicMax(&s_box[3], v);
    }
    __syncthreads();
    const float lo_u = o2f(s_box[0]), lo_v = o2f(s_box[1]);
    const float ext = fmaxf(fmaxf(o2f(s_box[2]) - lo_u, o2f(s_box[3]) - lo_v), 1e-30f);
    int32_t *cell = order + p.n_s;
    for (int i = threadIdx.x; i < p.n_s; i += blockDim.x) {
        const float3 x = f3(p.sensors[3 * i], p.sensors[3 * i + 1], p.sensors[3 * i + 2]);
        const int cu = min(max((int)((dot(x, tb) - lo_u) / ext * 32.0f), 0), 31);
        const int cv = min(max((int)((dot(x, bb) - lo_v) / ext * 32.0f), 0), 31);
        uint32_t m = 0;
        for (int k = 0; k < 5; ++k) m |= ((uint32_t)(cu >> k & 1) << (2 * k)) | ((uint32_t)(cv >> k & 1) << (2 * k + 1));
        cell[i] = (int)m;
        atomicAdd(&s_cnt[m], 1u);
    }
    __syncthreads();
    // exclusive scan of the 1024 counts
    const uint32_t c = s_cnt[threadIdx.x];
    uint32_t x = c;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
        if (lane >= d) x += y;
    }
    if (lane == 31) s_warp[w] = x;
    __syncthreads();
    if (w == 0) {
        uint32_t t = s_warp[lane];
        for (int d = 1; d < 32; d <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, t, d);
            if (lane >= d) t += y;
        }
        s_warp[lane] = t;
    }
    __syncthreads();
    s_cnt[threadIdx.x] = x - c + (w > 0 ? s_warp[w - 1] : 0u);
    __syncthreads();
    for (int i = threadIdx.x; i < p.n_s; i += blockDim.x) order[atomicAdd(&s_cnt[cell[i]], 1u)] = i;
}

// exhaustive grid: a warp takes 32 sensors of a laser, one per lane, and a run of p.run of its hidden
// samples; the lanes' shadow rays of one step leave the same point y, the next step's a point near it.  The runs of
// the same sensors are consecutive items, so their film rows stay in L2 while they are added to.  Against CTAs that
// own 32 film rows: no barrier between tiles, the steady sums in registers, samples in the order of the surface (16x16
// x 32x32 pairs, 1024 samples: 16.2 -> 14.8 ms; 4x4 x 16x16 pairs, 256 samples, 16 CTAs before: 441 -> 252 us).
template <bool CNT>
__global__ void __launch_bounds__(256, MT_NLOS_PAIRS_MINB) k_nlos_pairs(const DevScene s, const NlosParams p) {
    uint32_t conns = 0, contribs = 0, rays = 0;
    TraceCnt tc{0, 0};
    const int lane = threadIdx.x & 31;
    const int runs = (p.spp + p.run - 1) / p.run, groups = (p.n_s + 31) / 32;
    const long long items = (long long)p.n_l * groups * runs;
    for (;;) {
        int claim = 0;
        if (lane == 0) claim = atomicAdd(p.tile_counter, 1);
        const long long item = __shfl_sync(0xffffffffu, claim, 0);
        if (item >= items) break;
        const long long lg = item / runs;
        const int l = (int)(lg / groups), j0 = (int)(item - lg * runs) * p.run, j1 = min(p.spp, j0 + p.run);
        const int at = (int)(lg - (long long)l * groups) * 32 + lane;
        if (at >= p.n_s) continue;
        const int si = p.order ? __ldg(&p.order[at]) : at;
        const float3 xs = f3(p.sensors[3 * si], p.sensors[3 * si + 1], p.sensors[3 * si + 2]);
        const long long row = (long long)l * p.n_s + si;
        float steady = 0.f;
        for (int j = j0; j < j1; ++j) {
            const float4 ya = __ldg(&p.ysamp[2 * ((size_t)l * p.spp + j)]), yb = __ldg(&p.ysamp[2 * ((size_t)l * p.spp + j) + 1]);
            conns++;
            float opl = 0.f;
            const float H = sensor_value<CNT>(s, p, ya, yb, xs, opl, tc, rays);
            if (H > 0.f) {
                contribs++;
                const float v = H * p.scale;
                nlos_splat(p, row, opl, v);
                steady += v;
            }
        }
        if (p.steady && steady != 0.f) atomicAdd(&p.steady[row], steady);
    }
    __syncwarp();
    add_counters(s, conns, contribs, rays, tc);
}

template <bool DUMP, bool CNT>
__global__ void __launch_bounds__(256) k_nlos(const DevScene s, const NlosParams p) {
    extern __shared__ float4 smem4[];
    float *hist = reinterpret_cast<float *>(smem4);
    float *steady_s = hist + (size_t)p.tile * p.D;
    __shared__ int s_tile;
    uint32_t conns = 0, contribs = 0, rays = 0;
    TraceCnt tc{0, 0};
    const bool exh = p.mode == MT_EXHAUSTIVE;
    const long long rows = exh ? (long long)p.n_l * p.n_s : p.n_l;
    const int tiles_per_laser = exh ? (p.n_s + p.tile - 1) / p.tile : 0;
    for (;;) {
        if (threadIdx.x == 0) s_tile = atomicAdd(p.tile_counter, 1);
        for (int i = threadIdx.x; i < p.tile * (p.D + 1); i += blockDim.x) hist[i] = 0.f;
        __syncthreads();
        const int tile = s_tile;
        if (tile >= p.n_tiles) break;
        // rows [row0, row0 + nrows) of the film; laser l for the exhaustive grid
        long long row0;
        int nrows, l = 0, s0 = 0;
        if (exh) {
            l = tile / tiles_per_laser;
            s0 = (tile - l * tiles_per_laser) * p.tile;
            nrows = min(p.tile, p.n_s - s0);
            row0 = (long long)l * p.n_s + s0;
        } else {
            row0 = (long long)tile * p.tile;
            nrows = (int)min((long long)p.tile, rows - row0);
        }
        const int work = nrows * p.spp;
        // the exhaustive grid goes sensor-fastest: the lanes of a warp take consecutive sensors of the
        // tile and share one hidden sample, so their shadow rays leave the same point y (262 -> 190 ms
        // at 2-row tiles, 130 ms at 32-row tiles for 16x16 lasers x 64x64 sensors x 1024 samples);
        // scan points go sample-fastest
        for (int j = threadIdx.x; j < work; j += blockDim.x) {
            const int r = exh ? j % nrows : j / p.spp;
            const int sj = exh ? j / nrows : j - r * p.spp;
            const uint32_t smp = p.sample_offset + (uint32_t)sj;
            conns++;
            float H = 0.f, opl = 0.f;
            int tri = -1;
            if (!exh) {
                const int li = (int)row0 + r;
                const float3 xl = f3(p.lasers[3 * li], p.lasers[3 * li + 1], p.lasers[3 * li + 2]);
                const HiddenSample h = sample_hidden<CNT>(s, p, li, smp, xl, tc, rays);
                tri = h.tri;
                if (h.partial > 0.f) {
                    H = confocal_value(p, h);
                    opl = 2.0f * h.d1;
                }
            } else {
                const int si = s0 + r;
                const float3 xs = f3(p.sensors[3 * si], p.sensors[3 * si + 1], p.sensors[3 * si + 2]);
                const size_t yi = (size_t)l * p.spp + sj;
                tri = DUMP ? p.ysamp_tri[yi] : -1;
                H = sensor_value<CNT>(s, p, p.ysamp[2 * yi], p.ysamp[2 * yi + 1], xs, opl, tc, rays);
            }
            if (H > 0.f) {
                contribs++;
                const float x = (opl - p.start) / p.width;
                const bool in = x >= 0.f && x < (float)p.T;
                const int bin = in ? (int)x : -1;
                const float v = H * p.scale;
                if (in) {
                    if (p.aggregate) {
                        if (bin < p.D) splat_add<1, true>(&hist[r * p.D + bin], &v);
                        else splat_add<1, true>(&p.film[(size_t)(row0 + r) * p.T + bin], &v);
                    } else {
                        if (bin < p.D) atomicAdd(&hist[r * p.D + bin], v);
                        else atomicAdd(&p.film[(size_t)(row0 + r) * p.T + bin], v);
                    }
                }
                atomicAdd(&steady_s[r], v);
                if (DUMP) {
                    const unsigned long long slot = atomicAdd(p.dump_count, 1ull);
                    if ((long long)slot < p.dump_cap) {
                        mt_contrib c;
                        c.pixel = (int32_t)(row0 + r);
                        c.sample = (int32_t)smp;
                        c.depth = 2;
                        c.kind = 2;
                        c.tri = tri;
                        c.bin = in ? bin : (int)floorf(x);
                        c.opl = opl;
                        c.c[0] = H;
                        c.c[1] = 0.f;
                        c.c[2] = 0.f;
                        p.dump[slot] = c;
                    }
                }
            }
        }
        __syncthreads();
        const bool acc = p.flags & MT_ACCUMULATE;
        if (p.D == p.T) {
            const size_t n = (size_t)nrows * p.T;
            float *dst = p.film + (size_t)row0 * p.T;
            if (((n | (size_t)row0 * p.T) & 3) == 0 && (((uintptr_t)p.film) & 15) == 0) {
                float4 *d4 = reinterpret_cast<float4 *>(dst);
                const float4 *s4 = reinterpret_cast<const float4 *>(hist);
                for (size_t i = threadIdx.x; i < n / 4; i += blockDim.x) {
                    float4 v = s4[i];
                    if (acc) {
                        const float4 o = d4[i];
                        v = make_float4(v.x + o.x, v.y + o.y, v.z + o.z, v.w + o.w);
                    }
                    d4[i] = v;
                }
            } else {
                for (size_t i = threadIdx.x; i < n; i += blockDim.x) dst[i] = acc ? dst[i] + hist[i] : hist[i];
            }
        } else {
            for (int i = threadIdx.x; i < nrows * p.D; i += blockDim.x) {
                const int r = i / p.D, b = i - r * p.D;
                float *d = p.film + (size_t)(row0 + r) * p.T + b;
                *d = acc ? *d + hist[i] : hist[i];
            }
        }
        if (p.steady)
            for (int i = threadIdx.x; i < nrows; i += blockDim.x)
                p.steady[row0 + i] = acc ? p.steady[row0 + i] + steady_s[i] : steady_s[i];
        __syncthreads();
    }
    add_counters(s, conns, contribs, rays, tc);
}

template <bool DUMP, bool CNT>
mt_status launch_nlos(const DevScene &s, const NlosParams &p, const LaunchCfg &cfg, cudaStream_t st) {
    if (p.mode == MT_EXHAUSTIVE) {
        const long long total = (long long)p.n_l * p.spp;
        const int grid = (int)std::min<long long>((total + 255) / 256, (long long)cfg.num_sms * 16);
        k_nlos_ysample<CNT><<<grid, 256, 0, st>>>(s, p);
        MT_CUDA_TRY(cudaGetLastError());
    }
    auto kern = k_nlos<DUMP, CNT>;
    MT_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cfg.smem_bytes));
    int per_sm = 0;
    MT_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, cfg.threads, cfg.smem_bytes));
    if (per_sm < 1) {
        mt::set_error("nlos kernel does not fit: %d threads, %zu bytes of shared memory", cfg.threads, cfg.smem_bytes);
        return MT_ERR_UNSUPPORTED;
    }
    if (cfg.ctas_per_sm > 0) per_sm = std::min(per_sm, cfg.ctas_per_sm);
    const int grid = std::max(1, std::min(p.n_tiles, per_sm * cfg.num_sms));
    kern<<<grid, cfg.threads, cfg.smem_bytes, st>>>(s, p);
    MT_CUDA_TRY(cudaGetLastError());
    return MT_OK;
}

// persistent grid of the default forms
template <class K>
mt_status launch_default(K kern, const DevScene &s, const NlosParams &p, const LaunchCfg &cfg, long long ctas,
                         cudaStream_t st) {
    int per_sm = 0;
    MT_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, cfg.threads, 0));
    if (cfg.ctas_per_sm > 0) per_sm = std::min(per_sm, cfg.ctas_per_sm);
    const int grid = (int)std::max<long long>(1, std::min<long long>(ctas, (long long)std::max(1, per_sm) * cfg.num_sms));
    kern<<<grid, cfg.threads, 0, st>>>(s, p);
    MT_CUDA_TRY(cudaGetLastError());
    return MT_OK;
}

template <bool CNT>
mt_status launch_scan(const DevScene &s, const NlosParams &p, const LaunchCfg &cfg, cudaStream_t st) {
    return launch_default(k_nlos_scan<CNT>, s, p, cfg, p.n_l, st);
}

template <bool CNT>
mt_status launch_pairs(const DevScene &s, const NlosParams &p, const LaunchCfg &cfg, cudaStream_t st) {
    if (p.spp >= MT_NLOS_ORDER_SPP) {
        const long long batches = (long long)p.n_l * ((p.spp + MT_NLOS_BATCH - 1) / MT_NLOS_BATCH);
        k_nlos_ysample_ordered<CNT><<<(int)std::min<long long>(batches, (long long)cfg.num_sms * 16), 256, 0, st>>>(s, p);
    } else {
        const long long total = (long long)p.n_l * p.spp;
        k_nlos_ysample<CNT><<<(int)std::min<long long>((total + 255) / 256, (long long)cfg.num_sms * 16), 256, 0, st>>>(
            s, p);
    }
    MT_CUDA_TRY(cudaGetLastError());
    if (p.order) {
        k_nlos_sensor_order<<<1, 1024, 0, st>>>(p, const_cast<int32_t *>(p.order));
        MT_CUDA_TRY(cudaGetLastError());
    }
    const long long items = (long long)p.n_l * ((p.n_s + 31) / 32) * ((p.spp + p.run - 1) / p.run);
    const int warps = cfg.threads / 32;
    return launch_default(k_nlos_pairs<CNT>, s, p, cfg, (items + warps - 1) / warps, st);
}

}  // namespace

mt_status mt_launch_nlos(const DevScene &s, const NlosParams &p, const LaunchCfg &cfg, bool dump, bool counters,
                         cudaStream_t st) {
    if (p.scan && !dump) return counters ? launch_scan<true>(s, p, cfg, st) : launch_scan<false>(s, p, cfg, st);
    if (p.run && !dump) return counters ? launch_pairs<true>(s, p, cfg, st) : launch_pairs<false>(s, p, cfg, st);
    if (dump) return counters ? launch_nlos<true, true>(s, p, cfg, st) : launch_nlos<true, false>(s, p, cfg, st);
    return counters ? launch_nlos<false, true>(s, p, cfg, st) : launch_nlos<false, false>(s, p, cfg, st);
}
