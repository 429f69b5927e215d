// mt_trace.cuh -- BVH traversal and ray/triangle intersection (device code).
//
// Visibility V and segment lengths of the path integral (arXiv 2510.25660,
// Sec. 3 Eqs. 3 and 8) come from these queries.
//
// Node layout (32 bytes = one L2 sector, fetched by one 256-bit load): one
// 32-bit word per child and axis holds that axis' lower plane (low half) and
// upper plane (high half):
//   a.x = child 0 x   a.y = child 0 y   a.z = child 0 z   a.w = child 1 x
//   b.x = child 1 y   b.y = child 1 z   b.z = child 0 reference   b.w = child 1 reference
// Planes are 16-bit fixed point in the scene box, rounded outward by two steps
// (plane = q_lo + q * q_scale), so boxes are conservative.  A reference with
// bit 31 clear is an internal node index; with bit 31 set it is a leaf of
// ((ref >> 29) & 3) + 1 triangles starting at (ref & 0x1FFFFFFF); 0xFFFFFFFF
// is an empty child.  Triangles are 48-byte records in leaf order, one float4
// row per axis: (v0, v1, v2 of that axis, original triangle index as int bits).
#pragma once
#include "mt_common.cuh"

#define MT_EMPTY_REF 0xFFFFFFFFu

// An empty child also has inverted planes (lower 65535, upper 0 on every axis),
// which the slab test rejects for either direction sign, so the traversal does
// not look at its reference.

struct RayT {
    float3 o, d;
    float3 sa, sb;   // slab: t = (2^23 + q) * sa + sb for a quantised plane q
    float3 inv;      // 1 / direction (zero components replaced by +-1e-20)
    uint32_t oct;    // bit k set: direction component k is negative
    uint32_t sel_n[3];  // byte-permute selector of the near plane per axis (far = near ^ 0x22)
    // watertight test (Woop, Benthin, Wald, JCGT 2013): rows of a triangle record holding its shear axes
    // kx = kz + 1 and ky = kz + 2 (mod 3) and its dominant axis kz, the origin in that axis order, the shear
    int kx, ky, kz;
    float3 ok;
    float Sx, Sy, Sz;
};

__device__ __forceinline__ float comp3(float3 v, int k) { return k == 0 ? v.x : (k == 1 ? v.y : v.z); }

__device__ __forceinline__ RayT make_ray(const DevScene &s, float3 o, float3 d) {
    RayT r;
    r.o = o;
    r.d = d;
    // zero direction components are replaced by +-1e-20 for the slab test only
    const float dx = fabsf(d.x) < 1e-20f ? copysignf(1e-20f, d.x) : d.x;
    const float dy = fabsf(d.y) < 1e-20f ? copysignf(1e-20f, d.y) : d.y;
    const float dz = fabsf(d.z) < 1e-20f ? copysignf(1e-20f, d.z) : d.z;
    const float ix = 1.0f / dx, iy = 1.0f / dy, iz = 1.0f / dz;
    r.inv = f3(ix, iy, iz);
    r.oct = (dx < 0.0f ? 1u : 0u) | (dy < 0.0f ? 2u : 0u) | (dz < 0.0f ? 4u : 0u);
    r.sa = f3(s.q_scale.x * ix, s.q_scale.y * iy, s.q_scale.z * iz);
    // the 2^23 offset of the exponent trick below is folded into sb; the two
    // 2^23 * sa terms cancel exactly inside the FMA, leaving one rounding of sb
    // (at most half a quantisation step, inside the two-step padding)
    r.sb = f3((s.q_lo.x - o.x) * ix - 8388608.0f * r.sa.x, (s.q_lo.y - o.y) * iy - 8388608.0f * r.sa.y,
              (s.q_lo.z - o.z) * iz - 8388608.0f * r.sa.z);
    const float dd[3] = {dx, dy, dz};
#pragma unroll
    for (int k = 0; k < 3; ++k) r.sel_n[k] = dd[k] >= 0.0f ? 0x7610u : 0x7632u;  // low half = lower plane
    const float ax = fabsf(d.x), ay = fabsf(d.y), az = fabsf(d.z);
    // the original test swaps kx and ky for a negative dominant component to keep the winding; the swap
    // negates every edge function, the determinant and T exactly and leaves t = T / det as it is, so it
    // is left out and the axes are always a rotation
    const int kz = (ax >= ay && ax >= az) ? 0 : (ay >= az ? 1 : 2);
    const int kx = kz == 2 ? 0 : kz + 1;
    const int ky = kx == 2 ? 0 : kx + 1;
    r.kx = kx;
    r.ky = ky;
    r.kz = kz;
    r.ok = f3(comp3(o, kx), comp3(o, ky), comp3(o, kz));
    const float dk = comp3(d, kz);
    r.Sx = comp3(d, kx) / dk;
    r.Sy = comp3(d, ky) / dk;
    r.Sz = 1.0f / dk;
    return r;
}

// 16-bit fixed point q -> the float 2^23 + q (exact) by writing q under the
// exponent of 2^23 with one byte permute
__device__ __forceinline__ float q_plane(uint32_t word, uint32_t sel) {
    return __int_as_float(__byte_perm(word, 0x4B000000u, sel));
}

// One binary node (32 bytes, 32-byte aligned) in one 256-bit read-only load
// (sm_100-class); MT_NODE_V8 = 0: two 128-bit loads.
#ifndef MT_NODE_V8
#define MT_NODE_V8 1
#endif
__device__ __forceinline__ void ldg_node(const uint4 *p, uint4 &a, uint4 &b) {
#if MT_NODE_V8 && !MT_L2_KEEP_BVH
    asm("ld.global.nc.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
        : "l"(p));
#else
    a = ldg_keep(p);
    b = ldg_keep(p + 1);
#endif
}

// Packed arithmetic of sm_100-class GPUs: fma.rn.f32x2 (two independent FMAs,
// each rounded once, in one instruction) and three-input min/max.  Each lane
// gets the same values as the scalar forms, so switching MT_SLAB_PACKED off
// (scalar FMAs and two-input min/max) changes no result, only the count of
// issued instructions per node.
#ifndef MT_SLAB_PACKED
#define MT_SLAB_PACKED 1
#endif

__device__ __forceinline__ void fma_x2(float ax, float ay, float bx, float by, float cx, float cy, float &dx,
                                       float &dy) {
#if MT_SLAB_PACKED
    asm("{\n\t.reg .b64 a, b, c, d;\n\t"
        "mov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
        "fma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
        : "=f"(dx), "=f"(dy)
        : "f"(ax), "f"(ay), "f"(bx), "f"(by), "f"(cx), "f"(cy));
#else
    dx = fmaf(ax, bx, cx);
    dy = fmaf(ay, by, cy);
#endif
}

__device__ __forceinline__ float max3f(float a, float b, float c) {
#if MT_SLAB_PACKED
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
#else
    return fmaxf(fmaxf(a, b), c);
#endif
}

__device__ __forceinline__ float min3f(float a, float b, float c) {
#if MT_SLAB_PACKED
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
#else
    return fminf(fminf(a, b), c);
#endif
}

// entry / exit distance of one child box; wx, wy, wz are its three axis words
__device__ __forceinline__ void slab(const RayT &r, uint32_t wx, uint32_t wy, uint32_t wz, float tmax, float &tn,
                                     float &tf) {
    float nx, ny, fx, fy;
    fma_x2(q_plane(wx, r.sel_n[0]), q_plane(wy, r.sel_n[1]), r.sa.x, r.sa.y, r.sb.x, r.sb.y, nx, ny);
    fma_x2(q_plane(wx, r.sel_n[0] ^ 0x22u), q_plane(wy, r.sel_n[1] ^ 0x22u), r.sa.x, r.sa.y, r.sb.x, r.sb.y, fx,
           fy);
    const float nz = fmaf(q_plane(wz, r.sel_n[2]), r.sa.z, r.sb.z);
    const float fz = fmaf(q_plane(wz, r.sel_n[2] ^ 0x22u), r.sa.z, r.sb.z);
    tn = fmaxf(max3f(nx, ny, nz), 0.0f);
    tf = fminf(min3f(fx, fy, fz), tmax);
}

// entry / exit distances of both child boxes of a binary node (a, b = its two
// 128-bit halves)
__device__ __forceinline__ void slab2(const RayT &r, const uint4 &a, const uint4 &b, float tmax, float &tn0,
                                      float &tf0, float &tn1, float &tf1) {
    slab(r, a.x, a.y, a.z, tmax, tn0, tf0);
    slab(r, a.w, b.x, b.y, tmax, tn1, tf1);
}

// vertices of leaf-order triangle k (for shading and sampling)
__device__ __forceinline__ void tri_vertices(const DevScene &s, int k, float3 &v0, float3 &v1, float3 &v2) {
    const float4 *T = s.tris + 3 * (size_t)k;
    const float4 X = ldg_keep(T), Y = ldg_keep(T + 1), Z = ldg_keep(T + 2);
    v0 = f3(X.x, Y.x, Z.x);
    v1 = f3(X.y, Y.y, Z.y);
    v2 = f3(X.z, Y.z, Z.z);
}
__device__ __forceinline__ int tri_id(const DevScene &s, int k) {
    return __float_as_int(__ldg(&s.tris[3 * (size_t)k].w));
}

// Watertight ray/triangle test of the record at T.  The edge functions are
// evaluated without contraction so that a shared edge gives exactly opposite
// values in its two triangles (no gaps).  Returns true with t = T/det when the
// ray crosses the triangle (edges inclusive) at t > 0; id = original index.
// The axis permutation is in the choice of the rows that are loaded, so the
// test itself has no selects (with one float4 per vertex it took 18 selects
// and 6 comparisons of the axis numbers per triangle).  The traversal is bound
// by instruction issue at about nine active lanes per instruction, and most
// warp steps hold a lane in a leaf, so the shorter test shows in every render:
// 76.8 -> 70.1 ms for the 512x512x256-spp frame of the 1.16M-triangle scene,
// 4.59 -> 4.22 ms for a 135x241x19-spp frame of the 97k-triangle one.
__device__ __forceinline__ bool tri_hit(const RayT &r, const float4 *T, float &t, int &id) {
    const float4 X = ldg_keep(T + r.kx), Y = ldg_keep(T + r.ky), Z = ldg_keep(T + r.kz);
    id = __float_as_int(Z.w);
    const float Akz = Z.x - r.ok.z, Bkz = Z.y - r.ok.z, Ckz = Z.z - r.ok.z;
    const float Ax = (X.x - r.ok.x) - r.Sx * Akz, Ay = (Y.x - r.ok.y) - r.Sy * Akz;
    const float Bx = (X.y - r.ok.x) - r.Sx * Bkz, By = (Y.y - r.ok.y) - r.Sy * Bkz;
    const float Cx = (X.z - r.ok.x) - r.Sx * Ckz, Cy = (Y.z - r.ok.y) - r.Sy * Ckz;
    const float U = __fsub_rn(__fmul_rn(Cx, By), __fmul_rn(Cy, Bx));
    const float V = __fsub_rn(__fmul_rn(Ax, Cy), __fmul_rn(Ay, Cx));
    const float W = __fsub_rn(__fmul_rn(Bx, Ay), __fmul_rn(By, Ax));
    // edge functions of both signs: outside
    if (min3f(U, V, W) < 0.f && max3f(U, V, W) > 0.f) return false;
    const float det = U + V + W;
    if (det == 0.f) return false;
    // contraction spelled out, so that every kernel and trace_flat round the same way
    const float Tn = fmaf(W, r.Sz * Ckz, fmaf(U, r.Sz * Akz, V * (r.Sz * Bkz)));
    if (det > 0.f ? Tn <= 0.f : Tn >= 0.f) return false;
    t = Tn / det;
    return true;
}

struct TraceCnt {
    uint32_t nodes, tris;  // bytes of BVH nodes fetched, triangle records tested
};

// A leaf's triangles are tested one per iteration of the traversal loop (the
// leaf reference advances to the next triangle: first + 1, count - 1), so that
// in a warp whose lanes meet leaves at different steps the diverging leaf work
// of one step is one triangle test instead of up to four, while the other
// lanes go on with their nodes.  Measured on the 1.16M-triangle scene (fused
// traversal pass of the 512x512x256-spp render): 67.36 ms with the leaf's
// triangles in an inner loop, 65.35 ms so.
#define MT_LEAF_MORE 0x60000000u                // count - 1 field of a leaf reference
#define MT_LEAF_NEXT (1u - 0x20000000u)         // first + 1, count - 1 (mod 2^32)

// The binary traversals push without looking at the stack's size.  A ray's
// stack holds at most one entry per internal node on the way from the root to
// the node it visits, so never more than the depth of the tree, and a scene
// whose tree is deeper than MT_STACK - 2 is refused when it is built (scene
// creation validates every child reference too).  With the check, and the
// atomic on the error word behind it, the compiler kept the lanes of the
// descending branches apart from those that pop: 512x512x256-spp frame of the
// 1.16M-triangle scene 70.6 -> 64.6 ms, exhaustive NLOS scan 32.1 -> 16.1 ms,
// confocal scan 2.37 -> 1.76 ms, Cornell box render 369 -> 197 us.

// Closest hit with t in (0, tmax); ties in t go to the smaller original index.
// Returns the leaf-order triangle index (or -1) and writes t and the original index.
template <bool CNT>
__device__ __forceinline__ int trace_closest(const DevScene &s, const RayT &r, float tmax, float &t_out,
                                             int &orig_out, TraceCnt &cnt) {
    float tbest = tmax;
    int best_k = -1;
    uint2 st[MT_STACK];  // (reference, entry distance bits)
    int sp = 0;
    uint32_t ref = 0;
    for (;;) {
        if (!(ref & 0x80000000u)) {
            uint4 a, b;
            ldg_node(&s.nodes[2 * ref], a, b);
            if (CNT) cnt.nodes += 32;
            float tn0, tf0, tn1, tf1;
            slab2(r, a, b, tbest, tn0, tf0, tn1, tf1);
            const bool h0 = tn0 <= tf0;
            const bool h1 = tn1 <= tf1;
            if (h0 && h1) {
                const bool f0 = tn0 <= tn1;
                st[sp++] = make_uint2(f0 ? b.w : b.z, __float_as_uint(f0 ? tn1 : tn0));
                ref = f0 ? b.z : b.w;
                continue;
            }
            if (h0) { ref = b.z; continue; }
            if (h1) { ref = b.w; continue; }
        } else {
            // one triangle of the leaf per iteration; the rest stay in `ref`
            const int k = (int)(ref & 0x1FFFFFFFu);
            if (CNT) cnt.tris++;
            float t;
            int id;
            if (tri_hit(r, s.tris + 3 * (size_t)k, t, id) && t < tmax) {
                // the best hit's original index is read back only for a tie
                if (t < tbest || (t == tbest && id < tri_id(s, best_k))) {
                    tbest = t;
                    best_k = k;
                }
            }
            if (ref & MT_LEAF_MORE) {
                ref += MT_LEAF_NEXT;
                continue;
            }
        }
        // pop the next entry whose entry distance does not exceed the best hit
        for (;;) {
            if (sp == 0) {
                t_out = tbest;
                orig_out = best_k >= 0 ? tri_id(s, best_k) : 0x7fffffff;
                return best_k;
            }
            --sp;
            const uint2 e = st[sp];
            if (__uint_as_float(e.y) <= tbest) {
                ref = e.x;
                break;
            }
        }
    }
}

// Any hit with t in (0, tmax).
template <bool CNT>
__device__ __forceinline__ bool trace_any(const DevScene &s, const RayT &r, float tmax, TraceCnt &cnt) {
    uint32_t st_ref[MT_STACK];
    int sp = 0;
    uint32_t ref = 0;
    for (;;) {
        if (!(ref & 0x80000000u)) {
            uint4 a, b;
            ldg_node(&s.nodes[2 * ref], a, b);
            if (CNT) cnt.nodes += 32;
            float tn0, tf0, tn1, tf1;
            slab2(r, a, b, tmax, tn0, tf0, tn1, tf1);
            const bool h0 = tn0 <= tf0;
            const bool h1 = tn1 <= tf1;
            if (h0 && h1) {
                const bool f0 = tn0 <= tn1;
                st_ref[sp++] = f0 ? b.w : b.z;
                ref = f0 ? b.z : b.w;
                continue;
            }
            if (h0) { ref = b.z; continue; }
            if (h1) { ref = b.w; continue; }
        } else {
            const int k = (int)(ref & 0x1FFFFFFFu);
            if (CNT) cnt.tris++;
            float t;
            int id;
            if (tri_hit(r, s.tris + 3 * (size_t)k, t, id) && t < tmax) return true;
            if (ref & MT_LEAF_MORE) {
                ref += MT_LEAF_NEXT;
                continue;
            }
        }
        if (sp == 0) return false;
        --sp;
        ref = st_ref[sp];
    }
}

// ---------------------------------------------------------------------------
// Scenes of a few triangles (the rule is where s.flat is built): every triangle in
// turn instead of the tree, two per step in packed arithmetic.  All lanes of a warp do the same
// work, where in the tree of the 36-triangle box a lane in nine instructions of
// ten waits for another's node or leaf; the steps are independent, so few warps
// hide their latency.  The hit is the smallest (t, original index) all the same,
// from the same operations in the same order as tri_hit.  A ray almost in the
// plane of a triangle can pass the edge tests by rounding far from it; the tree
// never tests such a triangle, because the ray misses its leaf's box.  So the
// hit found is checked against the box of its leaf, and a ray that fails goes
// through the tree (a hit that passes is the tree's own: its ancestors' boxes
// contain the leaf's, and no triangle is nearer).
// Records (s.flat, leaf order, built at scene creation): per pair of triangles
// and axis a 32-byte row (v0, v0', v1, v1', v2, v2', index, index'); s.flat_box:
// per triangle the three plane words of its leaf.
// ---------------------------------------------------------------------------
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk(float a, float b) {
    f32x2 d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
    return d;
}
__device__ __forceinline__ void upk(f32x2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
    f32x2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
    f32x2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}

struct FlatRow {
    f32x2 v0, v1, v2;
    int id0, id1;
};
__device__ __forceinline__ FlatRow ld_flat(const float4 *p) {
    FlatRow r;
    float a, b, c, d, e, f, g, h;
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(a), "=f"(b), "=f"(c), "=f"(d), "=f"(e), "=f"(f), "=f"(g), "=f"(h)
        : "l"(p));
    r.v0 = pk(a, b);
    r.v1 = pk(c, d);
    r.v2 = pk(e, f);
    r.id0 = __float_as_int(g);
    r.id1 = __float_as_int(h);
    return r;
}

// the tests of tri_hit after the edge functions
__device__ __forceinline__ bool flat_hit(float U, float V, float W, float det, float Tn, float &t) {
    if (min3f(U, V, W) < 0.f && max3f(U, V, W) > 0.f) return false;
    if (det == 0.f) return false;
    if (det > 0.f ? Tn <= 0.f : Tn >= 0.f) return false;
    t = Tn / det;
    return true;
}

// leaf-order index of the closest hit or, ANY, of any hit; -1: none
template <bool ANY>
__device__ __forceinline__ int trace_flat(const DevScene &s, const RayT &r, float tmax, float &t_out, int &orig_out) {
    const float4 *px = s.flat + 2 * r.kx, *py = s.flat + 2 * r.ky, *pz = s.flat + 2 * r.kz;
    const f32x2 ox = pk(r.ok.x, r.ok.x), oy = pk(r.ok.y, r.ok.y), oz = pk(r.ok.z, r.ok.z);
    const f32x2 m1 = pk(-1.0f, -1.0f), nSx = pk(-r.Sx, -r.Sx), nSy = pk(-r.Sy, -r.Sy), Sz = pk(r.Sz, r.Sz);
    float tbest = tmax;
    int best_k = -1, best_id = 0x7fffffff;
    const int n = s.n_tris;
    for (int k = 0; k < n; k += 2, px += 6, py += 6, pz += 6) {
        const FlatRow X = ld_flat(px), Y = ld_flat(py), Z = ld_flat(pz);
        const f32x2 Akz = sub2(Z.v0, oz), Bkz = sub2(Z.v1, oz), Ckz = sub2(Z.v2, oz);
        const f32x2 Ax = fma2(nSx, Akz, sub2(X.v0, ox)), Ay = fma2(nSy, Akz, sub2(Y.v0, oy));
        const f32x2 Bx = fma2(nSx, Bkz, sub2(X.v1, ox)), By = fma2(nSy, Bkz, sub2(Y.v1, oy));
        const f32x2 Cx = fma2(nSx, Ckz, sub2(X.v2, ox)), Cy = fma2(nSy, Ckz, sub2(Y.v2, oy));
        // products and difference each rounded, as in tri_hit: a packed subtraction of packed products would be
        // contracted, an FMA with -1 is not
        const f32x2 U = fma2(mul2(Cy, Bx), m1, mul2(Cx, By));
        const f32x2 V = fma2(mul2(Ay, Cx), m1, mul2(Ax, Cy));
        const f32x2 W = fma2(mul2(By, Ax), m1, mul2(Bx, Ay));
        const f32x2 det = add2(add2(U, V), W);
        const f32x2 T = fma2(W, mul2(Sz, Ckz), fma2(U, mul2(Sz, Akz), mul2(V, mul2(Sz, Bkz))));
        float u[2], v[2], w[2], d[2], tn[2];
        upk(U, u[0], u[1]);
        upk(V, v[0], v[1]);
        upk(W, w[0], w[1]);
        upk(det, d[0], d[1]);
        upk(T, tn[0], tn[1]);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            float t;
            if (flat_hit(u[j], v[j], w[j], d[j], tn[j], t) && t < tmax) {
                if (ANY) return k + j;
                const int id = j ? Z.id1 : Z.id0;
                if (t < tbest || (t == tbest && id < best_id)) {
                    tbest = t;
                    best_k = k + j;
                    best_id = id;
                }
            }
        }
    }
    t_out = tbest;
    orig_out = best_id;
    return best_k;
}

// whether the ray enters the box of triangle k's leaf up to tmax, as the tree tests it
__device__ __forceinline__ bool flat_in_box(const DevScene &s, const RayT &r, int k, float tmax) {
    const uint4 w = __ldg(&s.flat_box[k]);
    float tn, tf;
    slab(r, w.x, w.y, w.z, tmax, tn, tf);
    return tn <= tf;
}

// the scene's own way: all triangles (FLAT, scenes that have s.flat) or the binary tree
template <bool CNT, bool FLAT>
__device__ __forceinline__ int scene_closest(const DevScene &s, const RayT &r, float tmax, float &t_out, int &orig_out,
                                             TraceCnt &cnt) {
    if (FLAT) {
        const int k = trace_flat<false>(s, r, tmax, t_out, orig_out);
        if (k < 0 || flat_in_box(s, r, k, t_out)) return k;
    }
    return trace_closest<CNT>(s, r, tmax, t_out, orig_out, cnt);
}
template <bool CNT, bool FLAT>
__device__ __forceinline__ bool scene_any(const DevScene &s, const RayT &r, float tmax, TraceCnt &cnt) {
    if (FLAT) {
        float t;
        int id;
        const int k = trace_flat<true>(s, r, tmax, t, id);
        if (k < 0) return false;
        if (flat_in_box(s, r, k, tmax)) return true;
    }
    return trace_any<CNT>(s, r, tmax, cnt);
}

// ---------------------------------------------------------------------------
// Traversal as a per-lane state machine, one node or leaf per call, for
// kernels whose lanes fetch a new ray as soon as their current one is done
// (persistent threads with dynamic ray fetch, Aila & Laine, HPG 2009).
// ---------------------------------------------------------------------------
struct TravState {
    uint32_t ref;
    int sp;
    float tbest;
    int best_k, best_id;
};

__device__ __forceinline__ void trav_init(TravState &ts, float tmax) {
    ts.ref = 0;
    ts.sp = 0;
    ts.tbest = tmax;
    ts.best_k = -1;
    ts.best_id = 0x7fffffff;
}

// Advance by one node or one leaf; returns true when the traversal is over
// (for ANY: also when a hit is found, signalled by best_k = 1).
template <bool ANY, bool CNT>
__device__ __forceinline__ bool trav_step(const DevScene &s, const RayT &r, float tmax, TravState &ts, uint2 *st,
                                          TraceCnt &cnt) {
    if (!(ts.ref & 0x80000000u)) {
        uint4 a, b;
        ldg_node(&s.nodes[2 * ts.ref], a, b);
        if (CNT) cnt.nodes += 32;
        float tn0, tf0, tn1, tf1;
        slab(r, a.x, a.y, a.z, ts.tbest, tn0, tf0);
        slab(r, a.w, b.x, b.y, ts.tbest, tn1, tf1);
        const bool h0 = tn0 <= tf0;
        const bool h1 = tn1 <= tf1;
        if (h0 && h1) {
            const bool f0 = tn0 <= tn1;
            st[ts.sp++] = make_uint2(f0 ? b.w : b.z, __float_as_uint(f0 ? tn1 : tn0));
            ts.ref = f0 ? b.z : b.w;
            return false;
        }
        if (h0) {
            ts.ref = b.z;
            return false;
        }
        if (h1) {
            ts.ref = b.w;
            return false;
        }
    } else {
        const int first = (int)(ts.ref & 0x1FFFFFFFu), n = (int)((ts.ref >> 29) & 3u) + 1;
        for (int k = first; k < first + n; ++k) {
            if (CNT) cnt.tris++;
            float t;
            int id;
            if (tri_hit(r, s.tris + 3 * (size_t)k, t, id) && t < tmax) {
                if (ANY) {
                    ts.best_k = 1;
                    return true;
                }
                if (t < ts.tbest || (t == ts.tbest && id < ts.best_id)) {
                    ts.tbest = t;
                    ts.best_k = k;
                    ts.best_id = id;
                }
            }
        }
    }
    while (ts.sp > 0) {
        --ts.sp;
        const uint2 e = st[ts.sp];
        if (ANY || __uint_as_float(e.y) <= ts.tbest) {
            ts.ref = e.x;
            return false;
        }
    }
    return true;
}

// ---------------------------------------------------------------------------
// 8-wide BVH with compressed child boxes (after Ylitie, Karras and Laine,
// "Efficient incoherent ray traversal on GPUs through compressed wide BVHs",
// HPG 2017; the node layout below is this library's own).
//
// Node = 80 bytes = five uint4:
//   w0.xyz  frame origin p (float), w0.w = ex | ey << 8 | ez << 16 | imask << 24
//           (biased float exponents of the per-axis step 2^e; imask bit i set:
//           child slot i is an internal node)
//   w1.x    index of the first internal child; the internal child in slot i
//           is w1.x + popc(imask & ((1 << i) - 1))
//   w1.y    first triangle of this node's leaf children
//   w1.z/w  one meta byte per slot (slots 0-3 / 4-7): a leaf child has
//           0x80 | (count - 1) << 5 | offset, triangles w1.y + offset ...
//   w2.xy qlo_x[8]  w2.zw qlo_y[8]  w3.xy qlo_z[8]  w3.zw qhi_x[8]
//   w4.xy qhi_y[8]  w4.zw qhi_z[8]   (one byte per slot, little-endian)
// A plane is p + q * 2^e, rounded outward by two steps; an empty slot has
// lower planes 255 and upper planes 0 and is never hit.  Slot bit k of a child
// says it lies on the upper side of the node along axis k, so visiting slots
// in increasing order of slot ^ oct(ray) is roughly front to back.
// ---------------------------------------------------------------------------
#define MT_WIDE_WORDS 5

// reorder the bits of an 8-bit mask so that bit k holds bit (k ^ m)
__device__ __forceinline__ uint32_t perm_xor8(uint32_t x, uint32_t m) {
    if (m & 1u) x = ((x & 0x55u) << 1) | ((x >> 1) & 0x55u);
    if (m & 2u) x = ((x & 0x33u) << 2) | ((x >> 2) & 0x33u);
    if (m & 4u) x = ((x & 0x0Fu) << 4) | ((x >> 4) & 0x0Fu);
    return x;
}

// byte i of the 8-byte pair (lo, hi) as the float 2^23 + q
__device__ __forceinline__ float q8(uint32_t lo, uint32_t hi, int i) {
    return __int_as_float(__byte_perm(i < 4 ? lo : hi, 0x4B000000u, 0x7440u | (uint32_t)(i & 3)));
}

// Hit mask of the eight child boxes of node w0..w4 against (0, tmax].
__device__ __forceinline__ uint32_t wide_hits(const RayT &r, const uint4 &w0, const uint4 &w2, const uint4 &w3,
                                              const uint4 &w4, float tmax) {
    // per-axis frame: t = (2^23 + q) * a + b with the 2^23 offset folded into b
    const float ax = __int_as_float((int)((w0.w & 0xFFu) << 23)) * r.inv.x;
    const float ay = __int_as_float((int)(((w0.w >> 8) & 0xFFu) << 23)) * r.inv.y;
    const float az = __int_as_float((int)(((w0.w >> 16) & 0xFFu) << 23)) * r.inv.z;
    const float bx = fmaf(-8388608.0f, ax, (__uint_as_float(w0.x) - r.o.x) * r.inv.x);
    const float by = fmaf(-8388608.0f, ay, (__uint_as_float(w0.y) - r.o.y) * r.inv.y);
    const float bz = fmaf(-8388608.0f, az, (__uint_as_float(w0.z) - r.o.z) * r.inv.z);
    // near planes: the lower ones for a positive direction component
    const bool nx = r.oct & 1u, ny = r.oct & 2u, nz = r.oct & 4u;
    const uint32_t nx0 = nx ? w3.z : w2.x, nx1 = nx ? w3.w : w2.y, fx0 = nx ? w2.x : w3.z, fx1 = nx ? w2.y : w3.w;
    const uint32_t ny0 = ny ? w4.x : w2.z, ny1 = ny ? w4.y : w2.w, fy0 = ny ? w2.z : w4.x, fy1 = ny ? w2.w : w4.y;
    const uint32_t nz0 = nz ? w4.z : w3.x, nz1 = nz ? w4.w : w3.y, fz0 = nz ? w3.x : w4.z, fz1 = nz ? w3.y : w4.w;
    uint32_t hits = 0;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const float tnx = fmaf(q8(nx0, nx1, i), ax, bx), tfx = fmaf(q8(fx0, fx1, i), ax, bx);
        const float tny = fmaf(q8(ny0, ny1, i), ay, by), tfy = fmaf(q8(fy0, fy1, i), ay, by);
        const float tnz = fmaf(q8(nz0, nz1, i), az, bz), tfz = fmaf(q8(fz0, fz1, i), az, bz);
        const float tn = fmaxf(fmaxf(tnx, tny), fmaxf(tnz, 0.0f));
        const float tf = fminf(fminf(tfx, tfy), fminf(tfz, tmax));
        hits |= (tn <= tf ? 1u : 0u) << i;
    }
    return hits;
}

// Closest hit (ANY = false: returns the triangle index or -1, writes t and the
// original index; ties in t go to the smaller original index) or any hit
// (ANY = true: returns 1 on a hit, else -1) with t in (0, tmax).
template <bool ANY, bool CNT>
__device__ __forceinline__ int trace_wide(const DevScene &s, const RayT &r, float tmax, float &t_out, int &orig_out,
                                          TraceCnt &cnt) {
    float tbest = tmax;
    int best_k = -1, best_id = 0x7fffffff;
    uint2 st[MT_STACK];  // (first internal child, imask << 8 | remaining visit-order mask)
    int sp = 0;
    uint32_t node = 0;
    for (;;) {
        const uint4 *np = s.wnodes + MT_WIDE_WORDS * (size_t)node;
        const uint4 w0 = ldg_keep(np), w1 = ldg_keep(np + 1), w2 = ldg_keep(np + 2), w3 = ldg_keep(np + 3), w4 = ldg_keep(np + 4);
        if (CNT) cnt.nodes += 80;
        const uint32_t hits = wide_hits(r, w0, w2, w3, w4, tbest);
        const uint32_t imask = w0.w >> 24;
        uint32_t leaves = hits & ~imask;
        while (leaves) {
            const int slot = __ffs(leaves) - 1;
            leaves &= leaves - 1u;
            const uint32_t meta = ((slot < 4 ? w1.z : w1.w) >> (8 * (slot & 3))) & 0xFFu;
            const int first = (int)w1.y + (int)(meta & 31u), last = first + (int)((meta >> 5) & 3u);
            for (int k = first; k <= last; ++k) {
                if (CNT) cnt.tris++;
                float t;
                int id;
                if (tri_hit(r, s.tris + 3 * (size_t)k, t, id) && t < tmax) {
                    if (ANY) return 1;
                    if (t < tbest || (t == tbest && id < best_id)) {
                        tbest = t;
                        best_k = k;
                        best_id = id;
                    }
                }
            }
        }
        uint32_t order = perm_xor8(hits & imask, r.oct);
        uint32_t base = w1.x, im = imask;
        if (!order) {
            // pop the next group that still has children to visit
            if (sp == 0) break;
            const uint2 g = st[sp - 1];
            base = g.x;
            im = g.y >> 8;
            order = g.y & 0xFFu;
            --sp;
        }
        const int k = __ffs(order) - 1;
        order &= order - 1u;
        const uint32_t slot = (uint32_t)k ^ r.oct;
        node = base + __popc(im & ((1u << slot) - 1u));
        if (order) {
            if (sp < MT_STACK) {
                st[sp] = make_uint2(base, (im << 8) | order);
                ++sp;
            } else {
                raise_err(s, MT_EFLAG_STACK);
            }
        }
    }
    t_out = tbest;
    orig_out = best_id;
    return best_k;
}
