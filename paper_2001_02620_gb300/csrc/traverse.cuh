// Device-side traversal of the two-level quad BVH (qrt_layout.h).
//
// Top level: four-wide TLAS over instance world boxes.  At a TLAS leaf the ray
// is re-centred at t_e, where it passes closest to the object origin (never
// before tmin), formed exactly with error-free FP32 transformations, and moved
// into the instance's object space (the direction is not renormalised, so t
// is shared by both levels); the object's BLAS is traversed on the same stack
// with a parameter s = t - t_e.  When the stack drains back to the level where
// the instance was entered, the world ray is restored.  Leaves of a BLAS hold
// up to 8 quads stored contiguously.
//
// Precision design.  Box tests are made conservative by widening every
// dequantised box by twice delta, an absolute bound on the position error of the
// FP32 ray in the current space (2^-20 (|o| + R) at the top level, where the
// world ray is exact; 2^-22 (kappa + 2) (|o''| + R) in object space, where o''
// is the re-centred origin, R the object's radius and kappa the condition
// number of the transform), so a node is never culled
// that the exact ray enters.  The quad test is the watertight test of Woop,
// Benthin and Wald (JCGT 2013) applied to both triangles of the quad with the
// diagonal v0-v2 shared; an edge function within the same error bound of zero,
// or a hit distance within its error bound of either end of the interval,
// makes the decision uncertain, and only then the quad is re-tested in FP64
// from the world ray and the FP64 transform (later, together with other lanes'
// quads: Traversal::resolve); two hits whose FP32 distances
// lie within their error bounds of each other are ordered by FP64 distances.
// Hit/miss decisions and the closest-hit choice therefore agree with exact
// arithmetic on the given FP32 ray except when a hit lies within FP64
// rounding of an edge or of another hit.
//
// Execution.  Persistent kernels run persistent_trace: each lane of a warp
// holds one ray; the warp tests inner nodes together, enters instances in
// groups, then lets every other lane enter its instance or test one leaf;
// finished lanes take the next ray at once (claimed for the warp, see there).
// What bounds it is the issue slots (60 to 70 % busy at 13 to 16 active lanes
// of 32; some 410 warp instructions per node step, all phases counted) and,
// behind them, each ray's chain of dependent node loads, hidden by resident
// warps.  So the registers hold what a node test reads and shared memory the
// rest of a ray and its stack: 64 registers (32 warps an SM) with few spills
// (bytes stored a thread: 16 for the renderer's closest-hit rays, 64 with
// textures, 4 for its any-hit rays, 24 for any-hit queries; none for
// closest-hit queries, at 72 registers).  Left to the compiler, the state
// spilled 476 bytes a thread at 48 registers, the 64-entry stacks lay in local
// memory, a node test sorted its children and the FP64 re-test sat in the leaf
// loop.  That against this on one GB300, ms: 2 M diffuse bounces on the mid
// scene 5.59 -> 2.82, 1.5 M sun rays 1.63 -> 0.81, 1 M rays of ambient
// occlusion on the island (0.40 re-tests a ray) 1.94 -> 0.80, the mid frame
// 18.0 -> 10.5, the island frame 34.5 -> 20.4.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "qrt_layout.h"

namespace qrt {

constexpr float kInfF = __builtin_huge_valf();

struct Hit {
    float t;
    uint32_t inst, prim;
    float u, v;
    uint32_t slot;  // global quad slot of the hit (for shading)
};

// A world-space ray (origin, direction).
struct WRay {
    float ox, oy, oz, dx, dy, dz;
};

// Ray in the current space: what a node test reads, in the two quadruples in
// which the world-space form also lies in shared memory (Traversal), so that
// one 128-bit load each restores it in place.
struct RaySetup {
    float4 o;    // origin; w: 2 delta, delta the bound on its position error
    float4 inv;  // reciprocal direction, |d| clamped away from 0; w: near end of the interval
};

// Watertight shear of the current-space ray in affine form,
// X = V . rx - cx, Y = V . ry - cy, Z = V . rz - cz.  Built at the start of
// each leaf rather than kept for the whole ray: it is needed only there, and
// twelve fewer live registers per ray buy resident warps.
struct Shear {
    float rx0, rx1, rx2, cx;
    float ry0, ry1, ry2, cy;
    float rz0, rz1, rz2, cz;
    float eps_t;  // bound on the error of an FP32 hit distance (t units)
};

__device__ __forceinline__ float clamp_dir(float d) {
    return fabsf(d) > 1e-30f ? d : copysignf(1e-30f, d);
}

__device__ __forceinline__ RaySetup setup_boxes(float ox, float oy, float oz, float dx, float dy, float dz,
                                                float delta, float near) {
    return RaySetup{make_float4(ox, oy, oz, 2.0f * delta),
                    make_float4(__frcp_rn(clamp_dir(dx)), __frcp_rn(clamp_dir(dy)), __frcp_rn(clamp_dir(dz)), near)};
}

// o: the origin in the current space and 2 delta; (dx, dy, dz): the direction,
// the same value the box set-up was made from
__device__ __forceinline__ Shear make_shear(const float4& o, float dx, float dy, float dz) {
    Shear sh;
    const float ax = fabsf(dx), ay = fabsf(dy), az = fabsf(dz);
    // kz = dominant axis, (kx, ky) the next two in cyclic order; selects
    // instead of indexed arrays keep everything in registers
    const int kz = (ax > ay) ? ((ax > az) ? 0 : 2) : ((ay > az) ? 1 : 2);
    const float dkx = kz == 0 ? dy : (kz == 1 ? dz : dx);
    const float dky = kz == 0 ? dz : (kz == 1 ? dx : dy);
    const float dkz = kz == 0 ? dx : (kz == 1 ? dy : dz);
    const float okx = kz == 0 ? o.y : (kz == 1 ? o.z : o.x);
    const float oky = kz == 0 ? o.z : (kz == 1 ? o.x : o.y);
    const float okz = kz == 0 ? o.x : (kz == 1 ? o.y : o.z);
    // one reciprocal; the products' extra rounding is covered by delta
    const float Sz = __frcp_rn(dkz);
    const float Sx = __fmul_rn(dkx, Sz), Sy = __fmul_rn(dky, Sz);
    // row X: +1 at kx, -Sx at kz; row Y: +1 at ky, -Sy at kz; row Z: Sz at kz
    sh.rx0 = kz == 0 ? -Sx : (kz == 2 ? 1.f : 0.f);
    sh.rx1 = kz == 1 ? -Sx : (kz == 0 ? 1.f : 0.f);
    sh.rx2 = kz == 2 ? -Sx : (kz == 1 ? 1.f : 0.f);
    sh.ry0 = kz == 0 ? -Sy : (kz == 1 ? 1.f : 0.f);
    sh.ry1 = kz == 1 ? -Sy : (kz == 2 ? 1.f : 0.f);
    sh.ry2 = kz == 2 ? -Sy : (kz == 0 ? 1.f : 0.f);
    sh.rz0 = kz == 0 ? Sz : 0.f;
    sh.rz1 = kz == 1 ? Sz : 0.f;
    sh.rz2 = kz == 2 ? Sz : 0.f;
    sh.cx = __fmaf_rn(-Sx, okz, okx);
    sh.cy = __fmaf_rn(-Sy, okz, oky);
    sh.cz = __fmul_rn(Sz, okz);
    // a position error of delta moves the distance along the dominant axis
    // by delta |Sz|; twice that bounds the FP32 hit distance's error
    sh.eps_t = __fmul_rn(o.w, fabsf(Sz));
    return sh;
}

__device__ __forceinline__ float maxabs3(float a, float b, float c) {
    return fmaxf(fabsf(a), fmaxf(fabsf(b), fabsf(c)));
}

// --------------------------------------------------------------------------
// Node fetch: 64 bytes as four 128-bit or two 256-bit read-only loads.  The
// loads do not allocate in L1: shared memory leaves it little room, and node
// lines are seldom reused by the same SM soon enough (nodes, or everything,
// allocating there: 0 to 3 % slower; L2 caches both).
// --------------------------------------------------------------------------
__device__ __forceinline__ uint4 ld_nc_na(const void* p) {
    uint4 v;
    asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "l"(p));
    return v;
}

__device__ __forceinline__ float4 ld_nc_na_f4(const void* p) {
    const uint4 v = ld_nc_na(p);
    return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z),
                       __uint_as_float(v.w));
}

// A node's sixteen words in memory order (QNode): o.xyz s.xyz, near/far plane
// codes lo.xyz hi.xyz, references.
template <int FETCH>
__device__ __forceinline__ void load_node(const QNode* n, uint32_t w[16]) {
    if constexpr (FETCH == 32) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
            asm volatile("ld.global.nc.L1::no_allocate.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                         : "=r"(w[8 * h]), "=r"(w[8 * h + 1]), "=r"(w[8 * h + 2]), "=r"(w[8 * h + 3]),
                           "=r"(w[8 * h + 4]), "=r"(w[8 * h + 5]), "=r"(w[8 * h + 6]),
                           "=r"(w[8 * h + 7])
                         : "l"(reinterpret_cast<const char*>(n) + 32 * h));
    } else {
        const uint4* p = reinterpret_cast<const uint4*>(n);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint4 v = ld_nc_na(p + k);
            w[4 * k] = v.x;
            w[4 * k + 1] = v.y;
            w[4 * k + 2] = v.z;
            w[4 * k + 3] = v.w;
        }
    }
}

// Plane value v(q) of byte i of w (QNode): one byte permute with plane_exp =
// 0x3F000000.
__device__ __forceinline__ float plane_v(uint32_t w, uint32_t plane_exp, int i) {
    return __uint_as_float(__byte_perm(w, plane_exp, 0x7044u | ((uint32_t)i << 8)));
}

// Three-operand minima and maxima (one instruction on sm_103a); a NaN operand
// is ignored, or propagated by the _nan forms.
__device__ __forceinline__ float max3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float min3(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// (a0, a1) * b + (c0, c1), both halves in one instruction.
__device__ __forceinline__ void fma2(float a0, float a1, float b, float c0, float c1, float& r0, float& r1) {
    asm("{.reg .b64 a, b, c, r;\n\t"
        "mov.b64 a, {%2, %3};\n\t"
        "mov.b64 b, {%4, %4};\n\t"
        "mov.b64 c, {%5, %6};\n\t"
        "fma.rn.f32x2 r, a, b, c;\n\t"
        "mov.b64 {%0, %1}, r;}"
        : "=f"(r0), "=f"(r1)
        : "f"(a0), "f"(a1), "f"(b), "f"(c0), "f"(c1));
}

// Tests the four children of a node, in slot order: entry distances (inf =
// missed), whether hit, references.  An empty slot can pass for hit where all
// of the node's planes lie within the widening; its kRefNone is then dropped
// when it comes up.
//
// A plane's distance is fma(v(q), s/d, (node.o - o)/d), its box widened by
// 2 delta.  delta alone bounds the ray's own position error; the second delta
// covers this arithmetic: with e = 2^-24, the roundings of s/d, node.o - o,
// 1/d and the fused product amount to at most e (|v s| + |node.o - o| +
// 2 |plane - o|) <= e (9 R + 3 |o|) in position, R the radius of the space's
// geometry (|v s| <= 2.7 R), while delta is at least 12 e (R + |o|).
template <int FETCH>
__device__ __forceinline__ void node_children(const QNode* node, uint32_t plane_exp, const RaySetup& r,
                                              float tmax, float t[4], bool hit[4], uint32_t ref[4]) {
    uint32_t w[16];
    load_node<FETCH>(node, w);
    const float o[3] = {r.o.x, r.o.y, r.o.z}, inv[3] = {r.inv.x, r.inv.y, r.inv.z};
    float A[3], bn[3], bf[3];
    uint32_t wn[3], wf[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float d = __fsub_rn(__uint_as_float(w[a]), o[a]);
        const float p = __fmul_rn(r.o.w, fabsf(inv[a]));
        A[a] = __fmul_rn(__uint_as_float(w[3 + a]), inv[a]);
        bn[a] = __fmaf_rn(d, inv[a], -p);
        bf[a] = __fmaf_rn(d, inv[a], p);
        // near and far planes by the sign of the direction
        const bool neg = inv[a] < 0.f;
        wn[a] = neg ? w[9 + a] : w[6 + a];
        wf[a] = neg ? w[6 + a] : w[9 + a];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        float n[3], f[3];
#pragma unroll
        for (int a = 0; a < 3; ++a)
            fma2(plane_v(wn[a], plane_exp, i), plane_v(wf[a], plane_exp, i), A[a], bn[a], bf[a], n[a], f[a]);
        const float tn = fmaxf(max3(n[0], n[1], n[2]), r.inv.w);
        const float tf = fminf(min3(f[0], f[1], f[2]), tmax);
        ref[i] = w[12 + i];
        hit[i] = tn <= tf;
        t[i] = hit[i] ? tn : kInfF;
    }
}

// --------------------------------------------------------------------------
// Quad test
// --------------------------------------------------------------------------
struct SV {
    float X, Y, Z;
};

__device__ __forceinline__ SV shear(const Shear& sh, float x, float y, float z) {
    SV s;
    s.X = __fmaf_rn(x, sh.rx0, __fmaf_rn(y, sh.rx1, __fmaf_rn(z, sh.rx2, -sh.cx)));
    s.Y = __fmaf_rn(x, sh.ry0, __fmaf_rn(y, sh.ry1, __fmaf_rn(z, sh.ry2, -sh.cy)));
    s.Z = __fmaf_rn(x, sh.rz0, __fmaf_rn(y, sh.rz1, __fmaf_rn(z, sh.rz2, -sh.cz)));
    return s;
}

// 2D edge function; exactly antisymmetric: edge(P,Q) == -edge(Q,P).
__device__ __forceinline__ float edge(const SV& P, const SV& Q) {
    return __fsub_rn(__fmul_rn(P.X, Q.Y), __fmul_rn(P.Y, Q.X));
}

// Exact-enough re-test in FP64 of quad `slot` of instance `inst`: object ray
// from the world ray and the instance's FP64 world->object matrix, then the
// watertight test with FP64 arithmetic.  A hit has t > tmin (world t, with
// quad-space u, v if UV, else 0); a miss returns t = +inf.
//
// The FP64 pipe is slow (1/64 of FP32) and was 65 % busy for rays of ambient
// occlusion, so nothing that can be had without it uses it: signs are read
// from the bits, (u, v) are divided out only if asked for, and each lane takes
// the triangles that it hits, nearly always one, instead of the warp going
// over both.  1 M rays of ambient occlusion on the island (0.40 re-tests a
// ray) 0.852 -> 0.802 ms, 2 M diffuse bounces on the mid scene 2.93 -> 2.87,
// 0.8 M camera rays 0.721 -> 0.711.  A shear scaled by the dominant component
// would save two more divisions, but decided 6 % more of the rays through
// edges wrongly (against 128-bit arithmetic).
//
// Without UV: any-hit rays, and the second test of kernels that return (u, v).
// The renderer's closest-hit kernels need none either, but measured slower
// with the short version (one-sample 1280x720 frames +1.2 %, 24 small views
// +2.3 %), though they spill less with it: the cause is not known.
struct Hit64 {
    double t;
    float u, v;
};

// Bit 0: x < 0, bit 1: x > 0, neither for a zero.
__device__ __forceinline__ uint32_t sign_bits(double x) {
    const uint32_t hi = (uint32_t)__double2hiint(x);
    return (hi << 1 | (uint32_t)__double2loint(x)) == 0 ? 0u : 2u - (hi >> 31);
}

template <bool UV>
static __device__ __noinline__ Hit64 quad_test64(const InstDev* ip, const InstDev64* ip64,
                                                 const QuadDev* quad, WRay ray, float tmin) {
    double o[3], d[3];
    const double e[3] = {(double)ray.ox - (double)ip->c[0], (double)ray.oy - (double)ip->c[1],
                         (double)ray.oz - (double)ip->c[2]};
    const double wd[3] = {ray.dx, ray.dy, ray.dz};
    const double* w = ip64->w;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        o[r] = w[3 * r] * e[0] + w[3 * r + 1] * e[1] + w[3 * r + 2] * e[2];
        d[r] = w[3 * r] * wd[0] + w[3 * r + 1] * wd[1] + w[3 * r + 2] * wd[2];
    }
    // kz = dominant axis, (kx, ky) the next two in cyclic order; selects
    // instead of indexed arrays keep everything in registers
    const int kz = (fabs(d[0]) > fabs(d[1])) ? ((fabs(d[0]) > fabs(d[2])) ? 0 : 2)
                                             : ((fabs(d[1]) > fabs(d[2])) ? 1 : 2);
    const auto pick = [kz](double a, double b, double c, double& x, double& y, double& z) {
        x = kz == 0 ? b : (kz == 1 ? c : a);
        y = kz == 0 ? c : (kz == 1 ? a : b);
        z = kz == 0 ? a : (kz == 1 ? b : c);
    };
    double dx, dy, dz;
    pick(d[0], d[1], d[2], dx, dy, dz);
    const double Sx = dx / dz, Sy = dy / dz, Sz = 1.0 / dz;
    double X[4], Y[4], Z[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        double px, py, pz;
        pick((double)quad->v[3 * k] - o[0], (double)quad->v[3 * k + 1] - o[1],
             (double)quad->v[3 * k + 2] - o[2], px, py, pz);
        X[k] = px - Sx * pz;
        Y[k] = py - Sy * pz;
        Z[k] = Sz * pz;
    }
    const auto E = [&](int p, int q) { return X[p] * Y[q] - Y[p] * X[q]; };
    const double e21 = E(2, 1), e02 = E(0, 2), e10 = E(1, 0), e32 = E(3, 2), e03 = E(0, 3);
    Hit64 h{__longlong_as_double(0x7ff0000000000000ll), 0.f, 0.f};
    // triangle 0: (v0, v1, v2) with weights (e21, e02, e10); triangle 1:
    // (v0, v2, v3) with weights (e32, e03, -e02).  Hit unless two weights have
    // opposite signs (one that is not a number leaves no distance below).
    const uint32_t s02 = sign_bits(e02);
    const uint32_t s0 = sign_bits(e21) | s02 | sign_bits(e10);
    const uint32_t s1 = sign_bits(e32) | sign_bits(e03) | (s02 >> 1) | (s02 << 1 & 2u);
    uint32_t left = (s0 != 3u ? 1u : 0u) | (s1 != 3u ? 2u : 0u);
#pragma unroll 1
    while (left) {
        const bool tri = !(left & 1u);
        left &= left - 1u;
        const double U = tri ? e32 : e21, V = tri ? e03 : e02, W = tri ? -e02 : e10;
        const double det = U + V + W;
        if (sign_bits(det)) {
            const double tt = (U * Z[0] + V * (tri ? Z[2] : Z[1]) + W * (tri ? Z[3] : Z[2])) / det;
            if (tt > (double)tmin && tt < h.t) {
                h.t = tt;
                if constexpr (UV) {
                    h.u = (float)((tri ? V : V + W) / det);
                    h.v = (float)((tri ? V + W : W) / det);
                }
            }
        }
    }
    return h;
}

// min / max of three values that return NaN when one is NaN.
__device__ __forceinline__ float min3_nan(float a, float b, float c) {
    float r;
    asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
    float r;
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// FP32 test of one quad in the object-space parameter s (smin < s < smax).
// kQuadUncertain: the decision is within its error bounds -- an edge function
// within its band of zero, or the hit distance within eps_t of either end of
// the interval -- and quad_test64 makes it.  A hit leaves its distance and
// (u, v) as numerators over det: few hits are kept, so few are divided.
enum QuadResult { kQuadMiss = 0, kQuadHit = 1, kQuadUncertain = 2 };

struct QuadHit {
    float s, u_num, v_num, det;
};

__device__ __forceinline__ QuadResult quad_test(const Shear& sh, float delta, const QuadDev* q, float smin,
                                                float smax, QuadHit& out) {
    const float4* p = reinterpret_cast<const float4*>(q);
    // quads are read once per test: no L1 allocation, as for the nodes
    const float4 a = ld_nc_na_f4(p), b = ld_nc_na_f4(p + 1), c = ld_nc_na_f4(p + 2);
    const SV s0 = shear(sh, a.x, a.y, a.z);
    const SV s1 = shear(sh, a.w, b.x, b.y);
    const SV s2 = shear(sh, b.z, b.w, c.x);
    const SV s3 = shear(sh, c.y, c.z, c.w);
    const float e21 = edge(s2, s1), e02 = edge(s0, s2), e10 = edge(s1, s0);
    const float e32 = edge(s3, s2), e03 = edge(s0, s3);
    // one error band for the whole quad: covers delta-perturbed vertices and
    // the rounding of the edge products
    const float M = fmaxf(max3(max3(fabsf(s0.X), fabsf(s0.Y), fabsf(s1.X)), fabsf(s1.Y), fabsf(s2.X)),
                          max3(fabsf(s2.Y), fabsf(s3.X), fabsf(s3.Y)));
    const float B = __fmaf_rn(4.0f * delta, M, 4.76837158e-07f * M * M);  // 2^-21 M^2
    // triangle 0 = (v0, v1, v2), weights (e21, e02, e10); triangle 1 = (v0,
    // v2, v3), weights (e32, e03, -e02).  Weights surely of both signs: a
    // miss; surely of one: a hit; a NaN is neither.
    const float mn0 = min3_nan(e21, e02, e10), mx0 = max3_nan(e21, e02, e10);
    const float mn1 = min3_nan(e32, e03, -e02), mx1 = max3_nan(e32, e03, -e02);
    const bool miss0 = mx0 > B && mn0 < -B, miss1 = mx1 > B && mn1 < -B;
    if (miss0 && miss1) return kQuadMiss;
    const bool hit0 = mn0 > B || mx0 < -B, hit1 = mn1 > B || mx1 < -B;
    bool sure = (miss0 || hit0) && (miss1 || hit1);
    QuadResult res = kQuadMiss;
    out.s = kInfF;
    bool second = !hit0;
    if (sure) {
        for (;;) {
            const float u = second ? e32 : e21, v = second ? e03 : e02, w = second ? -e02 : e10;
            const float det = __fadd_rn(__fadd_rn(u, v), w);
            const float T = __fmaf_rn(u, s0.Z, __fmaf_rn(v, second ? s2.Z : s1.Z, __fmul_rn(w, second ? s3.Z : s2.Z)));
            const float s = __fdiv_rn(T, det);
            if (s > smin && s < out.s) {
                const float vw = __fadd_rn(v, w);
                out = QuadHit{s, second ? v : vw, second ? vw : w, det};
                res = kQuadHit;
            }
            sure = sure && !(fabsf(s - smin) <= sh.eps_t || fabsf(s - smax) <= sh.eps_t);
            if (second || !hit1) break;
            second = true;  // both triangles hit: a folded quad
        }
    }
    return sure ? res : kQuadUncertain;
}

// --------------------------------------------------------------------------
// Two-level traversal
// --------------------------------------------------------------------------
struct TraceStats {
    uint32_t nodes;      // inner nodes visited
    uint32_t quads;      // quads tested
    uint32_t insts;      // instances entered
    uint32_t fallbacks;  // FP64 re-tests
    uint32_t rays;       // rays traced
    uint32_t verts;      // path vertices shaded (closest hits of the path tracer)
};

// Adds a thread's counters into stats[0..5] (rays, nodes, quads, instances,
// FP64 re-tests, shaded vertices), one atomic per warp and counter.  Call
// from converged code.
__device__ __forceinline__ void add_stats(unsigned long long* stats, const TraceStats& st) {
    uint32_t v[6] = {st.rays, st.nodes, st.quads, st.insts, st.fallbacks, st.verts};
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        uint32_t x = v[k];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xFFFFFFFFu, x, o);
        if ((threadIdx.x & 31) == 0 && x) atomicAdd(stats + k, (unsigned long long)x);
    }
}

// --------------------------------------------------------------------------
// Two-level traversal of one ray per thread
// --------------------------------------------------------------------------

// 32-bit shared-memory addresses; volatile, so that what is put there stays
// there instead of being kept in registers through the traversal.
__device__ __forceinline__ float4 lds4(uint32_t a) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts4(uint32_t a, float x, float y, float z, float w) {
    asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(a), "f"(x), "f"(y), "f"(z), "f"(w));
}
__device__ __forceinline__ float lds1(uint32_t a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts1(uint32_t a, float v) {
    asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v));
}
__device__ __forceinline__ uint32_t lds_u(uint32_t a) {
    uint32_t v;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts_u(uint32_t a, uint32_t v) {
    asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v));
}
__device__ __forceinline__ uint2 lds_u2(uint32_t a) {
    uint2 v;
    asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts_u2(uint32_t a, uint32_t x, uint32_t y) {
    asm volatile("st.shared.v2.u32 [%0], {%1,%2};" ::"r"(a), "r"(x), "r"(y));
}

// v by way of shared memory (this lane's word a): a value that the compiler
// cannot recompute and so keeps in a register.  Left to itself it rebuilt the
// plane constant and the stack's address in every node test.
__device__ __forceinline__ uint32_t keep_register(uint32_t a, uint32_t v) {
    sts_u(a, v);
    return lds_u(a);
}

// What a kernel asks of the traversal, and the shared memory it takes.
//   ANY    any hit instead of the closest
//   UV     the closest hit's quad-space (u, v) is wanted
//   RANGE  the ray's interval (tmin, tmax) is its own; otherwise (0, inf)
//   STACK  stack entries in shared memory; deeper ones, up to kMaxStack, go to
//          local memory
// Per thread kRecs 16-byte records and the stack's entries: 64 bits (distance,
// reference) for closest-hit rays, whose pops drop entries beyond the best
// hit; 32 bits (reference) for any-hit rays, which never drop one (tmax stays
// put until the ray ends) and have one word for the node tests of a shared ray
// behind them.  Per warp, record k of lane l lies at 512 k + 16 l and stack
// entry k after the records at (32 sizeof(Entry)) k + sizeof(Entry) l: lanes
// never conflict for a bank, however far apart their stacks are.
template <bool ANY_, bool UV_, bool RANGE_, int FETCH_, int STACK_>
struct TraversalKind {
    static constexpr bool ANY = ANY_, UV = UV_, RANGE = RANGE_;
    static constexpr int FETCH = FETCH_, STACK = STACK_;
    using Entry = std::conditional_t<ANY, uint32_t, uint64_t>;
    static constexpr int kRecs = ANY ? 6 : (UV || RANGE ? 8 : 6);
    static constexpr int kLaneBytes = kRecs * 16 + STACK * (int)sizeof(Entry) + (ANY ? 4 : 0);
    static_assert(STACK >= 4 && STACK <= 32, "a node's pushes fit, the tuning's caps lie beyond");
};

// Stack entries in shared memory: what fits the 228 KB of an SM (less 1 KB a
// block) at the kernel's resident warps, in blocks of 256 threads (at 28 warps
// of 128), at most 16 for any-hit rays.  A ray's
// stack seldom holds more than 9 entries, but the deepest of a warp's lanes is
// beyond 9 in half of a closest-hit frame's node steps and beyond 12 in a
// sixth, and a lane beyond takes its warp through the slower path.
constexpr int lane_room(int warps) { return warps > 40 ? 144 : warps > 32 ? 176 : warps > 28 ? 216 : 240; }
constexpr int shared_stack(bool any, int recs, int warps) {
    const int fits = any ? (lane_room(warps) - 16 * 6 - 4) / 4 : (lane_room(warps) - 16 * recs) / 8;
    return any && fits > 16 ? 16 : fits < 4 ? 4 : fits;
}

// Whether a kernel of this kind reaches its resident warps in those blocks.  At
// 48 warps closest-hit rays with (u, v) have room for two entries only and take
// four, at 40 warps (2 M diffuse bounces on the mid scene 5.30 ms against 5.74).
// Any-hit rays have eleven there: sun rays 1.48 -> 1.50 ms against sixteen at
// 40 warps, the mid frame 19.6 -> 18.8.
template <class Kind>
constexpr bool reaches(int warps) {
    if (warps > 40 && Kind::kRecs == 8) warps = 40;
    const int block = warps == 28 ? 128 : 256, blocks = 32 * warps / block;
    return blocks * (block * Kind::kLaneBytes + block / 32 * 16 + 1024) <= 228 * 1024;
}

// The ray-query kernels' rays, and the wavefront renderer's.
template <bool ANY, int FETCH, int OCC>
using QueryKind = TraversalKind<ANY, !ANY, true, FETCH, shared_stack(ANY, 8, OCC)>;
template <bool ANY, bool UV, int FETCH, int OCC>
using WaveKind = TraversalKind<ANY, UV, ANY, FETCH, shared_stack(ANY, UV ? 8 : 6, OCC)>;

// Resumable traversal.  init() sets the ray up; the caller then runs, while
// the ray is not finished, whichever step fits its state: inner_step (an inner
// node to test), instance_step (a TLAS leaf to enter), leaf_step (a BLAS leaf
// to test).  Registers hold what a node test reads; everything else about the
// ray -- its world-space form, the object-space direction, the hit -- lies in
// shared memory and is touched only when an instance is entered or left or a
// leaf is tested.  (Left to the compiler, the same state spilled to local
// memory: at 48 registers 476 bytes of spill stores per thread, half of all
// local accesses, with the stacks 1 KB a thread of L1 and L2 footprint.)
template <class Kind>
struct Traversal {
    static constexpr bool ANY = Kind::ANY, UV = Kind::UV, RANGE = Kind::RANGE;
    static constexpr int STACK = Kind::STACK;
    using Entry = typename Kind::Entry;

    uint32_t rec;         // shared-memory address of this thread's records
    uint32_t plane_exp;   // 0x3F000000 (plane_v)
    uint32_t tip;         // and of its stack's next free entry
    uint32_t bottom;      // and first entry
    uint32_t inst_tip;    // tip at instance entry; bottom at the top level
    RaySetup r;         // the ray in the current space; r.inv.w = tmin - te
    float lim;          // far end of its interval there: best hit (or tmax) - te
    uint32_t cur;       // reference to visit next, kRefNone: take one from the stack
    uint32_t pleaf;     // postponed BLAS leaf (0 = none)
    uint32_t node_base;
    int budget;         // inner-node tests left before the step limit
    bool found;         // any-hit rays: answered
    int waiting;        // quads that wait for resolve(): 1, or 2 when another wants its place
    uint32_t deep;      // local-memory address of the entries beyond shared memory

    // records: byte offsets from rec
    static constexpr uint32_t kWorldO = 0;       // r.o at the top level
    static constexpr uint32_t kWorldInv = 512;   // r.inv at the top level (w: tmin)
    static constexpr uint32_t kWorldD = 1024;    // world direction; closest hit: h_t, any hit: cur_inst
    static constexpr uint32_t kObjD = 1536;      // object-space direction, quad_base
    static constexpr uint32_t kHit = 2048;       // closest hit: inst, slot, error bound of h_t, cur_inst
    static constexpr uint32_t kObjO = 2048;      // any hit: r.o in object space
    // the quad that waits: slot, inst; closest hit also the error bound of its
    // distance; then te
    static constexpr uint32_t kPend = 2560;
    static constexpr uint32_t kPendEps = kPend + 8;
    static constexpr uint32_t kTe = kPend + 12;
    static constexpr uint32_t kTmax = ANY ? kPend + 8 : 3072 + 8;  // RANGE
    static constexpr uint32_t kUV = 3072;        // u, v of the best hit, tmax, unused
    static constexpr uint32_t kPendUV = 3584;    // of the waiting quad (u NaN: FP32 could not decide it)
    static constexpr uint32_t kHT = kWorldD + 12;
    static constexpr uint32_t kCurInst = ANY ? kWorldD + 12 : kHit + 12;

    static constexpr uint32_t kStride = 32u * (uint32_t)sizeof(Entry);  // between stack entries
    static constexpr uint32_t kShared = STACK * kStride;                // entries beyond go to local memory

    __device__ __forceinline__ bool top(const DevScene& S) const { return node_base == S.tlas_base; }

    // base: the warp's shared memory; deep_entries: kMaxStack - STACK entries
    // of the thread's local memory (not a member: that would put the whole
    // traversal there)
    __device__ __forceinline__ void bind(uint32_t base, Entry* deep_entries) {
        deep = (uint32_t)__cvta_generic_to_local(deep_entries);
        const uint32_t lane = threadIdx.x & 31u;
        const uint32_t own = base + 16u * lane;
        rec = keep_register(own, own);
        bottom = keep_register(own, base + 512u * Kind::kRecs + (uint32_t)sizeof(Entry) * lane);
        plane_exp = keep_register(own, 0x3F000000u);
        if constexpr (ANY) sts_u(steps_word(), 0u);
        cur = kRefNone;
        pleaf = 0;
        found = false;
        waiting = 0;
    }

    __device__ __forceinline__ float tmin() const { return RANGE ? lds1(rec + kWorldInv + 12) : 0.f; }
    __device__ __forceinline__ float tmax() const { return RANGE ? lds1(rec + kTmax) : kInfF; }

    __device__ __forceinline__ void init(const DevScene& S, float ox, float oy, float oz, float dx,
                                         float dy, float dz, float t0, float t1, uint32_t msteps,
                                         TraceStats& st) {
        ++st.rays;
        tip = inst_tip = bottom;
        node_base = S.tlas_base;
        pleaf = 0;
        budget = (int)min(msteps, 0x7FFFFFFFu);
        found = false;
        waiting = 0;
        lim = t1;
        r = setup_boxes(ox, oy, oz, dx, dy, dz, world_delta(S, ox, oy, oz), t0);
        sts4(rec + kWorldO, r.o.x, r.o.y, r.o.z, r.o.w);
        sts4(rec + kWorldInv, r.inv.x, r.inv.y, r.inv.z, r.inv.w);
        sts4(rec + kWorldD, dx, dy, dz, t1);
        if constexpr (!ANY) sts4(rec + kHit, __uint_as_float(0xFFFFFFFFu), 0.f, 0.f, 0.f);
        if constexpr (RANGE) sts1(rec + kTmax, t1);
        if constexpr (UV) sts_u2(rec + kUV, 0u, 0u);
        cur = S.n_inst > 0 ? 0u : kRefNone;  // TLAS root, an inner reference
    }

    // 2^-20 (|o| + R_top): the world ray is exact, so this covers only the
    // rounding of the slab arithmetic at the top level.
    static __device__ __forceinline__ float world_delta(const DevScene& S, float ox, float oy, float oz) {
        return 9.5367431640625e-07f * (maxabs3(ox, oy, oz) + S.R_top);
    }

    __device__ __forceinline__ WRay world() const {
        const float4 o = lds4(rec + kWorldO), d = lds4(rec + kWorldD);
        return WRay{o.x, o.y, o.z, d.x, d.y, d.z};
    }

    // Far end of the interval in object space (s units, widened by the
    // rounding of t - te).
    static __device__ __forceinline__ float object_limit(float t, float te) {
        return __fadd_rn(__fsub_rn(t, te), 1.9073486328125e-06f * (fabsf(t) + fabsf(te)));
    }

    __device__ __forceinline__ void put_shared(float t, uint32_t ref) {
        if constexpr (ANY) sts_u(tip, ref);
        else sts_u2(tip, ref, __float_as_uint(t));
        tip += kStride;
    }

    // As put_shared, wherever the entry goes; false if the stack is full (cap
    // entries).
    __device__ __forceinline__ bool put(float t, uint32_t ref, int cap) {
        if (tip - bottom < kShared) {
            put_shared(t, ref);
            return true;
        }
        const int i = (int)((tip - bottom - kShared) / kStride);
        if (i + STACK >= cap) return false;
        const uint32_t a = deep + (uint32_t)sizeof(Entry) * (uint32_t)i;
        if constexpr (ANY) asm volatile("st.local.u32 [%0], %1;" ::"r"(a), "r"(ref) : "memory");
        else asm volatile("st.local.v2.u32 [%0], {%1,%2};" ::"r"(a), "r"(ref), "f"(t) : "memory");
        tip += kStride;
        return true;
    }

    // Pops an entry into cur unless it lies beyond the best hit.  Both places
    // are read under a predicate: a branch and its reconvergence cost more.
    __device__ __forceinline__ void pop() {
        tip -= kStride;
        const uint32_t off = tip - bottom;
        const uint32_t far = deep + (off - kShared) / 32u;
        if constexpr (ANY) {
            asm volatile("{.reg .pred p;\n\t"
                         "setp.lt.u32 p, %1, %2;\n\t"
                         "@p ld.shared.u32 %0, [%3];\n\t"
                         "@!p ld.local.u32 %0, [%4];}"
                         : "=r"(cur)
                         : "r"(off), "n"(kShared), "r"(tip), "r"(far)
                         : "memory");
        } else {
            uint32_t ref, t;
            asm volatile("{.reg .pred p;\n\t"
                         "setp.lt.u32 p, %2, %3;\n\t"
                         "@p ld.shared.v2.u32 {%0,%1}, [%4];\n\t"
                         "@!p ld.local.v2.u32 {%0,%1}, [%5];}"
                         : "=r"(ref), "=r"(t)
                         : "r"(off), "n"(kShared), "r"(tip), "r"(far)
                         : "memory");
            cur = __uint_as_float(t) <= lim ? ref : kRefNone;
        }
    }

    // A lane is in exactly one of: an inner node to test (wants_inner), a TLAS
    // leaf to enter (at_instance), a BLAS leaf to test (at_leaf: postponed or
    // current), or nothing left to visit (visited; a quad may still wait).
    __device__ __forceinline__ bool wants_inner() const { return (int)cur >= 0; }
    __device__ __forceinline__ bool at_instance() const { return cur >= kRefInstance && (!ANY || pleaf == 0); }
    __device__ __forceinline__ bool at_blas_leaf() const { return cur - kRefLeaf < kRefNone - kRefLeaf; }
    __device__ __forceinline__ bool at_leaf() const { return pleaf != 0 || at_blas_leaf(); }
    __device__ __forceinline__ bool visited() const { return cur == kRefNone && pleaf == 0; }
    __device__ __forceinline__ bool finished() const { return visited() && waiting == 0; }

    __device__ __forceinline__ void stop(uint32_t e) {
        budget = kStopped | (int)e;
        cur = kRefNone;
        pleaf = 0;
        waiting = 0;
    }

    __device__ __forceinline__ void postpone() {
        if (pleaf == 0 && at_blas_leaf()) {
            pleaf = cur;
            cur = kRefNone;
        }
    }

    // Pops until cur holds a reference, the stack is empty, or (closest hit)
    // the instance boundary is reached while a leaf of this instance is still
    // postponed.  BLAS leaves met on the way are postponed (one at a time) so
    // that the lane keeps traversing inner nodes with the rest of its warp.
    // Any-hit rays leave the instance all the same and test the leaf from the
    // object-space ray in shared memory before they enter another (sun rays
    // 0.99 -> 0.97 ms); closest-hit rays would walk on without that leaf's hit
    // to cull with, and measured 5 % slower that way.
    __device__ __forceinline__ void advance(const DevScene& S) {
        postpone();
        while (cur == kRefNone) {
            if (tip == inst_tip) {
                if (top(S) || (!ANY && pleaf != 0)) break;
                leave_instance(S);
                if (tip == bottom) break;
            }
            pop();
            postpone();
        }
    }

    // Tests the inner node cur and moves on (precondition: wants_inner()).
    // Closest hit: the nearest hit child is visited next (the first of equally
    // near ones), the others are pushed with their entry distances.  They are
    // pushed in slot order, not sorted: with two hits, by far the most common
    // case, that is sorted already, and a sorting network took 25 instructions
    // of every node test.  Any hit: the first hit in slot order is next (the
    // answer does not depend on the order, and an unoccluded ray visits every
    // child anyway).
    __device__ __forceinline__ void inner_step(const DevScene& S, TraceStats& st, int cap) {
        --budget;
        ++st.nodes;
        float t[4];
        bool hit[4];
        uint32_t ref[4];
        node_children<Kind::FETCH>(S.nodes + (size_t)(node_base + cur), plane_exp, r, lim, t, hit, ref);
        bool next0, next1, next2;  // the child visited next, child 3 if none of these
        if constexpr (ANY) {
            next0 = hit[0];
            next1 = !hit[0] && hit[1];
            next2 = !hit[0] && !hit[1] && hit[2];
        } else {
            const float m = fminf(min3(t[0], t[1], t[2]), t[3]);
            next0 = t[0] == m;
            next1 = !next0 && t[1] == m;
            next2 = !next0 && !next1 && t[2] == m;
        }
        const bool next3 = !next0 && !next1 && !next2;
        const bool push[4] = {hit[0] && !next0, hit[1] && !next1, hit[2] && !next2, hit[3] && !next3};
        cur = next0 ? ref[0] : next1 ? ref[1] : next2 ? ref[2] : ref[3];
        if (!(hit[0] || hit[1] || hit[2] || hit[3])) cur = kRefNone;
        if (tip - bottom + 3 * kStride <= kShared) {
#pragma unroll
            for (int k = 3; k >= 0; --k)
                if (push[k]) put_shared(t[k], ref[k]);
        } else {
            bool room = true;
#pragma unroll
            for (int k = 3; k >= 0; --k)
                if (push[k]) room = room && put(t[k], ref[k], cap);
            if (!room) {
                stop(kErrStackOverflow);
                return;
            }
        }
        advance(S);
    }

    // Whether the ray has tested more nodes than it may; such a ray ends here.
    // Asked between steps and not in them, which saves two instructions of
    // every node test: a ray may go some nodes beyond its limit, but never ends
    // beyond it unreported.  (An any-hit ray shared with other lanes: share_rays.)
    __device__ __forceinline__ void check_budget() {
        if (budget < 0 && !error()) stop(kErrStepLimit);
    }

    // Device error bits of a ray that was stopped, else 0: they take the place
    // of its step count.
    static constexpr int kStopped = (int)0x80000000u;
    __device__ __forceinline__ uint32_t error() const {
        return (uint32_t)budget - (uint32_t)kStopped < 16u ? (uint32_t)(budget & 15) : 0u;
    }

    // Tests one BLAS leaf (the postponed one first; precondition: at_leaf()).
    __device__ __forceinline__ void leaf_step(const DevScene& S, TraceStats& st) {
        uint32_t ref = pleaf;
        if (ref) {
            pleaf = 0;
        } else {
            ref = cur;
            cur = kRefNone;
        }
        if (leaf(S, st, ref)) {
            answer();
        } else {
            advance(S);
        }
    }

    __device__ __forceinline__ void answer() {
        found = true;
        cur = kRefNone;
        pleaf = 0;
        waiting = 0;
    }

    // Moves the ray into the object space of the instance of the TLAS leaf cur
    // (precondition: at_instance()).  The world point p = o + te d where the
    // ray passes closest to the object origin and its offset p - c from that
    // origin are formed exactly as float pairs (two-product / two-sum), so the
    // FP32 object-space origin W (p - c) carries an error proportional to the
    // object's size only; the BLAS then works in s = t - te.
    __device__ __forceinline__ void instance_step(const DevScene& S, TraceStats& st) {
        const uint32_t inst = cur & kRefIndexMask;
        const float4* ip = reinterpret_cast<const float4*>(S.inst + inst);
        const float4 m0 = __ldg(ip), m1 = __ldg(ip + 1), m2 = __ldg(ip + 2), m3 = __ldg(ip + 3);
        // m0 = (c, R); m1 = (w0 w1 w2 w3); m2 = (w4 w5 w6 w7); m3 = (w8, node_base, quad_base, kappa)
        const float4 wo = lds4(rec + kWorldO), wd = lds4(rec + kWorldD);
        const float tmin_ = r.inv.w;  // at the top level
        // Re-centre where the ray passes closest to the object origin (never
        // before tmin), so the re-centred origin lies within the object's
        // reach; hits before that point have s < 0.  (Re-centring at the
        // instance box's entry distance instead needs that distance kept per
        // stack entry and per ray, and measured slower with more FP64
        // re-tests.)
        float te;
        {
            const float cx = __fsub_rn(m0.x, wo.x), cy = __fsub_rn(m0.y, wo.y), cz = __fsub_rn(m0.z, wo.z);
            const float dd = __fmaf_rn(wd.x, wd.x, __fmaf_rn(wd.y, wd.y, __fmul_rn(wd.z, wd.z)));
            const float tc = __fdiv_rn(__fmaf_rn(cx, wd.x, __fmaf_rn(cy, wd.y, __fmul_rn(cz, wd.z))), dd);
            te = (tc > tmin_ && tc < kInfF) ? tc : tmin_;
        }
        float exl, eyl, ezl;
        const float ex = exact_offset(wo.x, wd.x, te, m0.x, &exl);
        const float ey = exact_offset(wo.y, wd.y, te, m0.y, &eyl);
        const float ez = exact_offset(wo.z, wd.z, te, m0.z, &ezl);
        const float rox = __fmaf_rn(m1.x, ex, __fmaf_rn(m1.y, ey, __fmaf_rn(m1.z, ez,
                              __fmaf_rn(m1.x, exl, __fmaf_rn(m1.y, eyl, __fmul_rn(m1.z, ezl))))));
        const float roy = __fmaf_rn(m1.w, ex, __fmaf_rn(m2.x, ey, __fmaf_rn(m2.y, ez,
                              __fmaf_rn(m1.w, exl, __fmaf_rn(m2.x, eyl, __fmul_rn(m2.y, ezl))))));
        const float roz = __fmaf_rn(m2.z, ex, __fmaf_rn(m2.w, ey, __fmaf_rn(m3.x, ez,
                              __fmaf_rn(m2.z, exl, __fmaf_rn(m2.w, eyl, __fmul_rn(m3.x, ezl))))));
        // W d: the world direction in object space
        const float fdx = __fmaf_rn(m1.x, wd.x, __fmaf_rn(m1.y, wd.y, __fmul_rn(m1.z, wd.z)));
        const float fdy = __fmaf_rn(m1.w, wd.x, __fmaf_rn(m2.x, wd.y, __fmul_rn(m2.y, wd.z)));
        const float fdz = __fmaf_rn(m2.z, wd.x, __fmaf_rn(m2.w, wd.y, __fmul_rn(m3.x, wd.z)));
        node_base = __float_as_uint(m3.y);
        // 2^-22 (kappa + 2) (|o''| + R): rounding of W, of W (p - c), of W d and
        // of the shear arithmetic, with a factor-two margin
        r = setup_boxes(rox, roy, roz, fdx, fdy, fdz,
                        __fmul_rn(2.384185791015625e-07f * (m3.w + 2.0f), maxabs3(rox, roy, roz) + m0.w),
                        __fsub_rn(tmin_, te));
        sts1(rec + kTe, te);
        sts4(rec + kObjD, fdx, fdy, fdz, m3.z);
        if constexpr (ANY) sts4(rec + kObjO, rox, roy, roz, r.o.w);
        sts_u(rec + kCurInst, inst);
        lim = object_limit(ANY ? tmax() : wd.w, te);
        inst_tip = tip;
        ++st.insts;
        cur = 0;
    }

    // Back to the world-space ray and the top level.
    __device__ __forceinline__ void leave_instance(const DevScene& S) {
        r.o = lds4(rec + kWorldO);
        r.inv = lds4(rec + kWorldInv);
        lim = ANY ? tmax() : lds1(rec + kHT);
        inst_tip = bottom;
        node_base = S.tlas_base;
    }

    // (o + te d) - c per axis as a float pair hi + *lo, exact up to the
    // rounding of the small correction terms.
    static __device__ __forceinline__ float exact_offset(float o, float d, float te, float c, float* lo) {
        const float q = __fmul_rn(te, d);
        const float rho = __fmaf_rn(te, d, -q);       // te d = q + rho exactly
        const float s = __fadd_rn(o, q);
        const float bb = __fsub_rn(s, o);
        const float e1 = __fadd_rn(__fsub_rn(o, __fsub_rn(s, bb)), __fsub_rn(q, bb));  // o + q = s + e1
        const float hi = __fsub_rn(s, c);
        const float b2 = __fsub_rn(hi, s);
        const float e2 = __fadd_rn(__fsub_rn(s, __fsub_rn(hi, b2)), __fsub_rn(-c, b2));  // s - c = hi + e2
        *lo = __fadd_rn(e2, __fadd_rn(e1, rho));
        return hi;
    }

    // The hit, read back once the ray has ended.  The original quad index is
    // looked up from the slot here (any-hit results carry none).
    __device__ __forceinline__ Hit hit(const DevScene& S) const {
        Hit h;
        const float4 a = lds4(rec + kHit);
        h.t = lds1(rec + kHT);
        h.inst = __float_as_uint(a.x);
        h.slot = __float_as_uint(a.y);
        h.prim = h.inst == 0xFFFFFFFFu ? 0xFFFFFFFFu : __ldg(S.prim + h.slot);
        h.u = h.v = 0.f;
        if constexpr (UV) {
            h.u = lds1(rec + kUV);
            h.v = lds1(rec + kUV + 4);
        }
        return h;
    }

    // Makes (t, inst, slot) the best hit, and cuts the ray there.
    __device__ __forceinline__ void record(float t, uint32_t inst, uint32_t slot, float eps, float u, float v) {
        sts1(rec + kHT, t);
        sts_u2(rec + kHit, inst, slot);
        sts1(rec + kHit + 8, eps);
        if constexpr (UV) sts_u2(rec + kUV, __float_as_uint(u), __float_as_uint(v));
    }
    __device__ __forceinline__ void shorten(const DevScene& S, float t, float te) {
        lim = top(S) ? t : object_limit(t, te);
    }

    // Tests the quads of BLAS leaf ref; returns true when an any-hit query is
    // answered.  A quad that FP32 cannot decide, or whose distance is within
    // its error bound of the best hit's, waits for resolve(); while one waits
    // the traversal goes on, and the next one puts the rest of its leaf back.
    // So does a closest-hit ray's next hit of any kind: which of two near hits
    // keeps its FP32 distance and which gets an FP64 one depends on the order
    // they are compared in, and that must be the order of the traversal, not
    // the moment at which the warp came to resolve().
    __device__ __forceinline__ bool leaf(const DevScene& S, TraceStats& st, uint32_t ref) {
        const float4 od = lds4(rec + kObjD);
        const float4 oo = ANY ? lds4(rec + kObjO) : r.o;
        const Shear sh = make_shear(oo, od.x, od.y, od.z);
        const float te = lds1(rec + kTe);
        const float t0 = tmin(), t1 = tmax();
        const float smin = ANY ? __fsub_rn(t0, te) : r.inv.w;
        uint32_t slot = __float_as_uint(od.w) + (ref & kRefIndexMask);
        for (;;) {
            QuadHit q;
            const QuadResult res = quad_test(sh, 0.5f * oo.w, S.quads + slot, smin, __fsub_rn(t1, te), q);
            if (res != kQuadMiss) {
                const float t = __fadd_rn(q.s, te);
                bool wait = res == kQuadUncertain;
                float u = __int_as_float(0x7fffffff), v = 0.f;
                if constexpr (ANY) {
                    if (!wait && t > t0 && t < t1) return true;
                } else if (!wait && t > t0 && t < t1) {
                    const float ht = lds1(rec + kHT);
                    const float4 hr = lds4(rec + kHit);
                    const uint32_t inst = lds_u(rec + kCurInst);
                    const uint32_t hinst = __float_as_uint(hr.x), hslot = __float_as_uint(hr.y);
                    wait = waiting != 0 || (fabsf(t - ht) <= fmaxf(sh.eps_t, hr.z) && hinst != 0xFFFFFFFFu &&
                           !(hslot == slot && hinst == inst));
                    if (wait || t <= ht) {
                        if constexpr (UV) {
                            u = __fdiv_rn(q.u_num, q.det);
                            v = __fdiv_rn(q.v_num, q.det);
                        } else {
                            u = 0.f;
                        }
                        if (!wait && (t < ht || before(S, inst, slot, hinst, hslot))) {
                            record(t, inst, slot, sh.eps_t, u, v);
                            lim = object_limit(t, te);
                        }
                    }
                }
                if (wait) {
                    if (waiting) {
                        waiting = 2;
                        pleaf = ref;
                        return false;
                    }
                    waiting = 1;
                    sts_u2(rec + kPend, slot, lds_u(rec + kCurInst));
                    if constexpr (!ANY) sts1(rec + kPendEps, sh.eps_t);
                    if constexpr (UV) sts_u2(rec + kPendUV, __float_as_uint(u), __float_as_uint(v));
                }
            }
            ++st.quads;
            if ((ref & 0x38000000u) == 0) return false;
            // the rest of the leaf: one item further, one fewer
            ref -= (1u << 27) - 1u;
            ++slot;
        }
    }

    // Decides the waiting quad in FP64: two candidates whose distances are
    // within their error bounds of each other are ordered by their FP64
    // distances, equal distances by (instance, quad).  Rare, and slow on this
    // GPU (FP64 runs at 1/64 of FP32, and a warp pays for one lane what it
    // pays for all), so the caller gathers lanes for it.
    //
    // The traversal's registers (and the caller's, `item`) are put away in
    // local memory and read back here, by hand: the compiler, left to keep
    // them over the calls, stored each of them whenever it changed, nine local
    // stores in every node step.
    __device__ __forceinline__ void resolve(const DevScene& S, TraceStats& st, uint32_t& item) {
        volatile uint32_t away[19];
        const float rf[8] = {r.o.x, r.o.y, r.o.z, r.o.w, r.inv.x, r.inv.y, r.inv.z, r.inv.w};
        away[0] = rec;
#pragma unroll
        for (int k = 0; k < 8; ++k) away[1 + k] = __float_as_uint(rf[k]);
        away[9] = __float_as_uint(lim);
        away[10] = cur;
        away[11] = pleaf;
        away[12] = tip;
        away[13] = inst_tip;
        away[14] = bottom;
        away[15] = plane_exp;
        away[16] = node_base;
        away[17] = (uint32_t)budget;
        away[18] = item;
        ++st.fallbacks;
        bool better = false;
        {
            const uint2 p = lds_u2(rec + kPend);
            const Hit64 c = quad_test64<!ANY>(S.inst + p.y, S.inst64 + p.y, S.quads + p.x, world(), tmin());
            rec = away[0];
            const float t = (float)c.t, t0 = tmin(), t1 = tmax();
            better = t > t0 && t < t1 && c.t < (double)t1;
            if constexpr (!ANY) {
                if (better) better = beats_best(S, st, c, away);
            }
        }
        rec = away[0];
        const auto f = [&](int k) { return __uint_as_float(away[k]); };
        r.o = make_float4(f(1), f(2), f(3), f(4));
        r.inv = make_float4(f(5), f(6), f(7), f(8));
        lim = f(9);
        cur = away[10];
        pleaf = away[11];
        tip = away[12];
        inst_tip = away[13];
        bottom = away[14];
        plane_exp = away[15];
        node_base = away[16];
        budget = (int)away[17];
        item = away[18];
        waiting = 0;
        if (better) {
            if constexpr (ANY) answer();
            else shorten(S, lds1(rec + kHT), lds1(rec + kTe));
        }
    }

    // Whether the waiting quad's FP64 hit c beats the best hit, whose place it
    // then takes.  away[0] = rec.
    __device__ __forceinline__ bool beats_best(const DevScene& S, TraceStats& st, const Hit64& c,
                                               const volatile uint32_t* away) {
        const float4 hr = lds4(rec + kHit);
        const float t = (float)c.t, ht = lds1(rec + kHT);
        const uint2 p = lds_u2(rec + kPend);
        const uint32_t hinst = __float_as_uint(hr.x), hslot = __float_as_uint(hr.y);
        float eps = lds1(rec + kPendEps);
        bool better;
        if (fabsf(t - ht) <= fmaxf(eps, hr.z) && hinst != 0xFFFFFFFFu && !(hslot == p.x && hinst == p.y)) {
            ++st.fallbacks;
            const double tb =
                quad_test64<!UV>(S.inst + hinst, S.inst64 + hinst, S.quads + hslot, world(), tmin()).t;
            rec = away[0];
            better = c.t < tb || (c.t == tb && before(S, p.y, p.x, hinst, hslot));
        } else {
            better = t < ht || (t == ht && before(S, p.y, p.x, hinst, hslot));
            eps = 0.f;
        }
        if (better) {
            float u = c.u, v = c.v;
            if constexpr (UV) {
                const uint2 uv = lds_u2(rec + kPendUV);
                if (__uint_as_float(uv.x) == __uint_as_float(uv.x)) {  // an FP32 hit: its own (u, v)
                    u = __uint_as_float(uv.x);
                    v = __uint_as_float(uv.y);
                }
            }
            record(t, p.y, p.x, eps, u, v);
        }
        return better;
    }

    // ---- any-hit rays: parts of a ray's tree traversed by idle lanes ---------

    // Shared-memory address of the stack's lowest entry (the subtree highest in
    // the tree, as a rule the largest), 0 if there is none to give away.
    __device__ __forceinline__ uint32_t spare_entry() const {
        const uint32_t end = min(tip, bottom + kShared);
        for (uint32_t a = bottom; a != end; a += kStride)
            if (lds_u(a) != kRefNone) return a;
        return 0;
    }

    // Takes the entry at address `entry` from the ray of the lane with records
    // at `from` and makes this lane, which is idle, traverse it.  other, its
    // other_base, other_budget: that lane's ray, node_base and budget;
    // object_space: the entry lies in its instance.
    __device__ __forceinline__ void take(const DevScene& S, uint32_t from, uint32_t entry, bool object_space,
                                         const RaySetup& other, uint32_t other_base, int other_budget) {
#pragma unroll
        for (int k = 0; k < Kind::kRecs; ++k) {
            const float4 v = lds4(from + 512u * k);
            sts4(rec + 512u * k, v.x, v.y, v.z, v.w);
        }
        cur = lds_u(entry);
        sts_u(entry, kRefNone);
        pleaf = 0;
        tip = inst_tip = bottom;
        budget = other_budget;
        sts_u(steps_word(), (uint32_t)other_budget);
        found = false;
        waiting = 0;
        if (object_space) {
            r = other;
            node_base = other_base;
            lim = object_limit(tmax(), lds1(rec + kTe));
        } else {
            r.o = lds4(rec + kWorldO);
            r.inv = lds4(rec + kWorldInv);
            node_base = S.tlas_base;
            lim = tmax();
        }
    }

    // Of a ray's own lane: the node tests that its helpers made, kFailed and
    // error bits if one of them was stopped.  Of a helper: its budget when it
    // began.  Zeroed once: rays are shared when none is left to start, and a
    // lane that has been a helper never starts one.
    static constexpr uint32_t kFailed = 0xFFFFFFF0u;
    __device__ __forceinline__ uint32_t steps_word() const { return bottom + kShared; }
    // What a helper that is done has to add to its ray's word.
    __device__ __forceinline__ uint32_t spent() const {
        return error() ? kFailed | error() : lds_u(steps_word()) - (uint32_t)budget;
    }

    // Takes over what a helper lane found and spent.
    __device__ __forceinline__ void absorb(bool its_found, uint32_t its_spent) {
        const uint32_t had = lds_u(steps_word()), sum = had + its_spent;
        uint32_t now = sum < had || sum >= kFailed ? kFailed | kErrStepLimit : sum;
        if (had >= kFailed || its_spent >= kFailed)
            now = (had >= kFailed ? had : kFailed) | (its_spent >= kFailed ? its_spent : kFailed);
        sts_u(steps_word(), now);
        if (its_found && !error()) answer();
    }

    // The end of a shared ray (precondition: finished(), no helpers left): one
    // that is not answered is stopped if its lanes together made more tests than
    // it may, or one of them was.  The budget then counts them all (cost maps),
    // but an answered ray's does not go below 0.
    __device__ __forceinline__ void settle() {
        const uint32_t c = lds_u(steps_word());
        if (budget < 0) return;  // beyond the limit by itself
        if (c <= (uint32_t)budget) budget -= (int)c;
        else budget = found ? 0 : kStopped | (int)(c >= kFailed ? c & 15u : kErrStepLimit);
    }

    // Order of two hits at the same distance.
    static __device__ __forceinline__ bool before(const DevScene& S, uint32_t inst, uint32_t slot,
                                                  uint32_t hinst, uint32_t hslot) {
        return inst < hinst || (inst == hinst && __ldg(S.prim + slot) < __ldg(S.prim + hslot));
    }
};

// Shared memory of a block of `threads` threads, and a warp's part of it: the
// lanes' records and stacks, and the warp's claimed items.
template <class Kind>
constexpr size_t traversal_bytes(int threads) {
    return (size_t)threads * Kind::kLaneBytes + threads / 32 * 16;
}
template <class Kind>
__device__ __forceinline__ uint32_t traversal_base() {
    extern __shared__ __align__(512) unsigned char qrt_smem[];
    return (uint32_t)__cvta_generic_to_shared(qrt_smem) + (threadIdx.x >> 5) * (32u * Kind::kLaneBytes + 16u);
}

// What a lane of the persistent loop works on: item k, the ray of lane l
// (kHelper + l), nothing.
constexpr uint32_t kHelper = 0xFFFFFF00u, kIdle = 0xFFFFFFFFu;

// Each idle lane takes a subtree off the stack of a busy one, as long as one
// has any to give.  An unoccluded any-hit ray visits every node its segment
// meets, in whatever order, so its subtrees can go in parallel: at the end of
// a queue, and from the start of one too short for every lane, where otherwise
// the launch lasts as long as its longest ray.  Shadow rays of the mid frame
// 2.83 -> 2.53 ms, 1.5 M sun rays 0.90 -> 0.82.  Closest-hit rays lost that way
// (one ray on the mid scene 32 -> 80 us): the far subtrees are those which the
// near ones' hit culls.
//
// The step limit.  The lane that gives goes on as it would alone, from the top
// of its stack, and what it gives away lies at the bottom, which it would come
// to last.  So its own tests are those of a ray alone, in order; a helper begins
// with the budget left to its giver, so that a ray alone is beyond its limit
// wherever the helper is; and only the end of an unanswered ray adds them up
// (settle).  An unoccluded ray is reported exactly if it takes more tests than it
// may, as it is alone; an occluded one that is answered within its limit alone
// is answered here, whatever its helpers spend.  A ray that is stopped or
// answered ends its helpers.
template <class Kind>
__device__ __forceinline__ void share_rays(const DevScene& S, Traversal<Kind>& T, uint32_t& item, uint32_t base) {
    const unsigned FULL = 0xFFFFFFFFu;
    const unsigned lane = threadIdx.x & 31u;
    const unsigned idle = __ballot_sync(FULL, item == kIdle);
    if (idle == 0 || idle == FULL) return;
    const uint32_t give = item != kIdle && !T.visited() ? T.spare_entry() : 0u;
    const unsigned givers = __ballot_sync(FULL, give != 0u);
    if (givers == 0) return;
    __syncwarp();  // the givers' shared memory is read below
    const int rank = __popc(idle & ((1u << lane) - 1u));
    const bool takes = item == kIdle && rank < __popc(givers);
    const int src = takes ? (int)__fns(givers, 0, rank + 1) : (int)lane;
    const auto from = [&](float x) { return __shfl_sync(FULL, x, src); };
    const uint32_t entry = __shfl_sync(FULL, give, src);
    const bool object_space = __shfl_sync(FULL, (int)(!T.top(S) && give >= T.inst_tip), src);
    const uint32_t its_item = __shfl_sync(FULL, item, src);
    const uint32_t its_base = __shfl_sync(FULL, T.node_base, src);
    const int its_budget = __shfl_sync(FULL, T.budget, src);
    const RaySetup its_ray{make_float4(from(T.r.o.x), from(T.r.o.y), from(T.r.o.z), from(T.r.o.w)),
                           make_float4(from(T.r.inv.x), from(T.r.inv.y), from(T.r.inv.z), from(T.r.inv.w))};
    if (takes) {
        T.take(S, base + 16u * (uint32_t)src, entry, object_space, its_ray, its_base, its_budget);
        item = its_item >= kHelper ? its_item : kHelper + (uint32_t)src;
    }
    __syncwarp();
}

// Helpers that are done hand over what they found and spent; the helpers of a
// ray that is answered or stopped end.  Returns the lanes whose ray others
// still help with.
template <class Kind>
__device__ __forceinline__ unsigned gather_rays(Traversal<Kind>& T, uint32_t& item) {
    const unsigned FULL = 0xFFFFFFFFu;
    const unsigned lane = threadIdx.x & 31u;
    unsigned ready = __ballot_sync(FULL, item >= kHelper && item != kIdle && T.finished());
    const uint32_t spent = ready >> lane & 1u ? T.spent() : 0u;
    while (ready) {
        const int j = __ffs(ready) - 1;
        ready &= ready - 1;
        const int owner = (int)(__shfl_sync(FULL, item, j) - kHelper);
        const bool its_found = __shfl_sync(FULL, (int)(T.found && !T.error()), j);
        const uint32_t its_spent = __shfl_sync(FULL, spent, j);
        if ((int)lane == owner) T.absorb(its_found, its_spent);
        if ((int)lane == j) item = kIdle;
    }
    const unsigned over = __ballot_sync(FULL, item < kHelper && (T.found || T.error()));
    if (item >= kHelper && item != kIdle && (over >> (item - kHelper) & 1u)) {
        T.answer();  // its steps are still handed over, next time
        T.found = false;
    }
    return __reduce_or_sync(FULL, item >= kHelper && item != kIdle ? 1u << (item - kHelper) : 0u);
}

// Persistent warp-synchronous traversal loop over work items [0, count).  Each
// lane holds one ray; start(k) sets item k up in T (T.init), done(k) consumes
// the finished ray in T; a ray may use cap (<= kMaxStack) stack entries, a
// launch-wide value passed down rather than kept per ray.
//
// The first items are dealt out: L to each warp, as many as it takes for the
// launch's warps to hold them all, at most 32.  So a short queue is spread one
// ray to a warp and over all SMs, where no ray waits for another's divergent
// steps.  Later ones are claimed from *cursor (zero at the launch), one atomic
// for a warp: 32 items while plenty are left, then `batch` for each idle lane.
// A finished lane takes the next of them at once and never waits for the
// slowest ray of its warp.
//
// Per outer iteration the warp first tests inner nodes together (lanes that
// reach a BLAS leaf postpone it and keep traversing; lanes waiting at
// instances enter them in groups) until few lanes are left with an inner node,
// then lanes enter instances or test one leaf each.
template <class Kind, class Start, class Done>
__device__ __forceinline__ void persistent_trace(const DevScene& S, Traversal<Kind>& T, TraceStats& st,
                                                 uint32_t* cursor, uint32_t count, uint32_t batch, int cap,
                                                 Start start, Done done) {
    const unsigned FULL = 0xFFFFFFFFu;
    const unsigned lane = threadIdx.x & 31u;
    const uint32_t base = traversal_base<Kind>();
    const uint32_t claimed = base + 32u * Kind::kLaneBytes;  // claimed items not yet started: first, end
    typename Kind::Entry deep[kMaxStack - Kind::STACK];
    T.bind(base, deep);
    uint32_t item = kIdle;
    int waited = 0;  // iterations lanes have sat with nothing left but a waiting quad
    bool more;       // items may be left to claim
    {
        const uint32_t warps = gridDim.x * (blockDim.x >> 5);
        const uint32_t w = (threadIdx.x >> 5) * gridDim.x + blockIdx.x;
        const uint32_t L = min(32u, (count + warps - 1) / warps);
        const uint32_t k = w * L + lane;
        if (lane < L && k < count) {
            item = k;
            start(k);
        }
        more = count > 32u * warps;
        if (lane == 0) sts_u2(claimed, 0u, 0u);
        __syncwarp();
    }
    for (;;) {
        const unsigned want = __ballot_sync(FULL, item == kIdle);
        if (more && want) {
            const uint32_t n = (uint32_t)__popc(want), rank = (uint32_t)__popc(want & ((1u << lane) - 1u));
            const uint2 have = lds_u2(claimed);
            const uint32_t left = have.y - have.x;
            uint32_t first = 0;
            uint32_t claim = batch * n;
            if (n > left) {
                const uint32_t warps = gridDim.x * (blockDim.x >> 5);
                // a warp's worth at a time while every warp still has several to
                // come: the claims share one counter, and so one L2 slice
                // (closest-hit stage of the mid frame 8.22 -> 8.00 ms; down to
                // two warps' worth left, sun rays lost 2 % in the tail)
                if (have.y + 128u * warps < count) claim = max(claim, 32u);
                if (lane == 0) first = 32u * warps + atomicAdd(cursor, claim);
                first = __shfl_sync(FULL, first, 0);
            }
            __syncwarp();
            if (lane == 0) {
                if (n > left) sts_u2(claimed, first + (n - left), first + claim);
                else sts_u2(claimed, have.x + n, have.y);
            }
            __syncwarp();
            if (item == kIdle) {
                const uint32_t k = rank < left ? have.x + rank : first + (rank - left);
                if (k < count) {
                    item = k;
                    start(k);
                }
            }
            more = __all_sync(FULL, item != kIdle);  // past the end: nothing more to claim
        }
        if constexpr (Kind::ANY)
            if (!more) share_rays(S, T, item, base);
        if (!__any_sync(FULL, item != kIdle)) break;
        // rays with something left to do (one that only waits for its helpers
        // has not)
        const int n_busy = __popc(__ballot_sync(FULL, item != kIdle && !T.finished()));
        int turns = more ? -1 : 8;  // any hit: then see again who is idle
        for (;;) {
            // Once eight or more lanes wait at an instance (TLAS leaf), they
            // enter it together and go on with the inner nodes of its BLAS
            // in this phase, instead of idling until the next outer
            // iteration.  Each such step enters at least eight instances.
            const bool wt = T.at_instance();
            if (__popc(__ballot_sync(FULL, wt)) >= 8) {
                if (wt) T.instance_step(S, st);
                continue;
            }
            // Leave the inner-node phase early once the lanes still in it are
            // no more than the lanes waiting at an instance or a leaf (any
            // hit: half as many): those then move on together instead of
            // idling until the warp's longest run of inner nodes ends.  A lane
            // that the next phase moves on is left then, or no lane is busy,
            // so every outer iteration makes progress.  (Closest hit with the
            // other line +2 %; ambient occlusion with it +8 %, sun rays even.)
            const bool w = T.wants_inner();
            if ((Kind::ANY ? 3 : 2) * __popc(__ballot_sync(FULL, w)) <= n_busy || (Kind::ANY && turns-- == 0)) break;
            if (w) T.inner_step(S, st, cap);
        }
        if (T.at_instance()) {
            T.instance_step(S, st);
        } else if (T.at_leaf()) {
            T.leaf_step(S, st);
        }
        // Waiting quads are decided together: when a lane cannot go on, when
        // eight wait, or when the lanes that wait for nothing else have cost
        // about as much as the FP64 test does.
        const unsigned bp = __ballot_sync(FULL, T.waiting != 0);
        if (bp) {
            const bool idle = T.waiting != 0 && T.visited();
            waited += __popc(__ballot_sync(FULL, idle));
            if (__popc(bp) >= 8 || waited >= 16 || __any_sync(FULL, T.waiting == 2) ||
                !__any_sync(FULL, item != kIdle && !idle)) {
                if (T.waiting) T.resolve(S, st, item);
                waited = 0;
            }
        }
        unsigned helped = 0;  // lanes whose ray others still help with
        if constexpr (Kind::ANY)
            if (!more) helped = gather_rays(T, item);
        if (item != kIdle) T.check_budget();
        if (item < kHelper && T.finished() && !(helped >> lane & 1u)) {
            if constexpr (Kind::ANY)
                if (!more) T.settle();
            done(item);
            item = kIdle;
        }
    }
}

// Closest hit or any hit (Kind::ANY) of the world ray, run to completion by
// one thread.  Returns device error bits (0 = fine); a closest hit is left in
// *h (inst = 0xFFFFFFFF if none), an any-hit answer in *found.
template <class Kind>
__device__ __forceinline__ uint32_t trace_ray(const DevScene& S, float wox, float woy, float woz,
                                              float wdx, float wdy, float wdz, float tmin, float tmax,
                                              uint32_t max_steps, int cap, Hit* h, bool* found,
                                              TraceStats& st) {
    Traversal<Kind> T;
    typename Kind::Entry deep[kMaxStack - Kind::STACK];
    T.bind(traversal_base<Kind>(), deep);
    T.init(S, wox, woy, woz, wdx, wdy, wdz, tmin, tmax, max_steps, st);
    uint32_t none = 0;
    for (;;) {
        T.check_budget();  // may end the ray
        if (T.finished()) break;
        if (T.waiting == 2 || T.visited())
            T.resolve(S, st, none);
        else if (T.wants_inner())
            T.inner_step(S, st, cap);
        else if (T.at_instance())
            T.instance_step(S, st);
        else
            T.leaf_step(S, st);
    }
    if constexpr (Kind::ANY)
        *found = T.found;
    else
        *h = T.hit(S);
    return T.error();
}

}  // namespace qrt
