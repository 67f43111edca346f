// Device data layout of a qrt scene in HBM, shared by the host builder
// (bvh_build.cpp) and the CUDA kernels.
//
//   nodes   QNode[ sum of BLAS nodes | TLAS nodes ]   64 B each, 64-B aligned
//   quads   QuadDev[ all meshes, leaf order ]          48 B each (4 x float3)
//   prim    uint32[ same slots ]: original quad index within its mesh
//   inst    InstDev[ n_inst ]                          64 B each
//   inst64  InstDev64[ n_inst ]: FP64 transform for the exact re-test, 80 B
//
// All indices are 32-bit offsets from 64-bit bases.  Stack references are
// local to the current level (TLAS or one BLAS), so every object may hold up
// to 2^27 nodes and 2^27 quads.
#pragma once
#include <stdint.h>

namespace qrt {

// Four-wide node with conservatively quantised child boxes.
//
// A plane code q stands for the float v(q) with bits 0x3F000000 | q << 16:
// v = 0.5 + q/256 for q < 128 and q/128 above, 0.5 .. 1.9921875, and the plane
// lies at fma(v(q), s, o).  The traversal makes v(q) with one byte permute,
// with no integer-to-float conversion, and s need not be a power of two, so
// the 256 codes cover the node's extent exactly (192 to 384 steps per
// extent).  Boxes are rounded outward: a dequantised box always contains the
// exact child box.  An axis whose extent cannot be covered in FP32 (beyond
// about 5e38) has s = NaN and bounds nothing: slab tests take minima and
// maxima that ignore NaN.
struct alignas(64) QNode {
    float o[3], s[3];
    uint8_t qlo[3][4];  // [axis][child]
    uint8_t qhi[3][4];  // [axis][child]
    uint32_t ref[4];    // child references (below); kRefNone = empty slot (qlo 255, qhi 0)
};
static_assert(sizeof(QNode) == 64, "QNode must be 64 bytes");

constexpr uint32_t kMaxLeaf = 8;

// Stack/child reference.  Inner node: its index, local to its tree.  BLAS
// leaf: bit 31, (count-1) in bits 27..29, first local quad slot in bits 0..26.
// TLAS leaf: bits 31 and 30, the instance.  kRefNone is no leaf: eight quads
// cannot start at the last slot there is.  One unsigned comparison tells each
// kind from the others.
constexpr uint32_t kRefLeaf = 0x80000000u;
constexpr uint32_t kRefInstance = 0xC0000000u;
constexpr uint32_t kRefIndexMask = 0x07FFFFFFu;
constexpr uint32_t kMaxLocalIndex = kRefIndexMask;
constexpr uint32_t kRefNone = 0xBFFFFFFFu;

struct alignas(16) QuadDev {
    float v[12];  // v0, v1, v2, v3 as packed float3
};
static_assert(sizeof(QuadDev) == 48, "QuadDev must be 48 bytes");

// Instance record, 64 bytes.  A ray entering the instance is re-centred on
// the world ray with error-free FP32 transformations (the point o + t_e d and
// its offset from c are formed exactly as float pairs), so the FP32 object-
// space ray's error scales with the object's size and the transform's
// condition number kappa, not with the object's distance.
struct alignas(64) InstDev {
    float c[3];          // object origin in world space (translation of object->world)
    float R;             // max |coordinate| of the object's bounding box
    float w[9];          // world->object linear part, row-major (FP32 of the FP64 inverse)
    uint32_t node_base;  // global index of this object's BLAS root
    uint32_t quad_base;  // global slot of its first quad == its first albedo row
    float kappa;         // infinity-norm condition number of the linear part
};
static_assert(sizeof(InstDev) == 64, "InstDev must be 64 bytes");

// FP64 world->object linear part, read only by the exact quad re-test.
struct alignas(16) InstDev64 {
    double w[9];
    double pad;
};
static_assert(sizeof(InstDev64) == 80, "InstDev64 must be 80 bytes");

// Everything a kernel needs, passed by value.
struct DevScene {
    const QNode* nodes;
    const QuadDev* quads;
    const uint32_t* prim;
    const InstDev* inst;
    const InstDev64* inst64;
    uint32_t tlas_base;  // global node index of the TLAS root
    uint32_t n_inst;
    float R_top;         // max |coordinate| of the world box
    uint32_t pad;
    uint32_t* err;       // device error word [0] = bits, [1] = first bad index
};

// Device error bits.
constexpr uint32_t kErrStackOverflow = 1u;
constexpr uint32_t kErrStepLimit = 2u;

// Traversal stack entries per ray allocated by the ray-query and wavefront
// trace kernels; tuning.stack caps how many a ray may use (32 or 64).
constexpr int kMaxStack = 64;

}  // namespace qrt
