// Box quantisation of a four-wide node (QNode, qrt_layout.h), shared by the host
// builder (bvh_build.cpp) and the linear BVH builds on device and host
// (lbvh.cu): one rule, the same codes everywhere.
#pragma once
#include <math.h>
#include <stdint.h>

#include "bvh_build.h"
#include "qrt_layout.h"

#ifdef __CUDACC__
#define QRT_HD __host__ __device__
#else
#define QRT_HD
#endif

namespace qrt {

// v(q) of a plane code (see QNode).
QRT_HD inline float code_value(int q) {
    return q < 128 ? 0.5f + (float)q * (1.0f / 256.0f) : (float)q * (1.0f / 128.0f);
}

QRT_HD inline float dequant(int q, float s, float o) { return fmaf(code_value(q), s, o); }

// Quantises the [lo, hi] intervals of nc children along one axis.  Returns
// false if the extent cannot be covered in FP32.
QRT_HD inline bool quantize_axis(const float* lo, const float* hi, int nc, float* s_out, float* o_out,
                                 uint8_t* qlo, uint8_t* qhi) {
    const float inf = (float)INFINITY;
    float ulo = lo[0], uhi = hi[0];
    for (int i = 1; i < nc; ++i) {
        ulo = fminf(ulo, lo[i]);
        uhi = fmaxf(uhi, hi[i]);
    }
    // the step: v spans 1.4921875 s over the extent.  Rounding of the origin
    // can leave the top plane short of uhi; the step then grows, slowly at
    // first (a rounding's worth), then in large steps (the origin's own
    // spacing exceeds the extent).
    double step = ((double)uhi - (double)ulo) / 1.4921875;
    for (int k = 0; k < 64; ++k) {
        float s = (float)step;
        if ((double)s < step) s = nextafterf(s, inf);
        float o = (float)((double)ulo - 0.5 * (double)s);
        if (!(s <= 3.402823466e38f) || !(fabsf(o) <= 3.402823466e38f)) return false;
        while (dequant(0, s, o) > ulo) o = nextafterf(o, -inf);
        if (!(fabsf(o) <= 3.402823466e38f)) return false;
        if (dequant(255, s, o) >= uhi) {
            const double inv = s > 0.f ? 1.0 / (double)s : 0.0;
            for (int i = 0; i < nc; ++i) {
                const double xl = ((double)lo[i] - (double)o) * inv;
                const double fl = xl < 1.0 ? floor((xl - 0.5) * 256.0) : floor(xl * 128.0);
                int ql = (int)(fl < 0.0 ? 0.0 : (fl > 255.0 ? 255.0 : fl));
                while (ql > 0 && dequant(ql, s, o) > lo[i]) --ql;
                const double xh = ((double)hi[i] - (double)o) * inv;
                const double ch = xh <= 1.0 ? ceil((xh - 0.5) * 256.0) : ceil(xh * 128.0);
                int qh = (int)(ch < 0.0 ? 0.0 : (ch > 255.0 ? 255.0 : ch));
                while (qh < 255 && dequant(qh, s, o) < hi[i]) ++qh;
                qlo[i] = (uint8_t)ql;
                qhi[i] = (uint8_t)qh;
            }
            *s_out = s;
            *o_out = o;
            return true;
        }
        double next = step * (k < 4 ? 1.0 + 1e-6 : 1.25);
        const double floor_step = 1.5e-45;  // smallest FP32 subnormal
        step = next > floor_step ? next : floor_step;
    }
    return false;
}

// Fills the boxes of q from its nc child boxes (slots 0 .. nc-1; the others
// become empty).  An axis that cannot be covered bounds nothing.
QRT_HD inline void quantize_node(QNode& q, const FBox* cb, int nc) {
    for (int a = 0; a < 3; ++a) {
        float lo[4], hi[4];
        for (int i = 0; i < nc; ++i) {
            lo[i] = cb[i].lo[a];
            hi[i] = cb[i].hi[a];
        }
        for (int i = 0; i < 4; ++i) {
            q.qlo[a][i] = 255;
            q.qhi[a][i] = 0;
        }
        if (!quantize_axis(lo, hi, nc, &q.s[a], &q.o[a], q.qlo[a], q.qhi[a])) {
            q.s[a] = nanf("");
            q.o[a] = 0.f;
        }
    }
}

// The dequantised box of child i (infinite along an uncovered axis).
QRT_HD inline FBox child_bounds(const QNode& q, int i) {
    const float inf = (float)INFINITY;
    FBox b;
    for (int a = 0; a < 3; ++a) {
        const bool covered = q.s[a] == q.s[a];
        b.lo[a] = covered ? dequant(q.qlo[a][i], q.s[a], q.o[a]) : -inf;
        b.hi[a] = covered ? dequant(q.qhi[a][i], q.s[a], q.o[a]) : inf;
    }
    return b;
}

QRT_HD inline uint32_t leaf_ref(uint32_t first, uint32_t count) {
    return kRefLeaf | ((count - 1u) << 27) | first;
}
QRT_HD inline uint32_t instance_ref(uint32_t inst) { return kRefInstance | inst; }
QRT_HD inline bool is_inner(uint32_t ref) { return !(ref & kRefLeaf); }
QRT_HD inline uint32_t leaf_count(uint32_t ref) { return ((ref >> 27) & 0x7u) + 1u; }
QRT_HD inline uint32_t leaf_first(uint32_t ref) { return ref & kRefIndexMask; }

}  // namespace qrt
