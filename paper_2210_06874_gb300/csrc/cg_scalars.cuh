// cg_scalars.cuh -- the scalar state of the FP32 CG iterations, shared by every
// kind of FP32 iteration.
#pragma once

#include "tc_tile.cuh"

namespace hmc {
namespace tc {

enum SegmentEnd : int { kSegUpdate = 1, kSegMaxIter = 2, kSegNonfinite = 3 };

// Scalar state of the FP32 iteration, kept and updated by thread 0 alone
// and read by the other threads after a barrier, in FP32 (the iterates are
// FP32; FP64 arithmetic runs at a small fraction of the FP32 rate and with
// long latency on this part).  rr = |r|^2, pp = |p|^2 estimate (sets the
// vector scale of the tensor-core operands), rmax = |r|^2 at the last
// reliable update; stop and ru2 are the FP32 images of the FP64 criteria.
struct CgScalars {
    float rr, pp, rmax, alpha, beta, sc, inv, stop, ru2;
    int it, reason;
    int it0, every;   // iteration of the last reliable update; the most between two
};

// Thread 0, after qq = |q|^2: alpha and the scale of q.
__device__ __forceinline__ void cg_after_q(CgScalars& s, float qq) {
    int rs = 0;
    if (!isfinite(qq) || !(qq > 0.f)) {
        rs = kSegNonfinite;
    } else {
        s.alpha = s.rr / qq;
        vector_scale_f(qq, s.sc, s.inv);
    }
    s.reason = rs;
}

// Thread 0, after rr_new = |r|^2: segment end, or beta, pp and the scale of
// the next direction.
__device__ __forceinline__ void cg_after_r(CgScalars& s, float rr_new) {
    int rs = 0;
    s.it += 1;
    if (!isfinite(rr_new)) {
        rs = kSegNonfinite;
    } else if (rr_new <= s.stop || rr_new <= s.ru2 * s.rmax || s.it - s.it0 >= s.every) {
        rs = kSegUpdate;
    } else {
        const float b = rr_new / s.rr;
        s.beta = b;
        s.rr = rr_new;
        s.pp = fmaf(b * b, s.pp, rr_new);
        vector_scale_f(s.pp, s.sc, s.inv);
    }
    s.reason = rs;
}

}  // namespace tc
}  // namespace hmc
