// Where a record can be accepted: the half extents of the pixels whose FP32
// power may come out at or above the record's threshold.  The record's own
// half extents (ex, ey) are those of the undivided covariance; the conic that
// the blend evaluates was divided by a c - b^2, which cancels for needles, and
// the evaluated power carries the rounding of terms many times its size, so
// for needles of hundreds of pixels the accepted pixels reach beyond (ex, ey)
// by up to tens of pixels.  Every kernel that leaves records out by their
// extents uses the bound below.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace msgs {

__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// power log2(e) = A dx^2 + B dx dy + C dy^2, in the blend's FP32 operations,
// is within 6 u (|A| dx^2 + |B dx dy| + |C| dy^2) of exact (u = 2^-24).  On
// one pixel row the record is accepted between the roots in dx of that sum =
// thr, whose discriminant is d = -(4 A C - B^2) dy^2 + 4 A thr; the rounding
// moves those roots by no more than raising d by 54 u 4 A C dy^2 + 18 u 4 A thr.
// With kReachErr = 64 u the form below, 4 A C lowered by 2 kReachErr and thr
// raised by kReachErr, is raised by more than that and its own rounding: a
// row's accepted pixels have (B dy - sqrt(d)) / -2A <= dx <= (B dy + sqrt(d)) /
// -2A.  Where the product so lowered is above B^2 (condition 4 A C / (4 A C -
// B^2) below 1.3e5) the rows' intervals form an ellipse, else they only widen
// with dy.  An FP32 emulation of 1800 needles of 3 to 3000 px, every pixel at
// their tips and a sample of the tiles between, found none accepted outside.
// The ellipse has the plain extents to 1% below a condition of 2600.
constexpr float kReachErr = 3.8e-6f;
// The conic's entries are above 1e-16 in magnitude (splats of up to 1e8 px),
// so that their products are normal numbers; false also for NaN.
__device__ __forceinline__ bool reach_curved(float A, float C) {
    return A < -1e-16f && C < -1e-16f;
}
// 4 A C - B^2 lowered, and 4 thr raised.
__device__ __forceinline__ float reach_det(float A, float B, float C) {
    return fmaf(-B, B, 4.0f * (1.0f - 2.0f * kReachErr) * A * C);
}
__device__ __forceinline__ float reach_thr(float thr) { return 4.0f * (1.0f + kReachErr) * thr; }
// The ellipse's half extents; false without one.
__device__ __forceinline__ bool reach_extents(float A, float B, float C, float thr, float &ex,
                                              float &ey) {
    const float den = reach_det(A, B, C), q = __fdividef(reach_thr(thr), den);
    ex = sqrt_approx(C * q);
    ey = sqrt_approx(A * q);
    return reach_curved(A, C) && den > 0.0f;
}
// The same bound, coarser, on the record's own half extents, without B and C
// and the square roots (a mask pass forms one per list entry): A ex^2 / thr is
// the condition k = a c / (a c - b^2), and the pixels lie within ex (1 + 32 u
// k), ey (1 + 32 u k) while that factor is at most 1.25 (12 u k are the
// power's rounding, 5 u k the conic's, to first order; the emulation above
// agrees).  False beyond, and for NaN.  The list kernel's masks gather 32
// bytes a record for it instead of 16: the deepest lists' blend (71x38, 51k
// entries a tile) 688 -> 708 us, with reach_extents 720.
__device__ __forceinline__ bool reach_box(float A, float thr, float &ex, float &ey) {
    const float rho = 1.9073486328125e-6f * __fdividef(A * ex * ex, thr);
    ex = fmaf(rho, ex, ex);
    ey = fmaf(rho, ey, ey);
    return rho <= 0.25f;
}

}  // namespace msgs
