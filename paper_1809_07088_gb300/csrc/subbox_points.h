// Shared by the two routes of the sub-box sums at arbitrary wavevectors (subbox_dft.cu: every box on
// its own; subbox_cells.cu: cell amplitudes shared by the boxes): site constants, phases in cycles.
#pragma once

#include "api_internal.h"

enum { SB_OCC = 0, SB_SPIN = 1, SB_DISP = 2 };

// per-site constants of the sub-box sum (FP64, built on the host)
struct SbSite {
    double r[3];
    double b;
    double coef[9];
    int kind;
    int pad;
};

// Phases are carried in cycles (Q.x / 2 pi) and brought to [-1/2, 1/2] by subtracting the
// nearest integer before the sine and cosine, where the fast FP32 __sincosf / __cosf are
// accurate; FP64 uses sincospi / cospi.
// x minus its nearest integer.  FP32: adding and subtracting 1.5 * 2^23 rounds |x| < 2^22 to
// the nearest integer on the FMA pipe (rintf would take a slot of the SFU/conversion pipe that
// the sine and cosine need); phases here are a few cycles.
__device__ __forceinline__ double frac_w(double x) { return x - rint(x); }
__device__ __forceinline__ float frac_w(float x) {
    const float r = __fsub_rn(__fadd_rn(x, 12582912.0f), 12582912.0f);
    return __fsub_rn(x, r);
}
// cos 2 pi t for a phase t in cycles (reduced to [-1/2, 1/2] first)
__device__ __forceinline__ double cos_cycles(double t) { return cospi(2.0 * frac_w(t)); }
__device__ __forceinline__ float cos_cycles(float t) { return __cosf(frac_w(t) * 6.283185307179586f); }
// (cos 2 pi r, sin 2 pi r) for |r| <= 1/2
__device__ __forceinline__ void sincos_cycles(double r, double &c, double &s) { sincospi(2.0 * r, &s, &c); }
__device__ __forceinline__ void sincos_cycles(float r, float &c, float &s) { __sincosf(r * 6.283185307179586f, &s, &c); }
// S += phi (c + i s) = phi c + (i phi) s: two paired FP32 multiply-adds
__device__ __forceinline__ void cexp_acc(float2 &S, float2 phi, float2 iphi, float c, float s) {
    S = __ffma2_rn(phi, make_float2(c, c), S);
    S = __ffma2_rn(iphi, make_float2(s, s), S);
}
__device__ __forceinline__ void cexp_acc(double2 &S, double2 phi, double2 iphi, double c, double s) {
    S.x = fma(phi.x, c, S.x);
    S.x = fma(iphi.x, s, S.x);
    S.y = fma(phi.y, c, S.y);
    S.y = fma(iphi.y, s, S.y);
}

// the shared-amplitude route (subbox_cells.cu): true when it took the request (its kernels are queued
// on st); false leaves it to the box-by-box kernels.  fill: the share of the resident blocks that their
// launch would keep busy
template <typename T>
bool subbox_cells_run(ds_model *M, int kind, const SbSite *d_sites, const int4 *d_org, long long norigin,
                      const double *d_hkl, long long npts, const ds_opts *o, T *dout, double fill, Scratch &ws, cudaStream_t st);
