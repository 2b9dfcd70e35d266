// Sub-box sums at arbitrary wavevectors from cell amplitudes shared by the boxes (Section V A; the same
// sum as subbox_dft.cu, regrouped).
//
// With many origins a lattice point lies in several boxes: norigin n_sb^3 / (nmodels n1 n2 n3) of them
// on average.  The amplitude of a cell,
//     A_R(Q) = sum_mu phi_mu(Q) a_{R,mu}(Q),   a = delta, M or delta exp(i Q.u),
// carries no box, so it is formed once per cell and point instead of once per box; a box then costs
//     F_o = sum_d1 e1^d1 sum_d2 e2^d2 L_{o + (d1, d2, 0)},   L_R = sum_d3 e3^d3 A_{R + (0, 0, d3)},
// e_a = exp(2 pi i h_a), with cells wrapped and phases not (open boxes).  With tabulated powers the line
// sums of the ring leave out the phase e3^(nsb - 1), common to every box of a point.  The line sums L are formed as
// the cells of a row are walked (the last eight amplitudes stay in registers), so a box reads n_sb^2
// values per point.  For displacements the bound moves from one SFU (sin, cos) pair per atom and box to
// one per atom, plus the L2 traffic of the line sums.
//
// Points are taken in chunks whose line sums stay in the L2 (SX_L2 bytes), one point per thread: the
// loads and stores of a warp are 32 consecutive points.  Per chunk: line sums (grid: points x rows of
// cells), the Debye-Waller means from the same exponentials (DIFFUSE displacements), the boxes (grid:
// points x origin chunks).  Partial sums are added in a fixed order.
//
// fcc 32^3 (131,072 atoms), 2516 origins, n_sb = 5, 40,401 points, FP32: 10.5 ms (29.5 ms box by box, at
// 0.75 of the SFU rate); per chunk of 256 points, cold caches, the line sums take 35.5 us (instruction issue
// 72 %, 96 registers, five CTAs per SM), the mean 6.5, the boxes 26.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>

#include "api_internal.h"
#include "subbox_points.h"

using namespace ds;

namespace {

constexpr int SX_T = 128;                     // points per block
constexpr size_t SX_L2 = 64u << 20;           // line sums of a chunk
constexpr size_t SX_MOST = 1024u << 20;       // and at most, for one block of points over large ensembles
constexpr long long SX_PREP = 65536;          // points whose constants are held at once
constexpr int SX_RING = 8;                    // amplitudes of a row kept in registers

// FP32 displacements take tabulated powers of the cell phases, each formed in FP64 and rounded once: powers of a rounded
// phase drift by a rounding per cell (2.5e-7 of the result against 1.0e-7, boxes of 5^3, TOTAL), which the box-by-box
// kernel's per-atom phases do not.  Its occupancies and moments advance a rounded phase too, as here.
template <typename T, int KIND> constexpr bool sx_tab() { return sizeof(T) == 4 && KIND == SB_DISP; }

template <typename T> struct SxParams {
    int nsite, nsb, n1, n2, n3, ncell, nmodels, diffuse;
    const SbSite *site;
    const uint8_t *occ;
    const float *vec;
    const double *mean;
    const double *hkl;
    long long npts;                 // points of the request
    long long p0, np;               // points whose constants are held: [p0, p0 + np)
    long long q0;                   // first of them in this chunk, relative to p0
    int nq, ld;                     // points of the chunk, and padded to whole blocks
    long long ldp;                  // stride of the constants
    double recip[9];
    c_t<T> *phi;                    // [site][ldp]: phi_mu
    c_t<T> *e;                      // [axis][u][ldp]: e_axis^u for u < 8, e_axis^8
    T *Q;                           // [axis][ldp]: Q / 2 pi (cycles per A) for displacements, Q for moments
    double2 *phiB;                  // displacements: [site][ldp]: phi_mu exp(2 pi i off) times the box sum of exp(2 pi i Q.d)
    T off, off_c, off_s;            // displacements: phase added to every Q.u (cycles), its cosine and sine
    c_t<T> *K;                      // occupancies, moments: mean amplitude [comp][ldp]
    c_t<T> *A, *L;                  // [comp][model cell][ld]; A: amplitudes where the line sums take their own pass
    T *dwp;                         // [row block][site][ld]: sums of w cos(Q.u)
    c_t<T> *KB;                     // [ld]: the mean amplitude of a box
    int rows_per, nrb;              // rows of cells per block, row blocks
    const int4 *origins;
    long long norigin, per_chunk;
    T *partial;                     // [origin chunk][npts]
};

// per-point constants (FP64, stored in the working type)
template <typename T, int KIND> __global__ void __launch_bounds__(SX_T) k_sx_prep(const __grid_constant__ SxParams<T> p) {
    const long long j = (long long)blockIdx.x * SX_T + threadIdx.x;
    if (j >= p.ldp) return;
    const long long q = p.p0 + min(j, p.np - 1);   // padding repeats the last point
    const double h[3] = {p.hkl[3 * q], p.hkl[3 * q + 1], p.hkl[3 * q + 2]};
    double Qd[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        Qd[a] = h[0] * p.recip[a] + h[1] * p.recip[3 + a] + h[2] * p.recip[6 + a];
        p.Q[a * p.ldp + j] = (T)(KIND == SB_DISP ? Qd[a] / TWO_PI_D : Qd[a]);
    }
    const double s2 = (Qd[0] * Qd[0] + Qd[1] * Qd[1] + Qd[2] * Qd[2]) / (FOUR_PI_D * FOUR_PI_D);
    double Br = 1.0, Bi = 0.0, lr = 1.0, li = 0.0;   // (lr, li): what the line sums leave out, e_3^-(nsb - 1)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double sn, cs;
        sincospi(2.0 * frac_w(h[a]), &sn, &cs);
        double xr = 1.0, xi = 0.0, sr = 0.0, si = 0.0;   // sum_d e^d
        for (int d = 0; d < max(p.nsb, SX_RING + 1); ++d) {
            if (d <= SX_RING) p.e[(a * (SX_RING + 1) + d) * p.ldp + j] = mk<T>((T)xr, (T)xi);
            if (d < p.nsb) sr += xr, si += xi;
            if (sx_tab<T, KIND>() && a == 2 && d == p.nsb - 1 && p.nsb <= SX_RING) lr = xr, li = -xi;
            const double t = xr * cs - xi * sn;
            xi = xr * sn + xi * cs;
            xr = t;
        }
        const double t = Br * sr - Bi * si;
        Bi = Br * si + Bi * sr;
        Br = t;
    }
    {
        const double t = Br * lr - Bi * li;
        Bi = Br * li + Bi * lr;
        Br = t;
    }
    constexpr int NC = KIND == SB_SPIN ? 3 : 1;
    double Kr[NC], Ki[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) Kr[c] = Ki[c] = 0.0;
    for (int s = 0; s < p.nsite; ++s) {
        const SbSite &S = p.site[s];
        const double f = S.b * form_factor<double>(S.kind, S.coef, s2);
        const double t = frac_w(h[0] * S.r[0] + h[1] * S.r[1] + h[2] * S.r[2]);
        double sn, cs;
        sincospi(2.0 * t, &sn, &cs);
        p.phi[s * p.ldp + j] = mk<T>((T)(f * cs), (T)(f * sn));
        if (KIND == SB_DISP) sincospi(2.0 * (t + (double)p.off), &sn, &cs);
        if (KIND == SB_DISP && p.diffuse) p.phiB[s * p.ldp + j] = make_double2(f * cs * Br - f * sn * Bi, f * cs * Bi + f * sn * Br);
        if (KIND != SB_DISP && p.diffuse) {
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const double m = p.mean[KIND == SB_SPIN ? 3 * s + c : s];
                Kr[c] += f * cs * m;
                Ki[c] += f * sn * m;
            }
        }
    }
    if (KIND != SB_DISP)
#pragma unroll
        for (int c = 0; c < NC; ++c) p.K[c * p.ldp + j] = mk<T>((T)Kr[c], (T)Ki[c]);
}

// x e + a for complex x, e, a
template <typename C> __device__ __forceinline__ C cmad(C x, C e, C a) {
    C r;
    r.x = fma(x.x, e.x, fma(-x.y, e.y, a.x));
    r.y = fma(x.x, e.y, fma(x.y, e.x, a.y));
    return r;
}

// Line sums (LINE) or plain amplitudes of whole rows of cells.  The row loop is unrolled by the ring
// length, so the ring is indexed by constants.  Displacements: an atom costs three multiply-adds, one
// reduction, one (sin, cos) pair, the product with its site's factor (four multiply-adds; formed in FP64
// and rounded once, as box by box) and two adds into its site's sum, the Debye-Waller mean.
// DIFFUSE FP32 requests add the phase off = 1/16 cycle to every atom: the fast sine falls short by about
// 1.2e-7 on either side of the multiples of a quarter, 6e-7 of sin(Q.u) where |Q.u| stays below 0.3, and what
// is left of an intensity without its mean is sin(Q.u) (4.3e-7 of it without the phase, boxes of 2^3).  At 1/16
// the error has no slope.  The phase is common to F and K B.  TOTAL needs none: cosines near 1 are exact.  WGT:
// occupancies weight the displaced atoms.  GUARD: the sites beyond nsite are left out at run time (where a
// site is dear: sines and cosines, FP64); without it they are atoms of weight zero.
template <typename T, int KIND, int MAXS, bool LINE, bool WGT, bool GUARD>
__global__ void __launch_bounds__(SX_T, KIND == SB_SPIN ? 4 : (sizeof(T) == 8 ? (KIND == SB_DISP && MAXS > 8 ? 2 : 4) : (MAXS <= 4 ? (KIND == SB_DISP ? 5 : 8) : 4))) k_sx_rows(const __grid_constant__ SxParams<T> p) {
    using C = c_t<T>;
    constexpr int NC = KIND == SB_SPIN ? 3 : 1;
    extern __shared__ __align__(16) unsigned char sx_raw[];
    const int nsite = p.nsite, nsb = p.nsb, n3 = p.n3, tid = threadIdx.x;
    float4 *atoms = (float4 *)sx_raw;                        // [n3][MAXS]
    C *first = (C *)(sx_raw + sizeof(float4) * n3 * MAXS) + tid;   // LINE: [i][comp][SX_T], a row's first amplitudes
    const int ql = blockIdx.x * SX_T + tid;
    const long long j = p.q0 + ql;                     // < ldp: chunks are whole blocks
    C phi[MAXS];
    C wsum[KIND == SB_DISP ? MAXS : 1];
#pragma unroll
    for (int s = 0; s < MAXS; ++s) {
        phi[s] = s < nsite ? p.phi[s * p.ldp + j] : mk<T>(T(0), T(0));
        if (KIND == SB_DISP) wsum[KIND == SB_DISP ? s : 0] = mk<T>(T(0), T(0));
    }
    constexpr bool TAB = sx_tab<T, KIND>();
    const C e3 = p.e[(2 * (SX_RING + 1) + 1) * p.ldp + j];
    C q3[TAB ? SX_RING : 1];   // e_3^-i of the ring
    if (LINE && TAB) {
#pragma unroll
        for (int i = 0; i < SX_RING; ++i) {
            C q = i < nsb ? p.e[(2 * (SX_RING + 1) + i) * p.ldp + j] : mk<T>(T(0), T(0));
            q.y = -q.y;
            q3[TAB ? i : 0] = q;
        }
    }
    T Qx = T(0), Qy = T(0), Qz = T(0);
    C K[NC];
    if (KIND == SB_DISP) {
        Qx = p.Q[j], Qy = p.Q[p.ldp + j], Qz = p.Q[2 * p.ldp + j];
    } else {
#pragma unroll
        for (int c = 0; c < NC; ++c) K[c] = p.K[c * p.ldp + j];
    }
    const int nrow = p.nmodels * p.n1 * p.n2;
    const int row_lo = blockIdx.y * p.rows_per, row_hi = min(nrow, row_lo + p.rows_per);
    const size_t cstride = (size_t)p.nmodels * p.ncell * p.ld;
    for (int row = row_lo; row < row_hi; ++row) {
        const int m = row / (p.n1 * p.n2), rr = row - m * p.n1 * p.n2;
        __syncthreads();
        for (int i = tid; i < n3 * MAXS; i += SX_T) {
            const int s = i / n3, r3 = i - s * n3;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (s < nsite) {
                const size_t at = ((size_t)m * nsite + s) * p.ncell + (size_t)rr * n3 + r3;
                if (KIND == SB_OCC) v.x = (float)p.occ[at];
                else v = make_float4(p.vec[3 * at], p.vec[3 * at + 1], p.vec[3 * at + 2], WGT ? (float)p.occ[at] : 1.f);
            }
            atoms[r3 * MAXS + s] = v;
        }
        __syncthreads();
        C h[NC][SX_RING];
        C *dst = (LINE ? p.L : p.A) + ((size_t)row * n3) * p.ld + ql;
        const int npos = LINE ? n3 + nsb - 1 : n3;
        // STEADY: every cell of the group is on the row and ends a box line
        auto group = [&](int r0, auto steady) {
            constexpr bool STEADY = decltype(steady)::value;
            C *d0 = dst + (ptrdiff_t)(LINE ? r0 - nsb + 1 : r0) * p.ld;
#pragma unroll
            for (int u = 0; u < SX_RING; ++u) {
                const int r = r0 + u;
                if (!STEADY && r >= npos) break;
                C a[NC];
                if (STEADY || r < n3) {
                    const float4 *at = atoms + r * MAXS;
                    if (KIND == SB_DISP) {
                        a[0] = mk<T>(T(0), T(0));
#pragma unroll
                        for (int s = 0; s < MAXS; ++s) {
                            if (GUARD && s >= nsite) break;
                            const float4 v = at[s];
                            const T t = fma(Qx, (T)v.x, fma(Qy, (T)v.y, fma(Qz, (T)v.z, p.off)));
                            T cs, sn;
                            sincos_cycles(frac_w(t), cs, sn);
                            if (WGT) {
                                cs *= (T)v.w;
                                sn *= (T)v.w;
                            }
                            C &ws = wsum[KIND == SB_DISP ? s : 0];
                            ws.x += cs;
                            ws.y += sn;
                            a[0] = cmad(phi[s], mk<T>(cs, sn), a[0]);
                        }
                    } else {
#pragma unroll
                        for (int c = 0; c < NC; ++c) a[c] = mk<T>(-K[c].x, -K[c].y);
#pragma unroll
                        for (int s = 0; s < MAXS; ++s) {
                            if (GUARD && s >= nsite) break;
                            const float4 v = at[s];
                            const T x[3] = {(T)v.x, (T)v.y, (T)v.z};
#pragma unroll
                            for (int c = 0; c < NC; ++c) {
                                a[c].x = fma(phi[s].x, x[c], a[c].x);
                                a[c].y = fma(phi[s].y, x[c], a[c].y);
                            }
                        }
                    }
                    if (LINE && !STEADY && r < nsb - 1)
#pragma unroll
                        for (int c = 0; c < NC; ++c) first[(r * NC + c) * SX_T] = a[c];
                } else {
                    // the row wraps: its first amplitudes again
#pragma unroll
                    for (int c = 0; c < NC; ++c) a[c] = first[((r - n3) * NC + c) * SX_T];
                }
                if (LINE) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) h[c][u] = a[c];
                }
                if (!LINE || STEADY || r >= nsb - 1) {
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        C l = a[c];
                        if (LINE) {
#pragma unroll
                            for (int i = 1; i < SX_RING; ++i) {
                                if (i >= nsb) break;
                                const C hv = h[c][(u - i + SX_RING) % SX_RING];
                                l = TAB ? cmad(q3[TAB ? i : 0], hv, l) : cmad(l, e3, hv);
                            }
                        }
                        d0[c * cstride + (ptrdiff_t)u * p.ld] = l;
                    }
                }
            }
        };
        for (int r0 = 0; r0 < npos; r0 += SX_RING) {
            if (r0 >= SX_RING && r0 + SX_RING <= n3) group(r0, std::true_type{});
            else group(r0, std::false_type{});
        }
    }
    if (KIND == SB_DISP && p.diffuse) {
        // sum of w cos(Q.u) = Re[exp(-2 pi i off) sum of w exp(i Q.u + 2 pi i off)]
#pragma unroll
        for (int s = 0; s < MAXS; ++s)
            if (s < nsite) {
                const C ws = wsum[KIND == SB_DISP ? s : 0];
                p.dwp[((size_t)blockIdx.y * nsite + s) * p.ld + ql] = fma(ws.x, p.off_c, ws.y * p.off_s);
            }
    }
}

// line sums of boxes wider than the register ring, from the amplitudes
template <typename T, bool TAB> __global__ void __launch_bounds__(SX_T) k_sx_line(const __grid_constant__ SxParams<T> p, int nc) {
    using C = c_t<T>;
    const int ql = blockIdx.x * SX_T + threadIdx.x;
    const C e3 = p.e[(2 * (SX_RING + 1) + 1) * p.ldp + p.q0 + ql];
    C pw[SX_RING + 1];   // e_3^u
#pragma unroll
    for (int u = 0; u <= SX_RING; ++u) pw[u] = !TAB ? e3 : p.e[(2 * (SX_RING + 1) + u) * p.ldp + p.q0 + ql];
    const size_t cells = (size_t)p.nmodels * p.ncell;
    for (size_t i = blockIdx.y; i < cells * nc; i += gridDim.y) {
        const size_t row = i / p.n3;
        const int r3 = (int)(i - row * p.n3);
        const C *a = p.A + row * p.n3 * p.ld + ql;
        C l = mk<T>(T(0), T(0));
        if (TAB) {
            for (int d0 = (p.nsb - 1) / SX_RING * SX_RING; d0 >= 0; d0 -= SX_RING) {
                l = cmul(l, pw[SX_RING]);
#pragma unroll
                for (int u = 0; u < SX_RING; ++u) {
                    if (d0 + u >= p.nsb) break;
                    int w = r3 + d0 + u;
                    if (w >= p.n3) w -= p.n3;
                    l = cmad(pw[u], a[(size_t)w * p.ld], l);
                }
            }
        } else {
            for (int d = p.nsb - 1; d >= 0; --d) {
                int w = r3 + d;
                if (w >= p.n3) w -= p.n3;
                l = cmad(l, e3, a[(size_t)w * p.ld]);
            }
        }
        p.L[i * p.ld + ql] = l;
    }
}

// K B of the chunk's points, K = sum_mu phi_mu <w cos(Q.u)>_mu: the row blocks' sums by slices of 8 points and 128
// threads each, in a fixed order; K B in FP64, rounded once (it cancels against F at Bragg positions)
constexpr int SX_MP = 8, SX_MG = 128;
template <typename T> __global__ void __launch_bounds__(SX_MP * SX_MG) k_sx_mean(const __grid_constant__ SxParams<T> p) {
    __shared__ T red[SX_MG / 4][SX_MP + 1];
    __shared__ double2 term[MAX_SITES][SX_MP];
    const int tx = threadIdx.x % SX_MP, g = threadIdx.x / SX_MP, nsite = p.nsite;
    const int nsl = (SX_MG / nsite) & ~3, s = g / nsl, sl = g - s * nsl;   // slices of a site, the thread's site and slice
    const int ql = blockIdx.x * SX_MP + tx;
    double2 pb = make_double2(0.0, 0.0);
    if (g < nsite) pb = p.phiB[g * p.ldp + p.q0 + ql];
    T t = T(0);
    if (s < nsite) {
        const T *q = p.dwp + ((size_t)sl * nsite + s) * p.ld + ql;
        const size_t step = (size_t)nsl * nsite * p.ld;
        constexpr int NL = 16;   // loads in flight
        for (int b = sl; b < p.nrb; b += NL * nsl, q += NL * step) {
            T v[NL];
#pragma unroll
            for (int u = 0; u < NL; ++u) v[u] = b + u * nsl < p.nrb ? q[u * step] : T(0);
#pragma unroll
            for (int u = 0; u < NL; ++u) t += v[u];
        }
    }
    t += __shfl_xor_sync(0xffffffffu, t, SX_MP);   // the four slices of a warp are of one site
    t += __shfl_xor_sync(0xffffffffu, t, 2 * SX_MP);
    if (g % 4 == 0) red[g / 4][tx] = t;
    __syncthreads();
    if (g < nsite) {
        T sum = T(0);
        for (int i = 0; i < nsl / 4; ++i) sum += red[g * (nsl / 4) + i][tx];
        const double w = (double)(sum / (T)((double)p.nmodels * p.ncell));
        term[g][tx] = make_double2(pb.x * w, pb.y * w);
    }
    __syncthreads();
    if (g == 0) {
        double kr = 0.0, ki = 0.0;
        for (int i = 0; i < nsite; ++i) kr += term[i][tx].x, ki += term[i][tx].y;
        p.KB[ql] = mk<T>((T)kr, (T)ki);
    }
}

// The boxes: sums over the line sums of a box's rows, eight loads in flight per thread; the element
// offsets of each origin's wrapped rows are tabulated once per block.
template <typename T, int KIND>
__global__ void __launch_bounds__(SX_T) k_sx_boxes(const __grid_constant__ SxParams<T> p) {
    using C = c_t<T>;
    constexpr int NC = KIND == SB_SPIN ? 3 : 1;
    constexpr int NB = SX_RING;
    extern __shared__ __align__(16) unsigned char sx_raw[];
    constexpr bool TAB = sx_tab<T, KIND>();
    C *pw1 = (C *)sx_raw + threadIdx.x;             // TAB: [u][SX_T], e_1^u
    int *off1 = (int *)((C *)sx_raw + (TAB ? SX_RING * SX_T : 0));   // [origin][nsb]: element offset of (model, o1 + d1, 0, o3)
    int *off2 = off1 + p.per_chunk * p.nsb;         // [origin][nsb]: of row o2 + d2 within a plane
    const int nsb = p.nsb;
    const int ql = blockIdx.x * SX_T + threadIdx.x;
    const long long j = p.q0 + ql;
    const long long o0 = (long long)blockIdx.y * p.per_chunk;
    const int no = (int)(min(p.norigin, o0 + p.per_chunk) - o0);
    for (int i = threadIdx.x; i < no * nsb; i += SX_T) {
        const int oi = i / nsb, d = i - oi * nsb;
        const int4 og = p.origins[o0 + oi];
        int w1 = og.y + d, w2 = og.z + d;   // o < n and d < n_sb <= n
        if (w1 >= p.n1) w1 -= p.n1;
        if (w2 >= p.n2) w2 -= p.n2;
        off1[i] = ((og.x * p.n1 + w1) * p.n2 * p.n3 + og.w) * p.ld;
        off2[i] = w2 * p.n3 * p.ld;
    }
    // e_2^u below the box's width, and the eighth powers of wider boxes
    const C e1 = p.e[p.ldp + j], e2 = p.e[(SX_RING + 2) * p.ldp + j];
    C pw[NB], e1n = mk<T>(T(1), T(0)), e2n = e1n;
    pw[0] = e1n;
#pragma unroll
    for (int u = 1; u < NB; ++u) {
        if (!TAB) pw[u] = cmul(pw[u - 1], e2);
        else pw[u] = u < nsb ? p.e[(SX_RING + 1 + u) * p.ldp + j] : pw[0];
    }
    if (TAB) {
#pragma unroll
        for (int u = 0; u < NB; ++u)
            if (u < nsb) pw1[u * SX_T] = p.e[u * p.ldp + j];
        if (nsb > NB) e1n = p.e[SX_RING * p.ldp + j], e2n = p.e[(2 * SX_RING + 1) * p.ldp + j];
    } else {
        e2n = cmul(pw[NB - 1], e2);
    }
    C KB = mk<T>(T(0), T(0));
    if (KIND == SB_DISP && p.diffuse) KB = p.KB[ql];
    T Qv[3] = {T(0), T(0), T(0)};
    if (KIND == SB_SPIN)
#pragma unroll
        for (int a = 0; a < 3; ++a) Qv[a] = p.Q[a * p.ldp + j];
    const size_t cstride = (size_t)p.nmodels * p.ncell * p.ld;
    const C *L = p.L + ql;
    __syncthreads();
    T acc = T(0);
    for (int oi = 0; oi < no; ++oi) {
        C F[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) F[c] = mk<T>(T(0), T(0));
        for (int d1 = nsb - 1; d1 >= 0; --d1) {
            if (TAB && d1 % SX_RING == SX_RING - 1 && d1 < nsb - 1) {
#pragma unroll
                for (int c = 0; c < NC; ++c) F[c] = cmul(F[c], e1n);
            }
            const C *pl = L + off1[oi * nsb + d1];
            C G[NC];
#pragma unroll
            for (int c = 0; c < NC; ++c) G[c] = mk<T>(T(0), T(0));
            for (int t0 = (nsb - 1) / NB * NB; t0 >= 0; t0 -= NB) {
                const int *o2 = off2 + oi * nsb + t0;
                const int nt = nsb - t0;
                C v[NB][NC];
#pragma unroll
                for (int u = 0; u < NB; ++u) {
                    if (u >= nt) break;
                    const C *at = pl + o2[u];
#pragma unroll
                    for (int c = 0; c < NC; ++c) v[u][c] = at[c * cstride];
                }
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    if (NB < nsb) G[c] = cmul(G[c], e2n);
                    G[c] = cadd(G[c], v[0][c]);
                }
#pragma unroll
                for (int u = 1; u < NB; ++u) {
                    if (u >= nt) break;
#pragma unroll
                    for (int c = 0; c < NC; ++c) cfma(G[c], pw[u], v[u][c]);
                }
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) F[c] = TAB ? cmad(pw1[(d1 % SX_RING) * SX_T], G[c], F[c]) : cmad(F[c], e1, G[c]);
        }
        T tot = T(0);
        if (KIND == SB_DISP) F[0] = csub(F[0], KB);
#pragma unroll
        for (int c = 0; c < NC; ++c) tot += F[c].x * F[c].x + F[c].y * F[c].y;
        if (KIND == SB_SPIN) {
            const T q2 = Qv[0] * Qv[0] + Qv[1] * Qv[1] + Qv[2] * Qv[2];
            if (q2 > T(0)) {
                const T pr = Qv[0] * F[0].x + Qv[1] * F[1].x + Qv[2] * F[2].x;
                const T pi = Qv[0] * F[0].y + Qv[1] * F[1].y + Qv[2] * F[2].y;
                tot -= (pr * pr + pi * pi) / q2;
            } else {
                tot *= T(2) / T(3);
            }
        }
        acc += tot;
    }
    if (ql < p.nq) p.partial[(size_t)blockIdx.y * p.npts + p.p0 + j] = acc;
}

template <typename T>
__global__ void k_sx_sum(const T *__restrict__ partial, long long npts, int nchunk, double norm, T *__restrict__ out) {
    for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < npts; q += (long long)gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int c = 0; c < nchunk; ++c) s += (double)partial[(size_t)c * npts + q];
        out[q] = (T)(s * norm);
    }
}

template <typename T, int KIND, bool LINE, bool WGT> void launch_rows(const SxParams<T> &p, const dim3 &grid, cudaStream_t st) {
    auto go = [&](auto kern, int maxs) {
        // atoms of a row (<= 32 KB: n3 <= 128, nsite <= 16) and, for line sums, its first amplitudes
        const size_t sm = sizeof(float4) * p.n3 * maxs +
                          (LINE ? sizeof(c_t<T>) * (p.nsb - 1) * (KIND == SB_SPIN ? 3 : 1) * SX_T : 0);
        allow_smem(kern, sm);
        kern<<<grid, SX_T, sm, st>>>(p);
        count_launches(1);
    };
    const int ns = p.nsite;
    if constexpr (sizeof(T) == 4 && KIND == SB_DISP) {
        // the SFU-bound case: instances of exactly nsite sites up to eight
        if constexpr (LINE) {
            switch (ns) {
            case 1: return go(k_sx_rows<T, KIND, 1, LINE, WGT, false>, 1);
            case 2: return go(k_sx_rows<T, KIND, 2, LINE, WGT, false>, 2);
            case 3: return go(k_sx_rows<T, KIND, 3, LINE, WGT, false>, 3);
            case 4: return go(k_sx_rows<T, KIND, 4, LINE, WGT, false>, 4);
            case 5: return go(k_sx_rows<T, KIND, 5, LINE, WGT, false>, 5);
            case 6: return go(k_sx_rows<T, KIND, 6, LINE, WGT, false>, 6);
            case 7: return go(k_sx_rows<T, KIND, 7, LINE, WGT, false>, 7);
            case 8: return go(k_sx_rows<T, KIND, 8, LINE, WGT, false>, 8);
            default: break;
            }
        }
        ns == 16 ? go(k_sx_rows<T, KIND, 16, LINE, WGT, false>, 16) : go(k_sx_rows<T, KIND, 16, LINE, WGT, true>, 16);
    } else {
        // FP64 sums of occupancies and displacements leave idle sites out; moments (bound by the latency of
        // their three rings) and FP32 occupancies run faster with idle sites of weight zero
        constexpr bool G = sizeof(T) == 8 && KIND != SB_SPIN;
        if constexpr (LINE || !G)
            if (ns <= 4) return go(k_sx_rows<T, KIND, 4, LINE, WGT, G>, 4);
        if constexpr (LINE) {
            if (ns <= 8) return go(k_sx_rows<T, KIND, 8, LINE, WGT, G>, 8);
        } else if (G && ns == 16) {
            return go(k_sx_rows<T, KIND, 16, LINE, WGT, false>, 16);
        }
        go(k_sx_rows<T, KIND, 16, LINE, WGT, G>, 16);
    }
}
template <typename T, int KIND> void launch_rows(const SxParams<T> &p, bool line, const dim3 &grid, cudaStream_t st) {
    if constexpr (KIND == SB_DISP) {
        if (p.occ) return line ? launch_rows<T, KIND, true, true>(p, grid, st) : launch_rows<T, KIND, false, true>(p, grid, st);
    }
    return line ? launch_rows<T, KIND, true, false>(p, grid, st) : launch_rows<T, KIND, false, false>(p, grid, st);
}

template <typename T, int KIND> void run_kind(SxParams<T> p, double norm, int chunk_q, int nochunk, T *dout, cudaStream_t st) {
    using C = c_t<T>;
    constexpr int NC = KIND == SB_SPIN ? 3 : 1;
    const bool line = p.nsb <= SX_RING;
    for (p.p0 = 0; p.p0 < p.npts; p.p0 += SX_PREP) {
        p.np = std::min<long long>(SX_PREP, p.npts - p.p0);
        k_sx_prep<T, KIND><<<(unsigned)((p.ldp + SX_T - 1) / SX_T), SX_T, 0, st>>>(p);
        count_launches(1);
        for (p.q0 = 0; p.q0 < p.np; p.q0 += chunk_q) {
            p.nq = (int)std::min<long long>(chunk_q, p.np - p.q0);
            const unsigned qb = (unsigned)((p.nq + SX_T - 1) / SX_T);
            const dim3 rows(qb, (unsigned)p.nrb);
            launch_rows<T, KIND>(p, line, rows, st);
            if (!line) {
                const size_t lines = (size_t)p.nmodels * p.ncell * NC;
                k_sx_line<T, sx_tab<T, KIND>()><<<dim3(qb, (unsigned)std::min<size_t>(lines, 16384)), SX_T, 0, st>>>(p, NC);
                count_launches(1);
            }
            if (KIND == SB_DISP && p.diffuse) {
                k_sx_mean<T><<<qb * (SX_T / SX_MP), SX_MP * SX_MG, 0, st>>>(p);
                count_launches(1);
            }
            k_sx_boxes<T, KIND><<<dim3(qb, (unsigned)nochunk), SX_T,
                                    (sx_tab<T, KIND>() ? sizeof(C) * SX_RING * SX_T : 0) + sizeof(int) * 2 * p.per_chunk * p.nsb, st>>>(p);
            count_launches(1);
        }
    }
    const unsigned nb = (unsigned)std::max<long long>(1, std::min<long long>((p.npts + 255) / 256, 152 * 8));
    k_sx_sum<T><<<nb, 256, 0, st>>>(p.partial, p.npts, nochunk, norm, dout);
    count_launches(1);
}

// Rule: the cheaper route by a cost model, picoseconds per point, of both routes measured on GB300 in both
// precisions (768 pairs of times: 20^3 to 64^3 cells, 1 to 16 sites, boxes of 2^3 to 10^3 cells, 0.5 to 8
// boxes per cell; 22,500 points in FP32, 2,500 in FP64).  Box by box: a term per cell of a box, and the
// Debye-Waller pass of DIFFUSE displacements.  Shared: a term per cell, which grows with the box's width
// (the ring of the line sums; amplitudes written and read again where the ring is too short) and with
// the sites that are evaluated (FP64 moments: whole instances), and one per line sum read.
// Few points leave the box-by-box launch short of blocks (fill < 1; measured for FP32 occupancies and moments:
// 16^3 cells, six spins, 33 boxes of 8^3, 3600 points, fill 0.14: 1.00 box by box, 0.35 ms shared).
// The line lies where the two are equal, 20^3 cells, n_sb = 5, four sites, box by box and shared: FP32
// displacements 2.23 and 1.38 ms at 4 boxes per cell; occupancies 0.54 and 0.77 ms at 1.6, 1.17 and 0.85 at
// 4; FP64 displacements 14.0 and 7.8 ms at 0.6; occupancies 0.91 and 1.30 ms at 0.6, 1.71 and 1.34 at 1.6.
// Where the rule shares, sharing was at most 8 % slower than box by box at any overlap between the measured
// ones, and at most 3 % in 270 random requests.  From 48^3 cells on the line sums of one block of points
// exceed the L2; sharing gains there too (FP32, 64^3, four displaced sites, 2.5 boxes per cell, 1600 points:
// 7.5 and 2.5 ms).
bool cells_cheaper(bool fp64, int kind, bool diffuse, int nsite, int nsb, double cells, double norigin, double fill) {
    const int NC = kind == SB_SPIN ? 3 : 1;
    const double ns = nsite, w = nsb;
    const bool wide = nsb > SX_RING;
    double box_cell, cell, line, dw = 0.0;
    if (!fp64) {
        line = kind == SB_SPIN ? 3.3 : 0.9;
        if (kind == SB_DISP) box_cell = 0.4 + 0.5 * ns, cell = 3.8 + 0.5 * ns + 0.15 * std::max(0.0, ns - 6) + 0.1 * std::max(0.0, w - 5), dw = 0.48 * ns;
        else if (kind == SB_OCC) box_cell = 0.9 + 0.145 * ns, cell = 2.2 + 0.28 * ns + 0.7 * std::max(0.0, w - 5);
        else box_cell = 1.6 + 0.36 * ns, cell = 8.8 + 0.35 * ns + 0.55 * w;
        if (wide) {
            line = 0.9 * NC;
            cell = (kind == SB_DISP ? 3.8 + 0.5 * ns : (kind == SB_OCC ? 2.2 + 0.28 * ns : 4.5 + 0.97 * ns)) + 2.3 * NC * w;
        }
    } else {
        const double pad = nsite <= 4 ? 4 : (nsite <= 8 ? 8 : 16);
        if (kind == SB_DISP) box_cell = 50 + 60 * ns, cell = 6 + 85 * ns + (wide ? 9.5 : 7.2) * w, line = 13, dw = 150 * ns;
        else if (kind == SB_OCC) box_cell = 40 + 7 * ns, cell = 12 + 6.7 * ns + (wide ? 9.4 : 7.1) * w, line = 12;
        else box_cell = 30 + 22 * ns, cell = wide ? 30 + 13 * pad + 33 * w : 100 + 15 * pad + 27 * w, line = 40;
        if (wide) line = NC;
    }
    double by_box = norigin * w * w * w * box_cell + (diffuse ? dw * cells : 0.0);
    if (!fp64 && kind != SB_DISP) by_box += 2.3 * norigin;   // per box
    if (!fp64 && kind != SB_DISP) by_box *= std::pow(fill, -0.25);
    return cells * cell + norigin * w * w * line <= 0.95 * by_box;
}

}  // namespace

template <typename T>
bool subbox_cells_run(ds_model *M, int kind, const SbSite *d_sites, const int4 *d_org, long long norigin,
                      const double *d_hkl, long long npts, const ds_opts *o, T *dout, double fill, Scratch &ws, cudaStream_t st) {
    using C = c_t<T>;
    ds_ctx *ctx = M->ctx;
    const int nsb = o->subbox_n, nsite = M->nsite, NC = kind == SB_SPIN ? 3 : 1;
    const double cells = (double)M->nmodels * M->n[0] * M->n[1] * M->n[2];
    if (!cells_cheaper(sizeof(T) == 8, kind, o->mode == DS_DIFFUSE, nsite, nsb, cells, (double)norigin, fill)) return false;
    // points per chunk: line sums (and amplitudes, for boxes wider than the ring) within SX_L2
    const size_t per_q = (size_t)cells * NC * sizeof(C) * (nsb > SX_RING ? 2 : 1);
    long long blocks = std::max<long long>(1, (long long)(SX_L2 / (per_q * SX_T)));
    blocks = std::min<long long>(blocks, (std::min<long long>(npts, SX_PREP) + SX_T - 1) / SX_T);
    const int chunk_q = (int)blocks * SX_T;
    if ((size_t)chunk_q * per_q > SX_MOST) return false;
    SxParams<T> p;
    memset(&p, 0, sizeof(p));
    p.nsite = nsite;
    p.nsb = nsb;
    p.n1 = M->n[0];
    p.n2 = M->n[1];
    p.n3 = M->n[2];
    p.ncell = p.n1 * p.n2 * p.n3;
    p.nmodels = M->nmodels;
    p.diffuse = o->mode == DS_DIFFUSE;
    p.site = d_sites;
    p.occ = (kind == SB_OCC || (kind == SB_DISP && M->has_occ)) ? M->d_occ : nullptr;
    p.vec = kind == SB_SPIN ? M->d_spins : M->d_disp;
    p.mean = kind == SB_OCC ? (M->user_mean ? M->d_user_mean : M->d_mean_occ) : M->d_mean_spin;
    p.hkl = d_hkl;
    p.npts = npts;
    p.ld = chunk_q;
    // a chunk's last block may reach past the held points: the constants are padded by one chunk
    p.ldp = (std::min<long long>(npts, SX_PREP) + chunk_q - 1) / chunk_q * chunk_q;
    p.origins = d_org;
    p.norigin = norigin;
    for (int i = 0; i < 9; ++i) p.recip[i] = M->recip[i];
    p.off = sizeof(T) == 4 && p.diffuse ? T(0.0625) : T(0);
    p.off_c = (T)std::cos(TWO_PI_D * p.off);
    p.off_s = (T)std::sin(TWO_PI_D * p.off);
    // row blocks: about eight blocks per SM
    const long long nrow = (long long)p.nmodels * p.n1 * p.n2;
    const long long want = std::max<long long>(1, 152 * 8 / blocks);
    p.rows_per = (int)std::max<long long>(1, (nrow + want - 1) / want);
    if (nrow > (1LL << 31) - 1 || (nrow + p.rows_per - 1) / p.rows_per > 65535) return false;
    p.nrb = (int)((nrow + p.rows_per - 1) / p.rows_per);
    // origins per block: about eight blocks per SM, their row offsets within 32 KB of shared memory
    p.per_chunk = std::min<long long>(std::max<long long>(1, (norigin + want - 1) / want), 4096 / nsb);
    if ((norigin + p.per_chunk - 1) / p.per_chunk > 65535) return false;
    const int nochunk = (int)((norigin + p.per_chunk - 1) / p.per_chunk);
    // one block, so that nothing is held when it cannot be had: the box-by-box route needs less
    const size_t nk = (size_t)p.ldp;
    const bool mean_b = kind == SB_DISP && p.diffuse;
    size_t need = 0;
    std::vector<std::pair<void **, size_t>> parts;   // (pointer, offset)
    auto part = [&](auto *&ptr, size_t count) {
        parts.push_back({(void **)&ptr, need});
        need += (count * sizeof(*ptr) + 255) & ~(size_t)255;
    };
    part(p.phi, nk * nsite);
    part(p.e, nk * 3 * (SX_RING + 1));
    part(p.Q, nk * 3);
    if (mean_b) part(p.phiB, nk * nsite);
    part(p.K, nk * NC);
    part(p.L, (size_t)cells * NC * p.ld);
    if (nsb > SX_RING) part(p.A, (size_t)cells * NC * p.ld);
    if (mean_b) {
        part(p.dwp, (size_t)p.nrb * nsite * p.ld);
        part(p.KB, (size_t)p.ld);
    }
    part(p.partial, (size_t)nochunk * npts);
    if (ws.total + need > ctx->budget) return false;
    char *block = (char *)ws.get(need);
    if (!block) {
        ws.failed = false;
        return false;
    }
    for (auto &q : parts) *q.first = block + q.second;
    double norm = 1.0 / ((double)norigin * nsite * (double)nsb * nsb * nsb);
    if (kind == SB_SPIN) norm *= 0.07265;  // C of Eq. mag_intensity (barn)
    ProfScope ps(ctx, "subbox_cells", st);
    if (kind == SB_OCC) run_kind<T, SB_OCC>(p, norm, chunk_q, nochunk, dout, st);
    else if (kind == SB_SPIN) run_kind<T, SB_SPIN>(p, norm, chunk_q, nochunk, dout, st);
    else run_kind<T, SB_DISP>(p, norm, chunk_q, nochunk, dout, st);
    return true;
}

template bool subbox_cells_run<float>(ds_model *, int, const SbSite *, const int4 *, long long, const double *, long long,
                                      const ds_opts *, float *, double, Scratch &, cudaStream_t);
template bool subbox_cells_run<double>(ds_model *, int, const SbSite *, const int4 *, long long, const double *,
                                       long long, const ds_opts *, double *, double, Scratch &, cudaStream_t);
