// Rays: builders (tangent slab, axisymmetric lines of sight), the segment
// march with the angular reduction, and the spectral flux integral
// (Sec. 2.2.3).
//
// k_march (below) marches the bundles of every surface point over a range of
// wavelength columns and reduces them to the spectral flux at the point;
// k_wall_flux_part / _sum integrate that over the range.
#include <algorithm>

#include "rapral_internal.cuh"
#include "geom.cuh"

namespace {

// One segment of the march for one direction is I <- I e + ca j_far + cb j_near
// with t = dtau, e = e^{-t}, f = (1 - e)/t, the far-node coefficient
// ca = (f - e)/kappa and the near-node coefficient cb = (1 - f)/kappa.  With
// p = (1 - f)/t = sum_n (-t)^n / (n + 2)! it is
//   I + s B,  A = j_far - kappa I,  B = A + p ((j_near - j_far) - t A),
// which takes no exponential and no division where the series is short: FP64
// for |t| < 1/2, FP32 (seven terms, truncation below 4e-8 relative) likewise;
// beyond, the closed form loses at most two bits to 1 - e >= 0.39, and FP32
// takes e from an approximate ex2.
__device__ __forceinline__ float ex2f_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float recip(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// FP64.  The FP64 pipe has 1/64 of the FP32 rate here, so a step costs its
// count of FP64 operations.  The series is entered at the length |t| needs
// (truncation below 2e-17 relative: 3, 4, 5, 6, 9, 14 terms below 2^-17, 2^-13,
// 2^-10, 2^-7, 2^-4, 1/2; the lanes of a warp share the tail), and |t| is
// compared by its high word on the integer pipe.  A thin step is 8 to 20 FP64
// operations; with an expm1 and two divisions whatever its t it took the
// time of 75 (61 cells x 25 directions x 100,001 points: 18.8 -> 5.5 ms, 4.3
// with the directions split over warps).
constexpr int hi_2m(int k) { return (1023 - k) << 20; }   // high word of 2^-k
constexpr int T64_1 = hi_2m(1);
__device__ __forceinline__ int abs_hi(double t) { return __double2hiint(t) & 0x7fffffff; }
__device__ __forceinline__ double thin_series(double t, int hi) {
    double p;
    if (hi < hi_2m(17)) {
        p = 1.0 / 24.0;
    } else {
        if (hi < hi_2m(13)) {
            p = -1.0 / 120.0;
        } else {
            if (hi < hi_2m(10)) {
                p = 1.0 / 720.0;
            } else {
                if (hi < hi_2m(7)) {
                    p = -1.0 / 5040.0;
                } else {
                    if (hi < hi_2m(4)) {
                        p = 1.0 / 3628800.0;
                    } else {
                        p = fma(t, -1.0 / 1307674368000.0, 1.0 / 87178291200.0);
                        p = fma(t, p, -1.0 / 6227020800.0);
                        p = fma(t, p, 1.0 / 479001600.0);
                        p = fma(t, p, -1.0 / 39916800.0);
                        p = fma(t, p, 1.0 / 3628800.0);
                    }
                    p = fma(t, p, -1.0 / 362880.0);
                    p = fma(t, p, 1.0 / 40320.0);
                    p = fma(t, p, -1.0 / 5040.0);
                }
                p = fma(t, p, 1.0 / 720.0);
            }
            p = fma(t, p, -1.0 / 120.0);
        }
        p = fma(t, p, 1.0 / 24.0);
    }
    p = fma(t, p, -1.0 / 6.0);
    return fma(t, p, 0.5);
}
__device__ __noinline__ double thick_step(double I, double kf, double t, double jf, double jn) {
    const double em1 = expm1(-t), ik = 1.0 / kf;
    const double f = -em1 / t, e = 1.0 + em1;
    return I * e + (f - e) * ik * jf + (1.0 - f) * ik * jn;
}
__device__ __forceinline__ void seg_step(double& I, double kf, double s, double jf, double jn) {
    const double t = kf * s;
    const int hi = abs_hi(t);
    if (hi < T64_1) {
        const double p = thin_series(t, hi);
        const double A = fma(-kf, I, jf);
        I = fma(s, fma(p, fma(-t, A, jn - jf), A), I);
    } else {
        I = thick_step(I, kf, t, jf, jn);
    }
}
// FP32, thin (|dtau| < 0.5): with p = (1 - f)/dtau from its series
// p = sum_n (-dtau)^n / (n + 2)!, n = 0..6 (truncation below 4e-8 relative)
// and f = 1 - dtau p, the step I e + ca j_far + cb j_near is
// I + s f (j_far - kappa I) + s p (j_near - j_far): one series and no
// exponential (e = 1 - dtau f >= 0.6 keeps the subtraction within a factor
// 1/e of FP32 rounding).  Thick: e from ex2, f from one reciprocal.
__device__ __forceinline__ float thin_series(float t) {
    float p = fmaf(t, 1.0f / 40320.0f, -1.0f / 5040.0f);
    p = fmaf(t, p, 1.0f / 720.0f);
    p = fmaf(t, p, -1.0f / 120.0f);
    p = fmaf(t, p, 1.0f / 24.0f);
    p = fmaf(t, p, -1.0f / 6.0f);
    return fmaf(t, p, 0.5f);
}
__device__ __forceinline__ void seg_step(float& I, float kf, float s, float jf, float jn) {
    const float dtau = kf * s;
    if (fabsf(dtau) < (float)RAPRAL_THIN_F32) {
        const float p = thin_series(dtau);
        const float f = fmaf(-dtau, p, 1.0f);
        I = fmaf(s, fmaf(f, fmaf(-kf, I, jf), p * (jn - jf)), I);
        return;
    }
    const float e = ex2f_approx(-1.44269504f * dtau);
    const float r = recip(dtau);
    const float f = (1.0f - e) * r;
    I = fmaf(s * r, fmaf(f - e, jf, (1.0f - f) * jn), I * e);
}

// Two steps at once in FP32 (two wavelength columns, or two directions of a
// bundle): where both are optically thin the series and the update run as
// packed pairs (one instruction for both, each with the scalar step's IEEE
// result); otherwise each takes the scalar step.
__device__ __forceinline__ void seg_step2(float& I0, float& I1, float k0, float k1, float s0, float s1, float jf0,
                                          float jf1, float jn0, float jn1) {
    const float2 k = make_float2(k0, k1), s = make_float2(s0, s1);
    const float2 dt = __fmul2_rn(k, s);
    if (fabsf(dt.x) < (float)RAPRAL_THIN_F32 && fabsf(dt.y) < (float)RAPRAL_THIN_F32) {
        const auto c2 = [](float c) { return make_float2(c, c); };
        float2 p = __ffma2_rn(dt, c2(1.0f / 40320.0f), c2(-1.0f / 5040.0f));
        p = __ffma2_rn(dt, p, c2(1.0f / 720.0f));
        p = __ffma2_rn(dt, p, c2(-1.0f / 120.0f));
        p = __ffma2_rn(dt, p, c2(1.0f / 24.0f));
        p = __ffma2_rn(dt, p, c2(-1.0f / 6.0f));
        p = __ffma2_rn(dt, p, c2(0.5f));
        const float2 f = __ffma2_rn(make_float2(-dt.x, -dt.y), p, c2(1.0f));
        const float2 I = make_float2(I0, I1);
        const float2 A = __ffma2_rn(make_float2(-k0, -k1), I, make_float2(jf0, jf1));
        const float2 dJ = make_float2(jn0 - jf0, jn1 - jf1);
        const float2 r = __ffma2_rn(s, __ffma2_rn(f, A, __fmul2_rn(p, dJ)), I);
        I0 = r.x;
        I1 = r.y;
    } else {
        seg_step(I0, k0, s0, jf0, jn0);
        seg_step(I1, k1, s1, jf1, jn1);
    }
}

// The nd directions of one column (nd <= MAXD, the same for the whole warp;
// scmax: their largest scale).  With the common length s the step of a
// direction of scale c is I + c B, A = s j_far - s kappa I, B = A +
// p(c s kappa) (s (j_near - j_far) - c s kappa A), so s kappa, s j_far and
// s (j_near - j_far) are shared.  FP32 runs two directions a packed
// instruction, with t = -c s kappa carried so that no sign is flipped (FP32
// and integer instructions share one pipe, which bounds the slab): the
// largest scale decides once for all directions and, by a vote, for the warp
// (lanes on two paths would take both) whether the short series (|t| below
// 2^-5, four terms, truncation 3e-9: 8 packed instructions a pair) or the
// seven-term one (11) holds; only where it does not is each pair tested.
__device__ __forceinline__ float2 f2c(float c) { return make_float2(c, c); }
template <bool SHORT>
__device__ __forceinline__ void dir_pair(float& I0, float& I1, float2 t0, float2 jd, float2 dj, float2 sc) {
    const float2 t = __fmul2_rn(t0, sc);
    float2 p = f2c(1.0f / 120.0f);
    if (!SHORT) {
        p = __ffma2_rn(t, f2c(1.0f / 40320.0f), f2c(1.0f / 5040.0f));
        p = __ffma2_rn(t, p, f2c(1.0f / 720.0f));
        p = __ffma2_rn(t, p, f2c(1.0f / 120.0f));
    }
    p = __ffma2_rn(t, p, f2c(1.0f / 24.0f));
    p = __ffma2_rn(t, p, f2c(1.0f / 6.0f));
    p = __ffma2_rn(t, p, f2c(0.5f));
    const float2 I = make_float2(I0, I1);
    const float2 A = __ffma2_rn(t0, I, jd);
    const float2 r = __ffma2_rn(sc, __ffma2_rn(p, __ffma2_rn(t, A, dj), A), I);
    I0 = r.x;
    I1 = r.y;
}
template <class T, int MAXD>
__device__ __forceinline__ void dir_steps(T (&I)[MAXD], T kf, T ds, const T* sc, T scmax, int nd, T jf, T jn) {
    if constexpr (sizeof(T) == 4) {
        const float t0 = -kf * ds;
        const float2 t2 = f2c(t0), jd = f2c(ds * jf), dj = f2c(ds * (jn - jf));
        const float tm = fabsf(t0) * scmax;
        const auto pairs = [&](auto step) {
#pragma unroll
            for (int d = 0; d < MAXD; d += 2) {
                if (d % 4 == 0 && d >= nd) break;
                if (d + 1 < MAXD) {
                    step(I[d], I[d + 1], make_float2(sc[d], sc[d + 1]));
                } else {   // the last of an odd number, with an idle half of scale 0
                    float idle = 0.0f;
                    step(I[d], idle, make_float2(sc[d], 0.0f));
                }
            }
        };
        if (!__any_sync(0xffffffffu, tm >= 0.03125f)) {
            pairs([&](float& a, float& b, float2 s) { dir_pair<true>(a, b, t2, jd, dj, s); });
        } else if (!__any_sync(0xffffffffu, tm >= (float)RAPRAL_THIN_F32)) {
            pairs([&](float& a, float& b, float2 s) { dir_pair<false>(a, b, t2, jd, dj, s); });
        } else {
            pairs([&](float& a, float& b, float2 s) {
                if (fabsf(t0) * fmaxf(s.x, s.y) < (float)RAPRAL_THIN_F32) {
                    dir_pair<false>(a, b, t2, jd, dj, s);
                } else {
                    seg_step(a, kf, ds * s.x, jf, jn);
                    seg_step(b, kf, ds * s.y, jf, jn);
                }
            });
        }
    } else {
        const T t0 = kf * ds, jd = ds * jf, dj = ds * (jn - jf);
#pragma unroll
        for (int d = 0; d < MAXD; ++d) {
            if (d < nd) {
                const T t = t0 * sc[d];
                const int hi = abs_hi(t);
                if (hi < T64_1) {
                    const T p = thin_series(t, hi);
                    const T A = fma(-t0, I[d], jd);
                    I[d] = fma(sc[d], fma(p, fma(-t, A, dj), A), I[d]);
                } else {
                    I[d] = thick_step(I[d], kf, t, jf, jn);
                }
            }
        }
    }
}

// Checks of the ray set and, with `f` (the FP32 march), the FP32 copies of
// the path lengths (f), direction scales (fd) and weights (fw).
__global__ void k_validate_rays(const int32_t* __restrict__ seg_cell, const double* __restrict__ seg_ds, int64_t nseg,
                                int64_t C, const double* __restrict__ dir_scale,
                                const double* __restrict__ dir_weight, int64_t ndir, float* __restrict__ f,
                                float* __restrict__ fd, float* __restrict__ fw, int* status) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < nseg) {
        const int c = seg_cell[i];
        if (c < 0 || c >= C) fail(status, CHK_SEG_CELL, i);
        const double d = seg_ds[i];
        if (!(d >= 0.0) || !isfinite(d)) fail(status, CHK_SEG_DS, i);
        if (f) f[i] = (float)d;
    }
    if (i < ndir) {
        const double s = dir_scale[i];
        if (!(s > 0.0) || !isfinite(s)) fail(status, CHK_DIR, i);
        if (f) {
            fd[i] = (float)s;
            fw[i] = (float)dir_weight[i];
        }
    }
}

struct MarchArgs {
    const int64_t* point_off;
    const int64_t* seg_off;
    const int32_t* seg_cell;
    const double* seg_ds;
    const int64_t* dir_off;
    const double* dir_scale;
    const double* dir_weight;
    const float* seg_ds_f;       // FP32 copies (FP32 march only): no conversion per
    const float* dir_scale_f;    // (segment, direction, wavelength)
    const float* dir_weight_f;
    const int32_t* bundle_wall;
    double T_wall;
    const void* wall_row;        // Planck intensity at T_wall per column (null: T_wall = 0)
    const void* kappa;
    const void* emis;
    int64_t ld;
    double lam_min, h;
    int64_t k0, nk;
    void* q_lambda;
    void* I_out;
    Phys ph;
    const int* status;
};

template <class T> __device__ __forceinline__ T seg_len(const MarchArgs& a, int64_t i);
template <> __device__ __forceinline__ double seg_len<double>(const MarchArgs& a, int64_t i) { return a.seg_ds[i]; }
template <> __device__ __forceinline__ float seg_len<float>(const MarchArgs& a, int64_t i) { return a.seg_ds_f[i]; }
template <class T> __device__ __forceinline__ T dir_val(const double* d, const float* f, int64_t i);
template <> __device__ __forceinline__ double dir_val<double>(const double* d, const float*, int64_t i) { return d[i]; }
template <> __device__ __forceinline__ float dir_val<float>(const double*, const float* f, int64_t i) { return f[i]; }

// Planck intensity, temperature form (Sec. 2.2), W/cm^2/sr/um.
__device__ __forceinline__ double planck(double lam_nm, double T, const Phys& ph) {
    const double lcm = lam_nm * 1e-7;
    const double l2 = lcm * lcm;
    return 1e-7 * 2.0 * ph.h * ph.c * ph.c / (1e4 * l2 * l2 * lcm * expm1(ph.h * ph.c / (lcm * ph.kB * T)));
}

// One staged segment of a warp's bundle (march_nodes, march_multi, march_bundle).
template <class T> struct __align__(16) SegStage {
    const char* row;   // kappa row of the segment's next cell
    T ds;              // path length (x the direction scale for one-direction bundles)
};

#ifndef RAPRAL_MARCH_UNROLL
#define RAPRAL_MARCH_UNROLL 3
#endif
constexpr int kUnroll = RAPRAL_MARCH_UNROLL;

// Node-valued rays (one direction): rows are the LOS nodes, segment s of
// bundle b runs from node s + b to node s + b + 1, kappa held at the far
// node, j linear between the nodes (the same coefficients).
template <class T, int V>
__device__ __forceinline__ void march_nodes(const MarchArgs& a, int64_t b, T sc, SegStage<T>* stage, int lane,
                                            const char* kbase, int64_t ldb, int64_t offK, int64_t offJ,
                                            T (&I)[V][1]) {
    const int64_t s0 = a.seg_off[b], s1 = a.seg_off[b + 1];
    if (s1 <= s0) return;
    T kf[V], jf[V];
    {
        const char* row = kbase + (s0 + b) * ldb;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            kf[v] = *reinterpret_cast<const T*>(row + offK + 32 * v * sizeof(T));
            jf[v] = *reinterpret_cast<const T*>(row + offJ + 32 * v * sizeof(T));
        }
    }
    for (int64_t g = s0; g < s1; g += 32) {
        const int64_t mine = g + lane;
        __syncwarp();
        const bool in = mine < s1;
        stage[lane].row = in ? kbase + (mine + 1 + b) * ldb : kbase;
        stage[lane].ds = in ? seg_len<T>(a, mine) * sc : T(0);
        if (lane == 0) stage[32].row = kbase;
        __syncwarp();
        const int n = s1 - g < 32 ? (int)(s1 - g) : 32;
        T kx[V], jx[V];
        {
            const char* r0 = stage[0].row;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                kx[v] = *reinterpret_cast<const T*>(r0 + offK + 32 * v * sizeof(T));
                jx[v] = *reinterpret_cast<const T*>(r0 + offJ + 32 * v * sizeof(T));
            }
        }
        for (int j = 0; j < n; ++j) {
            const T ds = stage[j].ds;
            const char* rn = stage[j + 1].row;
            T ky[V], jy[V];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                ky[v] = *reinterpret_cast<const T*>(rn + offK + 32 * v * sizeof(T));
                jy[v] = *reinterpret_cast<const T*>(rn + offJ + 32 * v * sizeof(T));
            }
            if constexpr (V == 2 && sizeof(T) == 4) {
                seg_step2(I[0][0], I[1][0], kf[0], kf[1], ds, ds, jf[0], jf[1], jx[0], jx[1]);
            } else {
#pragma unroll
                for (int v = 0; v < V; ++v) seg_step(I[v][0], kf[v], ds, jf[v], jx[v]);
            }
#pragma unroll
            for (int v = 0; v < V; ++v) {
                kf[v] = kx[v]; jf[v] = jx[v];
                kx[v] = ky[v]; jx[v] = jy[v];
            }
        }
    }
}

// The march of a bundle of several directions over the lane's column: a step
// of 17 directions is about 150 FP32 instructions a warp.  The next MPF cells
// are in flight, across the staging seams: entry j of the stage holds the
// length of segment j and the row of the cell that step j + MPF needs (two,
// three, four and six ahead take the same time).  In FP32 two steps are
// unrolled: the ring's shift is then a renaming, where a copy of a value still
// in flight waits for it (200 cells x 17 directions x 262,144 columns: 573 ->
// 528 us; rings of three and four, unrolled by as many: 599 and 629).  In FP64
// the loads are far ahead in time and the longer body costs 2 %.
template <class T, int MAXD>
__device__ __forceinline__ void march_multi(const MarchArgs& a, int64_t b, int64_t d0, int nd, SegStage<T>* stage,
                                            int lane, const char* kbase, int64_t ldb, int64_t offK, int64_t offJ,
                                            int col0, T (&I)[1][MAXD]) {
    constexpr int MPF = 2, UNROLL = sizeof(T) == 4 ? MPF : 1;
    T sc[MAXD], scmax = T(0);
#pragma unroll
    for (int d = 0; d < MAXD; ++d) {
        sc[d] = d < nd ? dir_val<T>(a.dir_scale, a.dir_scale_f, d0 + d) : T(0);
        scmax = sc[d] > scmax ? sc[d] : scmax;
    }
    const T I0 = (a.wall_row && a.bundle_wall[b]) ? reinterpret_cast<const T*>(a.wall_row)[col0] : T(0);
#pragma unroll
    for (int d = 0; d < MAXD; ++d) I[0][d] = I0;
    const int64_t s0 = a.seg_off[b], s1 = a.seg_off[b + 1];
    if (s1 <= s0) return;
    const auto row_of = [&](int64_t i) { return i < s1 ? kbase + (int64_t)a.seg_cell[i] * ldb : kbase; };   // past the end: a valid row
    const char* r0 = row_of(s0);
    T kc = *reinterpret_cast<const T*>(r0 + offK), jc = *reinterpret_cast<const T*>(r0 + offJ);
    T kf = kc, jf = jc, rk[MPF], rj[MPF];
#pragma unroll
    for (int q = 0; q < MPF; ++q) {
        const char* r = row_of(s0 + 1 + q);
        rk[q] = *reinterpret_cast<const T*>(r + offK);
        rj[q] = *reinterpret_cast<const T*>(r + offJ);
    }
    for (int64_t g = s0; g < s1 - 1; g += 32) {
        const int64_t mine = g + lane;
        __syncwarp();
        stage[lane].row = row_of(mine + 1 + MPF);
        stage[lane].ds = mine < s1 - 1 ? seg_len<T>(a, mine) : T(0);
        __syncwarp();
        const int n = s1 - 1 - g < 32 ? (int)(s1 - 1 - g) : 32;
#pragma unroll UNROLL
        for (int j = 0; j < n; ++j) {
            const T ds = stage[j].ds;
            const char* r = stage[j].row;
            const T kx = rk[0], jx = rj[0];
#pragma unroll
            for (int q = 0; q + 1 < MPF; ++q) { rk[q] = rk[q + 1]; rj[q] = rj[q + 1]; }
            rk[MPF - 1] = *reinterpret_cast<const T*>(r + offK);
            rj[MPF - 1] = *reinterpret_cast<const T*>(r + offJ);
            const T kn = T(0.5) * (kc + kx), jn = T(0.5) * (jc + jx);
            dir_steps<T, MAXD>(I[0], kf, ds, sc, scmax, nd, jf, jn);
            kf = kn; jf = jn; kc = kx; jc = jx;
        }
    }
    // last segment: its near node is the cell's own value
    dir_steps<T, MAXD>(I[0], kf, seg_len<T>(a, s1 - 1), sc, scmax, nd, jf, jc);
}

template <class T, int V>
__device__ __forceinline__ void march_bundle(const MarchArgs& a, int64_t b, int64_t d0, SegStage<T>* stage,
                                             int lane, const char* kbase, int64_t ldb, int64_t offK, int64_t offJ,
                                             int col0, T (&I)[V][1]) {
    // the direction's scale goes into the staged length
    const T stage_scale = dir_val<T>(a.dir_scale, a.dir_scale_f, d0);
#pragma unroll
    for (int v = 0; v < V; ++v) {
        const T I0 = (a.wall_row && a.bundle_wall[b]) ? reinterpret_cast<const T*>(a.wall_row)[col0 + 32 * v] : T(0);
        I[v][0] = I0;
    }
    const int64_t s0 = a.seg_off[b], s1 = a.seg_off[b + 1];
    if (s1 <= s0) return;
    T kc[V], jc[V], kf[V], jf[V];
    {
        const char* row = kbase + (int64_t)a.seg_cell[s0] * ldb;
#pragma unroll
        for (int v = 0; v < V; ++v) {
            kc[v] = kf[v] = *reinterpret_cast<const T*>(row + offK + 32 * v * sizeof(T));
            jc[v] = jf[v] = *reinterpret_cast<const T*>(row + offJ + 32 * v * sizeof(T));
        }
    }
    // every segment but the last has a next cell: stage (row of the next
    // cell, length) for 32 segments, read back by all lanes
    for (int64_t g = s0; g < s1 - 1; g += 32) {
        const int64_t mine = g + lane;
        __syncwarp();
        // entries past the chunk point at row 0 (a valid row), so the
        // prefetch of entry j + 1 below never leaves the arrays
        const bool in = mine < s1 - 1;
        stage[lane].row = in ? kbase + (int64_t)a.seg_cell[mine + 1] * ldb : kbase;
        stage[lane].ds = in ? seg_len<T>(a, mine) * stage_scale : T(0);
        if (lane == 0) stage[32].row = kbase;
        __syncwarp();
        const int n = s1 - 1 - g < 32 ? (int)(s1 - 1 - g) : 32;
        T kx[V], jx[V];
        {
            const char* r0 = stage[0].row;
#pragma unroll
            for (int v = 0; v < V; ++v) {
                kx[v] = *reinterpret_cast<const T*>(r0 + offK + 32 * v * sizeof(T));
                jx[v] = *reinterpret_cast<const T*>(r0 + offJ + 32 * v * sizeof(T));
            }
        }
#pragma unroll kUnroll
        for (int j = 0; j < n; ++j) {
            const T ds = stage[j].ds;
            const char* rn = stage[j + 1].row;
            T ky[V], jy[V];   // next segment's next cell, loaded a step ahead
#pragma unroll
            for (int v = 0; v < V; ++v) {
                ky[v] = *reinterpret_cast<const T*>(rn + offK + 32 * v * sizeof(T));
                jy[v] = *reinterpret_cast<const T*>(rn + offJ + 32 * v * sizeof(T));
            }
            T kn[V], jn[V];
#pragma unroll
            for (int v = 0; v < V; ++v) {
                kn[v] = T(0.5) * (kc[v] + kx[v]);
                jn[v] = T(0.5) * (jc[v] + jx[v]);
            }
            if constexpr (V == 2 && sizeof(T) == 4) {
                seg_step2(I[0][0], I[1][0], kf[0], kf[1], ds, ds, jf[0], jf[1], jn[0], jn[1]);
            } else {
#pragma unroll
                for (int v = 0; v < V; ++v) seg_step(I[v][0], kf[v], ds, jf[v], jn[v]);
            }
#pragma unroll
            for (int v = 0; v < V; ++v) {
                kf[v] = kn[v]; jf[v] = jn[v];
                kc[v] = kx[v]; jc[v] = jx[v];
                kx[v] = ky[v]; jx[v] = jy[v];
            }
        }
    }
    {   // last segment: its near node is the cell's own value
        const T ds = seg_len<T>(a, s1 - 1) * stage_scale;
        if constexpr (V == 2 && sizeof(T) == 4) {
            seg_step2(I[0][0], I[1][0], kf[0], kf[1], ds, ds, jf[0], jf[1], jc[0], jc[1]);
        } else {
#pragma unroll
            for (int v = 0; v < V; ++v) seg_step(I[v][0], kf[v], ds, jf[v], jc[v]);
        }
    }
}

// k_march: the segment march with the angular reduction.  A block covers one
// (surface point, bundle group) and a tile of wavelength columns; lane l of a
// column group takes columns l, l + 32, ..., l + 32 (V - 1) of the group's 32
// V.  Each gather of a segment is then V coalesced row reads, and the
// per-segment work (next cell, length, row address) is shared by the V columns
// and the warp's directions.  Three forms:
//   SL = 8 (many bundles a point, as the axisymmetric rays): eight warps on the
//     same columns take the bundles of the group round-robin;
//   SL = 1, MAXD > 1 (a few bundles of many directions, as the tangent slab):
//     one warp a block, all of a bundle's directions, or DS > 0: up to DS warps
//     on the same columns share each bundle's directions;
//   SL = 1, MAXD = 1: eight warps on eight column groups, every bundle.
// A warp stages the next cell's row address and the length of 32 segments at
// a time in shared memory (one coalesced read of the segment list), so no
// kappa / j gather waits on a dependent load of the list, and loads cells'
// values one step (march_multi: two) ahead; the last segment of a bundle, whose near
// node is its own cell, is taken after the loop.  A point's bundles are
// split over 2^lgG blocks (groups) so that enough blocks share a wavelength
// tile for its kappa / j rows to stay in L2.  Each slice Kahan-sums its
// bundles' weighted intensities, the slices are added in a fixed order, and
// the groups' partial spectral fluxes are added in group order by
// k_group_sum: results do not depend on timing.  The last wavelength tile is
// shifted back to end at nk (columns below the tile are computed again and
// not written), so every load is in bounds; with V = 1 and nk below the
// tile a lane past nk reads column nk - 1 and writes nothing.
#ifndef RAPRAL_MARCH_MINB
#define RAPRAL_MARCH_MINB 4
#endif
// Warps a block: eight where they share a point's bundles; one for the slab,
// whose warps are independent and all take the same time, so that the last
// wave is spread over the chip.  FP32 slab, 200 cells x 17 directions x 262,144
// columns: blocks of 8 warps 669 us, 2 warps 632, 1 warp 619 at 24 resident
// warps an SM, 578 at 32 (28: 589, 40: 582).
constexpr int march_warps(int MAXD, int SL) { return SL == 1 && MAXD > 1 ? 1 : 8; }
// Resident blocks asked of the compiler.
template <class T>
constexpr int march_minb(int V, int MAXD, int SL) {
    return MAXD == 1 ? (sizeof(T) == 4 && V > 1 ? RAPRAL_MARCH_MINB : 1)
           : MAXD > 17 ? 1
           : SL > 1 ? (sizeof(T) == 4 ? 3 : 1)
                    : (sizeof(T) == 4 ? 32 : 12);
}
// A split bundle's blocks: 30 resident warps an SM asked in FP32, 18 in FP64
// (3 directions a warp) or 15 (7).
template <class T>
constexpr int march_minb_split(int MAXD, int DS) { return (sizeof(T) == 4 ? 32 : MAXD <= 3 ? 18 : 16) / DS; }
// DS > 0: the directions of each bundle are dealt to the block's warps (at most
// DS of them), MAXD or fewer each, all on the same 32 columns.
template <class T, int V, int MAXD, int SL, bool NODES = false, int DS = 0>
__global__ void __launch_bounds__(32 * (DS ? DS : march_warps(MAXD, SL)),
                                  DS ? march_minb_split<T>(MAXD, DS) : march_minb<T>(V, MAXD, SL))
    k_march(MarchArgs a, int lgG, T* __restrict__ part) {
    static_assert(!NODES || MAXD == 1, "node-valued rays have one direction a bundle");
    static_assert(MAXD == 1 || V == 1, "bundles of several directions take one column a lane");
    static_assert(DS == 0 || (SL == 1 && MAXD > 1), "a split of the directions has no bundle slices");
    if (*a.status) return;
    constexpr int W = DS ? DS : march_warps(MAXD, SL), CW = DS ? 1 : W / SL, TW = CW * 32 * V;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int slice = DS ? 0 : warp / CW, cgrp = DS ? 0 : warp % CW;
    const int nr = DS ? (int)(blockDim.x >> 5) : SL;   // partial sums a column
    // columns fit in int: nk <= 32 x 65535 (checked by the caller)
    const int nk = (int)a.nk;
    const int tile0 = (int)blockIdx.y * TW;
    const int base = (tile0 + TW > nk && nk >= TW) ? nk - TW : tile0;
    const int colu = base + cgrp * 32 * V + lane;   // unclamped first column
    const int col0 = colu < nk ? colu : nk - 1;     // only when V = 1 and nk < TW
    // byte addressing: row of cell c at kbase + c ldb; this lane's kappa and
    // j columns at offK, offJ from it
    const char* kbase = reinterpret_cast<const char*>(a.kappa);
    const int64_t ldb = a.ld * (int64_t)sizeof(T);
    const int64_t offK = (int64_t)col0 * sizeof(T);
    const int64_t offJ = (reinterpret_cast<const char*>(a.emis) - kbase) + offK;
    __shared__ SegStage<T> stage_all[W][33];
    SegStage<T>* stage = stage_all[warp];
    T acc[V], comp[V];
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = comp[v] = T(0);
    // G = 2^lgG groups of point p = blockIdx.x >> lgG; group g takes every
    // G-th run of SL bundles, slice s the s-th bundle of each run
    const unsigned p = blockIdx.x >> lgG, grp = blockIdx.x & ((1u << lgG) - 1u);
    const int64_t b1 = a.point_off[p + 1];
    for (int64_t b = a.point_off[p] + (int64_t)grp * SL + slice; b < b1; b += (int64_t)SL << lgG) {
        const int64_t db = a.dir_off[b];
        const int nb = (int)(a.dir_off[b + 1] - db);
        // a warp's share and where its next one starts (a second share only if
        // max_dirs understates the bundle: one of several directions is marched
        // whole in every form)
        const int q = DS ? min((nb + nr - 1) / nr, MAXD) : MAXD > 1 ? min(nb, MAXD) : nb;
        for (int first = DS ? warp * q : 0; first < nb; first += DS ? nr * q : q) {
            const int64_t d0 = db + first;
            const int nd = min(nb - first, q);
            T I[V][MAXD];
            if constexpr (NODES) {
                const bool wall = a.wall_row && a.bundle_wall[b];
#pragma unroll
                for (int v = 0; v < V; ++v) I[v][0] = wall ? reinterpret_cast<const T*>(a.wall_row)[col0 + 32 * v] : T(0);
                march_nodes<T, V>(a, b, dir_val<T>(a.dir_scale, a.dir_scale_f, d0), stage, lane, kbase, ldb, offK,
                                  offJ, I);
            } else {
                if constexpr (MAXD == 1) march_bundle<T, V>(a, b, d0, stage, lane, kbase, ldb, offK, offJ, col0, I);
                else march_multi<T, MAXD>(a, b, d0, nd, stage, lane, kbase, ldb, offK, offJ, col0, I);
            }
#pragma unroll
            for (int v = 0; v < V; ++v) {
                const int kk = colu + 32 * v;
                const bool own = kk >= tile0 && kk < nk;
                T part_v = T(0);
#pragma unroll
                for (int d = 0; d < MAXD; ++d) {
                    if (d < nd) {
                        part_v += dir_val<T>(a.dir_weight, a.dir_weight_f, d0 + d) * I[v][d];
                        if (a.I_out && own) reinterpret_cast<T*>(a.I_out)[(d0 + d) * a.nk + kk] = I[v][d];
                    }
                }
                // compensated sum over the slice's bundles
                const T y = part_v - comp[v];
                const T tt = acc[v] + y;
                comp[v] = (tt - acc[v]) - y;
                acc[v] = tt;
            }
        }
    }
    constexpr int NR = DS ? DS : SL;
    __shared__ T red[NR][TW];
#pragma unroll
    for (int v = 0; v < V; ++v) red[DS ? warp : slice][cgrp * 32 * V + lane + 32 * v] = acc[v];
    __syncthreads();
    T* dst = (lgG == 0 ? reinterpret_cast<T*>(a.q_lambda) : part) + (int64_t)blockIdx.x * a.nk;
    for (int i = threadIdx.x; i < TW; i += blockDim.x) {
        const int kk = base + i;
        if (kk < tile0 || kk >= nk) continue;
        T s = red[0][i];
        for (int q = 1; q < nr; ++q) s += red[q][i];
        dst[kk] = s;
    }
}

// ---------------------------------------------------------------------------
// k_march1: the FP32 march of single-direction, cell-valued bundles (the
// axisymmetric lines of sight), the hot kernel of the afterbody.
//
// Same work and results contract as k_march<float, 2, 1, 8>, organised for
// fewer instructions per segment-wavelength:
//  * lane l owns four or two ADJACENT columns: one 16- or 8-byte load fetches
//    them, for kappa and for j (a warp reads 512 or 256 contiguous bytes of a
//    row); where rows are not aligned for it, two columns 32 apart with one
//    coalesced 4-byte load each;
//  * node values are carried doubled (K = kappa_a + kappa_b, the sum of the
//    two cells at a face), with the segment length halved to match, which
//    removes the averaging multiplies;
//  * the step (m1_step) carries minus the intensity and minus the half length
//    and takes the series as long as the depth needs;
//  * equal rays of a point are marched once (k_ray_hash, k_ray_match);
//  * the staged list holds, for step j, the segment's halved length (as the
//    packed pair the step multiplies by) and the byte offset of the row of the
//    cell PF steps ahead (row x ld, computed once by the staging lane), so a
//    step does no address arithmetic beyond adding that offset to its lane's
//    base; each step issues the loads it will use PF steps later and no load
//    is exposed at the 32-segment staging seams;
//  * the bundles of a block are dealt to its eight warps longest first
//    (k_march_plan), so the warps finish together at the block's reduction.
// Every slice still Kahan-sums its bundles in a fixed order and the slices
// and groups are added in fixed order: results do not depend on timing.
// Four columns a lane at the 64 registers of four blocks an SM spill 184 bytes
// a thread (244 loaded); two columns do not, and are 6 % slower on wide ranges.

#ifndef RAPRAL_M1_PF
#define RAPRAL_M1_PF 2
#endif
#ifndef RAPRAL_M1_UNROLL
#define RAPRAL_M1_UNROLL 4
#endif
constexpr int M1_PF = RAPRAL_M1_PF;            // steps between a load and its use
constexpr int kM1Unroll = RAPRAL_M1_UNROLL;    // segment steps unrolled
constexpr int M1_SLICES = 8;    // warps (bundle slices) per block

struct __align__(16) M1Stage {
    float2 nsh;     // minus half the segment length (x the direction scale), twice: a packed pair
    int64_t off;    // byte offset of the row of the cell step j + M1_PF needs (its next cell); 0 past the end
};

// One step of one column with doubled node values Kf, Jf (far), Jn (near),
// minus the half length, nsh, and minus the intensity, M.
__device__ __forceinline__ float m1_step1(float M, float Kf, float Jf, float Jn, float nsh) {
    const float t = Kf * nsh;   // minus kappa_far x length
    const float dJ = Jn - Jf;
    if (fabsf(t) < (float)RAPRAL_THIN_F32) {
        float p = fmaf(t, 1.0f / 40320.0f, 1.0f / 5040.0f);
        p = fmaf(t, p, 1.0f / 720.0f);
        p = fmaf(t, p, 1.0f / 120.0f);
        p = fmaf(t, p, 1.0f / 24.0f);
        p = fmaf(t, p, 1.0f / 6.0f);
        p = fmaf(t, p, 0.5f);
        const float A = fmaf(Kf, M, Jf);
        return fmaf(nsh, fmaf(p, fmaf(t, A, dJ), A), M);
    }
    const float e = ex2f_approx(1.44269504f * t);
    const float r = recip(t);
    const float f = (e - 1.0f) * r;
    const float p = (f - 1.0f) * r;
    return fmaf(nsh, fmaf(f, Jf, p * dJ), M * e);
}

// One step of both columns: packed when both are thin.  Carrying -I and -h
// leaves no sign to flip (packed operands take none for free): 14 packed
// operations, 11 where both depths are below 2^-5 (four terms of the series,
// truncation 3e-9), as nearly all are.  FP32 and integer instructions share
// one pipe here, and the march is bound by it: the form with signs, the full
// series always and f beside p was 57 pipe slots for two columns.
constexpr float M1_SHORT = 0.03125f;
__device__ __forceinline__ void m1_step(float2& M, float2 Kf, float2 Jf, float2 Jn, float2 nsh) {
    const float2 t = __fmul2_rn(Kf, nsh);
    const float m = fmaxf(fabsf(t.x), fabsf(t.y));
    if (m < (float)RAPRAL_THIN_F32) {
        const auto c2 = [](float c) { return make_float2(c, c); };
        float2 p = c2(1.0f / 120.0f);
        if (m >= M1_SHORT) {
            p = __ffma2_rn(t, c2(1.0f / 40320.0f), c2(1.0f / 5040.0f));
            p = __ffma2_rn(t, p, c2(1.0f / 720.0f));
            p = __ffma2_rn(t, p, c2(1.0f / 120.0f));
        }
        p = __ffma2_rn(t, p, c2(1.0f / 24.0f));
        p = __ffma2_rn(t, p, c2(1.0f / 6.0f));
        p = __ffma2_rn(t, p, c2(0.5f));
        const float2 A = __ffma2_rn(Kf, M, Jf);
        const float2 u = __ffma2_rn(t, A, __ffma2_rn(Jf, c2(-1.0f), Jn));
        M = __ffma2_rn(nsh, __ffma2_rn(p, u, A), M);
    } else {
        M.x = m1_step1(M.x, Kf.x, Jf.x, Jn.x, nsh.x);
        M.y = m1_step1(M.y, Kf.y, Jf.y, Jn.y, nsh.x);
    }
}

// Equal rays.  In an axisymmetric field a line of sight and its mirror image
// cross the same cells with the same lengths, so half of the rays of such a
// set repeat the other half: a ray whose cells, FP32 lengths, FP32 scale and
// wall flag equal an earlier one's of its point, bit for bit, has the same
// intensity bit for bit, and the two are marched once.  Whether a set has such
// rays is found from its lists on every call (a hash a ray, then a full
// comparison of the candidates); sets without them march as they are.  With
// the step below, 100 x 50 cells, 20 points x 512 rays, 16,384 columns: 7.73 ->
// 4.16 ms.
constexpr int M1_PAIR_MAX = 2048;   // bundles of a point compared (16 KB of keys); more: no pairs
// The search takes 12 to 22 us (two launches and a plan of what is left): it
// pays from about 30 us of march on where a set has equal rays.  10 points x 512
// rays of 80 segments x 256 / 512 / 1,000 columns, none equal: 146 / 213 / 351 us
// searched, 131 / 198 / 336 not; every two equal: 99 / 135 / 205 and 132 / 198 /
// 336.  At 128 columns none would take 103 and 84, every two 72 and 84: below the
// limits the rays march as they are.
constexpr int64_t M1_PAIR_WORK = int64_t(1) << 25;   // segments x columns, and
constexpr int64_t M1_PAIR_COLUMNS = 256;             // columns, from which a set is searched

__device__ __forceinline__ unsigned mix32(unsigned x) {
    x ^= x >> 16; x *= 0x7feb352du;
    x ^= x >> 15; x *= 0x846ca68bu;
    return x ^ (x >> 16);
}

// key[b]: 64-bit hash of bundle b's segments, scale and wall flag (0: not one
// direction, never paired); cand[] and partner[] cleared.  One warp a bundle.
// The points' bundles are [point_off[0], point_off[P]); what a set holds
// before or after them belongs to no point, and its lists are not read.
__global__ void __launch_bounds__(256) k_ray_hash(MarchArgs a, int64_t P, int64_t B,
                                                  unsigned long long* __restrict__ key, int32_t* __restrict__ cand,
                                                  int32_t* __restrict__ partner) {
    if (*a.status) return;
    const int64_t b = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (b >= B) return;
    // everything that needs no other value is loaded at once: latency is all this pass costs
    const int64_t in0 = a.point_off[0], in1 = a.point_off[P];
    const int64_t s0 = a.seg_off[b], s1 = a.seg_off[b + 1], d0 = a.dir_off[b];
    const int64_t nd = a.dir_off[b + 1] - d0;
    const bool wall = a.bundle_wall[b] != 0;
    if (lane == 0) cand[b] = partner[b] = -1;
    unsigned long long k = 0ULL;
    if (b >= in0 && b < in1 && nd == 1) {
        const unsigned sc = __float_as_uint(a.dir_scale_f[d0]);
        unsigned h0 = 0, h1 = 0;
        for (int64_t i = s0 + lane; i < s1; i += 32) {
            const unsigned x = mix32((unsigned)a.seg_cell[i] * 0x9e3779b1u + (unsigned)(i - s0));
            const unsigned y = mix32(__float_as_uint(a.seg_ds_f[i]) ^ x);
            h0 += y;
            h1 += mix32(y + 0x68bc21ebu);
        }
        h0 = __reduce_add_sync(0xffffffffu, h0);
        h1 = __reduce_add_sync(0xffffffffu, h1);
        h0 = mix32(h0 ^ sc);
        h1 = mix32(h1 + (unsigned)(s1 - s0) * 2u + wall);
        k = ((unsigned long long)h0 << 32 | h1) | 1ULL;
    }
    if (lane == 0) key[b] = k;
}

// cand[b]: the earlier bundle of the point whose march bundle b shares (a key's
// odd ranks go to the one before them), -1 for the others; partner[] the other
// way.  Blocks (point, 32 bundles), eight lanes a bundle; a warp then compares
// each candidate with its bundle in full, and what differs marches on its own.
// One block a point, which took its bundles in turn, and a launch of its own for
// the comparison needed 13 us for 2 points x 512 rays, 81 for 2 x 2,048 and 15
// for 2,000 x 16; now 5, about 8 and 7.
constexpr int MATCH_LANES = 8, MATCH_THREADS = 256, MATCH_BUNDLES = MATCH_THREADS / MATCH_LANES;
__global__ void __launch_bounds__(MATCH_THREADS) k_ray_match(MarchArgs a, const unsigned long long* __restrict__ key,
                                                             int32_t* __restrict__ cand,
                                                             int32_t* __restrict__ partner) {
    if (*a.status) return;
    __shared__ unsigned long long ks[M1_PAIR_MAX];
    __shared__ int16_t cs[MATCH_BUNDLES];
    const int64_t pb0 = a.point_off[blockIdx.x];
    const int64_t nb = a.point_off[blockIdx.x + 1] - pb0;
    if (nb > M1_PAIR_MAX) return;
    const int n = (int)nb, step = (int)gridDim.y * MATCH_BUNDLES, first = (int)blockIdx.y * MATCH_BUNDLES;
    if (first >= n) return;
    // a second pass only if max_bundles_per_point understates the point
    const int read = first + step < n ? n : min(n, first + MATCH_BUNDLES);
    for (int k = threadIdx.x; k < read; k += MATCH_THREADS) ks[k] = key[pb0 + k];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int kb = first; kb < n; kb += step) {
        const int k = kb + (int)threadIdx.x / MATCH_LANES, own = threadIdx.x % MATCH_LANES;
        const unsigned long long x = k < n ? ks[k] : 0ULL;
        int rank = 0, prev = -1;
        if (x != 0ULL)
            for (int q = own; q < k; q += MATCH_LANES)
                if (ks[q] == x) { ++rank; prev = q; }
#pragma unroll
        for (int o = 1; o < MATCH_LANES; o <<= 1) {
            rank += __shfl_xor_sync(0xffffffffu, rank, o);
            prev = max(prev, __shfl_xor_sync(0xffffffffu, prev, o));
        }
        if (own == 0) cs[k - kb] = (rank & 1) ? (int16_t)prev : (int16_t)-1;
        __syncthreads();
        for (int i = warp; i < MATCH_BUNDLES; i += MATCH_THREADS / 32) {
            if (cs[i] < 0) continue;   // the same for the whole warp
            const int64_t b = pb0 + kb + i, q = pb0 + cs[i];
            const int64_t x0 = a.seg_off[q], y0 = a.seg_off[b], m = a.seg_off[q + 1] - x0;
            const int64_t dx = a.dir_off[q], dy = a.dir_off[b];
            bool eq = m == a.seg_off[b + 1] - y0 &&
                      __float_as_uint(a.dir_scale_f[dx]) == __float_as_uint(a.dir_scale_f[dy]) &&
                      (a.bundle_wall[q] != 0) == (a.bundle_wall[b] != 0);
            for (int64_t j = lane; eq && j < m; j += 32)
                eq = a.seg_cell[x0 + j] == a.seg_cell[y0 + j] &&
                     __float_as_uint(a.seg_ds_f[x0 + j]) == __float_as_uint(a.seg_ds_f[y0 + j]);
            eq = __all_sync(0xffffffffu, eq);
            if (eq && lane == 0) {
                cand[b] = (int32_t)q;
                partner[q] = (int32_t)b;
            }
        }
        __syncthreads();
    }
}

// Bundle plan: for each (point p, group g) the group's bundles (a contiguous
// run of the point's marched bundles: with the rays of a point in angular
// order, the neighbours a block marches cross the same cells near the point,
// which L1 then serves) dealt to M1_SLICES slices longest first (greedy to the
// least-loaded slice, ties to the lower slice; equal lengths in index order).
// plan[] lists each group's bundles slice by slice, starting at the group's
// base; soff[(p G + g)(M1_SLICES + 1) + s] is where slice s starts.  Groups of
// more than 1024 bundles are dealt round-robin in index order.
__global__ void __launch_bounds__(128) k_march_plan(const int64_t* __restrict__ point_off,
                                                    const int64_t* __restrict__ seg_off,
                                                    const int32_t* __restrict__ cand, int G,
                                                    int32_t* __restrict__ plan, int32_t* __restrict__ soff,
                                                    const int* status) {
    if (*status) return;
    const int64_t p = blockIdx.x / G;
    const int g = (int)(blockIdx.x % G);
    const int64_t pb0 = point_off[p];
    int64_t nb = point_off[p + 1] - pb0;
    // the point's marched bundles (those that are no one's partner), in index order
    __shared__ int16_t us[M1_PAIR_MAX];
    __shared__ int nu;
    const bool all = cand == nullptr || nb > M1_PAIR_MAX;
    if (!all) {
        // a word of flags a warp pass, then a warp's prefix over the words (one
        // warp in order, and the slices' loads by number below: 2,000 points x 16
        // bundles 26 us, now 15)
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = (int)nb, words = (n + 31) / 32;
        __shared__ unsigned keep[M1_PAIR_MAX / 32];
        __shared__ int before[M1_PAIR_MAX / 32];
#pragma unroll 4
        for (int w = warp; w < words; w += 4) {
            const int k = 32 * w + lane;
            const unsigned mk = __ballot_sync(0xffffffffu, k < n && cand[pb0 + (k < n ? k : 0)] < 0);
            if (lane == 0) keep[w] = mk;
        }
        __syncthreads();
        if (warp == 0) {   // two words a lane
            const int c0 = 2 * lane < words ? __popc(keep[2 * lane]) : 0;
            const int c1 = 2 * lane + 1 < words ? __popc(keep[2 * lane + 1]) : 0;
            int sum = c0 + c1;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, sum, o);
                if (lane >= o) sum += v;
            }
            before[2 * lane] = sum - c0 - c1;
            before[2 * lane + 1] = sum - c1;
            if (lane == 31) nu = sum;
        }
        __syncthreads();
        for (int w = warp; w < words; w += 4) {
            const unsigned mk = keep[w];
            if (mk >> lane & 1u) us[before[w] + __popc(mk & ((1u << lane) - 1u))] = (int16_t)(32 * w + lane);
        }
        __syncthreads();
        nb = nu;
    }
    const auto uniq = [&](int64_t i) { return (int32_t)(all ? i : pb0 + us[i - pb0]); };
    const int64_t m = nb > g ? (nb - g + G - 1) / G : 0;                     // bundles of this group
    const int64_t base = pb0 + (int64_t)g * (nb / G) + (g < nb % G ? g : nb % G);   // the group's first entry
    int32_t* so = soff + blockIdx.x * (M1_SLICES + 1);
    __shared__ int32_t len[1024];
    __shared__ int16_t order[1024], place[1024];   // bundle and place in its slice, by rank
    __shared__ int8_t slice_of[1024];
    __shared__ int32_t start[M1_SLICES];
    if (m > 1024) {   // round-robin in index order
        for (int64_t k = threadIdx.x; k < m; k += blockDim.x) {
            const int s = (int)(k % M1_SLICES);
            const int64_t per = m / M1_SLICES, extra = m % M1_SLICES;
            const int64_t start = s * per + (s < extra ? s : extra);
            plan[base + start + k / M1_SLICES] = uniq(base + k);
        }
        if (threadIdx.x <= M1_SLICES) {
            const int s = threadIdx.x;
            const int64_t per = m / M1_SLICES, extra = m % M1_SLICES;
            so[s] = (int32_t)(base + s * per + (s < extra ? s : extra));
        }
        return;
    }
    const int mm = (int)m;
    for (int k = threadIdx.x; k < mm; k += blockDim.x) {
        const int64_t b = uniq(base + k);
        len[k] = (int32_t)min(seg_off[b + 1] - seg_off[b], (int64_t)2147483647);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < mm; k += blockDim.x) {   // rank: longer first, then lower index
        const int32_t lk = len[k];
        int r = 0;
        for (int q = 0; q < mm; ++q) r += (len[q] > lk) || (len[q] == lk && q < k);
        order[r] = (int16_t)k;
    }
    __syncthreads();
    if (threadIdx.x == 0) {   // in registers: a slice's load or count by its number would go through memory
        int64_t load[M1_SLICES];
        int cnt[M1_SLICES];
#pragma unroll
        for (int s = 0; s < M1_SLICES; ++s) { load[s] = 0; cnt[s] = 0; }
        for (int r = 0; r < mm; ++r) {
            const int64_t l = (int64_t)len[order[r]] + 1;
            int best = 0, at = 0;
            int64_t least = load[0];
#pragma unroll
            for (int s = 1; s < M1_SLICES; ++s)
                if (load[s] < least) { least = load[s]; best = s; }
#pragma unroll
            for (int s = 0; s < M1_SLICES; ++s)
                if (s == best) { load[s] += l; at = cnt[s]++; }
            slice_of[r] = (int8_t)best;
            place[r] = (int16_t)at;
        }
        int acc = 0;
#pragma unroll
        for (int s = 0; s < M1_SLICES; ++s) {
            start[s] = acc;
            so[s] = (int32_t)(base + acc);
            acc += cnt[s];
        }
        so[M1_SLICES] = (int32_t)(base + acc);
    }
    __syncthreads();
    // each slice's bundles, longest first
    for (int r = threadIdx.x; r < mm; r += blockDim.x)
        plan[base + start[slice_of[r]] + place[r]] = uniq(base + order[r]);
}

// A lane's 2 NP adjacent columns of one row, as NP packed pairs.
template <int NP> struct M1V { float2 v[NP]; };

// The lane's columns of one row: one 8-byte (NP = 1) or 16-byte (NP = 2)
// load of adjacent columns when they are aligned (VEC), else one coalesced
// 4-byte load a column at the offsets dq[] from the first (32 apart; columns
// past the range repeat the last).
template <int NP, bool VEC>
__device__ __forceinline__ M1V<NP> m1_load(const float* __restrict__ p, const int (&dq)[2 * NP]) {
    M1V<NP> r;
    if constexpr (VEC && NP == 1) {
        r.v[0] = *reinterpret_cast<const float2*>(p);
    } else if constexpr (VEC) {
        const float4 x = *reinterpret_cast<const float4*>(p);
        r.v[0] = make_float2(x.x, x.y);
        r.v[1] = make_float2(x.z, x.w);
    } else {
#pragma unroll
        for (int q = 0; q < NP; ++q) r.v[q] = make_float2(p[dq[2 * q]], p[dq[2 * q + 1]]);
    }
    return r;
}

template <int NP>
__device__ __forceinline__ M1V<NP> m1_sum(const M1V<NP>& x, const M1V<NP>& y) {
    M1V<NP> r;
#pragma unroll
    for (int q = 0; q < NP; ++q) r.v[q] = __fadd2_rn(x.v[q], y.v[q]);
    return r;
}

// The lane's columns of one row of kappa and of emis: kb, jb point at the
// lane's first column in row 0, off is the row's byte offset.
template <int NP, bool VEC>
__device__ __forceinline__ M1V<NP> m1_rowload(const char* kb, const char* jb, int64_t off, const int (&dq)[2 * NP],
                                              M1V<NP>& j) {
    j = m1_load<NP, VEC>(reinterpret_cast<const float*>(jb + off), dq);
    return m1_load<NP, VEC>(reinterpret_cast<const float*>(kb + off), dq);
}

// The march of bundle b over the lane's columns (doubled node values).
template <int NP, bool VEC>
__device__ __forceinline__ M1V<NP> m1_bundle(const MarchArgs& a, int64_t b, float sc, M1Stage* st, int lane,
                                             const char* __restrict__ kb, const char* __restrict__ jb,
                                             const int (&dq)[2 * NP], int64_t ldb, M1V<NP> I) {
    const int64_t s0 = a.seg_off[b], s1 = a.seg_off[b + 1];
    if (s1 <= s0) return I;
    M1V<NP> kc, jc;
    kc = m1_rowload<NP, VEC>(kb, jb, (int64_t)a.seg_cell[s0] * ldb, dq, jc);
    M1V<NP> Kf = m1_sum(kc, kc), Jf = m1_sum(jc, jc);
    const float hs = -0.5f * sc;
#pragma unroll
    for (int q = 0; q < NP; ++q) I.v[q] = make_float2(-I.v[q].x, -I.v[q].y);   // minus the intensity on the way
    // ring of loads in flight: values of the next cells of the following PF segments
    M1V<NP> rk[M1_PF], rj[M1_PF];
#pragma unroll
    for (int q = 0; q < M1_PF; ++q) {
        const int64_t i = s0 + q;   // segment i's next cell is cell i + 1
        const int c = (i < s1 - 1) ? a.seg_cell[i + 1] : 0;
        rk[q] = m1_rowload<NP, VEC>(kb, jb, (int64_t)c * ldb, dq, rj[q]);
    }
    for (int64_t g = s0; g < s1 - 1; g += 32) {
        const int64_t mine = g + lane;
        __syncwarp();
        const int64_t ahead = mine + M1_PF;   // the segment whose next cell this entry fetches
        const float shl = mine < s1 - 1 ? seg_len<float>(a, mine) * hs : 0.0f;
        st[lane].nsh = make_float2(shl, shl);
        st[lane].off = ahead < s1 - 1 ? (int64_t)a.seg_cell[ahead + 1] * ldb : 0;
        __syncwarp();
        const int n = s1 - 1 - g < 32 ? (int)(s1 - 1 - g) : 32;
#pragma unroll kM1Unroll
        for (int j = 0; j < n; ++j) {
            const M1Stage e = st[j];
            const M1V<NP> kx = rk[0], jx = rj[0];
#pragma unroll
            for (int q = 0; q + 1 < M1_PF; ++q) { rk[q] = rk[q + 1]; rj[q] = rj[q + 1]; }
            rk[M1_PF - 1] = m1_rowload<NP, VEC>(kb, jb, e.off, dq, rj[M1_PF - 1]);
            const M1V<NP> Kn = m1_sum(kc, kx), Jn = m1_sum(jc, jx);
#pragma unroll
            for (int q = 0; q < NP; ++q) m1_step(I.v[q], Kf.v[q], Jf.v[q], Jn.v[q], e.nsh);
            Kf = Kn; Jf = Jn; kc = kx; jc = jx;
        }
    }
    {   // last segment: its near node is its own cell's value
        const float hl = seg_len<float>(a, s1 - 1) * hs;
        const M1V<NP> Jn = m1_sum(jc, jc);
#pragma unroll
        for (int q = 0; q < NP; ++q) m1_step(I.v[q], Kf.v[q], Jf.v[q], Jn.v[q], make_float2(hl, hl));
    }
#pragma unroll
    for (int q = 0; q < NP; ++q) I.v[q] = make_float2(-I.v[q].x, -I.v[q].y);
    return I;
}

// Stores of a lane's columns: one vector store when aligned and owned, else
// one 4-byte store a column it owns.
template <int NP, bool VEC>
__device__ __forceinline__ void m1_store(float* __restrict__ p, const M1V<NP>& x, const bool (&own)[2 * NP]) {
    if constexpr (VEC && NP == 1) {
        if (own[0]) *reinterpret_cast<float2*>(p) = x.v[0];
    } else if constexpr (VEC) {
        if (own[0]) *reinterpret_cast<float4*>(p) = make_float4(x.v[0].x, x.v[0].y, x.v[1].x, x.v[1].y);
    } else {
#pragma unroll
        for (int q = 0; q < NP; ++q) {
            if (own[2 * q]) p[64 * q] = x.v[q].x;
            if (own[2 * q + 1]) p[64 * q + 32] = x.v[q].y;
        }
    }
}

// Block (point, bundle group) x tile of 64 NP columns; warp w is slice w of
// the group's plan; lane l owns the 2 NP adjacent columns from 2 NP l.  The
// last tile is shifted back to end at nk when nk >= the tile (columns below
// the tile are computed again and not written); a range shorter than a tile
// clamps the reads of lanes past it and writes nothing there.
template <int NP, bool VEC>
__global__ void __launch_bounds__(256, RAPRAL_MARCH_MINB) k_march1(MarchArgs a, int lgG, const int32_t* __restrict__ plan,
                                                                   const int32_t* __restrict__ soff,
                                                                   const int32_t* __restrict__ partner,
                                                                   float* __restrict__ part) {
    if (*a.status) return;
    constexpr int TW = 64 * NP, SLC = M1_SLICES, NC = 2 * NP;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nk = (int)a.nk;
    const int tile0 = (int)blockIdx.y * TW;
    const int base = (tile0 + TW > nk && nk >= TW) ? nk - TW : tile0;
    // the lane's columns: col .. col + NC - 1 (VEC), or col, col + 32, ...
    constexpr int CS = VEC ? 1 : 32;
    const int col = base + (VEC ? NC * lane : lane);
    const int c0 = col < nk ? col : nk - 1;           // clamped reads (VEC: never clamped)
    int dq[NC];
    bool own[NC];
#pragma unroll
    for (int q = 0; q < NC; ++q) {
        dq[q] = (col + CS * q < nk ? col + CS * q : nk - 1) - c0;
        own[q] = col + CS * q >= tile0 && col + CS * q < nk;
    }
    const char* kb = reinterpret_cast<const char*>(reinterpret_cast<const float*>(a.kappa) + c0);
    const char* jb = reinterpret_cast<const char*>(reinterpret_cast<const float*>(a.emis) + c0);
    __shared__ M1Stage stage_all[SLC][32];
    M1Stage* st = stage_all[warp];
    M1V<NP> acc, comp;
#pragma unroll
    for (int q = 0; q < NP; ++q) acc.v[q] = comp.v[q] = make_float2(0.f, 0.f);
    const int32_t* so = soff + (int64_t)blockIdx.x * (SLC + 1);
    const int k1 = so[warp + 1];
    for (int k = so[warp]; k < k1; ++k) {
        const int64_t b = plan[k];
        const int64_t d0 = a.dir_off[b];
        if (a.dir_off[b + 1] == d0) continue;
        M1V<NP> I0;
#pragma unroll
        for (int q = 0; q < NP; ++q) I0.v[q] = make_float2(0.f, 0.f);
        if (a.wall_row && a.bundle_wall[b]) I0 = m1_load<NP, VEC>(reinterpret_cast<const float*>(a.wall_row) + c0, dq);
        const M1V<NP> I = m1_bundle<NP, VEC>(a, b, a.dir_scale_f[d0], st, lane, kb, jb, dq, a.ld * 4, I0);
        if (a.I_out) m1_store<NP, VEC>(reinterpret_cast<float*>(a.I_out) + d0 * a.nk + col, I, own);
        float w = a.dir_weight_f[d0];
        const int b2 = partner ? partner[b] : -1;
        if (b2 >= 0) {   // the equal ray: its weight, and its intensities
            const int64_t d2 = a.dir_off[b2];
            w += a.dir_weight_f[d2];
            if (a.I_out) m1_store<NP, VEC>(reinterpret_cast<float*>(a.I_out) + d2 * a.nk + col, I, own);
        }
#pragma unroll
        for (int q = 0; q < NP; ++q) {   // compensated sum over the slice's bundles
            const float2 y = make_float2(w * I.v[q].x - comp.v[q].x, w * I.v[q].y - comp.v[q].y);
            const float2 tt = make_float2(acc.v[q].x + y.x, acc.v[q].y + y.y);
            comp.v[q] = make_float2((tt.x - acc.v[q].x) - y.x, (tt.y - acc.v[q].y) - y.y);
            acc.v[q] = tt;
        }
    }
    __shared__ M1V<NP> red[SLC][32];
    red[warp][lane] = acc;
    __syncthreads();
    if (warp == 0) {
        M1V<NP> sum = red[0][lane];
        for (int w = 1; w < SLC; ++w) {
#pragma unroll
            for (int q = 0; q < NP; ++q)
                sum.v[q] = make_float2(sum.v[q].x + red[w][lane].v[q].x, sum.v[q].y + red[w][lane].v[q].y);
        }
        float* dst = (lgG == 0 ? reinterpret_cast<float*>(a.q_lambda) : part) + (int64_t)blockIdx.x * a.nk + col;
        m1_store<NP, VEC>(dst, sum, own);
    }
}

// Planck intensity at the wall temperature for the columns of a range.
template <class T>
__global__ void k_planck_row(double lam_min, double h, int64_t k0, int64_t nk, double T_wall, Phys ph, T* row) {
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nk; k += (int64_t)gridDim.x * blockDim.x)
        row[k] = (T)planck(lam_min + (double)(k0 + k) * h, T_wall, ph);
}

// q_lambda[p][k] = sum of the G bundle-group partials of point p, in group order.
template <class T>
__global__ void k_group_sum(const T* __restrict__ part, int G, int64_t P, int64_t nk, T* __restrict__ q,
                            const int* status) {
    if (*status) return;
    const int64_t n = P * nk;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = i / nk, k = i - p * nk;
        const T* src = part + p * G * nk + k;
        T s = src[0];
        for (int g = 1; g < G; ++g) s += src[g * nk];
        q[i] = s;
    }
}

// Spectral integral in two deterministic stages: blocks (point, slice)
// Neumaier-sum a slice of flux_span(nk) grid points each, eight a thread, then
// one warp per point adds the slices, each lane a strided part in order.
// Weights other than 1 (the grid's ends) are applied to their points, the
// spacing once at the end: five FP64 operations a point.  The slices are a
// grid's second extent, 65,535 at most: ranges past 65,535 x 1,024 points take
// slices of 4,096.
constexpr int64_t MAX_FLUX_PARTS = 65535;
static int64_t flux_span(int64_t nk) { return nk <= MAX_FLUX_PARTS * 1024 ? 1024 : 4096; }

// (s, c) += x, Neumaier; magnitudes are compared by their bits
__device__ __forceinline__ void neumaier_add(double& s, double& c, double x) {
    const double t = s + x;
    const bool big = (__double_as_longlong(s) & 0x7fffffffffffffffll) >= (__double_as_longlong(x) & 0x7fffffffffffffffll);
    const double hi = big ? s : x, lo = big ? x : s;
    c += (hi - t) + lo;
    s = t;
}

template <class T>
__global__ void __launch_bounds__(128) k_wall_flux_part(const T* __restrict__ qlam, int64_t nk, int64_t k0,
                                                        int64_t n, int64_t span, double* __restrict__ part,
                                                        const int* status) {
    if (*status) return;
    const int64_t p = blockIdx.x;
    const int64_t a = (int64_t)blockIdx.y * span, b = min(a + span, nk);
    double s = 0.0, c = 0.0;
    for (int64_t k = a + threadIdx.x; k < b; k += blockDim.x) {
        const int64_t kg = k0 + k;
        double x = (double)qlam[p * nk + k];
        if (kg == 0 || kg == n - 1) x *= 0.5;
        neumaier_add(s, c, x);
    }
    __shared__ double red[4];
    double v = s + c;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 4; ++w) v += red[w];
        part[p * gridDim.y + blockIdx.y] = v;
    }
}

__global__ void __launch_bounds__(32) k_wall_flux_sum(const double* __restrict__ part, int nparts, double h_um,
                                                      double* __restrict__ q, const int* status) {
    if (*status) return;
    const int64_t p = blockIdx.x;
    double s = 0.0, c = 0.0;
    for (int i = threadIdx.x; i < nparts; i += 32) neumaier_add(s, c, part[p * nparts + i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {   // lane l + o into lane l
        const double s2 = __shfl_down_sync(0xffffffffu, s, o), c2 = __shfl_down_sync(0xffffffffu, c, o);
        neumaier_add(s, c, s2);
        c += c2;
    }
    if (threadIdx.x == 0) q[p] += (s + c) * h_um;
}

// Tangent slab: directions are split into bundles of at most SLAB_DIRS
// (the normal ray first); every bundle repeats the cell path.
__global__ void k_slab_rays(const int32_t* cell_order, const double* dx, int32_t m, const double* mu,
                            const double* wmu, int32_t n_mu, int32_t normal_ray, int32_t wall_start,
                            int64_t* point_off, int64_t* seg_off, int32_t* seg_cell, double* seg_ds,
                            int64_t* dir_off, double* dir_scale, double* dir_weight, int32_t* bundle_wall) {
    const int nd = n_mu + (normal_ray ? 1 : 0);
    const int nb = (nd + RAPRAL_SLAB_DIRS - 1) / RAPRAL_SLAB_DIRS;
    for (int64_t i = threadIdx.x; i < (int64_t)m * nb; i += blockDim.x) {
        const int64_t j = i % m;
        seg_cell[i] = cell_order[j];
        seg_ds[i] = dx[j];
    }
    for (int d = threadIdx.x; d < nd; d += blockDim.x) {
        if (normal_ray && d == 0) { dir_scale[0] = 1.0; dir_weight[0] = 0.0; continue; }
        const int mm = d - (normal_ray ? 1 : 0);
        dir_scale[d] = 1.0 / mu[mm];
        dir_weight[d] = 2.0 * M_PI * wmu[mm] * mu[mm];
    }
    for (int b = threadIdx.x; b <= nb; b += blockDim.x) {
        seg_off[b] = (int64_t)b * m;
        dir_off[b] = min(b * RAPRAL_SLAB_DIRS, nd);
        if (b < nb) bundle_wall[b] = wall_start;
    }
    if (threadIdx.x == 0) { point_off[0] = 0; point_off[1] = nb; }
}

__device__ __forceinline__ void ray_dir(int64_t b, int32_t n_mu, int32_t n_phi, const double* mu, int64_t* p,
                                        int* m, double* dx, double* dn, double* dt) {
    const int64_t per = (int64_t)n_mu * n_phi;
    *p = b / per;
    const int64_t rem = b - *p * per;
    *m = (int)(rem / n_phi);
    const int a = (int)(rem - (int64_t)(*m) * n_phi);
    const double mm = mu[*m];
    const double st = sqrt(1.0 - mm * mm);
    const double psi = (a + 0.5) * (2.0 * M_PI / n_phi);
    *dx = st * cos(psi);
    *dn = mm;
    *dt = st * sin(psi);
}

__global__ void k_axisym_count(const double* xf, int32_t nx, const double* rf, int32_t nr, const double* surf_x,
                               int32_t P, const double* mu, int32_t n_mu, int32_t n_phi, int64_t* counts) {
    const int64_t B = (int64_t)P * n_mu * n_phi;
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (b >= B) return;
    int64_t p; int m; double dx, dn, dt;
    ray_dir(b, n_mu, n_phi, mu, &p, &m, &dx, &dn, &dt);
    counts[b] = walk_ray(xf, nx, rf, nr, surf_x[p], rf[0], dx, dn, dt, nullptr, nullptr, 0);
}

__global__ void k_axisym_fill(const double* xf, int32_t nx, const double* rf, int32_t nr, const double* surf_x,
                              int32_t P, const double* mu, const double* wmu, int32_t n_mu, int32_t n_phi,
                              const int64_t* seg_off, int32_t* seg_cell, double* seg_ds, int64_t* point_off,
                              int64_t* dir_off, double* dir_scale, double* dir_weight, int32_t* bundle_wall) {
    const int64_t B = (int64_t)P * n_mu * n_phi;
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (b > B) return;
    dir_off[b] = b;
    if (b <= P) point_off[b] = b * (int64_t)n_mu * n_phi;
    if (b == B) return;
    int64_t p; int m; double dx, dn, dt;
    ray_dir(b, n_mu, n_phi, mu, &p, &m, &dx, &dn, &dt);
    walk_ray(xf, nx, rf, nr, surf_x[p], rf[0], dx, dn, dt, seg_cell, seg_ds, seg_off[b + 1]);
    dir_scale[b] = 1.0;
    dir_weight[b] = wmu[m] * mu[m] * (2.0 * M_PI / n_phi);
    bundle_wall[b] = 0;
}

#ifndef RAPRAL_MARCH_V
#define RAPRAL_MARCH_V 2
#endif

template <class T, int V, int MAXD, int SL, bool NODES = false, int DS = 0>
cudaError_t march_launch(rapral_ctx* ctx, const MarchArgs& a, int64_t P, int64_t nk, int G, void* part,
                         int n_split = 0) {
    const int W = DS ? n_split : march_warps(MAXD, SL);
    constexpr int TW = DS ? 32 * V : (march_warps(MAXD, SL) / SL) * 32 * V;
    int lgG = 0;
    while ((1 << lgG) < G) ++lgG;
    MarchArgs b = a;
    b.wall_row = nullptr;
    if (a.T_wall > 0.0) {   // the wall row follows the group partials in the scratch
        T* row = reinterpret_cast<T*>(part) + (G > 1 ? P * G * nk : 0);
        k_planck_row<T><<<(unsigned)std::min<int64_t>(div_up(nk, 256), 1024), 256, 0, ctx->stream>>>(
            a.lam_min, a.h, a.k0, nk, a.T_wall, a.ph, row);
        b.wall_row = row;
    }
    dim3 g((unsigned)(P << lgG), div_up(nk, TW));
    k_march<T, V, MAXD, SL, NODES, DS><<<g, 32 * W, 0, ctx->stream>>>(b, lgG, reinterpret_cast<T*>(part));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess || G == 1) return e;
    k_group_sum<T><<<(unsigned)std::min<int64_t>(div_up(P * nk, 256), 152 * 16), 256, 0, ctx->stream>>>(
        reinterpret_cast<const T*>(part), G, P, nk, reinterpret_cast<T*>(a.q_lambda), a.status);
    return cudaGetLastError();
}

// k_march1 applies: FP32 cell-valued single-direction bundles, eight or more
// a point.
static bool march1_applies(const MarchArgs& a, int maxd, int maxb, bool nodes) {
    return !nodes && maxd <= 1 && maxb >= 8 && a.ld <= 2147483647LL;
}

// Whether a lane's 2 NP adjacent columns can be loaded and stored as one
// vector: every row of kappa / emis, q_lambda, I_out and the wall row starts
// aligned to 8 NP bytes, and the range is whole tiles or ends on a multiple of
// 2 NP columns past the first tile.
static bool march1_vec(const MarchArgs& a, int64_t nk, const void* part, int NP) {
    const unsigned al = 8u * NP - 1u;
    const auto ok = [al](const void* q) { return (reinterpret_cast<uintptr_t>(q) & al) == 0; };
    const int64_t nc = 2 * NP;
    return nk >= 64 * NP && nk % nc == 0 && a.ld % nc == 0 && ok(a.kappa) && ok(a.emis) && ok(a.q_lambda) &&
           ok(part) && (a.I_out == nullptr || ok(a.I_out));
}

// The march's plan: the equal rays and the slices of every (point, group).
struct M1Plan {
    unsigned long long* key;   // [n_bundles]
    int32_t *partner, *cand, *plan;   // [n_bundles]
    int32_t* soff;             // [n_points G (M1_SLICES + 1)]
};

static cudaError_t march1_launch(rapral_ctx* ctx, const MarchArgs& a, int64_t P, int64_t B, int64_t n_segments,
                                 int64_t nk, int maxb, int G, void* part, const M1Plan& pl) {
    int lgG = 0;
    while ((1 << lgG) < G) ++lgG;
    const bool pairs = B > 0 && nk >= M1_PAIR_COLUMNS && n_segments * nk >= M1_PAIR_WORK;
    int32_t *cand = pairs ? pl.cand : nullptr, *partner = pairs ? pl.partner : nullptr;
    if (pairs) {
        const dim3 gm((unsigned)P, div_up(std::min(maxb, M1_PAIR_MAX), MATCH_BUNDLES));
        k_ray_hash<<<div_up(B * 32, 256), 256, 0, ctx->stream>>>(a, P, B, pl.key, cand, partner);
        k_ray_match<<<gm, MATCH_THREADS, 0, ctx->stream>>>(a, pl.key, cand, partner);
    }
    k_march_plan<<<(unsigned)(P * G), 128, 0, ctx->stream>>>(a.point_off, a.seg_off, cand, G, pl.plan, pl.soff,
                                                             a.status);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    MarchArgs b = a;
    b.wall_row = nullptr;
    if (a.T_wall > 0.0) {   // the wall row follows the group partials in the scratch
        float* row = reinterpret_cast<float*>(part) + (G > 1 ? P * G * nk : 0);
        k_planck_row<float><<<(unsigned)std::min<int64_t>(div_up(nk, 256), 1024), 256, 0, ctx->stream>>>(
            a.lam_min, a.h, a.k0, nk, a.T_wall, a.ph, row);
        b.wall_row = row;
    }
    // four adjacent columns a lane where 16-byte loads are aligned (100 x 50
    // cells, 20 points x 512 rays, 16,384 columns: 3.93 ms, two columns 4.16),
    // two where 8-byte ones are (16,382: 4.24), else two columns 32 apart (16,383:
    // 4.72, four of them 4.95).  Four halve the blocks, so they wait for ten
    // blocks an SM, two and a half waves: 10 points x 512 rays of 80 segments,
    // 128 / 512 / 1,024 / 1,536 / 2,048 / 4,096 columns (160 to 5,120 blocks of
    // four) 146 / 252 / 377 / 506 / 637 / 1,199 us with four, 114 / 227 / 365 /
    // 516 / 656 / 1,251 with two; 200 points x 64 rays, 256 and 512 columns (800,
    // 1,600) 166 and 255 with four, 156 and 258 with two.
    float* pf = reinterpret_cast<float*>(part);
    const auto grid = [&](int np) { return dim3((unsigned)(P << lgG), div_up(nk, 64 * np)); };
    const bool four = (P << lgG) * (int64_t)div_up(nk, 128) >= 152 * 10;
    if (four && march1_vec(a, nk, part, 2))
        k_march1<2, true><<<grid(2), 32 * M1_SLICES, 0, ctx->stream>>>(b, lgG, pl.plan, pl.soff, partner, pf);
    else if (march1_vec(a, nk, part, 1))
        k_march1<1, true><<<grid(1), 32 * M1_SLICES, 0, ctx->stream>>>(b, lgG, pl.plan, pl.soff, partner, pf);
    else
        k_march1<1, false><<<grid(1), 32 * M1_SLICES, 0, ctx->stream>>>(b, lgG, pl.plan, pl.soff, partner, pf);
    e = cudaGetLastError();
    if (e != cudaSuccess || G == 1) return e;
    k_group_sum<float><<<(unsigned)std::min<int64_t>(div_up(P * nk, 256), 152 * 16), 256, 0, ctx->stream>>>(
        reinterpret_cast<const float*>(part), G, P, nk, reinterpret_cast<float*>(a.q_lambda), a.status);
    return cudaGetLastError();
}

// Eight bundle slices for eight or more bundles a point, else one; V > 1
// columns a lane only for one-direction bundles in FP32 and ranges of at
// least one tile.
template <class T>
cudaError_t march_t(rapral_ctx* ctx, const MarchArgs& a, int64_t P, int64_t nk, int maxd, int maxb, int G,
                    void* part, bool nodes) {
    constexpr int VR = sizeof(T) == 4 ? RAPRAL_MARCH_V : 1;
    if (nodes) {   // node-valued lines of sight: one direction a bundle (checked by the caller)
        if (maxb < 8) return march_launch<T, 1, 1, 1, true>(ctx, a, P, nk, G, part);
        if (VR > 1 && nk >= 32 * VR) return march_launch<T, VR, 1, 8, true>(ctx, a, P, nk, G, part);
        return march_launch<T, 1, 1, 8, true>(ctx, a, P, nk, G, part);
    }
    if (maxb >= 8) {
        if (maxd <= 1) {
            if (VR > 1 && nk >= 32 * VR) return march_launch<T, VR, 1, 8>(ctx, a, P, nk, G, part);
            return march_launch<T, 1, 1, 8>(ctx, a, P, nk, G, part);
        }
        if (maxd <= 17) return march_launch<T, 1, 17, 8>(ctx, a, P, nk, G, part);
        return march_launch<T, 1, RAPRAL_MAX_DIRS, 8>(ctx, a, P, nk, G, part);
    }
    if (maxd <= 1) return march_launch<T, 1, 1, 1>(ctx, a, P, nk, G, part);
    // A warp takes a bundle's directions one after the other, 1,400 cycles a
    // step of 17 in FP32 however idle the chip is.  Up to 11 column tiles an SM
    // they are split over warps of three: FP32, 200 cells x 17 directions x
    // 5,000 / 20,000 / 45,000 / 55,000 / 65,000 columns 183 / 201 / 234 / 248 /
    // 268 us in one warp, 76 / 105 / 160 / 237 / 301 split (five each: 104 / 127
    // / 173 / 199 / 242; 8 directions, 100 cells, 55,000: 89, 71 split by threes,
    // 70 by fives).  In FP64 the pipe is what bounds the march and the split
    // keeps it fed at every size: 60 cells x 17 directions x 5,000 / 20,000 /
    // 60,000 / 100,001 columns 1,160 / 1,405 / 2,762 / 3,240 us in one warp, 465 /
    // 840 / 1,820 / 2,820 by threes, 680 / 1,048 / 1,864 / 2,680 by sevens, which
    // are taken above the line.  In FP32 fives are the best form at 55,000 and
    // 65,000 columns and no branch takes them: where they stop paying has not
    // been measured.
    if (maxd <= 17 && P * div_up(nk, 32) <= 152 * 11)
        return march_launch<T, 1, 3, 1, false, 6>(ctx, a, P, nk, G, part, std::max(1, (int)div_up(maxd, 3)));
    if constexpr (sizeof(T) == 8) {
        if (maxd <= 17)
            return march_launch<T, 1, 7, 1, false, 3>(ctx, a, P, nk, G, part, std::max(1, (int)div_up(maxd, 7)));
    } else {
        if (maxd <= 17) return march_launch<T, 1, 17, 1>(ctx, a, P, nk, G, part);
    }
    return march_launch<T, 1, RAPRAL_MAX_DIRS, 1>(ctx, a, P, nk, G, part);
}

}  // namespace

// Bundle groups per point where a point has eight or more bundles (a power of two):
// enough blocks share a wavelength tile (points x groups >= 1536, about two
// waves of resident blocks) that the tiles in flight, and so the kappa / j
// rows they gather, stay few enough for L2; each group keeps at least 32
// bundles, and points x groups stays below 2^31.
#ifndef RAPRAL_MARCH_TILE_BLOCKS
#define RAPRAL_MARCH_TILE_BLOCKS 1536
#endif
static int march_groups(const rapral_rays* r) {
    if (r->max_bundles_per_point < 8 || r->n_points <= 0) return 1;
    int G = 1;
    while (G * r->n_points < RAPRAL_MARCH_TILE_BLOCKS && 2 * G * 32 <= r->max_bundles_per_point && G < 1024 &&
           2 * G * r->n_points < (int64_t)1 << 31)
        G *= 2;
    return G;
}

static size_t round256(size_t x) { return (x + 255) / 256 * 256; }

// FP32 scratch: the FP32 copies of lengths, scales and weights (each from a
// multiple of 64 floats), then k_march1's plan.
static size_t march_copy_bytes(const rapral_rays* r) {
    return round256((size_t)(r->n_segments + 2 * r->n_dirs + 128) * sizeof(float));
}
static size_t march_plan_bytes(const rapral_rays* r) {
    return round256((size_t)r->n_bundles * 8) + 3 * round256((size_t)r->n_bundles * 4) +
           round256((size_t)r->n_points * march_groups(r) * (M1_SLICES + 1) * 4);
}

size_t march_scratch_bytes(const rapral_rays* r, int64_t nk, int precision) {
    size_t bytes = 0;
    if (precision == RAPRAL_FP32) bytes = march_copy_bytes(r) + march_plan_bytes(r);
    const int G = march_groups(r);
    const size_t el = precision == RAPRAL_FP64 ? sizeof(double) : sizeof(float);
    if (G > 1) bytes += (size_t)r->n_points * G * nk * el;
    return bytes + nk * el + 256;   // + the wall's Planck row
}

cudaError_t launch_validate_rays(rapral_ctx* ctx, const rapral_rays* r, int64_t n_cells, void* copies) {
    const int64_t n = r->n_segments > r->n_dirs ? r->n_segments : r->n_dirs;
    if (n == 0) return cudaSuccess;
    float* f = reinterpret_cast<float*>(copies);
    float* fd = f ? f + ((r->n_segments + 63) / 64) * 64 : nullptr;
    float* fw = f ? fd + ((r->n_dirs + 63) / 64) * 64 : nullptr;
    k_validate_rays<<<div_up(n, 256), 256, 0, ctx->stream>>>(r->seg_cell, r->seg_ds, r->n_segments, n_cells,
                                                            r->dir_scale, r->dir_weight, r->n_dirs, f, fd, fw,
                                                            ctx->d_status);
    return cudaGetLastError();
}

cudaError_t launch_march(rapral_ctx* ctx, const rapral_rays* r, const void* kappa, const void* emis, int64_t ld,
                         const rapral_grid* g, double h, int64_t k0, int64_t nk, int precision, void* q_lambda,
                         void* I_out, const Phys& ph, void* scratch) {
    MarchArgs a;
    a.point_off = r->point_off; a.seg_off = r->seg_off; a.seg_cell = r->seg_cell; a.seg_ds = r->seg_ds;
    a.dir_off = r->dir_off; a.dir_scale = r->dir_scale; a.dir_weight = r->dir_weight;
    a.seg_ds_f = nullptr; a.dir_scale_f = nullptr; a.dir_weight_f = nullptr;
    a.bundle_wall = r->bundle_wall; a.T_wall = r->T_wall; a.wall_row = nullptr;
    a.kappa = kappa; a.emis = emis; a.ld = ld;
    a.lam_min = g->lam_min; a.h = h; a.k0 = k0; a.nk = nk;
    a.q_lambda = q_lambda; a.I_out = I_out; a.ph = ph; a.status = ctx->d_status;
    const int G = march_groups(r);
    if (precision == RAPRAL_FP64)
        return march_t<double>(ctx, a, r->n_points, nk, r->max_dirs, r->max_bundles_per_point, G, scratch,
                               r->node_values != 0);
    // the FP32 copies (written by launch_validate_rays), the plan, then the group partials
    char* at = reinterpret_cast<char*>(scratch);
    a.seg_ds_f = reinterpret_cast<float*>(at);
    a.dir_scale_f = a.seg_ds_f + ((r->n_segments + 63) / 64) * 64;
    a.dir_weight_f = a.dir_scale_f + ((r->n_dirs + 63) / 64) * 64;
    at += march_copy_bytes(r);
    void* part = at + march_plan_bytes(r);
    M1Plan pl;
    const auto take = [&at](size_t bytes) { char* p = at; at += round256(bytes); return p; };
    pl.key = reinterpret_cast<unsigned long long*>(take((size_t)r->n_bundles * 8));
    pl.partner = reinterpret_cast<int32_t*>(take((size_t)r->n_bundles * 4));
    pl.cand = reinterpret_cast<int32_t*>(take((size_t)r->n_bundles * 4));
    pl.plan = reinterpret_cast<int32_t*>(take((size_t)r->n_bundles * 4));
    pl.soff = reinterpret_cast<int32_t*>(take((size_t)r->n_points * G * (M1_SLICES + 1) * 4));
    if (march1_applies(a, r->max_dirs, r->max_bundles_per_point, r->node_values != 0))
        return march1_launch(ctx, a, r->n_points, r->n_bundles, r->n_segments, nk,
                              r->max_bundles_per_point, G, part, pl);
    return march_t<float>(ctx, a, r->n_points, nk, r->max_dirs, r->max_bundles_per_point, G, part,
                          r->node_values != 0);
}

int64_t wall_flux_parts(int64_t nk) { return (nk + flux_span(nk) - 1) / flux_span(nk); }

cudaError_t launch_wall_flux(rapral_ctx* ctx, const void* q_lambda, int precision, const rapral_grid* g, double h,
                             int64_t k0, int64_t nk, int64_t n_points, double* q, void* partials) {
    if (n_points == 0) return cudaSuccess;
    const double h_um = h * 1e-3;
    const int64_t np = wall_flux_parts(nk);
    double* part = reinterpret_cast<double*>(partials);
    dim3 grid((unsigned)n_points, (unsigned)np);
    if (precision == RAPRAL_FP64)
        k_wall_flux_part<double><<<grid, 128, 0, ctx->stream>>>(reinterpret_cast<const double*>(q_lambda), nk, k0,
                                                                g->n, flux_span(nk), part, ctx->d_status);
    else
        k_wall_flux_part<float><<<grid, 128, 0, ctx->stream>>>(reinterpret_cast<const float*>(q_lambda), nk, k0,
                                                               g->n, flux_span(nk), part, ctx->d_status);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_wall_flux_sum<<<(unsigned)n_points, 32, 0, ctx->stream>>>(part, (int)np, h_um, q, ctx->d_status);
    return cudaGetLastError();
}

cudaError_t launch_slab_rays(rapral_ctx* ctx, const int32_t* cell_order, const double* dx, int32_t m,
                             const double* mu, const double* wmu, int32_t n_mu, int32_t normal_ray,
                             int32_t wall_start, int64_t* point_off, int64_t* seg_off, int32_t* seg_cell,
                             double* seg_ds, int64_t* dir_off, double* dir_scale, double* dir_weight,
                             int32_t* bundle_wall) {
    k_slab_rays<<<1, 256, 0, ctx->stream>>>(cell_order, dx, m, mu, wmu, n_mu, normal_ray, wall_start, point_off,
                                           seg_off, seg_cell, seg_ds, dir_off, dir_scale, dir_weight, bundle_wall);
    return cudaGetLastError();
}

cudaError_t launch_axisym_count(rapral_ctx* ctx, const double* xf, int32_t nx, const double* rf, int32_t nr,
                                const double* surf_x, int32_t P, const double* mu, int32_t n_mu, int32_t n_phi,
                                int64_t* seg_off, int64_t* scan_tmp) {
    (void)scan_tmp;
    const int64_t B = (int64_t)P * n_mu * n_phi;
    if (B == 0) return cudaSuccess;
    k_axisym_count<<<div_up(B, 128), 128, 0, ctx->stream>>>(xf, nx, rf, nr, surf_x, P, mu, n_mu, n_phi, seg_off);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return launch_scan_i64(ctx, seg_off, B);
}

cudaError_t launch_axisym_fill(rapral_ctx* ctx, const double* xf, int32_t nx, const double* rf, int32_t nr,
                               const double* surf_x, int32_t P, const double* mu, const double* wmu, int32_t n_mu,
                               int32_t n_phi, const int64_t* seg_off, int32_t* seg_cell, double* seg_ds,
                               int64_t* point_off, int64_t* dir_off, double* dir_scale, double* dir_weight,
                               int32_t* bundle_wall) {
    const int64_t B = (int64_t)P * n_mu * n_phi;
    k_axisym_fill<<<div_up(B + 1, 128), 128, 0, ctx->stream>>>(xf, nx, rf, nr, surf_x, P, mu, wmu, n_mu, n_phi,
                                                               seg_off, seg_cell, seg_ds, point_off, dir_off,
                                                               dir_scale, dir_weight, bundle_wall);
    return cudaGetLastError();
}
