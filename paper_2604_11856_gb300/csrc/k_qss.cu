// Quasi-steady-state collisional-radiative populations (Sec. 2.1): per cell
// and atomic radiator, the rate matrix R and source b of the QSS master
// equation, solved by LU with partial pivoting.  One warp per cell: lanes
// compute the transitions' up / down rates and store them in the rows that gain
// by them (added in order where a pair of levels has several transitions);
// lane r sums column r, what its level loses, for the diagonal, pivots and
// eliminates its row, and the warp substitutes back column by column.  FP64
// throughout: the systems span many orders of magnitude in their rates.
//
// The FP64 pipe bounds it (a warp instruction of it takes 17 clocks of an SM,
// whatever lanes are on; it is 89 % busy), so the count
// of FP64 warp instructions a cell is what the layout keeps down: 32 sums for
// the diagonals of 32 rows (from lists of each row's transitions two a list
// entry, by transitions four with two lanes on, 1,984 for 496), exponentials
// and pivot comparisons on the integer pipe, divisions one Newton reciprocal a
// level or pivot, back substitution one instruction a column instead of one
// lane's 496.  The rates need no store of their own, so 16 warps an SM fit
// (eight with one).  20,000 cells of 32 + 4 levels, 496 transitions: 6.57 ->
// 2.25 ms, then 2.09 without the lists and the rates' store.
#include <algorithm>

#include "rapral_internal.cuh"
#include "exp_fix.cuh"

namespace {

constexpr int QW = 4;          // warps (cells) per block
constexpr int QMAXL = 32;      // levels solved
constexpr int QMAXT = QMAXL * (QMAXL - 1) / 2;
constexpr double N_AVOGADRO = 6.022e23;

// inf or NaN, on the integer pipe
__device__ __forceinline__ bool nonfinite(double x) { return (__double2hiint(x) & 0x7ff00000) == 0x7ff00000; }

// 1 / x: an FP32 reciprocal of the leading part and one Newton step of third
// order (relative error of the seed e: the result's is e^3 plus rounding),
// where x is well inside the FP32 range; the division elsewhere.
__device__ __forceinline__ double recip64(double x) {
    const int ex = (__double2hiint(x) >> 20) & 0x7ff;
    if (ex < 1023 - 100 || ex > 1023 + 100) return 1.0 / x;
    // x's leading 24 bits as a float, without the FP64 pipe's conversion
    const long long bits = __double_as_longlong(x);
    const unsigned fb = ((unsigned)(bits >> 32) & 0x80000000u) | ((unsigned)(ex - 896) << 23) |
                        (unsigned)((bits >> 29) & 0x7fffff);
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(__uint_as_float(fb)));
    const unsigned rb = __float_as_uint(r);
    const double y = __longlong_as_double(((long long)(rb & 0x80000000u) << 32) |
                                          ((long long)((rb >> 23 & 0xff) + 896) << 52) |
                                          ((long long)(rb & 0x7fffff) << 29));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

__global__ void __launch_bounds__(32 * QW, 4)
    k_qss(rapral_cr_model m, rapral_cells cells, Phys ph, double* n_out, int* status) {
    // one decision for the block: its warps fill the shared tables together,
    // and other blocks of this launch may be setting the status meanwhile
    if (__syncthreads_or(*status != 0)) return;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    __shared__ uint64_t tab[EXPFIX_N];
    __shared__ double Rs[QW][QMAXL][QMAXL + 1];
    __shared__ double bs[QW][QMAXL];
    __shared__ double Qh[QW][QMAXL], Qv[QW][QMAXL], iQh[QW][QMAXL], iQv[QW][QMAXL];
    __shared__ unsigned char slo[QMAXT], sup[QMAXT];
    __shared__ unsigned pairs[QMAXL], twice;   // level i: a bit per j > i with a transition; any pair has several
    const int l = m.n_levels, T = m.n_trans, nc = cells.n_cols;
    expfix_load(tab);
    if (threadIdx.x < QMAXL) pairs[threadIdx.x] = 0u;
    if (threadIdx.x == 0) twice = 0u;
    __syncthreads();
    // every transition is checked before any indexed use
    bool bad = false;
    for (int t = threadIdx.x; t < T; t += blockDim.x) {
        const int i = m.lo[t], j = m.up[t];
        if (i < 0 || j <= i || j >= l) {
            fail(status, CHK_CR_TRANS, t);
            bad = true;
            continue;
        }
        slo[t] = (unsigned char)i;
        sup[t] = (unsigned char)j;
    }
    if (__syncthreads_or(bad)) return;
    for (int t = threadIdx.x; t < T; t += blockDim.x)
        if (atomicOr(&pairs[slo[t]], 1u << sup[t]) >> sup[t] & 1u) twice = 1u;
    __syncthreads();
    double (*R)[QMAXL + 1] = Rs[w];
    double* b = bs[w];
    for (int64_t c = (int64_t)w * gridDim.x + blockIdx.x; c < cells.n_cells; c += (int64_t)gridDim.x * QW) {
        const double Ttr = cells.Ttr[c], Tve = cells.Tve[c];
        const double* dens = cells.n + c * nc;
        double nM = 0.0;
        for (int k = 0; k < nc; ++k)
            if (k != cells.ne_col) nM += dens[k];
        const double ne = dens[cells.ne_col];
        const double nion = m.ion_col >= 0 ? dens[m.ion_col] : 0.0;
        const double lnTtr = log(Ttr), lnTve = log(Tve), iTtr = 1.0 / Ttr, iTve = 1.0 / Tve;
        const double nMa = nM * (1.0 / N_AVOGADRO), nea = ne * (1.0 / N_AVOGADRO);
        __syncwarp();
        if (lane < l)
            for (int j = 0; j < l; ++j) R[j][lane] = 0.0;
        // level weights Q_i = g_i e^{-c2 E_i / T} at both temperatures
        if (lane < l) {
            const double g = m.g[lane], x = -ph.c2 * m.E[lane];
            const double qh = g * exp_fix(x * iTtr, tab), qv = g * exp_fix(x * iTve, tab);
            Qh[w][lane] = qh;
            Qv[w][lane] = qv;
            iQh[w][lane] = recip64(qh);
            iQv[w][lane] = recip64(qv);
        }
        __syncwarp();
        // transition rates per particle of the lower (up) / upper (down) level,
        // straight to the rows that gain by them: R[upper][lower], R[lower][upper]
        for (int t0 = 0; t0 < T; t0 += 32) {
            const int t = min(t0 + lane, T - 1);
            const int i = slo[t], j = sup[t];
            // C T^n e^{-theta/T} as C e^{n ln T - theta/T}: one exp a rate
            const double theta = ph.c2 * (m.E[j] - m.E[i]);
            const double kh_up = m.hp_C[t] * exp_fix(m.hp_n[t] * lnTtr - theta * iTtr, tab);
            const double ke_up = m.e_C[t] * exp_fix(m.e_n[t] * lnTve - theta * iTve, tab);
            double kh_dn = kh_up * Qh[w][i] * iQh[w][j];
            double ke_dn = ke_up * Qv[w][i] * iQv[w][j];
            if (nonfinite(kh_dn) || nonfinite(ke_dn)) {   // weights below 2^-1022 (cold cells)
                kh_dn = kh_up * Qh[w][i] / Qh[w][j];
                ke_dn = ke_up * Qv[w][i] / Qv[w][j];
            }
            const double rad = m.lam[t] >= 200.0 ? m.A[t] : 0.0;
            const double up = kh_up * nMa + ke_up * nea, dn = kh_dn * nMa + ke_dn * nea + rad;
            if (!twice) {
                R[j][i] = up;
                R[i][j] = dn;
            } else {   // pairs of levels with several transitions: added in their order
                for (int q = 0; q < 32 && t0 + q < T; ++q) {
                    if (lane == q) {
                        R[j][i] += up;
                        R[i][j] += dn;
                    }
                    __syncwarp();
                }
            }
        }
        // lane r completes row r; what level r loses is what the others gain, column r
        double diag = 0.0;
        __syncwarp();
        if (lane < l) {
            double d[4] = {0.0, 0.0, 0.0, 0.0};
            int j = 0;
            for (; j + 3 < l; j += 4)
#pragma unroll
                for (int q = 0; q < 4; ++q) d[q] -= R[j + q][lane];
            for (; j < l; ++j) d[0] -= R[j][lane];
            diag = (d[0] + d[1]) + (d[2] + d[3]);
        }
        __syncwarp();
        if (lane < l) {
            if (lane > 0) {
                // electron-impact ionisation and three-body recombination
                const double Qp = m.g_ion * exp_fix(-ph.c2 * m.E_ionize * iTve, tab);
                const double x = 2.0 * M_PI * ph.me * ph.kB * Tve / (ph.h * ph.h);
                const double Qe = 2.0 * (x * sqrt(x));
                const double kf = m.ii_C[lane] * exp_fix(m.ii_n[lane] * lnTve, tab) *
                                  exp_fix(-ph.c2 * (m.E_ionize - m.E[lane]) * iTve, tab);
                const double kr = kf * Qv[w][lane] / (Qp * Qe);
                R[lane][lane] = diag - kf * nea;
                b[lane] = -kr * nion * ne * nea;
            } else {   // closure: the levels and the lumped ones above sum to the density
                for (int j = 0; j < l; ++j) R[0][j] = 1.0;
                if (m.n_levels_all > l) {
                    double s = 0.0;
                    for (int p = l; p < m.n_levels_all; ++p) s += m.g[p] * exp_fix(-ph.c2 * m.E[p] * iTve, tab);
                    R[0][l - 1] = 1.0 + s / Qv[w][l - 1];
                }
                b[0] = dens[m.col];
            }
        }
        __syncwarp();
        // LU with partial pivoting (the first largest |R[r][k]| of rows r >= k;
        // non-negative doubles order like their bits)
        bool singular = false;
        double inv_own = 0.0;   // lane k: 1 / pivot k
        for (int k = 0; k < l; ++k) {
            const unsigned long long v =
                (lane >= k && lane < l) ? (unsigned long long)__double_as_longlong(R[lane][k]) & ~(1ull << 63) : 0ull;
            const unsigned hi = (unsigned)(v >> 32), mhi = __reduce_max_sync(0xffffffffu, hi);
            const unsigned lo = hi == mhi ? (unsigned)v : 0u, mlo = __reduce_max_sync(0xffffffffu, lo);
            if ((mhi | mlo) == 0u || mhi > 0x7ff00000u || (mhi == 0x7ff00000u && mlo)) {   // zero or NaN
                singular = true;
                break;
            }
            const unsigned at = __ballot_sync(0xffffffffu, lane >= k && lane < l && hi == mhi && lo == mlo);
            const int p = __ffs(at) - 1;
            if (p != k) {
                if (lane < l) { const double x = R[k][lane]; R[k][lane] = R[p][lane]; R[p][lane] = x; }
                if (lane == 0) { const double x = b[k]; b[k] = b[p]; b[p] = x; }
                __syncwarp();
            }
            const double piv = R[k][k], inv = recip64(piv);
            if (lane == k) inv_own = inv;
            if (lane > k && lane < l) {
                const double r = R[lane][k];
                double f = r * inv;
                f = fma(fma(-f, piv, r), inv, f);   // the quotient, rounded once
                if (nonfinite(f)) f = r / piv;      // pivots below 2^-1022
                R[lane][k] = f;
                int j = k + 1;
                for (; j + 3 < l; j += 4) {   // loads ahead of the stores, which the compiler has to keep in order
                    double x[4], y[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) x[q] = R[k][j + q], y[q] = R[lane][j + q];
#pragma unroll
                    for (int q = 0; q < 4; ++q) R[lane][j + q] = fma(-f, x[q], y[q]);
                }
                for (; j < l; ++j) R[lane][j] = fma(-f, R[k][j], R[lane][j]);
                b[lane] = fma(-f, b[k], b[lane]);
            }
            __syncwarp();
        }
        if (singular) {
            if (lane == 0) fail(status, CHK_CR_SINGULAR, c);
            continue;
        }
        // back substitution, a column at a time
        double x = lane < l ? b[lane] : 0.0;
        for (int i = l - 1; i >= 0; --i) {
            const double piv = R[i][i];
            double xi = x * inv_own;
            xi = fma(fma(-xi, piv, x), inv_own, xi);
            if (nonfinite(xi)) xi = x / piv;
            xi = __shfl_sync(0xffffffffu, xi, i);
            if (lane == i) x = xi;
            else if (lane < i) x = fma(-R[lane][i], xi, x);
        }
        if (lane < l) n_out[c * l + lane] = x;
    }
}

// Departure coefficients of the model's levels (Sec. 2.1): ln b_i = ln N_i -
// ln N_i^B with the Boltzmann population of the main path, ln N_i^B =
// lnpref + ln g_i - c2 E_i / T_ve.  One thread per (cell, level slot); slots
// past the model's levels hold 0 (b = 1).
__global__ void k_qss_departures(const double* __restrict__ E, const double* __restrict__ g, int l,
                                 const double* __restrict__ Tve, const double* __restrict__ lnpref,
                                 const double* __restrict__ n_qss, int64_t C, int s, int S, int n_lev, double c2,
                                 double* __restrict__ ln_b, int* status) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= C * n_lev) return;
    const int64_t c = i / n_lev;
    const int k = (int)(i - c * n_lev);
    double v = 0.0;
    if (k < l) {
        const double N = n_qss[c * l + k];
        if (!(N > 0.0)) {
            fail(status, CHK_CR_POP, c);
            v = 0.0;
        } else {
            v = log(N) - (lnpref[c * S + s] + log(g[k]) - c2 * E[k] / Tve[c]);
        }
    }
    ln_b[(c * S + s) * n_lev + k] = v;
}

__global__ void k_check_levels(const int32_t* __restrict__ u, const int32_t* __restrict__ lo, int64_t L, int n_lev,
                               int* status) {
    const int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= L) return;
    const int a = u[l], b = lo[l];
    if (a < -1 || a >= n_lev || b < -1 || b >= n_lev) fail(status, CHK_DEP_LEVEL, l);
}

}  // namespace

cudaError_t launch_qss(rapral_ctx* ctx, const rapral_cr_model* m, const rapral_cells* cells, double* n_out,
                       const Phys& ph) {
    if (cells->n_cells == 0) return cudaSuccess;
    if (m->n_trans > QMAXT || m->n_levels > QMAXL) return cudaErrorInvalidValue;
    // four blocks an SM fit (shared memory); each takes cells until none is
    // left, and the first cells go to a warp of every block
    const int64_t blocks = std::min<int64_t>(cells->n_cells, 152 * 4);
    k_qss<<<(unsigned)blocks, 32 * QW, 0, ctx->stream>>>(*m, *cells, ph, n_out, ctx->d_status);
    return cudaGetLastError();
}

cudaError_t launch_qss_departures(rapral_ctx* ctx, const rapral_cr_model* m, const rapral_cells* cells, int32_t s,
                                  int32_t S, const double* n_qss, double* ln_b, int32_t n_lev, const Phys& ph) {
    const int64_t n = cells->n_cells * n_lev;
    if (n == 0) return cudaSuccess;
    k_qss_departures<<<div_up(n, 256), 256, 0, ctx->stream>>>(m->E, m->g, m->n_levels, cells->Tve, cells->lnpref,
                                                             n_qss, cells->n_cells, s, S, n_lev, ph.c2, ln_b,
                                                             ctx->d_status);
    return cudaGetLastError();
}

cudaError_t launch_check_levels(rapral_ctx* ctx, const int32_t* lev_u, const int32_t* lev_l, int64_t L,
                                int32_t n_lev) {
    if (L == 0) return cudaSuccess;
    k_check_levels<<<div_up(L, 256), 256, 0, ctx->stream>>>(lev_u, lev_l, L, n_lev, ctx->d_status);
    return cudaGetLastError();
}
