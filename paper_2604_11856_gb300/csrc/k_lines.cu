// Line preparation, spectral-tile binning and the line-by-line sum
// (Sec. 2.2.1 atoms, Sec. 2.2.2 diatomics).
//
// Binning (deterministic, ordered by line index):
//   k_line_plan    per line, the checks, the tiles its window can touch in any
//                  cell of the request, from a conservative width: lamV <=
//                  lamL + lamG with both widths at their largest over the
//                  cells, and the record of a line that touches one
//   k_bin_count    one block per tile: scan the lines whose centre lies within
//                  the widest window of the tile, count those that reach it
//   scan           exclusive prefix of the counts -> CSR offsets
//   k_bin_fill     same scan, ordered compaction of the line indices
//
// Line sum, FP64: one block per (tile, cell).  Thread i owns the points i,
// i + 128, ... of the tile.  Lines of the tile are processed in batches of
// blockDim: each thread sets up one (line, cell) pair -- populations in log
// space, strengths, Doppler / Stark / Voigt widths, profile normalisation and
// the window -- into shared memory; then every thread evaluates the profile
// of each staged pair at its own points inside that pair's window and
// accumulates kappa and j.  Results are written once, coalesced.  FP32: one
// warp per (tile, cell), described with its kernel below.
//
// Optional per-context parts, each a template flag of the kernels so that the
// default path is unchanged: the full Lorentz width (Stark from the
// ionisation gap, resonance, van der Waals), departure coefficients of
// collisional-radiative levels, and the exact Voigt shape (voigt.cuh) in
// place of Whiting's fit.
#include "rapral_internal.cuh"
#include "exp_fix.cuh"

// the rational Faddeeva expansion's coefficients (exact Voigt line shape)
__constant__ VoigtCoef c_voigt;

namespace {

__device__ __forceinline__ double voigt_hwhm(double lamL, double lamG) {
    const double d = (lamL - lamG) / (lamL + lamG);
    return (1.0 - 0.18121 * (1.0 - d * d) - (0.023665 * exp(0.6 * d) + 0.00418 * exp(-1.9 * d)) * sin(M_PI * d)) *
           (lamL + lamG);
}

// Checks one line; a failed check is recorded and the line gets no record.
__device__ __forceinline__ bool check_line(const rapral_lines& ln, int32_t S, int64_t l, int* status) {
    bool ok = true;
    const int s = ln.species[l];
    if (s < 0 || s >= S) fail(status, CHK_LINE_SPECIES, l), ok = false;
    const double lam = ln.lam0[l];
    if (!(lam > 0.0) || !isfinite(lam) || !(ln.lamS0[l] >= 0.0) || !isfinite(ln.lamS0[l]))
        fail(status, CHK_LINE_LAM, l), ok = false;
    if (!(ln.gu[l] > 0.0) || !(ln.gl[l] > 0.0) || !isfinite(ln.gu[l]) || !isfinite(ln.gl[l]))
        fail(status, CHK_LINE_G, l), ok = false;
    if (!(ln.A[l] >= 0.0) || !isfinite(ln.A[l])) fail(status, CHK_LINE_A, l), ok = false;
    return ok;
}

// Conservative half-width of line l's window over the request's cells, nm:
// lamV <= lamL + lamG (the Voigt fit's factor never exceeds 1), both at their
// largest over the cells.  lamS0: the Stark width in use; c: the factors of
// the resonance and van der Waals terms (zero without them).
__device__ __forceinline__ double window_nm(double cD, double lamS0, double2 c, int s, bool broad,
                                            const unsigned long long* dmax) {
    const auto dm = [dmax](int i) { return __longlong_as_double((long long)dmax[i]); };
    double lamL = RAPRAL_LAM_NATURAL + lamS0 * dm(1);
    if (broad) lamL += c.x * dm(2 + 2 * s) + c.y * dm(3 + 2 * s);
    return RAPRAL_WINDOW * (lamL + cD * dm(0)) * (1.0 + 1e-9);
}

// One thread a line: the checks, the window's tiles and, for the lines whose
// window reaches the range, the records.  FP64 runs at 1/64 of the FP32 rate
// here, so what a line costs is its FP64 operations: three logarithms, a
// square root and four divisions for a record.  A chunk of a solve sees all
// lines of the list and keeps a few percent of them, so lines are turned away
// first by a bound of their window from FP32 widths (rounded up by 1e-4 and
// four grid points, against FP32 errors of 1e-6), which takes six FP64
// operations.  Checks, records and bounds of 320k lines took 342 us as three
// kernels (208 of them for one 64-bit atomicMax a line on one word, now one a
// block); 48 cells x 65,536 of 1e6 points, the whole call: 1.355 -> 1.060 ms.
__global__ void __launch_bounds__(256) k_line_plan(rapral_lines ln, const double* __restrict__ mass,
                                                   const int32_t* __restrict__ kind, int32_t S, double lam_min,
                                                   double h, Phys ph, int64_t k0, int64_t nk, int tile_w,
                                                   const unsigned long long* __restrict__ dmax,
                                                   LinePrep* __restrict__ out, LineF32* __restrict__ out32,
                                                   int2* __restrict__ line_tiles, unsigned long long* wmax,
                                                   int* unsorted, BroadArgs br, double2* lb, float2* lb32,
                                                   int* status) {
    __shared__ unsigned long long wblk;
    if (threadIdx.x == 0) wblk = 0ULL;
    __syncthreads();
    const int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    unsigned long long wbits = 0ULL;
    if (l < ln.n_lines && check_line(ln, S, l, status)) {
        const double lam0 = ln.lam0[l];
        if (l + 1 < ln.n_lines && ln.lam0[l + 1] < lam0) *unsorted = 1;
        const int s = ln.species[l];
        const bool atom = kind[s] == 0;
        const bool stark = (br.flags & RAPRAL_BROAD_STARK_IONIZE) && atom;
        bool near = true;
        if (!stark && !lb) {
            const float lamf = (float)lam0;
            const float wf =
                (float)RAPRAL_WINDOW *
                ((float)RAPRAL_LAM_NATURAL +
                 (float)ln.lamS0[l] * (float)__longlong_as_double((long long)dmax[1]) +
                 (float)RAPRAL_DOPPLER_HALF * lamf * rsqrtf((float)mass[s]) *
                     (float)__longlong_as_double((long long)dmax[0]));
            const double w = (double)(wf * 1.0001f) + 4.0 * h;   // NaN or inf: kept
            near = !(lam0 + w < lam_min + (double)k0 * h || lam0 - w > lam_min + (double)(k0 + nk - 1) * h);
        }
        int2 t = make_int2(1, 0);
        if (near) {
            LinePrep p;
            const double lcm = lam0 * 1e-7;
            const double A = ln.A[l];
            p.lam0 = lam0;
            p.cD = RAPRAL_DOPPLER_HALF * lam0 / sqrt(mass[s]);
            p.lamS0 = ln.lamS0[l];
            if (stark) {   // Stark coefficient from the ionisation gap
                const double dE = fmax(br.Eion[s] - ln.Eu_el[l], RAPRAL_E_IONIZE_H / 25.0);
                p.lamS0 = 1.69e3 * lam0 * lam0 / pow(dE, 2.623);
            }
            double2 c = make_double2(0.0, 0.0);
            if (lb) {   // per-line factors of the resonance and van der Waals widths
                if ((br.flags & RAPRAL_BROAD_RESONANCE) && atom && ln.El_el[l] == 0.0 && ln.El_v[l] == 0.0 &&
                    ln.El_j[l] == 0.0) {
                    const double f =
                        ph.me * ph.c * lcm * lcm / (8.0 * M_PI * M_PI * ph.e * ph.e) * ln.gu[l] / ln.gl[l] * A;
                    c.x = 4.3e-28 * lam0 * f * sqrt(ln.gl[l] / ln.gu[l]) * lam0 * lam0;
                }
                if ((br.flags & RAPRAL_BROAD_VDW) && atom) c.y = lam0 * lam0;
                lb[l] = c;
                lb32[l] = make_float2((float)c.x, (float)c.y);
            }
            p.tpos = (lam0 - lam_min) / h;
            const double w = window_nm(p.cD, p.lamS0, c, s, lb != nullptr, dmax) / h + 2.0;   // grid points
            const double lo = fmax(ceil(p.tpos - w), (double)k0);
            const double hi = fmin(floor(p.tpos + w), (double)(k0 + nk - 1));
            if (!(lo > hi)) {
                t.x = (int)(((int64_t)lo - k0) / tile_w);
                t.y = (int)(((int64_t)hi - k0) / tile_w);
                wbits = (unsigned long long)__double_as_longlong(w);
                p.lnAj = log(1e-7 * (ph.h * ph.c / (4.0 * M_PI)) * A / lcm);
                p.lnAk = log(1e4 * A * (lcm * lcm) * (lcm * lcm) / (8.0 * M_PI * ph.c));
                p.lngu = log(ln.gu[l]);
                p.lnAjg = p.lnAj + p.lngu;
                p.lnAkg = p.lnAk + p.lngu;
                p.Eve_u = ln.Eu_el[l] + ln.Eu_v[l];
                p.Er_u = ln.Eu_j[l];
                p.Eve_l = ln.El_el[l] + ln.El_v[l];
                p.Er_l = ln.El_j[l];
                p.dEve = p.Eve_u - p.Eve_l;
                p.dEr = p.Er_u - p.Er_l;
                p.dEve_f = (float)p.dEve;
                p.dEr_f = (float)p.dEr;
                p.cD_f = (float)p.cD;
                p.lamS0_f = (float)p.lamS0;
                const double kcd = rint(p.tpos);
                p.kc = (int32_t)fmin(fmax(kcd, -1e9), 2e9);
                p.delta_f = (float)(p.tpos - (double)p.kc);
                p.species = s;
                p.pad = 0;
                out[l] = p;
                if (out32) {
                    LineF32 f;
                    f.lnAjg = ff_from(p.lnAjg);
                    f.dAkj = ff_from(p.lnAk - p.lnAj);
                    f.Eve_u = ff_from(p.Eve_u);
                    f.Er_u = ff_from(p.Er_u);
                    f.dEve = ff_from(p.dEve);
                    f.dEr = ff_from(p.dEr);
                    f.cD = p.cD_f;
                    f.lamS0 = p.lamS0_f;
                    f.delta = p.delta_f;
                    f.kc = p.kc;
                    f.species = s;
                    f.kcf = (float)p.kc;
                    out32[l] = f;
                }
            }
        }
        line_tiles[l] = t;
    }
    // widest window of the lines that reach the range (positive doubles order
    // like their bits): one atomic a block
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long v = __shfl_xor_sync(0xffffffffu, wbits, o);
        wbits = v > wbits ? v : wbits;
    }
    if ((threadIdx.x & 31) == 0 && wbits) atomicMax(&wblk, wbits);
    __syncthreads();
    if (threadIdx.x == 0 && wblk) atomicMax(wmax, wblk);
}

// Entries of the sorted x[0, n) below v (UPPER: not above v), by one warp: 32
// probes a round (four rounds for 320k lines; a thread's bisection is a chain
// of 18 loads, twice, before a block could begin).
template <bool UPPER>
__device__ __forceinline__ int64_t warp_bound(const double* __restrict__ x, int64_t n, double v) {
    const int lane = threadIdx.x & 31;
    int64_t a = 0, b = n;
    while (a < b) {
        const int64_t step = (b - a + 31) / 32, p = a + lane * step;
        bool in = false;
        if (p < b) in = UPPER ? x[p] <= v : x[p] < v;
        const int c = __popc(__ballot_sync(0xffffffffu, in));   // the probes that are below come first
        if (c == 0) break;
        b = min(b, a + c * step);
        a += (c - 1) * step + 1;
    }
    return a;
}

// Lines whose centre can reach tile t: lam0 within the widest window of the
// tile's wavelength span (searched by two warps when lam0 is sorted, else
// all).  For the whole block; range: two shared words.
__device__ void tile_candidates(const double* lam0, int64_t L, int sorted, double wmax, double lam_min, double h,
                                int64_t kt0, int64_t kt1, int64_t* range, int64_t* b0, int64_t* b1) {
    if (!sorted) { *b0 = 0; *b1 = L; return; }
    const int warp = threadIdx.x >> 5;
    if (warp == 0) {
        const int64_t a = warp_bound<false>(lam0, L, lam_min + ((double)kt0 - wmax - 2.0) * h);
        if ((threadIdx.x & 31) == 0) range[0] = a;
    } else if (warp == 1) {
        const int64_t a = warp_bound<true>(lam0, L, lam_min + ((double)kt1 + wmax + 2.0) * h);
        if ((threadIdx.x & 31) == 0) range[1] = a;
    }
    __syncthreads();
    *b0 = range[0];
    *b1 = range[1];
}

__global__ void __launch_bounds__(256) k_bin_count(const double* __restrict__ lam0, int64_t L,
                                                   const int2* __restrict__ line_tiles, const int* unsorted,
                                                   const unsigned long long* wmaxp, double lam_min, double h,
                                                   int64_t k0, int64_t nk, int tile_w, int* __restrict__ counts,
                                                   const int* status) {
    if (*status) return;
    const int t = blockIdx.x;
    const int64_t kt0 = k0 + (int64_t)t * tile_w;
    const int64_t kt1 = min(kt0 + tile_w, k0 + nk) - 1;
    __shared__ int64_t range[2];
    int64_t b0, b1;
    tile_candidates(lam0, L, !*unsorted, __longlong_as_double((long long)*wmaxp), lam_min, h, kt0, kt1, range,
                    &b0, &b1);
    int cnt = 0;
    for (int64_t l = b0 + threadIdx.x; l < b1; l += blockDim.x) {
        const int2 r = line_tiles[l];
        cnt += (r.x <= t && t <= r.y);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
    __shared__ int ws[8];
    if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = cnt;
    __syncthreads();
    if (threadIdx.x == 0) {
        int s = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += ws[i];
        counts[t] = s;
    }
}

__global__ void __launch_bounds__(256) k_bin_fill(const double* __restrict__ lam0, int64_t L,
                                                  const int2* __restrict__ line_tiles, const int* unsorted,
                                                  const unsigned long long* wmaxp, double lam_min, double h,
                                                  int64_t k0, int64_t nk, int tile_w, const int* __restrict__ off,
                                                  int* __restrict__ out, unsigned long long* unit,
                                                  const int* status) {
    if (unit && blockIdx.x == 0 && threadIdx.x == 0) *unit = 0ULL;   // the line sum's work counter
    if (*status) return;
    const int t = blockIdx.x;
    const int64_t kt0 = k0 + (int64_t)t * tile_w;
    const int64_t kt1 = min(kt0 + tile_w, k0 + nk) - 1;
    __shared__ int64_t range[2];
    int64_t b0, b1;
    tile_candidates(lam0, L, !*unsorted, __longlong_as_double((long long)*wmaxp), lam_min, h, kt0, kt1, range,
                    &b0, &b1);
    __shared__ int wsum[8];
    __shared__ int base_s;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int base = off[t];
    for (int64_t r0 = b0; r0 < b1; r0 += blockDim.x) {
        const int64_t l = r0 + threadIdx.x;
        bool in = false;
        if (l < b1) { const int2 r = line_tiles[l]; in = (r.x <= t && t <= r.y); }
        const unsigned m = __ballot_sync(0xffffffffu, in);
        if (lane == 0) wsum[warp] = __popc(m);
        __syncthreads();
        if (threadIdx.x == 0) {
            int s = 0;
            for (int i = 0; i < nw; ++i) { int v = wsum[i]; wsum[i] = s; s += v; }
            base_s = s;
        }
        __syncthreads();
        if (in) out[base + wsum[warp] + __popc(m & ((1u << lane) - 1u))] = (int)l;
        base += base_s;
        __syncthreads();
    }
}

// Exclusive scan of the per-tile line counts into the int32 offsets of the
// tile lists, carried in int64 so that a total beyond 2^31 - 1 is seen:
// total[0] receives the exact sum, total[1] the status code (offsets past 2^31 - 1 wrap, and the
// callers refuse such a plan before the lists are filled).  Single block.
__global__ void __launch_bounds__(1024) k_scan_counts(int* data, int64_t n, long long* total, const int* status) {
    __shared__ long long part[32];
    __shared__ long long carry_s;
    if (threadIdx.x == 0) carry_s = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t c0 = 0; c0 < n; c0 += blockDim.x) {
        const int64_t i = c0 + threadIdx.x;
        const long long v = (i < n) ? (long long)data[i] : 0LL;
        long long x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) part[warp] = x;
        __syncthreads();
        if (warp == 0) {
            long long p = (lane < (int)(blockDim.x >> 5)) ? part[lane] : 0LL;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const long long y = __shfl_up_sync(0xffffffffu, p, o);
                if (lane >= o) p += y;
            }
            part[lane] = p;
        }
        __syncthreads();
        const long long carry = carry_s;
        const long long incl = x + (warp > 0 ? part[warp - 1] : 0LL);
        if (i < n) data[i] = (int)(unsigned)(unsigned long long)(carry + incl - v);
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry_s = carry + incl;
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        data[n] = (int)(unsigned)(unsigned long long)carry_s;
        total[0] = carry_s;
        total[1] = status[ST_CODE];   // read back with the total
    }
}

// Single-block exclusive scan over n entries; data[n] receives the total.
template <class T>
__global__ void __launch_bounds__(1024) k_scan(T* data, int64_t n) {
    __shared__ T part[32];
    __shared__ T carry_s;
    if (threadIdx.x == 0) carry_s = 0;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int64_t c0 = 0; c0 < n; c0 += blockDim.x) {
        const int64_t i = c0 + threadIdx.x;
        T v = (i < n) ? data[i] : T(0);
        T x = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            T y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) part[warp] = x;
        __syncthreads();
        if (warp == 0) {
            T p = (lane < (int)(blockDim.x >> 5)) ? part[lane] : T(0);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                T y = __shfl_up_sync(0xffffffffu, p, o);
                if (lane >= o) p += y;
            }
            part[lane] = p;
        }
        __syncthreads();
        const T carry = carry_s;
        const T incl = x + (warp > 0 ? part[warp - 1] : T(0));
        if (i < n) data[i] = carry + incl - v;
        __syncthreads();
        if (threadIdx.x == blockDim.x - 1) carry_s = carry + incl;
        __syncthreads();
    }
    if (threadIdx.x == 0) data[n] = carry_s;
}

// ------------------------------------------------------------ line sum FP64

// Block-wide sum of the per-thread work counters, one atomic per counter.
__device__ void block_count(unsigned long long* stats, int64_t ev, int64_t g, int64_t c, int64_t p) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ev += __shfl_xor_sync(0xffffffffu, ev, o);
        g += __shfl_xor_sync(0xffffffffu, g, o);
        c += __shfl_xor_sync(0xffffffffu, c, o);
        p += __shfl_xor_sync(0xffffffffu, p, o);
    }
    if ((threadIdx.x & 31) == 0 && p > 0) {   // one atomic set per warp
        atomicAdd(&stats[0], (unsigned long long)ev);
        atomicAdd(&stats[1], (unsigned long long)g);
        atomicAdd(&stats[2], (unsigned long long)c);
        atomicAdd(&stats[3], (unsigned long long)p);
    }
}

struct __align__(16) PairF64 {
    double lam0, w100, inv2V, r, omr, c16, aj, ak;
    double ug2, ue2;   // u^2 past which the Gaussian / correction exponential is left out
    int klo, khi, pad0, pad1;
};

// Exponentials of the Whiting bracket left out where they are below 1e-17 of
// its Lorentz part (at least r / (2 (1 + 4u^2)); the part is positive for
// every u), far below the FP64 rounding of the sum:
//   Gaussian (1 - r) e^{-2.772 x}, x = u^2: from the x with
//     2.772 x - ln(1 + 4x) = ln(2e17 (1 - r) / r), by fixed-point iteration
//     from below plus a margin, capped at the FP64 underflow (2.772 x = 745.5);
//   correction c16 e^{-0.4 x^1.125}: c16 / r <= 0.016 for every r, so one
//     bound serves all pairs, x = 65.14 (0.4 x^1.125 - ln(1 + 4x) = ln(3.2e15)).
constexpr double SKIP_CORR_U2 = 65.14;
__device__ double skip_gauss_u2(double omr, double r) {
    const double under = 745.5 / 2.772;
    if (!(omr > 0.0)) return 0.0;
    if (!(r > 0.0)) return under;
    const double K = log(2e17 * omr / r);
    double x = fmax(K, 0.0) / 2.772;
    for (int i = 0; i < 4; ++i) x = fmax(K + log1p(4.0 * x), 0.0) / 2.772;
    return fmin(1.05 * x + 0.5, under);
}

// Lorentz HWHM of line l in cell c in FP64: natural + Stark, plus the
// optional resonance and van der Waals terms.
__device__ __forceinline__ double lorentz64(const LineSumArgs& a, const LinePrep& L, const CellPrep& cp, int64_t l,
                                            int64_t c) {
    double lamL = RAPRAL_LAM_NATURAL + L.lamS0 * cp.stc;
    if (a.lb) {
        const double2 x = a.lb[l], y = a.cb[c * a.S + L.species];
        lamL += x.x * y.x;
        lamL += x.y * y.y;
    }
    return lamL;
}

// FP64 <-> FP32 of positive normal values in the FP32 range by their bits
// (truncating): the conversion instructions run on the FP64 pipe.
__device__ __forceinline__ float trunc_float(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    return __uint_as_float(((hi - (896u << 20)) << 3) | (lo >> 29));
}
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x);
    return __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29));
}
// u^(1/4) for u in [2^-60, 2^60]: w = u^(-1/4) to FP32 accuracy, e = 1 - u w^4
// (below 2^-19), u^(1/4) = u w^3 (1 - e)^(-3/4) with the series through e^2
// (e^3 < 2^-57): 7 FP64 operations, two square roots take 18 operation times.
__device__ __forceinline__ double root4(double u) {
    float r, wf;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(trunc_float(u)));
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(wf) : "f"(r));
    const double w = widen(wf), w2 = w * w, x = u * w2;
    const double e = fma(-x, w2, 1.0);
    const double y = x * w;
    return fma(y, e * fma(e, 0.65625, 0.75), y);
}
// n / d for d in [1, 2^100]: an FP32 reciprocal and one step of third order
// (4 operations; a division takes 9 operation times)
__device__ __forceinline__ double quotient(double n, double d) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(trunc_float(d)));
    const double y = widen(r), e = fma(-d, y, 1.0), q = n * y;
    return fma(q, fma(e, e, e), q);
}
// a <= b for non-negative a, b (their bits order like them; NaN a: false)
__device__ __forceinline__ bool le_bits(double a, double b) {
    return __double_as_longlong(a) <= __double_as_longlong(b);
}

// One block: one tile of 128 PPT points and one cell.  The FP64 pipe bounds it
// (1/64 of the FP32 rate), so an evaluation costs its FP64 warp instructions,
// whatever lanes are in the window: thread i owns points i, i + 128, ..., so
// that a warp's points are runs of 32 in a row and a run outside the window
// is skipped by the whole warp (with 128 points in a row a warp, a window of
// 70 points kept 37 % of the lanes busy), and an evaluation is 22 FP64
// operations: wavelengths formed once a tile, comparisons on the integer
// pipe, u^2.25 and the quotient by Newton steps from FP32 seeds, exponentials
// in fixed point.  24 cells x 50,001 points, 64,000 lines: 20.3 -> 4.9 ms.
template <int PPT, bool VG = false>
__global__ void __launch_bounds__(128) k_line_sum_f64(LineSumArgs a) {
    if (*a.status) return;
    const int W = 128 * PPT;
    const int t = blockIdx.y;
    const int64_t c = blockIdx.x;
    const int64_t kt0 = a.k0 + (int64_t)t * W;
    const int64_t kend = min(kt0 + W, a.k0 + a.nk);   // exclusive
    const int kp = (int)threadIdx.x;            // the thread's points kt0 + kp + 128 i
    const int wp = (int)(threadIdx.x & ~31u);   // the warp's runs kt0 + wp + 128 i .. + 31
    __shared__ PairF64 pr[128];
    __shared__ uint64_t tab[EXPFIX_N];
    expfix_load(tab);
    __syncthreads();
    int64_t n_ev = 0, n_g = 0, n_c = 0, n_pairs = 0;
    double acck[PPT], accj[PPT], lk[PPT];
#pragma unroll
    for (int i = 0; i < PPT; ++i) {
        acck[i] = 0.0;
        accj[i] = 0.0;
        lk[i] = __dadd_rn(a.lam_min, __dmul_rn((double)(kt0 + kp + 128 * i), a.h));
    }
    const CellPrep cp = a.cp[c];
    const double inv_h = 1.0 / a.h;
    const int beg = a.tile_off[t], end = a.tile_off[t + 1];
    for (int b = beg; b < end; b += 128) {
        const int nb = min(128, end - b);
        if ((int)threadIdx.x < nb) {
            const int l = a.tile_lines[b + threadIdx.x];
            const LinePrep L = a.lp[l];
            PairF64 P;
            P.klo = 1; P.khi = 0;
            double du = 0.0, dl = 0.0;   // departure coefficients (ln b) of the line's levels
            if (a.dep_lnb) {
                const double* row = a.dep_lnb + (c * a.S + L.species) * a.dep_nlev;
                const int iu = a.dep_u[l], il = a.dep_l[l];
                if (iu >= 0) du = row[iu];
                if (il >= 0) dl = row[il];
            }
            const double lnNu = a.lnpref[c * a.S + L.species] + L.lngu - (L.Eve_u * cp.bve + L.Er_u * cp.btr) + du;
            const double Sj = exp_fix(L.lnAj + lnNu, tab);
            if (Sj > 0.0) {
                const double x = L.dEve * cp.bve + L.dEr * cp.btr + (dl - du);
                const double Sk = exp_fix(L.lnAk + lnNu, tab) * expm1(x);
                const double lamG = L.cD * cp.sqrtT;
                const double lamL = lorentz64(a, L, cp, l, c);
                const double lamV = voigt_hwhm(lamL, lamG);
                double r = lamL / lamV;
                double pre = 1e3 / (2.0 * lamV * (1.065 + 0.447 * r + 0.058 * r * r));
                P.lam0 = L.lam0;
                P.w100 = RAPRAL_WINDOW * lamV;
                P.inv2V = 0.5 / lamV;
                if (VG) {   // exact Voigt: x = dlam / (sigma sqrt 2) = dlam sqrt(ln 2) / lamG, y = lamL sqrt(ln 2) / lamG
                    P.inv2V = 0.83255461115769775635 / lamG;
                    r = lamL * P.inv2V;
                    pre = 1e3 * 0.46971863934982566689 / lamG;   // 1e3 / (sigma sqrt(2 pi))
                }
                P.r = r;
                P.omr = 1.0 - r;
                P.c16 = 0.016 * r * (1.0 - r);
                if (!VG) {
                    P.ug2 = skip_gauss_u2(P.omr, r);
                    P.ue2 = P.c16 > 0.0 ? SKIP_CORR_U2 : 0.0;
                }
                P.aj = Sj * pre;
                P.ak = Sk * pre;
                const double lo = ceil((L.lam0 - P.w100 - a.lam_min) * inv_h) - 1.0;
                const double hi = floor((L.lam0 + P.w100 - a.lam_min) * inv_h) + 1.0;
                P.klo = (int)(fmax(lo, (double)kt0) - (double)kt0);   // offsets from kt0
                P.khi = (int)(fmin(hi, (double)(kend - 1)) - (double)kt0);
                if (P.klo <= P.khi) {
                    // counters: candidate points (the exact window is tested per point), and
                    // those where the two exponentials are above the FP64 underflow limit
                    const double kcen = L.tpos;
                    const double hg = 16.4 * 2.0 * lamV * inv_h, hc = 28.4 * 2.0 * lamV * inv_h;   // 2.772u^2, 0.4u^2.25 < 745.5
                    n_ev += min((int64_t)P.khi + kt0, (int64_t)floor(kcen + RAPRAL_WINDOW * lamV * inv_h)) -
                            max((int64_t)P.klo + kt0, (int64_t)ceil(kcen - RAPRAL_WINDOW * lamV * inv_h)) + 1;
                    n_g += max((int64_t)0, min((int64_t)P.khi + kt0, (int64_t)floor(kcen + hg)) -
                                               max((int64_t)P.klo + kt0, (int64_t)ceil(kcen - hg)) + 1);
                    n_c += max((int64_t)0, min((int64_t)P.khi + kt0, (int64_t)floor(kcen + hc)) -
                                               max((int64_t)P.klo + kt0, (int64_t)ceil(kcen - hc)) + 1);
                    ++n_pairs;
                }
            }
            pr[threadIdx.x] = P;
        }
        __syncthreads();
        for (int q = 0; q < nb; ++q) {
            const int klo = pr[q].klo, khi = pr[q].khi;
            if (khi < wp || klo > wp + 128 * (PPT - 1) + 31) continue;
            const PairF64 P = pr[q];
#pragma unroll
            for (int i = 0; i < PPT; ++i) {
                if (khi < wp + 128 * i || klo > wp + 128 * i + 31) continue;   // the same for the warp
                const int k = kp + 128 * i;
                const double dl = fabs(lk[i] - P.lam0);
                if (k < klo || k > khi || !le_bits(dl, P.w100)) continue;
                if (VG) {
                    const double br = voigt_re<double>(c_voigt, dl * P.inv2V, P.r);
                    accj[i] += P.aj * br;
                    acck[i] += P.ak * br;
                    continue;
                }
                const double u = dl * P.inv2V;
                const double u2 = u * u;
                // u^2.25: zero to FP64 beside 1 where u < 2^-60
                const double v = __double2hiint(u) >= 0x3C300000 ? u2 * root4(u) : 0.0;
                const double qd = fma(4.0, u2, 1.0);
                const double pd = fma(0.1, v, 1.0);
                double br = quotient(fma(P.r, pd, -P.c16 * qd), qd * pd);
                if (__double_as_longlong(u2) < __double_as_longlong(P.ue2)) br = fma(P.c16, exp_fix(-0.4 * v, tab), br);
                if (__double_as_longlong(u2) < __double_as_longlong(P.ug2))
                    br = fma(P.omr, exp_fix(-2.772 * u2, tab), br);
                accj[i] = fma(P.aj, br, accj[i]);
                acck[i] = fma(P.ak, br, acck[i]);
            }
        }
        __syncthreads();
    }
    block_count(a.stats, n_ev, n_g, n_c, n_pairs);
    double* K = reinterpret_cast<double*>(a.kappa) + c * a.ld - a.k0;
    double* J = reinterpret_cast<double*>(a.emis) + c * a.ld - a.k0;
#pragma unroll
    for (int i = 0; i < PPT; ++i) {
        const int64_t k = kt0 + kp + 128 * i;
        if (k < kend) { __stcs(K + k, acck[i]); __stcs(J + k, accj[i]); }   // streaming, as the FP32 path
    }
}


// ------------------------------------------------------ line sum FP32 (chosen)
//
// Set-up per (line, cell): log-space populations and strengths in FP64,
// exponentials of the reduced log (integer power of two times 2^f, f in
// [0, 1)) in FP32; widths, Voigt HWHM and profile constants in FP32.  The
// window [klo, khi] is found in grid units in FP32 and certified: when an edge
// lies within the FP32 error bound of a grid point, both edges are decided
// again with the FP64 Voigt width and the literal test |lam_k - lam0| <=
// 100 lamV, so every (line, point) inclusion matches the FP64 decision.
// Per point: u = |(k - kc) s - u0| (s = h / 2lamV), the Whiting bracket with
// MUFU ex2 / rsqrt / rcp, exponentials below FP32 rounding left out, and Kahan
// compensated sums of kappa and j over the tile's lines.

__device__ __forceinline__ float ex2_approx(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ bool in_window64(int64_t k, double lam_min, double h, double lam0, double w100) {
    const double lk = __dadd_rn(lam_min, __dmul_rn((double)k, h));
    return fabs(lk - lam0) <= w100;
}

// Exact edges near the FP32 estimates (the estimate is within a fraction of a
// grid point of the truth).
__device__ __noinline__ void exact_edges(const LinePrep* __restrict__ Lp, const CellPrep* __restrict__ cpp,
                                         const double2* lb, const double2* cbrow, double lam_min, double h,
                                         int64_t* klo, int64_t* khi) {
    const LinePrep& L = *Lp;
    const CellPrep& cp = *cpp;
    const double lamG = L.cD * cp.sqrtT;
    double lamL = RAPRAL_LAM_NATURAL + L.lamS0 * cp.stc;
    if (lb) {   // the optional resonance / van der Waals terms, as lorentz64
        const double2 x = *lb, y = cbrow[L.species];
        lamL += x.x * y.x;
        lamL += x.y * y.y;
    }
    const double w100 = RAPRAL_WINDOW * voigt_hwhm(lamL, lamG);
    int64_t k = *khi + 2;
    while (k > *khi - 3 && !in_window64(k, lam_min, h, L.lam0, w100)) --k;
    const int64_t hi = k;
    k = *klo - 2;
    while (k < *klo + 3 && !in_window64(k, lam_min, h, L.lam0, w100)) ++k;
    *klo = k;
    *khi = hi;
}

// Conversion-free helpers for the FP32 set-up.  On GB300 float/integer
// conversions and roundings share the narrow FP64 pipe, so the set-up keeps
// to FMA-pipe arithmetic and MUFU ex2 / rcp.

// Nearest integer of |x| < 2^22 (adding and removing 1.5 * 2^23).
__device__ __forceinline__ float round_near(float x) { return (x + 12582912.0f) - 12582912.0f; }
__device__ __forceinline__ float floor_f(float x) { const float n = round_near(x); return n > x ? n - 1.0f : n; }
__device__ __forceinline__ float ceil_f(float x) { const float n = round_near(x); return n < x ? n + 1.0f : n; }

// e^y for y = hi + lo: t = y log2(e) (float-float), t = n + f with n the
// nearest integer, 2^f and 2^n by MUFU ex2.
__device__ __forceinline__ float exp_ff(float2 y) {
    const float2 t = ff_mul(y, make_float2(1.4426950216293335f, 1.925963033500011e-08f));
    const float n = round_near(t.x);
    return ex2_approx((t.x - n) + t.y) * ex2_approx(n);
}

// e^z - 1 for z <= 0: Taylor series through z^9 for z > -1/2 (error below
// 3e-10 relative), else 2^(z log2 e) - 1 (|result| >= 0.39).
__device__ __forceinline__ float expm1_neg(float z) {
    if (z > -0.5f) {
        float p = 1.0f / 362880.0f;
        p = fmaf(p, z, 1.0f / 40320.0f);
        p = fmaf(p, z, 1.0f / 5040.0f);
        p = fmaf(p, z, 1.0f / 720.0f);
        p = fmaf(p, z, 1.0f / 120.0f);
        p = fmaf(p, z, 1.0f / 24.0f);
        p = fmaf(p, z, 1.0f / 6.0f);
        p = fmaf(p, z, 0.5f);
        p = fmaf(p, z, 1.0f);
        return p * z;
    }
    return ex2_approx(z * 1.44269504f) - 1.0f;
}

// sin(pi d) for |d| <= 1: sin(pi a) = sin(pi (1 - a)) maps |d| to [0, 1/2],
// then the Taylor series of sin(pi x) through x^13 (error below 1e-9).
__device__ __forceinline__ float sinpi_series(float d) {
    const float a = fabsf(d);
    const float x = a > 0.5f ? 1.0f - a : a;
    const float z = x * x;
    float p = 4.663027939386666e-4f;
    p = fmaf(p, z, -7.37043097615242e-3f);
    p = fmaf(p, z, 8.214588463306427e-2f);
    p = fmaf(p, z, -0.5992645025253296f);
    p = fmaf(p, z, 2.550163984298706f);
    p = fmaf(p, z, -5.167712688446045f);
    p = fmaf(p, z, 3.1415927410125732f);
    return copysignf(x * p, d);
}

// One (line, cell) pair set up for a warp's tile [kt0, kt0 + TW): window
// offsets inside the tile (as floats), u at the tile's first point, profile
// constants, and the part of the line where an exponential of the bracket is
// above the FP32 rounding of the rest.  Everything a warp needs per pair is
// computed here, by one lane per pair.
// Exponentials of the bracket: beyond |u| = 6 the correction 0.016 r (1 - r)
// e^{-0.4 u^2.25} is below 4e-10 of the Lorentz part r / (1 + 4u^2) for every
// r, and the Gaussian e^{-2.772 u^2} below 5e-44, under 1e-30 of it for the r
// that a natural width of 5.9e-6 nm leaves: both are left out there.
constexpr float NEAR_U = 6.0f;
// Constants of the profile whose rounding would lean one way for every line:
// the Gaussian's exponent -2.772 log2(e) u^2 to the nearest float; the
// approximate ex2 lies 5.1e-8 low on average over [-20, 0], which a shift of
// its argument takes back; 1.065 of the normalisation rounds up by 5.4e-8,
// which its factor 500 takes back (the next float, 6.1e-8 up).
constexpr float GAUSS_SCALE = -3.9991507f, GAUSS_SHIFT = 7.4e-8f, NORM_FACTOR = 500.00003f;

struct PairF32 {
    float lo, hi;     // window part inside the tile, offsets from kt0
    float x0, wn;     // line centre as an offset from kt0; points around it with |u| <= NEAR_U
    float ub, ub_lo;  // signed u at kt0, (kt0 - kc) s - u0, as a float-float pair
    float s;          // h / (2 lamV): step of u per grid point
    float r, aj, ak;
};

// What a warp's set-up reads of its cell, in shared memory: held in registers
// it was spilled through the sweep.  (The default form still spills 112 bytes a
// thread, 128 loaded, at the 64 registers of 32 warps an SM; at 80 registers
// and 24 warps it spills 4, and the line sums take 3 % longer.)
struct WarpCell {
    float2 bve_ff, btr_ff;
    float sqrtT_f, stc_f, pad[2];
    float2 lp[RAPRAL_MAX_SPECIES];   // ln(N_s / Z_s) as float-float pairs
    float2 cb[RAPRAL_MAX_SPECIES];   // (N_0, W) of the optional terms
};

// FL: bit 0 the optional Lorentz terms, bit 1 the departure coefficients.
template <int FL>
__device__ __forceinline__ bool setup_pair_f32(const LineSumArgs& a, const LineF32& L, const WarpCell& cp, float2 lp,
                                               float2 cb, int line, int64_t c, float hf, float inv_hf, int kt0,
                                               float kt0f, float kt1f, bool count, PairF32* P, int64_t* cnt) {
    constexpr bool BR = (FL & 1) != 0, DEP = (FL & 2) != 0, VG = (FL & 4) != 0;
    if (!(lp.x > -INFINITY)) return false;
    // widths first: most candidates of a tile list miss the tile in a given cell
    const float lamG = L.cD * cp.sqrtT_f;
    float lamL = (float)RAPRAL_LAM_NATURAL + L.lamS0 * cp.stc_f;
    if (BR) {   // resonance / van der Waals terms: c_R N_0 + c_W W
        const float2 x = a.lb32[line];
        lamL = fmaf(x.y, cb.y, fmaf(x.x, cb.x, lamL));
    }
    const float sum = lamL + lamG;
    {   // lamV <= lamL + lamG: cheap rejection before the Voigt fit
        const float wmax = (float)RAPRAL_WINDOW * sum * inv_hf * 1.0001f + 1.0f;
        if (kt1f - L.kcf < L.delta - wmax || kt0f - L.kcf > L.delta + wmax) return false;
    }
    const float d = (lamL - lamG) * rcp_approx(sum);
    const float F = 1.0f - 0.18121f * (1.0f - d * d) -
                    (0.023665f * ex2_approx(0.6f * 1.44269504f * d) + 0.00418f * ex2_approx(-1.9f * 1.44269504f * d)) *
                        sinpi_series(d);
    const float lamV = F * sum;
    const float wpts = (float)RAPRAL_WINDOW * lamV * inv_hf;
    const float hi = L.delta + wpts, lo = L.delta - wpts;
    const float fhi = floor_f(hi), clo = ceil_f(lo);
    // window in offsets from kt0 (exact: integers below 2^24)
    float lo_rel = L.kcf + clo - kt0f, hi_rel = L.kcf + fhi - kt0f;
    // Certification.  The FP32 edge positions are within 1.2e-6 wpts + 6e-8
    // grid units of the exact ones (lamV to 9e-7 relative through widths,
    // the Voigt fit, ex2 and the sin series; wpts and the sums to a few more
    // roundings).  Only an edge that lies inside this tile and within m of a
    // grid point is decided again in FP64.
    // (with the optional terms lamL carries two more roundings: a wider margin)
    const float m = (BR ? 2e-6f : 1.5e-6f) * wpts + 1e-6f;
    const float span = kt1f - kt0f;
    const bool lo_in = lo_rel >= -1.0f && lo_rel <= span + 1.0f;
    const bool hi_in = hi_rel >= -1.0f && hi_rel <= span + 1.0f;
    if ((hi_in && (hi - fhi < m || fhi + 1.0f - hi < m)) || (lo_in && (clo - lo < m || lo - (clo - 1.0f) < m))) {
        int64_t klo = (int64_t)L.kc + (int64_t)clo, khi = (int64_t)L.kc + (int64_t)fhi;
        exact_edges(a.lp + line, a.cp + c, BR ? a.lb + line : nullptr, BR ? a.cb + c * a.S : nullptr, a.lam_min, a.h,
                    &klo, &khi);
        lo_rel = (float)(klo - kt0);
        hi_rel = (float)(khi - kt0);
    }
    lo_rel = fmaxf(lo_rel, 0.0f);
    hi_rel = fminf(hi_rel, kt1f - kt0f);
    if (lo_rel > hi_rel) return false;
    // strengths: ln S_j = lnAj + ln g_u + ln(N_s/Z_s) - (E_el + E_V)_u c2/T_ve - E_J,u c2/T_tr
    // and x = ln(N_l g_u / (N_u g_l)) = dE_ve c2/T_ve + dE_J c2/T_tr, in float-float
    float2 yj = ff_add(ff_add(L.lnAjg, lp), ff_neg(ff_add(ff_mul(L.Eve_u, cp.bve_ff), ff_mul(L.Er_u, cp.btr_ff))));
    float2 x = ff_add(ff_mul(L.dEve, cp.bve_ff), ff_mul(L.dEr, cp.btr_ff));
    if (DEP) {   // departure coefficients: ln N_u += ln b_u, x += ln b_l - ln b_u
        const int iu = a.dep_u[line], il = a.dep_l[line];
        if (iu >= 0 || il >= 0) {
            const double* row = a.dep_lnb + ((int64_t)c * a.S + L.species) * a.dep_nlev;
            const double du = iu >= 0 ? row[iu] : 0.0, dl = il >= 0 ? row[il] : 0.0;
            yj = ff_add(yj, ff_from(du));
            x = ff_add(x, ff_from(dl - du));
        }
    }
    const float Sj = exp_ff(yj);
    float2 yk = ff_add(yj, L.dAkj);
    float fk;
    if (x.x >= 0.0f) {           // kappa0 = e^{lnAk + ln N_l g_u/g_l} (1 - e^{-x})
        yk = ff_add(yk, x);
        fk = -expm1_neg(-x.x);
    } else {                     // kappa0 = e^{lnAk + ln N_u} (e^{x} - 1)
        fk = expm1_neg(x.x);
    }
    const float Sk = exp_ff(yk) * fk;
    if (!(Sj > 0.0f) && Sk == 0.0f) return false;
    const float iv = rcp_approx(lamV);
    float r = lamL * iv;
    float pre = NORM_FACTOR * iv * rcp_approx(1.065f + 0.447f * r + 0.058f * r * r);   // 1e3 / (2 lamV ..)
    float s = 0.5f * fmaf(hf, iv, a.h_lo * iv);
    if (VG) {   // exact Voigt: u is x = dlam sqrt(ln 2) / lamG, r is y, pre 1e3 / (sigma sqrt(2 pi))
        const float ig = rcp_approx(lamG);
        r = 0.83255461f * lamL * ig;
        pre = 1e3f * 0.46971864f * ig;
        s = 0.83255461f * fmaf(hf, ig, a.h_lo * ig);
    }
    const float u0 = L.delta * s;                    // u of the centre's offset from kc
    {   // signed u at kt0 without rounding loss: (kt0 - kc) is exact, its
        // product with s and the sum with -u0 are split into hi + lo
        const float dk = kt0f - L.kcf;
        const float p = dk * s;
        const float pe = fmaf(dk, s, -p);
        const float uh = p - u0;
        const float bb = uh - p;
        const float e = (p - (uh - bb)) + (-u0 - bb);
        P->ub = uh;
        P->ub_lo = e + pe;
    }
    P->lo = lo_rel;
    P->hi = hi_rel;
    P->x0 = L.kcf - kt0f + L.delta;
    P->wn = 2.0f * NEAR_U * lamV * inv_hf;
    P->s = s;
    P->r = r;
    P->aj = Sj * pre;
    P->ak = Sk * pre;
    if (count) {
        // work counters: points in the window; those where the Gaussian core and
        // the exponential correction are above the FP32 underflow limits
        const int64_t klo = kt0 + (int64_t)lo_rel, khi = kt0 + (int64_t)hi_rel;
        cnt[0] += khi - klo + 1;
        const float kcen = L.kcf + L.delta;
        const float hg = 5.6125f / s, hc = 10.95f / s;   // u^2 < 31.5, u^2.25 < 218
        cnt[1] += max((int64_t)0, min(khi, (int64_t)floorf(kcen + hg)) - max(klo, (int64_t)ceilf(kcen - hg)) + 1);
        cnt[2] += max((int64_t)0, min(khi, (int64_t)floorf(kcen + hc)) - max(klo, (int64_t)ceilf(kcen - hc)) + 1);
        cnt[3] += 1;
    }
    return true;
}

// Kahan step: (s, c) += x.
__device__ __forceinline__ void kahan_add(float& s, float& c, float x) {
    const float y = x - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
}

// A batch's staged lines.  Lines whose window covers the whole tile: W0 = s,
// ub, ub_lo, r and W1 = aj, ak, those with no near part from the front, the
// others from the end.  The others (partial lines) two a slot in packed-pair
// order: G[0] = -mid, half (of the window part in the tile), G[1] = ub, ub_lo,
// G[2] = s, r, G[3] = aj, ak, each for both lines, and per line the runs it
// reaches (low half) and the runs that hold points of its near part (high).
template <int PB>
struct LineSlots {
    float4 G[4][PB / 2];
    float4 W0[PB];
    float2 W1[PB];
    unsigned runs[PB];
};

// Whiting's bracket of a slot's two lines at the lane's point of one run (the
// factor 1e3 / (2 lamV (1.065 + 0.447 r + 0.058 r^2)) is folded into aj, ak),
// added to the run's sums, a sum a line.  With q4 = 1 + 4u^2, p1 = 1 + 0.1
// u^2.25, c = 0.016 (1 - r): r ((p1 - c q4) / (q4 p1)), and in a near run
// + r c e^{-0.4 u^2.25} + (1 - r) e^{-2.772 u^2}.
//
// The MUFU pipe (16 rsqrt or rcp a clock and SM) takes 24 clocks a warp for a
// far evaluation with its own reciprocal; the two lines share the one of
// their denominators' product (20 clocks, beside 17 of the FP32 pipe).
// |u| is capped so that the product of a point in its window and one far out
// of it stays in range.
template <bool NEAR>
__device__ __forceinline__ void slot_eval(float k, float2 nmid, float2 half, float2 ub, float2 ubl, float2 s, float2 nc,
                                          float2 r, float2 aj, float2 ak, float& bj, float& bk) {
    const auto c2 = [](float x) { return make_float2(x, x); };
    // signed u at point k: one rounding of k s + ub (exact product), then the
    // low part; relative to u itself, so the Gaussian core keeps FP32 accuracy
    // however far the tile start lies from the line centre
    const float2 u = __fadd2_rn(__ffma2_rn(c2(k), s, ub), ubl);
    const float2 d = __fadd2_rn(c2(k), nmid);
    const float2 w = make_float2(fminf(fabsf(u.x), 1e4f), fminf(fabsf(u.y), 1e4f));
    const float2 u2 = __fmul2_rn(w, w);
    const float2 q = make_float2(rsqrt_approx(rsqrt_approx(w.x)), rsqrt_approx(rsqrt_approx(w.y)));
    const float2 v = __fmul2_rn(u2, q);                    // u^2.25
    const float2 q4 = __ffma2_rn(c2(4.0f), u2, c2(1.0f));
    const float2 p1 = __ffma2_rn(c2(0.1f), v, c2(1.0f));
    const float2 qp = __fmul2_rn(q4, p1);
    const float rp = rcp_approx(qp.x * qp.y);
    const float2 rd = make_float2(qp.y * rp, qp.x * rp);
    float2 h = __fmul2_rn(__ffma2_rn(nc, q4, p1), rd);
    if (NEAR) {
        const float2 xc = __fmul2_rn(c2(-0.5770780f), v);  // -0.4 log2(e) v
        const float2 xg = __ffma2_rn(c2(GAUSS_SCALE), u2, c2(GAUSS_SHIFT));
        const float2 e2 = make_float2(ex2_approx(xc.x), ex2_approx(xc.y));
        const float2 g = make_float2(ex2_approx(xg.x), ex2_approx(xg.y));
        const float2 omr = __ffma2_rn(c2(-1.0f), r, c2(1.0f));
        h = __ffma2_rn(__fmul2_rn(c2(0.016f), omr), e2, h);
        h = __ffma2_rn(omr, g, __fmul2_rn(r, h));
    }
    // predicated: outside its window a line adds nothing, whatever its strength
    // (a strength past the FP32 range times a zeroed profile would be NaN)
    if (fabsf(d.x) <= half.x) {
        bj = fmaf(aj.x, h.x, bj);
        bk = fmaf(ak.x, h.x, bk);
    }
    if (fabsf(d.y) <= half.y) {
        bj = fmaf(aj.y, h.y, bj);
        bk = fmaf(ak.y, h.y, bk);
    }
}

// The n staged lines over the lane's points lane + 32 i of the tile.  Lines
// of a slot are neighbours in the sorted list, so they reach nearly the same
// runs; a run is taken if either reaches it, and as near if either is.
template <int PPT, int PB>
__device__ __forceinline__ void sweep_slots(const LineSlots<PB>& sl, int n, float lanef, float (&bj)[PPT],
                                            float (&bk)[PPT]) {
    for (int j = 0; 2 * j < n; ++j) {
        const uint2 m = *reinterpret_cast<const uint2*>(&sl.runs[2 * j]);
        const unsigned runs = m.x | m.y;
        const float4 g0 = sl.G[0][j], g1 = sl.G[1][j], g2 = sl.G[2][j], g3 = sl.G[3][j];
        const float2 nmid = make_float2(g0.x, g0.y), half = make_float2(g0.z, g0.w);
        const float2 ub = make_float2(g1.x, g1.y), ubl = make_float2(g1.z, g1.w);
        const float2 s = make_float2(g2.x, g2.y), r = make_float2(g2.z, g2.w);
        const float2 aj = make_float2(g3.x, g3.y), ak = make_float2(g3.z, g3.w);
        const float2 nc = __ffma2_rn(make_float2(0.016f, 0.016f), r, make_float2(-0.016f, -0.016f));
        const float2 ajr = __fmul2_rn(aj, r), akr = __fmul2_rn(ak, r);
#pragma unroll
        for (int i = 0; i < PPT; ++i) {
            if (!(runs & (1u << i))) continue;   // the same for the whole warp
            if (runs & (0x10000u << i))
                slot_eval<true>(lanef + 32.0f * i, nmid, half, ub, ubl, s, nc, r, aj, ak, bj[i], bk[i]);
            else
                slot_eval<false>(lanef + 32.0f * i, nmid, half, ub, ubl, s, nc, r, ajr, akr, bj[i], bk[i]);
        }
    }
}

// One line whose window covers every point of the tile: no point needs the
// window test, and the runs are taken four at a time in packed pairs with one
// reciprocal for the four (|u| <= 50 in a window, so the denominators' product
// stays below 2e27), which overlaps their latencies and takes 18 clocks of the
// MUFU pipe an evaluation instead of 24.
template <int PPT, bool NEAR>
__device__ __forceinline__ void sweep_whole(float lanef, float s, float ub, float ub_lo, float r, float aj, float ak,
                                            float (&bj)[PPT], float (&bk)[PPT]) {
    static_assert(PPT % 4 == 0, "runs are taken four at a time");
    const auto c2 = [](float x) { return make_float2(x, x); };
    const float omr = 1.0f - r, c = 0.016f * omr;
    const float2 aj2 = c2(NEAR ? aj : aj * r), ak2 = c2(NEAR ? ak : ak * r);
#pragma unroll
    for (int i0 = 0; i0 < PPT; i0 += 4) {
        float2 u2[2], v[2], qp[2], num[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = i0 + 2 * h;
            const float2 k = make_float2(lanef + 32.0f * i, lanef + 32.0f * (i + 1));
            const float2 u = __fadd2_rn(__ffma2_rn(k, c2(s), c2(ub)), c2(ub_lo));     // signed u; only |u| and u^2 are used
            u2[h] = __fmul2_rn(u, u);
            const float2 q = make_float2(rsqrt_approx(rsqrt_approx(fabsf(u.x))), rsqrt_approx(rsqrt_approx(fabsf(u.y))));
            v[h] = __fmul2_rn(u2[h], q);                            // u^2.25
            const float2 q4 = __ffma2_rn(c2(4.0f), u2[h], c2(1.0f));
            const float2 p1 = __ffma2_rn(c2(0.1f), v[h], c2(1.0f));
            qp[h] = __fmul2_rn(q4, p1);
            num[h] = __ffma2_rn(c2(-c), q4, p1);
        }
        const float d0 = qp[0].x * qp[0].y, d1 = qp[1].x * qp[1].y;
        const float R = rcp_approx(d0 * d1);
        const float rr[2] = {R * d1, R * d0};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = i0 + 2 * h;
            float2 br = __fmul2_rn(num[h], make_float2(qp[h].y * rr[h], qp[h].x * rr[h]));
            if (NEAR) {
                const float2 xc = __fmul2_rn(c2(-0.5770780f), v[h]);
                const float2 xg = __ffma2_rn(c2(GAUSS_SCALE), u2[h], c2(GAUSS_SHIFT));
                const float2 e2 = make_float2(ex2_approx(xc.x), ex2_approx(xc.y));    // e^{-0.4 v}
                const float2 g = make_float2(ex2_approx(xg.x), ex2_approx(xg.y));     // e^{-2.772 u^2}
                br = __ffma2_rn(c2(c), e2, br);
                br = __ffma2_rn(c2(omr), g, __fmul2_rn(c2(r), br));
            }
            const float2 j2 = __ffma2_rn(aj2, br, make_float2(bj[i], bj[i + 1]));
            const float2 k2 = __ffma2_rn(ak2, br, make_float2(bk[i], bk[i + 1]));
            bj[i] = j2.x; bj[i + 1] = j2.y;
            bk[i] = k2.x; bk[i + 1] = k2.y;
        }
    }
}
template <int PPT, int PB, bool NEAR>
__device__ __forceinline__ void sweep_wholes(const LineSlots<PB>& sl, int q0, int q1, float lanef, float (&bj)[PPT],
                                             float (&bk)[PPT]) {
    for (int q = q0; q < q1; ++q) {
        const float4 A = sl.W0[q];
        const float2 B = sl.W1[q];
        sweep_whole<PPT, NEAR>(lanef, A.x, A.y, A.z, A.w, B.x, B.y, bj, bk);
    }
}

// The same sweep with the exact Voigt shape: r is y, u is x.
template <int PPT>
__device__ __forceinline__ void sweep_pair_voigt(const VoigtCoef& vc, float lo, float hi, float o0, float kf, float s, float ub,
                                                 float ub_lo, float y, float aj, float ak, float (&bj)[PPT],
                                                 float (&bk)[PPT]) {
#pragma unroll
    for (int i = 0; i < PPT; ++i) {
        const float p0 = o0 + 32.0f * i;
        if (p0 + 31.0f < lo || p0 > hi) continue;
        const float k = kf + 32.0f * i;
        const float br = voigt_re<float>(vc, fmaf(k, s, ub) + ub_lo, y);
        if (k >= lo && k <= hi) {
            bj[i] = fmaf(aj, br, bj[i]);
            bk[i] = fmaf(ak, br, bk[i]);
        }
    }
}

// Warp-level line sum: a warp owns one cell and the TW = 32 PPT points of
// tile t, lane l the points l, l + 32, ..., l + 32 (PPT - 1); it stages 32
// (line, cell) pairs at a time in its own shared-memory slice (one per lane),
// then sweeps them over its points.  With the points interleaved, whether a
// pair's window reaches the i-th run of 32 points is the same for the whole
// warp, so runs outside the window are skipped without a masked evaluation.
// Lines whose window covers the whole tile are swept one at a time over four
// runs, the others two at a time run by run.  Warps never wait for each other.
// Tiles of 256 and 512 points are swept in parts of 128, so that a line's
// set-up, a quarter of the time at 128, serves several parts: 256 points take
// 29.3 ms for 31.1 on 200 cells x 1e6 points and 63.8 for 65.3 on 80,000 cells x
// 4,096, but 1.01 for 0.98 on 48 cells x 65,536, where half as many units leave
// the last wave emptier.
//
// What bounds it: set-up takes a quarter, whole lines a quarter to a half,
// partial lines the rest (most of the afterbody's cool cells); issue slots are
// 70 % busy, the MUFU pipe about as much, and more resident warps help (32 an
// SM at 64 registers against 24 at 80).  Line sums in ms, before (one line
// at a time, a reciprocal a point, both exponentials in every run of a tile
// that holds the line's centre) and now: 200 cells x 1e6 points 33.9 -> 31.2,
// 80,000 cells x 4,096 points 76.9 -> 65.6, 48 x 65,536 1.04 -> 0.97, full
// Lorentz width 96 x 100,001 0.83 -> 0.74.
template <int PPT, int FL, int PB = 32>
__device__ __forceinline__ void warp_tile_f32(const LineSumArgs& a, int t, int64_t c, LineSlots<PB>& sl,
                                              WarpCell& wc, float4* acc, int lane, int64_t* cnt) {
    constexpr int TW = 32 * PPT;
    const int kt0 = (int)(a.k0 + (int64_t)t * TW);
    const int kt1 = (int)min(a.k0 + (int64_t)(t + 1) * TW, a.k0 + a.nk) - 1;   // inclusive
    const float kt0f = (float)kt0, kt1f = (float)kt1;
    const float lanef = (float)lane;       // lane's first point, relative to kt0
    // compensated sums (Kahan) of the per-batch partial sums, kept in shared
    // memory (acc[i * 32 + lane] = (s_j, c_j, s_k, c_k)); inside a batch of at
    // most PB lines the terms are added plainly in registers (error <= (PB - 1) u
    // of the batch's magnitude, u = 2^-24)
#pragma unroll
    for (int i = 0; i < PPT; ++i) acc[i * 32 + lane] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const float hf = (float)a.h;
    const float inv_hf = (float)(1.0 / a.h);
    const bool count = a.count != 0;
    if (lane == 0) {
        const CellPrep& cp = a.cp[c];
        wc.bve_ff = cp.bve_ff;
        wc.btr_ff = cp.btr_ff;
        wc.sqrtT_f = cp.sqrtT_f;
        wc.stc_f = cp.stc_f;
    }
    if (lane < a.S) {
        const double v = a.lnpref[c * a.S + lane];
        wc.lp[lane] = v > -INFINITY ? ff_from(v) : make_float2(-INFINITY, 0.0f);
        if (FL & 1) wc.cb[lane] = a.cb32[c * a.S + lane];
    }
    __syncwarp();
    const int beg = a.tile_off[t], end = a.tile_off[t + 1];
    constexpr int NH = PB / 32;   // staged halves of 32 pairs (one pair a lane each)
    for (int b = beg; b < end; b += PB) {
        PairF32 P[NH];
        bool valid[NH];
#pragma unroll
        for (int hh = 0; hh < NH; ++hh) {
            const int nb = min(32, end - (b + 32 * hh));
            valid[hh] = false;
            if (lane < nb) {
                const int l = a.tile_lines[b + 32 * hh + lane];
                const LineF32 L = a.lf[l];
                valid[hh] = setup_pair_f32<FL>(a, L, wc, wc.lp[L.species],
                                               (FL & 1) ? wc.cb[L.species] : make_float2(0.f, 0.f), l, c, hf, inv_hf,
                                               kt0, kt0f, kt1f, count, &P[hh], cnt);
            }
        }
        // the tile's parts of 128 points, four runs each: the lines' set-up serves all of them
#pragma unroll 1
        for (int g0 = 0; g0 < PPT; g0 += 4) {
            const float o0 = 32.0f * g0;
            int n = 0, nf = 0, nn = 0;   // lines staged: partial, whole far (from the front), whole near (from the end)
#pragma unroll
            for (int hh = 0; hh < NH; ++hh) {
                const PairF32& Q = P[hh];
                bool part = valid[hh] && Q.lo <= o0 + 127.0f && Q.hi >= o0;
                const bool whole = part && !(FL & 4) && Q.lo <= o0 && Q.hi >= o0 + 127.0f;
                const bool wnear = Q.x0 - Q.wn <= o0 + 127.0f && Q.x0 + Q.wn >= o0;
                const unsigned mf = __ballot_sync(0xffffffffu, whole && !wnear);
                const unsigned mn = __ballot_sync(0xffffffffu, whole && wnear);
                const unsigned lt = (1u << lane) - 1u;
                if (whole) {
                    const int q = wnear ? PB - 1 - nn - __popc(mn & lt) : nf + __popc(mf & lt);
                    sl.W0[q] = make_float4(Q.s, Q.ub, Q.ub_lo, Q.r);
                    sl.W1[q] = make_float2(Q.aj, Q.ak);
                    part = false;
                }
                nf += __popc(mf);
                nn += __popc(mn);
                const unsigned m = __ballot_sync(0xffffffffu, part);
                if (part) {
                    const int pos = n + __popc(m & lt), j = pos >> 1, o = pos & 1;
                    unsigned runs = 0;
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const float p0 = o0 + 32.0f * i;
                        if (Q.lo <= p0 + 31.0f && Q.hi >= p0)
                            runs |= (Q.x0 - Q.wn <= p0 + 31.0f && Q.x0 + Q.wn >= p0 ? 0x10001u : 1u) << i;
                    }
                    sl.runs[pos] = runs;
                    float* g = reinterpret_cast<float*>(&sl.G[0][j]) + o;
                    constexpr int GS = (int)(sizeof(sl.G[0]) / sizeof(float));
                    g[0] = -0.5f * (Q.lo + Q.hi);
                    g[2] = 0.5f * (Q.hi - Q.lo);
                    g[GS] = Q.ub;
                    g[GS + 2] = Q.ub_lo;
                    g[2 * GS] = Q.s;
                    g[2 * GS + 2] = Q.r;
                    g[3 * GS] = Q.aj;
                    g[3 * GS + 2] = Q.ak;
                }
                n += __popc(m);
            }
            if (n + nf + nn == 0) continue;   // the same for the whole warp
            if ((n & 1) && lane == 0) {   // an idle line beside the last one: u = 1 everywhere, in no window
                const int j = n >> 1;
                float* g = reinterpret_cast<float*>(&sl.G[0][j]) + 1;
                constexpr int GS = (int)(sizeof(sl.G[0]) / sizeof(float));
                sl.runs[n] = 0;
                g[0] = 0.0f;
                g[2] = -1.0f;
                g[GS] = 1.0f;
                g[GS + 2] = 0.0f;
                g[2 * GS] = 0.0f;
                g[2 * GS + 2] = 1.0f;
                g[3 * GS] = 0.0f;
                g[3 * GS + 2] = 0.0f;
            }
            __syncwarp();
            float bk[4], bj[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) bk[i] = bj[i] = 0.0f;
            const float kf = lanef + o0;
            if (FL & 4) {
                for (int q = 0; q < n; ++q) {
                    const float* g = reinterpret_cast<const float*>(&sl.G[0][q >> 1]) + (q & 1);
                    constexpr int GS = (int)(sizeof(sl.G[0]) / sizeof(float));
                    sweep_pair_voigt<4>(c_voigt, -g[0] - g[2], -g[0] + g[2], o0, kf, g[2 * GS], g[GS], g[GS + 2],
                                        g[2 * GS + 2], g[3 * GS], g[3 * GS + 2], bj, bk);
                }
            } else {
                sweep_wholes<4, PB, false>(sl, 0, nf, kf, bj, bk);
                sweep_wholes<4, PB, true>(sl, PB - nn, PB, kf, bj, bk);
                sweep_slots<4, PB>(sl, n, kf, bj, bk);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                float4 v = acc[(g0 + i) * 32 + lane];
                kahan_add(v.x, v.y, bj[i]);
                kahan_add(v.z, v.w, bk[i]);
                acc[(g0 + i) * 32 + lane] = v;
            }
            __syncwarp();
        }
    }
    float* K = reinterpret_cast<float*>(a.kappa) + c * a.ld - a.k0;
    float* J = reinterpret_cast<float*>(a.emis) + c * a.ld - a.k0;
#pragma unroll
    for (int i = 0; i < PPT; ++i) {
        const int k = kt0 + lane + 32 * i;
        const float4 v = acc[i * 32 + lane];
        // streaming stores: the rows are read back by the march of a later
        // chunk, long after they would have left L2, so they are marked
        // evict-first and leave L2 to the gathers running beside them
        if (k <= kt1) { __stcs(K + k, v.z); __stcs(J + k, v.x); }
    }
}

// Resident blocks per SM asked of the compiler: 32 warps per SM, so at most
// 64 registers per thread (200 cells x 1e6 points 31.2 ms, 28 warps 31.3, 24
// 32.2; 80,000 cells x 4,096 points 65.6, 66.2 and 67.3).  Tiles of 512 points
// keep 8 KB of sums a warp in shared memory: 16 warps.
#ifndef RAPRAL_LS_WARPS
#define RAPRAL_LS_WARPS 32
#endif
#define RAPRAL_LS_BLOCKS(PPT, WPB) (((PPT) > 8 ? 16 : RAPRAL_LS_WARPS) / (WPB))

template <int PPT, int WPB, int FL = 0, int PB = 32>
__global__ void __launch_bounds__(32 * WPB, RAPRAL_LS_BLOCKS(PPT, WPB)) k_line_sum_f32(LineSumArgs a) {
    if (*a.status) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t c = (int64_t)blockIdx.x * WPB + warp;
    if (c >= a.C) return;
    __shared__ __align__(16) LineSlots<PB> sl[WPB];
    __shared__ __align__(16) WarpCell wc[WPB];
    __shared__ float4 acc[WPB][32 * PPT];
    int64_t cnt[4] = {0, 0, 0, 0};
    warp_tile_f32<PPT, FL, PB>(a, blockIdx.y, c, sl[warp], wc[warp], acc[warp], lane, cnt);
    if (a.count) block_count(a.stats, cnt[0], cnt[1], cnt[2], cnt[3]);
}

// The same line sum as a persistent launch: a fixed number of blocks pull
// the units (tile, group of WPB cells) of k_line_sum_f32's grid, in its
// order (tile by tile), from an atomic counter; each warp does the same
// work as there, so the sums are bitwise the same.
template <int PPT, int WPB, int PB = 32>
__global__ void __launch_bounds__(32 * WPB, RAPRAL_LS_BLOCKS(PPT, WPB)) k_line_sum_f32_persist(LineSumArgs a, int64_t n_groups,
                                                                            int64_t total,
                                                                            unsigned long long* counter) {
    if (*a.status) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ __align__(16) LineSlots<PB> sl[WPB];
    __shared__ __align__(16) WarpCell wc[WPB];
    __shared__ float4 acc[WPB][32 * PPT];
    __shared__ long long unit_s;
    int64_t cnt[4] = {0, 0, 0, 0};
    for (;;) {
        if (threadIdx.x == 0) unit_s = (long long)atomicAdd(counter, 1ULL);
        __syncthreads();
        const int64_t u = unit_s;
        __syncthreads();
        if (u >= total) break;
        const int t = (int)(u / n_groups);
        const int64_t c = (u - (int64_t)t * n_groups) * WPB + warp;
        if (c < a.C) warp_tile_f32<PPT, 0, PB>(a, t, c, sl[warp], wc[warp], acc[warp], lane, cnt);
        __syncwarp();
    }
    if (a.count) block_count(a.stats, cnt[0], cnt[1], cnt[2], cnt[3]);
}

// Launches k_line_sum_f32_persist over the units of grid g: ctx->ls_persist
// blocks a SM, or as many as fit (-1); the unit counter (ctx->d_unit) was
// cleared by k_bin_fill.
template <int PPT, int WPB, int PB>
static cudaError_t launch_persist(rapral_ctx* ctx, const LineSumArgs& a, dim3 g) {
    int dev = 0, sms = 0, per_sm = ctx->ls_persist;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess && per_sm < 0)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_line_sum_f32_persist<PPT, WPB, PB>, 32 * WPB, 0);
    unsigned long long* counter = ctx->d_unit;
    if (e != cudaSuccess) return e;
    const int64_t total = (int64_t)g.x * g.y;
    const int64_t blocks = std::min<int64_t>(total, (int64_t)sms * std::max(1, per_sm));
    k_line_sum_f32_persist<PPT, WPB, PB><<<(unsigned)blocks, 32 * WPB, 0, ctx->stream>>>(a, (int64_t)g.x, total, counter);
    return cudaGetLastError();
}

// Persistent line sum over many independent requests: blocks pull work
// units (request, tile, group of WPB cells) from one atomic counter until the
// list is exhausted; units of a request are ordered tile by tile so blocks
// working at the same time share a tile's line list in L2.
template <int PPT, int WPB, bool BR = false, int PB = 32>
__global__ void __launch_bounds__(32 * WPB, RAPRAL_LS_BLOCKS(PPT, WPB)) k_line_sum_batch(const BatchItem* __restrict__ items,
                                                                       int n_items, int64_t total,
                                                                       unsigned long long* counter,
                                                                       unsigned long long* stats, const int* status) {
    if (*status) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ __align__(16) LineSlots<PB> sl[WPB];
    __shared__ __align__(16) WarpCell wc[WPB];
    __shared__ float4 acc[WPB][32 * PPT];
    __shared__ long long unit_s;
    int64_t cnt[4] = {0, 0, 0, 0};
    for (;;) {
        if (threadIdx.x == 0) unit_s = (long long)atomicAdd(counter, 1ULL);
        __syncthreads();
        const int64_t u = unit_s;
        __syncthreads();
        if (u >= total) break;
        int lo = 0, hi = n_items;     // last item whose first unit is <= u
        while (hi - lo > 1) {
            const int m = (lo + hi) >> 1;
            if (items[m].unit_off <= u) lo = m; else hi = m;
        }
        const BatchItem& it = items[lo];
        const int64_t local = u - it.unit_off;
        const int t = (int)(local / it.n_groups);
        const int64_t c = (local - (int64_t)t * it.n_groups) * WPB + warp;
        if (c < it.a.C)
            warp_tile_f32<PPT, BR ? 1 : 0, PB>(it.a, t, c, sl[warp], wc[warp], acc[warp],
                                               lane, cnt);
        __syncwarp();
    }
    if (items[0].a.count) block_count(stats, cnt[0], cnt[1], cnt[2], cnt[3]);
}

}  // namespace

cudaError_t launch_plan_reset(rapral_ctx* ctx, unsigned long long* d_max, const BinPlan* plan) {
    // maxima, widest window, total, status copy and the unsorted flag lie together in the arena
    const size_t n = (size_t)(reinterpret_cast<char*>(plan->unsorted + 1) - reinterpret_cast<char*>(d_max));
    return cudaMemsetAsync(d_max, 0, n, ctx->stream);
}

cudaError_t launch_line_plan(rapral_ctx* ctx, const rapral_species* sp, const rapral_lines* ln,
                             double lam_min, double h, const Phys& ph, const unsigned long long* d_max,
                             LinePrep* out, LineF32* out32, BinPlan* plan, const BroadArgs* br, double2* lb,
                             float2* lb32) {
    if (ln->n_lines == 0) return cudaSuccess;
    BroadArgs b = br ? *br : BroadArgs{};
    if (!broad_terms(br)) lb = nullptr, lb32 = nullptr;
    // a block's warps share one SM's FP64 pipe: a short list goes out a warp a
    // block (1,500 lines: 22 us as 6 blocks of eight warps)
    const int nt = ln->n_lines < 152 * 256 ? 32 : 256;
    k_line_plan<<<div_up(ln->n_lines, nt), nt, 0, ctx->stream>>>(
        *ln, sp->mass, sp->kind, sp->n_species, lam_min, h, ph, plan->k0, plan->nk, plan->tile_w, d_max, out, out32,
        plan->line_tiles, plan->wmax, plan->unsorted, b, lb, lb32, ctx->d_status);
    return cudaGetLastError();
}

cudaError_t launch_bin_count(rapral_ctx* ctx, const rapral_lines* ln, const rapral_grid* g, double h,
                             BinPlan* plan) {
    k_bin_count<<<(unsigned)plan->n_tiles, 256, 0, ctx->stream>>>(ln->lam0, ln->n_lines, plan->line_tiles,
                                                                  plan->unsorted, plan->wmax, g->lam_min, h,
                                                                  plan->k0, plan->nk, plan->tile_w, plan->tile_off,
                                                                  ctx->d_status);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_scan_counts<<<1, 1024, 0, ctx->stream>>>(plan->tile_off, plan->n_tiles, plan->total, ctx->d_status);
    return cudaGetLastError();
}

cudaError_t launch_bin_fill(rapral_ctx* ctx, const rapral_lines* ln, const rapral_grid* g, double h,
                            BinPlan* plan) {
    k_bin_fill<<<(unsigned)plan->n_tiles, 256, 0, ctx->stream>>>(ln->lam0, ln->n_lines, plan->line_tiles,
                                                                 plan->unsorted, plan->wmax, g->lam_min, h,
                                                                 plan->k0, plan->nk, plan->tile_w, plan->tile_off,
                                                                 plan->tile_lines, ctx->d_unit, ctx->d_status);
    return cudaGetLastError();
}

cudaError_t launch_scan_i64(rapral_ctx* ctx, int64_t* data, int64_t n) {
    k_scan<long long><<<1, 1024, 0, ctx->stream>>>(reinterpret_cast<long long*>(data), n);
    return cudaGetLastError();
}

static cudaError_t launch_line_sum_grid(rapral_ctx* ctx, const LineSumArgs& a, int precision, dim3 grid);

cudaError_t launch_line_sum(rapral_ctx* ctx, const LineSumArgs& a, int precision, int64_t n_tiles) {
    if (n_tiles == 0 || a.C == 0) return cudaSuccess;
    // cells along x (up to 2^31 - 1), tiles along y (<= 65535): consecutive
    // blocks share a tile's line list in L2
    dim3 grid((unsigned)a.C, (unsigned)n_tiles);
    if (ctx->ev_before) cudaEventRecord(ctx->ev_before, ctx->stream);
    cudaError_t e = launch_line_sum_grid(ctx, a, precision, grid);
    if (ctx->ev_after) cudaEventRecord(ctx->ev_after, ctx->stream);
    return e;
}

static cudaError_t launch_line_sum_grid(rapral_ctx* ctx, const LineSumArgs& a, int precision, dim3 grid) {
    if (precision == RAPRAL_FP64) {
        if (a.voigt) {   // one tiling with the exact line shape
            if (a.tile_w != 512) return cudaErrorInvalidValue;
            k_line_sum_f64<4, true><<<grid, 128, 0, ctx->stream>>>(a);
            return cudaGetLastError();
        }
        switch (a.tile_w) {
            case 128: k_line_sum_f64<1><<<grid, 128, 0, ctx->stream>>>(a); break;
            case 256: k_line_sum_f64<2><<<grid, 128, 0, ctx->stream>>>(a); break;
            case 512: k_line_sum_f64<4><<<grid, 128, 0, ctx->stream>>>(a); break;
            default: return cudaErrorInvalidValue;
        }
        return cudaGetLastError();
    }
    // FP32: warp-level kernel, WPB cells per block; with the optional
    // resonance / van der Waals terms four cells a block
    const int fl = (a.lb32 ? 1 : 0) | (a.dep_lnb ? 2 : 0) | (a.voigt ? 4 : 0);
    if (fl & 4) {   // exact Voigt shape: one tiling, 128 x 4
        if (a.tile_w != 128) return cudaErrorInvalidValue;
        dim3 gb(div_up(a.C, 4), grid.y);
        switch (fl) {
            case 4: k_line_sum_f32<4, 4, 4><<<gb, 128, 0, ctx->stream>>>(a); break;
            case 5: k_line_sum_f32<4, 4, 5><<<gb, 128, 0, ctx->stream>>>(a); break;
            case 6: k_line_sum_f32<4, 4, 6><<<gb, 128, 0, ctx->stream>>>(a); break;
            default: k_line_sum_f32<4, 4, 7><<<gb, 128, 0, ctx->stream>>>(a); break;
        }
        return cudaGetLastError();
    }
    if (fl) {
        dim3 gb(div_up(a.C, 4), grid.y);
#define RAPRAL_LSF(FL)                                                                   \
    switch (a.tile_w) {                                                                  \
        case 128: k_line_sum_f32<4, 4, FL><<<gb, 128, 0, ctx->stream>>>(a); break;      \
        case 256: k_line_sum_f32<8, 4, FL><<<gb, 128, 0, ctx->stream>>>(a); break;      \
        case 512: k_line_sum_f32<16, 4, FL><<<gb, 128, 0, ctx->stream>>>(a); break;     \
        default: return cudaErrorInvalidValue;                                           \
    }
        if (fl == 1) { RAPRAL_LSF(1) } else if (fl == 2) { RAPRAL_LSF(2) } else { RAPRAL_LSF(3) }
#undef RAPRAL_LSF
        return cudaGetLastError();
    }
    const int wpb = a.tile_w == 512 ? 4 : ctx->cells_per_block;
    dim3 g32(div_up(a.C, wpb), grid.y);
#define RAPRAL_LS32_PB(PPT, WPB, PB)                                                          \
    do {                                                                                      \
        if (ctx->ls_persist != 0 && ctx->d_unit) return launch_persist<PPT, WPB, PB>(ctx, a, g32); \
        k_line_sum_f32<PPT, WPB, 0, PB><<<g32, 32 * WPB, 0, ctx->stream>>>(a);                 \
    } while (0)
#define RAPRAL_LS32(PPT, WPB)                                  \
    do {                                                       \
        if (ctx->pairs_per_batch == 64) RAPRAL_LS32_PB(PPT, WPB, 64); \
        else RAPRAL_LS32_PB(PPT, WPB, 32);                     \
    } while (0)
    if (a.tile_w == 128 && wpb == 2) RAPRAL_LS32(4, 2);
    else if (a.tile_w == 128 && wpb == 4) RAPRAL_LS32(4, 4);
    else if (a.tile_w == 128 && wpb == 8) RAPRAL_LS32(4, 8);
    else if (a.tile_w == 256 && wpb == 2) RAPRAL_LS32(8, 2);
    else if (a.tile_w == 256 && wpb == 4) RAPRAL_LS32(8, 4);
    else if (a.tile_w == 256 && wpb == 8) RAPRAL_LS32(8, 8);
    else if (a.tile_w == 512) RAPRAL_LS32(16, 4);
    else return cudaErrorInvalidValue;
#undef RAPRAL_LS32
#undef RAPRAL_LS32_PB
    return cudaGetLastError();
}

template <int PPT, int WPB, bool BR = false, int PB = 32>
static cudaError_t batch_launch(rapral_ctx* ctx, const BatchItem* items, int n, int64_t total,
                                unsigned long long* counter, int* blocks_out, bool launch) {
    int per_sm = 0, dev = 0, sms = 0;
    cudaError_t e =
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_line_sum_batch<PPT, WPB, BR, PB>, 32 * WPB, 0);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int blocks = max(1, per_sm) * sms;
    if (blocks_out) *blocks_out = blocks;
    if (!launch) return cudaSuccess;
    k_line_sum_batch<PPT, WPB, BR, PB><<<blocks, 32 * WPB, 0, ctx->stream>>>(items, n, total, counter, ctx->d_stats,
                                                                             ctx->d_status);
    return cudaGetLastError();
}

cudaError_t launch_line_sum_batch(rapral_ctx* ctx, int tile_w, int wpb, int pb, const BatchItem* items, int n,
                                  int64_t total, unsigned long long* counter, int* blocks_out, bool launch, bool broad) {
    if (broad) {   // the optional Lorentz terms: four cells a block (the plan's group size), 32 pairs a pass
        if (wpb != 4 || pb != 32) return cudaErrorInvalidValue;
        if (tile_w == 128) return batch_launch<4, 4, true>(ctx, items, n, total, counter, blocks_out, launch);
        if (tile_w == 256) return batch_launch<8, 4, true>(ctx, items, n, total, counter, blocks_out, launch);
        if (tile_w == 512) return batch_launch<16, 4, true>(ctx, items, n, total, counter, blocks_out, launch);
        return cudaErrorInvalidValue;
    }
#define RAPRAL_BL(PPT, WPB)                                                                          \
    return pb == 64 ? batch_launch<PPT, WPB, false, 64>(ctx, items, n, total, counter, blocks_out, launch) \
                    : batch_launch<PPT, WPB, false, 32>(ctx, items, n, total, counter, blocks_out, launch)
    if (pb != 32 && pb != 64) return cudaErrorInvalidValue;
    if (tile_w == 128 && wpb == 2) RAPRAL_BL(4, 2);
    if (tile_w == 128 && wpb == 4) RAPRAL_BL(4, 4);
    if (tile_w == 128 && wpb == 8) RAPRAL_BL(4, 8);
    if (tile_w == 256 && wpb == 2) RAPRAL_BL(8, 2);
    if (tile_w == 256 && wpb == 4) RAPRAL_BL(8, 4);
    if (tile_w == 256 && wpb == 8) RAPRAL_BL(8, 8);
    if (tile_w == 512) RAPRAL_BL(16, 4);
#undef RAPRAL_BL
    return cudaErrorInvalidValue;
}

// Fourier coefficients a_1 .. a_N of f(t) = L^2 sec^2(t/2) e^{-L^2 tan^2(t/2)},
// L = (N / sqrt 2)^{1/2}, by the trapezoid rule on 4N points of [-pi, pi)
// (f vanishes at -pi): the coefficients of Weideman's rational expansion.
static void weideman(int N, double* a, double* L) {
    const int M = 2 * N, M2 = 2 * M;
    const double l = std::sqrt(N / std::sqrt(2.0));
    *L = l;
    for (int n = 1; n <= N; ++n) {
        double acc = 0.0;
        for (int j = -M + 1; j <= M - 1; ++j) {
            const double th = j * M_PI / M;
            const double t = l * std::tan(0.5 * th);
            acc += std::exp(-t * t) * (l * l + t * t) * std::cos(n * th);
        }
        a[n - 1] = acc / M2;
    }
}

const VoigtCoef& voigt_coefficients() {
    static const VoigtCoef vc = [] {
        VoigtCoef v{};
        weideman(RAPRAL_VOIGT_NW64, v.a64, &v.L64);
        double a32[RAPRAL_VOIGT_NW32], L32;
        weideman(RAPRAL_VOIGT_NW32, a32, &L32);
        for (int n = 0; n < RAPRAL_VOIGT_NW32; ++n) v.a32[n] = (float)a32[n];
        v.L32 = (float)L32;
        return v;
    }();
    return vc;
}

cudaError_t voigt_upload() {
    return cudaMemcpyToSymbol(c_voigt, &voigt_coefficients(), sizeof(VoigtCoef));
}
