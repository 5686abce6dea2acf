// Populations (Sec. 2.1) and per-cell preparation.
//
// k_populations: one block per (cell group, species).  Atoms: threads stride
// over the level list and sum g exp(-c2 E / T_ve).  Diatomics: threads stride
// over the rotational quantum number of each state and add
//   g_i exp(-c2 E_i / T_ve) exp(-c2 E_V / T_ve) / sigma (2J+1) L_alter exp(-c2 E_J / T_tr),
// which is the product form of g_i exp(-c2E_i/T_ee) Q_vr,i.  Fixed-order warp
// and block reductions keep the result deterministic.  FP64 accuracy
// throughout (partition sums are FP64 in both precisions).
#include "rapral_internal.cuh"
#include "exp_fix.cuh"

namespace {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ bool check_cell(const double* Ttr, const double* Tve, const double* n, int64_t i,
                                           int32_t ncol, int* status) {
    bool ok = true;
    const double a = Ttr[i], b = Tve[i];
    if (!(a > 0.0) || !(b > 0.0) || !isfinite(a) || !isfinite(b)) fail(status, CHK_CELL_T, i), ok = false;
    for (int j = 0; j < ncol; ++j) {
        const double v = n[i * ncol + j];
        if (!(v >= 0.0) || !isfinite(v)) { fail(status, CHK_CELL_N, i); ok = false; break; }
    }
    return ok;
}

__global__ void k_validate_cells(const double* Ttr, const double* Tve, const double* n, int64_t C,
                                 int32_t ncol, int* status) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < C) check_cell(Ttr, Tve, n, i, ncol, status);
}

// A block: one species, CC cells, its 256 threads along the levels (atoms) or
// the rotational ladders (diatomics).  What a term costs is its exponential;
// with expfix_boltzmann it is 95 integer operations and one FP64 multiply-add
// beside them (exp(double) kept the FP64 pipe busy at 21 operation times a
// term: 5000 cells, 53,000 terms a cell, 9.7 -> 0.96 ms).  A level is read and
// turned into fixed point once for its CC cells.
// The order of a cell's sum does not depend on CC.
template <int CC>
__global__ void __launch_bounds__(256) k_populations(rapral_species sp, const double* __restrict__ Ttr,
                                                     const double* __restrict__ Tve, const double* __restrict__ n,
                                                     int32_t ncol, int64_t C, double c2, double* __restrict__ lnpref,
                                                     int* status) {
    // one decision for the block: its warps share the tables and sums, and
    // other blocks of this launch may be setting the status meanwhile
    if (__syncthreads_or(*status != 0)) return;
    __shared__ uint64_t tab[EXPFIX_N];
    __shared__ double pv[CC][32];      // Boltzmann factors of 32 vibrational levels of a state, with its weight
    __shared__ double red[CC][8];
    expfix_load(tab);
    const int S = sp.n_species, s = blockIdx.y;
    const int64_t c0 = (int64_t)blockIdx.x * CC;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (s == 0 && tid < CC && c0 + tid < C) check_cell(Ttr, Tve, n, c0 + tid, ncol, status);
    __shared__ double sb[2][CC];       // c2 / T_ve, c2 / T_tr: a division a block and cell, not one a thread
    if (tid < 2 * CC) {
        const int q = tid >> 1;
        const int64_t c = c0 + q < C ? c0 + q : C - 1;
        sb[tid & 1][q] = c2 / ((tid & 1) ? Ttr : Tve)[c];
    }
    __syncthreads();
    double bve[CC], btr[CC], z[CC];
    ExpFixScale sc[CC];
#pragma unroll
    for (int q = 0; q < CC; ++q) {
        bve[q] = sb[0][q];
        btr[q] = sb[1][q];
        z[q] = 0.0;
    }
    if (sp.kind[s] == RAPRAL_ATOM) {
        const int64_t b = sp.atom_off[s + 1];
#pragma unroll
        for (int q = 0; q < CC; ++q) sc[q] = expfix_scale(bve[q]);
        for (int64_t l = sp.atom_off[s] + tid; l < b; l += 256) {
            const double E = sp.atom_E[l], g = sp.atom_g[l];
            const uint64_t Ef = expfix_energy(E);
#pragma unroll
            for (int q = 0; q < CC; ++q) z[q] = fma(g, expfix_boltzmann(Ef, sc[q], E, bve[q], tab), z[q]);
        }
    } else {
#pragma unroll
        for (int q = 0; q < CC; ++q) sc[q] = expfix_scale(btr[q]);
        for (int64_t i = sp.st_off[s]; i < sp.st_off[s + 1]; ++i) {
            const int nv = sp.st_nv[i], nj = sp.st_nj[i];
            const double La = sp.st_Lalt[2 * i], Lb = sp.st_Lalt[2 * i + 1];
            const double* rot = sp.rot_E + sp.st_rot_off[i];
            const double* vib = sp.vib_E + sp.st_vib_off[i];
            for (int v0 = 0; v0 < nv; v0 += 32) {
                const int nvc = nv - v0 < 32 ? nv - v0 : 32;
                __syncthreads();
                for (int x = tid; x < CC * nvc; x += 256) {   // a (cell, level) a thread
                    const int q = x / nvc, v = x - q * nvc;
                    const double b = sb[0][q];
                    pv[q][v] = sp.st_g[i] * exp_fix(-b * sp.st_E[i], tab) / sp.st_sigma[i] *
                               exp_fix(-b * vib[v0 + v], tab);
                }
                __syncthreads();
                for (int J = tid; J < nj; J += 256) {
                    double y[CC];
#pragma unroll
                    for (int q = 0; q < CC; ++q) y[q] = 0.0;
                    for (int v = 0; v < nvc; ++v) {
                        const double E = rot[(int64_t)(v0 + v) * nj + J];
                        const uint64_t Ef = expfix_energy(E);
#pragma unroll
                        for (int q = 0; q < CC; ++q)
                            y[q] = fma(pv[q][v], expfix_boltzmann(Ef, sc[q], E, btr[q], tab), y[q]);
                    }
                    const double w = (2.0 * J + 1.0) * ((J & 1) ? Lb : La);
#pragma unroll
                    for (int q = 0; q < CC; ++q) z[q] = fma(w, y[q], z[q]);
                }
            }
        }
    }
#pragma unroll
    for (int q = 0; q < CC; ++q) {
        z[q] = warp_sum(z[q]);
        if (lane == 0) red[q][warp] = z[q];
    }
    __syncthreads();
    if (tid < CC && c0 + tid < C) {
        const int64_t c = c0 + tid;
        double Z = red[tid][0];
        for (int w = 1; w < 8; ++w) Z += red[tid][w];
        const double N = n[c * ncol + sp.density_col[s]];
        lnpref[c * S + s] = (N > 0.0) ? log(N) - log(Z) : -INFINITY;
    }
}

// Largest of the block's positive doubles (as bits; 0: none) into *dst, one
// atomic a block: one a cell on the same word cost 0.1 ms on 80,000 cells.
__device__ __forceinline__ void block_max(unsigned long long v, unsigned long long* blk, unsigned long long* dst) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long x = __shfl_xor_sync(0xffffffffu, v, o);
        v = x > v ? x : v;
    }
    if (threadIdx.x == 0) *blk = 0ULL;
    __syncthreads();
    if ((threadIdx.x & 31) == 0 && v) atomicMax(blk, v);
    __syncthreads();
    if (threadIdx.x == 0 && *blk) atomicMax(dst, *blk);
    __syncthreads();
}

// Checks and record of one cell per thread.
__global__ void __launch_bounds__(256) k_cell_prep(const double* __restrict__ Ttr, const double* __restrict__ Tve,
                                                   const double* __restrict__ n, int32_t ncol, int32_t ne_col,
                                                   int64_t C, double c2, CellPrep* __restrict__ out,
                                                   unsigned long long* dmax, int* status) {
    __shared__ unsigned long long blk;
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    unsigned long long mT = 0ULL, mS = 0ULL;
    if (c < C && check_cell(Ttr, Tve, n, c, ncol, status)) {
        CellPrep p;
        const double tt = Ttr[c], tv = Tve[c];
        p.bve = c2 / tv;
        p.btr = c2 / tt;
        p.sqrtT = sqrt(tt);
        p.stc = pow(tv / 10000.0, 0.33) * (n[c * ncol + ne_col] / 1e16);
        p.bve_f = (float)p.bve;
        p.btr_f = (float)p.btr;
        p.sqrtT_f = (float)p.sqrtT;
        p.stc_f = (float)p.stc;
        p.bve_ff = ff_from(p.bve);
        p.btr_ff = ff_from(p.btr);
        out[c] = p;
        // positive doubles order like their bit patterns
        mT = (unsigned long long)__double_as_longlong(p.sqrtT);
        mS = (unsigned long long)__double_as_longlong(p.stc);
    }
    block_max(mT, &blk, &dmax[0]);
    block_max(mS, &blk, &dmax[1]);
}

// Ground-level weight of each atomic species: the summed g of its levels at
// E = 0 (0 for molecules).  A block a species, threads along its levels: what
// it takes is load latency (20,000 levels on two atoms, cold: one thread 1.2 ms,
// a warp 57 us, 512 threads 10 us).
constexpr int GROUND_THREADS = 512;
__global__ void __launch_bounds__(GROUND_THREADS) k_ground_weights(rapral_species sp, double* g0) {
    __shared__ double part[GROUND_THREADS / 32];
    const int s = blockIdx.x, lane = threadIdx.x & 31;
    double g = 0.0;
    if (sp.kind[s] == RAPRAL_ATOM) {
        const int64_t b = sp.atom_off[s + 1];
#pragma unroll 4
        for (int64_t k = sp.atom_off[s] + threadIdx.x; k < b; k += GROUND_THREADS)
            if (sp.atom_E[k] == 0.0) g += sp.atom_g[k];
    }
    g = warp_sum(g);
    if (lane == 0) part[threadIdx.x >> 5] = g;
    __syncthreads();
    if (threadIdx.x >= 32) return;
    g = warp_sum(lane < GROUND_THREADS / 32 ? part[lane] : 0.0);
    if (lane == 0) g0[s] = g;
}

// Per (cell, atomic species): ground-level density N_0 = n_s g_0 / Z_s and
// the van der Waals factor W = 6.65e-29 N (2T/M)^0.5 + 2.925e-29 N_o (2T/M_o)^0.5
// (the other heavy particles in column order); zeros for molecules or for
// terms that are off.  Largest values over the cells per species in dmax.  A
// thread a (cell, species): a few cells are a chain of FP64 exp, log and square
// roots (96 cells x 8 species: 28 us with the species in turn, 11 so).
__global__ void k_cell_broad(rapral_species sp, rapral_cells cells, BroadArgs br, const double* __restrict__ g0,
                             double2* __restrict__ cb, float2* __restrict__ cb32, unsigned long long* dmax,
                             const int* status) {
    if (*status) return;
    __shared__ unsigned long long blk;
    const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const bool in = c < cells.n_cells;
    const int S = sp.n_species, nc = cells.n_cols, s = blockIdx.y;
    double N0 = 0.0, W = 0.0;
    if (in && sp.kind[s] == RAPRAL_ATOM) {
        const double* n = cells.n + c * nc;
        if ((br.flags & RAPRAL_BROAD_RESONANCE) && g0[s] > 0.0) N0 = exp(cells.lnpref[c * S + s] + log(g0[s]));
        if (br.flags & RAPRAL_BROAD_VDW) {
            const double T = cells.Ttr[c];
            const int col = sp.density_col[s];
            double No = 0.0, NoM = 0.0;
            for (int k = 0; k < nc && k < br.ncol; ++k) {
                if (k == col || !(br.colmass[k] > 0.0)) continue;
                No += n[k];
                NoM += n[k] * br.colmass[k];
            }
            W = 6.65e-29 * n[col] * sqrt(2.0 * T / sp.mass[s]);
            if (No > 0.0) W += 2.925e-29 * No * sqrt(2.0 * T / (NoM / No));
        }
    }
    if (in) {
        cb[c * S + s] = make_double2(N0, W);
        cb32[c * S + s] = make_float2((float)N0, (float)W);
    }
    block_max((unsigned long long)__double_as_longlong(N0), &blk, &dmax[2 + 2 * s]);
    block_max((unsigned long long)__double_as_longlong(W), &blk, &dmax[3 + 2 * s]);
}

}  // namespace

cudaError_t launch_broad_cells(rapral_ctx* ctx, const rapral_species* sp, const rapral_cells* cells,
                               const BroadArgs& br, double* g0, double2* cb, float2* cb32, unsigned long long* d_max) {
    const int S = sp->n_species;
    k_ground_weights<<<S, GROUND_THREADS, 0, ctx->stream>>>(*sp, g0);   // d_max was cleared by launch_plan_reset
    if (cells->n_cells == 0) return cudaGetLastError();
    k_cell_broad<<<dim3(div_up(cells->n_cells, 128), (unsigned)S), 128, 0, ctx->stream>>>(*sp, *cells, br, g0, cb,
                                                                                          cb32, d_max, ctx->d_status);
    return cudaGetLastError();
}

cudaError_t launch_validate_cells(rapral_ctx* ctx, const rapral_cells* cells) {
    k_validate_cells<<<div_up(cells->n_cells, 256), 256, 0, ctx->stream>>>(
        cells->Ttr, cells->Tve, cells->n, cells->n_cells, cells->n_cols, ctx->d_status);
    return cudaGetLastError();
}

cudaError_t launch_populations(rapral_ctx* ctx, const rapral_species* sp, const rapral_cells* cells,
                               double* lnpref, const Phys& ph) {
    // Four cells a block share a level's load and conversion; one cell a block
    // where four would leave the chip with fewer than eight blocks an SM
    const int64_t C = cells->n_cells, S = sp->n_species;
    if (C * S >= 4 * 152 * 8)
        k_populations<4><<<dim3(div_up(C, 4), (unsigned)S), 256, 0, ctx->stream>>>(
            *sp, cells->Ttr, cells->Tve, cells->n, cells->n_cols, C, ph.c2, lnpref, ctx->d_status);
    else
        k_populations<1><<<dim3((unsigned)C, (unsigned)S), 256, 0, ctx->stream>>>(
            *sp, cells->Ttr, cells->Tve, cells->n, cells->n_cols, C, ph.c2, lnpref, ctx->d_status);
    return cudaGetLastError();
}

cudaError_t launch_cell_prep(rapral_ctx* ctx, const rapral_cells* cells, const Phys& ph, CellPrep* out,
                             unsigned long long* d_max) {
    k_cell_prep<<<div_up(cells->n_cells, 256), 256, 0, ctx->stream>>>(
        cells->Ttr, cells->Tve, cells->n, cells->n_cols, cells->ne_col, cells->n_cells, ph.c2, out, d_max,
        ctx->d_status);
    return cudaGetLastError();
}

// Saha-Boltzmann populations of an atomic radiator (Sec. 2.1): N_i =
// N_+ N_e (h^2 / (2 pi m_e k T))^1.5 g_i e^{hc (E_ion - E_i) / kT} / (2 Q_+),
// that is the prefactor ln(N / Z) of the Boltzmann form replaced by
// ln(N_+ N_e) + 1.5 ln(h^2 / (2 pi m_e k T)) + c2 E_ion / T - ln(2 Q_+), T = T_ve.
// No ions or electrons: -inf (no population).
__global__ void k_saha_prefactor(const double* __restrict__ Tve, const double* __restrict__ n, int ncol, int ne_col,
                                 int64_t C, int s, int S, double E_ion, int ion_col, int n_terms,
                                 const double* __restrict__ ion_E, const double* __restrict__ ion_g, Phys ph,
                                 double* __restrict__ lnpref, const int* status) {
    if (*status) return;
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= C) return;
    const double T = Tve[c];
    double Qp = 0.0;
    for (int k = 0; k < n_terms; ++k) Qp += ion_g[k] * exp(-ph.c2 * ion_E[k] / T);
    const double pe = n[c * ncol + ion_col] * n[c * ncol + ne_col];
    lnpref[c * S + s] = pe > 0.0 && Qp > 0.0
                            ? log(n[c * ncol + ion_col]) + log(n[c * ncol + ne_col]) +
                                  1.5 * log(ph.h * ph.h / (2.0 * M_PI * ph.me * ph.kB * T)) + ph.c2 * E_ion / T -
                                  log(2.0 * Qp)
                            : -INFINITY;
}

cudaError_t launch_saha_prefactor(rapral_ctx* ctx, const rapral_cells* cells, int s, int S, double E_ion,
                                  int ion_col, int n_terms, const double* ion_E, const double* ion_g,
                                  const Phys& ph, double* lnpref) {
    if (cells->n_cells == 0) return cudaSuccess;
    k_saha_prefactor<<<div_up(cells->n_cells, 256), 256, 0, ctx->stream>>>(
        cells->Tve, cells->n, cells->n_cols, cells->ne_col, cells->n_cells, s, S, E_ion, ion_col, n_terms, ion_E,
        ion_g, ph, lnpref, ctx->d_status);
    return cudaGetLastError();
}
