// Build orchestration for one J/K evaluation (Sections 2.5, 2.6 and 3.2 of
// arXiv:2410.22278) and the small bandwidth-bound kernels around it.
//
// Step order on the caller's stream:
//   1. D' = F o D with F_mn = f_m f_n the Cartesian component factors of
//      Eq. local_normalization, so every kernel works on raw Cartesian
//      functions; per-shell-block max |D'| for the precision policy.
//   2. real-space (erfc) quartet kernels per class pair -> X (Coulomb), Y
//      (exchange) accumulators, FP64 atomics.
//   3. reciprocal (erf) part per chunk of G: structure-factor slab M,
//      rho_D = M^T vec(D') and J_LR += M rho_D (Coulomb), Z = D' M per G and
//      K_LR += [M_1 .. M_g] [Z_1; ..; Z_g] (exchange).
//   4. removed K = 0 term in closed form: -(pi/(V w^2)) Tr(D'S) S and
//      -(pi/(V w^2)) S D' S.
//   5. J = F o (X + X^T + J_LR + J_bg), K = F o (Y + Y^T + K_LR + K_bg).
#include <algorithm>
#include <cstdio>
#include <map>
#include <string>

#include "jeng.cuh"
#include "kernels.cuh"
#include "launch.h"
#include "plan.h"
#include "real_units.h"

namespace jk {

__global__ void k_scale(int n, const double *__restrict__ f, const double *__restrict__ A, double *__restrict__ B)
{
    const size_t n2 = (size_t)n * n;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n2; i += (size_t)gridDim.x * blockDim.x)
        B[i] = f[i / n] * f[i % n] * A[i];
}

__global__ void k_to_float(size_t n, const double *__restrict__ a, float *__restrict__ b)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) b[i] = (float)a[i];
}

// max |D'| per shell block, its single-precision copy and the largest of all
// (dmaxf[nshell^2], zeroed before the launch)
__global__ void k_dmax(PlanDev pl, const double *__restrict__ Dp, double *__restrict__ dmax, float *__restrict__ dmaxf)
{
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const int nsh = pl.nshell;
    if (idx >= (long long)nsh * nsh) return;
    const int I = (int)(idx / nsh), J = (int)(idx % nsh);
    const ShellRec a = pl.shells[I], b = pl.shells[J];
    double m = 0;
    for (int i = 0; i < ncart(a.l); ++i)
        for (int j = 0; j < ncart(b.l); ++j) m = fmax(m, fabs(Dp[(size_t)(a.ao + i) * pl.nbf + b.ao + j]));
    dmax[idx] = m;
    dmaxf[idx] = (float)m;
    atomicMax(reinterpret_cast<int *>(dmaxf + (size_t)nsh * nsh), __float_as_int((float)m));  // m >= 0: ordered as integers
}

// out[k] += sum_i A_k[i] * B[i] for k = 0, 1 (two traces in one pass)
__global__ void k_dot2(size_t n2, const double *__restrict__ B, const double *__restrict__ A0, const double *__restrict__ A1,
                       double *__restrict__ out)
{
    double s0 = 0, s1 = 0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n2; i += (size_t)gridDim.x * blockDim.x) {
        if (A0) s0 += A0[i] * B[i];
        if (A1) s1 += A1[i] * B[i];
    }
    __shared__ double sh[2][32];
    s0 = warp_sum(s0);
    s1 = warp_sum(s1);
    if ((threadIdx.x & 31) == 0) {
        sh[0][threadIdx.x >> 5] = s0;
        sh[1][threadIdx.x >> 5] = s1;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        const int nw = blockDim.x >> 5;
        s0 = threadIdx.x < nw ? sh[0][threadIdx.x] : 0.0;
        s1 = threadIdx.x < nw ? sh[1][threadIdx.x] : 0.0;
        s0 = warp_sum(s0);
        s1 = warp_sum(s1);
        if (threadIdx.x == 0) {
            atomicAdd(out, s0);
            atomicAdd(out + 1, s1);
        }
    }
}

// Packed upper triangles (row-major, i <= j): entry (i, j) at
// i n - i (i - 1) / 2 + j - i.  The structure factors M_b are symmetric in
// their two basis indices (each unique shell pair writes both blocks), so
// the Coulomb contraction needs one triangle: rho_b = sum_{i<=j} M_b(ij)
// Ds(ij) with Ds the symmetrised density (D'_ij + D'_ji off the diagonal),
// and J_LR(ij) = J_LR(ji) = sum_b M_b(ij) rho_b.
__device__ __forceinline__ long long tri_index(long long n, long long i, long long j) { return i * n - i * (i - 1) / 2 + j - i; }

// Ap[b] = upper triangle of A[b] for nb matrices n x n
__global__ void k_pack_upper(int n, long long npk, int nb, const double *__restrict__ A, double *__restrict__ Ap)
{
    const long long n2 = (long long)n * n, tot = n2 * nb;
    for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < tot; idx += (long long)gridDim.x * blockDim.x) {
        const long long b = idx / n2, r = idx - b * n2, i = r / n, j = r - i * n;
        if (j >= i) Ap[b * npk + tri_index(n, i, j)] = A[idx];
    }
}

// Ds = packed D + D^T off the diagonal, D on it
__global__ void k_sym_density(int n, const double *__restrict__ D, double *__restrict__ Ds)
{
    const long long n2 = (long long)n * n;
    for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < n2; idx += (long long)gridDim.x * blockDim.x) {
        const long long i = idx / n, j = idx - i * n;
        if (j > i) Ds[tri_index(n, i, j)] = D[idx] + D[j * n + i];
        else if (j == i) Ds[tri_index(n, i, i)] = D[idx];
    }
}

// J (n x n) = the symmetric matrix of the packed Jp
__global__ void k_unpack_sym(int n, const double *__restrict__ Jp, double *__restrict__ J)
{
    const long long n2 = (long long)n * n;
    for (long long idx = (long long)blockIdx.x * blockDim.x + threadIdx.x; idx < n2; idx += (long long)gridDim.x * blockDim.x) {
        const long long i = idx / n, j = idx - i * n;
        J[idx] = Jp[i <= j ? tri_index(n, i, j) : tri_index(n, j, i)];
    }
}

// J = F o (X + X^T + JLR + c tr S), K = F o (Y + Y^T + KLR + c SDS)
__global__ void k_final(int n, const double *__restrict__ f, const double *__restrict__ X, const double *__restrict__ Y,
                        const double *__restrict__ JLR, const double *__restrict__ KLR, const double *__restrict__ S,
                        const double *__restrict__ SDS, const double *__restrict__ trDS, double c, const unsigned *__restrict__ err,
                        double *__restrict__ J, double *__restrict__ K)
{
    const size_t n2 = (size_t)n * n;
    const double tr = *trDS;
    // a wait of a tensor-core GEMM ran out: the result is not trusted
    const double poison = *err ? __longlong_as_double(0x7ff8000000000000ll) : 0.0;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n2; i += (size_t)gridDim.x * blockDim.x) {
        const size_t r = i / n, cidx = i % n, t = cidx * n + r;
        const double ff = f[r] * f[cidx];
        if (J) J[i] = ff * (X[i] + X[t] + 0.5 * (JLR[i] + JLR[t]) + c * tr * S[i]) + poison;
        if (K) K[i] = ff * (Y[i] + Y[t] + 0.5 * (KLR[i] + KLR[t]) + c * 0.5 * (SDS[i] + SDS[t])) + poison;
    }
}

template <int LA, int LB>
static void sfac_go(const PlanDev &pl, int sp0, int sp1, const double *gv, int g0, int gcur, const double *gtab, double *M,
                    cudaStream_t st)
{
    const long long nt = (long long)(sp1 - sp0) * gcur;
    if (nt <= 0) return;
    k_sfac<LA, LB><<<(unsigned)((nt + 127) / 128), 128, 0, st>>>(pl, sp0, sp1, gv, g0, gcur, gtab, M);
}

void launch_sfac(int cls, const PlanDev &pl, int sp0, int sp1, const double *gv, int g0, int gcur, const double *gtab, double *M,
                 cudaStream_t st)
{
    switch (cls) {
    case 0: sfac_go<0, 0>(pl, sp0, sp1, gv, g0, gcur, gtab, M, st); break;
    case 1: sfac_go<1, 0>(pl, sp0, sp1, gv, g0, gcur, gtab, M, st); break;
    case 2: sfac_go<1, 1>(pl, sp0, sp1, gv, g0, gcur, gtab, M, st); break;
    case 3: sfac_go<2, 0>(pl, sp0, sp1, gv, g0, gcur, gtab, M, st); break;
    case 4: sfac_go<2, 1>(pl, sp0, sp1, gv, g0, gcur, gtab, M, st); break;
    case 5: sfac_go<2, 2>(pl, sp0, sp1, gv, g0, gcur, gtab, M, st); break;
    default: break;
    }
}

template <int LA, int LB>
static void sfac_df_go(const PlanDev &pl, int sp0, int sp1, int g0, int gcur, const float2 *gtab, double *M, cudaStream_t st)
{
    const long long nt = (long long)(sp1 - sp0) * gcur;
    if (nt <= 0) return;
    k_sfac_df<LA, LB><<<(unsigned)((nt + 127) / 128), 128, 0, st>>>(pl, sp0, sp1, g0, gcur, gtab, M);
}

static void launch_sfac_df(int cls, const PlanDev &pl, int sp0, int sp1, int g0, int gcur, const float2 *gtab, double *M, cudaStream_t st)
{
    switch (cls) {
    case 0: sfac_df_go<0, 0>(pl, sp0, sp1, g0, gcur, gtab, M, st); break;
    case 1: sfac_df_go<1, 0>(pl, sp0, sp1, g0, gcur, gtab, M, st); break;
    case 2: sfac_df_go<1, 1>(pl, sp0, sp1, g0, gcur, gtab, M, st); break;
    case 3: sfac_df_go<2, 0>(pl, sp0, sp1, g0, gcur, gtab, M, st); break;
    case 4: sfac_df_go<2, 1>(pl, sp0, sp1, g0, gcur, gtab, M, st); break;
    case 5: sfac_df_go<2, 2>(pl, sp0, sp1, g0, gcur, gtab, M, st); break;
    default: break;
    }
}

// (pi/p)^{3/2} e^{-G^2/4p} for every distinct pair exponent p and every G of
// a chunk, laid out [p][g] (consecutive threads of the structure-factor
// kernel read consecutive g); into tab (FP64) or, when tab2 is given, into
// tab2 as double-floats times the weight sqrt(8 pi w(G) / V) of the G
__global__ void k_gauss_table(int npv, const double *__restrict__ pv, const double *__restrict__ gv, int g0, int gcur,
                              double *__restrict__ tab, float2 *__restrict__ tab2)
{
    const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= (long long)npv * gcur) return;
    const int ip = (int)(e / gcur), gi = (int)(e % gcur);
    const double *g = gv + 4 * (size_t)(g0 + gi);
    const double G2 = g[0] * g[0] + g[1] * g[1] + g[2] * g[2], p = pv[ip];
    const double v = (kPi / p) * sqrt(kPi / p) * exp(-G2 / (4.0 * p));
    if (tab2) {
        const dfl d = dfl_split(v * g[3]);
        tab2[e] = make_float2(d.hi, d.lo);
    } else {
        tab[e] = v;
    }
}

void launch_gauss_table(const Plan *P, int g0, int gcur, double *tab, cudaStream_t st)
{
    const long long ne = (long long)P->pvals.size() * gcur;
    if (ne > 0) k_gauss_table<<<(unsigned)((ne + 255) / 256), 256, 0, st>>>((int)P->pvals.size(), P->d_pvals, P->d_gvec, g0, gcur, tab, nullptr);
}

static int grid_for(size_t n) { return (int)std::min<size_t>((n + 255) / 256, 152 * 16); }

// Hermite densities (back = false) or the Hermite-to-Cartesian step (back =
// true) of the J-engine for the images of class cls (l_I >= l_J)
template <int LA, int LB>
static void hermite_go(bool back, const PlanDev &pl, int b0, int b1, const Workspace &w, const double *Dp, bool f32, double *X,
                       cudaStream_t st)
{
    if (b1 <= b0) return;
    const unsigned g = (unsigned)((b1 - b0 + 127) / 128);
    if (back)
        k_hermite_back<LA, LB><<<g, 128, 0, st>>>(pl, b0, b1, w.hs, w.JH, X);
    else
        k_hermite_density<LA, LB><<<g, 128, 0, st>>>(pl, b0, b1, Dp, w.hs, w.DhD, f32 ? w.DhF : nullptr);
}

static void launch_hermite(int cls, bool back, const PlanDev &pl, int b0, int b1, const Workspace &w, const double *Dp, bool f32,
                           double *X, cudaStream_t st)
{
    switch (cls) {
    case 0: hermite_go<0, 0>(back, pl, b0, b1, w, Dp, f32, X, st); break;
    case 1: hermite_go<1, 0>(back, pl, b0, b1, w, Dp, f32, X, st); break;
    case 2: hermite_go<1, 1>(back, pl, b0, b1, w, Dp, f32, X, st); break;
    case 3: hermite_go<2, 0>(back, pl, b0, b1, w, Dp, f32, X, st); break;
    case 4: hermite_go<2, 1>(back, pl, b0, b1, w, Dp, f32, X, st); break;
    case 5: hermite_go<2, 2>(back, pl, b0, b1, w, Dp, f32, X, st); break;
    default: break;
    }
}

// The warps of a warp-per-bra launch over the bras [b0, b1) and kets [k0, k1)
// (TileMap) of the bra class B.  kchunk is the mean number of kets of a warp: a
// warp gets the work of kchunk kets of the mean primitive count with a bra of
// the class's mean one (also where only a part of its bras is launched).
// Images are in descending order of primitive count inside a class, so a
// range of bras of similar count is contiguous; a new range starts where the
// count has fallen by a quarter.
static TileMap tile_map(const Plan *P, const ClassRange &B, int b0, int b1, int k0, int k1, int kchunk)
{
    TileMap m{};
    if (b1 <= b0 || k1 <= k0) return m;
    const auto prims = [&](int i0, int i1) {
        return (double)(P->spi[i1 - 1].pp0 + P->spi[i1 - 1].npp - P->spi[i0].pp0);
    };
    const double pk = prims(k0, k1);
    double work = (double)kchunk * (prims(B.b0, B.b1) / (B.b1 - B.b0)) * (pk / (k1 - k0));
    // at most 2^28 warps (blockIdx.x); only a hand-set schedule gets there
    work = std::max(work, prims(b0, b1) * pk / (double)(1 << 28));
    for (int b = b0; b < b1;) {
        const int top = P->spi[b].npp;
        int e = b1;
        if (m.n < 7)  // the eighth range takes what is left
            e = (int)(std::partition_point(P->spi.begin() + b, P->spi.begin() + b1, [&](const SpiRec &s) { return 4 * s.npp > 3 * top; }) -
                      P->spi.begin());
        TileMap::Range &g = m.g[m.n];
        g.b0 = b;
        g.b1 = e;
        g.W = (int)std::min(pk, std::max(1.0, work / top));
        g.nch = (int)((pk + g.W - 1) / g.W);
        g.first = m.items;
        m.items += (long long)(e - b) * g.nch;
        ++m.n;
        b = e;
    }
    return m;
}

static int cuda_check(const char *what)
{
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return fail(JK_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
    return JK_OK;
}

int compute_overlap_raw(Plan *P, cudaStream_t st)
{
    PlanDev pl = P->dev();
    for (int c = 0; c < JK_NCLASS_MAX; ++c)
        launch_sfac(c, pl, P->spair_class_off[c], P->spair_class_off[c + 1], P->d_g0, 0, 1, P->d_gtab0, P->ws.M, st);
    cudaMemcpyAsync(P->d_S, P->ws.M, sizeof(double) * P->nbf * P->nbf, cudaMemcpyDeviceToDevice, st);
    return cuda_check("overlap");
}

void PhaseTimer::begin(cudaStream_t s)
{
    st = cur = s;
    next = 0;
    marks.clear();
    for (int i = 0; i < kPhases; ++i) launches[i] = 0;
}
int PhaseTimer::start(int phase)
{
    (void)phase;
    if (next >= (int)pool.size()) {
        cudaEvent_t e;
        cudaEventCreate(&e);
        pool.push_back(e);
    }
    cudaEventRecord(pool[next], cur);
    return next++;
}
void PhaseTimer::stop(int phase, int ev_start, int nlaunch)
{
    int e = start(phase);
    marks.push_back({phase, {ev_start, e}});
    launches[phase] += nlaunch;
}
void PhaseTimer::destroy()
{
    for (auto e : pool) cudaEventDestroy(e);
    pool.clear();
}

// Reciprocal (erf) part of the build on stream st: structure factors (or
// the cache), the Coulomb slab passes and the exchange contraction, chunk
// by chunk of G.  Small plans enqueue it on a side stream, beside real space.
static int reciprocal_phase(Plan *P, double *J, double *K, cudaStream_t st)
{
    const int n = P->nbf;
    const size_t n2 = (size_t)n * n;
    PlanDev pl = P->dev();
    Workspace &w = P->ws;
    const bool mixed = P->precision == JK_MIXED;
    PhaseTimer &tm = P->timer;
    int ev, rc;
    const int ng = (int)(P->gvec.size() / 4);
    // mixed precision: structure factors in double-float on the FP32 pipe
    const bool sfac_df = mixed && P->sfac_df && w.gtab2;
    // the D-independent structure factors (and their exchange slices) come
    // from the reciprocal cache once a build has filled it; a mixed plan
    // caches them as packed upper triangles for the Coulomb contraction (the
    // exchange reads its BF16 slices), an FP64 plan in full
    RecipCache &cache = P->cache;
    const bool packed = cache.on && mixed;
    const long long npk = (long long)n * (n + 1) / 2;
    if (J && packed) {
        // symmetrised density and the packed J_LR accumulator in the
        // epilogue's scratch (free until the epilogue)
        k_sym_density<<<grid_for(n2), 256, 0, st>>>(n, w.Dp, w.T1);
        cudaMemsetAsync(w.T2, 0, npk * sizeof(double), st);
    }
    for (int g0 = 0, chunk = 0; g0 < ng; g0 += w.gc, ++chunk) {
        const int gcur = std::min(w.gc, ng - g0);
        // Mf: full structure factors of the chunk (formed here when needed);
        // Mc: what the Coulomb contraction reads
        double *Mf = w.M, *Mc = w.M;
        bool form = true;
        if (cache.on && !mixed) {
            Mf = Mc = cache.M + 2 * (size_t)g0 * n2;
            form = !cache.m_valid;
        } else if (packed) {
            Mc = cache.M + 2 * (size_t)g0 * npk;
            form = !cache.m_valid || (K && !cache.s_valid);  // the exchange slices are cut from the full form
        }
        if (form) {
            ev = tm.start(2);
            int nsf = 0;
            const long long ne = (long long)P->pvals.size() * gcur;
            k_gauss_table<<<(unsigned)((ne + 255) / 256), 256, 0, st>>>((int)P->pvals.size(), P->d_pvals, P->d_gvec, g0, gcur, w.gtab,
                                                                         sfac_df ? w.gtab2 : nullptr);
            for (int c = 0; c < JK_NCLASS_MAX; ++c) {
                if (sfac_df)
                    launch_sfac_df(c, pl, P->spair_class_off[c], P->spair_class_off[c + 1], g0, gcur, w.gtab2, Mf, st);
                else
                    launch_sfac(c, pl, P->spair_class_off[c], P->spair_class_off[c + 1], P->d_gvec, g0, gcur, w.gtab, Mf, st);
                nsf += P->spair_class_off[c + 1] > P->spair_class_off[c];
            }
            if (packed && !cache.m_valid) {
                k_pack_upper<<<152 * 16, 256, 0, st>>>(n, npk, 2 * gcur, Mf, Mc);
                ++nsf;
            }
            if ((rc = cuda_check("structure factors"))) return rc;
            tm.stop(2, ev, nsf + 1);
        }
        const int m2 = 2 * gcur;
        if (J) {
            // rho_D = M^T vec(D'), J_LR += M rho_D (two passes over the slab)
            ev = tm.start(3);
            if (packed) {
                slab_gemv_t(Mc, npk, m2, w.T1, w.rho_part, w.rho, st);
                slab_gemv_n(Mc, npk, m2, w.rho, 1.0, w.T2, st);
            } else {
                slab_sym_t(Mc, n, m2, w.Dp, w.T1, w.rho_part, w.rho, g0 == 0, st);
                slab_sym_n(Mc, n, m2, w.rho, w.JLR, st);
            }
            tm.stop(3, ev, 3);
        }
        if (K) {
            ev = tm.start(4);
            if (mixed) {
                // split-precision BF16 tensor-core GEMMs, slices per chunk from its G bound
                if ((rc = ozaki_exchange_chunk(P, chunk, Mf, m2, w.chunk_slices[chunk], st))) return rc;
                tm.stop(4, ev, 4);
            } else {
                // the plain FP64 form: Z_b = D' M_b, then K_LR += sum_b M_b Z_b
                // (upper tiles; the product is symmetric), FP64 GEMMs
                dgemm_batched(n, n, n, w.Dp, n, 0, Mf, n, (long long)n2, w.Z, n, (long long)n2, m2, 1.0, 0.0, false, st);
                dgemm_batched(n, n, n, Mf, n, (long long)n2, w.Z, n, (long long)n2, w.KLR, n, 0, m2, 1.0, 0.0, true, st);
                tm.stop(4, ev, 2);
            }
        }
    }
    // filled in stream order: later builds on this plan are ordered after this one
    if (J && packed) k_unpack_sym<<<grid_for(n2), 256, 0, st>>>(n, w.T2, w.JLR);
    if (cache.on) {
        cache.m_valid = true;
        if (mixed && K) cache.s_valid = true;
    }
    if (mixed && K) {
        ev = tm.start(4);
        if ((rc = ozaki_finish(P, st))) return rc;
        tm.stop(4, ev, 1);
    } else if (K && ng > 0) {
        mirror_upper(n, w.KLR, st);
    }
    return cuda_check("reciprocal phase");
}

// The caller holds P->build_mu (jk_build), so the stream ordering against
// the previous build on this plan and the use of its workspace are one
// critical section.
int run_build(Plan *P, const double *D, double *J, double *K, cudaStream_t st)
{
    if (cudaSetDevice(P->device) != cudaSuccess) return fail_cuda(JK_ERR_CUDA, "cudaSetDevice failed");
    const int n = P->nbf;
    const size_t n2 = (size_t)n * n;
    PlanDev pl = P->dev();
    Workspace &w = P->ws;
    const bool mixed = P->precision == JK_MIXED;
    PhaseTimer &tm = P->timer;
    tm.begin(st);
    const int ev_all = tm.start(6);
    int ev = tm.start(0);

    k_scale<<<grid_for(n2), 256, 0, st>>>(n, P->d_compf, D, w.Dp);
    if (mixed) {
        const long long ns2 = (long long)P->nshell * P->nshell;
        cudaMemsetAsync(w.dmaxf + ns2, 0, sizeof(float), st);
        k_dmax<<<(unsigned)((ns2 + 255) / 256), 256, 0, st>>>(pl, w.Dp, w.dmax, w.dmaxf);
        k_to_float<<<grid_for(n2), 256, 0, st>>>(n2, w.Dp, w.Dpf);
    }
    cudaMemsetAsync(w.X, 0, n2 * sizeof(double), st);
    cudaMemsetAsync(w.Y, 0, n2 * sizeof(double), st);
    cudaMemsetAsync(w.JLR, 0, n2 * sizeof(double), st);
    cudaMemsetAsync(w.KLR, 0, n2 * sizeof(double), st);
    cudaMemsetAsync(w.scal, 0, 16 * sizeof(double), st);
    cudaMemsetAsync(w.cnt, 0, kCounters * sizeof(unsigned long long), st);
    if (w.nbig) cudaMemsetAsync(w.nbig, 0, 2 * sizeof(unsigned) * w.nlist, st);
    int rc;
    if ((rc = cuda_check("prologue"))) return rc;
    // mixed precision: slices of D' and its low-rank factorisation for the
    // exchange contraction (decided on the device; nothing waits for it)
    if (mixed && K && (rc = ozaki_begin(P, st))) return rc;
    tm.stop(0, ev, mixed ? (K ? 7 : 3) : 1);

    // Coulomb-only build: the J-engine (Hermite densities in, Hermite J out)
    // (only the classes with a d shell, l_I = 2, take part: kJengClass)
    constexpr int kJengClass = 3;
    bool have_d = false;
    for (int c = kJengClass; c < JK_NCLASS_MAX; ++c) have_d = have_d || P->classes[c].b1 > P->classes[c].b0;
    const bool jeng = J && !K && have_d;
    if (jeng) {
        const int eh = tm.start(0);
        cudaMemsetAsync(w.JH, 0, std::max<size_t>(1, P->ppi.size()) * w.hs * sizeof(double), st);
        for (int c = kJengClass; c < JK_NCLASS_MAX; ++c)
            launch_hermite(c, false, pl, P->classes[c].b0, P->classes[c].b1, w, w.Dp, mixed, nullptr, st);
        tm.stop(0, eh, JK_NCLASS_MAX - kJengClass + 1);
    }

    // ---- real space.  Large cells: one class pair after another on the
    // caller's stream (the tile kernels fill every SM; on streams of their own
    // they gained nothing on the water box).  Small plans deal the class pairs
    // out over the caller's stream and three more, forked and joined by events
    // (they only meet in the atomics on X, Y and the counters), with the
    // reciprocal phase, which shares nothing with them, on a fifth.
    ev = tm.start(1);
    int nreal = 0;
    if (P->nside > 0) {
        cudaEventRecord(P->side_fork, st);
        for (int i = 0; i < P->nside; ++i) cudaStreamWaitEvent(P->side[i], P->side_fork, 0);
    }
    const auto join = [&](int i0, int i1) {
        tm.use(st);
        for (int i = i0; i < i1; ++i) {
            cudaEventRecord(P->side_join[i], P->side[i]);
            cudaStreamWaitEvent(st, P->side_join[i], 0);
        }
    };
    if (P->nside > 0) {
        tm.use(P->side[P->nside - 1]);
        if ((rc = reciprocal_phase(P, J, K, P->side[P->nside - 1]))) {
            join(0, P->nside);
            return rc;
        }
        tm.use(st);
    }
    int turn = 0;
    for (int cb = 0; cb < JK_NCLASS_MAX; ++cb)
        for (int ck = cb; ck < JK_NCLASS_MAX; ++ck) {
            const ClassRange &B = P->classes[cb], &Kc = P->classes[ck];
            if (B.b1 <= B.b0 || Kc.b1 <= Kc.b0) continue;
            RealLaunch a{};
            a.pl = pl;
            a.b0 = B.b0;
            a.b1 = B.b1;
            a.k0 = Kc.b0;
            a.k1 = Kc.b1;
            a.same = cb == ck;
            a.kchunk = P->kchunk[cb][ck];
            a.map = tile_map(P, B, a.b0, a.b1, a.k0, a.k1, a.kchunk);
            a.variant = P->kvariant[cb][ck];
            a.tau = P->mixed_tau;
            a.Dp = w.Dp;
            a.dmax = w.dmax;
            a.Dpf = w.Dpf;
            a.dmaxf = w.dmaxf;
            a.X = w.X;
            a.Y = K ? w.Y : nullptr;
            // the next lane whose list holds the class pair (FP64 plans have no lists)
            const int nlane = mixed ? w.nlist : std::max(1, P->nside);
            int lane = turn++ % nlane;
            if (mixed)
                while (lane > 0 && w.list_cap[lane] < std::min<long long>(w.list_cap[0], P->class_quartets(cb, ck))) lane = (lane + 1) % nlane;
            cudaStream_t ls = lane ? P->side[lane - 1] : st;
            tm.use(ls);
            const QuartetList big{w.big ? (char *)w.big + w.list_off[lane] : nullptr, w.list_elt == 4};
            unsigned *nbig = w.nbig ? w.nbig + 2 * lane : nullptr;
            a.st = ls;
            a.DhD = w.DhD;
            a.DhF = w.DhF;
            a.JH = w.JH;
            a.hs = w.hs;
            // Coulomb-only builds take the J-engine for class pairs with a d
            // shell on both sides, where the Hermite contraction is smaller
            // than the Cartesian block (measured: for s and p classes the
            // Cartesian kernels with the exchange digestion skipped are
            // faster); its tiles are lane-per-bra, 32 kets each
            const bool use_jeng = jeng && cb >= kJengClass && ck >= kJengClass;
            if (use_jeng) a.kchunk = 32;
            if (use_jeng && !mixed) {
                a.mode = 0;
                a.fp32 = false;
                a.cnt = w.cnt;
                const int et = tm.start(10);
                launch_jeng(cb, ck, a);
                tm.stop(10, et, 1);
                nreal += 1;
            } else if (use_jeng) {
                cudaMemsetAsync(nbig, 0, sizeof(unsigned), ls);
                a.mode = 2;
                a.fp32 = true;
                a.cnt = w.cnt + 1;
                a.big = big;
                a.nbig = nbig;
                a.ovf = nbig + 1;
                a.cap = w.list_cap[lane];
                const int et = tm.start(10);
                launch_jeng(cb, ck, a);
                tm.stop(10, et, 1);
                // the listed large quartets: the Cartesian FP64 pass, Coulomb only
                a.list_pass = true;
                a.cnt64 = w.cnt;
                const int el = tm.start(9);
                launch_real(cb, ck, a);
                tm.stop(9, el, 1);
                nreal += 2;
            } else if (!mixed) {
                a.mode = 0;
                a.fp32 = false;
                a.cnt = w.cnt;
                const int et = tm.start(10);
                launch_real(cb, ck, a);
                tm.stop(10, et, 1);
                nreal += 1;
            } else {
                // FP32 pass over every quartet, collecting the large ones ...
                cudaMemsetAsync(nbig, 0, sizeof(unsigned), ls);
                a.mode = 2;
                a.fp32 = true;
                a.cnt = w.cnt + 1;
                a.big = big;
                a.nbig = nbig;
                a.ovf = nbig + 1;
                a.cap = w.list_cap[lane];
                const int et = tm.start(10);
                launch_real(cb, ck, a);
                tm.stop(10, et, 1);
                // ... then FP64 over the compact list
                a.list_pass = true;
                a.cnt64 = w.cnt;
                const int el = tm.start(9);
                launch_real(cb, ck, a);
                tm.stop(9, el, 1);
                nreal += 2;
            }
            if ((rc = cuda_check("real-space kernel"))) {
                join(0, P->nside);
                return rc;
            }
        }
    join(0, P->nside - 1);
    if (jeng) {
        // Hermite J of every primitive pair back to Cartesian, into X
        for (int c = kJengClass; c < JK_NCLASS_MAX; ++c)
            launch_hermite(c, true, pl, P->classes[c].b0, P->classes[c].b1, w, nullptr, false, w.X, st);
        nreal += JK_NCLASS_MAX - kJengClass;
    }
    tm.stop(1, ev, nreal);

    // ---- reciprocal space
    if (P->nside > 0) join(P->nside - 1, P->nside);
    else if ((rc = reciprocal_phase(P, J, K, st))) return rc;

    ev = tm.start(5);

    // ---- removed K = 0 term: c = -pi / (V w^2)
    const double cbg = -kPi / (P->volume * P->omega * P->omega);
    k_dot2<<<grid_for(n2), 256, 0, st>>>(n2, P->d_S, w.Dp, nullptr, w.scal);
    if (K) {
        // S D' S (both factors symmetric; FP64 GEMMs)
        dgemm_batched(n, n, n, w.Dp, n, 0, P->d_S, n, 0, w.T1, n, (long long)n2, 1, 1.0, 0.0, false, st);
        dgemm_batched(n, n, n, P->d_S, n, 0, w.T1, n, 0, w.T2, n, (long long)n2, 1, 1.0, 0.0, false, st);
    }
    k_final<<<grid_for(n2), 256, 0, st>>>(n, P->d_compf, w.X, w.Y, w.JLR, w.KLR, P->d_S, w.T2, w.scal, cbg, w.err, J, K);
    tm.stop(5, ev, K ? 4 : 2);
    tm.stop(6, ev_all, 0);
    return cuda_check("epilogue");
}

// Autotuner: for every class pair with work, time the real-space tile kernel of
// the plan's precision with each candidate over two sub-ranges of at most 2048
// bras against all kets, and the two fastest, with the plan's untuned schedule,
// over the whole class where that takes less than about a second.  A candidate
// replaces the untuned schedule only if it is faster by 2%: the sub-ranges alone
// preferred few kets per warp, and the 64-water tiles so tuned took 389 ms
// against 354 untuned.  Results are cached in a text file (one line per GPU
// name, precision, class pair and size bucket: family * 65536 + kets, or 0
// where the untuned schedule stays) when cache_path is given.
int autotune(Plan *P, const double *D, cudaStream_t st, const char *cache_path, int *chosen)
{
    if (cudaSetDevice(P->device) != cudaSuccess) return fail_cuda(JK_ERR_CUDA, "cudaSetDevice failed");
    cudaDeviceProp prop;
    cudaGetDeviceProperties(&prop, P->device);
    const bool mixed = P->precision == JK_MIXED;
    const int n = P->nbf;
    const size_t n2 = (size_t)n * n;
    Workspace &w = P->ws;
    PlanDev pl = P->dev();
    k_scale<<<grid_for(n2), 256, 0, st>>>(n, P->d_compf, D, w.Dp);
    if (mixed) k_to_float<<<grid_for(n2), 256, 0, st>>>(n2, w.Dp, w.Dpf);
    // existing cache entries
    std::map<std::string, int> cache;
    if (cache_path) {
        FILE *f = fopen(cache_path, "r");
        if (f) {
            char key[512];
            int v;
            while (fscanf(f, "%511s %d", key, &v) == 2) cache[key] = v;
            fclose(f);
        }
    }
    auto bucket = [](int x) { int b = 0; while ((1 << b) < x) ++b; return b; };
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    // device time of choice c over the bras [b0, b1) of a class pair, the
    // shortest of reps launches; negative if a launch failed
    const auto timed = [&](int cb, int ck, int b0, int b1, int c, int reps) -> float {
        const ClassRange &B = P->classes[cb], &Kc = P->classes[ck];
        float best = 1e30f;
        for (int r = 0; r < reps; ++r) {
            RealLaunch a{};
            a.pl = pl;
            a.b0 = b0;
            a.b1 = b1;
            a.k0 = Kc.b0;
            a.k1 = Kc.b1;
            a.same = cb == ck;
            a.kchunk = c & 65535;
            a.map = tile_map(P, B, a.b0, a.b1, a.k0, a.k1, a.kchunk);
            a.variant = c >> 16;
            a.mode = 0;
            a.fp32 = mixed;
            a.Dp = w.Dp;
            a.dmax = w.dmax;
            a.Dpf = w.Dpf;
            a.dmaxf = w.dmaxf;
            a.X = w.X;
            a.Y = w.Y;
            a.cnt = w.cnt;
            a.st = st;
            cudaEventRecord(e0, st);
            launch_real(cb, ck, a);
            cudaEventRecord(e1, st);
            float ms = 0;
            if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) return -1.0f;
            best = std::min(best, ms);
            if (ms > (b1 - b0 < B.b1 - B.b0 ? 2.0f : 20.0f)) break;  // long enough not to need another
        }
        return best;
    };
    // candidates: for s and p class pairs the lane-per-bra kernels with 8 .. 128
    // kets per tile, the warp kernels with 8 .. 2048 kets per warp (1 .. 256
    // where a warp takes one image quartet) and the pair-queue kernels with 32
    // .. 512 kets per tile; for class pairs with a d shell their one kernel with
    // 1 .. 2048 kets per warp
    constexpr float kMargin = 0.98f;
    int k = 0;
    bool dirty = false;
    for (int cb = 0; cb < JK_NCLASS_MAX; ++cb)
        for (int ck = cb; ck < JK_NCLASS_MAX; ++ck, ++k) {
            const ClassRange &B = P->classes[cb], &Kc = P->classes[ck];
            if (chosen) {
                chosen[2 * k] = P->kvariant[cb][ck];
                chosen[2 * k + 1] = P->kchunk[cb][ck];
            }
            if (B.b1 <= B.b0 || Kc.b1 <= Kc.b0) continue;
            char key[512];
            snprintf(key, sizeof key, "%s|%s|v5|%d%d|%d|%d", prop.name, mixed ? "mixed" : "fp64", cb, ck, bucket(B.b1 - B.b0),
                     bucket(Kc.b1 - Kc.b0));
            for (char *q = key; *q; ++q)
                if (*q == ' ') *q = '_';
            int family, kets;
            P->default_schedule(cb, ck, family, kets);
            const int own = family << 16 | kets;
            int best = 0;
            auto it = cache.find(key);
            if (it != cache.end()) {
                best = it->second;
            } else {
                std::vector<int> cands;
                if (real_has_warp_kernel(cb, ck)) {
                    for (int c : {8, 16, 32, 64, 128}) cands.push_back(c);
                    if (P->warp_per_quartet(cb, ck))
                        for (int c : {1, 4, 16, 64, 256}) cands.push_back(65536 + c);
                    else
                        for (int c : {8, 32, 128, 256, 512, 1024, 2048}) cands.push_back(65536 + c);
                    for (int c : {32, 64, 128, 256, 512}) cands.push_back(2 * 65536 + c);
                } else {
                    for (int c : {1, 4, 16, 64, 128, 512, 2048}) cands.push_back(c);
                }
                cands.erase(std::remove(cands.begin(), cands.end(), own), cands.end());
                // the class is sorted by primitive count, so the start and the middle differ
                const int nbc = B.b1 - B.b0, m0 = std::max(B.b0 + std::min(nbc, 2048), B.b0 + nbc / 2), m1 = std::min(B.b1, m0 + 2048);
                const auto sample = [&](int c) -> float {
                    const float t0 = timed(cb, ck, B.b0, std::min(B.b1, B.b0 + 2048), c, 3);
                    const float t1 = m1 > m0 ? timed(cb, ck, m0, m1, c, 3) : 0.0f;
                    return t0 < 0 || t1 < 0 ? -1.0f : t0 + t1;
                };
                float t_own = sample(own);
                bool failed = t_own < 0;
                std::vector<std::pair<float, int>> t;
                for (int c : cands) {
                    t.push_back({sample(c), c});
                    failed = failed || t.back().first < 0;
                }
                std::sort(t.begin(), t.end());
                if (nbc > 2048) {
                    const auto prims = [&](int i0, int i1) { return i1 > i0 ? P->spi[i1 - 1].pp0 + P->spi[i1 - 1].npp - P->spi[i0].pp0 : 0; };
                    const double part = (double)prims(B.b0, B.b0 + 2048) + prims(m0, m1);
                    if (t_own * prims(B.b0, B.b1) / part < 1000.0) {
                        t_own = timed(cb, ck, B.b0, B.b1, own, 2);
                        failed = failed || t_own < 0;
                        t.resize(std::min<size_t>(t.size(), 2));
                        for (auto &x : t) {
                            x.first = timed(cb, ck, B.b0, B.b1, x.second, 2);
                            failed = failed || x.first < 0;
                        }
                        std::sort(t.begin(), t.end());
                    }
                }
                if (failed) {
                    cudaEventDestroy(e0);
                    cudaEventDestroy(e1);
                    return fail_cuda(JK_ERR_CUDA, "autotune launch failed");
                }
                if (!t.empty() && t[0].first < kMargin * t_own) best = t[0].second;
                cache[key] = best;
                dirty = true;
            }
            if (best >> 16 > 2 || (best >> 16 > 0 && !real_has_warp_kernel(cb, ck)) || best <= 0 || (best & 65535) == 0) best = own;
            P->kchunk[cb][ck] = best & 65535;
            P->kvariant[cb][ck] = best >> 16;
            if (chosen) {
                chosen[2 * k] = best >> 16;
                chosen[2 * k + 1] = best & 65535;
            }
        }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (cache_path && dirty) {
        FILE *f = fopen(cache_path, "w");
        if (f) {
            for (auto &kv : cache) fprintf(f, "%s %d\n", kv.first.c_str(), kv.second);
            fclose(f);
        }
    }
    P->tuned = true;
    return cuda_check("autotune");
}

// Real-space schedule given by the caller: (family, kets per tile) per
// class pair in the order of jk_autotune's output.
int set_schedule(Plan *P, const int *sched, int n)
{
    int k = 0;
    for (int cb = 0; cb < JK_NCLASS_MAX; ++cb)
        for (int ck = cb; ck < JK_NCLASS_MAX; ++ck, ++k) {
            if (k >= n) return JK_OK;
            const int fam = sched[2 * k], kets = sched[2 * k + 1];
            if (fam < 0 || fam > 2 || (fam >= 1 && !real_has_warp_kernel(cb, ck)) || kets < 1 || kets > 65535)
                return fail(JK_ERR_INVALID, "schedule entry " + std::to_string(k) + " out of range");
        }
    k = 0;
    for (int cb = 0; cb < JK_NCLASS_MAX; ++cb)
        for (int ck = cb; ck < JK_NCLASS_MAX && k < n; ++ck, ++k) {
            P->kvariant[cb][ck] = sched[2 * k];
            P->kchunk[cb][ck] = sched[2 * k + 1];
        }
    return JK_OK;
}

int build_counts(Plan *P, long long *counts, int n)
{
    unsigned long long h[kCounters] = {};
    unsigned hb[2 * Workspace::kLists] = {};
    if (P->timer.next > 0 && cudaEventSynchronize(P->timer.pool[P->timer.next - 1]) != cudaSuccess)
        return fail_cuda(JK_ERR_CUDA, "build did not finish");
    if (cudaMemcpy(h, P->ws.cnt, sizeof h, cudaMemcpyDeviceToHost) != cudaSuccess) return fail_cuda(JK_ERR_CUDA, "count copy failed");
    if (P->ws.nbig && cudaMemcpy(hb, P->ws.nbig, 2 * sizeof(unsigned) * P->ws.nlist, cudaMemcpyDeviceToHost) != cudaSuccess)
        return fail_cuda(JK_ERR_CUDA, "count copy failed");
    for (int i = 1; i < P->ws.nlist; ++i) hb[1] += hb[2 * i + 1];
    // rank and form of the density factorisation (mixed builds with K)
    int dyn[4] = {0, 0, 0, 0};
    if (P->precision == JK_MIXED && P->ws.lr.dyn && cudaMemcpy(dyn, P->ws.lr.dyn, sizeof dyn, cudaMemcpyDeviceToHost) != cudaSuccess)
        return fail_cuda(JK_ERR_CUDA, "status copy failed");
    // public layout (jk_build_counts)
    const long long out[13] = {(long long)h[0], (long long)h[1], (long long)hb[1], dyn[3], (long long)h[4], (long long)h[5], dyn[0],
                               (long long)h[8], (long long)h[9], (long long)h[12], (long long)h[14], (long long)h[13], (long long)h[15]};
    for (int i = 0; i < n && i < 13; ++i) counts[i] = out[i];
    unsigned e = 0;
    if (cudaMemcpy(&e, P->ws.err, sizeof e, cudaMemcpyDeviceToHost) != cudaSuccess) return fail_cuda(JK_ERR_CUDA, "check word copy failed");
    if (e) return fail(JK_ERR_TIMEOUT, "a bounded wait in a tensor-core GEMM ran out; J and K of that build are NaN");
    return JK_OK;
}

int build_times(Plan *P, double *ms, int *launches, int n)
{
    PhaseTimer &tm = P->timer;
    for (int i = 0; i < n; ++i) {
        if (ms) ms[i] = 0;
        if (launches) launches[i] = 0;
    }
    if (tm.marks.empty()) return JK_OK;
    if (cudaEventSynchronize(tm.pool[tm.next - 1]) != cudaSuccess) return fail_cuda(JK_ERR_CUDA, "build did not finish");
    // a phase's intervals add up, unless they lie on several streams: then the
    // time during which at least one of them ran (from the build's first event)
    std::vector<std::pair<float, float>> iv[PhaseTimer::kPhases];
    for (auto &m : tm.marks) {
        float t0 = 0, t = 0;
        cudaEventElapsedTime(&t, tm.pool[m.second.first], tm.pool[m.second.second]);
        if (P->nside > 0) cudaEventElapsedTime(&t0, tm.pool[0], tm.pool[m.second.first]);
        if (P->nside > 0) iv[m.first].push_back({t0, t0 + t});
        else if (m.first < n && ms) ms[m.first] += t;
    }
    for (int p = 0; p < PhaseTimer::kPhases && p < n && ms; ++p) {
        std::sort(iv[p].begin(), iv[p].end());
        float end = -1.0f;
        for (auto &x : iv[p]) {
            ms[p] += std::max(0.0f, x.second - std::max(x.first, end));
            end = std::max(end, x.second);
        }
    }
    for (int i = 0; i < n && i < PhaseTimer::kPhases; ++i)
        if (launches) launches[i] = tm.launches[i];
    int tot = 0;
    for (int i = 0; i < 6; ++i) tot += tm.launches[i];
    if (launches && n > 6) launches[6] = tot;
    if (ms && n > 11) {
        // slot 11: BF16 MMA flops issued (for the tensor roofline), from the
        // form and rank the device chose
        int dyn[3] = {0, 0, 0};
        if (P->precision == JK_MIXED && P->ws.lr.dyn &&
            cudaMemcpy(dyn, P->ws.lr.dyn, sizeof dyn, cudaMemcpyDeviceToHost) != cudaSuccess)
            return fail_cuda(JK_ERR_CUDA, "status copy failed");
        ms[11] = P->precision == JK_MIXED ? ozaki_mma_flops(P, dyn) : 0.0;
    }
    return JK_OK;
}

}  // namespace jk
