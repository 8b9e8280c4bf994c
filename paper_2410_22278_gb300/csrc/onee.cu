// One-electron operators of the cell on the device: the kinetic-energy
// matrix and the nuclear attraction of point charges with their periodic
// images, Ewald-split at the plan's omega (Sections 2.1 and 2.2 of the
// paper; the kinetic formula is in its Supporting Information).  Both are
// sums over the plan's unique shell-pair images of local integrals between
// mu at A and nu at B + R, like the overlap.
//
// Nuclear attraction, per charge Z_C at C (Eq. pbc_v1e_base_case_final):
//   real part    -Z (2 pi/p) K sum_t E^{ab}_t R_t(P - C - R_C) over the images
//                R_C inside the screening sphere, seeds (-2p)^m G_m(p X^2, c),
//                c = w / sqrt(p + w^2) (the attenuated Boys difference of Eq.
//                boys_function_split written as one integral);
//   reciprocal   -(4 pi / V) sum_{G != 0} e^{-G^2/4w^2}/G^2 Re[conj(rho_ab(G))
//                rho_N(G)], rho_N(G) = sum_C Z_C e^{-iG.C}: the same
//                sum as in the Coulomb build, taken pair by pair against the
//                nuclear structure factor (k_onee_recip);
//   self term    +(pi / (V w^2)) Z_tot S_ab (Eq. v1e_self_term).
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <vector>

#include "kernels.cuh"
#include "launch.h"
#include "plan.h"

namespace jk {
namespace {

// 1-D overlaps s[i][j] = sqrt(pi/p) E^{ij}_0, i <= LA, j <= LB + 2 (the
// Gaussian factor is in K), and the kinetic block of one primitive pair:
//   t(i, j) = -1/2 [ j(j-1) s(i,j-2) - 2b(2j+1) s(i,j) + 4b^2 s(i,j+2) ],
//   T = tx sy sz + sx ty sz + sx sy tz.
template <int LA, int LB>
__device__ __forceinline__ void kinetic_block(const PpiRec &x, double b, double *blk)
{
    constexpr int NA = ncart(LA), NB = ncart(LB), LB2 = LB + 2, NT = LA + LB2 + 1;
    double s[3][LA + 1][LB2 + 1], t[3][LA + 1][LB + 1];
    const double rp = sqrt(kPi / x.p);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        double E[(LA + 1) * (LB2 + 1) * NT];
        herm_E<LA, LB2, double>(x.PA[k], x.PB[k], 0.5 / x.p, E);
#pragma unroll
        for (int i = 0; i <= LA; ++i)
#pragma unroll
            for (int j = 0; j <= LB2; ++j) s[k][i][j] = rp * E[(i * (LB2 + 1) + j) * NT];
#pragma unroll
        for (int i = 0; i <= LA; ++i)
#pragma unroll
            for (int j = 0; j <= LB; ++j) {
                double v = -2.0 * b * (2 * j + 1) * s[k][i][j] + 4.0 * b * b * s[k][i][j + 2];
                if (j >= 2) v += j * (j - 1) * s[k][i][j - 2];
                t[k][i][j] = -0.5 * v;
            }
    }
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
        for (int c = 0; c < NB; ++c) {
            const int ax = cexp(LA, a, 0), ay = cexp(LA, a, 1), az = cexp(LA, a, 2);
            const int bx = cexp(LB, c, 0), by = cexp(LB, c, 1), bz = cexp(LB, c, 2);
            blk[a * NB + c] += x.K * (t[0][ax][bx] * s[1][ay][by] * s[2][az][bz] + s[0][ax][bx] * t[1][ay][by] * s[2][az][bz] +
                                      s[0][ax][bx] * s[1][ay][by] * t[2][az][bz]);
        }
}

// Where the images of a class start, where their blocks do, its first shell
// pair and its first element among all (first[JK_NCLASS_MAX]: their number).
struct ImageBlocks {
    int b0[JK_NCLASS_MAX], sp0[JK_NCLASS_MAX];
    size_t off[JK_NCLASS_MAX];
    long long first[JK_NCLASS_MAX + 1];
};

// Every kernel below leaves the block of a shell-pair image of its own (blk:
// those of one class, NA x NB elements an image); this sums the images of each
// shell pair into the raw matrix, gsz lanes an element and in a fixed order, so
// a repeated call gives the same bits (images added by atomics did not).  For
// I = J an image with R != 0 stands for its mirror too.  Bound by latency: all
// classes in one launch, eight chains an element, or 32 in small cells, whose
// shell pairs have ten and more images (launched class by class with one chain
// an element, a call on the 8-function cell took 0.90 ms instead of 0.87, on one
// water molecule 4.26 instead of 4.07; those are the times with atomics).
__global__ void __launch_bounds__(128) k_onee_gather(PlanDev pl, ImageBlocks ib, int gsz, const double *__restrict__ blk, double *__restrict__ Out)
{
    const long long x = (blockIdx.x * 128LL + threadIdx.x) / gsz;
    const int part = threadIdx.x & (gsz - 1);
    const bool on = x < ib.first[JK_NCLASS_MAX];
    int c = 0;
    while (c + 1 < JK_NCLASS_MAX && x >= ib.first[c + 1]) ++c;
    const int la = c == 0 ? 0 : c <= 2 ? 1 : 2, lb = c - la * (la + 1) / 2, NB = ncart(lb), NAB = ncart(la) * NB;
    double sum = 0.0;
    SpairRec rec{};
    int e = 0;
    if (on) {
        rec = pl.spair[ib.sp0[c] + (int)((x - ib.first[c]) / NAB)];
        e = (int)((x - ib.first[c]) % NAB);
        for (int q = part; q < rec.nspi; q += gsz) {
            const int img = pl.spi_order[rec.spi0 + q];
            const double *v = blk + ib.off[c] + (size_t)(img - ib.b0[c]) * NAB;
            sum += v[e];
            if (rec.I == rec.J) {
                const SpiRec &si = pl.spi[img];
                if (si.n[0] || si.n[1] || si.n[2]) sum += v[(e % NB) * NB + e / NB];
            }
        }
    }
    __syncwarp();
    for (int o = gsz >> 1; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (!on || part != 0) return;
    const size_t n = pl.nbf, r = pl.shells[rec.I].ao + e / NB, k = pl.shells[rec.J].ao + e % NB;
    Out[r * n + k] = sum;
    if (rec.I != rec.J) Out[k * n + r] = sum;
}

// Kinetic energy: one warp per shell-pair image, one primitive pair per lane.
template <int LA, int LB>
__global__ void __launch_bounds__(128) k_onee_kinetic(PlanDev pl, int b0, int b1, const double2 *__restrict__ ab, double *__restrict__ out)
{
    constexpr int NA = ncart(LA), NB = ncart(LB);
    const int img = b0 + blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (img >= b1) return;
    const SpiRec si = pl.spi[img];
    double blk[NA * NB];
#pragma unroll
    for (int k = 0; k < NA * NB; ++k) blk[k] = 0.0;
    for (int q = lane; q < si.npp; q += 32) {
        const PpiRec x = pl.ppi[si.pp0 + q];
        kinetic_block<LA, LB>(x, ab[si.pp0 + q].y, blk);
    }
#pragma unroll
    for (int k = 0; k < NA * NB; ++k) {
        const double v = warp_sum(blk[k]);
        if (lane == (k & 31)) out[(size_t)(img - b0) * (NA * NB) + k] = v;
    }
}

// Real part of the attraction: one warp per shell-pair image.  A group of
// gsz lanes (32, or 8 for few charges) takes one primitive pair and shares
// its charges: the radius and the image search in single precision (they
// decide which terms are formed), the seeds and the R table in FP64, summed
// over charges and images in registers and over the group by shuffles; then
// the group's lanes form the Cartesian elements.  One thread per shell pair
// walked up to 36 primitive pairs x 81 charges x images alone (27-water box:
// 200 ms for 30 thousand threads of very different length).
template <int LA, int LB>
__global__ void __launch_bounds__(128) k_onee_real(PlanDev pl, int b0, int b1, int natom, const double *__restrict__ Zc,
                                                   const double *__restrict__ xyz, const double *__restrict__ cand, int ncand, int gsz,
                                                   double *__restrict__ out)
{
    constexpr int NA = ncart(LA), NB = ncart(LB), NAB = NA * NB, L = LA + LB, NT = L + 1, D = L + 1;
    constexpr int NK = (NAB + 7) / 8;
    const int img = b0 + blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (img >= b1) return;
    const SpiRec si = pl.spi[img];
    const int gl = lane & (gsz - 1), grp = lane / gsz, ngrp = 32 / gsz;
    const double w2 = pl.omega * pl.omega;
    double blk[NK];
#pragma unroll
    for (int k = 0; k < NK; ++k) blk[k] = 0.0;
    for (int q0 = 0; q0 < si.npp; q0 += ngrp) {
        const int q = q0 + grp;
        double Rs[D * D * D];
#pragma unroll
        for (int k = 0; k < D * D * D; ++k) Rs[k] = 0.0;
        PpiRec x{};
        if (q < si.npp) {
            x = pl.ppi[si.pp0 + q];
            const double wp = 1.0 / (x.p + w2), aw = x.p * w2 * wp, c = sqrt(w2 * wp);
            const float awf = (float)aw, pre = (float)(2.0 * kPi / x.p * fabs(x.K) * (1.0 - c));
            for (int C = gl; C < natom; C += gsz) {
                const double z = Zc[C];
                // screening radius of Eq. pbc_eri_real_cutoff_implementation for a
                // point charge: (2 pi/p) |K Z| (1 - c) e^{-aw r^2} above delta_R / 10
                const float lg = logf(pre * fabsf((float)z)) - pl.log_ewald_R;
                if (!(lg > 0.0f)) continue;
                float r = sqrtf(lg / awf);
                if (L > 0) {
                    r = sqrtf((lg + L * logf(1.0f + 2.0f * awf * r)) / awf);
                    r = sqrtf((lg + L * logf(1.0f + 2.0f * awf * r)) / awf) + 0.5f + 0.25f * L;
                }
                const float r2 = r * r;
                double X0[3] = {x.P[0] - xyz[3 * C], x.P[1] - xyz[3 * C + 1], x.P[2] - xyz[3 * C + 2]};
                double f[3];
#pragma unroll
                for (int a = 0; a < 3; ++a) f[a] = rint(pl.Finv[3 * a] * X0[0] + pl.Finv[3 * a + 1] * X0[1] + pl.Finv[3 * a + 2] * X0[2]);
#pragma unroll
                for (int a = 0; a < 3; ++a) X0[a] -= f[0] * pl.L[a] + f[1] * pl.L[3 + a] + f[2] * pl.L[6 + a];
                const float F0[3] = {(float)X0[0], (float)X0[1], (float)X0[2]};
                const float x0n = sqrtf(F0[0] * F0[0] + F0[1] * F0[1] + F0[2] * F0[2]);
                for (int k = 0; k < ncand; ++k) {
                    const float cx = (float)cand[4 * k], cy = (float)cand[4 * k + 1], cz = (float)cand[4 * k + 2];
                    if ((float)cand[4 * k + 3] - x0n >= r) break;
                    const float fx = F0[0] - cx, fy = F0[1] - cy, fz = F0[2] - cz;
                    if (fx * fx + fy * fy + fz * fz >= r2) continue;
                    const double Xx = X0[0] - cand[4 * k], Xy = X0[1] - cand[4 * k + 1], Xz = X0[2] - cand[4 * k + 2];
                    const double x2 = Xx * Xx + Xy * Xy + Xz * Xz;
                    double G[L + 1], s[L + 1];
                    boys_attenuated_tab<L>(x.p * x2, aw * x2, c, pl.boys_t, G);
                    double fm = -z;  // (-2p)^m times the charge of the attraction
#pragma unroll
                    for (int m = 0; m <= L; ++m) {
                        s[m] = fm * G[m];
                        fm *= -2.0 * x.p;
                    }
                    double B[D * D * D];
                    herm_R<L, double>(s, Xx, Xy, Xz, B);
#pragma unroll
                    for (int t = 0; t <= L; ++t)
#pragma unroll
                        for (int u = 0; u <= L - t; ++u)
#pragma unroll
                            for (int v = 0; v <= L - t - u; ++v) Rs[(t * D + u) * D + v] += B[(t * D + u) * D + v];
                }
            }
        }
        __syncwarp();
#pragma unroll
        for (int t = 0; t <= L; ++t)
#pragma unroll
            for (int u = 0; u <= L - t; ++u)
#pragma unroll
                for (int v = 0; v <= L - t - u; ++v) {
                    double y = Rs[(t * D + u) * D + v];
                    for (int o = gsz >> 1; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
                    Rs[(t * D + u) * D + v] = y;
                }
        if (q < si.npp) {
            double E[3][(LA + 1) * (LB + 1) * NT];
#pragma unroll
            for (int k = 0; k < 3; ++k) herm_E<LA, LB, double>(x.PA[k], x.PB[k], 0.5 / x.p, E[k]);
            const double pref = 2.0 * kPi / x.p * x.K;
#pragma unroll
            for (int a = 0; a < NA; ++a)
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    const int o = a * NB + b;
                    if ((o & 7) != (gl & 7) || (gsz == 32 && gl >= 8)) continue;
                    const int ax = cexp(LA, a, 0), ay = cexp(LA, a, 1), az = cexp(LA, a, 2);
                    const int bx = cexp(LB, b, 0), by = cexp(LB, b, 1), bz = cexp(LB, b, 2);
                    double v = 0.0;
#pragma unroll
                    for (int tx = 0; tx <= ax + bx; ++tx)
#pragma unroll
                        for (int ty = 0; ty <= ay + by; ++ty)
#pragma unroll
                            for (int tz = 0; tz <= az + bz; ++tz)
                                v += E[0][(ax * (LB + 1) + bx) * NT + tx] * E[1][(ay * (LB + 1) + by) * NT + ty] *
                                     E[2][(az * (LB + 1) + bz) * NT + tz] * Rs[(tx * D + ty) * D + tz];
                    blk[o >> 3] += pref * v;
                }
        }
    }
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        // lane l of each group of eight holds element 8 k + l
        double v = blk[k];
        v += __shfl_xor_sync(0xffffffffu, v, 8);
        v += __shfl_xor_sync(0xffffffffu, v, 16);
        const int o = 8 * k + lane;
        if (lane < 8 && o < NAB) out[(size_t)(img - b0) * NAB + o] = v;
    }
}

// Reciprocal part: one block per shell-pair image, the G of a chunk over its
// threads.  For each primitive pair the phases e^{i n 2 pi f_k} of the three
// fractional coordinates f_k of P stand in shared memory, so a G costs two
// complex products instead of a dot product and a sincos; the sum over G is
// taken for the Hermite moments (i G)^t, and the E coefficients enter once
// per primitive pair instead of once per G.  Bound by the FP64 pipe: about 13
// FP64 instructions per (primitive pair, G) for s-s.
//   v[g] = -8 pi w(G) / V rho_N(G) (the weights of both structure factors),
//   gtab[pidx * gcur + g] = (pi / p)^{3/2} e^{-G^2 / 4p}.
template <int LA, int LB>
__global__ void __launch_bounds__(128) k_onee_recip(PlanDev pl, int b0, int g0, int gcur, int nmax, const double2 *__restrict__ v,
                                                    const double *__restrict__ gtab, double *__restrict__ out)
{
    constexpr int NA = ncart(LA), NB = ncart(LB), NAB = NA * NB, L = LA + LB, NT = L + 1, D = L + 1, NH = nherm(L);
    extern __shared__ double2 ph[];  // [3][2 nmax + 1]
    __shared__ double red[4][NH], H[NH];
    const int img = b0 + blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const SpiRec si = pl.spi[img];
    const int nph = 2 * nmax + 1;
    double acc = 0.0;  // element threadIdx.x of the block
    for (int q = 0; q < si.npp; ++q) {
        const PpiRec x = pl.ppi[si.pp0 + q];
        __syncthreads();
        for (int e = threadIdx.x; e < 3 * nph; e += 128) {
            const int k = e / nph, nn = e - k * nph - nmax;
            const double f = pl.Finv[3 * k] * x.P[0] + pl.Finv[3 * k + 1] * x.P[1] + pl.Finv[3 * k + 2] * x.P[2];
            double sn, cs;
            sincospi(2.0 * nn * (f - rint(f)), &sn, &cs);
            ph[e] = make_double2(cs, sn);
        }
        __syncthreads();
        const double *gt = gtab + (size_t)pl.ppi_pidx[si.pp0 + q] * gcur;
        double m[NH];
#pragma unroll
        for (int h = 0; h < NH; ++h) m[h] = 0.0;
        for (int g = threadIdx.x; g < gcur; g += 128) {
            const float4 gn = __ldg(pl.gdf + 3 * (size_t)(g0 + g));
            const double2 ea = ph[nmax + (int)gn.x], eb = ph[nph + nmax + (int)gn.y], ec = ph[2 * nph + nmax + (int)gn.z];
            const double2 w = __ldg(v + g);
            const double gf = __ldg(gt + g);
            double zr = ea.x * eb.x - ea.y * eb.y, zi = ea.x * eb.y + ea.y * eb.x;
            const double yr = zr * ec.x - zi * ec.y, yi = zr * ec.y + zi * ec.x;
            zr = gf * (yr * w.x - yi * w.y);
            if constexpr (L == 0) {
                m[0] += zr;
            } else {
                zi = gf * (yr * w.y + yi * w.x);
                // Re[i^t z]: zr, -zi, -zr, zi, zr
                const double ph4[5] = {zr, -zi, -zr, zi, zr};
                double pw[3][L + 1];
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const double G = __ldg(pl.gvec + 4 * (size_t)(g0 + g) + k);
                    pw[k][0] = 1.0;
#pragma unroll
                    for (int t = 1; t <= L; ++t) pw[k][t] = pw[k][t - 1] * G;
                }
                int h = 0;
#pragma unroll
                for (int t = 0; t <= L; ++t)
#pragma unroll
                    for (int u = 0; u <= L - t; ++u)
#pragma unroll
                        for (int w3 = 0; w3 <= L - t - u; ++w3, ++h) m[h] += pw[0][t] * pw[1][u] * pw[2][w3] * ph4[t + u + w3];
            }
        }
#pragma unroll
        for (int h = 0; h < NH; ++h) {
            const double y = warp_sum(m[h]);
            if (lane == 0) red[wid][h] = y;
        }
        __syncthreads();
        for (int h = threadIdx.x; h < NH; h += 128) H[h] = (red[0][h] + red[1][h]) + (red[2][h] + red[3][h]);
        __syncthreads();
        if (threadIdx.x < NAB) {
            double E[3][(LA + 1) * (LB + 1) * NT];
#pragma unroll
            for (int k = 0; k < 3; ++k) herm_E<LA, LB, double>(x.PA[k], x.PB[k], 0.5 / x.p, E[k]);
            double Hr[D * D * D];
            {
                int h = 0;
#pragma unroll
                for (int t = 0; t <= L; ++t)
#pragma unroll
                    for (int u = 0; u <= L - t; ++u)
#pragma unroll
                        for (int w3 = 0; w3 <= L - t - u; ++w3, ++h) Hr[(t * D + u) * D + w3] = H[h];
            }
#pragma unroll
            for (int a = 0; a < NA; ++a)
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    if (threadIdx.x != a * NB + b) continue;
                    const int ax = cexp(LA, a, 0), ay = cexp(LA, a, 1), az = cexp(LA, a, 2);
                    const int bx = cexp(LB, b, 0), by = cexp(LB, b, 1), bz = cexp(LB, b, 2);
                    double y = 0.0;
#pragma unroll
                    for (int tx = 0; tx <= ax + bx; ++tx)
#pragma unroll
                        for (int ty = 0; ty <= ay + by; ++ty)
#pragma unroll
                            for (int tz = 0; tz <= az + bz; ++tz)
                                y += E[0][(ax * (LB + 1) + bx) * NT + tx] * E[1][(ay * (LB + 1) + by) * NT + ty] *
                                     E[2][(az * (LB + 1) + bz) * NT + tz] * Hr[(tx * D + ty) * D + tz];
                    acc += x.K * y;
                }
        }
    }
    if (threadIdx.x < NAB) out[(size_t)(img - b0) * NAB + threadIdx.x] += acc;  // the real part is there already
}

// one launch per class of shell-pair images (op 0 kinetic, 1 real part, 2
// reciprocal part of the attraction)
struct OneeArgs {
    PlanDev pl;
    int op = 0;
    const double2 *ab;
    int natom;
    const double *Z, *xyz, *cand;
    int ncand;
    int g0, gcur, nmax;
    const double2 *v;
    const double *gtab;
    double *blk;   // blocks of all images, class after class
    double *Out;   // raw matrix
    cudaStream_t st;
};
template <int LA, int LB>
static size_t onee_go(const OneeArgs &a, int b0, int b1, size_t off)
{
    constexpr int NAB = ncart(LA) * ncart(LB);
    if (b1 <= b0) return off;
    const unsigned nb = (unsigned)(b1 - b0);
    double *blk = a.blk + off;
    if (a.op == 0) k_onee_kinetic<LA, LB><<<(nb + 3) / 4, 128, 0, a.st>>>(a.pl, b0, b1, a.ab, blk);
    else if (a.op == 1)
        k_onee_real<LA, LB><<<(nb + 3) / 4, 128, 0, a.st>>>(a.pl, b0, b1, a.natom, a.Z, a.xyz, a.cand, a.ncand, a.natom > 16 ? 32 : 8, blk);
    else
        k_onee_recip<LA, LB><<<nb, 128, 3 * (2 * a.nmax + 1) * sizeof(double2), a.st>>>(a.pl, b0, a.g0, a.gcur, a.nmax, a.v, a.gtab, blk);
    return off + (size_t)nb * NAB;
}

static void launch_onee(const Plan *P, OneeArgs a, int op)
{
    a.op = op;
    size_t off = 0;
    for (int c = 0; c < JK_NCLASS_MAX; ++c) {
        const int b0 = P->classes[c].b0, b1 = P->classes[c].b1;
        switch (c) {
        case 0: off = onee_go<0, 0>(a, b0, b1, off); break;
        case 1: off = onee_go<1, 0>(a, b0, b1, off); break;
        case 2: off = onee_go<1, 1>(a, b0, b1, off); break;
        case 3: off = onee_go<2, 0>(a, b0, b1, off); break;
        case 4: off = onee_go<2, 1>(a, b0, b1, off); break;
        case 5: off = onee_go<2, 2>(a, b0, b1, off); break;
        default: break;
        }
    }
}

static void launch_gather(const Plan *P, const OneeArgs &a)
{
    ImageBlocks ib{};
    for (int c = 0; c < JK_NCLASS_MAX; ++c) {
        const ClassRange &r = P->classes[c];
        const long long nab = ncart(r.la) * ncart(r.lb);
        ib.b0[c] = r.b0;
        ib.sp0[c] = P->spair_class_off[c];
        if (c + 1 < JK_NCLASS_MAX) ib.off[c + 1] = ib.off[c] + (size_t)((r.b1 - r.b0) * nab);
        ib.first[c + 1] = ib.first[c] + (P->spair_class_off[c + 1] - P->spair_class_off[c]) * nab;
    }
    const int gsz = P->spi.size() > 8 * P->spair.size() ? 32 : 8;
    const long long threads = gsz * ib.first[JK_NCLASS_MAX];
    if (threads > 0) k_onee_gather<<<(unsigned)((threads + 127) / 128), 128, 0, a.st>>>(a.pl, ib, gsz, a.blk, a.Out);
}

// sign (8 pi w(G) / V)^{pw/2} (Re, Im) of rho_N(G) = sum_C Z_C e^{-iG.C}, one
// warp per G (pw 1: the column weight of the structure-factor slab; pw 2:
// both weights)
__global__ void __launch_bounds__(128) k_nuclear_sfac(int natom, const double *__restrict__ Zc, const double *__restrict__ xyz,
                                                      const double *__restrict__ gv, int g0, int gcur, int pw, double sign,
                                                      double2 *__restrict__ out)
{
    const int gi = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (gi >= gcur) return;
    const double *g = gv + 4 * (size_t)(g0 + gi);
    double re = 0, im = 0;
    for (int C = lane; C < natom; C += 32) {
        double sn, cs;
        sincos(g[0] * xyz[3 * C] + g[1] * xyz[3 * C + 1] + g[2] * xyz[3 * C + 2], &sn, &cs);
        re += Zc[C] * cs;
        im -= Zc[C] * sn;
    }
    re = warp_sum(re);
    im = warp_sum(im);
    const double f = sign * (pw == 2 ? g[3] * g[3] : g[3]);
    if (lane == 0) out[gi] = make_double2(f * re, f * im);
}

// Out = F o (A + c S_raw): component factors and the self term; A is read from
// its upper triangle, so Out is symmetric to the bit
__global__ void k_onee_final(int n, const double *__restrict__ f, const double *__restrict__ A, const double *__restrict__ S, double c,
                             double *__restrict__ Out)
{
    const size_t n2 = (size_t)n * n;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n2; i += (size_t)gridDim.x * blockDim.x)
    {
        const size_t r = i / n, q = i % n;
        Out[i] = f[r] * f[q] * (A[min(r, q) * n + max(r, q)] + c * S[i]);
    }
}

}  // namespace

int one_electron(Plan *P, int natom, const double *Z, const double *xyz, double *T, double *V, cudaStream_t st)
{
    const int n = P->nbf;
    const size_t n2 = (size_t)n * n;
    Workspace &w = P->ws;
    const PlanDev pl = P->dev();
    auto ok = [](cudaError_t e) { return e == cudaSuccess; };
    const int grid = (int)std::min<size_t>((n2 + 255) / 256, 152 * 16);
    // blocks of the images, in the build's exchange scratch (rewritten by every
    // build before it is read) where they take at most half of it
    size_t nblk = 0;
    for (const ClassRange &c : P->classes) nblk += (size_t)(c.b1 - c.b0) * ncart(c.la) * ncart(c.lb);
    nblk += nblk & 1;
    const size_t scratch = 2 * (size_t)w.gc * n2;
    const bool inside = nblk <= scratch / 2;
    OneeArgs a{};
    a.pl = pl;
    a.st = st;
    a.blk = w.Z;
    if (!inside && !ok(cudaMallocAsync((void **)&a.blk, nblk * sizeof(double), st))) return fail_cuda(JK_ERR_OOM, "one-electron scratch");
    // end of the call on any path: the scratch goes back and the stream is waited for
    const auto finish = [&] {
        if (!inside) cudaFreeAsync(a.blk, st);
        return ok(cudaStreamSynchronize(st));
    };
    if (T) {
        bool good = ok(cudaMemsetAsync(w.T1, 0, n2 * sizeof(double), st));
        a.ab = P->d_ppi_ab;
        a.Out = w.T1;
        launch_onee(P, a, 0);
        launch_gather(P, a);
        k_onee_final<<<grid, 256, 0, st>>>(n, P->d_compf, w.T1, P->d_S, 0.0, T);
        if (!ok(cudaGetLastError()) || !good) {
            finish();
            return fail_cuda(JK_ERR_CUDA, "kinetic-energy kernels failed");
        }
    }
    if (!V || natom <= 0) return finish() ? JK_OK : fail_cuda(JK_ERR_CUDA, "one-electron kernels failed");

    // lattice candidates for the charges' images: |R| up to the largest
    // screening radius plus the cell's circumradius (the reduced X0 is at
    // most that long), sorted by length
    double zmax = 0, ztot = 0;
    for (int C = 0; C < natom; ++C) {
        zmax = std::max(zmax, std::fabs(Z[C]));
        ztot += Z[C];
    }
    const double w2 = P->omega * P->omega, lgd = std::log(P->cut.ewald_R * 1e-1);
    double rmax = 0;
    for (size_t q = 0; q < P->pvals.size(); ++q) {
        // the radius grows with |K|: the largest one of each exponent decides
        const double p = P->pvals[q], c = std::sqrt(w2 / (p + w2)), aw = p * w2 / (p + w2);
        const double lg = std::log(2.0 * kPi / p * P->pval_kmax[q] * zmax * (1.0 - c)) - lgd;
        if (lg <= 0) continue;
        double r = std::sqrt(lg / aw);
        for (int it = 0; it < 2; ++it) r = std::sqrt((lg + 4.0 * std::log(1.0 + 2.0 * aw * r)) / aw);
        rmax = std::max(rmax, r + 1.5);
    }
    double hd = 0;
    for (int s1 = -1; s1 <= 1; s1 += 2)
        for (int s2 = -1; s2 <= 1; s2 += 2)
            for (int s3 = -1; s3 <= 1; s3 += 2) {
                double v[3];
                for (int k = 0; k < 3; ++k) v[k] = 0.5 * (s1 * P->L[k] + s2 * P->L[3 + k] + s3 * P->L[6 + k]);
                hd = std::max(hd, std::sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]));
            }
    std::vector<std::array<double, 4>> cv;
    {
        const double R = rmax + hd;
        int nr[3];
        for (int a = 0; a < 3; ++a) {
            const double inv = std::sqrt(P->Finv[3 * a] * P->Finv[3 * a] + P->Finv[3 * a + 1] * P->Finv[3 * a + 1] +
                                         P->Finv[3 * a + 2] * P->Finv[3 * a + 2]);
            nr[a] = (int)std::ceil(R * inv) + 1;
        }
        for (int i = -nr[0]; i <= nr[0]; ++i)
            for (int j = -nr[1]; j <= nr[1]; ++j)
                for (int k = -nr[2]; k <= nr[2]; ++k) {
                    double v[3];
                    for (int a = 0; a < 3; ++a) v[a] = i * P->L[a] + j * P->L[3 + a] + k * P->L[6 + a];
                    const double len = std::sqrt(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
                    if (len < R) cv.push_back({v[0], v[1], v[2], len});
                }
        std::sort(cv.begin(), cv.end(), [](const std::array<double, 4> &a, const std::array<double, 4> &b) { return a[3] < b[3]; });
    }
    const int ncand = (int)cv.size();
    // scratch of the call in one piece: charges, positions, candidates, rho_N(G)
    const int ng = (int)(P->gvec.size() / 4);
    const size_t oX = ((size_t)natom + 1) / 2 * 2, oC = oX + (3 * (size_t)natom + 1) / 2 * 2, oN = oC + 4 * (size_t)std::max(1, ncand);
    double *dZ = nullptr;
    if (!ok(cudaMallocAsync((void **)&dZ, sizeof(double) * (oN + 2 * (size_t)std::max(1, ng)), st))) {
        finish();
        return fail_cuda(JK_ERR_OOM, "one-electron scratch");
    }
    double *dX = dZ + oX, *dC = dZ + oC;
    double2 *dn = reinterpret_cast<double2 *>(dZ + oN);
    cudaMemcpyAsync(dZ, Z, sizeof(double) * natom, cudaMemcpyHostToDevice, st);
    cudaMemcpyAsync(dX, xyz, sizeof(double) * 3 * natom, cudaMemcpyHostToDevice, st);
    if (ncand) cudaMemcpyAsync(dC, cv.data(), sizeof(double) * 4 * ncand, cudaMemcpyHostToDevice, st);
    bool good = ok(cudaMemsetAsync(w.T2, 0, n2 * sizeof(double), st));
    a.natom = natom;
    a.Z = dZ;
    a.xyz = dX;
    a.cand = dC;
    a.ncand = ncand;
    a.Out = w.T2;
    launch_onee(P, a, 1);
    // reciprocal part.  The phase tables of k_onee_recip hold every integer
    // coordinate of G (nmax up to 64: 6 KB); a lattice that needs more takes
    // the structure-factor slab chunk by chunk, as the build does
    if (ng > 0 && P->g_nmax <= 64) {
        // Gaussian factors of as many G as fit what is left of that scratch
        const size_t used = inside ? nblk : 0, cap = scratch - used, np = std::max<size_t>(1, P->pvals.size());
        const int gch = (int)std::max<size_t>(1, std::min<size_t>((size_t)ng, cap / np));
        k_nuclear_sfac<<<(ng + 3) / 4, 128, 0, st>>>(natom, dZ, dX, P->d_gvec, 0, ng, 2, -1.0, dn);
        a.nmax = P->g_nmax;
        const bool fits = cap >= np;
        a.gtab = fits ? w.Z + used : w.gtab;  // w.gtab holds at least one G
        for (int g0 = 0; g0 < ng; g0 += a.gcur) {
            a.g0 = g0;
            a.gcur = std::min(fits ? gch : w.gc, ng - g0);
            a.v = dn + g0;
            launch_gauss_table(P, g0, a.gcur, const_cast<double *>(a.gtab), st);
            launch_onee(P, a, 2);
        }
        launch_gather(P, a);
    } else {
        launch_gather(P, a);
        for (int g0 = 0; g0 < ng; g0 += w.gc) {
            const int gcur = std::min(w.gc, ng - g0);
            launch_gauss_table(P, g0, gcur, w.gtab, st);
            for (int c = 0; c < JK_NCLASS_MAX; ++c)
                launch_sfac(c, pl, P->spair_class_off[c], P->spair_class_off[c + 1], P->d_gvec, g0, gcur, w.gtab, w.M, st);
            k_nuclear_sfac<<<(gcur + 3) / 4, 128, 0, st>>>(natom, dZ, dX, P->d_gvec, g0, gcur, 1, 1.0, dn);
            slab_gemv_n(w.M, (long long)n2, 2 * gcur, reinterpret_cast<const double *>(dn), -1.0, w.T2, st, false);
        }
    }
    // self term +(pi/(V w^2)) Z_tot S and the component factors
    k_onee_final<<<grid, 256, 0, st>>>(n, P->d_compf, w.T2, P->d_S, kPi / (P->volume * w2) * ztot, V);
    cudaFreeAsync(dZ, st);
    good = ok(cudaGetLastError()) && good;
    good = finish() && good;  // also where a launch failed: the copies above read the caller's host arrays
    return good ? JK_OK : fail_cuda(JK_ERR_CUDA, "nuclear-attraction kernels failed");
}

}  // namespace jk
