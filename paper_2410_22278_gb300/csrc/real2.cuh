// Warp-cooperative real-space quartet kernels (erfc part of Eq.
// pbc_eri_general_final) for the classes of s and p shells.
//
// The lane-per-bra tile kernel of kernels.cuh lets the 32 lanes of a warp
// walk one ket with 32 different bras; lanes whose bra cannot reach the ket,
// or whose primitive quartet is screened out, idle while the others work.
// Here one warp owns one bra image and a range of kets, and every stage --
// image quartets, primitive quartets, terms, digestion -- is refilled to 32
// lanes from the one before (k_real_w below).
// Primitive pairs are stored in descending order of B = |K| p^{-5/4}: every
// primitive prefactor 2 pi^{5/2} |K_i K_j| / (pq sqrt(p+q)) is at most
// 2 pi^{5/2} 2^{-1/2} B_i B_j (p + q >= 2 sqrt(pq)), so a loop over
// primitives ends at the first pair whose B_i B_j lies below the
// per-term threshold (PlanDev::mag_thr): the magnitude test of Eq.
// pbc_eri_real_cutoff_implementation fails for it and for every later one.
// Which kernel family (this one, the lane-per-bra one of kernels.cuh or the
// pair-queue one below) runs a class pair is chosen by the autotuner.
// The FP64 pass over the large quartets of the mixed path refills its lanes the
// same way, from groups of list entries (k_real_list_w).
#pragma once
#include "kernels.cuh"
#include "launch.h"

namespace jk {

// Pair data plus its Hermite coefficients in the kernel's precision.
template <int LA, int LB, typename T>
struct PrimE {
    PairT<T> x;
    T E[3][(LA + 1) * (LB + 1) * (LA + LB + 1)];
};

template <int LA, int LB, typename T>
__device__ __forceinline__ void load_prim(const PlanDev &pl, int k, PrimE<LA, LB, T> &o, PpiF &f)
{
    f = pl.ppf[k];
    load_pair(pl, k, f, o.x);
    const T oo2p = T(0.5) * o.x.ip;
#pragma unroll
    for (int a = 0; a < 3; ++a) herm_E<LA, LB, T>(o.x.PA[a], o.x.PB[a], oo2p, o.E[a]);
}

// Screening of one primitive quartet, all in single precision: true if some
// lattice image of P - Q lies inside the sphere of Eq.
// pbc_eri_real_cutoff_implementation (the same radius and image test as
// prim_term).  The minimum image decides at once when it lies inside; else
// no other image can, unless the shortest non-zero candidate vector is
// shorter than |X0| + r (|X0 - R1| >= |R1| - |X0|).
template <int L>
__device__ __forceinline__ bool prim_reaches(const PlanDev &pl, const PpiF &bf, const PpiF &kf)
{
    const float ipf = bf.pad, iqf = kf.pad;
    const float awf = frcp_fast(ipf + iqf + pl.inv_omega2f);
    const float cwf = fsqrt_fast(awf * (ipf + iqf));
    const float preff = 34.986836655249725f * bf.K * kf.K * ipf * iqf * rsqrtf(bf.p + kf.p);
    const float lg = __logf(fabsf(preff) * (1.0f - cwf)) - pl.log_ewald_R;
    if (!(lg > 0.0f)) return false;
    float r = fsqrt_fast(fdiv_fast(lg, awf));
    if (L > 0) {
        r = fsqrt_fast(fdiv_fast(lg + L * __logf(1.0f + 2.0f * awf * r), awf));
        r = fsqrt_fast(fdiv_fast(lg + L * __logf(1.0f + 2.0f * awf * r), awf));
        r += 0.5f + 0.25f * L;
    }
    float X0[3] = {bf.P[0] - kf.P[0], bf.P[1] - kf.P[1], bf.P[2] - kf.P[2]};
    float f[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) f[a] = rintf(pl.Finvf[3 * a] * X0[0] + pl.Finvf[3 * a + 1] * X0[1] + pl.Finvf[3 * a + 2] * X0[2]);
#pragma unroll
    for (int a = 0; a < 3; ++a) X0[a] -= f[0] * pl.Lf[a] + f[1] * pl.Lf[3 + a] + f[2] * pl.Lf[6 + a];
    const float x2 = X0[0] * X0[0] + X0[1] * X0[1] + X0[2] * X0[2];
    const float r2 = r * r;
    if (x2 < r2) return true;
    const float x0n = fsqrt_fast(x2);
    for (int c = 1; c < pl.nr1; ++c) {
        if (pl.r1f[4 * c + 3] - x0n >= r) return false;
        const float Xx = X0[0] - pl.r1f[4 * c], Xy = X0[1] - pl.r1f[4 * c + 1], Xz = X0[2] - pl.r1f[4 * c + 2];
        if (Xx * Xx + Xy * Xy + Xz * Xz < r2) return true;
    }
    return false;
}

// Exact screening radius of one primitive quartet (Eq.
// pbc_eri_real_cutoff_implementation, single precision); false when the
// quartet has no term above the threshold.
template <int L>
__device__ __forceinline__ bool prim_radius(const PlanDev &pl, const PpiF &bf, const PpiF &kf, float &r)
{
    const float ipf = bf.pad, iqf = kf.pad;
    const float awf = frcp_fast(ipf + iqf + pl.inv_omega2f);
    const float cwf = fsqrt_fast(awf * (ipf + iqf));
    const float preff = 34.986836655249725f * bf.K * kf.K * ipf * iqf * rsqrtf(bf.p + kf.p);
    const float lg = __logf(fabsf(preff) * (1.0f - cwf)) - pl.log_ewald_R;
    if (!(lg > 0.0f)) return false;
    r = fsqrt_fast(fdiv_fast(lg, awf));
    if (L > 0) {
        r = fsqrt_fast(fdiv_fast(lg + L * __logf(1.0f + 2.0f * awf * r), awf));
        r = fsqrt_fast(fdiv_fast(lg + L * __logf(1.0f + 2.0f * awf * r), awf));
        r += 0.5f + 0.25f * L;  // the Gaussian bound is derived for s functions; widen for L > 0
    }
    return true;
}

// alpha = 1/(1/p + 1/q), alpha_w = 1/(1/p + 1/q + 1/w^2), c_w = sqrt(alpha_w / alpha).
// FP64: one reciprocal square root instead of two divisions and a square
// root (about 12 FP64 instructions against 30; within 3 ulp).
__device__ __forceinline__ void alphas(double ipq, double iw2, double &alpha, double &aw, double &cw)
{
    const double b = ipq + iw2, y = rsqrt(ipq * b), t = y * y;
    alpha = t * b;
    aw = t * ipq;
    cw = ipq * y;
}
__device__ __forceinline__ void alphas(float ipq, float iw2, float &alpha, float &aw, float &cw)
{
    aw = rcp_nr(ipq + iw2);
    alpha = rcp_nr(ipq);
    cw = sqrt_nr(aw * ipq);
}
__device__ __forceinline__ double inv_sqrt(double x) { return rsqrt(x); }
__device__ __forceinline__ float inv_sqrt(float x) { return rsqrt_nr(x); }

// Geometry of one primitive quartet: its screening sphere, the nearest image
// of P - Q (single precision F0 for the image search, X0 for the terms) and
// its exponents.
template <typename T>
struct PrimGeo {
    float F0[3], r, x0n;
    T X0[3], alpha, aw, cw;
};

template <int L, typename T>
__device__ __forceinline__ bool prim_geo(const PlanDev &pl, const PairT<T> &x, const PpiF &bf, const PairT<T> &y, const PpiF &kf,
                                         PrimGeo<T> &g, Tally &tl)
{
    ++tl.screen;
    if (!prim_radius<L>(pl, bf, kf, g.r)) return false;
    ++tl.radius;
    float f[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        g.F0[a] = bf.P[a] - kf.P[a];
        g.X0[a] = x.P[a] - y.P[a];
    }
    if (pl.orth == 2) {
        // diagonal lattice: rounding by adding and subtracting 1.5 * 2^23
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            f[a] = fmaf(g.F0[a], pl.Finvf[4 * a], 12582912.0f) - 12582912.0f;
            g.F0[a] = fmaf(-f[a], pl.Lf[4 * a], g.F0[a]);
        }
        if (sizeof(T) == 4 || f[0] != 0.0f || f[1] != 0.0f || f[2] != 0.0f)
#pragma unroll
            for (int a = 0; a < 3; ++a) g.X0[a] -= T(f[a]) * latc(pl.L, pl.Lf, 4 * a, T(0));
    } else {
#pragma unroll
        for (int a = 0; a < 3; ++a)
            f[a] = rintf(pl.Finvf[3 * a] * g.F0[0] + pl.Finvf[3 * a + 1] * g.F0[1] + pl.Finvf[3 * a + 2] * g.F0[2]);
        if (f[0] != 0.0f || f[1] != 0.0f || f[2] != 0.0f) {
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                g.F0[a] -= f[0] * pl.Lf[a] + f[1] * pl.Lf[3 + a] + f[2] * pl.Lf[6 + a];
                g.X0[a] -= T(f[0]) * latc(pl.L, pl.Lf, a, T(0)) + T(f[1]) * latc(pl.L, pl.Lf, 3 + a, T(0)) +
                           T(f[2]) * latc(pl.L, pl.Lf, 6 + a, T(0));
            }
        }
    }
    g.x0n = fsqrt_fast(g.F0[0] * g.F0[0] + g.F0[1] * g.F0[1] + g.F0[2] * g.F0[2]);
    alphas(x.ip + y.ip, latc(&pl.inv_omega2, &pl.inv_omega2f, 0, T(0)), g.alpha, g.aw, g.cw);
    return true;
}

// Index of the first lattice vector from c on whose image lies inside the
// sphere, pl.nr1 if there is none.
template <typename T>
__device__ __forceinline__ int next_image(const PlanDev &pl, const PrimGeo<T> &g, int c, Tally &tl)
{
    const float4 *lat = reinterpret_cast<const float4 *>(pl.r1f);
    const float r2 = g.r * g.r;
#pragma unroll 1
    for (; c < pl.nr1; ++c) {
        const float4 R = __ldg(lat + c);
        if (R.w - g.x0n >= g.r) break;
        ++tl.cand;
        const float fx = g.F0[0] - R.x, fy = g.F0[1] - R.y, fz = g.F0[2] - R.z;
        if (fx * fx + fy * fy + fz * fz < r2) return c;
    }
    return pl.nr1;
}

// Rs += Hermite R table of the image c.
template <int L, typename T>
__device__ __forceinline__ void add_image(const PlanDev &pl, const T *X0, T alpha, T aw, T cw, int c, T *Rs)
{
    constexpr int D = L + 1;
    const T Xx = X0[0] - lat_at(pl, 4 * c, T(0)), Xy = X0[1] - lat_at(pl, 4 * c + 1, T(0)), Xz = X0[2] - lat_at(pl, 4 * c + 2, T(0));
    T s[L + 1];
    seeds<L>(Xx * Xx + Xy * Xy + Xz * Xz, alpha, aw, cw, pl, s);
    T Bt[D * D * D];
    herm_R<L, T>(s, Xx, Xy, Xz, Bt);
#pragma unroll
    for (int t = 0; t <= L; ++t)
#pragma unroll
        for (int u = 0; u <= L - t; ++u)
#pragma unroll
            for (int v = 0; v <= L - t - u; ++v) Rs[(t * D + u) * D + v] += Bt[(t * D + u) * D + v];
}

// One lane's images one after another; false if there is none.  The image
// search runs in single precision (it only decides which terms are formed)
// and each lane walks on to its next image before the terms are formed, so
// the lanes of a warp form them together.
template <int L, typename T>
__device__ __forceinline__ bool all_images(const PlanDev &pl, const PrimGeo<T> &g, T *Rs, Tally &tl)
{
    int n = 0;
#pragma unroll 1
    for (int c = next_image(pl, g, 0, tl); c < pl.nr1; c = next_image(pl, g, c + 1, tl)) {
        add_image<L, T>(pl, g.X0, g.alpha, g.aw, g.cw, c, Rs);
        ++n;
    }
    tl.img += n;
    return n > 0;
}

// V += contraction of the Hermite table Rs of one primitive quartet with both
// E tables.
template <int LA, int LB, int LC, int LD, typename T>
__device__ __forceinline__ void contract(const PrimE<LA, LB, T> &b, const PrimE<LC, LD, T> &k, const T *Rs, T *V)
{
    constexpr int NA = ncart(LA), NB = ncart(LB), NC = ncart(LC), ND = ncart(LD);
    constexpr int L = LA + LB + LC + LD, LAB = LA + LB, LCD = LC + LD;
    constexpr int NTA = LAB + 1, NTC = LCD + 1, D = L + 1;
    const PairT<T> &x = b.x, &y = k.x;
    const T tp = T(kTwoPi52) * x.K * y.K * x.ip * y.ip * inv_sqrt(x.p + y.p);
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            const int cx = cexp(LC, c, 0), cy = cexp(LC, c, 1), cz = cexp(LC, c, 2);
            const int dx = cexp(LD, d, 0), dy = cexp(LD, d, 1), dz = cexp(LD, d, 2);
            T W[NTA * NTA * NTA];
#pragma unroll
            for (int tx = 0; tx <= LAB; ++tx)
#pragma unroll
                for (int ty = 0; ty <= LAB - tx; ++ty)
#pragma unroll
                    for (int tz = 0; tz <= LAB - tx - ty; ++tz) {
                        T acc = T(0);
#pragma unroll
                        for (int sx = 0; sx <= cx + dx; ++sx)
#pragma unroll
                            for (int sy = 0; sy <= cy + dy; ++sy)
#pragma unroll
                                for (int sz = 0; sz <= cz + dz; ++sz) {
                                    const T e = k.E[0][(cx * (LD + 1) + dx) * NTC + sx] * k.E[1][(cy * (LD + 1) + dy) * NTC + sy] *
                                                k.E[2][(cz * (LD + 1) + dz) * NTC + sz];
                                    const T rv = Rs[((tx + sx) * D + ty + sy) * D + tz + sz];
                                    if ((sx + sy + sz) & 1)
                                        acc -= e * rv;
                                    else
                                        acc += e * rv;
                                }
                        W[(tx * NTA + ty) * NTA + tz] = acc;
                    }
#pragma unroll
            for (int a = 0; a < NA; ++a)
#pragma unroll
                for (int bb = 0; bb < NB; ++bb) {
                    const int ax = cexp(LA, a, 0), ay = cexp(LA, a, 1), az = cexp(LA, a, 2);
                    const int bx = cexp(LB, bb, 0), by = cexp(LB, bb, 1), bz = cexp(LB, bb, 2);
                    T v = T(0);
#pragma unroll
                    for (int tx = 0; tx <= ax + bx; ++tx)
#pragma unroll
                        for (int ty = 0; ty <= ay + by; ++ty)
#pragma unroll
                            for (int tz = 0; tz <= az + bz; ++tz)
                                v += b.E[0][(ax * (LB + 1) + bx) * NTA + tx] * b.E[1][(ay * (LB + 1) + by) * NTA + ty] *
                                     b.E[2][(az * (LB + 1) + bz) * NTA + tz] * W[(tx * NTA + ty) * NTA + tz];
                    V[((a * NB + bb) * NC + c) * ND + d] += tp * v;
                }
        }
}

// One primitive quartet (bra pair b, ket pair k) into the Cartesian block V;
// the events go to the lane's tally (flops.h).
template <int LA, int LB, int LC, int LD, typename T>
__device__ __forceinline__ void prim_term(const PlanDev &pl, const PrimE<LA, LB, T> &b, const PpiF &bf, const PrimE<LC, LD, T> &k,
                                          const PpiF &kf, T *V, Tally &tl)
{
    constexpr int L = LA + LB + LC + LD, D = L + 1;
    PrimGeo<T> g;
    if (!prim_geo<L, T>(pl, b.x, bf, k.x, kf, g, tl)) return;
    T Rs[D * D * D];
#pragma unroll
    for (int q = 0; q < D * D * D; ++q) Rs[q] = T(0);
    if (!all_images<L, T>(pl, g, Rs, tl)) return;
    ++tl.term;
    contract<LA, LB, LC, LD, T>(b, k, Rs, V);
}

// Digest the block V of an image quartet (first basis functions aoI .. aoL of
// its shells, n in all) with orbit weight w: ket-side Coulomb X_kl += 2w sum_ij V D_ij (atomics), exchange in its
// four index assignments (the other four of the orbit are transposes, added
// at assembly), and the bra-side Coulomb term into the lane's jb.
template <int LA, int LB, int LC, int LD, typename T>
__device__ __forceinline__ void digest(int n, int aoI, int aoJ, int aoK, int aoL, const T *V, T w, const T *__restrict__ Dp, const T *Dij,
                                       Acc<T> *jb, double *__restrict__ X, double *__restrict__ Y)
{
    constexpr int NA = ncart(LA), NB = ncart(LB), NC = ncart(LC), ND = ncart(LD);
    auto Dd = [&](int r, int c) { return __ldg(Dp + (size_t)r * n + c); };
#pragma unroll
    for (int ab = 0; ab < NA * NB; ++ab) {
        T s = T(0);
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
            for (int d = 0; d < ND; ++d) s += V[ab * NC * ND + c * ND + d] * Dd(aoK + c, aoL + d);
        jb[ab].add(T(2) * w * s);
    }
#pragma unroll
    for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int d = 0; d < ND; ++d) {
            T s = T(0);
#pragma unroll
            for (int ab = 0; ab < NA * NB; ++ab) s += V[ab * NC * ND + c * ND + d] * Dij[ab];
            atomicAdd(X + (size_t)(aoK + c) * n + aoL + d, to_f64(T(2) * w * s));
        }
    if (!Y) return;  // a Coulomb-only build
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
        for (int d = 0; d < ND; ++d) {  // K_il += w V_ijkl D_jk
            T s = T(0);
#pragma unroll
            for (int b = 0; b < NB; ++b)
#pragma unroll
                for (int c = 0; c < NC; ++c) s += V[((a * NB + b) * NC + c) * ND + d] * Dd(aoJ + b, aoK + c);
            atomicAdd(Y + (size_t)(aoI + a) * n + aoL + d, to_f64(w * s));
        }
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int d = 0; d < ND; ++d) {  // K_jl += w V_ijkl D_ik
            T s = T(0);
#pragma unroll
            for (int a = 0; a < NA; ++a)
#pragma unroll
                for (int c = 0; c < NC; ++c) s += V[((a * NB + b) * NC + c) * ND + d] * Dd(aoI + a, aoK + c);
            atomicAdd(Y + (size_t)(aoJ + b) * n + aoL + d, to_f64(w * s));
        }
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
        for (int c = 0; c < NC; ++c) {  // K_ik += w V_ijkl D_jl
            T s = T(0);
#pragma unroll
            for (int b = 0; b < NB; ++b)
#pragma unroll
                for (int d = 0; d < ND; ++d) s += V[((a * NB + b) * NC + c) * ND + d] * Dd(aoJ + b, aoL + d);
            atomicAdd(Y + (size_t)(aoI + a) * n + aoK + c, to_f64(w * s));
        }
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
        for (int c = 0; c < NC; ++c) {  // K_jk += w V_ijkl D_il
            T s = T(0);
#pragma unroll
            for (int a = 0; a < NA; ++a)
#pragma unroll
                for (int d = 0; d < ND; ++d) s += V[((a * NB + b) * NC + c) * ND + d] * Dd(aoI + a, aoL + d);
            atomicAdd(Y + (size_t)(aoJ + b) * n + aoK + c, to_f64(w * s));
        }
}

constexpr int kWarpsPerBlock = 4;

// Image quartets a warp evaluates together (slots of its shared Cartesian
// blocks): as many as 4.6 KB of shared memory per warp hold, so that the last
// partly filled batch of primitive quartets of a group counts little.
template <int NV, typename T>
struct BatchShape {
    static constexpr int per = NV * (int)sizeof(T);
    static constexpr int SL = per <= 24 ? 128 : per <= 36 ? 64 : per <= 144 ? 32 : per <= 216 ? 16 : 8;
    static constexpr int LO = sizeof(T) == 4 ? SL / 2 * NV : 0;  // rounding errors of the sums of a deep bra (k_real_w)
    static constexpr int KQ = SL == 128 ? 256 : SL == 64 ? 128 : 64;  // ring of queued kets, at least SL + 31
};
constexpr int kBraChunk = 16;    // bra primitives screened per round (bits of a lane's mask)
constexpr int kTermRing = 1024;  // at most 31 + 32 * kBraChunk entries are in flight
constexpr int kListRing = 64;    // of the list kernel: at most 31 + 32

// Resident blocks asked for: the FP32 kernels of low momentum wait on
// dependent instructions and need the warps (24 per SM: at most 85 registers).
template <typename T>
constexpr int tile_blocks(int L)
{
    return sizeof(T) == 4 ? (L == 0 ? 6 : L <= 1 ? 5 : L <= 2 ? 4 : 3) : (L == 0 ? 4 : 3);
}

// Quartet-level screening of one image quartet from the packed records (spq,
// spr): quartet_reaches of kernels.cuh with ln S instead of a logarithm per
// pair and, for L > 0, one logarithm instead of two (Lc bounds the correction
// inside it, so the sphere contains the former one).  big_bound receives
// quartet_estimate_bound, brief whether [c_w, 1] is short (the two reasons to
// look at the FP64 list).  All pairs of a launch come through here (7.2e9 for
// (ss|ss) of the 64-water box, of which 17% pass); read from the 72-byte image
// records with the density maxima of every passing pair it was 37% of the
// kernel's time.
template <int L>
__device__ __forceinline__ bool pair_reaches(const PlanDev &pl, const float4 &bq, const float4 &br, const float4 &kq, const float4 &kr,
                                             float Lc, float &big_bound, bool &brief)
{
    const float s = br.y + kr.y + (3.2094f - pl.log_ewald_R);  // ln(2 pi^{5/2} / sqrt 2) + 1e-3
    if (!(s > 0.0f)) return false;
    const float ipq = br.z + kr.z, inv = ipq + pl.inv_omega2f, aw = frcp_fast(inv);
    float u = s;
    if (L > 0) u += L * __logf(1.0f + 2.0f * fsqrt_fast(aw * (s + Lc)));
    const float ext = bq.w + kq.w;
    const float r = 1.0002f * fsqrt_fast(u * inv) + (L > 0 ? 0.5f + 0.25f * L : 0.0f) + ext + 1e-3f;
    float X[3] = {bq.x - kq.x, bq.y - kq.y, bq.z - kq.z}, d2, e2;
    if (pl.orth == 2) {
#pragma unroll
        for (int a = 0; a < 3; ++a) X[a] = fmaf(-(fmaf(X[a], pl.Finvf[4 * a], 12582912.0f) - 12582912.0f), pl.Lf[4 * a], X[a]);
        d2 = e2 = X[0] * X[0] + X[1] * X[1] + X[2] * X[2];
    } else {
        float f[3], Y[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            f[a] = pl.Finvf[3 * a] * X[0] + pl.Finvf[3 * a + 1] * X[1] + pl.Finvf[3 * a + 2] * X[2];
            f[a] -= rintf(f[a]);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) Y[a] = f[0] * pl.Lf[a] + f[1] * pl.Lf[3 + a] + f[2] * pl.Lf[6 + a];
        d2 = e2 = Y[0] * Y[0] + Y[1] * Y[1] + Y[2] * Y[2];
        if (!pl.orth) {
            // skewed: the rounded image need not be the nearest; plane spacings bound the distance
            const float dp = fmaxf(fmaxf(pl.hplane[0] * fabsf(f[0]), pl.hplane[1] * fabsf(f[1])), pl.hplane[2] * fabsf(f[2]));
            d2 = dp * dp;
        }
    }
    const float dd = fmaxf(0.0f, fsqrt_fast(e2) - ext);
    big_bound = 24.7394241f * 1.002f * br.x * kr.x * __expf(-0.9999f * aw * dd * dd);
    brief = ipq > 0.7224f * (ipq + pl.inv_omega2f);
    return d2 < r * r;
}

// Mixed precision: true if the image quartet (bra, kt) goes to the FP64 list,
// decided as in k_real; called for the few that may (pair_reaches).
template <typename T>
__device__ __noinline__ bool list_quartet(const PlanDev &pl, int bra, int kt, float tauf, const T *__restrict__ dmax, QuartetList big,
                                          unsigned *__restrict__ nbig, unsigned cap, unsigned *__restrict__ ovf)
{
    const SpiRec sb = pl.spi[bra], sk = pl.spi[kt];
    const float dm = quartet_dmax(reinterpret_cast<const float *>(dmax), pl.nshell, sb, sk);
    const float est = quartet_estimate_bound(pl, sb, sk) * dm >= tauf ? quartet_estimate(pl, sb, sk) * dm : 0.0f;
    const float ipq = frcp_fast(sb.pmin) + frcp_fast(sk.pmin);
    if (!(est >= tauf || ipq > 0.7225f * (ipq + pl.inv_omega2f))) return false;
    const unsigned slot = atomicAdd(nbig, 1u);
    if (slot < cap) {
        big.put(slot, bra, kt);
        return true;
    }
    atomicAdd(ovf, 1u);
    return false;
}

// Largest ln(1 + 2 alpha_w r) correction of a screening radius over the plan
// (alpha_w r = sqrt(alpha_w u) <= omega sqrt(u), u the exponent at the edge).
template <int L>
__device__ __forceinline__ float radius_correction(const PlanDev &pl, float smax)
{
    if (L == 0) return 0.0f;
    const float om2 = 2.0f * rsqrtf(pl.inv_omega2f);
    float u = smax;
#pragma unroll 1
    for (int it = 0; it < 4; ++it) u = smax + L * __logf(1.0f + om2 * fsqrt_fast(fmaxf(u, 0.0f)));
    return 1.05f * fmaxf(u - smax, 0.0f);
}

// Images of a batch of primitive quartets shared out evenly over the lanes of
// a warp (FP64, total momentum up to 2, where the sum of the R table over lanes
// is cheap).  A small cell has several images per primitive quartet, one to
// twenty: lane by lane, the batch takes as many rounds as its largest count,
// three times the mean, and an FP64 instruction costs the same however few
// lanes take part.  FP64 build of 6 water molecules: (ss|ss) 49.7 -> 25.7 ms,
// (ss|ps) 49.5 -> 37.2 ms.  In single precision the bookkeeping cost more than
// it saved ((ss|ss) of 5 molecules 7.0 -> 10.0 ms), and so it did for the
// listed quartets, which have ten and more images each.
constexpr int kImgRound = 8;  // images a lane lists per round
template <int L, typename T>
struct ImgShare {
    static constexpr bool on = L <= 2 && sizeof(T) == 8;
    unsigned short list[on ? 32 * kImgRound : 1];  // owner lane and lattice vector
    T R[on ? 32 * nherm(L) : 1];                    // sums of the owners' R tables
};

// Rs = R table of the lane's primitive quartet (g, if act), summed over its
// images; every lane of the warp calls this.  n and total: images of this lane
// and of the warp.
template <int L, typename T>
__device__ __forceinline__ void shared_images(const PlanDev &pl, const PrimGeo<T> &g, int n, ImgShare<L, T> &sh, T *Rs)
{
    constexpr int D = L + 1, NH = nherm(L);
    const int lane = threadIdx.x & 31;
    Tally none;
#pragma unroll
    for (int h = 0; h < NH; ++h) sh.R[h * 32 + lane] = T(0);
    int c = -1;
#pragma unroll 1
    while (__any_sync(0xffffffffu, n > 0)) {
        const int now = min(n, kImgRound);
        int pos = now;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, pos, o);
            if (lane >= o) pos += t;
        }
        const int total = __shfl_sync(0xffffffffu, pos, 31);
        pos -= now;
#pragma unroll 1
        for (int i = 0; i < now; ++i) {
            c = next_image(pl, g, c + 1, none);
            sh.list[pos + i] = (unsigned short)(lane << 11 | c);
        }
        n -= now;
        __syncwarp();
#pragma unroll 1
        for (int e0 = 0; e0 < total; e0 += 32) {
            const bool on = e0 + lane < total;
            const unsigned it = on ? sh.list[e0 + lane] : 0u;
            const int src = (int)(it >> 11);
            T X0[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) X0[a] = __shfl_sync(0xffffffffu, g.X0[a], src);
            const T alpha = __shfl_sync(0xffffffffu, g.alpha, src), aw = __shfl_sync(0xffffffffu, g.aw, src),
                    cw = __shfl_sync(0xffffffffu, g.cw, src);
            T Ri[D * D * D];
#pragma unroll
            for (int q = 0; q < D * D * D; ++q) Ri[q] = T(0);
            if (on) add_image<L, T>(pl, X0, alpha, aw, cw, (int)(it & 2047u), Ri);
            __syncwarp();
            // sum over the lanes of one owner (adjacent), then its first lane adds
            const int key = on ? src : 32 + lane;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int ok = __shfl_down_sync(0xffffffffu, key, o);
                const bool add = lane + o < 32 && ok == key;
                if (!__any_sync(0xffffffffu, add)) break;
#pragma unroll
                for (int t = 0; t <= L; ++t)
#pragma unroll
                    for (int u = 0; u <= L - t; ++u)
#pragma unroll
                        for (int v = 0; v <= L - t - u; ++v) {
                            const T y = __shfl_down_sync(0xffffffffu, Ri[(t * D + u) * D + v], o);
                            if (add) Ri[(t * D + u) * D + v] += y;
                        }
            }
            const int prev = __shfl_up_sync(0xffffffffu, key, 1);
            if (on && (lane == 0 || prev != key)) {
                int h = 0;
#pragma unroll
                for (int t = 0; t <= L; ++t)
#pragma unroll
                    for (int u = 0; u <= L - t; ++u)
#pragma unroll
                        for (int v = 0; v <= L - t - u; ++v, ++h) sh.R[h * 32 + src] += Ri[(t * D + u) * D + v];
            }
            __syncwarp();
        }
    }
    int h = 0;
#pragma unroll
    for (int t = 0; t <= L; ++t)
#pragma unroll
        for (int u = 0; u <= L - t; ++u)
#pragma unroll
            for (int v = 0; v <= L - t - u; ++v, ++h) Rs[(t * D + u) * D + v] = sh.R[h * 32 + lane];
    __syncwarp();
}

// First index in [lo, hi) whose primitive pairs start at or after `val` (hi if
// none); the whole warp searches, 32 probes per step.
__device__ __forceinline__ int first_at(const SpiRec *__restrict__ spi, int lo, int hi, long long val)
{
    const int lane = threadIdx.x & 31;
    while (lo < hi) {
        const int step = (hi - lo + 31) / 32, idx = lo + lane * step;
        const unsigned m = __ballot_sync(0xffffffffu, idx < hi && spi[idx].pp0 < val);
        const int c = __popc(m);
        if (c == 0) return lo;
        hi = min(hi, lo + c * step);
        lo += (c - 1) * step + 1;
    }
    return lo;
}

// Bra and ket range of warp `item` of a launch (TileMap); false if it has none.
__device__ __forceinline__ bool tile_of(const PlanDev &pl, const TileMap &map, long long item, int k0, int k1, int same, int &bra, int &kbeg,
                                        int &kend)
{
    if (item >= map.items) return false;
    int r = 0;
    while (r + 1 < map.n && item >= map.g[r + 1].first) ++r;
    const TileMap::Range &g = map.g[r];
    const int rel = (int)((item - g.first) / g.nch), ch = (int)((item - g.first) % g.nch);
    bra = g.b0 + rel;
    const long long p0 = pl.spi[k0].pp0 + (long long)ch * g.W;
    kbeg = ch == 0 ? k0 : first_at(pl.spi, k0, k1, p0);
    kend = ch + 1 == g.nch ? k1 : first_at(pl.spi, kbeg, k1, p0 + g.W);
    if (same) kbeg = max(kbeg, bra);
    return kbeg < kend;
}

// Superset test of prim_radius and the image search for one primitive
// quartet, without a logarithm or a division: ln of the magnitude bound
// 2 pi^{5/2} 2^{-1/2} B_i B_j over the threshold is a sum (s = lb_i + lb_j +
// const, > 0), 1 - c_w <= 1 and ln(1 + 2 alpha_w r) <= its largest value over
// the plan (Lc), so the sphere drawn here contains the exact one.
template <int L>
__device__ __forceinline__ bool prim_maybe(const PlanDev &pl, const float4 &b, const float4 &k, float s, float Lc, float r1min)
{
    const float inv = b.w + k.w + pl.inv_omega2f;  // 1 / alpha_w
    float X[3] = {b.x - k.x, b.y - k.y, b.z - k.z};
    if (pl.orth == 2) {
        // diagonal lattice: nearest image by adding and subtracting 1.5 * 2^23
#pragma unroll
        for (int a = 0; a < 3; ++a) X[a] = fmaf(-(fmaf(X[a], pl.Finvf[4 * a], 12582912.0f) - 12582912.0f), pl.Lf[4 * a], X[a]);
    } else {
        float f[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) f[a] = rintf(pl.Finvf[3 * a] * X[0] + pl.Finvf[3 * a + 1] * X[1] + pl.Finvf[3 * a + 2] * X[2]);
#pragma unroll
        for (int a = 0; a < 3; ++a) X[a] -= f[0] * pl.Lf[a] + f[1] * pl.Lf[3 + a] + f[2] * pl.Lf[6 + a];
    }
    const float x2 = X[0] * X[0] + X[1] * X[1] + X[2] * X[2];
    if (L == 0 && pl.orth) return x2 < 1.001f * s * inv;
    const float r = 1.0005f * fsqrt_fast((s + Lc) * inv) + (L > 0 ? 0.5f + 0.25f * L : 0.0f);
    // a skewed cell's rounded image may not be the nearest one
    return x2 < r * r || (!pl.orth && r1min - fsqrt_fast(x2) < r);
}

// Evaluate count (<= 32) queued primitive quartets from ring position qd on,
// one per lane, and add the lanes of each image quartet into its block Vs[slot].
// A ring entry holds the slot, the positions i and j of the bra and ket
// primitive pairs in their images (first ones: bra0(slot), ket0(slot)) and a
// group: the entries of one slot and group are adjacent.  several: a slot may
// come with more than one group, and (LO > 0) the blocks are sums with their
// rounding errors LO elements further on.
template <int LA, int LB, int LC, int LD, typename T, int RING, bool SHARE, int LO, class BraFn, class KetFn>
__device__ __forceinline__ void eval_terms(const PlanDev &pl, const unsigned *ring, unsigned qd, unsigned count, BraFn bra0, KetFn ket0,
                                           bool several, T *Vs, Tally &tl, unsigned &used, bool share = false,
                                           ImgShare<LA + LB + LC + LD, T> *img = nullptr)
{
    constexpr int NV = ncart(LA) * ncart(LB) * ncart(LC) * ncart(LD), L = LA + LB + LC + LD;
    const int lane = threadIdx.x & 31;
    const bool on = lane < count;
    unsigned key = 0xffffff80u + lane;  // a segment of its own (group 511 is not used)
    T V[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) V[q] = T(0);
    if constexpr (SHARE) {
        PrimE<LA, LB, T> bp;
        PrimE<LC, LD, T> kp;
        PpiF bf, kf;
        PrimGeo<T> g;
        bool act = false;
        if (on) {
            const unsigned it = ring[(qd + lane) & (RING - 1)];
            key = it & 0xff80007fu;
            load_prim<LA, LB, T>(pl, bra0(it & 127u) + (int)((it >> 7) & 255u), bp, bf);
            load_prim<LC, LD, T>(pl, ket0(it & 127u) + (int)((it >> 15) & 255u), kp, kf);
            ++tl.brap;
            ++tl.ketp;
            act = prim_geo<L, T>(pl, bp.x, bf, kp.x, kf, g, tl);
            ++used;
        }
        T Rs[(L + 1) * (L + 1) * (L + 1)];
#pragma unroll
        for (int q = 0; q < (L + 1) * (L + 1) * (L + 1); ++q) Rs[q] = T(0);
        if (share) {
            int n = 0;
            if (act)
#pragma unroll 1
                for (int c = next_image(pl, g, 0, tl); c < pl.nr1; c = next_image(pl, g, c + 1, tl)) ++n;
            tl.img += n;
            act = n > 0;
            shared_images<L, T>(pl, g, n, *img, Rs);
        } else if (act) {
            act = all_images<L, T>(pl, g, Rs, tl);
        }
        if (act) {
            ++tl.term;
            contract<LA, LB, LC, LD, T>(bp, kp, Rs, V);
        }
    } else if (on) {
        const unsigned it = ring[(qd + lane) & (RING - 1)];
        key = it & 0xff80007fu;
        PrimE<LA, LB, T> bp;
        PrimE<LC, LD, T> kp;
        PpiF bf, kf;
        load_prim<LA, LB, T>(pl, bra0(it & 127u) + (int)((it >> 7) & 255u), bp, bf);
        load_prim<LC, LD, T>(pl, ket0(it & 127u) + (int)((it >> 15) & 255u), kp, kf);
        ++tl.brap;
        ++tl.ketp;
        prim_term<LA, LB, LC, LD, T>(pl, bp, bf, kp, kf, V, tl);
        ++used;
    }
    __syncwarp();
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned ok = __shfl_down_sync(0xffffffffu, key, o);
        const bool add = lane + o < 32 && ok == key;
        if (!__any_sync(0xffffffffu, add)) break;
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const T t = __shfl_down_sync(0xffffffffu, V[q], o);
            if (add) V[q] += t;
        }
    }
    const unsigned prev = __shfl_up_sync(0xffffffffu, key, 1);
    const bool head = on && (lane == 0 || prev != key);
    T *dst = Vs + (head ? key & 127u : 0u) * NV;
    const auto add_compensated = [&] {  // two-sum
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            const T h = dst[q], t = h + V[q], b = t - h;
            dst[q] = t;
            dst[LO + q] += (h - (t - b)) + (V[q] - b);
        }
    };
    if (!several) {
        if (head)
#pragma unroll
            for (int q = 0; q < NV; ++q) dst[q] += V[q];
    } else {
        // one slot can head several segments here: one after another
        const unsigned m = __match_any_sync(0xffffffffu, head ? (key & 127u) : 128u + lane);
        const int rank = __popc(m & ((1u << lane) - 1u));
#pragma unroll 1
        for (int rr = 0; __any_sync(0xffffffffu, head && rank >= rr); ++rr) {
            if (head && rank == rr) {
                if constexpr (LO > 0) {
                    add_compensated();
                } else {
#pragma unroll
                    for (int q = 0; q < NV; ++q) dst[q] += V[q];
                }
            }
            __syncwarp();
        }
    }
    __syncwarp();
}

// Warp-per-bra tile kernel.  Block = 4 warps, each with a bra and a range of
// kets (TileMap).  mode and the FP64 list as in k_real.
//   1. 32 kets at a time are tested (block bound, quartet bound, precision
//      policy); the ones that pass are queued until SL of them are held.
//   2. Their primitive pairs are laid out one per lane; each lane marks the
//      bra primitives whose quartet may have a term (prim_maybe, kBraChunk at
//      a time) and the marked quartets go into a ring ordered by ket.
//   3. Whenever 32 are queued they are evaluated, one per lane, and the lanes
//      of one ket are summed (segmented reduction) into its shared block.
//   4. The SL blocks are digested, one ket per lane.
// The work of a warp is bounded by its primitive quartets, not its kets: cut
// by kets alone, the (ss|ss) launch of a 5-molecule box waited for one warp
// (36 x 36 primitive quartets, up to 20 images each) for 80% of its 63 ms.
// Against one ket's primitives per step and kets alone, when this split came
// in: mixed J+K build of 5 water molecules 77 -> 29 ms, of 31 (reciprocal cache)
// 223 -> 193 ms, of 64 962 -> 801 ms; FP64 build of 6 molecules 325 -> 131 ms
// (with what followed 22.9, 176, 713 and 85.6 ms).  Bound by
// instruction issue (0.53 a clock and scheduler, 17 of 32 lanes active).
// The stages have very different pass rates (water box, (ss|ss): 17% of the
// pairs, then 1.3 terms out of 6.7 screened primitive quartets per pair), so
// each stage refills the warp; with one ket's primitives per step and the
// screening, the terms and the digestion in one loop body about a tenth of
// the lanes were active.
// The sums of a deep bra are compensated in single precision: rounded at every
// batch, the K of a diamond cell with every quartet in FP32 was 1.2e-7 off
// (rms) against 0.7e-7 now and 0.95e-7 with the terms of a ket primitive summed
// in a lane.
// Counters (cnt, one precision's base): [0] image quartets evaluated, [4]
// algorithmic flops, [8] screening and bookkeeping flops, [12] primitive
// quartets evaluated and [14] lane slots offered to them (their ratio is the
// lane occupancy).
template <int LA, int LB, int LC, int LD, typename T>
__global__ void __launch_bounds__(32 * kWarpsPerBlock, tile_blocks<T>(LA + LB + LC + LD)) k_real_w(PlanDev pl, TileMap map, int k0, int k1, int same, int mode, double tau,
                                                                const T *__restrict__ Dp, const T *__restrict__ dmax,
                                                                double *__restrict__ X, double *__restrict__ Y,
                                                                unsigned long long *__restrict__ cnt, QuartetList big,
                                                                unsigned *__restrict__ nbig, unsigned cap, unsigned *__restrict__ ovf)
{
    constexpr int NA = ncart(LA), NB = ncart(LB), NC = ncart(LC), ND = ncart(LD), NV = NA * NB * NC * ND;
    constexpr int L = LA + LB + LC + LD;
    constexpr int SL = BatchShape<NV, T>::SL, KQ = BatchShape<NV, T>::KQ, LO = BatchShape<NV, T>::LO;
    __shared__ unsigned ring_s[kWarpsPerBlock][kTermRing];
    __shared__ int kq_s[kWarpsPerBlock][KQ], pp0_s[kWarpsPerBlock][SL];
    __shared__ T V_s[kWarpsPerBlock][SL * NV];
    __shared__ ImgShare<L, T> img_s[kWarpsPerBlock];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int bra, kbeg, kend;
    // whole warps return; no block-wide barrier below
    if (!tile_of(pl, map, (long long)blockIdx.x * kWarpsPerBlock + wid, k0, k1, same, bra, kbeg, kend)) return;
    unsigned *ring = ring_s[wid];
    int *kq = kq_s[wid], *kpp0 = pp0_s[wid];
    T *Vs = V_s[wid];
    const SpiRec sb = pl.spi[bra];
    const int n = pl.nbf;
    const int aoI = pl.shells[sb.I].ao, aoJ = pl.shells[sb.J].ao;
    // A bra of many primitives adds up to 65536 terms to a block, 32 at a time:
    // in single precision its sums carry their rounding errors along, in the
    // upper half of the slots (its batches are full with half as many kets).
    const bool deep = LO > 0 && sb.npp > kBraChunk;
    const int nslot = deep ? SL / 2 : SL;
    T Dij[NA * NB];
    Acc<T> jb[NA * NB];
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
        for (int b = 0; b < NB; ++b) Dij[a * NB + b] = __ldg(Dp + (size_t)(aoI + a) * n + aoJ + b);
    const float tauf = (float)tau;
    // constants of prim_maybe
    const float lbc = 3.2094f - pl.log_ewald_R;  // ln(2 pi^{5/2} / sqrt 2) + 1e-3
    const float r1min = pl.nr1 > 1 ? pl.r1f[7] : 1e30f;
    const bool share = pl.img_share;  // several images per primitive quartet
    const float Lc = radius_correction<L>(pl, 2.0f * pl.lb_max + lbc);
    const float Lq = radius_correction<L>(pl, 2.0f * pl.ls_max + lbc);  // the same for whole images
    const float4 bq = __ldg(pl.spq + bra), br = __ldg(pl.spr + bra);
    const bool policy = sizeof(T) == 4 && mode;
    const float dall = policy ? (float)__ldg(dmax + (size_t)pl.nshell * pl.nshell) : 0.0f;
    Tally tl;
    unsigned used = 0, slots = 0;  // primitive quartets evaluated and lane slots offered
    unsigned nq = 0, kn = 0, kd = 0;

    unsigned qn = 0, qd = 0;
    // evaluate the next count queued primitive quartets
    auto eval = [&](unsigned count) {
        eval_terms<LA, LB, LC, LD, T, kTermRing, ImgShare<L, T>::on, LO>(
            pl, ring, qd, count, [&](unsigned) { return sb.pp0; }, [&](unsigned slot) { return kpp0[slot]; }, sb.npp > kBraChunk, Vs, tl,
            used, share, &img_s[wid]);
        slots += lane == 0 ? 32u : 0u;
        qd += count;
    };
    // screen, evaluate and digest the next count queued kets
    auto process = [&](int count) {
#pragma unroll 1
        for (int q = lane; q < (deep ? SL : count) * NV; q += 32) Vs[q] = T(0);
        unsigned grp = 0;
#pragma unroll 1
        for (int s0 = 0; s0 < count; s0 += 32) {
            int np = 0;
            if (s0 + lane < count) {
                const int kt = kq[(kd + s0 + lane) & (KQ - 1)];
                const int first = __float_as_int(__ldg(&pl.spr[kt].w));
                np = __float_as_int(__ldg(&pl.spr[kt + 1].w)) - first;
                kpp0[s0 + lane] = first;
            }
            int incl = np;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += t;
            }
            const int total = __shfl_sync(0xffffffffu, incl, 31);
            const int excl = incl - np;
            __syncwarp();
            int e0 = 0, ic = 0, src = 0, j = 0;
            float4 kv = make_float4(0.f, 0.f, 0.f, 0.f);
            float ks = -1e30f;
#pragma unroll 1
            while (e0 < total) {
                if (ic == 0) {
                    const int e = e0 + lane;
                    // owner: the first lane whose inclusive prefix exceeds e
                    int own = 0;
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1) {
                        const int v = __shfl_sync(0xffffffffu, incl, own + step - 1);
                        if (v <= e) own += step;
                    }
                    src = s0 + own;
                    j = e - __shfl_sync(0xffffffffu, excl, own);
                    ks = -1e30f;
                    if (e < total) {
                        const int kpp = kpp0[src] + j;
                        kv = __ldg(pl.pps + kpp);
                        ks = __ldg(pl.pplb + kpp) + lbc;
                    }
                }
                unsigned mask = 0;
                const int ie = min(kBraChunk, sb.npp - ic);
                // bra primitives in descending order of their bound: the first one
                // below the magnitude threshold ends the loop
                int i = 0;
                float lb = __ldg(pl.pplb + sb.pp0 + ic);
                float4 bv = __ldg(pl.pps + sb.pp0 + ic);
#pragma unroll 1
                for (; i < ie; ++i) {
                    const float s = ks + lb;
                    if (!(s > 0.0f)) break;
                    ++tl.screen;
                    // the next one is on its way while this one is tested
                    const float4 cur = bv;
                    const int nx = sb.pp0 + ic + min(i + 1, ie - 1);
                    lb = __ldg(pl.pplb + nx);
                    bv = __ldg(pl.pps + nx);
                    if (prim_maybe<L>(pl, cur, kv, s, Lc, r1min)) mask |= 1u << i;
                }
                const int cm = __popc(mask);
                int pre = cm;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int t = __shfl_up_sync(0xffffffffu, pre, o);
                    if (lane >= o) pre += t;
                }
                unsigned pos = qn + pre - cm;
                const unsigned base = (unsigned)src | ((unsigned)ic << 7) | ((unsigned)j << 15) | (grp << 23);
#pragma unroll 1
                while (mask) {
                    const unsigned b = __ffs(mask) - 1;
                    mask &= mask - 1;
                    ring[pos++ & (kTermRing - 1)] = base + (b << 7);
                }
                qn += __shfl_sync(0xffffffffu, pre, 31);
                // the quartets of one ket stay adjacent in the ring unless the bra
                // takes several rounds; then each round is a group of its own
                if (sb.npp > kBraChunk) grp = grp == 510u ? 0u : grp + 1u;
                ic += kBraChunk;
                if (ic >= sb.npp || !__any_sync(0xffffffffu, i == kBraChunk)) {
                    ic = 0;
                    e0 += 32;
                }
                __syncwarp();
                const unsigned lim = e0 < total || s0 + 32 < count ? 32u : 1u;
#pragma unroll 1
                while (qn - qd >= lim) eval(min(32u, qn - qd));
            }
        }
        __syncwarp();
#pragma unroll 1
        for (int sl = lane; sl < count; sl += 32) {
            T V[NV];
            bool any = false;
#pragma unroll
            for (int q = 0; q < NV; ++q) {
                V[q] = Vs[sl * NV + q];
                if (LO > 0 && deep) V[q] += Vs[LO + sl * NV + q];
                any = any || V[q] != T(0);
            }
            if (any) {
                const int kt = kq[(kd + sl) & (KQ - 1)];
                const int4 kd4 = __ldg(pl.spd + kt);
                const T w = T(sb.w) * T(__int_as_float(kd4.z)) * ((same && kt == bra) ? T(0.5) : T(1));
                digest<LA, LB, LC, LD, T>(n, aoI, aoJ, kd4.x, kd4.y, V, w, Dp, Dij, jb, X, Y);
            }
            ++tl.quart;
        }
        kd += count;
        __syncwarp();
    };

    // 32 blocks of 32 kets at a time: one block bound per lane, then the kets
    // of the blocks that may be reached
#pragma unroll 1
    for (int g0 = kbeg >> 5; g0 * 32 < kend; g0 += 32) {
        unsigned bm = __ballot_sync(0xffffffffu, (g0 + lane) * 32 < kend && block_reaches<L>(pl, sb, g0 + lane));
        const bool last = (g0 + 32) * 32 >= kend;
        do {
            const int kt = bm ? (g0 + __ffs(bm) - 1) * 32 + lane : kend;
            bm &= bm - 1;
            bool valid = kt >= kbeg && kt < kend;
            if (valid) {
                float eb;
                bool brief;
                valid = pair_reaches<L>(pl, bq, br, __ldg(pl.spq + kt), __ldg(pl.spr + kt), Lq, eb, brief);
                // large quartets (and short [c_w, 1] intervals) go to the FP64 list
                if (policy && valid && (eb * dall >= tauf || brief))
                    valid = !list_quartet(pl, bra, kt, tauf, dmax, big, nbig, cap, ovf);
            }
            const unsigned vmask = __ballot_sync(0xffffffffu, valid);
            nq += lane == 0 ? __popc(vmask) : 0;
            if (valid) kq[(kn + __popc(vmask & ((1u << lane) - 1u))) & (KQ - 1)] = kt;
            kn += __popc(vmask);
            __syncwarp();
            const unsigned lim = last && !bm ? 1u : (unsigned)nslot;
#pragma unroll 1
            while (kn - kd >= lim) process((int)min((unsigned)nslot, kn - kd));
        } while (bm);
    }
    // bra-side Coulomb: one atomic per element for the warp
#pragma unroll
    for (int a = 0; a < NA; ++a)
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            const double v = warp_sum(jb[a * NB + b].value());
            if (lane == 0 && v != 0.0) atomicAdd(X + (size_t)(aoI + a) * n + aoJ + b, v);
        }
    unsigned long long fl = tally_alg<LA, LB, LC, LD>(tl), fs = tally_screen<LA, LB, LC, LD>(tl), u64 = used, s64 = slots;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        fl += __shfl_xor_sync(0xffffffffu, fl, o);
        fs += __shfl_xor_sync(0xffffffffu, fs, o);
        u64 += __shfl_xor_sync(0xffffffffu, u64, o);
        s64 += __shfl_xor_sync(0xffffffffu, s64, o);
    }
    if (lane == 0) {
        if (nq) atomicAdd(cnt, (unsigned long long)nq);
        if (fl) atomicAdd(cnt + 4, fl);
        if (fs) atomicAdd(cnt + 8, fs);
        if (u64) atomicAdd(cnt + 12, u64);
        if (s64) atomicAdd(cnt + 14, s64);
    }
}

// Pair-queue tile kernel (third family for s and p class pairs): as the
// lane-per-bra kernel, a warp holds 32 consecutive bras and walks the kets of
// its chunk; but every (bra, ket) image pair that passes the quartet-level
// bound goes into a per-warp queue in shared memory, and the queue is
// evaluated 32 pairs at a time, one pair per lane, so lanes whose own bra
// misses a ket do not idle while the others work.  The pairs of one batch
// are ordered by ket, so the ket-side Coulomb term is summed over the lanes
// of a ket by a segmented warp reduction; the bra-side term is added to the
// bra's FP64 partial in shared memory; exchange as in the other kernels.
template <int LA, int LB, int LC, int LD, typename T>
__global__ void __launch_bounds__(kRealThreads) k_real_q(PlanDev pl, int b0, int b1, int k0, int k1, int same, int kchunk, int mode,
                                                          double tau, const T *__restrict__ Dp, const T *__restrict__ dmax,
                                                          double *__restrict__ X, double *__restrict__ Y,
                                                          unsigned long long *__restrict__ cnt, QuartetList big,
                                                          unsigned *__restrict__ nbig, unsigned cap, unsigned *__restrict__ ovf)
{
    constexpr int NA = ncart(LA), NB = ncart(LB), NC = ncart(LC), ND = ncart(LD), NV = NA * NB * NC * ND;
    constexpr int L = LA + LB + LC + LD;
    constexpr int NW = kRealThreads / 32;
    __shared__ int qall[NW][64];
    __shared__ double jball[NW][32 * NA * NB];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int *qb = qall[wid];
    double *jbs = jball[wid];
    const int wbra0 = b0 + blockIdx.x * kRealThreads + 32 * wid;  // the warp's first bra
    const int bra = wbra0 + lane;
    int kbeg = k0 + blockIdx.y * kchunk;
    const int kend = min(k1, kbeg + kchunk);
    if (same) kbeg = max(kbeg, wbra0);
    if (kbeg >= kend || wbra0 >= b1) return;  // whole warp; no block-wide barrier below
    const bool act = bra < b1;
    const SpiRec sb = pl.spi[act ? bra : b0];
    const int n = pl.nbf, nsh = pl.nshell;
#pragma unroll
    for (int q = 0; q < NA * NB; ++q) jbs[lane * NA * NB + q] = 0.0;
    __syncwarp();
    const float tauf = (float)tau;
    unsigned nq = 0, qn = 0, qd = 0;
    Tally tl;
    // evaluate `count` queued pairs, one per lane
    auto process = [&](unsigned count) {
        const bool on = lane < count;
        int o = 0, kt = 0;
        if (on) {
            const int item = qb[(qd + lane) & 63];
            o = item & 31;
            kt = item >> 5;
        }
        T V[NV];
#pragma unroll
        for (int q = 0; q < NV; ++q) V[q] = T(0);
        SpiRec sbo{}, sk{};
        if (on) {
            sbo = pl.spi[wbra0 + o];
            sk = pl.spi[kt];
            quartet_block<LA, LB, LC, LD, T>(pl, sbo, sk, V, tl);
            ++tl.quart;
            ++nq;
        }
        const T w = on ? T(sbo.w) * T(sk.w) * ((same && kt == wbra0 + o) ? T(0.5) : T(1)) : T(0);
        const int aoI = pl.shells[on ? sbo.I : sb.I].ao, aoJ = pl.shells[on ? sbo.J : sb.J].ao;
        const int aoK = pl.shells[on ? sk.I : sb.I].ao, aoL = pl.shells[on ? sk.J : sb.J].ao;
        auto Dd = [&](int r, int c) { return __ldg(Dp + (size_t)r * n + c); };
        // bra-side Coulomb: the bra's FP64 partial in shared memory
        if (on) {
#pragma unroll
            for (int ab = 0; ab < NA * NB; ++ab) {
                T s2 = T(0);
#pragma unroll
                for (int c = 0; c < NC; ++c)
#pragma unroll
                    for (int d = 0; d < ND; ++d) s2 += V[ab * NC * ND + c * ND + d] * Dd(aoK + c, aoL + d);
                if (s2 != T(0)) atomicAdd(jbs + o * NA * NB + ab, to_f64(T(2) * w * s2));
            }
        }
        // ket-side Coulomb: segmented sum over the lanes of one ket (the batch is ordered by ket)
        const int key = on ? kt : -1 - lane;
#pragma unroll
        for (int cd = 0; cd < NC * ND; ++cd) {
            T s2 = T(0);
            if (on) {
                T Dij[NA * NB];
#pragma unroll
                for (int a = 0; a < NA; ++a)
#pragma unroll
                    for (int b = 0; b < NB; ++b) Dij[a * NB + b] = Dd(aoI + a, aoJ + b);
#pragma unroll
                for (int ab = 0; ab < NA * NB; ++ab) s2 += V[ab * NC * ND + cd] * Dij[ab];
                s2 *= T(2) * w;
            }
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const int ok2 = __shfl_down_sync(0xffffffffu, key, off);
                const T t2 = __shfl_down_sync(0xffffffffu, s2, off);
                if (lane + off < 32 && ok2 == key) s2 += t2;
            }
            const int prevk = __shfl_up_sync(0xffffffffu, key, 1);
            if (on && (lane == 0 || prevk != key) && s2 != T(0))
                atomicAdd(X + (size_t)(aoK + cd / ND) * n + aoL + cd % ND, to_f64(s2));
        }
        // exchange: the four index assignments of the orbit (the other four are transposes)
        if (on && Y) {
#pragma unroll
            for (int a = 0; a < NA; ++a)
#pragma unroll
                for (int d = 0; d < ND; ++d) {
                    T s2 = T(0);
#pragma unroll
                    for (int b = 0; b < NB; ++b)
#pragma unroll
                        for (int c = 0; c < NC; ++c) s2 += V[((a * NB + b) * NC + c) * ND + d] * Dd(aoJ + b, aoK + c);
                    atomicAdd(Y + (size_t)(aoI + a) * n + aoL + d, to_f64(w * s2));
                }
#pragma unroll
            for (int b = 0; b < NB; ++b)
#pragma unroll
                for (int d = 0; d < ND; ++d) {
                    T s2 = T(0);
#pragma unroll
                    for (int a = 0; a < NA; ++a)
#pragma unroll
                        for (int c = 0; c < NC; ++c) s2 += V[((a * NB + b) * NC + c) * ND + d] * Dd(aoI + a, aoK + c);
                    atomicAdd(Y + (size_t)(aoJ + b) * n + aoL + d, to_f64(w * s2));
                }
#pragma unroll
            for (int a = 0; a < NA; ++a)
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    T s2 = T(0);
#pragma unroll
                    for (int b = 0; b < NB; ++b)
#pragma unroll
                        for (int d = 0; d < ND; ++d) s2 += V[((a * NB + b) * NC + c) * ND + d] * Dd(aoJ + b, aoL + d);
                    atomicAdd(Y + (size_t)(aoI + a) * n + aoK + c, to_f64(w * s2));
                }
#pragma unroll
            for (int b = 0; b < NB; ++b)
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    T s2 = T(0);
#pragma unroll
                    for (int a = 0; a < NA; ++a)
#pragma unroll
                        for (int d = 0; d < ND; ++d) s2 += V[((a * NB + b) * NC + c) * ND + d] * Dd(aoI + a, aoL + d);
                    atomicAdd(Y + (size_t)(aoJ + b) * n + aoK + c, to_f64(w * s2));
                }
        }
        qd += count;
        __syncwarp();
    };
    for (int kt = kbeg; kt < kend; ++kt) {
        // one bound per block of 32 kets for the whole warp first
        if (kt == kbeg || (kt & 31) == 0) {
            if (!__any_sync(0xffffffffu, act && block_reaches<L>(pl, sb, kt >> 5))) {
                kt = min(kend, ((kt >> 5) + 1) << 5) - 1;
                continue;
            }
        }
        const SpiRec sk = pl.spi[kt];
        bool valid = act && (!same || kt >= bra) && quartet_reaches<L>(pl, sb, sk);
        if (sizeof(T) == 4 && valid && mode) {
            const float dm = quartet_dmax(reinterpret_cast<const float *>(dmax), nsh, sb, sk);
            const float est = quartet_estimate_bound(pl, sb, sk) * dm >= tauf ? quartet_estimate(pl, sb, sk) * dm : 0.0f;
            const float ipq = frcp_fast(sb.pmin) + frcp_fast(sk.pmin);
            if (est >= tauf || ipq > 0.7225f * (ipq + pl.inv_omega2f)) {
                const unsigned slot = atomicAdd(nbig, 1u);
                if (slot < cap) {
                    big.put(slot, bra, kt);
                    valid = false;
                } else {
                    atomicAdd(ovf, 1u);
                }
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, valid);
        if (!m) continue;
        if (valid) qb[(qn + __popc(m & ((1u << lane) - 1u))) & 63] = (kt << 5) | lane;
        qn += __popc(m);
        __syncwarp();
        if (qn - qd >= 32) process(32);
    }
    while (qn > qd) process(min(32u, qn - qd));
    // the bra-side Coulomb partials of the warp's bras
    if (act) {
        const int aoI = pl.shells[sb.I].ao, aoJ = pl.shells[sb.J].ao;
#pragma unroll
        for (int a = 0; a < NA; ++a)
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                const double v = jbs[lane * NA * NB + a * NB + b];
                if (v != 0.0) atomicAdd(X + (size_t)(aoI + a) * n + aoJ + b, v);
            }
    }
    unsigned long long fl = tally_alg<LA, LB, LC, LD>(tl), fs = tally_screen<LA, LB, LC, LD>(tl);
    unsigned tot = nq;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        tot += __shfl_xor_sync(0xffffffffu, tot, o);
        fl += __shfl_xor_sync(0xffffffffu, fl, o);
        fs += __shfl_xor_sync(0xffffffffu, fs, o);
    }
    if (lane == 0) {
        if (tot) atomicAdd(cnt, (unsigned long long)tot);
        if (fl) atomicAdd(cnt + 4, fl);
        if (fs) atomicAdd(cnt + 8, fs);
    }
}

// FP64 pass over the listed large quartets.  A warp takes up to SL entries at
// a time (fewer when the list is too short for eight such turns per warp: with
// one turn, its heaviest entries side by side in one warp, a short list took
// twice as long): their
// primitive quartets are laid out one per lane and screened, the ones that pass
// go into the ring of k_real_w and are evaluated 32 at a time into the entries'
// blocks, which are digested one entry per lane.  With one entry per warp the
// last batch of an entry was half empty (33 primitive quartets on average for
// (ss|pp) of the 64-water box: two batches) and one lane digested alone.
// Counters as k_real_w (cnt points at the FP64 slots).
template <int LA, int LB, int LC, int LD>
__global__ void __launch_bounds__(32 * kWarpsPerBlock, LA + LB + LC + LD <= 3 ? 3 : 2) k_real_list_w(PlanDev pl, QuartetList big,
                                                                        const unsigned *__restrict__ nbig, unsigned cap, int same,
                                                                        const double *__restrict__ Dp, double *__restrict__ X,
                                                                        double *__restrict__ Y, unsigned long long *__restrict__ cnt)
{
    constexpr int NA = ncart(LA), NB = ncart(LB), NC = ncart(LC), ND = ncart(LD), NV = NA * NB * NC * ND;
    constexpr int L = LA + LB + LC + LD;
    constexpr int SL = NV <= 18 ? 32 : 16;
    __shared__ unsigned ring_s[kWarpsPerBlock][kListRing];
    __shared__ int bpp0_s[kWarpsPerBlock][SL], kpp0_s[kWarpsPerBlock][SL];
    __shared__ double V_s[kWarpsPerBlock][SL * NV];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned *ring = ring_s[wid];
    int *bpp0 = bpp0_s[wid], *kpp0 = kpp0_s[wid];
    double *Vs = V_s[wid];
    const unsigned total = min(*nbig, cap), nwarps = gridDim.x * kWarpsPerBlock, warp = blockIdx.x * kWarpsPerBlock + wid;
    const unsigned per = min((unsigned)SL, max(1u, total / (8 * nwarps)));
    const int n = pl.nbf;
    const float lbc = 3.2094f - pl.log_ewald_R;  // ln(2 pi^{5/2} / sqrt 2) + 1e-3
    const float r1min = pl.nr1 > 1 ? pl.r1f[7] : 1e30f;
    const float Lc = radius_correction<L>(pl, 2.0f * pl.lb_max + lbc);
    Tally tl;
    unsigned used = 0, slots = 0, done = 0;
#pragma unroll 1
    for (unsigned base = warp * per; base < total; base += nwarps * per) {
        const int cnt_e = (int)min(per, total - base);
        int nk = 1, nterm = 0;
        if (lane < cnt_e) {
            const int2 pr = big.get(base + lane);
            const int b0 = __float_as_int(__ldg(&pl.spr[pr.x].w)), k0 = __float_as_int(__ldg(&pl.spr[pr.y].w));
            nk = __float_as_int(__ldg(&pl.spr[pr.y + 1].w)) - k0;
            nterm = (__float_as_int(__ldg(&pl.spr[pr.x + 1].w)) - b0) * nk;
            bpp0[lane] = b0;
            kpp0[lane] = k0;
        }
        for (int q = lane; q < cnt_e * NV; q += 32) Vs[q] = 0.0;
        int incl = nterm;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += t;
        }
        const int all = __shfl_sync(0xffffffffu, incl, 31), excl = incl - nterm;
        __syncwarp();
        unsigned qn = 0, qd = 0;
#pragma unroll 1
        for (int e0 = 0; e0 < all; e0 += 32) {
            const int e = e0 + lane;
            // owner: the first lane whose inclusive prefix exceeds e
            int own = 0;
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
                const int v = __shfl_sync(0xffffffffu, incl, own + step - 1);
                if (v <= e) own += step;
            }
            const int t = e - __shfl_sync(0xffffffffu, excl, own), k = __shfl_sync(0xffffffffu, nk, own);
            const int i = t / k, j = t - i * k;
            bool pass = false;
            if (e < all) {
                const int ib = bpp0[own] + i, ik = kpp0[own] + j;
                const float s = __ldg(pl.pplb + ib) + __ldg(pl.pplb + ik) + lbc;
                ++tl.screen;
                pass = s > 0.0f && prim_maybe<L>(pl, __ldg(pl.pps + ib), __ldg(pl.pps + ik), s, Lc, r1min);
            }
            const unsigned m = __ballot_sync(0xffffffffu, pass);
            if (pass)
                ring[(qn + __popc(m & ((1u << lane) - 1u))) & (kListRing - 1)] = (unsigned)own | ((unsigned)i << 7) | ((unsigned)j << 15);
            qn += __popc(m);
            __syncwarp();
            const unsigned lim = e0 + 32 < all ? 32u : 1u;
#pragma unroll 1
            while (qn - qd >= lim) {
                const unsigned count = min(32u, qn - qd);
                eval_terms<LA, LB, LC, LD, double, kListRing, false, 0>(
                    pl, ring, qd, count, [&](unsigned s) { return bpp0[s]; }, [&](unsigned s) { return kpp0[s]; }, false, Vs, tl, used);
                qd += count;
                slots += lane == 0 ? 32u : 0u;
            }
        }
        __syncwarp();
        if (lane < cnt_e) {
            const int2 pr = big.get(base + lane);
            const int4 b4 = __ldg(pl.spd + pr.x), k4 = __ldg(pl.spd + pr.y);
            double V[NV], Dij[NA * NB];
            Acc<double> jb[NA * NB];
#pragma unroll
            for (int q = 0; q < NV; ++q) V[q] = Vs[lane * NV + q];
#pragma unroll
            for (int a = 0; a < NA; ++a)
#pragma unroll
                for (int b = 0; b < NB; ++b) Dij[a * NB + b] = __ldg(Dp + (size_t)(b4.x + a) * n + b4.y + b);
            const double w = (double)__int_as_float(b4.z) * (double)__int_as_float(k4.z) * ((same && pr.x == pr.y) ? 0.5 : 1.0);
            digest<LA, LB, LC, LD, double>(n, b4.x, b4.y, k4.x, k4.y, V, w, Dp, Dij, jb, X, Y);
#pragma unroll
            for (int a = 0; a < NA; ++a)
#pragma unroll
                for (int b = 0; b < NB; ++b) atomicAdd(X + (size_t)(b4.x + a) * n + b4.y + b, jb[a * NB + b].value());
            ++tl.quart;
            ++done;
        }
        __syncwarp();
    }
    unsigned long long fl = tally_alg<LA, LB, LC, LD>(tl), fs = tally_screen<LA, LB, LC, LD>(tl), u64 = used, s64 = slots, d64 = done;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        fl += __shfl_xor_sync(0xffffffffu, fl, o);
        fs += __shfl_xor_sync(0xffffffffu, fs, o);
        u64 += __shfl_xor_sync(0xffffffffu, u64, o);
        s64 += __shfl_xor_sync(0xffffffffu, s64, o);
        d64 += __shfl_xor_sync(0xffffffffu, d64, o);
    }
    if (lane == 0) {
        if (d64) atomicAdd(cnt, d64);
        if (fl) atomicAdd(cnt + 4, fl);
        if (fs) atomicAdd(cnt + 8, fs);
        if (u64) atomicAdd(cnt + 12, u64);
        if (s64) atomicAdd(cnt + 14, s64);
    }
}

}  // namespace jk
