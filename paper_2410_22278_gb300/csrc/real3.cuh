// Warp-cooperative real-space quartet kernels for the class pairs whose
// Cartesian block is too large for one lane (more than 36 elements: p and d
// shells, up to 1296 elements and a Hermite table of 165).
//
// One warp evaluates one image quartet:
//   1. its primitive quartets are screened 32 at a time;
//   2. the ones that pass are taken four at a time, eight lanes each (the last
//      two or one with 16 or 32 lanes): the lanes share the lattice images (seeds and R table in registers, then a
//      sum over the eight lanes) -- a small cell has 10 to 60 images per
//      primitive quartet, a large one a few;
//   3. for each of the four, the R table and the E tables of both pairs go to
//      shared memory and all 32 lanes form the Cartesian block from them,
//      W[t][cd] = sum_s E_cd,s R_{t+s}, V[ab][cd] += sum_t E_ab,t W[t][cd],
//      one output element per lane and step, V in shared memory;
//   4. the digestion sums one J or K element per lane.
// What bounds it: the serial chain of one quartet.  With one thread per
// quartet (the lane-per-bra kernel this replaces here) the whole chain ran in
// one lane with its arrays in local memory, and a class pair with a few
// thousand quartets kept a few warps busy for tens of milliseconds.  With the
// split of real2.cuh for the smaller classes, when they came in: FP64 build of
// a 20-function s/p/d cell 321 -> 7.2 ms, mixed build of one diamond cell 386 ->
// 26 ms, of 2 x 2 x 2 cells 745 -> 340 ms (with what followed 1.93, 16.3 and 299
// ms).  (pp|pp) of 16 water molecules: 0.20 ms, issue slots 15% busy, waiting
// on global and shared memory in turn; its FP64 list 1.4 ms.
#pragma once
#include "real2.cuh"

namespace jk {

template <int LA, int LB, int LC, int LD, typename T>
struct CoopShared {
    static constexpr int NA = ncart(LA), NB = ncart(LB), NC = ncart(LC), ND = ncart(LD);
    static constexpr int L = LA + LB + LC + LD, D = L + 1, LAB = LA + LB, LCD = LC + LD, NTA = LAB + 1, NTC = LCD + 1;
    static constexpr int NH = nherm(LAB), NAB = NA * NB, NCD = NC * ND;
    static constexpr int EA = (LA + 1) * (LB + 1) * NTA, EC = (LC + 1) * (LD + 1) * NTC;
    T V[NAB * NCD], W[NH * NCD], R[D * D * D], Ea[3 * EA], Ec[3 * EC];
    unsigned char tab[NH][3];            // (tx, ty, tz) of a Hermite index of the bra
    unsigned char tix[NTA * NTA * NTA];  // and back
    unsigned char eab[NAB][6], ecd[NCD][6];
};

// index tables of the shared structure (once per block of one warp)
template <int LA, int LB, int LC, int LD, typename T>
__device__ __forceinline__ void coop_init(CoopShared<LA, LB, LC, LD, T> &s)
{
    using S = CoopShared<LA, LB, LC, LD, T>;
    const int lane = threadIdx.x & 31;
    if (lane == 0) {
        int h = 0;
        for (int x = 0; x <= S::LAB; ++x)
            for (int y = 0; y <= S::LAB - x; ++y)
                for (int z = 0; z <= S::LAB - x - y; ++z, ++h) {
                    s.tab[h][0] = x;
                    s.tab[h][1] = y;
                    s.tab[h][2] = z;
                    s.tix[(x * S::NTA + y) * S::NTA + z] = h;
                }
    }
    for (int o = lane; o < S::NAB; o += 32)
        for (int k = 0; k < 3; ++k) {
            s.eab[o][k] = cexp(LA, o / S::NB, k);
            s.eab[o][3 + k] = cexp(LB, o % S::NB, k);
        }
    for (int o = lane; o < S::NCD; o += 32)
        for (int k = 0; k < 3; ++k) {
            s.ecd[o][k] = cexp(LC, o / S::ND, k);
            s.ecd[o][3 + k] = cexp(LD, o % S::ND, k);
        }
    __syncwarp();
}

// V (shared) = Cartesian block of the image quartet (sb, sk); false if it has
// no term.
template <int LA, int LB, int LC, int LD, typename T>
__device__ __forceinline__ bool coop_quartet(const PlanDev &pl, const SpiRec &sb, const SpiRec &sk, CoopShared<LA, LB, LC, LD, T> &s,
                                             Tally &tl)
{
    using S = CoopShared<LA, LB, LC, LD, T>;
    constexpr int L = S::L, D = S::D, NTA = S::NTA, NTC = S::NTC;
    const int lane = threadIdx.x & 31;
    const int nterm = sb.npp * sk.npp;
    const float4 *lat = reinterpret_cast<const float4 *>(pl.r1f);
    bool some = false;
    // Rounding errors of the block's sums over the primitive quartets, in
    // registers (single precision, up to four elements a lane: (pp|pp) and the
    // smaller blocks with d).  (pp|pp) adds up to 1296 terms; rounded at each,
    // the K of water boxes with every quartet in FP32 was 1.8e-7 off (rms, 5
    // molecules) against 1.1e-7 for sums over ket primitives by a tree.
    constexpr int NV = S::NAB * S::NCD, LV = (NV + 31) / 32;
    constexpr bool comp = sizeof(T) == 4 && LV <= 4;
    T lo[comp ? LV : 1];
#pragma unroll
    for (int k = 0; k < (comp ? LV : 1); ++k) lo[k] = T(0);
    for (int o = lane; o < NV; o += 32) s.V[o] = T(0);
    for (int t0 = 0; t0 < nterm; t0 += 32) {
        const int tt = t0 + lane;
        bool pass = false;
        if (tt < nterm) {
            const int i = tt / sk.npp, j = tt - i * sk.npp;
            pass = __ldg(pl.ppB + sb.pp0 + i) * __ldg(pl.ppB + sk.pp0 + j) >= pl.mag_thr &&
                   prim_reaches<L>(pl, pl.ppf[sb.pp0 + i], pl.ppf[sk.pp0 + j]);
            ++tl.screen;
        }
        unsigned m = __ballot_sync(0xffffffffu, pass);
        while (m) {
            // four primitive quartets, one per group of eight lanes (or two of
            // 16, or one of 32 when no more are left)
            const int left = __popc(m), gsz = left > 2 ? 8 : left == 2 ? 16 : 32;
            const int gl = lane & (gsz - 1), grp = lane / gsz;
            int mine = -1, ng = 0;
            int tid4[4];
#pragma unroll
            for (int g = 0; g < 4; ++g) {
                tid4[g] = m ? t0 + __ffs(m) - 1 : -1;
                ng += m != 0;
                m &= m - 1;
                if (g == grp) mine = tid4[g];
            }
            T Rs[D * D * D];
#pragma unroll
            for (int q = 0; q < D * D * D; ++q) Rs[q] = T(0);
            if (mine >= 0) {
                const int i = mine / sk.npp, j = mine - i * sk.npp;
                const PpiF bf = pl.ppf[sb.pp0 + i], kf = pl.ppf[sk.pp0 + j];
                PairT<T> x, y;
                load_pair(pl, sb.pp0 + i, bf, x);
                load_pair(pl, sk.pp0 + j, kf, y);
                float r;
                if (!prim_radius<L>(pl, bf, kf, r)) r = -1.0f;
                tl.radius += gl == 0;
                tl.term += gl == 0;
                const float r2 = r > 0.0f ? r * r : -1.0f;
                float F0[3] = {bf.P[0] - kf.P[0], bf.P[1] - kf.P[1], bf.P[2] - kf.P[2]}, f[3];
                T X0[3] = {x.P[0] - y.P[0], x.P[1] - y.P[1], x.P[2] - y.P[2]};
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    f[a] = rintf(pl.Finvf[3 * a] * F0[0] + pl.Finvf[3 * a + 1] * F0[1] + pl.Finvf[3 * a + 2] * F0[2]);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    F0[a] -= f[0] * pl.Lf[a] + f[1] * pl.Lf[3 + a] + f[2] * pl.Lf[6 + a];
                    X0[a] -= T(f[0]) * latc(pl.L, pl.Lf, a, T(0)) + T(f[1]) * latc(pl.L, pl.Lf, 3 + a, T(0)) +
                             T(f[2]) * latc(pl.L, pl.Lf, 6 + a, T(0));
                }
                const float x0n = fsqrt_fast(F0[0] * F0[0] + F0[1] * F0[1] + F0[2] * F0[2]);
                T alpha, aw, cw;
                alphas(x.ip + y.ip, latc(&pl.inv_omega2, &pl.inv_omega2f, 0, T(0)), alpha, aw, cw);
                int c = gl;
                while (true) {
                    bool hit = false;
                    while (c < pl.nr1) {
                        const float4 R = __ldg(lat + c);
                        if (R.w - x0n >= r) break;
                        ++tl.cand;
                        const float fx = F0[0] - R.x, fy = F0[1] - R.y, fz = F0[2] - R.z;
                        if (fx * fx + fy * fy + fz * fz < r2) {
                            hit = true;
                            break;
                        }
                        c += gsz;
                    }
                    if (!hit) break;
                    const T Xx = X0[0] - lat_at(pl, 4 * c, T(0)), Xy = X0[1] - lat_at(pl, 4 * c + 1, T(0)),
                            Xz = X0[2] - lat_at(pl, 4 * c + 2, T(0));
                    const T x2 = Xx * Xx + Xy * Xy + Xz * Xz;
                    c += gsz;
                    ++tl.img;
                    T sd[L + 1];
                    seeds<L>(x2, alpha, aw, cw, pl, sd);
                    T Bt[D * D * D];
                    herm_R<L, T>(sd, Xx, Xy, Xz, Bt);
#pragma unroll
                    for (int t = 0; t <= L; ++t)
#pragma unroll
                        for (int u = 0; u <= L - t; ++u)
#pragma unroll
                            for (int v = 0; v <= L - t - u; ++v) Rs[(t * D + u) * D + v] += Bt[(t * D + u) * D + v];
                }
            }
            __syncwarp();
            some = true;
#pragma unroll
            for (int t = 0; t <= L; ++t)
#pragma unroll
                for (int u = 0; u <= L - t; ++u)
#pragma unroll
                    for (int v = 0; v <= L - t - u; ++v) {
                        T q = Rs[(t * D + u) * D + v];
                        q += __shfl_xor_sync(0xffffffffu, q, 1);
                        q += __shfl_xor_sync(0xffffffffu, q, 2);
                        q += __shfl_xor_sync(0xffffffffu, q, 4);
                        if (gsz > 8) q += __shfl_xor_sync(0xffffffffu, q, 8);
                        if (gsz > 16) q += __shfl_xor_sync(0xffffffffu, q, 16);
                        Rs[(t * D + u) * D + v] = q;
                    }
#pragma unroll 1
            for (int g = 0; g < ng; ++g) {
                const int term = g == 0 ? tid4[0] : g == 1 ? tid4[1] : g == 2 ? tid4[2] : tid4[3];
                const int i = term / sk.npp, j = term - i * sk.npp;
                if (grp == g) {
#pragma unroll
                    for (int t = 0; t <= L; ++t)
#pragma unroll
                        for (int u = 0; u <= L - t; ++u)
#pragma unroll
                            for (int v = 0; v <= L - t - u; ++v) {
                                const int q = (t * D + u) * D + v;
                                if (((t + u + v) & 7) == gl) s.R[q] = Rs[q];
                            }
                }
                // E tables, one axis per lane; the ket's carry (-1)^s and, on
                // the first axis, the prefactor
                if (lane < 6) {
                    const bool brs = lane < 3;
                    const int ax = brs ? lane : lane - 3;
                    PairT<T> p;
                    const int ip = brs ? sb.pp0 + i : sk.pp0 + j;
                    const PpiF pf = pl.ppf[ip];
                    load_pair(pl, ip, pf, p);
                    const T PA = ax == 0 ? p.PA[0] : ax == 1 ? p.PA[1] : p.PA[2];
                    const T PB = ax == 0 ? p.PB[0] : ax == 1 ? p.PB[1] : p.PB[2];
                    if (brs) {
                        T E[S::EA];
                        herm_E<LA, LB, T>(PA, PB, T(0.5) * p.ip, E);
#pragma unroll
                        for (int q = 0; q < S::EA; ++q) s.Ea[ax * S::EA + q] = E[q];
                    } else {
                        T E[S::EC];
                        herm_E<LC, LD, T>(PA, PB, T(0.5) * p.ip, E);
                        T sc = T(1);
                        if (ax == 0) {
                            PairT<T> b;
                            const PpiF bf = pl.ppf[sb.pp0 + i];
                            load_pair(pl, sb.pp0 + i, bf, b);
                            sc = T(kTwoPi52) * b.K * p.K * b.ip * p.ip * inv_sqrt(b.p + p.p);
                        }
#pragma unroll
                        for (int q = 0; q < S::EC; ++q) s.Ec[ax * S::EC + q] = ((q % NTC) & 1) ? -sc * E[q] : sc * E[q];
                    }
                }
                __syncwarp();
                for (int o = lane; o < S::NH * S::NCD; o += 32) {
                    const int h = o / S::NCD, cd = o - h * S::NCD;
                    const int tx = s.tab[h][0], ty = s.tab[h][1], tz = s.tab[h][2];
                    const int cx = s.ecd[cd][0], cy = s.ecd[cd][1], cz = s.ecd[cd][2];
                    const int dx = s.ecd[cd][3], dy = s.ecd[cd][4], dz = s.ecd[cd][5];
                    const T *e0 = s.Ec + (cx * (LD + 1) + dx) * NTC, *e1 = s.Ec + S::EC + (cy * (LD + 1) + dy) * NTC,
                            *e2 = s.Ec + 2 * S::EC + (cz * (LD + 1) + dz) * NTC;
                    T acc = T(0);
                    for (int sx = 0; sx <= cx + dx; ++sx)
                        for (int sy = 0; sy <= cy + dy; ++sy) {
                            const T *Rp = s.R + ((tx + sx) * D + ty + sy) * D + tz;
                            T in = T(0);
                            for (int sz = 0; sz <= cz + dz; ++sz) in += e2[sz] * Rp[sz];
                            acc += e0[sx] * e1[sy] * in;
                        }
                    s.W[o] = acc;
                }
                __syncwarp();
                const auto element = [&](int o) {
                    const int ab = o / S::NCD, cd = o - ab * S::NCD;
                    const int ax = s.eab[ab][0], ay = s.eab[ab][1], az = s.eab[ab][2];
                    const int bx = s.eab[ab][3], by = s.eab[ab][4], bz = s.eab[ab][5];
                    const T *e0 = s.Ea + (ax * (LB + 1) + bx) * NTA, *e1 = s.Ea + S::EA + (ay * (LB + 1) + by) * NTA,
                            *e2 = s.Ea + 2 * S::EA + (az * (LB + 1) + bz) * NTA;
                    T acc = T(0);
                    for (int ux = 0; ux <= ax + bx; ++ux)
                        for (int uy = 0; uy <= ay + by; ++uy) {
                            T in = T(0);
                            for (int uz = 0; uz <= az + bz; ++uz) in += e2[uz] * s.W[s.tix[(ux * NTA + uy) * NTA + uz] * S::NCD + cd];
                            acc += e0[ux] * e1[uy] * in;
                        }
                    return acc;
                };
                if constexpr (comp) {
#pragma unroll
                    for (int k = 0; k < LV; ++k) {
                        const int o = lane + 32 * k;
                        if (o >= NV) break;
                        const T x = element(o), h = s.V[o], t = h + x, b = t - h;
                        s.V[o] = t;
                        lo[k] += (h - (t - b)) + (x - b);
                    }
                } else {
                    for (int o = lane; o < NV; o += 32) s.V[o] += element(o);
                }
                __syncwarp();
            }
        }
    }
    if constexpr (comp) {
#pragma unroll
        for (int k = 0; k < LV; ++k)
            if (lane + 32 * k < NV) s.V[lane + 32 * k] += lo[k];
        __syncwarp();
    }
    return some;
}

// J and K contributions of the block in s.V with orbit weight w (as digest in
// real2.cuh), one output element per lane.
template <int LA, int LB, int LC, int LD, typename T>
__device__ __forceinline__ void coop_digest(const PlanDev &pl, const SpiRec &sb, const SpiRec &sk, const CoopShared<LA, LB, LC, LD, T> &s,
                                            T w, const T *__restrict__ Dp, double *__restrict__ X, double *__restrict__ Y)
{
    using S = CoopShared<LA, LB, LC, LD, T>;
    constexpr int NA = S::NA, NB = S::NB, NC = S::NC, ND = S::ND;
    const int lane = threadIdx.x & 31, n = pl.nbf;
    const int aoI = pl.shells[sb.I].ao, aoJ = pl.shells[sb.J].ao, aoK = pl.shells[sk.I].ao, aoL = pl.shells[sk.J].ao;
    auto Dd = [&](int r, int c) { return __ldg(Dp + (size_t)r * n + c); };
    auto V = [&](int a, int b, int c, int d) { return s.V[((a * NB + b) * NC + c) * ND + d]; };
    for (int o = lane; o < NA * NB; o += 32) {
        const int a = o / NB, b = o % NB;
        T v = T(0);
        for (int c = 0; c < NC; ++c)
            for (int d = 0; d < ND; ++d) v += V(a, b, c, d) * Dd(aoK + c, aoL + d);
        atomicAdd(X + (size_t)(aoI + a) * n + aoJ + b, to_f64(T(2) * w * v));
    }
    for (int o = lane; o < NC * ND; o += 32) {
        const int c = o / ND, d = o % ND;
        T v = T(0);
        for (int a = 0; a < NA; ++a)
            for (int b = 0; b < NB; ++b) v += V(a, b, c, d) * Dd(aoI + a, aoJ + b);
        atomicAdd(X + (size_t)(aoK + c) * n + aoL + d, to_f64(T(2) * w * v));
    }
    if (!Y) return;  // a Coulomb-only build
    for (int o = lane; o < NA * ND; o += 32) {  // K_il += w V_ijkl D_jk
        const int a = o / ND, d = o % ND;
        T v = T(0);
        for (int b = 0; b < NB; ++b)
            for (int c = 0; c < NC; ++c) v += V(a, b, c, d) * Dd(aoJ + b, aoK + c);
        atomicAdd(Y + (size_t)(aoI + a) * n + aoL + d, to_f64(w * v));
    }
    for (int o = lane; o < NB * ND; o += 32) {  // K_jl += w V_ijkl D_ik
        const int b = o / ND, d = o % ND;
        T v = T(0);
        for (int a = 0; a < NA; ++a)
            for (int c = 0; c < NC; ++c) v += V(a, b, c, d) * Dd(aoI + a, aoK + c);
        atomicAdd(Y + (size_t)(aoJ + b) * n + aoL + d, to_f64(w * v));
    }
    for (int o = lane; o < NA * NC; o += 32) {  // K_ik += w V_ijkl D_jl
        const int a = o / NC, c = o % NC;
        T v = T(0);
        for (int b = 0; b < NB; ++b)
            for (int d = 0; d < ND; ++d) v += V(a, b, c, d) * Dd(aoJ + b, aoL + d);
        atomicAdd(Y + (size_t)(aoI + a) * n + aoK + c, to_f64(w * v));
    }
    for (int o = lane; o < NB * NC; o += 32) {  // K_jk += w V_ijkl D_il
        const int b = o / NC, c = o % NC;
        T v = T(0);
        for (int a = 0; a < NA; ++a)
            for (int d = 0; d < ND; ++d) v += V(a, b, c, d) * Dd(aoI + a, aoL + d);
        atomicAdd(Y + (size_t)(aoJ + b) * n + aoK + c, to_f64(w * v));
    }
}

template <int LA, int LB, int LC, int LD>
__device__ __forceinline__ void coop_counts(const Tally &tl, unsigned nq, unsigned long long *__restrict__ cnt)
{
    unsigned long long fl = tally_alg<LA, LB, LC, LD>(tl), fs = tally_screen<LA, LB, LC, LD>(tl);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        fl += __shfl_xor_sync(0xffffffffu, fl, o);
        fs += __shfl_xor_sync(0xffffffffu, fs, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (nq) atomicAdd(cnt, (unsigned long long)nq);
        if (fl) atomicAdd(cnt + 4, fl);
        if (fs) atomicAdd(cnt + 8, fs);
    }
}

// Tile form: block = one warp with a bra and a range of kets (TileMap); mode,
// the precision policy and the FP64 list as in k_real_w.
template <int LA, int LB, int LC, int LD, typename T>
__global__ void __launch_bounds__(32) k_real_c(PlanDev pl, TileMap map, int k0, int k1, int same, int mode, double tau,
                                               const T *__restrict__ Dp, const T *__restrict__ dmax, double *__restrict__ X,
                                               double *__restrict__ Y, unsigned long long *__restrict__ cnt, QuartetList big,
                                               unsigned *__restrict__ nbig, unsigned cap, unsigned *__restrict__ ovf)
{
    constexpr int L = LA + LB + LC + LD;
    __shared__ CoopShared<LA, LB, LC, LD, T> s;
    const int lane = threadIdx.x & 31;
    int bra, kbeg, kend;
    if (!tile_of(pl, map, blockIdx.x, k0, k1, same, bra, kbeg, kend)) return;
    const SpiRec sb = pl.spi[bra];
    const float tauf = (float)tau;
    const float Lq = radius_correction<L>(pl, 2.0f * pl.ls_max + 3.2094f - pl.log_ewald_R);
    const float4 bq = __ldg(pl.spq + bra), br = __ldg(pl.spr + bra);
    const bool policy = sizeof(T) == 4 && mode;
    const float dall = policy ? (float)__ldg(dmax + (size_t)pl.nshell * pl.nshell) : 0.0f;
    Tally tl;
    unsigned nq = 0;
    bool ready = false;
    for (int kb = kbeg & ~31; kb < kend; kb += 32) {
        const int kt = kb + lane;
        bool valid = kt >= kbeg && kt < kend && block_reaches<L>(pl, sb, kb >> 5);
        if (valid) {
            float eb;
            bool brief;
            valid = pair_reaches<L>(pl, bq, br, __ldg(pl.spq + kt), __ldg(pl.spr + kt), Lq, eb, brief);
            if (policy && valid && (eb * dall >= tauf || brief)) valid = !list_quartet(pl, bra, kt, tauf, dmax, big, nbig, cap, ovf);
        }
        unsigned m = __ballot_sync(0xffffffffu, valid);
        nq += __popc(m);
        if (m && !ready) {
            coop_init(s);
            ready = true;
        }
        while (m) {
            const int kq = kb + __ffs(m) - 1;
            m &= m - 1;
            const SpiRec sk = pl.spi[kq];
            tl.quart += lane == 0;
            if (!coop_quartet<LA, LB, LC, LD, T>(pl, sb, sk, s, tl)) continue;
            const T w = T(sb.w) * T(sk.w) * ((same && kq == bra) ? T(0.5) : T(1));
            coop_digest<LA, LB, LC, LD, T>(pl, sb, sk, s, w, Dp, X, Y);
            __syncwarp();
        }
    }
    coop_counts<LA, LB, LC, LD>(tl, nq, cnt);
}

// FP64 pass over the listed large quartets: one warp per list entry.
template <int LA, int LB, int LC, int LD>
__global__ void __launch_bounds__(32) k_real_list_c(PlanDev pl, QuartetList big, const unsigned *__restrict__ nbig,
                                                    unsigned cap, int same, const double *__restrict__ Dp, double *__restrict__ X,
                                                    double *__restrict__ Y, unsigned long long *__restrict__ cnt)
{
    __shared__ CoopShared<LA, LB, LC, LD, double> s;
    const unsigned total = min(*nbig, cap);
    if (blockIdx.x >= total) return;
    Tally tl;
    unsigned nq = 0;
    coop_init(s);
    for (unsigned q = blockIdx.x; q < total; q += gridDim.x) {
        const int2 pr = big.get(q);
        const SpiRec sb = pl.spi[pr.x], sk = pl.spi[pr.y];
        ++nq;
        tl.quart += (threadIdx.x & 31) == 0;
        if (!coop_quartet<LA, LB, LC, LD, double>(pl, sb, sk, s, tl)) continue;
        const double w = double(sb.w) * double(sk.w) * ((same && pr.x == pr.y) ? 0.5 : 1.0);
        coop_digest<LA, LB, LC, LD, double>(pl, sb, sk, s, w, Dp, X, Y);
        __syncwarp();
    }
    coop_counts<LA, LB, LC, LD>(tl, nq, cnt);
}

}  // namespace jk
