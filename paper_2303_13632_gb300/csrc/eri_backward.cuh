// eri_backward.cuh -- adjoint of the ERI kernel: gradients of E = sum_q sum_abcd G_abcd (ab|cd)
// with respect to the shell centres and the primitive exponents, recomputing the recurrences.
//
// For a primitive g_a = c N(alpha, L) prod_xi (r_xi - A_xi)^{a_xi} exp(-alpha |r - A|^2):
//   d g_a / d A_xi  = 2 alpha g_{a + 1_xi} - a_xi g_{a - 1_xi}
//   d g_a / d alpha = (2L + 3) / (4 alpha) g_a - sum_xi g_{a + 2_xi}
// (shifted functions keep the coefficient and normalisation of g_a).  In the Rys form of Eq. 8 each
// shift touches one axis factor only (n_Rys = floor((L+2)/2) + 1 roots, exact for the shifted
// integrals of total degree <= L + 2), so with W = sum G I_y I_z over the outputs that share their
// components w = (i0, i1, i2, i3) along an axis,
//   dE/dA = sum_mu sum_w W(w) [2 alpha I(w + 1_a) - a I(w - 1_a)]   on that axis,
// and the same with w + 2_a for the exponents.
//
// No integral beyond the class's own index ranges is formed.  I(w) is the mean of a product of
// powers of x - A, x - B, x' - C, x' - D over a Gaussian in (x, x'), so raising an index is
//   I(w + 1_a) = C00_A I(w) + B10 D I(w) + B00 K I(w),
// where D I(w) = a I(w - 1_a) + b I(w - 1_b) and K I(w) = c I(w - 1_c) + d I(w - 1_d) (the
// derivatives along x and x').  The sums over w of W times I, its four lowered forms, DD I, DK I and
// KK I (S0, Sa..Sd, SDD, SDK, SKK; SD = Sa + Sb, SK = Sc + Sd) then give everything: with
// P = B10 SD + B00 SK and V = B10^2 SDD + 2 B10 B00 SDK + B00^2 SKK,
//   U1 = sum W I(w + 1_a) = C00_A S0 + P,   U2 = sum W I(w + 2_a) = C00_A (U1 + P) + B10 S0 + V,
// for B with C00_B, and for C and D with C00', B01 and the bra and ket sums exchanged.  On the ranges
// extended by two this took 625 instead of 81 2-D integrals per (root, axis) of [dd|dd] (90 KB of
// shared memory instead of 8 per primitive quartet in FP64) and 12 of them per w and centre.
//
// GPU mapping.  A unit is a primitive quartet; a CTA owns a range of consecutive units of a class and
// takes QG of them at a time, so that every CTA has the same number whatever the contraction
// degrees.  Geometry, roots and the B, C records are made for a batch of units at once (one thread
// per unit, then per (unit, root): all threads busy in FP64).  Then per QG units:
//   1  2-D integrals: the lanes of rows_direct per (unit, root, axis)
//   2  W: one thread per (unit, root, a, c, b-chunk) with its outputs' G in registers (kept while the
//      units belong to one quartet) and the (b, d) blocks of I_x, I_y, I_z at its (a, c): five
//      operations per output for all three axes; the partial W blocks go to shared memory
//   3  one thread per (unit, axis, root, i0, i2): sums the partial blocks over the (a, c) with these
//      components, forms the eight sums from the neighbouring blocks of I and adds to the centre and
//      exponent gradients in registers (in FP32 as pairs of a sum and its rounding error, exact to
//      about 2^-40) until the quartet or the primitive changes; then the pairs are summed over the
//      segment's lanes and added to global memory in FP64.
// Step 3 of a unit and step 1 of the next one share a barrier interval (the first from the low
// threads up, the second from the high ones down, I in two buffers): two barriers per QG units.
// Bound by barriers between short steps and issue in FP32 (two CTAs per SM, 35% of the issue slots),
// by the FP64 pipe in FP64.  Measured on the 16 classes of p and d shells, K = 3, forward and backward:
// 1024 quartets per class in mixed precision 115 -> 13.3 ms, 384 in FP64 220 -> 47.3 ms.  In FP32 the
// pairs cost 0.9 ms over compensated sums rounded to one number before the lanes are summed, and FP64
// registers in their place 3.1 ms for the same results; relative error of both gradients against 64 bits
// 5.8e-8 with them, 1.2e-7 without, 8.5e-8 with FP32 sums per primitive quartet and FP64 beyond.  36
// instead of 18 G values per thread in FP64 (one pass over the roots of [dd|dd], no b-chunks) took that
// from 50.4 ms.
#pragma once

#include "eri_bwd_table.h"
#include "eri_kernels.cuh"

namespace eri {

template <int La_, int Lb_, int Lc_, int Ld_, typename R_>
struct GCfg {
    using R = R_;
    static constexpr int La = La_, Lb = Lb_, Lc = Lc_, Ld = Ld_;
    static constexpr int NA = ncart(La), NB = ncart(Lb), NC = ncart(Lc), ND = ncart(Ld);
    static constexpr int NERI = NA * NB * NC * ND;
    static constexpr int NRYS = (La + Lb + Lc + Ld + 2) / 2 + 1;
    static constexpr bool SWAB_OK = false, SWCD_OK = false;
    static constexpr int S_CB = S_N, S_CD = S_N + 3, SN = S_N + 6;
    static constexpr int NI = La + 1, NJ = Lb + 1, NK = Lc + 1, NL = Ld + 1, JL = NJ * NL;
    using IB_ = JBlock<JL, NK, (int)sizeof(R)>;
    static constexpr int VJ = IB_::V, JP = IB_::P;
    static constexpr int AC = NI * NK;
    static constexpr int IR = IB_::ROW, IB = NI * IR;  // 2-D integrals per row and per (root, axis)
    static constexpr int THREADS = 256;
    // outputs (G values) per thread of step 2
    static constexpr int BCH = imax(1, imin(NB, (sizeof(R) == 8 ? 36 : 50) / ND));
    static constexpr int NCH = cdiv(NB, BCH);
    static constexpr int ACN = NA * NC * NCH;
    // roots taken together, in passes of equal length
    static constexpr int NPASS = cdiv(NRYS, imin(NRYS, imax(1, THREADS / ACN)));
    static constexpr int RG = cdiv(NRYS, NPASS);
    static constexpr int WT = RG * ACN;
    // threads of step 3 per (unit, axis), padded to whole segments of a warp
    static constexpr int SA = RG * AC;
    static constexpr int SEG = SA <= 32 ? pow2ceil(SA) : cdiv(SA, 32) * 32;
    static constexpr int SW = SEG < 32 ? SEG : 32;   // lanes summed by shuffles
    static constexpr int NSW = SEG / SW;
    static constexpr int ST = 3 * SEG;
    static constexpr int I_VALS = 3 * NRYS * IB;     // per unit
    static constexpr int W_VALS = 3 * RG * ACN * JP;
    static constexpr int UNIT_BYTES = (2 * I_VALS + W_VALS) * (int)sizeof(R);
    static constexpr int QG = imax(1, imin(imin(THREADS / WT, THREADS / ST), (48 * 1024) / UNIT_BYTES));
    // units per batch of the setup stages
    static constexpr int NBU = imax(1, imin(32, THREADS / (QG * NRYS))) * QG;
    static constexpr int align16(int n) { return (n + 15) / 16 * 16; }
    static constexpr int OFF_BC = 0;
    static constexpr int OFF_META = align16(NBU * NRYS * SN * (int)sizeof(R));
    static constexpr int OFF_EA = align16(OFF_META + NBU * 8 * 4);
    static constexpr int OFF_I = align16(OFF_EA + NBU * 12 * (int)sizeof(R));
    static constexpr int OFF_W = align16(OFF_I + 2 * QG * I_VALS * (int)sizeof(R));  // I in two buffers
    // the batch's geometry is dead before steps 1 to 3 start
    static constexpr int SMEM = imax(OFF_W + QG * W_VALS * (int)sizeof(R), OFF_I + NBU * G_N * 8) + 16;
};

// a + b = sum + err exactly (Knuth's two-sum).
__device__ __forceinline__ float two_sum(float a, float b, float &err) {
    const float s = __fadd_rn(a, b), z = __fsub_rn(s, a);
    err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z));
    return s;
}

// Units of a class: its quartets' primitive quartets, quartet after quartet.
struct GradUnits {
    const long long *ps;  // prefix sum of the primitive quartets at the class's first quartet, or
                          // null for a primitive plan (one unit per quartet)
    long long units;
    int steps;            // groups of QG units per CTA
};

template <class C, int CH>
__device__ __forceinline__ void load_g(const double *__restrict__ G, const ClassArgs &args, int a, int c,
                                       typename C::R (&g)[C::BCH][C::ND]) {
#pragma unroll
    for (int bb = 0; bb < C::BCH; ++bb)
#pragma unroll
        for (int d = 0; d < C::ND; ++d)
            if (CH * C::BCH + bb < C::NB)
                g[bb][d] = to_r<typename C::R>(__ldg(G + a * args.ostride[0] + (CH * C::BCH + bb) * args.ostride[1] +
                                                     c * args.ostride[2] + d * args.ostride[3]));
}

// Step 2 for b-chunk CH: the thread's partial W blocks along the three axes.
template <class C, int CH>
__device__ __forceinline__ void w_chunk(const typename C::R (&g)[C::BCH][C::ND], const typename C::R (&X)[C::JL],
                                        const typename C::R (&Y)[C::JL], const typename C::R (&Z)[C::JL],
                                        typename C::R (&WX)[C::JL], typename C::R (&WY)[C::JL],
                                        typename C::R (&WZ)[C::JL]) {
    using R = typename C::R;
#pragma unroll
    for (int bb = 0; bb < C::BCH; ++bb) {
        if constexpr (CH * C::BCH < C::NB) {
            const int b = CH * C::BCH + bb;
            if (b < C::NB) {
#pragma unroll
                for (int d = 0; d < C::ND; ++d) {
                    const int jx = cart_x(C::Lb, b) * C::NL + cart_x(C::Ld, d);
                    const int jy = cart_y(C::Lb, b) * C::NL + cart_y(C::Ld, d);
                    const int jz = cart_z(C::Lb, b) * C::NL + cart_z(C::Ld, d);
                    const R gy = g[bb][d] * Y[jy], gx = g[bb][d] * X[jx];
                    WX[jx] = fma(gy, Z[jz], WX[jx]);
                    WZ[jz] = fma(gy, X[jx], WZ[jz]);
                    WY[jy] = fma(gx, Z[jz], WY[jy]);
                }
            }
        }
    }
}

template <class C>
__device__ __forceinline__ void backward_units(const ShellsDev &sh, const Tables &tb, const ClassArgs &args,
                                               const GradUnits &un, const double *__restrict__ G,
                                               double *__restrict__ dR, double *__restrict__ dalpha) {
    using R = typename C::R;
    constexpr int T = C::THREADS, JL = C::JL, JP = C::JP;
    extern __shared__ __align__(16) unsigned char smem[];
    R *bc_s = reinterpret_cast<R *>(smem + C::OFF_BC);
    int *meta_s = reinterpret_cast<int *>(smem + C::OFF_META);  // quartet, its four shells' primitives
    // 2 alpha, (2L+3) / (4 alpha) of the four and what the latter's rounding to R leaves: it multiplies the
    // same sign of term in every unit of the primitive, so its rounding would not average out
    R *ea_s = reinterpret_cast<R *>(smem + C::OFF_EA);
    R *I_s = reinterpret_cast<R *>(smem + C::OFF_I);
    R *W_s = reinterpret_cast<R *>(smem + C::OFF_W);
    double *geo_s = reinterpret_cast<double *>(smem + C::OFF_I);
    __shared__ int range_s[2];

    const int tid = threadIdx.x;
    const long long U0 = (long long)blockIdx.x * un.steps * C::QG;
    const long long U1 = min(un.units, U0 + (long long)un.steps * C::QG);
    const long long base = un.ps ? un.ps[0] : 0;
    if (un.ps && tid < 2) {  // quartets of the CTA's first and last unit
        const long long u = tid ? U1 - 1 : U0;
        int lo = 0, hi = (int)args.nq - 1;
        while (lo < hi) {
            const int mid = lo + (hi - lo + 1) / 2;
            if (__ldg(un.ps + mid) - base <= u) lo = mid; else hi = mid - 1;
        }
        range_s[tid] = lo;
    }
    // step 2: (group, root of the pass, a, c, chunk); step 3: (group, axis, root of the pass, i0, i2)
    const int wg = tid / C::WT, wr = tid - wg * C::WT;
    const int wmu = wr / C::ACN, witem = wr - wmu * C::ACN;
    // the chunk is the slowest part of an item, so that most warps run the code of one chunk
    const int wch = witem / (C::NA * C::NC), wc = witem % C::NC, wa = (witem / C::NC) % C::NA;
    int wo[3];
#pragma unroll
    for (int x = 0; x < 3; ++x) wo[x] = c_cart[C::La][wa][x] * C::IR + c_cart[C::Lc][wc][x] * JP;
    R g[C::BCH][C::ND];
    int gq = -1;  // the quartet whose G the thread holds
    const int sg = tid / C::ST, sx = (tid - sg * C::ST) / C::SEG, se = (tid - sg * C::ST) % C::SEG;
    const bool s_on = sg < C::QG && se < C::SA;
    const int smu = se / C::AC, si = (se % C::AC) / C::NK, sk = se % C::NK;
    // centre gradients of the quartet (0..3) and exponent gradients (4..7); FP32: with their errors
    R dacc[8], derr[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) dacc[k] = derr[k] = (R)0;
    auto add = [&](int k, R t) {
        if constexpr (sizeof(R) == 4) {
            R e;
            dacc[k] = two_sum(dacc[k], t, e);
            derr[k] += e;
        } else {
            dacc[k] += t;
        }
    };
    // 1: 2-D integrals of the units u0.. of the batch (nu of them) into buffer buf, by the CTA's warps
    // from the last one down
    auto integrals = [&](int u0, int nu, int buf) {
        constexpr int NIP = pow2ceil(C::NI), RITEMS = C::QG * C::NRYS * 3 * NIP;
        R *Id = I_s + buf * C::QG * C::I_VALS;
        for (int it = (T / 32 - 1 - tid / 32) * 32 + tid % 32; it < cdiv(RITEMS, 32) * 32; it += T) {
            const int blk = it / NIP, i = it % NIP;
            const int gu = blk / (3 * C::NRYS);
            const bool live = it < RITEMS && u0 + gu < nu;
            // lanes without a unit repeat the first one (in range, not stored)
            const int r = live ? blk - gu * 3 * C::NRYS : 0, unit = live ? u0 + gu : u0;
            rows_direct<C, typename C::IB_, NIP>(bc_s + (unit * C::NRYS + r / 3) * C::SN, r % 3, i, live,
                                                 Id + (live ? gu : 0) * C::I_VALS + ((r % 3) * C::NRYS + r / 3) * C::IB);
        }
    };

    for (long long ub = U0; ub < U1; ub += C::NBU) {
        const int nu = (int)min((long long)C::NBU, U1 - ub);
        __syncthreads();
        for (int i = tid; i < nu; i += T) {
            const long long u = ub + i;
            int q, prim = 0;
            if (un.ps) {
                int lo = range_s[0], hi = range_s[1];
                while (lo < hi) {
                    const int mid = lo + (hi - lo + 1) / 2;
                    if (__ldg(un.ps + mid) - base <= u) lo = mid; else hi = mid - 1;
                }
                q = lo;
                prim = (int)(u - (__ldg(un.ps + q) - base));
            } else {
                q = (int)u;
            }
            const int4 gqt = args.quartets[q];
            const int4 qt = make_int4(pick(gqt, args.perm[0]), pick(gqt, args.perm[1]), pick(gqt, args.perm[2]),
                                      pick(gqt, args.perm[3]));
            int np = 0;
            geometry_of<C>(sh, args, qt, prim, geo_s + i * G_N, np);
            const int nb = sh.nprim[qt.y], nc = sh.nprim[qt.z], nd = sh.nprim[qt.w];
            int t = prim;
            const int id = t % nd;
            t /= nd;
            const int ic = t % nc;
            t /= nc;
            const int pk[4] = {sh.pofs[qt.x] + t / nb, sh.pofs[qt.y] + t % nb, sh.pofs[qt.z] + ic,
                               sh.pofs[qt.w] + id};
            meta_s[i * 8] = q;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                constexpr int Lk[4] = {C::La, C::Lb, C::Lc, C::Ld};
                const double al = sh.exps[pk[k]];
                meta_s[i * 8 + 1 + k] = pk[k];
                const double ce = (0.25 * (2 * Lk[k] + 3)) / al;
                const R ch = to_r<R>(ce);
                ea_s[i * 12 + k] = to_r<R>(2.0 * al);
                ea_s[i * 12 + 4 + k] = ch;
                ea_s[i * 12 + 8 + k] = to_r<R>(ce - RTraits<R>::to_f64(ch));
            }
        }
        __syncthreads();
        for (int it = tid; it < nu * C::NRYS; it += T) {
            const int i = it / C::NRYS, mu = it - i * C::NRYS;
            const double *geo = geo_s + i * G_N;
            double x, w;
            rys_root<sizeof(R) == 4>(tb, C::NRYS, mu, geo[G_T], x, w);
            R *b = bc_s + it * C::SN;
            const double ipq = geo[G_IPQ], fq = geo[G_Q] * x * ipq, fp = geo[G_P] * x * ipq;
            b[S_WZ] = to_r<R>(geo[G_PREF] * w);
            b[S_B00] = to_r<R>(0.5 * x * ipq);
            b[S_B10] = to_r<R>((1.0 - fq) * (0.5 * geo[G_IP]));
            b[S_B01] = to_r<R>((1.0 - fp) * (0.5 * geo[G_IQ]));
#pragma unroll
            for (int s = 0; s < 3; ++s) {
                const double pq = geo[G_PQX + s];
                b[S_C0X + s] = to_r<R>(geo[G_PAX + s] - fq * pq);
                b[C::S_CB + s] = to_r<R>((geo[G_PAX + s] + geo[G_ABX + s]) - fq * pq);
                b[S_C1X + s] = to_r<R>(geo[G_QCX + s] + fp * pq);
                b[C::S_CD + s] = to_r<R>((geo[G_QCX + s] + geo[G_CDX + s]) + fp * pq);
            }
        }
        __syncthreads();  // records are written
        integrals(0, nu, 0);
        for (int u0 = 0, buf = 0; u0 < nu; u0 += C::QG, buf ^= 1) {
            __syncthreads();  // I of these units is written, W of the units before is read
            const R *Ic = I_s + buf * C::QG * C::I_VALS;
            const bool w_unit = wg < C::QG && u0 + wg < nu;
            if (w_unit) {
                const int q = meta_s[(u0 + wg) * 8];
                if (q != gq) {
                    gq = q;
                    with_chunk<C::NCH>(wch, [&](auto ch) {
                        load_g<C, decltype(ch)::value>(G + (long long)q * C::NERI, args, wa, wc, g);
                    });
                }
            }
            const bool s_unit = s_on && u0 + sg < nu;
#pragma unroll 1
            for (int pass = 0; pass < C::NPASS; ++pass) {
                const int m0 = pass * C::RG;
                if (pass > 0) __syncthreads();
                // 2: partial W blocks
                if (w_unit && m0 + wmu < C::NRYS) {
                    const R *Iu = Ic + wg * C::I_VALS + (m0 + wmu) * C::IB;
                    R X[JL], Y[JL], Z[JL], WX[JL], WY[JL], WZ[JL];
                    load_block<JL, C::VJ>(Iu + wo[0], X);
                    load_block<JL, C::VJ>(Iu + C::NRYS * C::IB + wo[1], Y);
                    load_block<JL, C::VJ>(Iu + 2 * C::NRYS * C::IB + wo[2], Z);
#pragma unroll
                    for (int t = 0; t < JL; ++t) WX[t] = WY[t] = WZ[t] = (R)0;
                    with_chunk<C::NCH>(wch, [&](auto ch) { w_chunk<C, decltype(ch)::value>(g, X, Y, Z, WX, WY, WZ); });
                    R *Wu = W_s + wg * C::W_VALS + (wmu * C::ACN + witem) * JP;
                    store_block<JL, C::VJ>(Wu, WX);
                    store_block<JL, C::VJ>(Wu + C::RG * C::ACN * JP, WY);
                    store_block<JL, C::VJ>(Wu + 2 * C::RG * C::ACN * JP, WZ);
                }
                __syncthreads();
                // 3: the sums over w of the thread's (i0, i2)
                if (s_unit && m0 + smu < C::NRYS) {
                    const R *Wu = W_s + sg * C::W_VALS + (sx * C::RG + smu) * C::ACN * JP;
                    R Wb[JL];
#pragma unroll
                    for (int t = 0; t < JL; ++t) Wb[t] = (R)0;
                    for (int na = 0; na <= C::La - si; ++na) {
                        const int ca = axis_component(C::La, sx, si, na);
                        for (int nc = 0; nc <= C::Lc - sk; ++nc) {
                            const R *p = Wu + (ca * C::NC + axis_component(C::Lc, sx, sk, nc)) * JP;
#pragma unroll
                            for (int ch = 0; ch < C::NCH; ++ch, p += C::NA * C::NC * JP) {
                                R v[JL];
                                load_block<JL, C::VJ>(p, v);
#pragma unroll
                                for (int t = 0; t < JL; ++t) Wb[t] += v[t];
                            }
                        }
                    }
                    const R *Ib = Ic + sg * C::I_VALS + (sx * C::NRYS + m0 + smu) * C::IB + si * C::IR + sk * JP;
                    const R fi = (R)si, fk = (R)sk;
                    R S0 = (R)0, Sa = (R)0, Sb = (R)0, Sc = (R)0, Sd = (R)0, DD = (R)0, DK = (R)0, KK = (R)0;
                    R v[JL];
                    // sum of W(j, l) v(j - dj, l - dl) f(j, l) with f = 1, j, l, j (j-1), l (l-1) or j l, the
                    // factor applied once per row or column
                    auto over_j = [&](int dj) -> R {
                        R s = (R)0;
#pragma unroll
                        for (int j = dj; j < C::NJ; ++j) {
                            R r = (R)0;
#pragma unroll
                            for (int l = 0; l < C::NL; ++l) r = fma(Wb[j * C::NL + l], v[(j - dj) * C::NL + l], r);
                            s = dj == 0 ? s + r : fma((R)(dj == 1 ? j : j * (j - 1)), r, s);
                        }
                        return s;
                    };
                    auto over_l = [&](int dl) -> R {
                        R s = (R)0;
#pragma unroll
                        for (int l = dl; l < C::NL; ++l) {
                            R r = (R)0;
#pragma unroll
                            for (int j = 0; j < C::NJ; ++j) r = fma(Wb[j * C::NL + l], v[j * C::NL + l - dl], r);
                            s = fma((R)(dl == 1 ? l : l * (l - 1)), r, s);
                        }
                        return s;
                    };
                    load_block<JL, C::VJ>(Ib, v);
                    S0 = over_j(0);
                    if constexpr (C::NJ > 1) Sb = over_j(1);
                    if constexpr (C::NL > 1) Sd = over_l(1);
                    if constexpr (C::NJ > 2) DD = over_j(2);
                    if constexpr (C::NL > 2) KK = over_l(2);
                    if constexpr (C::NJ > 1 && C::NL > 1) {
#pragma unroll
                        for (int j = 1; j < C::NJ; ++j) {
                            R r = (R)0;
#pragma unroll
                            for (int l = 1; l < C::NL; ++l)
                                r = fma((R)l * Wb[j * C::NL + l], v[(j - 1) * C::NL + l - 1], r);
                            DK = fma((R)j, r, DK);
                        }
                    }
                    if constexpr (C::La > 0) {
                        if (si > 0) {
                            load_block<JL, C::VJ>(Ib - C::IR, v);
                            Sa = fi * over_j(0);
                            if constexpr (C::NJ > 1) DD = fma((R)2 * fi, over_j(1), DD);
                            if constexpr (C::NL > 1) DK = fma(fi, over_l(1), DK);
                        }
                    }
                    if constexpr (C::Lc > 0) {
                        if (sk > 0) {
                            load_block<JL, C::VJ>(Ib - JP, v);
                            Sc = fk * over_j(0);
                            if constexpr (C::NL > 1) KK = fma((R)2 * fk, over_l(1), KK);
                            if constexpr (C::NJ > 1) DK = fma(fk, over_j(1), DK);
                        }
                    }
                    auto dot = [&](const R *p) -> R {
                        R s = (R)0;
                        load_block<JL, C::VJ>(p, v);
#pragma unroll
                        for (int t = 0; t < JL; ++t) s = fma(Wb[t], v[t], s);
                        return s;
                    };
                    if constexpr (C::La > 1)
                        if (si > 1) DD = fma(fi * (fi - (R)1), dot(Ib - 2 * C::IR), DD);
                    if constexpr (C::Lc > 1)
                        if (sk > 1) KK = fma(fk * (fk - (R)1), dot(Ib - 2 * JP), KK);
                    if constexpr (C::La > 0 && C::Lc > 0)
                        if (si > 0 && sk > 0) DK = fma(fi * fk, dot(Ib - C::IR - JP), DK);
                    const R *b = bc_s + ((u0 + sg) * C::NRYS + m0 + smu) * C::SN;
                    const R b00 = b[S_B00], b10 = b[S_B10], b01 = b[S_B01];
                    const R SD = Sa + Sb, SK = Sc + Sd;
                    const R P = fma(b10, SD, b00 * SK), Q = fma(b01, SK, b00 * SD);
                    const R x2 = (R)2 * b00 * DK;
                    const R VP = fma(b10, fma(b10, DD, x2), b00 * b00 * KK) + b10 * S0;
                    const R VQ = fma(b01, fma(b01, KK, x2), b00 * b00 * DD) + b01 * S0;
                    const R *ea = ea_s + (u0 + sg) * 12;
                    const R cf[4] = {b[S_C0X + sx], b[C::S_CB + sx], b[S_C1X + sx], b[C::S_CD + sx]};
                    const R low[4] = {Sa, Sb, Sc, Sd};
                    const R e0 = sx == 0 ? S0 : (R)0;  // sum over mu of e0: the quartet's energy
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const R p = k < 2 ? P : Q;
                        const R u1 = fma(cf[k], S0, p);
                        add(k, fma(ea[k], u1, -low[k]));
                        R x = -fma(cf[k], u1 + p, k < 2 ? VP : VQ);
                        if constexpr (sizeof(R) == 4) x = fma(ea[8 + k], e0, x);
                        add(4 + k, fma(ea[4 + k], e0, x));
                    }
                }
            }
            if (u0 + C::QG < nu) integrals(u0 + C::QG, nu, buf ^ 1);
            // sums that end here: the exponent gradients whose primitive, and the centre gradients whose
            // quartet is not that of the group's next unit (in this batch)
            unsigned int ends = 0u;
            const int *mine = meta_s + (u0 + sg) * 8;
            if (sg < C::QG && u0 + sg < nu) {
                const bool last = u0 + sg + C::QG >= nu;
                const int *next = mine + C::QG * 8;
                ends = (last || next[0] != mine[0]) ? 1u : 0u;
#pragma unroll
                for (int k = 0; k < 4; ++k) ends |= (last || next[1 + k] != mine[1 + k]) ? 2u << k : 0u;
            }
            const unsigned int any = __reduce_or_sync(0xffffffffu, ends);
            auto total = [&](int k, bool end) -> double {  // of the segment, on its first lane; the sum starts anew
                R v = (R)0, err = (R)0;
                if (end) {
                    v = dacc[k];
                    err = derr[k];
                    dacc[k] = derr[k] = (R)0;
                }
#pragma unroll
                for (int off = C::SW / 2; off > 0; off >>= 1) {
                    const R o = __shfl_down_sync(0xffffffffu, v, off, C::SW);
                    if constexpr (sizeof(R) == 4) {
                        const R oe = __shfl_down_sync(0xffffffffu, err, off, C::SW);
                        R e;
                        v = two_sum(v, o, e);
                        err += oe + e;
                    } else {
                        v += o;
                    }
                }
                if constexpr (sizeof(R) == 4)  // (an infinite sum has no error term; plain conversions are the
                    return RTraits<R>::finite(v) ? (double)v + (double)err : (double)v;  // faster ones here)
                else
                    return v;
            };
            const bool leader = se % C::SW == 0;
            if (any & 1u) {
                const bool end = ends & 1u;
                int4 gqt = make_int4(0, 0, 0, 0);
                if (end && leader) gqt = args.quartets[mine[0]];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const double v = total(k, end);
                    if (end && leader) atomicAdd(dR + 3LL * pick(gqt, args.perm[k]) + sx, v);
                }
            }
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (any & (2u << k)) {
                    const bool end = ends & (2u << k);
                    const double v = total(4 + k, end);
                    if (end && leader) atomicAdd(dalpha + mine[1 + k], v);
                }
        }
    }
}

template <class C, int MINB>
__global__ void __launch_bounds__(C::THREADS, MINB)
eri_backward_kernel(ShellsDev sh, Tables tb, ClassArgs args, GradUnits un, const double *__restrict__ G,
                    double *__restrict__ dR, double *__restrict__ dalpha) {
    backward_units<C>(sh, tb, args, un, G, dR, dalpha);
}

template <int La, int Lb, int Lc, int Ld, typename R>
cudaError_t launch_backward(const ShellsDev &sh, const Tables &tb, const ClassArgs &args,
                            const long long *ps, long long units, const double *G, double *dR,
                            double *dalpha, cudaStream_t stream) {
    using C = GCfg<La, Lb, Lc, Ld, R>;
    static_assert(C::SMEM <= 227 * 1024, "adjoint tile exceeds shared memory");
    static_assert(C::WT <= C::THREADS && C::ST <= C::THREADS, "adjoint thread layout");
    if (args.nq <= 0 || units <= 0) return cudaSuccess;
    // registers: two CTAs per SM; the wide blocks of f shells and FP64 take the register file of one
    constexpr int MINB = (sizeof(R) == 8 || C::JL > 9) ? 1 : 2;
    auto kern = eri_backward_kernel<C, MINB>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    if (e != cudaSuccess) return e;
    // whole batches per CTA, at most 64 steps, about eight CTAs per SM when there are enough units
    constexpr int batch = C::NBU / C::QG;
    const long long want = units / ((long long)C::QG * 152 * 8);
    GradUnits un{ps, units, (int)std::max<long long>(1, std::min<long long>(64, want))};
    if (un.steps > batch) un.steps = un.steps / batch * batch;
    const long long per = (long long)un.steps * C::QG, grid = (units + per - 1) / per;
    if (grid > 0x7fffffffLL) return cudaErrorInvalidValue;
    kern<<<(unsigned)grid, C::THREADS, C::SMEM, stream>>>(sh, tb, args, un, G, dR, dalpha);
    return cudaGetLastError();
}

}  // namespace eri
