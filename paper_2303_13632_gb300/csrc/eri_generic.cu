// eri_generic.cu -- ERIs of the classes with a g shell (L = 4) by one kernel whose angular
// momenta are run-time values.
//
// The per-class kernels of eri_kernels.cuh are specialised for each canonical class: every loop
// over components is unrolled and the intermediates live in registers.  For the 65 canonical
// classes with a g shell that specialisation would take the library build from minutes to the
// better part of an hour ([gg|gg] alone compiles for more than seven minutes in three variants),
// so these classes share one kernel per precision with the same stages of Sec. II-C in run-time
// loops over shared memory:
//   geometry and prefactor        FP64, as the specialised kernels
//   Rys root/weight, B and C      FP64, rounded to R
//   2-D integrals I(i, j, k, l)   the four-index Rys recursion in which every index is raised with
//                                 the C value of its own centre (the recurrences behind Eqs. 6-7
//                                 before the transfer relation; exact arithmetic gives the VRR +
//                                 HRR values)
//   quadrature (Eq. 8)            summed over the roots in R and over primitives in FP64 (in the
//                                 output or the scratch)
// Compressed output (Sec. II-D) then takes one more launch over the FP64 values (pack_kernel of
// eri_contract.cu).
#include <algorithm>
#include <vector>

#include "eri_internal.h"
#include "eri_kernels.cuh"

namespace eri {

namespace {

constexpr int kGenThreads = 256;
constexpr int kGenQmax = 64;      // quartets per tile
constexpr int kGenUnits = 128;    // units (primitive quartets) per batch of the setup stages
constexpr int kGenBcBytes = 28 * 1024;  // shared memory of a batch's B, C records
constexpr int kGenSmem = 96 * 1024, kGenSmemPrim = 72 * 1024;  // contracted plans, primitive plans
// Limit of the kernels' dynamic shared memory (the static part is below 2 KB).  It is state of the
// function, shared by all host threads, so every launch sets the same one, whatever it takes itself.
constexpr int kGenSmemLimit = 227 * 1024 - 2048;
// B, C values per (unit, root): the slots of phase_setup plus C00 relative to B and C00'
// relative to D
constexpr int kGenCB = S_N, kGenCD = S_N + 3, kGenSN = S_N + 6;
constexpr int kGenSNP = kGenSN + 1;  // odd stride of the (unit, root) records: distinct banks

// geometry without the choice of transfer direction (the four-index recursion needs none)
struct GenGeo {
    static constexpr bool SWAB_OK = false, SWCD_OK = false;
};

struct GenShape {
    int L[4];        // canonical angular momenta
    int n[4];        // Cartesian components per shell
    int nrys, neri;  // roots, ERIs per quartet
    int iblkp;       // stride of the (La+1)(Lb+1)(Lc+1)(Ld+1) integrals of a (unit, root, axis), odd
                     // so that the blocks the lanes of a warp build start in distinct banks
    int lanes;       // lanes per (unit, root, axis): (La+1)(Lb+1) rounded up to a power of two, or 1
    int q;           // quartets per tile
    int setup;       // units per batch of the setup stages
    int units;       // units per batch of the 2-D integrals
    unsigned m_neri, m_ncd;  // ceil(2^32 / d) for n_ERIQ, n_c n_d (0: d = 1)
    int geo_off, bc_off, i_off, smem;  // dynamic shared memory layout (bytes)
};

unsigned div_magic(int d) { return d == 1 ? 0u : (unsigned)(((1ull << 32) + d - 1) / d); }
// n / d for n d < 2^32 with the magic of d
__device__ __forceinline__ int div_by(int n, unsigned m) { return m ? (int)__umulhi((unsigned)n, m) : n; }

// Shape of a class; q_most: quartets per tile of a primitive plan at most.
//   Primitive plans: a tile is one batch of the setup stages, its records no more than the tile's, and 72 KB
// of shared memory leave three CTAs per SM (96 KB and records for 26 to 128 units whatever the tile held
// left two).  A second batch of the integrals that would be only partly filled is left to the next tile.
//   Contracted quartets have setup batches of their own, and short tiles keep the longest of them from
// holding up the end of a launch.
//   FP64: the recursion on lanes costs 25 FP64 instructions per lane ahead of the first plane and five per
// plane, on idle lanes too, and the FP64 pipe is what bounds it.  One thread per (unit, root, axis) issues
// fewer but has their whole chain, so it takes the classes with few planes and the batches that fill a warp.
//   369 classes in FP64, 2^15 / 2^20 / 2^22 ERIs each: 1.11 / 26.2 / 103.9 ms before these three rules,
// 0.64 / 15.2 / 59.5 with them; one class at a time (the canonical ones) 23.0 -> 13.9 ms at 2^22.
template <typename R>
GenShape gen_shape(const int L[4], bool contracted, int q_most = kGenQmax) {
    GenShape g{};
    for (int k = 0; k < 4; ++k) {
        g.L[k] = L[k];
        g.n[k] = ncart(L[k]);
    }
    g.nrys = (L[0] + L[1] + L[2] + L[3]) / 2 + 1;
    g.neri = g.n[0] * g.n[1] * g.n[2] * g.n[3];
    g.iblkp = ((L[0] + 1) * (L[1] + 1) * (L[2] + 1) * (L[3] + 1)) | 1;
    g.m_neri = div_magic(g.neri);
    g.m_ncd = div_magic(g.n[2] * g.n[3]);
    const int tab = 2 * 4 * (g.n[0] * g.n[1] + g.n[2] * g.n[3]) + 4 * (kGenUnits + 2 * kGenQmax + 2);
    g.bc_off = (tab + 15) / 16 * 16;
    // the records of a setup batch, and behind them the integrals of a smaller one, whose place the
    // batch's geometry takes before
    const int rec = g.nrys * kGenSNP * (int)sizeof(R), ints = 3 * g.nrys * g.iblkp * (int)sizeof(R);
    const int budget = contracted ? kGenSmem : kGenSmemPrim;
    auto records = [&](int setup) { return (g.bc_off + setup * rec + 15) / 16 * 16; };
    auto units = [&](int setup) { return std::max(1, std::min(setup, (budget - records(setup)) / ints)); };
    g.setup = std::max(1, std::min(kGenUnits, kGenBcBytes / rec));
    if (contracted) {
        g.q = g.neri >= 64 ? 1 : 4;  // whatever the call: the order of a quartet's sums depends on it
    } else {
        const int fit = std::max(1, (budget - g.bc_off) / (rec + ints));  // whose integrals fit at a time
        g.q = std::min({q_most, kGenQmax, g.setup, std::max(fit, 16384 / g.neri)});
        const int u = units(g.q);
        if (g.q < 2 * u) g.q = std::min(g.q, u);
        g.setup = g.q;
    }
    g.i_off = records(g.setup);
    g.units = units(g.setup);
    g.geo_off = g.i_off;
    g.smem = g.i_off + std::max(g.units * ints, g.setup * G_N * 8);
    const int planes = (L[2] + 1) * (L[3] + 1);
    g.lanes = 1;
    if (sizeof(R) == 4 || (planes > 6 && g.units * g.nrys * 3 < 36))
        while (g.lanes < (L[0] + 1) * (L[1] + 1)) g.lanes *= 2;
    return g;
}

// 2-D integrals of one (unit, root, axis) by g.lanes lanes of a warp, lane (i, j) holding its value of
// the plane (k, l).  Raising k or l takes the values of lanes (i - 1, j) and (i, j - 1) by shuffles
// and the lane's own lower planes from registers; every index is raised with its own centre.  Every
// lane of the warp calls it; live lanes store I(i, j, k, l) at i si + j sj + k sk + l.
template <typename R>
__device__ __forceinline__ void plane_recursion(const GenShape &g, const R *b, int xi, int e, bool live, R *I) {
    const int La = g.L[0], Lb = g.L[1], Lc = g.L[2], Ld = g.L[3], nj = Lb + 1, w = g.lanes;
    const int i = e / nj, j = e - i * nj;
    const int sk = Ld + 1, sj = (Lc + 1) * sk, si = nj * sj;
    const R cA = b[S_C0X + xi], cB = b[kGenCB + xi], cC = b[S_C1X + xi], cD = b[kGenCD + xi];
    const R b00 = b[S_B00], b10 = b[S_B10], b01 = b[S_B01];
    const R ib00 = (R)i * b00, jb00 = (R)j * b00, ib10 = (R)i * b10;
    // the plane (0, 0): I(i, 0), then up to I(i, j) on every lane of row i
    R lo = (R)0, v = xi == 2 ? b[S_WZ] : (R)1, mine;
    for (int t = 1; t <= La; ++t) {
        R n = cA * v;
        if (t > 1) n = fma((R)(t - 1) * b10, lo, n);
        if (t <= i) {
            lo = v;
            v = n;
        }
    }
    mine = v;
    lo = (R)0;
    for (int t = 1; t <= Lb; ++t) {
        const R u = __shfl_up_sync(0xffffffffu, v, nj, w);
        R n = cB * v;
        if (t > 1) n = fma((R)(t - 1) * b10, lo, n);
        if (i > 0) n = fma(ib10, u, n);
        lo = v;
        v = n;
        if (t == j) mine = n;
    }
    R *out = I + i * si + j * sj;
    R p1 = (R)0, p2 = (R)0, low[kLmax + 1];  // (k-1, 0), (k-2, 0), (k-1, l)
#pragma unroll
    for (int l = 0; l <= kLmax; ++l) low[l] = (R)0;
    for (int k = 0; k <= Lc; ++k, out += sk) {
        if (k > 0) {
            const R u = __shfl_up_sync(0xffffffffu, p1, nj, w), s = __shfl_up_sync(0xffffffffu, p1, 1, w);
            R n = cC * p1;
            if (k > 1) n = fma((R)(k - 1) * b01, p2, n);
            if (i > 0) n = fma(ib00, u, n);
            if (j > 0) n = fma(jb00, s, n);
            mine = n;
        }
        p2 = p1;
        p1 = mine;
        if (live) out[0] = mine;
        R q1 = mine, q2 = (R)0, below = low[0];
        low[0] = mine;
        const R kb01 = (R)k * b01;
#pragma unroll
        for (int l = 1; l <= kLmax; ++l) {
            if (l <= Ld) {
                const R u = __shfl_up_sync(0xffffffffu, q1, nj, w), s = __shfl_up_sync(0xffffffffu, q1, 1, w);
                R n = cD * q1;
                if (l > 1) n = fma((R)(l - 1) * b01, q2, n);
                if (k > 0) n = fma(kb01, below, n);
                if (i > 0) n = fma(ib00, u, n);
                if (j > 0) n = fma(jb00, s, n);
                if (live) out[l] = n;
                q2 = q1;
                q1 = n;
                below = low[l];
                low[l] = n;
            }
        }
    }
}

// The same by one thread, each value from the lower ones in shared memory, by the operations of
// plane_recursion in their order.
template <typename R>
__device__ __forceinline__ void chain_recursion(const GenShape &g, const R *b, int xi, R *I) {
    const int La = g.L[0], Lb = g.L[1], Lc = g.L[2], Ld = g.L[3];
    const int sk = Ld + 1, sj = (Lc + 1) * sk, si = (Lb + 1) * sj;
    const R cA = b[S_C0X + xi], cB = b[kGenCB + xi], cC = b[S_C1X + xi], cD = b[kGenCD + xi];
    const R b00 = b[S_B00], b10 = b[S_B10], b01 = b[S_B01];
    I[0] = xi == 2 ? b[S_WZ] : (R)1;
    for (int i = 1; i <= La; ++i) {
        R v = cA * I[(i - 1) * si];
        if (i > 1) v = fma((R)(i - 1) * b10, I[(i - 2) * si], v);
        I[i * si] = v;
    }
    for (int j = 1; j <= Lb; ++j)
        for (int i = 0; i <= La; ++i) {
            const int e = i * si + j * sj;
            R v = cB * I[e - sj];
            if (j > 1) v = fma((R)(j - 1) * b10, I[e - 2 * sj], v);
            if (i > 0) v = fma((R)i * b10, I[e - si - sj], v);
            I[e] = v;
        }
    for (int k = 1; k <= Lc; ++k)
        for (int i = 0; i <= La; ++i)
            for (int j = 0; j <= Lb; ++j) {
                const int e = i * si + j * sj + k * sk;
                R v = cC * I[e - sk];
                if (k > 1) v = fma((R)(k - 1) * b01, I[e - 2 * sk], v);
                if (i > 0) v = fma((R)i * b00, I[e - si - sk], v);
                if (j > 0) v = fma((R)j * b00, I[e - sj - sk], v);
                I[e] = v;
            }
    for (int l = 1; l <= Ld; ++l)
        for (int k = 0; k <= Lc; ++k)
            for (int i = 0; i <= La; ++i)
                for (int j = 0; j <= Lb; ++j) {
                    const int e = i * si + j * sj + k * sk + l;
                    R v = cD * I[e - 1];
                    if (l > 1) v = fma((R)(l - 1) * b01, I[e - 2], v);
                    if (k > 0) v = fma((R)k * b01, I[e - sk - 1], v);
                    if (i > 0) v = fma((R)i * b00, I[e - si - 1], v);
                    if (j > 0) v = fma((R)j * b00, I[e - sj - 1], v);
                    I[e] = v;
                }
}

// One tile: quartets [q0, q0 + qn) of the class of `args`, ERIs summed over primitive quartets
// in FP64 into out[q * n_ERIQ + generic index], q = 0..qn-1 (out = the tile's first quartet).
// The tile's primitive quartets are taken in batches, whatever quartet they belong to, of g.setup for
// the first two stages (short chains of FP64 work, nothing but their number hides their latency) and of
// g.units for the others (their integrals fill the shared memory):
//   geometry        one thread per unit
//   roots, B and C  one thread per (unit, root)
//   2-D integrals   plane_recursion, (La+1)(Lb+1) lanes per (unit, root, axis), or chain_recursion, one thread
//   quadrature      one thread per (quartet, output), or several that share the quartet's units
// One primitive quartet per quartet at a time left most of the CTA idle in all but the last of these:
// 35,000 quartets of a 40-atom molecule (K up to 6, FP32) from the work queue 133 -> 9.0 ms; the 369
// classes with a g shell, 2^20 ERIs each, 16-bit codes 45 -> 38 ms (10.6 ms with the classes spread
// over side streams).  Bound by shared-memory reads: three per root and output for two operations.
// Every thread of the CTA calls it; it begins and ends with a barrier.
template <typename R>
__device__ __forceinline__ void generic_tile(const ShellsDev &sh, const Tables &tb, const ClassArgs &args,
                                             const GenShape &g, long long q0, int qn, double *__restrict__ out,
                                             unsigned char *smem) {
    const int nab = g.n[0] * g.n[1], ncd = g.n[2] * g.n[3];
    // per (a, b) and (c, d): offsets of the components in a block along the three axes (10 bits
    // each; they add without carry) and the position in the caller's order
    unsigned *off_s = reinterpret_cast<unsigned *>(smem);
    int *pos_s = reinterpret_cast<int *>(off_s + nab + ncd);
    int *uq_s = pos_s + nab + ncd;        // quartet of each unit of the batch
    int *first_s = uq_s + kGenUnits;      // first unit of each quartet of the tile; [qn] = units
    double *geo_s = reinterpret_cast<double *>(smem + g.geo_off);
    R *bc_s = reinterpret_cast<R *>(smem + g.bc_off);
    R *I_s = reinterpret_cast<R *>(smem + g.i_off);
    const int tid = threadIdx.x;
    const int La = g.L[0], Lb = g.L[1], Lc = g.L[2], Ld = g.L[3];
    const int sk = Ld + 1, sj = (Lc + 1) * sk, si = (Lb + 1) * sj;
    auto shells_of = [&](int q) {
        const int4 gq = args.quartets[q0 + q];
        return make_int4(pick(gq, args.perm[0]), pick(gq, args.perm[1]), pick(gq, args.perm[2]), pick(gq, args.perm[3]));
    };
    __syncthreads();
    for (int t = tid; t < nab + ncd; t += kGenThreads) {
        const bool bra = t < nab;
        const int e = bra ? t : t - nab, n2 = bra ? g.n[1] : g.n[3];
        const int e1 = e / n2, e2 = e - e1 * n2;
        const int l1 = bra ? La : Lc, l2 = bra ? Lb : Ld, s1 = bra ? si : sk, s2 = bra ? sj : 1;
        unsigned o = 0;
        for (int x = 0; x < 3; ++x) o |= (unsigned)(c_cart[l1][e1][x] * s1 + c_cart[l2][e2][x] * s2) << (10 * x);
        off_s[t] = o;
        pos_s[t] = e1 * args.ostride[bra ? 0 : 2] + e2 * args.ostride[bra ? 1 : 3];
    }
    if (tid == 0) first_s[0] = 0;
    for (int q = tid; q < qn; q += kGenThreads) {
        const int4 qt = shells_of(q);
        first_s[q + 1] = sh.nprim[qt.x] * sh.nprim[qt.y] * sh.nprim[qt.z] * sh.nprim[qt.w];
    }
    __syncthreads();
    if (tid == 0)
        for (int q = 0; q < qn; ++q) first_s[q + 1] += first_s[q];
    __syncthreads();
    const int total = first_s[qn];
    for (int sb = 0; sb < total; sb += g.setup) {
        const int ns = min(g.setup, total - sb);
        for (int i = tid; i < ns; i += kGenThreads) {
            int lo = 0, hi = qn - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) / 2;
                if (first_s[mid] <= sb + i) lo = mid; else hi = mid - 1;
            }
            int np = 0;
            geometry_of<GenGeo>(sh, args, shells_of(lo), sb + i - first_s[lo], geo_s + i * G_N, np);
            uq_s[i] = lo;
        }
        __syncthreads();
        for (int it = tid; it < ns * g.nrys; it += kGenThreads) {
            const int u = it / g.nrys, mu = it - u * g.nrys;
            const double *geo = geo_s + u * G_N;
            double x, w;
            rys_root<sizeof(R) == 4>(tb, g.nrys, mu, geo[G_T], x, w);
            R *b = bc_s + (size_t)it * kGenSNP;
            const double ipq = geo[G_IPQ];
            const double fq = geo[G_Q] * x * ipq, fp = geo[G_P] * x * ipq;
            b[S_B00] = to_r<R>(0.5 * x * ipq);
            b[S_B10] = to_r<R>((1.0 - fq) * (0.5 * geo[G_IP]));
            b[S_B01] = to_r<R>((1.0 - fp) * (0.5 * geo[G_IQ]));
            for (int s = 0; s < 3; ++s) {
                const double pq = geo[G_PQX + s];
                b[S_C0X + s] = to_r<R>(geo[G_PAX + s] - fq * pq);
                b[kGenCB + s] = to_r<R>((geo[G_PAX + s] + geo[G_ABX + s]) - fq * pq);
                b[S_C1X + s] = to_r<R>(geo[G_QCX + s] + fp * pq);
                b[kGenCD + s] = to_r<R>((geo[G_QCX + s] + geo[G_CDX + s]) + fp * pq);
            }
            b[S_WZ] = to_r<R>(geo[G_PREF] * w);
        }
        __syncthreads();
        for (int ub = sb; ub < sb + ns; ub += g.units) {
            const int nu = min(g.units, sb + ns - ub);
            const R *bc_u = bc_s + (size_t)(ub - sb) * g.nrys * kGenSNP;
            const int groups = nu * g.nrys * 3, nij = (La + 1) * (Lb + 1);
            if (sizeof(R) == 8 && g.lanes == 1) {
                for (int it = tid; it < groups; it += kGenThreads)
                    chain_recursion<R>(g, bc_u + (size_t)(it / 3) * kGenSNP, it % 3, I_s + (size_t)it * g.iblkp);
            } else {
                for (int it = tid; it - (tid & 31) < groups * g.lanes; it += kGenThreads) {
                    const int r = it / g.lanes, e = it % g.lanes;
                    const bool live = r < groups && e < nij;
                    const int m = r < groups ? r : 0;  // lanes past the last group repeat the first (not stored)
                    plane_recursion<R>(g, bc_u + (size_t)(m / 3) * kGenSNP, m % 3, e < nij ? e : 0, live,
                                       I_s + (size_t)m * g.iblkp);
                }
            }
            __syncthreads();
            // quadrature: `parts` neighbouring lanes share the units of one (quartet, output)
            const int qa = uq_s[ub - sb], nseg = uq_s[ub - sb + nu - 1] - qa + 1, ms = 3 * g.iblkp;
            int parts = 1;
            while (parts < 32 && 2 * parts * nseg * g.neri <= kGenThreads && 2 * parts * nseg <= nu) parts *= 2;
            const int items = nseg * g.neri * parts;
            for (int it = tid; it - (tid & 31) < items; it += kGenThreads) {
                const bool on = it < items;
                const int t = on ? it / parts : 0, part = it & (parts - 1);
                const int seg = div_by(t, g.m_neri), o = t - seg * g.neri, q = qa + seg;
                const int ab = div_by(o, g.m_ncd), cd = o - ab * ncd;
                const unsigned off = off_s[ab] + off_s[nab + cd];
                const int u0 = max(first_s[q] - ub, 0), u1 = on ? min(first_s[q + 1] - ub, nu) : 0;
                double sum = 0.0;
                for (int u = u0 + part; u < u1; u += parts) {
                    const R *I0 = I_s + (size_t)u * g.nrys * ms;
                    const R *Ix = I0 + (off & 1023u), *Iy = I0 + g.iblkp + ((off >> 10) & 1023u),
                            *Iz = I0 + 2 * g.iblkp + (off >> 20);
                    R s = (R)0;
                    for (int mu = 0; mu < g.nrys; ++mu, Ix += ms, Iy += ms, Iz += ms) s = fma(*Ix * *Iy, *Iz, s);
                    sum += RTraits<R>::to_f64(s);
                }
                for (int d = parts / 2; d > 0; d >>= 1) sum += __shfl_down_sync(0xffffffffu, sum, d, parts);
                if (on && part == 0) {
                    double *dst = out + (long long)q * g.neri + pos_s[ab] + pos_s[nab + cd];
                    if (first_s[q] < ub) sum += *dst;
                    *dst = sum;
                    if (first_s[q + 1] <= ub + nu && !(fabs(sum) <= 1.7976931348623157e308)) atomicOr(args.err, 1);
                }
            }
            __syncthreads();
        }
    }
}

template <typename R>
__global__ void __launch_bounds__(kGenThreads)
eri_generic_kernel(ShellsDev sh, Tables tb, ClassArgs args, GenShape g, double *__restrict__ out) {
    extern __shared__ __align__(16) unsigned char smem[];
    const long long q0 = (long long)blockIdx.x * g.q;
    const int qn = (int)((args.nq - q0) < g.q ? (args.nq - q0) : g.q);
    generic_tile<R>(sh, tb, args, g, q0, qn, out + q0 * (long long)g.neri, smem);
}

template <typename R>
cudaError_t run_values(const ShellsDev &sh, const Tables &tb, const ClassArgs &a, const GenShape &g,
                       double *out, cudaStream_t stream) {
    auto kern = eri_generic_kernel<R>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kGenSmemLimit);
    if (e != cudaSuccess) return e;
    const long long tiles = (a.nq + g.q - 1) / g.q;
    if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
    kern<<<(unsigned)tiles, kGenThreads, g.smem, stream>>>(sh, tb, a, g, out);
    return cudaGetLastError();
}

// quartets per compressed chunk: a multiple of 32 (every chunk starts on a packed word)
long long chunk_quartets(int neri, size_t scratch_bytes) {
    long long c = (long long)(scratch_bytes / (sizeof(double) * (size_t)neri)) / 32 * 32;
    return c;
}

// ---------------------------------------------------------------------------------------------
// One persistent launch for every class of a plan: a work queue of tiles (class, quartets
// [q0, q0 + q)) over all classes, pulled by the resident CTAs from one atomic counter, so
// quartets of uneven class and contraction degree balance across the GPU.  Each tile's FP64
// values go to the CTA's slot of a scratch buffer and are compressed in the same launch: b_max
// and eps per quartet (Eq. 9), then the codes (Eq. 10) packed one output word per thread; words
// that a tile shares with its neighbour tile are OR-ed in (the output is zeroed before the
// launch), the others stored.

struct QueueClass {
    ClassArgs a;           // quartets, permutation, output strides, packed segment and scales
    GenShape g;            // shape and shared-memory layout (common quartet cap)
    long long first_tile;  // first tile of the class in the queue
};

// The CTA's share of a queue: tiles by the counter until it is past the last one.  bits = 0: FP64
// output, one tile per CTA (no counter, no slot).
template <typename R>
__device__ __forceinline__ void queue_tiles(const ShellsDev &sh, const Tables &tb, const QueueClass *classes,
                                            int n_classes, long long n_tiles, unsigned long long *counter,
                                            double *__restrict__ scratch, long long slot_doubles, int bits,
                                            unsigned char *smem) {
    __shared__ long long item_s;
    __shared__ int cls_s;
    __shared__ unsigned long long bmax_s[kGenQmax];
    __shared__ double inv_s[kGenQmax];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    double *vals = scratch + (long long)blockIdx.x * slot_doubles;
    const double M = bits ? (double)((1u << (bits - 1)) - 1u) : 0.0;
    const uint32_t mask = (1u << bits) - 1u;
    for (;;) {
        if (tid == 0) {
            item_s = bits ? (long long)atomicAdd(counter, 1ull) : (long long)blockIdx.x;
            int lo = 0, hi = n_classes - 1;  // last class whose first tile <= item
            while (lo < hi) {
                const int mid = (lo + hi + 1) / 2;
                if (classes[mid].first_tile <= item_s) lo = mid; else hi = mid - 1;
            }
            cls_s = lo;
        }
        __syncthreads();
        const long long item = item_s;
        if (item >= n_tiles) break;
        const QueueClass &qc = classes[cls_s];
        const ClassArgs a = qc.a;
        const GenShape g = qc.g;
        const long long q0 = (item - qc.first_tile) * g.q;
        const int qn = (int)((a.nq - q0) < g.q ? (a.nq - q0) : g.q);
        generic_tile<R>(sh, tb, a, g, q0, qn, bits ? vals : a.out_fp64 + q0 * (long long)g.neri, smem);
        if (bits == 0) return;
        // b_max per quartet (non-negative IEEE values order like their bit patterns): all warps on
        // a large quartet, a warp per small one
        for (int q = tid; q < qn; q += kGenThreads) bmax_s[q] = 0ull;
        __syncthreads();
        const int wstep = g.neri >= 512 ? kGenThreads : 32, wfirst = g.neri >= 512 ? tid : lane;
        for (int q = g.neri >= 512 ? 0 : warp; q < qn; q += g.neri >= 512 ? 1 : kGenThreads / 32) {
            unsigned long long m = 0ull;
            for (int o = wfirst; o < g.neri; o += wstep)
                m = max(m, (unsigned long long)__double_as_longlong(fabs(vals[(long long)q * g.neri + o])));
            for (int d = 16; d > 0; d >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, d));
            if (lane == 0) atomicMax(bmax_s + q, m);
        }
        __syncthreads();
        for (int q = tid; q < qn; q += kGenThreads) {
            const float e = (float)(__longlong_as_double((long long)bmax_s[q]) / M);
            inv_s[q] = e > 0.0f ? 1.0 / (double)e : 0.0;
            a.scales[q0 + q] = e;
        }
        __syncthreads();
        // the tile's words of the stream, positions relative to the tile's first bit
        const long long bit0 = q0 * g.neri * bits, bit1 = (q0 + qn) * (long long)g.neri * bits;
        const long long w0 = bit0 >> 5;
        const int head = (int)(bit0 & 31), nw = (int)(((bit1 + 31) >> 5) - w0), nv = qn * g.neri;
        for (int w = tid; w < nw; w += kGenThreads) {
            const int b0 = w * 32 - head;
            int c = b0 <= 0 ? 0 : (int)((unsigned)b0 / (unsigned)bits);
            uint32_t word = 0u;
            for (int s = c * bits - b0; s < 32 && c < nv; ++c, s += bits) {
                double r = round(vals[c] * inv_s[div_by(c, g.m_neri)]);
                r = r > M ? M : (r < -M ? -M : r);
                const uint32_t code = (uint32_t)(int)r & mask;
                word |= s >= 0 ? code << s : code >> (-s);
            }
            if (b0 >= 0 && b0 + 32 <= nv * bits)
                a.packed[w0 + w] = word;
            else
                atomicOr(a.packed + w0 + w, word);
        }
        __syncthreads();
    }
}

template <typename R>
__global__ void __launch_bounds__(kGenThreads)
eri_queue_kernel(ShellsDev sh, Tables tb, const QueueClass *__restrict__ classes, int n_classes,
                 long long n_tiles, unsigned long long *counter, double *__restrict__ scratch,
                 long long slot_doubles, int bits) {
    extern __shared__ __align__(16) unsigned char smem[];
    queue_tiles<R>(sh, tb, classes, n_classes, n_tiles, counter, scratch, slot_doubles, bits, smem);
}

// The same with the class table as a kernel parameter: calls over all classes run the classes with a g
// shell in sets of kGenericSet while they are small.  They keep no table on the device for it, and a
// captured launch carries its own.  With two launches per class the 369 classes took 3.24 ms however
// few their quartets; at 2^15 ERIs per class in sets 0.42 ms, bound by the quadrature of generic_tile.
struct GenSet {
    QueueClass c[kGenericSet];
};
static_assert(sizeof(GenSet) + 512 <= 32764, "kernel parameters");

template <typename R>
__global__ void __launch_bounds__(kGenThreads)
eri_generic_set_kernel(ShellsDev sh, Tables tb, const __grid_constant__ GenSet set, int n_classes, long long n_tiles,
                       unsigned long long *counter, double *__restrict__ scratch, long long slot_doubles, int bits) {
    extern __shared__ __align__(16) unsigned char smem[];
    queue_tiles<R>(sh, tb, set.c, n_classes, n_tiles, counter, scratch, slot_doubles, bits, smem);
}

// Table of a queue (n classes, into qc) and what its launch takes.
struct QueueShape {
    long long tiles = 0, slot = 1;  // tiles; FP64 values of the largest
    int smem = 0;
};

QueueShape queue_table(const QueueSpec *classes, int n, bool mixed, bool contracted, QueueClass *qc) {
    // the classes with the most work per quartet first: a long quartet of a high class that starts last
    // keeps one CTA busy after all others are done (5 of 6.5 ms on a 40-atom molecule's 8,000 quartets)
    std::vector<int> order(n);
    for (int i = 0; i < n; ++i) order[i] = i;
    auto work = [&](int i) {
        const int *L = classes[i].L;
        return (L[0] + L[1] + L[2] + L[3] + 2) * ncart(L[0]) * ncart(L[1]) * ncart(L[2]) * ncart(L[3]);
    };
    std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return work(x) > work(y); });
    QueueShape s;
    for (int i = 0; i < n; ++i) {
        const QueueSpec &c = classes[order[i]];
        qc[i].a = c.a;
        qc[i].g = mixed ? gen_shape<float>(c.L, contracted) : gen_shape<double>(c.L, contracted);
        qc[i].first_tile = s.tiles;
        s.tiles += (c.a.nq + qc[i].g.q - 1) / qc[i].g.q;
        s.smem = std::max(s.smem, qc[i].g.smem);
        s.slot = std::max(s.slot, (long long)qc[i].g.q * qc[i].g.neri);
    }
    return s;
}

// Grid of a queue: the CTAs that the GPU holds at a time, as far as there are tiles and slots for them.
template <class K>
cudaError_t queue_grid(K kern, const QueueShape &s, size_t scratch_bytes, int device, long long *grid) {
    int per_sm = 0, sms = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kGenThreads, s.smem);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device);
    if (e != cudaSuccess) return e;
    *grid = std::min<long long>(s.tiles, (long long)std::max(1, per_sm) * sms);
    *grid = std::min<long long>(*grid, (long long)(scratch_bytes / (sizeof(double) * (size_t)s.slot)));
    return *grid < 1 ? cudaErrorInvalidValue : cudaSuccess;
}

template <typename R>
cudaError_t run_set(const ShellsDev &sh, const Tables &tb, const QueueSpec *classes, int n, bool contracted, int bits,
                    void *scratch, size_t scratch_bytes, int device, cudaStream_t stream) {
    constexpr size_t kHead = 256;  // the counter, ahead of the slots
    GenSet set;
    const QueueShape s = queue_table(classes, n, sizeof(R) == 4, contracted, set.c);
    if (s.smem > kGenSmemLimit || s.tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
    auto kern = eri_generic_set_kernel<R>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kGenSmemLimit);
    if (e != cudaSuccess) return e;
    long long grid = s.tiles;
    if (bits) {
        if (!scratch || scratch_bytes <= kHead) return cudaErrorInvalidValue;
        if ((e = queue_grid(kern, s, scratch_bytes - kHead, device, &grid)) != cudaSuccess) return e;
        if ((e = cudaMemsetAsync(scratch, 0, sizeof(unsigned long long), stream)) != cudaSuccess) return e;
    }
    kern<<<(unsigned)grid, kGenThreads, s.smem, stream>>>(
        sh, tb, set, n, s.tiles, static_cast<unsigned long long *>(scratch),
        bits ? reinterpret_cast<double *>(static_cast<char *>(scratch) + kHead) : nullptr, s.slot, bits);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_queue(const ShellsDev &sh, const Tables &tb, const QueueSpec *classes, int n_classes,
                         bool mixed, bool contracted, int bits, void *d_table, unsigned long long *d_counter,
                         double *scratch, size_t scratch_bytes, int device, cudaStream_t stream) {
    if (n_classes <= 0) return cudaSuccess;
    std::vector<QueueClass> qc(n_classes);
    const QueueShape s = queue_table(classes, n_classes, mixed, contracted, qc.data());
    if (s.smem > kGenSmemLimit) return cudaErrorInvalidValue;
    auto kern = mixed ? eri_queue_kernel<float> : eri_queue_kernel<double>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kGenSmemLimit);
    if (e != cudaSuccess) return e;
    long long grid = 0;
    if ((e = queue_grid(kern, s, scratch_bytes, device, &grid)) != cudaSuccess) return e;
    if ((size_t)n_classes * sizeof(QueueClass) > queue_table_bytes()) return cudaErrorInvalidValue;
    e = cudaMemcpyAsync(d_table, qc.data(), (size_t)n_classes * sizeof(QueueClass), cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(d_counter, 0, sizeof(unsigned long long), stream);
    if (e != cudaSuccess) return e;
    kern<<<(unsigned)grid, kGenThreads, s.smem, stream>>>(sh, tb, static_cast<const QueueClass *>(d_table), n_classes,
                                                          s.tiles, d_counter, scratch, s.slot, bits);
    return cudaGetLastError();
}

cudaError_t launch_generic_set(const ShellsDev &sh, const Tables &tb, const QueueSpec *classes, int n, bool mixed,
                               bool contracted, int bits, void *scratch, size_t scratch_bytes, int device,
                               cudaStream_t stream) {
    if (n <= 0) return cudaSuccess;
    if (n > kGenericSet) return cudaErrorInvalidValue;
    return mixed ? run_set<float>(sh, tb, classes, n, contracted, bits, scratch, scratch_bytes, device, stream)
                 : run_set<double>(sh, tb, classes, n, contracted, bits, scratch, scratch_bytes, device, stream);
}

size_t queue_table_bytes() { return (size_t)kNumClassIds * sizeof(QueueClass); }

cudaError_t launch_generic(const ShellsDev &sh, const Tables &tb, const ClassArgs &a, const int L[4],
                           bool mixed, bool contracted, double *scratch, size_t scratch_bytes,
                           int n_streams, cudaStream_t stream) {
    if (a.nq <= 0) return cudaSuccess;
    // two tiles per SM of the stream's share at least: one tile's stages take the same time however few
    // the others are (the canonical classes one at a time at 2^18 ERIs, FP64 10.4 -> 4.2 ms, FP32 with 16-bit
    // codes 6.6 -> 4.3; with full tiles and the rules of gen_shape FP64 took 8.0)
    const long long share = 2 * 152 / n_streams;
    const int q_most = (int)std::min<long long>(kGenQmax, (a.nq + share - 1) / share);
    const GenShape g = mixed ? gen_shape<float>(L, contracted, q_most) : gen_shape<double>(L, contracted, q_most);
    if (g.smem > kGenSmemLimit) return cudaErrorInvalidValue;
    if (a.out_fp64)
        return mixed ? run_values<float>(sh, tb, a, g, a.out_fp64, stream)
                     : run_values<double>(sh, tb, a, g, a.out_fp64, stream);
    const long long chunk = chunk_quartets(g.neri, scratch_bytes);
    if (chunk < 32 || !scratch) return cudaErrorInvalidValue;
    for (long long c0 = 0; c0 < a.nq; c0 += chunk) {
        ClassArgs ac = a;
        ac.quartets = a.quartets + c0;
        ac.nq = std::min(chunk, a.nq - c0);
        cudaError_t e = mixed ? run_values<float>(sh, tb, ac, g, scratch, stream)
                              : run_values<double>(sh, tb, ac, g, scratch, stream);
        if (e != cudaSuccess) return e;
        const long long w0 = c0 * g.neri * a.bits / 32;
        ac.packed = a.packed + w0;
        ac.scales = a.scales + c0;
        ac.seg_words = (c0 + ac.nq == a.nq) ? a.seg_words - w0 : ac.nq * g.neri * a.bits / 32;
        if ((e = pack_values(ac, g.neri, scratch, stream)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

int generic_launches(long long nq, int neri, bool compressed, size_t scratch_bytes) {
    if (nq <= 0) return 0;
    if (!compressed) return 1;
    const long long chunk = chunk_quartets(neri, scratch_bytes);
    return chunk > 0 ? 2 * (int)((nq + chunk - 1) / chunk) : 0;
}

const char *generic_kernel_names(bool mixed, bool compressed) {
    if (compressed)
        return mixed ? "eri_generic_kernel<float> + pack_kernel<double>" : "eri_generic_kernel<double> + pack_kernel<double>";
    return mixed ? "eri_generic_kernel<float>" : "eri_generic_kernel<double>";
}

}  // namespace eri
