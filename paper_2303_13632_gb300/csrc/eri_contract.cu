// eri_contract.cu -- contracted quartets as sums over primitive quartets.
//
// A contracted quartet (Sec. II-A) is the sum of nprim_a nprim_b nprim_c nprim_d primitive ones,
// from one to over a thousand of them, uneven within a class.  Walking them one after the other in
// the CTA that owns the quartet leaves the GPU to the longest quartet and the few threads of each
// phase; here every primitive quartet is a unit of its own, as in a primitive plan:
//   unit_setup_kernel   one thread per unit: geometry, roots and weights, B and C (FP64)
//   class kernel        the class's recurrence and quadrature kernel over the units' records
//   contract_kernel     one thread per (quartet, output): the sum over the quartet's units, in
//                       order, so that the FP32 Kahan sums are those of a sequential loop
//   pack_kernel         b_max, eps and the codes of the finished quartets (compressed output)
// The values of a unit pass through memory once in each direction (8 n_ERIQ bytes in FP32), little
// next to the n_Rys n_ERIQ multiply-adds behind them.  The units of a class are cut into spans that
// fill the scratch; a quartet may be cut, its partial sums are carried to the next span.
//
// Measured against the primitive loop inside the class kernel: a diatomic's 3,081 unique quartets
// (s, s, p, p, d, f per atom, K up to 6, FP64) 501 -> 5.4 ms; 70,000 quartets of a 40-atom molecule
// (K up to 6, FP32, 16-bit codes) 300 -> 10.3 ms, same codes bit for bit.  The sums are bound by the
// latency of a long quartet's chain: with 32 values of a chain in flight instead of 8 those two
// fell from 7.1 and 11.6 ms.
#include <algorithm>
#include <type_traits>

#include "eri_internal.h"
#include "eri_kernels.cuh"

namespace eri {

namespace {

constexpr int kThreads = 256;
constexpr int kBatch = 32;  // units a thread of contract_kernel loads ahead of their sum

template <bool AB, bool CD>
struct UnitGeo {
    static constexpr bool SWAB_OK = AB, SWCD_OK = CD;
};

// last quartet q in [lo, hi] whose first unit is <= u
__device__ __forceinline__ int quartet_of(const long long *__restrict__ ps, long long base, long long u,
                                          int lo, int hi) {
    while (lo < hi) {
        const int mid = lo + (hi - lo + 1) / 2;
        if (__ldg(ps + mid) - base <= u) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__global__ void unit_counts_kernel(const int4 *__restrict__ q, long long n, const int *__restrict__ nprim,
                                   long long *__restrict__ out) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i > n) return;
    if (i == n) {
        out[i] = 0;
        return;
    }
    const int4 t = q[i];
    out[i] = (long long)nprim[t.x] * nprim[t.y] * nprim[t.z] * nprim[t.w];
}

// The records of eri_setup_kernel for the units of a span, the B and C values formed in FP64 and
// rounded (as phase_setup).
template <typename R, bool SWAB, bool SWCD>
__global__ void __launch_bounds__(128)
unit_setup_kernel(ShellsDev sh, Tables tb, ClassArgs args, KernelInfo k, UnitSpan span, R *out, int st) {
    __shared__ int range_s[2];
    const int first = blockIdx.x * 128, last = min(first + 127, span.nu - 1);
    const long long base = span.ps[0];
    if (threadIdx.x < 2)
        range_s[threadIdx.x] = quartet_of(span.ps, base, span.u0 + (threadIdx.x ? last : first), 0, (int)span.nq - 1);
    __syncthreads();
    const int u = first + threadIdx.x;
    if (u > last) return;
    const int q = quartet_of(span.ps, base, span.u0 + u, range_s[0], range_s[1]);
    const int prim = (int)(span.u0 + u - (__ldg(span.ps + q) - base));
    const int4 g = args.quartets[q];
    const int4 qt = make_int4(pick(g, args.perm[0]), pick(g, args.perm[1]), pick(g, args.perm[2]),
                              pick(g, args.perm[3]));
    double geo[G_N];
    int np = 0;
    geometry_of<UnitGeo<SWAB, SWCD>>(sh, args, qt, prim, geo, np);
    R *o = out + u;
    o[0 * st] = to_r<R>(geo[G_ABX]);
    o[1 * st] = to_r<R>(geo[G_ABY]);
    o[2 * st] = to_r<R>(geo[G_ABZ]);
    o[3 * st] = to_r<R>(geo[G_CDX]);
    o[4 * st] = to_r<R>(geo[G_CDY]);
    o[5 * st] = to_r<R>(geo[G_CDZ]);
    o[6 * st] = to_r<R>(geo[G_SWAB]);
    o[7 * st] = to_r<R>(geo[G_SWCD]);
    o += kSetupGeo * st;
    if (k.ltot == 0) {
        double F0, F1;
        if constexpr (sizeof(R) == 4)
            boys_f01_mixed<false>(geo[G_T], tb.boys_t01, tb.boys_t01_f, F0, F1);
        else
            boys_f01<false>(geo[G_T], tb.boys_t01, F0, F1);
        for (int f = 0; f < S_WZ; ++f) o[f * st] = (R)0;
        o[S_WZ * st] = to_r<R>(geo[G_PREF] * F0);
        return;
    }
    const double p = geo[G_P], q2 = geo[G_Q], ipq = geo[G_IPQ];
#pragma unroll 1
    for (int mu = 0; mu < k.nrys; ++mu, o += k.sn * st) {
        double x, w;
        rys_root<sizeof(R) == 4>(tb, k.nrys, mu, geo[G_T], x, w);
        const double fq = q2 * x * ipq, fp = p * x * ipq;
        o[S_WZ * st] = to_r<R>(geo[G_PREF] * w);
        o[S_B00 * st] = to_r<R>(0.5 * x * ipq);
        o[S_B10 * st] = to_r<R>((1.0 - fq) * (0.5 * geo[G_IP]));
        o[S_B01 * st] = to_r<R>((1.0 - fp) * (0.5 * geo[G_IQ]));
#pragma unroll
        for (int s = 0; s < 3; ++s) {
            const double pq = geo[G_PQX + s];
            o[(S_C0X + s) * st] = to_r<R>(geo[G_PAX + s] - fq * pq);
            o[(S_C1X + s) * st] = to_r<R>(geo[G_QCX + s] + fp * pq);
        }
        if constexpr (sizeof(R) == 4) {
            if (k.cb)
#pragma unroll
                for (int s = 0; s < 3; ++s)
                    o[(k.cb + s) * st] = to_r<R>((geo[G_PAX + s] + geo[G_ABX + s]) - fq * geo[G_PQX + s]);
            if (k.cd)
#pragma unroll
                for (int s = 0; s < 3; ++s)
                    o[(k.cd + s) * st] = to_r<R>((geo[G_QCX + s] + geo[G_CDX + s]) + fp * geo[G_PQX + s]);
        }
    }
}

// One thread per (quartet of the span, output): the sum over the quartet's units in order (for
// R = float the Kahan sum of a sequential loop).  The loads of a quartet's units are independent
// and one n_ERIQ row apart, so neighbouring threads read neighbouring values.
template <typename R, bool OUT64>
__global__ void __launch_bounds__(kThreads)
contract_kernel(ClassArgs args, int neri, UnitSpan span, R *values, R *carry, int parity) {
    __shared__ int q_s[2];
    const long long base = span.ps[0], u1 = span.u0 + span.nu;
    if (threadIdx.x < 2)
        q_s[threadIdx.x] = quartet_of(span.ps, base, threadIdx.x ? u1 - 1 : span.u0, 0, (int)span.nq - 1);
    __syncthreads();
    const unsigned int n = (unsigned int)(q_s[1] - q_s[0] + 1) * (unsigned int)neri;
    const R *cin = carry + (size_t)parity * 2 * neri;
    R *cout = carry + (size_t)(1 - parity) * 2 * neri;
    bool bad = false;
    for (unsigned int t = blockIdx.x * kThreads + threadIdx.x; t < n; t += gridDim.x * kThreads) {
        const int q = q_s[0] + (int)(t / (unsigned int)neri), o = (int)(t % (unsigned int)neri);
        const long long f = __ldg(span.ps + q) - base, l = __ldg(span.ps + q + 1) - base;
        const int a = (int)(max(f, span.u0) - span.u0), b = (int)(min(l, u1) - span.u0);
        const R *v = values + (size_t)a * neri + o;
        R acc = (R)0, comp = (R)0;
        int left = b - a;
        if (f < span.u0) {
            acc = cin[o];
            if constexpr (sizeof(R) == 4) comp = cin[neri + o];
        } else {
            acc = *v;
            v += neri;
            --left;
        }
        // kBatch loads in flight: the chain of sums of a long quartet waits on memory otherwise
        R x[kBatch];
        for (; left > 0; left -= kBatch, v += (size_t)kBatch * neri) {
#pragma unroll
            for (int i = 0; i < kBatch; ++i)
                if (i < left) x[i] = v[(size_t)i * neri];
#pragma unroll
            for (int i = 0; i < kBatch; ++i)
                if (i < left) {
                    if constexpr (sizeof(R) == 4) {
                        const R y = __fsub_rn(x[i], comp);
                        const R s = __fadd_rn(acc, y);
                        comp = __fsub_rn(__fsub_rn(s, acc), y);
                        acc = s;
                    } else {
                        acc += x[i];
                    }
                }
        }
        if (l > u1) {
            cout[o] = acc;
            if constexpr (sizeof(R) == 4) cout[neri + o] = comp;
        } else {
            bad |= !RTraits<R>::finite(acc);
            if constexpr (OUT64)
                args.out_fp64[(long long)q * neri + o] = RTraits<R>::to_f64(acc);
            else
                values[(size_t)a * neri + o] = acc;
        }
    }
    if (bad) atomicOr(args.err, 1);
}

// b_max, eps (Eq. 9) and codes (Eq. 10) of the quartets that end in the span, qt per CTA, with the
// arithmetic of the class kernels' epilogue in the value type; one thread packs one output word.
// Words shared with a neighbouring tile are merged with atomics on the tile's own bits.
template <typename R>
__global__ void __launch_bounds__(kThreads)
pack_kernel(ClassArgs args, int neri, int qt, UnitSpan span, const R *__restrict__ values) {
    constexpr int kMaxQ = 128;
    __shared__ int q_s[2];
    __shared__ int slot_s[kMaxQ];
    __shared__ R inv_s[kMaxQ];
    __shared__ unsigned long long part_raw_s[kThreads / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long base = span.ps ? span.ps[0] : 0, u1 = span.u0 + span.nu;
    if (tid == 0) {
        if (span.ps) {
            q_s[0] = quartet_of(span.ps, base, span.u0, 0, (int)span.nq - 1);
            int b = quartet_of(span.ps, base, u1 - 1, 0, (int)span.nq - 1);
            if (span.ps[b + 1] - base > u1) --b;  // continues in the next span
            q_s[1] = b;
        } else {  // values of whole quartets
            q_s[0] = 0;
            q_s[1] = span.nu - 1;
        }
    }
    __syncthreads();
    const long long q0 = q_s[0] + (long long)blockIdx.x * qt;
    if (q0 > q_s[1]) return;
    const int qn = (int)min((long long)qt, q_s[1] + 1 - q0);
    const int bits = args.bits;
    const R M = (R)((1u << (bits - 1)) - 1u);
    for (int q = tid; q < qn; q += kThreads)
        slot_s[q] = span.ps ? (int)(max(span.ps[q0 + q] - base, span.u0) - span.u0) : (int)(q0 + q);
    __syncthreads();
    // non-negative IEEE values order like their bit patterns (and a NaN stays the largest)
    using U = std::conditional_t<sizeof(R) == 8, unsigned long long, unsigned int>;
    U *part_s = reinterpret_cast<U *>(part_raw_s);
    auto absbits = [](R x) -> U {
        if constexpr (sizeof(R) == 8)
            return (U)__double_as_longlong(x) & 0x7fffffffffffffffull;
        else
            return (U)__float_as_uint(x) & 0x7fffffffu;
    };
    auto finish = [&](int q, U u) {
        R m;
        if constexpr (sizeof(R) == 8)
            m = __longlong_as_double((long long)u);
        else
            m = __uint_as_float(u);
        float eps;
        R inv;
        if constexpr (sizeof(R) == 8) {
            eps = (float)(m / M);
            inv = eps > 0.0f ? (R)(1.0 / (double)eps) : (R)0;
        } else {
            eps = m / M;
            inv = eps > 0.0f ? (R)(1.0f / eps) : (R)0;
        }
        args.scales[q0 + q] = eps;
        inv_s[q] = inv;
    };
    if (neri >= 512) {  // all threads on one quartet
        for (int q = 0; q < qn; ++q) {
            const R *v = values + (size_t)slot_s[q] * neri;
            U m = 0;
            for (int o = tid; o < neri; o += kThreads) m = max(m, absbits(v[o]));
            for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, off));
            if (lane == 0) part_s[warp] = m;
            __syncthreads();
            if (tid == 0) {
                for (int w = 1; w < kThreads / 32; ++w) m = max(m, part_s[w]);
                finish(q, m);
            }
            __syncthreads();
        }
    } else {  // a warp per quartet
        for (int q = warp; q < qn; q += kThreads / 32) {
            const R *v = values + (size_t)slot_s[q] * neri;
            U m = 0;
            for (int o = lane; o < neri; o += 32) m = max(m, absbits(v[o]));
            for (int off = 16; off > 0; off >>= 1) m = max(m, __shfl_down_sync(0xffffffffu, m, off));
            if (lane == 0) finish(q, m);
        }
        __syncthreads();
    }
    const uint32_t mask = (1u << bits) - 1u;
    const long long bit0 = q0 * (long long)neri * bits, bit1 = (q0 + qn) * (long long)neri * bits;
    const long long w0 = bit0 >> 5, w1 = (bit1 + 31) >> 5;
    const int head = (int)(bit0 & 31), nw = (int)(w1 - w0), nv = qn * neri;
    const bool last_tile = q0 + qn >= span.nq;
    const int tail = (int)(bit1 & 31);
    for (int w = tid; w < nw; w += kThreads) {
        // tile bit of the word's first bit, and the codes that reach into the word
        const int b0 = w * 32 - head;
        int c = b0 <= 0 ? 0 : (int)((unsigned int)b0 / (unsigned int)bits);
        uint32_t word = 0u;
        for (int s = c * bits - b0; s < 32 && c < nv; ++c, s += bits) {
            const int q = (int)((unsigned int)c / (unsigned int)neri);
            R r = RTraits<R>::round_away(values[(size_t)slot_s[q] * neri + (c - q * neri)] * inv_s[q]);
            r = r > M ? M : (r < -M ? -M : r);
            const uint32_t code = to_code<R>(r, bits) & mask;
            word |= s >= 0 ? code << s : code >> (-s);
        }
        uint32_t keep = 0xffffffffu;  // bits of this word owned by this tile
        if (w == 0 && head) keep &= ~((1u << head) - 1u);
        if (w == nw - 1 && tail && !last_tile) keep &= (1u << tail) - 1u;
        if (keep == 0xffffffffu) {
            args.packed[w0 + w] = word;
        } else {
            atomicAnd(args.packed + w0 + w, ~keep);
            atomicOr(args.packed + w0 + w, word & keep);
        }
    }
    if (last_tile)
        for (long long w = w1 + tid; w < args.seg_words; w += kThreads) args.packed[w] = 0u;
}

template <typename R>
cudaError_t setup_r(const ShellsDev &sh, const Tables &tb, const ClassArgs &a, const KernelInfo &k,
                    const UnitSpan &span, R *rec, int stride, cudaStream_t s) {
    const unsigned blocks = (unsigned)((span.nu + 127) / 128);
    if (k.swab && k.swcd)
        unit_setup_kernel<R, true, true><<<blocks, 128, 0, s>>>(sh, tb, a, k, span, rec, stride);
    else if (k.swab)
        unit_setup_kernel<R, true, false><<<blocks, 128, 0, s>>>(sh, tb, a, k, span, rec, stride);
    else if (k.swcd)
        unit_setup_kernel<R, false, true><<<blocks, 128, 0, s>>>(sh, tb, a, k, span, rec, stride);
    else
        unit_setup_kernel<R, false, false><<<blocks, 128, 0, s>>>(sh, tb, a, k, span, rec, stride);
    return cudaGetLastError();
}

// nq: quartets the span can hold at most
template <typename R>
cudaError_t pack_r(const ClassArgs &a, int neri, long long nq, const UnitSpan &span, const R *values, cudaStream_t s) {
    const int qt = std::max(1, std::min(128, 4096 / neri));
    pack_kernel<R><<<(unsigned)((nq + qt - 1) / qt), kThreads, 0, s>>>(a, neri, qt, span, values);
    return cudaGetLastError();
}

template <typename R>
cudaError_t contract_r(const ClassArgs &a, int neri, const UnitSpan &span, R *values, R *carry, int parity,
                       cudaStream_t s) {
    // quartets the span can touch
    const long long nq = std::min<long long>(span.nq, (long long)span.nu + 1);
    const unsigned blocks = (unsigned)std::min<long long>((nq * neri + kThreads - 1) / kThreads, 152LL * 16);
    if (a.out_fp64) {
        contract_kernel<R, true><<<blocks, kThreads, 0, s>>>(a, neri, span, values, carry, parity);
        return cudaGetLastError();
    }
    contract_kernel<R, false><<<blocks, kThreads, 0, s>>>(a, neri, span, values, carry, parity);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return pack_r(a, neri, nq, span, values, s);
}

}  // namespace

cudaError_t unit_counts(const int4 *q, long long n, const int *nprim, long long *out, cudaStream_t s) {
    unit_counts_kernel<<<(unsigned)((n + 256) / 256), 256, 0, s>>>(q, n, nprim, out);
    return cudaGetLastError();
}

cudaError_t unit_setup(const ShellsDev &sh, const Tables &tb, const ClassArgs &a, const KernelInfo &k,
                       bool mixed, const UnitSpan &span, void *records, int stride, cudaStream_t s) {
    return mixed ? setup_r(sh, tb, a, k, span, static_cast<float *>(records), stride, s)
                 : setup_r(sh, tb, a, k, span, static_cast<double *>(records), stride, s);
}

cudaError_t pack_values(const ClassArgs &a, int neri, const double *values, cudaStream_t s) {
    UnitSpan whole{};
    whole.nq = a.nq;
    whole.nu = (int)a.nq;
    return pack_r(a, neri, a.nq, whole, values, s);
}

cudaError_t unit_contract(const ClassArgs &a, bool mixed, int neri, const UnitSpan &span, void *values,
                          void *carry, int parity, cudaStream_t s) {
    return mixed ? contract_r(a, neri, span, static_cast<float *>(values), static_cast<float *>(carry), parity, s)
                 : contract_r(a, neri, span, static_cast<double *>(values), static_cast<double *>(carry), parity, s);
}

}  // namespace eri
