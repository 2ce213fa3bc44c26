// eri_contract.cu -- contracted quartets as sums over primitive quartets.
//
// A contracted quartet (Sec. II-A) is the sum of nprim_a nprim_b nprim_c nprim_d primitive ones,
// from one to over a thousand of them, uneven within a class.  Walking them one after the other in
// the CTA that owns the quartet leaves the GPU to the longest quartet and the few threads of each
// phase; here every primitive quartet is a unit of its own, as in a primitive plan:
//   unit_setup_kernel   one thread per unit: geometry; then one per (unit, root): root and weight, B and
//                       C (FP64)
//   class kernel        the class's recurrence and quadrature kernel over the units' records
//   contract_kernel     one thread per (quartet, output): the sum over the quartet's units, in
//                       order, so that the FP32 Kahan sums are those of a sequential loop
//   pack_kernel         b_max, eps and the codes of the finished quartets (compressed output)
// The values of a unit pass through memory once in each direction (8 n_ERIQ bytes in FP32), little
// next to the n_Rys n_ERIQ multiply-adds behind them.  The units of a class are cut into spans that
// fill the scratch; a quartet may be cut, its partial sums are carried to the next span.
//
// Measured against the primitive loop inside the class kernel: a diatomic's 3,081 unique quartets
// (s, s, p, p, d, f per atom, K up to 6, FP64) 501 -> 3.2 ms; 70,000 quartets of a 40-atom molecule
// (K up to 6, FP32, 16-bit codes) 300 -> 8.6 ms, same codes bit for bit.  The sums are bound by the
// latency of a long quartet's chain: kBatch values of it are added while the next kBatch are loaded
// (with 32 values in flight instead of 8, before the setup ran by (unit, root), those two fell from 7.1
// and 11.6 to 5.4 and 10.3 ms).
#include <algorithm>
#include <type_traits>

#include "eri_internal.h"
#include "eri_kernels.cuh"

namespace eri {

namespace {

constexpr int kThreads = 256;
constexpr int kBatch = 24;  // units a thread of contract_kernel loads at a time

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

// The same by the lanes of a warp: 32 probes at a time, so that a search of a class's quartets waits
// for memory two or three times instead of a dozen (8 of the 19 us of a small pack_kernel).
__device__ __forceinline__ int quartet_of_warp(const long long *__restrict__ ps, long long base, long long u,
                                               int lo, int hi) {
    const int lane = threadIdx.x & 31;
    while (lo < hi) {
        const int step = (hi - lo + 31) / 32;  // probes lo + step, lo + 2 step, .. (those above hi fail)
        const long long at = lo + (long long)(lane + 1) * step;
        const bool le = at <= hi && __ldg(ps + at) - base <= u;
        const int n = __popc(__ballot_sync(0xffffffffu, le));  // the prefix sum ascends
        const long long next = lo + (long long)(n + 1) * step - 1;
        lo += n * step;
        hi = next < hi ? (int)next : hi;
    }
    return lo;
}

// Quartets of the span's first and last unit, to q_s[0] and q_s[1] (warps 0 and 1; a barrier follows).
__device__ __forceinline__ void span_quartets(const UnitSpan &span, long long base, long long first,
                                              long long last, int *q_s) {
    const int warp = threadIdx.x >> 5;
    if (warp < 2) {
        const int q = quartet_of_warp(span.ps, base, warp ? last : first, 0, (int)span.nq - 1);
        if ((threadIdx.x & 31) == 0) q_s[warp] = q;
    }
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

__global__ void class_ends_kernel(const long long *__restrict__ ps, const __grid_constant__ ClassEnds at,
                                  long long *__restrict__ ends) {
    for (int c = threadIdx.x; c < kNumClassIds; c += blockDim.x) ends[c] = ps[at.i[c]];
}

// Setup records of the units of a span, B and C formed in FP64 and rounded (as phase_setup): geometry
// by one thread per unit, then roots, weights, B and C by one per (unit, root).  kSetupUnits units per
// CTA: a warp for the geometry, all four for the roots, stores coalesced over the units.  Bound by the
// FP64 pipe on many units, by the latency of its chains on few: with one thread walking the roots of a
// unit a class of some hundred quartets took about 30 us.
constexpr int kSetupUnits = 32;

template <typename R, bool SWAB, bool SWCD>
__global__ void __launch_bounds__(128)
unit_setup_kernel(ShellsDev sh, Tables tb, ClassArgs args, KernelInfo k, UnitSpan span, R *out, int st) {
    __shared__ int range_s[2];
    __shared__ double geo_s[kSetupUnits * G_N];
    const int first = blockIdx.x * kSetupUnits, n = min(kSetupUnits, span.nu - first), tid = threadIdx.x;
    out += first;
    if (span.ps) {
        const long long base = span.ps[0];
        span_quartets(span, base, span.u0 + first, span.u0 + first + n - 1, range_s);
        __syncthreads();
    }
    if (tid < n) {
        int q = first + tid, prim = 0;
        if (span.ps) {
            const long long base = span.ps[0], u = span.u0 + first + tid;
            q = quartet_of(span.ps, base, u, range_s[0], range_s[1]);
            prim = (int)(u - (__ldg(span.ps + q) - base));
        }
        const int4 g = args.quartets[q];
        const int4 qt = make_int4(pick(g, args.perm[0]), pick(g, args.perm[1]), pick(g, args.perm[2]),
                                  pick(g, args.perm[3]));
        double *geo = geo_s + tid * G_N;
        int np = 0;
        geometry_of<UnitGeo<SWAB, SWCD>>(sh, args, qt, prim, geo, np);
        if (!k.direct) {  // the four-index path reads no transfer vectors
            R *o = out + tid;
            o[0 * st] = to_r<R>(geo[G_ABX]);
            o[1 * st] = to_r<R>(geo[G_ABY]);
            o[2 * st] = to_r<R>(geo[G_ABZ]);
            o[3 * st] = to_r<R>(geo[G_CDX]);
            o[4 * st] = to_r<R>(geo[G_CDY]);
            o[5 * st] = to_r<R>(geo[G_CDZ]);
            o[6 * st] = to_r<R>(geo[G_SWAB]);
            o[7 * st] = to_r<R>(geo[G_SWCD]);
        }
    }
    __syncthreads();
    out += kSetupGeo * st;
    for (int it = tid; it < kSetupUnits * k.nrys; it += 128) {
        const int u = it % kSetupUnits, mu = it / kSetupUnits;
        if (u >= n) continue;
        const double *geo = geo_s + u * G_N;
        R *o = out + mu * k.sn * st + u;
        if (k.ltot == 0) {
            double F0, F1;
            if constexpr (sizeof(R) == 4)
                boys_f01_mixed<false>(geo[G_T], tb.boys_t01, tb.boys_t01_f, F0, F1);
            else
                boys_f01<false>(geo[G_T], tb.boys_t01, F0, F1);
            for (int f = 0; f < S_WZ; ++f) o[f * st] = (R)0;
            o[S_WZ * st] = to_r<R>(geo[G_PREF] * F0);
            continue;
        }
        double x, w;
        rys_root<sizeof(R) == 4>(tb, k.nrys, mu, geo[G_T], x, w);
        const double ipq = geo[G_IPQ];
        const double fq = geo[G_Q] * x * ipq, fp = geo[G_P] * x * ipq;
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
            if (k.cb) {
#pragma unroll
                for (int s = 0; s < 3; ++s)
                    o[(k.cb + s) * st] = to_r<R>((geo[G_PAX + s] + geo[G_ABX + s]) - fq * geo[G_PQX + s]);
            }
            if (k.cd) {
#pragma unroll
                for (int s = 0; s < 3; ++s)
                    o[(k.cd + s) * st] = to_r<R>((geo[G_QCX + s] + geo[G_CDX + s]) + fp * geo[G_PQX + s]);
            }
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
    span_quartets(span, base, span.u0, u1 - 1, q_s);
    __syncthreads();
    const unsigned int n = (unsigned int)(q_s[1] - q_s[0] + 1) * (unsigned int)neri;
    // two halves of kCarryBytes: a sum and, in FP32, its compensation per output
    constexpr int kHalf = sizeof(R) == 4 ? 2 : 1;
    const R *cin = carry + (size_t)parity * kHalf * neri;
    R *cout = carry + (size_t)(1 - parity) * kHalf * neri;
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
        // the loads of the next kBatch units are under way while one batch is summed: the chain of a
        // long quartet waits on memory otherwise
        R x[kBatch], y2[kBatch];
        auto fetch = [&](R (&d)[kBatch], int n) {
#pragma unroll
            for (int i = 0; i < kBatch; ++i)
                if (i < n) d[i] = v[(size_t)i * neri];
            v += (size_t)kBatch * neri;
        };
        auto sum = [&](const R (&d)[kBatch], int n) {
#pragma unroll
            for (int i = 0; i < kBatch; ++i)
                if (i < n) {
                    if constexpr (sizeof(R) == 4) {
                        const R y = __fsub_rn(d[i], comp);
                        const R s = __fadd_rn(acc, y);
                        comp = __fsub_rn(__fsub_rn(s, acc), y);
                        acc = s;
                    } else {
                        acc += d[i];
                    }
                }
        };
        fetch(x, left);
        while (left > 0) {
            fetch(y2, left - kBatch);
            sum(x, left);
            left -= kBatch;
            if (left <= 0) break;
            fetch(x, left - kBatch);
            sum(y2, left);
            left -= kBatch;
        }
        if (l > u1) {
            cout[o] = acc;
            if constexpr (sizeof(R) == 4) cout[neri + o] = comp;
        } else {
            // the zeros up to the longest quartet of the group: a Kahan step with zero changes the sum
            // only where the compensation left over rounds it to a neighbour, so the others are not searched
            if constexpr (sizeof(R) == 4) {
                if (__fsub_rn(acc, comp) != acc) {
                    const long long g0 = (long long)(q / span.group) * span.group;
                    const long long g1 = min(g0 + span.group, span.nq);
                    long long longest = 0;
                    for (long long i = g0; i < g1; ++i) longest = max(longest, __ldg(span.ps + i + 1) - __ldg(span.ps + i));
                    for (long long i = l - f; i < longest; ++i) {
                        const R y = -comp, s = __fadd_rn(acc, y);
                        if (!(s != acc)) break;
                        comp = __fsub_rn(__fsub_rn(s, acc), y);
                        acc = s;
                    }
                }
            }
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
    if (span.ps) {
        span_quartets(span, base, span.u0, u1 - 1, q_s);
        __syncthreads();
        if (tid == 0 && span.ps[q_s[1] + 1] - base > u1) --q_s[1];  // continues in the next span
    } else if (tid == 0) {  // values of whole quartets
        q_s[0] = 0;
        q_s[1] = span.nu - 1;
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
    const unsigned blocks = (unsigned)((span.nu + kSetupUnits - 1) / kSetupUnits);
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

cudaError_t class_ends(const long long *ps, const ClassEnds &at, long long *ends, cudaStream_t s) {
    class_ends_kernel<<<1, 256, 0, s>>>(ps, at, ends);
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
