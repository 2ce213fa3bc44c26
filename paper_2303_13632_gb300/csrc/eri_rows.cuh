// eri_rows.cuh -- the four-index recursion of phase_direct spread over the lanes of a warp.
//
// The 2-D integrals I(i, j, k, l) of one (quartet, root, axis) are built by a group of NIP lanes
// (La + 1 rounded up to a power of two), lane i holding the rows j = 0..Lb of index i.  Raising k or
// l needs the row of lane i - 1 (one shuffle per value) and the lane's own rows of lower planes,
// which stay in registers, so a plane costs no shared-memory read and its Lb + 1 values are
// independent.  One thread per (quartet, root, axis) instead walks (La+1)(Lb+1)(Lc+1)(Ld+1)
// dependent steps through shared memory: for [ff|ff] 21 busy threads and 256 steps per quartet.
#pragma once

#include "eri_kernels.cuh"

namespace eri {

__host__ __device__ constexpr int pow2ceil(int n) { return n <= 1 ? 1 : 2 * pow2ceil((n + 1) / 2); }

// C: La..Ld, R, S_CB, S_CD (the slots of C00 on B and C00' on D).  b: the B, C record of the root;
// xi: axis; i: the lane's row; blk: the block of (quartet, root, axis), laid out [i][k][j][l] with
// KP values from one k to the next; live: the lane stores its row.  Every lane of the warp calls it.
// Each value is formed by the operations of phase_direct in their order.
template <class C, int KP>
__device__ __forceinline__ void rows_direct(const typename C::R *b, int xi, int i, bool live,
                                            typename C::R *blk) {
    using R = typename C::R;
    constexpr int NJ = C::Lb + 1, NK = C::Lc + 1, NL = C::Ld + 1, NIP = pow2ceil(C::La + 1);
    const R cA = b[S_C0X + xi], cC = b[S_C1X + xi];
    R cB = (R)0, cD = (R)0;
    if constexpr (C::Lb > 0) cB = b[C::S_CB + xi];
    if constexpr (C::Ld > 0) cD = b[C::S_CD + xi];
    const R b00 = b[S_B00], b10 = b[S_B10], b01 = b[S_B01];
    const R ib00 = (R)i * b00, ib10 = (R)i * b10;
    const auto below = [](R v) -> R {  // the value of lane i - 1
        if constexpr (NIP == 1)
            return v;
        else
            return __shfl_up_sync(0xffffffffu, v, 1, NIP);
    };
    // plane (0, 0): I(i, 0), every lane running the chain up to its own row, then the row
    R r[NJ];
    {
        R lo = (R)0, v = (xi == 2) ? b[S_WZ] : (R)1;
        r[0] = v;
#pragma unroll
        for (int t = 1; t <= C::La; ++t) {
            const R n = t > 1 ? fma((R)(t - 1) * b10, lo, cA * v) : cA * v;
            lo = v;
            v = n;
            if (t == i) r[0] = v;
        }
    }
#pragma unroll
    for (int j = 1; j < NJ; ++j) {
        const R u = below(r[j - 1]);
        R v = cB * r[j - 1];
        if (j > 1) v = fma((R)(j - 1) * b10, r[j - 2], v);
        if (i > 0) v = fma(ib10, u, v);
        r[j] = v;
    }
    R *row = blk + i * NK * KP;
    R p1[NJ], p2[NJ];       // rows (k-1, 0) and (k-2, 0)
    R lo[NL][NJ];           // rows (k-1, l), l > 0
#pragma unroll
    for (int j = 0; j < NJ; ++j) p1[j] = p2[j] = (R)0;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        if (k > 0) {
            R n[NJ];
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const R u = below(p1[j]);
                R v = cC * p1[j];
                if (k > 1) v = fma((R)(k - 1) * b01, p2[j], v);
                if (i > 0) v = fma(ib00, u, v);
                if (j > 0) v = fma((R)j * b00, p1[j - 1], v);
                n[j] = v;
            }
#pragma unroll
            for (int j = 0; j < NJ; ++j) r[j] = n[j];
        }
        R q1[NJ], q2[NJ];  // rows (k, l-1) and (k, l-2)
        R cur[NL][NJ];
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            if (live) row[k * KP + j * NL] = r[j];
            q1[j] = r[j];
            q2[j] = (R)0;
            cur[0][j] = r[j];
        }
#pragma unroll
        for (int l = 1; l < NL; ++l) {
            R n[NJ];
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                const R u = below(q1[j]);
                R v = cD * q1[j];
                if (l > 1) v = fma((R)(l - 1) * b01, q2[j], v);
                if (k > 0) v = fma((R)k * b01, lo[l - 1][j], v);
                if (i > 0) v = fma(ib00, u, v);
                if (j > 0) v = fma((R)j * b00, q1[j - 1], v);
                n[j] = v;
            }
#pragma unroll
            for (int j = 0; j < NJ; ++j) {
                if (live) row[k * KP + j * NL + l] = n[j];
                q2[j] = q1[j];
                q1[j] = n[j];
                cur[l][j] = n[j];
            }
        }
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            p2[j] = p1[j];
            p1[j] = r[j];
#pragma unroll
            for (int l = 0; l < NL; ++l) lo[l][j] = cur[l][j];
        }
    }
}

}  // namespace eri
