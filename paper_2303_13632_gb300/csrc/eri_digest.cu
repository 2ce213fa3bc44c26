// eri_digest.cu -- consumer side of the compressed ERIs: decompression (Sec. II-D, Eq. 11)
// fused with their contraction against a density matrix into the Coulomb and exchange
// matrices,
//   J[mu, nu]  += (mu nu | lam sig) D[lam, sig],     K[mu, lam] += (mu nu | lam sig) D[nu, sig],
// the use Sec. I and Sec. II-D give for computing and storing ERIs compressed (the matrices
// an SCF or AIMD step rebuilds from the stored integrals).
//
// A quartet's block e[a][b][c][d] (codes q times the quartet's eps) contributes through each of
// the eight index permutations of Sec. II-B that give a distinct ordered shell quartet
// (permutations that map the quartet onto itself are counted once).  For the eight
// permutations the twelve contractions needed fall into six "index-pair passes": a pass fixes
// two positions (x, y) of the block and sums over the other two (u, w) against the D block
// D[u, w] and its transpose D[w, u]:
//   pass (a,b): T1 = sum e D[c,d] -> J[a,b] (perm 1), J[b,a] (perm 2);
//               T2 = sum e D[d,c] -> J[a,b] (perm 3), J[b,a] (perm 4)
//   pass (c,d): T3 = sum e D[a,b] -> J[c,d] (5), J[d,c] (6); T4 = sum e D[b,a] -> J[c,d] (7), J[d,c] (8)
//   pass (a,c): sum e D[b,d] -> K[a,c] (1);  sum e D[d,b] -> K[c,a] (5)
//   pass (b,c): sum e D[a,d] -> K[b,c] (2);  sum e D[d,a] -> K[c,b] (7)
//   pass (a,d): sum e D[b,c] -> K[a,d] (3);  sum e D[c,b] -> K[d,a] (6)
//   pass (b,d): sum e D[a,c] -> K[b,d] (4);  sum e D[c,a] -> K[d,b] (8)
// with the permutations 1..8 = (abcd), (bacd), (abdc), (badc), (cdab), (dcab), (cdba), (dcba).
//
// GPU mapping: one CTA per tile of consecutive quartets of one class.  The tile's codes are decoded
// into shared memory as FP32 integers (exact for widths <= 24) and the D blocks between the
// quartet's four shells that the passes read are staged in FP32 (six for a symmetric D, else
// twelve).  A warp owns a few (pass, x, y), neighbours in the list of items, and its lanes the tile's
// quartets: the sums of a warp have the same length, what depends on the pass alone is formed once,
// and the strides between quartets are odd, so that lanes read distinct banks.  Values with the same
// destination (neighbours in a list of unique quartets share their bra, many also the shell c) are
// summed in FP64 over a lane's quartets and, where all its lanes end on one destination, over the
// lanes before they are added to J and K (device atomics, so the summation order of the FP64
// accumulation varies between runs).  3.45 million unique quartets of s to f shells (12 atoms, 16
// bits): 10.5 -> 6.0 ms with a symmetric D.  Bound by shared-memory reads (two per product) and issue.
#include <algorithm>
#include <type_traits>
#include <vector>

#include "eri_internal.h"

namespace eri {

namespace {

constexpr int kDigestThreads = 256;
// dynamic shared memory of a tile: 47 KB, so that with the kernel's static shared memory (the
// class parameters) a CTA stays within the 48 KB available without an opt-in
constexpr int kDigestSmem = 47 * 1024;

// pass p fixes positions (PX, PY) and sums over (PU, PW)
__constant__ int c_px[6] = {0, 2, 0, 1, 0, 1};
__constant__ int c_py[6] = {1, 3, 2, 2, 3, 3};
__constant__ int c_pu[6] = {2, 0, 1, 0, 1, 0};
__constant__ int c_pw[6] = {3, 1, 3, 3, 2, 2};

struct DigestArgs {
    const int4 *quartets;  // class-sorted shell ids of the class
    long long nq;
    const uint32_t *packed;  // class segment of the packed stream
    const float *scales;     // eps of the class's quartets
    const int *bfoff;        // first basis function of every shell
    const float *D;          // density matrix, FP32, row major
    long long nbf;
    double *J, *K;
    int bits;
    int unique8;
    int n[4];      // Cartesian components of the four positions
    int st[4];     // strides of the four positions in the quartet's block
    int neri;
    int T;         // quartets per tile
    int lanes;     // lanes of a warp over the tile's quartets (power of two); 32 / lanes items per warp
    int se, sd;    // values per quartet in shared memory: codes, D (odd)
    unsigned m_neri;  // ceil(2^32 / n_ERIQ): quartet of a code of the tile (0: one value per quartet)
    int nblk;      // staged D blocks
    int bx[12], by[12];  // block b holds D[x][y] of positions (bx, by)
    int boff[16];  // offset of D block (x, y) (index x*4 + y) in a quartet's D area
    int rstart[13];  // first row of each staged block; [nblk] = rows
    int NI;        // items per quartet
    int ioff[7];   // first item of each pass
};

// Which of the eight permutations give a distinct ordered shell quartet (bit p-1 for
// permutation p): a permutation equal, as a tuple of shell ids, to an earlier one is dropped.
__device__ __forceinline__ int perm_mask(int4 s, bool unique8) {
    if (!unique8) return 1;
    const int t[8][4] = {{s.x, s.y, s.z, s.w}, {s.y, s.x, s.z, s.w}, {s.x, s.y, s.w, s.z},
                         {s.y, s.x, s.w, s.z}, {s.z, s.w, s.x, s.y}, {s.w, s.z, s.x, s.y},
                         {s.z, s.w, s.y, s.x}, {s.w, s.z, s.y, s.x}};
    int mask = 0;
#pragma unroll
    for (int p = 0; p < 8; ++p) {
        bool fresh = true;
#pragma unroll
        for (int r = 0; r < p; ++r)
            fresh &= !(t[p][0] == t[r][0] && t[p][1] == t[r][1] && t[p][2] == t[r][2] &&
                       t[p][3] == t[r][3]);
        mask |= fresh ? (1 << p) : 0;
    }
    return mask;
}

// Coefficients (0 or 1) of the two sums of pass p in its two destinations, four bits per pass:
// dest 1 = M[x, y] gets bit 0 S + bit 1 S', dest 2 = M[y, x] gets bit 2 S + bit 3 S'.
__device__ __forceinline__ unsigned int pass_bits(int m) {
    auto b = [m](int perm) { return (unsigned int)(m >> (perm - 1)) & 1u; };
    return (b(1) | b(3) << 1 | b(2) << 2 | b(4) << 3) | (b(5) | b(7) << 1 | b(6) << 2 | b(8) << 3) << 4 |
           (b(1) | b(5) << 3) << 8 | (b(2) | b(7) << 3) << 12 | (b(3) | b(6) << 3) << 16 | (b(4) | b(8) << 3) << 20;
}

// SYM: the caller's D is symmetric.  Then S = S' in every pass (D[u][w] = D[w][u]) and the two
// destinations M[x][y], M[y][x] of an item receive equal totals over the whole sum, so each item
// forms one sum and adds all of its coefficient to M[x][y] alone; the finished matrices are
// symmetrised afterwards, M = (M + M^T) / 2 (symmetrise_kernel), which restores every entry.
//
// One launch covers every class: CTA b takes tile b - tile_start[c] of the class c with
// tile_start[c] <= b < tile_start[c + 1] (the classes' parameters in `args`, copied to shared
// memory by the CTA), so small classes do not leave the GPU idle between launches.
template <bool SYM>
__global__ void __launch_bounds__(kDigestThreads)
digest_kernel(const DigestArgs *__restrict__ args, const long long *__restrict__ tile_start, int n_classes) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ DigestArgs A;
    __shared__ long long tile_s;
    if (threadIdx.x == 0) {
        int lo = 0, hi = n_classes - 1;  // last class with tile_start <= blockIdx.x
        while (lo < hi) {
            const int mid = (lo + hi + 1) / 2;
            if (tile_start[mid] <= (long long)blockIdx.x)
                lo = mid;
            else
                hi = mid - 1;
        }
        tile_s = ((long long)blockIdx.x - tile_start[lo]) | ((long long)lo << 40);
    }
    __syncthreads();
    {
        const int c = (int)(tile_s >> 40);
        const int *src = reinterpret_cast<const int *>(args + c);
        int *dst = reinterpret_cast<int *>(&A);
        for (int i = threadIdx.x; i < (int)(sizeof(DigestArgs) / 4); i += kDigestThreads) dst[i] = src[i];
    }
    __syncthreads();
    int *meta = reinterpret_cast<int *>(smem);               // T x 8: bf offsets, mask, eps
    float *e_s = reinterpret_cast<float *>(meta + A.T * 8);  // T x se codes
    float *d_s = e_s + (size_t)A.T * A.se;                   // T x sd D values
    const long long q0 = (tile_s & ((1LL << 40) - 1)) * A.T;
    const int tn = (int)((A.nq - q0) < A.T ? (A.nq - q0) : A.T);
    const int tid = threadIdx.x;

    for (int t = tid; t < tn; t += kDigestThreads) {
        const int4 s = A.quartets[q0 + t];
        int *m = meta + t * 8;
        m[0] = A.bfoff[s.x];
        m[1] = A.bfoff[s.y];
        m[2] = A.bfoff[s.z];
        m[3] = A.bfoff[s.w];
        m[4] = (int)pass_bits(perm_mask(s, A.unique8 != 0));
        m[5] = __float_as_int(A.scales[q0 + t]);
    }
    // codes of the tile: fields q0*neri .. (q0+tn)*neri of the class's stream (Eq. 11 without
    // the scale, which is applied once per sum), at bits relative to the tile's first word
    const int nv = tn * A.neri;
    const unsigned long long bit0 = (unsigned long long)q0 * (unsigned)A.neri * (unsigned)A.bits;
    const uint32_t *words = A.packed + (bit0 >> 5);
    const int head = (int)(bit0 & 31), up = 32 - A.bits;
    // place of the tile's value v: quartets se apart
    const int pad = A.se - A.neri;
    auto place = [&](int v) { return v + pad * (A.m_neri ? (int)__umulhi((unsigned)v, A.m_neri) : v); };
    if (A.bits == 16) {
        const int16_t *codes = reinterpret_cast<const int16_t *>(words) + (head >> 4);
        for (int v = tid; v < nv; v += kDigestThreads) e_s[place(v)] = (float)__ldg(codes + v);
    } else {
        for (int v = tid; v < nv; v += kDigestThreads) {
            const int bit = head + v * A.bits, w = bit >> 5, off = bit & 31;
            uint32_t raw = __ldg(words + w) >> off;
            if (off + A.bits > 32) raw |= __ldg(words + w + 1) << (32 - off);
            e_s[place(v)] = (float)((int)(raw << up) >> up);  // sign extension
        }
    }
    __syncthreads();
    // lane = (item of the warp, quartet)
    const int lane = tid & 31, tl = lane & (A.lanes - 1), il = lane / A.lanes, items = 32 / A.lanes;
    // the D blocks between the quartet's shells, D[o_x + i][o_y + j]: a block row per item, whose at
    // most 10 loads are independent
    const int rows = A.rstart[A.nblk];
    for (int r = (tid >> 5) * items + il; r < rows; r += kDigestThreads / 32 * items) {
        int b = 0;
        for (int k = 1; k < A.nblk; ++k) b += r >= A.rstart[k];
        const int x = A.bx[b], y = A.by[b];
        const int i = r - A.rstart[b], ny = A.n[y];
        float *dst = d_s + A.boff[x * 4 + y] + i * ny;
        for (int t = tl; t < tn; t += A.lanes) {
            const int *m = meta + t * 8;
            const float *src = A.D + (long long)(m[x] + i) * A.nbf + m[y];
#pragma unroll 10
            for (int j = 0; j < ny; ++j) dst[t * A.sd + j] = __ldg(src + j);
        }
    }
    __syncthreads();
    for (int r0 = (tid >> 5) * items; r0 < A.NI; r0 += kDigestThreads / 32 * items) {
        const int r = r0 + il;
        const bool on = r < A.NI;
        int p = 0;
#pragma unroll
        for (int k = 1; k < 6; ++k) p += r >= A.ioff[k];
        const int x = c_px[p], y = c_py[p], u = c_pu[p], w = c_pw[p];
        const int loc = r - A.ioff[p];
        const int ix = loc / A.n[y], iy = loc - ix * A.n[y];
        const int nu = A.n[u], nw = A.n[w], su = A.st[u], sw = A.st[w];
        const float *e0 = e_s + ix * A.st[x] + iy * A.st[y];
        const float *d1 = d_s + A.boff[u * 4 + w];  // D[u][w], row length nw
        const float *d2 = d_s + A.boff[w * 4 + u];  // D[w][u], row length nu
        double *M = p < 2 ? A.J : A.K;
        int row = -1, col = -1;  // the pending sums' destination
        double acc1 = 0.0, acc2 = 0.0;
        unsigned int pend = 0u;
        auto flush = [&]() {
            if (pend & 1u) atomicAdd(M + (long long)row * A.nbf + col, acc1);
            if (pend & 2u) atomicAdd(M + (long long)col * A.nbf + row, acc2);
            acc1 = acc2 = 0.0;
            pend = 0u;
        };
        for (int t = tl; on && t < tn; t += A.lanes) {
            const int *m = meta + t * 8;
            const unsigned int c = ((unsigned int)m[4] >> (4 * p)) & 15u;
            if (c == 0u) continue;
            const float *ep = e0 + t * A.se, *dp = d1 + t * A.sd, *dq = d2 + t * A.sd;
            const float eps = __int_as_float(m[5]);
            const int rw = m[x] + ix, cl = m[y] + iy;
            if (rw != row || cl != col) {
                flush();
                row = rw;
                col = cl;
            }
            float S = 0.0f, S2 = 0.0f;
            auto rows_of = [&](auto n) {  // rows of a compile-time length, in order
                constexpr int N = decltype(n)::value;
                for (int iu = 0; iu < nu; ++iu, ep += su, dp += N, ++dq) {
#pragma unroll
                    for (int iw = 0; iw < N; ++iw) {
                        const float e = ep[iw * sw];
                        S = fmaf(e, dp[iw], S);
                        if constexpr (!SYM) S2 = fmaf(e, dq[iw * nu], S2);
                    }
                }
            };
            switch (nw) {
                case 1: rows_of(std::integral_constant<int, 1>{}); break;
                case 3: rows_of(std::integral_constant<int, 3>{}); break;
                case 6: rows_of(std::integral_constant<int, 6>{}); break;
                default: rows_of(std::integral_constant<int, 10>{}); break;
            }
            if constexpr (SYM) {
                const float k = (float)__popc(c);
                acc1 += f32_to_f64(S * (k * eps));
                pend = 1u;
            } else {
                const float v1 = ((c & 1u) ? S : 0.0f) + ((c & 2u) ? S2 : 0.0f);
                const float v2 = ((c & 4u) ? S : 0.0f) + ((c & 8u) ? S2 : 0.0f);
                if (c & 3u) acc1 += f32_to_f64(v1 * eps);
                if (c & 12u) acc2 += f32_to_f64(v2 * eps);
                pend |= ((c & 3u) ? 1u : 0u) | ((c & 12u) ? 2u : 0u);
            }
        }
        // one destination over the item's lanes: one sum (lanes with nothing pending add zeros)
        if (A.lanes > 1) {
            const int src = lane & ~(A.lanes - 1);
            const int row0 = __shfl_sync(0xffffffffu, row, src), col0 = __shfl_sync(0xffffffffu, col, src);
            const bool same = pend == 0u || (row == row0 && col == col0);
            if (__all_sync(0xffffffffu, same)) {
                for (int off = A.lanes / 2; off > 0; off >>= 1) {
                    acc1 += __shfl_down_sync(0xffffffffu, acc1, off, A.lanes);
                    if constexpr (!SYM) acc2 += __shfl_down_sync(0xffffffffu, acc2, off, A.lanes);
                    pend |= __shfl_down_sync(0xffffffffu, pend, off, A.lanes);
                }
                if (tl != 0) pend = 0u;
            }
        }
        flush();
    }
}

// M = (M + M^T) / 2 for an n x n row-major matrix, one thread per pair i < j.
__global__ void symmetrise_kernel(double *__restrict__ M, long long n) {
    const long long pairs = n * (n - 1) / 2;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < pairs;
         t += (long long)gridDim.x * blockDim.x) {
        long long i = (long long)((sqrt(8.0 * (double)t + 1.0) + 1.0) * 0.5);  // row, i >= 1
        while (i * (i - 1) / 2 > t) --i;
        while ((i + 1) * i / 2 <= t) ++i;
        const long long j = t - i * (i - 1) / 2;  // 0 <= j < i
        const double v = 0.5 * (M[i * n + j] + M[j * n + i]);
        M[i * n + j] = v;
        M[j * n + i] = v;
    }
}

__global__ void density_to_f32_kernel(const double *__restrict__ D, long long n, float *__restrict__ out) {
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        out[i] = f64_to_f32(D[i]);
}

int ncart_d(int L) { return (L + 1) * (L + 2) / 2; }

}  // namespace

cudaError_t digest_density_f32(const double *D, long long n, float *out, cudaStream_t stream) {
    if (n <= 0) return cudaSuccess;
    long long blocks = (n + 255) / 256;
    if (blocks > 4096) blocks = 4096;
    density_to_f32_kernel<<<(unsigned)blocks, 256, 0, stream>>>(D, n, out);
    return cudaGetLastError();
}

cudaError_t digest_symmetrise(double *M, long long n, cudaStream_t stream) {
    if (n < 2) return cudaSuccess;
    const long long pairs = n * (n - 1) / 2;
    long long blocks = (pairs + 255) / 256;
    if (blocks > 8192) blocks = 8192;
    symmetrise_kernel<<<(unsigned)blocks, 256, 0, stream>>>(M, n);
    return cudaGetLastError();
}

size_t digest_table_bytes() { return 256 * sizeof(DigestArgs) + 257 * sizeof(long long); }

cudaError_t digest_all(const DigestClass *classes, int n_classes, int bits, bool unique8, bool symmetric,
                       const int *bfoff, const float *D32, long long nbf, double *J, double *K,
                       void *d_table, cudaStream_t stream) {
    if (n_classes <= 0) return cudaSuccess;
    if (n_classes > 256) return cudaErrorInvalidValue;
    std::vector<DigestArgs> args(n_classes);
    std::vector<long long> start(n_classes + 1);
    size_t smem_max = 0;
    long long tiles = 0;
    for (int k = 0; k < n_classes; ++k) {
        const DigestClass &c = classes[k];
        DigestArgs &A = args[k];
        A = DigestArgs{};
        A.quartets = c.quartets;
        A.nq = c.nq;
        A.packed = c.packed;
        A.scales = c.scales;
        A.bfoff = bfoff;
        A.D = D32;
        A.nbf = nbf;
        A.J = J;
        A.K = K;
        A.bits = bits;
        A.unique8 = unique8 ? 1 : 0;
        const int L[4] = {(c.cls >> 6) & 3, (c.cls >> 4) & 3, (c.cls >> 2) & 3, c.cls & 3};
        for (int x = 0; x < 4; ++x) A.n[x] = ncart_d(L[x]);
        A.st[3] = 1;
        for (int x = 2; x >= 0; --x) A.st[x] = A.st[x + 1] * A.n[x + 1];
        A.neri = A.st[0] * A.n[0];
        // the blocks the passes read: D[u][w], and D[w][u] unless D is symmetric
        const int pu[6] = {2, 0, 1, 0, 1, 0}, pw[6] = {3, 1, 3, 3, 2, 2};
        int o = 0;
        A.nblk = 0;
        A.rstart[0] = 0;
        for (int p = 0; p < 6; ++p)
            for (int h = 0; h < (symmetric ? 1 : 2); ++h) {
                const int x = h ? pw[p] : pu[p], y = h ? pu[p] : pw[p];
                A.bx[A.nblk] = x;
                A.by[A.nblk] = y;
                A.boff[x * 4 + y] = o;
                o += A.n[x] * A.n[y];
                A.rstart[A.nblk + 1] = A.rstart[A.nblk] + A.n[x];
                ++A.nblk;
            }
        A.se = A.neri | 1;
        A.sd = o | 1;
        const int px[6] = {0, 2, 0, 1, 0, 1}, py[6] = {1, 3, 2, 2, 3, 3};
        A.ioff[0] = 0;
        for (int p = 0; p < 6; ++p) A.ioff[p + 1] = A.ioff[p] + A.n[px[p]] * A.n[py[p]];
        A.NI = A.ioff[6];
        const int perq = 4 * (8 + A.se + A.sd);
        int T = kDigestSmem / perq;
        T = T < 1 ? 1 : (T > 128 ? 128 : T);
        A.lanes = 1;
        while (A.lanes < 32 && 2 * A.lanes <= T) A.lanes *= 2;
        T = T / A.lanes * A.lanes;  // all lanes busy on every quartet of a full tile
        A.T = T;
        A.m_neri = A.neri == 1 ? 0u : (unsigned)(((1ull << 32) + A.neri - 1) / A.neri);
        if ((size_t)T * perq > (size_t)kDigestSmem) return cudaErrorInvalidValue;
        smem_max = std::max(smem_max, (size_t)T * perq);
        start[k] = tiles;
        tiles += (c.nq + T - 1) / T;
    }
    start[n_classes] = tiles;
    if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
    DigestArgs *d_args = static_cast<DigestArgs *>(d_table);
    long long *d_start = reinterpret_cast<long long *>(static_cast<char *>(d_table) + 256 * sizeof(DigestArgs));
    cudaError_t e = cudaMemcpyAsync(d_args, args.data(), n_classes * sizeof(DigestArgs), cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(d_start, start.data(), (n_classes + 1) * sizeof(long long), cudaMemcpyHostToDevice, stream);
    if (e != cudaSuccess) return e;
    if (symmetric)
        digest_kernel<true><<<(unsigned)tiles, kDigestThreads, smem_max, stream>>>(d_args, d_start, n_classes);
    else
        digest_kernel<false><<<(unsigned)tiles, kDigestThreads, smem_max, stream>>>(d_args, d_start, n_classes);
    return cudaGetLastError();
}

}  // namespace eri
