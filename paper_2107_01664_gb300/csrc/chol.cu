// Pre-factorised cotan-Laplacian solves (§5.2): supernodal sparse Cholesky of
// C with one pinned vertex per connected component, on the device.
//
// The ordering, supernodal tree and index maps come from chol_symbolic.h
// (host, once per topology). Per set of positions the values of C change and
// the factor is recomputed:
//
//   factor (two launches per tree level): k_chol_panel, one block per supernode
//   J, assembles the panel (t x nJ, shared memory) from the entries of C in J's
//   columns and the children's update matrices, factors its diagonal block
//   (right-looking, in blocks of eight columns) with L11^-1 formed along the way, and
//   stores L11^-1 and L21; k_chol_update, one block per 64 x 64 tile, forms
//   U_J = (children's share of struct x struct) - L21 L21^T (global memory).
//
//   solve (forward levels leaves -> root, backward levels root -> leaves):
//   with L11^-1 stored, each supernode's step is two small dense mat-vecs on
//   K columns, so the substitution's only sequential chain is the tree height.
//
// The factor is FP32 (64x the FP64 issue rate of this GPU); the solve is
// wrapped in FP64 iterative refinement x += L^-T L^-1 (b - C x), with the
// residual in FP64, until every column meets |r| <= tol |b| (the same test
// as the CG path). Refinement that stops reducing the residual hands the
// solve to the CG path.
#include <algorithm>
#include <cmath>
#include <memory>
#include <string>
#include <vector>

#include "chol_symbolic.h"
#include "tp_internal.cuh"

namespace tp {

constexpr int CH_KMAX = 9;
constexpr int CH_LEAF = 64;                    // vertices per leaf supernode
constexpr int CHF_TILE = 64;                   // tile of an update matrix (k_chol_update)
constexpr int CHF_KC = 32;                     // columns of L21 staged at a time
constexpr int CHS_T = 256;                     // solve block
constexpr int CHR_T = 256;                     // residual block
constexpr size_t CHS_SMALL = 70 * 1024;        // solve step of which an SM holds three blocks
constexpr size_t CH_SMEM_MAX = 220 * 1024;     // dynamic shared memory of a factor panel or a solve step

struct CholNode {   // 64 bytes
    int p0, nJ, mJ, t;
    long long loff, uoff;
    int voff, child0, child1, s0;
    int asm0, asm1, ldu, flags;   // leading dimension of U
};
static_assert(sizeof(CholNode) == 64, "CholNode layout");
// the node's one child has exactly the rows of its front: its U is the trailing
// part of the child's U, updated in place (the links of a separator's chain)
constexpr int CHN_INPLACE = 1;
// the children's update vectors are read from global memory in the solve
constexpr int CHN_DIRECT = 2;

struct CholCtl {
    int done;       // 1: every column converged (or the refinement gave up)
    int stalled;    // 1: the residual stopped decreasing
    int iters;      // refinement sweeps done
    int err;        // 1: a cross-block wait of a sweep gave up
    unsigned ticket[3], bcount, arrive;   // sweep scheduling (zero between sweeps)
    int bad_pivot;  // 1: a non-positive pivot appeared in the factorisation
    double bb[CH_KMAX], rr[CH_KMAX];
    unsigned epoch;  // sweeps finished; never cleared (the node flags compare against it)
};

struct CholState {
    CholSymbolic S;
    bool ok = false;
    std::string why;
    int H = 0;                            // number of levels
    std::vector<int> lvl_max_t;           // rows of the level's largest front
    std::vector<size_t> lvl_factor_smem;  // bytes
    std::vector<int> lvl_tile;            // first entry of each level in `tiles`
    std::vector<double> lvl_factor_flops;
    int64_t usize = 0;                    // floats of the update matrices (those in place share their child's)
    double solve_bytes = 0.0;             // factor bytes read by one forward + backward sweep
    Buf nodes, level_nodes, child_idx, rel, struct_pos, asm_dst, asm_src, perm, comp_ptr, comp_verts, comp_of;
    Buf parent, fdone, bdone, trace, tiles;
    // dynamic shared memory of the sweep kernel by column count: the largest of all
    // nodes, and of the leading tree levels that leave room for three blocks per SM
    // (small_n nodes)
    size_t solve_smem[CH_KMAX + 1] = {}, small_smem[CH_KMAX + 1] = {};
    int small_n[CH_KMAX + 1] = {};
    bool wide = false;         // a front has more than 256 rows, or CHN_DIRECT
    Buf L, U, uvec, ybuf, xbuf, ctl, part, x, r, bp;
    bool factored = false;
    int ncomp = 1;
    // refinement sweeps captured as CUDA graphs, one per column count, keyed
    // by the buffers and scalars baked into their launches
    // deferred solves (inside flexible GMRES): the pivot check of the current
    // factor is read once, and the sweeps' wait errors and poor columns accumulate in
    // dflags [2] for the caller to read (chol_deferred_flags)
    bool pivot_known = false, pivot_ok = false;
    Buf dflags;
    struct SweepGraph {
        cudaGraphExec_t exec = nullptr;
        const void* key[4] = {};
        double tol2 = 0.0;
        int cap = 0, kernels = 0;
    } graph[CH_KMAX + 1];
    cudaStream_t capture = nullptr;
};

// ---------------------------------------------------------------------------
// factorisation
// ---------------------------------------------------------------------------

// Panel of one supernode per block: assembly, Cholesky of the diagonal block
// and its inverse, in blocks of CHF_NB columns. Latency-bound: the blocks of
// columns come one after the other, and the levels above the leaves hold fewer
// supernodes than the GPU has SMs. Hence few barriers (three per block of
// columns: every thread factors the CHF_NB x CHF_NB diagonal block for itself
// and substitutes into its own rows), and a trailing update of rank CHF_NB with
// the row factors in registers, which takes the remaining panel columns and the
// columns of L11^-1 alike (the same row operations on the identity). 25,000
// vertices, 9 levels: 31 us a level on average, 84 us one column at a time.
constexpr int CHF_NB = 8;

// shared floats of a panel of t rows and n columns: P (t x n), X (n x n, leading
// dimension a multiple of 8), the block's rows below it (n x NB), the rows of the
// largest child
__host__ __device__ inline int chf_ldx(int n) { return (n + CHF_NB - 1) / CHF_NB * CHF_NB; }
inline size_t chf_smem(size_t t, size_t n, size_t child) {
    return sizeof(float) * (((t * n + 3) & ~size_t(3)) + (size_t)chf_ldx((int)n) * n + chf_ldx((int)n) * CHF_NB + child);
}

__global__ void __launch_bounds__(512)
k_chol_panel(const CholNode* __restrict__ nodes, const int* __restrict__ lvl, const int* __restrict__ child_idx,
             const int* __restrict__ rel, const int* __restrict__ asm_dst, const int* __restrict__ asm_src,
             const double* __restrict__ val, float* __restrict__ L, const float* __restrict__ U,
             CholCtl* __restrict__ ctl) {
    constexpr int NB = CHF_NB;
    extern __shared__ float4 smem4_f[];
    float* smem = reinterpret_cast<float*>(smem4_f);
    const CholNode nd = nodes[lvl[blockIdx.x]];
    const int n = nd.nJ, m = nd.mJ, t = nd.t;
    const int ldx = chf_ldx(n);
    float* P = smem;                                   // panel t x n, column-major
    float* X = smem + ((t * n + 3) & ~3);              // L11^-1, n columns, leading dimension ldx
    float* B = X + (size_t)ldx * n;                    // rows of the block's L: B[row][NB]
    const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, warp = tid >> 5, NW = T >> 5;

    if (nd.flags & CHN_INPLACE) {
        // the panel is the first n columns of the child's update matrix
        const float* Uc = U + nodes[child_idx[nd.child0]].uoff;
        for (int y = warp; y < n; y += NW)
#pragma unroll 8
            for (int x = lane; x < t; x += 32) P[x + y * t] = x >= y ? Uc[x + (size_t)y * nd.ldu] : 0.f;
    } else {
        for (int i = tid; i < t * n; i += T) P[i] = 0.f;
    }
    for (int i = tid; i < ldx * n; i += T) X[i] = i % ldx == i / ldx ? 1.f : 0.f;
    for (int i = tid; i < ldx * NB; i += T) B[i] = 0.f;
    __syncthreads();
    // entries of C in J's columns (each panel position at most once)
    for (int e = nd.asm0 + tid; e < nd.asm1; e += T) P[asm_dst[e]] += (float)val[asm_src[e]];
    __syncthreads();
    if (!(nd.flags & CHN_INPLACE)) {
        // extend-add of the children's columns that fall into the panel (the
        // first ones: a child's rows are sorted), one child at a time, its rows'
        // places in the front staged first
        int* rl = reinterpret_cast<int*>(B + ldx * NB);
        for (int ci = nd.child0; ci < nd.child1; ++ci) {
            const CholNode cn = nodes[child_idx[ci]];
            const int mc = cn.mJ;
            const float* Uc = U + cn.uoff;
            for (int x = tid; x < mc; x += T) rl[x] = rel[cn.s0 + x];
            __syncthreads();
            int lo = 0, hi = mc;     // columns with a place before n
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (rl[mid] < n) lo = mid + 1;
                else hi = mid;
            }
            const int cnt = lo * mc;
            for (int e0 = tid; e0 < cnt; e0 += 4 * T) {
                float v[4];
                int at[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int e = e0 + q * T, y = e / mc, x = e - y * mc;
                    at[q] = -1;
                    if (e < cnt && x >= y) {
                        v[q] = Uc[x + (size_t)y * cn.ldu];
                        at[q] = rl[x] + rl[y] * t;
                    }
                }
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    if (at[q] >= 0) P[at[q]] += v[q];
            }
            __syncthreads();
        }
    }
    for (int kb = 0; kb < n; kb += NB) {
        const int nb = min(NB, n - kb);
        // the diagonal block (columns past n: identity), factored by every thread;
        // D[k][l] = L entries below the diagonal, rd = reciprocal diagonal
        float D[NB][NB], rd[NB];
#pragma unroll
        for (int l = 0; l < NB; ++l)
#pragma unroll
            for (int k = l; k < NB; ++k) D[k][l] = k < nb ? P[kb + k + (kb + l) * t] : (k == l ? 1.f : 0.f);
        bool bad = false;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
            float d = D[k][k];
            if (!(d > 0.f)) {
                bad = true;
                d = 1.f;
            }
            // correctly rounded steps: rsqrtf with a Newton step made the refinement
            // take a sweep more (163,842 vertices)
            rd[k] = 1.f / sqrtf(d);
#pragma unroll
            for (int i = k + 1; i < NB; ++i) D[i][k] *= rd[k];
#pragma unroll
            for (int j = k + 1; j < NB; ++j)
#pragma unroll
                for (int i = j; i < NB; ++i) D[i][j] = fmaf(-D[i][k], D[j][k], D[i][j]);
        }
        if (bad && tid == 0) ctl->bad_pivot = 1;
        // rows below the block: substitution, row by row; rows of the diagonal
        // block's own columns go to B too
        for (int i = kb + nb + tid; i < t; i += T) {
            float r[NB];
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                float x = k < nb ? P[i + (kb + k) * t] : 0.f;
#pragma unroll
                for (int l = 0; l < k; ++l) x = fmaf(-r[l], D[k][l], x);
                r[k] = x * rd[k];
            }
#pragma unroll
            for (int k = 0; k < NB; ++k)
                if (k < nb) P[i + (kb + k) * t] = r[k];
            if (i < n) {
                float4* br = reinterpret_cast<float4*>(B + i * NB);
                br[0] = make_float4(r[0], r[1], r[2], r[3]);
                br[1] = make_float4(r[4], r[5], r[6], r[7]);
            }
        }
        // the block's rows of the inverse: X_b <- L_bb^-1 X_b, a thread per column
        for (int c = T - 1 - tid; c < kb + nb; c += T) {
            float4* xc = reinterpret_cast<float4*>(X + kb + (size_t)c * ldx);
            const float4 x0 = xc[0], x1 = xc[1];
            float r[NB] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
#pragma unroll
            for (int k = 0; k < NB; ++k) {
                float x = r[k];
#pragma unroll
                for (int l = 0; l < k; ++l) x = fmaf(-r[l], D[k][l], x);
                r[k] = x * rd[k];
            }
            xc[0] = make_float4(r[0], r[1], r[2], r[3]);
            xc[1] = make_float4(r[4], r[5], r[6], r[7]);
        }
        __syncthreads();
        const int k1 = kb + nb;
        if (k1 >= n) break;
        // trailing update: work items are (32 rows, eight columns); panel columns
        // k1 .. n with all rows from k1, inverse columns 0 .. k1 with rows k1 .. n
        const int pch = (t - k1 + 31) / 32, pgr = (n - k1 + 7) / 8;
        const int xch = (n - k1 + 31) / 32, xgr = (k1 + 7) / 8;
        const int items = pch * pgr + xch * xgr;
        for (int w = warp; w < items; w += NW) {
            const bool inv = w >= pch * pgr;
            const int q = inv ? w - pch * pgr : w, ch = inv ? xch : pch;
            const int i = k1 + (q % ch) * 32 + lane, j0 = (inv ? 0 : k1) + (q / ch) * 8;
            const int iend = inv ? n : t, jend = inv ? k1 : n;
            if (i >= iend) continue;
            float r[NB];
#pragma unroll
            for (int k = 0; k < NB; ++k) r[k] = k < nb ? P[i + (kb + k) * t] : 0.f;
            float* out = inv ? X + i : P + i;
            const int ldo = inv ? ldx : t;
#pragma unroll
            for (int jj = 0; jj < 8; ++jj) {
                const int j = j0 + jj;
                if (j < jend) {
                    const float4* bj = reinterpret_cast<const float4*>(inv ? X + kb + (size_t)j * ldx : B + j * NB);
                    const float4 b0 = bj[0], b1 = bj[1];
                    float x = out[(size_t)j * ldo];
                    x = fmaf(-r[0], b0.x, x);
                    x = fmaf(-r[1], b0.y, x);
                    x = fmaf(-r[2], b0.z, x);
                    x = fmaf(-r[3], b0.w, x);
                    x = fmaf(-r[4], b1.x, x);
                    x = fmaf(-r[5], b1.y, x);
                    x = fmaf(-r[6], b1.z, x);
                    x = fmaf(-r[7], b1.w, x);
                    out[(size_t)j * ldo] = x;
                }
            }
        }
        __syncthreads();
    }
    const int ldn = n | 1, ldm = m == 0 ? 0 : (m | 1);
    float* Lj = L + nd.loff;   // n x n, leading dimension ldn
    float* L21 = Lj + (size_t)n * ldn;   // m x n, leading dimension ldm
    for (int c = warp; c < n; c += NW) {
        for (int r = lane; r < n; r += 32) Lj[r + c * ldn] = r >= c ? X[r + c * ldx] : 0.f;
        for (int x = lane; x < m; x += 32) L21[x + c * ldm] = P[n + x + c * t];
    }
}

// A 64 x 64 tile (lower part) of one supernode's update matrix: the children's
// entries that fall into it (contiguous row and column ranges of each child,
// whose rows are sorted; in place: the tile itself), minus L21 L21^T. tiles:
// (node, first row, first column). A level's tiles run side by side (12 us a level
// on 25,000 vertices, mostly its chain of dependent loads); one block per supernode
// did this work and the panel in 127 us.
__global__ void __launch_bounds__(256)
k_chol_update(const CholNode* __restrict__ nodes, const int4* __restrict__ tiles, const int* __restrict__ child_idx,
              const int* __restrict__ rel, const float* __restrict__ L, float* __restrict__ U) {
    constexpr int TB = CHF_TILE, KC = CHF_KC;
    __shared__ float S[TB][TB + 1];          // [column][row]
    __shared__ __align__(16) float As[KC][TB], Bs[KC][TB];
    __shared__ int s_rng[4];
    const int4 tl = tiles[blockIdx.x];
    const CholNode nd = nodes[tl.x];
    const int n = nd.nJ, m = nd.mJ, r0 = tl.y, c0 = tl.z, tid = threadIdx.x;
    const int rn = min(TB, m - r0), cn = min(TB, m - c0);
    const int ldm = m | 1;
    const float* L21 = L + nd.loff + (size_t)n * (n | 1);
    float* UJ = U + nd.uoff;
    const bool inplace = nd.flags & CHN_INPLACE;
    if (!inplace) {
        for (int i = tid; i < TB * (TB + 1); i += 256) (&S[0][0])[i] = 0.f;
        __syncthreads();
        for (int ci = nd.child0; ci < nd.child1; ++ci) {
            const CholNode ch = nodes[child_idx[ci]];
            const int* rl = rel + ch.s0;
            if (tid < 4) {   // first child row at or after front rows n + r0, n + r0 + rn, n + c0, n + c0 + cn
                const int want = n + (tid == 0 ? r0 : tid == 1 ? r0 + rn : tid == 2 ? c0 : c0 + cn);
                int lo = 0, hi = ch.mJ;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (rl[mid] < want) lo = mid + 1;
                    else hi = mid;
                }
                s_rng[tid] = lo;
            }
            __syncthreads();
            const int x0 = s_rng[0], x1 = s_rng[1], y0 = s_rng[2], y1 = s_rng[3];
            const float* Uc = U + ch.uoff;
            for (int y = y0 + (tid >> 5); y < y1; y += 8) {
                const int c = rl[y] - n - c0;
                for (int x = max(x0, y) + (tid & 31); x < x1; x += 32) S[c][rl[x] - n - r0] += Uc[x + (size_t)y * ch.ldu];
            }
            __syncthreads();
        }
    }
    const int tx = tid & 15, ty = tid >> 4;   // rows tx + 16 i, columns 4 ty + j
    float acc[4][4] = {};
    for (int k0 = 0; k0 < n; k0 += KC) {
        const int kn = min(KC, n - k0);
        __syncthreads();
#pragma unroll
        for (int u = 0; u < KC * TB / 256; ++u) {
            const int i = tid + u * 256, k = i / TB, r = i % TB;
            As[k][r] = k < kn && r < rn ? L21[r0 + r + (size_t)(k0 + k) * ldm] : 0.f;
            Bs[k][r] = k < kn && r < cn ? L21[c0 + r + (size_t)(k0 + k) * ldm] : 0.f;
        }
        __syncthreads();
        const int ke = (kn + 7) & ~7;
#pragma unroll 8
        for (int k = 0; k < ke; ++k) {
            const float4 b = *reinterpret_cast<const float4*>(&Bs[k][4 * ty]);
            const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float av = As[k][tx + 16 * i];
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av, bv[j], acc[i][j]);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int r = tx + 16 * i, c = 4 * ty + j;
            if (r >= rn || c >= cn || r0 + r < c0 + c) continue;
            float* u = UJ + (r0 + r) + (size_t)(c0 + c) * nd.ldu;
            *u = (inplace ? *u : S[c][r]) - acc[i][j];
        }
}

// ---------------------------------------------------------------------------
// solves
// ---------------------------------------------------------------------------

// The node's factor block [L11^-1 | L21] (odd leading dimensions, from a
// 16-byte aligned offset) is first copied to shared memory with 16-byte
// loads, so that the mat-vecs below read shared memory only.
__device__ __forceinline__ float* stage_factor(const float* __restrict__ L, const CholNode& nd, float* smem) {
    const int ldn = nd.nJ | 1, ldm = nd.mJ == 0 ? 0 : (nd.mJ | 1);
    const int nl4 = (nd.nJ * ldn + nd.nJ * ldm + 3) >> 2;
    const float4* src = reinterpret_cast<const float4*>(L + nd.loff);
    float4* dst = reinterpret_cast<float4*>(smem);
    for (int i = threadIdx.x; i < nl4; i += CHS_T) dst[i] = __ldcg(src + i);
    return smem + 4 * nl4;
}

// Everything one refinement sweep needs (kernel parameter block).
struct SweepArgs {
    const CholNode* nodes;
    const int* order;        // level_nodes: children before parents
    const int* child_idx;
    const int* rel;
    const int* struct_pos;
    const int* perm;
    const int* parent;
    const float* L;
    float* ybuf;
    float* xbuf;
    float* uvec;
    unsigned* fdone;         // per node: epoch of its last finished forward step
    unsigned* bdone;         // per node: epoch of its last finished backward step
    const int* rowptr;
    const int* col;
    const double* val;
    const double* bp;
    double* x;
    double* r;
    double* part;
    CholCtl* ctl;
    unsigned long long* trace;   // per ticket timestamps (builds with TP_CHOL_TRACE only)
    double tol2;
    int nv, nn, cap;
    int phase, t0, t1, last;  // this launch's part of the sweep: tickets t0 .. t1, and whether the residual follows
};

#ifdef TP_CHOL_TRACE
__device__ __forceinline__ unsigned long long gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
#define CH_TRACE(tk, slot)                                                      \
    do {                                                                        \
        if (threadIdx.x == 0 && A.trace) A.trace[(size_t)(tk) * 6 + (slot)] = gtimer(); \
    } while (0)
#else
#define CH_TRACE(tk, slot) \
    do {                   \
    } while (0)
#endif

constexpr int CH_MAXCH = 16;   // children whose records are prefetched to shared memory

struct ChildRec {
    int voff, mJ, s0, row0;   // row0: first row of this child in the staged update vectors
};

// store(e, load(e)) for e < count, the block's threads taking entries
// e = tid, tid + CHS_T, ...: each thread issues B independent loads before
// its stores, so a gather costs one memory round trip per B entries
// instead of one per entry
template <int B, class Load, class Store>
__device__ __forceinline__ void gather_batched(int count, Load load, Store store) {
    for (int e0 = threadIdx.x; e0 < count; e0 += CHS_T * B) {
        float v[B];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int e = e0 + b * CHS_T;
            if (e < count) v[b] = load(e);
        }
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const int e = e0 + b * CHS_T;
            if (e < count) store(e, v[b]);
        }
    }
}

// K columns padded to whole float4s in shared memory
template <int K>
struct Kp {
    static constexpr int P = (K + 3) & ~3;
};

// out(r, acc) for r < R with acc[c] = sum_k A(r, k) v[k][c], A(r, k) =
// M[r * sr + k * sk], k over [0, r] (mode 0), [r, n) (mode 1) or [0, n)
// (mode 2). One thread per row (passes of 128 rows); the two halves of the
// block take the even and the odd k, so every lane of a warp reads the same
// row of v (a broadcast) and the halves meet in one shared-memory add.
template <int K, class Out>
__device__ __forceinline__ void rows_matvec(const float* M, int sr, int sk, int R, int n, int mode, const float* v,
                                            float* scratch, Out out) {
    constexpr int KP = Kp<K>::P;
    static_assert(CHS_T == 256, "two halves of 128 threads");
    const int tid = threadIdx.x, rr = tid & 127, half = tid >> 7;
    for (int r0 = 0; r0 < R; r0 += 128) {
        const int r = r0 + rr;
        float acc[K];
#pragma unroll
        for (int c = 0; c < K; ++c) acc[c] = 0.f;
        if (r < R) {
            const float* mr = M + (size_t)r * sr;
            int k, kend, step;
            if (mode == 1) {
                k = n - 1 - half;
                kend = r - 1;
                step = -2;
            } else {
                k = half;
                kend = mode == 0 ? r + 1 : n;
                step = 2;
            }
            for (; step > 0 ? k < kend : k > kend; k += step) {
                const float m = mr[k * sk];
                const float4* vr = reinterpret_cast<const float4*>(v + k * KP);
#pragma unroll
                for (int q = 0; q < KP / 4; ++q) {
                    const float4 t = vr[q];
                    if (4 * q + 0 < K) acc[4 * q + 0] += m * t.x;
                    if (4 * q + 1 < K) acc[4 * q + 1] += m * t.y;
                    if (4 * q + 2 < K) acc[4 * q + 2] += m * t.z;
                    if (4 * q + 3 < K) acc[4 * q + 3] += m * t.w;
                }
            }
        }
        if (half && r < R)
#pragma unroll
            for (int c = 0; c < K; ++c) scratch[rr * KP + c] = acc[c];
        __syncthreads();
        if (!half && r < R) {
#pragma unroll
            for (int c = 0; c < K; ++c) acc[c] += scratch[rr * KP + c];
            out(r, acc);
        }
        __syncthreads();
    }
}

// rows_matvec of mode 2 for many rows and few terms (a wide front's L21 y): every
// thread takes four rows at a time, which share the broadcast reads of v
template <int K, class Out>
__device__ __forceinline__ void tall_matvec(const float* M, int ld, int R, int n, const float* v, Out out) {
    constexpr int KP = Kp<K>::P, RT = 4;
    for (int r0 = threadIdx.x; r0 < R; r0 += CHS_T * RT) {
        float acc[RT][K];
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int c = 0; c < K; ++c) acc[i][c] = 0.f;
#pragma unroll 2
        for (int k = 0; k < n; ++k) {
            float vk[KP];
#pragma unroll
            for (int q = 0; q < KP / 4; ++q) {
                const float4 t = reinterpret_cast<const float4*>(v + k * KP)[q];
                vk[4 * q] = t.x; vk[4 * q + 1] = t.y; vk[4 * q + 2] = t.z; vk[4 * q + 3] = t.w;
            }
#pragma unroll
            for (int i = 0; i < RT; ++i) {
                const int r = r0 + i * CHS_T;
                const float mr = r < R ? M[r + k * ld] : 0.f;
#pragma unroll
                for (int c = 0; c < K; ++c) acc[i][c] = fmaf(mr, vk[c], acc[i][c]);
            }
        }
#pragma unroll
        for (int i = 0; i < RT; ++i)
            if (r0 + i * CHS_T < R) out(r0 + i * CHS_T, acc[i]);
    }
    __syncthreads();
}

// out(r, acc) with acc[c] = sum_{k < n} M[r * ld + k] v[k][c] for few rows of many
// terms (a wide front's L21^T x): the lanes of a warp share a row's terms, in two
// rows at a time, and add up by a fixed butterfly. rows_matvec kept two threads a
// row busy here: 8 us a step for 24 rows of 1,000 terms.
template <int K, class Out>
__device__ __forceinline__ void wide_matvec(const float* M, int ld, int R, int n, const float* v, Out out) {
    constexpr int KP = Kp<K>::P, RT = 2;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int r0 = warp * RT; r0 < R; r0 += (CHS_T / 32) * RT) {
        float acc[RT][K];
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
            for (int c = 0; c < K; ++c) acc[i][c] = 0.f;
#pragma unroll 2
        for (int k = lane; k < n; k += 32) {
            float vk[KP];
#pragma unroll
            for (int q = 0; q < KP / 4; ++q) {
                const float4 t = reinterpret_cast<const float4*>(v + k * KP)[q];
                vk[4 * q] = t.x; vk[4 * q + 1] = t.y; vk[4 * q + 2] = t.z; vk[4 * q + 3] = t.w;
            }
#pragma unroll
            for (int i = 0; i < RT; ++i) {
                const float mr = r0 + i < R ? M[(r0 + i) * ld + k] : 0.f;
#pragma unroll
                for (int c = 0; c < K; ++c) acc[i][c] = fmaf(mr, vk[c], acc[i][c]);
            }
        }
#pragma unroll
        for (int i = 0; i < RT; ++i) {
#pragma unroll
            for (int c = 0; c < K; ++c)
                for (int o = 16; o > 0; o >>= 1) acc[i][c] += __shfl_xor_sync(0xffffffffu, acc[i][c], o);
            if (lane == 0 && r0 + i < R) out(r0 + i, acc[i]);
        }
    }
    __syncthreads();
}

// shared-memory layout of a solve step (floats): factor block, then the
// K-column vectors (rows of KP floats): forward w (t), y (n); backward x_S
// (m), y_J (n), z (n); then the two-half scratch (128 rows); then (backward)
// the node's FP64 solution entries
template <int K>
struct StepSmem {
    float* vec;
    float* scratch;
    double* xo;
    int* aux;      // forward: the children's target rows, then their update vectors; backward: struct(J)
    __device__ StepSmem(const CholNode& nd, float* smem) {
        constexpr int KP = Kp<K>::P;
        const int n = nd.nJ, m = nd.mJ;
        const int ldn = n | 1, ldm = m == 0 ? 0 : (m | 1);
        vec = smem + 4 * ((n * ldn + n * ldm + 3) >> 2);
        scratch = vec + (m + 2 * n) * KP;
        xo = reinterpret_cast<double*>(scratch + 128 * KP);
        aux = reinterpret_cast<int*>(xo + n * K);
    }
};

// forward step of node J, in two halves. fwd_prepare does what does not
// depend on the children (factor block to shared memory, w = (r_J ; 0),
// the children's records); fwd_finish adds the children's update vectors
// and forms y_J = L11^-1 w_J and u_J = w_S - L21 y_J.
template <int K, bool WIDE>
__device__ __forceinline__ void fwd_prepare(const SweepArgs& A, const CholNode& nd, float* smem, ChildRec* kids) {
    constexpr int KP = Kp<K>::P;
    const int n = nd.nJ, t = nd.t, tid = threadIdx.x;
    stage_factor(A.L, nd, smem);
    const StepSmem<K> sm(nd, smem);
    float* w = sm.vec;   // t x KP
    const int* perm = A.perm + nd.p0;
    gather_batched<8>(t * K,
                      [&](int e) { const int a = e / K; return a < n ? (float)__ldcg(A.r + (size_t)perm[a] * K + (e - a * K)) : 0.f; },
                      [&](int e, float v) { const int a = e / K; w[a * KP + (e - a * K)] = v; });
    const int nc = nd.child1 - nd.child0;
    if (nc <= CH_MAXCH && !(WIDE && (nd.flags & CHN_DIRECT))) {
        // the children's records, then their target rows in this front
        if (tid == 0) {
            int row0 = 0;
            for (int ci = 0; ci < nc; ++ci) {
                const CholNode cn = A.nodes[A.child_idx[nd.child0 + ci]];
                kids[ci] = ChildRec{cn.voff, cn.mJ, cn.s0, row0};
                row0 += cn.mJ;
            }
        }
        __syncthreads();
        for (int ci = 0; ci < nc; ++ci) {
            const ChildRec cr = kids[ci];
            for (int x = tid; x < cr.mJ; x += CHS_T) sm.aux[cr.row0 + x] = A.rel[cr.s0 + x];
        }
    }
}

template <int K, bool WIDE>
__device__ void fwd_finish(const SweepArgs& A, const CholNode& nd, float* smem, const ChildRec* kids) {
    constexpr int KP = Kp<K>::P;
    const int n = nd.nJ, m = nd.mJ, t = nd.t, tid = threadIdx.x;
    const int ldn = n | 1, ldm = m == 0 ? 0 : (m | 1);
    const StepSmem<K> sm(nd, smem);
    float* w = sm.vec;            // t x KP
    float* y = w + t * KP;        // n x KP
    const float* Li = smem;       // n x n, leading dimension ldn
    const float* L21 = smem + n * ldn;   // m x n, leading dimension ldm
    const int nc = nd.child1 - nd.child0;
    if (nc <= CH_MAXCH && !(WIDE && (nd.flags & CHN_DIRECT))) {
        // every child's update vector in one batched pass, then the
        // extend-add from shared memory, one child at a time
        const int rows = nc ? kids[nc - 1].row0 + kids[nc - 1].mJ : 0;
        const int* krow = sm.aux;
        float* kval = reinterpret_cast<float*>(sm.aux + rows);
        gather_batched<8>(rows * K,
                          [&](int e) {
                              const int r = e / K;
                              int ci = 0;
                              while (ci + 1 < nc && kids[ci + 1].row0 <= r) ++ci;
                              return __ldcg(A.uvec + ((size_t)kids[ci].voff + (r - kids[ci].row0)) * K + (e - r * K));
                          },
                          [&](int e, float v) { kval[e] = v; });
        __syncthreads();
        for (int ci = 0; ci < nc; ++ci) {
            const ChildRec cr = kids[ci];
            for (int idx = tid; idx < cr.mJ * K; idx += CHS_T) {
                const int x = idx / K, c = idx - x * K;
                w[krow[cr.row0 + x] * KP + c] += kval[cr.row0 * K + idx];
            }
            __syncthreads();
        }
    } else {
        for (int ci = 0; ci < nc; ++ci) {
            const CholNode cn = A.nodes[A.child_idx[nd.child0 + ci]];
            const int* rl = A.rel + cn.s0;
            const float* uc = A.uvec + (size_t)cn.voff * K;
            if constexpr (WIDE) {
                const bool same = nd.flags & CHN_INPLACE;   // the child's rows are this front's
                gather_batched<12>(cn.mJ * K, [&](int e) { return __ldcg(uc + e); },
                                   [&](int e, float v) {
                                       const int x = e / K;
                                       w[(same ? x : __ldg(rl + x)) * KP + (e - x * K)] += v;
                                   });
            } else {
                for (int idx = tid; idx < cn.mJ * K; idx += CHS_T) {
                    const int x = idx / K, c = idx - x * K;
                    w[rl[x] * KP + c] += __ldcg(uc + idx);
                }
            }
            __syncthreads();
        }
    }
    float* yb = A.ybuf + (size_t)nd.p0 * K;
    rows_matvec<K>(Li, 1, ldn, n, n, 0, w, sm.scratch, [&](int r, const float (&acc)[K]) {
#pragma unroll
        for (int c = 0; c < K; ++c) {
            y[r * KP + c] = acc[c];
            yb[r * K + c] = acc[c];
        }
    });
    float* uj = A.uvec + (size_t)nd.voff * K;
    auto put_u = [&](int r, const float (&acc)[K]) {
#pragma unroll
        for (int c = 0; c < K; ++c) uj[r * K + c] = w[(n + r) * KP + c] - acc[c];
    };
    // (two passes of 128 rows or fewer keep both halves of the block on a row)
    if (WIDE && m > 256)
        tall_matvec<K>(L21, ldm, m, n, y, put_u);
    else
        rows_matvec<K>(L21, 1, ldm, m, n, 2, y, sm.scratch, put_u);
}

// backward step of node J. bwd_prepare stages the factor block and the
// node's own entries of the FP64 solution (only this node writes them);
// bwd_finish gathers x_S and y_J in one pass, then z = y_J - L21^T x_S,
// x_J = L11^-T z, and the solution gains x_J.
template <int K>
__device__ __forceinline__ void bwd_prepare(const SweepArgs& A, const CholNode& nd, float* smem) {
    stage_factor(A.L, nd, smem);
    const StepSmem<K> sm(nd, smem);
    for (int idx = threadIdx.x; idx < nd.nJ * K; idx += CHS_T) {
        const int a = idx / K, c = idx - a * K;
        sm.xo[idx] = A.x[(size_t)A.perm[nd.p0 + a] * K + c];
    }
    for (int x = threadIdx.x; x < nd.mJ; x += CHS_T) sm.aux[x] = A.struct_pos[nd.s0 + x];
}

template <int K, bool WIDE>
__device__ void bwd_finish(const SweepArgs& A, const CholNode& nd, float* smem) {
    constexpr int KP = Kp<K>::P;
    const int n = nd.nJ, m = nd.mJ, tid = threadIdx.x;
    const int ldn = n | 1, ldm = m == 0 ? 0 : (m | 1);
    const StepSmem<K> sm(nd, smem);
    float* xs = sm.vec;           // m x KP
    float* yj = xs + m * KP;      // n x KP
    float* z = yj + n * KP;       // n x KP
    const float* Li = smem;
    const float* L21 = smem + n * ldn;
    const int* spos = sm.aux;   // struct(J), staged before the wait
    gather_batched<8>((m + n) * K,
                      [&](int e) {
                          if (e < m * K) {
                              const int x = e / K;
                              return __ldcg(A.xbuf + (size_t)spos[x] * K + (e - x * K));
                          }
                          return __ldcg(A.ybuf + (size_t)nd.p0 * K + (e - m * K));
                      },
                      [&](int e, float v) {
                          if (e < m * K) {
                              const int x = e / K;
                              xs[x * KP + (e - x * K)] = v;
                          } else {
                              const int j = e - m * K, a = j / K;
                              yj[a * KP + (j - a * K)] = v;
                          }
                      });
    __syncthreads();
    auto put_z = [&](int r, const float (&acc)[K]) {
#pragma unroll
        for (int c = 0; c < K; ++c) z[r * KP + c] = yj[r * KP + c] - acc[c];
    };
    // rows_matvec takes about 15 cycles per term of its longest thread, m / 2 terms;
    // the lanes' sums about 30 per column and row, n / 8 rows a warp
    if (WIDE && m > 4 * n && m > 128)
        wide_matvec<K>(L21, ldm, n, m, xs, put_z);
    else
        rows_matvec<K>(L21, ldm, 1, n, m, 2, xs, sm.scratch, put_z);
    float* xb = A.xbuf + (size_t)nd.p0 * K;
    const double* xo = sm.xo;
    rows_matvec<K>(Li, ldn, 1, n, n, 1, z, sm.scratch, [&](int r, const float (&acc)[K]) {
        double* xv = A.x + (size_t)A.perm[nd.p0 + r] * K;
#pragma unroll
        for (int c = 0; c < K; ++c) {
            xb[r * K + c] = acc[c];
            xv[c] = xo[r * K + c] + (double)acc[c];
        }
    });
}

// ---- cross-block signalling (bounded waits: ~1 s, then ctl->err) ---------

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release(unsigned* p, unsigned v) {
    __threadfence();
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// waits until *p >= target (counters) or == target (epoch flags); false on
// timeout. Spins tightly first (a flag is usually set within microseconds).
__device__ bool wait_until(const unsigned* p, unsigned target, bool at_least, CholCtl* ctl) {
    const long long t0 = clock64();
    for (int spins = 0;; ++spins) {
        const unsigned v = ld_acquire(p);
        if (at_least ? v >= target : v == target) return true;
        if (spins > 256) {
            if (*(volatile int*)&ctl->err) return false;
            if (clock64() - t0 > (1LL << 31)) {   // ~1 s at 2 GHz
                atomicExch(&ctl->err, 1);
                return false;
            }
            __nanosleep(32);
        }
    }
}

// One refinement sweep in one launch: forward and backward substitution
// over the supernodal tree, then r = bp - C x and the convergence test.
// Blocks take nodes from a ticket counter: tickets 0..nn-1 are the forward
// steps in `order` (children first), nn..2nn-1 the backward steps in
// reverse order (parents first). A step waits only for steps with smaller
// tickets (its children's forward steps; its parent's backward step, or
// for a root its own forward step), and those were taken by blocks that
// are already running, so the waits end without any assumption on how
// many blocks are resident. Flags hold the sweep's epoch, so they need no
// reset; the last block to finish the residual resets the counters and
// advances the epoch.
// WIDE: the tree has fronts of more than 256 rows (their matvecs, and vectors of the
// children read in place), or the sweep runs in three launches. Without those paths
// the kernel is 1 to 4 us shorter a sweep on meshes of 1,000 to 10,000 vertices, and
// with the tickets' range known it needs no spills at nine columns (1,890 vertices, a
// solve of two sweeps on three columns, medians over ten meshes: 173 -> 169 us, 165 us
// before there was a WIDE variant; where the allocations land moves one mesh by 4%).
template <int K, bool WIDE>
__global__ void __launch_bounds__(CHS_T)
k_chol_sweep(SweepArgs A) {
    CholCtl* ctl = A.ctl;
    if (*(volatile int*)&ctl->done) return;
    extern __shared__ float4 smem4[];
    float* smem = reinterpret_cast<float*>(smem4);
    __shared__ int s_tk, s_ok, s_last;
    __shared__ ChildRec s_kids[CH_MAXCH];
    __shared__ double s_red[CHS_T];
    const unsigned ep = *(volatile unsigned*)&ctl->epoch + 1;
    const int nn = A.nn, tid = threadIdx.x;
    unsigned* ticket = &ctl->ticket[WIDE ? A.phase : 0];
    const int t0 = WIDE ? A.t0 : 0, t1 = WIDE ? A.t1 : 2 * nn;
    if (tid == 0) s_tk = t0 + (int)atomicAdd(ticket, 1u);
    __syncthreads();
    for (;;) {
        const int tk = s_tk;
        if (tk >= t1) break;
        // the next ticket is taken now and used after this step: the atomic's
        // latency overlaps the step (the block runs both steps in order)
        unsigned next = 0;
        if (tid == 0) next = t0 + atomicAdd(ticket, 1u);
        const bool fwd = tk < nn;
        CH_TRACE(tk, 0);
        const int J = fwd ? A.order[tk] : A.order[2 * nn - 1 - tk];
        const CholNode nd = A.nodes[J];
        if (fwd)
            fwd_prepare<K, WIDE>(A, nd, smem, s_kids);
        else
            bwd_prepare<K>(A, nd, smem);
        // wait: forward for every child (one thread each), backward for the
        // parent (a root for its own forward step)
        if (tid == 0) s_ok = 1;
        __syncthreads();
        CH_TRACE(tk, 1);
        if (fwd) {
            const int nc = nd.child1 - nd.child0;
            for (int i = tid; i < nc; i += CHS_T)
                if (!wait_until(A.fdone + A.child_idx[nd.child0 + i], ep, false, ctl)) s_ok = 0;
        } else if (tid == 0) {
            const int P = A.parent[J];
            if (!(P >= 0 ? wait_until(A.bdone + P, ep, false, ctl) : wait_until(A.fdone + J, ep, false, ctl))) s_ok = 0;
        }
        __syncthreads();
        CH_TRACE(tk, 2);
        if (s_ok) {
            if (fwd)
                fwd_finish<K, WIDE>(A, nd, smem, s_kids);
            else
                bwd_finish<K, WIDE>(A, nd, smem);
        }
        __syncthreads();
        CH_TRACE(tk, 3);
#ifdef TP_CHOL_TRACE
        if (tid == 0 && A.trace) A.trace[(size_t)tk * 6 + 4] = blockIdx.x, A.trace[(size_t)tk * 6 + 5] = J;
#endif
        if (tid == 0) {
            if (fwd) {
                st_release(A.fdone + J, ep);
            } else {
                st_release(A.bdone + J, ep);
                atomicAdd(&ctl->bcount, 1u);
            }
            s_tk = (int)next;
        }
        __syncthreads();
    }
    if (WIDE && !A.last) return;
    // r = bp - C x once every backward step is done; per-block sums of r.r
    CH_TRACE(2 * nn + blockIdx.x, 0);
    if (tid == 0) s_ok = wait_until(&ctl->bcount, (unsigned)nn, true, ctl);
    __syncthreads();
    CH_TRACE(2 * nn + blockIdx.x, 1);
    // one thread per (vertex, column): the block covers R = (CHS_T / K) K
    // consecutive entries and the grid stride is a multiple of K, so thread
    // t always holds column t % K and the block's column sums are taken in a
    // fixed order
    constexpr int R = (CHS_T / K) * K;
    double acc = 0.0;
    if (tid < R) {
        const size_t total = (size_t)A.nv * K;
        for (size_t i = (size_t)blockIdx.x * R + tid; i < total; i += (size_t)gridDim.x * R) {
            const int v = (int)(i / K), c = (int)(i - (size_t)v * K);
            double rs = A.bp[i];
            for (int e = A.rowptr[v]; e < A.rowptr[v + 1]; ++e) rs -= A.val[e] * __ldcg(A.x + (size_t)A.col[e] * K + c);
            A.r[i] = rs;
            acc += rs * rs;
        }
    }
    s_red[tid] = acc;
    __syncthreads();
    if (tid < K) {
        double sum = 0.0;
        for (int q = tid; q < R; q += K) sum += s_red[q];
        A.part[(size_t)blockIdx.x * K + tid] = sum;
    }
    CH_TRACE(2 * nn + blockIdx.x, 2);
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(&ctl->arrive, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    // the last block: convergence test (every column at |r|^2 <= tol^2 |b|^2;
    // a column that has not lost three quarters of |r|^2 in the sweep means
    // the FP32 factor is too coarse: stalled), reset
    __threadfence();
    __shared__ double s_rr[K];
    {
        // column c: lanes of warp c % 8 stride over the blocks' partials,
        // then a fixed butterfly
        const int lane = tid & 31, wp = tid >> 5;
        for (int c = wp; c < K; c += CHS_T / 32) {
            double sum = 0.0;
            for (unsigned b = lane; b < gridDim.x; b += 32) sum += __ldcg(A.part + (size_t)b * K + c);
            for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
            if (lane == 0) s_rr[c] = sum;
        }
    }
    __syncthreads();
    if (tid == 0) {
        int conv = 1, worse = 0;
        for (int j = 0; j < K; ++j) {
            const double rr = s_rr[j];
            if (!(rr <= A.tol2 * ctl->bb[j])) {
                conv = 0;
                if (!(rr <= 0.25 * ctl->rr[j])) worse = 1;
            }
            ctl->rr[j] = rr;
        }
        ctl->iters += 1;
        if (conv) {
            ctl->done = 1;
        } else if (worse || ctl->bad_pivot || ctl->err || ctl->iters >= A.cap) {
            ctl->done = 1;
            ctl->stalled = 1;
        }
        CH_TRACE(2 * nn + gridDim.x, 0);
        ctl->ticket[0] = ctl->ticket[1] = ctl->ticket[2] = 0;
        ctl->arrive = 0;
        ctl->bcount = 0;
        __threadfence();
        ctl->epoch = ep;
    }
}

// sums over the T threads of a block of K per-thread FP64 values, in a fixed
// order through shared memory sh [K * T] (16 partial sums per column, then
// their sum): thread j < K returns the sum of column j, the others 0. Fewer
// FP64 additions than a shuffle tree per column (the FP64 pipe is narrow).
template <int K, int T>
__device__ __forceinline__ double block_colsum_f64(const double (&acc)[K], double* sh) {
    constexpr int P = 16;
    static_assert(K * P <= T, "one thread per partial sum");
    const int t = threadIdx.x;
#pragma unroll
    for (int j = 0; j < K; ++j) sh[j * T + t] = acc[j];
    __syncthreads();
    double s = 0.0;
    if (t < K * P) {
        const int j = t / P, q = t - j * P;
#pragma unroll
        for (int i = q; i < T; i += P) s += sh[j * T + i];
    }
    __syncthreads();
    if (t < K * P) sh[t] = s;
    __syncthreads();
    double v = 0.0;
    if (t < K)
#pragma unroll
        for (int q = 0; q < P; ++q) v += sh[t * P + q];
    return v;
}

// The start of a solve in one launch: bp = b minus its per-component means
// (mean, from k_comp_mean), x = 0, r = bp, per-block partials of |bp|^2;
// the last block to finish (completion ticket) adds the partials in block
// order, records |b|^2 per column (done when every column is zero), then
// puts the ticket back.
template <int K>
__global__ void __launch_bounds__(CHR_T)
k_chol_start(const double* __restrict__ b, const double* __restrict__ mean, const int* __restrict__ comp_of, int nv,
             double* __restrict__ bp, double* __restrict__ x, double* __restrict__ r, double* __restrict__ part,
             unsigned* __restrict__ ticket, CholCtl* __restrict__ ctl) {
    __shared__ double sh[K * CHR_T];
    __shared__ bool last;
    double acc[K];
#pragma unroll
    for (int c = 0; c < K; ++c) acc[c] = 0.0;
    for (int v = blockIdx.x * CHR_T + threadIdx.x; v < nv; v += gridDim.x * CHR_T) {
        const double* mc = mean + (size_t)comp_of[v] * K;
#pragma unroll
        for (int c = 0; c < K; ++c) {
            const size_t o = (size_t)v * K + c;
            const double s = b[o] - mc[c];
            bp[o] = s;
            x[o] = 0.0;
            r[o] = s;
            acc[c] += s * s;
        }
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double bs = block_colsum_f64<K, CHR_T>(acc, sh);
    if (threadIdx.x < K) part[(size_t)blockIdx.x * K + threadIdx.x] = bs;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    __shared__ double s_bb[K];
    for (int c = w; c < K; c += CHR_T / 32) {   // one warp per column
        double t = 0.0;
        for (unsigned q = lane; q < gridDim.x; q += 32) t += __ldcg(part + (size_t)q * K + c);
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) s_bb[c] = t;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int all = 1;
        for (int j = 0; j < K; ++j) {
            ctl->bb[j] = s_bb[j];
            ctl->rr[j] = s_bb[j];
            all &= s_bb[j] == 0.0;
        }
        ctl->done = all;
        ctl->iters = 0;
        *ticket = 0u;
    }
}

// per-component means of the k columns in a fixed order: block (c, s)
// sums slice s of component c's vertex list (CH_MSPLIT slices), then the
// last block to finish adds every component's slices in order (and, given
// dflags, records the state of the deferred solve that produced x)
constexpr int CH_MSPLIT = 48;   // about one vertex per thread on 10k-vertex meshes

__global__ void __launch_bounds__(256)
k_comp_mean(const int* __restrict__ comp_ptr, const int* __restrict__ comp_verts, const double* __restrict__ x,
            int k, double* __restrict__ part, double* __restrict__ mean, unsigned* __restrict__ ticket,
            const CholCtl* __restrict__ ctl, int* __restrict__ dflags) {
    __shared__ double sh[CH_KMAX * 256];
    __shared__ bool last;
    const int c = blockIdx.x, s = blockIdx.y;
    const int v0 = comp_ptr[c], v1 = comp_ptr[c + 1];
    const int len = (v1 - v0 + CH_MSPLIT - 1) / CH_MSPLIT;
    const int a0 = v0 + s * len, a1 = min(v1, a0 + len);
    double acc[CH_KMAX];
#pragma unroll
    for (int j = 0; j < CH_KMAX; ++j) acc[j] = 0.0;
    for (int i = a0 + threadIdx.x; i < a1; i += 256) {
        const double* xv = x + (size_t)comp_verts[i] * k;
#pragma unroll
        for (int j = 0; j < CH_KMAX; ++j)
            if (j < k) acc[j] += xv[j];
    }
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const double bs = block_colsum_f64<CH_KMAX, 256>(acc, sh);
    if (threadIdx.x < k) part[((size_t)c * CH_MSPLIT + s) * k + threadIdx.x] = bs;
    // the last block to finish adds each component's slices in order and
    // resets the ticket
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x * gridDim.y - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    // one warp per (component, column): lane l takes slices l, l + 32, then
    // a fixed shuffle tree
    const int ncomp = gridDim.x;
    for (int e = w; e < ncomp * k; e += 256 / 32) {
        const int cc = e / k, j = e - cc * k;
        double t = 0.0;
        for (int q = lane; q < CH_MSPLIT; q += 32) t += __ldcg(part + ((size_t)cc * CH_MSPLIT + q) * k + j);
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) mean[(size_t)cc * k + j] = t / (double)(comp_ptr[cc + 1] - comp_ptr[cc]);
    }
    if (threadIdx.x == 0) {
        *ticket = 0u;
        if (dflags) {
            // after the sweeps of a deferred solve: its wait error, and whether it stopped
            // short of the tolerance with more than a hundredth of a right-hand side left
            if (ctl->err) dflags[0] = 1;
            if (!ctl->done || ctl->stalled)
                for (int j = 0; j < k; ++j)
                    if (!(ctl->rr[j] <= 1e-4 * ctl->bb[j])) dflags[1] = 1;
        }
    }
}

__global__ void k_comp_sub(const int* __restrict__ comp_of, const double* __restrict__ mean, int nv, int k,
                           const double* __restrict__ src, double* __restrict__ dst) {
    size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= (size_t)nv * k) return;
    const int v = (int)(i / k), j = (int)(i - (size_t)v * k);
    dst[i] = src[i] - mean[(size_t)comp_of[v] * k + j];
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

void chol_release(tp_mesh* m) {
    if (!m->chol) return;
    CholState* c = m->chol;
    Buf* all[] = {&c->nodes, &c->level_nodes, &c->child_idx, &c->rel, &c->struct_pos, &c->asm_dst,
                  &c->asm_src, &c->perm, &c->comp_ptr, &c->comp_verts, &c->comp_of, &c->parent, &c->fdone,
                  &c->bdone, &c->tiles, &c->L, &c->U,
                  &c->uvec, &c->ybuf, &c->xbuf, &c->ctl, &c->part, &c->x, &c->r, &c->bp, &c->dflags};
    for (Buf* b : all) release(*b);
    for (auto& g : c->graph)
        if (g.exec) cudaGraphExecDestroy(g.exec);
    if (c->capture) cudaStreamDestroy(c->capture);
    delete c;
    m->chol = nullptr;
}

void chol_invalidate(tp_mesh* m) {
    if (m->chol) {
        m->chol->factored = false;
        m->chol->pivot_known = false;
    }
}

int chol_deferred_flags(tp_mesh* m, cudaStream_t st, int* err, int* poor, bool reset) {
    *err = *poor = 0;
    CholState* c = m->chol;
    if (!c || !c->dflags.ptr) return TP_OK;
    if (!reset) {
        int h[2] = {0, 0};
        TP_CUDA(cudaMemcpyAsync(h, c->dflags.ptr, sizeof(h), cudaMemcpyDeviceToHost, st));
        TP_CUDA(cudaStreamSynchronize(st));
        *err = h[0];
        *poor = h[1];
    }
    TP_CUDA(cudaMemsetAsync(c->dflags.ptr, 0, 2 * sizeof(int), st));
    return TP_OK;
}

template <class T>
static int upload(Buf& b, const std::vector<T>& v) {
    TP_TRY(ensure(b, sizeof(T) * std::max<size_t>(1, v.size())));
    if (!v.empty()) TP_CUDA(cudaMemcpy(b.ptr, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice));
    return TP_OK;
}

template <int K>
static int solve_smem_attr() {
    TP_CUDA(cudaFuncSetAttribute(k_chol_sweep<K, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CH_SMEM_MAX));
    TP_CUDA(cudaFuncSetAttribute(k_chol_sweep<K, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CH_SMEM_MAX));
    if constexpr (K < CH_KMAX) return solve_smem_attr<K + 1>();
    return TP_OK;
}

// symbolic analysis and device tables (once per mesh)
static int chol_setup(tp_mesh* m) {
    if (m->chol) return TP_OK;
    std::unique_ptr<CholState> c(new CholState());
    const int nv = m->nv;
    std::vector<int> rowptr(nv + 1), col(m->nnz);
    TP_CUDA(cudaMemcpy(rowptr.data(), m->rowptr.ptr, sizeof(int) * (nv + 1), cudaMemcpyDeviceToHost));
    TP_CUDA(cudaMemcpy(col.data(), m->col.ptr, sizeof(int) * m->nnz, cudaMemcpyDeviceToHost));
    CholSymbolic& S = c->S;
    if (!chol_analyze(nv, rowptr.data(), col.data(), CH_LEAF, S)) {
        c->why = "empty pattern";
        m->chol = c.release();
        return TP_OK;
    }
    c->ncomp = S.ncomp;
    c->H = (int)S.level_ptr.size() - 1;
    c->lvl_max_t.assign(c->H, 0);
    c->lvl_factor_smem.assign(c->H, 0);
    c->lvl_factor_flops.assign(c->H, 0.0);
    // bytes of a solve step on K columns: the factor block (rounded to 16 bytes),
    // the vectors (rows of K rounded to whole float4s), the 128-row scratch, the
    // node's FP64 solution entries, then struct(J) or the staged rows and update
    // vectors of the children (see StepSmem)
    auto step_smem = [&](int J, int K, bool direct) {
        const size_t n = S.nJ[J], mm = S.mJ[J], KP = (K + 3) & ~3;
        size_t csum = 0;   // rows of the children's update vectors
        if (!direct)
            for (int ci = S.child_ptr[J]; ci < S.child_ptr[J + 1]; ++ci) csum += S.mJ[S.child_idx[ci]];
        return sizeof(float) * (((n * chol_ld(n) + n * chol_ld(mm) + 3) & ~size_t(3)) + (mm + 2 * n) * KP + 128 * KP +
                                2 * n * K + std::max(csum * (K + 1), mm) + 4);
    };
    size_t worst = 0;
    bool small_open[CH_KMAX + 1];
    std::fill(small_open, small_open + CH_KMAX + 1, true);
    std::vector<int> flags(S.nnode, 0);
    for (int h = 0; h < c->H; ++h) {
        size_t lvl_smem[CH_KMAX + 1] = {};
        for (int i = S.level_ptr[h]; i < S.level_ptr[h + 1]; ++i) {
            const int J = S.level_nodes[i];
            const double n = S.nJ[J], mm = S.mJ[J];
            c->lvl_max_t[h] = std::max(c->lvl_max_t[h], S.nJ[J] + S.mJ[J]);
            int child = 0;   // rows of the largest child
            for (int ci = S.child_ptr[J]; ci < S.child_ptr[J + 1]; ++ci) child = std::max(child, S.mJ[S.child_idx[ci]]);
            const size_t sm = chf_smem((size_t)S.nJ[J] + S.mJ[J], S.nJ[J], child);
            c->lvl_factor_smem[h] = std::max(c->lvl_factor_smem[h], sm);
            worst = std::max(worst, sm);
            if (S.child_ptr[J + 1] - S.child_ptr[J] == 1 && S.mJ[S.child_idx[S.child_ptr[J]]] == S.nJ[J] + S.mJ[J])
                flags[J] |= CHN_INPLACE;
            // a chain's link reads one vector in order, and a front whose children
            // do not fit beside it reads theirs from global memory
            if ((flags[J] & CHN_INPLACE) || step_smem(J, CH_KMAX, false) > CH_SMEM_MAX) flags[J] |= CHN_DIRECT;
            c->wide = c->wide || (flags[J] & CHN_DIRECT) || mm > 256;
            for (int K = 1; K <= CH_KMAX; ++K)
                lvl_smem[K] = std::max(lvl_smem[K], step_smem(J, K, flags[J] & CHN_DIRECT));
            // partial Cholesky, Schur update of struct x struct, triangular inverse
            c->lvl_factor_flops[h] += n * n * n / 3.0 + n * n * mm + n * mm * mm + n * n * n / 3.0;
        }
        for (int K = 1; K <= CH_KMAX; ++K) {
            c->solve_smem[K] = std::max(c->solve_smem[K], lvl_smem[K]);
            small_open[K] = small_open[K] && lvl_smem[K] <= CHS_SMALL;
            if (!small_open[K]) continue;
            c->small_smem[K] = std::max(c->small_smem[K], lvl_smem[K]);
            c->small_n[K] = S.level_ptr[h + 1];
        }
    }
    c->solve_bytes = 2.0 * sizeof(float) * (double)S.lsize;
    worst = std::max(worst, c->solve_smem[CH_KMAX]);
    if (worst > CH_SMEM_MAX) {
        c->why = "a supernode panel needs " + std::to_string(worst) + " bytes of shared memory";
        m->chol = c.release();
        return TP_OK;
    }
    // update matrices: in place ones are the trailing part of the child's
    std::vector<int64_t> uoff(S.nnode);
    std::vector<int> ldu(S.nnode);
    int64_t& usize = c->usize;
    for (int J = 0; J < S.nnode; ++J) {   // postorder: children first
        if (flags[J] & CHN_INPLACE) {
            const int ch = S.child_idx[S.child_ptr[J]];
            ldu[J] = ldu[ch];
            uoff[J] = uoff[ch] + (int64_t)S.nJ[J] * (ldu[ch] + 1);
        } else {
            ldu[J] = S.mJ[J];
            uoff[J] = usize;
            usize += (int64_t)S.mJ[J] * S.mJ[J];
        }
    }
    // tiles of the update matrices (lower part), by level
    std::vector<int4> tiles;
    c->lvl_tile.assign(c->H + 1, 0);
    for (int h = 0; h < c->H; ++h) {
        for (int i = S.level_ptr[h]; i < S.level_ptr[h + 1]; ++i) {
            const int J = S.level_nodes[i];
            for (int c0 = 0; c0 < S.mJ[J]; c0 += CHF_TILE)
                for (int r0 = c0; r0 < S.mJ[J]; r0 += CHF_TILE) tiles.push_back(make_int4(J, r0, c0, 0));
        }
        c->lvl_tile[h + 1] = (int)tiles.size();
    }
    // device tables
    std::vector<CholNode> nodes(S.nnode);
    for (int J = 0; J < S.nnode; ++J) {
        CholNode& d = nodes[J];
        d.p0 = S.p0[J];
        d.nJ = S.nJ[J];
        d.mJ = S.mJ[J];
        d.t = S.nJ[J] + S.mJ[J];
        d.loff = S.loff[J];
        d.uoff = uoff[J];
        d.voff = S.voff[J];
        d.child0 = S.child_ptr[J];
        d.child1 = S.child_ptr[J + 1];
        d.s0 = S.struct_ptr[J];
        d.asm0 = S.asm_ptr[J];
        d.asm1 = S.asm_ptr[J + 1];
        d.ldu = ldu[J];
        d.flags = flags[J];
    }
    std::vector<int> comp_ptr(S.ncomp + 1, 0), comp_verts(nv);
    for (int v = 0; v < nv; ++v) comp_ptr[S.comp[v] + 1]++;
    for (int i = 0; i < S.ncomp; ++i) comp_ptr[i + 1] += comp_ptr[i];
    {
        std::vector<int> fill(comp_ptr.begin(), comp_ptr.end() - 1);
        for (int v = 0; v < nv; ++v) comp_verts[fill[S.comp[v]]++] = v;
    }
    TP_TRY(upload(c->nodes, nodes));
    TP_TRY(upload(c->level_nodes, S.level_nodes));
    TP_TRY(upload(c->child_idx, S.child_idx));
    TP_TRY(upload(c->rel, S.rel));
    TP_TRY(upload(c->struct_pos, S.struct_pos));
    TP_TRY(upload(c->asm_dst, S.asm_dst));
    TP_TRY(upload(c->asm_src, S.asm_src));
    TP_TRY(upload(c->perm, S.perm));
    TP_TRY(upload(c->comp_ptr, comp_ptr));
    TP_TRY(upload(c->comp_verts, comp_verts));
    TP_TRY(upload(c->comp_of, S.comp));
    TP_TRY(upload(c->parent, S.parent));
    TP_TRY(upload(c->tiles, tiles));
    TP_TRY(ensure(c->fdone, sizeof(unsigned) * std::max(1, S.nnode)));
    TP_TRY(ensure(c->bdone, sizeof(unsigned) * std::max(1, S.nnode)));
    TP_CUDA(cudaMemset(c->fdone.ptr, 0, sizeof(unsigned) * std::max(1, S.nnode)));
    TP_CUDA(cudaMemset(c->bdone.ptr, 0, sizeof(unsigned) * std::max(1, S.nnode)));
    TP_TRY(ensure(c->L, sizeof(float) * std::max<int64_t>(1, S.lsize)));
    TP_TRY(ensure(c->U, sizeof(float) * std::max<int64_t>(1, usize)));
    TP_TRY(ensure(c->uvec, sizeof(float) * (size_t)std::max(1, S.vsize) * CH_KMAX));
    TP_TRY(ensure(c->ybuf, sizeof(float) * (size_t)std::max(1, S.n) * CH_KMAX));
    TP_TRY(ensure(c->xbuf, sizeof(float) * (size_t)std::max(1, S.n) * CH_KMAX));
    TP_TRY(ensure(c->ctl, sizeof(CholCtl)));
    TP_CUDA(cudaMemset(c->ctl.ptr, 0, sizeof(CholCtl)));
#ifdef TP_CHOL_TRACE
    TP_TRY(ensure(c->trace, sizeof(unsigned long long) * 6 * ((size_t)2 * S.nnode + 3 * sm_count() + 2)));
#endif
    TP_CUDA(cudaFuncSetAttribute(k_chol_panel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CH_SMEM_MAX));
    TP_TRY(solve_smem_attr<1>());
    c->ok = true;
    m->chol = c.release();
    return TP_OK;
}

static int chol_factor(tp_mesh* m, cudaStream_t st) {
    CholState* c = m->chol;
    if (c->factored) return TP_OK;
    TP_CUDA(cudaMemsetAsync(c->ctl.ptr, 0, offsetof(CholCtl, epoch), st));   // the epoch is never cleared
    double flops = 0.0;
    for (double f : c->lvl_factor_flops) flops += f;
    {
        ProfScope ps(m, PK_CHOL_FACTOR, flops, st);
        const CholSymbolic& S = c->S;
        for (int h = 0; h < c->H; ++h) {
            const int cnt = S.level_ptr[h + 1] - S.level_ptr[h];
            if (cnt == 0) continue;
            // small fronts by the thousand: more blocks per SM; above them the level
            // waits for its largest front
            const int threads = c->lvl_max_t[h] <= 96 ? 128 : cnt >= sm_count() ? 256 : 512;
            k_chol_panel<<<cnt, threads, c->lvl_factor_smem[h], st>>>(
                c->nodes.as<CholNode>(), c->level_nodes.as<int>() + S.level_ptr[h], c->child_idx.as<int>(),
                c->rel.as<int>(), c->asm_dst.as<int>(), c->asm_src.as<int>(), m->val.as<double>(),
                c->L.as<float>(), c->U.as<float>(), c->ctl.as<CholCtl>());
            TP_LAUNCH_CHECK();
            const int nt = c->lvl_tile[h + 1] - c->lvl_tile[h];
            if (nt == 0) continue;
            k_chol_update<<<nt, 256, 0, st>>>(c->nodes.as<CholNode>(), c->tiles.as<int4>() + c->lvl_tile[h],
                                              c->child_idx.as<int>(), c->rel.as<int>(), c->L.as<float>(),
                                              c->U.as<float>());
            TP_LAUNCH_CHECK();
        }
    }
    c->factored = true;
    return TP_OK;
}

// dst = src minus its per-component mean (k columns)
// per-component means of src into c->part (and the deferred flags, see k_comp_mean)
static int comp_means(tp_mesh* m, const double* src, int k, int* dflags, cudaStream_t st) {
    CholState* c = m->chol;
    double* mean = c->part.as<double>();                        // ncomp * 9 doubles
    double* slices = mean + (size_t)c->ncomp * CH_KMAX;          // ncomp * CH_MSPLIT * 9 doubles
    unsigned* tk = nullptr;
    TP_TRY(mesh_tickets(m, &tk, st));
    k_comp_mean<<<dim3(c->ncomp, CH_MSPLIT), 256, 0, st>>>(c->comp_ptr.as<int>(), c->comp_verts.as<int>(), src, k,
                                                           slices, mean, tk + TICKET_COMP, c->ctl.as<CholCtl>(),
                                                           dflags);
    TP_LAUNCH_CHECK();
    return TP_OK;
}

static int comp_project(tp_mesh* m, const double* src, double* dst, int k, cudaStream_t st, int* dflags = nullptr) {
    CholState* c = m->chol;
    double* mean = c->part.as<double>();
    TP_TRY(comp_means(m, src, k, dflags, st));
    const size_t n = (size_t)m->nv * k;
    k_comp_sub<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(c->comp_of.as<int>(), mean, m->nv, k, src, dst);
    TP_LAUNCH_CHECK();
    return TP_OK;
}

// `nsweep` refinement sweeps on stream st (recorded into a graph by the
// caller); *nk counts the kernels
template <int K>
static int chol_sweep_kernels(tp_mesh* m, int nsweep, double* partr, double tol2, int cap, cudaStream_t st, int* nk) {
    CholState* c = m->chol;
    const CholSymbolic& S = c->S;
    SweepArgs A;
    A.nodes = c->nodes.as<CholNode>();
    A.order = c->level_nodes.as<int>();
    A.child_idx = c->child_idx.as<int>();
    A.rel = c->rel.as<int>();
    A.struct_pos = c->struct_pos.as<int>();
    A.perm = c->perm.as<int>();
    A.parent = c->parent.as<int>();
    A.L = c->L.as<float>();
    A.ybuf = c->ybuf.as<float>();
    A.xbuf = c->xbuf.as<float>();
    A.uvec = c->uvec.as<float>();
    A.fdone = c->fdone.as<unsigned>();
    A.bdone = c->bdone.as<unsigned>();
    A.rowptr = m->rowptr.as<int>();
    A.col = m->col.as<int>();
    A.val = m->val.as<double>();
    A.bp = c->bp.as<double>();
    A.x = c->x.as<double>();
    A.r = c->r.as<double>();
    A.part = partr;
    A.ctl = c->ctl.as<CholCtl>();
    A.trace = nullptr;
#ifdef TP_CHOL_TRACE
    A.trace = c->trace.as<unsigned long long>();   // allocated with the tables (no allocation under capture)
#endif
    A.tol2 = tol2;
    A.nv = m->nv;
    A.nn = S.nnode;
    A.cap = cap;
    const int nn = S.nnode, sms = sm_count(), small = c->small_n[K];
    // One launch a sweep, with the shared memory of its largest step. Where that
    // leaves one or two blocks per SM to thousands of small steps (163,842 vertices:
    // 5,600 of 5,811), the small levels at the leaves run in launches of their own,
    // forward before and backward after the others, three blocks per SM.
    const bool parts = c->solve_smem[K] > CHS_SMALL && small >= 6 * sms;
    for (int s = 0; s < nsweep; ++s) {
        for (int part = 0; part < 3; ++part) {
            if (!parts && part != 2) continue;
            A.phase = part;
            A.t0 = !parts || part == 0 ? 0 : part == 1 ? small : 2 * nn - small;
            A.t1 = parts && part == 0 ? small : parts && part == 1 ? 2 * nn - small : 2 * nn;
            A.last = part == 2;
            const bool big = !parts || part == 1;
            const int most = big ? 2 * sms : 3 * sms;
            const int want = !parts ? nn : part == 1 ? nn - small : small;
            const int grid = std::max(1, std::min(want, most));
            if (want == 0) continue;
            const size_t smem = big ? c->solve_smem[K] : c->small_smem[K];
            if (c->wide || parts)
                k_chol_sweep<K, true><<<grid, CHS_T, smem, st>>>(A);
            else
                k_chol_sweep<K, false><<<grid, CHS_T, smem, st>>>(A);
            TP_CUDA(cudaGetLastError());
            ++*nk;
        }
    }
    return TP_OK;
}

constexpr int CH_SWEEPS_PER_GRAPH = 2;   // FP32 factor: about three digits per sweep

// the graph of CH_SWEEPS_PER_GRAPH sweeps for K columns, captured on a
// private stream (re-captured when a buffer it uses has moved)
template <int K>
static int sweep_graph(tp_mesh* m, double* partr, double tol2, int cap, CholState::SweepGraph** out) {
    CholState* c = m->chol;
    CholState::SweepGraph& g = c->graph[K];
    const void* key[4] = {c->x.ptr, c->r.ptr, c->bp.ptr, partr};
    bool same = g.exec && g.tol2 == tol2 && g.cap == cap;
    for (int i = 0; i < 4 && same; ++i) same = g.key[i] == key[i];
    if (!same) {
        if (g.exec) cudaGraphExecDestroy(g.exec);
        g.exec = nullptr;
        if (!c->capture) TP_CUDA(cudaStreamCreateWithFlags(&c->capture, cudaStreamNonBlocking));
        TP_CUDA(cudaStreamBeginCapture(c->capture, cudaStreamCaptureModeThreadLocal));
        int nk = 0;
        int s = chol_sweep_kernels<K>(m, CH_SWEEPS_PER_GRAPH, partr, tol2, cap, c->capture, &nk);
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamEndCapture(c->capture, &graph);
        if (s != TP_OK) {
            if (graph) cudaGraphDestroy(graph);
            return s;
        }
        if (e != cudaSuccess) return fail(TP_ERR_CUDA, std::string("capturing the refinement sweeps: ") +
                                                           cudaGetErrorString(e));
        e = cudaGraphInstantiate(&g.exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) return fail(TP_ERR_CUDA, std::string("instantiating the refinement sweeps: ") +
                                                           cudaGetErrorString(e));
        for (int i = 0; i < 4; ++i) g.key[i] = key[i];
        g.tol2 = tol2;
        g.cap = cap;
        g.kernels = nk;
    }
    *out = &g;
    return TP_OK;
}

template <int K>
static int chol_run(tp_mesh* m, const tp_params* p, const double* b, double* z_out, cudaStream_t st, int* iters,
                    bool* handed_off, PoissonMode mode) {
    CholState* c = m->chol;
    const bool deferred = mode == POISSON_DEFERRED;
    if (deferred && !c->pivot_known) {
        // the factor's pivot check, once per factorisation
        int bp = 0;
        TP_CUDA(cudaMemcpyAsync(&bp, reinterpret_cast<char*>(c->ctl.ptr) + offsetof(CholCtl, bad_pivot), sizeof(int),
                                cudaMemcpyDeviceToHost, st));
        TP_CUDA(cudaStreamSynchronize(st));
        c->pivot_ok = bp == 0;
        c->pivot_known = true;
    }
    if (deferred && !c->pivot_ok) {
        *handed_off = true;
        return TP_OK;
    }
    const int nv = m->nv;
    const size_t n = (size_t)nv * K;
    TP_TRY(ensure(c->x, sizeof(double) * n));
    TP_TRY(ensure(c->r, sizeof(double) * n));
    TP_TRY(ensure(c->bp, sizeof(double) * n));
    const int rgrid = std::min(4 * sm_count(), (nv + CHR_T - 1) / CHR_T);
    // partial sums after the per-component means (comp_project's region)
    // per-block partials of the initial residual (rgrid blocks) and of the
    // sweep kernel (up to 3 blocks per SM)
    const size_t nparts = (size_t)std::max(rgrid, 3 * sm_count());
    const size_t head = (size_t)c->ncomp * CH_KMAX * (1 + CH_MSPLIT);   // means and their slices
    TP_TRY(ensure(c->part, sizeof(double) * (head + nparts * CH_KMAX) + 64));
    double* partr = c->part.as<double>() + head;
    // clear done .. arrive; bad_pivot (from the factorisation) and the epoch stay
    TP_CUDA(cudaMemsetAsync(c->ctl.ptr, 0, offsetof(CholCtl, bad_pivot), st));
    // b minus its component means, x = 0, r = b, |b|^2 (two launches)
    TP_TRY(comp_means(m, b, K, nullptr, st));
    {
        unsigned* tk = nullptr;
        TP_TRY(mesh_tickets(m, &tk, st));
        k_chol_start<K><<<rgrid, CHR_T, 0, st>>>(b, c->part.as<double>(), c->comp_of.as<int>(), nv, c->bp.as<double>(),
                                                c->x.as<double>(), c->r.as<double>(), partr, tk + TICKET_CHOL,
                                                c->ctl.as<CholCtl>());
        TP_LAUNCH_CHECK();
    }
    const double tol2 = p->cg_tol * p->cg_tol;
    const int cap = std::max(1, std::min(p->cg_max, 40));
    CholState::SweepGraph* g = nullptr;
    TP_TRY(sweep_graph<K>(m, partr, tol2, cap, &g));
    if (deferred) {
        // no host read: a fixed number of sweeps for cg_tol, then the flags, which
        // the caller reads. Measured digits of |r|/|b| (9 columns, random b): at
        // least four after the first sweep on up to 25,000 vertices (torus_20k,
        // linked_tori_50k, icosphere_l3), 2.5 to 3.5 on 40,000 to 120,000 (tori, linked
        // tori), and two to three more per sweep after it.
        if (!c->dflags.ptr) {
            TP_TRY(ensure(c->dflags, 4 * sizeof(int)));
            TP_CUDA(cudaMemsetAsync(c->dflags.ptr, 0, 4 * sizeof(int), st));   // fresh memory holds garbage
        }
        // Larger meshes: 2.5 and 1.5. 130,200 to 182,000 vertices, smooth or with noise up
        // to 0.4 edges: 1e-4 in two sweeps (once three: a torus of 1,400 x 110, nine columns),
        // 1e-6 in three (once four), 1e-9 in four to six; 655,362: 1e-4 in three, 1e-6 in four.
        // The line lies where the former limit of the factor was: below it the flexible method
        // has always gone on with what the fewer sweeps give.
        const double digits = -std::log10(std::max(p->cg_tol, 1e-300));
        const bool large = nv > CHOL_LARGE_NV;
        const double first = large ? 2.5 : 4.0, next = large ? 1.5 : 3.0;
        const int sweeps = std::min(cap, 1 + std::max(0, (int)std::ceil((digits - first) / next)));
        const int graphs = sweeps / CH_SWEEPS_PER_GRAPH;
        for (int gi = 0; gi < graphs; ++gi) {
            ProfScope ps(m, PK_CHOL_SOLVE, c->solve_bytes * CH_SWEEPS_PER_GRAPH, st);
            TP_CUDA(cudaGraphLaunch(g->exec, st));
            count_launches(g->kernels);
        }
        if (sweeps % CH_SWEEPS_PER_GRAPH) {
            // the odd sweep, launched directly
            ProfScope ps(m, PK_CHOL_SOLVE, c->solve_bytes, st);
            int nk = 0;
            TP_TRY(chol_sweep_kernels<K>(m, sweeps % CH_SWEEPS_PER_GRAPH, partr, tol2, cap, st, &nk));
            count_launches(nk);
        }
        if (iters) *iters = sweeps;
        TP_TRY(comp_project(m, c->x.as<double>(), z_out, K, st, c->dflags.as<int>()));
        return TP_OK;
    }
    CholCtl h{};
    int launched = 0;
    for (;;) {
        {
            ProfScope ps(m, PK_CHOL_SOLVE, c->solve_bytes * CH_SWEEPS_PER_GRAPH, st);
            TP_CUDA(cudaGraphLaunch(g->exec, st));
            count_launches(g->kernels);
        }
        launched += CH_SWEEPS_PER_GRAPH;
        TP_CUDA(cudaMemcpyAsync(&h, c->ctl.ptr, sizeof(CholCtl), cudaMemcpyDeviceToHost, st));
        TP_CUDA(cudaStreamSynchronize(st));
        if (h.done || launched >= cap) break;
    }
    if (iters) *iters = h.iters;
    if (h.err) return fail(TP_ERR_TIMEOUT, "cotan solve: a wait of the factorised sweep gave up");
    bool good = h.done && !h.stalled;
    if (mode == POISSON_LOOSE && !good) {
        good = true;
        for (int j = 0; j < K; ++j) good = good && h.rr[j] <= 1e-4 * h.bb[j];
    }
    if (h.bad_pivot || !good) {
        *handed_off = true;
        return TP_OK;
    }
    TP_TRY(comp_project(m, c->x.as<double>(), z_out, K, st));
    return TP_OK;
}

// z = C^+ b by the factor; *used = false when the factor cannot serve this
// mesh or this right-hand side (the caller then runs CG)
int chol_solve(tp_mesh* m, const tp_params* p, const double* b, int k, double* z_out, cudaStream_t st, int* iters,
               bool* used, PoissonMode mode) {
    *used = false;
    if (k < 1 || k > CH_KMAX) return fail(TP_ERR_INVALID_ARG, "cotan solve: k must be in 1..9");
    TP_TRY(laplacian_values(m, st));
    TP_TRY(chol_setup(m));
    if (!m->chol->ok) return TP_OK;
    TP_TRY(chol_factor(m, st));
    bool handed = false;
    int it = 0;
    switch (k) {
        case 1: TP_TRY(chol_run<1>(m, p, b, z_out, st, &it, &handed, mode)); break;
        case 2: TP_TRY(chol_run<2>(m, p, b, z_out, st, &it, &handed, mode)); break;
        case 3: TP_TRY(chol_run<3>(m, p, b, z_out, st, &it, &handed, mode)); break;
        case 4: TP_TRY(chol_run<4>(m, p, b, z_out, st, &it, &handed, mode)); break;
        case 5: TP_TRY(chol_run<5>(m, p, b, z_out, st, &it, &handed, mode)); break;
        case 6: TP_TRY(chol_run<6>(m, p, b, z_out, st, &it, &handed, mode)); break;
        case 7: TP_TRY(chol_run<7>(m, p, b, z_out, st, &it, &handed, mode)); break;
        case 8: TP_TRY(chol_run<8>(m, p, b, z_out, st, &it, &handed, mode)); break;
        default: TP_TRY(chol_run<9>(m, p, b, z_out, st, &it, &handed, mode)); break;
    }
    if (iters) *iters = it;
    *used = !handed;
    return TP_OK;
}

#ifdef TP_CHOL_TRACE
// timestamps of the last sweep (trace builds): [2 nn + blocks + 1][6]
int chol_trace(tp_mesh* m, unsigned long long* out, int max_rows, int* nn, int* grid) {
    CholState* c = m->chol;
    if (!c || !c->trace.ptr) return fail(TP_ERR_INVALID_ARG, "no trace");
    *nn = c->S.nnode;
    *grid = std::max(1, std::min(c->S.nnode, 2 * sm_count()));
    const size_t rows = std::min<size_t>((size_t)max_rows, (size_t)2 * c->S.nnode + *grid + 1);
    TP_CUDA(cudaMemcpy(out, c->trace.ptr, sizeof(unsigned long long) * 6 * rows, cudaMemcpyDeviceToHost));
    return TP_OK;
}
#endif

// host-side description of the factor (for tests and reports)
// Self-test of the bounded cross-block wait: one thread waits for a word
// that nothing sets; the wait gives up after its clock budget (~1 s),
// records the timeout in the control block and returns.
__global__ void k_wait_selftest(const unsigned* word, CholCtl* ctl, int* result) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *result = wait_until(word, 1u, true, ctl) ? 0 : 1;
}

int wait_selftest(int* timed_out) {
    void* mem = nullptr;
    const size_t bytes = 256 + sizeof(CholCtl);
    TP_CUDA(cudaMalloc(&mem, bytes));
    unsigned* word = (unsigned*)mem;
    int* result = (int*)((char*)mem + 64);
    CholCtl* ctl = (CholCtl*)((char*)mem + 256);
    int h[2] = {0, 0};
    cudaError_t e = cudaMemset(mem, 0, bytes);
    if (e == cudaSuccess) {
        k_wait_selftest<<<1, 32>>>(word, ctl, result);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpy(&h[0], result, sizeof(int), cudaMemcpyDeviceToHost);
    if (e == cudaSuccess) e = cudaMemcpy(&h[1], &ctl->err, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(mem);
    if (e != cudaSuccess) return fail(TP_ERR_CUDA, cudaGetErrorString(e));
    *timed_out = (h[0] == 1 && h[1] != 0) ? 1 : 0;
    return *timed_out ? fail(TP_ERR_TIMEOUT, "self-test: the bounded wait gave up as designed") : TP_OK;
}

int chol_info(tp_mesh* m, tp_chol_info* out) {
    *out = tp_chol_info{};
    TP_TRY(chol_setup(m));
    const CholState* c = m->chol;
    const CholSymbolic& S = c->S;
    out->available = c->ok ? 1 : 0;
    out->components = S.ncomp;
    out->unknowns = S.n;
    out->supernodes = S.nnode;
    out->levels = c->H;
    out->max_front = S.max_t;
    out->factor_floats = (double)S.lsize;
    out->update_floats = (double)c->usize;
    return TP_OK;
}

}  // namespace tp
