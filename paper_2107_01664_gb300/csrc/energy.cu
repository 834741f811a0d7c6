// Direct energy and differential of Eq. 10 at p = 6 with FP32 pair terms: the
// all-pairs kernels of the default mode (pairs.cu holds the other exponents, FP64
// and the per-target rows).
//
// Both are bound by the FP32 pipe, so the work is in the operations of a pair.
//   Energy: only the sum is wanted, so an unordered pair is taken once with both of
//   its terms: K(S,T) + K(T,S) share d, |d|^2 and its reciprocal: 21 operations
//   and one MUFU in place of 28 and two. Only source tiles at or after the target
//   block's own are visited; inside the block's own tiles every ordered pair is
//   taken with one term (no pair is left out or counted twice there).
//   Differential: with t = u / |d|^2 and f = 2 / |d|^2 (the doubling is an integer
//   addition to the exponent, off the FP32 pipe) the terms are powers of t^ = u f
//   times a_T f, which keeps the ratio 2 between the two parts of dE/dX and needs
//   neither K nor the energy's own sum: 36 operations against 41. The 12 sums become
//   8: N_S . sum(w d) gives a K_ST's part of dE/da after the loop.
//
// Targets go in pairs through packed f32x2 instructions; a source's coordinates,
// normal and area are staged in shared memory already doubled ({x, x}, ...). Tiles
// near a block's targets take the same path with the differences of the low parts
// added. A block takes an equal run of units (32 sources against a row of targets),
// so no wave of blocks is left partly empty whatever the size. FP32 sums over 32
// sources (16 for dE of small meshes), Kahan pairs across them, FP64 from there.
//
// Measured: E on 20,000 / 69,690 faces 259 / 2,588 us -> 172 / 1,822 us; a call for dE
// and E on 2,176 / 20,000 / 69,690 faces 103 / 674 / 6,605 us -> 71 / 610 / 6,416 us. The
// FP32 pipe is busy 73% (E) and 70% (dE) of the SMs' active cycles; four targets a thread
// for dE (half the shared-memory reads) ran slower.
#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>

#include "tp_internal.cuh"

namespace tp {

namespace {

using u64 = unsigned long long;

constexpr int ET = 128;    // threads per block, sources per shared-memory tile
constexpr int EC = 32;     // sources per unit and FP32 sum
// blocks per resident block: tiles near a row's targets cost more, so equal runs of
// units do not take equal time, and several runs per slot even that out (20,000
// faces: 181 -> 172 us for E, 609 -> 566 us for dE)
constexpr long long GE = 4, GD = 2;

__device__ __forceinline__ u64 pk(float a, float b) {
    u64 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float2 up(u64 r) {
    float2 v;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v.x), "=f"(v.y) : "l"(r));
    return v;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
    u64 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 sub2(u64 a, u64 b) {
    u64 d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
    u64 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
    u64 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ float rcpf(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ u64 rcp2(u64 a) {
    const float2 v = up(a);
    return pk(rcpf(v.x), rcpf(v.y));
}
// twice the reciprocal, the factor 2 by the exponent (an argument of 2^126 or more
// gives 2^-126 in place of 0)
__device__ __forceinline__ u64 rcp2_twice(u64 a) {
    const float2 v = up(a);
    return pk(__uint_as_float(__float_as_uint(rcpf(v.x)) + 0x00800000u),
              __uint_as_float(__float_as_uint(rcpf(v.y)) + 0x00800000u));
}

struct alignas(16) Kahan2 {   // two compensated FP32 sums
    u64 s = 0ull, c = 0ull;
    __device__ __forceinline__ void add(u64 x) {
        const u64 y = sub2(x, c), t = add2(s, y);
        c = sub2(sub2(t, s), y);
        s = t;
    }
    __device__ __forceinline__ double value(int lane) const {
        const float2 a = up(s), b = up(c);
        return lane ? (double)a.y - (double)b.y : (double)a.x - (double)b.x;
    }
};

// a source tile: {x,x,y,y} {z,z,a,a} {nx,nx,ny,ny} {nz,nz,.,.} and the low parts
// {lx,lx,ly,ly} {lz,lz,.,.} per source
struct Tile {
    ulonglong2 g[ET][4];
    ulonglong2 l[ET][2];
};

__device__ __forceinline__ void stage(Tile& t, const float4* __restrict__ fa, const float4* __restrict__ fb,
                                      const float4* __restrict__ fl, int src, int nf, bool low) {
    // sources past the end: far away, zero area and normal (all their terms are zero)
    const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 A = src < nf ? fa[src] : make_float4(PAD_X, 0.f, 0.f, 0.f), N = src < nf ? fb[src] : z;
    ulonglong2* g = t.g[threadIdx.x];
    g[0] = make_ulonglong2(pk(A.x, A.x), pk(A.y, A.y));
    g[1] = make_ulonglong2(pk(A.z, A.z), pk(A.w, A.w));
    g[2] = make_ulonglong2(pk(N.x, N.x), pk(N.y, N.y));
    g[3] = make_ulonglong2(pk(N.z, N.z), 0ull);
    if (low) {
        const float4 L = src < nf ? fl[src] : z;
        t.l[threadIdx.x][0] = make_ulonglong2(pk(L.x, L.x), pk(L.y, L.y));
        t.l[threadIdx.x][1] = make_ulonglong2(pk(L.z, L.z), 0ull);
    }
}

// PP pairs of targets of a thread: 2 j and 2 j + 1 sit ET faces apart
template <int PP>
struct Targets {
    u64 x[PP], y[PP], z[PP], nx[PP], ny[PP], nz[PP], lx[PP], ly[PP], lz[PP];
    __device__ __forceinline__ void load(const float4* __restrict__ fa, const float4* __restrict__ fb,
                                         const float4* __restrict__ fl, int base, int nf, float (&lo)[3],
                                         float (&hi)[3]) {
        for (int c = 0; c < 3; ++c) lo[c] = 3e38f, hi[c] = -3e38f;
#pragma unroll
        for (int j = 0; j < PP; ++j) {
            float4 A[2], N[2], L[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int f = base + (2 * j + h) * ET + threadIdx.x;
                A[h] = N[h] = L[h] = make_float4(0.f, 0.f, 0.f, 0.f);   // past the end: zero normal
                if (f < nf) {
                    A[h] = fa[f];
                    N[h] = fb[f];
                    L[h] = fl[f];
                    lo[0] = fminf(lo[0], A[h].x); lo[1] = fminf(lo[1], A[h].y); lo[2] = fminf(lo[2], A[h].z);
                    hi[0] = fmaxf(hi[0], A[h].x); hi[1] = fmaxf(hi[1], A[h].y); hi[2] = fmaxf(hi[2], A[h].z);
                }
            }
            x[j] = pk(A[0].x, A[1].x); y[j] = pk(A[0].y, A[1].y); z[j] = pk(A[0].z, A[1].z);
            nx[j] = pk(N[0].x, N[1].x); ny[j] = pk(N[0].y, N[1].y); nz[j] = pk(N[0].z, N[1].z);
            lx[j] = pk(L[0].x, L[1].x); ly[j] = pk(L[0].y, L[1].y); lz[j] = pk(L[0].z, L[1].z);
        }
    }
    template <bool COMP>
    __device__ __forceinline__ void diff(int j, const Tile& t, int q, const ulonglong2& g0, const ulonglong2& g1,
                                         u64& dx, u64& dy, u64& dz) const {
        dx = sub2(x[j], g0.x);
        dy = sub2(y[j], g0.y);
        dz = sub2(z[j], g1.x);
        if (COMP) {
            const ulonglong2 l0 = t.l[q][0], l1 = t.l[q][1];
            dx = add2(dx, sub2(lx[j], l0.x));
            dy = add2(dy, sub2(ly[j], l0.y));
            dz = add2(dz, sub2(lz[j], l1.x));
        }
    }
};

// the warp's targets against a tile's box: whether any pair may be near
__device__ __forceinline__ void warp_box(float (&lo)[3], float (&hi)[3]) {
    for (int o = 16; o > 0; o >>= 1)
        for (int c = 0; c < 3; ++c) {
            lo[c] = fminf(lo[c], __shfl_xor_sync(0xffffffffu, lo[c], o));
            hi[c] = fmaxf(hi[c], __shfl_xor_sync(0xffffffffu, hi[c], o));
        }
}
__device__ __forceinline__ bool near_tile(const float4* __restrict__ tbox, int tile, const float (&lo)[3],
                                          const float (&hi)[3], float thr2) {
    const float4 l = tbox[2 * tile], h = tbox[2 * tile + 1];
    const float gx = fmaxf(fmaxf(l.x - hi[0], lo[0] - h.x), 0.f), gy = fmaxf(fmaxf(l.y - hi[1], lo[1] - h.y), 0.f),
                gz = fmaxf(fmaxf(l.z - hi[2], lo[2] - h.z), 0.f);
    return gx * gx + gy * gy + gz * gz < thr2;
}

// ---- energy -----------------------------------------------------------------

// 32 sources against PP pairs of targets; BOTH: with the reversed term
template <int PP, bool BOTH, bool COMP>
__device__ __forceinline__ void energy_chunk(const Tile& t, int c0, const Targets<PP>& T, u64 (&P)[PP]) {
    const u64 EPS = pk(1e-18f, 1e-18f);   // keeps the self pair finite (its terms are zero)
#pragma unroll 4
    for (int q = c0; q < c0 + EC; ++q) {
        const ulonglong2 g0 = t.g[q][0], g1 = t.g[q][1];
        ulonglong2 g2{}, g3{};
        if (BOTH) {
            g2 = t.g[q][2];
            g3 = t.g[q][3];
        }
#pragma unroll
        for (int j = 0; j < PP; ++j) {
            u64 dx, dy, dz;
            T.template diff<COMP>(j, t, q, g0, g1, dx, dy, dz);
            const u64 ir2 = rcp2(fma2(dx, dx, fma2(dy, dy, fma2(dz, dz, EPS))));
            const u64 tS = mul2(fma2(T.nx[j], dx, fma2(T.ny[j], dy, mul2(T.nz[j], dz))), ir2);
            const u64 qS = mul2(tS, tS);
            u64 K = mul2(mul2(qS, qS), qS);
            if (BOTH) {
                const u64 tT = mul2(fma2(g2.x, dx, fma2(g2.y, dy, mul2(g3.x, dz))), ir2);
                const u64 qT = mul2(tT, tT);
                K = fma2(mul2(qT, qT), qT, K);
            }
            P[j] = fma2(K, g1.y, P[j]);
        }
    }
}

// first unit of target row b (2 PP tiles of targets, nt source tiles): rows before
// it hold the units of the tiles at or after their own
__host__ __device__ __forceinline__ long long energy_row(long long b, long long nt, int tt) {
    return (ET / EC) * (b * nt - tt * (b * (b - 1) / 2));
}

// E = sum_S a_S sum_{T != S} K(S,T) a_T into *E: every block adds its runs, the last
// one to finish (completion ticket) the blocks' sums in order
template <int PP>
__global__ void __launch_bounds__(ET, PP == 2 ? 4 : 6)
k_energy_total(const float4* __restrict__ fa, const float4* __restrict__ fb, const float4* __restrict__ fl,
               const float4* __restrict__ tbox, const double* __restrict__ center, const d4* __restrict__ f64a, int nf,
               int nt, int rows, long long units, double* __restrict__ part, unsigned* __restrict__ ticket,
               double* __restrict__ E) {
    constexpr int TT = 2 * PP;
    __shared__ Tile t;
    __shared__ double red[ET / 32];
    __shared__ bool last;
    const int tid = threadIdx.x;
    const long long u1 = units * (blockIdx.x + 1) / gridDim.x;
    long long u = units * blockIdx.x / gridDim.x;
    const float thr2 = (float)center[3];
    double e = 0.0;
    int b;
    {   // the row of the first unit
        int lo = 0, hi = rows - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (energy_row(mid, nt, TT) <= u) lo = mid;
            else hi = mid - 1;
        }
        b = lo;
    }
    for (; u < u1; ++b) {
        const long long r0 = energy_row(b, nt, TT), r1 = min(u1, energy_row(b + 1, nt, TT));
        Targets<PP> T;
        float lo[3], hi[3];
        T.load(fa, fb, fl, b * TT * ET, nf, lo, hi);
        warp_box(lo, hi);
        Kahan2 acc[PP];
        while (u < r1) {
            const int c = (int)(u - r0), tile = b * TT + c / (ET / EC), q0 = c % (ET / EC);
            const int q1 = (int)min((long long)(ET / EC), q0 + (r1 - u));
            const bool own = tile < (b + 1) * TT;        // the block's own tiles: one term per ordered pair
            const bool near = near_tile(tbox, tile, lo, hi, thr2);
            __syncthreads();
            stage(t, fa, fb, fl, tile * ET + tid, nf, true);
            __syncthreads();
            for (int q = q0; q < q1; ++q) {
                u64 P[PP];
#pragma unroll
                for (int j = 0; j < PP; ++j) P[j] = 0ull;
                if (own)
                    energy_chunk<PP, false, true>(t, q * EC, T, P);
                else if (near)
                    energy_chunk<PP, true, true>(t, q * EC, T, P);
                else
                    energy_chunk<PP, true, false>(t, q * EC, T, P);
#pragma unroll
                for (int j = 0; j < PP; ++j) acc[j].add(P[j]);
            }
            u += q1 - q0;
        }
#pragma unroll
        for (int j = 0; j < PP; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int f = (b * TT + 2 * j + h) * ET + tid;
                if (f < nf) e = fma(f64a[f].w, acc[j].value(h), e);
            }
    }
    auto block_sum = [&](double v) {   // in thread 0
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        __syncthreads();
        if ((tid & 31) == 0) red[tid >> 5] = v;
        __syncthreads();
        return ((red[0] + red[1]) + red[2]) + red[3];
    };
    const double s = block_sum(e);
    if (tid == 0) {
        part[blockIdx.x] = s;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double v = 0.0;
    for (unsigned q = tid; q < gridDim.x; q += ET) v += __ldcg(part + q);
    const double tot = block_sum(v);
    if (tid == 0) {
        *E = tot;
        *ticket = 0u;
    }
}

// ---- differential -----------------------------------------------------------

// sums over the sources T (with f = 2 / |d|^2, u_S = N_S.d, u_T = N_T.d, t = u f):
// 0 a f t_S^5 | 1-3 the same times d | 4-6 a f t_T^5 N_T - (a f (t_S^6 + t_T^6)) d
// | 7 a f t_T^5 u_T. In the terms of the differential
//   a c_S = (0) / 64,  a (K_ST + K_TS) = (N_S . (1-3) + (7)) / 64,
//   p a c_T N_T - 2 p a (K_ST + K_TS) d / |d|^2 = p (4-6) / 64.
constexpr int DA = 8;
constexpr int DS = DA + 3;   // the FP32 sums keep the two parts of 4-6 apart: less rounding (they cancel)

template <bool COMP, int NC>
__device__ __forceinline__ void diff_chunk(const Tile& t, int c0, const Targets<1>& T, u64 (&s)[DS]) {
    const u64 EPS = pk(1e-18f, 1e-18f);
#pragma unroll 8
    for (int q = c0; q < c0 + NC; ++q) {
        const ulonglong2 g0 = t.g[q][0], g1 = t.g[q][1], g2 = t.g[q][2], g3 = t.g[q][3];
        u64 dx, dy, dz;
        T.template diff<COMP>(0, t, q, g0, g1, dx, dy, dz);
        const u64 r2 = fma2(dx, dx, fma2(dy, dy, fma2(dz, dz, EPS)));
        const u64 f = rcp2_twice(r2);
        const u64 tS = mul2(fma2(T.nx[0], dx, fma2(T.ny[0], dy, mul2(T.nz[0], dz))), f);
        const u64 uT = fma2(g2.x, dx, fma2(g2.y, dy, mul2(g3.x, dz))), tT = mul2(uT, f);
        const u64 qS = mul2(tS, tS), qT = mul2(tT, tT);
        const u64 af = mul2(g1.y, f);
        const u64 w = mul2(mul2(mul2(qS, qS), tS), af);
        const u64 v = mul2(mul2(mul2(qT, qT), tT), af);
        const u64 k = fma2(v, tT, mul2(w, tS));
        const float2 kf = up(k);
        const u64 nk = pk(-kf.x, -kf.y);
        s[0] = add2(s[0], w);
        s[1] = fma2(w, dx, s[1]);
        s[2] = fma2(w, dy, s[2]);
        s[3] = fma2(w, dz, s[3]);
        s[4] = fma2(v, g2.x, s[4]);
        s[5] = fma2(v, g2.y, s[5]);
        s[6] = fma2(v, g3.x, s[6]);
        s[8] = fma2(nk, dx, s[8]);
        s[9] = fma2(nk, dy, s[9]);
        s[10] = fma2(nk, dz, s[10]);
        s[7] = fma2(v, uT, s[7]);
    }
}

constexpr int DROW = 2 * ET;   // targets per row

// FP32 sums of dE over 16 sources up to this many faces, over 32 beyond. The error of dE
// against FP64 sums (noisy tori, means over 16 to 64 meshes): 512 / 2,176 / 6,820 /
// 10,080 faces 4.40 / 2.68 / 3.93 / 3.17e-7 with 32, 4.21 / 2.71 / 3.48 / 3.23e-7 with
// 16, against 4.35 / 2.78 / 3.75 / 3.62e-7 of the kernel with 12 sums; 16 sources cost
// nothing at 6,820 faces (133 us), 3 and 4% at 10,080 and 20,000 (208 -> 213, 610 -> 634).
constexpr int DIFF_SHORT = 8192;

// units of block b of G: [b U / G, (b + 1) U / G); row r's units start at r * per
__host__ __device__ __forceinline__ long long diff_block(long long u, long long U, long long G) {
    return ((u + 1) * G - 1) / U;
}

template <int NC>
__global__ void __launch_bounds__(ET, 5)
k_diff_sums(const float4* __restrict__ fa, const float4* __restrict__ fb, const float4* __restrict__ fl,
            const float4* __restrict__ tbox, const double* __restrict__ center, int nf, long long per, long long units,
            double* __restrict__ part) {
    __shared__ Tile t;
    __shared__ Kahan2 acc[DA][ET];   // in shared memory: the registers go to eight sources in flight
    const int tid = threadIdx.x;
    const long long u1 = units * (blockIdx.x + 1) / gridDim.x;
    long long u = units * blockIdx.x / gridDim.x;
    const float thr2 = (float)center[3];
    while (u < u1) {
        const long long row = u / per, r0 = row * per, r1 = min(u1, r0 + per);
        Targets<1> T;
        float lo[3], hi[3];
        T.load(fa, fb, fl, (int)row * DROW, nf, lo, hi);
        warp_box(lo, hi);
#pragma unroll
        for (int i = 0; i < DA; ++i) acc[i][tid] = Kahan2();
        while (u < r1) {
            const int c = (int)(u - r0), tile = c / (ET / EC), q0 = c % (ET / EC);
            const int q1 = (int)min((long long)(ET / EC), q0 + (r1 - u));
            const bool near = near_tile(tbox, tile, lo, hi, thr2);
            __syncthreads();
            stage(t, fa, fb, fl, tile * ET + tid, nf, true);
            __syncthreads();
            for (int q = q0 * (EC / NC); q < q1 * (EC / NC); ++q) {   // q * NC: source of the tile
                u64 s[DS];
#pragma unroll
                for (int i = 0; i < DS; ++i) s[i] = 0ull;
                if (near)
                    diff_chunk<true, NC>(t, q * NC, T, s);
                else
                    diff_chunk<false, NC>(t, q * NC, T, s);
#pragma unroll
                for (int i = 0; i < DA; ++i) {
                    Kahan2 k = acc[i][tid];
                    k.add(i >= 4 && i < 7 ? add2(s[i], s[i + 4]) : s[i]);
                    acc[i][tid] = k;
                }
            }
            u += q1 - q0;
        }
        // this run's sums, in the slot of the block among the row's blocks
        const long long slot = (long long)blockIdx.x - diff_block(r0, units, gridDim.x);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int f = (int)row * DROW + h * ET + tid;
            if (f < nf)
#pragma unroll
                for (int i = 0; i < DA; ++i) part[((size_t)slot * DA + i) * nf + f] = acc[i][tid].value(h);
        }
    }
}

// The slots' sums per face, then the face's adjoints (CORNER = false: adj [nf*7] and
// energy rows) or straight its corner gradients (§3.1, the chain rule of
// k_adj_to_corner) and the energy: E = 1/2 sum a_S sum a_T (K_ST + K_TS), block sums
// added by the last block to finish. 32 faces a block, a thread per (face, sum).
template <bool CORNER>
__global__ void __launch_bounds__(32 * DA)
k_diff_finish(const double* __restrict__ part, int nf, long long per, long long units, long long G, double p,
              const d4* __restrict__ f64a, const d4* __restrict__ f64b, const double* __restrict__ pos,
              const int* __restrict__ faces, double* __restrict__ out, double* __restrict__ erow,
              double* __restrict__ epart, unsigned* __restrict__ ticket, double* __restrict__ E) {
    __shared__ double sh[DA][33];
    __shared__ double red[DA];
    __shared__ bool last;
    const int fl = threadIdx.x & 31, i = threadIdx.x >> 5, S = blockIdx.x * 32 + fl;
    const long long row = blockIdx.x * 32 / DROW;   // 32 divides DROW: one row per block
    const int slots = (int)(diff_block((row + 1) * per - 1, units, G) - diff_block(row * per, units, G)) + 1;
    double x = 0.0;
    if (S < nf) {
        const double* ps = part + (size_t)i * nf + S;
#pragma unroll 4
        for (int s = 0; s < slots; ++s) x += ps[(size_t)s * DA * nf];
    }
    sh[i][fl] = x;
    __syncthreads();
    if (i == 0) {
        double er = 0.0;
        if (S < nf) {
            const d4 fa = f64a[S], fb = f64b[S];
            const double a = fa.w, N[3] = {fb.x, fb.y, fb.z};
            const double c = a * p * (1.0 / 64.0);
            double gX[3], gN[3];
            for (int q = 0; q < 3; ++q) {
                gX[q] = c * fma(x, N[q], sh[4 + q][fl]);
                gN[q] = c * sh[1 + q][fl];
            }
            // (the normal that the pair kernel had)
            const double ga = (sh[7][fl] + (double)(float)N[0] * sh[1][fl] + (double)(float)N[1] * sh[2][fl] +
                               (double)(float)N[2] * sh[3][fl]) * (1.0 / 64.0);
            er = 0.5 * a * ga;
            if (CORNER) {
                const double nn = 2.0 * a;
                const bool mid = nn > 1e-280 && nn < 1e280;
                const double rn = mid ? rcp64(nn) : 1.0 / nn;
                const size_t vi = faces[3 * S], vj = faces[3 * S + 1], vk = faces[3 * S + 2];
                double e1[3], e2[3], w[3];
                for (int q = 0; q < 3; ++q) {
                    e1[q] = pos[3 * vj + q] - pos[3 * vi + q];
                    e2[q] = pos[3 * vk + q] - pos[3 * vi + q];
                }
                const double gNn = gN[0] * N[0] + gN[1] * N[1] + gN[2] * N[2];
                for (int q = 0; q < 3; ++q) w[q] = div64(gN[q] - gNn * N[q], nn, rn) + 0.5 * ga * N[q];
                const double gj[3] = {e2[1] * w[2] - e2[2] * w[1], e2[2] * w[0] - e2[0] * w[2],
                                      e2[0] * w[1] - e2[1] * w[0]};
                const double gk[3] = {w[1] * e1[2] - w[2] * e1[1], w[2] * e1[0] - w[0] * e1[2],
                                      w[0] * e1[1] - w[1] * e1[0]};
                double* cr = out + 9 * (size_t)S;
                for (int q = 0; q < 3; ++q) {
                    const double third = third64(gX[q]);
                    cr[q] = -(gj[q] + gk[q]) + third;
                    cr[3 + q] = gj[q] + third;
                    cr[6 + q] = gk[q] + third;
                }
            } else {
                for (int q = 0; q < 3; ++q) {
                    out[7 * (size_t)S + q] = gX[q];
                    out[7 * (size_t)S + 3 + q] = gN[q];
                }
                out[7 * (size_t)S + 6] = ga;
                erow[S] = er;
            }
        }
        if (CORNER) {
            for (int o = 16; o > 0; o >>= 1) er += __shfl_xor_sync(0xffffffffu, er, o);
            if (fl == 0) {
                epart[blockIdx.x] = er;
                __threadfence();
                last = atomicAdd(ticket, 1u) == gridDim.x - 1;
            }
        }
    }
    if (!CORNER) return;
    __syncthreads();
    if (!last) return;
    __threadfence();
    double v = 0.0;
    for (unsigned q = threadIdx.x; q < gridDim.x; q += 32 * DA) v += __ldcg(epart + q);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (fl == 0) red[i] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int q = 0; q < DA; ++q) tot += red[q];
        *E = tot;
        *ticket = 0u;
    }
}

// resident blocks per SM of a kernel (cached per kernel and device)
int resident(const void* fn) {
    static std::mutex mu;
    static std::map<std::pair<const void*, int>, int> cache;
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lock(mu);
    const auto key = std::make_pair(fn, dev);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, ET, 0) != cudaSuccess || n < 1) {
        cudaGetLastError();
        n = 1;
    }
    return cache[key] = n;
}

template <int PP>
int launch_energy(tp_mesh* m, double* E_dev, cudaStream_t st) {
    const int nf = m->nf, nt = (nf + ET - 1) / ET, rows = (nt + 2 * PP - 1) / (2 * PP);
    const long long units = energy_row(rows, nt, 2 * PP);
    const long long G = std::min<long long>(units, GE * sm_count() * resident((const void*)k_energy_total<PP>));
    unsigned* tk = nullptr;
    TP_TRY(mesh_tickets(m, &tk, st));
    TP_TRY(ensure(m->part2, sizeof(double) * (size_t)G));
    const double pairs = (double)nf * (nf - 1);
    m->pairs += pairs;
    ProfScope ps(m, PK_ENERGY, pairs, st);
    k_energy_total<PP><<<(unsigned)G, ET, 0, st>>>(m->f32a.as<float4>(), m->f32b.as<float4>(), m->f32c.as<float4>(),
                                                   m->tilebox.as<float4>(), m->center.as<double>(), m->f64a.as<d4>(),
                                                   nf, nt, rows, units, m->part2.as<double>(), tk + TICKET_ENERGY,
                                                   E_dev);
    TP_LAUNCH_CHECK();
    return TP_OK;
}

}  // namespace

bool p6_fp32_direct(const tp_params* p) {
    return p->theta == 0.0 && p->precision == TP_PREC_FP32 && p->p == 6.0;
}

int energy_total_p6(tp_mesh* m, double* E_dev, cudaStream_t st) {
    // four targets a thread share each source's shared-memory reads; two where four
    // leave fewer units than two rounds of the SMs' four blocks (up to 24 tiles, 3,072
    // faces, on 152 SMs)
    const long long nt = (m->nf + ET - 1) / ET;
    return 2 * nt * nt / 4 * (ET / EC) >= 8LL * sm_count() ? launch_energy<2>(m, E_dev, st)
                                                           : launch_energy<1>(m, E_dev, st);
}

long long diff_p6_slots_max(int nf, int sms) {
    const long long per = (nf + ET - 1) / ET * (long long)(ET / EC), rows = (nf + DROW - 1) / DROW;
    return std::min(per, GD * sms * 8 / std::max(1LL, rows) + 2);
}

int diff_p6(tp_mesh* m, double* adj, double* erow, double* corner, double* E_dev, cudaStream_t st) {
    const int nf = m->nf, nt = (nf + ET - 1) / ET, rows = (nf + DROW - 1) / DROW;
    const long long per = (long long)nt * (ET / EC), units = per * rows;
    const auto kernel = nf <= DIFF_SHORT ? k_diff_sums<EC / 2> : k_diff_sums<EC>;
    const long long G = std::min<long long>(units, GD * sm_count() * resident((const void*)kernel));
    long long slots = 1;   // most blocks that share a row
    for (long long r = 0; r < rows; ++r)
        slots = std::max(slots, diff_block((r + 1) * per - 1, units, G) - diff_block(r * per, units, G) + 1);
    TP_TRY(ensure(m->part, sizeof(double) * (size_t)slots * DA * nf));
    const double pairs = (double)nf * (nf - 1);
    m->pairs += pairs;
    {
        ProfScope ps(m, PK_DIFF, pairs, st);
        kernel<<<(unsigned)G, ET, 0, st>>>(m->f32a.as<float4>(), m->f32b.as<float4>(), m->f32c.as<float4>(),
                                           m->tilebox.as<float4>(), m->center.as<double>(), nf, per, units,
                                           m->part.as<double>());
        TP_LAUNCH_CHECK();
    }
    const int nb = (nf + 31) / 32;
    unsigned* tk = nullptr;
    TP_TRY(mesh_tickets(m, &tk, st));
    TP_TRY(ensure(m->part2, sizeof(double) * (size_t)nb));
    if (corner)
        k_diff_finish<true><<<nb, 32 * DA, 0, st>>>(m->part.as<double>(), nf, per, units, G, 6.0, m->f64a.as<d4>(),
                                                    m->f64b.as<d4>(), m->pos.as<double>(), m->faces.as<int>(), corner,
                                                    nullptr, m->part2.as<double>(), tk + TICKET_ENERGY, E_dev);
    else
        k_diff_finish<false><<<nb, 32 * DA, 0, st>>>(m->part.as<double>(), nf, per, units, G, 6.0, m->f64a.as<d4>(),
                                                     m->f64b.as<d4>(), m->pos.as<double>(), m->faces.as<int>(), adj,
                                                     erow, nullptr, nullptr, nullptr);
    TP_LAUNCH_CHECK();
    return TP_OK;
}

}  // namespace tp
