// Tiled two-pass block H*V for spin-1/2 models on the full 2^N space, 32 real
// columns in FP32 or FP64 (16 complex columns: the cTPQ block of Sec. 3.5.2 and the
// real-time evolution of Sec. 3.4).
//
// Row s (an N-bit spin string) holds 32 columns, 128 (FP32) or 256 (FP64)
// contiguous bytes.  An
// exchange bond (i, j) with Jxy != 0 couples s with s ^ (2^i | 2^j) where the
// two bits differ (Sec. 3.1.1).  The single-pass kernels gather about 20 such
// rows per row from all over the 8.6 GB block and move about 6x the
// algorithmic bytes from DRAM.
//
// Here the off-diagonal bonds are split over two passes.  Pass k works on a
// bit set S_k: it walks the rows tile by tile, a tile being the 2^|S_k| rows
// that share the bits outside S_k, every thread block on the same tile at a
// time, and applies only bonds with both sites in S_k, so every gather stays
// inside the current tile, which is sized to a fraction of L2 and comes from
// DRAM once.  The sets come from the bond graph: A and B disjoint site sets
// with no bond between them, S_1 = all sites but A, S_2 = all sites but B;
// a bond touching A lies in S_2, one touching B in S_1, the rest in both
// (split for balance).  So each pass reads x once and the pair moves
//   pass 1: x, diagonal (one value per row), t written;
//   pass 2: x, t, v (the gamma term), y written
// instead of x about 17 times.
//   pass 1:  t[s] = d[s] x[s] + sum_{bonds of pass 1} c_b x[s ^ m_b]
//   pass 2:  acc = t[s] + sum_{bonds of pass 2} c_b x[s ^ m_b],
//            y = alpha acc + beta y + gamma v  (pair swap, fused reductions)
// d is the diagonal, sum_b Jz_b S^z_i S^z_j, stored once per Hamiltonian and
// precision.  t lives in y when y's old value is not read (beta = 0 and
// v != y), else in a context buffer.
//
// Inside a pass, a warp owns an item: the rows that share all bits but the
// first item bits of S_k (16 rows in FP32, 4 per lane, 16 bytes of a row per lane;
// 8 in FP64, all in every lane, one column per lane).  What a bond does to an item
// is decided once, one bond per lane: with both sites outside the item it applies
// to all its rows or to none; with one site inside, to the rows whose bit is the
// opposite of the other site's; with both inside, to the rows where the two
// differ, in two parts.  In every case the target rows lie at one fixed row
// offset, so an applicable bond is an entry (first target row, coefficient, masks
// of the rows and lane groups it touches) of the warp's list, and costs one address
// and, for 16 (8) rows, 4 (8) loads per lane and their FMAs; only bonds with a site
// inside test anything per row.  Every row sums its terms in a fixed order: deterministic.
//
// What bounds it: FP32 L2-to-SM traffic (22 sites, pass 1: 8.4 reads of 128 bytes
// per row at 10.1 TB/s; 26 sites about 11 per row and pass), FP64 the FP64 pipe
// (21-site chain, pass 1: 94 % busy, 5.5 operations per element).  Before, 8 lanes walked the bonds row
// by row, testing each bond on each row (74 to 80 warp instructions per row and
// pass).  ms per cTPQ step (6 stages), before and now: 26 sites of a 3-regular
// graph FP32 116 -> 102, 25-site chain FP32 50.7 -> 43.4, 21-site ladder FP64
// 25.6 -> 14.2, 22 sites FP64 57 -> 29.5.  Tried (26 sites): 24 warps per SM 123, 32
// 206 (more rows in flight leave L2 early), 2 rows per lane 122 to 217.
#include "fixed.cuh"
#include "hvcommon.cuh"

#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

namespace hphi {

namespace {

constexpr int kTileThreads = 256;
constexpr int kTileItemBits = 5;  // smallest tile
// sites of an FP32 item order's leading cluster: 2^7 rows are in a thread block at a
// time (26 sites: 103 against 106 ms a step in ascending order; FP64, bound by its
// pipe, was 3 % slower with it, so ascending there)
constexpr int kTileCluster = 8;
constexpr int kTileSlack = 1;     // half tiles that a block may be ahead of the average
constexpr int kTileWaits = 64;    // pacing polls at most
constexpr int kTileMin = 2;       // thread blocks per SM
// list entries in flight (FP32 12 16-byte, FP64 16 8-byte loads per lane)
template <typename T> constexpr int kTileUnroll = sizeof(T) == 4 ? 3 : 2;

// Lane layout of a 32-column row: E columns per lane, LPR lanes per row, 2^QB rows
// per warp access, 2^RB rows per lane, 2^IB rows per item.  FP32 lanes move 16
// bytes.  FP64 rows take a whole warp, so that which rows a bond touches is the
// same for all lanes and the FP64 pipe gets no FMA for the others (with two rows
// per access, masked, pass 1 of a 21-site chain ran 11 FP64 operations per
// element, 6.3 of them needed).
template <typename T>
struct TileShape {
    static constexpr int E = sizeof(T) == 4 ? 4 : 1;
    static constexpr int LPR = 32 / E;
    static constexpr int QB = sizeof(T) == 4 ? 2 : 0;
    static constexpr int RB = sizeof(T) == 4 ? 2 : 3;
    static constexpr int R = 1 << RB;
    static constexpr int IB = QB + RB;
};

// One applicable bond of a warp's item.
template <typename T>
struct alignas(16) TileHit;
template <>
struct alignas(16) TileHit<float> {
    int row;        // target of the item's first row
    uint32_t mask;  // rows (bits 0-3) and lane groups (bits 4-7) it applies to; FP64: rows (bits 0-7)
    float c;
};
template <>
struct alignas(16) TileHit<double> {
    double c;
    int row;
    uint32_t mask;
};

__device__ __forceinline__ void ldrow(const float *p, float (&v)[4]) {
    asm("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "l"(p));
}
__device__ __forceinline__ void ldrow(const double *p, double (&v)[1]) {
    asm("ld.global.nc.f64 %0, [%1];" : "=d"(v[0]) : "l"(p));
}
// streamed rows (t, the old y and v, the stores), evicted from L2 first
__device__ __forceinline__ void ldrow_rw(const float *p, float (&v)[4], uint64_t pol) {  // coherent: may alias y
    asm volatile("ld.global.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                 : "l"(p), "l"(pol)
                 : "memory");
}
__device__ __forceinline__ void ldrow_rw(const double *p, double (&v)[1], uint64_t pol) {
    asm volatile("ld.global.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v[0]) : "l"(p), "l"(pol) : "memory");
}
__device__ __forceinline__ void strow(float *p, const float (&v)[4], uint64_t pol) {
    asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1, %2, %3, %4}, %5;" ::"l"(p), "f"(v[0]), "f"(v[1]),
                 "f"(v[2]), "f"(v[3]), "l"(pol)
                 : "memory");
}
__device__ __forceinline__ void strow(double *p, const double (&v)[1], uint64_t pol) {
    asm volatile("st.global.L2::cache_hint.f64 [%0], %1, %2;" ::"l"(p), "d"(v[0]), "l"(pol) : "memory");
}

template <typename T>
__global__ void k_tile_diag(const DTerm *terms, int nt, int64_t D, T *d) {
    for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < D; s += (int64_t)gridDim.x * blockDim.x) {
        double v = 0.0;
        for (int k = 0; k < nt; k++) {
            const DTerm &t = terms[k];
            if (t.kind != DT_SPIN) continue;
            v += (((s >> t.i) ^ (s >> t.j)) & 1) ? -0.25 * t.a : 0.25 * t.a;
        }
        d[s] = (T)v;
    }
}

__device__ __forceinline__ void tile_fma(float c, const float (&v)[4], float (&acc)[4]) {
    fma2(acc[0], acc[1], c, v[0], v[1]);
    fma2(acc[2], acc[3], c, v[2], v[3]);
}
__device__ __forceinline__ void tile_fma(double c, const double (&v)[1], double (&acc)[1]) {
    acc[0] = fma(c, v[0], acc[0]);
}

// One bond on the rows of MASK only (FP64; no instruction for the other rows).
template <uint32_t MASK>
__device__ __forceinline__ void tile_some(const double *p, const int64_t (&roff)[8], double c, double (&acc)[8][1]) {
    double v[8][1];
#pragma unroll
    for (int j = 0; j < 8; j++)
        if ((MASK >> j) & 1u) ldrow(p + roff[j], v[j]);
#pragma unroll
    for (int j = 0; j < 8; j++)
        if ((MASK >> j) & 1u) tile_fma(c, v[j], acc[j]);
}

// One pass.  PASS 1 writes t; PASS 2 reads t and applies the epilogue.
template <typename T, int PASS, int RED>
__global__ void __launch_bounds__(kTileThreads, kTileMin)
    k_tile(const __grid_constant__ HvArgs<T> a, const __grid_constant__ TileArgs ta, const T *__restrict__ diag,
           T *tbuf) {
    using S = TileShape<T>;
    constexpr int E = S::E, LPR = S::LPR, QB = S::QB, IB = S::IB, RB = S::RB, R = S::R;
    constexpr int UN = kTileUnroll<T>;
    constexpr int W = kTileThreads / 32, P = PASS - 1;
    constexpr int NR = RED == 2 ? 3 : (RED ? 1 : 0);
    __shared__ uint32_t pin[4][256], pout[4][256];
    extern __shared__ __align__(16) unsigned char s_raw[];  // per warp the list of hits; the entries
    const int ne = ta.ne[P];
    TileHit<T> *hit = (TileHit<T> *)s_raw + (threadIdx.x >> 5) * ne;
    TileEnt *ents = (TileEnt *)((TileHit<T> *)s_raw + W * ne);
    // reductions of a thread (they would not fit in registers next to the sums)
    __shared__ RedAcc<T> racc[NR > 0 ? NR * E : 1][NR > 0 ? kTileThreads : 1];
    const uint32_t *tab = ta.tab + (size_t)P * 8 * 256;
    for (int i = threadIdx.x; i < 4 * 256; i += kTileThreads) {
        pin[i >> 8][i & 255] = tab[i];
        pout[i >> 8][i & 255] = tab[4 * 256 + i];
    }
    for (int i = threadIdx.x; i < ne; i += kTileThreads) ents[i] = ta.ent[P][i];
    if constexpr (NR > 0)
        for (int r = 0; r < NR * E; r++) racc[r][threadIdx.x] = RedAcc<T>();
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int gl = lane % LPR, rsub = lane / LPR;
    const int nin = ta.nin[P], nfull = ta.nfull[P];
    const int64_t per_tile = (int64_t)1 << (nin - IB);
    const int64_t items = per_tile << ta.nout[P];
    const T *__restrict__ X = a.x;
    // row offsets of the item's rows: lane group, register rows; lane l also holds row
    // l of the item (group l mod 2^QB, register row l >> QB) for the diagonal
    int drow = 0;
#pragma unroll
    for (int b = 0; b < IB; b++) drow += ((lane >> b) & 1) ? ta.site[P][b] : 0;
    int64_t roff[R];
#pragma unroll
    for (int j = 0; j < R; j++) {
        int r = 0;
#pragma unroll
        for (int b = 0; b < QB; b++) r += ((rsub >> b) & 1) ? ta.site[P][b] : 0;
#pragma unroll
        for (int b = 0; b < RB; b++) r += ((j >> b) & 1) ? ta.site[P][QB + b] : 0;
        roff[j] = (int64_t)r * 32 + E * gl;
    }
    const bool use_beta = a.beta != 0.0, use_v = a.v != nullptr;
    const uint32_t lt = (1u << lane) - 1u;
    const uint64_t stream = spol(1, 1);
    // Items in a fixed stride drift apart (SMs differ in speed by some percent, several
    // tiles over a pass), and tiles that are no longer worked on together leave L2 early:
    // N = 24 pass 1 read x 2.8 times.  Without reductions the warps draw pairs of items by
    // ticket instead (the next ticket when a pair is begun) and x is read 1.2 times.  With
    // reductions the stride stays fixed, so that their order does, and the blocks pace one
    // another: every half tile a block reports, and waits (a bounded number of short polls;
    // a hint that nothing depends on) while the average is more than kTileSlack reports
    // behind it.
    constexpr int G = 2;
    const bool dyn = RED == 0 && ta.ticket[P] != nullptr;
    const int64_t stride = (int64_t)gridDim.x * W, iters = (items + stride - 1) / stride;
    const int period = per_tile / 2 > stride ? (int)(per_tile / 2 / stride) : 1;
    auto draw = [&]() -> int64_t {
        unsigned n = 0;
        if (lane == 0) n = atomicAdd(ta.ticket[P], 1u);
        return (int64_t)n * G;
    };
    int64_t w = 0, next = 0;
    int left = 0;
    if (dyn) next = draw();
#pragma unroll 1
    for (int64_t it = 0;; it++) {
        if (dyn) {
            if (left == 0) {
                w = __shfl_sync(0xffffffffu, next, 0);
                left = G;
                if (w < items) next = draw();
            } else {
                w++;
            }
            left--;
            if (w >= items) break;
        } else {
            if (it >= iters) break;
            if (RED != 0 && ta.ticket[P] != nullptr && it > 0 && it % period == 0) {
                __syncthreads();
                if (threadIdx.x == 0) {
                    atomicAdd(ta.ticket[P], 1u);
                    const int64_t need = (it / period - kTileSlack) * (int64_t)gridDim.x;
                    for (int i = 0; i < kTileWaits && need > 0; i++) {
                        unsigned n;
                        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(n) : "l"(ta.ticket[P]) : "memory");
                        if ((int64_t)n >= need) break;
                        __nanosleep(500);
                    }
                }
                __syncthreads();
            }
            w = (int64_t)blockIdx.x * W + warp + it * stride;
            if (w >= items) continue;
        }
        const uint32_t t = (uint32_t)(w >> (nin - IB));
        const uint32_t inner = (uint32_t)(w & (per_tile - 1)) << IB;
        const uint32_t s = pin[0][inner & 255] | pin[1][(inner >> 8) & 255] | pin[2][(inner >> 16) & 255] |
                           pin[3][inner >> 24] | pout[0][t & 255] | pout[1][(t >> 8) & 255] |
                           pout[2][(t >> 16) & 255] | pout[3][t >> 24];
        // the item's bonds: those that touch whole items first
        int nf = 0, nh = 0;
        __syncwarp();  // the previous item is done with the list
#pragma unroll 1
        for (int k0 = 0; k0 < ne; k0 += 32) {
            const int k = k0 + lane;
            bool app = false;
            TileHit<T> h;
            if (k < ne) {
                const TileEnt b = ents[k];
                const uint32_t m = s & b.mo;
                app = k >= nfull || (m != 0 && m != b.mo);
                h.row = (int)(s ^ b.mo) + (m ? b.d0 : b.d1);
                h.mask = m ? b.mask & 0xFFu : b.mask >> 8;
                h.c = (T)b.c;
            }
            const unsigned bal = __ballot_sync(0xffffffffu, app);
            if (app) hit[nh + __popc(bal & lt)] = h;
            nh += __popc(bal);
            const int left = nfull - k0;
            nf += __popc(bal & (left >= 32 ? 0xffffffffu : left > 0 ? (1u << left) - 1u : 0u));
        }
        __syncwarp();
        const int64_t base = (int64_t)s * 32;
        T acc[R][E];
        if constexpr (PASS == 1) {
            const T dv = lane < (1 << IB) ? __ldg(diag + (int64_t)s + drow) : (T)0;
#pragma unroll
            for (int j = 0; j < R; j++) ldrow(X + base + roff[j], acc[j]);
#pragma unroll
            for (int j = 0; j < R; j++) {
                const T dj = __shfl_sync(0xffffffffu, dv, (j << QB) | rsub);
#pragma unroll
                for (int e = 0; e < E; e++) acc[j][e] *= dj;
            }
        } else {
#pragma unroll
            for (int j = 0; j < R; j++) ldrow_rw(tbuf + base + roff[j], acc[j], stream);
        }
        int k = 0;
#pragma unroll 1
        for (; k + UN <= nf; k += UN) {
            T v[UN][R][E], c[UN];
#pragma unroll
            for (int u = 0; u < UN; u++) {
                const TileHit<T> h = hit[k + u];
                c[u] = h.c;
                const T *p = X + (int64_t)h.row * 32;
#pragma unroll
                for (int j = 0; j < R; j++) ldrow(p + roff[j], v[u][j]);
            }
#pragma unroll
            for (int u = 0; u < UN; u++)
#pragma unroll
                for (int j = 0; j < R; j++) tile_fma(c[u], v[u][j], acc[j]);
        }
        // the rest: whole items left over and bonds with a site inside the item
        if constexpr (sizeof(T) == 8) {
#pragma unroll 1
            for (; k < nh; k++) {
                const TileHit<T> h = hit[k];
                const T *p = X + (int64_t)h.row * 32;
                switch (h.mask & 0xFFu) {  // by the values of one item bit, or of two that differ
                case 0x55u: tile_some<0x55u>(p, roff, h.c, acc); break;
                case 0xAAu: tile_some<0xAAu>(p, roff, h.c, acc); break;
                case 0x33u: tile_some<0x33u>(p, roff, h.c, acc); break;
                case 0xCCu: tile_some<0xCCu>(p, roff, h.c, acc); break;
                case 0x0Fu: tile_some<0x0Fu>(p, roff, h.c, acc); break;
                case 0xF0u: tile_some<0xF0u>(p, roff, h.c, acc); break;
                case 0x22u: tile_some<0x22u>(p, roff, h.c, acc); break;
                case 0x44u: tile_some<0x44u>(p, roff, h.c, acc); break;
                case 0x0Au: tile_some<0x0Au>(p, roff, h.c, acc); break;
                case 0x50u: tile_some<0x50u>(p, roff, h.c, acc); break;
                case 0x0Cu: tile_some<0x0Cu>(p, roff, h.c, acc); break;
                case 0x30u: tile_some<0x30u>(p, roff, h.c, acc); break;
                default: tile_some<0xFFu>(p, roff, h.c, acc); break;
                }
            }
        } else {
            // what is not loaded is 0
#pragma unroll 1
            for (; k < nh; k += UN) {
                T v[UN][R][E], c[UN];
                uint32_t rows[UN];
#pragma unroll
                for (int u = 0; u < UN; u++) {
                    const TileHit<T> h = hit[k + u < nh ? k + u : k];
                    c[u] = h.c;
                    rows[u] = k + u < nh ? h.mask & 0xFu : 0u;
                    const bool mine = (h.mask >> (4 + rsub)) & 1u;
                    const T *p = X + (int64_t)h.row * 32;
#pragma unroll
                    for (int j = 0; j < R; j++) {
#pragma unroll
                        for (int e = 0; e < E; e++) v[u][j][e] = (T)0;
                        if (mine && ((rows[u] >> j) & 1u)) ldrow(p + roff[j], v[u][j]);
                    }
                }
#pragma unroll
                for (int u = 0; u < UN; u++)
#pragma unroll
                    for (int j = 0; j < R; j++)
                        tile_fma(c[u], v[u][j], acc[j]);
            }
        }
        if constexpr (PASS == 1) {
#pragma unroll
            for (int j = 0; j < R; j++) strow(tbuf + base + roff[j], acc[j], stream);
        } else {
            if constexpr (RED == 2) {
                RedAcc<T> r[3][E];
#pragma unroll
                for (int i = 0; i < 3 * E; i++) r[i / E][i % E] = racc[i][threadIdx.x];
#pragma unroll
                for (int j = 0; j < R; j++) {
                    T xo[E];
                    ldrow(X + base + roff[j], xo);
#pragma unroll
                    for (int e = 0; e < E; e++) {
                        r[0][e].add(xo[e], acc[j][e]);
                        r[1][e].add(acc[j][e], acc[j][e]);
                        r[2][e].add(xo[e], xo[e]);
                    }
                }
#pragma unroll
                for (int i = 0; i < 3 * E; i++) racc[i][threadIdx.x] = r[i / E][i % E];
            }
            T al[E], ga[E];
#pragma unroll
            for (int e = 0; e < E; e++) {
                al[e] = (T)(a.alpha_dev ? a.alpha_dev[E * gl + e] : a.alpha[E * gl + e]);
                ga[e] = (T)(a.gamma_dev ? a.gamma_dev[E * gl + e] : a.gamma[E * gl + e]);
            }
            T out[R][E];
#pragma unroll
            for (int j = 0; j < R; j++)
#pragma unroll
                for (int e = 0; e < E; e++) {
                    T hx = acc[j][e];
                    if (a.swap) {  // the partner column: in this lane, or in the next
                        if constexpr (E == 1) hx = __shfl_xor_sync(0xffffffffu, hx, 1);
                        else hx = acc[j][e ^ 1];
                    }
                    out[j][e] = al[e] * hx;
                }
            if (use_beta) {
                const T be = (T)a.beta;
                T o[R][E];
#pragma unroll
                for (int j = 0; j < R; j++) ldrow_rw(a.y + base + roff[j], o[j], stream);
#pragma unroll
                for (int j = 0; j < R; j++)
#pragma unroll
                    for (int e = 0; e < E; e++) out[j][e] = fma(be, o[j][e], out[j][e]);
            }
            if (use_v) {
                T o[R][E];
#pragma unroll
                for (int j = 0; j < R; j++) ldrow_rw(a.v + base + roff[j], o[j], stream);
#pragma unroll
                for (int j = 0; j < R; j++)
#pragma unroll
                    for (int e = 0; e < E; e++) out[j][e] = fma(ga[e], o[j][e], out[j][e]);
            }
#pragma unroll
            for (int j = 0; j < R; j++) strow(a.y + base + roff[j], out[j], stream);
            if constexpr (RED == 1 || RED == 3) {
                RedAcc<T> r[E];
#pragma unroll
                for (int e = 0; e < E; e++) r[e] = racc[e][threadIdx.x];
#pragma unroll
                for (int j = 0; j < R; j++) {
                    T xo[E];
                    if constexpr (RED == 1) ldrow(X + base + roff[j], xo);
#pragma unroll
                    for (int e = 0; e < E; e++) r[e].add(RED == 1 ? xo[e] : out[j][e], out[j][e]);
                }
#pragma unroll
                for (int e = 0; e < E; e++) racc[e][threadIdx.x] = r[e];
            }
        }
    }
    if constexpr (PASS == 2 && RED != 0) {
        // lanes gl, gl + LPR, ... hold the same columns
        __shared__ double red_sm[W][3][32];
#pragma unroll
        for (int r = 0; r < NR; r++)
#pragma unroll
            for (int e = 0; e < E; e++) {
                double v = racc[r * E + e][threadIdx.x].value();
#pragma unroll
                for (int off = LPR; off < 32; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
                if (rsub == 0) red_sm[warp][r][E * gl + e] = v;
            }
        __syncthreads();
        for (int i = threadIdx.x; i < 3 * 32; i += kTileThreads) {
            const int r = i / 32, c = i % 32;
            double sum = 0.0;
            if (r < NR)
                for (int w2 = 0; w2 < W; w2++) sum += red_sm[w2][r][c];
            a.partials[((int64_t)blockIdx.x * 3 + r) * a.ncol + c] = sum;
        }
    }
}

uint32_t pdep32(uint32_t v, uint32_t mask) {
    uint32_t out = 0;
    for (int b = 0; b < 32 && v; b++)
        if ((mask >> b) & 1u) {
            if (v & 1u) out |= 1u << b;
            v >>= 1;
        }
    return out;
}

struct TileBond {
    int i, j;
    double c;
};

// The sites of S: first a cluster of `size` of them (or all) grown greedily by the
// site with the most bonds into it, from the start that ends with the most inner
// bonds; then the others, ascending.
std::vector<int> site_order(int N, uint64_t S, const std::vector<TileBond> &bonds, int size) {
    std::vector<int> best;
    int best_in = -1;
    for (int st = 0; st < N; st++) {
        if (!((S >> st) & 1)) continue;
        std::vector<int> c{st};
        uint64_t in = 1ull << st;
        int inner = 0;
        while ((int)c.size() < size && in != S) {
            int pick = -1, most = -1;
            for (int v = 0; v < N; v++) {
                if (!((S >> v) & 1) || ((in >> v) & 1)) continue;
                int n = 0;
                for (const TileBond &b : bonds)
                    n += (b.i == v && ((in >> b.j) & 1)) || (b.j == v && ((in >> b.i) & 1));
                if (n > most) {
                    most = n;
                    pick = v;
                }
            }
            c.push_back(pick);
            in |= 1ull << pick;
            inner += most;
        }
        if (inner > best_in) {
            best_in = inner;
            best = c;
        }
    }
    uint64_t in = 0;
    for (int v : best) in |= 1ull << v;
    for (int v = 0; v < N; v++)
        if (((S & ~in) >> v) & 1) best.push_back(v);
    return best;
}

// Two disjoint site sets A, B with no off-diagonal bond between them and
// N - |A|, N - |B| <= smax: A grown greedily from each start site by the
// neighbour that adds the fewest new neighbours, B taken from the sites
// neither in A nor next to it.  Returns false when no start site gives both
// sizes.
bool find_cover(int N, const std::vector<uint64_t> &adj, int smax, uint64_t *A_out, uint64_t *B_out) {
    const int need = N - smax;
    if (need <= 0) {
        *A_out = 0;
        *B_out = 0;
        return true;
    }
    const uint64_t all = N == 64 ? ~0ull : ((1ull << N) - 1);
    auto nbr = [&](uint64_t A) {
        uint64_t n = 0;
        for (int v = 0; v < N; v++)
            if ((A >> v) & 1) n |= adj[v];
        return n & ~A;
    };
    for (int st = 0; st < N; st++) {
        uint64_t A = 1ull << st;
        while (true) {
            const uint64_t R = all & ~(A | nbr(A));
            if (__builtin_popcountll(A) >= need && __builtin_popcountll(R) >= need) {
                // B: `need` sites of R (the fewest that bring pass 2 within smax;
                // the sites left out keep their bonds free for either pass)
                uint64_t B = 0;
                for (int v = 0; v < N && __builtin_popcountll(B) < need; v++)
                    if ((R >> v) & 1) B |= 1ull << v;
                *A_out = A;
                *B_out = B;
                return true;
            }
            if (__builtin_popcountll(A) >= need) break;
            const uint64_t cand = nbr(A) ? nbr(A) : (all & ~A);
            int best = -1, bc = 1 << 30;
            for (int v = 0; v < N; v++) {
                if (!((cand >> v) & 1)) continue;
                const int c = __builtin_popcountll(nbr(A | (1ull << v)));
                if (c < bc) {
                    bc = c;
                    best = v;
                }
            }
            if (best < 0) break;
            A |= 1ull << best;
        }
    }
    return false;
}

template <typename T>
size_t tile_smem(const TileArgs &ta, int p) {
    return (size_t)ta.ne[p] * (kTileThreads / 32 * sizeof(TileHit<T>) + sizeof(TileEnt)) + 16;
}

template <typename T, int PASS>
int go_tile(hphi_ctx *ctx, const HvArgs<T> &a, const TileArgs &ta, const T *diag, T *tbuf, int red_mode, int grid) {
#define HPHI_TILE(R) \
    k_tile<T, PASS, R><<<grid, kTileThreads, tile_smem<T>(ta, PASS - 1), ctx->stream>>>(a, ta, diag, tbuf)
    if constexpr (PASS == 1) {
        HPHI_TILE(0);
    } else {
        switch (red_mode) {
        case 0: HPHI_TILE(0); break;
        case 1: HPHI_TILE(1); break;
        case 2: HPHI_TILE(2); break;
        case 3: HPHI_TILE(3); break;
        default: return HPHI_E_INVAL;
        }
    }
#undef HPHI_TILE
    HPHI_CUDA(ctx, cudaGetLastError());
    return HPHI_OK;
}

}  // namespace

// Bit sets, bond split and tables of the tiled kernel for a full-space spin
// Hamiltonian (built on the first launch that asks for it).  Leaves
// ham->tile[prec] null when the model is not eligible or no split fits L2.
// prec 0: FP32 rows (128 bytes), 1: FP64 rows (256 bytes).
int build_tile_tables(hphi_ctx *ctx, hphi_ham *H, int prec) {
    if (prec < 0 || prec > 1) return set_err(ctx, HPHI_E_INVAL, "tiled kernel tables: unknown precision");
    if (H->tile[prec] || H->tile_tried[prec]) return HPHI_OK;
    H->tile_tried[prec] = 1;
    const double row_bytes = prec ? 256.0 : 128.0;
    const size_t es = prec ? sizeof(double) : sizeof(float);
    if (H->model != HPHI_SPIN_HALF_GC) return HPHI_OK;
    const int N = H->basis->N;
    if (N < kTileItemBits || N > 31) return HPHI_OK;
    std::vector<uint64_t> adj(N, 0);
    std::vector<TileBond> bonds;
    for (const DTerm &t : H->dterms) {
        if (t.kind != DT_SPIN || t.b == 0.0) continue;
        if (!(fabs(t.b) < 1e30)) return HPHI_OK;  // FP32 rows that a bond does not touch add Jxy/2 times 0
        adj[t.i] |= 1ull << t.j;
        adj[t.j] |= 1ull << t.i;
        bonds.push_back(TileBond{t.i, t.j, 0.5 * t.b});
    }
    int l2 = 0;
    if (cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, ctx->device) != cudaSuccess || l2 <= 0) {
        cudaGetLastError();
        return HPHI_OK;
    }
    // a tile of 2^s rows within 30 % of L2
    int smax = kTileItemBits;
    while (smax < N && (row_bytes * (double)(2ull << smax)) <= 0.3 * (double)l2) smax++;
    uint64_t A = 0, B = 0;
    if (!find_cover(N, adj, smax, &A, &B)) return HPHI_OK;
    const uint64_t all = (N == 64) ? ~0ull : ((1ull << N) - 1);
    TileArgs ta{};
    const uint64_t S[2] = {all & ~A, all & ~B};
    std::vector<TileBond> part[2];
    for (const TileBond &b : bonds) {
        const uint64_t m = (1ull << b.i) | (1ull << b.j);
        const bool in1 = (m & A) == 0, in2 = (m & B) == 0;
        if (in1 && in2) part[part[0].size() <= part[1].size() ? 0 : 1].push_back(b);
        else if (in1) part[0].push_back(b);
        else part[1].push_back(b);
    }
    std::vector<uint32_t> tab(2 * 8 * 256);
    std::vector<TileEnt> ents[2];
    for (int p = 0; p < 2; p++) {
        if ((int)part[p].size() > kTileMaxBonds) return HPHI_OK;
        ta.nin[p] = __builtin_popcountll(S[p]);
        ta.nout[p] = N - ta.nin[p];
        if (ta.nin[p] < kTileItemBits) return HPHI_OK;
        // order of the tile's sites in the item counter: a cluster of sites joined by as
        // many of the pass's bonds as possible first (their gathers stay among the rows
        // that a thread block works on, in L1), then the others ascending
        const std::vector<int> order = site_order(N, S[p], part[p], prec ? 0 : kTileCluster);
        // item bits: the first sites of that order (lane groups, then register rows)
        const int qb = prec ? TileShape<double>::QB : TileShape<float>::QB;
        const int rb = prec ? TileShape<double>::RB : TileShape<float>::RB;
        int where[32];  // item bit of a site, -1: none
        for (int v = 0; v < 32; v++) where[v] = -1;
        int nitem = 0;
        for (int v : order)
            if (nitem < qb + rb) {
                ta.site[p][nitem] = 1 << v;
                where[v] = nitem++;
            }
        // rows (low bits) and lane groups (bits 4-7, FP32) whose item bit b has the value val
        auto rows_with = [&](int b, int val) {
            uint32_t m = 0;
            for (int j = 0; j < (1 << rb); j++)
                if (b < qb || ((j >> (b - qb)) & 1) == val) m |= 1u << j;
            for (int g = 0; qb > 0 && g < (1 << qb); g++)
                if (b >= qb || ((g >> b) & 1) == val) m |= 1u << (4 + g);
            return m;
        };
        const uint32_t all_rows = 0xFFu;
        std::vector<TileEnt> full, rest;
        for (const TileBond &b : part[p]) {
            const int wi = where[b.i], wj = where[b.j];
            TileEnt e{};
            e.c = b.c;
            if (wi < 0 && wj < 0) {
                e.mo = (1u << b.i) | (1u << b.j);
                e.mask = all_rows | all_rows << 8;
                full.push_back(e);
            } else if (wi < 0 || wj < 0) {
                const int in = wi < 0 ? b.j : b.i, wb = wi < 0 ? wj : wi;
                e.mo = 1u << (wi < 0 ? b.i : b.j);
                e.d0 = 1 << in;     // outer site up: rows whose inner bit is down
                e.d1 = -(1 << in);  // outer site down: rows whose inner bit is up
                e.mask = rows_with(wb, 0) | rows_with(wb, 1) << 8;
                rest.push_back(e);
            } else {
                for (int v = 0; v < 2; v++) {  // i up, j down; then the other way round
                    e.d1 = (v ? 1 : -1) * (1 << b.i) + (v ? -1 : 1) * (1 << b.j);
                    e.mask = (rows_with(wi, 1 - v) & rows_with(wj, v)) << 8;
                    rest.push_back(e);
                }
            }
        }
        ta.nfull[p] = (int)full.size();
        full.insert(full.end(), rest.begin(), rest.end());
        ta.ne[p] = (int)full.size();
        ents[p] = full;
        const uint32_t out_mask = (uint32_t)(all & ~S[p]);
        for (int byte = 0; byte < 4; byte++)
            for (uint32_t v = 0; v < 256; v++) {
                uint32_t in = 0;
                for (int b = 0; b < 8; b++)
                    if (((v >> b) & 1u) && 8 * byte + b < (int)order.size()) in |= 1u << order[8 * byte + b];
                tab[(size_t)p * 2048 + byte * 256 + v] = in;
                tab[(size_t)p * 2048 + 1024 + byte * 256 + v] = pdep32(v << (8 * byte), out_mask);
            }
    }
    const int64_t D = H->D;
    // one device block: deposit tables, then the entries of both passes
    size_t at_ent[2];
    for (int p = 0; p < 2; p++) {
        at_ent[p] = tab.size();
        tab.resize(tab.size() + ents[p].size() * (sizeof(TileEnt) / sizeof(uint32_t)));
        if (!ents[p].empty()) memcpy(tab.data() + at_ent[p], ents[p].data(), ents[p].size() * sizeof(TileEnt));
    }
    cudaError_t e = cudaMalloc((void **)&H->tile_tab[prec], tab.size() * sizeof(uint32_t));
    if (e == cudaSuccess)
        e = cudaMemcpy(H->tile_tab[prec], tab.data(), tab.size() * sizeof(uint32_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMalloc(&H->tile_diag[prec], (size_t)D * es);
    if (e != cudaSuccess) {
        cudaFree(H->tile_tab[prec]);
        H->tile_tab[prec] = nullptr;
        return cuda_err(ctx, e, "tiled kernel tables");
    }
    const int gd = (int)std::min<int64_t>((D + 255) / 256, (int64_t)ctx->sm_count * 16);
    if (prec)
        k_tile_diag<double><<<gd, 256, 0, ctx->stream>>>(H->dterms_d, (int)H->dterms.size(), D,
                                                         (double *)H->tile_diag[prec]);
    else
        k_tile_diag<float><<<gd, 256, 0, ctx->stream>>>(H->dterms_d, (int)H->dterms.size(), D,
                                                        (float *)H->tile_diag[prec]);
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
    if (e != cudaSuccess) return cuda_err(ctx, e, "tiled kernel diagonal");
    ta.tab = H->tile_tab[prec];
    for (int p = 0; p < 2; p++) ta.ent[p] = (const TileEnt *)(H->tile_tab[prec] + at_ent[p]);
    H->tile[prec] = new (std::nothrow) TileArgs(ta);
    if (!H->tile[prec]) return set_err(ctx, HPHI_E_NOMEM, "tiled kernel tables");
    return HPHI_OK;
}

template <typename T>
int launch_tile(hphi_ctx *ctx, const hphi_ham *ham, HvArgs<T> &a, int red_mode, int *grid) {
    constexpr int prec = std::is_same<T, float>::value ? 0 : 1;
    if (!ham->tile[prec]) return set_err(ctx, HPHI_E_INVAL, "tiled H*V: not available for this Hamiltonian");
    const TileArgs &ta = *ham->tile[prec];
    const size_t need = (size_t)ham->D * 32 * sizeof(T);
    T *tbuf = nullptr;
    if (a.beta == 0.0 && (a.v == nullptr || a.v != a.y)) {
        tbuf = a.y;
    } else {
        if (ctx->seg_tmp_bytes < need) {
            HPHI_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
            cudaFree(ctx->seg_tmp);
            ctx->seg_tmp = nullptr;
            ctx->seg_tmp_bytes = 0;
            cudaError_t e = cudaMalloc(&ctx->seg_tmp, need);
            if (e != cudaSuccess) return cuda_err(ctx, e, "tiled H*V buffer");
            ctx->seg_tmp_bytes = need;
        }
        tbuf = (T *)ctx->seg_tmp;
    }
    if (red_mode < 0 || red_mode > 3) return set_err(ctx, HPHI_E_INVAL, "tiled H*V: unknown reduction mode");
    static const void *const pass2[4] = {(const void *)k_tile<T, 2, 0>, (const void *)k_tile<T, 2, 1>,
                                         (const void *)k_tile<T, 2, 2>, (const void *)k_tile<T, 2, 3>};
    // no more thread blocks than the partials of an H*x launch hold (8 per SM)
    auto grid_of = [&](const void *f, int p) {
        int occ = dyn_occupancy(ctx, f, kTileThreads, tile_smem<T>(ta, p));
        if (occ < 1) return 0;
        occ = occ < 8 ? occ : 8;
        int64_t g = (int64_t)occ * ctx->sm_count;
        if (g > ham->nh) g = ham->nh;
        return (int)(g < 1 ? 1 : g);
    };
    const int g1 = grid_of((const void *)k_tile<T, 1, 0>, 0), g2 = grid_of(pass2[red_mode], 1);
    if (!g1 || !g2) return set_err(ctx, HPHI_E_INVAL, "tiled H*V: the bond lists do not fit in shared memory");
    *grid = g2;
    const T *diag = (const T *)ham->tile_diag[prec];
    TileArgs tp = ta;
    if (ta.nout[0] >= 2 || ta.nout[1] >= 2) {
        HPHI_CUDA(ctx, cudaMemsetAsync(ctx->ticket, 0, 2 * sizeof(unsigned), ctx->stream));
        for (int p = 0; p < 2; p++) tp.ticket[p] = ta.nout[p] >= 2 ? ctx->ticket + p : nullptr;
    }
    const int slot = prof_begin(ctx, PROF_HV);
    int st = go_tile<T, 1>(ctx, a, tp, diag, tbuf, 0, g1);
    if (!st) st = go_tile<T, 2>(ctx, a, tp, diag, tbuf, red_mode, g2);
    prof_end(ctx, slot);
    if (st) return st;
    snprintf(ctx->last_kernel, sizeof ctx->last_kernel, "k_tile<%s,RED%d>x2@" HPHI_SRC_TAG, tname<T>(), red_mode);
    return HPHI_OK;
}

template int launch_tile<float>(hphi_ctx *, const hphi_ham *, HvArgs<float> &, int, int *);
template int launch_tile<double>(hphi_ctx *, const hphi_ham *, HvArgs<double> &, int, int *);

}  // namespace hphi
