// Segment H*x kernel for the spin-1/2 S^z sector, one column.
//
// Cut the spin string at bit s: u = the upper N - s bits, l0 = the lowest s
// bits (10, or the low half's where that is shorter).  The rows that share u
// form a segment: consecutive rows, the C(s, c) strings l0 of popcount c = n -
// |u| in ascending order.  One warp owns a segment, lane t its rows t, t + 32,
// ... (at most 8, in registers), so everything that depends on u alone is done
// once per segment, one bond per lane:
//   - a bond with both sites in u ("uniform") applies to the whole segment or
//     to none of it, and its target is the same rows of segment u ^ m: the
//     applicable ones are listed as (row offset, coefficient) and each is one
//     coalesced load and one FMA per row;
//   - a bond with one site b in l0 ("mixed") applies to the rows whose bit b
//     equals 1 - u_a; its target is row rank(l0 ^ 2^b) of segment u ^ 2^a;
//   - a bond inside l0 ("inner") keeps the segment; its target is rank(l0 ^ m),
//     read from a copy of the segment in shared memory.
// The last two take the ranks from byte tables in shared memory, one table per
// (bit b, needed value) or bond, 255 marking rows that the bond does not touch;
// the bytes of a lane's rows lie next to each other, so a lane reads all of them
// with one load.  No row tests a uniform bond, none walks a list, and nothing is
// accumulated through shared memory.
//
// The diagonal is summed in fixed point (integers, scaled by a power of two so
// that it stays below 2^30, in 64 bits 2^62; partial sums may wrap): the part of
// u by one warp reduction, the mixed part from two 32-entry tables kept one
// entry per lane (l0's low and high five bits), the part of l0 from a table.  That
// costs no FP64 adds.  A grid step is 2^-32 (2^-64) of a power of two above the sum
// of all |Jz|, more than a weak coupling can do without where strong ones cancel:
// build_warp_tables chooses the integers, or leaves the kernel out.
//
// Thread blocks take row blocks h (the high half of the spin string) in the
// traversal order of set_traversal, the warps of a block its segments, so that
// the in-block targets stay in L1.  A row sums its terms in a fixed order and
// the work split is static: deterministic.  (Sec. 3.1.1: the exchange terms on
// the bit-encoded basis.)
//
// What bounds it: FP32 the latency of the gathers (6x5 lattice: 12.8 warp
// instructions per row, 57 % of the issue slots, DRAM 2.6 TB/s), FP64 the FP64
// pipe (94 % busy).  Measured against the bond-major kernel (hv_phased.cu, 25
// warp instructions per row), ms per product: 4x8 FP32 24.6 -> 14.2, 6x5 FP32
// 6.02 -> 2.75, 14-rung ladder FP32 1.58 -> 0.49, FP64 3.92 -> 2.91, 24-site
// chain FP64 0.39 -> 0.125, 16-site chain FP64 0.025 -> 0.010.  Splits tried: 9
// segment bits 6x5 3.66, 8 bits 5.68 (lanes idle in short segments); 8 uniform
// loads in flight per lane 3.27, 16: 2.87, 24: 2.79; 16 mixed loads 3.32; two
// batches in flight at a time 5.9 (spills at 64 registers); 16 warps per SM 3.4.
#include "fixed.cuh"
#include "hvcommon.cuh"

#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <vector>

namespace hphi {

namespace {

constexpr int kLoadsU = 24, kLoadsM = 8;  // loads per lane in flight: uniform bonds, mixed bonds
// threads per block: one block per SM, registers for 32 (FP64: 16) warps
template <typename T> constexpr int kSegThreads = sizeof(T) == 4 ? 1024 : 512;
constexpr int kSegStage = 256;  // staged values per warp (a slot behind every segment stays 0)
constexpr int kSegBits = 62;  // the diagonal lies below 2^62 grid steps
constexpr int kSegRows = 8;   // rows of a lane held in registers (C(10, 5) = 252 rows per segment)

// FP64 couplings are stored over the diagonal's scale (a power of two, so exact) and H x
// is scaled with alpha in one multiplication: the FP64 pipe is the bound.  FP32 ones are
// not: the scaled sums of vectors above 1e19 would overflow.  There alpha goes into the
// couplings and the diagonal's scale (RED 2 needs H x itself): a multiplication per row
// costs 20 Lanczos steps of the 6x5 lattice 3 %, and their alphas are no closer to 64
// bits with it (6x4 lattice, 8 start vectors: 1.36e-7 with, 1.33e-7 without).
template <typename T> constexpr bool seg_scaled = sizeof(T) == 8;
template <typename T, int RED> constexpr bool seg_fold = !seg_scaled<T> && RED != 2;

// A bond of the image, in T's precision.
struct WarpBond {     // a bond as the builder collects it
    double cxy;       // Jxy/2
    long long cz;     // -Jz/2 in fixed point
    uint32_t mask;    // its sites above the segment bits
    uint32_t tab;     // rank table (mixed: of needed value 0; the next one of 1)
};
template <typename T, typename I>
struct SmemBond {
    T cxy;
    I cz;
    uint32_t mask, tab;
};

// One entry of a warp's bond list: row offset of the target, coefficient, and
// for mixed / inner bonds the byte offset of the rank table.
template <typename T>
struct SegEnt;
template <>
struct __align__(16) SegEnt<float> {
    int delta;
    int tab;
    float c;
    int pad;
};
template <>
struct __align__(16) SegEnt<double> {
    double c;
    int delta;
    int tab;
};

__device__ __forceinline__ int seg_isum(int v) { return __reduce_add_sync(0xffffffffu, v); }
__device__ __forceinline__ long long seg_isum(long long v) {
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// The NC table bytes of one lane (padded to 1, 2, 4 or 8).
template <int NC>
__device__ __forceinline__ void load_ranks(const unsigned char *tab, int lane, uint32_t (&w)[2]) {
    if constexpr (NC > 4) {
        const uint2 v = *reinterpret_cast<const uint2 *>(tab + lane * 8);
        w[0] = v.x;
        w[1] = v.y;
    } else if constexpr (NC > 2) {
        w[0] = *reinterpret_cast<const uint32_t *>(tab + lane * 4);
    } else if constexpr (NC == 2) {
        w[0] = *reinterpret_cast<const uint16_t *>(tab + lane * 2);
    } else {
        w[0] = tab[lane];
    }
}
template <typename T>
__device__ __forceinline__ T lds(uint32_t a) {
    T v;
    if constexpr (sizeof(T) == 4) asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    else asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}

// acc += c v, two rows per instruction in FP32 (each rounded as a single fma)
template <int NC>
__device__ __forceinline__ void fma_rows(float c, const float (&v)[NC], float (&acc)[NC]) {
#pragma unroll
    for (int i = 0; i + 1 < NC; i += 2)
        fma2(acc[i], acc[i + 1], c, v[i], v[i + 1]);
    if constexpr (NC % 2) acc[NC - 1] = fma(c, v[NC - 1], acc[NC - 1]);
}
template <int NC>
__device__ __forceinline__ void fma_rows(double c, const double (&v)[NC], double (&acc)[NC]) {
#pragma unroll
    for (int i = 0; i < NC; i++) acc[i] = fma(c, v[i], acc[i]);
}

// Byte offsets of the Hamiltonian's tables in their image: the segment strings'
// diagonal, the segment strings, Lin offsets of the segments, jb in two parts,
// the bonds (uniform, mixed, mixed diagonal, inner), the rank tables (mixed,
// inner).  Every part is a multiple of 16 bytes.
template <typename T, typename I>
struct WarpLayout {
    uint32_t l0s, so, jp, bonds, tabs, bytes;
    __host__ __device__ explicit WarpLayout(const WarpArgs &g) {
        uint32_t o = (uint32_t)sizeof(I) * g.nrow;
        auto part = [&](uint32_t n) {
            const uint32_t at = o;
            o += (n + 15u) & ~15u;
            return at;
        };
        l0s = part(2u * g.nrow);
        so = part(2u * (uint32_t)((g.nlo + 1) << g.n1));
        jp = part(4u * (uint32_t)(g.jhi + ((g.jw + 1) << g.jl)));
        bonds = part((uint32_t)sizeof(SmemBond<T, I>) * (g.nu + g.nx + g.nm + g.ni));
        tabs = part((uint32_t)g.tab_stride * (g.ntab + g.ni));
        bytes = o;
    }
};

__device__ __forceinline__ double seg_diag(long long d, double) { return (double)d; }
template <typename I>
__device__ __forceinline__ float seg_diag(I d, float scale) { return (float)d * scale; }

// What a warp needs to know of its segment.
template <typename T, typename I>
struct Seg {
    const SegEnt<T> *list;        // mixed bonds, then the applicable uniform ones
    int nml, nall;
    const SmemBond<T, I> *ib;        // inner bonds
    int nib;
    const unsigned char *tabs;    // rank tables of the mixed bonds, this class
    const unsigned char *itabs;   // rank tables of the inner bonds, this class
    int stride;                   // bytes of one table
    const I *dl0;
    const uint16_t *l0s;
    I du, tlo, thi;
    T *stage;                     // 256 values of the warp: x of the segment, zeros behind it
    uint32_t base, len;
};
template <typename T>
struct Epi {
    const T *al;  // in shared memory: one register less through the bonds
    T ga, be, dscale;
    bool use_beta, use_v;
    uint64_t keep, stream;
};

// Epilogue of NC rows row, row + 32, ... (the last one only if `tail`; xs: their
// x, 32 apart): the old y and v of all rows are loaded before the first store.
// acc is H x, in FP64 over the diagonal's scale, in FP32 times alpha unless RED is 2.
template <typename T, int NC, int RED>
__device__ __forceinline__ void seg_out(const HvArgs<T> &a, const Epi<T> &e, uint32_t row, bool tail, const T *xs,
                                        T (&acc)[NC], RedAcc<T> (&racc)[RED == 2 ? 3 : 1]) {
    if constexpr (RED == 2) {
#pragma unroll
        for (int c = 0; c < NC; c++) {
            if constexpr (seg_scaled<T>) acc[c] = e.dscale * acc[c];
            if (c + 1 < NC || tail) {
                const T xo = xs[32 * c];
                racc[0].add(xo, acc[c]);
                racc[1].add(acc[c], acc[c]);
                racc[2].add(xo, xo);
            }
        }
    }
    if constexpr (!seg_fold<T, RED>) {
        const T al = *e.al;
#pragma unroll
        for (int c = 0; c < NC; c++) acc[c] = al * acc[c];
    }
    if (e.use_beta) {
        T t[NC];
#pragma unroll
        for (int c = 0; c < NC; c++) {
            t[c] = (T)0;
            if (c + 1 < NC || tail) t[c] = cload<T>(a.y + row + 32 * c, e.stream);
        }
        fma_rows<NC>(e.be, t, acc);
    }
    if (e.use_v) {
        T t[NC];
#pragma unroll
        for (int c = 0; c < NC; c++) {
            t[c] = (T)0;
            if (c + 1 < NC || tail) t[c] = cload<T>(a.v + row + 32 * c, e.stream);
        }
        fma_rows<NC>(e.ga, t, acc);
    }
#pragma unroll
    for (int c = 0; c < NC; c++)
        if (c + 1 < NC || tail) {
            cstore<T>(a.y + row + 32 * c, e.stream, acc[c]);
            if constexpr (RED == 1) racc[0].add(xs[32 * c], acc[c]);
            if constexpr (RED == 3) racc[0].add(acc[c], acc[c]);
        }
}

// The rows of one segment, NC = ceil(len / 32) per lane.  Loads of whole rows of
// 32 run past the segment's end into the rows behind it (whose sums are not
// stored): the caller has checked that they stay inside x.
template <typename T, typename I, int NC, int RED>
__device__ __forceinline__ void seg_rows(const HvArgs<T> &a, const Seg<T, I> &g, const Epi<T> &e, int lane,
                                         RedAcc<T> (&racc)[RED == 2 ? 3 : 1]) {
    constexpr int UB = kLoadsU / NC, UM = kLoadsM / NC;  // uniform and mixed bonds in flight
    const T *__restrict__ xs = a.x + g.base;
    const T *__restrict__ xl = xs + lane;
    T acc[NC];
    {
        T xo[NC];
#pragma unroll
        for (int c = 0; c < NC; c++) xo[c] = gload<T>(xl + 32 * c, e.keep);
        if (lane + 32 * (NC - 1) >= g.len) xo[NC - 1] = (T)0;
#pragma unroll
        for (int c = 0; c < NC; c++) {
            g.stage[lane + 32 * c] = xo[c];
            const uint32_t l0 = g.l0s[lane + 32 * c];
            const I d = g.du + g.dl0[lane + 32 * c] + __shfl_sync(0xffffffffu, g.tlo, l0 & 31u) +
                        __shfl_sync(0xffffffffu, g.thi, l0 >> 5);
            acc[c] = seg_diag(d, e.dscale) * xo[c];
        }
    }
    __syncwarp();
    // inner bonds, from the staged segment (rows a bond does not touch read the zero
    // in slot 255)
    const uint32_t st = (uint32_t)__cvta_generic_to_shared(g.stage);
    auto inner = [&](int k) {
        uint32_t w[2];
        T v[NC];
        load_ranks<NC>(g.itabs + k * g.stride, lane, w);
        const T cf = g.ib[k].cxy;
#pragma unroll
        for (int c = 0; c < NC; c++)
            v[c] = lds<T>(__dp4a(w[c >> 2], (uint32_t)sizeof(T) << (8 * (c & 3)), st));
        fma_rows<NC>(cf, v, acc);
    };
    // mixed bonds.  A value that is not loaded is 0, so that every FMA runs
    // unpredicated and no register stays live from one segment to the next.
#pragma unroll 1
    for (int k = 0; k < g.nib; k++) inner(k);
    int k = 0;
#pragma unroll 1
    for (; k < g.nml; k += UM) {
        T v[UM][NC], cf[UM];
#pragma unroll
        for (int u = 0; u < UM; u++) {
            const bool on = UM == 1 || k + u < g.nml;
            const SegEnt<T> n = g.list[on ? k + u : k];
            const T *p = xs + n.delta;
            cf[u] = n.c;
            uint32_t w[2];
            load_ranks<NC>(g.tabs + n.tab, lane, w);
#pragma unroll
            for (int c = 0; c < NC; c++) {
                const uint32_t t = (w[c >> 2] >> (8 * (c & 3))) & 255u;
                v[u][c] = (T)0;
                if (on && t != 255u) v[u][c] = gload<T>(p + t, e.keep);
            }
        }
#pragma unroll
        for (int u = 0; u < UM; u++) fma_rows<NC>(cf[u], v[u], acc);
    }
    // uniform bonds
    const SegEnt<T> *ul = g.list + g.nml;
    const int nul = g.nall - g.nml;
#pragma unroll 1
    for (k = 0; k + UB <= nul; k += UB) {
        T v[UB][NC], cf[UB];
#pragma unroll
        for (int u = 0; u < UB; u++) {
            const SegEnt<T> n = ul[k + u];
            cf[u] = n.c;
#pragma unroll
            for (int c = 0; c < NC; c++) v[u][c] = gload<T>(xl + n.delta + 32 * c, e.keep);
        }
#pragma unroll
        for (int u = 0; u < UB; u++) fma_rows<NC>(cf[u], v[u], acc);
    }
#pragma unroll 1
    for (; UB > 1 && k < nul; k++) {
        T v[NC];
        const SegEnt<T> n = ul[k];
#pragma unroll
        for (int c = 0; c < NC; c++) v[c] = gload<T>(xl + n.delta + 32 * c, e.keep);
        fma_rows<NC>(n.c, v, acc);
    }
    seg_out<T, NC, RED>(a, e, g.base + lane, lane + 32 * (NC - 1) < g.len, g.stage + lane, acc, racc);
}

// The same for segments whose padded rows would reach past the end of x: 32
// rows at a time, every access predicated, inner bonds read from x.
template <typename T, typename I, int RED>
__device__ __noinline__ void seg_edge(const HvArgs<T> &a, const Seg<T, I> &g, const Epi<T> &e, int lane, int nc,
                                      RedAcc<T> (&racc)[RED == 2 ? 3 : 1]) {
    const T *__restrict__ xs = a.x + g.base;
    const int nb = nc > 4 ? 8 : nc > 2 ? 4 : nc;  // entries of a lane in the tables
    for (int c = 0; c < nc; c++) {
        const uint32_t r = lane + 32 * c;
        const bool in = r < g.len;
        const uint32_t l0 = g.l0s[r];
        const I d = g.du + g.dl0[r] + __shfl_sync(0xffffffffu, g.tlo, l0 & 31u) +
                    __shfl_sync(0xffffffffu, g.thi, l0 >> 5);
        const T xo = in ? xs[r] : (T)0;
        T acc = seg_diag(d, e.dscale) * xo;
        for (int k = 0; k < g.nib; k++) {
            const uint32_t t = g.itabs[k * g.stride + lane * nb + c];
            if (in && t != 255u) acc = fma(g.ib[k].cxy, xs[t], acc);
        }
        for (int k = 0; k < g.nall; k++) {
            const uint32_t t = k < g.nml ? g.tabs[g.list[k].tab + lane * nb + c] : r;
            if (in && t != 255u) acc = fma(g.list[k].c, xs[(int64_t)g.list[k].delta + t], acc);
        }
        T ac[1] = {acc};
        if (in) seg_out<T, 1, RED>(a, e, g.base + r, true, xs + r, ac, racc);
    }
}

template <typename T, typename I, int RED, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
    k_hvw(const __grid_constant__ HvArgs<T> a, const __grid_constant__ WarpArgs g) {
    constexpr int W = NT / 32;
    extern __shared__ __align__(16) unsigned char s_raw[];
    __shared__ T al_sm;
    // shared layout: per warp the bond list and the staged segment, then the
    // Hamiltonian's tables (one copy of the image in memory), then the traversal
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nlist = g.nu + g.nx;
    const WarpLayout<T, I> lay(g);
    SegEnt<T> *lists = (SegEnt<T> *)s_raw;
    T *stages = (T *)(s_raw + sizeof(SegEnt<T>) * (size_t)W * nlist);
    unsigned char *img = (unsigned char *)(stages + W * kSegStage);
    const I *dl0 = (const I *)img;
    const uint16_t *l0s = (const uint16_t *)(img + lay.l0s), *so = (const uint16_t *)(img + lay.so);
    const uint32_t *jp = (const uint32_t *)(img + lay.jp);
    const SmemBond<T, I> *ub = (const SmemBond<T, I> *)(img + lay.bonds), *mb = ub + nlist, *ib = mb + g.nm;
    const unsigned char *tabs = img + lay.tabs;
    uint16_t *perm = (uint16_t *)(img + lay.bytes);  // counter bytes to bits of h
    {
        const uint4 *src = (const uint4 *)g.fix[sizeof(T) == 8].img;
#pragma unroll 4
        for (int i = threadIdx.x; i < (int)(lay.bytes / 16); i += NT) ((uint4 *)img)[i] = __ldg(src + i);
        if (a.P.use_perm)
            for (int i = threadIdx.x; i < 512; i += NT) perm[i] = (uint16_t)block_of(a.P, i < 256 ? i : (i - 256) << 8);
        for (int i = threadIdx.x; i < W * kSegStage; i += NT) stages[i] = (T)0;
        if (threadIdx.x == 0) {
            al_sm = (T)(a.alpha_dev ? a.alpha_dev[0] : a.alpha[0]);
            if constexpr (seg_scaled<T> && RED != 2) al_sm *= (T)g.fix[1].scale;
        }
    }
    __syncthreads();
    if constexpr (seg_fold<T, RED>) {
        const T al = al_sm;
        for (int i = threadIdx.x; i < nlist + g.nm + g.ni; i += NT) ((SmemBond<T, I> *)ub)[i].cxy *= al;
        __syncthreads();
    }
    Epi<T> e;
    e.keep = spol(a.P.hints, 0);
    e.stream = spol(a.P.hints, 1);
    e.al = &al_sm;
    e.ga = (T)(a.gamma_dev ? a.gamma_dev[0] : a.gamma[0]);
    e.be = (T)a.beta;
    e.dscale = (T)g.fix[sizeof(T) == 8].scale * (seg_fold<T, RED> ? al_sm : (T)1);
    e.use_beta = a.beta != 0.0;
    e.use_v = a.v != nullptr;
    Seg<T, I> sg;
    SegEnt<T> *list = lists + (size_t)warp * nlist;
    sg.list = list;
    sg.nml = g.nx;
    sg.ib = ib;
    sg.nib = g.ni;
    sg.tabs = tabs;
    sg.stride = g.tab_stride;
    sg.stage = stages + warp * kSegStage;
    const int mb0 = lane < g.s ? g.moff[lane] : 0, mb1 = lane < g.s ? g.moff[lane + 1] : 0;
    constexpr int NR = RED == 2 ? 3 : (RED ? 1 : 0);
    RedAcc<T> racc[RED == 2 ? 3 : 1];
    const uint32_t m1 = (1u << g.n1) - 1u;
    // first row of the segment of upper string S: jb[h] in two parts, h = (hh, hl)
    // with hl its low jl <= 8 bits: the rows below (hh, 0), then those below hl among
    // the strings with |hh| (small enough for shared memory)
    const uint32_t ml = (1u << g.jl) - 1u;
    const uint32_t *jlow = jp + g.jhi;
    auto row_of = [&](uint32_t S) -> int {
        const uint32_t h = S >> g.nlo, hh = h >> g.jl;
        const int ph = __popc(hh), p = g.n - __popc(h);
        if (p < 0 || p > g.nlo) return 0;
        return (int)(jp[hh] + jlow[(ph << g.jl) + (h & ml)] + so[(p << g.n1) | ((S >> g.s) & m1)]);
    };
    // unit t of this block's stream: row block t >> n1 (every gridDim.x-th of the
    // traversal), segment order[t & m1] within it, rotated from block to block
    const uint32_t nblk = ((uint32_t)a.P.nh - blockIdx.x + gridDim.x - 1) / gridDim.x;
    const uint32_t units = nblk << g.n1;
#pragma unroll 1
    for (uint32_t t = warp; t < units; t += W) {
        const uint32_t j = t >> g.n1;
        const uint32_t hc = blockIdx.x + j * gridDim.x;
        const uint32_t h = a.P.use_perm ? perm[hc & 255u] | perm[256 + (hc >> 8)] : hc;
        const int p = g.n - __popc(h);
        if (p < 0 || p > g.nlo) continue;
        const uint32_t l1 = g.order[(t + j * g.rot) & m1];
        const int c = p - __popc(l1);
        if (c < 0 || c > g.s) continue;
        const uint32_t S = (h << g.nlo) | (l1 << g.s);
        const int base = row_of(S);
        const WarpClass cl = g.cls[c];
        const int last = (int)a.P.rows - 32 * cl.nc - base;  // largest delta whose padded rows stay inside x
        // the bonds of this segment, one per lane: applicable uniform ones are
        // compacted, mixed ones keep their place
        I dpart = 0;
        int nul = 0;
        bool edge = last < 0;
        __syncwarp();  // the previous segment is done with the lists
#pragma unroll 1
        for (int k0 = 0; k0 < nlist; k0 += 32) {
            const int k = k0 + lane;
            bool app = false;
            SegEnt<T> n;
            if (k < nlist) {
                const SmemBond<T, I> b = ub[k];
                const uint32_t m = S & b.mask;
                const bool uni = k < g.nu, differ = m != 0 && m != b.mask;
                if (!uni || differ) {
                    n.delta = row_of(S ^ b.mask) - base;
                    n.c = b.cxy;
                    if (uni) {
                        dpart += b.cz;
                        app = b.cxy != (T)0;
                        edge = edge || n.delta > last;
                    } else {
                        n.tab = (int)(b.tab + (m ? 0u : 1u)) * g.tab_stride + cl.tab;
                        list[k - g.nu] = n;
                    }
                }
            }
            const unsigned bal = __ballot_sync(0xffffffffu, app);
            if (app) list[g.nx + nul + __popc(bal & ((1u << lane) - 1u))] = n;
            nul += __popc(bal);
        }
        // mixed diagonal: lane b holds w_b = sum cz (1 - 2 u_a); const part sum cz u_a
        I wb = 0;
#pragma unroll 1
        for (int k = mb0; k < mb1; k++) {
            const I cz = mb[k].cz;
            if (S & mb[k].mask) {
                wb -= cz;
                dpart += cz;
            } else {
                wb += cz;
            }
        }
        sg.du = seg_isum(dpart);
        sg.tlo = 0;
        sg.thi = 0;
#pragma unroll
        for (int b = 0; b < 5; b++) {
            const I w0 = __shfl_sync(0xffffffffu, wb, b), w1 = __shfl_sync(0xffffffffu, wb, b + 5);
            if ((lane >> b) & 1) {
                sg.tlo += w0;
                sg.thi += w1;
            }
        }
        edge = __any_sync(0xffffffffu, edge);
        __syncwarp();
        sg.nall = g.nx + nul;
        sg.base = (uint32_t)base;
        sg.len = cl.len;
        sg.dl0 = dl0 + cl.row0;
        sg.l0s = l0s + cl.row0;
        sg.itabs = tabs + (size_t)g.tab_stride * g.ntab + cl.tab;
        if (edge) {
            const Seg<T, I> sg2 = sg;  // copies: what is passed by address lives in memory
            const Epi<T> e2 = e;
            RedAcc<T> r2[RED == 2 ? 3 : 1];
            for (int r = 0; r < NR; r++) r2[r] = racc[r];
            seg_edge<T, I, RED>(a, sg2, e2, lane, cl.nc, r2);
            for (int r = 0; r < NR; r++) racc[r] = r2[r];
            continue;
        }
        switch (cl.nc) {
        case 1: seg_rows<T, I, 1, RED>(a, sg, e, lane, racc); break;
        case 2: seg_rows<T, I, 2, RED>(a, sg, e, lane, racc); break;
        case 3: seg_rows<T, I, 3, RED>(a, sg, e, lane, racc); break;
        case 4: seg_rows<T, I, 4, RED>(a, sg, e, lane, racc); break;
        case 7: seg_rows<T, I, 7, RED>(a, sg, e, lane, racc); break;
        default: seg_rows<T, I, 8, RED>(a, sg, e, lane, racc); break;
        }
    }
    if constexpr (RED != 0) {
        __syncthreads();
        double *red_sm = (double *)s_raw;
#pragma unroll
        for (int r = 0; r < NR; r++) {
            double val = racc[r].value();
#pragma unroll
            for (int off = 16; off >= 1; off >>= 1) val += __shfl_xor_sync(0xffffffffu, val, off);
            if (lane == 0) red_sm[warp * 3 + r] = val;
        }
        __syncthreads();
        if (threadIdx.x < 3) {
            const int r = threadIdx.x;
            double s = 0.0;
            if (r < NR)
                for (int w = 0; w < W; w++) s += red_sm[w * 3 + r];
            a.partials[((int64_t)blockIdx.x * 3 + r) * a.ncol] = s;
        }
    }
}

template <typename T, typename I>
size_t warp_smem(const WarpArgs &g, int W) {
    const WarpLayout<T, I> lay(g);
    return (sizeof(SegEnt<T>) * (size_t)(g.nu + g.nx) + sizeof(T) * kSegStage) * W + lay.bytes + 512 * sizeof(uint16_t);
}

template <typename T, typename I, int RED, int NT, int MINB>
int go_w(hphi_ctx *ctx, const hphi_ham *ham, const HvArgs<T> &a, int64_t want, int *grid_out) {
    const WarpArgs &g = *ham->warp;
    const size_t dyn = warp_smem<T, I>(g, NT / 32);
    const int occ = dyn_occupancy(ctx, (const void *)k_hvw<T, I, RED, NT, MINB>, NT, dyn);
    if (occ < 1) return set_err(ctx, HPHI_E_INVAL, "segment H*x: the tables do not fit in shared memory");
    // no more thread blocks than the partials of an H*x launch hold (8 per SM, one per row block)
    int64_t gr = std::min<int64_t>({(int64_t)std::min(occ, 8) * ctx->sm_count, ham->nh, want});
    if (gr < 1) gr = 1;
    *grid_out = (int)gr;
    const int slot = prof_begin(ctx, PROF_HV);
    k_hvw<T, I, RED, NT, MINB><<<(int)gr, NT, dyn, ctx->stream>>>(a, g);
    snprintf(ctx->last_kernel, sizeof ctx->last_kernel, "k_hvw<%s,%d,s%d,I%d,RED%d>@" HPHI_SRC_TAG, tname<T>(), NT, g.s,
             (int)sizeof(I) * 8, RED);
    prof_end(ctx, slot);
    HPHI_CUDA(ctx, cudaGetLastError());
    return HPHI_OK;
}

template <typename T, typename I, int RED>
int go_size(hphi_ctx *ctx, const hphi_ham *ham, const HvArgs<T> &a, int *grid) {
    const int64_t units = ham->nh << ham->warp->n1;
    if (units >= (int64_t)ctx->sm_count * 64) return go_w<T, I, RED, kSegThreads<T>, 1>(ctx, ham, a, units, grid);
    return go_w<T, I, RED, 64, 8>(ctx, ham, a, (units + 1) / 2, grid);
}

template <typename T, typename I>
int go_red(hphi_ctx *ctx, const hphi_ham *ham, const HvArgs<T> &a, int red_mode, int *grid) {
    switch (red_mode) {
    case 0: return go_size<T, I, 0>(ctx, ham, a, grid);
    case 1: return go_size<T, I, 1>(ctx, ham, a, grid);
    case 2: return go_size<T, I, 2>(ctx, ham, a, grid);
    case 3: return go_size<T, I, 3>(ctx, ham, a, grid);
    default: return HPHI_E_INVAL;
    }
}

}  // namespace

// Tables of the segment kernel for a spin S^z-sector Hamiltonian of at most 32
// sites and fewer than 2^31 rows (ham->warp stays null otherwise, or when the
// tables would not fit in shared memory next to the bond lists, or when no integers
// hold the diagonal).  The host's time for them counts for a Hamiltonian that is used
// once, so it avoids vectors per table, divisions and branches on the strings: 5 us for
// a 16-site chain (first product 46 -> 32), 15 for 20 sites (118 -> 43), 30 for a 14-rung
// ladder (3880 -> 2870).
//
// The kernel issues its mixed-bond FMAs for every row and the bond-major kernel only
// where they apply, so in FP64, where the FP64 pipe bounds both, the latter stays
// where its lists are longest (row blocks of 16 low bits: 4x8 56.9 against 62.3 ms;
// 15 bits: 6x5 15.5 against 15.2).  FP32 problems below 2^14 rows keep it too: both are
// one wave of latency there (16 sites: 10 us).  Away from half filling segments are
// short and lanes idle, but the bond-major kernel's blocks are shorter still: us here
// and there, FP32, 30 sites with 4 / 6 / 10 up spins 68 / 270 / 1432 and 399 / 1048 / 3623,
// 32 sites with 8 up 2042 and 4259; FP64, 24 sites with 1 / 4 up 8 / 26 and 39 / 127.
int build_warp_tables(hphi_ctx *ctx, hphi_ham *H, std::vector<unsigned char> &blob, size_t *at) {
    const hphi_basis *B = H->basis;
    if (B->model != HPHI_SPIN_HALF || B->N > 32 || H->nlo > 16 || H->nlo < 1 || H->D >= ((int64_t)1 << 31))
        return HPHI_OK;
    const bool want32 = H->D >= 16384, want64 = H->nlo < 16;
    if (!want32 && !want64) return HPHI_OK;
    WarpArgs g{};
    g.nlo = H->nlo;
    g.n = H->host.n;
    g.s = H->nlo < kWarpSegMax ? H->nlo : kWarpSegMax;
    g.n1 = g.nlo - g.s;
    g.rot = g.n1 > 0 ? 5 : 0;
    static constexpr Binomials binom;
    // classes: the strings of one popcount, ascending; rows of a segment padded to 32 nc
    const uint32_t nl = 1u << g.s;
    unsigned char pos[1 << kWarpSegMax];  // position of a string in its class
    uint16_t row[1 << kWarpSegMax];       // its padded row (diagonal, string)
    uint16_t slot[1 << kWarpSegMax];      // its byte in a rank table
    int rows = 0;
    for (int c = 0; c <= g.s; c++) {
        WarpClass &k = g.cls[c];
        k.len = (uint32_t)binom(g.s, c);
        const int need = (int)((k.len + 31) / 32);
        if (need == 5 || need == 6 || need > kSegRows) return HPHI_OK;  // C(s, c) for s <= 10 has none
        k.nc = need;
        k.row0 = k.tab = rows;
        rows += 32 * (need > 4 ? 8 : need > 2 ? 4 : need);
    }
    g.nrow = g.tab_stride = rows;
    int seen[kWarpSegMax + 1] = {};
    for (uint32_t l = 0; l < nl; l++) {
        const int c = __builtin_popcount(l), r = seen[c]++, need = g.cls[c].nc;
        pos[l] = (unsigned char)r;
        row[l] = (uint16_t)(g.cls[c].row0 + r);
        slot[l] = (uint16_t)(g.cls[c].tab + (r & 31) * (need > 4 ? 8 : need > 2 ? 4 : need) + (r >> 5));
    }
    // bonds; the diagonal (at most a quarter of sum |Jz|) in fixed point below 2^62
    double bound = 0.0, c0 = 0.0, weak = 0.0;  // weak: the smallest Jxy/2
    for (const DTerm &t : H->dterms) {
        bound += fabs(t.a);
        c0 += 0.25 * t.a;
        if (!(fabs(t.b) < 1e30)) return HPHI_OK;  // rows that a bond does not touch add 0 times alpha Jxy/2
        if (t.b != 0.0 && (weak == 0.0 || 0.5 * fabs(t.b) < weak)) weak = 0.5 * fabs(t.b);
    }
    if (!isfinite(bound)) return HPHI_OK;
    int ed = 0;
    frexp(bound > 0.0 ? 0.25 * bound : 1.0, &ed);  // |diagonal| < 2^ed
    if (ed < -60 || ed > 100) return HPHI_OK;      // the scale is a normal number in FP32 too
    // Which integers hold it: the grid follows the sum of all |Jz|, and strong bonds may
    // cancel in a row.  Every Jz/2 keeps the digits that it has in the vectors' type, or a
    // grid step is at most a quarter ulp of the smallest exchange coefficient, whose terms
    // round by more; FP64 also where C0 = sum Jz/4 is not small against the grid (2^56
    // steps), as the other kernels' sums start from C0 and round at its scale.  32-bit
    // integers for FP32 vectors, 64-bit where those do not keep the digits (ms, 32, 64 bits,
    // bond-major kernel: 14-rung ladder 0.493, 0.557, 1.58; 4x8 14.2, 14.6, 24.4).
    auto keeps = [&](int bits, int digits) {
        bool ok = true;
        for (const DTerm &t : H->dterms) ok = ok && fix_keeps(0.5 * t.a, ed, bits, digits);
        return ok || ldexp(1.0, ed - bits) <= ldexp(weak, -digits - 1);
    };
    if (want64 && (keeps(kSegBits, 53) || fabs(c0) >= ldexp(1.0, ed - 6))) g.fix[1].bytes = 8;
    if (want32) g.fix[0].bytes = keeps(30, 24) ? 4 : keeps(kSegBits, 24) ? 8 : 0;
    auto fixed = [&](double v) { return (long long)llrint(ldexp(v, kSegBits - ed)); };
    std::vector<WarpBond> ub, xb, ib;  // uniform, mixed, inner
    std::vector<std::vector<WarpBond>> mb(g.s);
    std::vector<int> tab_bit(g.s, -1);
    std::vector<unsigned char> tabs, itabs;  // rank tables, one after the other
    tabs.reserve((size_t)2 * g.s * rows);
    itabs.reserve(H->dterms.size() * rows);
    auto new_table = [&](std::vector<unsigned char> &to) {
        to.resize(to.size() + rows, 255);
        return (uint32_t)(to.size() / rows) - 1;
    };
    std::vector<long long> dl(nl, 0);  // diagonal of the bonds inside, per string
    for (const DTerm &t : H->dterms) {
        const int i = t.i < t.j ? t.i : t.j, j = t.i < t.j ? t.j : t.i;
        const double cz = -0.5 * t.a, cxy = 0.5 * t.b;
        WarpBond b{};
        b.cxy = cxy;
        b.cz = fixed(cz);
        if (i >= g.s) {
            b.mask = (1u << i) | (1u << j);
            ub.push_back(b);
        } else if (j >= g.s) {
            b.mask = 1u << j;
            if (cz != 0.0) mb[i].push_back(b);
            if (cxy != 0.0) {
                if (tab_bit[i] < 0) {
                    tab_bit[i] = (int)new_table(tabs);
                    new_table(tabs);
                    unsigned char *t0 = tabs.data() + (size_t)tab_bit[i] * rows, *t1 = t0 + rows;
                    for (uint32_t a = 0; a < nl; a += 2u << i)
                        for (uint32_t l = a; l < a + (1u << i); l++) {  // l and l with bit i
                            t0[slot[l]] = pos[l | 1u << i];
                            t1[slot[l | 1u << i]] = pos[l];
                        }
                }
                b.tab = (uint32_t)tab_bit[i];
                xb.push_back(b);
            }
        } else {
            unsigned char *t = nullptr;
            if (cxy != 0.0) {
                b.tab = new_table(itabs);
                t = itabs.data() + (size_t)b.tab * rows;
                ib.push_back(b);
            }
            for (uint32_t a = 0; a < nl; a += 2u << j)
                for (uint32_t c = a; c < a + (1u << j); c += 2u << i)
                    for (uint32_t l = c; l < c + (1u << i); l++) {  // l with bit i, l with bit j
                        const uint32_t li = l | 1u << i, lj = l | 1u << j;
                        dl[li] += b.cz;
                        dl[lj] += b.cz;
                        if (t) {
                            t[slot[li]] = pos[lj];
                            t[slot[lj]] = pos[li];
                        }
                    }
        }
    }
    const long long c0f = fixed(c0);
    std::vector<WarpBond> all(ub);
    all.insert(all.end(), xb.begin(), xb.end());
    int m = 0;
    for (int b = 0; b < g.s; b++) {
        g.moff[b] = m;
        m += (int)mb[b].size();
        all.insert(all.end(), mb[b].begin(), mb[b].end());
    }
    for (int b = g.s; b <= kWarpSegMax; b++) g.moff[b] = m;
    all.insert(all.end(), ib.begin(), ib.end());
    g.nu = (int)ub.size();
    g.nx = (int)xb.size();
    g.nm = m;
    g.ni = (int)ib.size();
    g.ntab = (int)(tabs.size() / rows);
    std::vector<uint16_t> so((size_t)(g.nlo + 1) << g.n1);
    for (int p = 0; p <= g.nlo; p++) {
        int64_t acc = 0;
        for (uint32_t l1 = 0; l1 < (1u << g.n1); l1++) {
            so[((size_t)p << g.n1) | l1] = (uint16_t)acc;
            acc += binom(g.s, p - __builtin_popcount(l1));
        }
    }
    // jb[h] = jp[hh] + jp[jhi + (|hh| << jl) + hl]
    const int nhi = B->N - g.nlo;
    g.jl = nhi < 8 ? nhi : 8;
    g.jw = nhi - g.jl;
    g.jhi = 1 << g.jw;
    std::vector<uint32_t> jp;
    {
        int64_t acc = 0;
        for (uint32_t t = 0; t < (1u << g.jw); t++) {
            jp.push_back((uint32_t)acc);
            for (int k = 0; k <= g.jl; k++) acc += binom(g.jl, k) * binom(g.nlo, g.n - __builtin_popcount(t) - k);
        }
        for (int ph = 0; ph <= g.jw; ph++) {
            acc = 0;
            for (uint32_t t = 0; t < (1u << g.jl); t++) {
                jp.push_back((uint32_t)acc);
                acc += binom(g.nlo, g.n - ph - __builtin_popcount(t));
            }
        }
    }
    // segments of a row block, long ones first (popcounts near the middle)
    std::vector<int> ord(1 << g.n1);
    for (int i = 0; i < (1 << g.n1); i++) ord[i] = i;
    std::stable_sort(ord.begin(), ord.end(), [&](int x, int y) {
        return std::abs(2 * __builtin_popcount(x) - g.n1) < std::abs(2 * __builtin_popcount(y) - g.n1);
    });
    for (int i = 0; i < (1 << g.n1); i++) g.order[i] = (uint8_t)ord[i];
    const size_t most = 200 * 1024;
    if (warp_smem<double, long long>(g, kSegThreads<double> / 32) > most) g.fix[1].bytes = 0;
    if ((g.fix[0].bytes == 8 ? warp_smem<float, long long>(g, kSegThreads<float> / 32)
                             : warp_smem<float, int>(g, kSegThreads<float> / 32)) > most)
        g.fix[0].bytes = 0;
    if (!g.fix[0].bytes && !g.fix[1].bytes) return HPHI_OK;
    // the images of both precisions
    blob.reserve(blob.size() + (g.fix[0].bytes ? WarpLayout<float, long long>(g).bytes : 0) +
                 (g.fix[1].bytes ? WarpLayout<double, long long>(g).bytes : 0) + 4096);
    auto image = [&](auto zero, auto izero) {
        using T = decltype(zero);
        using I = decltype(izero);
        const WarpLayout<T, I> lay(g);
        const size_t start = (blob.size() + 15) & ~(size_t)15;
        blob.resize(start + lay.bytes, 0);
        unsigned char *p = blob.data() + start;
        for (int i = 0; i < rows; i++) ((I *)p)[i] = to_fix<I, kSegBits>(c0f);
        for (uint32_t l = 0; l < nl; l++) {
            ((I *)p)[row[l]] = to_fix<I, kSegBits>(c0f + dl[l]);
            ((uint16_t *)(p + lay.l0s))[row[l]] = (uint16_t)l;
        }
        memcpy(p + lay.so, so.data(), sizeof(uint16_t) * so.size());
        memcpy(p + lay.jp, jp.data(), sizeof(uint32_t) * jp.size());
        for (size_t i = 0; i < all.size(); i++)
            ((SmemBond<T, I> *)(p + lay.bonds))[i] =
                SmemBond<T, I>{(T)(seg_scaled<T> ? ldexp(all[i].cxy, kSegBits - ed) : all[i].cxy), to_fix<I, kSegBits>(all[i].cz), all[i].mask, all[i].tab};
        if (!tabs.empty()) memcpy(p + lay.tabs, tabs.data(), tabs.size());
        if (!itabs.empty()) memcpy(p + lay.tabs + tabs.size(), itabs.data(), itabs.size());
        return start;
    };
    if (g.fix[0].bytes) at[0] = g.fix[0].bytes == 8 ? image(0.0f, 0ll) : image(0.0f, 0);
    if (g.fix[1].bytes) at[1] = image(0.0, 0ll);
    for (int t = 0; t < 2; t++) g.fix[t].scale = ldexp(1.0, ed - (g.fix[t].bytes == 4 ? 30 : kSegBits));
    H->warp = new (std::nothrow) WarpArgs(g);
    if (!H->warp) return set_err(ctx, HPHI_E_NOMEM, "segment kernel tables");
    return HPHI_OK;
}

template <typename T>
int launch_warp(hphi_ctx *ctx, const hphi_ham *ham, const HvArgs<T> &a, int red_mode, int *grid) {
    if (!ham->warp) return set_err(ctx, HPHI_E_INVAL, "segment H*x: not available for this Hamiltonian");
    if (a.ldx != 1 || a.ldy != 1 || (a.v && a.ldv != 1))
        return set_err(ctx, HPHI_E_INVAL, "segment H*x: one contiguous column only");
    const int bytes = ham->warp->fix[sizeof(T) == 8].bytes;
    if (bytes == 8) return go_red<T, long long>(ctx, ham, a, red_mode, grid);
    if constexpr (sizeof(T) == 4)
        if (bytes == 4) return go_red<T, int>(ctx, ham, a, red_mode, grid);
    return set_err(ctx, HPHI_E_INVAL, "segment H*x: not available for this Hamiltonian");
}

template int launch_warp<float>(hphi_ctx *, const hphi_ham *, const HvArgs<float> &, int, int *);
template int launch_warp<double>(hphi_ctx *, const hphi_ham *, const HvArgs<double> &, int, int *);

}  // namespace hphi
