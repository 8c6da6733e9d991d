// Hubbard H*x kernel: one real column, or one pair of columns (a complex vector).
//
// Row (up, dn) = up * D_dn + dn.  The down hops of a row depend on dn alone, the
// up hops on up alone (Sec. 3.4 H_quench, Sec. 5): a thread block owns U
// consecutive up strings and stages their U * D_dn rows in shared memory, the
// values of one dn side by side in 16 bytes (U up strings x C columns: U = 4 in
// FP32, 2 in FP64, half of that for a pair of columns).  A thread owns one dn:
//   - a down hop is one list entry (target, coefficient), read once for all U C
//     values, one 16-byte shared load and U C FMAs;
//   - an up hop of string u is the same for the whole block: a coalesced load of
//     row block u' and one FMA per value.
// So the sums stay in registers and the list entries are read once per 16 bytes
// of result.  The diagonal sum_i U_i n_iu n_id + sum V n_i n_j is summed in fixed
// point: per up string, tables over groups of 6 sites of dn.  The grid follows the
// sum of the couplings' magnitudes, and a row without a doubly occupied site has no
// U in it, so the integers are chosen by what the grid does to the smallest coupling
// (build_hub_tables): FP32 vectors take 32 bits where every coupling keeps its 24,
// else 64; FP64 vectors one grid or two, one for U and one for V, and the kernel
// only where these cost less than the hops round.
//
// What bounds it: FP64 the FP64 pipe (89 % busy; a warp's down hops run as many
// rounds as its longest list), FP32 the latency of the up-hop loads (4x4: 6 stalls per
// issue at 32 warps per SM, 17.9 GB from L2 at 5.4 TB/s) and the bank conflicts of the
// 16-byte gathers (36 % of the shared-load wavefronts).  ms per product, before and
// now: 4x4 FP32 5.66 -> 3.3, FP64 17.1 -> 12.6; 7x2 ladder FP32 0.400 -> 0.148, complex
// FP64 1.75 -> 1.36; 6x2 complex FP64 0.149 -> 0.107.  (Before: the bond-major kernel,
// hv_phased.cu, which walks a list per (hop pair, sign) through a shared
// accumulator, 22 warp instructions per row against 11 here; for pairs the
// generic kernel, which issues its FMAs for every slot of a batch of eight.)
// Tried: 8 down hops in flight 44: 3.67, 16 up hops 3.69, 512 threads 4.2, thread
// counts that leave no lane idle 7x2 FP32 0.179.
#include "fixed.cuh"
#include "hvcommon.cuh"

#include <math.h>
#include <string.h>

#include <algorithm>
#include <new>
#include <type_traits>
#include <vector>

namespace hphi {

namespace {

constexpr int kHubGroup = 6;  // sites per diagonal table
constexpr int kHubBits = 62;  // the diagonal lies below 2^62 grid steps

template <typename T>
struct alignas(16) HubPack {
    T e[16 / sizeof(T)];
};

template <typename I, int U>
struct alignas(sizeof(I) * U < 16 ? sizeof(I) * U : 16) IntPack {  // the diagonal parts of U up strings
    I e[U];
};

template <typename T>
struct alignas(2 * sizeof(T)) HubHop {   // an up hop: first row of the target's block, coefficient
    uint32_t row;
    T c;
};

// C columns of row r (C = 2: one 8- or 16-byte access)
template <typename T, int C>
__device__ __forceinline__ void hub_load(const T *__restrict__ x, uint32_t r, T (&v)[C]) {
    if constexpr (C == 1) {
        v[0] = __ldg(x + r);
    } else if constexpr (sizeof(T) == 4) {
        const float2 t = __ldg(reinterpret_cast<const float2 *>(x) + r);
        v[0] = t.x;
        v[1] = t.y;
    } else {
        const double2 t = __ldg(reinterpret_cast<const double2 *>(x) + r);
        v[0] = t.x;
        v[1] = t.y;
    }
}
template <typename T, int C>
__device__ __forceinline__ void hub_load_rw(const T *x, uint32_t r, T (&v)[C]) {  // may alias the output
    if constexpr (C == 1) {
        v[0] = x[r];
    } else if constexpr (sizeof(T) == 4) {
        const float2 t = *(reinterpret_cast<const float2 *>(x) + r);
        v[0] = t.x;
        v[1] = t.y;
    } else {
        const double2 t = *(reinterpret_cast<const double2 *>(x) + r);
        v[0] = t.x;
        v[1] = t.y;
    }
}
template <typename T, int C>
__device__ __forceinline__ void hub_store(T *y, uint32_t r, const T (&v)[C]) {
    if constexpr (C == 1) y[r] = v[0];
    else if constexpr (sizeof(T) == 4) *(reinterpret_cast<float2 *>(y) + r) = make_float2(v[0], v[1]);
    else *(reinterpret_cast<double2 *>(y) + r) = make_double2(v[0], v[1]);
}

// Sums that a diagonal is made of: 2 where V has a grid of its own.
template <typename T>
__host__ __device__ __forceinline__ int hub_parts(const HubArgs &g) { return sizeof(T) == 8 ? g.fix[1].parts : 1; }

// dn strings of a thread at a time (an FP64 pair fills the pipe with one)
template <typename T, int C> constexpr int hub_dn = sizeof(T) == 8 && C == 2 ? 1 : 2;

// acc[i] += c v[i] over one pack
__device__ __forceinline__ void pack_fma(float c, const HubPack<float> &v, float (&acc)[4]) {
#pragma unroll
    for (int i = 0; i < 4; i += 2) fma2(acc[i], acc[i + 1], c, v.e[i], v.e[i + 1]);
}
__device__ __forceinline__ void pack_fma(double c, const HubPack<double> &v, double (&acc)[2]) {
    acc[0] = fma(c, v.e[0], acc[0]);
    acc[1] = fma(c, v.e[1], acc[1]);
}

template <typename T, typename I, int C, int RED, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
    k_hub(const __grid_constant__ HvArgs<T> a, const __grid_constant__ HubArgs g) {
    constexpr int P = 16 / (int)sizeof(T), U = P / C;
    constexpr int QB = hub_dn<T, C>;
    constexpr int HB = 8 / C / ((int)sizeof(T) / 4);        // up hops in flight
    constexpr int DB = 4;                                   // down hops in flight
    extern __shared__ __align__(16) unsigned char s_raw[];
    const uint32_t ddn = g.ddn;
    HubPack<T> *xs = (HubPack<T> *)s_raw;
    HubHop<T> *hops = (HubHop<T> *)(xs + ddn);              // [U][up_pad], zeros behind the list
    I *tab = (I *)(hops + U * g.up_pad);                    // [ngrp][64][U]
    const HubFix &fx = g.fix[sizeof(T) == 8];
    const int parts = hub_parts<T>(g);                      // sums of a diagonal: U and V apart, or together
    I *wj = tab + parts * U * g.ngrp * 64;                  // [U][32]; a second set of both for V
    T *coef = (T *)(wj + parts * U * 32);                   // [n_coef]
    __shared__ int nup[U];
    __shared__ I du[U];
    const HamDesc &D = *a.P.desc;
    __shared__ T al_sm[C];  // (registers less through the hops)
    T ga[C];
#pragma unroll
    for (int c = 0; c < C; c++) ga[c] = (T)(a.gamma_dev ? a.gamma_dev[c] : a.gamma[c]);
    // FP64 hops are taken over the diagonal's scale (a power of two, so exact) and H x is
    // scaled with alpha in one multiplication: the FP64 pipe is the bound.  FP32 ones are
    // not: the scaled sums of vectors above 1e19 would overflow (FP64's only above 1e288).
    constexpr bool PRE = sizeof(T) == 8;
    const T dscale = (T)fx.scale, vscale = (T)(PRE ? fx.vscale / fx.scale : fx.vscale);
    const T cscale = (T)(PRE ? 1.0 / fx.scale : 1.0);
    if (threadIdx.x < C) {
        const T al = (T)(a.alpha_dev ? a.alpha_dev[threadIdx.x] : a.alpha[threadIdx.x]);
        al_sm[threadIdx.x] = PRE && RED != 2 ? al * dscale : al;
    }
    for (int i = threadIdx.x; i < D.n_ncoef; i += NT) coef[i] = (T)D.coef[i] * cscale;
    const T be = (T)a.beta;
    const bool use_beta = a.beta != 0.0, use_v = a.v != nullptr;
    const T *__restrict__ X = a.x;
    constexpr int NR = RED == 2 ? 3 : (RED ? 1 : 0);
    RedAcc<T> racc[NR > 0 ? NR : 1][C];
    // unit blk: U up strings and every g.split-th round of their down strings
    const uint32_t nblk = (g.nh + U - 1) / U * g.split;
    for (uint32_t blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
        const uint32_t u0 = blk / g.split * U, part = blk % g.split;
        __syncthreads();  // the previous block is done with the shared arrays
        // up hops, down-site weights w_j = U_j n_j + sum V n_other, rows of the block
        for (int i = threadIdx.x; i < U * g.up_pad; i += NT) {
            const int u = i / g.up_pad, e = i - u * g.up_pad;
            const uint32_t h = u0 + u;
            HubHop<T> hp;
            hp.row = 0;
            hp.c = (T)0;
            if (h < g.nh && e < a.P.up_cnt[h]) {
                hp.row = a.P.up_tgt[(int64_t)e * g.nh + h] * ddn;
                hp.c = coef[a.P.up_cf[(int64_t)e * g.nh + h]];
            }
            hops[i] = hp;
        }
        for (int i = threadIdx.x; i < U * 32; i += NT) {
            const int u = i >> 5, j = i & 31;
            const uint32_t h = u0 + u;
            I w = 0, wv = 0;
            if (h < g.nh && j < g.N) {
                const uint32_t su = a.P.states_up[h];
                if ((su >> j) & 1u) w += to_fix<I, kHubBits>(fx.ufix[j]);
                for (int k = 0; k < g.nv; k++) {
                    const HubV v = fx.vfix[k];
                    if (v.j == j && ((su >> v.i) & 1u)) wv += to_fix<I, kHubBits>(v.v);
                    if (v.i == j && ((su >> v.j) & 1u)) wv += to_fix<I, kHubBits>(v.v);
                }
            }
            wj[i] = parts == 2 ? w : w + wv;
            if (parts == 2) wj[U * 32 + i] = wv;
            if (j == 0) {
                nup[u] = h < g.nh ? a.P.up_cnt[h] : 0;
                du[u] = h < g.nh && fx.dup ? to_fix<I, kHubBits>(fx.dup[h]) : (I)0;
            }
        }
        for (uint32_t q = threadIdx.x; q < ddn; q += NT) {
            HubPack<T> x;
#pragma unroll
            for (int u = 0; u < U; u++) {
                T v[C];
#pragma unroll
                for (int c = 0; c < C; c++) v[c] = (T)0;
                if (u0 + u < g.nh) hub_load<T, C>(X, (u0 + u) * ddn + q, v);
#pragma unroll
                for (int c = 0; c < C; c++) x.e[u * C + c] = v[c];
            }
            xs[q] = x;
        }
        __syncthreads();
        for (int i = threadIdx.x; i < parts * U * g.ngrp * 64; i += NT) {
            const int u = i % U, r = i / U, gr = r >> 6, v = parts == 2 && gr >= g.ngrp;
            const int j0 = (gr - (v ? g.ngrp : 0)) * kHubGroup;
            I s = 0;
#pragma unroll
            for (int k = 0; k < kHubGroup; k++)
                if ((r >> k) & 1) s += wj[(v * U + u) * 32 + (j0 + k < 32 ? j0 + k : 31)];
            tab[i] = s;
        }
        __syncthreads();
        for (uint32_t q0 = threadIdx.x + part * (NT * QB); q0 < ddn; q0 += NT * QB * g.split) {
            T acc[QB][P];
            uint32_t q[QB];
            bool on[QB];
            int cnt[QB];
#pragma unroll
            for (int b = 0; b < QB; b++) {
                on[b] = q0 + b * NT < ddn;
                q[b] = on[b] ? q0 + b * NT : q0;
                const uint32_t s = __ldg(a.P.states_dn + q[b]);
                cnt[b] = on[b] ? __ldg(a.P.ll_cnt + q[b]) : 0;
                const I dl = fx.ddnf ? to_fix<I, kHubBits>(__ldg(fx.ddnf + q[b])) : (I)0;
                const HubPack<T> x = xs[q[b]];
                // sum of one set of tables, on top of d
                auto add = [&](const I *tb, I (&d)[U]) {
                    for (int k = 0; k < g.ngrp; k++) {
                        const IntPack<I, U> t = *(const IntPack<I, U> *)(tb + (k * 64 + ((s >> (kHubGroup * k)) & 63u)) * U);
#pragma unroll
                        for (int u = 0; u < U; u++) d[u] += t.e[u];
                    }
                };
                I d[U];
#pragma unroll
                for (int u = 0; u < U; u++) d[u] = dl + du[u];
                T dt[U];
                if (parts == 2) {  // the V part apart (FP64)
                    T dv[U];
                    add(tab + U * g.ngrp * 64, d);
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        dv[u] = (T)d[u] * vscale;
                        d[u] = 0;
                    }
                    add(tab, d);
#pragma unroll
                    for (int u = 0; u < U; u++) dt[u] = (T)d[u] + dv[u];
                } else {
                    add(tab, d);
#pragma unroll
                    for (int u = 0; u < U; u++) dt[u] = PRE ? (T)d[u] : (T)d[u] * dscale;
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
#pragma unroll
                    for (int c = 0; c < C; c++) acc[b][u * C + c] = dt[u] * x.e[u * C + c];
                }
            }
            // the down hops wait on shared memory, the up hops on L2: odd warps take them the
            // other way round, so that one half of the warps covers the other's waits
#pragma unroll 1
            for (int ph = 0; ph < 2; ph++) {
                if (((threadIdx.x >> 5) & 1) == ph) {
                    // down hops: DB list entries of every dn in flight
                    int most = cnt[0];
#pragma unroll
                    for (int b = 1; b < QB; b++) most = cnt[b] > most ? cnt[b] : most;
#pragma unroll 1
                    for (int e0 = 0; e0 < most; e0 += DB) {
                        uint32_t pk[QB][DB];
#pragma unroll
                        for (int b = 0; b < QB; b++)
#pragma unroll
                            for (int e = 0; e < DB; e++) {
                                pk[b][e] = 0u;
                                if (e0 + e < cnt[b]) pk[b][e] = __ldg(a.P.ll_pk + (uint32_t)(e0 + e) * ddn + q[b]);
                            }
#pragma unroll
                        for (int b = 0; b < QB; b++)
#pragma unroll
                            for (int e = 0; e < DB; e++)
                                if (e0 + e < cnt[b]) pack_fma(coef[pk[b][e] >> 24], xs[pk[b][e] & 0xFFFFFFu], acc[b]);
                    }
                } else {
                    // up hops, string by string, HB in flight; a value that is not loaded is 0
#pragma unroll
                    for (int u = 0; u < U; u++) {
                        const HubHop<T> *hp = hops + u * g.up_pad;
                        const int n = nup[u];
#pragma unroll 1
                        for (int k = 0; k < n; k += HB) {
                            T v[HB][QB][C], cf[HB];
#pragma unroll
                            for (int e = 0; e < HB; e++) {
                                const bool in = k + e < n;
                                const HubHop<T> h = hp[k + e];
                                cf[e] = h.c;
#pragma unroll
                                for (int b = 0; b < QB; b++) {
#pragma unroll
                                    for (int c = 0; c < C; c++) v[e][b][c] = (T)0;
                                    if (in) hub_load<T, C>(X, h.row + q[b], v[e][b]);
                                }
                            }
#pragma unroll
                            for (int e = 0; e < HB; e++) {
                                if (sizeof(T) == 8 && k + e >= n) break;  // FP64: no FMA that adds nothing
#pragma unroll
                                for (int b = 0; b < QB; b++)
#pragma unroll
                                    for (int c = 0; c < C; c++) acc[b][u * C + c] = fma(cf[e], v[e][b][c], acc[b][u * C + c]);
                            }
                        }
                    }
                }
            }
            // epilogue: y = alpha (H x) + beta y + gamma v, old values loaded before any store
            auto finish = [&](int b, auto times_alpha) {
                const HubPack<T> x = xs[q[b]];
                T out[P];
                if constexpr (PRE && RED == 2) {
#pragma unroll
                    for (int i = 0; i < P; i++) acc[b][i] *= dscale;
                }
                T al[C];
#pragma unroll
                for (int c = 0; c < C; c++) al[c] = al_sm[c];
#pragma unroll
                for (int u = 0; u < U; u++)
#pragma unroll
                    for (int c = 0; c < C; c++) {
                        const T hx = acc[b][u * C + c], other = acc[b][u * C + (C == 2 ? c ^ 1 : c)];
                        if constexpr (decltype(times_alpha)::value) out[u * C + c] = al[c] * (C == 2 && a.swap ? other : hx);
                        else out[u * C + c] = hx;
                    }
                if (use_beta) {
#pragma unroll
                    for (int u = 0; u < U; u++)
                        if (u0 + u < g.nh) {
                            T t[C];
                            hub_load_rw<T, C>(a.y, (u0 + u) * ddn + q[b], t);
#pragma unroll
                            for (int c = 0; c < C; c++) out[u * C + c] = fma(be, t[c], out[u * C + c]);
                        }
                }
                if (use_v) {
#pragma unroll
                    for (int u = 0; u < U; u++)
                        if (u0 + u < g.nh) {
                            T t[C];
                            hub_load_rw<T, C>(a.v, (u0 + u) * ddn + q[b], t);
#pragma unroll
                            for (int c = 0; c < C; c++) out[u * C + c] = fma(ga[c], t[c], out[u * C + c]);
                        }
                }
#pragma unroll
                for (int u = 0; u < U; u++) {
                    if (u0 + u >= g.nh) continue;
                    T o[C];
#pragma unroll
                    for (int c = 0; c < C; c++) o[c] = out[u * C + c];
                    hub_store<T, C>(a.y, (u0 + u) * ddn + q[b], o);
#pragma unroll
                    for (int c = 0; c < C; c++) {
                        const T xo = x.e[u * C + c], hx = acc[b][u * C + c];
                        if constexpr (RED == 1) racc[0][c].add(xo, o[c]);
                        if constexpr (RED == 2) {
                            racc[0][c].add(xo, hx);
                            racc[1][c].add(hx, hx);
                            racc[2][c].add(xo, xo);
                        }
                        if constexpr (RED == 3) racc[0][c].add(o[c], o[c]);
                    }
                }
            };
            // one FP32 column with alpha = 1 (the usual product) has an epilogue of its own: the
            // multiplications cost it 2 to 9 % at 12 to 14 sites
            const bool plain = C == 1 && !PRE && al_sm[0] == (T)1;
#pragma unroll
            for (int b = 0; b < QB; b++) {
                if (!on[b]) continue;
                if (plain) finish(b, std::false_type());
                else finish(b, std::true_type());
            }
        }
    }
    if constexpr (RED != 0) {
        __shared__ double red_sm[NT / 32][3][C];
        const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
        for (int r = 0; r < NR; r++)
#pragma unroll
            for (int c = 0; c < C; c++) {
                double val = racc[r][c].value();
#pragma unroll
                for (int off = 16; off >= 1; off >>= 1) val += __shfl_xor_sync(0xffffffffu, val, off);
                if (lane == 0) red_sm[warp][r][c] = val;
            }
        __syncthreads();
        if (threadIdx.x < 3 * C) {
            const int r = threadIdx.x / C, c = threadIdx.x % C;
            double s = 0.0;
            if (r < NR)
                for (int w = 0; w < NT / 32; w++) s += red_sm[w][r][c];
            a.partials[((int64_t)blockIdx.x * 3 + r) * a.ncol + c] = s;
        }
    }
}

template <typename T, int C>
size_t hub_smem(const HubArgs &g, int ncoef, int int_bytes) {
    const size_t U = 16 / sizeof(T) / C;
    return (size_t)g.ddn * 16 + U * g.up_pad * sizeof(HubHop<T>) +
           hub_parts<T>(g) * U * (g.ngrp * 64 + 32) * (size_t)int_bytes + ncoef * sizeof(T);
}

template <typename T, typename I, int C, int RED, int NT, int MINB>
int go_hub(hphi_ctx *ctx, const hphi_ham *ham, const HvArgs<T> &a, int *grid) {
    HubArgs g = *ham->hub;
    const size_t dyn = hub_smem<T, C>(g, ham->host.n_ncoef, (int)sizeof(I));
    const int occ = dyn_occupancy(ctx, (const void *)k_hub<T, I, C, RED, NT, MINB>, NT, dyn);
    if (occ < 1) return set_err(ctx, HPHI_E_INVAL, "Hubbard H*x: the rows of an up string do not fit in shared memory");
    constexpr int U = 16 / (int)sizeof(T) / C;
    // few up strings: several thread blocks share them, each with a part of the down strings
    // (they all stage the rows), as long as every one gets an SM and a round of its own
    // (us: 16 sites, 1 up 7 down, FP64 180 -> 39, bond-major kernel 109; FP32 67 -> 20, 66)
    const int64_t blocks = (g.nh + U - 1) / U, rounds = (g.ddn + NT * hub_dn<T, C> - 1) / (NT * hub_dn<T, C>);
    g.split = (uint32_t)std::max<int64_t>(1, std::min<int64_t>(rounds, ctx->sm_count / blocks));
    // no more thread blocks than the partials of an H*x launch hold (8 per SM)
    const int64_t gr = std::min<int64_t>((int64_t)std::min(occ, 8) * ctx->sm_count, blocks * g.split);
    *grid = (int)(gr < 1 ? 1 : gr);
    const int slot = prof_begin(ctx, PROF_HV);
    k_hub<T, I, C, RED, NT, MINB><<<*grid, NT, dyn, ctx->stream>>>(a, g);
    snprintf(ctx->last_kernel, sizeof ctx->last_kernel, "k_hub<%s,C%d,%d,I%d,RED%d>@" HPHI_SRC_TAG, tname<T>(), C, NT,
             (int)sizeof(I) * 8, RED);
    prof_end(ctx, slot);
    HPHI_CUDA(ctx, cudaGetLastError());
    return HPHI_OK;
}

template <typename T, typename I, int C, int RED>
int go_hub_size(hphi_ctx *ctx, const hphi_ham *ham, const HvArgs<T> &a, int *grid) {
    // Where the blocks leave SMs or the wave half empty, wider ones run fewer rounds one after
    // the other: 1024 threads up to one block per SM, 256 up to four, as far as the down
    // strings fill them (FP64 real: two per thread keep the pipe busy up to 1024).  us: 14
    // sites, 2 up 7 down, FP32 45 -> 16, bond-major kernel 31; 10 sites, 2 up 5 down, complex
    // FP64 20.5 -> 9.9, generic kernel 12.4.
    constexpr int U = 16 / (int)sizeof(T) / C;
    const int64_t blocks = (ham->hub->nh + U - 1) / U, ddn = ham->hub->ddn;
    if (blocks <= ctx->sm_count && ddn > (sizeof(T) == 8 && C == 1 ? 1024 : 512))
        return go_hub<T, I, C, RED, 1024, 1>(ctx, ham, a, grid);
    if (blocks <= 4 * ctx->sm_count && ddn > 64 && ddn <= 512)
        return go_hub<T, I, C, RED, 256, 4>(ctx, ham, a, grid);
    if (ham->hub->ddn > 4096) return go_hub<T, I, C, RED, 1024, 1>(ctx, ham, a, grid);
    if (ham->hub->ddn > 512) return go_hub<T, I, C, RED, 256, 4>(ctx, ham, a, grid);
    return go_hub<T, I, C, RED, 64, 8>(ctx, ham, a, grid);
}

template <typename T, typename I, int C>
int go_hub_red(hphi_ctx *ctx, const hphi_ham *ham, const HvArgs<T> &a, int red_mode, int *grid) {
    switch (red_mode) {
    case 0: return go_hub_size<T, I, C, 0>(ctx, ham, a, grid);
    case 1: return go_hub_size<T, I, C, 1>(ctx, ham, a, grid);
    case 2: return go_hub_size<T, I, C, 2>(ctx, ham, a, grid);
    case 3: return go_hub_size<T, I, C, 3>(ctx, ham, a, grid);
    default: return HPHI_E_INVAL;
    }
}

}  // namespace

// Fixed-point diagonal tables of the Hubbard kernel.  ham->hub stays null when
// the packed down-hop lists are missing, or the rows of one up string (16 bytes
// per down string) do not fit in shared memory, or the model has more than 32
// sites or 2^32 rows, or no integers hold its diagonal.
int build_hub_tables(hphi_ctx *ctx, hphi_ham *H) {
    const hphi_basis *B = H->basis;
    if (B->model != HPHI_HUBBARD || B->N > 32 || H->D >= ((int64_t)1 << 32)) return HPHI_OK;
    if (H->ll_w > 0 && !H->ll_pk) return HPHI_OK;
    HubArgs g{};
    g.N = B->N;
    g.nh = (uint32_t)H->nh;
    if (H->L > ((int64_t)1 << 20)) return HPHI_OK;
    g.ddn = (uint32_t)H->L;
    g.up_pad = (H->up_w + 7) & ~7;  // whole batches of up hops
    g.ngrp = (B->N + kHubGroup - 1) / kHubGroup;
    g.nv = H->host.n_v;
    // |U part| <= sum |U|, |V part| <= 4 sum |V|, each (or both together) below 2^e2;
    // fixed point: 2^(62 - e2) per unit, the upper 32 bits of that in 32-bit integers
    double ubound = 0.0, vbound = 0.0, hop = 0.0;
    for (int i = 0; i < B->N; i++) ubound += fabs(H->host.U[i]);
    for (int k = 0; k < g.nv; k++) vbound += 4.0 * fabs(H->host.v[k].v);
    for (int k = 0; k < H->host.n_ncoef; k++) hop = k ? std::min(hop, fabs(H->host.coef[k])) : fabs(H->host.coef[k]);
    if (!isfinite(ubound + vbound)) return HPHI_OK;
    for (int k = 0; k < H->host.n_ncoef; k++)
        if (!(fabs(H->host.coef[k]) < 1e30)) return HPHI_OK;  // FP64 hops are scaled by up to 2^122
    auto grid = [](double b) {
        int e2 = 0;
        frexp(b > 0.0 ? b : 1.0, &e2);
        return e2;
    };
    const int eu = grid(ubound), ev = grid(vbound), e2 = grid(ubound + vbound);
    if (std::min(eu, ev) < -60 || e2 > 100) return HPHI_OK;  // the scales are normal numbers in FP32 too
    // Which integers: every coupling keeps the digits that it has in the vectors' type, or
    // a grid step is at most a quarter ulp of the smallest hop, whose terms round by more
    // (a row without U in its diagonal still gets hops).  V = 0.3 next to U = 100 on 14
    // sites: off by 1.2e-6 of it on a 32-bit grid, 3e-16 on the same grid in 64 bits, 1e-18
    // on its own.  ms per product of the 7x2 ladder with V, FP32: 32 bits 0.154, 64 bits
    // 0.165, bond-major kernel 0.448; FP64: one grid 0.697, two 0.763, bond-major 1.075.
    auto keeps = [&](int eu, int ev, int bits, int digits) {
        bool ok = true;
        for (int i = 0; i < B->N; i++) ok = ok && fix_keeps(H->host.U[i], eu, bits, digits);
        for (int k = 0; k < g.nv; k++) ok = ok && fix_keeps(H->host.v[k].v, ev, bits, digits);
        return ok || ldexp(1.0, std::max(eu, ev) - bits) <= ldexp(hop, -digits - 1);
    };
    const size_t most = 222 * 1024;
    g.fix[0].parts = g.fix[1].parts = 1;
    if (keeps(e2, e2, kHubBits, 53)) {
        g.fix[1].bytes = 8;
    } else if (g.nv > 0 && keeps(eu, ev, kHubBits, 53)) {
        g.fix[1].bytes = 8;
        g.fix[1].parts = 2;
    }
    if (g.fix[1].bytes && hub_smem<double, 1>(g, H->host.n_ncoef, 8) > most) g.fix[1].bytes = 0;
    if (keeps(e2, e2, 30, 24)) g.fix[0].bytes = 4;
    else if (keeps(e2, e2, kHubBits, 24)) g.fix[0].bytes = 8;
    if (g.fix[0].bytes && hub_smem<float, 1>(g, H->host.n_ncoef, g.fix[0].bytes) > most) g.fix[0].bytes = 0;
    if (!g.fix[0].bytes && !g.fix[1].bytes) return HPHI_OK;
    std::vector<uint32_t> st[2];
    if (g.nv > 0)
        for (int s = 0; s < 2; s++) {
            st[s].resize((size_t)B->sp[s].dim);
            HPHI_CUDA(ctx, cudaMemcpy(st[s].data(), B->sp[s].states, st[s].size() * sizeof(uint32_t),
                                      cudaMemcpyDeviceToHost));
        }
    std::vector<long long> blob;  // per precision: vfix | V of one species alone, per string
    size_t at_v[2], at_s[2][2];
    for (int t = 0; t < 2; t++) {
        const bool own = g.fix[t].parts == 2;
        const int tu = own ? eu : e2, tv = own ? ev : e2;
        auto fixed = [](double v, int e) { return (long long)llrint(ldexp(v, kHubBits - e)); };
        for (int i = 0; i < B->N; i++) g.fix[t].ufix[i] = fixed(H->host.U[i], tu);
        const int bits = g.fix[t].bytes == 4 ? 30 : kHubBits;
        g.fix[t].scale = ldexp(1.0, tu - bits);
        g.fix[t].vscale = ldexp(1.0, tv - bits);
        if (g.nv == 0) continue;
        std::vector<HubV> vf;
        for (int k = 0; k < g.nv; k++) vf.push_back(HubV{H->host.v[k].i, H->host.v[k].j, fixed(H->host.v[k].v, tv)});
        at_v[t] = blob.size();
        blob.resize(at_v[t] + vf.size() * (sizeof(HubV) / sizeof(long long)));
        memcpy(blob.data() + at_v[t], vf.data(), vf.size() * sizeof(HubV));
        for (int s = 0; s < 2; s++) {
            at_s[t][s] = blob.size();
            for (uint32_t x : st[s]) {
                long long d = 0;
                for (const HubV &v : vf)
                    if (((x >> v.i) & 1u) && ((x >> v.j) & 1u)) d += v.v;
                blob.push_back(d);
            }
        }
    }
    if (g.nv > 0) {
        cudaError_t e = cudaMalloc((void **)&H->hub_tab, blob.size() * sizeof(long long));
        if (e == cudaSuccess)
            e = cudaMemcpy(H->hub_tab, blob.data(), blob.size() * sizeof(long long), cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return cuda_err(ctx, e, "Hubbard kernel tables");
        for (int t = 0; t < 2; t++) {
            g.fix[t].vfix = (const HubV *)(H->hub_tab + at_v[t]);
            g.fix[t].dup = H->hub_tab + at_s[t][0];
            g.fix[t].ddnf = H->hub_tab + at_s[t][1];
        }
    }
    H->hub = new (std::nothrow) HubArgs(g);
    if (!H->hub) return set_err(ctx, HPHI_E_NOMEM, "Hubbard kernel tables");
    return HPHI_OK;
}

template <typename T>
int launch_hub(hphi_ctx *ctx, const hphi_ham *ham, const HvArgs<T> &a, int red_mode, int *grid) {
    if (!ham->hub) return set_err(ctx, HPHI_E_INVAL, "Hubbard H*x: not available for this Hamiltonian");
    const int bytes = ham->hub->fix[sizeof(T) == 8].bytes;
    if (bytes == 8) {
        if (a.ncol == 1) return go_hub_red<T, long long, 1>(ctx, ham, a, red_mode, grid);
        return go_hub_red<T, long long, 2>(ctx, ham, a, red_mode, grid);
    }
    if constexpr (sizeof(T) == 4) {
        if (bytes == 4 && a.ncol == 1) return go_hub_red<T, int, 1>(ctx, ham, a, red_mode, grid);
        if (bytes == 4) return go_hub_red<T, int, 2>(ctx, ham, a, red_mode, grid);
    }
    return set_err(ctx, HPHI_E_INVAL, "Hubbard H*x: not available for this Hamiltonian");
}

template int launch_hub<float>(hphi_ctx *, const hphi_ham *, const HvArgs<float> &, int, int *);
template int launch_hub<double>(hphi_ctx *, const hphi_ham *, const HvArgs<double> &, int, int *);

}  // namespace hphi
