// The Krylov side of one step: the BSR SpMV and the GMRES / ORTHOMIN vector and state kernels
// (modified Gram-Schmidt Arnoldi with Givens rotations, and ORTHOMIN(k) projections, Section 2).
// Every kernel reads its system's control words, so systems at different points of their solve
// share the same launches.
#include <algorithm>
#include <cooperative_groups.h>

#include "asm2_internal.h"

namespace asm2 {

namespace {

// ------------------------------------------------------------------------------------------
// SpMV y = A x or y = b - A x (ELL, one thread per block row, 3x3 blocks).  Bound by the FP64 unit (63 FMAs a
// row of seven blocks: 105 us at a million rows) and by HBM (85 us) at once, so the next block's values and x are
// requested before the arithmetic of this one, and the column after that; the values are read once (streaming
// loads).  With the loads of a block after the arithmetic of the last, 256 threads and 64 registers: 148.9 us a
// launch at 128 x 128 x 64 (0.71 of the FP64 rate), now 129.5 (0.81); 97 x 83 x 29 46 -> 38 us, 64 x 64 x 16
// 22 -> 16.4, 10 x 10 x 5 12.3 -> 10.2 (with the gaps between events).  256 threads and three CTAs per SM: 133.7.
// ------------------------------------------------------------------------------------------
constexpr int kSpmvThreads = 128;

__global__ void __launch_bounds__(kSpmvThreads, 6) k_spmv(const SysTab* __restrict__ tab, const RowItem* __restrict__ items) {
    constexpr int per = 256 / kSpmvThreads;  // CTAs per item of 256 rows
    const RowItem it = items[blockIdx.x / per];
    const SysTab& st = tab[it.sys];
    const int in = st.ctl[C_SPMV_IN];
    if (in < 0) return;
    const int row = it.r0 + kSpmvThreads * (blockIdx.x % per) + threadIdx.x;
    if (row >= st.n_cells) return;
    const int out = st.ctl[C_SPMV_OUT];
    const int bs = st.ctl[C_SPMV_B];
    const double* __restrict__ x = st.ws + (long long)in * st.n3p;
    double* __restrict__ y = st.ws + (long long)out * st.n3p;
    const long long rp = st.rows_pad;
    const int W = st.ell_w;
    const int* __restrict__ cp = st.ell_col + row;
    const double* __restrict__ vp = st.ell_val + row;
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    double v[2][9], xx[2][3];
    int c1 = 0;
    const auto load = [&](int h, int c, const double* q) {
#pragma unroll
        for (int k = 0; k < 9; k++) v[h][k] = __ldcs(q + k * rp);
        xx[h][0] = x[3LL * c], xx[h][1] = x[3LL * c + 1], xx[h][2] = x[3LL * c + 2];
    };
    // one FMA per product into the running sums: an FP64 instruction costs a warp ~64 cycles
    // here, and a separate product-then-add form would take four per three products
    const auto mac = [&](int h) {
        a0 = fma(v[h][2], xx[h][2], fma(v[h][1], xx[h][1], fma(v[h][0], xx[h][0], a0)));
        a1 = fma(v[h][5], xx[h][2], fma(v[h][4], xx[h][1], fma(v[h][3], xx[h][0], a1)));
        a2 = fma(v[h][8], xx[h][2], fma(v[h][7], xx[h][1], fma(v[h][6], xx[h][0], a2)));
    };
    if (W > 0) {
        const int c0 = cp[0];
        c1 = W > 1 ? cp[rp] : 0;
        load(0, c0, vp);
    }
    for (int w = 0; w < W; w += 2) {
        if (w + 1 < W) {
            const int c = c1;
            if (w + 2 < W) c1 = cp[(w + 2) * rp];
            load(1, c, vp + (w + 1) * 9 * rp);
        }
        mac(0);
        if (w + 1 < W) {
            if (w + 2 < W) {
                const int c = c1;
                if (w + 3 < W) c1 = cp[(w + 3) * rp];
                load(0, c, vp + (w + 2) * 9 * rp);
            }
            mac(1);
        }
    }
    if (bs >= 0) {
        const double* b = st.ws + (long long)bs * st.n3p;
        a0 = b[3LL * row] - a0;
        a1 = b[3LL * row + 1] - a1;
        a2 = b[3LL * row + 2] - a2;
    }
    y[3LL * row] = a0;
    y[3LL * row + 1] = a1;
    y[3LL * row + 2] = a2;
}

// ------------------------------------------------------------------------------------------
// GMRES vector kernels.  A chunk is a work item of one system (vec_item_len elements); reductions write one
// partial per chunk and the last chunk to arrive sums the partials in index order, so every
// result is independent of scheduling and of the other systems in the launch.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ double* vec(const SysTab& st, int slot) { return st.ws + (long long)slot * st.n3p; }

__device__ __forceinline__ int zslot(const SysTab& st, int k) { return VV0 + st.m + 1 + k; }

// block sum of two values; result valid in thread 0.  The 256 partials go through shared memory
// and one warp reduces them (8 sequential adds + a 5-round tree): FP64 adds are scarce here, so
// this issues ~4x fewer of them than a shuffle tree in every warp.
__device__ __forceinline__ void block_sum2(double& a, double& b) {
    __shared__ double s0[VEC_THREADS], s1[VEC_THREADS];
    s0[threadIdx.x] = a;
    s1[threadIdx.x] = b;
    __syncthreads();
    if (threadIdx.x < 32) {
        double x = 0.0, y = 0.0;
        for (int i = threadIdx.x; i < (int)blockDim.x; i += 32) {
            x += s0[i];
            y += s1[i];
        }
        for (int o = 16; o > 0; o >>= 1) {
            x += __shfl_down_sync(0xffffffffu, x, o);
            y += __shfl_down_sync(0xffffffffu, y, o);
        }
        a = x;
        b = y;
    }
    __syncthreads();
}

// single-value form of block_sum2 (the same summation order for that value)
__device__ __forceinline__ void block_sum1(double& a) {
    __shared__ double s0[VEC_THREADS];
    s0[threadIdx.x] = a;
    __syncthreads();
    if (threadIdx.x < 32) {
        double x = 0.0;
        for (int i = threadIdx.x; i < (int)blockDim.x; i += 32) x += s0[i];
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
        a = x;
    }
    __syncthreads();
}

// Publish this chunk's partials; returns true in thread 0.. of the last chunk of its system,
// with (s0, s1) = the ordered total.
__device__ bool finish_reduction(const SysTab& st, int chunk, double& s0, double& s1) {
    __shared__ bool last;
    block_sum2(s0, s1);
    if (threadIdx.x == 0) {
        st.partial[2 * chunk] = s0;
        st.partial[2 * chunk + 1] = s1;
        __threadfence();
        const int prev = atomicAdd(&st.ctl[C_CNT_RED], 1);
        last = (prev == st.nchunk - 1);
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < st.nchunk; i += blockDim.x) {
        a += __ldcg(&st.partial[2 * i]);
        b += __ldcg(&st.partial[2 * i + 1]);
    }
    block_sum2(a, b);
    s0 = a;
    s1 = b;
    if (threadIdx.x == 0) st.ctl[C_CNT_RED] = 0;
    return true;
}

__global__ void k_gather_ctl(const SysTab* __restrict__ tab, int* __restrict__ out) {
    if (threadIdx.x < C_NCTL) out[blockIdx.x * C_NCTL + threadIdx.x] = tab[blockIdx.x].ctl[threadIdx.x];
}

__global__ void __launch_bounds__(VEC_THREADS) k_init(const SysTab* __restrict__ tab, const VecItem* __restrict__ items) {
    const VecItem it = items[blockIdx.x];
    const SysTab& st = tab[it.sys];
    if (st.ctl[C_PHASE] != PH_INIT) return;
    double* x = vec(st, VX);
    const double* b = vec(st, VB);
    double* r = vec(st, VR);
    const long long e0 = (long long)it.chunk * st.vchunk;
    for (int i = threadIdx.x; i < st.vchunk; i += blockDim.x) {
        x[e0 + i] = 0.0;
        r[e0 + i] = b[e0 + i];
    }
}

// restart phase: u = V y (then u goes through B^{-1}), or x += Z y (flexible)
__global__ void __launch_bounds__(VEC_THREADS) k_prep(const SysTab* __restrict__ tab, const VecItem* __restrict__ items) {
    const VecItem it = items[blockIdx.x];
    const SysTab& st = tab[it.sys];
    if (st.ctl[C_PHASE] != PH_RESTART) return;
    const int jend = st.ctl[C_JEND];
    const ScalLayout SL = ScalLayout::make(st.m);
    const double* yv = st.scal + SL.y;
    const long long e0 = (long long)it.chunk * st.vchunk;
    double* dst = st.flexible ? vec(st, VX) : vec(st, VU);
    for (int i = threadIdx.x; i < st.vchunk; i += blockDim.x) {
        double acc = st.flexible ? dst[e0 + i] : 0.0;
        for (int k = 0; k < jend; k++) acc += yv[k] * vec(st, st.flexible ? zslot(st, k) : VV0 + k)[e0 + i];
        dst[e0 + i] = acc;
    }
}

// restart phase (non-flexible): x += z
__global__ void __launch_bounds__(VEC_THREADS) k_post(const SysTab* __restrict__ tab, const VecItem* __restrict__ items) {
    const VecItem it = items[blockIdx.x];
    const SysTab& st = tab[it.sys];
    if (st.ctl[C_PHASE] != PH_RESTART || st.flexible) return;
    double* x = vec(st, VX);
    const double* z = vec(st, VZ);
    const long long e0 = (long long)it.chunk * st.vchunk;
    for (int i = threadIdx.x; i < st.vchunk; i += blockDim.x) x[e0 + i] += z[e0 + i];
}

// ------------------------------------------------------------------------------------------
// Blocked modified Gram-Schmidt.  Modified Gram-Schmidt takes each coefficient h_k = (w, v_k) from
// the w that all earlier projections have already been subtracted from, so by itself it needs a
// global reduction per basis vector.  Within a block of vectors the same coefficients follow from
// the inner products with the block's first w and the block's Gram matrix:
//   h_k = (w, v_k) - sum_{i in block, i < k} (v_k, v_i) h_i,
// a forward substitution with the unit lower triangle of V^T V (the low-synchronisation form of
// modified Gram-Schmidt of Swirydowicz, Langou, Ananthan, Yang and Thomas, 2021, whose loss of
// orthogonality is that of modified Gram-Schmidt).  The Gram entries are of the size of the loss
// of orthogonality; v_j's row is taken at step j, in the same sweep as (w, v_i), and kept.  One
// reduction per block of st.gs_block vectors replaces one per vector.
//
// Two block sizes (gs_block_size): a whole restart cycle of up to kGsMaxBlock vectors in one
// block costs half as many multiply-adds again (every (v_j, v_i) of the cycle), which short vectors
// do not notice; long vectors, bound by the FP64 pipe, take blocks of kGsGroup (batches) or
// kGsLong (the cooperative kernel).
// ------------------------------------------------------------------------------------------
template <int W>
__device__ __forceinline__ void load_w(const double* p, double (&x)[W]) {
    if constexpr (W == 2) {
        const double2 t = *reinterpret_cast<const double2*>(p);
        x[0] = t.x;
        x[1] = t.y;
    } else {
        x[0] = p[0];
    }
}
template <int W>
__device__ __forceinline__ void store_w(double* p, const double (&x)[W]) {
    if constexpr (W == 2)
        *reinterpret_cast<double2*>(p) = make_double2(x[0], x[1]);
    else
        p[0] = x[0];
}

// One sweep over the elements [e0, e1) of this CTA (W per thread and iteration):
//   w -= sum_{i < np} hp[i] vp_i   (vp = the vectors from slot prev on; np = 0: w is left alone)
//   acc[d] += (w, v_{nxt + d}), d < nn <= kGsGroup
//   acc[kGsGroup + d] += (v_j, v_{nxt + d}), d < ng   (v_j at slot jslot)
//   ww += (w, w) when NORM
template <int W, bool NORM>
__device__ __forceinline__ void gs_sweep(const SysTab& st, long long e0, long long e1, int prev, int np,
                                         const double* hp, int nxt, int nn, int ng, int jslot, double (&acc)[16],
                                         double& ww) {
    double* w = vec(st, VW);
    const double* vp = vec(st, prev);
    const double* vn = vec(st, nxt);
    const double* vj = vec(st, jslot);
    const long long n = st.n3p;
    constexpr int kL = W == 2 ? 4 : kGsGroup;  // vectors loaded together (registers)
#pragma unroll 1
    for (long long e = e0 + W * threadIdx.x; e < e1; e += W * VEC_THREADS) {
        double x[W], y[W];
        load_w<W>(w + e, x);
        if (ng > 0) load_w<W>(vj + e, y);
#pragma unroll 1
        for (int i0 = 0; i0 < np; i0 += kL) {
            double c[kL][W];
#pragma unroll
            for (int d = 0; d < kL; d++)
                if (i0 + d < np) load_w<W>(vp + (i0 + d) * n + e, c[d]);
#pragma unroll
            for (int d = 0; d < kL; d++)
                if (i0 + d < np) {
                    const double h = hp[i0 + d];
#pragma unroll
                    for (int u = 0; u < W; u++) x[u] = fma(-h, c[d][u], x[u]);
                }
        }
        if (np > 0) store_w<W>(w + e, x);
#pragma unroll
        for (int d0 = 0; d0 < kGsGroup; d0 += kL) {
            if (d0 >= nn) break;
            double b[kL][W];
#pragma unroll
            for (int d = 0; d < kL; d++)
                if (d0 + d < nn) load_w<W>(vn + (d0 + d) * n + e, b[d]);
#pragma unroll
            for (int d = 0; d < kL; d++)
                if (d0 + d < nn)
#pragma unroll
                    for (int u = 0; u < W; u++) acc[d0 + d] = fma(x[u], b[d][u], acc[d0 + d]);
#pragma unroll
            for (int d = 0; d < kL; d++)
                if (d0 + d < ng)
#pragma unroll
                    for (int u = 0; u < W; u++)
                        acc[kGsGroup + d0 + d] = fma(y[u], b[d][u], acc[kGsGroup + d0 + d]);
        }
        if constexpr (NORM)
#pragma unroll
            for (int u = 0; u < W; u++) ww = fma(x[u], x[u], ww);
    }
}

// The CTA's sums of N (4, 8 or 16) values per thread: value q valid in thread q < N.  Within a warp the
// values are halved as the lanes are (N adds and one more per spare lane bit, against 5 N for a
// shuffle tree per value: an FP64 add holds a sub-partition's FP64 unit for ~64 cycles); the eight
// warps' results are added in index order.  All threads call it; sm holds 8 * 16 doubles.
// The lanes that hold the same value all store it: with the store under a condition on the lane, nvcc 13.0 lost
// warp 0's share of a sum once a loop around this function was unrolled (up to four groups, the third with one vector).
template <int N>
__device__ __forceinline__ double cta_sums(double (&v)[16], double* sm) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int c = N, o = 16;
#pragma unroll
    for (int step = 0; step < 4; step++) {
        if (c == 1) break;
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < N / 2; i++)
            if (i < c / 2) {
                const double keep = up ? v[i + c / 2] : v[i], send = up ? v[i] : v[i + c / 2];
                v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        c >>= 1;
        o >>= 1;
    }
    for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    constexpr int kRep = 32 / N;  // lanes that hold the same value
    __syncthreads();
    sm[16 * warp + lane / kRep] = v[0];
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x < N) {
#pragma unroll
        for (int k = 0; k < VEC_THREADS / 32; k++) t += sm[16 * k + threadIdx.x];
    }
    return t;
}

// Sums of a block's values over its nparts partials, into tot[]: values 0 .. nd - 1 (the dots) and
// nd .. nd + ng - 1 (the Gram row, from row bs on) and, last, (w, w) (row 2 bs) when ww.  Value q's
// partials are at part[row(q) * rs + k * ks].  A power-of-two group of lanes per value.
__device__ __forceinline__ void gs_totals(const double* part, long long rs, long long ks, int nparts, int nd, int ng, bool ww,
                                          int bs, double* tot) {
    const int nv = nd + ng + (ww ? 1 : 0);
    const int tpv = nv <= 8 ? 32 : nv <= 16 ? 16 : nv <= 32 ? 8 : 4;
    const int per = VEC_THREADS / tpv, sub = threadIdx.x & (tpv - 1);
    for (int q0 = 0; q0 < nv; q0 += per) {
        const int q = q0 + (int)threadIdx.x / tpv;
        double a = 0.0;
        if (q < nv) {
            const double* p = part + (q < nd ? q : q < nd + ng ? bs + q - nd : 2 * bs) * rs;
            int k = sub;
            for (; k + 3 * tpv < nparts; k += 4 * tpv) {
                const double l0 = __ldcg(p + k * ks), l1 = __ldcg(p + (k + tpv) * ks), l2 = __ldcg(p + (k + 2 * tpv) * ks),
                             l3 = __ldcg(p + (k + 3 * tpv) * ks);
                a += (l0 + l1) + (l2 + l3);
            }
            for (; k < nparts; k += tpv) a += __ldcg(p + k * ks);
        }
        for (int o = tpv >> 1; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
        if (sub == 0 && q < nv) tot[q] = a;
    }
}

// h_lo .. h_{hi-1} of a block from its dots tot[0 ..] (forward substitution with the Gram rows; the
// last block's last vector is v_j, whose row follows the dots in tot).  gram: the kept rows
// (kGsMaxBlock per vector, entry i - lo), from row lo on.  Warp 0 of the CTA; h into hs[0 ..].
__device__ __forceinline__ void gs_substitute(const double* tot, int nd, int ng, const double* gram, double* hs) {
    const int lane = threadIdx.x & 31;
    double c = lane < nd ? tot[lane] : 0.0;
    const double* row = ng > 0 && lane == nd - 1 ? tot + nd : gram + (long long)lane * kGsMaxBlock;
    for (int k = 0; k + 1 < nd; k++) {
        const double h = __shfl_sync(0xffffffffu, c, k);
        if (lane > k && lane < nd) c = fma(-row[k], h, c);
    }
    if (lane < nd) hs[lane] = c;
}

// Pass b of a step of the batched path: subtract block b - 1's projections, then block b's
// coefficients (b < number of blocks) or ||w||; pass 0 also gives ||w|| before orthogonalisation.
// Restart/init systems compute beta = ||r|| at pass 0.  The last chunk of a system to arrive adds
// the chunks' partials up.
__global__ void __launch_bounds__(VEC_THREADS, 2) k_mgs(const SysTab* __restrict__ tab, const VecItem* __restrict__ items,
                                                        int b) {
    const VecItem it = items[blockIdx.x];
    const SysTab& st = tab[it.sys];
    if (st.krylov != 0) return;
    const int ph = st.ctl[C_PHASE];
    const ScalLayout SL = ScalLayout::make(st.m);
    const long long e0 = (long long)it.chunk * st.vchunk, e1 = e0 + st.vchunk;
    if (ph == PH_ARNOLDI) {
        __shared__ double hp[kGsMaxBlock], sm[8 * 16], tot[2 * kGsMaxBlock + 1], hs[kGsMaxBlock];
        __shared__ bool last;
        const int j = st.ctl[C_J], bs = st.gs_block, m = st.m;
        const int lo = b * bs, plo = lo - bs;
        if (plo > j) return;
        const int np = b > 0 ? min(bs, j + 1 - plo) : 0;
        const int nd = max(0, min(bs, j + 1 - lo));
        const bool fin = nd == 0, lastb = lo + nd == j + 1;
        const int ngram = !fin && lastb ? nd - 1 : 0;
        if ((int)threadIdx.x < np) hp[threadIdx.x] = st.scal[SL.H + (plo + threadIdx.x) * m + j];
        __syncthreads();
        const int rows = 2 * bs + 1;
        double* part = st.partial + (long long)it.chunk * rows;
#pragma unroll 1
        for (int g0 = 0; g0 < max(1, nd); g0 += kGsGroup) {
            double acc[16], ww = 0.0;
#pragma unroll
            for (int q = 0; q < 16; q++) acc[q] = 0.0;
            const int nn = max(0, min(kGsGroup, nd - g0)), ng = max(0, min(kGsGroup, ngram - g0));
            const int p = g0 == 0 ? np : 0;
            if (g0 == 0 && (b == 0 || fin))
                gs_sweep<2, true>(st, e0, e1, VV0 + max(0, plo), p, hp, VV0 + lo, nn, ng, VV0 + j, acc, ww);
            else
                gs_sweep<2, false>(st, e0, e1, VV0 + max(0, plo), p, hp, VV0 + lo + g0, nn, ng, VV0 + j, acc, ww);
            if (!fin) {
                if (ng > 0) {
                    const double t = cta_sums<16>(acc, sm);
                    if ((int)threadIdx.x < nn) part[g0 + threadIdx.x] = t;
                    if ((int)threadIdx.x >= kGsGroup && (int)threadIdx.x < kGsGroup + ng)
                        part[bs + g0 + threadIdx.x - kGsGroup] = t;
                } else {
                    const double t = cta_sums<8>(acc, sm);
                    if ((int)threadIdx.x < nn) part[g0 + threadIdx.x] = t;
                }
            }
            if (g0 == 0 && (b == 0 || fin)) {
                block_sum1(ww);
                if (threadIdx.x == 0) part[2 * bs] = ww;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            last = atomicAdd(&st.ctl[C_CNT_RED], 1) == st.nchunk - 1;
        }
        __syncthreads();
        if (!last) return;
        __threadfence();
        if (threadIdx.x == 0) st.ctl[C_CNT_RED] = 0;
        gs_totals(st.partial, 1, rows, st.nchunk, nd, ngram, b == 0 || fin, bs, tot);
        __syncthreads();
        double* gram = st.scal + SL.gram;
        if (fin) {
            if (threadIdx.x == 0) {
                const double hn = sqrt(tot[0]);
                st.scal[SL.hn] = hn;
                st.scal[SL.H + (j + 1) * m + j] = hn;
            }
            return;
        }
        if (threadIdx.x < 32) {
            gs_substitute(tot, nd, ngram, gram + (long long)lo * kGsMaxBlock, hs);
            const int t = threadIdx.x;
            if (t < nd) st.scal[SL.H + (lo + t) * m + j] = hs[t];
            if (t < ngram) gram[(long long)j * kGsMaxBlock + t] = tot[nd + t];
            if (t == 0 && b == 0) st.scal[SL.w0] = sqrt(tot[nd + ngram]);
        }
    } else if (ph == PH_RESTART || ph == PH_INIT) {
        if (b != 0) return;
        const double* r = vec(st, VR);
        double s0 = 0.0, s1 = 0.0;
        for (int i = threadIdx.x; i < st.vchunk; i += blockDim.x) s0 = fma(r[e0 + i], r[e0 + i], s0);
        if (!finish_reduction(st, it.chunk, s0, s1)) return;
        if (threadIdx.x == 0) st.scal[SL.beta] = sqrt(s0);
    }
}

__device__ void set_slots(const SysTab& st, int ph, int j) {
    int* c = st.ctl;
    if (ph == PH_ARNOLDI) {
        c[C_APPLY_IN] = VV0 + j;
        c[C_APPLY_OUT] = st.flexible ? zslot(st, j) : VZ;
        c[C_SPMV_IN] = c[C_APPLY_OUT];
        c[C_SPMV_OUT] = VW;
        c[C_SPMV_B] = -1;
    } else if (ph == PH_RESTART) {
        c[C_APPLY_IN] = st.flexible ? -1 : VU;
        c[C_APPLY_OUT] = VZ;
        c[C_SPMV_IN] = VX;
        c[C_SPMV_OUT] = VR;
        c[C_SPMV_B] = VB;
    } else {
        c[C_APPLY_IN] = -1;
        c[C_SPMV_IN] = -1;
    }
}

// Givens rotation of column j and the GMRES state machine of one system, by one warp (all lanes
// call it with the same arguments).  Every FP64 operation takes ~85 cycles here and every global
// load more, so the operands are loaded by the lanes together and only the recurrences run in order:
// one multiply-add per earlier rotation, and in the back substitution a division and a multiply-add
// per column.
__device__ void step_state(const SysTab& st, int ph) {
    const ScalLayout SL = ScalLayout::make(st.m);
    const int m = st.m, lane = threadIdx.x & 31;
    constexpr unsigned kAll = 0xffffffffu;
    int* c = st.ctl;
    double* s = st.scal;
    double* H = s + SL.H;
    if (ph == PH_ARNOLDI) {
        const int j = c[C_J], iters = c[C_ITERS] + 1, maxit = c[C_MAXIT];
        const double hn = s[SL.hn], w0 = s[SL.w0], tol = s[SL.tol], bnorm = s[SL.bnorm], gj = s[SL.g + j];
        // H[k], H[k+1] <- rotation k of them: t is the running H[k]
        double t = H[j];
        for (int k0 = 0; k0 < j; k0 += 32) {
            const int k = k0 + lane;
            double ck = 1.0, sk = 0.0, hk = 0.0, tk = 0.0;
            if (k < j) {
                ck = s[SL.cs + k];
                sk = s[SL.sn + k];
                hk = H[(k + 1) * m + j];
            }
            const double up = ck * hk;
            const int nk = min(32, j - k0);
            for (int i = 0; i < nk; i++) {
                if (lane == i) tk = t;
                t = fma(-__shfl_sync(kAll, sk, i), t, __shfl_sync(kAll, up, i));
            }
            if (k < j) H[k * m + j] = fma(ck, tk, sk * hk);
        }
        const double b = hn, rr = hypot(t, b);  // (t, b) = H[j], H[j+1] of this column
        double cs = 1.0, sn = 0.0;
        if (rr != 0.0) {
            cs = t / rr;
            sn = b / rr;
        }
        const double gn = -sn * gj;
        const bool breakdown = hn <= 1e-14 * w0;
        const bool small = fabs(gn) <= tol * bnorm;
        const bool stop = small || breakdown || iters >= maxit || j + 1 == m;
        __syncwarp();
        if (lane == 0) {
            s[SL.cs + j] = cs;
            s[SL.sn + j] = sn;
            H[j * m + j] = cs * t + sn * b;
            H[(j + 1) * m + j] = 0.0;
            s[SL.g + j + 1] = gn;
            s[SL.g + j] = cs * gj;
            c[C_ITERS] = iters;
            if (breakdown) c[C_BREAKDOWN] = 1;
            if (stop) {
                c[C_JEND] = j + 1;
                c[C_PHASE] = PH_RESTART;
                set_slots(st, PH_RESTART, 0);
            } else {
                c[C_J] = j + 1;
                set_slots(st, PH_ARNOLDI, j + 1);
            }
        }
        __syncwarp();
        if (stop) {  // y = H^{-1} g, last column first; lane k holds y_k of each 32 rows
            const int jend = j + 1;
            for (int r0 = (jend - 1) / 32 * 32; r0 >= 0; r0 -= 32) {
                const int r = r0 + lane, nr = min(32, jend - r0);
                double acc = 0.0, d = 1.0;
                if (r < jend) {
                    acc = s[SL.g + r];
                    d = H[r * m + r];
                    for (int l = jend - 1; l >= r0 + 32; l--) acc = fma(-H[r * m + l], s[SL.y + l], acc);
                }
                for (int k = nr - 1; k >= 0; k--) {
                    const double yk = __shfl_sync(kAll, acc / d, k);
                    const double h = r < r0 + k ? H[r * m + r0 + k] : 0.0;
                    if (lane == k) acc = yk;
                    else if (lane < k) acc = fma(-h, yk, acc);
                    if (lane == k) d = 1.0;
                }
                if (r < jend) s[SL.y + r] = acc;
                __syncwarp();
            }
        }
        return;
    }
    if (lane != 0) return;
    const double beta = s[SL.beta];
    if (ph == PH_INIT) {
        s[SL.bnorm] = beta;
        if (beta == 0.0) {
            c[C_CONVERGED] = 1;
            c[C_STATUS] = 0;
            c[C_PHASE] = PH_DONE;
            set_slots(st, PH_DONE, 0);
            return;
        }
    } else {
        c[C_RESTARTS] += 1;
    }
    const double rel = beta / s[SL.bnorm];
    if (rel <= s[SL.tol]) {
        c[C_CONVERGED] = 1;
        c[C_STATUS] = 0;
        c[C_PHASE] = PH_DONE;
        set_slots(st, PH_DONE, 0);
    } else if (c[C_ITERS] >= c[C_MAXIT] || beta == 0.0) {
        c[C_STATUS] = 4;  // ASM_ERR_NOT_CONVERGED
        c[C_PHASE] = PH_DONE;
        set_slots(st, PH_DONE, 0);
    } else {
        for (int k = 0; k <= m; k++) s[SL.g + k] = 0.0;
        s[SL.g] = beta;
        c[C_J] = 0;
        c[C_PHASE] = PH_ARNOLDI;
        set_slots(st, PH_ARNOLDI, 0);
    }
}


// End of a step: vector scaling (v_{j+1} = w / h_{j+1,j}, or v_0 = r / beta), then the last chunk
// of each system applies the Givens rotations and moves its state machine.
__global__ void __launch_bounds__(VEC_THREADS) k_finish(const SysTab* __restrict__ tab,
                                                        const VecItem* __restrict__ items) {
    const VecItem it = items[blockIdx.x];
    const SysTab& st = tab[it.sys];
    const int ph = st.ctl[C_PHASE];
    if (ph == PH_DONE || st.krylov != 0) return;
    const ScalLayout SL = ScalLayout::make(st.m);
    const long long e0 = (long long)it.chunk * st.vchunk;
    if (ph == PH_ARNOLDI) {
        const int j = st.ctl[C_J];
        const double hn = st.scal[SL.hn];
        if (hn > 0.0) {
            const double inv = 1.0 / hn;
            const double* w = vec(st, VW);
            double* v = vec(st, VV0 + j + 1);
            for (int i = threadIdx.x; i < st.vchunk; i += blockDim.x) v[e0 + i] = w[e0 + i] * inv;
        }
    } else {
        const double beta = st.scal[SL.beta];
        if (beta > 0.0) {
            const double inv = 1.0 / beta;
            const double* r = vec(st, VR);
            double* v = vec(st, VV0);
            for (int i = threadIdx.x; i < st.vchunk; i += blockDim.x) v[e0 + i] = r[e0 + i] * inv;
        }
    }
    __shared__ bool last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&st.ctl[C_CNT_FIN], 1) == st.nchunk - 1;
    }
    __syncthreads();
    if (!last || threadIdx.x >= 32) return;
    __threadfence();
    if (threadIdx.x == 0) st.ctl[C_CNT_FIN] = 0;
    step_state(st, ph);
}

// ------------------------------------------------------------------------------------------
// ORTHOMIN(k) (Section 2): the new direction p = B^{-1} r, q = A p is A-orthogonalised against the
// k most recent directions (newest first, each projection on the q already updated), then
// alpha = (r, q) / (q, q), x += alpha p, r -= alpha q.  The directions sit in a ring of k + 1
// slots: P_s = VV0 + s, Q_s = VV0 + k + 1 + s.
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ int om_p(const SysTab& st, int s) { return VV0 + s; }
__device__ __forceinline__ int om_q(const SysTab& st, int s) { return VV0 + st.m + 1 + s; }

__device__ void om_set_slots(const SysTab& st, int ph) {
    int* c = st.ctl;
    if (ph == PH_OM) {
        const int s = c[C_OM_SLOT];
        c[C_APPLY_IN] = VR;
        c[C_APPLY_OUT] = om_p(st, s);
        c[C_SPMV_IN] = om_p(st, s);
        c[C_SPMV_OUT] = om_q(st, s);
        c[C_SPMV_B] = -1;
    } else if (ph == PH_OM_FINAL) {
        c[C_APPLY_IN] = -1;
        c[C_SPMV_IN] = VX;
        c[C_SPMV_OUT] = VW;
        c[C_SPMV_B] = VB;
    } else {
        c[C_APPLY_IN] = -1;
        c[C_SPMV_IN] = -1;
    }
}

// ORTHOMIN state machine of one system (one thread).  nrm = ||r|| (initial and after an update)
// or ||b - A x|| (final).
__device__ void om_state(const SysTab& st, int ph, double nrm) {
    const ScalLayout SL = ScalLayout::make(st.m);
    int* c = st.ctl;
    double* s = st.scal;
    int next = PH_OM;
    if (ph == PH_INIT) {
        s[SL.bnorm] = nrm;
        s[SL.beta] = nrm;
        if (nrm == 0.0) {
            c[C_CONVERGED] = 1;
            c[C_STATUS] = 0;
            next = PH_DONE;
        } else {
            c[C_OM_STORED] = 0;
            c[C_OM_SLOT] = 0;
        }
    } else if (ph == PH_OM) {
        c[C_ITERS] += 1;
        if (c[C_OM_STORED] < st.m) c[C_OM_STORED] += 1;
        if (nrm <= s[SL.tol] * s[SL.bnorm] || c[C_ITERS] >= c[C_MAXIT])
            next = PH_OM_FINAL;
        else
            c[C_OM_SLOT] = (c[C_OM_SLOT] + 1) % (st.m + 1);
    } else {  // PH_OM_FINAL
        s[SL.beta] = nrm;
        const bool conv = nrm <= s[SL.tol] * s[SL.bnorm];
        c[C_CONVERGED] = conv ? 1 : 0;
        c[C_STATUS] = conv ? 0 : 4;  // ASM_ERR_NOT_CONVERGED
        next = PH_DONE;
    }
    c[C_PHASE] = next;
    om_set_slots(st, next);
}

// Pass b of a direction step: the projections of block b - 1 are applied (p -= beta_l P_l, q -= beta_l Q_l, l the
// l-th most recent stored direction, block b holding l = 32 b + 1 .. 32 b + 32), then the next block's coefficients
// or, after the last block, (q, q) and (r, q).  Each beta_l belongs to the q that the projections before it have
// already been subtracted from; within a block it follows from the products with the block's first q,
//   beta_l = ((q, Q_l) - sum_{l' < l in block} beta_l' (Q_l', Q_l)) / (Q_l, Q_l),
// so a block takes one reduction instead of one per direction.  The products (Q_l', Q_l) of directions less than a
// block apart are kept: the newest direction's are taken in pass 0 of the step after its own, in the sweep that
// reads the same vectors.  What bounded a step was its serial launches: at 30x30x9, k = 30, up to 31 of 15 us are
// now three, and a solve of 29 steps takes 5.1 ms instead of 9.2.
// MINB: CTAs per SM that the registers are limited for (0: no limit, 156 registers).  Launches of more CTAs than SMs
// take two (128 registers, 32 bytes spilled): they are bound by the FP64 unit, which eight warps
// alone do not keep busy.  128 x 128 x 64 FP32, a solve with k = 5: 79.5 ms with one, 71.2 with two (77.5 with a launch per
// direction); k = 30 76.9 and 65.5; two systems of 64 x 64 x 48, k = 30 17.0 and 15.3.  Where one CTA per SM is all
// there is, the limit costs: 64 x 64 x 48 alone 11.6 and 12.2.
template <int MINB>
__global__ void __launch_bounds__(VEC_THREADS, MINB) k_om(const SysTab* __restrict__ tab,
                                                          const VecItem* __restrict__ items, int b) {
    const VecItem it = items[blockIdx.x];
    const SysTab& st = tab[it.sys];
    if (st.krylov != 1) return;
    const int ph = st.ctl[C_PHASE];
    const long long e0 = (long long)it.chunk * st.vchunk, e1 = e0 + st.vchunk;
    const ScalLayout SL = ScalLayout::make(st.m);
    if (ph == PH_OM) {
        constexpr int W = 2, kB = kGsMaxBlock, kL = 4, kRows = 2 * kB + 1;
        __shared__ double hp[kB], sm[8 * 16], tot[kRows];
        __shared__ long long prev_at[kB], next_at[kB];  // offsets of Q_l of the previous and of the next block
        __shared__ bool last;
        const int stored = st.ctl[C_OM_STORED], K1 = st.m + 1, slot = st.ctl[C_OM_SLOT];
        const int lo = 1 + kB * b, plo = lo - kB;
        if (plo > stored) return;
        const int np = b > 0 ? min(kB, stored + 1 - plo) : 0, nd = max(0, min(kB, stored + 1 - lo));
        const int ngram = b == 0 ? max(0, nd - 1) : 0;  // (Q_1, Q_l), l = 2 ..
        const bool fin = nd == 0;
        const auto dir = [&](int l) { return (slot - l + K1) % K1; };
        double* p = vec(st, om_p(st, slot));
        double* q = vec(st, om_q(st, slot));
        const double* newest = vec(st, om_q(st, dir(1)));
        const double* r = vec(st, VR);
        if ((int)threadIdx.x < np) {
            hp[threadIdx.x] = st.scal[SL.om_beta + plo - 1 + threadIdx.x];
            prev_at[threadIdx.x] = om_q(st, dir(plo + threadIdx.x)) * st.n3p;
        }
        if ((int)threadIdx.x < nd) next_at[threadIdx.x] = om_q(st, dir(lo + threadIdx.x)) * st.n3p;
        const double* ws = st.ws;
        const long long p_of_q = (long long)(om_p(st, 0) - om_q(st, 0)) * st.n3p;  // from Q_s to P_s
        __syncthreads();
        double* part = st.partial + (long long)it.chunk * kRows;
#pragma unroll 1
        for (int g0 = 0; g0 < max(1, nd); g0 += kGsGroup) {
            const int nn = min(kGsGroup, nd - g0), ng = max(0, min(kGsGroup, 1 + ngram - g0));  // (entry 0: (Q_1, Q_1))
            double acc[16], qq = 0.0, rq = 0.0;
#pragma unroll
            for (int k = 0; k < 16; k++) acc[k] = 0.0;
#pragma unroll 1
            for (long long e = e0 + W * threadIdx.x; e < e1; e += W * VEC_THREADS) {
                double x[W], y[W];
                load_w<W>(q + e, x);
                if (g0 == 0 && np > 0) {
                    double t[W];
                    load_w<W>(p + e, t);
#pragma unroll 1
                    for (int i0 = 0; i0 < np; i0 += kL) {
                        double cp[kL][W], cq[kL][W];
#pragma unroll
                        for (int d = 0; d < kL; d++)
                            if (i0 + d < np) {
                                const double* qo = ws + prev_at[i0 + d] + e;
                                load_w<W>(qo + p_of_q, cp[d]);
                                load_w<W>(qo, cq[d]);
                            }
#pragma unroll
                        for (int d = 0; d < kL; d++)
                            if (i0 + d < np) {
                                const double h = hp[i0 + d];
#pragma unroll
                                for (int u = 0; u < W; u++) {
                                    t[u] = fma(-h, cp[d][u], t[u]);
                                    x[u] = fma(-h, cq[d][u], x[u]);
                                }
                            }
                    }
                    store_w<W>(p + e, t);
                    store_w<W>(q + e, x);
                }
                if (fin) {
                    load_w<W>(r + e, y);
#pragma unroll
                    for (int u = 0; u < W; u++) {
                        qq = fma(x[u], x[u], qq);
                        rq = fma(y[u], x[u], rq);
                    }
                } else {
                    if (ng > 0) load_w<W>(newest + e, y);
#pragma unroll
                    for (int d0 = 0; d0 < kGsGroup; d0 += kL) {
                        if (d0 >= nn) break;
                        double v[kL][W];
#pragma unroll
                        for (int d = 0; d < kL; d++)
                            if (d0 + d < nn) load_w<W>(ws + next_at[g0 + d0 + d] + e, v[d]);
#pragma unroll
                        for (int d = 0; d < kL; d++)
                            if (d0 + d < nn)
#pragma unroll
                                for (int u = 0; u < W; u++) acc[d0 + d] = fma(x[u], v[d][u], acc[d0 + d]);
#pragma unroll
                        for (int d = 0; d < kL; d++)
                            if (d0 + d < ng)
#pragma unroll
                                for (int u = 0; u < W; u++)
                                    acc[kGsGroup + d0 + d] = fma(y[u], v[d][u], acc[kGsGroup + d0 + d]);
                    }
                }
            }
            const int t = threadIdx.x;
            if (fin) {
                block_sum2(qq, rq);
                if (t == 0) {
                    part[0] = qq;
                    part[1] = rq;
                }
            } else {
                const double v = ng > 0 ? cta_sums<16>(acc, sm) : cta_sums<8>(acc, sm);
                if (t < nn) part[g0 + t] = v;
                if (t >= kGsGroup && t < kGsGroup + ng) part[kB + g0 + t - kGsGroup] = v;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            last = atomicAdd(&st.ctl[C_CNT_RED], 1) == st.nchunk - 1;
        }
        __syncthreads();
        if (!last) return;
        __threadfence();
        if (threadIdx.x == 0) st.ctl[C_CNT_RED] = 0;
        gs_totals(st.partial, 1, kRows, st.nchunk, fin ? 2 : nd, fin || b > 0 ? 0 : 1 + ngram, false, kB, tot);
        __syncthreads();
        if (fin) {
            if (threadIdx.x == 0) {
                st.scal[SL.om_qq + slot] = tot[0];
                st.scal[SL.om_alpha] = tot[0] != 0.0 ? tot[1] / tot[0] : 0.0;
            }
            return;
        }
        if (threadIdx.x >= 32) return;
        // lane i: beta of l = lo + i
        const int i = threadIdx.x;
        double* gram = st.scal + SL.gram;  // entry (slot, distance): the product with the direction that much older
        if (b == 0 && i >= 1 && i < nd) gram[dir(1) * kB + i] = tot[nd + i];
        __syncwarp();
        // One reciprocal per lane, not a division per link of the chain.  1 / (Q_l, Q_l) overflows below 2^-1024 (a
        // right-hand side of 1e-150, eight digits later), so where a (Q_l, Q_l) is small it and the products that
        // its reciprocal multiplies are scaled by a power of two, which leaves their bits alone.  (A chain of its own:
        // one chain for both cases took 1.3 us a step longer at 30 x 30 x 9, k = 30.)
        const double qq = i < nd ? st.scal[SL.om_qq + dir(lo + i)] : 1.0;
        double c = i < nd ? tot[i] : 0.0, inv = i < nd ? 1.0 / qq : 0.0;
        if (__any_sync(0xffffffffu, qq < 0x1p-1000)) {
            const double sc = qq < 0x1p-1000 ? 0x1p600 : 1.0;
            c *= sc;
            inv = i < nd ? 1.0 / (qq * sc) : 0.0;
            for (int k = 0; k + 1 < nd; k++) {
                const double beta = __shfl_sync(0xffffffffu, c * inv, k);
                if (i > k && i < nd) c = fma(-(gram[dir(lo + k) * kB + i - k] * sc), beta, c);
            }
        } else {
            for (int k = 0; k + 1 < nd; k++) {
                const double beta = __shfl_sync(0xffffffffu, c * inv, k);
                if (i > k && i < nd) c = fma(-gram[dir(lo + k) * kB + i - k], beta, c);
            }
        }
        if (i < nd) st.scal[SL.om_beta + lo - 1 + i] = c * inv;
    } else if (ph == PH_INIT || ph == PH_OM_FINAL) {
        if (b != 0) return;
        const double* r = vec(st, ph == PH_INIT ? VR : VW);
        double s0 = 0.0, s1 = 0.0;
        for (int i = threadIdx.x; i < st.vchunk; i += blockDim.x) {
            const double a = r[e0 + i];
            s0 = fma(a, a, s0);
        }
        if (!finish_reduction(st, it.chunk, s0, s1)) return;
        if (threadIdx.x == 0) om_state(st, ph, sqrt(s0));
    }
}

// x += alpha p, r -= alpha q and ||r||; a direction with (q, q) = 0 ends the iteration instead.
__global__ void __launch_bounds__(VEC_THREADS) k_om_update(const SysTab* __restrict__ tab,
                                                           const VecItem* __restrict__ items) {
    const VecItem it = items[blockIdx.x];
    const SysTab& st = tab[it.sys];
    if (st.krylov != 1 || st.ctl[C_PHASE] != PH_OM) return;
    const ScalLayout SL = ScalLayout::make(st.m);
    const int slot = st.ctl[C_OM_SLOT];
    const bool dead = st.scal[SL.om_qq + slot] == 0.0;
    const long long e0 = (long long)it.chunk * st.vchunk;
    double s0 = 0.0, s1 = 0.0;
    if (!dead) {
        const double alpha = st.scal[SL.om_alpha];
        const double* p = vec(st, om_p(st, slot));
        const double* q = vec(st, om_q(st, slot));
        double* x = vec(st, VX);
        double* r = vec(st, VR);
        for (int i = threadIdx.x; i < st.vchunk; i += blockDim.x) {
            x[e0 + i] += alpha * p[e0 + i];
            const double a = r[e0 + i] - alpha * q[e0 + i];
            r[e0 + i] = a;
            s0 += a * a;
        }
    }
    if (!finish_reduction(st, it.chunk, s0, s1)) return;
    if (threadIdx.x != 0) return;
    if (dead) {
        st.ctl[C_PHASE] = PH_OM_FINAL;
        om_set_slots(st, PH_OM_FINAL);
    } else {
        om_state(st, PH_OM, sqrt(s0));
    }
}

// sum of one partial per CTA, in every CTA in the same order
__device__ __forceinline__ double grid_total1(const double* part, int G) {
    double a = 0.0;
    for (int i = threadIdx.x; i < G; i += blockDim.x) a += __ldcg(&part[i]);
    block_sum1(a);
    __shared__ double bc;
    if (threadIdx.x == 0) bc = a;
    __syncthreads();
    const double t = bc;
    __syncthreads();
    return t;
}

// Classical Gram-Schmidt for step j (asm_options.ortho = ASM_ORTHO_CGS): every coefficient
// h_i = (w, v_i), i = 0..j, and (w, w) from the same w, one sweep per dot and one grid reduction
// for all of them; then w' = w - sum_i h_i v_i (i in order) in one sweep, stored in w, and its norm
// from a second grid reduction.  Two grid barriers per step instead of MGS's j + 2; the rounding
// differs from MGS.  Partials: part2[i G + b] for value i of CTA b, the norm's after them.  The
// caller scales w' into v_{j+1}.  j + 2 <= kCgsMax.
__device__ void cgs_project(const SysTab& st, double* part2, cooperative_groups::grid_group& grid, int j,
                            const ScalLayout& SL, double& w0, double& hn) {
    constexpr int kU = 4;
    const int G = gridDim.x, nv = j + 2, m = st.m;
    const long long n = st.n3p;
    const long long stride = (long long)G * blockDim.x;
    const long long e_begin = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    double* w = vec(st, VW);
    // kD dots per sweep over w (vector i of the sweep: v_{i0 + i}, or w itself for the norm);
    // each thread keeps one partial per dot and element slot
    constexpr int kD = 4;
    __shared__ double red[kD][VEC_THREADS];
    for (int i0 = 0; i0 < nv; i0 += kD) {
        const double* vs[kD];
#pragma unroll
        for (int d = 0; d < kD; d++) {
            const int i = i0 + d;
            vs[d] = i <= j ? vec(st, VV0 + i) : (i == j + 1 ? w : nullptr);
        }
        double p[kD][2];
#pragma unroll
        for (int d = 0; d < kD; d++) p[d][0] = p[d][1] = 0.0;
        double a[2], b[kD][2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const long long e = e_begin + u * stride;
            a[u] = e < n ? w[e] : 0.0;
#pragma unroll
            for (int d = 0; d < kD; d++) b[d][u] = e < n && vs[d] ? vs[d][e] : 0.0;
        }
        for (long long e0 = e_begin; e0 < n; e0 += 2 * stride) {
            double an[2], bn[kD][2];
#pragma unroll
            for (int u = 0; u < 2; u++) {
                const long long e = e0 + (2 + u) * stride;
                an[u] = e < n ? w[e] : 0.0;
#pragma unroll
                for (int d = 0; d < kD; d++) bn[d][u] = e < n && vs[d] ? vs[d][e] : 0.0;
            }
#pragma unroll
            for (int d = 0; d < kD; d++)
                if (vs[d] != nullptr)
#pragma unroll
                    for (int u = 0; u < 2; u++) p[d][u] = fma(a[u], b[d][u], p[d][u]);
#pragma unroll
            for (int u = 0; u < 2; u++) {
                a[u] = an[u];
#pragma unroll
                for (int d = 0; d < kD; d++) b[d][u] = bn[d][u];
            }
        }
        // the kD block sums: warp d adds column d (eight entries per lane, then five shuffles)
#pragma unroll
        for (int d = 0; d < kD; d++) red[d][threadIdx.x] = p[d][0] + p[d][1];
        __syncthreads();
        const int wd = threadIdx.x >> 5, lane = threadIdx.x & 31;
        if (wd < kD) {
            double x = 0.0;
            for (int t = lane; t < (int)blockDim.x; t += 32) x += red[wd][t];
            for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
            if (lane == 0 && i0 + wd < nv) part2[(size_t)(i0 + wd) * G + blockIdx.x] = x;
        }
        __syncthreads();
    }
    grid.sync();
    // the nv totals in every CTA: eight threads per value over its G partials (index order within
    // each thread, then three butterfly adds), 32 values per round
    __shared__ double htot[kCgsMax];
    for (int base = 0; base < nv; base += 32) {
        const int i = base + (int)(threadIdx.x >> 3), q = threadIdx.x & 7;
        double a = 0.0;
        if (i < nv) {
            const double* pi = part2 + (size_t)i * G;
            int c = q;
            for (; c + 24 < G; c += 32) {
                const double l0 = __ldcg(&pi[c]), l1 = __ldcg(&pi[c + 8]), l2 = __ldcg(&pi[c + 16]), l3 = __ldcg(&pi[c + 24]);
                a += l0;
                a += l1;
                a += l2;
                a += l3;
            }
            for (; c < G; c += 8) a += __ldcg(&pi[c]);
        }
        a += __shfl_xor_sync(0xffffffffu, a, 4);
        a += __shfl_xor_sync(0xffffffffu, a, 2);
        a += __shfl_xor_sync(0xffffffffu, a, 1);
        if (q == 0 && i < nv) htot[i] = a;
    }
    __syncthreads();
    w0 = htot[j + 1];
    double p[kU];
#pragma unroll
    for (int u = 0; u < kU; u++) p[u] = 0.0;
    for (long long e0 = e_begin; e0 < n; e0 += kU * stride) {
        double x[kU];
#pragma unroll
        for (int u = 0; u < kU; u++) x[u] = e0 + u * stride < n ? w[e0 + u * stride] : 0.0;
        // kV basis vectors at a time: all their loads are issued before their multiply-adds (which
        // keep the order i = 0..j), so that enough loads are in flight to stream V from memory
        constexpr int kV = 4;
        int i = 0;
        for (; i + kV <= j + 1; i += kV) {
            double b[kV][kU];
#pragma unroll
            for (int d = 0; d < kV; d++) {
                const double* vi = vec(st, VV0 + i + d);
#pragma unroll
                for (int u = 0; u < kU; u++) b[d][u] = e0 + u * stride < n ? vi[e0 + u * stride] : 0.0;
            }
#pragma unroll
            for (int d = 0; d < kV; d++) {
                const double h = htot[i + d];
#pragma unroll
                for (int u = 0; u < kU; u++) x[u] = fma(-h, b[d][u], x[u]);
            }
        }
        for (; i <= j; i++) {
            const double h = htot[i];
            const double* vi = vec(st, VV0 + i);
            double b[kU];
#pragma unroll
            for (int u = 0; u < kU; u++) b[u] = e0 + u * stride < n ? vi[e0 + u * stride] : 0.0;
#pragma unroll
            for (int u = 0; u < kU; u++) x[u] = fma(-h, b[u], x[u]);
        }
#pragma unroll
        for (int u = 0; u < kU; u++) {
            if (e0 + u * stride < n) w[e0 + u * stride] = x[u];
            p[u] = fma(x[u], x[u], p[u]);
        }
    }
    double sum = (p[0] + p[1]) + (p[2] + p[3]);
    block_sum1(sum);
    double* pn = part2 + (size_t)nv * G;
    if (threadIdx.x == 0) pn[blockIdx.x] = sum;
    grid.sync();
    hn = sqrt(grid_total1(pn, G));
    if (blockIdx.x == 0 && threadIdx.x == 0)
        for (int i = 0; i <= j; i++) st.scal[SL.H + i * m + j] = htot[i];
}

// ------------------------------------------------------------------------------------------
// The whole orthogonalisation of one step of one system in one cooperative launch, every CTA on
// its slice [e0, e1) of the vectors: one grid barrier per block of basis vectors and one for the norm.
// ------------------------------------------------------------------------------------------
struct GsBlock {  // the vectors v_lo .. v_{lo + nd - 1}; ngram: Gram entries taken with them
    int lo, nd, ngram;
};
__device__ __forceinline__ GsBlock gs_block_at(int lo, int bs, int j) {
    const int nd = min(bs, j + 1 - lo);
    return GsBlock{lo, nd, lo + nd == j + 1 ? nd - 1 : 0};
}

struct GsShared {
    double sm[8 * 16], tot[2 * kGsMaxBlock + 1], hs[kGsMaxBlock];
    double gram[kGsMaxBlock * kGsMaxBlock];
};

// A group's CTA sums into the partials of its block: row q of the block's dots, Gram row and (row
// 2 bs) w's norm, one value per CTA.  GP: vectors per group (dots acc[0 ..], Gram entries acc[GP ..])
template <int GP>
__device__ __forceinline__ void gs_store_partials(GsShared& S, double (&acc)[16], double ww, bool norm, double* part, int bs,
                                                  int g0, int nn, int ng) {
    const int G = gridDim.x, q = threadIdx.x;
    const double t = ng > 0 ? cta_sums<2 * GP>(acc, S.sm) : cta_sums<GP>(acc, S.sm);
    if (q < nn) part[(long long)(g0 + q) * G + blockIdx.x] = t;
    if (q >= GP && q < GP + ng) part[(long long)(bs + g0 + q - GP) * G + blockIdx.x] = t;
    if (norm) {
        block_sum1(ww);
        if (q == 0) part[(long long)2 * bs * G + blockIdx.x] = ww;
    }
}

// The coefficients of a block, in S.hs of every CTA, from the partials (this is the grid barrier);
// CTA 0 keeps them and v_j's Gram row.  Each CTA adds the CTAs' partials up itself, in the same
// order.  Where that is many values from many CTAs (a whole cycle in one block), CTA q adds value q up
// and a second barrier hands it round: 152 partials of 60 values in every CTA would be ~40
// dependent FP64 adds of ~128 cycles.
__device__ __forceinline__ void gs_coefficients(const SysTab& st, GsShared& S, cooperative_groups::grid_group& grid,
                                                double* part, const GsBlock& B, int bs, int j, const ScalLayout& SL,
                                                double& w0) {
    const int G = gridDim.x, m = st.m;
    double* gram = st.scal + SL.gram;
    // the kept Gram rows, loaded while the barrier is waited for
    for (int t = threadIdx.x; t < B.nd * kGsMaxBlock; t += blockDim.x)
        S.gram[t] = t / kGsMaxBlock + B.lo < j ? gram[(long long)B.lo * kGsMaxBlock + t] : 0.0;
    grid.sync();
    const int nv = B.nd + B.ngram + (B.lo == 0 ? 1 : 0);
    if (nv > 16 && G > 32) {
        double* all = part + (long long)(2 * bs + 1) * G;
        const int q = blockIdx.x + G * (threadIdx.x >> 5);
        if (q < nv) {
            const int lane = threadIdx.x & 31;
            const double* p = part + (long long)(q < B.nd ? q : q < B.nd + B.ngram ? bs + q - B.nd : 2 * bs) * G;
            double a = 0.0;
            for (int k = lane; k < G; k += 32) a += __ldcg(p + k);
            for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if (lane == 0) all[q] = a;
        }
        grid.sync();
        if ((int)threadIdx.x < nv) S.tot[threadIdx.x] = __ldcg(all + threadIdx.x);
    } else {
        gs_totals(part, G, 1, G, B.nd, B.ngram, B.lo == 0, bs, S.tot);
    }
    __syncthreads();
    if (threadIdx.x < 32) gs_substitute(S.tot, B.nd, B.ngram, S.gram, S.hs);
    if (B.lo == 0) w0 = S.tot[B.nd + B.ngram];
    __syncthreads();
    if (blockIdx.x == 0) {
        const int t = threadIdx.x;
        if (t < B.nd) st.scal[SL.H + (B.lo + t) * m + j] = S.hs[t];
        if (t < B.ngram) gram[(long long)j * kGsMaxBlock + t] = S.tot[B.nd + t];
    }
}

// doubles of one of the two sets of partials (a block's are read while the next block's are written)
__device__ __forceinline__ long long gs_part_set(int bs) { return (long long)(2 * bs + 1) * gridDim.x + 2 * kGsMaxBlock + 1; }

// a sum over the CTAs, in every CTA (the other grid barrier)
__device__ __forceinline__ double gs_grid_sum(double s, double* part, cooperative_groups::grid_group& grid) {
    block_sum1(s);
    if (threadIdx.x == 0) part[blockIdx.x] = s;
    grid.sync();
    return grid_total1(part, gridDim.x);
}

// End of a step: v_{j+1} = w / h_{j+1,j}, or v_0 = r / beta (scale: that norm).  The state machine takes a few
// microseconds of dependent scalar operations: warp 0 of CTA 0 runs it while the other warps scale.
template <int W>
__device__ __forceinline__ void ortho_finish(const SysTab& st, int ph, int j, const ScalLayout& SL, long long e0, long long e1,
                                             double w0, double scale) {
    constexpr int kU = 8;
    const double* src = vec(st, ph == PH_ARNOLDI ? VW : VR);
    const int dst = ph == PH_ARNOLDI ? VV0 + j + 1 : VV0;
    int first = threadIdx.x, step = VEC_THREADS;
    if (blockIdx.x == 0) {
        if (threadIdx.x < 32) {
            if (threadIdx.x == 0) {
                if (ph == PH_ARNOLDI) {
                    st.scal[SL.w0] = sqrt(w0);
                    st.scal[SL.hn] = scale;
                    st.scal[SL.H + (j + 1) * st.m + j] = scale;
                } else {
                    st.scal[SL.beta] = scale;
                }
            }
            __syncwarp();
            step_state(st, ph);
            return;
        }
        first -= 32;
        step -= 32;
    }
    if (scale > 0.0) {
        const double inv = 1.0 / scale;
        double* v = vec(st, dst);
        for (long long e = e0 + W * first; e < e1; e += kU * W * step) {
            double a[kU][W];
#pragma unroll
            for (int u = 0; u < kU; u++)
                if (e + u * W * step < e1) load_w<W>(src + e + u * W * step, a[u]);
#pragma unroll
            for (int u = 0; u < kU; u++)
                if (e + u * W * step < e1) {
#pragma unroll
                    for (int k = 0; k < W; k++) a[u][k] *= inv;
                    store_w<W>(v + e + u * W * step, a[u]);
                }
        }
    }
}

// this CTA's slice of the vectors: whole 64-element pieces (the vectors are zero beyond n3)
__device__ __forceinline__ void gs_slice(const SysTab& st, long long& e0, long long& e1) {
    const long long n = (st.n3 + 63) & ~63;
    const long long len = ((n + gridDim.x - 1) / gridDim.x + 63) & ~63LL;
    e0 = min(n, len * blockIdx.x);
    e1 = min(n, e0 + len);
}

// ||r|| of an initial or restarting system
__device__ __forceinline__ double ortho_beta(const SysTab& st, double* part2, cooperative_groups::grid_group& grid,
                                             long long e0, long long e1) {
    const double* r = vec(st, VR);
    constexpr int kU = 8;
    double s0 = 0.0;
    for (long long e = e0 + threadIdx.x; e < e1; e += kU * VEC_THREADS) {
        double a[kU];
#pragma unroll
        for (int u = 0; u < kU; u++) a[u] = e + u * VEC_THREADS < e1 ? r[e + u * VEC_THREADS] : 0.0;
#pragma unroll
        for (int u = 0; u < kU; u++) s0 = fma(a[u], a[u], s0);
    }
    return sqrt(gs_grid_sum(s0, part2, grid));
}

// Short vectors (st.gs_block = kGsMaxBlock: up to 131,072 values, 862 per SM): a handful of elements per thread, so
// what counts is the number of barriers and of dependent FP64 operations.
__global__ void __launch_bounds__(VEC_THREADS, 1) k_ortho_short(const SysTab* __restrict__ tab, double* __restrict__ part2) {
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    __shared__ GsShared S;
    const SysTab& st = tab[0];
    const int ph = st.ctl[C_PHASE];
    if (ph == PH_DONE) return;
    const ScalLayout SL = ScalLayout::make(st.m);
    long long e0, e1;
    gs_slice(st, e0, e1);
    if (ph != PH_ARNOLDI) {
        ortho_finish<1>(st, ph, 0, SL, e0, e1, 0.0, ortho_beta(st, part2, grid, e0, e1));
        return;
    }
    const int j = st.ctl[C_J], bs = st.gs_block;
    double w0 = 0.0, norm = 0.0;
    int turn = 0;
    for (int lo = 0; lo <= j; lo += bs, turn ^= 1) {
        const GsBlock B = gs_block_at(lo, bs, j);
        double* part = part2 + turn * gs_part_set(bs);
#pragma unroll 1
        for (int g0 = 0; g0 < B.nd; g0 += kGsGroup) {
            double acc[16], ww = 0.0;
#pragma unroll
            for (int q = 0; q < 16; q++) acc[q] = 0.0;
            const int nn = min(kGsGroup, B.nd - g0), ng = max(0, min(kGsGroup, B.ngram - g0));
            const bool start = lo == 0 && g0 == 0;
            if (start)
                gs_sweep<1, true>(st, e0, e1, VV0, 0, S.hs, VV0, nn, ng, VV0 + j, acc, ww);
            else
                gs_sweep<1, false>(st, e0, e1, VV0, 0, S.hs, VV0 + lo + g0, nn, ng, VV0 + j, acc, ww);
            gs_store_partials<kGsGroup>(S, acc, ww, start, part, bs, g0, nn, ng);
        }
        gs_coefficients(st, S, grid, part, B, bs, j, SL, w0);
        double acc[16];
        norm = 0.0;
        gs_sweep<1, true>(st, e0, e1, VV0 + lo, B.nd, S.hs, VV0, 0, 0, VV0, acc, norm);
    }
    ortho_finish<1>(st, ph, j, SL, e0, e1, w0, sqrt(gs_grid_sum(norm, part2 + turn * gs_part_set(bs), grid)));
}

// gs_sweep for blocks of kGsLong vectors, with loads ahead of the arithmetic: the next vectors of an
// iteration are requested before its subtractions, the previous block's vectors of the next iteration
// before the products; with vectors on one side only, those of the next iteration.
template <bool PREV, bool GRAM>
__device__ __forceinline__ void gs_sweep_pipe(const SysTab& st, long long e0, long long e1, int prev, int np,
                                              const double* hp, int nxt, int nn, int ng, int jslot, bool norm,
                                              double (&acc)[16], double& ww) {
    constexpr int W = 2;
    const long long n = st.n3p;
    const long long first = e0 + W * threadIdx.x, step = W * VEC_THREADS;
    if (first >= e1) return;
    double* w = vec(st, VW);
    const double* vp = vec(st, prev);
    const double* vn = vec(st, nxt);
    const double* vj = vec(st, jslot);
    double h[kGsLong], x[W], y[W], b[kGsLong][W], c[kGsLong][W];
    auto load_group = [&](const double* base, int cnt, long long e, double (&v)[kGsLong][W]) {
        // no branch around the loads: a vector past the last one reads the last one again (its products
        // are skipped); q is opaque so that no address register per vector lives across the loop
        const double* q = base + e;
        asm volatile("" : "+l"(q));
#pragma unroll
        for (int d = 0; d < kGsLong; d++) {
            load_w<W>(q, v[d]);
            q += d + 1 < cnt ? n : 0;
        }
    };
    load_w<W>(w + first, x);
    if (PREV) {
#pragma unroll
        for (int d = 0; d < kGsLong; d++) h[d] = d < np ? hp[d] : 0.0;
        load_group(vp, np, first, c);
    } else {
        load_group(vn, nn, first, b);
        if (GRAM) load_w<W>(vj + first, y);
    }
#pragma unroll 1
    for (long long e = first; e < e1; e += step) {
        const long long en = e + step < e1 ? e + step : first;  // the last iteration's loads are not used
        double x1[W], y1[W];
        if (PREV) {
            if (nn > 0) {
                load_group(vn, nn, e, b);
                if (GRAM) load_w<W>(vj + e, y);
            } else {
                load_group(vp, np, en, b);
            }
#pragma unroll
            for (int d = 0; d < kGsLong; d++)
                if (d < np)
#pragma unroll
                    for (int u = 0; u < W; u++) x[u] = fma(-h[d], c[d][u], x[u]);
            store_w<W>(w + e, x);
            if (nn > 0) {
                load_group(vp, np, en, c);
            } else {
#pragma unroll
                for (int d = 0; d < kGsLong; d++)
#pragma unroll
                    for (int u = 0; u < W; u++) c[d][u] = b[d][u];
            }
        } else {
            load_group(vn, nn, en, c);
            if (GRAM) load_w<W>(vj + en, y1);
        }
        load_w<W>(w + en, x1);
#pragma unroll
        for (int d = 0; d < kGsLong; d++)
            if (d < nn)
#pragma unroll
                for (int u = 0; u < W; u++) acc[d] = fma(x[u], b[d][u], acc[d]);
        if (GRAM)
#pragma unroll
            for (int d = 0; d < kGsLong; d++)
                if (d < ng)
#pragma unroll
                    for (int u = 0; u < W; u++) acc[kGsLong + d] = fma(y[u], b[d][u], acc[kGsLong + d]);
        if (norm)
#pragma unroll
            for (int u = 0; u < W; u++) ww = fma(x[u], x[u], ww);
#pragma unroll
        for (int u = 0; u < W; u++) {
            x[u] = x1[u];
            if (!PREV) {
                if (GRAM) y[u] = y1[u];
#pragma unroll
                for (int d = 0; d < kGsLong; d++) b[d][u] = c[d][u];
            }
        }
    }
}

// Long vectors: blocks of kGsLong, two CTAs per SM.  An FP64 multiply-add holds a sub-partition's
// FP64 unit for 64 cycles, so what matters is that some warp always has its operands: 16 warps per SM
// with blocks of four (18 operands in registers) do that better than eight warps with blocks of
// eight, although those sweep w half as often (128x128x64, one solve: 21.6 against 26.9 ms; one reduction per
// vector: 24.5 ms).
__global__ void __launch_bounds__(VEC_THREADS, 2) k_ortho_long(const SysTab* __restrict__ tab, double* __restrict__ part2) {
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    __shared__ GsShared S;
    const SysTab& st = tab[0];
    const int ph = st.ctl[C_PHASE];
    if (ph == PH_DONE) return;
    const ScalLayout SL = ScalLayout::make(st.m);
    long long e0, e1;
    gs_slice(st, e0, e1);
    if (ph != PH_ARNOLDI) {
        ortho_finish<2>(st, ph, 0, SL, e0, e1, 0.0, ortho_beta(st, part2, grid, e0, e1));
        return;
    }
    const int j = st.ctl[C_J], bs = kGsLong;
    double w0 = 0.0, norm = 0.0;
    int turn = 0, np = 0;
    for (int lo = 0; lo <= j; lo += bs, turn ^= 1) {
        const GsBlock B = gs_block_at(lo, bs, j);
        double acc[16], ww = 0.0;
#pragma unroll
        for (int q = 0; q < 16; q++) acc[q] = 0.0;
        if (lo == 0 && B.ngram == 0)
            gs_sweep_pipe<false, false>(st, e0, e1, VV0, 0, S.hs, VV0, B.nd, 0, VV0 + j, true, acc, ww);
        else if (lo == 0)
            gs_sweep_pipe<false, true>(st, e0, e1, VV0, 0, S.hs, VV0, B.nd, B.ngram, VV0 + j, true, acc, ww);
        else if (B.ngram == 0)
            gs_sweep_pipe<true, false>(st, e0, e1, VV0 + lo - bs, np, S.hs, VV0 + lo, B.nd, 0, VV0 + j, false, acc, ww);
        else
            gs_sweep_pipe<true, true>(st, e0, e1, VV0 + lo - bs, np, S.hs, VV0 + lo, B.nd, B.ngram, VV0 + j, false, acc, ww);
        double* part = part2 + turn * gs_part_set(bs);
        gs_store_partials<kGsLong>(S, acc, ww, lo == 0, part, bs, 0, B.nd, B.ngram);
        gs_coefficients(st, S, grid, part, B, bs, j, SL, w0);
        np = B.nd;
    }
    double acc[16];
    gs_sweep_pipe<true, false>(st, e0, e1, VV0 + j / bs * bs, np, S.hs, VV0, 0, 0, VV0, true, acc, norm);
    ortho_finish<2>(st, ph, j, SL, e0, e1, w0, sqrt(gs_grid_sum(norm, part2 + turn * gs_part_set(bs), grid)));
}

__global__ void __launch_bounds__(VEC_THREADS, 2) k_ortho_cgs(const SysTab* __restrict__ tab, double* __restrict__ part2) {
    namespace cg = cooperative_groups;
    cg::grid_group grid = cg::this_grid();
    const SysTab& st = tab[0];
    const int ph = st.ctl[C_PHASE];
    if (ph == PH_DONE) return;
    const ScalLayout SL = ScalLayout::make(st.m);
    long long e0, e1;
    gs_slice(st, e0, e1);
    if (ph != PH_ARNOLDI) {
        ortho_finish<2>(st, ph, 0, SL, e0, e1, 0.0, ortho_beta(st, part2, grid, e0, e1));
        return;
    }
    const int j = st.ctl[C_J];
    double w0 = 0.0, hn = 0.0;
    cgs_project(st, part2, grid, j, SL, w0, hn);
    ortho_finish<2>(st, ph, j, SL, e0, e1, w0, hn);
}

}  // namespace

void launch_spmv(const SysTab* tab, const RowItem* items, int nitems, cudaStream_t st) {
    if (nitems > 0) k_spmv<<<256 / kSpmvThreads * nitems, kSpmvThreads, 0, st>>>(tab, items);
}

void launch_gather_ctl(const SysTab* tab, int n, int* out, cudaStream_t st) {
    if (n > 0) k_gather_ctl<<<n, 32, 0, st>>>(tab, out);
}
void launch_init(const SysTab* tab, const VecItem* items, int nitems, cudaStream_t st) {
    if (nitems > 0) k_init<<<nitems, VEC_THREADS, 0, st>>>(tab, items);
}
void launch_prep(const SysTab* tab, const VecItem* items, int nitems, cudaStream_t st) {
    if (nitems > 0) k_prep<<<nitems, VEC_THREADS, 0, st>>>(tab, items);
}
void launch_post(const SysTab* tab, const VecItem* items, int nitems, cudaStream_t st) {
    if (nitems > 0) k_post<<<nitems, VEC_THREADS, 0, st>>>(tab, items);
}
void launch_mgs(const SysTab* tab, const VecItem* items, int nitems, int pass, cudaStream_t st) {
    if (nitems > 0) k_mgs<<<nitems, VEC_THREADS, 0, st>>>(tab, items, pass);
}
namespace {
const void* ortho_kernel(int ortho, int n3) {
    if (ortho == 1) return (const void*)k_ortho_cgs;
    if (gs_block_size(n3) == kGsMaxBlock) return (const void*)k_ortho_short;
    return (const void*)k_ortho_long;
}
}  // namespace

int ortho_coop_grid(int device, int ortho, int n3) {
    int per_sm = 0, sms = 0;
    const void* f = ortho_kernel(ortho, n3);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, VEC_THREADS, 0) != cudaSuccess) return 0;
    if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess) return 0;
    // two CTAs per SM for their loads in flight; short vectors: one, for fewer partials, with 128
    // elements per CTA (one warp per SM sub-partition) until the chip is full
    const bool is_short = f == (const void*)k_ortho_short;
    const int max_grid = std::min(per_sm, is_short ? 1 : 2) * sms;
    return is_short ? std::max(1, std::min(max_grid, (n3 + 127) / 128)) : max_grid;
}

cudaError_t launch_ortho_coop(const SysTab* tab, double* part2, int grid, int ortho, int n3, cudaStream_t st) {
    void* args[] = {(void*)&tab, (void*)&part2};
    return cudaLaunchCooperativeKernel(ortho_kernel(ortho, n3), dim3(grid), dim3(VEC_THREADS), args, 0, st);
}

void launch_om(const SysTab* tab, const VecItem* items, int nitems, int pass, int sms, cudaStream_t st) {
    if (nitems <= 0) return;
    if (nitems <= sms)
        k_om<0><<<nitems, VEC_THREADS, 0, st>>>(tab, items, pass);
    else
        k_om<2><<<nitems, VEC_THREADS, 0, st>>>(tab, items, pass);
}
void launch_om_update(const SysTab* tab, const VecItem* items, int nitems, cudaStream_t st) {
    if (nitems > 0) k_om_update<<<nitems, VEC_THREADS, 0, st>>>(tab, items);
}

void launch_finish(const SysTab* tab, const VecItem* items, int nitems, cudaStream_t st) {
    if (nitems > 0) k_finish<<<nitems, VEC_THREADS, 0, st>>>(tab, items);
}

}  // namespace asm2
