// Nested factorisation (Appendix A) as the local solver of local problems without lumps: each
// subdomain's A_i is hepta-banded on its box of bx * by * bz cells (local cell p = z + bz (x + bx y)),
// A = D + L1 + U1 + L2 + U2 + L3 + U3, and
//   B = (P + L3)(I + P^{-1} U3),  P = (T + L2)(I + T^{-1} U2),  T = (G + L1)(I + G^{-1} U1)
// with G block diagonal, G = D - L1 G^{-1} U1 (Eq. A.6), with colsum also minus the block column sums
// of L2 T^{-1} U2 and L3 P^{-1} U3 (Eq. A.7).
//
// Both the factorisation and the solve are sequential along the cells of a subdomain: every line
// depends on the previous line of its plane, every plane on the previous plane.  So one CTA takes
// one subdomain: in the factorisation one of its warps runs the recurrences of a line (FP64 and the
// 3x3 block algebra of G: lane 3 r + c holds element (r, c) of a block), the others fetch the next
// line's operands, and all share the independent per-cell products.  The apply (one warp that solves, one
// that issues the copies) streams one packet per line -- G^{-1}, G^{-1} L1, G^{-1} U1, their two-step products, L2, L3, U3, U2 of the line's
// cells, packed after the factorisation -- through a shared-memory ring of 2-4 slots by bulk copies,
// ahead of the line being solved.  The products that do not depend on the line recurrences run on
// all lanes of the first warp; the two recurrences of T^{-1}, with one level of recursive doubling, run from shared
// memory on one lane (FP32) or three (FP64, one row each: an FP64 instruction costs the same for one
// lane as for 32).
#include <cuda_runtime.h>

#include <algorithm>

#include "asm2_internal.h"
#include "f64cvt.h"
#include "tma.h"

namespace asm2 {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// ---- the factorisation: 3x3 blocks held one element per lane (lanes 0..8; others carry zeros) ----

// Each cell's seven band blocks D, L1, U1, L2, U2, L3, U3 (zero where the neighbour is missing),
// gathered from the assembled slots into the compute type before the sequential factorisation,
// so that its operand loads need no index and can be issued early.
enum { BD_D = 0, BD_L1, BD_U1, BD_L2, BD_U2, BD_L3, BD_U3, BD_N };

template <typename TC>
__global__ void __launch_bounds__(128) k_nf_gather(const NFDesc* __restrict__ descs) {
    const NFDesc& d = descs[blockIdx.y];
    const int t = blockIdx.x * blockDim.x + threadIdx.x;  // (cell, band)
    if (t >= BD_N * d.n) return;
    const int sl = d.bands[t];
    TC* o = static_cast<TC*>(d.fband) + 9LL * t;
    for (int e = 0; e < 9; e++) o[e] = sl >= 0 ? (TC)d.slot[9LL * sl + e] : TC(0);
}

// a * b for blocks held per lane
template <typename TC>
__device__ __forceinline__ TC bmul(TC a, TC b, int lane) {
    const int r = lane < 9 ? lane / 3 : 0, c = lane < 9 ? lane - 3 * (lane / 3) : 0;
    const TC a0 = __shfl_sync(kFull, a, 3 * r), a1 = __shfl_sync(kFull, a, 3 * r + 1), a2 = __shfl_sync(kFull, a, 3 * r + 2);
    const TC b0 = __shfl_sync(kFull, b, c), b1 = __shfl_sync(kFull, b, 3 + c), b2 = __shfl_sync(kFull, b, 6 + c);
    return lane < 9 ? a0 * b0 + a1 * b1 + a2 * b2 : TC(0);
}

// Inverse of a block held per lane by cofactors: lane 3 r + c gets C_cr / det, with the cofactor
// C_ij = a_{i+1,j+1} a_{i+2,j+2} - a_{i+1,j+2} a_{i+2,j+1} (indices mod 3) and det = sum_k a_0k C_0k.
// Twelve dependent operations instead of the ~60 of an elimination on one lane (a dependent FP64
// operation costs ~100 cycles here).  false (on every lane) when det = 0.
template <typename TC>
__device__ __forceinline__ bool binv(TC a, TC& inv, int lane) {
    const int r = lane < 9 ? lane / 3 : 0, c = lane < 9 ? lane - 3 * (lane / 3) : 0;
    const int i1 = c == 2 ? 0 : c + 1, i2 = c == 0 ? 2 : c - 1, j1 = r == 2 ? 0 : r + 1, j2 = r == 0 ? 2 : r - 1;
    const TC p = __shfl_sync(kFull, a, 3 * i1 + j1), q = __shfl_sync(kFull, a, 3 * i2 + j2);
    const TC u = __shfl_sync(kFull, a, 3 * i1 + j2), v = __shfl_sync(kFull, a, 3 * i2 + j1);
    const TC cof = p * q - u * v;                       // C_cr
    const TC term = __shfl_sync(kFull, a, r) * cof;     // lanes 3 r (c = 0): a_0r C_0r
    const TC det = __shfl_sync(kFull, term, 0) + __shfl_sync(kFull, term, 3) + __shfl_sync(kFull, term, 6);
    if (det == TC(0)) return false;
    inv = lane < 9 ? cof / det : TC(0);
    return true;
}

// Working buffers of a line: bz blocks each, a block's rows LayF<TC>::RS values apart (FP32 pads a row
// to four values, so that it is one 16-byte access).  Fixed ones, then per stage the operands of a line.
enum { NB_N = 0, NB_K, NB_GI, NB_RHS, NB_VT, NB_W, NB_CS2, NB_G, NB_FIXED };
enum { ST_SRC = 0, ST_POST, ST_N, ST_K, ST_GI, ST_MX };   // of a line of a plane solve
enum { ST_D = 2, ST_L1, ST_U1, ST_C3, ST_FIELDS };         // of a line being factorised (with ST_SRC, ST_POST)

template <typename TC>
struct LayF {
    static constexpr int RS = sizeof(TC) == 4 ? 4 : 3, BS = 3 * RS;
};

// Rows of blocks along a line, one block product a step: x_0 = s_0, x_i = s_i - x_{i-1} A_i, where step i is
// cell first + dir i and A_i the block of that cell + mo.  Warp 0; dst may be src.
// FP32: three lanes, one row each, the row in registers: a step is the four dependent operations of the
// product (16 cycles), its operands loaded three steps ahead; with one element per lane the row has to
// go round by shuffles (~45 cycles).
__device__ __forceinline__ void chain_rows(const float* src, const float* A, int mo, float* dst, int bz, int first, int dir,
                                           int lane) {
    if (lane >= 3) return;
    const float4* s4 = reinterpret_cast<const float4*>(src) + lane;
    const float4* a4 = reinterpret_cast<const float4*>(A);
    float4* d4 = reinterpret_cast<float4*>(dst) + lane;
    float4 c[4], m[4][3];
    // steps past the end read the last one's operands again, and step 0 multiplies a zero row: no branch in
    // the ring, whose slots then stay in registers
    const auto load = [&](int i, int k) {
        const int j = min(i, bz - 1), q = first + dir * j, qa = j > 0 ? q + mo : first;
        c[k] = s4[3 * q];
        m[k][0] = a4[3 * qa];
        m[k][1] = a4[3 * qa + 1];
        m[k][2] = a4[3 * qa + 2];
    };
#pragma unroll
    for (int i = 0; i < 3; i++) load(i, i);
    float x0 = 0.f, x1 = 0.f, x2 = 0.f;
#pragma unroll 1
    for (int i0 = 0; i0 < bz; i0 += 4) {
#pragma unroll
        for (int k = 0; k < 4; k++) {
            load(i0 + k + 3, (k + 3) & 3);
            const float y0 = c[k].x - (x0 * m[k][0].x + x1 * m[k][1].x + x2 * m[k][2].x);
            const float y1 = c[k].y - (x0 * m[k][0].y + x1 * m[k][1].y + x2 * m[k][2].y);
            const float y2 = c[k].z - (x0 * m[k][0].z + x1 * m[k][1].z + x2 * m[k][2].z);
            x0 = y0;
            x1 = y1;
            x2 = y2;
            if (i0 + k < bz) d4[3 * (first + dir * (i0 + k))] = make_float4(x0, x1, x2, 0.f);
        }
    }
}
// FP64: nine lanes, one element each (an FP64 instruction holds the unit ~64 cycles for one lane as for 32)
__device__ __forceinline__ void chain_rows(const double* src, const double* A, int mo, double* dst, int bz, int first, int dir,
                                           int lane) {
    const int e = lane < 9 ? lane : 0, r = e / 3, col = e - 3 * r;
    double x = 0.0, c = src[9 * first + e], m = 0.0;
#pragma unroll 1
    for (int i = 0; i < bz; i++) {
        const int q = first + dir * i;
        const double y = c, b = m;
        if (i + 1 < bz) {
            c = src[9 * (q + dir) + e];
            m = A[9 * (q + dir + mo) + e];
        }
        const double a0 = __shfl_sync(kFull, x, 3 * r), a1 = __shfl_sync(kFull, x, 3 * r + 1),
                     a2 = __shfl_sync(kFull, x, 3 * r + 2);
        const double b0 = __shfl_sync(kFull, b, col), b1 = __shfl_sync(kFull, b, 3 + col), b2 = __shfl_sync(kFull, b, 6 + col);
        x = i > 0 ? fma(-a2, b2, fma(-a1, b1, fma(-a0, b0, y))) : y;
        if (lane < 9) dst[9 * q + e] = x;
    }
}

// f(cell, row, column, padded element offset) for each element of a line's blocks, by the threads [t0, t0 + nt)
template <typename TC, typename F>
__device__ __forceinline__ void elements(int bz, int t0, int nt, F f) {
#pragma unroll 2
    for (int t = (int)threadIdx.x - t0; t < 9 * bz; t += nt) {
        const int q = t / 9, e = t - 9 * q, r = e / 3, c = e - 3 * r;
        f(t, q, r, c, LayF<TC>::BS * q + LayF<TC>::RS * r + c);
    }
}

// element (r, c) of A B for blocks of working buffers
template <typename TC>
__device__ __forceinline__ TC prod(const TC* a, const TC* b, int r, int c) {
    constexpr int RS = LayF<TC>::RS;
    return a[RS * r] * b[c] + a[RS * r + 1] * b[RS + c] + a[RS * r + 2] * b[2 * RS + c];
}

// Factorisation in the compute type TC: G and G^{-1} (stored in FP64) of every cell, plane by plane, line by
// line, cell by cell, and with colsum, before each plane j > 0, cs3 = the block column sums of
// L3 P_{j-1}^{-1} U3, from W = u P^{-1} with u = L3 (a row of blocks):
//   vb (I + T^{-1} U2) = u:  vb_l = u_l - (vb_{l-1} T_{l-1}^{-1}) U2_{l-1}
//   W (T + L2) = vb:         W_l = (vb_l - W_{l+1} L2_{l+1}) T_l^{-1}
// and before each line l > 0 cs2 = those of L2 T_{l-1}^{-1} U2.  W = u T^{-1} on a line
// (W (G + L1)(I + G^{-1} U1) = u) with N_q = G_q^{-1} U1_q and K_q = L1_{q+1} G_q^{-1} is
//   forward   v_q = u_q - v_{q-1} N_{q-1}
//   backward  W_q = v_q G_q^{-1} - W_{q+1} K_q       (v_q G_q^{-1} for all cells first)
//
// Serial along the cells of a subdomain: what bounds it is the latency of a step of a line's two recurrences
// and of G's own.  A CTA per subdomain keeps a line's operands in shared memory: warp 0 runs the
// recurrences while the other warps fetch the next line's operands into the second stage, and the
// products of independent cells go over all threads.  With one warp per subdomain and the operands in device
// memory, 64 boxes of 12 x 12 x 32 cells with column sums took 8.4 ms (FP32; FP64 15.5, FP32 boxes of
// 4 x 3 x 150 1.77), now 2.6 (9.8, 0.55), the same FP32 bits; half of what is left is G's recurrence.
// `stages` 2, or 1 (no overlap of the fetch) for lines whose two stages do not fit.
template <typename TC, int T>
__global__ void __launch_bounds__(T, T == 128 ? 4 : 2) k_nf_factor(const NFDesc* __restrict__ descs, int stages, FactErr* err) {
    constexpr int BS = LayF<TC>::BS, RS = LayF<TC>::RS;
    extern __shared__ __align__(16) unsigned char nf_smem[];
    __shared__ bool bad;
    const NFDesc d = descs[blockIdx.x];  // by value: its fields stay in registers across the stores
    const int bz = d.bz, bx = d.bx, by = d.by, S = bz * bx, lane = threadIdx.x & 31;
    const bool seq = threadIdx.x < 32;
    // device scratch: cs3 and vb (9 S each), N, K and (FP32) G^{-1} (9 n each)
    TC* cs3 = reinterpret_cast<TC*>(d.work);
    TC* vb = cs3 + 9 * S;
    TC* gn = vb + 9 * S;
    TC* gk = gn + 9LL * d.n;
    TC* gg = sizeof(TC) == 8 ? reinterpret_cast<TC*>(d.gi) : gk + 9LL * d.n;
    TC* const buf = reinterpret_cast<TC*>(nf_smem);
    const auto fix = [&](int f) { return buf + (long long)f * BS * bz; };
    const auto st = [&](int b, int f) { return buf + (long long)(NB_FIXED + ST_FIELDS * b + f) * BS * bz; };
    const TC* fband = static_cast<const TC*>(d.fband);
    const auto band = [&](int k, int q0, int t, int q) { return fband[9LL * (BD_N * (q0 + q) + k) + t - 9 * q]; };
    if (threadIdx.x == 0) bad = false;

    // operands of line solve i of the solve with plane j - 1 (forward lines 0 .. bx-1, back to 0)
    const auto stage_plane = [&](int j, int i, int b, int t0, int nt) {
        const int c0 = (j - 1) * S, l = i < bx ? i : 2 * bx - 2 - i, p0 = c0 + l * bz;
        TC *sn = st(b, ST_N), *sk = st(b, ST_K), *sg = st(b, ST_GI), *ss = st(b, ST_SRC), *sm = st(b, ST_MX),
           *sp = st(b, ST_POST);
        elements<TC>(bz, t0, nt, [&](int t, int q, int, int, int o) {
            const TC n = gn[9LL * p0 + t], k = gk[9LL * p0 + t], g = gg[9LL * p0 + t];
            const TC s = i < bx ? band(BD_L3, c0 + S + l * bz, t, q) : vb[9 * l * bz + t];
            const TC m = i == 0 ? TC(0) : i < bx ? band(BD_U2, p0 - bz, t, q) : band(BD_L2, p0 + bz, t, q);
            const TC u = i >= bx - 1 ? band(BD_U3, p0, t, q) : TC(0);
            sn[o] = n;
            sk[o] = k;
            sg[o] = g;
            ss[o] = s;
            sm[o] = m;
            sp[o] = u;
        });
    };
    // operands of line l of plane j
    const auto stage_line = [&](int j, int l, int b, bool line_term, bool plane_term, int t0, int nt) {
        const int p0 = j * S + l * bz;
        TC *sd = st(b, ST_D), *s1 = st(b, ST_L1), *u1 = st(b, ST_U1), *ss = st(b, ST_SRC), *sp = st(b, ST_POST), *c3 = st(b, ST_C3);
        elements<TC>(bz, t0, nt, [&](int t, int q, int, int, int o) {
            const TC a = band(BD_D, p0, t, q), b1 = band(BD_L1, p0, t, q), c = band(BD_U1, p0, t, q);
            const TC s = line_term ? band(BD_L2, p0, t, q) : TC(0), u = line_term ? band(BD_U2, p0 - bz, t, q) : TC(0);
            const TC e = plane_term ? cs3[9 * l * bz + t] : TC(0);
            sd[o] = a;
            s1[o] = b1;
            u1[o] = c;
            ss[o] = s;
            sp[o] = u;
            c3[o] = e;
        });
    };
    // NB_W = u T^{-1}; `meanwhile` runs on the other warps during the forward recurrence
    const auto line_solve = [&](const TC* u, const TC* N, const TC* K, const TC* GI, auto meanwhile) {
        TC *v = fix(NB_VT), *W = fix(NB_W);
        if (seq)
            chain_rows(u, N, -1, v, bz, 0, 1, lane);
        else
            meanwhile();
        __syncthreads();
        elements<TC>(bz, 0, T, [&](int, int q, int r, int c, int o) { W[o] = prod(v + BS * q, GI + BS * q, r, c); });
        __syncthreads();
        if (seq) chain_rows(W, K, 0, W, bz, bz - 1, -1, lane);
        __syncthreads();
    };

    for (int j = 0; j < by; j++) {
        const bool plane_term = d.colsum && j > 0;
        if (plane_term) {
            stage_plane(j, 0, 0, 0, T);
            __syncthreads();
            for (int i = 0; i < 2 * bx - 1; i++) {
                const int b = stages == 2 ? i & 1 : 0, l = i < bx ? i : 2 * bx - 2 - i;
                TC *rhs = fix(NB_RHS), *W = fix(NB_W);
                const TC *src = st(b, ST_SRC), *mx = st(b, ST_MX), *post = st(b, ST_POST);
                elements<TC>(bz, 0, T, [&](int t, int q, int r, int c, int o) {
                    TC v = src[o];
                    if (i > 0) v -= prod(W + BS * q, mx + BS * q, r, c);
                    rhs[o] = v;
                    if (i < bx - 1) vb[9 * l * bz + t] = v;
                });
                __syncthreads();
                line_solve(rhs, st(b, ST_N), st(b, ST_K), st(b, ST_GI), [&] {
                    if (stages == 2 && i + 1 < 2 * bx - 1) stage_plane(j, i + 1, b ^ 1, 32, T - 32);
                });
                if (i >= bx - 1)
                    elements<TC>(bz, 0, T, [&](int t, int q, int r, int c, int) {
                        cs3[9 * l * bz + t] = prod(W + BS * q, post + BS * q, r, c);
                    });
                if (stages != 2 && i + 1 < 2 * bx - 1) {
                    __syncthreads();
                    stage_plane(j, i + 1, 0, 0, T);
                    __syncthreads();
                }
            }
            __syncthreads();
        }
        stage_line(j, 0, 0, false, plane_term, 0, T);
        __syncthreads();
        for (int l = 0; l < bx; l++) {
            const int b = stages == 2 ? l & 1 : 0, p0 = j * S + l * bz;
            const bool line_term = d.colsum && l > 0;
            const auto next = [&] {
                if (stages == 2 && l + 1 < bx) stage_line(j, l + 1, b ^ 1, d.colsum, plane_term, 32, T - 32);
            };
            TC *cs2 = fix(NB_CS2), *G = fix(NB_G), *GI = fix(NB_GI);
            if (line_term) {
                line_solve(st(b, ST_SRC), fix(NB_N), fix(NB_K), GI, next);
                const TC *W = fix(NB_W), *post = st(b, ST_POST);
                elements<TC>(bz, 0, T,
                             [&](int, int q, int r, int c, int o) { cs2[o] = prod(W + BS * q, post + BS * q, r, c); });
                __syncthreads();
            }
            if (seq) {
                // G_p = D_p - L1_p G_{p-1}^{-1} U1_{p-1} - (line and plane column sums); the previous
                // cell's G^{-1} stays in a register, the next cell's operands load early
                const int e = lane < 9 ? lane : 0, o = RS * (e / 3) + e % 3;
                const TC *D = st(b, ST_D) + o, *L1 = st(b, ST_L1) + o, *U1 = st(b, ST_U1) + o, *c2 = cs2 + o, *c3 = st(b, ST_C3) + o;
                TC gprev = 0, nd = D[0], nl1 = 0, nu1 = 0, nc2 = line_term ? c2[0] : TC(0), nc3 = plane_term ? c3[0] : TC(0);
#pragma unroll 1
                for (int q = 0; q < bz; q++) {
                    const TC cd = nd, cl1 = nl1, cu1 = nu1, cc2 = nc2, cc3 = nc3;
                    if (q + 1 < bz) {
                        nd = D[BS * (q + 1)];
                        nl1 = L1[BS * (q + 1)];
                        nu1 = U1[BS * q];
                        if (line_term) nc2 = c2[BS * (q + 1)];
                        if (plane_term) nc3 = c3[BS * (q + 1)];
                    }
                    TC g = cd;
                    if (q > 0) g -= bmul(bmul(cl1, gprev, lane), cu1, lane);
                    g -= cc2;
                    g -= cc3;
                    TC gi;
                    if (!binv(g, gi, lane)) {  // (warp-uniform)
                        if (lane == 0) {
                            bad = true;
                            if (atomicCAS(&err->flag, 0, 1) == 0) {
                                err->sub = d.sub;
                                err->row = p0 + q;
                            }
                        }
                        break;
                    }
                    if (lane < 9) {
                        G[BS * q + o] = g;
                        GI[BS * q + o] = gi;
                    }
                    gprev = gi;
                }
            } else if (!line_term) {
                next();
            }
            __syncthreads();
            if (bad) return;
            // G, G^{-1} and, for the line and plane solves, N_q and K_q
            TC *N = fix(NB_N), *K = fix(NB_K);
            const TC *L1 = st(b, ST_L1), *U1 = st(b, ST_U1);
            elements<TC>(bz, 0, T, [&](int t, int q, int r, int c, int o) {
                const long long at = 9LL * p0 + t;
                const TC n = prod(GI + BS * q, U1 + BS * q, r, c);
                const TC k = q + 1 < bz ? prod(L1 + BS * (q + 1), GI + BS * q, r, c) : TC(0), gi = GI[o];
                d.g[at] = (double)G[o];
                d.gi[at] = (double)gi;
                if (sizeof(TC) == 4) gg[at] = gi;
                N[o] = n;
                K[o] = k;
                gn[at] = n;
                gk[at] = k;
            });
            __syncthreads();
            if (stages != 2 && l + 1 < bx) {
                stage_line(j, l + 1, 0, d.colsum, plane_term, 0, T);
                __syncthreads();
            }
        }
    }
}

// ---- the apply ---------------------------------------------------------------------------------

// fields of a line packet, each bz blocks, field after field.  A line solve copies only the fields
// it reads into a ring slot of SL_FIELDS fields: G^{-1}, M, N, P, Q always (slot fields 0-4),
// then L2 and L3 on a forward line of a forward plane, L2 and U3 on a forward line of a backward
// plane, U2 on a backward line (slot fields 5, 6).
enum { PK_GI = 0, PK_M, PK_N, PK_P, PK_Q, PK_L2, PK_L3, PK_U3, PK_U2, PK_FIELDS };
enum { SL_X = 5, SL_Y = 6, SL_FIELDS = 7 };

// Layout of the compute type: a 3x3 block is 3 rows of RS values (row r at r RS), a cell's
// 3-vector takes VS values in shared memory.  FP32 pads both to 4, so that a row or a vector is one
// 16-byte access; FP64 keeps them dense (its packets are twice as large already).
template <typename T>
struct Lay {
    static constexpr int RS = 3, VS = 3;
};
template <>
struct Lay<float> {
    static constexpr int RS = 4, VS = 4;
};

__device__ __forceinline__ void ld3(const float* p, float& a, float& b, float& c) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    a = v.x;
    b = v.y;
    c = v.z;
}
__device__ __forceinline__ void ld3(const double* p, double& a, double& b, double& c) {
    a = p[0];
    b = p[1];
    c = p[2];
}
__device__ __forceinline__ void st3(float* p, float a, float b, float c) {
    *reinterpret_cast<float4*>(p) = make_float4(a, b, c, 0.f);
}
__device__ __forceinline__ void st3(double* p, double a, double b, double c) {
    p[0] = a;
    p[1] = b;
    p[2] = c;
}

// y -= a x for a 3x3 block a and 3-vectors, one fused chain per row
template <typename T>
__device__ __forceinline__ void sub_mv(const T* a, T x0, T x1, T x2, T& y0, T& y1, T& y2) {
    constexpr int RS = Lay<T>::RS;
    T a0, a1, a2;
    ld3(a, a0, a1, a2);
    y0 = fma(-a2, x2, fma(-a1, x1, fma(-a0, x0, y0)));
    ld3(a + RS, a0, a1, a2);
    y1 = fma(-a2, x2, fma(-a1, x1, fma(-a0, x0, y1)));
    ld3(a + 2 * RS, a0, a1, a2);
    y2 = fma(-a2, x2, fma(-a1, x1, fma(-a0, x0, y2)));
}

// packets of every line, one thread per cell: G^{-1}, M = G^{-1} L1 (the forward recurrence of
// (G + L1) s = u is s_q = G_q^{-1} u_q - M_q s_{q-1}), N = G^{-1} U1 (the backward recurrence of
// (I + G^{-1} U1) w = s is w_q = s_q - N_q w_{q+1}), the two-step products P_q = M_q M_{q-1} and
// Q_q = N_q N_{q+1}, and the blocks L2, U2, L3, U3 (zero where the neighbour is missing); products
// in FP64, stored in the compute type (row padding stays zero)
// bytes of one field of a line packet: bz blocks, rounded up to 16 bytes (a bulk-copy unit)
template <typename T>
__host__ __device__ __forceinline__ size_t field_bytes(int bz) {
    return ((size_t)9 * Lay<T>::RS / 3 * sizeof(T) * bz + 15) & ~(size_t)15;
}

template <typename T>
__global__ void __launch_bounds__(128) k_nf_pack(const NFDesc* __restrict__ descs) {
    constexpr int RS = Lay<T>::RS, BS = 3 * RS;
    const NFDesc& d = descs[blockIdx.y];
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= d.n) return;
    const int bz = d.bz, line = p / bz, q = p - line * bz;
    T* pk = reinterpret_cast<T*>(static_cast<unsigned char*>(d.pack) + (size_t)line * d.line_bytes);
    const auto band = [&](int k) -> const double* {
        const int s = d.bands[7 * p + k];
        return s >= 0 ? d.slot + 9LL * s : nullptr;
    };
    const auto put = [&](int f, const double* b) {
        T* o = pk + (size_t)f * (field_bytes<T>(bz) / sizeof(T)) + (size_t)q * BS;
        for (int r = 0; r < 3; r++)
            for (int c = 0; c < 3; c++) o[r * RS + c] = b ? (T)b[3 * r + c] : T(0);
    };
    const auto mul = [](const double* a, const double* b, double* c) {
        for (int r = 0; r < 3; r++)
            for (int k = 0; k < 3; k++) c[3 * r + k] = a[3 * r] * b[k] + a[3 * r + 1] * b[3 + k] + a[3 * r + 2] * b[6 + k];
    };
    // G^{-1} L1 (k = 1) or G^{-1} U1 (k = 2) of cell pp; false where that band block is missing
    const auto gib = [&](int pp, int k, double* out) {
        const int sl = d.bands[7 * pp + k];
        if (sl < 0) return false;
        mul(d.gi + 9LL * pp, d.slot + 9LL * sl, out);
        return true;
    };
    double m[9], m2[9], pq[9];
    put(PK_GI, d.gi + 9LL * p);
    const bool hm = gib(p, 1, m);
    put(PK_M, hm ? m : nullptr);
    put(PK_P, hm && q > 0 && gib(p - 1, 1, m2) ? (mul(m, m2, pq), pq) : nullptr);
    const bool hn = gib(p, 2, m);
    put(PK_N, hn ? m : nullptr);
    put(PK_Q, hn && q + 1 < bz && gib(p + 1, 2, m2) ? (mul(m, m2, pq), pq) : nullptr);
    put(PK_L2, band(3));
    put(PK_U2, band(4));
    put(PK_L3, band(5));
    put(PK_U3, band(6));
}

// The line solves of one apply, in order: forward planes j = 0 .. by-1, then backward planes
// j = by-2 .. 0; in each plane the forward lines l = 0 .. bx-1 of (T + L2) z = t, then the
// backward lines l = bx-2 .. 0 of (I + T^{-1} U2) o = z.  P counts the plane passes, i the line
// solves of the pass; next() advances without divisions.
struct LineStep {
    int P = 0, i = 0, j = 0, l = 0;
    bool fwd_plane = true, fwd_line = true, plane_first = true, plane_done = false;
    __device__ __forceinline__ void set(int bx, int by) {
        fwd_plane = P < by;
        j = fwd_plane ? P : 2 * by - 2 - P;
        fwd_line = i < bx;
        l = fwd_line ? i : 2 * bx - 2 - i;
        plane_first = i == 0;
        plane_done = i == 2 * bx - 2;
    }
    __device__ __forceinline__ void next(int bx, int by) {
        if (++i == 2 * bx - 1) {
            i = 0;
            ++P;
        }
        set(bx, by);
    }
};

__host__ __device__ size_t nf_rline_bytes(int bz) { return ((size_t)24 * bz + 32 + 15) & ~(size_t)15; }

// bytes of a plane vector (VS values per cell, rounded up to 16)
template <typename T>
__host__ __device__ __forceinline__ size_t nf_plane_bytes(int S) {
    return ((size_t)Lay<T>::VS * S * sizeof(T) + 15) & ~(size_t)15;
}

// z[owned cells of plane j] = x_j (held in pv)
template <typename T>
__device__ __forceinline__ void write_owned(const NFDesc& d, int j, const T* pv, double* z, int lane) {
    constexpr int VS = Lay<T>::VS;
    if (j < d.own_lo[1] || j >= d.own_hi[1]) return;
    const int wx = d.own_hi[0] - d.own_lo[0], wz = d.own_hi[2] - d.own_lo[2];
    for (int t = lane; t < wx * wz; t += 32) {
        const int x = d.own_lo[0] + t / wz, zz = d.own_lo[2] + t % wz;
        const long long cell = d.c0 + zz + (long long)d.gnz * (x + (long long)d.gnx * j);
        const T* v = pv + VS * (x * d.bz + zz);
        z[3 * cell] = (double)v[0];
        z[3 * cell + 1] = (double)v[1];
        z[3 * cell + 2] = (double)v[2];
    }
}

// One chain step x <- c + A x for a 3x3 block A (three float4 rows) and 3-vectors, one fused
// chain per row
__device__ __forceinline__ void chain_step(const float4* a, float4 c, float& x0, float& x1, float& x2) {
    const float n0 = fmaf(a[0].z, x2, fmaf(a[0].y, x1, fmaf(a[0].x, x0, c.x)));
    const float n1 = fmaf(a[1].z, x2, fmaf(a[1].y, x1, fmaf(a[1].x, x0, c.y)));
    const float n2 = fmaf(a[2].z, x2, fmaf(a[2].y, x1, fmaf(a[2].x, x0, c.z)));
    x0 = n0;
    x1 = n1;
    x2 = n2;
}

// x_q = c_q + A_q x_{q-d} for q = q0, q0 + d, ... (d = +-2; the x before q0 is zero), in place
// in cb, on one lane (FP32).  The operands are loaded three steps ahead into a ring of registers (steps past
// the end read the last one's again, so that the ring has no branches): four steps loaded together and then
// computed left the loads' latency exposed once per group.
__device__ __forceinline__ void chain(const float* A, float* cb, int q0, int d, int count) {
    if (count <= 0) return;
    const float4* Av = reinterpret_cast<const float4*>(A);
    float4* cv = reinterpret_cast<float4*>(cb);
    float4 a[4][3], c[4];
    const auto load = [&](int i, int k) {
        const int q = q0 + d * min(i, count - 1);
        a[k][0] = Av[3 * q];
        a[k][1] = Av[3 * q + 1];
        a[k][2] = Av[3 * q + 2];
        c[k] = cv[q];
    };
#pragma unroll
    for (int i = 0; i < 3; i++) load(i, i);
    float x0 = 0.f, x1 = 0.f, x2 = 0.f;
#pragma unroll 1
    for (int i0 = 0; i0 < count; i0 += 4) {
#pragma unroll
        for (int k = 0; k < 4; k++) {
            load(i0 + k + 3, (k + 3) & 3);
            chain_step(a[k], c[k], x0, x1, x2);
            if (i0 + k < count) cv[q0 + d * (i0 + k)] = make_float4(x0, x1, x2, 0.f);
        }
    }
}

// The same on three lanes (FP64: lane r takes row r, the state goes round by shuffles; an FP64
// instruction costs the same for one lane as for 32)
__device__ __forceinline__ void chain(const double* A, double* cb, int q0, int d, int count, int lane) {
    constexpr unsigned kRow = 0x7u;
    double x = 0.0;
    for (int i = 0; i < count; i++) {
        const int q = q0 + d * i;
        const double* a = A + 9 * q + 3 * lane;
        const double a0 = a[0], a1 = a[1], a2 = a[2], c = cb[3 * q + lane];
        const double x0 = __shfl_sync(kRow, x, 0), x1 = __shfl_sync(kRow, x, 1), x2 = __shfl_sync(kRow, x, 2);
        x = fma(a2, x2, fma(a1, x1, fma(a0, x0, c)));
        cb[3 * q + lane] = x;
    }
}

// T^{-1} of one line, c = G^{-1} u given in cb: s_q = c_q - M_q s_{q-1} (s_{-1} = 0), then
// w_q = s_q - N_q w_{q+1} (w_bz = 0), with one level of recursive doubling: the sequential chains
// visit every other cell,
//   s_q = (c_q - M_q c_{q-1}) + P_q s_{q-2},  P_q = M_q M_{q-1}    (q odd)
//   w_q = (s_q - N_q s_{q+1}) + Q_q w_{q+2},  Q_q = N_q N_{q+1}    (chain cells q = bz-2, bz-4, ...)
// and the cells in between follow from their neighbours on all lanes, each lane finishing the
// cells next to its own (three passes over the line besides the two chains).  On return o_q = w_q
// (forward line) or o_q -= w_q (backward line).  Called by the whole warp.
template <typename T>
__device__ __forceinline__ void line_solve(const T* M, const T* N, const T* P, const T* Q, T* cb, T* o, int bz,
                                           bool fwd_line, int lane) {
    constexpr int BS = 3 * Lay<T>::RS, VS = Lay<T>::VS;
    // y_q - B_q x_{q'} for cells of cb (a missing q' contributes nothing)
    const auto sub = [&](const T* B, int q, int qx, T& y0, T& y1, T& y2) {
        if (qx < 0 || qx >= bz) return;
        T x0, x1, x2;
        ld3(cb + VS * qx, x0, x1, x2);
        sub_mv(B + BS * q, x0, x1, x2, y0, y1, y2);
    };
    // odd q: c_q - M_q c_{q-1}
    for (int q = 1 + 2 * lane; q < bz; q += 64) {
        T y0, y1, y2;
        ld3(cb + VS * q, y0, y1, y2);
        sub(M, q, q - 1, y0, y1, y2);
        st3(cb + VS * q, y0, y1, y2);
    }
    __syncwarp();
    if constexpr (sizeof(T) == 4) {
        if (lane == 0) chain(P, cb, 1, 2, bz / 2);
    } else {
        if (lane < 3) chain(P, cb, 1, 2, bz / 2, lane);
    }
    __syncwarp();
    // chain cells q = bz-2-2i: t_q = s_q - N_q s_{q+1}, the even one of q and q + 1 first finished
    // as s_e = c_e - M_e s_{e-1} (it is this lane's: bz even, e = q; bz odd, e = q + 1)
    for (int i = lane;; i += 32) {
        const int q = bz - 2 - 2 * i;
        if (q < 0) break;
        T s0, s1, s2, n0, n1, n2;
        ld3(cb + VS * q, s0, s1, s2);
        ld3(cb + VS * (q + 1), n0, n1, n2);
        if ((q & 1) == 0) {
            sub(M, q, q - 1, s0, s1, s2);  // s_q
        } else {
            sub_mv(M + BS * (q + 1), s0, s1, s2, n0, n1, n2);  // s_{q+1} = c_{q+1} - M_{q+1} s_q
            st3(cb + VS * (q + 1), n0, n1, n2);
        }
        sub_mv(N + BS * q, n0, n1, n2, s0, s1, s2);
        st3(cb + VS * q, s0, s1, s2);
    }
    __syncwarp();
    if constexpr (sizeof(T) == 4) {
        if (lane == 0) chain(Q, cb, bz - 2, -2, bz / 2);
    } else {
        if (lane < 3) chain(Q, cb, bz - 2, -2, bz / 2, lane);
    }
    __syncwarp();
    // the other cells q = bz-1-2i: w_q = s_q - N_q w_{q+1} (w_bz = 0); this lane then writes the
    // output of q and of the chain cell q - 1 below it
    const auto out = [&](int q, T w0, T w1, T w2) {
        if (!fwd_line) {
            T a0, a1, a2;
            ld3(o + VS * q, a0, a1, a2);
            w0 = a0 - w0;
            w1 = a1 - w1;
            w2 = a2 - w2;
        }
        st3(o + VS * q, w0, w1, w2);
    };
    for (int i = lane;; i += 32) {
        const int q = bz - 1 - 2 * i;
        if (q < 0) break;
        T w0, w1, w2;
        ld3(cb + VS * q, w0, w1, w2);
        sub(N, q, q + 1, w0, w1, w2);
        out(q, w0, w1, w2);
        if (q > 0) {
            ld3(cb + VS * (q - 1), w0, w1, w2);
            out(q - 1, w0, w1, w2);
        }
    }
}

// an element of r in the compute type (FP32: the integer conversion, off the FP64 unit)
template <typename T>
__device__ __forceinline__ T to_compute(double v) {
    if constexpr (sizeof(T) == 4)
        return f64_to_f32(v);
    else
        return v;
}

// B_i^{-1} R_i r for one subdomain per CTA, owned cells written to the apply output.  Warp 0 solves the lines;
// warp 1 issues the copies, a slot's next line as soon as warp 0 has released it (SPREAD may exchange them).  What
// bounds the kernel is the serial path of warp 0, ~3,600 cycles a line of 32 cells in FP32 (the two recurrences 850
// each at 16 steps,
// G^{-1} u 460, the wait 300, the other passes 240 - 410): addresses and copies of the next line, and the
// conversion of r, are off it (64 boxes of 12 x 12 x 32 cells, an apply as called: FP32 1,084 -> 985 us, FP64
// 4,360 -> 4,160).
// SPREAD, for launches of more than two CTAs per SM: which of its two warps solves, a CTA takes from its place in the SM
// (%warpid, read once; any value is right), so that the solving warps of four CTAs are in four sub-partitions.  The first
// warps of every other CTA share one, and two line recurrences then take each other's issue slots.  512 boxes
// (128 x 128 x 64), an apply as called, FP32: 1,452 us with first warps, 1,220 spread (1,222 with one warp per CTA), FP64
// 4,953 and 4,918; 320 boxes 1,057 and 918.  With one or two CTAs per SM first warps are apart, and this form is 1 %
// slower (64 boxes: 964 and 974).
// Shared memory: SLOTS + 1 pairs of mbarriers (16 bytes: a slot is full | is free; y_j has come | the producer's
// two words) | SLOTS packet slots | SLOTS slots for the
// line's part of r (FP64) | plane vector pv [VS S] | y_j of a backward plane [VS S] | line vector
// cb [VS bz].  pv holds, in turn, y_{j-1} and z / o of plane j during the forward planes, then
// x_{j+1} and z / o of plane j during the backward ones: every line reads the previous plane's
// value of a line before it overwrites it.  y_j goes to device memory (yv, one plane every
// nf_plane_bytes) when its forward plane is done, and comes back by a bulk copy issued at the start
// of its backward plane.
template <typename T, int SLOTS, bool SPREAD>
__global__ void __launch_bounds__(64) k_nf_apply(const SysTab* __restrict__ tab, const NFDesc* __restrict__ descs) {
    constexpr int BS = 3 * Lay<T>::RS, VS = Lay<T>::VS;
    extern __shared__ __align__(16) unsigned char nf_smem[];
    const NFDesc d = descs[blockIdx.x];  // by value: its fields stay in registers across the stores
    const SysTab& st = tab[d.sys];
    const int in = st.ctl[C_APPLY_IN];
    if (in < 0) return;
    const double* __restrict__ r = st.ws + (long long)in * st.n3p;
    double* __restrict__ z = st.ws + (long long)st.ctl[C_APPLY_OUT] * st.n3p;
    const int lane = threadIdx.x & 31;
    const int bx = d.bx, by = d.by, bz = d.bz, S = bx * bz;
    const unsigned fb = (unsigned)field_bytes<T>(bz);
    const size_t LB = (size_t)d.line_bytes, SB = (size_t)SL_FIELDS * fb, RB = nf_rline_bytes(bz),
                 PB = nf_plane_bytes<T>(S);
    unsigned long long* bar = reinterpret_cast<unsigned long long*>(nf_smem);  // full: even words, free: odd
    unsigned long long* ybar = bar + 2 * SLOTS;
    volatile int* stop = reinterpret_cast<volatile int*>(ybar + 1);  // warp 0 has given up
    volatile int* issued = stop + 1;                                 // line solves issued when warp 1 ends
    unsigned char* const pk_base = nf_smem + 16 * (SLOTS + 1);
    unsigned char* const r_base = pk_base + SLOTS * SB;
    T* pv = reinterpret_cast<T*>(r_base + SLOTS * RB);
    T* yb = reinterpret_cast<T*>(reinterpret_cast<unsigned char*>(pv) + PB);
    T* cb = reinterpret_cast<T*>(reinterpret_cast<unsigned char*>(yb) + PB);
    unsigned char* yv = static_cast<unsigned char*>(d.yv);
    const int K = (2 * by - 1) * (2 * bx - 1);
    const size_t fe = fb / sizeof(T);

    // the grid cell of a line's first cell; the line's cells follow it (z is the fastest index)
    const auto cell0_of = [&](const LineStep& s) {
        return d.c0 + (long long)d.gnz * (s.l + (long long)d.gnx * s.j);
    };
    // packet of a line solve into slot b, plus the line's part of r for a forward line of a forward
    // plane (the copy starts at the 16-byte boundary at or below it: one leading double when the
    // cell is odd); only the fields the line solve reads
    const auto issue = [&](const LineStep& s, int b) {
        unsigned rbytes = 0;
        const unsigned char* rsrc = nullptr;
        if (s.fwd_plane && s.fwd_line) {
            const long long c0 = cell0_of(s);
            const long long a = (24 * c0) & ~15LL, e = (24 * (c0 + bz) + 15) & ~15LL;
            rbytes = (unsigned)(e - a);
            rsrc = reinterpret_cast<const unsigned char*>(r) + a;
        }
        // (packet field, slot field, count) of each copy
        int f[3][3] = {{PK_GI, 0, PK_Q + 1}, {0, 0, 0}, {0, 0, 0}};
        if (!s.fwd_line) {
            f[1][0] = PK_U2, f[1][1] = SL_X, f[1][2] = 1;
        } else if (s.fwd_plane) {
            f[1][0] = PK_L2, f[1][1] = SL_X, f[1][2] = 2;  // L2, L3
        } else {
            f[1][0] = PK_L2, f[1][1] = SL_X, f[1][2] = 1;
            f[2][0] = PK_U3, f[2][1] = SL_Y, f[2][2] = 1;
        }
        if (f[1][2] > 0 && f[1][0] == f[0][0] + f[0][2] && f[1][1] == f[0][1] + f[0][2]) {
            f[0][2] += f[1][2];  // adjacent in the packet and in the slot: one copy
            f[1][2] = 0;
        }
        unsigned tx = rbytes;
        for (int i = 0; i < 3; i++) tx += (unsigned)f[i][2] * fb;
        tma::mbar_expect_tx(&bar[2 * b], tx);
        const unsigned char* src = static_cast<const unsigned char*>(d.pack) + (size_t)(s.j * bx + s.l) * LB;
        for (int i = 0; i < 3; i++)
            if (f[i][2] > 0)
                tma::bulk_load(pk_base + b * SB + (size_t)f[i][1] * fb, src + (size_t)f[i][0] * fb,
                               (unsigned)f[i][2] * fb, &bar[2 * b]);
        if (rbytes) tma::bulk_load(r_base + b * RB, rsrc, rbytes, &bar[2 * b]);
    };

    if (threadIdx.x == 0) {
        for (int b = 0; b < SLOTS; b++) {
            tma::mbar_init(&bar[2 * b], 1);
            tma::mbar_init(&bar[2 * b + 1], 1);
        }
        tma::mbar_init(ybar, 1);
        *stop = 0;
        if constexpr (SPREAD) {
            unsigned slot;
            asm volatile("mov.u32 %0, %%warpid;" : "=r"(slot));
            *issued = (int)(slot >> 2) & 1;
        }
        tma::fence_mbar_init();
    }
    __syncthreads();
    bool solver = threadIdx.x < 32;
    if constexpr (SPREAD) {
        solver = (int)(threadIdx.x >> 5) == *issued;
        __syncthreads();
    }
    if (!solver) {
        if (lane == 0) {
            LineStep nx;  // the next line solve to issue
            nx.set(bx, by);
            int ni = 0, bi = 0;
            unsigned fph = 1;  // phase of "slot bi is free"
            for (; ni < K; ni++) {
                if (ni >= SLOTS) {
                    bool ok = false;
                    for (long long i = 0; i < tma::kWaitLimit && !ok && !*stop; i++) {
                        ok = tma::mbar_try_wait(&bar[2 * bi + 1], fph);
                        if (!ok) __nanosleep(200);  // (polling takes the shared-memory cycles of warp 0)
                    }
                    if (!ok) break;
                }
                issue(nx, bi);
                nx.next(bx, by);
                if (++bi == SLOTS) {
                    bi = 0;
                    fph ^= 1u;
                }
            }
            *issued = ni;
        }
        __syncthreads();
        return;
    }
    LineStep s;
    s.set(bx, by);
    bool ypend = false;
    // a wait that expired: report it, have warp 1 stop, wait (bounded) for the copies still in flight, and leave
    const auto fail = [&](int k) {
        if (lane == 0) {
            atomicExch(st.dev_err, 7);
            *stop = 1;
        }
        __syncthreads();
        if (lane == 0) {
            const int ni = *issued;
            for (int k2 = k; k2 < ni; k2++) tma::mbar_wait(&bar[2 * (k2 % SLOTS)], (unsigned)(k2 / SLOTS) & 1u);
            if (ypend) tma::mbar_wait(ybar, (unsigned)(by - 2 - s.j) & 1u);
        }
    };
    int bc = 0;
    unsigned ph = 0;  // slot and barrier phase of the line solve in progress
    for (int k = 0; k < K; k++) {
        if (s.plane_first && !s.fwd_plane) {  // y_j of this backward plane, needed when it is done
            if (lane == 0) {
                tma::mbar_expect_tx(ybar, (unsigned)PB);
                tma::bulk_load(yb, yv + (size_t)s.j * PB, (unsigned)PB, ybar);
            }
            ypend = true;
        }
        const bool ok = tma::mbar_wait(&bar[2 * bc], ph, st.wait_limit);
        if (!__all_sync(kFull, ok)) {
            fail(k);
            return;
        }
        const T* pk = reinterpret_cast<const T*>(pk_base + bc * SB);
        const auto blk = [&](int f, int q) { return pk + f * fe + (size_t)q * BS; };
        T* pl = pv + (size_t)VS * s.l * bz;  // this line's part of the plane vector
        // c = G^{-1} u, u the line's right-hand side:
        //   forward line of a forward plane:   u = r - L3 y_{j-1} - L2 z_{l-1}
        //   forward line of a backward plane:  u = U3 x_{j+1} - L2 z_{l-1}
        //   backward line:                     u = U2 o_{l+1}
        // (a product that is added goes through sub_mv with the vector negated, which is exact)
        const double* rl = reinterpret_cast<const double*>(r_base + bc * RB) + (cell0_of(s) & 1);
        for (int q = lane; q < bz; q += 32) {
            T u0 = 0, u1 = 0, u2 = 0, x0, x1, x2;
            const T* cur = pl + VS * q;
            if (s.fwd_line) {
                if (s.fwd_plane) {
                    u0 = to_compute<T>(rl[3 * q]);
                    u1 = to_compute<T>(rl[3 * q + 1]);
                    u2 = to_compute<T>(rl[3 * q + 2]);
                    if (s.j > 0) {
                        ld3(cur, x0, x1, x2);
                        sub_mv(blk(SL_Y, q), x0, x1, x2, u0, u1, u2);  // L3
                    }
                } else {
                    ld3(cur, x0, x1, x2);
                    sub_mv(blk(SL_Y, q), -x0, -x1, -x2, u0, u1, u2);  // U3
                }
                if (s.l > 0) {
                    ld3(cur - VS * bz, x0, x1, x2);
                    sub_mv(blk(SL_X, q), x0, x1, x2, u0, u1, u2);  // L2
                }
            } else {
                ld3(cur + VS * bz, x0, x1, x2);
                sub_mv(blk(SL_X, q), -x0, -x1, -x2, u0, u1, u2);  // U2
            }
            T c0 = 0, c1 = 0, c2 = 0;
            sub_mv(blk(PK_GI, q), -u0, -u1, -u2, c0, c1, c2);
            st3(cb + VS * q, c0, c1, c2);
        }
        __syncwarp();
        line_solve(blk(PK_M, 0), blk(PK_N, 0), blk(PK_P, 0), blk(PK_Q, 0), cb, pl, bz, s.fwd_line, lane);
        __syncwarp();
        if (lane == 0) tma::mbar_arrive(&bar[2 * bc + 1]);  // the slot is free
        if (s.plane_done) {  // pv = P_j^{-1} t
            if (s.fwd_plane) {
                if (s.j < by - 1) {  // y_j to device memory, ordered before its later bulk copy back
                    T* yj = reinterpret_cast<T*>(yv + (size_t)s.j * PB);
                    for (int e = lane; e < VS * S; e += 32) yj[e] = pv[e];
                    asm volatile("fence.proxy.async;" ::: "memory");
                } else {
                    write_owned(d, s.j, pv, z, lane);  // x_{by-1} = y_{by-1}
                }
            } else {
                const bool yok = tma::mbar_wait(ybar, (unsigned)(by - 2 - s.j) & 1u, st.wait_limit);
                if (!__all_sync(kFull, yok)) {
                    fail(k + 1);
                    return;
                }
                ypend = false;
                for (int e = lane; e < VS * S; e += 32) pv[e] = yb[e] - pv[e];  // x_j = y_j - pv
                __syncwarp();
                write_owned(d, s.j, pv, z, lane);
            }
            __syncwarp();
        }
        s.next(bx, by);
        if (++bc == SLOTS) {
            bc = 0;
            ph ^= 1u;
        }
    }
    __syncthreads();  // (with warp 1's end)
}

template <typename T, int SLOTS>
void nf_apply_t(const SysTab* tab, const NFDesc* descs, int ndesc, size_t smem, int sms, cudaStream_t st) {
    const auto apply = [&](auto kernel) {
        allow_dynamic_smem((const void*)kernel, (int)smem);
        kernel<<<ndesc, 64, smem, st>>>(tab, descs);
    };
    if (ndesc <= 2 * sms)
        apply(k_nf_apply<T, SLOTS, false>);
    else
        apply(k_nf_apply<T, SLOTS, true>);
}

template <typename T>
void nf_apply_s(const SysTab* tab, const NFDesc* descs, int ndesc, int slots, size_t smem, int sms, cudaStream_t st) {
    if (slots >= 4)
        nf_apply_t<T, 4>(tab, descs, ndesc, smem, sms, st);
    else if (slots == 3)
        nf_apply_t<T, 3>(tab, descs, ndesc, smem, sms, st);
    else
        nf_apply_t<T, 2>(tab, descs, ndesc, smem, sms, st);
}

}  // namespace

size_t nf_line_bytes(int bz, int prec) {
    return PK_FIELDS * (prec == 0 ? field_bytes<double>(bz) : field_bytes<float>(bz));
}

size_t nf_plane_bytes(int S, int prec) { return prec == 0 ? nf_plane_bytes<double>(S) : nf_plane_bytes<float>(S); }

size_t nf_apply_smem(int bx, int bz, int prec, int slots) {
    const size_t t = prec == 0 ? 8 : 4, vs = prec == 0 ? 3 : 4;
    const size_t fb = prec == 0 ? field_bytes<double>(bz) : field_bytes<float>(bz);
    return 16 * (size_t)(slots + 1) + slots * (SL_FIELDS * fb + nf_rline_bytes(bz)) +
           2 * nf_plane_bytes(bx * bz, prec) + vs * (size_t)bz * t;
}

size_t nf_work_doubles(int bx, int by, int bz) { return 18 * (size_t)bx * bz + 18 * (size_t)bx * by * bz; }

namespace {
size_t nf_factor_smem(int bz, int prec, int stages) {
    return (size_t)(NB_FIXED + ST_FIELDS * stages) * bz * (prec == 0 ? LayF<double>::BS * 8 : LayF<float>::BS * 4);
}

template <typename TC>
void nf_factor_t(const NFDesc* descs, int ndesc, int nmax, int bz_max, int prec, int dev_smem, int sms, FactErr* err,
                 cudaStream_t st) {
    const dim3 ggrid((unsigned)((BD_N * nmax + 127) / 128), (unsigned)ndesc);
    const dim3 grid((unsigned)((nmax + 127) / 128), (unsigned)ndesc);
    // one stage always fits where the apply's two ring slots (1,056 bytes a cell in FP64 and 720 in FP32,
    // against 1,008 and 672 here) and its plane vectors do
    const int stages = nf_factor_smem(bz_max, prec, 2) <= (size_t)dev_smem - 1024 ? 2 : 1;
    const size_t smem = nf_factor_smem(bz_max, prec, stages);
    k_nf_gather<TC><<<ggrid, 128, 0, st>>>(descs);
    // CTAs of 256 threads fit an SM twice (registers); where that does not hold the launch and shared memory has room
    // for more, CTAs of 128, up to four: a re-factor of 128 x 128 x 64 cells in 512 boxes, FP64 24.5 -> 14.4 ms (22.5
    // with one warp per box), FP32 8.6 -> 6.6; 128 x 128 x 32 in 320, 15.4 -> 10.8 and 4.9 -> 4.0.
    const auto factor = [&](auto kernel, int threads) {
        allow_dynamic_smem((const void*)kernel, (int)smem);
        kernel<<<ndesc, threads, smem, st>>>(descs, stages, err);
    };
    if (ndesc <= 2 * sms || 3 * (smem + 1024) > (size_t)dev_smem)
        factor(k_nf_factor<TC, 256>, 256);
    else
        factor(k_nf_factor<TC, 128>, 128);
    k_nf_pack<TC><<<grid, 128, 0, st>>>(descs);
}
}  // namespace

void launch_nf_factor(const NFDesc* descs, int ndesc, int nmax, int bz_max, int prec, int dev_smem, int sms, FactErr* err,
                      cudaStream_t st) {
    if (ndesc <= 0) return;
    if (prec == 0)
        nf_factor_t<double>(descs, ndesc, nmax, bz_max, prec, dev_smem, sms, err, st);
    else
        nf_factor_t<float>(descs, ndesc, nmax, bz_max, prec, dev_smem, sms, err, st);
}

void launch_nf_apply(const SysTab* tab, const NFDesc* descs, int ndesc, int prec, int slots, size_t smem,
                     int sms, cudaStream_t st) {
    if (ndesc <= 0) return;
    if (prec == 0)
        nf_apply_s<double>(tab, descs, ndesc, slots, smem, sms, st);
    else
        nf_apply_s<float>(tab, descs, ndesc, slots, smem, sms, st);
}

int nf_apply_slots(int ndesc, int bx_max, int bz_max, int prec, int sm_smem, int sms, int dev_smem) {
    // the deepest ring with which every CTA of the launch is resident at once; else the shallowest
    // that fits a CTA at all
    const long long per_sm = (ndesc + std::max(1, sms) - 1) / std::max(1, sms);
    for (int s = 4; s >= 2; s--) {
        const size_t b = nf_apply_smem(bx_max, bz_max, prec, s);
        if (b <= (size_t)dev_smem && per_sm * (long long)(b + 1024) <= (long long)sm_smem) return s;
    }
    return 2;
}

}  // namespace asm2
