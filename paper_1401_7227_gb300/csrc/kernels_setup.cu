// Setup kernels: ELL fill of A, far-box coarse matrix, assembly of the local matrices
// A_i = R_i A R_i^T (Eq. 3.4 with the R_i of Eq. 4.1; Eq. B.3), the level-scheduled block ILU(0)
// with column-sum compensation (Section 2; cf. Eq. A.7) and the packing of the factor streams.
#include <cuda_fp16.h>

#include "asm2_internal.h"
#include "packets.h"

namespace asm2 {

namespace {


// ELL slot w of row r <- BSR block rp[r] + w (the w-th stored block of the row).  Threads run over
// (w, r) with r fastest, so the nine element planes are written with unit stride across a warp;
// each thread reads its block's 72 contiguous bytes.  Padding slots keep their zeros.
__global__ void k_ell_fill(const double* __restrict__ bsr, const int* __restrict__ rp, int n, int ell_w,
                           double* __restrict__ ell, int rows_pad) {
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (long long)ell_w * n) return;
    const int w = (int)(t / n), r = (int)(t - (long long)w * n);
    const int e = rp[r] + w;
    if (e >= rp[r + 1]) return;
    const double* b = bsr + 9LL * e;
    double v[9];
#pragma unroll
    for (int k = 0; k < 9; k++) v[k] = b[k];
#pragma unroll
    for (int k = 0; k < 9; k++) ell[((long long)w * 9 + k) * rows_pad + r] = v[k];
}

// C[J, J'] = sum of the blocks of A coupling far box J to far box J' (one CTA per C block); block
// lists hold BSR block indices into the array-of-blocks copy of A
__global__ void k_coarse(const int* __restrict__ cptr, const int* __restrict__ cloc,
                         const double* __restrict__ bsr, double* __restrict__ cval) {
    const int c = blockIdx.x;
    double acc[9];
#pragma unroll
    for (int e = 0; e < 9; e++) acc[e] = 0.0;
    for (int i = cptr[c] + threadIdx.x; i < cptr[c + 1]; i += blockDim.x) {
        const int L = cloc[i];
#pragma unroll
        for (int e = 0; e < 9; e++) acc[e] += bsr[9LL * L + e];
    }
    __shared__ double red[9][256];
#pragma unroll
    for (int e = 0; e < 9; e++) red[e][threadIdx.x] = acc[e];
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s)
#pragma unroll
            for (int e = 0; e < 9; e++) red[e][threadIdx.x] += red[e][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x < 9) cval[(long long)c * 9 + threadIdx.x] = red[threadIdx.x][0];
}

// slot value = C block (far-far pairs) + signed sum of A blocks from the slot's list
__global__ void k_assemble(const int* __restrict__ aptr, const int* __restrict__ aloc, const int* __restrict__ acs,
                           const double* __restrict__ bsr, const double* __restrict__ cval,
                           double* __restrict__ slot, long long nslot, int long_min) {
    long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nslot * 9) return;
    long long s = t / 9;
    int e = (int)(t - s * 9);
    const int i0 = aptr[s], i1 = aptr[s + 1];
    if (i1 - i0 >= long_min) return;  // a whole warp sums this one (k_assemble_long)
    double acc = 0.0;
    int c = acs[s];
    if (c >= 0) acc = cval[(long long)c * 9 + e];
    for (int i = i0; i < i1; i++) {
        int L = aloc[i];
        if (L >= 0)
            acc += bsr[9LL * L + e];
        else
            acc -= bsr[9LL * ~L + e];
    }
    slot[t] = acc;
}

// Slots with long lists (far-lump blocks: the box-pair block minus thousands of near-region
// couplings): one warp per slot, lanes over the list four entries at a time with the loads issued
// first, nine partial sums per lane combined by shuffles
__global__ void __launch_bounds__(256) k_assemble_long(const int* __restrict__ aptr, const int* __restrict__ aloc,
                                                       const int* __restrict__ acs, const double* __restrict__ bsr,
                                                       const double* __restrict__ cval,
                                                       double* __restrict__ slot, const int* __restrict__ long_slots,
                                                       int nlong) {
    const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (w >= nlong) return;
    const int s = long_slots[w];
    const int i0 = aptr[s], i1 = aptr[s + 1];
    double acc[9];
#pragma unroll
    for (int e = 0; e < 9; e++) acc[e] = 0.0;
    constexpr int kU = 4;
    for (int b = i0 + lane; b < i1; b += 32 * kU) {
        int L[kU];
#pragma unroll
        for (int u = 0; u < kU; u++) L[u] = b + 32 * u < i1 ? aloc[b + 32 * u] : 0x7fffffff;
#pragma unroll
        for (int u = 0; u < kU; u++) {
            if (L[u] == 0x7fffffff) continue;
            const int loc = L[u] >= 0 ? L[u] : ~L[u];
            const double sg = L[u] >= 0 ? 1.0 : -1.0;
#pragma unroll
            for (int e = 0; e < 9; e++) acc[e] = fma(sg, bsr[9LL * loc + e], acc[e]);
        }
    }
#pragma unroll
    for (int e = 0; e < 9; e++)
        for (int o = 16; o > 0; o >>= 1) acc[e] += __shfl_xor_sync(0xffffffffu, acc[e], o);
    if (lane < 9) {
        double v = 0.0;
#pragma unroll
        for (int e = 0; e < 9; e++)
            if (e == lane) v = acc[e];
        const int c = acs[s];
        if (c >= 0) v += cval[(long long)c * 9 + lane];
        slot[(long long)s * 9 + lane] = v;
    }
}

// 3x3 inverse in place by Gauss-Jordan elimination with partial pivoting; false on a zero pivot (m is then
// undefined).  The operations on [A | I], without those on the zeros and ones of I: ~60 instructions of the
// FP64 unit instead of ~100.
__device__ __forceinline__ bool inverse3(double (&m)[3][3]) {
    int piv[2] = {0, 1};
#pragma unroll
    for (int c = 0; c < 3; c++) {
        int p = c;
        double big = fabs(m[c][c]);
#pragma unroll
        for (int r = c + 1; r < 3; r++)
            if (fabs(m[r][c]) > big) {
                p = r;
                big = fabs(m[r][c]);
            }
        if (big == 0.0) return false;
#pragma unroll
        for (int r = c + 1; r < 3; r++)
            if (p == r)
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    const double t = m[c][k];
                    m[c][k] = m[r][k];
                    m[r][k] = t;
                }
        if (c < 2) piv[c] = p;
        // one reciprocal per pivot column: FP64 division expands to many FP64-pipe instructions
        const double id = 1.0 / m[c][c];
        m[c][c] = id;
#pragma unroll
        for (int k = 0; k < 3; k++)
            if (k != c) m[c][k] *= id;
#pragma unroll
        for (int r = 0; r < 3; r++) {
            if (r == c) continue;
            const double f = m[r][c];
#pragma unroll
            for (int k = 0; k < 3; k++)
                if (k != c) m[r][k] = fma(-f, m[c][k], m[r][k]);
            m[r][c] = -(f * id);
        }
    }
    // the inverse of the row-swapped matrix: its columns in the order of the rows
#pragma unroll
    for (int c = 1; c >= 0; c--)
#pragma unroll
        for (int r = 0; r < 3; r++)
#pragma unroll
            for (int k = c + 1; k < 3; k++)
                if (piv[c] == k) {
                    const double t = m[r][c];
                    m[r][c] = m[r][k];
                    m[r][k] = t;
                }
    return true;
}

// Right-looking block ILU(0) (+ colsum) in "pull" form, one CTA per subdomain.  Level by level:
// (A) every slot finalised at this level subtracts its (L, U) pairs in the order the
// right-looking update would apply them (compensations of dropped fill are pairs of the
// diagonal slots); (B) the level's pivots are inverted; (C) its L column blocks are scaled by
// D^{-1}.  All pairs reference slots finalised at lower levels.
//
// What bounds it is latency: a level of 40-65 rows has three phases with a barrier each, and each phase is a chain
// of dependent loads (~1,000 cycles a link) and of dependent FP64 operations (69 cycles; a level's longest
// target has 10-100 pairs of three).  So T threads and MINB CTAs per SM fill the SM's registers for the number of
// subdomains in the launch, a phase's first indices are loaded in the phase before, and a target's next KP pairs
// and a thread's KC blocks of L are in flight together.  Re-factor before -> after: 64 x 64 x 16 cells
// (64 subdomains) 1.27 -> 0.94 ms, 97 x 83 x 29 (120) 2.95 -> 2.28, 128 x 128 x 32 (256) 4.71 -> 4.07,
// 128 x 128 x 64 (512) 8.98 -> 8.35.
template <int T, int MINB, int KP, int KC>
__global__ void __launch_bounds__(T, MINB) k_factor(const FactDesc* __restrict__ fds, const int* __restrict__ ids,
                                                    FactErr* err) {
    const FactDesc fd = fds[ids ? ids[blockIdx.x] : blockIdx.x];
    double* slot = fd.slot;
    // nine lanes per 3x3 result (lane = 3 r + c within a group), three groups per warp: each FP64
    // instruction then serves three targets instead of one thread's nine elements
    const int lane = threadIdx.x & 31, grp = lane / 9, e9 = lane - 9 * grp, er = e9 / 3, ec = e9 - 3 * er;
    const int warp = threadIdx.x >> 5, nwarp = T >> 5;
    const bool lane_on = grp < 3;
    // What a level reads first -- its ranges, the first target, pivot row and L block of each thread -- is
    // requested a phase or a level ahead: those loads are links of a serial chain of ~1,000 cycles each.
    int tl0 = fd.tgt_lv[0], lp0 = fd.lv_pos0[0], l0 = fd.ls_lv[0];
    int tl1 = fd.tgt_lv[1], lp1 = fd.lv_pos0[1], l1 = fd.ls_lv[1];
    int nsl = 0, nq0 = 0, nq1 = 0;
    const auto target = [&](int t) {
        nsl = fd.tgt[t];
        nq0 = fd.pp[t];
        nq1 = fd.pp[t + 1];
    };
    if (lane_on && tl0 + 3 * warp + grp < tl1) target(tl0 + 3 * warp + grp);
    for (int lv = 0; lv < fd.nlev; lv++) {
        const int lvn = min(lv + 2, fd.nlev);
        const int tl2 = fd.tgt_lv[lvn], lp2 = fd.lv_pos0[lvn], l2 = fd.ls_lv[lvn];
        const int p0 = lp0 + threadIdx.x;
        const int dpos = p0 < lp1 ? fd.diag_of_pos[p0] : 0, rpos = p0 < lp1 ? fd.row_of_pos[p0] : 0;
        int t = tl0 + 3 * warp + grp;
        bool on = lane_on && t < tl1;
        while (on) {
            double* s = slot + (long long)nsl * 9;
            const int q0 = nq0, q1 = nq1;
            t += 3 * nwarp;
            on = t < tl1;
            if (on) target(t);
            double acc = s[e9];
            // KP pairs at a time, in the order of one at a time: the blocks of the next ones and the indices of
            // those after them are requested before the arithmetic
            int2 pa[KP], pb[KP];
            double la[KP][3], ua[KP][3], lb[KP][3], ub[KP][3];
            const auto pairs = [&](int q, int2(&pr)[KP]) {
#pragma unroll
                for (int u = 0; u < KP; u++) pr[u] = q + u < q1 ? fd.pair[q + u] : make_int2(0, 0);
            };
            const auto blocks = [&](const int2(&pr)[KP], double(&l)[KP][3], double(&uu)[KP][3]) {
#pragma unroll
                for (int u = 0; u < KP; u++) {
                    const double* L = slot + (long long)pr[u].x * 9 + 3 * er;
                    const double* U = slot + (long long)pr[u].y * 9 + ec;
#pragma unroll
                    for (int k = 0; k < 3; k++) {
                        l[u][k] = L[k];
                        uu[u][k] = U[3 * k];
                    }
                }
            };
            const auto subtract = [&](int q, const double(&l)[KP][3], const double(&uu)[KP][3]) {
#pragma unroll
                for (int u = 0; u < KP; u++)
                    if (q + u < q1)  // three FMAs into the running value (not product, sum, subtract)
                        acc = fma(-l[u][2], uu[u][2], fma(-l[u][1], uu[u][1], fma(-l[u][0], uu[u][0], acc)));
            };
            pairs(q0, pa);
            blocks(pa, la, ua);
            pairs(q0 + KP, pb);
            for (int q = q0; q < q1;) {
                if (q + KP < q1) {
                    blocks(pb, lb, ub);
                    pairs(q + 2 * KP, pa);
                }
                subtract(q, la, ua);
                q += KP;
                if (q >= q1) break;
                if (q + KP < q1) {
                    blocks(pa, la, ua);
                    pairs(q + 2 * KP, pb);
                }
                subtract(q, lb, ub);
                q += KP;
            }
            s[e9] = acc;
        }
        if (lane_on && tl1 + 3 * warp + grp < tl2) target(tl1 + 3 * warp + grp);  // of the next level
        int2 lq[KC];
#pragma unroll
        for (int u = 0; u < KC; u++) {
            const int i = l0 + 3 * (warp + nwarp * u) + grp;
            lq[u] = lane_on && i < l1 ? fd.ls[i] : make_int2(-1, -1);
        }
        __syncthreads();
        for (int p = p0; p < lp1; p += T) {
            double* d = slot + (long long)(p == p0 ? dpos : fd.diag_of_pos[p]) * 9;
            const int row = p == p0 ? rpos : fd.row_of_pos[p];
            double D[3][3];
#pragma unroll
            for (int e = 0; e < 9; e++) D[e / 3][e % 3] = d[e];
            double* dp = fd.dpiv + (long long)row * 9;
#pragma unroll
            for (int e = 0; e < 9; e++) dp[e] = D[e / 3][e % 3];
            if (!inverse3(D)) {
                if (atomicCAS(&err->flag, 0, 1) == 0) {
                    err->sub = ids ? ids[blockIdx.x] : blockIdx.x;
                    err->row = row;
                }
#pragma unroll
                for (int e = 0; e < 9; e++) D[e / 3][e % 3] = (e % 4 == 0) ? 1.0 : 0.0;
            }
#pragma unroll
            for (int e = 0; e < 9; e++) d[e] = D[e / 3][e % 3];
        }
        __syncthreads();
        // KC items of a lane at a time: their blocks, and the next ones' indices, are loaded before any arithmetic
        for (int i0 = l0 + 3 * warp; i0 < l1; i0 += 3 * nwarp * KC) {
            int2 q[KC];
            double a[KC][3], di[KC][3];
#pragma unroll
            for (int u = 0; u < KC; u++) {
                q[u] = lq[u];
                const int i = i0 + grp + 3 * nwarp * (KC + u);
                lq[u] = lane_on && i < l1 ? fd.ls[i] : make_int2(-1, -1);
            }
#pragma unroll
            for (int u = 0; u < KC; u++) {
                const double* A = slot + (long long)max(q[u].x, 0) * 9 + 3 * er;
                const double* Di = slot + (long long)max(q[u].y, 0) * 9 + ec;
#pragma unroll
                for (int k = 0; k < 3; k++) {
                    a[u][k] = q[u].x >= 0 ? A[k] : 0.0;
                    di[u][k] = q[u].x >= 0 ? Di[3 * k] : 0.0;
                }
            }
            __syncwarp();  // every lane of a group has read its row of L before any writes
#pragma unroll
            for (int u = 0; u < KC; u++)
                if (q[u].x >= 0)
                    slot[(long long)q[u].x * 9 + e9] = a[u][0] * di[u][0] + a[u][1] * di[u][1] + a[u][2] * di[u][2];
        }
        __syncthreads();
        tl0 = tl1, tl1 = tl2, lp0 = lp1, lp1 = lp2, l0 = l1, l1 = l2;
    }
}

// One thread per 3x3 block.  FP16 blocks are stored as 9 halves of v * 2^-e followed by e (int16),
// with e chosen so that the largest magnitude lands in [0.5, 1): U (~T) and D^{-1} (~1/T) then both
// keep FP16's full relative precision instead of overflowing or underflowing.
template <typename T>
__global__ void k_pack(const long long* __restrict__ off, const int* __restrict__ src, long long n,
                       unsigned char* __restrict__ base, const double* __restrict__ slot) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double* v = slot + (long long)src[i] * 9;
    if constexpr (sizeof(T) == 2) {
        double mx = 0.0;
#pragma unroll
        for (int e = 0; e < 9; e++) mx = fmax(mx, fabs(v[e]));
        int ex = 0;
        if (mx > 0.0) ex = ilogb(mx) + 1;
        __half* dst = reinterpret_cast<__half*>(base + off[i]);
#pragma unroll
        for (int e = 0; e < 9; e++) dst[e] = __double2half(ldexp(v[e], -ex));
        reinterpret_cast<short*>(dst)[9] = (short)ex;
    } else {
        T* dst = reinterpret_cast<T*>(base + off[i]);
#pragma unroll
        for (int e = 0; e < 9; e++) dst[e] = (T)v[e];
    }
}

// The same blocks into the packets of the stream by lane: element (k, t) of a block lies 30 t + lane
// values from its offset, the lanes of k = 0, 1, 2 next to each other (eight apart in the packet of a
// long lump row); an FP16 row's record is {three halves, exponent} per lane.  Neighbouring threads hold
// neighbouring rows of a packet.
template <typename T>
__global__ void k_pack_lanes(const long long* __restrict__ off, const int* __restrict__ src, long long n,
                             unsigned char* __restrict__ base, const double* __restrict__ slot) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double* v = slot + (long long)src[i] * 9;
    const long long o = off[i];
    unsigned char* dst = base + (o >= 0 ? o : ~o);
    if constexpr (sizeof(T) == 2) {
        double mx = 0.0;
#pragma unroll
        for (int e = 0; e < 9; e++) mx = fmax(mx, fabs(v[e]));
        const int ex = mx > 0.0 ? ilogb(mx) + 1 : 0;
#pragma unroll
        for (int k = 0; k < 3; k++) {
            unsigned short h[3];
#pragma unroll
            for (int t = 0; t < 3; t++) h[t] = __half_as_ushort(__double2half(ldexp(v[3 * k + t], -ex)));
            reinterpret_cast<uint2*>(dst)[k] =
                make_uint2(h[0] | (unsigned)h[1] << 16, h[2] | (unsigned)(unsigned short)(short)ex << 16);
        }
    } else {
        const int lane = o >= 0 ? 1 : 8;
#pragma unroll
        for (int k = 0; k < 3; k++)
#pragma unroll
            for (int t = 0; t < 3; t++) reinterpret_cast<T*>(dst)[30 * t + lane * k] = (T)v[3 * k + t];
    }
}

// a warp per part (a few hundred bytes; a few MB in all, once per structure)
__global__ void __launch_bounds__(256) k_place(const PkPiece* __restrict__ pieces, int n, const int4* __restrict__ src,
                                               int4* __restrict__ dst) {
    const int i = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    if (i >= n) return;
    const PkPiece p = pieces[i];
    for (int k = threadIdx.x & 31; k < p.n; k += 32) dst[(long long)p.dst + k] = src[(long long)p.src + k];
}

inline unsigned blocks_for(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace

void launch_ell_fill(const double* bsr_vals, const int* row_ptr, int n, int ell_w, double* ell_val, int rows_pad,
                     cudaStream_t st) {
    if (n <= 0 || ell_w <= 0) return;
    k_ell_fill<<<blocks_for((long long)ell_w * n, 256), 256, 0, st>>>(bsr_vals, row_ptr, n, ell_w, ell_val, rows_pad);
}

void launch_coarse(const int* cptr, const int* cloc, const double* bsr_val, double* cval, int nc,
                   cudaStream_t st) {
    if (nc <= 0) return;
    k_coarse<<<nc, 256, 0, st>>>(cptr, cloc, bsr_val, cval);
}

void launch_assemble(const int* aptr, const int* aloc, const int* acs, const double* bsr_val,
                     const double* cval, double* slot, long long nslot, cudaStream_t st, const int* long_slots,
                     int nlong) {
    if (nslot <= 0) return;
    const int long_min = long_slots ? kLongAssembly : 0x7fffffff;
    k_assemble<<<blocks_for(nslot * 9, 256), 256, 0, st>>>(aptr, aloc, acs, bsr_val, cval, slot, nslot,
                                                           long_min);
    if (long_slots && nlong > 0)
        k_assemble_long<<<(nlong + 7) / 8, 256, 0, st>>>(aptr, aloc, acs, bsr_val, cval, slot, long_slots,
                                                         nlong);
}

void launch_factor(const FactDesc* fd, int nsub, int sms, FactErr* err, const int* sub_ids, cudaStream_t st) {
    if (nsub <= 0) return;
    // As many threads as are resident with every CTA of the launch on the chip at once.  128 x 128 x 32 cells in
    // 256 subdomains, the whole re-factor: 4.07 ms with 512 threads and two CTAs per SM, 4.60 with one, 4.34 with
    // four of 256 threads; 64 subdomains (64 x 64 x 16): 0.94 with 512 threads of 126 registers, 0.99 with 1,024 of
    // 64, 1.17 with 256; 512 subdomains (128 x 128 x 64): 8.35 with four of 256, 8.92 with two of 512.
    if (nsub <= sms)
        k_factor<512, 1, 2, 3><<<nsub, 512, 0, st>>>(fd, sub_ids, err);
    else if (nsub <= 2 * sms)
        k_factor<512, 2, 2, 2><<<nsub, 512, 0, st>>>(fd, sub_ids, err);
    else
        k_factor<256, 4, 2, 2><<<nsub, 256, 0, st>>>(fd, sub_ids, err);
}

void launch_pack(const long long* off, const int* src, long long n, int prec, unsigned char* stream_base,
                 const double* slot_base, cudaStream_t st) {
    if (n <= 0) return;
    unsigned g = blocks_for(n, 256);
    if (prec == 0)
        k_pack<double><<<g, 256, 0, st>>>(off, src, n, stream_base, slot_base);
    else if (prec == 1)
        k_pack<float><<<g, 256, 0, st>>>(off, src, n, stream_base, slot_base);
    else
        k_pack<__half><<<g, 256, 0, st>>>(off, src, n, stream_base, slot_base);
}

void launch_place(const PkPiece* pieces, int n, const void* src, void* dst, cudaStream_t st) {
    if (n <= 0) return;
    k_place<<<blocks_for(32LL * n, 256), 256, 0, st>>>(pieces, n, static_cast<const int4*>(src), static_cast<int4*>(dst));
}

void launch_pack_lanes(const long long* off, const int* src, long long n, int prec, unsigned char* stream_base,
                       const double* slot_base, cudaStream_t st) {
    if (n <= 0) return;
    const unsigned g = blocks_for(n, 256);
    if (prec == 0)
        k_pack_lanes<double><<<g, 256, 0, st>>>(off, src, n, stream_base, slot_base);
    else if (prec == 1)
        k_pack_lanes<float><<<g, 256, 0, st>>>(off, src, n, stream_base, slot_base);
    else
        k_pack_lanes<__half><<<g, 256, 0, st>>>(off, src, n, stream_base, slot_base);
}

}  // namespace asm2
