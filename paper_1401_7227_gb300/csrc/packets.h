// The factor stream by lane: the rows of every stream chunk (symbolic.h) laid out in packets of one
// warp, so that a lane of the apply finds its operands and values at fixed offsets from one pointer
// and decodes nothing.  A chunk's packets hold its rows with the same entries in the same order, and
// the lanes that share a row are those of the other layout, so both layouts give the same bits.
//
// Chunk:   byte end[16]: warp w takes the packets end[w - 1] .. end[w] - 1; int4 {byte offset of the packet, of its
//          values, kind, 0} per packet; the packets, each on a 16-byte boundary (as is every array below).
// Packet:  ten positions p (a row, or a row's entry slot), three lanes each -- lane 3 p + k computes output
//          component k; in a kPkLong packet one row over eight slots, lane 8 k + p.
//          int out[10]      byte offset of the position's row in the local vectors, or -1
//          int idx[E][10]   byte offset of the operand row of the position's e-th entry
//          val[E][3][30]    element (k, t) of that entry's block at [e][t][lane] (FP16 rows: one 8-byte record
//                           {(k,0), (k,1), (k,2), exponent} at [e][lane])
//          dinv[3][30]      backward chunks: element (k, t) of D^{-1} at [t][lane of the row's first position]
// Positions and entries a row does not have point at a zero row behind the local vectors, with zero values.
#pragma once

#include <algorithm>
#include <cstring>
#include <vector>

#include "asm2_internal.h"

namespace asm2 {

// kind word of a packet: entries | type << 8 | log2(slots per row) << 12 | backward << 16
enum { kPkFine = 0, kPkLump = 1, kPkLong = 2 };
constexpr int kPkMaxEntries = 255;  // longer rows (a cell coupled to hundreds of others) are not laid out by lane
constexpr int kPkPos = 10, kPkLanes = 30;  // positions and lanes of a packet
constexpr int kPkIdx = 48;  // byte offset of idx in a packet (out[10], padded)

inline int pk_val_offset(int entries) { return (kPkIdx + 4 * kPkPos * entries + 15) & ~15; }

// End of the chunks whose copies are in flight when the apply gives up at chunk ci of n: the first `slots` are issued
// ahead, and after chunk c the copy of chunk c + slots, but not after chunk ci - 1, where the wait for ci ran out.
__host__ __device__ inline int pk_issued_end(int ci, int slots, int n) {
    const int end = ci > 0 ? ci - 1 + slots : slots;
    return end < n ? end : n;
}

// A part of a stream, in units of 16 bytes: its place in the stream and in the bytes that hold such parts back to back.
struct PkPiece {
    int dst, src, n;
};

// The parts of a subdomain's stream by rows that are not values (symbolic.h): of each chunk the header with the fine
// rows' pointers and columns, and the lump rows' pointers and columns.  add(byte offset, bytes) for each.
template <class F>
void rows_index_pieces(const std::vector<unsigned char>& stream, const std::vector<long long>& chunk_off, int n_fwd, int prec,
                       F add) {
    const auto a16 = [](size_t x) { return (x + 15) & ~(size_t)15; };
    const size_t fbb = prec == 0 ? 72 : (prec == 1 ? 36 : 20);
    for (size_t i = 0; i < chunk_off.size(); i++) {
        int h[8];
        std::memcpy(h, stream.data() + chunk_off[i], sizeof(h));
        const size_t nf = (size_t)h[1], nc = (size_t)h[3], ef = (size_t)h[4], ec = (size_t)h[5];
        const size_t fine = 32 + a16(4 * (nf + 1)) + a16(4 * ef), values = a16(fbb * ef) + ((int)i < n_fwd ? 0 : a16(fbb * nf));
        add(chunk_off[i], fine);
        add(chunk_off[i] + (long long)(fine + values), a16(4 * (nc + 1)) + a16(4 * ec));
    }
}

struct Packets {
    std::vector<unsigned char> stream;  // out and idx filled in, values zero
    std::vector<long long> chunk_off;
    std::vector<int> chunk_bytes;
    int cap = 0;  // the largest chunk
    // value blocks: byte offset of element (0, 0), ~ for a kPkLong packet's (lane stride 8), and
    // the slot that holds the block; fine rows, then lump rows
    std::vector<long long> off_f, off_c;
    std::vector<int> src_f, src_c;
};

// stream, chunk_off, src_f, src_c: a subdomain's chunks and the slots of its value blocks in stream order
// (SubSym).  prec / lump32 as in build_symbolic; not for FP64 lump rows under narrower fine rows.  P is left
// empty where a chunk does not fit the format.
inline void build_packets(const std::vector<unsigned char>& stream, const std::vector<long long>& chunk_off, int n_fwd,
                          const std::vector<int>& src_f, const std::vector<int>& src_c, int nf_all, int nc_all, int prec,
                          bool lump32, Packets& P) {
    const YLayout L = y_layout(nf_all, nc_all, prec, lump32);
    const int row = prec == 0 ? 24 : 16, wl = prec == 0 ? 8 : 4;
    const auto y_of = [&](int c) { return c >= 0 ? (int)L.fine + row * c : row * ~c; };
    const int zero = (int)L.total;
    const auto a16 = [](size_t x) { return (x + 15) & ~(size_t)15; };
    // bytes of one entry's values in a packet, and from one t to the next
    const auto entry_bytes = [&](bool fine) { return (size_t)(fine && prec == 2 ? 8 * kPkLanes : 3 * kPkLanes * wl); };
    struct Row {
        int out, e0, ne, src0, dsrc;  // entries e0 ..; value slots src0 .., D^{-1} slot
        const int* col;
    };
    struct Pk {
        int type, lg, entries, first, rows;
        size_t bytes;
    };
    P = Packets();
    P.stream.reserve(stream.size() / 2 * 3);
    P.off_f.reserve(src_f.size());
    P.src_f.reserve(src_f.size());
    P.off_c.reserve(src_c.size());
    P.src_c.reserve(src_c.size());
    size_t kf = 0, kc = 0;
    std::vector<Row> rows;
    std::vector<Pk> pks;
    for (size_t i = 0; i < chunk_off.size(); i++) {
        const bool lower = (int)i < n_fwd;
        const unsigned char* base = stream.data() + chunk_off[i];
        int h[8];
        std::memcpy(h, base, 32);
        const int f0 = h[0], nf = h[1], c0 = h[2], nc = h[3], ef = h[4], ec = h[5], lump_lg = (h[6] >> 8) & 15;
        const size_t fbb = prec == 0 ? 72 : (prec == 1 ? 36 : 20), lbb = lump32 ? 36 : 72;
        const int* fptr = reinterpret_cast<const int*>(base + 32);
        const int* fcol = reinterpret_cast<const int*>(base + 32 + a16(4 * (size_t)(nf + 1)));
        size_t w = 32 + a16(4 * (size_t)(nf + 1)) + a16(4 * (size_t)ef) + a16(fbb * ef) + (lower ? 0 : a16(fbb * nf));
        const int* cptr = reinterpret_cast<const int*>(base + w);
        const int* ccol = reinterpret_cast<const int*>(base + w + a16(4 * (size_t)(nc + 1)));
        (void)lbb;
        rows.clear();
        pks.clear();
        const auto add = [&](int type, int lg, std::vector<Row>& rs) {
            // rows of similar length share a packet
            std::stable_sort(rs.begin(), rs.end(), [](const Row& a, const Row& b) { return a.ne > b.ne; });
            const int S = 1 << lg, per = type == kPkLong ? 1 : kPkPos / S;
            for (size_t r = 0; r < rs.size(); r += per) {
                Pk k{type, lg, 0, (int)rows.size(), (int)std::min<size_t>(per, rs.size() - r), 0};
                for (int q = 0; q < k.rows; q++) {
                    k.entries = std::max(k.entries, (rs[r + q].ne + S - 1) / S);
                    rows.push_back(rs[r + q]);
                }
                const bool fine = type == kPkFine;
                k.bytes = a16(pk_val_offset(k.entries) + entry_bytes(fine) * (k.entries + (lower ? 0 : 1)));
                pks.push_back(k);
            }
        };
        std::vector<Row> fine, shrt, lng;
        for (int r = 0; r < nf; r++)
            fine.push_back(Row{y_of(f0 + r), fptr[r], fptr[r + 1] - fptr[r], (int)(kf + fptr[r]), (int)(kf + ef + r), fcol});
        for (int r = 0; r < nc; r++) {
            const Row q{y_of(~(c0 + r)), cptr[r], cptr[r + 1] - cptr[r], (int)(kc + cptr[r]), (int)(kc + ec + r), ccol};
            (q.ne > kLongLumpRow ? lng : shrt).push_back(q);
        }
        kf += ef + (lower ? 0 : nf);
        kc += ec + (lower ? 0 : nc);
        add(kPkFine, 0, fine);
        add(kPkLump, lump32 ? 0 : lump_lg, shrt);
        add(kPkLong, 3, lng);
        // The longest packets first, each to the warp with the least to do: in FP64 to the SM sub-partition
        // (warps w, w + 4, ...) with the fewest FP64 operations, whose unit they share, and within it to the
        // warp with fewest; in FP32, where a packet costs ~150 cycles and ~13 per entry, by that.
        const auto cost = [&](const Pk& k) {
            return prec == 0 ? 3 * k.entries + (lower ? 1 : 4) + k.lg : 150 + 13 * k.entries;
        };
        std::stable_sort(pks.begin(), pks.end(), [&](const Pk& a, const Pk& b) { return cost(a) > cost(b); });
        int load[kPkWarps] = {};
        std::vector<int> warp_of(pks.size());
        for (size_t q = 0; q < pks.size(); q++) {
            int best = 0;
            const auto part = [&](int w) { return load[w & 3] + load[(w & 3) + 4] + load[(w & 3) + 8] + load[(w & 3) + 12]; };
            for (int w = 1; w < kPkWarps - 1; w++)  // (the last one waits for the next chunk)
                if (prec == 0 ? part(w) < part(best) || (part(w) == part(best) && load[w] < load[best]) : load[w] < load[best])
                    best = w;
            load[best] += cost(pks[q]);
            warp_of[q] = best;
        }
        std::vector<Pk> by_warp;
        static_assert(kPkWarps == 16, "four warps per SM sub-partition, a 16-byte table");
        unsigned char end[kPkWarps] = {};
        for (int w = 0; w < kPkWarps; w++) {
            for (size_t q = 0; q < pks.size(); q++)
                if (warp_of[q] == w) by_warp.push_back(pks[q]);
            end[w] = (unsigned char)by_warp.size();
        }
        bool fits = by_warp.size() <= 255;  // (a chunk of at most 24 KB holds fewer)
        for (const Pk& k : by_warp) fits = fits && k.entries <= kPkMaxEntries;
        if (!fits) {
            P = Packets();
            return;
        }
        pks.swap(by_warp);
        size_t total = 16 + 16 * pks.size();
        const size_t head = total;
        for (const Pk& k : pks) total += k.bytes;
        const size_t off0 = P.stream.size();
        P.chunk_off.push_back((long long)off0);
        P.chunk_bytes.push_back((int)total);
        P.cap = std::max(P.cap, (int)total);
        P.stream.resize(off0 + total, 0);
        int* hd = reinterpret_cast<int*>(P.stream.data() + off0);
        std::memcpy(hd, end, sizeof(end));
        size_t at = head;
        for (size_t q = 0; q < pks.size(); q++) {
            const Pk& k = pks[q];
            hd[4 + 4 * q] = (int)at;
            hd[5 + 4 * q] = (int)at + pk_val_offset(k.entries);
            hd[6 + 4 * q] = k.entries | k.type << 8 | k.lg << 12 | (lower ? 0 : 1) << 16;
            int* out = reinterpret_cast<int*>(P.stream.data() + off0 + at);
            int* idx = out + kPkIdx / 4;
            for (int p = 0; p < kPkPos; p++) out[p] = -1;
            for (int p = 0; p < kPkPos * k.entries; p++) idx[p] = zero;
            const int S = 1 << k.lg;
            const bool is_fine = k.type == kPkFine, is_long = k.type == kPkLong;
            const size_t val = off0 + at + pk_val_offset(k.entries), eb = entry_bytes(is_fine);
            const int w1 = is_fine && prec == 2 ? 8 : wl;  // bytes from one lane to the next
            std::vector<long long>& off = is_fine ? P.off_f : P.off_c;
            std::vector<int>& src = is_fine ? P.src_f : P.src_c;
            const std::vector<int>& from = is_fine ? src_f : src_c;
            // entry by entry, so that consecutive blocks are neighbours in the packet
            const auto place = [&](int pos, size_t o, int s) {
                const long long b = (long long)(o + (size_t)(is_long ? pos : 3 * pos) * w1);
                off.push_back(is_long ? ~b : b);
                src.push_back(s);
            };
            for (int q2 = 0; q2 < k.rows; q2++)
                for (int s = 0; s < S; s++) out[q2 * S + s] = rows[k.first + q2].out;
            for (int e = 0; e < k.entries; e++)
                for (int q2 = 0; q2 < k.rows; q2++) {
                    const Row& r = rows[k.first + q2];
                    for (int s = 0; s < S; s++)
                        if (e * S + s < r.ne) {
                            idx[kPkPos * e + q2 * S + s] = y_of(r.col[r.e0 + e * S + s]);
                            place(q2 * S + s, val + eb * e, from[r.src0 + e * S + s]);
                        }
                }
            if (!lower)
                for (int q2 = 0; q2 < k.rows; q2++) place(q2 * S, val + eb * k.entries, from[rows[k.first + q2].dsrc]);
            at += k.bytes;
        }
    }
}

}  // namespace asm2
