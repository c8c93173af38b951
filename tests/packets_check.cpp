// Test-only: builds both layouts of the factor stream (symbolic.cpp) on the CPU and compares them chunk by
// chunk.  Not part of the library.
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <vector>

#include "symbolic.h"

using namespace asm2;

namespace {

struct RowOf {
    int type = 0, lg = 0;
    std::vector<std::pair<int, int>> entries;  // operand row (byte offset), value slot
    int dsrc = -1;
    bool operator==(const RowOf& o) const {
        return type == o.type && lg == o.lg && entries == o.entries && dsrc == o.dsrc;
    }
};

std::string check_sub(const SubSym& o, int prec, bool lump32) {
    const YLayout L = y_layout(o.nf, o.n - o.nf, prec, lump32);
    const int row = prec == 0 ? 24 : 16, wl = prec == 0 ? 8 : 4;
    const auto y_of = [&](int c) { return c >= 0 ? (int)L.fine + row * c : row * ~c; };
    const auto a16 = [](size_t x) { return (x + 15) & ~(size_t)15; };
    if (o.pk.chunk_off.size() != o.chunk_off.size()) return "chunk count";
    // value slots by place: fine rows' and lump rows' blocks of the stream by lane
    std::map<long long, int> src;
    std::set<long long> bytes;  // 4-byte words taken by values
    for (int g = 0; g < 2; g++) {
        const auto& off = g ? o.pk.off_c : o.pk.off_f;
        const auto& s = g ? o.pk.src_c : o.pk.src_f;
        if (off.size() != (g ? o.pk_off_c : o.pk_off_f).size()) return "value count";
        for (size_t i = 0; i < off.size(); i++) {
            const bool lng = off[i] < 0;
            const long long b = lng ? ~off[i] : off[i];
            if (!src.emplace(b, s[i]).second) return "two blocks at one place";
            const bool half = g == 0 && prec == 2;
            for (int k = 0; k < 3; k++)
                for (int t = 0; t < (half ? 1 : 3); t++)
                    for (int w = 0; w < (half ? 8 : wl); w += 4) {
                        const long long at = b + (half ? 8 * k : (30LL * t + (lng ? 8 : 1) * k) * wl) + w;
                        if (at % 4 != 0 || !bytes.insert(at).second) return "values overlap";
                    }
        }
    }
    size_t kf = 0, kc = 0;
    for (size_t i = 0; i < o.chunk_off.size(); i++) {
        const bool lower = (int)i < o.n_fwd_chunks;
        // by rows
        std::map<int, RowOf> want, got;
        const unsigned char* b = o.stream.data() + o.chunk_off[i];
        int h[8];
        std::memcpy(h, b, 32);
        size_t w = 32;
        for (int g = 0; g < 2; g++) {
            const int n = h[g ? 3 : 1], ne = h[g ? 5 : 4], r0 = h[g ? 2 : 0];
            const size_t bb = g ? (lump32 ? 36 : 72) : (prec == 0 ? 72 : prec == 1 ? 36 : 20);
            const int* ptr = reinterpret_cast<const int*>(b + w);
            const int* col = reinterpret_cast<const int*>(b + w + a16(4 * (size_t)(n + 1)));
            w += a16(4 * (size_t)(n + 1)) + a16(4 * (size_t)ne) + a16(bb * ne) + (lower ? 0 : a16(bb * n));
            const std::vector<int>& ps = g ? o.pk_src_c : o.pk_src_f;
            size_t& k0 = g ? kc : kf;
            for (int r = 0; r < n; r++) {
                RowOf R;
                R.type = g == 0 ? kPkFine : ptr[r + 1] - ptr[r] > kLongLumpRow ? kPkLong : kPkLump;
                R.lg = R.type == kPkLong ? 3 : R.type == kPkLump && !lump32 ? (h[6] >> 8) & 15 : 0;
                for (int e = ptr[r]; e < ptr[r + 1]; e++) R.entries.push_back({y_of(col[e]), ps[k0 + e]});
                if (!lower) R.dsrc = ps[k0 + ne + r];
                want[y_of(g ? ~(r0 + r) : r0 + r)] = R;
            }
            k0 += ne + (lower ? 0 : n);
        }
        // by lane
        const long long c0 = o.pk.chunk_off[i], cb = o.pk.chunk_bytes[i];
        const unsigned char* p = o.pk.stream.data() + c0;
        if (cb > o.pk.cap || cb % 16 != 0) return "chunk size";
        int np = 0;
        for (int q = 0; q < kPkWarps; q++) {
            if (p[q] < np) return "warp table";
            np = p[q];
        }
        for (int q = 0; q < np; q++) {
            int d[4];
            std::memcpy(d, p + kPkWarps + 16 * q, 16);
            const int E = d[2] & 255, type = (d[2] >> 8) & 15, lg = (d[2] >> 12) & 15, S = 1 << lg;
            if ((d[2] >> 16 == 0) != lower || d[0] % 16 != 0 || d[1] != d[0] + pk_val_offset(E)) return "packet head";
            const bool half = type == kPkFine && prec == 2;
            const long long eb = half ? 240 : 90LL * wl;
            if (d[1] + eb * (E + (lower ? 0 : 1)) > cb) return "packet past its chunk";
            const int* out = reinterpret_cast<const int*>(p + d[0]);
            const int* idx = out + kPkIdx / 4;
            for (int r = 0; r < kPkPos / S || (type == kPkLong && r < 1); r++) {
                const int pos0 = r * S;
                if (pos0 + S > kPkPos) break;
                if (out[pos0] < 0) continue;
                RowOf R;
                R.type = type;
                R.lg = lg;
                const auto place = [&](int pos, int e) {
                    return c0 + d[1] + eb * e + (long long)(type == kPkLong ? pos : 3 * pos) * (half ? 8 : wl);
                };
                for (int e = 0; e < E * S; e++) {
                    const int pos = pos0 + e % S;
                    if (out[pos] != out[pos0]) return "a row's positions differ";
                    const auto f = src.find(place(pos, e / S));
                    const int x = idx[kPkPos * (e / S) + pos];
                    if (f == src.end()) {
                        if (x != (int)L.total) return "padding reads a row";
                        continue;
                    }
                    R.entries.push_back({x, f->second});
                }
                if (!lower) {
                    const auto f = src.find(place(pos0, E));
                    if (f == src.end()) return "no D^{-1}";
                    R.dsrc = f->second;
                }
                if (!got.emplace(out[pos0], R).second) return "a row twice";
            }
        }
        if (got.size() != want.size()) return "row count";
        for (const auto& kv : want)
            if (!got.count(kv.first) || !(got[kv.first] == kv.second)) return "a row's entries differ";
    }
    return "";
}

}  // namespace

namespace {

// the stream by rows is its index parts over zeros (the values are not filled in on the host)
std::string check_rows_pieces(const SubSym& o, int prec) {
    std::vector<unsigned char> out(o.stream.size(), 0);
    std::string e;
    size_t bytes = 0;
    rows_index_pieces(o.stream, o.chunk_off, o.n_fwd_chunks, prec, [&](long long at, size_t n) {
        if (at < 0 || at % 16 != 0 || n % 16 != 0 || n == 0 || at + n > out.size()) {
            e = "piece range";
            return;
        }
        std::memcpy(out.data() + at, o.stream.data() + at, n);
        bytes += n;
    });
    if (!e.empty()) return e;
    // and none of it is a value's place: every block's bytes lie outside the parts
    std::vector<char> index(o.stream.size(), 0);
    rows_index_pieces(o.stream, o.chunk_off, o.n_fwd_chunks, prec,
                      [&](long long at, size_t n) { std::memset(index.data() + at, 1, n); });
    const size_t fbb = prec == 0 ? 72 : (prec == 1 ? 36 : 20), lbb = prec == 0 ? 72 : 36;
    for (long long at : o.pk_off_f)
        for (size_t k = 0; k < fbb; k++)
            if (index[at + k]) return "a value in a part";
    for (long long at : o.pk_off_c)
        for (size_t k = 0; k < lbb; k++)
            if (index[at + k]) return "a value in a part";
    return out == o.stream && bytes < o.stream.size() ? "" : "parts";
}

}  // namespace

// geo as in host_symbolic_shim.cpp; 0, or 1 with the first difference in err
extern "C" int pk_check(const int* geo, int n, int nnzb, const int* rp, const int* ci, int prec, int chunk_force, char* err,
                        int errlen) {
    Geom g;
    g.nx = geo[0], g.ny = geo[1], g.nz = geo[2], g.px = geo[3], g.py = geo[4], g.pz = geo[5], g.ov = geo[6], g.nw = geo[7];
    for (int d = 0; d < 3; d++) g.cn[d] = geo[8 + d], g.cf[d] = geo[12 + d];
    g.far_mode = geo[11];
    Pattern P;
    SysSym S;
    const bool lump32 = prec != 0;
    std::string e = build_pattern(n, rp, ci, nnzb, P);
    if (e.empty()) e = build_symbolic(g, P, prec, lump32, 1, S, 0, chunk_force, true);
    for (size_t s = 0; e.empty() && s < S.subs.size(); s++) e = check_rows_pieces(S.subs[s], prec);
    for (size_t s = 0; e.empty() && s < S.subs.size(); s++) e = check_sub(S.subs[s], prec, lump32);
    std::strncpy(err, e.c_str(), (size_t)errlen - 1);
    err[errlen - 1] = 0;
    return e.empty() ? 0 : 1;
}

// wants_lanes of a geometry; in *fits whether every subdomain's local vectors and the row of zeros fit smem bytes
extern "C" int pk_wanted(const int* geo, int n, int nnzb, const int* rp, const int* ci, int prec, int sms, int smem, int* fits) {
    Geom g;
    g.nx = geo[0], g.ny = geo[1], g.nz = geo[2], g.px = geo[3], g.py = geo[4], g.pz = geo[5], g.ov = geo[6], g.nw = geo[7];
    for (int d = 0; d < 3; d++) g.cn[d] = geo[8 + d], g.cf[d] = geo[12 + d];
    g.far_mode = geo[11];
    Pattern P;
    SysSym S;
    if (!build_pattern(n, rp, ci, nnzb, P).empty() || !build_symbolic(g, P, prec, prec != 0, 1, S, 0).empty()) return -1;
    *fits = 1;
    for (const SubSym& o : S.subs)
        if ((long long)y_layout(o.nf, o.n - o.nf, prec, prec != 0).total + 32 > smem) *fits = 0;
    return wants_lanes(g, prec, sms, smem);
}

// The ring of k_apply_packets step by step: the wait for chunk `expire` runs out.  0 if the chunks expire ..
// pk_issued_end - 1 are just those whose copies were issued and not waited for.
extern "C" int pk_drain_check(int slots, int n, int expire) {
    std::set<int> flying;
    for (int k = 0; k < slots && k < n; k++) flying.insert(k);
    for (int ci = 0; ci < expire; ci++) {
        flying.erase(ci);                               // landed before chunk ci was worked on
        const bool expired = ci + 1 == expire;          // the wait for the next one, before the refill
        if (!expired && ci + slots < n) flying.insert(ci + slots);
    }
    std::set<int> drained;
    for (int k = expire; k < pk_issued_end(expire, slots, n); k++) drained.insert(k);
    return drained == flying ? 0 : 1;
}
