// Strip kernels of fused groups (Section 5: code generated per fused
// partition of the graph).
//
// The tile form (codegen.cpp) passes every image of a group through shared
// memory, one int32 cell per operation.  A group whose images are all U8, S16
// or UYVY can do better: a thread owns a strip of 8 columns and R rows and
// walks down it, keeping for every image the few rows its consumers' windows
// reach as pixel pairs in 16-bit lanes of registers.  One 32-bit operation
// then works on two pixels, every row of every image is computed once per
// strip, and shared memory holds only the input tile, brought by one TMA box.
// What bounds it is instruction issue (the halo columns of chained local
// operators are recomputed by each strip) or, for short groups, HBM.
//
// Measured against the tile form (GB300, one launch): FChain 16 x 1080p 126.5
// -> 52 us (106 -> 35 instructions per pixel), Unsharp 16 x 2043x1361 77.8 ->
// 26 us (43 -> 11 instructions, 5.1 TB/s of reads and writes), Laplacian 16 x
// 1080p 47.9 -> 20.5 us, a morphology graph on one 1080p frame 18.7 -> 5.5 us,
// 64x48 frames equal.  Tried and left out, at 61.7 and 37 us on the first two:
// persistent CTAs with two box stages (FChain 65, Unsharp 48 us: the second
// box costs more resident CTAs than the overlap gains back), one step
// function with run-time stage conditions instead of the phases below (97 us:
// the windows no longer rotate by renaming).
//
// Exactness.  Every image has a static range [lo, hi] of values and a bias B;
// a lane holds v + B in [0, 65535].  A linear combination of lane words is
// computed in 32-bit arithmetic modulo 2^32: with integer coefficients the
// word of the sums is the sum of the words, whatever happens in between, so
// only the final lanes have to lie in [0, 65535], which a constant added to
// both lanes ensures (checked here from the ranges; a group that does not fit
// keeps the tile form).  Lanes that no stored output depends on hold values of
// the same ranges, so they never disturb their neighbours.  Operators that
// are not linear, minima, maxima or bit operations are evaluated per pixel on
// unpacked lanes with the shared scalar arithmetic.
//
// Rows.  At the step of output row y, image b receives its row y + h_b (h_b its
// halo); a window of D_b rows, the newest last, serves its consumers.  The
// steps before the first output row (the prologue, S < 0) run only the images
// that are needed from there on: b from step -2 h_b.
//
// Borders.  Tiles whose cells all lie in every image's valid region run
// without tests.  The others (EDGE) give the box cells outside the image
// their border value first, zero every lane outside an image's valid region,
// and fill the rows and lanes of intermediate images that lie outside the
// image as their consumers read them: rows above the image get row 0 when it
// has been computed (REPLICATE), rows below repeat the last one.
#include "codegen_strip.h"

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <sstream>

#include "../../include/hvx.h"

namespace hvx {
namespace {

typedef long long ll;

bool local_op(int op) {
    return op == OP_GAUSS || op == OP_BOX || op == OP_SOBEL_X || op == OP_SOBEL_Y ||
           op == OP_CONV || op == OP_DILATE || op == OP_ERODE || op == OP_MEDIAN;
}

std::string hex(uint32_t v) {
    char s[16];
    std::snprintf(s, sizeof(s), "0x%xu", v);
    return s;
}

// Both lanes equal to v (0 <= v <= 65535).
std::string dup(ll v) { return hex((uint32_t)(v & 0xFFFF) * 0x10001u); }

// expr with k added to both lanes (k may be negative).
std::string add_lanes(const std::string& e, ll k) {
    if (k == 0) return e;
    return "(" + e + " + " + hex((uint32_t)((uint64_t)k * 65537ull)) + ")";
}

struct Lane {
    ll lo = 0, hi = 0;  // range of the values
    ll bias = 0;        // a lane holds value + bias
};

struct StripEmitter {
    const GenericDesc& d;
    std::ostringstream o;
    std::vector<int> producer, ext_in;
    std::vector<bool> full;  // the image's valid region is the whole image
    std::vector<Lane> lane;
    std::vector<int> D, E;   // window rows; columns kept left and right of the strip (even)
    int unroll = 0;
    std::string acc_param, acc_arg;  // the global operators' accumulators, if any
    std::string mem_rows, mem_decl;  // inputs without a halo, read straight from memory
    int mem_words = 0;               // ... registers of a row of theirs
    std::vector<StripBox> boxes;
    std::vector<int> globals;     // stages that are global operators, in result order
    std::vector<bool> need_rect;  // the image's valid rectangle is read by EDGE tiles

    explicit StripEmitter(const GenericDesc& desc) : d(desc) {}

    int halo(int b) const { return d.buf[b].halo; }
    int words(int b) const { return 4 + E[b]; }

    // Row of buffer b that a stage of output halo ho reads at dy, as a window index.
    int row_at(int b, int ho, int dy) const { return D[b] - 1 - (halo(b) - ho - dy); }

    std::string word(int b, int row, int off) const {
        const int k = std::min(std::max(off, -E[b]), 6 + E[b]);
        return "w.b" + std::to_string(b) + "[" + std::to_string(row) + "][" +
               std::to_string((k + E[b]) / 2) + "]";
    }

    // The magnitude whose threshold a THRESH stage decides from the gradients.
    int fused_mag(const GenStage& st) const {
        if (st.op != OP_THRESH || st.i3 || st.i0 != HVX_THRESHOLD_BINARY) return -1;
        const int k = producer[st.in[0]];
        return k >= 0 && d.st[k].op == OP_MAG ? k : -1;
    }

    bool plan() {
        producer.assign(d.n_buf, -1);
        ext_in.assign(d.n_buf, -1);
        full.assign(d.n_buf, true);
        lane.assign(d.n_buf, Lane{});
        D.assign(d.n_buf, 1);
        E.assign(d.n_buf, 0);
        for (int e = 0; e < d.n_in; ++e) ext_in[d.in[e].buf] = e;
        for (int b = 0; b < d.n_buf; ++b) {
            const GenBuf& g = d.buf[b];
            if (g.fmt != HVX_DF_U8 && g.fmt != HVX_DF_S16 && g.fmt != HVX_DF_UYVY) return false;
            full[b] = g.valid[0] == 0 && g.valid[1] == 0 && g.valid[2] == d.W && g.valid[3] == d.H;
            E[b] = (g.halo + 1) & ~1;
            if (g.halo > GEN_MAX_HALO) return false;
        }
        need_rect.assign(d.n_buf, false);
        for (int b = 0; b < d.n_buf; ++b) need_rect[b] = !full[b];
        for (int k = 0; k < d.n_stage; ++k) {
            const GenStage& st = d.st[k];
            if (op_is_global(st.op)) {
                const int b = st.in[0];
                globals.push_back(k);
                need_rect[b] = true;
                D[b] = std::max(D[b], 1 + halo(b));
                if (d.buf[b].fmt == HVX_DF_UYVY) return false;
                continue;
            }
            producer[st.out] = k;
            const int ho = halo(st.out), r = local_op(st.op) ? st.ry : 0;
            for (int i = 0; i < 3; ++i)
                if (st.in[i] >= 0)
                    D[st.in[i]] = std::max(D[st.in[i]], 1 + halo(st.in[i]) - ho + r);
            const int m = fused_mag(st);
            if (m >= 0)
                for (int i = 0; i < 2; ++i)
                    D[d.st[m].in[i]] =
                        std::max(D[d.st[m].in[i]], 1 + halo(d.st[m].in[i]) - ho);
        }
        for (int e = 0; e < d.n_out; ++e) {
            const int b = d.out[e].buf;
            D[b] = std::max(D[b], 1 + halo(b));
            if (d.out[e].fmt != HVX_DF_U8 && d.out[e].fmt != HVX_DF_S16) return false;
        }
        int most = 1;
        for (int b = 0; b < d.n_buf; ++b) most = std::max(most, D[b]);
        // three steps a trip let a 3-row window rotate by renaming; longer loops
        // lost more to instruction fetch than they saved in moves (FChain, 16 x
        // 1080p: 62 us at 3, 64 at 1, 65 at 5)
        unroll = most == 1 ? 4 : 3;
        for (int e = 0; e < d.n_in; ++e) {
            const int b = d.in[e].buf, f = d.in[e].fmt;
            Lane& L = lane[b];
            if (f == HVX_DF_U8)
                L.hi = 255;
            else if (f == HVX_DF_UYVY)
                L.hi = 65535;
            else
                L = Lane{-32768, 32767, 32768};
            // 16-bit inputs are read by point operators alone
            if (f != HVX_DF_U8 && d.buf[b].fill != FILL_NONE) return false;
            if (halo(b) > 0) boxes.push_back({e, f == HVX_DF_U8 ? 1 : 2, halo(b)});
        }
        return true;
    }

    // ---- operators ---------------------------------------------------------

    std::string ind = "    ";
    int tmp = 0;

    std::string fresh(const char* p) { return p + std::to_string(tmp++); }

    // Clamps word expression e (range L) to [lo, hi] and moves it to the
    // smallest bias; updates L.
    std::string clamp(std::string e, Lane& L, ll lo, ll hi) {
        if (L.hi > hi) {
            e = "hvx_min2(" + e + ", " + dup(hi + L.bias) + ")";
            L.hi = hi;
        }
        if (L.lo < lo) {
            e = "hvx_max2(" + e + ", " + dup(lo + L.bias) + ")";
            L.lo = lo;
        }
        if (L.hi < L.lo) L.hi = L.lo;
        const ll nb = std::max(0ll, -L.lo);
        if (nb != L.bias) {
            e = add_lanes(e, nb - L.bias);
            L.bias = nb;
        }
        return e;
    }

    static void fmt_range(int fmt, ll* lo, ll* hi) {
        *lo = fmt == HVX_DF_U8 ? 0 : -32768;
        *hi = fmt == HVX_DF_U8 ? 255 : 32767;
    }

    // sum of c[i] * e[i], equal coefficients gathered
    static std::string combine(const std::vector<int>& c, const std::vector<std::string>& e) {
        std::map<int, std::vector<std::string>> by;
        for (size_t i = 0; i < c.size(); ++i)
            if (c[i]) {
                bool neg = by.count(-c[i]) && !by.count(c[i]);
                if (neg)
                    by[-c[i]].push_back("-" + e[i]);
                else
                    by[c[i]].push_back("+" + e[i]);
            }
        std::string s;
        // positive coefficients first
        for (auto it = by.rbegin(); it != by.rend(); ++it) {
            std::string g;
            for (const std::string& t : it->second)
                g += g.empty() ? (t[0] == '-' ? "0u - " + t.substr(1) : t.substr(1))
                               : std::string(t[0] == '-' ? " - " : " + ") + t.substr(1);
            const int m = std::abs(it->first);
            const bool many = it->second.size() > 1;
            std::string v = many ? "(" + g + ")" : g;
            if (m != 1) v = std::to_string(m) + "u * " + v;
            if (it->first > 0)
                s += (s.empty() ? "" : " + ") + v;
            else
                s += (s.empty() ? "0u - " : " - ") + v;
        }
        return s.empty() ? "0u" : s;
    }

    // A linear window operator: floor((sum c v + r0) / 2^shift) clamped to
    // the output format; box: divided by 9 instead.
    bool emit_conv(const GenStage& st, const std::vector<int>& c, int rx, int ry, ll r0, int shift,
                   int fmt, bool box) {
        const int b = st.in[0], ob = st.out, ho = halo(ob);
        const int kw = 2 * rx + 1, kh = 2 * ry + 1;
        const Lane in = lane[b];
        // distinct column vectors: base * m
        struct Col {
            std::vector<int> base;
            Lane L;
            std::vector<std::string> v;  // by word of the input
            bool plain = false;          // the base is one row, unscaled
            int plain_row = 0;
        };
        std::vector<Col> cols;
        std::vector<int> col_of(kw, -1), mult(kw, 0);
        for (int x = 0; x < kw; ++x) {
            std::vector<int> v(kh);
            int g = 0, sign = 0;
            for (int y = 0; y < kh; ++y) {
                v[y] = c[y * kw + x];
                int a = std::abs(v[y]);
                while (a) {
                    const int t = g % a;
                    g = a;
                    a = t;
                }
                if (v[y] && !sign) sign = v[y] > 0 ? 1 : -1;
            }
            if (!g) continue;
            for (int& y : v) y /= g * sign;
            mult[x] = g * sign;
            for (size_t i = 0; i < cols.size(); ++i)
                if (cols[i].base == v) col_of[x] = (int)i;
            if (col_of[x] < 0) {
                col_of[x] = (int)cols.size();
                Col n;
                n.base = v;
                cols.push_back(n);
            }
        }
        // ranges of the column sums and of the whole sum
        ll tlo = 0, thi = 0, konst = 0;
        for (Col& q : cols) {
            ll sum = 0;
            int nz = 0;
            for (int y = 0; y < kh; ++y) {
                const ll k = q.base[y];
                q.L.lo += k * (k > 0 ? in.lo : in.hi);
                q.L.hi += k * (k > 0 ? in.hi : in.lo);
                sum += k;
                if (k) {
                    ++nz;
                    q.plain_row = y - ry;
                }
            }
            q.plain = nz == 1 && sum == 1;
            q.L.bias = q.plain ? in.bias : std::max(0ll, -q.L.lo);
            if (q.L.hi + q.L.bias > 65535 || q.L.lo < -65535) return false;
            q.v.assign(words(b), "");
        }
        for (int x = 0; x < kw; ++x)
            if (mult[x]) {
                const Lane& L = cols[col_of[x]].L;
                const ll m = mult[x];
                tlo += m * (m > 0 ? L.lo : L.hi);
                thi += m * (m > 0 ? L.hi : L.lo);
                konst += m * L.bias;
            }
        const ll unit = box ? 1 : 1ll << shift;
        ll K = std::max(0ll, -(tlo + r0));
        K = (K + unit - 1) / unit * unit;
        if (thi + r0 + K > 65535 || tlo + r0 + K < 0) return false;
        if (box && (tlo < 0 || thi + r0 > 2299)) return false;
        if (shift > 15) return false;
        // column sums
        auto col_word = [&](Col& q, int off) -> std::string {
            const int j = (std::min(std::max(off, -E[b]), 6 + E[b]) + E[b]) / 2;
            if (q.plain) return word(b, row_at(b, ho, q.plain_row), 2 * j - E[b]);
            if (q.v[j].empty()) {
                q.v[j] = fresh("v");
                std::vector<std::string> e;
                ll sum = 0;
                for (int y = 0; y < kh; ++y) {
                    // rows with a zero coefficient may lie outside the window
                    e.push_back(q.base[y] ? word(b, row_at(b, ho, y - ry), 2 * j - E[b]) : "");
                    sum += q.base[y];
                }
                o << ind << "const unsigned " << q.v[j] << " = "
                  << add_lanes(combine(q.base, e), q.L.bias - in.bias * sum) << ";\n";
            }
            return q.v[j];
        };
        std::vector<std::map<int, std::string>> odd(cols.size());
        auto col_pair = [&](int ci, int s) -> std::string {  // lanes s, s + 1
            if (!(s & 1)) return col_word(cols[ci], s);
            auto it = odd[ci].find(s);
            if (it != odd[ci].end()) return it->second;
            // a neighbour word outside the kept columns is replaced by the other
            // one (its lane belongs to no needed output)
            const int l = s - 1 < -E[b] ? s + 1 : s - 1, r = s + 1 > 6 + E[b] ? s - 1 : s + 1;
            const std::string wl = col_word(cols[ci], l), wr = col_word(cols[ci], r);
            const std::string n = fresh("s");
            o << ind << "const unsigned " << n << " = __funnelshift_r(" << wl << ", " << wr
              << ", 16);\n";
            odd[ci][s] = n;
            return n;
        };
        Lane out;
        for (int j = 0; j < words(ob); ++j) {
            const int t = 2 * j - E[ob];
            std::vector<std::string> e;
            std::vector<int> m;
            for (int x = 0; x < kw; ++x)
                if (mult[x]) {
                    e.push_back(col_pair(col_of[x], t + x - rx));
                    m.push_back(mult[x]);
                }
            Lane L{tlo + r0, thi + r0, K};
            std::string s = add_lanes(combine(m, e), r0 + K - konst);
            if (box) {
                const std::string u = fresh("u");
                o << ind << "const unsigned " << u << " = " << s << ";\n";
                // t / 9 = (7282 t) >> 16 for t <= 2299
                s = "__byte_perm((" + u + " & 0xffffu) * 7282u, (" + u + " >> 16) * 7282u, 0x7632)";
                L.lo /= 9;
                L.hi /= 9;
            } else if (shift > 0) {
                if (shift == 8)
                    s = "__byte_perm(" + s + ", 0u, 0x4341)";
                else
                    s = "((" + s + " >> " + std::to_string(shift) + ") & " + dup(0xFFFF >> shift) + ")";
                L.lo >>= shift;
                L.hi >>= shift;
                L.bias = K >> shift;
            }
            ll lo, hi;
            fmt_range(fmt, &lo, &hi);
            s = clamp(s, L, lo, hi);
            o << ind << "w.b" << ob << "[" << D[ob] - 1 << "][" << j << "] = " << s << ";\n";
            out = L;
        }
        lane[ob] = out;
        return true;
    }

    void emit_minmax(const GenStage& st) {
        const int b = st.in[0], ob = st.out, ho = halo(ob);
        const bool med = st.op == OP_MEDIAN;
        const char* f = st.op == OP_ERODE ? "hvx_min2" : "hvx_max2";
        // per column word: the rows' maximum / minimum, or (min, med, max)
        const int n = med ? 3 : 1;
        std::map<std::pair<int, int>, std::string> v, s;
        auto colw = [&](int which, int off) {
            const int k = std::min(std::max(off, -E[b]), 6 + E[b]);
            auto it = v.find({which, k});
            if (it != v.end()) return it->second;
            std::string r[3];
            for (int y = 0; y < 3; ++y) r[y] = word(b, row_at(b, ho, y - 1), k);
            if (!med) {
                const std::string t = fresh("v");
                o << ind << "const unsigned " << t << " = " << f << "(" << f << "(" << r[0] << ", "
                  << r[1] << "), " << r[2] << ");\n";
                v[{0, k}] = t;
            } else {
                const std::string a = fresh("v"), c = fresh("v");
                std::string t[3];
                for (auto& x : t) x = fresh("v");
                o << ind << "const unsigned " << a << " = hvx_min2(" << r[0] << ", " << r[1] << "), "
                  << c << " = hvx_max2(" << r[0] << ", " << r[1] << ");\n"
                  << ind << "const unsigned " << t[0] << " = hvx_min2(" << a << ", " << r[2] << "), "
                  << t[1] << " = hvx_max2(" << a << ", hvx_min2(" << c << ", " << r[2] << ")), "
                  << t[2] << " = hvx_max2(" << c << ", " << r[2] << ");\n";
                for (int i = 0; i < 3; ++i) v[{i, k}] = t[i];
            }
            return v[{which, k}];
        };
        auto pair = [&](int which, int at) {  // odd offset: lanes at, at + 1
            auto it = s.find({which, at});
            if (it != s.end()) return it->second;
            const int l = at - 1 < -E[b] ? at + 1 : at - 1, r = at + 1 > 6 + E[b] ? at - 1 : at + 1;
            const std::string wl = colw(which, l), wr = colw(which, r), t = fresh("s");
            o << ind << "const unsigned " << t << " = __funnelshift_r(" << wl << ", " << wr
              << ", 16);\n";
            s[{which, at}] = t;
            return t;
        };
        for (int j = 0; j < words(ob); ++j) {
            const int t = 2 * j - E[ob];
            std::string L[3], C[3], R[3];
            for (int i = 0; i < n; ++i) {
                L[i] = pair(i, t - 1);
                C[i] = colw(i, t);
                R[i] = pair(i, t + 1);
            }
            std::string e;
            if (!med) {
                e = std::string(f) + "(" + f + "(" + L[0] + ", " + C[0] + "), " + R[0] + ")";
            } else {
                // median of nine = median of (largest minimum, median of the
                // medians, smallest maximum) of the sorted columns
                e = "hvx_med2(hvx_max2(hvx_max2(" + L[0] + ", " + C[0] + "), " + R[0] + "), hvx_med2(" +
                    L[1] + ", " + C[1] + ", " + R[1] + "), hvx_min2(hvx_min2(" + L[2] + ", " + C[2] +
                    "), " + R[2] + "))";
            }
            o << ind << "w.b" << ob << "[" << D[ob] - 1 << "][" << j << "] = " << e << ";\n";
        }
        lane[ob] = lane[b];
    }

    // Lane k of word expression e (range L) as an int value.
    static std::string unpack(const std::string& e, const Lane& L, int k) {
        std::string s = k ? "(int)(" + e + " >> 16)" : "(int)(" + e + " & 0xffffu)";
        return L.bias ? "(" + s + " - " + std::to_string(L.bias) + ")" : "(" + s + ")";
    }

    static std::string lit64(ll v) { return "(" + std::to_string(v) + "LL)"; }

    // A point operator evaluated pixel by pixel: expr(a, b) as int code.
    template <class F>
    void emit_scalar(const GenStage& st, const int* ins, int n_in, Lane out, F expr) {
        const int ob = st.out, ho = halo(ob);
        for (int j = 0; j < words(ob); ++j) {
            const int t = 2 * j - E[ob];
            std::string r[2];
            for (int k = 0; k < 2; ++k) {
                std::string v[2];
                for (int i = 0; i < n_in; ++i) {
                    v[i] = fresh("i");
                    o << ind << "const int " << v[i] << " = "
                      << unpack(word(ins[i], row_at(ins[i], ho, 0), t), lane[ins[i]], k) << ";\n";
                }
                r[k] = fresh("i");
                o << ind << "const int " << r[k] << " = " << expr(v[0], v[1]);
                if (out.bias) o << " + " << out.bias;
                o << ";\n";
            }
            o << ind << "w.b" << ob << "[" << D[ob] - 1 << "][" << j << "] = __byte_perm((unsigned)"
              << r[0] << ", (unsigned)" << r[1] << ", 0x5410);\n";
        }
        lane[ob] = out;
    }

    static std::string range_test(const GenStage& st, const std::string& v) {
        return "!((ll)" + v + " > " + lit64(st.k1) + " || (ll)" + v + " < " + lit64(st.k0) + ")";
    }

    bool emit_point(const GenStage& st) {
        const int ob = st.out, ho = halo(ob), a = st.in[0], b = st.in[1];
        auto W = [&](int buf, int j) { return word(buf, row_at(buf, ho, 0), 2 * j - E[ob]); };
        // every word by f(j); all have range L
        auto each = [&](Lane L, auto f) {
            for (int j = 0; j < words(ob); ++j)
                o << ind << "w.b" << ob << "[" << D[ob] - 1 << "][" << j << "] = " << f(j) << ";\n";
            lane[ob] = L;
        };
        const Lane u8{0, 255, 0}, s16{-32768, 32767, 32768};
        switch (st.op) {
            case OP_CHX:
                each(u8, [&](int j) { return "__byte_perm(" + W(a, j) + ", 0u, 0x4341)"; });
                return true;
            case OP_AND:
            case OP_OR:
            case OP_XOR: {
                const char* f = st.op == OP_AND ? " & " : st.op == OP_OR ? " | " : " ^ ";
                each(u8, [&](int j) { return W(a, j) + f + W(b, j); });
                return true;
            }
            case OP_NOT:
                each(u8, [&](int j) { return W(a, j) + " ^ 0x00ff00ffu"; });
                return true;
            case OP_ADD:
            case OP_SUB:
            case OP_ABSDIFF: {
                const Lane A = lane[a], B = lane[b];
                ll lo, hi;
                fmt_range(st.i1, &lo, &hi);
                if (st.op == OP_ABSDIFF) {
                    const ll nb = std::max(A.bias, B.bias);
                    const ll m = std::max(std::llabs(A.hi - B.lo), std::llabs(B.hi - A.lo));
                    if (A.hi + nb <= 65535 && B.hi + nb <= 65535) {
                        Lane L{0, m, 0};
                        const Lane L0 = L;
                        Lane last = L;
                        each(L0, [&](int j) {
                            const std::string x = add_lanes(W(a, j), nb - A.bias),
                                              y = add_lanes(W(b, j), nb - B.bias);
                            last = L0;
                            std::string e = "(hvx_max2(" + x + ", " + y + ") - hvx_min2(" + x + ", " +
                                            y + "))";
                            // wrap or saturate as the policy says
                            if (st.i0 || L0.hi <= hi) return clamp(e, last, lo, hi);
                            last = st.i1 == HVX_DF_U8 ? u8 : last;
                            return e + " & " + dup(0xFF);
                        });
                        if (!st.i0 && st.i1 != HVX_DF_U8 && m > hi) return false;
                        lane[ob] = last;
                        return true;
                    }
                } else {
                    const bool add = st.op == OP_ADD;
                    Lane L{add ? A.lo + B.lo : A.lo - B.hi, add ? A.hi + B.hi : A.hi - B.lo, 0};
                    L.bias = std::max(0ll, -L.lo);
                    const bool wrap = !st.i0 && (L.lo < lo || L.hi > hi);
                    if (wrap && st.i1 == HVX_DF_U8) L.bias = (L.bias + 255) / 256 * 256;
                    if (L.hi + L.bias <= 65535 && !(wrap && st.i1 != HVX_DF_U8)) {
                        Lane last = L;
                        each(L, [&](int j) {
                            last = L;
                            std::string e = add_lanes(
                                "(" + W(a, j) + (add ? " + " : " - ") + W(b, j) + ")",
                                L.bias - (add ? A.bias + B.bias : A.bias - B.bias));
                            if (!wrap) return clamp(e, last, lo, hi);
                            last = u8;
                            return e + " & " + dup(0xFF);
                        });
                        lane[ob] = last;
                        return true;
                    }
                }
                // wide ranges: pixel by pixel
                const int ins[2] = {a, b};
                emit_scalar(st, ins, 2, st.i1 == HVX_DF_U8 ? u8 : s16,
                            [&](const std::string& x, const std::string& y) {
                                const std::string r = st.op == OP_ADD   ? "(" + x + " + " + y + ")"
                                                      : st.op == OP_SUB ? "(" + x + " - " + y + ")"
                                                                        : "abs(" + x + " - " + y + ")";
                                if (st.i1 == HVX_DF_U8)
                                    return st.i0 ? "sat_u8(" + r + ")" : "(" + r + " & 0xFF)";
                                return st.i0 ? "sat_s16(" + r + ")" : "(int)(short)(" + r + ")";
                            });
                return true;
            }
            case OP_THRESH: {
                if (st.i3) return false;
                if (st.i1 < 0 || st.i1 > 255 || st.i2 < 0 || st.i2 > 255) return false;
                const std::string tv = std::to_string(st.i1), fv = std::to_string(st.i2);
                const int m = fused_mag(st);
                if (m >= 0) {
                    // round(sqrt(s)) > T is s > T^2 + T for 0 <= T < 32767 (codegen.cpp)
                    const ll T = st.k0;
                    const int* ins = d.st[m].in;
                    emit_scalar(st, ins, 2, u8, [&](const std::string& x, const std::string& y) {
                        if (T < 0 || T >= 32767) return T < 0 ? tv : fv;
                        return "((unsigned)(" + x + " * " + x + ") + (unsigned)(" + y + " * " + y +
                               ") > " + std::to_string(T * T + T) + "u ? " + tv + " : " + fv + ")";
                    });
                    return true;
                }
                if (st.i0 == HVX_THRESHOLD_BINARY) {
                    const Lane A = lane[a];
                    const ll T = st.k0;
                    if (T < A.lo || T >= A.hi) {
                        each(u8, [&](int) { return dup(T < A.lo ? st.i1 : st.i2); });
                        return true;
                    }
                    // the top bit of lane + (32767 - T - bias) is v > T
                    if (A.hi - T <= 32768 && T - A.lo <= 32767) {
                        each(u8, [&](int j) {
                            std::string e = "hvx_sign2(" +
                                            add_lanes(W(a, j), 32767 - T - A.bias) + ")";
                            if (st.i1 == 255 && st.i2 == 0) return e;
                            if ((st.i1 ^ st.i2) != 255) e = "(" + e + " & " + dup(st.i1 ^ st.i2) + ")";
                            return st.i2 ? e + " ^ " + dup(st.i2) : e;
                        });
                        return true;
                    }
                }
                emit_scalar(st, &a, 1, u8, [&](const std::string& x, const std::string&) {
                    const std::string t = st.i0 == HVX_THRESHOLD_BINARY
                                              ? "(ll)" + x + " > " + lit64(st.k0)
                                              : range_test(st, x);
                    return "((" + t + ") ? " + tv + " : " + fv + ")";
                });
                return true;
            }
            case OP_MAG: {
                const int ins[2] = {a, b};
                emit_scalar(st, ins, 2, Lane{0, 32767, 0},
                            [&](const std::string& x, const std::string& y) {
                                return "magnitude_s16(" + x + ", " + y + ")";
                            });
                return true;
            }
            case OP_PHASE: {
                const int ins[2] = {a, b};
                emit_scalar(st, ins, 2, u8, [&](const std::string& x, const std::string& y) {
                    return "(int)phase_u8(" + x + ", " + y + ")";
                });
                return true;
            }
            case OP_MULTIPLY: {
                const int ins[2] = {a, b};
                emit_scalar(st, ins, 2, st.i1 == HVX_DF_U8 ? u8 : s16,
                            [&](const std::string& x, const std::string& y) {
                                const std::string v = "multiply_scaled(" + x + ", " + y + ", " +
                                                      lit64(st.k0) + ", " + std::to_string(st.i3) +
                                                      ", " + (st.i2 ? "true" : "false") + ")";
                                if (st.i1 == HVX_DF_U8)
                                    return st.i0 ? "sat64_u8(" + v + ")" : "(int)(" + v + " & 0xFF)";
                                return st.i0 ? "sat64_s16(" + v + ")" : "wrap64_s16(" + v + ")";
                            });
                return true;
            }
            case OP_CONVDEPTH: {
                const Lane A = lane[a];
                const int s = st.i0;
                if (st.i1 == st.i3) {  // Copy
                    each(A, [&](int j) { return W(a, j); });
                    return true;
                }
                if (st.i1 == HVX_DF_S16) {
                    if (A.bias || A.hi > 255 || s > 7) return false;
                    each(Lane{0, A.hi << s, 0},
                         [&](int j) { return "(" + W(a, j) + " << " + std::to_string(s) + ")"; });
                    return true;
                }
                // S16 -> U8: floor(v / 2^s), the bias made a multiple of 2^s
                // (of 2^(s + 8) when the result wraps)
                const ll unit = 1ll << (st.i2 ? s : s + 8);
                const ll nb = (A.bias + unit - 1) / unit * unit;
                if (A.hi + nb > 65535) return false;
                Lane last;
                each(u8, [&](int j) {
                    std::string e = add_lanes(W(a, j), nb - A.bias);
                    if (s) e = "((" + e + " >> " + std::to_string(s) + ") & " + dup(0xFFFF >> s) + ")";
                    if (!st.i2) return e + " & " + dup(0xFF);
                    last = Lane{A.lo >> s, A.hi >> s, nb >> s};
                    return clamp(e, last, 0, 255);
                });
                lane[ob] = st.i2 ? last : u8;
                return true;
            }
        }
        return false;
    }

    bool emit_stage(const GenStage& st) {
        switch (st.op) {
            case OP_GAUSS:
                return emit_conv(st, {1, 2, 1, 2, 4, 2, 1, 2, 1}, 1, 1,
                                 st.rounding == HVX_ROUND_TO_NEAREST ? 8 : 0, 4, HVX_DF_U8, false);
            case OP_BOX:
                return emit_conv(st, std::vector<int>(9, 1), 1, 1,
                                 st.rounding == HVX_ROUND_TO_NEAREST ? 4 : 0, 0, HVX_DF_U8, true);
            case OP_SOBEL_X:
                return emit_conv(st, {-1, 0, 1, -2, 0, 2, -1, 0, 1}, 1, 1, 0, 0, HVX_DF_S16, false);
            case OP_SOBEL_Y:
                return emit_conv(st, {-1, -2, -1, 0, 0, 0, 1, 2, 1}, 1, 1, 0, 0, HVX_DF_S16, false);
            case OP_CONV: {
                const int n = (2 * st.rx + 1) * (2 * st.ry + 1);
                std::vector<int> c(d.coeff + st.coeff_off, d.coeff + st.coeff_off + n);
                // (coefficients beyond 16 bits never fit the lanes)
                for (int v : c)
                    if (v > 65535 || v < -65535) return false;
                return emit_conv(st, c, st.rx, st.ry, 0, st.shift, st.i0, false);
            }
            case OP_DILATE:
            case OP_ERODE:
            case OP_MEDIAN: emit_minmax(st); return true;
            default: return emit_point(st);
        }
    }

    // Lanes of tiles on the image's border also hold 0 (outside the valid
    // region) and the border constant.
    bool widen(int b) {
        Lane& L = lane[b];
        if (!full[b]) {
            L.lo = std::min(L.lo, 0ll);
            L.hi = std::max(L.hi, 0ll);
        }
        if (d.buf[b].fill == FILL_CONSTANT) {
            L.lo = std::min(L.lo, (ll)d.buf[b].cval);
            L.hi = std::max(L.hi, (ll)d.buf[b].cval);
        }
        return L.lo + L.bias >= 0 && L.hi + L.bias <= 65535;
    }

    // ---- the row step --------------------------------------------------------

    // EDGE tiles, after the newest row of buffer b (an op's output) was computed:
    // zeros outside its valid region, then the cells outside the image as its
    // local consumers read them.
    void emit_edge_fix(int b) {
        const int h = halo(b), n = words(b), nw = D[b] - 1;
        const std::string B = std::to_string(b), row = "w.b" + B + "[" + std::to_string(nw) + "]";
        const int fill = d.buf[b].fill;
        const bool fills = h > 0 && (fill == FILL_REPLICATE || fill == FILL_CONSTANT);
        if (full[b] && !fills) return;
        o << "      if (EDGE) {\n        const int yr = t.yb + i + " << h << ";\n";
        if (!full[b])
            o << "        hvx_valid<" << n << ", " << E[b] << ">(" << row << ", t.x, yr, t.v" << B
              << ", " << dup(lane[b].bias) << ");\n";
        if (fills) {
            const bool rep = fill == FILL_REPLICATE;
            const std::string cv = dup(d.buf[b].cval + lane[b].bias);
            o << "        hvx_cols<" << n << ", " << E[b] << ", " << (rep ? "true" : "false") << ">("
              << row << ", t.x, t.W, " << cv << ");\n";
            if (rep) {
                if (nw > 0)
                    o << "        if (__any_sync(__activemask(), yr == 0 || yr >= t.H)) {\n"
                      << "        #pragma unroll\n        for (int j = 0; j < " << n << "; ++j) {\n"
                      << "          if (yr >= t.H) " << row << "[j] = w.b" << B << "[" << nw - 1
                      << "][j];\n          #pragma unroll\n          for (int r = 0; r < " << nw
                      << "; ++r)\n            if (yr == 0) w.b" << B << "[r][j] = " << row
                      << "[j];\n        }\n        }\n";
            } else {
                o << "        #pragma unroll\n        for (int j = 0; j < " << n
                  << "; ++j)\n          if (yr < 0 || yr >= t.H) " << row << "[j] = " << cv << ";\n";
            }
        }
        o << "      }\n";
    }

    // The newest row of external input e from its box (or as read from memory).
    void emit_input(int e, int box) {
        const int b = d.in[e].buf, f = d.in[e].fmt, nw = D[b] - 1;
        const std::string row = "w.b" + std::to_string(b) + "[" + std::to_string(nw) + "]";
        const std::string flip = f == HVX_DF_S16 ? "true" : "false";
        if (box >= 0) {
            const int elem = boxes[box].elem;
            o << "      hvx_box_row<" << elem << ", " << E[b] << ", " << flip << ">(" << row << ", t.box"
              << box << " + (i + " << 2 * halo(b) << ") * " << STRIP_BOX_W * elem << ");\n";
        } else {
            const std::string E_ = std::to_string(e);
            o << "      hvx_mem_row<" << flip << ">(" << row << ", m.in" << E_ << ");\n";
            mem_rows += "  hvx_mem_load<EDGE>(m.in" + E_ + ", t.in" + E_ + ", t.ip" + E_ +
                        ", t.x, t.yb + i, t.W, t.H);\n";
            mem_words += f == HVX_DF_U8 ? 2 : 4;
            mem_decl += std::string(f == HVX_DF_U8 ? "  uint2" : "  uint4") + " in" + E_ + ";\n";
        }
    }

    void emit_outputs() {
        for (int e = 0; e < d.n_out; ++e) {
            const int b = d.out[e].buf;
            const int r = row_at(b, 0, 0), c = E[b] / 2;
            o << "      hvx_store<" << (d.out[e].fmt == HVX_DF_U8 ? 1 : 2) << ", EDGE>(";
            for (int j = 0; j < 4; ++j)
                o << (j ? ", " : "")
                  << add_lanes("w.b" + std::to_string(b) + "[" + std::to_string(r) + "][" +
                                   std::to_string(c + j) + "]",
                               d.out[e].fmt == HVX_DF_S16 ? 32768 - lane[b].bias : -lane[b].bias);
            o << ", t.out" << e << ", t.op" << e << ", t.x, t.yb + i, t.W, t.H);\n";
        }
    }

    // Row y of the global operators' inputs.
    void emit_globals() {
        for (int k : globals) {
            const GenStage& st = d.st[k];
            const int b = st.in[0], r = row_at(b, 0, 0), c = E[b] / 2;
            const Lane& L = lane[b];
            const std::string g = "acc.g" + std::to_string(k);
            std::string w;
            for (int j = 0; j < 4; ++j)
                w += (j ? ", w.b" : "w.b") + std::to_string(b) + "[" + std::to_string(r) + "][" +
                     std::to_string(c + j) + "]";
            const std::string at = ", t.x, t.yb + i, t.W, t.v" + std::to_string(b) + ");\n";
            if (st.op == OP_MEANSTD)
                o << "      hvx_sum_row<" << (L.bias == 0 && L.hi <= 255 ? "true" : "false") << ", "
                  << L.bias << ", EDGE>(" << g << ", " << w << at;
            else if (st.op == OP_MINMAX)
                o << "      hvx_mm_strip<EDGE>(" << g << ", " << w << at;
            else
                o << "      hvx_hist_row<" << L.bias << ", " << st.i0 << ", " << st.i1 << ", " << st.i2
                  << ", EDGE>(" << g << ", " << w << at;
        }
    }

    static const char* reduction_prelude() {
        return R"STRIP(
// ---- global operators: per-thread totals over all tiles of a CTA, one partial
// result per CTA, combined by the last CTA to finish.  Scratch of each: a counter
// of finished CTAs (the first one's is used), then sums, per-CTA extrema or bins;
// the last CTA leaves counter, sums and bins at zero for the next launch.  Against atomics per warp
// and tile on one result word (compare-and-swap for the counts): luma of a
// 3840x2160 UYVY frame with MeanStdDev, MinMaxLoc and a 256-bin Histogram 1110 ->
// 25.2 us (cold L2). ----
struct HvxSum {
  long long s1;
  unsigned long long s2;
  unsigned n;
  unsigned u1, u2;  // this tile's sums of U8 values (at most 8 x 24 pixels a thread)
};
__device__ __forceinline__ void hvx_sum_flush(HvxSum& a) {
  a.s1 += a.u1;
  a.s2 += a.u2;
  a.u1 = a.u2 = 0u;
}
__device__ __forceinline__ bool hvx_inside(int j, int x, int y, const int* v) {
  return y >= v[1] && y < v[3] && x + j >= v[0] && x + j < v[2];
}
template <int BIAS>
__device__ __forceinline__ int hvx_lane(const unsigned (&w)[4], int j) {
  return (int)((j & 1) ? w[j >> 1] >> 16 : w[j >> 1] & 0xffffu) - BIAS;
}
// a row of 8 values; BYTES: 0 .. 255 in the lanes
template <bool BYTES, int BIAS, bool EDGE>
__device__ __forceinline__ void hvx_sum_row(HvxSum& a, unsigned w0, unsigned w1, unsigned w2, unsigned w3,
                                            int x, int y, int, const int* v) {
  const unsigned w[4] = {w0, w1, w2, w3};
  if (BYTES && !EDGE) {
    const unsigned p = __byte_perm(w0, w1, 0x6420), q = __byte_perm(w2, w3, 0x6420);
    a.u1 = __dp4a(q, 0x01010101u, __dp4a(p, 0x01010101u, a.u1));
    a.u2 = __dp4a(q, q, __dp4a(p, p, a.u2));
    a.n += 8;
    return;
  }
  #pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int l = hvx_lane<BIAS>(w, j);
    if (!EDGE || hvx_inside(j, x, y, v)) {
      a.s1 += l;
      a.s2 += (unsigned long long)((long long)l * l);
      ++a.n;
    }
  }
}
// lanes of a row equal to v (at most 8)
__device__ __forceinline__ unsigned hvx_count(unsigned w0, unsigned w1, unsigned w2, unsigned w3, int v) {
  const unsigned d = (unsigned)v * 0x10001u, one = 0x10001u;
  const unsigned s = hvx_min2(w0 ^ d, one) + hvx_min2(w1 ^ d, one) + hvx_min2(w2 ^ d, one) +
                     hvx_min2(w3 ^ d, one);
  return 8u - (s & 0xffffu) - (s >> 16);
}
// the first lane of a row equal to v (one is)
__device__ __forceinline__ unsigned hvx_first(const unsigned (&w)[4], int v) {
  unsigned f = 0u;
  #pragma unroll
  for (int j = 7; j >= 0; --j)
    if (hvx_lane<0>(w, j) == v) f = j;
  return f;
}
// extrema of the lanes (values + bias).  Most rows reach neither extremum;
// one that equals it is counted by lane pairs, and its place matters only
// where a later tile of the thread starts further up.
template <bool EDGE>
__device__ __forceinline__ void hvx_mm_strip(HvxMinMaxAcc& a, unsigned w0, unsigned w1, unsigned w2,
                                             unsigned w3, int x, int y, int W, const int* v) {
  const unsigned w[4] = {w0, w1, w2, w3};
  const unsigned at = (unsigned)y * (unsigned)W + (unsigned)x;
  if (!EDGE) {
    const unsigned m = hvx_min2(hvx_min2(w0, w1), hvx_min2(w2, w3));
    const unsigned h = hvx_max2(hvx_max2(w0, w1), hvx_max2(w2, w3));
    const int lo = (int)min(m & 0xffffu, m >> 16), hi = (int)max(h & 0xffffu, h >> 16);
    if (lo <= a.minv) {
      const unsigned n = hvx_count(w0, w1, w2, w3, lo);
      a.minc = lo < a.minv ? n : a.minc + n;
      if (lo < a.minv || at < a.mini) a.mini = at + hvx_first(w, lo);
      a.minv = lo;
    }
    if (hi >= a.maxv) {
      const unsigned n = hvx_count(w0, w1, w2, w3, hi);
      a.maxc = hi > a.maxv ? n : a.maxc + n;
      if (hi > a.maxv || at < a.maxi) a.maxi = at + hvx_first(w, hi);
      a.maxv = hi;
    }
    return;
  }
  #pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int l = hvx_lane<0>(w, j);
    if (!hvx_inside(j, x, y, v)) continue;
    if (l <= a.minv) {
      a.mini = l < a.minv ? at + j : min(a.mini, at + j);
      a.minc = l < a.minv ? 1u : a.minc + 1u;
      a.minv = l;
    }
    if (l >= a.maxv) {
      a.maxi = l > a.maxv ? at + j : min(a.maxi, at + j);
      a.maxc = l > a.maxv ? 1u : a.maxc + 1u;
      a.maxv = l;
    }
  }
}
// 8 copies of each bin, one per lane modulo 8: half the bank conflicts of one
template <int BIAS, int BINS, int OFFSET, int RANGE, bool EDGE>
__device__ __forceinline__ void hvx_hist_row(unsigned* bins, unsigned w0, unsigned w1, unsigned w2,
                                             unsigned w3, int x, int y, int, const int* v) {
  const unsigned w[4] = {w0, w1, w2, w3};
  #pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int l = hvx_lane<BIAS>(w, j) - OFFSET;
    const bool in = (OFFSET == 0 && RANGE == 256 && BIAS == 0) || (l >= 0 && l < RANGE);
    if (in && (!EDGE || hvx_inside(j, x, y, v)))
      atomicAdd(bins + (BINS == RANGE ? l : l * BINS / RANGE) * 8 + (threadIdx.x & 7), 1u);
  }
}
// phase `parity` of bar, for at most ~2^31 cycles: on time-out the error is
// recorded, the same bound is waited once more, and false is returned
__device__ __forceinline__ bool hvx_mbar_wait_parity(unsigned long long* bar, unsigned parity, int* err) {
  for (int round = 0; round < 2; ++round) {
    const long long c0 = clock64();
    do {
      unsigned ok;
      asm volatile("{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\n\t"
                   "selp.u32 %0, 1, 0, q;\n\t}" : "=r"(ok) : "r"(hvx_smem(bar)), "r"(parity) : "memory");
      if (ok) return round == 0;
    } while (clock64() - c0 <= (1ll << 31));
    if (round == 0 && err) atomicCAS(err, 0, 1);
  }
  return false;
}
// the warp's totals into lane 0
__device__ __forceinline__ void hvx_sum_warp(HvxSum& a) {
  #pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a.s1 += __shfl_xor_sync(0xFFFFFFFFu, a.s1, o);
    a.s2 += __shfl_xor_sync(0xFFFFFFFFu, a.s2, o);
    a.n += __shfl_xor_sync(0xFFFFFFFFu, a.n, o);
  }
}
// accumulators of the CTA's warps combined into thread 0's
template <int WARPS>
__device__ __forceinline__ void hvx_mm_block(HvxMinMaxAcc& a, HvxMinMaxAcc* s) {
  hvx_mm_warp(a);
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = a;
  __syncthreads();
  if (threadIdx.x == 0)
    for (int k = 1; k < WARPS; ++k)
      hvx_mm_merge(a, s[k].minv, s[k].mini, s[k].minc, s[k].maxv, s[k].maxi, s[k].maxc);
  __syncthreads();
}
// the result words of MinMaxLoc (all ones where nothing was seen)
__device__ __forceinline__ void hvx_mm_result(unsigned long long* r, const HvxMinMaxAcc& a) {
  const unsigned lo = (unsigned)(a.minv + 32768), hi = 65535u - (unsigned)(a.maxv + 32768);
  r[0] = a.minc ? ((unsigned long long)lo << 32) | a.mini : ~0ull;
  r[1] = a.maxc ? ((unsigned long long)hi << 32) | a.maxi : ~0ull;
  r[2] = a.minc ? ((unsigned long long)lo << 40) | a.minc : ~0ull;
  r[3] = a.maxc ? ((unsigned long long)hi << 40) | a.maxc : ~0ull;
}
)STRIP";
    }

    // The kernels of a group with global operators: CTA c of p.ctas works on
    // the image's tiles c, c + p.ctas, ..
    void emit_reduction_kernels(const std::string& bounds) {
        const bool boxed = !boxes.empty();
        const int warps = STRIP_THREADS / 32;
        o << "template <bool GMAP>\n"
          << "__device__ __forceinline__ void hvx_image(const HvxJitParams& p, unsigned char* sm, int cta) {\n"
          << "  const int R = p.rows, gx = (p.W + " << STRIP_TW - 1 << ") / " << STRIP_TW
          << ", tiles = gx * ((p.H + 8 * R - 1) / (8 * R));\n"
          << "  const HvxBoxes x = hvx_boxes(sm + 128, R);\n"
          << "  unsigned long long* const bar = (unsigned long long*)sm;\n"
          << "  HvxAcc acc;\n";
        bool mm = false;
        for (int k : globals) {
            const std::string K = std::to_string(k);
            if (d.st[k].op == OP_MEANSTD) {
                o << "  acc.g" << K << " = HvxSum{0, 0, 0, 0, 0};\n"
                  << "  __shared__ HvxSum s" << K << "[" << warps << "];\n";
            } else if (d.st[k].op == OP_MINMAX) {
                mm = true;
                o << "  acc.g" << K << " = HvxMinMaxAcc{0x10000, -1, 0xFFFFFFFFu, 0xFFFFFFFFu, 0, 0};\n";
            } else {
                o << "  __shared__ unsigned h" << K << "[" << 8 * d.st[k].i0 << "];\n"
                  << "  acc.g" << K << " = h" << K << ";\n"
                  << "  for (int i = threadIdx.x; i < " << 8 * d.st[k].i0 << "; i += " << STRIP_THREADS
                  << ") h" << K << "[i] = 0u;\n";
            }
        }
        if (mm) o << "  __shared__ HvxMinMaxAcc smm[" << warps << "];\n";
        o << "  __shared__ bool last;\n";
        if (boxed) o << "  if (threadIdx.x == 0) hvx_mbar_init(bar);\n";
        o << "  __syncthreads();\n"
          << "  asm volatile(\"griddepcontrol.wait;\" ::: \"memory\");\n"
          << "  unsigned k = 0;\n"
          << "  for (int t = cta; t < tiles; t += p.ctas, ++k) {\n"
          << "    const int ty = t / gx, tx = t - ty * gx;\n";
        if (boxed)
            o << "    if (threadIdx.x == 0) {\n"
              << "      asm volatile(\"fence.proxy.async.shared::cta;\" ::: \"memory\");\n"
              << "      hvx_issue<GMAP>(p, x, bar, tx * " << STRIP_TW << ", ty * 8 * R);\n    }\n"
              << "    if (__syncthreads_or(!hvx_mbar_wait_parity(bar, k & 1, p.err))) break;\n";
        o << "    hvx_strip_tile(p, x, tx, ty, acc);\n";
        if (boxed) o << "    __syncthreads();\n";
        o << "  }\n";
        // this CTA's partial results
        for (size_t j = 0; j < globals.size(); ++j) {
            const int k = globals[j];
            const std::string K = std::to_string(k),
                              scr = "((unsigned char*)p.scratch[" + std::to_string(j) + "] + 16)";
            if (d.st[k].op == OP_MEANSTD) {
                o << "  hvx_sum_warp(acc.g" << K << ");\n"
                  << "  if ((threadIdx.x & 31) == 0) s" << K << "[threadIdx.x >> 5] = acc.g" << K << ";\n"
                  << "  __syncthreads();\n"
                  << "  if (threadIdx.x == 0) {\n    HvxSum q = s" << K << "[0];\n"
                  << "    for (int i = 1; i < " << warps << "; ++i) {\n      q.s1 += s" << K
                  << "[i].s1;\n      q.s2 += s" << K << "[i].s2;\n      q.n += s" << K << "[i].n;\n    }\n"
                  << "    unsigned long long* const r = (unsigned long long*)" << scr << ";\n"
                  << "    atomicAdd(r, (unsigned long long)q.s1);\n    atomicAdd(r + 1, q.s2);\n"
                  << "    atomicAdd(r + 2, (unsigned long long)q.n);\n  }\n";
            } else if (d.st[k].op == OP_MINMAX) {
                const ll bias = lane[d.st[k].in[0]].bias;
                o << "  hvx_mm_block<" << warps << ">(acc.g" << K << ", smm);\n"
                  << "  if (threadIdx.x == 0) {\n"
                  << "    acc.g" << K << ".minv -= " << bias << ";\n    acc.g" << K << ".maxv -= " << bias
                  << ";\n    ((HvxMinMaxAcc*)" << scr << ")[cta] = acc.g" << K << ";\n  }\n";
            } else {
                o << "  __syncthreads();\n"
                  << "  for (int i = threadIdx.x; i < " << d.st[k].i0 << "; i += " << STRIP_THREADS
                  << ") {\n    unsigned n = 0;\n    #pragma unroll\n"
                  << "    for (int c = 0; c < 8; ++c) n += h" << K << "[8 * i + c];\n"
                  << "    if (n) atomicAdd((unsigned*)" << scr << " + i, n);\n  }\n";
            }
        }
        // (the barrier orders the CTA's writes before thread 0's cumulative fence)
        o << "  __syncthreads();\n"
          << "  unsigned* const done = (unsigned*)p.scratch[0];\n"
          << "  if (threadIdx.x == 0) {\n    __threadfence();\n"
          << "    last = atomicAdd(done, 1u) == (unsigned)p.ctas - 1u;\n  }\n"
          << "  __syncthreads();\n"
          << "  if (!last) return;\n"
          << "  __threadfence();\n";
        for (size_t j = 0; j < globals.size(); ++j) {
            const int k = globals[j];
            const std::string res = "p.res[" + std::to_string(j) + "]",
                              mir = "p.mirror[" + std::to_string(j) + "]",
                              scr = "((unsigned char*)p.scratch[" + std::to_string(j) + "] + 16)";
            if (d.st[k].op == OP_MEANSTD) {
                o << "  if (threadIdx.x < 3) {\n    const unsigned long long v = atomicExch((unsigned long "
                     "long*)"
                  << scr << " + threadIdx.x, 0ull);\n    ((unsigned long long*)" << res
                  << ")[threadIdx.x] = v;\n    if (" << mir << ") ((unsigned long long*)" << mir
                  << ")[threadIdx.x] = v;\n  }\n";
            } else if (d.st[k].op == OP_MINMAX) {
                o << "  {\n    HvxMinMaxAcc a;\n    hvx_mm_init(a);\n"
                  << "    const volatile int* const q = (const volatile int*)" << scr << ";\n"
                  << "    for (int i = threadIdx.x; i < p.ctas; i += " << STRIP_THREADS << ")\n"
                  << "      hvx_mm_merge(a, q[6 * i], q[6 * i + 2], q[6 * i + 4], q[6 * i + 1], "
                     "q[6 * i + 3], q[6 * i + 5]);\n"
                  << "    hvx_mm_block<" << warps << ">(a, smm);\n"
                  << "    if (threadIdx.x == 0) {\n      hvx_mm_result((unsigned long long*)" << res
                  << ", a);\n      if (" << mir << ") hvx_mm_result((unsigned long long*)" << mir
                  << ", a);\n    }\n  }\n";
            } else {
                o << "  for (int i = threadIdx.x; i < " << d.st[k].i0 << "; i += " << STRIP_THREADS
                  << ") {\n    const unsigned v = atomicExch((unsigned*)" << scr
                  << " + i, 0u);\n    ((unsigned*)" << res << ")[i] = v;\n    if (" << mir
                  << ") ((unsigned*)" << mir << ")[i] = v;\n  }\n";
            }
        }
        o << "  if (threadIdx.x == 0) *done = 0u;\n}\n\n"
          << "extern \"C\" __global__ void " << bounds
          << " hvx_generated_strips(const __grid_constant__ HvxJitParams p) {\n"
          << "  asm volatile(\"griddepcontrol.launch_dependents;\");\n"
          << "  extern __shared__ __align__(128) unsigned char hvx_box[];\n"
          << "  hvx_image<false>(p, hvx_box, blockIdx.x);\n}\n"
          << "// n images: block t is CTA t - cta_start[i] of the last image i with cta_start[i] <= t\n"
          << "extern \"C\" __global__ void " << bounds
          << " hvx_generated_strips_batch(const HvxJitParams* __restrict__ ps, const int* __restrict__ "
             "cta_start, int n, int) {\n"
          << "  asm volatile(\"griddepcontrol.launch_dependents;\");\n"
          << "  extern __shared__ __align__(128) unsigned char hvx_box[];\n"
          << "  const int t = blockIdx.x;\n  int lo = 0, hi = n - 1;\n"
          << "  while (lo < hi) {\n    const int mid = (lo + hi + 1) >> 1;\n"
          << "    if (__ldg(cta_start + mid) <= t) lo = mid; else hi = mid - 1;\n  }\n"
          << "  hvx_image<true>(ps[lo], hvx_box, t - __ldg(cta_start + lo));\n}\n";
    }

    static const char* prelude() {
        static_assert(HVX_DF_U8 == 1 && HVX_DF_UYVY == 5, "hvx_ld's formats below");
        return R"STRIP(
// ---- strip form: 8 columns x R rows per thread, pixel pairs in 16-bit lanes ----
typedef long long ll;
__device__ __forceinline__ unsigned hvx_min2(unsigned a, unsigned b) {
  unsigned r;
  asm("min.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ unsigned hvx_max2(unsigned a, unsigned b) {
  unsigned r;
  asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ unsigned hvx_med2(unsigned a, unsigned b, unsigned c) {
  return hvx_max2(hvx_min2(a, b), hvx_min2(hvx_max2(a, b), c));
}
// 255 in each lane whose top bit is set, else 0 (prmt's sign-replicating nibbles)
__device__ __forceinline__ unsigned hvx_sign2(unsigned a) {
  unsigned r;
  asm("prmt.b32 %0, %1, 0, 0x4b49;" : "=r"(r) : "r"(a));
  return r;
}
// one box row as pairs (x - E, x - E + 1) .. (x + 6 + E, x + 7 + E)
template <int ELEM, int E, bool FLIP>
__device__ __forceinline__ void hvx_box_row(unsigned (&w)[4 + E], const unsigned char* s) {
  if (ELEM == 1) {
    const uint2 m = *(const uint2*)s;
    w[E / 2 + 0] = __byte_perm(m.x, 0u, 0x4140);
    w[E / 2 + 1] = __byte_perm(m.x, 0u, 0x4342);
    w[E / 2 + 2] = __byte_perm(m.y, 0u, 0x4140);
    w[E / 2 + 3] = __byte_perm(m.y, 0u, 0x4342);
    #pragma unroll
    for (int k = 0; k < E; k += 4) {
      const unsigned l = *(const unsigned*)(s - 4 - k), r = *(const unsigned*)(s + 8 + k);
      w[E / 2 - 1 - k / 2] = __byte_perm(l, 0u, 0x4342);
      w[E / 2 + 4 + k / 2] = __byte_perm(r, 0u, 0x4140);
      if (k + 2 < E) {
        w[E / 2 - 2 - k / 2] = __byte_perm(l, 0u, 0x4140);
        w[E / 2 + 5 + k / 2] = __byte_perm(r, 0u, 0x4342);
      }
    }
  } else {
    const uint4 m = *(const uint4*)s;
    w[E / 2 + 0] = m.x;
    w[E / 2 + 1] = m.y;
    w[E / 2 + 2] = m.z;
    w[E / 2 + 3] = m.w;
    #pragma unroll
    for (int k = 0; k < E / 2; ++k) {
      w[E / 2 - 1 - k] = *(const unsigned*)(s - 4 - 4 * k);
      w[E / 2 + 4 + k] = *(const unsigned*)(s + 16 + 4 * k);
    }
    if (FLIP) {
      #pragma unroll
      for (int j = 0; j < 4 + E; ++j) w[j] ^= 0x80008000u;
    }
  }
}
// 8 pixels of row y of an image in memory as stored, rows 16-byte aligned
// (ordinary loads, as hvx_ld's)
template <bool EDGE>
__device__ __forceinline__ void hvx_mem_load(uint2& m, const void* base, unsigned long long pitch, int x,
                                             int y, int W, int H) {
  const unsigned char* const r = (const unsigned char*)base + (unsigned long long)y * pitch;
  if (!EDGE || (y < H && x + 8 <= W)) {
    __builtin_assume(__isGlobal(r));
    m = *(const uint2*)(r + x);
    return;
  }
  unsigned v[2] = {0u, 0u};
  #pragma unroll
  for (int k = 0; k < 8; ++k)
    if (y < H && x + k < W) v[k >> 2] |= (unsigned)hvx_ld<1>(r, 0, x + k, 0) << (8 * (k & 3));
  m = make_uint2(v[0], v[1]);
}
template <bool EDGE>
__device__ __forceinline__ void hvx_mem_load(uint4& m, const void* base, unsigned long long pitch, int x,
                                             int y, int W, int H) {
  const unsigned char* const r = (const unsigned char*)base + (unsigned long long)y * pitch;
  if (!EDGE || (y < H && x + 8 <= W)) {
    __builtin_assume(__isGlobal(r));
    m = *(const uint4*)(r + 2 * x);
    return;
  }
  unsigned v[4] = {0u, 0u, 0u, 0u};
  #pragma unroll
  for (int k = 0; k < 8; ++k)
    if (y < H && x + k < W) v[k >> 1] |= (unsigned)hvx_ld<5>(r, 0, x + k, 0) << (16 * (k & 1));
  m = make_uint4(v[0], v[1], v[2], v[3]);
}
template <bool FLIP>
__device__ __forceinline__ void hvx_mem_row(unsigned (&w)[4], const uint2& m) {
  w[0] = __byte_perm(m.x, 0u, 0x4140);
  w[1] = __byte_perm(m.x, 0u, 0x4342);
  w[2] = __byte_perm(m.y, 0u, 0x4140);
  w[3] = __byte_perm(m.y, 0u, 0x4342);
}
template <bool FLIP>
__device__ __forceinline__ void hvx_mem_row(unsigned (&w)[4], const uint4& m) {
  const unsigned flip = FLIP ? 0x80008000u : 0u;
  w[0] = m.x ^ flip;
  w[1] = m.y ^ flip;
  w[2] = m.z ^ flip;
  w[3] = m.w ^ flip;
}
// 8 outputs of row y; 16-bit lanes of S16 images arrive as value + 32768
template <int ELEM, bool EDGE>
__device__ __forceinline__ void hvx_store(unsigned a, unsigned b, unsigned c, unsigned e, void* base,
                                          unsigned long long pitch, int x, int y, int W, int H) {
  if (EDGE && y >= H) return;
  unsigned char* const r = (unsigned char*)base + (unsigned long long)y * pitch;
  if (!EDGE || x + 8 <= W) {
    if (ELEM == 1)
      *(uint2*)(r + x) = make_uint2(__byte_perm(a, b, 0x6420), __byte_perm(c, e, 0x6420));
    else
      *(uint4*)(r + 2 * x) = make_uint4(a ^ 0x80008000u, b ^ 0x80008000u, c ^ 0x80008000u,
                                        e ^ 0x80008000u);
    return;
  }
  const unsigned v[4] = {a, b, c, e};
  #pragma unroll
  for (int j = 0; j < 8; ++j) {
    const unsigned l = (v[j >> 1] >> (16 * (j & 1))) & 0xffffu;
    if (x + j < W) {
      if (ELEM == 1)
        r[x + j] = (unsigned char)l;
      else
        ((unsigned short*)r)[x + j] = (unsigned short)(l ^ 0x8000u);
    }
  }
}
// lanes of row y outside rectangle v become `zero`
template <int NW, int E>
__device__ __forceinline__ void hvx_valid(unsigned (&w)[NW], int x, int y, const int* v, unsigned zero) {
  const bool row = y >= v[1] && y < v[3];
  #pragma unroll
  for (int j = 0; j < NW; ++j) {
    const int c = x - E + 2 * j;
    if (!row || c < v[0] || c >= v[2]) w[j] = __byte_perm(w[j], zero, 0x3254);
    if (!row || c + 1 < v[0] || c + 1 >= v[2]) w[j] = __byte_perm(w[j], zero, 0x5410);
  }
}
// lanes left and right of the image: the nearest image lane, or a constant
template <int NW, int E, bool REP>
__device__ __forceinline__ void hvx_cols(unsigned (&w)[NW], int x, int W, unsigned cval) {
  if (x == 0) {
    const unsigned v = REP ? __byte_perm(w[E / 2], 0u, 0x1010) : cval;
    #pragma unroll
    for (int j = 0; j < E / 2; ++j) w[j] = v;
  }
  if (x + 8 + E > W) {
    #pragma unroll
    for (int j = E / 2; j < NW; ++j) {
      const int c = x - E + 2 * j;
      if (c >= W) w[j] = REP ? __byte_perm(w[j - 1], 0u, 0x3232) : cval;  // (c = x lies inside)
      else if (c + 1 >= W) w[j] = __byte_perm(w[j], REP ? w[j] : cval, REP ? 0x1010 : 0x5410);
    }
  }
}
)STRIP";
    }

    bool emit() {
        if (!plan()) return false;
        if (!globals.empty()) {
            acc_param = ", HvxAcc& acc";
            acc_arg = ", acc";
        }
        // the row step's body first: it decides the lanes of every image
        std::ostringstream head;
        for (int e = 0; e < d.n_in; ++e) {
            int box = -1;
            for (size_t i = 0; i < boxes.size(); ++i)
                if (boxes[i].ext == e) box = (int)i;
            const int b = d.in[e].buf;
            o << "    if constexpr (S >= " << -2 * halo(b) << ") {\n";
            emit_shift(b);
            emit_input(e, box);
            o << "    }\n";
        }
        ind = "      ";
        for (int k = 0; k < d.n_stage; ++k) {
            const GenStage& st = d.st[k];
            if (op_is_global(st.op)) continue;
            o << "    if constexpr (S >= " << -2 * halo(st.out) << ") {  // op " << k << "\n";
            emit_shift(st.out);
            if (!emit_stage(st) || !widen(st.out)) return false;
            emit_edge_fix(st.out);
            o << "    }\n";
        }
        o << "    if constexpr (S == 0) {\n";
        emit_outputs();
        emit_globals();
        o << "    }\n";
        const std::string body = o.str();
        o.str("");
        o.clear();
        o << "\n#ifdef HVX_STRIPS" << prelude();
        if (!globals.empty()) {
            o << reduction_prelude() << "struct HvxAcc {\n";
            for (int k : globals)
                if (d.st[k].op != OP_HIST)
                    o << "  " << (d.st[k].op == OP_MEANSTD ? "HvxSum" : "HvxMinMaxAcc") << " g" << k
                      << ";\n";
                else
                    o << "  unsigned* g" << k << ";\n";
            o << "};\n";
        }
        // a thread's windows, and what it knows about its strip
        o << "struct HvxWin {\n";
        for (int b = 0; b < d.n_buf; ++b)
            o << "  unsigned b" << b << "[" << D[b] << "][" << words(b) << "];  // lanes "
              << lane[b].lo << " .. " << lane[b].hi << ", bias " << lane[b].bias << "\n";
        o << "};\nstruct HvxStrip {\n  int x, yb, W, H;\n";
        for (size_t i = 0; i < boxes.size(); ++i) o << "  const unsigned char* box" << i << ";\n";
        for (int e = 0; e < d.n_in; ++e)
            o << "  const void* in" << e << ";\n  unsigned long long ip" << e << ";\n";
        for (int e = 0; e < d.n_out; ++e)
            o << "  void* out" << e << ";\n  unsigned long long op" << e << ";\n";
        for (int b = 0; b < d.n_buf; ++b)
            if (need_rect[b]) o << "  const int* v" << b << ";\n";
        o << "};\n";
        o << "// row i of the inputs that are read straight from memory\n"
          << "struct HvxRow {\n" << mem_decl << "};\n"
          << "template <bool EDGE>\n"
          << "__device__ __forceinline__ void hvx_rows(HvxRow& m, const HvxStrip& t, int i) {\n"
          << mem_rows << "}\n";
        o << "// step i of a strip: output row yb + i (S = 0), or a prologue step i < 0 of the\n"
          << "// images needed from step S on\n"
          << "template <bool EDGE, int S>\n"
          << "__device__ __forceinline__ void hvx_step(HvxWin& w, const HvxStrip& t, const HvxRow& m, "
             "int i"
          << acc_param << ") {\n"
          << body << "}\n";
        emit_kernels();
        o << "#endif\n";
        return true;
    }

    // The window of buffer b moves up one row.
    void emit_shift(int b) {
        for (int r = 0; r + 1 < D[b]; ++r)
            o << "      #pragma unroll\n      for (int j = 0; j < " << words(b) << "; ++j) w.b" << b << "[" << r
              << "][j] = w.b" << b << "[" << r + 1 << "][j];\n";
    }

    void emit_kernels() {
        // the prologue in phases of equal work: from step -2 h on images of halo h run
        std::vector<int> phase;
        for (int b = 0; b < d.n_buf; ++b)
            if (halo(b) > 0) phase.push_back(-2 * halo(b));
        std::sort(phase.begin(), phase.end());
        phase.erase(std::unique(phase.begin(), phase.end()), phase.end());
        phase.push_back(0);
        o << "template <bool EDGE>\n"
          << "__device__ __forceinline__ void hvx_strip(const HvxStrip& t, int R" << acc_param << ") {\n"
          << "  HvxWin w = {};\n";
        for (size_t k = 0; k + 1 < phase.size(); ++k)
            o << "  #pragma unroll 1\n  for (int i = " << phase[k] << "; i < " << phase[k + 1]
              << "; ++i) hvx_step<EDGE, " << phase[k] << ">(w, t, HvxRow{}, i" << acc_arg << ");\n";
        o << "  const int n = EDGE ? min(R, t.H - t.yb) : R;  // R is a multiple of " << unroll << "\n"
          << "  #pragma unroll 1\n"
          << "  for (int i = 0; i < n; i += " << unroll << ") {\n";
        // Inputs from memory: several rows' loads ahead of the first store after
        // them, as many as 32 registers hold (luma statistics of a 3840x2160 UYVY
        // frame: the whole call 49.6 us with 4 rows, 53.7 with 2)
        const int ahead = std::max(1, std::min(unroll, mem_words ? 32 / mem_words : unroll));
        o << "    HvxRow m[" << ahead << "];\n";
        for (int u = 0; u < unroll; ++u) {
            for (int k = u; u % ahead == 0 && k < std::min(u + ahead, unroll); ++k)
                o << "    hvx_rows<EDGE>(m[" << k % ahead << "], t, i + " << k << ");\n";
            o << "    hvx_step<EDGE, 0>(w, t, m[" << u % ahead << "], i + " << u << acc_arg << ");\n";
        }
        o << "  }\n";
        for (int k : globals)
            if (d.st[k].op == OP_MEANSTD) o << "  hvx_sum_flush(acc.g" << k << ");\n";
        o << "}\n";
        // box cells outside the image that some strip reads
        for (size_t i = 0; i < boxes.size(); ++i) {
            const int e = boxes[i].ext, b = d.in[e].buf, h = halo(b), fill = d.buf[b].fill;
            if (fill == FILL_NONE) continue;
            const std::string E_ = std::to_string(e);
            const std::string ld = "hvx_ld<" + std::to_string(d.in[e].fmt) + ">(p.in[" + E_ +
                                   "], p.in_pitch[" + E_ + "], ";
            // (the nearest pixel lies in the box: every tile reaches into the image)
            const char* at = fill == FILL_MIRROR ? "hvx_mirror(x, W), hvx_mirror(y, H))"
                                                 : "hvx_repeat(x, W), hvx_repeat(y, H))";
            const std::string near_x = "min(max(x, 0), W - 1)", near_y = "min(max(y, 0), H - 1)";
            o << "__device__ void hvx_fill" << i
              << "(const HvxJitParams& p, unsigned char* box, int x0, int y0, int R) {\n"
              << "  const int W = p.W, H = p.H;\n  constexpr int h = " << h << ";\n"
              << "  const int c0 = x0 - h, c1 = min(x0 + " << STRIP_TW << ", W) + h;\n"
              << "  const int r0 = y0 - h, r1 = min(y0 + 8 * R, H) + h;\n"
              << "  auto put = [&](int x, int y) {\n"
              << "    box[(y - r0) * " << STRIP_BOX_W << " + x - x0 + 16] = (unsigned char)"
              << (fill == FILL_CONSTANT    ? std::to_string(d.buf[b].cval) + "u"
                  : fill == FILL_REPLICATE ? "box[(" + near_y + " - r0) * " + std::to_string(STRIP_BOX_W) +
                                                 " + " + near_x + " - x0 + 16]"
                                           : ld + at)
              << ";\n  };\n"
              << "  // rows above and below the image, then the sides of the rows inside\n"
              << "  #pragma unroll 1\n  for (int k = 1; k <= h; ++k)\n"
              << "    for (int x = c0 + (int)threadIdx.x; x < c1; x += " << STRIP_THREADS << ") {\n"
              << "      if (-k >= r0) put(x, -k);\n      if (H - 1 + k < r1) put(x, H - 1 + k);\n    }\n"
              << "  const int ra = max(r0, 0), rb = min(r1, H);\n"
              << "  for (int i = threadIdx.x; i < (rb - ra) * h; i += " << STRIP_THREADS << ") {\n"
              << "    const int y = ra + i / h, k = i % h + 1;\n"
              << "    if (-k >= c0) put(-k, y);\n    if (W - 1 + k < c1) put(W - 1 + k, y);\n  }\n}\n";
        }
        // the boxes of one stage, their loads, and one tile on them
        const bool boxed = !boxes.empty();
        bool fills = false;
        o << "struct HvxBoxes {\n  unsigned char* b[" << std::max<size_t>(boxes.size(), 1) << "];\n"
          << "  unsigned bytes;\n};\n"
          << "__device__ __forceinline__ HvxBoxes hvx_boxes(unsigned char* sm, int R) {\n"
          << "  HvxBoxes x;\n  int end = 0;\n  x.bytes = 0;\n  x.b[0] = sm;\n";
        for (size_t i = 0; i < boxes.size(); ++i) {
            fills = fills || d.buf[d.in[boxes[i].ext].buf].fill != FILL_NONE;
            o << "  x.b[" << i << "] = sm + end;\n  x.bytes += " << STRIP_BOX_W * boxes[i].elem
              << "u * (8 * R + " << 2 * boxes[i].halo << ");\n  end += (" << STRIP_BOX_W * boxes[i].elem
              << " * (8 * R + " << 2 * boxes[i].halo << ") + 127) & ~127;\n";
        }
        o << "  return x;\n}\n";
        if (boxed) {
            o << "template <bool GMAP>\n"
              << "__device__ __forceinline__ void hvx_issue(const HvxJitParams& p, const HvxBoxes& x, "
                 "unsigned long long* bar, int x0, int y0) {\n"
              << "  hvx_expect_tx(bar, x.bytes);\n";
            for (size_t i = 0; i < boxes.size(); ++i)
                o << "  if (GMAP) hvx_tmap_acquire(&p.tmap[" << boxes[i].ext << "]);\n"
                  << "  hvx_tma_2d(x.b[" << i << "], &p.tmap[" << boxes[i].ext << "], bar, x0 - 16, y0 - "
                  << boxes[i].halo << ");\n";
            o << "}\n";
        }
        o << "__device__ __forceinline__ void hvx_strip_tile(const HvxJitParams& p, const HvxBoxes& bx, int tx, "
             "int ty"
          << acc_param << ") {\n"
          << "  const int R = p.rows, x0 = tx * " << STRIP_TW << ", y0 = ty * 8 * R;\n"
          << "  const int q = threadIdx.x & 15, g = threadIdx.x >> 4;\n"
          << "  const bool edge = tx < p.ix0 || tx > p.ix1 || ty < p.iy0 || ty > p.iy1;\n";
        if (fills) {
            o << "  if (edge) {\n";
            for (size_t i = 0; i < boxes.size(); ++i)
                if (d.buf[d.in[boxes[i].ext].buf].fill != FILL_NONE)
                    o << "    hvx_fill" << i << "(p, bx.b[" << i << "], x0, y0, R);\n";
            o << "    __syncthreads();\n  }\n";
        }
        o << "  HvxStrip t;\n  t.x = x0 + 8 * q;\n  t.yb = y0 + R * g;\n  t.W = p.W;\n  t.H = p.H;\n"
          << "  if (t.x >= t.W || t.yb >= t.H) return;\n";
        for (size_t i = 0; i < boxes.size(); ++i)
            o << "  t.box" << i << " = bx.b[" << i << "] + R * g * " << STRIP_BOX_W * boxes[i].elem << " + "
              << boxes[i].elem << " * (16 + 8 * q);\n";
        for (int e = 0; e < d.n_in; ++e)
            o << "  t.in" << e << " = p.in[" << e << "];\n  t.ip" << e << " = p.in_pitch[" << e << "];\n";
        for (int e = 0; e < d.n_out; ++e)
            o << "  t.out" << e << " = p.out[" << e << "];\n  t.op" << e << " = p.out_pitch[" << e
              << "];\n";
        for (int b = 0; b < d.n_buf; ++b)
            if (need_rect[b]) o << "  t.v" << b << " = p.valid[" << b << "];\n";
        // 5 resident CTAs (at most 102 registers): FChain and the morphology graph
        // run 1-2 % faster than at 4 or 6
        const std::string bounds = "__launch_bounds__(" + std::to_string(STRIP_THREADS) + ", 5)";
        o << "  if (edge) hvx_strip<true>(t, R" << acc_arg << ");\n  else hvx_strip<false>(t, R" << acc_arg
          << ");\n}\n\n";
        if (!globals.empty()) {
            emit_reduction_kernels(bounds);
            return;
        }
        o << "extern \"C\" __global__ void " << bounds
          << " hvx_generated_strips(const __grid_constant__ HvxJitParams p) {\n"
          << "  asm volatile(\"griddepcontrol.launch_dependents;\");\n"
          << "  extern __shared__ __align__(128) unsigned char hvx_box[];\n"
          << "  const int tx = blockIdx.x, ty = blockIdx.y;\n"
          << "  const HvxBoxes x = hvx_boxes(hvx_box + 128, p.rows);\n";
        if (boxed)
            o << "  unsigned long long* const bar = (unsigned long long*)hvx_box;\n"
              << "  if (threadIdx.x == 0) hvx_mbar_init(bar);\n  __syncthreads();\n";
        o << "  asm volatile(\"griddepcontrol.wait;\" ::: \"memory\");\n";
        if (boxed)
            o << "  if (threadIdx.x == 0) hvx_issue<false>(p, x, bar, tx * " << STRIP_TW
              << ", ty * 8 * p.rows);\n  hvx_mbar_wait(bar, p.err);\n";
        o << "  hvx_strip_tile(p, x, tx, ty);\n}\n\n"
          << "// n images in one launch.  Images of one size (rows > 0): block (x, y, z) is\n"
          << "// tile (x, y) of image z with `rows` rows per thread, so that its boxes are\n"
          << "// requested before any parameter has been read.  Otherwise block t is tile\n"
          << "// t - tile_start[i] of the last image i with tile_start[i] <= t.\n"
          << "extern \"C\" __global__ void " << bounds
          << " hvx_generated_strips_batch(const HvxJitParams* __restrict__ ps, const int* __restrict__ "
             "tile_start, int n, int rows) {\n"
          << "  asm volatile(\"griddepcontrol.launch_dependents;\");\n"
          << "  extern __shared__ __align__(128) unsigned char hvx_box[];\n"
          << "  int img, tx, ty;\n"
          << "  if (rows > 0) {\n    img = blockIdx.z;\n    tx = blockIdx.x;\n    ty = blockIdx.y;\n"
          << "  } else {\n"
          << "    const int t = blockIdx.x;\n"
          << "    int lo = 0, hi = n - 1;\n"
          << "    while (lo < hi) {\n"
          << "      const int mid = (lo + hi + 1) >> 1;\n"
          << "      if (__ldg(tile_start + mid) <= t) lo = mid; else hi = mid - 1;\n"
          << "    }\n"
          << "    const int local = t - __ldg(tile_start + lo), gx = (ps[lo].W + " << STRIP_TW - 1 << ") / "
          << STRIP_TW << ";\n"
          << "    img = lo;\n    ty = local / gx;\n    tx = local - ty * gx;\n"
          << "    rows = ps[lo].rows;\n  }\n"
          << "  const HvxJitParams& p = ps[img];\n"
          << "  const HvxBoxes x = hvx_boxes(hvx_box + 128, rows);\n";
        if (boxed)
            o << "  unsigned long long* const bar = (unsigned long long*)hvx_box;\n"
              << "  if (threadIdx.x == 0) {\n    hvx_mbar_init(bar);\n"
              << "    asm volatile(\"griddepcontrol.wait;\" ::: \"memory\");\n"
              << "    hvx_issue<true>(p, x, bar, tx * " << STRIP_TW << ", ty * 8 * rows);\n  }\n"
              << "  __syncthreads();\n";
        o << "  asm volatile(\"griddepcontrol.wait;\" ::: \"memory\");\n";
        if (boxed) o << "  hvx_mbar_wait(bar, p.err);\n";
        o << "  hvx_strip_tile(p, x, tx, ty);\n}\n";
    }
};

}  // namespace

bool emit_strips(const GenericDesc& d, std::string* source, StripPlan* plan) {
    StripEmitter em(d);
    if (!em.emit()) return false;
    *source = em.o.str();
    plan->unroll = em.unroll;
    plan->boxes = em.boxes;
    plan->reduces = !em.globals.empty();
    return true;
}

}  // namespace hvx
