// The slice, contraction and walk compilers, checked on the host: what they build is interpreted as the kernels do it and compared with
// the recurrences themselves (Eq. 1 for every node, tails, Alg. 1 for time intervals), every index against its array, every 32-bit sum
// against its range.  Built and called by test_host_programs.py.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>

#include "../paper_2607_12324_b200/csrc/emo_contract.h"
#include "../paper_2607_12324_b200/csrc/emo_slice.h"
#include "../paper_2607_12324_b200/csrc/emo_walk.h"

using namespace emo;

namespace {

struct Failed {};
char g_what[256];
#define CHECK(x)                                                                    \
    do {                                                                            \
        if (!(x)) {                                                                 \
            std::snprintf(g_what, sizeof(g_what), "line %d: %s", __LINE__, #x);      \
            throw Failed();                                                         \
        }                                                                           \
    } while (0)

struct Input {
    HostGraph g;
    std::vector<int64_t> lat;
    std::vector<double> energy;
    GraphBounds b;
};

Input take(int32_t n, const int64_t *rp, const int32_t *col, const int32_t *group, int32_t rows, int32_t L, const int64_t *lat, const double *energy)
{
    Input in;
    in.g.n = n;
    in.g.L = L;
    in.g.rows = rows;
    in.g.m = rp[n];
    in.g.row_ptr.assign(rp, rp + n + 1);
    in.g.col.assign(col, col + rp[n]);
    in.g.group.assign(group, group + n);
    in.lat.assign(lat, lat + (size_t)n * L);
    in.energy.assign(energy, energy + (size_t)n * L);
    graph_bounds(in.g, lat, energy, in.b);
    return in;
}

int add32(int64_t a, int64_t b)
{
    CHECK(a + b >= INT32_MIN && a + b <= INT32_MAX);
    return (int)(a + b);
}

constexpr int kAbsent = -(1 << 30);

// One direction of a slice as a thread walks it: V the values' type, none the operand that an operation begins with.
template <typename V>
void walk_ops(const uint32_t *ops, unsigned steps, unsigned slots, unsigned unread, const std::vector<uint32_t> &inc, std::vector<V> &val, std::vector<char> &known)
{
    V acc = kAbsent;
    for (unsigned k = 0; k < steps; ++k, ops += kSliceStepWords) {
        V x[2];
        for (int i = 0; i < 2; ++i) {
            const unsigned slot = ops[i] & 0xFFFFu, entry = ops[i] >> 16;
            CHECK(slot < slots && entry < inc.size() && slot != unread && known[slot]);
            const int64_t y = (int64_t)val[slot] + inc[entry];
            CHECK(sizeof(V) == 8 || (y >= INT32_MIN && y <= INT32_MAX));
            x[i] = (V)y;
        }
        const V y = std::max(acc, std::max(x[0], x[1]));
        CHECK(ops[2] < slots && ops[3] < 2 && (ops[3] || ops[2] == unread));
        val[ops[2]] = y;
        known[ops[2]] = 1;
        acc = ops[3] ? (V)kAbsent : y;
    }
}

int check_slices(const Input &in, unsigned seed, int32_t *info)
{
    const HostGraph &g = in.g;
    const int n = g.n, L = g.L;
    Slices s;
    compile_slices(g, in.lat.data(), in.energy.data(), in.b, s);
    if (!s.ok) return 0;
    info[0] = s.count;
    info[1] = s.cols;
    info[2] = s.groups;
    info[3] = s.group;
    std::mt19937 rng(seed);
    std::vector<int> lv((size_t)std::max(g.rows, 1));
    for (int &x : lv) x = (int)(rng() % (unsigned)L);
    std::vector<int64_t> t((size_t)n), ES((size_t)n, 0), C((size_t)n), Q((size_t)n, 0);
    int64_t T = 0;
    double E = 0.0;
    for (int v = 0; v < n; ++v) {
        const size_t at = (size_t)v * L + (g.group[v] >= 0 ? lv[g.group[v]] : 0);
        t[v] = in.lat[at];
        E += in.energy[at];
        for (int64_t e = g.row_ptr[v]; e < g.row_ptr[v + 1]; ++e) ES[v] = std::max(ES[v], C[g.col[e]]);
        C[v] = ES[v] + t[v];
        T = std::max(T, C[v]);
    }
    for (int v = n - 1; v >= 0; --v) {
        Q[v] += t[v];
        for (int64_t e = g.row_ptr[v]; e < g.row_ptr[v + 1]; ++e) Q[g.col[e]] = std::max(Q[g.col[e]], Q[v]);
    }

    const int CW = s.cols;
    const size_t size = (size_t)CW * CW;
    CHECK(CW % 4 == 0 && CW <= kSliceMaxCols && (int)s.off.size() == s.count + 1);
    std::vector<SliceHdr> H((size_t)s.count);
    std::vector<std::vector<int>> M[2];
    std::vector<std::vector<uint32_t>> inc[2];
    uint32_t placed = 0;
    double E2 = 0.0;
    for (int k = 0; k < s.count; ++k) {
        const uint32_t *const w = s.blob.data() + s.off[(size_t)k];
        SliceHdr &h = H[(size_t)k];
        std::memcpy(&h, w, sizeof(h));
        CHECK(s.off[(size_t)k] % 4 == 0 && h.words % 4 == 0 && h.head % 4 == 0 && s.off[(size_t)k + 1] - s.off[(size_t)k] == h.words);
        CHECK(h.nodes > 0 && h.nodes <= (uint32_t)kSliceNodes && h.node0 == placed);
        placed += h.nodes;
        for (int d = 0; d < 2; ++d) {
            const SliceDirHdr &D = h.dir[d];
            CHECK(D.off_path + D.paths <= h.head && D.off_out + D.outs <= h.head && D.off_ops1 >= h.head && D.off_ops1 % 4 == 0 && D.off_ops2 % 4 == 0);
            CHECK(D.off_ops1 + kSliceStepWords * (D.steps + 1) <= h.words && D.off_ops2 + kSliceStepWords * (D.steps + 1) <= h.words);
            CHECK(D.cols <= (uint32_t)CW && D.outs <= (uint32_t)CW && D.cols < D.slots1 && D.cols < D.slots2);
            // durations, then running sums along the paths
            std::vector<uint32_t> a(D.len, 0xDEADBEEFu);
            for (uint32_t i = 0; i < h.nodes; ++i) {
                const size_t at = (size_t)(h.node0 + i);
                const uint32_t *const r = s.rec.data() + at * 4;
                const uint32_t entry = d ? r[2] >> 16 : r[2] & 0xFFFFu;
                CHECK(entry > 0 && entry < D.len && (d ? r[3] >> 16 : r[3] & 0xFFFFu) < D.slots2);
                CHECK((r[0] == kNone || r[0] < (uint32_t)g.rows) && r[1] < (uint32_t)n);
                const size_t e = at * (size_t)s.Lp + (size_t)(r[0] != kNone ? lv[r[0]] : 0);
                a[entry] = s.tabT[e];
                CHECK((int64_t)a[entry] == t[r[1]]);
                if (d == 0) E2 += s.tabE[e];
            }
            uint32_t all = 0;
            for (uint32_t p = 0; p < D.paths; ++p) {
                const uint32_t first = w[D.off_path + p] & 0xFFFFu, len = w[D.off_path + p] >> 16;
                CHECK(first + len < D.len && (p > 0 || first == 0));
                a[first] = 0;
                for (uint32_t i = 1; i <= len; ++i) a[first + i] += a[first + i - 1];
                all += len + 1;
            }
            CHECK(all == D.len);
            inc[d].push_back(a);
            // the matrix, column by column
            std::vector<int> m(size, kAbsent);
            for (uint32_t c = 0; c < D.cols; ++c) {
                std::vector<int> val(D.slots1, 0);
                std::vector<char> known(D.slots1, 0);
                for (uint32_t j = 0; j < D.cols; ++j) {
                    val[j] = j == c ? 0 : kAbsent;
                    known[j] = 1;
                }
                walk_ops<int>(w + D.off_ops1, D.steps, D.slots1, D.cols, inc[d].back(), val, known);
                for (uint32_t i = 0; i < D.outs; ++i) {
                    const uint32_t o = w[D.off_out + i];
                    CHECK((o & 0xFFFFu) < D.slots1 && (o >> 16) < D.len && known[o & 0xFFFFu]);
                    m[i * (size_t)CW + c] = std::max(add32(val[o & 0xFFFFu], inc[d].back()[o >> 16]), kAbsent);
                }
            }
            M[d].push_back(m);
        }
    }
    CHECK(placed == (uint32_t)n && std::fabs(E - E2) <= 1e-12 * std::max(1.0, std::fabs(E)));
    CHECK((int64_t)s.group * s.groups >= s.count && (int64_t)s.group * (s.groups - 1) < s.count);

    // the values that enter every slice: matrix by matrix, and by the products of whole groups
    std::vector<std::vector<int64_t>> st[2];
    int64_t T2 = 0;
    for (int d = 0; d < 2; ++d) {
        st[d].resize((size_t)s.count);
        std::vector<int64_t> c((size_t)CW, 0), cg((size_t)CW, 0);
        std::vector<int> P(size);
        int64_t Tg = 0;
        for (int x = 0; x < s.count; ++x) {
            const int k = d ? s.count - 1 - x : x;
            const std::vector<int> &m = M[d][(size_t)k];
            CHECK(x ? H[(size_t)(d ? k + 1 : k - 1)].dir[d].outs == H[(size_t)k].dir[d].cols : H[(size_t)k].dir[d].cols == 1);
            st[d][(size_t)k] = c;
            std::vector<int64_t> o((size_t)CW, 0);
            for (int i = 0; i < CW; ++i)
                for (int j = 0; j < CW; ++j)
                    if (m[(size_t)i * CW + j] >= 0) o[(size_t)i] = std::max(o[(size_t)i], c[(size_t)j] + m[(size_t)i * CW + j]);
            if (d == 0) T2 = std::max(T2, o[0]);
            o[0] = 0;
            c = o;
            if (s.groups > 1) {
                // groups run from the first slice on in both directions; a group's product, row 0 collecting its maximum
                const bool begins = d ? x == 0 || (k + 1) % s.group == 0 : k % s.group == 0;
                const bool ends = d ? k % s.group == 0 : (k + 1) % s.group == 0 || k == s.count - 1;
                if (begins)
                    for (int i = 0; i < CW; ++i)
                        for (int j = 0; j < CW; ++j) P[(size_t)i * CW + j] = i == j ? 0 : kAbsent;
                std::vector<int> first(begins ? std::vector<int>((size_t)CW, kAbsent) : std::vector<int>(P.begin(), P.begin() + CW));
                std::vector<int> R(size);
                for (int j = 0; j < CW; ++j) {
                    std::vector<int> col((size_t)CW);
                    for (int i = 0; i < CW; ++i) col[(size_t)i] = i ? P[(size_t)i * CW + j] : (j ? kAbsent : 0);
                    for (int i = 0; i < CW; ++i) {
                        int best = kAbsent;
                        for (int l = 0; l < CW; ++l) best = std::max(best, add32(m[(size_t)i * CW + l], col[(size_t)l]));
                        R[(size_t)i * CW + j] = i ? best : std::max(best, first[(size_t)j]);
                    }
                }
                P = R;
                if (ends) {
                    std::vector<int64_t> og((size_t)CW, 0);
                    for (int i = 0; i < CW; ++i)
                        for (int j = 0; j < CW; ++j)
                            if (P[(size_t)i * CW + j] >= 0) og[(size_t)i] = std::max(og[(size_t)i], cg[(size_t)j] + P[(size_t)i * CW + j]);
                    Tg = std::max(Tg, og[0]);
                    og[0] = 0;
                    cg = og;
                    CHECK(cg == c);
                }
            }
        }
        CHECK(d == 1 || s.groups == 1 || Tg == T);
    }
    CHECK(T2 == T);
    for (int k = 0; k < s.count; ++k) {
        const SliceHdr &h = H[(size_t)k];
        const uint32_t *const w = s.blob.data() + s.off[(size_t)k];
        std::vector<int64_t> val[2];
        for (int d = 0; d < 2; ++d) {
            const SliceDirHdr &D = h.dir[d];
            val[d].assign(D.slots2, 0);
            std::vector<char> known(D.slots2, 0);
            for (uint32_t j = 0; j < D.cols; ++j) {
                val[d][j] = st[d][(size_t)k][j];
                known[j] = 1;
            }
            walk_ops<int64_t>(w + D.off_ops2, D.steps, D.slots2, D.cols, inc[d][(size_t)k], val[d], known);
        }
        CHECK(s.count > 1 || val[0][h.dir[0].term] == T);
        for (uint32_t i = 0; i < h.nodes; ++i) {
            const uint32_t *const r = s.rec.data() + (size_t)(h.node0 + i) * 4;
            CHECK(val[0][r[3] & 0xFFFFu] + inc[0][(size_t)k][(r[2] & 0xFFFFu) - 1u] == ES[r[1]]);
            CHECK(val[1][r[3] >> 16] + inc[1][(size_t)k][r[2] >> 16] == Q[r[1]]);
        }
    }
    return 1;
}

int check_contract(const Input &in, unsigned seed, int32_t *info)
{
    const HostGraph &g = in.g;
    const int L = g.L;
    Contracted c;
    contract_forward(g, in.lat.data(), in.energy.data(), in.b, false, c);
    info[0] = c.n;
    CHECK(c.n <= g.n && (int)c.group.size() == c.n && (int)c.row_ptr.size() == c.n + 1 && c.row_ptr.back() == (int64_t)c.col.size());
    std::mt19937 rng(seed);
    for (int trial = 0; trial < 3; ++trial) {
        std::vector<int> lv((size_t)std::max(g.rows, 1));
        for (int &x : lv) x = trial ? (int)(rng() % (unsigned)L) : L - 1;
        auto evaluate = [&](int32_t n, const std::vector<int64_t> &rp, const std::vector<int32_t> &col, const std::vector<int32_t> &group, const std::vector<int64_t> &lat,
                            const std::vector<double> &energy, double &E) {
            std::vector<int64_t> C((size_t)n);
            int64_t T = 0;
            for (int32_t v = 0; v < n; ++v) {
                CHECK(group[v] < g.rows);
                int64_t start = 0;
                for (int64_t e = rp[v]; e < rp[v + 1]; ++e) {
                    CHECK(col[e] >= 0 && col[e] < v);
                    start = std::max(start, C[col[e]]);
                }
                const size_t at = (size_t)v * L + (group[v] >= 0 ? lv[group[v]] : 0);
                CHECK(lat[at] >= 0 && lat[at] < (int64_t)1 << 32);
                C[v] = start + lat[at];
                E += energy[at];
                T = std::max(T, C[v]);
            }
            return T;
        };
        double E = 0.0, Ec = 0.0;
        const int64_t T = evaluate(g.n, g.row_ptr, g.col, g.group, in.lat, in.energy, E), Tc = evaluate(c.n, c.row_ptr, c.col, c.group, c.lat, c.energy, Ec);
        CHECK(T == Tc && std::fabs(E - Ec) <= 1e-12 * std::max(1.0, std::fabs(E)));
    }
    return 1;
}

int check_walk(const Input &in, unsigned seed, int32_t *info)
{
    const HostGraph &g = in.g;
    const int n = g.n, L = g.L;
    Walk w;
    compile_walk(g, in.lat.data(), in.energy.data(), in.b, w);
    if (!w.ok) return 0;
    info[0] = w.chunks;
    info[1] = w.slots;
    info[2] = (int32_t)w.chunk_bytes;
    CHECK(w.blob.size() == (size_t)w.chunks * w.chunk_bytes && w.chunk_bytes % 16 == 0 && w.off_dur % 16 == 0 && w.off_en % 16 == 0);
    constexpr int kBig = (1 << 30) - 1;
    std::mt19937 rng(seed);
    for (int trial = 0; trial < 3; ++trial) {
        const int I = 1 + (int)(rng() % 10u);
        int64_t T0 = 0;
        for (int v = 0; v < n; ++v) T0 = std::max(T0, in.b.lbC[v]);
        const int64_t delta = std::max<int64_t>(1, T0 / (1 + rng() % (2u * (unsigned)I)));
        if (delta >= kWalkMaxDur) continue;
        const int rows = std::max(g.rows, 1);
        std::vector<int> F((size_t)rows * I);
        for (int &x : F) x = (int)(rng() % (unsigned)L);
        std::vector<int64_t> C((size_t)n), busy((size_t)rows * I, 0), busy2(busy);
        double E = 0.0, E2 = w.energy0;
        int64_t T = 0, T2 = 0;
        for (int v = 0; v < n; ++v) {
            int64_t start = 0;
            for (int64_t e = g.row_ptr[v]; e < g.row_ptr[v + 1]; ++e) start = std::max(start, C[g.col[e]]);
            const size_t at = (size_t)v * L + (size_t)(g.group[v] >= 0 ? F[(size_t)g.group[v] * I + (size_t)std::min<int64_t>(start / delta, I - 1)] : 0);
            C[v] = start + in.lat[at];
            E += in.energy[at];
            T = std::max(T, C[v]);
            if (g.group[v] >= 0)
                for (int i = 0; i < I; ++i) {
                    const int64_t lo = i * delta, hi = i + 1 < I ? lo + delta : INT64_MAX;
                    busy[(size_t)g.group[v] * I + i] += std::max<int64_t>(0, std::min(hi, C[v]) - std::max(lo, start));
                }
        }
        // one policy's walk, node by node
        std::vector<int64_t> slot((size_t)w.slots, -1);
        slot[0] = 0;
        int64_t t = 0, iend = 0, bacc = 0;
        int left = 1, i = 0, row = 0, la = 0, la2 = 0;
        auto level = [&](int r, int k) { return F[(size_t)r * I + (size_t)std::min(k, I - 1)]; };
        auto flush = [&](int64_t x) {
            CHECK(x >= 0);
            busy2[(size_t)row * I + i] += x;
        };
        for (int k = 0; k < w.chunks; ++k) {
            const unsigned char *const p = w.blob.data() + (size_t)k * w.chunk_bytes;
            const uint32_t *q = reinterpret_cast<const uint32_t *>(p);
            const uint32_t items = q[0];
            CHECK((1 + items + 1) * 16 <= w.off_dur);
            for (uint32_t a = 0; a < items; ++a) {
                q += 4;
                if (q[0] & kWalkStart) {
                    const uint32_t x = q[1] & 0xFFFFu, y = q[1] >> 16;
                    CHECK((int)x < w.slots && (int)y < w.slots && slot[x] >= 0 && slot[y] >= 0);
                    const int64_t z = std::max(slot[x], slot[y]);
                    t = (q[0] & kWalkMore) ? std::max(t, z) : z;
                }
                if (q[0] & kWalkFix) t += q[2];
                const int nodes = (int)(q[0] & 15u);
                if (nodes) {
                    CHECK(nodes <= kWalkRun && (int)q[2] < rows && q[3] + (uint32_t)nodes <= (uint32_t)kWalkRows);
                    if (q[0] & kWalkFresh) {
                        const int x = (int)std::min<int64_t>(t / delta, I - 1);
                        if (x != i || (int)q[2] != row) {
                            flush(bacc);
                            bacc = 0;
                        }
                        i = x;
                        row = (int)q[2];
                        la = level(row, x);
                        la2 = level(row, x + 1);
                        iend = x == I - 1 ? t + kBig : (x + 1) * delta;
                        left = (int)(iend - t);
                    }
                    CHECK(row == (int)q[2] && left > 0 && t == iend - left);
                    int64_t longest = 0;
                    for (int j = 0; j < nodes; ++j) {
                        const uint32_t *const d = reinterpret_cast<const uint32_t *>(p + w.off_dur) + (size_t)(q[3] + (uint32_t)j) * w.Lp;
                        const double *const e = reinterpret_cast<const double *>(p + w.off_en) + (size_t)(q[3] + (uint32_t)j) * w.Lp;
                        longest += *std::max_element(d, d + w.Lp);
                        E2 += e[la];
                        bacc += d[la];
                        left = add32(left, -(int64_t)d[la]);
                        while (left <= 0) {
                            flush(bacc + left);
                            bacc = -left;
                            const int next = std::min(i + 1, I - 1), step = next == I - 1 ? kBig : (int)delta;
                            i = next;
                            iend += step;
                            left += step;
                            la = la2;
                            la2 = level(row, next + 1);
                        }
                    }
                    CHECK(longest < kWalkMaxDur);      // (a run's sums are signed 32-bit numbers at any levels)
                    t = iend - left;
                }
                if (q[0] & kWalkPub) {
                    CHECK((int)(q[0] >> 16) < w.slots && (q[0] >> 16) > 0);
                    slot[q[0] >> 16] = t;
                }
                if (q[0] & kWalkTerm) T2 = std::max(T2, t);
            }
        }
        flush(bacc);
        CHECK(T == T2 && busy == busy2 && std::fabs(E - E2) <= 1e-12 * std::max(1.0, std::fabs(E)));
    }
    return 1;
}

}  // namespace

extern "C" {

const char *program_failure() { return g_what; }

// 1: built and right, 0: the compiler leaves the graph to others, -1: program_failure() says what.  kind: 0 slices (info: slices, columns,
// groups, slices of a group), 1 contraction (nodes left), 2 walk (chunks, slots, bytes of a chunk).
int program_check(int kind, int32_t n, const int64_t *rp, const int32_t *col, const int32_t *group, int32_t rows, int32_t L, const int64_t *lat, const double *energy, uint32_t seed,
                  int32_t *info)
{
    try {
        const Input in = take(n, rp, col, group, rows, L, lat, energy);
        return kind == 0 ? check_slices(in, seed, info) : (kind == 1 ? check_contract(in, seed, info) : check_walk(in, seed, info));
    } catch (const Failed &) {
        return -1;
    }
}

// Compiles only (bounds included).  Walk: -1 where a program that is refused is kept all the same.
int program_compile(int kind, int32_t n, const int64_t *rp, const int32_t *col, const int32_t *group, int32_t rows, int32_t L, const int64_t *lat, const double *energy)
{
    const Input in = take(n, rp, col, group, rows, L, lat, energy);
    if (kind == 0) {
        Slices s;
        compile_slices(in.g, lat, energy, in.b, s);
        return s.ok;
    }
    if (kind == 1) {
        Contracted c;
        contract_forward(in.g, lat, energy, in.b, false, c);
        return c.n;
    }
    Walk w;
    compile_walk(in.g, lat, energy, in.b, w);
    return w.ok ? 1 : (w.blob.empty() ? 0 : -1);
}

}  // extern "C"
