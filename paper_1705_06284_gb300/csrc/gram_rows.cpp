// Row layouts of the shared-operand tensor-core contraction.
#include "gram_rows.h"

#include <algorithm>
#include <set>

namespace fbs {

namespace {

typedef std::array<int, 2> Row;

Row pair_row(int x, int y) { return x <= y ? Row{x, y} : Row{y, x}; }

// Rows ordered so that units of 16, chunks of 8 and halves of 4 rows need few
// distinct factors, as far as the rows allow it: first units of 4 x 4 bins
// (8 factors for 16 rows), then chunks of 2 x 4 (6 for 8), then groups of four
// with a common bin, then the rest, then the single bins.
class RowOrder {
  public:
    explicit RowOrder(const std::vector<Row> &r) {
        for (const Row &x : r) {
            if (x[1] < 0) {
                single_.push_back(x);
            } else {
                nb_ = std::max(nb_, x[1] + 1);
                pairs_.insert(x);
            }
        }
        std::sort(single_.begin(), single_.end());
        // the searches are over the bins that occur, at most 64 of them
        if (nb_ <= 64) {
            adj_.assign(nb_, 0);
            for (const Row &x : pairs_)
                if (x[0] != x[1]) {
                    adj_[x[0]] |= 1ULL << x[1];
                    adj_[x[1]] |= 1ULL << x[0];
                }
            if (nb_ <= 24) blocks(4);
            blocks(2);
        }
        stars();
        out_.insert(out_.end(), pairs_.begin(), pairs_.end());
        ngrouped_ = out_.size() - pairs_.size();
        out_.insert(out_.end(), single_.begin(), single_.end());
    }
    std::vector<Row> rows() const { return out_; }
    size_t grouped() const { return ngrouped_; }  // rows before the rest and the single bins

  private:
    void take(int x, int y) {
        const Row r = pair_row(x, y);
        pairs_.erase(r);
        out_.push_back(r);
        adj_[x] &= ~(1ULL << y);
        adj_[y] &= ~(1ULL << x);
    }
    // nx x 4 blocks of rows (nx bins times four others), while there are any:
    // the two bins that have the fewest partners in common, four at least,
    // and for nx = 4 the two that keep the most of those
    void blocks(int nx) {
        for (;;) {
            unsigned long long best = 0, bx = 0;
            int common = 65;
            for (int a = 0; a < nb_; ++a) {
                if (!adj_[a]) continue;
                for (int b = a + 1; b < nb_; ++b) {
                    unsigned long long x = 1ULL << a | 1ULL << b, m = adj_[a] & adj_[b] & ~x;
                    for (int k = 2; k < nx; ++k) {
                        int add = -1, most = 3;
                        for (int c = 0; c < nb_; ++c) {
                            const unsigned long long v = 1ULL << c;
                            const int n = x & v ? 0 : __builtin_popcountll(m & adj_[c] & ~v);
                            if (n > most) {
                                most = n;
                                add = c;
                            }
                        }
                        if (add < 0) {
                            m = 0;
                            break;
                        }
                        x |= 1ULL << add;
                        m &= adj_[add] & ~x;
                    }
                    const int n = __builtin_popcountll(m);
                    if (n >= 4 && n < common) {
                        best = m;
                        bx = x;
                        common = n;
                    }
                }
            }
            if (!best) return;
            for (; bx; bx &= bx - 1) {
                unsigned long long m = best;
                for (int k = 0; k < 4; ++k, m &= m - 1) take(__builtin_ctzll(bx), __builtin_ctzll(m));
            }
        }
    }
    void stars() {
        std::vector<int> deg(nb_, 0);
        for (const Row &x : pairs_) {
            ++deg[x[0]];
            if (x[1] != x[0]) ++deg[x[1]];
        }
        for (;;) {
            const int c = nb_ ? (int)(std::max_element(deg.begin(), deg.end()) - deg.begin()) : -1;
            if (c < 0 || deg[c] < 4) return;
            std::vector<Row> of;
            for (const Row &x : pairs_)
                if (x[0] == c || x[1] == c) of.push_back(x);
            // partners with the fewest rows left first: they fit few other groups
            std::stable_sort(of.begin(), of.end(), [&](const Row &u, const Row &v) {
                return deg[u[0] == c ? u[1] : u[0]] < deg[v[0] == c ? v[1] : v[0]];
            });
            for (int k = 0; k < 4; ++k) {
                --deg[of[k][0]];
                if (of[k][1] != of[k][0]) --deg[of[k][1]];
                pairs_.erase(of[k]);
                out_.push_back(of[k]);
            }
        }
    }
    int nb_ = 0;
    size_t ngrouped_ = 0;
    std::set<Row> pairs_;
    std::vector<Row> single_, out_;
    std::vector<unsigned long long> adj_;
};

void sort_rows(std::vector<Row> &r) { r = RowOrder(r).rows(); }

// Rows numbered: single bins, then pairs x <= y.
size_t row_key(const Row &r, int nb) { return r[1] < 0 ? (size_t)r[0] : (size_t)nb * (1 + r[0]) + r[1]; }
size_t row_keys(int nb) { return (size_t)nb * (nb + 1); }

void pad_rows(std::vector<Row> &r, int multiple) {
    while (r.size() % multiple) r.push_back(Row{-1, -1});
}

// Greedy vertex cover: vertices of the candidates (allowed[v]) until every
// item has one in one of its edges; at most `most`, else empty with ok = false.
std::vector<int> greedy_cover(int nv, const std::vector<std::vector<std::pair<int, int>>> &edges,
                              const std::vector<char> &allowed, int most, bool &ok) {
    std::vector<std::vector<int>> of(nv);
    std::vector<int> cnt(nv, 0);
    for (int i = 0; i < (int)edges.size(); ++i)
        for (const auto &e : edges[i])
            for (int v : {e.first, e.second})
                if (allowed[v] && (of[v].empty() || of[v].back() != i)) {
                    of[v].push_back(i);
                    ++cnt[v];
                }
    std::vector<char> done(edges.size(), 0);
    size_t left = edges.size();
    std::vector<int> cover;
    ok = true;
    while (left > 0) {
        const int best = (int)(std::max_element(cnt.begin(), cnt.end()) - cnt.begin());
        if (cnt[best] == 0 || (int)cover.size() >= most) {
            ok = false;
            return {};
        }
        cover.push_back(best);
        for (int i : of[best]) {
            if (done[i]) continue;
            done[i] = 1;
            --left;
            std::vector<int> seen;
            for (const auto &e : edges[i])
                for (int v : {e.first, e.second})
                    if (allowed[v] && std::find(seen.begin(), seen.end(), v) == seen.end()) {
                        seen.push_back(v);
                        --cnt[v];
                    }
        }
    }
    return cover;
}

// Rows that B need not hold when there are more than 128: operand A's first 32
// rows (`own`) are its own, the single bins and pairs of the cover that no item
// needs on the B side; the cover's other pairs are shared (32 rows, the rest
// formed a second time among A's own), and further pairs join A alone until
// 128 are left for B (one MMA of N = 256).  False when that does not fit.
template <typename Held>
bool own_a_rows(const std::vector<Row> &vert, const std::vector<std::vector<std::pair<int, int>>> &edges,
                std::vector<char> &in_a, std::vector<char> &in_b, const Held &held, std::vector<Row> &own) {
    const int nv = (int)vert.size();
    std::vector<char> pairs(nv, 0);
    int npairs = 0;
    for (int v = 0; v < nv; ++v) {
        pairs[v] = vert[v][1] >= 0;
        npairs += pairs[v];
        if (!pairs[v]) {
            own.push_back(vert[v]);
            in_a[v] = 1;
            in_b[v] = 0;
        }
    }
    std::vector<std::vector<std::pair<int, int>>> open;  // items that need a pair of operand A
    std::vector<std::vector<int>> of(nv);
    for (int i = 0; i < (int)edges.size(); ++i) {
        bool quad = true;
        for (const auto &k : edges[i])
            for (int v : {k.first, k.second}) {
                quad &= pairs[v];
                if (of[v].empty() || of[v].back() != i) of[v].push_back(i);
            }
        if (quad) open.push_back(edges[i]);
    }
    if ((int)own.size() > 32) return false;
    bool ok = true;
    const std::vector<int> cover = greedy_cover(nv, open, pairs, kGramARows - (int)own.size(), ok);
    if (!ok) return false;
    for (int v : cover) in_a[v] = 1;
    int left = npairs, shared = (int)cover.size();
    auto move = [&](int v) {  // v on A alone, if every item keeps a slot
        const char was = in_a[v];
        in_a[v] = 1;
        in_b[v] = 0;
        for (int i : of[v])
            if (!held(edges[i])) {
                in_a[v] = was;
                in_b[v] = 1;
                return false;
            }
        own.push_back(vert[v]);
        --left;
        return true;
    };
    for (int k = (int)cover.size() - 1; k >= 0 && own.size() < 32 && (shared > 32 || left > 128); --k)
        if (move(cover[k])) --shared;
    for (int v = 0; v < nv && left > 128 && own.size() < 32; ++v)
        if (pairs[v] && !in_a[v]) move(v);
    for (int k = (int)cover.size() - 1; k >= 0 && shared > 32 && own.size() < 32; --k)
        if (in_b[cover[k]]) {
            own.push_back(vert[cover[k]]);
            --shared;
        }
    return left <= 128 && shared <= 32;
}

}  // namespace

bool gram_rows_shared(int nb, const std::vector<std::array<int, 4>> &items, GramRows &out) {
    std::vector<int> id(row_keys(nb), -1);
    std::vector<Row> vert;
    auto vertex = [&](Row r) {
        int &v = id[row_key(r, nb)];
        if (v < 0) {
            v = (int)vert.size();
            vert.push_back(r);
        }
        return v;
    };
    std::vector<std::vector<std::pair<int, int>>> edges(items.size());
    for (size_t i = 0; i < items.size(); ++i) {
        const auto &t = items[i];
        auto add = [&](Row p, Row q) {
            std::pair<int, int> e(vertex(p), vertex(q));
            if (e.first > e.second) std::swap(e.first, e.second);
            if (std::find(edges[i].begin(), edges[i].end(), e) == edges[i].end()) edges[i].push_back(e);
        };
        if (t[3] < 0) {
            add(pair_row(t[1], t[2]), Row{t[0], -1});
            add(pair_row(t[0], t[2]), Row{t[1], -1});
            add(pair_row(t[0], t[1]), Row{t[2], -1});
        } else {
            add(pair_row(t[0], t[1]), pair_row(t[2], t[3]));
            add(pair_row(t[0], t[2]), pair_row(t[1], t[3]));
            add(pair_row(t[0], t[3]), pair_row(t[1], t[2]));
        }
    }
    const int nv = (int)vert.size();
    std::vector<char> in_a(nv, 0), in_b(nv, 1);
    auto held = [&](const std::vector<std::pair<int, int>> &e) {
        for (const auto &k : e)
            if ((in_a[k.first] && in_b[k.second]) || (in_a[k.second] && in_b[k.first])) return true;
        return false;
    };
    std::vector<Row> own, rows;  // rows of operand A alone, then all rows
    bool ok = nv > 128 && own_a_rows(vert, edges, in_a, in_b, held, own);
    if (!ok) {  // every row on both sides: A is a cover of the items, B all rows
        std::fill(in_b.begin(), in_b.end(), 1);
        std::fill(in_a.begin(), in_a.end(), 0);
        own.clear();
        if (nv > kGramBRows) return false;
        for (int v : greedy_cover(nv, edges, std::vector<char>(nv, 1), kGramARows, ok)) in_a[v] = 1;
        if (!ok) return false;
    }
    std::vector<Row> ab, b;
    std::vector<int> at_a(nv, -1), at_b(nv, -1);  // the A and B row of every vertex
    for (int v = 0; v < nv; ++v) {
        const bool twice = std::find(own.begin(), own.end(), vert[v]) != own.end();
        if (in_b[v]) (in_a[v] && !twice ? ab : b).push_back(vert[v]);
    }
    sort_rows(own);
    sort_rows(ab);
    const RowOrder ob(b);
    b = ob.rows();
    rows = own;
    if (!own.empty()) pad_rows(rows, 32);
    out.jb0 = (int)rows.size() / 8;
    rows.insert(rows.end(), ab.begin(), ab.end());
    // the rest of B starts on a unit: its rows outside any group fill up the last one of A
    size_t lead = std::min((16 - rows.size() % 16) % 16, b.size() - ob.grouped());
    if ((rows.size() + lead) % 16) lead = 0;
    rows.insert(rows.end(), b.begin() + ob.grouped(), b.begin() + ob.grouped() + lead);
    b.erase(b.begin() + ob.grouped(), b.begin() + ob.grouped() + lead);
    rows.insert(rows.end(), b.begin(), b.end());
    out.nbch = ((int)rows.size() - 8 * out.jb0 + 7) / 8;
    for (int r = 0; r < (int)rows.size(); ++r) {
        if (rows[r][0] < 0) continue;
        const int v = vertex(rows[r]);
        if (r < kGramARows && at_a[v] < 0) at_a[v] = r;
        if (r >= 8 * out.jb0 && at_b[v] < 0) at_b[v] = r - 8 * out.jb0;
    }
    out.items.clear();
    for (size_t i = 0; i < items.size(); ++i) {
        bool placed = false;
        for (const auto &e : edges[i])
            for (int k = 0; k < 2 && !placed; ++k) {
                const int p = at_a[k ? e.second : e.first], q = at_b[k ? e.first : e.second];
                if (p < 0 || q < 0) continue;
                out.items.push_back({p, q, (int)i});
                placed = true;
            }
        if (!placed) return false;
    }
    std::sort(out.items.begin(), out.items.end());
    pad_rows(rows, 16);
    out.rows = rows;
    return true;
}

namespace {

// The third bin of a triplet carried by the pair with this key.
int rest_of(const std::array<int, 3> &t, int key, int nb) { return t[0] + t[1] + t[2] - key / nb - key % nb; }

}  // namespace

bool gram_rows_pairs(int nb, const std::vector<std::array<int, 3>> &trip, const std::vector<int> &key,
                     GramRows &out) {
    std::vector<int> arow((size_t)nb * nb, -1), brow(nb, -1);
    std::vector<Row> rows;
    for (size_t i = 0; i < trip.size(); ++i) {
        if (arow[key[i]] < 0) rows.push_back(Row{key[i] / nb, key[i] % nb});
        arow[key[i]] = 0;
        brow[rest_of(trip[i], key[i], nb)] = 0;
        if ((int)rows.size() > kGramARows) return false;
    }
    sort_rows(rows);
    for (int r = 0; r < (int)rows.size(); ++r) arow[rows[r][0] * nb + rows[r][1]] = r;
    pad_rows(rows, 32);
    out.jb0 = (int)rows.size() / 8;
    for (int b = 0; b < nb; ++b)
        if (brow[b] >= 0) {
            brow[b] = (int)rows.size() - 8 * out.jb0;
            rows.push_back(Row{b, -1});
        }
    out.nbch = ((int)rows.size() - 8 * out.jb0 + 7) / 8;
    if (out.nbch > kGramBRows / 8) return false;
    out.items.clear();
    for (size_t i = 0; i < trip.size(); ++i)
        out.items.push_back({arow[key[i]], brow[rest_of(trip[i], key[i], nb)], (int)i});
    std::sort(out.items.begin(), out.items.end());
    pad_rows(rows, 16);
    out.rows = rows;
    return true;
}

bool gram_rows_wide(int nb, const std::vector<std::array<int, 3>> &trip, const std::vector<int> &key,
                    std::vector<GramRows> &out) {
    std::vector<int> arow(nb, -1), brow((size_t)nb * nb, -1);  // of a single bin; of a pair, among all B rows
    std::vector<Row> left, right;
    for (size_t i = 0; i < trip.size(); ++i) {
        arow[rest_of(trip[i], key[i], nb)] = 0;
        if (brow[key[i]] < 0) right.push_back(Row{key[i] / nb, key[i] % nb});
        brow[key[i]] = 0;
    }
    for (int b = 0; b < nb; ++b)
        if (arow[b] >= 0) {
            arow[b] = (int)left.size();
            left.push_back(Row{b, -1});
        }
    if ((int)left.size() > kGramARows || right.empty()) return false;
    pad_rows(left, 32);
    const int np = (int)right.size(), groups = (np + kGramBRows - 1) / kGramBRows;
    const int per = ((np + groups - 1) / groups + 15) / 16 * 16;  // whole 16-row units, balanced
    out.assign((np + per - 1) / per, GramRows{});
    for (auto &g : out) {
        g.rows = left;
        g.jb0 = (int)left.size() / 8;
    }
    sort_rows(right);
    for (int n = 0; n < np; ++n) {
        brow[right[n][0] * nb + right[n][1]] = n;
        out[n / per].rows.push_back(right[n]);
    }
    for (size_t i = 0; i < trip.size(); ++i) {
        const int b = brow[key[i]];
        out[b / per].items.push_back({arow[rest_of(trip[i], key[i], nb)], b % per, (int)i});
    }
    for (auto &g : out) {
        g.nbch = ((int)g.rows.size() - 8 * g.jb0 + 7) / 8;
        std::sort(g.items.begin(), g.items.end());
        pad_rows(g.rows, 16);
    }
    return true;
}

}  // namespace fbs
