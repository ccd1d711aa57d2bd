// elim.cpp -- plans the eliminated walk (elim.hpp) and writes its generated kernel.
#include "elim.hpp"

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <sstream>

namespace perm {

namespace {

inline int pc(uint64_t v) { return __builtin_popcountll(v); }

// Elimination of the low columns `L` from tables with the given scopes, cost
// only: the column whose tables have the smallest joint scope goes first, its
// tables are multiplied in order of growing joint scope, and the last product
// is fused with the subtraction of the column-on half.
struct Sim {
    double ops = 0.0;
    int order[kNMax];
};

// The order in which the tables of a bucket are multiplied: smallest scope
// first, then always the table that grows the joint scope least.
// (`late`, if given, marks tables to come after all others.)
int bucket_order(const uint64_t *scope, const int *idx, int t, int *seq, const int *late = nullptr) {
    bool used[2 * kNMax] = {};
    uint64_t u = 0;
    for (int s = 0; s < t; ++s) {
        int best = -1, bk = 1 << 30;
        for (int i = 0; i < t; ++i) {
            if (used[i]) continue;
            const int key = pc(u | scope[idx[i]]) * 64 + pc(scope[idx[i]]) + (late && late[idx[i]] >= 0 ? 1 << 16 : 0);
            if (key < bk) { bk = key; best = i; }
        }
        used[best] = true;
        seq[s] = idx[best];
        u |= scope[idx[best]];
    }
    return pc(u);
}

// (The column graph is enough to pick the next column: adj[c] is the joint scope
// of the tables that mention c.  `cap` gives up once the count passes it.)
void simulate(const uint64_t *rowmask, int n, uint64_t L, int max_width, double cap, Sim &S) {
    uint64_t tabs[2 * kNMax], adj[kNMax];
    int nt = 0, scalars = 0;
    double ops = 0.0;
    S.ops = 1e30;
    for (uint64_t x = L; x; x &= x - 1) adj[__builtin_ctzll(x)] = 0;
    for (int i = 0; i < n; ++i) {
        const uint64_t s = rowmask[i] & L;
        if (!s) { ++scalars; continue; }
        const int w = pc(s);
        if (w > max_width) return;
        ops += (double)((1u << w) - 1u);
        tabs[nt++] = s;
        for (uint64_t x = s; x; x &= x - 1) adj[__builtin_ctzll(x)] |= s;
    }
    uint64_t rem = L;
    int done = 0;
    while (rem) {
        int c = -1, bw = 1 << 30;
        for (uint64_t x = rem; x; x &= x - 1) {
            const int j = __builtin_ctzll(x), w = pc(adj[j]);
            if (w < bw) { bw = w; c = j; }
        }
        if (bw > max_width) return;
        const uint64_t b = 1ull << c;
        // the bucket's tables by scope size: multiplied smallest first
        uint64_t bucket[2 * kNMax];
        int t = 0, keep = 0;
        for (int i = 0; i < nt; ++i) {
            if (!(tabs[i] & b)) { tabs[keep++] = tabs[i]; continue; }
            int p = t++;
            for (; p > 0 && pc(bucket[p - 1]) > pc(tabs[i]); --p) bucket[p] = bucket[p - 1];
            bucket[p] = tabs[i];
        }
        nt = keep;
        uint64_t u = bucket[0];
        if (t == 1) ops += 0.5 * (double)(1u << pc(u));
        for (int i = 1; i < t; ++i) {
            u |= bucket[i];
            ops += (double)(1u << pc(u));
        }
        if (ops > cap) return;
        u &= ~b;
        if (u) tabs[nt++] = u; else ++scalars;
        for (uint64_t x = u; x; x &= x - 1) {
            const int j = __builtin_ctzll(x);
            adj[j] = (adj[j] | u) & ~b;
        }
        S.order[done++] = c;
        rem &= ~b;
    }
    S.ops = ops + std::max(0, scalars - 1);
}

// Compresses the bits of `v` selected by `mask` (software pext; n <= 64).
inline uint32_t compress(uint64_t v, uint64_t mask) {
    uint32_t r = 0;
    int k = 0;
    for (; mask; mask &= mask - 1, ++k)
        if (v & (mask & (~mask + 1))) r |= 1u << k;
    return r;
}
inline uint64_t expand(uint32_t e, uint64_t mask) {
    uint64_t r = 0;
    for (int k = 0; mask; mask &= mask - 1, ++k)
        if ((e >> k) & 1u) r |= mask & (~mask + 1);
    return r;
}

struct Table {
    uint64_t scope;
    std::vector<int> v;   // value ids by compressed setting of the scope's columns
};

struct Builder {
    const Matrix &m;
    ElimPlan &E;
    bool exact;
    Builder(const Matrix &mm, ElimPlan &e) : m(mm), E(e), exact(mm.is_int) {
        E.ops.clear();
        E.bound.clear();
        for (int i = 0; i < m.n; ++i) {
            double b = 0.0;
            for (int j = 0; j < m.n; ++j) b += std::fabs(m.fval(i, j));
            E.bound.push_back(std::max(b, 1.0));
        }
    }
    int add(int a, int row, int col) {   // |x_i| stays within the row's absolute sum
        E.ops.push_back({kElimAdd, a, row, col});
        E.bound.push_back(E.bound[row]);
        return (int)E.bound.size() - 1;
    }
    int mul(int a, int b) {
        E.ops.push_back({kElimMul, a, b, 0});
        E.bound.push_back(E.bound[a] * E.bound[b]);
        return (int)E.bound.size() - 1;
    }
    int mulsub(int a, int b, int c) {
        E.ops.push_back({kElimMulSub, a, b, c});
        E.bound.push_back(E.bound[c] + E.bound[a] * E.bound[b]);
        return (int)E.bound.size() - 1;
    }
    int sub(int a, int b) {
        E.ops.push_back({kElimSub, a, b, 0});
        E.bound.push_back(E.bound[a] + E.bound[b]);
        return (int)E.bound.size() - 1;
    }
    // a row's table: x_i plus every subset of its low entries
    Table row_table(int i, uint64_t L) {
        Table t;
        t.scope = m.rowmask[i] & L;
        t.v.assign(1u << pc(t.scope), -1);
        t.v[0] = i;
        for (uint32_t e = 1; e < t.v.size(); ++e) {
            const uint32_t low = e & (~e + 1);
            t.v[e] = add(t.v[e ^ low], i, __builtin_ctzll(expand(low, t.scope)));
        }
        return t;
    }
    void run(uint64_t L, const int *order, int k) {
        // rows wait untouched until the first of their columns is summed out
        struct Item { uint64_t scope; int row; int tab; };
        std::vector<Table> store;
        std::vector<Item> items;
        std::vector<int> scalars;
        for (int i = 0; i < m.n; ++i) {
            const uint64_t s = m.rowmask[i] & L;
            if (s) items.push_back({s, i, -1}); else scalars.push_back(i);
        }
        for (int q = 0; q < k; ++q) {
            const uint64_t b = 1ull << order[q];
            std::vector<uint64_t> sc;
            std::vector<int> idx, seq;
            for (size_t i = 0; i < items.size(); ++i) {
                sc.push_back(items[i].scope);
                if (items[i].scope & b) idx.push_back((int)i);
            }
            if (idx.empty()) continue;   // (a column without rows: no perfect matching; never planned)
            seq.resize(idx.size());
            bucket_order(sc.data(), idx.data(), (int)idx.size(), seq.data());
            auto table = [&](int it) { return items[it].tab >= 0 ? store[items[it].tab] : row_table(items[it].row, L); };
            Table cur = table(seq[0]);
            Table out;
            for (size_t s = 1; s < seq.size(); ++s) {
                const Table t = table(seq[s]);
                Table r;
                r.scope = cur.scope | t.scope;
                if (s + 1 < seq.size()) {
                    r.v.resize(1u << pc(r.scope));
                    for (uint32_t e = 0; e < r.v.size(); ++e) {
                        const uint64_t x = expand(e, r.scope);
                        r.v[e] = mul(cur.v[compress(x, cur.scope)], t.v[compress(x, t.scope)]);
                    }
                    cur = std::move(r);
                } else {   // the last product, fused with the signed sum over column b
                    out.scope = r.scope & ~b;
                    out.v.resize(1u << pc(out.scope));
                    for (uint32_t e = 0; e < out.v.size(); ++e) {
                        const uint64_t x0 = expand(e, out.scope), x1 = x0 | b;
                        const int off = mul(cur.v[compress(x0, cur.scope)], t.v[compress(x0, t.scope)]);
                        out.v[e] = mulsub(cur.v[compress(x1, cur.scope)], t.v[compress(x1, t.scope)], off);
                    }
                }
            }
            if (seq.size() == 1) {
                out.scope = cur.scope & ~b;
                out.v.resize(1u << pc(out.scope));
                for (uint32_t e = 0; e < out.v.size(); ++e) {
                    const uint64_t x0 = expand(e, out.scope), x1 = x0 | b;
                    out.v[e] = sub(cur.v[compress(x0, cur.scope)], cur.v[compress(x1, cur.scope)]);
                }
            }
            std::vector<Item> rest;
            for (const Item &it : items)
                if (!(it.scope & b)) rest.push_back(it);
            if (out.scope) {
                rest.push_back({out.scope, -1, (int)store.size()});
                store.push_back(out);
            } else {
                scalars.push_back(out.v[0]);
            }
            items = rest;
        }
        // the scalars' product (exact: smallest bounds first, so that the
        // factors stay in 32 bits as long as they can)
        if (exact) std::stable_sort(scalars.begin(), scalars.end(), [&](int a, int b) { return E.bound[a] < E.bound[b]; });
        // (FP64: pairwise, so that the last products do not wait on one another)
        if (!exact)
            while (scalars.size() > 2) {
                std::vector<int> half;
                for (size_t i = 0; i + 1 < scalars.size(); i += 2) half.push_back(mul(scalars[i], scalars[i + 1]));
                if (scalars.size() & 1) half.push_back(scalars.back());
                scalars = half;
            }
        int r = scalars[0];
        for (size_t i = 1; i < scalars.size(); ++i) r = mul(r, scalars[i]);
        E.result = r;
    }
};

// The program by tables (scopes in elimination-order bits).
void build_tables(const Matrix &m, ElimPlan &E, const int *order, int k) {
    const int n = m.n;
    E.tables.clear();
    E.tops.clear();
    E.factors.clear();
    E.table_ops = 0.0;
    uint64_t live[kNMax];   // scope of each row by elimination place
    for (int i = 0; i < n; ++i) live[i] = 0;
    for (int q = 0; q < k; ++q)
        for (uint64_t rows = m.colmask[order[q]]; rows; rows &= rows - 1) live[__builtin_ctzll(rows)] |= 1ull << q;
    int item_tab[2 * kNMax], nitems = 0;   // tables (or rows still to be made tables: -1 - row) by scope
    uint64_t item_scope[2 * kNMax];
    for (int i = 0; i < n; ++i) {
        double b = 0.0;
        if (m.is_int)
            for (int j = 0; j < n; ++j) b += std::fabs(m.fval(i, j));
        E.tables.push_back({0, std::max(b, 1.0), i});
        if (live[i]) {
            item_scope[nitems] = live[i];
            item_tab[nitems++] = -1 - i;
        } else {
            E.factors.push_back(i);
        }
    }
    auto make = [&](uint64_t scope, double bound) {
        E.tables.push_back({scope, bound, -1});
        return (int)E.tables.size() - 1;
    };
    for (int q = 0; q < k; ++q) {
        const uint64_t b = 1ull << q;
        int idx[2 * kNMax], seq[2 * kNMax], t = 0;
        for (int i = 0; i < nitems; ++i)
            if (item_scope[i] & b) idx[t++] = i;
        if (!t) continue;
        // FP64: the order with all rows first where that is cheaper, an entry of a
        // product with a summed-out table (a magnitude too) counted as two
        bucket_order(item_scope, idx, t, seq);
        if (!m.is_int) {
            auto cost = [&](const int *order) {
                uint64_t u = item_scope[order[0]];
                bool summed = item_tab[order[0]] >= 0;
                double c = 0.0;
                for (int s = 1; s < t; ++s) {
                    u |= item_scope[order[s]];
                    summed |= item_tab[order[s]] >= 0;
                    c += (double)(1ull << pc(u)) * (summed ? 2.0 : 1.0);
                }
                return c;
            };
            int rows_first[2 * kNMax];
            bucket_order(item_scope, idx, t, rows_first, item_tab);
            if (cost(rows_first) < cost(seq)) std::copy(rows_first, rows_first + t, seq);
        }
        // a row becomes a table just before it is multiplied, and up to three more of
        // the bucket's rows of the same small size with it (one instruction)
        auto make_row = [&](int it) {
            const int row = -1 - item_tab[it];
            item_tab[it] = make(item_scope[it], E.tables[row].bound);
            E.tops.push_back({kTabRow, item_tab[it], row, 0, 0});
            E.table_ops += (double)(1ull << pc(item_scope[it])) - 1.0;
        };
        auto table = [&](int at) {
            const int it = seq[at];
            if (item_tab[it] >= 0) return item_tab[it];
            make_row(it);
            const int w = pc(item_scope[it]);
            for (int s = at + 1, more = 3; s < t && more > 0 && w <= 3; ++s)
                if (item_tab[seq[s]] < 0 && pc(item_scope[seq[s]]) == w) { make_row(seq[s]); --more; }
            return item_tab[it];
        };
        int cur = table(0), out;
        uint64_t scope = item_scope[seq[0]];
        if (t == 1) {
            out = make(scope & ~b, 2.0 * E.tables[cur].bound);
            E.tops.push_back({kTabSub, out, cur, cur, q});
            E.table_ops += (double)(1ull << (pc(scope) - 1));
        } else {
            for (int s = 1; s < t; ++s) {
                const int r = table(s);
                scope |= item_scope[seq[s]];
                const double bound = E.tables[cur].bound * E.tables[r].bound;
                const bool last = s + 1 == t;
                const int d = last ? make(scope & ~b, 2.0 * bound) : make(scope, bound);
                E.tops.push_back({(uint8_t)(last ? kTabSum : kTabMul), d, cur, r, q});
                E.table_ops += (double)(1ull << pc(scope));
                cur = d;
            }
            out = cur;
        }
        int keep = 0;
        for (int i = 0; i < nitems; ++i)
            if (!(item_scope[i] & b)) {
                item_scope[keep] = item_scope[i];
                item_tab[keep++] = item_tab[i];
            }
        nitems = keep;
        const uint64_t left = scope & ~b;
        if (left) {
            item_scope[nitems] = left;
            item_tab[nitems++] = out;
        } else {
            E.factors.push_back(out);
        }
    }
    E.table_ops += (double)E.factors.size() - 1.0;
}

}  // namespace

bool elim_plan(const Matrix &m, const int *col_order, int free_cols, double range_log2, const ElimLimits &lim,
               ElimPlan &E) {
    const int n = m.n;
    if (n < 4) return false;
    uint64_t rows[kNMax];
    for (int i = 0; i < n; ++i) rows[i] = m.rowmask[i];
    const int free_n = std::min(free_cols, n - 1);
    // candidates: the free columns by ascending size
    int cand[kNMax], nc = 0;
    for (int p = 0; p < free_n; ++p) cand[nc++] = col_order[p];
    insertion_sort(cand, cand + nc, [&](int a, int b) { return pc(m.colmask[a]) < pc(m.colmask[b]); });
    // Greedy growth of the low set: the column that lowers the modelled time
    // most.  time = (program + the outer flips' updates + loop) x outer steps,
    // where fewer steps than fill the GPU take as long as those.
    uint64_t L = 0;
    int k = 0;
    double best_time = 1e300;
    Sim best, S;
    best.ops = n - 1;
    auto model = [&](double ops, int kk, uint64_t LL) {
        double flip = 0.0;
        int got = 0;
        for (int i = 0; i < nc && got < 2; ++i)
            if (!((LL >> cand[i]) & 1ull)) { flip += pc(m.colmask[cand[i]]) * 0.75; ++got; }
        return (ops + flip + 8.0) * std::max(std::exp2(range_log2 - kk), lim.full_blocks);
    };
    if (lim.allow_none) best_time = model(n - 1, 0, 0);
    for (;;) {
        int pick = -1;
        Sim pick_sim;
        double pick_time = best_time;
        int tried = 0;
        for (int i = 0; i < nc && tried < lim.candidates; ++i) {
            const int c = cand[i];
            if ((L >> c) & 1ull) continue;
            ++tried;
            if (range_log2 - (k + 1) < 0.0) continue;
            simulate(rows, n, L | (1ull << c), lim.max_width, lim.max_ops, S);
            if (S.ops > lim.max_ops) continue;
            const double t = model(S.ops, k + 1, L | (1ull << c));
            if (t < pick_time) { pick_time = t; pick = c; pick_sim = S; }
        }
        if (pick < 0) break;
        best_time = pick_time;
        best = pick_sim;
        L |= 1ull << pick;
        ++k;
    }
    if (k < 1 && !lim.allow_none) return false;
    E.n = n;
    E.k = k;
    E.h = n - 1 - k;
    for (int i = 0; i < k; ++i) E.low[i] = best.order[i];
    // outer columns: the free ones by ascending size (the most frequent flips
    // touch the fewest rows), then the others at their own Gray positions
    int h = 0;
    for (int i = 0; i < nc; ++i)
        if (!((L >> cand[i]) & 1ull)) E.outer[h++] = cand[i];
    for (int p = free_n; p < n - 1; ++p) E.outer[h++] = col_order[p];
    E.last = col_order[n - 1];
    E.scale = 0;
    for (int i = 0; i < n; ++i) {
        E.exp2[i] = 0;
        if (m.is_int) continue;
        double rs = 0.0;
        for (int j = 0; j < n; ++j) rs += std::fabs(m.fval(i, j));
        if (!(rs > 0.0) || !std::isfinite(rs)) return false;
        std::frexp(rs / 2.0, &E.exp2[i]);
        E.exp2[i] -= elim_row_bits(n, k, i);
        E.scale += E.exp2[i];
    }
    double count;
    if (lim.tables_only) {
        build_tables(m, E, E.low, k);
        count = E.table_ops;
    } else {
        Builder(m, E).run(L, E.low, k);
        count = (double)E.ops.size();
    }
    double flips = 0.0;
    for (int p = 0; p < h; ++p) flips += pc(m.colmask[E.outer[p]]) * std::ldexp(1.0, -(p + 1));
    E.ops_per_step = std::ldexp(count + flips + 1.0, -k);
    return true;
}

bool elim_magnitudes_hold(const Matrix &m, const ElimPlan &E, const int *col_order, int free_cols, uint64_t g_lo,
                          uint64_t g_hi) {
    const int n = m.n;
    free_cols = std::min(free_cols, n - 1);
    // Scaled rows: |x_i| <= 2^b_i, and a nonzero x_i is at least one unit of the last
    // place of the row's finest entry, 2^g_i.
    int g[kNMax], bmin = 1 << 20;
    double x0[kNMax];
    for (int i = 0; i < n; ++i) {
        bmin = std::min(bmin, elim_row_bits(n, E.k, i));
        g[i] = 1 << 20;
        double rs = 0.0;
        for (uint64_t c = m.rowmask[i]; c; c &= c - 1) {
            const double v = m.fval(i, __builtin_ctzll(c));
            int e;
            const int64_t bits = (int64_t)std::ldexp(std::frexp(std::fabs(v), &e), 53);
            g[i] = std::min(g[i], e - 53 + __builtin_ctzll((uint64_t)bits) - 1 - E.exp2[i]);
            rs += v;
        }
        x0[i] = m.fval(i, E.last) - rs / 2.0;
    }
    // the fewest rows whose product may be below FP32's normal numbers
    insertion_sort(g, g + n, [](int a, int b) { return a < b; });
    int rows = 0;
    for (int sum = 0; sum >= -126; sum += g[rows++])
        if (rows == n) return true;
    // Each of a step's at most 2^7 tables may lose 2^-150 an entry (a single value
    // 2^-126: it is cut off there), times the largest magnitudes of the rows that are
    // still to come and the settings of the low columns: 2^(120 - rows bmin) at most.
    // The mean step's sum of magnitudes has to be 2^20 times that.
    const double need = 20.0 + 7.0 + (rows == 1 ? -126.0 : -150.0) + 120.0 - rows * bmin;
    // It is at least one term of the range over the number of its steps.  The free
    // columns take every setting: none and all of them (the largest terms of matrices
    // without negative entries), then each improved column by column.
    const double floor_log2 = E.k - std::log2((double)(g_hi - g_lo));
    double x[kNMax];
    auto fill = [&](uint64_t set) {
        for (int i = 0; i < n; ++i) {
            x[i] = x0[i];
            for (uint64_t c = m.rowmask[i] & set; c; c &= c - 1) x[i] += m.fval(i, __builtin_ctzll(c));
        }
    };
    auto term_log2 = [&] {
        double mant = 1.0;
        int exp = 0;
        for (int i = 0; i < n && mant != 0.0; ++i) {
            int e;
            mant = std::frexp(mant * std::fabs(std::ldexp(x[i], -E.exp2[i])), &e);
            exp += e;
        }
        return mant == 0.0 ? -1e300 : exp + std::log2(mant);
    };
    auto columns = [&](uint64_t q) {   // the columns set at Gray index q
        uint64_t set = 0;
        for (uint64_t u = q ^ (q >> 1); u; u &= u - 1) set |= 1ull << col_order[__builtin_ctzll(u)];
        return set;
    };
    uint64_t free = 0;
    for (int p = 0; p < free_cols; ++p) free |= 1ull << col_order[p];
    const uint64_t start[2] = {columns(g_lo) & ~free, columns(g_lo) | free};
    for (int improve = 0; improve < 2; ++improve)
        for (uint64_t set : start) {
            fill(set);
            for (uint64_t left = improve ? free : 0; left; left &= left - 1) {
                const int j = __builtin_ctzll(left);
                const double sign = (set >> j) & 1ull ? -1.0 : 1.0;
                double now = 1.0, then = 1.0;   // (factors from 2^-20: zeros are left where they can be)
                for (uint64_t r = m.colmask[j]; r; r &= r - 1) {
                    const int i = __builtin_ctzll(r);
                    now *= std::max(std::fabs(std::ldexp(x[i], -E.exp2[i])), 0x1p-20);
                    then *= std::max(std::fabs(std::ldexp(x[i] + sign * m.fval(i, j), -E.exp2[i])), 0x1p-20);
                }
                if (then <= now) continue;
                set ^= 1ull << j;
                for (uint64_t r = m.colmask[j]; r; r &= r - 1) x[__builtin_ctzll(r)] += sign * m.fval(__builtin_ctzll(r), j);
            }
            if (term_log2() + floor_log2 >= need) return true;
        }
    // Last, the mean of sampled |terms|, from below: the largest over the number of samples.
    uint64_t seed = 0x9e3779b97f4a7c15ull;
    double top = -1e300;
    int draws = 0;
    for (int terms = 0; terms < 8 && draws < 1024; ++draws) {
        seed += 0x9e3779b97f4a7c15ull;   // splitmix64
        uint64_t z = seed;
        z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
        z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
        fill(columns(g_lo + (z ^ (z >> 31)) % (g_hi - g_lo)));
        const double t = term_log2();
        if (t > -1e300) ++terms;
        top = std::max(top, t);
    }
    return top - std::log2((double)draws) + E.k >= need;
}

// ------------------------------------------------------------------ generated kernel

namespace {

std::string dlit(double v) {
    char buf[64];
    std::snprintf(buf, sizeof buf, "%a", v);
    return v < 0 || std::signbit(v) ? "(" + std::string(buf) + ")" : std::string(buf);
}
std::string ilit(int64_t v) { return v < 0 ? "(" + std::to_string(v) + ")" : std::to_string(v); }

}  // namespace

std::string elim_source(const Matrix &m, const ElimPlan &E, int limbs, bool want_abs) {
    const int n = E.n;
    const bool fp = limbs == 0;
    want_abs = want_abs && fp;
    std::ostringstream o;
    o << "// generated: eliminated permanent walk for one " << n << "x" << n << " matrix\n";
    o << "// low columns k=" << E.k << " outer columns h=" << E.h << " operations per outer step " << E.ops.size() << "\n";
    o << "#include \"core.cuh\"\n#ifndef PERM_HOST_EMULATION\n#include \"finish.cuh\"\n#endif\n\nnamespace pk {\n";
    if (fp) o << "typedef ArithF64 A;\n";
    else o << "typedef ArithExact<" << limbs << "> A;\n";
    o << "struct ElimPol {\n    static constexpr int NX = " << n << ";\n";
    o << "    static constexpr bool kAbs = " << (want_abs ? "true" : "false") << ";\n";
    o << "    static constexpr int scale = " << E.scale << ";   // the walk's sums are the true ones times 2^-scale\n";
    o << "    typedef A::X X;\n";
    auto entry = [&](int r, int c) {
        return fp ? dlit(std::ldexp(m.fval(r, c), -E.exp2[r])) : ilit(2 * m.ival(r, c));
    };
    o << "    static __device__ __forceinline__ void flip_dyn(int j, X (&x)[NX], int s) {\n        switch (j) {\n";
    for (int p = 0; p < E.h; ++p) {
        o << "        case " << p << ":\n";
        for (int i = 0; i < n; ++i)
            if (m.nz(i, E.outer[p]))
                o << "            x[" << i << "] = A::upd_rt(x[" << i << "], " << entry(i, E.outer[p]) << ", s);\n";
        o << "            break;\n";
    }
    o << "        default: break;\n        }\n    }\n";
    // the start vector: the lanes' outer columns added with weight 0 or 1
    o << "    static __device__ __forceinline__ void init_x(X (&x)[NX], u64 G) {\n";
    for (int i = 0; i < n; ++i) {
        if (fp) {
            double rowsum = 0.0;
            for (int j = 0; j < n; ++j) rowsum += m.fval(i, j);
            o << "        x[" << i << "] = " << dlit(std::ldexp(m.fval(i, E.last) - rowsum / 2.0, -E.exp2[i])) << ";\n";
        } else {
            int64_t rowsum = 0;
            for (int j = 0; j < n; ++j) rowsum += m.ival(i, j);
            o << "        x[" << i << "] = " << ilit(2 * m.ival(i, E.last) - rowsum) << ";\n";
        }
    }
    o << "        u64 U = warp_or64(G);\n        while (U) {\n            const int p = ctz64(U);\n            U &= U - 1;\n";
    o << "            flip_dyn(p, x, (int)((G >> p) & 1ull));\n        }\n    }\n";
    // the step: exact values take the narrowest type their bound allows
    auto type_of = [&](int v) {   // 0: int, 1: 64 bits, 2: the ring
        if (E.bound[v] < 2147483647.0) return 0;
        return limbs == 2 || E.bound[v] < 9.2e18 ? 1 : 2;
    };
    auto name = [&](int v) { return v < n ? "x[" + std::to_string(v) + "]" : "v" + std::to_string(v); };
    static const char *const tn[3] = {"int", "i64", "Ring<A::L>"};
    o << "    static __device__ __forceinline__ void step(const X (&x)[NX], A::Blk &blk, bool odd) {\n";
    if (want_abs)
        for (int i = 0; i < n; ++i) o << "        const float f" << i << " = abs_f32_full(x[" << i << "]);\n";
    for (size_t q = 0; q < E.ops.size(); ++q) {
        const ElimOp &op = E.ops[q];
        const int v = n + (int)q;
        if (fp) {
            o << "        const double v" << v << " = ";
            switch (op.kind) {
            case kElimAdd: o << name(op.a) << " + " << entry(op.b, op.c); break;
            case kElimMul: o << name(op.a) << " * " << name(op.b); break;
            case kElimMulSub: o << "fma(-" << name(op.a) << ", " << name(op.b) << ", " << name(op.c) << ")"; break;
            default: o << name(op.a) << " - " << name(op.b); break;
            }
            o << ";\n";
            if (!want_abs) continue;
            o << "        const float f" << v << " = ";
            switch (op.kind) {
            case kElimAdd: o << "abs_f32_full(v" << v << ")"; break;
            case kElimMul: o << "f" << op.a << " * f" << op.b; break;
            case kElimMulSub: o << "f" << op.a << " * f" << op.b << " + f" << op.c; break;
            default: o << "f" << op.a << " + f" << op.b; break;
            }
            o << ";\n";
        } else {
            const int t = type_of(v);
            o << "        const " << tn[t] << " v" << v << " = ";
            auto mul = [&](int a, int b) -> std::string {
                int ta = type_of(a), tb = type_of(b);
                std::string na = name(a), nb = name(b);
                if (ta < tb) { std::swap(ta, tb); std::swap(na, nb); }
                if (t == 0) return na + " * " + nb;
                if (t == 1) return "(i64)((u64)(i64)" + na + " * (u64)(i64)" + nb + ")";   // wraps modulo 2^64
                if (ta < 2) na = "ring_of<A::L>((i64)" + na + ")";
                return "ring_times(" + na + ", " + nb + ")";
            };
            auto as = [&](int a) -> std::string {
                const int ta = type_of(a);
                if (t == 0) return name(a);
                if (t == 1) return "(u64)(i64)" + name(a);
                return ta == 2 ? name(a) : "ring_of<A::L>((i64)" + name(a) + ")";
            };
            auto minus = [&](const std::string &a, const std::string &b) -> std::string {
                if (t == 0) return a + " - " + b;
                if (t == 1) return "(i64)(" + a + " - (u64)" + b + ")";
                return "ring_minus(" + a + ", " + b + ")";
            };
            switch (op.kind) {
            case kElimAdd: o << name(op.a) << " + " << entry(op.b, op.c); break;
            case kElimMul: o << mul(op.a, op.b); break;
            case kElimMulSub: o << minus(as(op.c), mul(op.a, op.b)); break;
            default: o << minus(as(op.a), as(op.b)); break;
            }
            o << ";\n";
        }
    }
    const int r = E.result;
    if (fp) {
        o << "        if (odd) A::blk_add<-1>(blk, " << name(r) << "); else A::blk_add<1>(blk, " << name(r) << ");\n";
        if (want_abs) o << "        A::blk_abs_f(blk, f" << r << ");\n";
    } else {
        o << "        const Ring<A::L> t = " << (type_of(r) == 2 ? name(r) : "ring_of<A::L>((i64)" + name(r) + ")") << ";\n";
        o << "        if (odd) A::blk_add<-1>(blk, t); else A::blk_add<1>(blk, t);\n";
    }
    o << "    }\n";
    o << "};\n}  // namespace pk\n\n";
    // One block per SM (255 registers): FP64 steps are bound by the FP64 pipe (2
    // lane-operations per clock and SM), which eight warps keep 85 % busy (ncu).
    o << "extern \"C\" __global__ void __launch_bounds__(256, 1) perm_walk(pk::WalkArgs wa, void *) {\n";
    o << "    pk::elim_tasks<pk::ElimPol, pk::A>(wa);\n";
    o << "#ifndef PERM_HOST_EMULATION\n    pk::finish_walk<pk::A>(wa.finish);\n#endif\n}\n";
    return o.str();
}

}  // namespace perm
