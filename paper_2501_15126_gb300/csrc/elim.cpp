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
    int width = 0;
    int order[kNMax];
};

// The order in which the tables of a bucket are multiplied: smallest scope
// first, then always the table that grows the joint scope least.
int bucket_order(const uint64_t *scope, const int *idx, int t, int *seq) {
    bool used[2 * kNMax] = {};
    uint64_t u = 0;
    for (int s = 0; s < t; ++s) {
        int best = -1, bk = 1 << 30;
        for (int i = 0; i < t; ++i) {
            if (used[i]) continue;
            const int key = pc(u | scope[idx[i]]) * 64 + pc(scope[idx[i]]);
            if (key < bk) { bk = key; best = i; }
        }
        used[best] = true;
        seq[s] = idx[best];
        u |= scope[idx[best]];
    }
    return pc(u);
}

void simulate(const uint64_t *rowmask, int n, uint64_t L, int max_width, Sim &S) {
    uint64_t tabs[2 * kNMax];
    int nt = 0, scalars = 0;
    S.ops = 0.0;
    S.width = 0;
    for (int i = 0; i < n; ++i) {
        const uint64_t s = rowmask[i] & L;
        if (!s) { ++scalars; continue; }
        S.ops += (double)(1ull << pc(s)) - 1.0;
        tabs[nt++] = s;
        S.width = std::max(S.width, pc(s));
    }
    if (S.width > max_width) { S.ops = 1e30; return; }
    uint64_t rem = L;
    int done = 0;
    while (rem) {
        int bw = 1 << 30;
        uint64_t bb = 0;
        for (uint64_t x = rem; x; x &= x - 1) {
            const uint64_t b = x & (~x + 1);
            uint64_t u = 0;
            int cnt = 0;
            for (int t = 0; t < nt; ++t)
                if (tabs[t] & b) { u |= tabs[t]; ++cnt; }
            const int key = pc(u) * 256 + cnt;
            if (key < bw) { bw = key; bb = b; }
        }
        int idx[2 * kNMax], seq[2 * kNMax], t = 0;
        for (int i = 0; i < nt; ++i)
            if (tabs[i] & bb) idx[t++] = i;
        const int w = bucket_order(tabs, idx, t, seq);
        S.width = std::max(S.width, w);
        if (w > max_width) { S.ops = 1e30; return; }
        uint64_t u = tabs[seq[0]];
        if (t == 1) S.ops += std::ldexp(1.0, pc(u) - 1);
        for (int i = 1; i < t; ++i) {
            u |= tabs[seq[i]];
            S.ops += std::ldexp(1.0, pc(u));
        }
        int keep = 0;
        for (int i = 0; i < nt; ++i)
            if (!(tabs[i] & bb)) tabs[keep++] = tabs[i];
        nt = keep;
        u &= ~bb;
        if (u) tabs[nt++] = u; else ++scalars;
        S.order[done++] = __builtin_ctzll(bb);
        rem &= ~bb;
    }
    S.ops += std::max(0, scalars - 1);
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
        int r = scalars[0];
        for (size_t i = 1; i < scalars.size(); ++i) r = mul(r, scalars[i]);
        E.result = r;
    }
};

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
    std::stable_sort(cand, cand + nc, [&](int a, int b) { return pc(m.colmask[a]) < pc(m.colmask[b]); });
    // Greedy growth of the low set: the column that lowers the modelled time
    // most.  time = (program + the outer flips' updates + loop) x outer steps,
    // where fewer steps than fill the GPU take as long as those.
    uint64_t L = 0;
    int k = 0;
    double best_time = 1e300;
    Sim best, S;
    auto model = [&](double ops, int kk, uint64_t LL) {
        double flip = 0.0;
        int got = 0;
        for (int i = 0; i < nc && got < 2; ++i)
            if (!((LL >> cand[i]) & 1ull)) { flip += pc(m.colmask[cand[i]]) * 0.75; ++got; }
        return (ops + flip + 8.0) * std::max(std::exp2(range_log2 - kk), lim.full_blocks);
    };
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
            simulate(rows, n, L | (1ull << c), lim.max_width, S);
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
    if (k < 1) return false;
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
        E.scale += E.exp2[i];
    }
    Builder(m, E).run(L, E.low, k);
    double flips = 0.0;
    for (int p = 0; p < h; ++p) flips += pc(m.colmask[E.outer[p]]) * std::ldexp(1.0, -(p + 1));
    E.ops_per_step = std::ldexp((double)E.ops.size() + flips + 1.0, -k);
    return true;
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
    o << "#include \"core.cuh\"\n\nnamespace pk {\n";
    if (fp) o << "typedef ArithF64 A;\n";
    else o << "typedef ArithExact<" << limbs << "> A;\n";
    o << "struct ElimPol {\n    static constexpr int NX = " << n << ";\n";
    o << "    static constexpr bool kAbs = " << (want_abs ? "true" : "false") << ";\n";
    o << "    // the walk's sum is the true one times 2^-scale, its sum of |terms| times 2^-abs_shift\n";
    o << "    static constexpr int scale = " << E.scale << ";\n";
    o << "    static constexpr int abs_shift = " << E.scale - (fp ? n * elim_abs_bits(n, E.k) : 0) << ";\n";
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
        for (int i = 0; i < n; ++i) o << "        const float f" << i << " = abs_scaled_f32(x[" << i << "], kAbsRow);\n";
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
            case kElimAdd: o << "abs_scaled_f32(v" << v << ", kAbsRow)"; break;
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
    if (want_abs) o << "    static constexpr int kAbsRow = " << -elim_abs_bits(n, E.k) << ";\n";
    o << "};\n}  // namespace pk\n\n";
    // One block per SM (255 registers): FP64 steps are bound by the FP64 pipe (2
    // lane-operations per clock and SM), which eight warps fill, and the tables
    // of a 2^5-entry elimination need the registers (the n=36 workload: 398
    // operations per step, 202 registers, no spills, 2^21 steps in 2.7 ms).
    o << "extern \"C\" __global__ void __launch_bounds__(256, 1) perm_walk(pk::WalkArgs wa, void *) {\n";
    o << "    pk::elim_tasks<pk::ElimPol, pk::A>(wa);\n}\n";
    return o.str();
}

}  // namespace perm
