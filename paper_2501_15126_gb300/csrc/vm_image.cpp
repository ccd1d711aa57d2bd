// vm_image.cpp -- program images of the eliminated walk (vm.h).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "plan.hpp"
#include "vm.hpp"

namespace perm {

namespace {

size_t up16(size_t v) { return (v + 15) & ~(size_t)15; }

// Consecutive slots for tables, first fit.
struct SlotRanges {
    std::pmr::vector<char> used;
    explicit SlotRanges(std::pmr::memory_resource *mem) : used(mem) {}
    int top = 0;
    int take(int count) {
        int run = 0;
        for (int s = 0;; ++s) {
            if (s >= (int)used.size()) used.push_back(0);
            run = used[s] ? 0 : run + 1;
            if (run == count) {
                const int b = s + 1 - count;
                for (int i = b; i <= s; ++i) used[i] = 1;
                top = std::max(top, s + 1);
                return b;
            }
        }
    }
    void give(int b, int count) {
        for (int i = b; i < b + count; ++i) used[i] = 0;
    }
};

}  // namespace

size_t vm_slot_area(int img, int limbs, int nslots, int nextra) {
    // FP64: a double per slot and lane, FP32 magnitudes in slots of their own;
    // double-double: pairs; exact: 64 bits, and the ring's 64-bit words
    const size_t lane = img == kImgDD ? 16 : 8, extra = img == kImgInt ? 8 * (size_t)((limbs + 1) / 2) : 4;
    return 32 * (lane * (size_t)nslots + extra * (size_t)nextra);
}

bool vm_image(const Matrix &m, const ElimPlan &E, int img, int limbs, int max_slots, std::pmr::vector<unsigned char> &out) {
    // working vectors in one block from where the image is (threads of small stacks call this)
    std::pmr::monotonic_buffer_resource local(48 * 1024, out.get_allocator().resource());
    std::pmr::memory_resource *mem = &local;
    const int n = m.n;
    const bool exact = img == kImgInt;
    const int ntab = (int)E.tables.size();
    const std::pmr::vector<ElimTableOp> &tops = E.tops;
    // literals: the entries that the program and the flips add; literal 0 pads
    std::pmr::vector<short> lit_of((size_t)n * n, -1, mem);
    std::pmr::vector<std::pair<int, int>> lits(1, {-1, -1}, mem);
    auto lit = [&](int r, int c) -> int {
        short &l = lit_of[(size_t)r * n + c];
        if (l >= 0) return l;
        lits.push_back({r, c});
        return l = (short)(lits.size() - 1);
    };
    // ring tables: 64-bit slots hold what their bound allows (everything, modulo 2^64, in a 64-bit ring)
    auto is_ring = [&](int t) { return exact && limbs > 2 && !(E.tables[t].bound < 9.2e18); };
    auto size_of = [&](int t) { return 1 << __builtin_popcountll(E.tables[t].scope); };
    std::pmr::vector<int> last(ntab, -1, mem), slot(ntab, -1, mem);
    for (int q = 0; q < (int)tops.size(); ++q) {
        if (tops[q].kind != kTabRow) last[tops[q].a] = last[tops[q].b] = q;
    }
    const int end = (int)tops.size();
    for (int f : E.factors) last[f] = end;
    // `extra` holds ring tables (exact) or the magnitudes of tables in which a
    // column has been summed out (FP64)
    SlotRanges plain(mem), extra(mem);
    plain.used.assign(n + 1, 1);   // x, padding
    plain.top = n + 1;
    std::pmr::vector<int> mag(ntab, -1, mem);
    std::pmr::vector<char> summed(ntab, 0, mem);
    if (!exact)
        for (const ElimTableOp &op : tops)
            summed[op.dst] = op.kind == kTabSum || op.kind == kTabSub || (op.kind == kTabMul && (summed[op.a] || summed[op.b]));
    for (int i = 0; i < n; ++i) slot[i] = i;
    // A bucket's running product keeps one range from its first row on: the range
    // is as large as the product will become, new columns take the upper index
    // bits, and the walk multiplies blocks of entries from the top down, so that
    // every product overwrites its own operand last.
    struct Bits { int count = 0, at[pk::kVmBits] = {}; };
    std::pmr::vector<int> room(ntab, 0, mem);
    std::pmr::vector<Bits> bits(ntab, Bits(), mem);   // a table's columns (elimination places) by index bit
    auto has = [](const Bits &b, int col) { return std::find(b.at, b.at + b.count, col) != b.at + b.count; };
    auto grown = [&](int t) {
        int size = size_of(t);
        for (int u = t; last[u] >= 0 && last[u] < end;) {
            const ElimTableOp &op = tops[last[u]];
            if (op.kind != kTabMul || op.a != u || op.b == u || is_ring(op.dst) != is_ring(t)) break;
            u = op.dst;
            size = size_of(u);
        }
        return size;
    };
    auto take = [&](int t, int size) {
        room[t] = size;
        slot[t] = (is_ring(t) ? extra : plain).take(size);
    };
    auto own_bits = [&](int t) {
        for (uint64_t x = E.tables[t].scope; x; x &= x - 1) bits[t].at[bits[t].count++] = __builtin_ctzll(x);
    };
    auto take_mag = [&](int t) {
        if (summed[t]) mag[t] = extra.take(size_of(t));
    };
    auto give = [&](int t, int q, bool keep_slot) {
        if (t < n || last[t] != q) return;
        if (!keep_slot) (is_ring(t) ? extra : plain).give(slot[t], room[t]);
        if (summed[t]) extra.give(mag[t], size_of(t));
    };
    auto ref = [&](int t) { return (unsigned short)(is_ring(t) ? slot[t] | (int)pk::kVmRingSlot : slot[t]); };
    auto mref = [&](int t) { return (unsigned short)(mag[t] >= 0 ? mag[t] : (int)pk::kVmNoMag); };
    // the stride of column place q in table t, and operand t's strides over the
    // result's index bits
    auto step = [&](int t, int q, int unit) {
        for (int k = 0; k < bits[t].count; ++k)
            if (bits[t].at[k] == q) return (unsigned short)(unit << k);
        return (unsigned short)0;
    };
    auto strides = [&](int t, int dst, int unit, unsigned short *s) {
        for (int k = 0; k < bits[dst].count; ++k) s[k] = step(t, bits[dst].at[k], unit);
    };
    const int slot_bytes = img == kImgDD ? 512 : 256;
    std::pmr::vector<pk::VmIns> prog(mem);
    prog.reserve(tops.size() + 4);
    for (int q = 0; q < end; ++q) {
        const ElimTableOp &op = tops[q];
        pk::VmIns I;
        std::memset(&I, 0, sizeof I);
        const uint64_t scope = E.tables[op.dst].scope;
        const int w = __builtin_popcountll(scope);
        if (w > pk::kVmBits) return false;
        I.w = (unsigned char)w;
        if (op.kind == kTabRow) {
            take(op.dst, grown(op.dst));
            own_bits(op.dst);
            if (w > pk::kVmRowBits) {
                I.kind = pk::kVmBigRow;
                I.dst = (unsigned short)slot[op.dst];
                I.big.x = (unsigned short)op.a;
                int k = 0;
                for (uint64_t x = scope; x; x &= x - 1)
                    I.big.lit[k++] = (unsigned short)lit(op.a, E.low[__builtin_ctzll(x)]);
                prog.push_back(I);
                continue;
            }
            const bool join = q > 0 && tops[q - 1].kind == kTabRow && !prog.empty() && prog.back().kind == pk::kVmRow &&
                              prog.back().w == w && prog.back().dst < pk::kVmRowsMost;
            if (!join) {
                I.kind = pk::kVmRow;
                prog.push_back(I);
            }
            pk::VmIns &R = prog.back();
            auto &row = R.row[R.dst++];
            row.dst = (unsigned short)slot[op.dst];
            row.x = (unsigned short)op.a;
            int k = 0;
            for (uint64_t x = scope; x; x &= x - 1) row.lit[k++] = (unsigned short)lit(op.a, E.low[__builtin_ctzll(x)]);
            continue;
        }
        const bool in_place = op.kind == kTabMul && op.a >= n && last[op.a] == q && op.a != op.b &&
                              is_ring(op.a) == is_ring(op.dst) && room[op.a] >= size_of(op.dst);
        if (op.kind == kTabMul) {   // A's columns first: what is left of the index is new
            Bits &d = bits[op.dst] = bits[op.a];
            for (int k = 0; k < bits[op.b].count; ++k)
                if (!has(d, bits[op.b].at[k])) d.at[d.count++] = bits[op.b].at[k];
        } else {
            own_bits(op.dst);
        }
        if (in_place) {
            slot[op.dst] = slot[op.a];
            room[op.dst] = room[op.a];
        } else {
            take(op.dst, op.kind == kTabMul ? grown(op.dst) : size_of(op.dst));
        }
        take_mag(op.dst);
        I.kind = (unsigned char)(op.kind == kTabSum   ? pk::kVmSum
                                 : op.kind == kTabSub ? pk::kVmSub
                                 : summed[op.dst]     ? pk::kVmMulF
                                                      : pk::kVmMul);
        I.dst = ref(op.dst);
        I.t.a = ref(op.a);
        I.t.b = ref(op.b);
        I.t.fdst = mref(op.dst);
        I.t.fa = mref(op.a);
        I.t.fb = mref(op.b);
        const int unit = is_ring(op.dst) ? 1 : slot_bytes;
        strides(op.a, op.dst, unit, I.t.sa);
        strides(op.b, op.dst, unit, I.t.sb);
        I.t.ea = step(op.a, op.col, unit);
        I.t.eb = step(op.b, op.col, unit);
        give(op.a, q, in_place);
        if (op.b != op.a) give(op.b, q, false);
        prog.push_back(I);
    }
    // the step's sum: the product of the single factors, the exact ones that fit
    // 64 bits first (by bound, in runs whose product still fits), ring ones one by one
    std::pmr::vector<int> plain_f(mem), ring_f(mem);
    for (int f : E.factors) (is_ring(f) ? ring_f : plain_f).push_back(f);
    if (exact)
        insertion_sort(plain_f.begin(), plain_f.end(), [&](int a, int b) { return E.tables[a].bound < E.tables[b].bound; });
    const bool narrow = exact && limbs > 2;
    bool any = false;
    unsigned short acc = 0, facc = (unsigned short)pk::kVmNoMag;
    double acc_bound = 1.0;
    for (size_t at = 0; at < plain_f.size();) {
        pk::VmIns I;
        std::memset(&I, 0, sizeof I);
        I.kind = pk::kVmProd;
        int c = 0;
        double bound = 1.0;
        if (any && (!narrow || (!(acc & pk::kVmRingSlot) && acc_bound * E.tables[plain_f[at]].bound < 9.2e18))) {
            I.prod.f[c].slot = acc;   // the running product leads the next run
            I.prod.f[c++].fslot = facc;
            bound = acc_bound;
            any = false;
        }
        while (at < plain_f.size() && c < pk::kVmProdMost) {
            const int f = plain_f[at];
            if (narrow && c && !(bound * E.tables[f].bound < 9.2e18)) break;
            bound *= E.tables[f].bound;
            I.prod.f[c].slot = (unsigned short)slot[f];
            I.prod.f[c++].fslot = mref(f);
            ++at;
        }
        I.w = (unsigned char)c;
        unsigned short d, fd = (unsigned short)pk::kVmNoMag;
        if (c == 1) {
            d = I.prod.f[0].slot;
            fd = I.prod.f[0].fslot;
        } else {
            d = (unsigned short)plain.take(1);
            if (!exact) fd = (unsigned short)extra.take(1);
            I.dst = d;
            I.prod.fdst = fd;
            prog.push_back(I);
        }
        if (any) {   // (ring walks) the running product times this run's
            pk::VmIns M;
            std::memset(&M, 0, sizeof M);
            M.kind = pk::kVmMul;
            M.t.a = acc;
            M.t.b = d;
            d = (unsigned short)(extra.take(1) | (int)pk::kVmRingSlot);
            M.dst = d;
            prog.push_back(M);
            bound *= acc_bound;
        }
        acc = d;
        facc = fd;
        acc_bound = bound;
        any = true;
    }
    for (int f : ring_f) {
        if (!any) { acc = ref(f); any = true; continue; }
        pk::VmIns M;
        std::memset(&M, 0, sizeof M);
        M.kind = pk::kVmMul;
        M.t.a = ref(f);
        M.t.b = acc;
        acc = (unsigned short)(extra.take(1) | (int)pk::kVmRingSlot);
        M.dst = acc;
        prog.push_back(M);
    }
    if (plain.top + extra.top > max_slots) return false;

    std::pmr::vector<unsigned short> flipptr(E.h + 1, 0, mem), flip(mem);   // bundles of four (slot, literal) pairs
    for (int p = 0; p < E.h; ++p) {
        flipptr[p] = (unsigned short)(flip.size() / 8);
        int cnt = 0;
        for (uint64_t rows = m.colmask[E.outer[p]]; rows; rows &= rows - 1, ++cnt) {
            const int r = __builtin_ctzll(rows);
            flip.push_back((unsigned short)r);
            flip.push_back((unsigned short)lit(r, E.outer[p]));
        }
        for (; cnt % 4; ++cnt) {
            flip.push_back((unsigned short)n);
            flip.push_back(0);
        }
    }
    flipptr[E.h] = (unsigned short)(flip.size() / 8);

    const size_t vsz = exact ? 4 : 8, x0sz = img == kImgDD ? 16 : vsz;
    pk::VmHeader H;
    std::memset(&H, 0, sizeof H);
    H.n = n;
    H.h = E.h;
    H.nslots = plain.top;
    H.nextra = extra.top;
    H.nins = (int)prog.size();
    H.result = acc;
    H.fresult = facc;
    size_t off = sizeof H;
    H.off_x0 = (int)off;
    off = up16(off + x0sz * n);
    H.off_lit = (int)off;
    off = up16(off + vsz * lits.size());
    H.off_flipptr = (int)off;
    off = up16(off + 2 * flipptr.size());
    H.off_flip = (int)off;
    off = up16(off + 2 * flip.size());
    H.off_prog = (int)off;
    off = up16(off + sizeof(pk::VmIns) * prog.size());
    H.off_base = (int)off;
    off = up16(off + x0sz * n);
    H.bytes = (int)off;
    out.assign(off, 0);
    unsigned char *base = out.data();
    std::memcpy(base, &H, sizeof H);
    for (int i = 0; i < n; ++i) {
        unsigned char *d = base + H.off_x0 + x0sz * i;
        if (exact) {
            int64_t rs = 0;
            for (int j = 0; j < n; ++j) rs += m.ival(i, j);
            const int v = (int)(2 * m.ival(i, E.last) - rs);
            std::memcpy(d, &v, 4);
        } else if (img == kImgDD) {
            double v[2];
            x0_dd(m, i, E.last, &v[0], &v[1]);
            v[0] = std::ldexp(v[0], -E.exp2[i]);
            v[1] = std::ldexp(v[1], -E.exp2[i]);
            std::memcpy(d, v, 16);
        } else {
            double rs = 0.0;
            for (int j = 0; j < n; ++j) rs += m.fval(i, j);
            const double v = std::ldexp(m.fval(i, E.last) - rs / 2.0, -E.exp2[i]);
            std::memcpy(d, &v, 8);
        }
    }
    for (size_t l = 1; l < lits.size(); ++l) {
        const int r = lits[l].first, c = lits[l].second;
        unsigned char *d = base + H.off_lit + vsz * l;
        if (exact) { const int v = (int)(2 * m.ival(r, c)); std::memcpy(d, &v, 4); }
        else { const double v = std::ldexp(m.fval(r, c), -E.exp2[r]); std::memcpy(d, &v, 8); }
    }
    std::memcpy(base + H.off_flipptr, flipptr.data(), 2 * flipptr.size());
    if (!flip.empty()) std::memcpy(base + H.off_flip, flip.data(), 2 * flip.size());
    std::memcpy(base + H.off_prog, prog.data(), sizeof(pk::VmIns) * prog.size());
    return true;
}

}  // namespace perm
