// vm_impl.cuh -- the eliminated walk (elim.hpp) run from a program image by
// precompiled kernels: batches, serving and single matrices too small to be
// worth a compilation.
//
// What bounds it: an FP64 operation occupies the FP64 pipe for 16 clocks of an
// SM per warp, so a program interpreted from shared memory can keep the pipe as
// busy as compiled code, given few enough instructions and enough warps around
// each operation.  An instruction therefore works on a whole table (vm.h), eight
// entries at a time: its decoding is shared, the operands' addresses follow by
// additions, the results' are immediate offsets, and eight independent products
// hide one another's latency.  The value slots of a warp (10-40 KB) set how many
// warps an SM holds, so there is one value per lane and slot.
//
// Measured (an n=28 p=0.3 FP64 matrix of 3.1 operations per Gray step, 2^27 steps;
// most of its family count 2.5 and take 0.8-0.9 ms): 1.22 ms, 6 warps per SM; with a
// range of slots per partial product, 10 % more slots and 5 warps, 1.33 ms at
// 58 % FP64-pipe activity.  Taken back: scalar instructions in bundles of four, one
// value per slot, 1.24 ms with 9 % fewer operations (56 % of the pipe); two values
// per lane and slot (half the decoding, half the warps) 1.86 ms; tables of 2^4
// entries (7 warps, 24 % more operations) 1.50 ms, of 2^6 (4 warps, 15 % fewer)
// 1.30 ms, but 3.1 against 2.7 ms at p=0.4.
//
// Each warp has its own shared-memory region: the image, then the value slots
// (slot-major, one word per lane: conflict-free).  Slots belong to one lane,
// so nothing is exchanged between lanes before the final shuffle reduction.
#pragma once

#ifndef PERM_HOST_EMULATION
#include <cuda_runtime.h>

#include "finish.cuh"
#include "vm.hpp"
#endif
#include "core.cuh"
#include "vm.h"

namespace pk {

// ------------------------------------------------------------------ shared-memory addresses
// 32-bit shared-window addresses with explicit loads and stores: a table
// instruction holds up to sixteen addresses at once, which would be 64-bit
// generic pointers otherwise.  (The host emulation uses plain pointers.)
#ifdef PERM_HOST_EMULATION
typedef unsigned char *VmAddr;
__device__ __forceinline__ VmAddr vm_addr(unsigned char *p) { return p; }
__device__ __forceinline__ double vm_ld_f64(VmAddr a) { return *reinterpret_cast<const double *>(a); }
__device__ __forceinline__ u64 vm_ld_u64(VmAddr a) { return *reinterpret_cast<const u64 *>(a); }
__device__ __forceinline__ float vm_ld_f32(VmAddr a) { return *reinterpret_cast<const float *>(a); }
__device__ __forceinline__ int vm_ld_s32(VmAddr a) { return *reinterpret_cast<const int *>(a); }
__device__ __forceinline__ uint4 vm_ld_v4(VmAddr a) { return *reinterpret_cast<const uint4 *>(a); }
__device__ __forceinline__ void vm_st(VmAddr a, double v) { *reinterpret_cast<double *>(a) = v; }
__device__ __forceinline__ void vm_st(VmAddr a, u64 v) { *reinterpret_cast<u64 *>(a) = v; }
__device__ __forceinline__ void vm_st(VmAddr a, float v) { *reinterpret_cast<float *>(a) = v; }
#else
typedef u32 VmAddr;
__device__ __forceinline__ VmAddr vm_addr(unsigned char *p) { return (u32)__cvta_generic_to_shared(p); }
__device__ __forceinline__ double vm_ld_f64(VmAddr a) {
    double v;
    asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ u64 vm_ld_u64(VmAddr a) {
    u64 v;
    asm volatile("ld.shared.u64 %0, [%1];" : "=l"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float vm_ld_f32(VmAddr a) {
    float v;
    asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ int vm_ld_s32(VmAddr a) {
    int v;
    asm volatile("ld.shared.s32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ uint4 vm_ld_v4(VmAddr a) {
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void vm_st(VmAddr a, double v) { asm volatile("st.shared.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory"); }
__device__ __forceinline__ void vm_st(VmAddr a, u64 v) { asm volatile("st.shared.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory"); }
__device__ __forceinline__ void vm_st(VmAddr a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }
#endif

// ------------------------------------------------------------------ slots of each arithmetic
struct VmF64 {
    typedef ArithF64 A;
    typedef double Lit;
    typedef double X0;
    typedef double Cell;
    static constexpr int kBits = 3;       // 2^kBits table entries in flight
    static constexpr int kSlot = 256;     // bytes of a slot
    static constexpr bool kMag = true;    // sums of |terms| are kept
    VmAddr bv, bf, lits;
    __device__ __forceinline__ void bind(unsigned char *area, const VmHeader *H, VmAddr l, int lane) {
        bv = vm_addr(area) + lane * 8;
        bf = vm_addr(area) + H->nslots * kSlot + lane * 4;
        lits = l;
    }
    static __device__ __forceinline__ Cell get(VmAddr p) { return vm_ld_f64(p); }
    static __device__ __forceinline__ void put(VmAddr p, Cell c) { vm_st(p, c); }
    __device__ __forceinline__ Lit lit(unsigned i) const { return vm_ld_f64(lits + i * 8); }
    static __device__ __forceinline__ float mag(Cell v) { return abs_f32_full(v); }
    static __device__ __forceinline__ Cell start(X0 x) { return x; }
    static __device__ __forceinline__ Cell plus(Cell x, Lit l) { return x + l; }
    static __device__ __forceinline__ Cell plus_rt(Cell x, Lit l, int s) { return A::upd_rt(x, l, s); }
    static __device__ __forceinline__ X0 base_add(X0 x, Lit l) { return x + l; }
    static __device__ __forceinline__ Cell mul(Cell a, Cell b) { return a * b; }
    static __device__ __forceinline__ Cell mulsub(Cell a, Cell b, Cell c) { return fma(-a, b, c); }   // c - a b
    static __device__ __forceinline__ Cell sub(Cell a, Cell b) { return a - b; }
    static __device__ __forceinline__ void add_result(A::Blk &b, Cell c, bool odd) { b.s += odd ? -c : c; }
};

struct VmDD {
    typedef ArithDD A;
    typedef double Lit;
    typedef DD X0;
    typedef DD Cell;
    static constexpr int kBits = 2;
    static constexpr int kSlot = 512;     // high parts, then low parts
    static constexpr bool kMag = true;
    VmAddr bv, bf, lits;
    __device__ __forceinline__ void bind(unsigned char *area, const VmHeader *H, VmAddr l, int lane) {
        bv = vm_addr(area) + lane * 8;
        bf = vm_addr(area) + H->nslots * kSlot + lane * 4;
        lits = l;
    }
    static __device__ __forceinline__ Cell get(VmAddr p) { return A::mk(vm_ld_f64(p), vm_ld_f64(p + 256)); }
    static __device__ __forceinline__ void put(VmAddr p, const Cell &c) {
        vm_st(p, c.h);
        vm_st(p + 256, c.l);
    }
    __device__ __forceinline__ Lit lit(unsigned i) const { return vm_ld_f64(lits + i * 8); }
    static __device__ __forceinline__ float mag(const Cell &v) { return abs_f32_full(v.h); }
    static __device__ __forceinline__ Cell start(X0 x) { return x; }
    static __device__ __forceinline__ Cell plus(Cell x, Lit l) { return A::add_d(x, l); }
    static __device__ __forceinline__ Cell plus_rt(Cell x, Lit l, int s) { return A::upd_rt(x, l, s); }
    static __device__ __forceinline__ X0 base_add(X0 x, Lit l) { return A::add_d(x, l); }
    static __device__ __forceinline__ Cell mul(Cell a, Cell b) { return A::mul(a, b); }
    static __device__ __forceinline__ Cell mulsub(Cell a, Cell b, Cell c) { return A::diff(c, A::mul(a, b)); }
    static __device__ __forceinline__ Cell sub(Cell a, Cell b) { return A::diff(a, b); }
    static __device__ __forceinline__ void add_result(A::Blk &b, Cell c, bool odd) {
        if (odd) A::template blk_add<-1>(b, c); else A::template blk_add<1>(b, c);
    }
};

// Exact values: 64-bit slots while their a-priori bound fits (always, modulo
// 2^64, for the 64-bit ring), ring slots of L limbs beyond.
template <int NL>
struct VmExact {
    typedef ArithExact<NL> A;
    typedef int Lit;
    typedef int X0;
    typedef u64 Cell;
    static constexpr int kBits = 3;
    static constexpr int kSlot = 256;
    static constexpr bool kMag = false;
    static constexpr int W = (NL + 1) / 2;
    VmAddr bv, bf, lits;
    __device__ __forceinline__ void bind(unsigned char *area, const VmHeader *H, VmAddr l, int lane) {
        bv = vm_addr(area) + lane * 8;
        bf = bv + H->nslots * kSlot;   // ring slots: W words of 256 bytes
        lits = l;
    }
    static __device__ __forceinline__ Cell get(VmAddr p) { return vm_ld_u64(p); }
    static __device__ __forceinline__ void put(VmAddr p, Cell c) { vm_st(p, c); }
    __device__ __forceinline__ Lit lit(unsigned i) const { return vm_ld_s32(lits + i * 4); }
    static __device__ __forceinline__ float mag(Cell) { return 0.f; }
    static __device__ __forceinline__ Cell start(X0 x) { return (u64)(i64)x; }
    static __device__ __forceinline__ Cell plus(Cell x, Lit l) { return x + (u64)(i64)l; }
    static __device__ __forceinline__ Cell plus_rt(Cell x, Lit l, int s) { return x + (u64)(i64)(s * l); }
    static __device__ __forceinline__ X0 base_add(X0 x, Lit l) { return x + l; }
    static __device__ __forceinline__ Cell mul(Cell a, Cell b) { return a * b; }
    static __device__ __forceinline__ Cell mulsub(Cell a, Cell b, Cell c) { return c - a * b; }
    static __device__ __forceinline__ Cell sub(Cell a, Cell b) { return a - b; }
    // entry `e` of table s (ring or 64-bit) as a ring element
    __device__ __forceinline__ Ring<NL> ld_ring(unsigned s, int e) const {
        const int q = (int)(s & kVmSlotMask) + e;
        if (!(s & kVmRingSlot)) return ring_of<NL>((i64)get(bv + q * kSlot));
        Ring<NL> r;
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const u64 w = get(bf + (q * W + i) * kSlot);
            r.w[2 * i] = (u32)w;
            if (2 * i + 1 < NL) r.w[(2 * i + 1) % NL] = (u32)(w >> 32);
        }
        return r;
    }
    __device__ __forceinline__ void st_ring(int q, const Ring<NL> &r) {
#pragma unroll
        for (int i = 0; i < W; ++i) {
            const u64 hi = (2 * i + 1 < NL) ? (u64)r.w[(2 * i + 1) % NL] : 0ull;
            put(bf + (q * W + i) * kSlot, (hi << 32) | r.w[2 * i]);
        }
    }
    // a table instruction into ring slots, entry by entry
    __device__ __forceinline__ void ring_table(int kind, int w, unsigned dst, unsigned a, unsigned b, const int *sa,
                                               const int *sb, int ea, int eb) {
#pragma unroll 1
        for (int e = (1 << w) - 1; e >= 0; --e) {   // (from the top down: vm_blocks)
            int oa = 0, ob = 0;
#pragma unroll
            for (int k = 0; k < kVmBits; ++k)
                if ((e >> k) & 1) { oa += sa[k]; ob += sb[k]; }
            Ring<NL> r;
            if (kind == kVmSub) {
                r = ring_minus(ld_ring(a, oa), ld_ring(a, oa + ea));
            } else {
                r = ring_times(ld_ring(a, oa), ld_ring(b, ob));
                if (kind == kVmSum) r = ring_minus(r, ring_times(ld_ring(a, oa + ea), ld_ring(b, ob + eb)));
            }
            st_ring((int)(dst & kVmSlotMask) + e, r);
        }
    }
};

template <class Vm> struct VmRings { static constexpr bool v = false; };
template <int NL> struct VmRings<VmExact<NL>> { static constexpr bool v = NL > 2; };

// ------------------------------------------------------------------ instructions
// Addresses of 2^NB consecutive result indices: base + the strides of their set bits.
template <int NB>
__device__ __forceinline__ void vm_addresses(VmAddr (&o)[1 << NB], VmAddr base, const int *s) {
    o[0] = base;
#pragma unroll
    for (int k = 0; k < NB; ++k)
#pragma unroll
        for (int i = 0; i < (1 << k); ++i) o[i | (1 << k)] = o[i] + s[k];
}

// Operand tables of an instruction: value and magnitude tables (bytes), and
// whether the magnitudes are the entries' own.
struct VmTab { VmAddr v, f; bool own; };

template <class Vm>
__device__ __forceinline__ float vm_mag(const Vm &vm, const VmTab &t, VmAddr p, typename Vm::Cell c) {
    if (t.own) return vm.mag(c);
    return vm_ld_f32(t.f + (int)(p - t.v) / (Vm::kSlot / 128));   // a magnitude slot: 128 bytes
}

template <class Vm, int NB>
__device__ __forceinline__ void vm_mul_block(VmAddr d, VmAddr a, VmAddr b, const int *sa, const int *sb) {
    VmAddr pa[1 << NB], pb[1 << NB];
    vm_addresses<NB>(pa, a, sa);
    vm_addresses<NB>(pb, b, sb);
    typename Vm::Cell r[1 << NB];
#pragma unroll
    for (int i = 0; i < (1 << NB); ++i) r[i] = Vm::mul(Vm::get(pa[i]), Vm::get(pb[i]));
#pragma unroll
    for (int i = 0; i < (1 << NB); ++i) Vm::put(d + i * Vm::kSlot, r[i]);
}
// entries with magnitudes: a product (kVmMulF), a summed-out pair of products
// (kVmSum) or a difference (kVmSub)
template <class Vm, int KIND, int NB>
__device__ __forceinline__ void vm_mag_block(const Vm &vm, VmAddr d, VmAddr fd, VmAddr a, VmAddr b,
                                             const VmTab &ta, const VmTab &tb, const int *sa, const int *sb,
                                             int ea, int eb) {
    typedef typename Vm::Cell Cell;
    VmAddr pa[1 << NB], pb[1 << NB];
    vm_addresses<NB>(pa, a, sa);
    if (KIND != kVmSub) vm_addresses<NB>(pb, b, sb);
    Cell r[1 << NB];
    float g[1 << NB];
#pragma unroll
    for (int i = 0; i < (1 << NB); ++i) {
        const Cell x = Vm::get(pa[i]);
        if constexpr (KIND == kVmSub) {
            const Cell y = Vm::get(pa[i] + ea);
            r[i] = Vm::sub(x, y);
            if (Vm::kMag) g[i] = vm_mag(vm, ta, pa[i], x) + vm_mag(vm, ta, pa[i] + ea, y);
        } else {
            const Cell y = Vm::get(pb[i]);
            r[i] = Vm::mul(x, y);
            if (Vm::kMag) g[i] = vm_mag(vm, ta, pa[i], x) * vm_mag(vm, tb, pb[i], y);
        }
    }
    if constexpr (KIND == kVmSum) {
#pragma unroll
        for (int i = 0; i < (1 << NB); ++i) {
            const Cell x = Vm::get(pa[i] + ea), y = Vm::get(pb[i] + eb);
            r[i] = Vm::mulsub(x, y, r[i]);
            if (Vm::kMag) g[i] = fma(vm_mag(vm, ta, pa[i] + ea, x), vm_mag(vm, tb, pb[i] + eb, y), g[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < (1 << NB); ++i) {
        Vm::put(d + i * Vm::kSlot, r[i]);
        if (Vm::kMag) vm_st(fd + i * 128, g[i]);
    }
}
template <class Vm, int NB>
__device__ __forceinline__ void vm_row_block(VmAddr d, typename Vm::Cell x, const typename Vm::Lit *l) {
    typename Vm::Cell r[1 << NB];
    r[0] = x;
#pragma unroll
    for (int k = 0; k < NB; ++k)
#pragma unroll
        for (int i = 0; i < (1 << k); ++i) r[i | (1 << k)] = Vm::plus(r[i], l[k]);
#pragma unroll
    for (int i = 0; i < (1 << NB); ++i) Vm::put(d + i * Vm::kSlot, r[i]);
}
// up to four rows of NB columns, side by side
template <class Vm, int NB, int FROM, int TO>
__device__ __forceinline__ void vm_rows(Vm &vm, int rows, const unsigned (&f)[kVmRowsMost * (2 + kVmRowBits)]) {
    typedef typename Vm::Cell Cell;
    constexpr int F = 2 + kVmRowBits;
    Cell r[kVmRowsMost][1 << NB];
#pragma unroll
    for (int q = FROM; q < TO; ++q) {   // (rows beyond the count repeat row 0's loads: their fields are zero)
        r[q][0] = Vm::get(vm.bv + f[q * F + 1] * Vm::kSlot);
    }
#pragma unroll
    for (int k = 0; k < NB; ++k)
#pragma unroll
        for (int q = FROM; q < TO; ++q)
            if (q < rows) {
                const typename Vm::Lit l = vm.lit(f[q * F + 2 + k]);
#pragma unroll
                for (int i = 0; i < (1 << k); ++i) r[q][i | (1 << k)] = Vm::plus(r[q][i], l);
            }
#pragma unroll
    for (int q = FROM; q < TO; ++q)
        if (q < rows) {
            const VmAddr d = vm.bv + f[q * F] * Vm::kSlot;
#pragma unroll
            for (int i = 0; i < (1 << NB); ++i) Vm::put(d + i * Vm::kSlot, r[q][i]);
        }
}

// Blocks of 2^NB entries over all index bits of a table instruction, from the
// top down: a result may share its lower part with its first operand (vm_image.cpp).
template <class Vm, int KIND, int NB>
__device__ __forceinline__ void vm_blocks(Vm &vm, int w, VmAddr d, VmAddr fd, const VmTab &ta, const VmTab &tb,
                                          const int *sa, const int *sb, int ea, int eb) {
#pragma unroll 1
    for (int o = (1 << (w - NB)) - 1; o >= 0; --o) {
        VmAddr a = ta.v, b = tb.v;
#pragma unroll
        for (int k = 0; k + NB < kVmBits; ++k)
            if ((o >> k) & 1) { a += sa[k + NB]; b += sb[k + NB]; }
        const VmAddr e = d + o * (Vm::kSlot << NB);
        if constexpr (KIND == kVmMul) vm_mul_block<Vm, NB>(e, a, b, sa, sb);
        else vm_mag_block<Vm, KIND, NB>(vm, e, fd + o * (128 << NB), a, b, ta, tb, sa, sb, ea, eb);
    }
}

// One instruction (its 48 bytes).
template <class Vm>
__device__ __forceinline__ void vm_step(Vm &vm, const uint4 &w0, const uint4 &w1, const uint4 &w2) {
    typedef typename Vm::Cell Cell;
    constexpr int KB = Vm::kBits, S = Vm::kSlot;
    const int kind = w0.x & 0xff, w = (w0.x >> 8) & 0xff;
    const unsigned dst = w0.x >> 16;
    if (kind == kVmRow) {
        const unsigned f[kVmRowsMost * (2 + kVmRowBits)] = {
            w0.y & 0xffff, w0.y >> 16, w0.z & 0xffff, w0.z >> 16, w0.w & 0xffff, w0.w >> 16, w1.x & 0xffff, w1.x >> 16,
            w1.y & 0xffff, w1.y >> 16, w1.z & 0xffff, w1.z >> 16, w1.w & 0xffff, w1.w >> 16, w2.x & 0xffff, w2.x >> 16,
            w2.y & 0xffff, w2.y >> 16, w2.z & 0xffff, w2.z >> 16};
        const int rows = (int)dst;
        if (w == 1) {
            vm_rows<Vm, 1, 0, 4>(vm, rows, f);
        } else if (w == 2) {
            vm_rows<Vm, 2, 0, 4>(vm, rows, f);
        } else {   // eight entries a row: two rows at once
            vm_rows<Vm, 3, 0, 2>(vm, rows, f);
            if (rows > 2) vm_rows<Vm, 3, 2, 4>(vm, rows, f);
        }
        return;
    }
    if (kind == kVmBigRow) {
        const unsigned li[kVmBits] = {w0.y >> 16, w0.z & 0xffff, w0.z >> 16, w0.w & 0xffff, w0.w >> 16, w1.x & 0xffff};
        typename Vm::Lit l[kVmBits];
#pragma unroll
        for (int k = 0; k < kVmBits; ++k) l[k] = vm.lit(li[k]);   // (literal 0 where the table has fewer columns)
        const Cell x = Vm::get(vm.bv + (w0.y & 0xffff) * S);
        VmAddr d = vm.bv + dst * S;
#pragma unroll 1
        for (int o = 0; o < (1 << (w - KB)); ++o, d += S << KB) {
            Cell y = x;
#pragma unroll
            for (int k = 0; k + KB < kVmBits; ++k)
                if ((o >> k) & 1) y = Vm::plus(y, l[k + KB]);
            vm_row_block<Vm, KB>(d, y, l);
        }
        return;
    }
    if (kind == kVmProd) {
        const unsigned e[kVmProdMost] = {w0.z, w0.w, w1.x, w1.y, w1.z, w1.w, w2.x, w2.y, w2.z, w2.w};
        Cell p[2];
        float g[2] = {1.f, 1.f};
#pragma unroll
        for (int i = 0; i < kVmProdMost; ++i)
            if (i < w) {   // two running products
                const Cell c = Vm::get(vm.bv + (e[i] & 0xffff) * S);
                p[i & 1] = i < 2 ? c : Vm::mul(p[i & 1], c);
                if (Vm::kMag)
                    g[i & 1] *= (e[i] >> 16) == kVmNoMag ? vm.mag(c) : vm_ld_f32(vm.bf + (e[i] >> 16) * 128);
            }
        Vm::put(vm.bv + dst * S, Vm::mul(p[0], p[1]));   // (two factors or more)
        if (Vm::kMag) vm_st(vm.bf + (w0.y & 0xffff) * 128, g[0] * g[1]);
        return;
    }
    const unsigned na = w0.y & 0xffff, nb = w0.y >> 16;
    const int sa[kVmBits] = {(int)(w1.x & 0xffff), (int)(w1.x >> 16), (int)(w1.y & 0xffff), (int)(w1.y >> 16), (int)(w1.z & 0xffff), (int)(w1.z >> 16)};
    const int sb[kVmBits] = {(int)(w1.w & 0xffff), (int)(w1.w >> 16), (int)(w2.x & 0xffff), (int)(w2.x >> 16), (int)(w2.y & 0xffff), (int)(w2.y >> 16)};
    const int ea = w2.z & 0xffff, eb = w2.z >> 16;
    if constexpr (VmRings<Vm>::v) {
        if (dst & kVmRingSlot) {
            vm.ring_table(kind, w, dst, na, nb, sa, sb, ea, eb);
            return;
        }
    }
    const unsigned fa = w0.z >> 16, fb = w0.w & 0xffff;
    VmTab ta, tb;
    ta.v = vm.bv + na * S;
    tb.v = vm.bv + nb * S;
    ta.f = vm.bf + fa * 128;
    tb.f = vm.bf + fb * 128;
    ta.own = fa == kVmNoMag;
    tb.own = fb == kVmNoMag;
    const VmAddr d = vm.bv + dst * S, fd = vm.bf + (w0.z & 0xffff) * 128;
    if (kind == kVmMul) {
        if (w >= KB) vm_blocks<Vm, kVmMul, KB>(vm, w, d, fd, ta, tb, sa, sb, ea, eb);
        else if (w == 2) vm_mul_block<Vm, 2>(d, ta.v, tb.v, sa, sb);
        else if (w == 1) vm_mul_block<Vm, 1>(d, ta.v, tb.v, sa, sb);
        else vm_mul_block<Vm, 0>(d, ta.v, tb.v, sa, sb);
    } else if (kind == kVmSum) {
        if (w >= 2) vm_blocks<Vm, kVmSum, 2>(vm, w, d, fd, ta, tb, sa, sb, ea, eb);
        else if (w == 1) vm_mag_block<Vm, kVmSum, 1>(vm, d, fd, ta.v, tb.v, ta, tb, sa, sb, ea, eb);
        else vm_mag_block<Vm, kVmSum, 0>(vm, d, fd, ta.v, tb.v, ta, tb, sa, sb, ea, eb);
    } else if (kind == kVmSub) {
        if (w >= 2) vm_blocks<Vm, kVmSub, 2>(vm, w, d, fd, ta, tb, sa, sb, ea, eb);
        else vm_blocks<Vm, kVmSub, 0>(vm, w, d, fd, ta, tb, sa, sb, ea, eb);
    } else if (Vm::kMag) {
        if (w >= 2) vm_blocks<Vm, kVmMulF, 2>(vm, w, d, fd, ta, tb, sa, sb, ea, eb);
        else vm_blocks<Vm, kVmMulF, 0>(vm, w, d, fd, ta, tb, sa, sb, ea, eb);
    }
}

// ------------------------------------------------------------------ the walk

// Adds outer column j to x, s times (+1, -1, or a lane's weight 0 or 1).
template <class Vm>
__device__ __forceinline__ void vm_flip(Vm &vm, const unsigned char *img, int j, int s) {
    const VmHeader *H = reinterpret_cast<const VmHeader *>(img);
    const unsigned short *ptr = reinterpret_cast<const unsigned short *>(img + H->off_flipptr);
    const uint4 *fl = reinterpret_cast<const uint4 *>(img + H->off_flip);
    const int e = ptr[j + 1];
    for (int b = ptr[j]; b < e; ++b) {   // four rows at a time (padded with slot n)
        const uint4 w = fl[b];
        const unsigned sl[4] = {w.x & 0xffff, w.y & 0xffff, w.z & 0xffff, w.w & 0xffff};
        const unsigned li[4] = {w.x >> 16, w.y >> 16, w.z >> 16, w.w >> 16};
        typename Vm::Cell x[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = Vm::plus_rt(Vm::get(vm.bv + sl[i] * Vm::kSlot), vm.lit(li[i]), s);
#pragma unroll
        for (int i = 0; i < 4; ++i) Vm::put(vm.bv + sl[i] * Vm::kSlot, x[i]);
    }
}

// Work that the warp shares lane by lane; the host emulation's one lane does all of it.
#ifdef PERM_HOST_EMULATION
#define PERM_VM_LANES(i, lane, count) for (int i = 0; i < (count); ++i)
#else
#define PERM_VM_LANES(i, lane, count) for (int i = (lane); i < (count); i += 32)
#endif

// x at the chunk's first outer index.  The columns set in every lane's code
// (all but the few lowest of the outer columns' high ones) are added once per
// warp, a lane per entry, to a common vector; the rest lane by lane with weight
// 0 or 1.
template <class Vm>
__device__ __forceinline__ void vm_start(Vm &vm, unsigned char *img, int lane, u64 G) {
    const VmHeader *H = reinterpret_cast<const VmHeader *>(img);
    typedef typename Vm::X0 X0;
    const X0 *x0 = reinterpret_cast<const X0 *>(img + H->off_x0);
    X0 *base = reinterpret_cast<X0 *>(img + H->off_base);
    const unsigned short *ptr = reinterpret_cast<const unsigned short *>(img + H->off_flipptr);
    const unsigned short *fl = reinterpret_cast<const unsigned short *>(img + H->off_flip);
    const int n = H->n;
    const u64 any = warp_or64(G), common = ~warp_or64(~G);
    __syncwarp();   // the warp has read the vector of its last task
    PERM_VM_LANES(i, lane, n) base[i] = x0[i];
    for (u64 U = common; U; U &= U - 1) {
        const int p = ctz64(U);
        __syncwarp();
        const int b = 4 * ptr[p], e = 4 * ptr[p + 1];   // a column's rows are distinct: one lane each
        PERM_VM_LANES(t, lane, e - b) {
            const int s = fl[2 * (b + t)];
            if (s < n) base[s] = Vm::base_add(base[s], vm.lit(fl[2 * (b + t) + 1]));   // (not a padding pair)
        }
    }
    __syncwarp();
    for (int i = 0; i < n; ++i) Vm::put(vm.bv + i * Vm::kSlot, Vm::start(base[i]));
    Vm::put(vm.bv + n * Vm::kSlot, Vm::start(X0()));   // the padding slot
    for (u64 U = any & ~common; U; U &= U - 1) {
        const int p = ctz64(U);
        vm_flip(vm, img, p, (int)((G >> p) & 1ull));
    }
}

// Adds the step's signed sum (and its sum of magnitudes) to the block sum.
template <class Vm>
__device__ __forceinline__ void vm_result(const Vm &vm, const VmHeader *H, typename Vm::A::Blk &b, bool odd) {
    if constexpr (Vm::kMag) {
        const typename Vm::Cell c = Vm::get(vm.bv + H->result * Vm::kSlot);
        Vm::add_result(b, c, odd);
        Vm::A::blk_abs_f(b, H->fresult == (int)kVmNoMag ? vm.mag(c) : vm_ld_f32(vm.bf + H->fresult * 128));
    } else {
        const auto t = vm.ld_ring((unsigned)H->result, 0);
        if (odd) Vm::A::template blk_add<-1>(b, t); else Vm::A::template blk_add<1>(b, t);
    }
}

// One chunk of 2^K outer steps of the image's matrix (q counts chunks); the
// slots start at `area`.
template <class Vm>
__device__ __forceinline__ typename Vm::A::Acc vm_chunk(unsigned char *img, unsigned char *area, int lane, u64 q, int K) {
    typedef typename Vm::A A;
    const VmHeader *H = reinterpret_cast<const VmHeader *>(img);
    const VmAddr prog = vm_addr(img) + H->off_prog;
    const int ni = H->nins;
    Vm vm;
    vm.bind(area, H, vm_addr(img) + H->off_lit, lane);
    const u64 g0 = q << K;
    vm_start(vm, img, lane, g0 ^ (g0 >> 1));
    typename A::Acc acc = A::acc_zero();
    typename A::Blk mid = A::blk_zero();
    const u64 len = 1ull << K;
    u64 l = 0;
    for (;;) {
        uint4 w0 = vm_ld_v4(prog), w1 = vm_ld_v4(prog + 16), w2 = vm_ld_v4(prog + 32);
#pragma unroll 1
        for (int i = 0; i < ni; ++i) {
            const uint4 c0 = w0, c1 = w1, c2 = w2;
            const VmAddr nx = prog + 48 * (i + 1 < ni ? i + 1 : i);   // the next instruction's words, ahead of this one's stores
            w0 = vm_ld_v4(nx);
            w1 = vm_ld_v4(nx + 16);
            w2 = vm_ld_v4(nx + 32);
            vm_step(vm, c0, c1, c2);
        }
        vm_result(vm, H, mid, ((g0 + l) & 1ull) != 0);
        if (++l >= len) break;
        if ((l & 7) == 0) {   // merged into the compensated accumulator every 8 steps
            A::acc_merge(acc, mid);
            mid = A::blk_zero();
        }
        const int j = ctz64(l);
        vm_flip(vm, img, j, (((g0 + l) >> (j + 1)) & 1ull) ? -1 : 1);
        __syncwarp();
    }
    A::acc_merge(acc, mid);
    return acc;
}

// Warps take 32-chunk tasks from one counter, as in the chained generic walk
// (generic_impl.cuh): same task table, same result places.
template <class Vm>
__device__ __forceinline__ void vm_task_loop(const BatchArgs &ba, unsigned char *slot) {
    typedef typename Vm::A A;
    const int lane = threadIdx.x & 31;
    int cached = -1;
    for (;;) {
        u64 task = 0;
        if (lane == 0) task = past_deadline(ba.timeout_ns, ba.deadline_word, ba.abort_flag) ? ~0ull : atomicAdd(ba.task_counter, 1ull);
        task = __shfl_sync(PERM_FULLMASK, task, 0);
        if (task >= ba.ntasks) break;
        int m = 0;
        if (lane == 0) {
            int lo = 0, hi = ba.nmat - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (ba.mats[mid].task_begin <= task) lo = mid; else hi = mid - 1;
            }
            m = lo;
        }
        m = __shfl_sync(PERM_FULLMASK, m, 0);
        const BatchMat bm = ba.mats[m];
        if (bm.image != cached) {
            __syncwarp();
            const uint4 *src = reinterpret_cast<const uint4 *>(
                reinterpret_cast<const unsigned char *>(ba.devmats) + (size_t)bm.image * 16);
            const int words = reinterpret_cast<const int *>(src)[3] / 16;   // the image's own size
            uint4 *dst = reinterpret_cast<uint4 *>(slot);
            for (int i = lane; i < words; i += 32) dst[i] = src[i];
            __syncwarp();
            cached = bm.image;
        }
        u64 q = bm.chunk_lo + (task - bm.task_begin) * 32ull + (u64)lane;
        const bool live = q < bm.chunk_hi;
        if (!live) q = bm.chunk_hi - 1;     // idle lanes shadow a real chunk to stay in step
        typename A::Acc acc = vm_chunk<Vm>(slot, slot + reinterpret_cast<const VmHeader *>(slot)->bytes, lane, q, bm.K);
        if (!live) acc = A::acc_zero();
#pragma unroll
        for (int d = 16; d >= 1; d >>= 1) acc = A::acc_add(acc, A::shfl_down(acc, d));
        if (lane == 0) A::acc_store(ba.task_out + (bm.out_offset + (task - bm.task_begin)) * (u64)A::ACC_WORDS, acc);
    }
}

#ifndef PERM_HOST_EMULATION
// One warp per block: a program's slots take 10-45 KB of shared memory, and
// single-warp blocks fill an SM's 227 KB to the last warp that fits.
template <class Vm>
__global__ void __launch_bounds__(32, 8) k_walk_vm(BatchArgs ba) {
    extern __shared__ __align__(16) unsigned char vm_smem[];
    vm_task_loop<Vm>(ba, vm_smem);
    finish_walk<typename Vm::A>(ba.finish);
}

#endif

}  // namespace pk

#ifndef PERM_HOST_EMULATION
namespace perm {

// The same limit from every caller: threads that launch programs of different
// sizes at once never lower it under each other's launch.
template <class Vm>
static cudaError_t vm_set_smem() {
    return cudaFuncSetAttribute(pk::k_walk_vm<Vm>, cudaFuncAttributeMaxDynamicSharedMemorySize, kVmMaxWarpBytes);
}
template <class Vm>
static cudaError_t vm_launch_t(const pk::BatchArgs &ba, int grid, int block, cudaStream_t st) {
    const size_t smem = (size_t)ba.slot_bytes;
    cudaError_t e = vm_set_smem<Vm>();
    if (e != cudaSuccess) return e;
    pk::k_walk_vm<Vm><<<grid, block, smem, st>>>(ba);
    return cudaGetLastError();
}
template <class Vm>
static cudaError_t vm_attr_t(cudaFuncAttributes *attr) {
    return cudaFuncGetAttributes(attr, pk::k_walk_vm<Vm>);
}
template <class Vm>
static cudaError_t vm_occ_t(int block, size_t slot_bytes, int *blocks_per_sm) {
    cudaError_t e = vm_set_smem<Vm>();
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, pk::k_walk_vm<Vm>, block, slot_bytes);
}
template <class Vm>
static GenericFns vm_make_fns() {
    GenericFns f;
    f.walk = vm_launch_t<Vm>;
    f.attr = vm_attr_t<Vm>;
    f.occ = vm_occ_t<Vm>;
    f.block_log2 = 0;
    return f;
}

}  // namespace perm
#endif
