// vm.h -- the step program of the eliminated walk as the precompiled kernels
// read it (plain data, shared by the host code and the kernels).
//
// A program image is a header, the start values of x, the matrix entries the
// program and the flips add (literals), the flip lists of the outer columns
// and the step's program.  Values live in numbered slots, one word per lane:
// slots 0..n-1 hold x, slot n pads, the rest hold tables, reused once dead.  A
// table over w low columns is 2^w consecutive slots, its lowest index bit the
// column summed out first.  An instruction works on whole tables: entry e of
// its result takes entries of its operands at strides given per index bit (0
// where the operand does not mention that column), so one decoding serves up to
// 64 entries and the addresses follow by additions.
//
// FP64 walks also sum |terms| (core.cuh).  A table of plain products has its
// entries' own magnitudes; only where a column has been summed out does the sum
// of magnitudes differ from the magnitude of the sum, and only such tables have
// a second, FP32 table in the magnitude slots.
#pragma once

namespace pk {

enum VmKind {
    kVmRow = 0,    // dst_i[e] = x_i + the literals of e's set bits, for up to four rows of w <= 3 columns
    kVmBigRow = 1, // the same for one row of w > 3 columns
    kVmMul = 2,    // dst[e] = A[e] * B[e]
    kVmMulF = 3,   // the same with magnitudes
    kVmSum = 4,    // dst[e] = A[e] * B[e] - A[e + ea] * B[e + eb]: a column summed out (and the magnitudes' sum)
    kVmSub = 5,    // dst[e] = A[e] - A[e + ea] (and the magnitudes' sum)
    kVmProd = 6    // dst = the product of the listed single slots (and magnitudes)
};
constexpr int kVmBits = 6;                // index bits an instruction can stride over
constexpr unsigned kVmRingSlot = 0x8000;  // table number names ring slots (exact walks wider than 64 bits)
constexpr unsigned kVmSlotMask = 0x7fff;
constexpr unsigned kVmNoMag = 0xffff;     // the operand's magnitudes are its entries' own
constexpr int kVmRowsMost = 4;
constexpr int kVmRowBits = 3;
constexpr int kVmProdMost = 10;

struct VmIns {                // 48 bytes
    unsigned char kind, w;    // w: index bits of the result (kVmProd: factors)
    unsigned short dst;       // kVmRow: rows
    union {
        struct {
            unsigned short a, b, fdst, fa, fb, pad;
            unsigned short sa[kVmBits], sb[kVmBits];   // strides in bytes (ring results: in slots)
            unsigned short ea, eb;
        } t;
        struct { unsigned short dst, x, lit[kVmRowBits]; } row[kVmRowsMost];
        struct { unsigned short x, lit[kVmBits]; } big;
        struct { unsigned short fdst, pad; struct { unsigned short slot, fslot; } f[kVmProdMost]; } prod;
    };
};

struct VmHeader {       // 64 bytes; offsets in bytes from the image's start, all multiples of 16
    int n;              // x slots; slot n pads
    int h;              // outer columns
    int off_base;       // scratch for a warp's common start vector (n start values)
    int bytes;          // size of the image (the staging code reads it here)
    int nslots;         // value slots
    int nextra;         // ring slots (exact) or magnitude slots (FP64, double-double)
    int nins;           // instructions of the program
    int result;         // slot of the step's signed sum
    int fresult;        // its magnitude slot, or kVmNoMag
    int off_x0, off_lit, off_flipptr, off_flip, off_prog;
    int reserved1, reserved2;
};

}  // namespace pk
