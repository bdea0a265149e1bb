// The diagonal window of the persistent and shared-string verifiers: one
// column step, the window's minimum and the meeting of two halves.
//
// Rows i follow x, columns j follow y. Of column j the window keeps the cells on
// the diagonals i - j = -klo .. -klo + 32W: the value of the top one, T =
// D(j - klo, j), and the vertical differences of the 32W rows below it, bit b of
// P (+1) and M (-1) standing for row j + 1 - klo + b. The next column looks at
// the same bit for row (j+1) - klo + b, so the window moves down its diagonal
// without a shift of P and M: of the bit-vector recurrence for unit-cost edit
// distance (Myers 1999, Hyyro 2001) only the diagonal zero-difference vector D0
// is shifted, by one bit and in the other direction (Hyyro 2003, the diagonally
// tiled band). With E the match mask of rows j - klo + b against y[j-1]:
//     D0 = (((E & P) + P) ^ P) | E | M        HP = M | ~(D0 | P)   HN = D0 & P
//     P' = HN | ~((D0 >> 1) | HP)             M' = HP & (D0 >> 1)
// and T' = T + 1 - (D0 & 1). Ten 32-bit instructions per word (the match mask's
// own funnel shift included), as many as the block-aligned form needs, but the
// window holds exactly the band's diagonals in 32-bit words, where the block-
// aligned one has to hold 63 rows more in 64-bit words (K = 40: 2 words against
// 4; K = 150: 5 against 8; K = 250: 8 against 10).
//
// Boundaries. The cell above the window is never used (its horizontal difference
// enters as 0 or +1, an upper bound), the row entering at the bottom is the
// minimum of a substitution and of one more than the row above it, rows outside
// x never match, and rows above row 0 start at D(i, 0) = -i, so that D(0, j) = j.
// Every value is >= the true one and equal to it where that is <= K and its path
// stays on the window's diagonals.
//
// A common prefix of both strings changes neither the distance nor this state
// (the window of |i - j| maps to itself), so a half may start with any number of
// columns on which both strings are padded with the same symbol: the persistent
// verifier pads both halves of a pair to the same multiple of 32 columns, and no
// column of its loop needs a test.
#pragma once
#include "ej_bitpar.cuh"

namespace ej {

// S = A + Bv as one (32 W)-bit addition (the carry runs through the carry flag
// inside one asm block).
template <int W>
__device__ __forceinline__ void add_chain32(uint32_t (&S)[W], const uint32_t (&A)[W], const uint32_t (&Bv)[W]);
template <>
__device__ __forceinline__ void add_chain32<1>(uint32_t (&S)[1], const uint32_t (&A)[1], const uint32_t (&Bv)[1]) {
    S[0] = A[0] + Bv[0];
}
template <>
__device__ __forceinline__ void add_chain32<2>(uint32_t (&S)[2], const uint32_t (&A)[2], const uint32_t (&Bv)[2]) {
    asm("add.cc.u32 %0, %2, %4;\n\taddc.u32 %1, %3, %5;"
        : "=r"(S[0]), "=r"(S[1])
        : "r"(A[0]), "r"(A[1]), "r"(Bv[0]), "r"(Bv[1]));
}
template <>
__device__ __forceinline__ void add_chain32<3>(uint32_t (&S)[3], const uint32_t (&A)[3], const uint32_t (&Bv)[3]) {
    asm("add.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, %7;\n\taddc.u32 %2, %5, %8;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]));
}
template <>
__device__ __forceinline__ void add_chain32<4>(uint32_t (&S)[4], const uint32_t (&A)[4], const uint32_t (&Bv)[4]) {
    asm("add.cc.u32 %0, %4, %8;\n\taddc.cc.u32 %1, %5, %9;\n\taddc.cc.u32 %2, %6, %10;\n\taddc.u32 %3, %7, %11;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2]), "=r"(S[3])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]), "r"(Bv[3]));
}
template <>
__device__ __forceinline__ void add_chain32<5>(uint32_t (&S)[5], const uint32_t (&A)[5], const uint32_t (&Bv)[5]) {
    asm("add.cc.u32 %0, %5, %10;\n\taddc.cc.u32 %1, %6, %11;\n\taddc.cc.u32 %2, %7, %12;\n\taddc.cc.u32 %3, %8, %13;\n\taddc.u32 %4, %9, %14;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2]), "=r"(S[3]), "=r"(S[4])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(A[4]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]), "r"(Bv[3]), "r"(Bv[4]));
}
template <>
__device__ __forceinline__ void add_chain32<6>(uint32_t (&S)[6], const uint32_t (&A)[6], const uint32_t (&Bv)[6]) {
    asm("add.cc.u32 %0, %6, %12;\n\taddc.cc.u32 %1, %7, %13;\n\taddc.cc.u32 %2, %8, %14;\n\taddc.cc.u32 %3, %9, %15;\n\taddc.cc.u32 %4, %10, %16;\n\taddc.u32 %5, %11, %17;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2]), "=r"(S[3]), "=r"(S[4]), "=r"(S[5])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(A[4]), "r"(A[5]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]), "r"(Bv[3]), "r"(Bv[4]), "r"(Bv[5]));
}
template <>
__device__ __forceinline__ void add_chain32<7>(uint32_t (&S)[7], const uint32_t (&A)[7], const uint32_t (&Bv)[7]) {
    asm("add.cc.u32 %0, %7, %14;\n\taddc.cc.u32 %1, %8, %15;\n\taddc.cc.u32 %2, %9, %16;\n\taddc.cc.u32 %3, %10, %17;\n\taddc.cc.u32 %4, %11, %18;\n\taddc.cc.u32 %5, %12, %19;\n\taddc.u32 %6, %13, %20;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2]), "=r"(S[3]), "=r"(S[4]), "=r"(S[5]), "=r"(S[6])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(A[4]), "r"(A[5]), "r"(A[6]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]), "r"(Bv[3]), "r"(Bv[4]), "r"(Bv[5]), "r"(Bv[6]));
}
template <>
__device__ __forceinline__ void add_chain32<8>(uint32_t (&S)[8], const uint32_t (&A)[8], const uint32_t (&Bv)[8]) {
    asm("add.cc.u32 %0, %8, %16;\n\taddc.cc.u32 %1, %9, %17;\n\taddc.cc.u32 %2, %10, %18;\n\taddc.cc.u32 %3, %11, %19;\n\taddc.cc.u32 %4, %12, %20;\n\taddc.cc.u32 %5, %13, %21;\n\taddc.cc.u32 %6, %14, %22;\n\taddc.u32 %7, %15, %23;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2]), "=r"(S[3]), "=r"(S[4]), "=r"(S[5]), "=r"(S[6]), "=r"(S[7])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(A[4]), "r"(A[5]), "r"(A[6]), "r"(A[7]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]), "r"(Bv[3]), "r"(Bv[4]), "r"(Bv[5]), "r"(Bv[6]), "r"(Bv[7]));
}
template <>
__device__ __forceinline__ void add_chain32<9>(uint32_t (&S)[9], const uint32_t (&A)[9], const uint32_t (&Bv)[9]) {
    asm("add.cc.u32 %0, %9, %18;\n\taddc.cc.u32 %1, %10, %19;\n\taddc.cc.u32 %2, %11, %20;\n\taddc.cc.u32 %3, %12, %21;\n\taddc.cc.u32 %4, %13, %22;\n\taddc.cc.u32 %5, %14, %23;\n\taddc.cc.u32 %6, %15, %24;\n\taddc.cc.u32 %7, %16, %25;\n\taddc.u32 %8, %17, %26;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2]), "=r"(S[3]), "=r"(S[4]), "=r"(S[5]), "=r"(S[6]), "=r"(S[7]), "=r"(S[8])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(A[4]), "r"(A[5]), "r"(A[6]), "r"(A[7]), "r"(A[8]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]), "r"(Bv[3]), "r"(Bv[4]), "r"(Bv[5]), "r"(Bv[6]), "r"(Bv[7]), "r"(Bv[8]));
}
template <>
__device__ __forceinline__ void add_chain32<10>(uint32_t (&S)[10], const uint32_t (&A)[10], const uint32_t (&Bv)[10]) {
    asm("add.cc.u32 %0, %10, %20;\n\taddc.cc.u32 %1, %11, %21;\n\taddc.cc.u32 %2, %12, %22;\n\taddc.cc.u32 %3, %13, %23;\n\taddc.cc.u32 %4, %14, %24;\n\taddc.cc.u32 %5, %15, %25;\n\taddc.cc.u32 %6, %16, %26;\n\taddc.cc.u32 %7, %17, %27;\n\taddc.cc.u32 %8, %18, %28;\n\taddc.u32 %9, %19, %29;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2]), "=r"(S[3]), "=r"(S[4]), "=r"(S[5]), "=r"(S[6]), "=r"(S[7]), "=r"(S[8]), "=r"(S[9])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(A[4]), "r"(A[5]), "r"(A[6]), "r"(A[7]), "r"(A[8]), "r"(A[9]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]), "r"(Bv[3]), "r"(Bv[4]), "r"(Bv[5]), "r"(Bv[6]), "r"(Bv[7]), "r"(Bv[8]), "r"(Bv[9]));
}
template <>
__device__ __forceinline__ void add_chain32<11>(uint32_t (&S)[11], const uint32_t (&A)[11], const uint32_t (&Bv)[11]) {
    asm("add.cc.u32 %0, %11, %22;\n\taddc.cc.u32 %1, %12, %23;\n\taddc.cc.u32 %2, %13, %24;\n\taddc.cc.u32 %3, %14, %25;\n\taddc.cc.u32 %4, %15, %26;\n\taddc.cc.u32 %5, %16, %27;\n\taddc.cc.u32 %6, %17, %28;\n\taddc.cc.u32 %7, %18, %29;\n\taddc.cc.u32 %8, %19, %30;\n\taddc.cc.u32 %9, %20, %31;\n\taddc.u32 %10, %21, %32;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2]), "=r"(S[3]), "=r"(S[4]), "=r"(S[5]), "=r"(S[6]), "=r"(S[7]), "=r"(S[8]), "=r"(S[9]), "=r"(S[10])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(A[4]), "r"(A[5]), "r"(A[6]), "r"(A[7]), "r"(A[8]), "r"(A[9]), "r"(A[10]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]), "r"(Bv[3]), "r"(Bv[4]), "r"(Bv[5]), "r"(Bv[6]), "r"(Bv[7]), "r"(Bv[8]), "r"(Bv[9]), "r"(Bv[10]));
}
template <>
__device__ __forceinline__ void add_chain32<12>(uint32_t (&S)[12], const uint32_t (&A)[12], const uint32_t (&Bv)[12]) {
    asm("add.cc.u32 %0, %12, %24;\n\taddc.cc.u32 %1, %13, %25;\n\taddc.cc.u32 %2, %14, %26;\n\taddc.cc.u32 %3, %15, %27;\n\taddc.cc.u32 %4, %16, %28;\n\taddc.cc.u32 %5, %17, %29;\n\taddc.cc.u32 %6, %18, %30;\n\taddc.cc.u32 %7, %19, %31;\n\taddc.cc.u32 %8, %20, %32;\n\taddc.cc.u32 %9, %21, %33;\n\taddc.cc.u32 %10, %22, %34;\n\taddc.u32 %11, %23, %35;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2]), "=r"(S[3]), "=r"(S[4]), "=r"(S[5]), "=r"(S[6]), "=r"(S[7]), "=r"(S[8]), "=r"(S[9]), "=r"(S[10]), "=r"(S[11])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(A[4]), "r"(A[5]), "r"(A[6]), "r"(A[7]), "r"(A[8]), "r"(A[9]), "r"(A[10]), "r"(A[11]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]), "r"(Bv[3]), "r"(Bv[4]), "r"(Bv[5]), "r"(Bv[6]), "r"(Bv[7]), "r"(Bv[8]), "r"(Bv[9]), "r"(Bv[10]), "r"(Bv[11]));
}
template <>
__device__ __forceinline__ void add_chain32<14>(uint32_t (&S)[14], const uint32_t (&A)[14], const uint32_t (&Bv)[14]) {
    asm("add.cc.u32 %0, %14, %28;\n\taddc.cc.u32 %1, %15, %29;\n\taddc.cc.u32 %2, %16, %30;\n\taddc.cc.u32 %3, %17, %31;\n\taddc.cc.u32 %4, %18, %32;\n\taddc.cc.u32 %5, %19, %33;\n\taddc.cc.u32 %6, %20, %34;\n\taddc.cc.u32 %7, %21, %35;\n\taddc.cc.u32 %8, %22, %36;\n\taddc.cc.u32 %9, %23, %37;\n\taddc.cc.u32 %10, %24, %38;\n\taddc.cc.u32 %11, %25, %39;\n\taddc.cc.u32 %12, %26, %40;\n\taddc.u32 %13, %27, %41;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2]), "=r"(S[3]), "=r"(S[4]), "=r"(S[5]), "=r"(S[6]), "=r"(S[7]), "=r"(S[8]), "=r"(S[9]), "=r"(S[10]), "=r"(S[11]), "=r"(S[12]), "=r"(S[13])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(A[4]), "r"(A[5]), "r"(A[6]), "r"(A[7]), "r"(A[8]), "r"(A[9]), "r"(A[10]), "r"(A[11]), "r"(A[12]), "r"(A[13]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]), "r"(Bv[3]), "r"(Bv[4]), "r"(Bv[5]), "r"(Bv[6]), "r"(Bv[7]), "r"(Bv[8]), "r"(Bv[9]), "r"(Bv[10]), "r"(Bv[11]), "r"(Bv[12]), "r"(Bv[13]));
}
template <>
__device__ __forceinline__ void add_chain32<16>(uint32_t (&S)[16], const uint32_t (&A)[16], const uint32_t (&Bv)[16]) {
    asm("add.cc.u32 %0, %16, %32;\n\taddc.cc.u32 %1, %17, %33;\n\taddc.cc.u32 %2, %18, %34;\n\taddc.cc.u32 %3, %19, %35;\n\taddc.cc.u32 %4, %20, %36;\n\taddc.cc.u32 %5, %21, %37;\n\taddc.cc.u32 %6, %22, %38;\n\taddc.cc.u32 %7, %23, %39;\n\taddc.cc.u32 %8, %24, %40;\n\taddc.cc.u32 %9, %25, %41;\n\taddc.cc.u32 %10, %26, %42;\n\taddc.cc.u32 %11, %27, %43;\n\taddc.cc.u32 %12, %28, %44;\n\taddc.cc.u32 %13, %29, %45;\n\taddc.cc.u32 %14, %30, %46;\n\taddc.u32 %15, %31, %47;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2]), "=r"(S[3]), "=r"(S[4]), "=r"(S[5]), "=r"(S[6]), "=r"(S[7]), "=r"(S[8]), "=r"(S[9]), "=r"(S[10]), "=r"(S[11]), "=r"(S[12]), "=r"(S[13]), "=r"(S[14]), "=r"(S[15])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(A[4]), "r"(A[5]), "r"(A[6]), "r"(A[7]), "r"(A[8]), "r"(A[9]), "r"(A[10]), "r"(A[11]), "r"(A[12]), "r"(A[13]), "r"(A[14]), "r"(A[15]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]), "r"(Bv[3]), "r"(Bv[4]), "r"(Bv[5]), "r"(Bv[6]), "r"(Bv[7]), "r"(Bv[8]), "r"(Bv[9]), "r"(Bv[10]), "r"(Bv[11]), "r"(Bv[12]), "r"(Bv[13]), "r"(Bv[14]), "r"(Bv[15]));
}
template <>
__device__ __forceinline__ void add_chain32<18>(uint32_t (&S)[18], const uint32_t (&A)[18], const uint32_t (&Bv)[18]) {
    asm("add.cc.u32 %0, %18, %36;\n\taddc.cc.u32 %1, %19, %37;\n\taddc.cc.u32 %2, %20, %38;\n\taddc.cc.u32 %3, %21, %39;\n\taddc.cc.u32 %4, %22, %40;\n\taddc.cc.u32 %5, %23, %41;\n\taddc.cc.u32 %6, %24, %42;\n\taddc.cc.u32 %7, %25, %43;\n\taddc.cc.u32 %8, %26, %44;\n\taddc.cc.u32 %9, %27, %45;\n\taddc.cc.u32 %10, %28, %46;\n\taddc.cc.u32 %11, %29, %47;\n\taddc.cc.u32 %12, %30, %48;\n\taddc.cc.u32 %13, %31, %49;\n\taddc.cc.u32 %14, %32, %50;\n\taddc.cc.u32 %15, %33, %51;\n\taddc.cc.u32 %16, %34, %52;\n\taddc.u32 %17, %35, %53;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2]), "=r"(S[3]), "=r"(S[4]), "=r"(S[5]), "=r"(S[6]), "=r"(S[7]), "=r"(S[8]), "=r"(S[9]), "=r"(S[10]), "=r"(S[11]), "=r"(S[12]), "=r"(S[13]), "=r"(S[14]), "=r"(S[15]), "=r"(S[16]), "=r"(S[17])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(A[4]), "r"(A[5]), "r"(A[6]), "r"(A[7]), "r"(A[8]), "r"(A[9]), "r"(A[10]), "r"(A[11]), "r"(A[12]), "r"(A[13]), "r"(A[14]), "r"(A[15]), "r"(A[16]), "r"(A[17]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]), "r"(Bv[3]), "r"(Bv[4]), "r"(Bv[5]), "r"(Bv[6]), "r"(Bv[7]), "r"(Bv[8]), "r"(Bv[9]), "r"(Bv[10]), "r"(Bv[11]), "r"(Bv[12]), "r"(Bv[13]), "r"(Bv[14]), "r"(Bv[15]), "r"(Bv[16]), "r"(Bv[17]));
}
template <>
__device__ __forceinline__ void add_chain32<20>(uint32_t (&S)[20], const uint32_t (&A)[20], const uint32_t (&Bv)[20]) {
    asm("add.cc.u32 %0, %20, %40;\n\taddc.cc.u32 %1, %21, %41;\n\taddc.cc.u32 %2, %22, %42;\n\taddc.cc.u32 %3, %23, %43;\n\taddc.cc.u32 %4, %24, %44;\n\taddc.cc.u32 %5, %25, %45;\n\taddc.cc.u32 %6, %26, %46;\n\taddc.cc.u32 %7, %27, %47;\n\taddc.cc.u32 %8, %28, %48;\n\taddc.cc.u32 %9, %29, %49;\n\taddc.cc.u32 %10, %30, %50;\n\taddc.cc.u32 %11, %31, %51;\n\taddc.cc.u32 %12, %32, %52;\n\taddc.cc.u32 %13, %33, %53;\n\taddc.cc.u32 %14, %34, %54;\n\taddc.cc.u32 %15, %35, %55;\n\taddc.cc.u32 %16, %36, %56;\n\taddc.cc.u32 %17, %37, %57;\n\taddc.cc.u32 %18, %38, %58;\n\taddc.u32 %19, %39, %59;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2]), "=r"(S[3]), "=r"(S[4]), "=r"(S[5]), "=r"(S[6]), "=r"(S[7]), "=r"(S[8]), "=r"(S[9]), "=r"(S[10]), "=r"(S[11]), "=r"(S[12]), "=r"(S[13]), "=r"(S[14]), "=r"(S[15]), "=r"(S[16]), "=r"(S[17]), "=r"(S[18]), "=r"(S[19])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(A[4]), "r"(A[5]), "r"(A[6]), "r"(A[7]), "r"(A[8]), "r"(A[9]), "r"(A[10]), "r"(A[11]), "r"(A[12]), "r"(A[13]), "r"(A[14]), "r"(A[15]), "r"(A[16]), "r"(A[17]), "r"(A[18]), "r"(A[19]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]), "r"(Bv[3]), "r"(Bv[4]), "r"(Bv[5]), "r"(Bv[6]), "r"(Bv[7]), "r"(Bv[8]), "r"(Bv[9]), "r"(Bv[10]), "r"(Bv[11]), "r"(Bv[12]), "r"(Bv[13]), "r"(Bv[14]), "r"(Bv[15]), "r"(Bv[16]), "r"(Bv[17]), "r"(Bv[18]), "r"(Bv[19]));
}
template <>
__device__ __forceinline__ void add_chain32<22>(uint32_t (&S)[22], const uint32_t (&A)[22], const uint32_t (&Bv)[22]) {
    asm("add.cc.u32 %0, %22, %44;\n\taddc.cc.u32 %1, %23, %45;\n\taddc.cc.u32 %2, %24, %46;\n\taddc.cc.u32 %3, %25, %47;\n\taddc.cc.u32 %4, %26, %48;\n\taddc.cc.u32 %5, %27, %49;\n\taddc.cc.u32 %6, %28, %50;\n\taddc.cc.u32 %7, %29, %51;\n\taddc.cc.u32 %8, %30, %52;\n\taddc.cc.u32 %9, %31, %53;\n\taddc.cc.u32 %10, %32, %54;\n\taddc.cc.u32 %11, %33, %55;\n\taddc.cc.u32 %12, %34, %56;\n\taddc.cc.u32 %13, %35, %57;\n\taddc.cc.u32 %14, %36, %58;\n\taddc.cc.u32 %15, %37, %59;\n\taddc.cc.u32 %16, %38, %60;\n\taddc.cc.u32 %17, %39, %61;\n\taddc.cc.u32 %18, %40, %62;\n\taddc.cc.u32 %19, %41, %63;\n\taddc.cc.u32 %20, %42, %64;\n\taddc.u32 %21, %43, %65;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2]), "=r"(S[3]), "=r"(S[4]), "=r"(S[5]), "=r"(S[6]), "=r"(S[7]), "=r"(S[8]), "=r"(S[9]), "=r"(S[10]), "=r"(S[11]), "=r"(S[12]), "=r"(S[13]), "=r"(S[14]), "=r"(S[15]), "=r"(S[16]), "=r"(S[17]), "=r"(S[18]), "=r"(S[19]), "=r"(S[20]), "=r"(S[21])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(A[4]), "r"(A[5]), "r"(A[6]), "r"(A[7]), "r"(A[8]), "r"(A[9]), "r"(A[10]), "r"(A[11]), "r"(A[12]), "r"(A[13]), "r"(A[14]), "r"(A[15]), "r"(A[16]), "r"(A[17]), "r"(A[18]), "r"(A[19]), "r"(A[20]), "r"(A[21]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]), "r"(Bv[3]), "r"(Bv[4]), "r"(Bv[5]), "r"(Bv[6]), "r"(Bv[7]), "r"(Bv[8]), "r"(Bv[9]), "r"(Bv[10]), "r"(Bv[11]), "r"(Bv[12]), "r"(Bv[13]), "r"(Bv[14]), "r"(Bv[15]), "r"(Bv[16]), "r"(Bv[17]), "r"(Bv[18]), "r"(Bv[19]), "r"(Bv[20]), "r"(Bv[21]));
}
template <>
__device__ __forceinline__ void add_chain32<24>(uint32_t (&S)[24], const uint32_t (&A)[24], const uint32_t (&Bv)[24]) {
    asm("add.cc.u32 %0, %24, %48;\n\taddc.cc.u32 %1, %25, %49;\n\taddc.cc.u32 %2, %26, %50;\n\taddc.cc.u32 %3, %27, %51;\n\taddc.cc.u32 %4, %28, %52;\n\taddc.cc.u32 %5, %29, %53;\n\taddc.cc.u32 %6, %30, %54;\n\taddc.cc.u32 %7, %31, %55;\n\taddc.cc.u32 %8, %32, %56;\n\taddc.cc.u32 %9, %33, %57;\n\taddc.cc.u32 %10, %34, %58;\n\taddc.cc.u32 %11, %35, %59;\n\taddc.cc.u32 %12, %36, %60;\n\taddc.cc.u32 %13, %37, %61;\n\taddc.cc.u32 %14, %38, %62;\n\taddc.cc.u32 %15, %39, %63;\n\taddc.cc.u32 %16, %40, %64;\n\taddc.cc.u32 %17, %41, %65;\n\taddc.cc.u32 %18, %42, %66;\n\taddc.cc.u32 %19, %43, %67;\n\taddc.cc.u32 %20, %44, %68;\n\taddc.cc.u32 %21, %45, %69;\n\taddc.cc.u32 %22, %46, %70;\n\taddc.u32 %23, %47, %71;"
        : "=r"(S[0]), "=r"(S[1]), "=r"(S[2]), "=r"(S[3]), "=r"(S[4]), "=r"(S[5]), "=r"(S[6]), "=r"(S[7]), "=r"(S[8]), "=r"(S[9]), "=r"(S[10]), "=r"(S[11]), "=r"(S[12]), "=r"(S[13]), "=r"(S[14]), "=r"(S[15]), "=r"(S[16]), "=r"(S[17]), "=r"(S[18]), "=r"(S[19]), "=r"(S[20]), "=r"(S[21]), "=r"(S[22]), "=r"(S[23])
        : "r"(A[0]), "r"(A[1]), "r"(A[2]), "r"(A[3]), "r"(A[4]), "r"(A[5]), "r"(A[6]), "r"(A[7]), "r"(A[8]), "r"(A[9]), "r"(A[10]), "r"(A[11]), "r"(A[12]), "r"(A[13]), "r"(A[14]), "r"(A[15]), "r"(A[16]), "r"(A[17]), "r"(A[18]), "r"(A[19]), "r"(A[20]), "r"(A[21]), "r"(A[22]), "r"(A[23]), "r"(Bv[0]), "r"(Bv[1]), "r"(Bv[2]), "r"(Bv[3]), "r"(Bv[4]), "r"(Bv[5]), "r"(Bv[6]), "r"(Bv[7]), "r"(Bv[8]), "r"(Bv[9]), "r"(Bv[10]), "r"(Bv[11]), "r"(Bv[12]), "r"(Bv[13]), "r"(Bv[14]), "r"(Bv[15]), "r"(Bv[16]), "r"(Bv[17]), "r"(Bv[18]), "r"(Bv[19]), "r"(Bv[20]), "r"(Bv[21]), "r"(Bv[22]), "r"(Bv[23]));
}

// One column. row: the match words of the column's symbol from the window's
// first word on, `stride` entries apart (W + 1 words); sh: (j - 1) mod 32. The
// low bits of D0 (1: T unchanged) enter tacc from the top.
template <int W>
__device__ __forceinline__ void diag_step(uint32_t (&P)[W], uint32_t (&M)[W], uint32_t &tacc,
                                          const uint32_t *__restrict__ row, int stride, uint32_t sh) {
    uint32_t r[W + 1], E[W], A[W], S[W];
#pragma unroll
    for (int v = 0; v <= W; v++) r[v] = row[v * stride];
#pragma unroll
    for (int v = 0; v < W; v++) {
        E[v] = __funnelshift_r(r[v], r[v + 1], sh);
        A[v] = E[v] & P[v];
    }
    add_chain32<W>(S, A, P);
    uint32_t U[W], D[W];
#pragma unroll
    for (int v = 0; v < W; v++) {
        U[v] = (S[v] ^ P[v]) | E[v];
        D[v] = U[v] | M[v];
    }
    tacc = __funnelshift_r(tacc, D[0], 1);
#pragma unroll
    for (int v = 0; v < W; v++) {
        const uint32_t D1 = v + 1 < W ? __funnelshift_r(D[v], D[v + 1 < W ? v + 1 : v], 1) : D[v] >> 1;
        const uint32_t HP = M[v] | ~(U[v] | P[v]);
        const uint32_t HN = U[v] & P[v];   // P and M have no common bit
        P[v] = HN | ~(D1 | HP);
        M[v] = HP & D1;
    }
}

// The window before column 1: rows 1 - klo .. 0 one less, rows from 1 on one
// more than the row above; T = klo.
template <int W>
__device__ __forceinline__ void diag_init(uint32_t (&P)[W], uint32_t (&M)[W], int32_t klo) {
#pragma unroll
    for (int v = 0; v < W; v++) {
        const int nb = klo - 32 * v;
        M[v] = nb <= 0 ? 0u : nb >= 32 ? ~0u : (1u << nb) - 1u;
        P[v] = ~M[v];
    }
}

// Nibble table of diag_min, 256 entries in shared memory: of the four rows with
// P bits idx & 15 and M bits idx >> 4 the sum of the differences (low half) and
// their smallest prefix sum (high half).
__device__ __forceinline__ void diag_fill_table(uint32_t *tab) {
    for (int t = threadIdx.x; t < 256; t += blockDim.x) {
        const uint32_t P = t & 15u, M = t >> 4;
        int run = 0, mn = 1 << 14;
        for (int k = 0; k < 4; k++) {
            run += (int)((P >> k) & 1u) - (int)((M >> k) & 1u);
            mn = run < mn ? run : mn;
        }
        tab[t] = ((uint32_t)mn << 16) | ((uint32_t)run & 0xFFFFu);
    }
}

// Minimum of the window minus T (at most 0: the top cell takes part). Two 16-bit
// lanes per register: the running sum twice, against the entry's (prefix
// minimum, sum), with the minimum so far as the bound of the high lane.
template <int W>
__device__ __forceinline__ int32_t diag_min(const uint32_t (&P)[W], const uint32_t (&M)[W], const uint32_t *tab) {
    uint32_t run2 = 0, bound = 0x00007FFFu;   // (minimum so far, no bound)
#pragma unroll
    for (int v = 0; v < W; v++) {
        const uint32_t even = (P[v] & 0x0F0F0F0Fu) | ((M[v] & 0x0F0F0F0Fu) << 4);
        const uint32_t odd = ((P[v] >> 4) & 0x0F0F0F0Fu) | (M[v] & 0xF0F0F0F0u);
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const uint32_t idx = __byte_perm((k & 1) ? odd : even, 0u, 0x4440 | (k >> 1));
            const uint32_t x = __viaddmin_s16x2(run2, tab[idx], bound);
            run2 = __byte_perm(x, 0u, 0x1010);
            bound = (x & 0xFFFF0000u) | 0x7FFFu;
        }
    }
    return (int32_t)bound >> 16;
}

// The same minimum as the return value, and *alive: whether some row may lie on an
// alignment of cost <= K, judged per half word: T + its minimum + the distance of
// the half's rows (16 h + 1 .. 16 h + 16 below the top cell, which counts to half 0)
// to the diagonal on which the alignment ends, rt rows below the top cell, is <= K.
// On every alignment of cost <= K there is such a row, and random strings run out
// of them about 7% of the columns before the plain minimum exceeds K.
template <int W>
__device__ __forceinline__ int32_t diag_alive(const uint32_t (&P)[W], const uint32_t (&M)[W], const uint32_t *tab,
                                              int32_t T, int32_t rt, int32_t K, bool *alive) {
    uint32_t run2 = 0;
    int32_t low = 0, best = 0x7FFFFFFF;   // smallest minimum, smallest minimum + distance
#pragma unroll
    for (int v = 0; v < W; v++) {
        const uint32_t even = (P[v] & 0x0F0F0F0Fu) | ((M[v] & 0x0F0F0F0Fu) << 4);
        const uint32_t odd = ((P[v] >> 4) & 0x0F0F0F0Fu) | (M[v] & 0xF0F0F0F0u);
#pragma unroll
        for (int h = 0; h < 2; h++) {
            uint32_t bound = v + h == 0 ? 0x00007FFFu : 0x7FFF7FFFu;
#pragma unroll
            for (int k = 4 * h; k < 4 * h + 4; k++) {
                const uint32_t idx = __byte_perm((k & 1) ? odd : even, 0u, 0x4440 | (k >> 1));
                const uint32_t x = __viaddmin_s16x2(run2, tab[idx], bound);
                run2 = __byte_perm(x, 0u, 0x1010);
                bound = (x & 0xFFFF0000u) | 0x7FFFu;
            }
            const int32_t mn = (int32_t)bound >> 16;
            low = min(low, mn);
            const int first = 32 * v + 16 * h + (v + h == 0 ? 0 : 1), last = 32 * v + 16 * h + 16;
            best = min(best, mn + max(max(first - rt, rt - last), 0));
        }
    }
    *alive = T + best <= K;
    return low;
}

// Sum of the differences of the first `cnt` rows of a dumped window (entries v
// and W + v, `stride` apart: words v of P and M).
template <int W>
__device__ __forceinline__ int32_t diag_prefix(const uint32_t *d, int stride, int32_t cnt) {
    int32_t acc = 0;
    for (int v = 0; v < W; v++) {
        const int32_t left = cnt - 32 * v;
        if (left <= 0) break;
        const uint32_t msk = left >= 32 ? ~0u : (1u << left) - 1u;
        acc += __popc(d[v * stride] & msk) - __popc(d[(W + v) * stride] & msk);
    }
    return acc;
}

// min_i F(i) + B(m - i) over the rows i that both dumped windows hold (the
// forward one at column n1, the backward one at column n2 of the reversed
// strings); `part` 0 / 1: the upper / lower half of those rows (the two lanes of
// a pair share the work). INT_MAX when there is none.
template <int W>
__device__ __forceinline__ int32_t diag_meet(const uint32_t *f, const uint32_t *b, int stride, int32_t m, int32_t n1,
                                             int32_t n2, int32_t klo, int part) {
    const int32_t rf = n1 - klo, rb = n2 - klo;   // rows of the two top cells
    int32_t lo = max(max(rf, m - (rb + 32 * W)), 0), hi = min(min(rf + 32 * W, m - rb), m);
    int32_t best = 0x7FFFFFFF;
    if (lo > hi) return best;
    const int32_t mid = (lo + hi) >> 1;
    if (part) lo = mid;
    else hi = mid;
    int32_t F = (int32_t)f[2 * W * stride] + diag_prefix<W>(f, stride, lo - rf);
    int32_t G = (int32_t)b[2 * W * stride] + diag_prefix<W>(b, stride, m - lo - rb);
    best = F + G;
    for (int32_t i = lo; i < hi; i++) {
        const uint32_t qf = (uint32_t)(i - rf), qb = (uint32_t)(m - i - 1 - rb);
        const int wf = (int)(qf >> 5) * stride, wb = (int)(qb >> 5) * stride;
        F += (int32_t)((f[wf] >> (qf & 31u)) & 1u) - (int32_t)((f[W * stride + wf] >> (qf & 31u)) & 1u);
        G -= (int32_t)((b[wb] >> (qb & 31u)) & 1u) - (int32_t)((b[W * stride + wb] >> (qb & 31u)) & 1u);
        best = min(best, F + G);
    }
    return best;
}

// Words of P, M and T as diag_prefix / diag_meet read them.
template <int W>
__device__ __forceinline__ void diag_dump(uint32_t *d, int stride, const uint32_t (&P)[W], const uint32_t (&M)[W],
                                          int32_t T) {
#pragma unroll
    for (int v = 0; v < W; v++) {
        d[v * stride] = P[v];
        d[(W + v) * stride] = M[v];
    }
    d[2 * W * stride] = (uint32_t)T;
}

}  // namespace ej
