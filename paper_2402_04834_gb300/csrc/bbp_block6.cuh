// The fused block update of a full 6 x 6 block (k = 6, d = 31's blocks), one
// coset per warp: the sums and roundings of fused_sweep's node-by-node passes
// (bbp_fused.cuh), column by column in registers.
//
// As in the 4 x 4 register form (bbp_reg.cuh), along a column the checks tie
// the chain legs to row bits, so a column is three 2-point XOR butterflies
// over the qubits' row bits.  A lane takes the rows that differ in those
// three bits (eight entries in registers) for one assignment of the check
// bits and open side legs, so a column is one pass over shared memory where
// the node-by-node form makes five (side message, three node pairs, side
// message).  Side legs that a check ties to a row bit are not stored, and
// where a qubit's in-leg is such a leg its factor is one of two constants, so
// only the two scaled copies ("E" for pi(X), "I" for pi(I)) are carried in
// place of the four combinations: at most 1024 entries a buffer instead of
// 4096 (16 warps per SM instead of 6).  The node-by-node form issued 12,300
// warp instructions an update with 6 warps per SM; this one issues 2,900 with
// 16, and its loops are kept rolled so that both forms stay in the
// instruction cache (unrolled it took 75 ms, waiting for instructions).  152
// syndromes at d = 31, p = 0.12: 102.4 -> 28.8 ms.
//
// Rounding follows the node-by-node form exactly: a butterfly's two terms
// are one product and one multiply-add, and which of the two is fused depends
// on how that form pairs the nodes of a column (bf's `own`); the messages of
// both forms are the same bits.
// Only blocks whose nodes, but for the first column's and the top row's, are
// inside the grid come here: full blocks always are, since the grid's side is
// odd.
#pragma once

#include "bbp_reg.cuh"

namespace bbp {

constexpr int kBlock6Buf = 1024;             // entries of each of the two state buffers

template <typename T>
struct Block6 {
  T* A;                                      // state buffers; the outgoing vector ends in A[0 .. 63]
  T* B;
  const T* mt;                               // side messages in consumption order, 64 entries each
  const T* mb;
  const T* in;                               // message opposite the outgoing side, or null on the grid border
  T pI, pE;
  bool a;                                    // the upper side has a message (the lower always has)
  bool chk0;                                 // column 0 starts with a check
  int ids;                                   // lane 3 t + u: id (alpha, beta) of qubit u of column t
  int lane;

  __device__ __forceinline__ int id(int t, int u) const { return __shfl_sync(kFull, ids, 3 * t + u); }
  __device__ __forceinline__ T g(int id, int al, int be) const { return id == ((al << 1) | be) ? pI : pE; }
  // Row index of chain bits s0 .. s5.
  static __device__ __forceinline__ int row(int s0, int s1, int s2, int s3, int s4, int s5) {
    return (s0 << 5) | (s1 << 4) | (s2 << 3) | (s3 << 2) | (s4 << 1) | s5;
  }
  // Butterfly over bit BIT of the entry index of e[N]; own: where the pair is
  // taken check first, output 0 fuses its own input's product (x0), otherwise
  // output 0 fuses x1; output 1 fuses x1 in both.
  template <int N, int BIT>
  __device__ __forceinline__ void bf(T (&e)[N], int id, int be, bool own) const {
    const T g0 = g(id, 0, be), g1 = g(id, 1, be);
#pragma unroll
    for (int i = 0; i < N; ++i)
      if (!(i & BIT)) {
        const T x0 = e[i], x1 = e[i | BIT];
        if (own) e[i] = fma(x0, g0, x1 * g1);
        else e[i] = fma(x1, g1, x0 * g0);
        e[i | BIT] = fma(x1, g0, x0 * g1);
      }
  }
  // Four products, and the lower message's steps, in the roundings of the
  // node-by-node form's expressions as compiled.
  static __device__ __forceinline__ T dot4(T a0, T c0, T a1, T c1, T a2, T c2, T a3, T c3) {
    return fma(a3, c3, fma(a2, c2, fma(a0, c0, a1 * c1)));
  }
  static __device__ __forceinline__ T dot2(T v, T m0, T x0, T m1, T x1) {
    return radd(v, fma(m0, x0, m1 * x1));
  }
  static __device__ __forceinline__ T dot1(T v, T m, T x) {    // dot2 with one of its products zero
    return radd(v, m * x);
  }
  // First qubit of a column with its upper leg u summed: y[r] over l, u of
  // x[u][l] g[l ^ r][u ^ r1], the four terms in the order (l, u) = 00, 01, 10, 11.
  __device__ __forceinline__ void bf4(const T (&x0)[8], const T (&x1)[8], int id, int r1, T (&y)[8]) const {
    const T g00 = g(id, 0, r1), g01 = g(id, 0, r1 ^ 1), g10 = g(id, 1, r1), g11 = g(id, 1, r1 ^ 1);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      y[i] = dot4(x0[i], g00, x1[i], g01, x0[4 + i], g10, x1[4 + i], g11);
      y[4 + i] = dot4(x0[i], g10, x1[i], g11, x0[4 + i], g00, x1[4 + i], g01);
    }
  }
  __device__ __forceinline__ T start(int H, int qubits) const { return in ? in[H] : ((H & qubits) ? T(0) : T(1)); }

  // Columns Q (qubits at chain positions 0, 2, 4) and C (1, 3, 5) in turn,
  // beginning with Q.
  __device__ __forceinline__ void run_q() const {
    const int b4 = (lane >> 4) & 1, b3 = (lane >> 3) & 1, b2 = (lane >> 2) & 1, b1 = (lane >> 1) & 1, b0 = lane & 1;
    T e[8];
    {  // t = 0 (Q): a0 = u recorded, b0 tied to r5.  A[a0][row]
      const int a0 = a ? b3 : 0, r1 = b2, r3 = b1, r5 = b0;
#pragma unroll
      for (int i = 0; i < 8; ++i) e[i] = start(row(i >> 2, r1, ((i >> 1) & 1), r3, (i & 1), r5), 42);
      bf<8, 4>(e, id(0, 0), a0 ^ r1, false);
      bf<8, 2>(e, id(0, 1), r1 ^ r3, !a);
      bf<8, 1>(e, id(0, 2), r3 ^ r5, !a);
      if (lane < (a ? 16 : 8))
#pragma unroll
        for (int i = 0; i < 8; ++i) A[64 * a0 + row(i >> 2, r1, ((i >> 1) & 1), r3, (i & 1), r5)] = e[i];
    }
    __syncwarp();
    {  // t = 1 (C): a1 tied to r0, l5 = b0, b1 = w recorded.  B[a0][row][b0][b1]
      const int a0 = a ? b4 : 0, w = b3, r0 = b2, r2 = b1, r4 = b0;
#pragma unroll
      for (int i = 0; i < 8; ++i) e[i] = A[64 * a0 + row(r0, (i >> 2), r2, ((i >> 1) & 1), r4, i & 1)];
      bf<8, 4>(e, id(1, 0), r0 ^ r2, a);
      bf<8, 2>(e, id(1, 1), r2 ^ r4, a);
      const int i5 = id(1, 2);
      const T g0 = g(i5, 0, r4 ^ w), g1 = g(i5, 1, r4 ^ w);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int l5 = i & 1, at = 64 * a0 + row(r0, (i >> 2), r2, ((i >> 1) & 1), r4, 0);
        B[4 * at + 2 * l5 + w] = e[i] * (l5 ? g1 : g0);              // r5 = 0
        B[4 * (at + 1) + 2 * l5 + w] = e[i] * (l5 ? g0 : g1);        // r5 = 1
      }
    }
    __syncwarp();
    const int i20 = id(2, 0);
    {  // t = 2 (Q): l0 = a1, a2 = u recorded, b2 tied to r5.
      const int r1 = b4, r3 = b3, r5 = b2, bb = lane & 3;
      const int i1 = id(2, 1), i2 = id(2, 2);
      if (!a) {  // A[row][b0 b1]
#pragma unroll
        for (int i = 0; i < 8; ++i) e[i] = B[4 * row(i >> 2, r1, ((i >> 1) & 1), r3, (i & 1), r5) + bb];
        bf<8, 4>(e, i20, r1, false);
        bf<8, 2>(e, i1, r1 ^ r3, true);
        bf<8, 1>(e, i2, r3 ^ r5, true);
#pragma unroll
        for (int i = 0; i < 8; ++i) A[4 * row(i >> 2, r1, ((i >> 1) & 1), r3, (i & 1), r5) + bb] = e[i];
      }
      // A[a0][a1][E / I][row without r0][b0 b1]
#pragma unroll 1
      for (int a01 = 0; a01 < (a ? 4 : 0); ++a01) {
        T x[4], y[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const T v = B[4 * (64 * (a01 >> 1) + row(a01 & 1, r1, (i >> 1), r3, (i & 1), r5)) + bb];
          x[i] = pE * v;
          y[i] = pI * v;
        }
        bf<4, 2>(x, i1, r1 ^ r3, false);
        bf<4, 1>(x, i2, r3 ^ r5, false);
        bf<4, 2>(y, i1, r1 ^ r3, false);
        bf<4, 1>(y, i2, r3 ^ r5, false);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int at = row(0, r1, (i >> 1), r3, (i & 1), r5);
          A[4 * (64 * a01 + at) + bb] = x[i];
          A[4 * (64 * a01 + 32 + at) + bb] = y[i];
        }
      }
    }
    __syncwarp();
    // t = 3 (C), the data column: the upper message over a (v = r0) leaves
    // its legs 4, 5 (al), qubits 1 and 3, then l5 = b2 and the lower message
    // over b and w.
    {  // B[al][r0 .. r4][b2][b0 b1]
      const int r0 = b4, r2 = b3, r4 = b2, bb = lane & 3;
      const int i1 = id(3, 0), i3 = id(3, 1);
      const int hb = i20 & 1, ha = i20 >> 1;
      T acc[4][8];
#pragma unroll
      for (int al = 0; al < 4; ++al)
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[al][i] = T(0);
      if (!a) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          acc[0][i] = A[4 * row(r0, (i >> 2), r2, ((i >> 1) & 1), r4, i & 1) + bb];
      }
#pragma unroll 1
      for (int a01 = 0; a01 < (a ? 4 : 0); ++a01) {
        const bool hit = r0 == (ha ^ (a01 & 1));
        T m0[4], m1[4];                      // a2 = 0, 1
        vcopy4(mt + 4 * (4 * a01 + r0), m0);
        vcopy4(mt + 4 * (4 * a01 + 2 + r0), m1);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int l1 = i >> 2;
          const int at = 64 * a01 + row(0, l1, r2, ((i >> 1) & 1), r4, i & 1);
          const T x = A[4 * at + bb], y = A[4 * (at + 32) + bb];
          const T x0 = hit && l1 == hb ? y : x;                // a2 = 0
          const T x1 = hit && l1 != hb ? y : x;                // a2 = 1
#pragma unroll
          for (int al = 0; al < 4; ++al) acc[al][i] = fma(m1[al], x1, fma(m0[al], x0, acc[al][i]));
        }
      }
#pragma unroll
      for (int al = 0; al < 4; ++al) {
        bf<8, 4>(acc[al], i1, r0 ^ r2, a);
        bf<8, 2>(acc[al], i3, r2 ^ r4, a);
#pragma unroll
        for (int i = 0; i < 8; ++i)
          B[4 * (64 * al + row(r0, (i >> 2), r2, ((i >> 1) & 1), r4, i & 1)) + bb] = acc[al][i];
      }
    }
    __syncwarp();
    {  // A[al][row][legs 4, 5 of the lower message]; lane = r0 .. r4
      const int i5 = id(3, 2), ha = i5 >> 1;
      const bool w0 = b0 == (i5 & 1);        // the id's beta is met by w = 0 (else by w = 1)
#pragma unroll 1
      for (int al = 0; al < (a ? 4 : 1); ++al) {
        T val[2][4];                         // [r5 ^ ha][leg values]
#pragma unroll
        for (int q = 0; q < 4; ++q) val[0][q] = val[1][q] = T(0);
#pragma unroll 1
        for (int b01 = 0; b01 < 4; ++b01)
#pragma unroll
          for (int b2 = 0; b2 < 2; ++b2) {
            T m0[4], m1[4];                  // w = 0, 1
            vcopy4(mb + 16 * b01 + 8 * b2, m0);
            vcopy4(mb + 16 * b01 + 8 * b2 + 4, m1);
            const T v = B[4 * (64 * al + 2 * lane + b2) + b01];
            const T xe = pE * v, xi = pI * v;
            const T x0 = w0 ? xi : xe, x1 = w0 ? xe : xi;
#pragma unroll
            for (int q = 0; q < 4; ++q) {    // the row r5 with b2 ^ r5 = ha meets the id
              val[b2][q] = dot2(val[b2][q], m0[q], x0, m1[q], x1);
              val[b2 ^ 1][q] = dot2(val[b2 ^ 1][q], m0[q], xe, m1[q], xe);
            }
          }
        vstore4(A + 4 * (64 * al + 2 * lane + ha), val[0]);
        vstore4(A + 4 * (64 * al + 2 * lane + (ha ^ 1)), val[1]);
      }
    }
    __syncwarp();
    {  // t = 4 (Q): u = leg 4, the lower leg 4 is r5.  B[leg 5][row][lower leg 5]
      const int r1 = b4, r3 = b3, r5 = b2, a5 = a ? b1 : 0;
      T x0[8], x1[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int at = row(i >> 2, r1, ((i >> 1) & 1), r3, (i & 1), r5);
        x0[i] = A[4 * (64 * a5 + at) + 2 * r5 + b0];
        x1[i] = a ? A[4 * (64 * (2 + a5) + at) + 2 * r5 + b0] : T(0);   // (no message: u = 0 alone)
      }
      bf4(x0, x1, id(4, 0), r1, e);
      bf<8, 2>(e, id(4, 1), r1 ^ r3, !a);
      bf<8, 1>(e, id(4, 2), r3 ^ r5, !a);
#pragma unroll
        for (int i = 0; i < 8; ++i)
          B[2 * (64 * a5 + row(i >> 2, r1, ((i >> 1) & 1), r3, (i & 1), r5)) + b0] = e[i];
    }
    __syncwarp();
    {  // t = 5 (C): leg 5 is r0; the lower leg 5 is w, summed.
      const int r0 = b3, r2 = b2, r4 = b1, w = b0;
#pragma unroll
      for (int i = 0; i < 8; ++i)
        e[i] = B[2 * ((a ? 64 * r0 : 0) + row(r0, (i >> 2), r2, ((i >> 1) & 1), r4, (i & 1))) + w];
      bf<8, 4>(e, id(5, 0), r0 ^ r2, a);
      bf<8, 2>(e, id(5, 1), r2 ^ r4, a);
      bf<8, 1>(e, id(5, 2), r4 ^ w, a);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const T v = radd(e[i], shx(e[i], 1));
        if (lane < 16 && w == 0) A[row(r0, (i >> 2), r2, ((i >> 1) & 1), r4, (i & 1))] = v;
      }
    }
    __syncwarp();
  }

  // Columns C and Q in turn, beginning with C.
  __device__ __forceinline__ void run_c() const {
    const int b4 = (lane >> 4) & 1, b3 = (lane >> 3) & 1, b2 = (lane >> 2) & 1, b1 = (lane >> 1) & 1, b0 = lane & 1;
    T e[8];
    {  // t = 0 (C): a0 tied to r0, b0 = w recorded.  A[row][b0]
      const int w = b3, r0 = b2, r2 = b1, r4 = b0;
#pragma unroll
      for (int i = 0; i < 8; ++i) e[i] = start(row(r0, (i >> 2), r2, ((i >> 1) & 1), r4, (i & 1)), 21);
      bf<8, 4>(e, id(0, 0), r0 ^ r2, a);
      bf<8, 2>(e, id(0, 1), r2 ^ r4, a);
      bf<8, 1>(e, id(0, 2), r4 ^ w, a);
      if (lane < 16)
#pragma unroll
        for (int i = 0; i < 8; ++i) A[2 * row(r0, (i >> 2), r2, ((i >> 1) & 1), r4, (i & 1)) + w] = e[i];
    }
    __syncwarp();
    const int i10 = id(1, 0);
    {  // t = 1 (Q): l0 = a0, a1 = u recorded, b1 tied to r5.
      const int r1 = b3, r3 = b2, r5 = b1;
      const int i1 = id(1, 1), i2 = id(1, 2);
      if (!a) {  // B[row][b0]
#pragma unroll
        for (int i = 0; i < 8; ++i) e[i] = A[2 * row(i >> 2, r1, ((i >> 1) & 1), r3, (i & 1), r5) + b0];
        bf<8, 4>(e, i10, r1, false);
        bf<8, 2>(e, i1, r1 ^ r3, true);
        bf<8, 1>(e, i2, r3 ^ r5, true);
        if (lane < 16)
#pragma unroll
          for (int i = 0; i < 8; ++i) B[2 * row(i >> 2, r1, ((i >> 1) & 1), r3, (i & 1), r5) + b0] = e[i];
      } else {   // B[a0][E / I][row without r0][b0]
      const int a0 = b4;
      T x[4], y[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const T v = A[2 * row(a0, r1, (i >> 1), r3, (i & 1), r5) + b0];
        x[i] = pE * v;
        y[i] = pI * v;
      }
      bf<4, 2>(x, i1, r1 ^ r3, false);
      bf<4, 1>(x, i2, r3 ^ r5, false);
      bf<4, 2>(y, i1, r1 ^ r3, false);
      bf<4, 1>(y, i2, r3 ^ r5, false);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int at = 64 * a0 + row(0, r1, (i >> 1), r3, (i & 1), r5);
        B[2 * at + b0] = x[i];
        B[2 * (at + 32) + b0] = y[i];
      }
      }
    }
    __syncwarp();
    {  // t = 2 (C): a2 tied to r0; qubits 1 and 3 (qubit 5, l5 = b1, is left to t = 3).  A[a0 a1][row, l5][b0]
      const int r0 = b4, r2 = b3, r4 = b2, a0 = b0;
      const int i1 = id(2, 0), i3 = id(2, 1);
      const int hb = i10 & 1;
      const bool hit = r0 == ((i10 >> 1) ^ a0);
#pragma unroll 1
      for (int a1 = 0; a1 < (a ? 2 : 1); ++a1) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int l1 = (i >> 2), l3 = ((i >> 1) & 1), l5 = i & 1;
          const int sel = hit && a1 == (hb ^ l1) ? 32 : 0;
          e[i] = B[2 * (a ? 64 * a0 + sel + row(0, l1, r2, l3, r4, l5) : row(r0, l1, r2, l3, r4, l5)) + b1];
        }
        bf<8, 4>(e, i1, r0 ^ r2, a);
        bf<8, 2>(e, i3, r2 ^ r4, a);
        if (a || a0 == 0)
#pragma unroll
          for (int i = 0; i < 8; ++i)
            A[2 * ((a ? 64 * (2 * a0 + a1) : 0) + row(r0, (i >> 2), r2, ((i >> 1) & 1), r4, i & 1)) + b1] = e[i];
      }
    }
    __syncwarp();
    // t = 3 (Q), the data column: qubit 5 of t = 2 scales by pE or pI by
    // (r5, b2 = w), so both scaled copies take the upper message (over a with
    // a2 = l0), qubit 0 (u summed) and qubit 2; the copy is picked per (r5, b2)
    // at qubit 4, and the lower message (over b, its leg w = r5) closes.
    const int i25 = id(2, 2);
    {  // B[E / I][al][r0 .. r3, l4][b1][b0]
      const int r1 = b4, r3 = b3, l4 = b2;
      const int i0 = id(3, 0), i2 = id(3, 1);
#pragma unroll 1
      for (int ei = 0; ei < 2; ++ei) {
        const T p = ei ? pI : pE;
        if (!a) {
          T y[4];                            // [r0][l2]
#pragma unroll
          for (int i = 0; i < 4; ++i) y[i] = p * A[2 * row(i >> 1, r1, (i & 1), r3, l4, b1) + b0];
          bf<4, 2>(y, i0, r1, false);
          bf<4, 1>(y, i2, r1 ^ r3, true);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            B[4 * (128 * ei + (row(i >> 1, r1, (i & 1), r3, l4, 0) >> 1)) + 2 * b1 + b0] = y[i];
          continue;
        }
        T acc[4][2][4];                      // [al][u][l0 l2]
#pragma unroll
        for (int al = 0; al < 4; ++al)
#pragma unroll
          for (int i = 0; i < 8; ++i) acc[al][i >> 2][i & 3] = T(0);
#pragma unroll 1
        for (int a01 = 0; a01 < 4; ++a01)
#pragma unroll
          for (int l0 = 0; l0 < 2; ++l0) {
            T m0[4], m1[4];                  // u = 0, 1
            vcopy4(mt + 8 * (2 * a01 + l0), m0);
            vcopy4(mt + 8 * (2 * a01 + l0) + 4, m1);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              const T x = p * A[2 * (64 * a01 + row(l0, r1, q, r3, l4, b1)) + b0];
#pragma unroll
              for (int al = 0; al < 4; ++al) {
                acc[al][0][2 * l0 + q] = fma(m0[al], x, acc[al][0][2 * l0 + q]);
                acc[al][1][2 * l0 + q] = fma(m1[al], x, acc[al][1][2 * l0 + q]);
              }
            }
          }
        const T g00 = g(i0, 0, r1), g01 = g(i0, 0, r1 ^ 1), g10 = g(i0, 1, r1), g11 = g(i0, 1, r1 ^ 1);
#pragma unroll
        for (int al = 0; al < 4; ++al) {
          T y[4];                            // [r0][l2]
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const T(&x0)[4] = acc[al][0];
            const T(&x1)[4] = acc[al][1];
            y[q] = dot4(x0[q], g00, x1[q], g01, x0[2 + q], g10, x1[2 + q], g11);
            y[2 + q] = dot4(x0[q], g10, x1[q], g11, x0[2 + q], g00, x1[2 + q], g01);
          }
          bf<4, 1>(y, i2, r1 ^ r3, false);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            B[4 * (32 * (4 * ei + al) + (row(i >> 1, r1, (i & 1), r3, l4, 0) >> 1)) + 2 * b1 + b0] = y[i];
        }
      }
    }
    __syncwarp();
    {  // A[al][row][legs 4, 5 of the lower message]; lane = (al's low bit, r0 .. r3)
      const int r3 = b0, i4 = id(3, 2), ha = i25 >> 1, hb = i25 & 1;
      const T g0[2] = {g(i4, 0, r3), g(i4, 0, r3 ^ 1)}, g1[2] = {g(i4, 1, r3), g(i4, 1, r3 ^ 1)};   // by r5
#pragma unroll 1
      for (int k = 0; k < (a ? 2 : 1); ++k) {
        const int al = a ? 2 * k + b4 : 0;
        const T* E = B + 4 * (32 * al + 2 * (lane & 15));
        T val[2][2][4];                      // [r5][r4][leg values]
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int q = 0; q < 4; ++q) val[r >> 1][r & 1][q] = T(0);
#pragma unroll 1
        for (int b01 = 0; b01 < 4; ++b01) {
          const int at = 2 * (b01 & 1) + (b01 >> 1);           // b1, b0
          const T xe0 = E[at], xe1 = E[4 + at];                // l4 = 0, 1
#pragma unroll
          for (int w = 0; w < 2; ++w) {      // b2
            const int hl = hb ^ w;           // the l4 whose (l4, w) meets the id's beta
            const T xi = E[512 + 4 * hl + at];
#pragma unroll
            for (int r5 = 0; r5 < 2; ++r5) {
              const bool hit = ((b01 & 1) ^ r5) == ha;
              const T x0 = hit && hl == 0 ? xi : xe0, x1 = hit && hl == 1 ? xi : xe1;
              T m[4];
              vcopy4(mb + 16 * b01 + 8 * w + 4 * r5, m);
              const T y0 = a ? fma(x1, g1[r5], x0 * g0[r5]) : fma(x0, g0[r5], x1 * g1[r5]);   // qubit 4, as bf(!a)
              const T y1 = fma(x1, g0[r5], x0 * g1[r5]);
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                val[r5][0][q] = dot1(val[r5][0][q], m[q], y0);
                val[r5][1][q] = dot1(val[r5][1][q], m[q], y1);
              }
            }
          }
        }
        if (a || lane < 16)
#pragma unroll
          for (int r = 0; r < 4; ++r)
            vstore4(A + 4 * (64 * al + 4 * (lane & 15) + 2 * ((r & 1)) + (r >> 1)), val[r >> 1][r & 1]);
      }
    }
    __syncwarp();
    {  // t = 4 (C): leg 4 is r0; the lower leg 4 is w, summed.  B[leg 5][row][lower leg 5]
      const int r0 = b4, r2 = b3, r4 = b2, a5 = a ? b1 : 0;
      const int i1 = id(4, 0), i3 = id(4, 1), i5 = id(4, 2);
      T s[8];
#pragma unroll
      for (int w = 0; w < 2; ++w) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          e[i] = A[4 * ((a ? 64 * (2 * r0 + a5) : 0) + row(r0, (i >> 2), r2, ((i >> 1) & 1), r4, (i & 1))) +
                   2 * w + b0];
        bf<8, 4>(e, i1, r0 ^ r2, a);
        bf<8, 2>(e, i3, r2 ^ r4, a);
        bf<8, 1>(e, i5, r4 ^ w, a);
#pragma unroll
        for (int i = 0; i < 8; ++i) s[i] = w ? radd(s[i], e[i]) : e[i];
      }
#pragma unroll
        for (int i = 0; i < 8; ++i)
          B[2 * (64 * a5 + row(r0, (i >> 2), r2, ((i >> 1) & 1), r4, (i & 1))) + b0] = s[i];
    }
    __syncwarp();
    {  // t = 5 (Q): u = leg 5, the lower leg 5 is r5.
      const int r1 = b2, r3 = b1, r5 = b0;
      T x0[8], x1[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int at = row(i >> 2, r1, ((i >> 1) & 1), r3, (i & 1), r5);
        x0[i] = B[2 * at + r5];
        x1[i] = a ? B[2 * (64 + at) + r5] : T(0);
      }
      bf4(x0, x1, id(5, 0), r1, e);
      bf<8, 2>(e, id(5, 1), r1 ^ r3, !a);
      bf<8, 1>(e, id(5, 2), r3 ^ r5, !a);
      if (lane < 8)
#pragma unroll
        for (int i = 0; i < 8; ++i) A[row(i >> 2, r1, ((i >> 1) & 1), r3, (i & 1), r5)] = e[i];
    }
    __syncwarp();
  }
};

}  // namespace bbp
