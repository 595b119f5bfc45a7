// Register form of the fused block update (Remark 9) for 4 x 4 blocks and the
// one-node-wide blocks that the last block row / column leaves at odd d.
//
// Along a column of a block checks and qubits alternate.  A check is a copy
// tensor (Sec. III.A), so its row leg, its two chain legs and (in the top or
// bottom row) the side message's leg are one and the same bit; a qubit's
// tensor pi(f + (x, z)) depends only on the parity of its in/out legs (alpha)
// and of its chain legs (beta): g[alpha][beta].  A column therefore acts on
// the 16-entry row state as two 2-point XOR convolutions (one per qubit row)
// whose beta is a parity of bits that the checks fix, and the side messages'
// legs are either tied to a row bit (check in the top / bottom row) or enter
// a qubit's beta.  Sides on the grid border have no message; they act as the
// product vector of their nodes' missing legs: ones for a check (a copy
// tensor over its remaining legs) and e_0 for a qubit (a missing leg carries
// 0), which is what the node-by-node path computes there.
//
// Work is handed out as jobs (message, coset), eight to a warp pass, four
// lanes each.  Row bits r0 and r2 of the chain live in registers (a lane
// holds four rows), r1 and r3 in the lanes (lane bit 1 and bit 0 of the
// group): column 2, the widest state (four open side legs), exchanges only
// over r0 and r2 and needs no shuffle, and the coefficient of each qubit is
// formed once per lane for four rows.  A pass takes any eight jobs of one
// shape, so cosets that have converged leave no idle lanes.  The kernel is
// bound by instruction issue; the form with two rows per lane, one message
// and its cosets to a pass, which this replaced, issued 416 instructions for
// at most four jobs, mostly shuffles, coefficient selects and staging.  At
// d = 11, p = 0.10, FP32, 10^4 syndromes: 10.34 -> 5.09 ms (the read-out and
// the prologue by the same jobs and by arithmetic instead of compactions:
// 1.19 -> 0.45 ms of it, timed at 0 iterations).
#pragma once

#include "bbp_kernels.cuh"

namespace bbp {

constexpr int kRegVec = 16;                 // entries of a message vector
constexpr int kBorderVecs = 2;              // product vectors of the grid border, after the messages
// Shapes (chain height x columns): 4 x 4; 4 x 1, 1 x 4 and 1 x 1, the last
// blocks of odd d; 4 x 3, 3 x 4 and 3 x 3, those of even d.
constexpr int kShapeNone = 0, kShapeQuad = 1, kShapeCol = 2, kShapeRow = 3, kShapeDot = 4;
constexpr int kShape43 = 5, kShape34 = 6, kShape33 = 7, kShapes = 7;

// Index of the directed edge leaving block (I, J) towards dir in (I, J, dir)
// order (R, L, D, U); the edge must exist.
BBP_HD int message_index(int nb, int I, int J, int dir) {
  int idx = I * 2 * (nb - 1) + (imin(I, nb - 1) + imax(I - 1, 0)) * nb;      // rows above
  const int up = I > 0, down = I + 1 < nb, left = J > 0, right = J + 1 < nb;
  idx += J + imax(J - 1, 0) + J * (up + down);                               // blocks to the left
  if (dir > kDirR) idx += right;
  if (dir > kDirL) idx += left;
  if (dir > kDirD) idx += down;
  return idx;
}

// A job's message: vector indices (< M a message, M + b the border vector b)
// of the incoming message opposite the outgoing side, of the side messages
// at the chain's upper (s' = 0) and lower end, and of the outgoing message;
// chk0: column 0 starts with a check (a chain of more than one node is then
// read bottom to top: both node tensors are symmetric in their chain legs, so
// one form covers both); srev: the side messages are consumed in reverse
// site order; shape.
struct RegTask {
  uint16_t in, up, lo, out;                 // 12 bits of index; top bits: in chk0, up srev, out shape
};
constexpr int kTaskIdx = 0xFFF, kTaskFlag = 0x8000, kTaskShape = 12;
static_assert(sizeof(RegTask) == 8, "a task is one 8-byte load");

// Border vector b of w legs: leg u from the last is e_0 (a qubit) where bit u
// of the mask is set, (1, 1) (a check) elsewhere.  Legs alternate, so the
// masks are 1010 (b = 0) and 0101 (b = 1); entries 0 and 1 serve one leg.
__device__ __forceinline__ bool border_entry(int b, int i) { return (i & (b ? 5 : 10)) == 0; }

// The side geometry of a block update: the chain's height and columns, and
// the node positions, as in make_frame but from arithmetic alone.
struct RegFrame {
  int dir, h, ncols, r0, r1, c0, c1;
  __device__ __forceinline__ void node(int t, int s, int* i, int* j) const {
    switch (dir) {
      case kDirR: *i = r0 + s; *j = c0 + t; break;
      case kDirL: *i = r0 + s; *j = c1 - 1 - t; break;
      case kDirD: *i = r0 + t; *j = c0 + s; break;
      default:    *i = r1 - 1 - t; *j = c0 + s; break;
    }
  }
  __device__ __forceinline__ bool rowwise() const { return dir == kDirR || dir == kDirL; }
  __device__ __forceinline__ bool chk0() const {
    int i, j;
    node(0, 0, &i, &j);
    return (i + j) & 1;
  }
  // Blocks three nodes wide or high keep the node-by-node form's chain order.
  __device__ __forceinline__ bool wide3() const { return h == 3 || ncols == 3; }
  __device__ __forceinline__ bool srev() const { return dir == kDirL || dir == kDirU; }
  __device__ __forceinline__ int shape() const {
    if (h == 4 && ncols == 4) return kShapeQuad;
    if (h == 4 && ncols == 1) return kShapeCol;
    if (h == 1 && ncols == 4) return kShapeRow;
    if (h == 1 && ncols == 1) return kShapeDot;
    if (h == 4 && ncols == 3) return kShape43;
    if (h == 3 && ncols == 4) return kShape34;
    if (h == 3 && ncols == 3) return kShape33;
    return kShapeNone;
  }
};

__device__ __forceinline__ RegFrame reg_frame(const Geo& g, int I, int J, int dir) {
  RegFrame f;
  f.dir = dir;
  f.r0 = g.lo(I); f.r1 = g.hi(I); f.c0 = g.lo(J); f.c1 = g.hi(J);
  const int hr = f.r1 - f.r0, hc = f.c1 - f.c0;
  f.h = f.rowwise() ? hr : hc;
  f.ncols = f.rowwise() ? hc : hr;
  return f;
}

__device__ __forceinline__ RegTask reg_task(const Geo& g, int M, int I, int J, const RegFrame& f) {
  const int nb = g.nb;
  const bool chk0 = f.chk0(), srev = f.srev(), rev = chk0 && f.h > 1 && !f.wide3();
  // The border vector of a side whose leg nearest the vector's last entry
  // belongs to node (i, j): mask bit 0 is set at a qubit.
  auto border = [&](int i, int j) { return M + (((i + j) & 1) ? 0 : 1); };
  auto side = [&](int towards) {            // message from the neighbour in direction `towards`, or -1
    const int i = I + (towards == kDirD) - (towards == kDirU), j = J + (towards == kDirR) - (towards == kDirL);
    if (i < 0 || j < 0 || i >= nb || j >= nb) return -1;
    return message_index(nb, i, j, towards ^ 1);
  };
  int i, j;
  int in = side(f.dir ^ 1);
  if (in < 0) {
    f.node(0, f.h - 1, &i, &j);
    in = border(i, j);
  }
  const int first = f.rowwise() ? kDirU : kDirL, last = f.rowwise() ? kDirD : kDirR;
  int ends[2] = {side(rev ? last : first), side(rev ? first : last)};       // upper (s' = 0), lower
#pragma unroll
  for (int e = 0; e < 2; ++e)
    if (ends[e] < 0) {
      // Stored in site order: with srev its last entry belongs to the first node consumed.
      f.node(srev ? 0 : f.ncols - 1, (e == 0) == rev ? f.h - 1 : 0, &i, &j);
      ends[e] = border(i, j);
    }
  RegTask q;
  q.in = (uint16_t)(in | (chk0 ? kTaskFlag : 0));
  q.up = (uint16_t)(ends[0] | (srev ? kTaskFlag : 0));
  q.lo = (uint16_t)ends[1];
  q.out = (uint16_t)((g.has(I, J, f.dir) ? message_index(nb, I, J, f.dir) : 0) | (f.shape() << kTaskShape));
  return q;
}

// Prefix parities of the pure error f_s: bit c of px[r] is the x bit of the
// horizontal-edge qubit (2 r, 2 c), bit r of pz[c] its z bit (vertical-edge
// qubits carry nothing).
__device__ __forceinline__ unsigned long long prefix_parity(unsigned long long v) {   // bit c: parity of bits < c
#pragma unroll
  for (int s = 1; s < 64; s <<= 1) v ^= v << s;
  return v << 1;
}

// Pauli-frame bits (x, z << 1) of f_s at node (i, j).
__device__ __forceinline__ int frame_bits(const unsigned long long* px, const unsigned long long* pz, int i, int j) {
  if ((i | j) & 1) return 0;
  return (int)((px[i >> 1] >> (j >> 1)) & 1ull) | ((int)((pz[j >> 1] >> (i >> 1)) & 1ull) << 1);
}

// Ids (2 bits each, pi(I) at (alpha, beta)) of a block's qubits for coset I,
// and the bits that the logical strings X-bar (grid row 0) and Z-bar (column
// 0) flip.  4 x 4: the upper (u = 0) and lower qubit of column t at bits
// 2 (2 t + u); 4 x 1: the qubits at s' = 0 and 2; 1 x 4: the qubits of columns
// 0 and 2, or 1 and 3; 1 x 1: the node; three wide or high: field 2 t + u the
// qubit at chain position 2 u, or 2 u + 1 in a column that starts with a check.
struct RegIds {
  unsigned id, fx, fz;
};
__device__ __forceinline__ void add_id(RegIds& v, const RegFrame& f, int t, int s, int field,
                                       const unsigned long long* px, const unsigned long long* pz) {
  int i, j;
  f.node(t, s, &i, &j);
  const int fv = frame_bits(px, pz, i, j);
  const bool alpha_is_z = ((i & 1) == 0) == f.rowwise();
  const bool hq = ((i | j) & 1) == 0;
  v.id |= (unsigned)(alpha_is_z ? fv : (((fv & 1) << 1) | (fv >> 1))) << (2 * field);
  v.fx |= (unsigned)(hq && i == 0 ? (alpha_is_z ? 1 : 2) : 0) << (2 * field);
  v.fz |= (unsigned)(hq && j == 0 ? (alpha_is_z ? 2 : 1) : 0) << (2 * field);
}
// Column t's part of a quad's ids (fields 2 t, 2 t + 1).
__device__ __forceinline__ void add_quad_column(RegIds& v, const RegFrame& f, int t, bool chk0,
                                                const unsigned long long* px, const unsigned long long* pz) {
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int sq = (t & 1) + 2 * u;
    add_id(v, f, t, chk0 ? 3 - sq : sq, 2 * t + u, px, pz);
  }
}
__device__ __forceinline__ RegIds reg_ids(const RegFrame& f, const unsigned long long* px,
                                          const unsigned long long* pz) {
  RegIds v{0u, 0u, 0u};
  const bool chk0 = f.chk0();
  const int shape = f.shape();
  if (shape == kShapeQuad) {
    for (int t = 0; t < 4; ++t) add_quad_column(v, f, t, chk0, px, pz);
  } else if (shape == kShapeCol) {
    add_id(v, f, 0, chk0 ? 3 : 0, 0, px, pz);
    add_id(v, f, 0, chk0 ? 1 : 2, 1, px, pz);
  } else if (shape == kShapeRow) {
    add_id(v, f, chk0 ? 1 : 0, 0, 0, px, pz);
    add_id(v, f, chk0 ? 3 : 2, 0, 1, px, pz);
  } else if (shape == kShapeDot) {
    add_id(v, f, 0, 0, 0, px, pz);
  } else if (shape != kShapeNone) {
    for (int t = 0; t < f.ncols; ++t) {
      const int c = ((t & 1) != 0) != chk0 ? 1 : 0;
      for (int u = 0; 2 * u + c < f.h; ++u) add_id(v, f, t, 2 * u + c, 2 * t + u, px, pz);
    }
  }
  return v;
}
__device__ __forceinline__ unsigned coset_id(const RegIds& v, int coset) {
  return v.id ^ ((coset == 1 || coset == 2) ? v.fx : 0u) ^ ((coset == 2 || coset == 3) ? v.fz : 0u);
}

// ---------------------------------------------------------------------------
// The G x M message vectors of a CTA.  In shared memory the border vectors
// follow each coset's messages; messages in a workspace slot (GM) have their
// border vectors in shared memory.
template <typename T, bool GM>
struct RegMsgs {
  T* base;
  int stride;                               // scalars from coset to coset
  const T* border;                          // GM only
  int M;
  __device__ __forceinline__ const T* at(int cq, int v) const {
    if constexpr (GM) {
      if (v >= M) return border + (v - M) * kRegVec;
    }
    return base + cq * stride + v * kRegVec;
  }
  __device__ __forceinline__ T* out(int cq, int v) const { return base + cq * stride + v * kRegVec; }
};

// What a pass needs to finish a message update itself (Remarks 3, 4, 7).
template <typename T>
struct RegUpd {
  T eta, one_m_eta;
  T* ovl;                                   // Delta term of each (coset, message)
  int M;
};

// One lane's view of its job.
template <typename T, bool GM>
struct RegJob {
  RegTask q;
  int cq;                                   // coset within the CTA
  unsigned id;                              // qubit ids of (message, coset)
  bool on;                                  // a repeated job that keeps the warp's shuffles company stores nothing
  __device__ __forceinline__ int in() const { return q.in & kTaskIdx; }
  __device__ __forceinline__ int up() const { return q.up & kTaskIdx; }
  __device__ __forceinline__ int lo() const { return q.lo & kTaskIdx; }
  __device__ __forceinline__ int out() const { return q.out & kTaskIdx; }
  __device__ __forceinline__ bool chk0() const { return (q.in & kTaskFlag) != 0; }
  __device__ __forceinline__ bool srev() const { return (q.up & kTaskFlag) != 0; }
};

template <typename T>
__device__ __forceinline__ T shx(T v, int mask) { return __shfl_xor_sync(kFull, v, mask); }

// Adds that are never contracted with the product feeding them, so that
// every kernel compiled from this gives the same bits.
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double radd(double a, double b) { return __dadd_rn(a, b); }

// Coefficient v (0 .. 3) of the qubit in field f of t = ids ^ lane pattern:
// pI where the field equals v.  With the lane's bit be at the field's beta
// position, the field is (alpha, beta ^ be): g[0][be], g[1][be] are
// v = 0, 2 and g[0][be ^ 1], g[1][be ^ 1] are v = 1, 3.
template <typename T>
__device__ __forceinline__ T qco(unsigned t, int f, unsigned v, T pI, T pE) {
  return ((t ^ (v << (2 * f))) & (3u << (2 * f))) == 0u ? pI : pE;   // constant masks: one logic op
}
// g[0][be] and g[1][be] of a qubit whose pi(I) entry sits at id = (alpha, beta).
template <typename T>
__device__ __forceinline__ void qpair(int id, int be, T pI, T pE, T& g0, T& g1) {
  const bool hit = (id & 1) == be;
  const bool hi = (id >> 1) & 1;
  g0 = (hit && !hi) ? pI : pE;
  g1 = (hit && hi) ? pI : pE;
}
template <typename T>
__device__ __forceinline__ T qval(int id, int al, int be, T pI, T pE) {
  return ((al << 1) | be) == id ? pI : pE;
}

// Four consecutive scalars at a 16-byte aligned address.
__device__ __forceinline__ void vcopy4(const float* p, float (&v)[4]) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void vcopy4(const double* p, double (&v)[4]) {
  const double2 q0 = reinterpret_cast<const double2*>(p)[0], q1 = reinterpret_cast<const double2*>(p)[1];
  v[0] = q0.x; v[1] = q0.y; v[2] = q1.x; v[3] = q1.y;
}
__device__ __forceinline__ void vstore4(float* p, const float (&v)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void vstore4(double* p, const double (&v)[4]) {
  reinterpret_cast<double2*>(p)[0] = make_double2(v[0], v[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(v[2], v[3]);
}

// Where a lane's four rows (q0, q2) of a 16-entry chain vector sit: row
// (r0 r1 r2 r3) at its own index, or bit-reversed when the chain is read
// bottom to top.
struct RowAt {
  int base, s0, s2;
  __device__ __forceinline__ RowAt(bool rev, int r1, int r3)
      : base(rev ? 2 * r1 + 8 * r3 : 4 * r1 + r3), s0(rev ? 1 : 8), s2(rev ? 4 : 2) {}
  __device__ __forceinline__ int operator()(int q0, int q2) const { return base + (q0 ? s0 : 0) + (q2 ? s2 : 0); }
};

// Sum of the 16 entries of a job, v[q0][q2] in this lane, over row bits in
// the order r0, r1, r2, r3; every lane of the group gets the same bits.
template <typename T>
__device__ __forceinline__ T job_sum(const T (&v)[2][2]) {
  T s0 = radd(v[0][0], v[1][0]), s1 = radd(v[0][1], v[1][1]);
  s0 = radd(s0, shx(s0, 2));
  s1 = radd(s1, shx(s1, 2));
  const T s = radd(s0, s1);
  return radd(s, shx(s, 1));
}

// The message update of a 16-entry vector: normalisation (Remark 3), damping
// with the stored message y (Remark 7), normalisation, and the Delta term
// 2 - 2 <x, y>^2 (Remark 4).  FP32 evaluates that term as s (2 - s / 2) with
// s = ||x - y||^2, an identity for unit vectors: no cancellation when a
// message barely moved, and no FP64 instruction per update (FP64 issues at
// 1/64 of the FP32 rate here).
template <typename T, bool GM>
__device__ __forceinline__ void reg_update16(const T (&out)[2][2], const RegMsgs<T, GM>& ms, const RegJob<T, GM>& jb,
                                             const RowAt& at, bool writer, const RegUpd<T>& up) {
  T* old = ms.out(jb.cq, jb.out());
  T x[2][2], y[2][2], w[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      y[a][b] = old[at(a, b)];
      w[a][b] = out[a][b] * out[a][b];
    }
  const T i1 = inv_norm(job_sum(w));
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      x[a][b] = fma(up.one_m_eta, out[a][b] * i1, up.eta * y[a][b]);
      w[a][b] = x[a][b] * x[a][b];
    }
  const T i2 = inv_norm(job_sum(w));
  T term;
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      x[a][b] = x[a][b] * i2;
      if constexpr (sizeof(T) == 4) {
        const T t = x[a][b] - y[a][b];
        w[a][b] = t * t;
      } else {
        w[a][b] = x[a][b] * y[a][b];
      }
    }
  const T sq = job_sum(w);
  if constexpr (sizeof(T) == 4) term = sq * fma(T(-0.5), sq, T(2));
  else term = fma(T(-2) * sq, sq, T(2));
  if (jb.on) {
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) old[at(a, b)] = x[a][b];
    if (writer) up.ovl[jb.cq * up.M + jb.out()] = term;
  }
}

// The same for a 2-entry vector (v0, v1) that every lane of the group holds
// whole; the writer lane stores it.
template <typename T, bool GM>
__device__ __forceinline__ void reg_update2(T v0, T v1, const RegMsgs<T, GM>& ms, const RegJob<T, GM>& jb, bool writer,
                                            const RegUpd<T>& up) {
  T* old = ms.out(jb.cq, jb.out());
  const T y0 = old[0], y1 = old[1];
  T inv = inv_norm(radd(v0 * v0, v1 * v1));
  T x0 = fma(up.one_m_eta, v0 * inv, up.eta * y0), x1 = fma(up.one_m_eta, v1 * inv, up.eta * y1);
  inv = inv_norm(radd(x0 * x0, x1 * x1));
  x0 = x0 * inv;
  x1 = x1 * inv;
  T term;
  if constexpr (sizeof(T) == 4) {
    const T t0 = x0 - y0, t1 = x1 - y1;
    const T sq = radd(t0 * t0, t1 * t1);
    term = sq * fma(T(-0.5), sq, T(2));
  } else {
    const T o = radd(x0 * y0, x1 * y1);
    term = fma(T(-2) * o, o, T(2));
  }
  __syncwarp();   // every lane has read the stored message
  if (jb.on && writer) {
    old[0] = x0;
    old[1] = x1;
    up.ovl[jb.cq * up.M + jb.out()] = term;
  }
}

// Per-warp staging: 16 scalars a job.
constexpr int kRegStage = 8 * 16;

// Eight 4 x 4 block updates.  Columns t = 0 .. 3 hold qubits at chain
// positions {0, 2} or {1, 3}, alternating.  UPD: the message update;
// otherwise the outgoing vectors go to stage + 16 job.
template <typename T, bool GM, bool UPD>
__device__ __forceinline__ void quad_pass(T* stage, T pI, T pE, const RegMsgs<T, GM>& ms, const RegJob<T, GM>& jb,
                                          int lane, const RegUpd<T>& upd) {
  const int r1 = (lane >> 1) & 1, r3 = lane & 1, g = lane >> 2;
  // The qubit ids (field 2 t + u: the upper, u = 0, or lower qubit of column
  // t) against the lane's row bits: be of each field's first use at r0 = r2 =
  // 0 is r1 (0, 0), r1 ^ r3 (0, 1), r1 (2, 0), r1 ^ r3 (2, 1); and r3 at the
  // alpha bit of (1, 1), whose coefficients the lanes of odd rows take
  // swapped.  Where be holds r0 or r2, the coefficients are picked by row.
  const unsigned tq = jb.id ^ (r1 ? 0x0505u : 0u) ^ (r3 ? 0x0484u : 0u);
  // The upper side message's part of column 2 (data column, upper qubit),
  // sum over v of A[a0 a1 v e] g[a][v ^ r1] with e = q0, a1 = q0 ^ a: the
  // lanes of a job that differ in r3 need the same eight values, so each
  // forms those of a0 = r3 and they are exchanged through shared memory.
  T* sj = stage + (g << 4);
  {
    const T* A = ms.at(jb.cq, jb.up());
    T a[8];                                                // [a1][v][e]
    if (jb.srev()) {
#pragma unroll
      for (int i = 0; i < 8; ++i) a[i] = A[r3 + 2 * (i >> 2) + 4 * ((i >> 1) & 1) + 8 * (i & 1)];
    } else {
      T lo[4], hi[4];
      vcopy4(A + 8 * r3, lo);
      vcopy4(A + 8 * r3 + 4, hi);
#pragma unroll
      for (int i = 0; i < 4; ++i) { a[i] = lo[i]; a[4 + i] = hi[i]; }
    }
    const T g00 = qco(tq, 4, 0u, pI, pE), g10 = qco(tq, 4, 2u, pI, pE);   // v = 0
    const T g01 = qco(tq, 4, 1u, pI, pE), g11 = qco(tq, 4, 3u, pI, pE);   // v = 1
    T c[4];                                                // [alpha][q0]
    c[0] = fma(a[2], g01, a[0] * g00);
    c[1] = fma(a[7], g01, a[5] * g00);
    c[2] = fma(a[6], g11, a[4] * g10);
    c[3] = fma(a[3], g11, a[1] * g10);
    vstore4(sj + 8 * r1 + 4 * r3, c);
  }
  __syncwarp();
  const RowAt at(jb.chk0(), r1, r3);
  T x[2][2];                                               // [q0][q2]
  {
    const T* X = ms.at(jb.cq, jb.in());
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) x[a][b] = X[at(a, b)];
  }
  // Column 0 (qubits at 0, 2): the upper leg a0 is recorded, the lower leg b0
  // is tied to r3 by the check at 3.
  T S0[2][2][2];                                           // [a0][q0][q2]
  {
    const T k0 = qco(tq, 1, 0u, pI, pE), k1 = qco(tq, 1, 2u, pI, pE);
    T u[2][2];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) u[a][b] = fma(k1, x[a][b ^ 1], k0 * x[a][b]);
#pragma unroll
    for (int a0 = 0; a0 < 2; ++a0) {
      const T h0 = qco(tq, 0, (unsigned)a0, pI, pE), h1 = qco(tq, 0, 2u + a0, pI, pE);
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) S0[a0][a][b] = fma(h1, u[a ^ 1][b], h0 * u[a][b]);
    }
  }
  // Column 1 (qubits at 1, 3): a1 is tied to r0 by the check at 0; the lower
  // leg b1 is recorded.  S1[b0][b1] for one a0 at a time, folded into column 2
  // at once.  Column 2 (qubits at 0, 2) is the data column of both side
  // messages: the upper leg v is summed against A (above), the lower leg
  // w = r3 against B[b0 b1 w f].
  T h0[2], h1[2];                                          // by r0 ^ r2
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    h0[b] = qco(tq, 2, (unsigned)b, pI, pE);
    h1[b] = qco(tq, 2, 2u + b, pI, pE);
  }
  // Column 1's lower qubit scales T_b0 by g[b0 ^ r3][r2 ^ b1]: pE for the b0
  // that its id does not meet (O), whatever b1, so S1, u and Y of that b0 are
  // formed once for both b1; for the other b0 (h) pI where r2 ^ b1 meets the id.
  const bool h = tq & 0x80u;
  const T kh[2] = {(tq & 0x40u) ? pE : pI, (tq & 0x40u) ? pI : pE};   // by r2 ^ b1
  const int lane_h = (lane & ~1) | (h ? 1 : 0), lane_o = lane_h ^ 1;
  const T c2k0 = qco(tq, 5, 0u, pI, pE), c2k1 = qco(tq, 5, 2u, pI, pE);
  // Column 3's upper leg e is tied to r0 by its check: only e = r0 of
  // A[a0 a1 v e] and of everything after it reaches a row's output.
  T YO[2][2], Yh[2][2][2];                                 // [q0][q2], [b1][q0][q2], e = r0
#pragma unroll
  for (int a0 = 0; a0 < 2; ++a0) {
    T cA[4];
    vcopy4(sj + 8 * r1 + 4 * a0, cA);                      // [alpha][q0]
    T TO[2][2], Th[2][2];                                  // the upper qubit's butterfly over r1, r3 = !h and h
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const T o = S0[a0][a][b];
        const T t = fma(h1[a ^ b], shx(o, 2), h0[a ^ b] * o);
        TO[a][b] = __shfl_sync(kFull, t, lane_o);
        Th[a][b] = __shfl_sync(kFull, t, lane_h);
      }
#pragma unroll
    for (int k = 0; k < 3; ++k) {                          // O, then h with b1 = 0, 1
      T S1[2][2], u[2][2];
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) S1[a][b] = k == 0 ? pE * TO[a][b] : kh[(k - 1) ^ b] * Th[a][b];
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) u[a][b] = fma(c2k1, S1[a][b ^ 1], c2k0 * S1[a][b]);
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          T& y = k == 0 ? YO[a][b] : Yh[k == 0 ? 0 : k - 1][a][b];
          y = a0 == 0 ? fma(cA[a], u[a][b], cA[2 + a] * u[a ^ 1][b])
                      : fma(cA[a], u[a][b], fma(cA[2 + a], u[a ^ 1][b], y));
        }
    }
  }
  T S2[2][2][2];                                           // [ff][q0][q2]
  {
    const T* B = ms.at(jb.cq, jb.lo());
    T bm[2][2][2];                                         // B[b0 b1 r3 ff]
    if (jb.srev()) {
#pragma unroll
      for (int i = 0; i < 8; ++i) bm[i >> 2][(i >> 1) & 1][i & 1] = B[(i >> 2) + 2 * ((i >> 1) & 1) + 4 * r3 + 8 * (i & 1)];
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) bm[i >> 2][(i >> 1) & 1][i & 1] = B[4 * (i >> 1) + 2 * r3 + (i & 1)];
    }
#pragma unroll
    for (int f = 0; f < 2; ++f)
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b)
          S2[f][a][b] = fma(bm[1][1][f], h ? Yh[1][a][b] : YO[a][b],
                            fma(bm[1][0][f], h ? Yh[0][a][b] : YO[a][b],
                                fma(bm[0][1][f], h ? YO[a][b] : Yh[1][a][b],
                                    bm[0][0][f] * (h ? YO[a][b] : Yh[0][a][b]))));
  }
  // Column 3 (qubits at 1, 3): the upper leg e is tied to r0, the lower leg f
  // closes against B's expected value.
  T out[2][2];
  {
    T c7[4], c6[4];
#pragma unroll
    for (unsigned v = 0; v < 4; ++v) {
      c7[v] = qco(tq, 7, v, pI, pE);
      c6[v] = qco(tq, 6, v, pI, pE);
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        const T z0 = S2[0][a][b], z1 = S2[1][a][b];
        const T p0 = shx(z0, 1), p1 = shx(z1, 1);
        const T uu = fma(c7[3 ^ b], p1, fma(c7[1 ^ b], z1, fma(c7[2 ^ b], p0, c7[b] * z0)));
        out[a][b] = fma(c6[2 ^ a ^ b], shx(uu, 2), c6[a ^ b] * uu);
      }
  }
  if constexpr (UPD) {
    reg_update16(out, ms, jb, at, (lane & 3) == 0, upd);
    __syncwarp();
  } else {
    __syncwarp();                                          // every lane has taken its part of the staging
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) sj[at(a, b)] = out[a][b];
    __syncwarp();
  }
}

// Eight blocks of one column of 4 nodes: as quad_pass's column 0, both side
// messages have one leg.
template <typename T, bool GM, bool UPD>
__device__ __forceinline__ void col_pass(T* stage, T pI, T pE, const RegMsgs<T, GM>& ms, const RegJob<T, GM>& jb,
                                         int lane, const RegUpd<T>& upd) {
  const int r1 = (lane >> 1) & 1, r3 = lane & 1, g = lane >> 2;
  // The top qubit (field 0) with be = r1, the lower one (field 1) with be = r1 ^ r3.
  const unsigned tq = jb.id ^ (r1 ? 5u : 0u) ^ (r3 ? 4u : 0u);
  const RowAt at(jb.chk0(), r1, r3);
  const T* X = ms.at(jb.cq, jb.in());
  const T* A = ms.at(jb.cq, jb.up());
  const T a0 = A[0], a1 = A[1];
  const T bb = ms.at(jb.cq, jb.lo())[r3];
  const T k0 = qco(tq, 1, 0u, pI, pE), k1 = qco(tq, 1, 2u, pI, pE);
  const T h0 = qco(tq, 0, 0u, pI, pE), h1 = qco(tq, 0, 2u, pI, pE);   // top leg 0
  const T m0 = qco(tq, 0, 1u, pI, pE), m1 = qco(tq, 0, 3u, pI, pE);   // top leg 1
  T x[2][2], u[2][2], out[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) x[a][b] = X[at(a, b)];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) u[a][b] = fma(k1, x[a][b ^ 1], k0 * x[a][b]);
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const T uf = u[a ^ 1][b];
      out[a][b] = bb * fma(a1, fma(m1, uf, m0 * u[a][b]), a0 * fma(h1, uf, h0 * u[a][b]));
    }
  if constexpr (UPD) {
    reg_update16(out, ms, jb, at, (lane & 3) == 0, upd);
  } else {
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b) stage[(g << 4) + at(a, b)] = out[a][b];
  }
  __syncwarp();
}

// Eight blocks of one row of 4 nodes: a lane takes the assignments (x0, x2,
// y0, y2) of the four side legs that the qubits see with (x2, y2) = lane bits
// and x0, y0 in registers; the legs at the checks are tied to the row leg.
// The group sums over x0, x2, y0, y2 in that order.
template <typename T, bool GM, bool UPD>
__device__ __forceinline__ void row_pass(T* stage, T pI, T pE, const RegMsgs<T, GM>& ms, const RegJob<T, GM>& jb,
                                         int lane, const RegUpd<T>& upd) {
  const int x2 = (lane >> 1) & 1, y2 = lane & 1, g = lane >> 2;
  const bool srev = jb.srev();
  const int s3 = srev ? 1 : 8, s2 = srev ? 2 : 4, s1 = srev ? 4 : 2, s0 = srev ? 8 : 1;   // strides of side legs 0 .. 3
  const int ia = (int)(jb.id & 3u), ib = (int)((jb.id >> 2) & 3u);
  const T* X = ms.at(jb.cq, jb.in());
  const T in0 = X[0], in1 = X[1];
  T pq[2][2][2];                                           // [x0][y0][r]
  if (!jb.chk0()) {
    // qubit, check, qubit, check: the qubits see legs 0 (x0, y0) and 2 (x2,
    // y2); the checks tie legs 1 to the row leg l1 and legs 3 to r.
    const T* A = ms.at(jb.cq, jb.up()) + (x2 ? s1 : 0);
    const T* B = ms.at(jb.cq, jb.lo()) + (y2 ? s1 : 0);
    T mA[2][2][2], mB[2][2][2];                            // [leg 0][leg 1][leg 3]
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int o = (a ? s3 : 0) + (b ? s2 : 0) + (c ? s0 : 0);
          mA[a][b][c] = A[o];
          mB[a][b][c] = B[o];
        }
#pragma unroll
    for (int x0 = 0; x0 < 2; ++x0)
#pragma unroll
      for (int y0 = 0; y0 < 2; ++y0) {
        T* part = pq[x0][y0];
        part[0] = part[1] = T(0);
#pragma unroll
        for (int l1 = 0; l1 < 2; ++l1) {
          T g0, g1;
          qpair(ia, x0 ^ y0, pI, pE, g0, g1);
          const T hh = l1 ? in0 * g1 + in1 * g0 : in0 * g0 + in1 * g1;
#pragma unroll
          for (int r = 0; r < 2; ++r) part[r] += hh * mA[x0][l1][r] * mB[y0][l1][r] * qval(ib, l1 ^ r, x2 ^ y2, pI, pE);
        }
      }
  } else {
    // check, qubit, check, qubit: the qubits see legs 1 (x0, y0) and 3 (x2,
    // y2); the checks tie legs 0 to l0 and legs 2 to l2.
    const T* A = ms.at(jb.cq, jb.up()) + (x2 ? s0 : 0);
    const T* B = ms.at(jb.cq, jb.lo()) + (y2 ? s0 : 0);
#pragma unroll
    for (int x0 = 0; x0 < 2; ++x0)
#pragma unroll
      for (int y0 = 0; y0 < 2; ++y0) {
        T* part = pq[x0][y0];
        part[0] = part[1] = T(0);
#pragma unroll
        for (int l0 = 0; l0 < 2; ++l0)
#pragma unroll
          for (int l2 = 0; l2 < 2; ++l2) {
            const int o = (l0 ? s3 : 0) + (l2 ? s1 : 0);
            const T w = (l0 ? in1 : in0) * A[o + (x0 ? s2 : 0)] * B[o + (y0 ? s2 : 0)] *
                        qval(ia, l0 ^ l2, x0 ^ y0, pI, pE);
            part[0] += w * qval(ib, l2, x2 ^ y2, pI, pE);
            part[1] += w * qval(ib, l2 ^ 1, x2 ^ y2, pI, pE);
          }
      }
  }
  T part[2];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    T s0v = pq[0][0][r] + pq[1][0][r], s1v = pq[0][1][r] + pq[1][1][r];
    s0v += shx(s0v, 2);
    s1v += shx(s1v, 2);
    part[r] = s0v + s1v;
    part[r] += shx(part[r], 1);
  }
  if constexpr (UPD) {
    reg_update2(part[0], part[1], ms, jb, (lane & 3) == 0, upd);
  } else {
    if ((lane & 3) < 2) stage[(g << 4) + (lane & 3)] = (lane & 1) ? part[1] : part[0];
  }
  __syncwarp();
}

// Eight single nodes: the legs (l, a, b, r), a and r in the lanes, summed
// over l, a, b in that order.
template <typename T, bool GM, bool UPD>
__device__ __forceinline__ void dot_pass(T* stage, T pI, T pE, const RegMsgs<T, GM>& ms, const RegJob<T, GM>& jb,
                                         int lane, const RegUpd<T>& upd) {
  const int a = (lane >> 1) & 1, r = lane & 1, g = lane >> 2;
  const bool chk = jb.chk0();
  const int id = (int)(jb.id & 3u);
  const T* X = ms.at(jb.cq, jb.in());
  const T* B = ms.at(jb.cq, jb.lo());
  const T ma = ms.at(jb.cq, jb.up())[a];
  T s[2];
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    T v[2];
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      const T nv = chk ? ((l == r && a == r && b == r) ? T(1) : T(0)) : qval(id, l ^ r, a ^ b, pI, pE);
      v[l] = X[l] * ma * B[b] * nv;
    }
    s[b] = radd(v[0], v[1]);
    s[b] += shx(s[b], 2);
  }
  const T v = s[0] + s[1];
  const T w = shx(v, 1);                                   // the other entry
  if constexpr (UPD) {
    reg_update2(r ? w : v, r ? v : w, ms, jb, (lane & 3) == 0, upd);
  } else {
    if ((lane & 3) < 2) stage[(g << 4) + r] = v;
  }
  __syncwarp();
}

// ---------------------------------------------------------------------------
// Updates of the blocks three nodes wide or high that the last block row and
// column hold at even d, in the roundings of the node-by-node form
// (fused_sweep, as compiled), whose bits they reproduce: of a butterfly's two
// terms the input with row bit 1 is the fused one.  Through that form these
// blocks, a quarter of the messages at d = 12, took most of the time.  Eight
// jobs a pass, four lanes each, as above.  2000 syndromes at d = 12, p = 0.10:
// 11.1 -> 2.9 ms.

// Table entry g[al][be] of the qubit in field f.
template <typename T>
__device__ __forceinline__ T qat(unsigned id, int f, int al, int be, T pI, T pE) {
  return ((id >> (2 * f)) & 3u) == (unsigned)((al << 1) | be) ? pI : pE;
}
// Butterfly over a row bit held by lane bit `mask`, r the lane's own.
template <typename T>
__device__ __forceinline__ T lane_bf(T x, int mask, int r, T g0, T g1) {
  const T y = shx(x, mask);
  return fma(r ? x : y, r ? g0 : g1, r ? y * g1 : x * g0);
}
// First qubit of a column, its row bit in registers: inputs x[l], output r,
// the upper leg u given (in the table entries) or summed.
template <typename T>
__device__ __forceinline__ T reg_bf(T x0, T x1, int r, T g0, T g1) {
  return r ? fma(x1, g0, x0 * g1) : fma(x1, g1, x0 * g0);
}
template <typename T>
__device__ __forceinline__ T reg_bf4(T x00, T x01, T x10, T x11, T ga, T gb, T gc, T gd) {   // x[l][u]
  return fma(x11, gd, fma(x10, gc, fma(x00, ga, x01 * gb)));
}

// The update of an 8-entry vector out[q0], (r1, r2) = lane bits: reg_update16
// with sums over r0, r1, r2.
template <typename T, bool GM>
__device__ __forceinline__ void reg_update8(const T (&out)[2], const RegMsgs<T, GM>& ms, const RegJob<T, GM>& jb,
                                            int lane, const RegUpd<T>& up) {
  T* old = ms.out(jb.cq, jb.out()) + (lane & 3);
  auto sum = [&](T a, T b) {
    T v = radd(a, b);
    v = radd(v, shx(v, 2));
    return radd(v, shx(v, 1));
  };
  const T y0 = old[0], y1 = old[4];
  const T i1 = inv_norm(sum(out[0] * out[0], out[1] * out[1]));
  T x0 = fma(up.one_m_eta, out[0] * i1, up.eta * y0), x1 = fma(up.one_m_eta, out[1] * i1, up.eta * y1);
  const T i2 = inv_norm(sum(x0 * x0, x1 * x1));
  x0 = x0 * i2;
  x1 = x1 * i2;
  T term;
  if constexpr (sizeof(T) == 4) {
    const T t0 = x0 - y0, t1 = x1 - y1;
    const T sq = sum(t0 * t0, t1 * t1);
    term = sq * fma(T(-0.5), sq, T(2));
  } else {
    const T o = sum(x0 * y0, x1 * y1);
    term = fma(T(-2) * o, o, T(2));
  }
  if (jb.on) {
    old[0] = x0;
    old[4] = x1;
    if ((lane & 3) == 0) up.ovl[jb.cq * up.M + jb.out()] = term;
  }
}

// 4 x 3: columns Q (qubits at 0, 2), C (1, 3), Q; column 0 lies on the grid
// border (no incoming message), the lower side has a message, the upper one
// unless the block is in the first row.  (r1, r3) = lane bits, r0, r2 = q0, q2.
template <typename T, bool GM>
__device__ __forceinline__ void pass43(T pI, T pE, const RegMsgs<T, GM>& ms, const RegJob<T, GM>& jb, int lane,
                                       const RegUpd<T>& upd) {
  const int r1 = (lane >> 1) & 1, r3 = lane & 1;
  const unsigned id = jb.id;
  const bool a = jb.up() < ms.M, srev = jb.srev();
  const T* A = ms.at(jb.cq, jb.up());
  const int s0 = srev ? 1 : 4, s2 = srev ? 4 : 1;            // strides of side legs 0 and 2 (leg 1: 2)
  const T* B = ms.at(jb.cq, jb.lo()) + (r3 ? s2 : 0);        // only its leg 2 = r3 reaches column 2's rows
  // Column 0: the incoming side is e_0 at the qubits, so each output is a
  // product of two table entries.  Column 1's upper side message over a0
  // (v = r0) leaves its leg 2.
  T x[2][2][2];                                              // [a2][q0][q2]
#pragma unroll
  for (int q0 = 0; q0 < 2; ++q0)
#pragma unroll
    for (int q2 = 0; q2 < 2; ++q2) {
      const T g2 = qat(id, 1, q2, r1 ^ r3, pI, pE);
      const T e0 = qat(id, 0, q0, r1, pI, pE) * g2, e1 = qat(id, 0, q0, r1 ^ 1, pI, pE) * g2;   // a0 = 0, 1
#pragma unroll
      for (int a2 = 0; a2 < 2; ++a2) {
        const T* m = A + 2 * q0 + (a2 ? s2 : 0);
        x[a2][q0][q2] = a ? fma(m[s0], e1, m[0] * e0) : (a2 ? T(0) : e0);
      }
    }
  // Qubit 1, then qubit 3 with l3 = b0, and the lower message over b0 and w.
  T z[2][2][2];
  const T b00 = B[0], b01 = B[2], b10 = B[s0], b11 = B[s0 + 2];
#pragma unroll
  for (int q0 = 0; q0 < 2; ++q0)
#pragma unroll
    for (int q2 = 0; q2 < 2; ++q2) {
      const T g0 = qat(id, 2, 0, q0 ^ q2, pI, pE), g1 = qat(id, 2, 1, q0 ^ q2, pI, pE);
      const T h00 = qat(id, 3, r3, q2, pI, pE), h01 = qat(id, 3, r3, q2 ^ 1, pI, pE);           // b0 = 0; w = 0, 1
      const T h10 = qat(id, 3, r3 ^ 1, q2, pI, pE), h11 = qat(id, 3, r3 ^ 1, q2 ^ 1, pI, pE);   // b0 = 1
#pragma unroll
      for (int a2 = 0; a2 < 2; ++a2) {
        const T t = lane_bf(x[a2][q0][q2], 2, r1, g0, g1);
        const T t0 = __shfl_sync(kFull, t, lane & ~1), t1 = __shfl_sync(kFull, t, lane | 1);
        const T v = fma(b00, t0 * h00, b01 * (t0 * h01));
        z[a2][q0][q2] = radd(v, fma(b10, t1 * h10, b11 * (t1 * h11)));
      }
    }
  // Column 2: qubit 0 with its upper leg a2 summed, then qubit 2.
  const T g0 = qat(id, 4, 0, r1, pI, pE), g1 = qat(id, 4, 1, r1, pI, pE);
  const T h0 = qat(id, 4, 0, r1 ^ 1, pI, pE), h1 = qat(id, 4, 1, r1 ^ 1, pI, pE);
  const T k0 = qat(id, 5, 0, r1 ^ r3, pI, pE), k1 = qat(id, 5, 1, r1 ^ r3, pI, pE);
  T out[2][2];
#pragma unroll
  for (int q0 = 0; q0 < 2; ++q0) {
    T y[2];
#pragma unroll
    for (int q2 = 0; q2 < 2; ++q2)
      y[q2] = q0 ? reg_bf4(z[0][0][q2], z[1][0][q2], z[0][1][q2], z[1][1][q2], g1, h1, g0, h0)
                 : reg_bf4(z[0][0][q2], z[1][0][q2], z[0][1][q2], z[1][1][q2], g0, h0, g1, h1);
    out[q0][0] = fma(y[1], k1, y[0] * k0);
    out[q0][1] = fma(y[1], k0, y[0] * k1);
  }
  reg_update16(out, ms, jb, RowAt(false, r1, r3), (lane & 3) == 0, upd);
  __syncwarp();
}

// 3 x 4 (chains of three nodes ending on the grid border: no lower message,
// the upper one always), and 3 x 3 (the corner block: no incoming message
// either).  r0 = q0, (r1, r2) = lane bits.  A qubit at position 2 has no lower
// leg (beta = r1), a check there no constraint.
template <typename T, bool GM, bool CORNER>
__device__ __forceinline__ void pass3(T pI, T pE, const RegMsgs<T, GM>& ms, const RegJob<T, GM>& jb, int lane,
                                      const RegUpd<T>& upd) {
  const int r1 = (lane >> 1) & 1, r2 = lane & 1;
  const unsigned id = jb.id;
  const bool srev = jb.srev(), chk0 = jb.chk0();
  const T* A = ms.at(jb.cq, jb.up());
  auto bf1 = [&](T x, int f, int q0) {                       // qubit 1 of a C column, field f
    return lane_bf(x, 2, r1, qat(id, f, 0, q0 ^ r2, pI, pE), qat(id, f, 1, q0 ^ r2, pI, pE));
  };
  auto bf2 = [&](T x, int f) {                               // qubit 2 of a Q column, field f
    return lane_bf(x, 1, r2, qat(id, f, 0, r1, pI, pE), qat(id, f, 1, r1, pI, pE));
  };
  auto first4 = [&](T x00, T x01, T x10, T x11, int f, int r) {   // qubit 0 with u summed, x[l][u]
    const T ga = qat(id, f, r, r1, pI, pE), gb = qat(id, f, r, r1 ^ 1, pI, pE);
    const T gc = qat(id, f, r ^ 1, r1, pI, pE), gd = qat(id, f, r ^ 1, r1 ^ 1, pI, pE);
    return reg_bf4(x00, x01, x10, x11, ga, gb, gc, gd);
  };
  T out[2] = {T(0), T(0)};
  if constexpr (CORNER) {
    const int s0 = srev ? 1 : 4, s2 = srev ? 4 : 1;          // strides of side legs 0 and 2 (leg 1: 2)
    T z[2][2];                                               // [a2][r0]
#pragma unroll
    for (int q0 = 0; q0 < 2; ++q0) {
      const T g2 = qat(id, 1, r2, r1, pI, pE);
      const T e0 = qat(id, 0, q0, r1, pI, pE) * g2, e1 = qat(id, 0, q0, r1 ^ 1, pI, pE) * g2;   // a0 = 0, 1
#pragma unroll
      for (int a2 = 0; a2 < 2; ++a2) {
        const T* m = A + 2 * q0 + (a2 ? s2 : 0);
        z[a2][q0] = bf1(fma(m[s0], e1, m[0] * e0), 2, q0);
      }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) out[r] = bf2(first4(z[0][0], z[1][0], z[0][1], z[1][1], 4, r), 5);
  } else {
    const int s0 = srev ? 1 : 8, s1 = srev ? 2 : 4, s2 = srev ? 4 : 2, s3 = srev ? 8 : 1;   // strides of the side legs
    const T* X = ms.at(jb.cq, jb.in()) + (lane & 3);
    const T x0 = X[0], x1 = X[4];
    // The lists keep the two forms apart, so a pass mostly runs one; where it
    // holds both, each job keeps its own.
    if (__any_sync(kFull, !chk0)) {  // Q, C, Q, C
      T y[2][2];                                             // [a0][r0], a0 = u
#pragma unroll
      for (int a0 = 0; a0 < 2; ++a0) {
        const T g0 = qat(id, 0, 0, a0 ^ r1, pI, pE), g1 = qat(id, 0, 1, a0 ^ r1, pI, pE);
#pragma unroll
        for (int r = 0; r < 2; ++r) y[a0][r] = bf1(bf2(reg_bf(x0, x1, r, g0, g1), 1), 2, r);
      }
      // The message over a0 (a1 = l0) and, at qubit 0, its leg 2 = u; leg 3 = r0 of the last column.
      T w[2][2][2];                                          // [leg 3][u][l0]
#pragma unroll
      for (int l0 = 0; l0 < 2; ++l0)
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int a3 = 0; a3 < 2; ++a3) {
            const T* m = A + (l0 ? s1 : 0) + (u ? s2 : 0) + (a3 ? s3 : 0);
            w[a3][u][l0] = fma(m[s0], y[1][l0], m[0] * y[0][l0]);
          }
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const T v = bf1(bf2(first4(w[r][0][0], w[r][1][0], w[r][0][1], w[r][1][1], 4, r), 5), 6, r);
        out[r] = chk0 ? out[r] : v;
      }
    }
    if (__any_sync(kFull, chk0)) {   // C, Q, C, Q
      const T c0 = bf1(x0, 0, 0), c1 = bf1(x1, 0, 1);        // a0 = r0
      T w[2][2];                                             // [leg 3][r0]
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        T y[2][2];                                           // [a0][a1]: qubit 0 with l0 = a0, a1 = u
#pragma unroll
        for (int a0 = 0; a0 < 2; ++a0)
#pragma unroll
          for (int a1 = 0; a1 < 2; ++a1)
            y[a0][a1] = bf2((a0 ? c1 : c0) * qat(id, 2, a0 ^ r, a1 ^ r1, pI, pE), 3);
#pragma unroll
        for (int a3 = 0; a3 < 2; ++a3) {
          const T* m = A + (r ? s2 : 0) + (a3 ? s3 : 0);     // leg 2 = r0
          const T v = fma(m[s0 + s1], y[1][1], fma(m[s0], y[1][0], fma(m[s1], y[0][1], m[0] * y[0][0])));
          w[a3][r] = bf1(v, 4, r);
        }
      }
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const T v = bf2(first4(w[0][0], w[1][0], w[0][1], w[1][1], 6, r), 7);
        out[r] = chk0 ? v : out[r];
      }
    }
  }
  reg_update8(out, ms, jb, lane, upd);
  __syncwarp();
}

template <typename T, bool GM, bool UPD, int SHAPE>
__device__ __forceinline__ void reg_pass(T* stage, T pI, T pE, const RegMsgs<T, GM>& ms, const RegJob<T, GM>& jb,
                                         int lane, const RegUpd<T>& upd) {
  if constexpr (SHAPE == kShapeQuad) quad_pass<T, GM, UPD>(stage, pI, pE, ms, jb, lane, upd);
  else if constexpr (SHAPE == kShapeCol) col_pass<T, GM, UPD>(stage, pI, pE, ms, jb, lane, upd);
  else if constexpr (SHAPE == kShapeRow) row_pass<T, GM, UPD>(stage, pI, pE, ms, jb, lane, upd);
  else if constexpr (SHAPE == kShapeDot) dot_pass<T, GM, UPD>(stage, pI, pE, ms, jb, lane, upd);
  else if constexpr (SHAPE == kShape43) pass43<T, GM>(pI, pE, ms, jb, lane, upd);
  else pass3<T, GM, SHAPE == kShape33>(pI, pE, ms, jb, lane, upd);
}

// Message item of job j when every message has n jobs (n = 1 .. 4).
__device__ __forceinline__ int job_item(int j, int n) { return n == 4 ? j >> 2 : n == 2 ? j >> 1 : n == 1 ? j : j / 3; }

// This warp's passes over the cnt messages of one shape whose tasks start at
// list position pos0, n cosets (cos_of) each: passes are dealt to the NW
// warps in turn, `first` counting those of the shapes before.  Returns the
// passes of this shape.
template <typename T, bool GM, int SHAPE, int NW>
__device__ __forceinline__ int reg_updates(T* stage, T pI, T pE, const RegMsgs<T, GM>& ms, const RegTask* tasks,
                                           const uint16_t* qid, int M, int pos0, int cnt, unsigned cos_of, int n,
                                           int first, int warp, int lane, const RegUpd<T>& upd) {
  const int passes = (cnt * n + 7) >> 3;
  int p = warp - first % NW;
  if (p < 0) p += NW;
  for (; p < passes; p += NW) {
    const int j = p * 8 + (lane >> 2);
    RegJob<T, GM> jb;
    int item = job_item(j, n);
    const int slot = j - item * n;
    jb.on = item < cnt;
    if (!jb.on) item = cnt - 1;
    jb.cq = (int)((cos_of >> (2 * slot)) & 3u);
    const int pos = pos0 + item;
    jb.q = tasks[pos];
    jb.id = qid[jb.cq * M + pos];
    reg_pass<T, GM, true, SHAPE>(stage, pI, pE, ms, jb, lane, upd);
  }
  return passes;
}

}  // namespace bbp
