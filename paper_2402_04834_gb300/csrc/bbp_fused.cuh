// Fused-block BP (Remark 9; the form the paper ran for k = 1, 2, 4): every
// k x k block acts as one vertex with four legs of dimension 2^k and the
// messages are dense vectors, so there is no MPS truncation at all.  Where
// the MPS form of Sec. III.D truncates nothing, both compute the same
// numbers.
//
// One CTA decodes G of the four cosets of one syndrome (G = 1, 2 or 4); all
// their messages live in shared memory (G x M dense vectors of 2^k).  The
// cosets share the network's geometry, and every node off the first row
// and column has the same Pauli frame in all of them (the logical strings
// of Sec. II run along row 0 and column 0), so a warp updates one directed
// block edge for all cosets of the CTA that are still iterating at once:
// index arithmetic, node tables and synchronisation are paid once for G
// vectors.  A coset whose Delta drops below delta0 is frozen (its messages
// and iteration count stay as they were), exactly as if it ran alone.
//
// A warp contracts one block with its incoming messages node by node on a
// dense state indexed by
//     [slot | a | rows of the chain | b | v]   (most to least significant bits)
// where slot picks the coset, v is the vertical leg inside the current
// column and a / b carry the top / bottom side message.  A side message
// m(t_0 .. t_{w-1}) is fed one leg per column through its exact copy / data /
// copy factorisation: the first floor(w/2) legs are recorded in a, the
// middle column contracts a with m and leaves in a the values expected for
// the remaining legs, which the last columns check off.  All dimensions are
// powers of two, so every index is a bit field.  Every loop is bounded and
// no CTA waits on another.
#pragma once

#include "bbp_kernels.cuh"
#include "bbp_block6.cuh"
#include "bbp_reg.cuh"

namespace bbp {

constexpr int kFusedK = 4;                 // block side of the learned warm start's messages
constexpr int kFusedVec = 1 << kFusedK;    // their dense length
constexpr int kFusedMaxG = 4;              // cosets per CTA

// Sizes of the kernels compiled for block sides up to K (K = 4 or 6): dense
// messages of 2^K entries and a per-coset state of at most 2^(2K) entries
// (a block with h rows and nc columns never holds more than h + nc bits:
// a and b together carry at most nc).
template <int K> struct FusedDim {
  static constexpr int vec = 1 << K;
  static constexpr int slot = 1 << (2 * K);
};

// Per-warp scratch for G cosets, carved from shared memory.
template <typename T>
struct FusedWS {   // (sizes for block side K: slot = FusedDim<K>::slot, vec = FusedDim<K>::vec)
  T* s0;   // state, G * slot; at k = 4 also the register form's staging (kRegStage <= slot)
  T* s1;   // state, G * slot
  T* wn;   // node tensors, 16 per coset
  T* mt;   // side message A in consumption order, vec per coset
  T* mb;   // side message B in consumption order, vec per coset
};

// Entries of a state buffer.  lean at k = 4: every block update of the
// kernel runs in register form, whose staging is all a warp needs.  lean at
// k = 5, 6: full 6 x 6 blocks are updated column by column in registers
// (bbp_block6.cuh), so the buffers need only hold that form's states and the
// node-by-node states of the partial blocks; the read-out, which contracts
// full blocks node by node, takes full-size buffers from the same memory with
// fewer warps.
template <int K>
BBP_HD int fused_slot(int lean) {
  return K <= 4 || !lean ? FusedDim<K>::slot : kBlock6Buf;
}

// Geometries whose block states at k = 5, 6 fit the small buffers: all but
// those with 6 x 5 blocks, whose widest state has 2^11 entries (k = 6 and d a
// multiple of 3).  With buffers of that size at most 8 FP32 warps, and fewer
// than 8 in FP64, would fit an SM; these distances take the kernels with
// full-size buffers (6 warps, 3 in FP64).
BBP_HD bool small_states(const Geo& g) { return g.k == 5 || (g.k == 6 && g.W % 6 != 5); }

template <typename T, int K>
BBP_HD int fused_ws_bytes(int G, int lean = 0) {
  if (K == 4 && lean) return align_up((int)sizeof(T) * kRegStage, 16);
  return align_up((int)sizeof(T) * G * (2 * fused_slot<K>(lean) + 16 + 2 * FusedDim<K>::vec), 16);
}

template <typename T, int K>
__device__ __forceinline__ FusedWS<T> fused_ws_at(unsigned char* base, int G, int slot) {
  static_assert(K != 4 || kRegStage <= FusedDim<K>::slot, "the staging fits in a state buffer");
  FusedWS<T> w;
  T* p = reinterpret_cast<T*>(base);
  w.s0 = p;
  w.s1 = p + G * slot;
  w.wn = p + 2 * G * slot;
  w.mt = w.wn + 16 * G;
  w.mb = w.mt + FusedDim<K>::vec * G;
  return w;
}

// Geometries whose every block has a register form at k = 4: the last
// block row / column is one node wide (W = 4 n + 1, every odd d).
BBP_HD bool register_form_only(const Geo& g) { return g.k == 4 && g.W % 4 == 1; }

// Scalars from one coset's messages to the next in shared memory: at k <= 4
// the border vectors follow the messages, and the offset of half a vector
// puts the same message of two cosets in different banks.
template <int K>
BBP_HD int fused_coset_stride(int M, bool gm) {
  if (K > 4 || gm) return M * FusedDim<K>::vec;
  return (M + kBorderVecs) * FusedDim<K>::vec + 8;
}

// Shared-memory layout of one fused CTA.
struct FusedLayout {
  int parity, frame, msg_of, meta, work, ovl, rlog, misc, tasks, qid, border, msgs, ws, ws_stride, total;
};

// gm: the messages live in a workspace slot of the CTA (always for k = 5,
// 6; on request for k <= 4), not in shared memory.  lean: the kernels with
// small per-warp buffers; at k = 4, 1 where every block is four or one node
// wide, 2 where any distance may come: blocks three nodes wide are then read
// out node by node by kReadWarps warps, a coset at a time, in the buffers'
// place.
constexpr int kReadWarps = 4;
constexpr int kEvenLB = 10;                 // template argument LB of the kernels with lean = 2: kEvenLB + CTAs per SM
template <typename T, int K>
BBP_HD FusedLayout fused_layout(const Geo& g, int M, int nwarps, int G, bool gm = (K > 4), int lean = 0) {
  FusedLayout L;
  int o = 0;
  L.parity = o; o = align_up(o + 2 * g.d * 8, 16);             // the pure error, as prefix parities
  L.frame = o;  if (lean != 1 || K > 4) o = align_up(o + G * g.W * g.W, 16);
  L.msg_of = o; if (lean != 1 || K > 4) o = align_up(o + 2 * g.nb * g.nb * 4, 16);
  L.meta = o;   o = align_up(o + 2 * M, 16);
  L.work = o;   o = align_up(o + 2 * M, 16);                   // lists of both colours
  L.ovl = o;    o = align_up(o + (int)sizeof(T) * G * M, 16);
  L.rlog = o;   o = align_up(o + 8 * G * (g.nb * g.nb + M / 2), 16);
  L.misc = o;   o = align_up(o + 336, 16);
  // Register form (k = 4): a task per message and the qubit ids of each
  // (coset, message), by list position, built once per syndrome.
  L.tasks = o;  if (K == 4 && g.k == 4) o = align_up(o + (int)sizeof(RegTask) * M, 16);
  L.qid = o;    if (K == 4 && g.k == 4) o = align_up(o + 2 * G * M, 16);
  L.border = o; if (K == 4 && gm) o = align_up(o + (int)sizeof(T) * kBorderVecs * kRegVec, 16);
  L.msgs = o;   // the messages, unless they live in the workspace
  if (!gm) o = align_up(o + (int)sizeof(T) * G * fused_coset_stride<K>(M, gm), 16);
  L.ws = o;
  L.ws_stride = fused_ws_bytes<T, K>(G, lean);
  int ws = nwarps * L.ws_stride;
  if (K == 4 && lean == 2) ws = imax(ws, kReadWarps * fused_ws_bytes<T, K>(1));
  o = align_up(o + ws, 16);
  L.total = o;
  return L;
}

template <typename T> struct Vec2;
template <> struct Vec2<float> { using type = float2; };
template <> struct Vec2<double> { using type = double2; };

// (Index fields below occupy disjoint bits; they are added rather than or-ed
// so that the compiler can advance the addresses instead of rebuilding them.)
//
// The data column of side message A with SD recorded legs and NF legs still
// to come (k = 5, 6: NF = 2), one coset, the message in registers: each
// lane takes groups hbv of (rows, b), reads in[a, hbv] for the 2^SD values
// of a once and writes out[a2, hbv, v] = sum_a m[a, v, a2] in[a, hbv].
template <typename T, int SD, int NF>
__device__ __forceinline__ void data_column_a(const T* mt, const T* cur, T* nxt, int ib, int ob, int hb,
                                              int lane) {
  using V2 = typename Vec2<T>::type;
  constexpr int NA = 1 << SD, NO = 1 << NF, NM = 1 << (SD + 1 + NF);
  T mr[NM];
#pragma unroll
  for (int i = 0; i < NM; ++i) mr[i] = mt[i];
  const int low = (1 << hb) - 1;
  for (int hbv = lane; hbv <= low; hbv += 32) {
    T x[NA];
#pragma unroll
    for (int a = 0; a < NA; ++a) x[a] = cur[ib + (a << hb) + hbv];
#pragma unroll
    for (int a2 = 0; a2 < NO; ++a2) {
      T s0 = T(0), s1 = T(0);
#pragma unroll
      for (int a = 0; a < NA; ++a) {
        s0 += mr[((a << 1) << NF) | a2] * x[a];
        s1 += mr[(((a << 1) | 1) << NF) | a2] * x[a];
      }
      V2 o;
      o.x = s0; o.y = s1;
      *reinterpret_cast<V2*>(nxt + 2 * (ob + (a2 << hb) + hbv)) = o;
    }
  }
}

// The data column of side message B (SD recorded legs, NF to come), one
// coset: each lane takes groups al of (a, rows), reads the 2^SD pairs
// in[al, b, v] once and writes out[al, b2] = sum_{b,v} m[b, v, b2] in[al, b, v].
template <typename T, int SD, int NF>
__device__ __forceinline__ void data_column_b(const T* mb, const T* cur, T* nxt, int ab0, int hah, int lane) {
  using V2 = typename Vec2<T>::type;
  constexpr int NB = 1 << SD, NO = 1 << NF, NM = 1 << (SD + 1 + NF);
  T mr[NM];
#pragma unroll
  for (int i = 0; i < NM; ++i) mr[i] = mb[i];
  for (int al = lane; al < (1 << hah); al += 32) {
    const int ah = ab0 + al;
    V2 x[NB];
#pragma unroll
    for (int b = 0; b < NB; ++b) x[b] = *reinterpret_cast<const V2*>(cur + (((ah << SD) + b) << 1));
#pragma unroll
    for (int b2 = 0; b2 < NO; ++b2) {
      T val = T(0);
#pragma unroll
      for (int b = 0; b < NB; ++b)
        val += mr[((b << 1) << NF) | b2] * x[b].x + mr[(((b << 1) | 1) << NF) | b2] * x[b].y;
      nxt[(ah << NF) | b2] = val;
    }
  }
}

__device__ __forceinline__ int bitrev(int x, int w) {
  return (int)(__brev((unsigned)x) >> (32 - w));
}

struct FState {
  int ab, h, bb, hv;   // bit widths of a, rows, b, v (per coset)
  __device__ __forceinline__ int bits() const { return ab + h + bb + hv; }
  __device__ __forceinline__ int size() const { return 1 << bits(); }
};

// Coset (0 .. G-1 within the CTA) held by slot s; slots are packed 2 bits each.
__device__ __forceinline__ int slot_coset(unsigned cos_of, int s) { return (int)((cos_of >> (2 * s)) & 3u); }

// The qubit table g[alpha][beta] = pi(f (+) (x, z)) of an interior qubit:
// one of x, z is the parity of its in/out legs (alpha), the other the
// parity of its chain legs (beta); alpha is z for horizontal-edge qubits
// swept along rows and for vertical-edge qubits swept along columns.
// Exactly one entry is pi(I): the one whose (x, z) equals the frame's
// (fx, fz), at index q = (alpha, beta) = (fz, fx) = the frame byte itself
// when alpha is z, and (fx, fz) = the byte with its two bits swapped when
// alpha is x.
template <typename T, int K>
__device__ __forceinline__ void qubit_table(const Ctx<T, K>& c, int qi, int qj, bool rowwise, T gt[4]) {
  const int fr = c.frame[qi * c.g.W + qj];
  const bool alpha_is_z = ((qi & 1) == 0) == rowwise;
  const int qi_id = alpha_is_z ? fr : (((fr & 1) << 1) | (fr >> 1));
#pragma unroll
  for (int q = 0; q < 4; ++q) gt[q] = q == qi_id ? c.pI : c.pE;
}

// Log of a product of positive factors, for the read-out (Lemma 1).  FP64
// sums the factors' logs; FP32 keeps the product as a float mantissa and a
// binary exponent and takes one FP64 log at the end (FP64 issues at 1/64
// of the FP32 rate here).  Used by one lane.
template <typename T> struct LogAcc;
template <> struct LogAcc<double> {
  double s = 0.0;
  __device__ __forceinline__ void mul(double x) { s += log(x); }
  __device__ __forceinline__ double value() const { return s; }
};
template <> struct LogAcc<float> {
  float m = 1.f;
  int e = 0;
  __device__ __forceinline__ void mul(float x) {
    int ex;
    m *= frexpf(x, &ex);
    e += ex;
    m = frexpf(m, &ex);
    e += ex;
  }
  __device__ __forceinline__ void mul(const LogAcc<float>& o) {
    int ex;
    m = frexpf(m * o.m, &ex);
    e += o.e + ex;
  }
  __device__ __forceinline__ double value() const { return log((double)m) + (double)e * 0.6931471805599453; }
};

// Contract block f (rotated so that f.dir points right) with its incoming
// dense messages for the n cosets of cos_of (messages of coset q at
// msgs + q * stride; c.frame is the frame of slot 0's coset and frames holds
// all G frames).  Leaves the outgoing vectors over the chain in ws.s0, slot
// s at s << h.  For the read-out (ls not null) every column's state is
// renormalised per coset and the norms taken out go to ls[slot] (lane 0).
template <typename T, int K>
__device__ __forceinline__ void fused_sweep_body(const FusedWS<T>& ws, const Ctx<T, K>& c, const T* msgs, int stride,
                                                 unsigned cos_of, int n, const uint8_t* frames, const Frame& f,
                                                 LogAcc<T>* ls, int lane) {
  using V2 = typename Vec2<T>::type;
  const int h = f.h, nc = f.ncols;
  T* cur = ws.s0;
  T* nxt = ws.s1;
  // Initial state: the message on the side opposite the outgoing one.
  for (int e = lane; e < (n << h); e += 32) {
    const int H = e & ((1 << h) - 1);
    const T* ms = msgs + slot_coset(cos_of, e >> h) * stride;
    cur[e] = f.in_idx >= 0 ? ms[f.in_idx * FusedDim<K>::vec + H] : (H == 0 ? T(1) : T(0));
  }
  // Side messages in consumption order.
  for (int e = lane; e < (n << nc); e += 32) {
    const int i = e & ((1 << nc) - 1);
    const int j = f.rev ? bitrev(i, nc) : i;
    const T* ms = msgs + slot_coset(cos_of, e >> nc) * stride;
    ws.mt[e] = f.a_idx >= 0 ? ms[f.a_idx * FusedDim<K>::vec + j] : T(0);
    ws.mb[e] = f.b_idx >= 0 ? ms[f.b_idx * FusedDim<K>::vec + j] : T(0);
  }
  __syncwarp();
  FState st{0, h, 0, 0};
  const int sd = nc >> 1;               // the column that holds the data site
  const int nf = nc - sd - 1;           // legs still expected after it
  const bool rowwise = f.dir == kDirR || f.dir == kDirL;
  const int WW = c.g.W * c.g.W;
  for (int t = 0; t < nc; ++t) {
    // Side message A: enters the column as its vertical leg v.  Output
    // entries come in pairs (v = 0, 1) sharing (slot, a, rows, b).
    {
      FState ns = st;
      ns.hv = 1;
      if (f.a_idx < 0) ns.ab = 0;
      else if (t < sd) ns.ab = st.ab + 1;
      else if (t == sd) ns.ab = nf;
      else ns.ab = st.ab - 1;
      const int np = n << (ns.bits() - 1);
      const int hb = h + st.bb;                        // bits of (rows, b)
      const int low = (1 << hb) - 1;
      if (K > 4 && t == sd && f.a_idx >= 0 && hb >= 5 && nf == 2 && (sd == 2 || sd == 3)) {
        for (int s = 0; s < n; ++s) {
          const int ib = s << (st.ab + hb), ob = s << (nf + hb);
          if (sd == 3) data_column_a<T, 3, 2>(ws.mt + (s << nc), cur, nxt, ib, ob, hb, lane);
          else data_column_a<T, 2, 2>(ws.mt + (s << nc), cur, nxt, ib, ob, hb, lane);
        }
      } else if (t == sd && f.a_idx >= 0 && hb >= 5 && nf <= 1) {
        // The data column, one coset at a time with its side message in
        // registers: each lane reads the 2^ab values in[a, rows, b] of its
        // (rows, b) once and writes all outputs (a2, v) of that group.
        const int na = 1 << st.ab;                     // st.ab = sd <= 2
        for (int s = 0; s < n; ++s) {
          T mr[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) mr[i] = i < (1 << nc) ? ws.mt[(s << nc) + i] : T(0);
          const int ib = s << (st.ab + hb), ob = s << (nf + hb);
          for (int hbv = lane; hbv <= low; hbv += 32) {
            T x[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) x[a] = a < na ? cur[ib + (a << hb) + hbv] : T(0);
            if (nf == 1) {
#pragma unroll
              for (int a2 = 0; a2 < 2; ++a2) {
                T s0 = T(0), s1 = T(0);
#pragma unroll
                for (int a = 0; a < 4; ++a) {
                  s0 += mr[(a << 2) | a2] * x[a];
                  s1 += mr[(((a << 1) | 1) << 1) | a2] * x[a];
                }
                V2 o;
                o.x = s0; o.y = s1;
                *reinterpret_cast<V2*>(nxt + 2 * (ob + (a2 << hb) + hbv)) = o;
              }
            } else {
              T s0 = T(0), s1 = T(0);
#pragma unroll
              for (int a = 0; a < 4; ++a) {
                s0 += mr[a << 1] * x[a];
                s1 += mr[(a << 1) | 1] * x[a];
              }
              V2 o;
              o.x = s0; o.y = s1;
              *reinterpret_cast<V2*>(nxt + 2 * (ob + hbv)) = o;
            }
          }
        }
      } else if (f.a_idx >= 0 && t < sd) {
        // Record v as a's new low bit: out[(slot, a, a'), hbv, v] = [a' = v]
        // in[(slot, a), hbv]; each input entry is read once and written to
        // both of its output pairs.
        const int nin = n << st.bits();
        constexpr int U = K > 4 ? 2 : 1;               // entries per lane and step (loads first)
        for (int e00 = lane; e00 < nin; e00 += 32 * U) {
          T xs[U];
          int es[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            es[u] = U == 1 ? e00 : min(e00 + 32 * u, nin - 1);
            xs[u] = cur[es[u]];
          }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int e = es[u];
            const int e0 = (((e >> hb) << 1) << hb) | (e & low);   // a' = 0
            V2 o0, o1;
            o0.x = xs[u]; o0.y = T(0);
            o1.x = T(0); o1.y = xs[u];
            *reinterpret_cast<V2*>(nxt + 2 * e0) = o0;
            *reinterpret_cast<V2*>(nxt + 2 * (e0 | (1 << hb))) = o1;
          }
        }
      } else if (K > 4 && f.a_idx >= 0 && t > sd) {
        // Move a's top bit into v: out[(slot, a), hbv, v] = in[(slot, v, a), hbv]
        // (two entries per lane and step, loads first).
        const int top = 1 << (st.ab - 1);
        for (int e20 = lane; e20 < np; e20 += 64) {
          V2 os[2];
          int es[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int e2 = min(e20 + 32 * u, np - 1);
            const int a2f = e2 >> hb, hbv = e2 & low;
            const int ai = ((a2f >> ns.ab) << st.ab) | (a2f & ((1 << ns.ab) - 1));
            os[u].x = cur[(ai << hb) | hbv];
            os[u].y = cur[((ai | top) << hb) | hbv];
            es[u] = e2;
          }
#pragma unroll
          for (int u = 0; u < 2; ++u) *reinterpret_cast<V2*>(nxt + 2 * es[u]) = os[u];
        }
      } else
      for (int e2 = lane; e2 < np; e2 += 32) {
        const int a2f = e2 >> hb, hbv = e2 & low;      // a2f = (slot, a); (rows, b) is shared by in and out
        V2 o;
        if (f.a_idx < 0) {
          o.x = cur[e2]; o.y = T(0);
        } else if (t < sd) {
          const T x = cur[((a2f >> 1) << hb) | hbv];
          if (a2f & 1) { o.x = T(0); o.y = x; } else { o.x = x; o.y = T(0); }
        } else if (t == sd) {
          const int s = a2f >> nf, a2 = a2f & ((1 << nf) - 1);
          const T* mt = ws.mt + (s << nc);
          const int ib = s << (st.ab + hb);
          T s0 = T(0), s1 = T(0);
          for (int a = 0; a < (1 << st.ab); ++a) {
            const T x = cur[ib | (a << hb) | hbv];
            s0 += mt[((a << 1) << nf) | a2] * x;
            s1 += mt[(((a << 1) | 1) << nf) | a2] * x;
          }
          o.x = s0; o.y = s1;
        } else {
          const int ai = ((a2f >> ns.ab) << st.ab) | (a2f & ((1 << ns.ab) - 1));
          o.x = cur[(ai << hb) | hbv];
          o.y = cur[((ai | (1 << (st.ab - 1))) << hb) | hbv];
        }
        *reinterpret_cast<V2*>(nxt + 2 * e2) = o;
      }
      __syncwarp();
      T* tmp = cur; cur = nxt; nxt = tmp;
      st = ns;
    }
    // The column's nodes, top to bottom: chain position s is row bit h-1-s.
    // Each lane takes quads of entries that differ only in the node's row bit
    // (l -> r) and in v (u -> d): out[r][d] = sum_{l,u} in[l][u] w[l][r][u][d],
    // read and written as two pairs of adjacent entries.
    const int lnq = st.bits() - 2;                    // quads per coset, log2
    const int nq = n << lnq;
    // The base of a quad has the row bit P and bit 0 (v) clear, so the other
    // entries of the quad are at base + bitP, base + 1, base + bitP + 1.
    // k = 5, 6 (few warps per SM): each lane loads U quads before it stores
    // any; a lane past the end repeats the last quad (same values, same
    // addresses).  Quad g sits at base 4g - 2 (g & low); for k <= 4 the row
    // bit P is at most h + b <= 4 + 2 (b holds at most nc / 2 legs), so
    // 2^(P-1) divides 32, g & low stays lane & low and a lane's base grows by
    // exactly 128 per step.
    constexpr int U = K > 4 ? 4 : 1;
    for (int s = 0; s < h; ++s) {
      const int P = (h - 1 - s) + st.bb + 1;          // bit of the node's row in the index
      const int bitP = 1 << P;
      const int lowmask = (1 << (P - 1)) - 1;
      int ni, nj;
      f.node(t, s, &ni, &nj);
      const bool interior = ni > 0 && nj > 0 && ni < c.g.W - 1 && nj < c.g.W - 1;
      if (interior && s + 1 < h) {
        int mi, mj;
        f.node(t, s + 1, &mi, &mj);
        if (mi > 0 && mj > 0 && mi < c.g.W - 1 && mj < c.g.W - 1) {
          // Two interior chain neighbours, one check and one qubit, in one
          // pass: the check's copy tensor ties the vertical leg between them
          // to the check's own row bit c.
          const bool check_first = (ni + nj) & 1;
          T gt[4];
          qubit_table(c, check_first ? mi : ni, check_first ? mj : nj, rowwise, gt);
          if (check_first) {
            // out[c, r, d] = sum_l in[c, l, v=c] g[l^r][c^d]; rows bits P (c) and P-1 (qubit).
            const int Q = P - 1, bitQ = 1 << Q, lowq = (1 << (Q - 1)) - 1;
            int bq = 4 * lane - 2 * (lane & lowq);   // k <= 4: base of quad g0, +128 per step
            // k <= 4: bit P <= 6 of the base does not change in steps of 128,
            // so the check bit and its table entries are fixed per lane.
            const int cbl = (bq >> P) & 1;
            const T l00 = cbl ? gt[1] : gt[0], l01 = cbl ? gt[0] : gt[1];
            const T l10 = cbl ? gt[3] : gt[2], l11 = cbl ? gt[2] : gt[3];
            for (int g0 = lane; g0 < nq; g0 += 32 * U, bq += 128) {
              int bs[U], cbs[U];
              T x0s[U], x1s[U];
#pragma unroll
              for (int u = 0; u < U; ++u) {
                const int g = U == 1 ? g0 : min(g0 + 32 * u, nq - 1);
                bs[u] = K <= 4 ? bq : ((g >> (Q - 1)) << (Q + 1)) | ((g & lowq) << 1);
                cbs[u] = K <= 4 ? cbl : (bs[u] >> P) & 1;
                x0s[u] = cur[bs[u] + cbs[u]];
                x1s[u] = cur[bs[u] + bitQ + cbs[u]];
              }
#pragma unroll
              for (int u = 0; u < U; ++u) {
                const int base = bs[u], cb = cbs[u];
                const T x0 = x0s[u], x1 = x1s[u];
                // g[a][c ^ d] by selects (a dynamic index would put gt in local memory)
                const T g00 = K <= 4 ? l00 : (cb ? gt[1] : gt[0]), g01 = K <= 4 ? l01 : (cb ? gt[0] : gt[1]);
                const T g10 = K <= 4 ? l10 : (cb ? gt[3] : gt[2]), g11 = K <= 4 ? l11 : (cb ? gt[2] : gt[3]);
                V2 o0, o1;
                o0.x = x0 * g00 + x1 * g10;   // r = 0, d = 0
                o0.y = x0 * g01 + x1 * g11;   // r = 0, d = 1
                o1.x = x0 * g10 + x1 * g00;   // r = 1, d = 0
                o1.y = x0 * g11 + x1 * g01;   // r = 1, d = 1
                *reinterpret_cast<V2*>(nxt + base) = o0;
                *reinterpret_cast<V2*>(nxt + (base + bitQ)) = o1;
              }
            }
          } else {
            // out[r, c, v] = [v = c] sum_{l,u} in[l, c, u] g[l^r][u^c]; qubit bit P, check bit P-1.
            const int cpos = P - 1;
            // k <= 4: bit P - 1 <= 5 of the base is fixed per lane (see above).
            const int cbl = ((4 * lane - 2 * (lane & lowmask)) >> cpos) & 1;
            const T l00 = cbl ? gt[1] : gt[0], l01 = cbl ? gt[0] : gt[1];
            const T l10 = cbl ? gt[3] : gt[2], l11 = cbl ? gt[2] : gt[3];
            for (int g0 = lane, bq = 4 * lane - 2 * (lane & lowmask); g0 < nq; g0 += 32 * U, bq += 128) {
              int bs[U];
              V2 i0s[U], i1s[U];
#pragma unroll
              for (int u = 0; u < U; ++u) {
                const int g = U == 1 ? g0 : min(g0 + 32 * u, nq - 1);
                bs[u] = K <= 4 ? bq : ((g >> (P - 1)) << (P + 1)) | ((g & lowmask) << 1);
                i0s[u] = *reinterpret_cast<const V2*>(cur + bs[u]);          // in[0][u=0,1]
                i1s[u] = *reinterpret_cast<const V2*>(cur + (bs[u] + bitP)); // in[1][u=0,1]
              }
#pragma unroll
              for (int u = 0; u < U; ++u) {
                const int base = bs[u];
                const int cb = K <= 4 ? cbl : (base >> cpos) & 1;
                const V2 i0 = i0s[u], i1 = i1s[u];
                // g[l ^ r][u ^ c]
                const T g00 = K <= 4 ? l00 : (cb ? gt[1] : gt[0]), g01 = K <= 4 ? l01 : (cb ? gt[0] : gt[1]);
                const T g10 = K <= 4 ? l10 : (cb ? gt[3] : gt[2]), g11 = K <= 4 ? l11 : (cb ? gt[2] : gt[3]);
                const T r0 = i0.x * g00 + i0.y * g01 + i1.x * g10 + i1.y * g11;
                const T r1 = i0.x * g10 + i0.y * g11 + i1.x * g00 + i1.y * g01;
                V2 o0, o1;
                o0.x = cb ? T(0) : r0; o0.y = cb ? r0 : T(0);
                o1.x = cb ? T(0) : r1; o1.y = cb ? r1 : T(0);
                *reinterpret_cast<V2*>(nxt + base) = o0;
                *reinterpret_cast<V2*>(nxt + (base + bitP)) = o1;
              }
            }
          }
          __syncwarp();
          T* tmp = cur; cur = nxt; nxt = tmp;
          ++s;
          continue;
        }
      }
      if (interior && !((ni + nj) & 1)) {
        // Interior qubit: out[r][d] = sum_{l,u} in[l][u] g[l^r][u^d], an XOR
        // convolution with the 2 x 2 table g[alpha][beta].
        T gt[4];
        qubit_table(c, ni, nj, rowwise, gt);
        for (int g0 = lane, bq = 4 * lane - 2 * (lane & lowmask); g0 < nq; g0 += 32 * U, bq += 128) {
          int bs[U];
          V2 i0s[U], i1s[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int g = U == 1 ? g0 : min(g0 + 32 * u, nq - 1);
            bs[u] = K <= 4 ? bq : ((g >> (P - 1)) << (P + 1)) | ((g & lowmask) << 1);
            i0s[u] = *reinterpret_cast<const V2*>(cur + bs[u]);          // in[0][0], in[0][1]
            i1s[u] = *reinterpret_cast<const V2*>(cur + (bs[u] + bitP)); // in[1][0], in[1][1]
          }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const V2 i0 = i0s[u], i1 = i1s[u];
            V2 o0, o1;
            o0.x = i0.x * gt[0] + i0.y * gt[1] + i1.x * gt[2] + i1.y * gt[3];
            o0.y = i0.x * gt[1] + i0.y * gt[0] + i1.x * gt[3] + i1.y * gt[2];
            o1.x = i0.x * gt[2] + i0.y * gt[3] + i1.x * gt[0] + i1.y * gt[1];
            o1.y = i0.x * gt[3] + i0.y * gt[2] + i1.x * gt[1] + i1.y * gt[0];
            *reinterpret_cast<V2*>(nxt + bs[u]) = o0;
            *reinterpret_cast<V2*>(nxt + (bs[u] + bitP)) = o1;
          }
        }
        __syncwarp();
        T* tmp = cur; cur = nxt; nxt = tmp;
        continue;
      }
      if (interior) {
        // Interior check: a copy tensor over four legs, out[r][d] = [r = d] in[r][r].
        for (int g0 = lane, bq = 4 * lane - 2 * (lane & lowmask); g0 < nq; g0 += 32 * U, bq += 128) {
          int bs[U];
          T i0x[U], i1y[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int g = U == 1 ? g0 : min(g0 + 32 * u, nq - 1);
            bs[u] = K <= 4 ? bq : ((g >> (P - 1)) << (P + 1)) | ((g & lowmask) << 1);
            i0x[u] = reinterpret_cast<const V2*>(cur + bs[u])->x;
            i1y[u] = reinterpret_cast<const V2*>(cur + (bs[u] + bitP))->y;
          }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            V2 o0, o1;
            o0.x = i0x[u]; o0.y = T(0);
            o1.x = T(0); o1.y = i1y[u];
            *reinterpret_cast<V2*>(nxt + bs[u]) = o0;
            *reinterpret_cast<V2*>(nxt + (bs[u] + bitP)) = o1;
          }
        }
        __syncwarp();
        T* tmp = cur; cur = nxt; nxt = tmp;
        continue;
      }
      // Border node: the general 16-entry tensor (missing legs carry 0).  On
      // row 0 and column 0 the frame, hence the tensor, depends on the coset.
      const bool per_coset = n > 1 && (ni == 0 || nj == 0);
      if (!per_coset) {
        if (lane < 16)
          ws.wn[lane] = node_value<T>(c.frame, c.g.W, c.pI, c.pE, ni, nj, f.dir, (lane >> 3) & 1,
                                      (lane >> 2) & 1, (lane >> 1) & 1, lane & 1);
      } else {
        for (int q = lane; q < 16 * n; q += 32)
          ws.wn[q] = node_value<T>(frames + slot_coset(cos_of, q >> 4) * WW, c.g.W, c.pI, c.pE, ni, nj, f.dir,
                                   (q >> 3) & 1, (q >> 2) & 1, (q >> 1) & 1, q & 1);
      }
      __syncwarp();
      T w[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) w[q] = ws.wn[q];
      for (int g = lane; g < nq; g += 32) {
        if (per_coset) {
          const T* wq = ws.wn + ((g >> lnq) << 4);
#pragma unroll
          for (int q = 0; q < 16; ++q) w[q] = wq[q];
        }
        const int base = ((g >> (P - 1)) << (P + 1)) | ((g & lowmask) << 1);
        const V2 i0 = *reinterpret_cast<const V2*>(cur + base);          // (l=0,u=0), (l=0,u=1)
        const V2 i1 = *reinterpret_cast<const V2*>(cur + (base + bitP)); // (l=1,u=0), (l=1,u=1)
        V2 o0, o1;
        // w index: ((l*2 + r)*2 + u)*2 + d
        o0.x = i0.x * w[0] + i0.y * w[2] + i1.x * w[8] + i1.y * w[10];     // r=0, d=0
        o0.y = i0.x * w[1] + i0.y * w[3] + i1.x * w[9] + i1.y * w[11];     // r=0, d=1
        o1.x = i0.x * w[4] + i0.y * w[6] + i1.x * w[12] + i1.y * w[14];    // r=1, d=0
        o1.y = i0.x * w[5] + i0.y * w[7] + i1.x * w[13] + i1.y * w[15];    // r=1, d=1
        *reinterpret_cast<V2*>(nxt + base) = o0;
        *reinterpret_cast<V2*>(nxt + (base + bitP)) = o1;
      }
      __syncwarp();
      T* tmp = cur; cur = nxt; nxt = tmp;
    }
    // Side message B: closes the column's vertical leg.
    {
      FState ns = st;
      ns.hv = 0;
      if (f.b_idx < 0) ns.bb = 0;
      else if (t < sd) ns.bb = st.bb + 1;
      else if (t == sd) ns.bb = nf;
      else ns.bb = st.bb - 1;
      const int nt = n << ns.bits();
      const int hah = st.ab + h;                       // bits of (a, rows)
      if (K > 4 && t == sd && f.b_idx >= 0 && hah >= 5 && nf == 2 && (sd == 2 || sd == 3)) {
        for (int s = 0; s < n; ++s) {
          if (sd == 3) data_column_b<T, 3, 2>(ws.mb + (s << nc), cur, nxt, s << hah, hah, lane);
          else data_column_b<T, 2, 2>(ws.mb + (s << nc), cur, nxt, s << hah, hah, lane);
        }
        __syncwarp();
        T* tmp = cur; cur = nxt; nxt = tmp;
      } else if (t == sd && f.b_idx >= 0 && hah >= 5 && nf <= 1) {
        // The data column, one coset at a time with its side message in
        // registers: each lane reads the 2^bb pairs in[a, rows, b, v] of its
        // (a, rows) once and writes all outputs b2 of that group.
        const int nbb = 1 << st.bb;                    // st.bb = sd <= 2
        for (int s = 0; s < n; ++s) {
          T mr[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) mr[i] = i < (1 << nc) ? ws.mb[(s << nc) + i] : T(0);
          for (int al = lane; al < (1 << hah); al += 32) {
            const int ah = (s << hah) + al;
            V2 x[4];
#pragma unroll
            for (int b = 0; b < 4; ++b) {
              if (b < nbb) {
                x[b] = *reinterpret_cast<const V2*>(cur + (((ah << st.bb) + b) << 1));
              } else {
                x[b].x = T(0); x[b].y = T(0);
              }
            }
            if (nf == 1) {
              V2 o;
              T val = T(0);
#pragma unroll
              for (int b = 0; b < 4; ++b) val += mr[(b << 2)] * x[b].x + mr[(((b << 1) | 1) << 1)] * x[b].y;
              o.x = val;
              val = T(0);
#pragma unroll
              for (int b = 0; b < 4; ++b) val += mr[(b << 2) | 1] * x[b].x + mr[(((b << 1) | 1) << 1) | 1] * x[b].y;
              o.y = val;
              *reinterpret_cast<V2*>(nxt + (ah << 1)) = o;
            } else {
              T val = T(0);
#pragma unroll
              for (int b = 0; b < 4; ++b) val += mr[b << 1] * x[b].x + mr[(b << 1) | 1] * x[b].y;
              nxt[ah] = val;
            }
          }
        }
        __syncwarp();
        T* tmp = cur; cur = nxt; nxt = tmp;
      } else if (K > 4 && f.b_idx >= 0 && t > sd) {
        // Close v against b's top bit: out[(slot, a, rows), b] = in[.., (0, b), v = 0]
        // + in[.., (1, b), v = 1] (two outputs per lane and step, loads first).
        const int top = 1 << (st.bb - 1);
        for (int e0 = lane; e0 < nt; e0 += 64) {
          T vs[2];
          int es[2];
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int e = min(e0 + 32 * u, nt - 1);
            const int b2 = e & ((1 << ns.bb) - 1), ah = e >> ns.bb;
            vs[u] = cur[((ah << st.bb) | b2) << 1] + cur[(((ah << st.bb) | top | b2) << 1) | 1];
            es[u] = e;
          }
#pragma unroll
          for (int u = 0; u < 2; ++u) nxt[es[u]] = vs[u];
        }
        __syncwarp();
        T* tmp = cur; cur = nxt; nxt = tmp;
      } else if (!(f.b_idx >= 0 && t < sd)) {   // recording v as b's new low bit changes no index
        for (int e = lane; e < nt; e += 32) {
          T val;
          if (f.b_idx < 0) {
            val = cur[e << 1];                          // v = 0, b has no bits
          } else if (t == sd) {
            const int b2 = e & ((1 << ns.bb) - 1), ah = e >> ns.bb;   // (slot, a, rows)
            const T* mb = ws.mb + ((ah >> (st.ab + h)) << nc);
            val = T(0);
            for (int b = 0; b < (1 << st.bb); ++b) {
              const int bi = ((ah << st.bb) | b) << 1;
              val += mb[((b << 1) << nf) | b2] * cur[bi] + mb[(((b << 1) | 1) << nf) | b2] * cur[bi | 1];
            }
          } else {
            const int b2 = e & ((1 << ns.bb) - 1), ah = e >> ns.bb;
            const int hi0 = ((ah << st.bb) | b2) << 1;                        // b top bit 0, v = 0
            const int hi1 = ((ah << st.bb) | (1 << (st.bb - 1)) | b2) << 1 | 1; // b top bit 1, v = 1
            val = cur[hi0] + cur[hi1];
          }
          nxt[e] = val;
        }
        __syncwarp();
        T* tmp = cur; cur = nxt; nxt = tmp;
      }
      st = ns;
    }
    if (ls) {   // keep each coset's block value in range; the logs go to the read-out
      const int S = st.size();
#pragma unroll
      for (int q = 0; q < kFusedMaxG; ++q) {
        if (q < n) {
          T* cq = cur + q * S;
          T acc = 0;
          for (int e = lane; e < S; e += 32) acc += cq[e] * cq[e];
          acc = warp_sum(acc);
          const T nrm = xsqrt(acc);
          if (nrm > T(0)) {
            const T inv = T(1) / nrm;
            for (int e = lane; e < S; e += 32) cq[e] *= inv;
            if (lane == 0) ls[q].mul(nrm);
          }
        }
      }
      __syncwarp();
    }
  }
  if (cur != ws.s0) {
    for (int e = lane; e < (n << h); e += 32) ws.s0[e] = cur[e];
    __syncwarp();
  }
}

// The outgoing vector of a full 6 x 6 block (one coset) into ws.s0, as
// fused_sweep leaves it.
template <typename T, int K>
__device__ __forceinline__ void block6_update(const FusedWS<T>& ws, const Ctx<T, K>& c, const T* msgs, const Frame& f,
                                              int lane) {
  constexpr int VEC = FusedDim<K>::vec;
  Block6<T> k;
  int i0, j0;
  f.node(0, 0, &i0, &j0);
  k.chk0 = (i0 + j0) & 1;
  // Side messages in consumption order; the qubits' ids, one per lane.
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int i = lane + 32 * u, j = f.rev ? bitrev(i, 6) : i;
    if (f.a_idx >= 0) ws.mt[i] = msgs[f.a_idx * VEC + j];
    ws.mb[i] = msgs[f.b_idx * VEC + j];
  }
  k.ids = 0;
  if (lane < 18) {
    const int t = lane / 3, u = lane - 3 * t;
    int i, j;
    f.node(t, 2 * u + ((((t & 1) != 0) != k.chk0) ? 1 : 0), &i, &j);
    const int fr = c.frame[i * c.g.W + j];
    const bool alpha_is_z = ((i & 1) == 0) == (f.dir == kDirR || f.dir == kDirL);
    k.ids = alpha_is_z ? fr : (((fr & 1) << 1) | (fr >> 1));
  }
  k.A = ws.s0; k.B = ws.s1; k.mt = ws.mt; k.mb = ws.mb;
  k.in = f.in_idx >= 0 ? msgs + f.in_idx * VEC : nullptr;
  k.pI = c.pI; k.pE = c.pE;
  k.a = f.a_idx >= 0;
  k.lane = lane;
  __syncwarp();
  if (k.chk0) k.run_c();
  else k.run_q();
}

// Block sides up to 4: one out-of-line copy (the kernels that also hold the
// register forms keep their hot loop small in the instruction cache);
// block sides 5 and 6 inline it (their loop is this sweep).
template <typename T, int K>
__device__ __noinline__ void fused_sweep_call(const FusedWS<T>& ws, const Ctx<T, K>& c, const T* msgs, int stride,
                                              unsigned cos_of, int n, const uint8_t* frames, const Frame& f,
                                              LogAcc<T>* ls, int lane) {
  fused_sweep_body<T, K>(ws, c, msgs, stride, cos_of, n, frames, f, ls, lane);
}

template <typename T, int K>
__device__ __forceinline__ void fused_sweep(const FusedWS<T>& ws, const Ctx<T, K>& c, const T* msgs, int stride,
                                            unsigned cos_of, int n, const uint8_t* frames, const Frame& f,
                                            LogAcc<T>* ls, int lane) {
  if constexpr (K <= 4) fused_sweep_call<T, K>(ws, c, msgs, stride, cos_of, n, frames, f, ls, lane);
  else fused_sweep_body<T, K>(ws, c, msgs, stride, cos_of, n, frames, f, ls, lane);
}

// <x, y> over n <= 64 entries for the read-out, in the working precision.
template <typename T>
__device__ __forceinline__ T read_dot(const T* x, const T* y, int n, int lane) {
  T acc = lane < n ? x[lane] * y[lane] : T(0);
  if (n > 32 && lane + 32 < n) acc += x[lane + 32] * y[lane + 32];
  return warp_sum(acc);
}

// The per-message term 2 - 2 <x, y>^2 of Delta (Remark 4) for unit vectors
// x (new) and y (old), each held one entry per lane in a group of lanes.
// FP64 evaluates it as written.  FP32 evaluates the same quantity as
// s (2 - s / 2) with s = ||x - y||^2 (an identity for unit vectors): no
// cancellation when a message barely moved, and no FP64 instruction per
// update (FP64 issues at 1/64 of the FP32 rate here).
template <typename T> struct DeltaTerm;
template <> struct DeltaTerm<double> {
  static __device__ __forceinline__ double eval(double x, double y, int width) {
    const double o = group_sum(x * y, width);
    return fma(-2.0 * o, o, 2.0);
  }
  // A 64-entry vector held as entries lane and lane + 32.
  static __device__ __forceinline__ double eval2(double x0, double y0, double x1, double y1) {
    const double o = warp_sum(x0 * y0 + x1 * y1);
    return fma(-2.0 * o, o, 2.0);
  }
};
template <> struct DeltaTerm<float> {
  static __device__ __forceinline__ float eval(float x, float y, int width) {
    const float t = x - y;
    const float s = group_sum(t * t, width);
    return s * fmaf(-0.5f, s, 2.f);
  }
  static __device__ __forceinline__ float eval2(float x0, float y0, float x1, float y1) {
    const float t0 = x0 - y0, t1 = x1 - y1;
    const float s = warp_sum(t0 * t0 + t1 * t1);
    return s * fmaf(-0.5f, s, 2.f);
  }
};

// Unit L2 norm (Remark 3) of the vector held by a group of lanes.
template <typename T>
__device__ __forceinline__ T group_normalize(T v, int width) {
  return v * inv_norm(group_sum(v * v, width));
}

// After a sweep: normalise the new messages in ws.s0 (Remark 3), damp them
// with the stored ones (Remark 7), normalise again, record each coset's
// Delta term in ovl[coset * M + idx] and store the result.  Entry e of the
// n x 2^h outgoing vectors sits in lane e % 32 (e < 64: G <= 4, h <= 4 or
// G = 1, h <= 6); a vector of 64 entries spans both halves.
template <typename T, int K>
__device__ __forceinline__ void fused_update(const FusedWS<T>& ws, T* msgs, int stride, unsigned cos_of, int n,
                                             int idx, int h, T eta, T one_m_eta, T* ovl, int M, int lane) {
  const int width = 1 << h, tot = n << h;
  if (K > 5 && width > 32) {
    // One vector of 64 entries (k = 6, one coset): entries lane and lane + 32
    // are reduced together.
    const int q = slot_coset(cos_of, 0);
    T* old0 = msgs + q * stride + idx * FusedDim<K>::vec + lane;
    T* old1 = old0 + 32;
    T x0 = ws.s0[lane], x1 = ws.s0[lane + 32];
    const T y0 = *old0, y1 = *old1;
    T nrm = xsqrt(warp_sum(x0 * x0 + x1 * x1));
    T inv = nrm > T(0) ? T(1) / nrm : T(0);
    x0 = fma(one_m_eta, x0 * inv, eta * y0);
    x1 = fma(one_m_eta, x1 * inv, eta * y1);
    nrm = xsqrt(warp_sum(x0 * x0 + x1 * x1));
    inv = nrm > T(0) ? T(1) / nrm : T(0);
    x0 *= inv;
    x1 *= inv;
    const T term = DeltaTerm<T>::eval2(x0, y0, x1, y1);
    *old0 = x0;
    *old1 = x1;
    if (lane == 0) ovl[q * M + idx] = term;
    __syncwarp();
    return;
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    if (r == 1 && tot <= 32) break;
    const int e = lane + 32 * r;
    const bool on = e < tot;
    const int q = on ? slot_coset(cos_of, e >> h) : 0;
    T* old = msgs + q * stride + idx * FusedDim<K>::vec + (e & (width - 1));
    T x = on ? ws.s0[e] : T(0);
    const T y = on ? *old : T(0);
    x = group_normalize(x, width);
    x = fma(one_m_eta, x, eta * y);
    x = group_normalize(x, width);
    const T term = DeltaTerm<T>::eval(x, y, width);
    if (on) {
      *old = x;
      if ((e & (width - 1)) == 0) ovl[q * M + idx] = term;
    }
  }
  __syncwarp();
}

// 2^-e exactly (0 <= e < 126), from the exponent bits.
template <typename T> __device__ __forceinline__ T pow2_neg(int e);
template <> __device__ __forceinline__ float pow2_neg<float>(int e) { return __int_as_float((127 - e) << 23); }
template <> __device__ __forceinline__ double pow2_neg<double>(int e) {
  return __longlong_as_double((long long)(1023 - e) << 52);
}

// Resident CTAs per SM the register budget is sized for: 16 warps per SM in
// FP32 and 8 in FP64; with k = 6 states (16 KB a buffer in FP32) the shared
// memory decides.  LB > 0: the kernel with small per-warp buffers
// (fused_slot), sized for LB resident CTAs per SM.
template <typename T, int NW, int G, int K, int LB = 0> struct FusedMinBlocks {
  static constexpr int warps = K > 4 ? NW : (sizeof(T) == 4 ? 16 : 8);
  static constexpr int value = LB > 0 ? LB % kEvenLB : (warps / NW > 1 ? warps / NW : 1);
};

// Position lists of a CTA: each colour's messages grouped by class, the
// register forms first (class 2 shape + srev, so that a pass rarely mixes
// both orders of the side messages), the node-by-node path last; within a
// class in any order, but in that of the blocks where every message is updated
// node by node (k <= 3: neighbouring blocks share what L1 holds, and the short
// updates of the edge blocks come last).
constexpr int kClassNone = 2 * kShapes;
constexpr int kClasses = kClassNone + 2;    // per colour: shapes x 2 orders, then none (R and D, L and U)
template <int V> struct IntC { static constexpr int value = V; };

// Messages of block (I, J)'s colour before its own in (I, J, dir) order.  A row's
// blocks of one parity of J have two horizontal sides each, less one at either
// end of the row.
__device__ __forceinline__ int colour_rank(int nb, int I, int J) {
  int n = 0;
  for (int i = 0; i <= I; ++i) {
    const int q = (I + J + i) & 1, end = i < I ? nb : J;               // blocks j < end, j = q mod 2
    const int cnt = (end + 1 - q) >> 1, vertical = (i + 1 < nb) + (i > 0);
    n += cnt * (2 + vertical) - (q == 0 && end > 0) - (end == nb && ((nb - 1) & 1) == q);
  }
  return n;
}

// Cosets c0 .. c0 + G - 1 of one syndrome decoded by the whole CTA: syn_src
// holds the syndrome's m bytes and outputs go to row syn * 4 + coset.
// GM: the messages live in gmsgs, this CTA's slot in global memory (the slot
// is L2-resident and touched only a few times per block sweep); always for
// k = 5, 6.  Otherwise they live in shared memory and gmsgs is null.
template <typename T, int NW, int G, int K, bool GM, int LB = 0>
__device__ __forceinline__ void fused_item(const KArgs<T>& a, const Geo g, const int M, const uint8_t* syn_src,
                                           const long long syn, const int c0, unsigned char* smem, T* gmsgs) {
  const int W = g.W, d = g.d, nb = g.nb, WW = W * W;
  static_assert(K <= 4 || G == 1, "k = 6 states hold one coset per CTA");
  constexpr int VEC = FusedDim<K>::vec;
  constexpr bool kLean = LB > 0 && K == 4;   // every block update in register form
  constexpr bool kEven = kLean && LB >= kEvenLB;   // ... blocks three nodes wide included
  constexpr int kMode = LB == 0 ? 0 : (kEven ? 2 : 1);
  static_assert(LB == 0 || K != 4 || !GM, "register-form-only kernels keep their messages in shared memory");
  const FusedLayout Lo = fused_layout<T, K>(g, M, NW, G, GM, kMode);
  unsigned long long* px = reinterpret_cast<unsigned long long*>(smem + Lo.parity);
  unsigned long long* pz = px + d;
  uint8_t* frames = smem + Lo.frame;
  int16_t* msg_of = reinterpret_cast<int16_t*>(smem + Lo.msg_of);
  int16_t* meta = reinterpret_cast<int16_t*>(smem + Lo.meta);
  int16_t* work = reinterpret_cast<int16_t*>(smem + Lo.work);
  T* ovl = reinterpret_cast<T*>(smem + Lo.ovl);                // Delta term of each (coset, message)
  int16_t* rank = reinterpret_cast<int16_t*>(smem + Lo.ovl);   // before that, each message's rank in its class
  RegTask* tasks = reinterpret_cast<RegTask*>(smem + Lo.tasks);
  uint16_t* qid = reinterpret_cast<uint16_t*>(smem + Lo.qid);
  double* rlog = reinterpret_cast<double*>(smem + Lo.rlog);
  // misc: [0], [1] work counters of the two colours' node-by-node messages,
  // [2] the read-out's, [3] cosets converged (bit q), [4 + q] flags, [8 + q]
  // iterations done, [12 .. 43] messages per (colour, class), [44 .. 75]
  // their list positions; dsh[q]: the sum of coset q's Delta terms at its
  // last iteration.
  int* misc = reinterpret_cast<int*>(smem + Lo.misc);
  double* dsh = reinterpret_cast<double*>(smem + Lo.misc + 304);
  int* cls_n = misc + 12;
  int* cls_at = misc + 12 + 2 * kClasses;
  T* msgs = GM ? gmsgs : reinterpret_cast<T*>(smem + Lo.msgs);
  const int stride = fused_coset_stride<K>(M, GM);           // from one coset's messages to the next

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if constexpr (kLean && !kEven) {
    // The host launches register-form-only kernels only where every block has
    // a register form; in a mixed batch the caller vouches for it.
    if (!register_form_only(g)) {
      if (tid < G) {
        const long long row = syn * 4 + c0 + tid;
        a.logp[row] = __longlong_as_double(0x7ff8000000000000ll);
        a.delta[row] = __longlong_as_double(0x7ff8000000000000ll);
        a.iters[row] = 0;
        a.flags[row] = kFlagCapacity | kFlagNonfinite;
      }
      return;
    }
  }
  const bool reg = kLean || (K == 4 && g.k == 4);            // blocks with a register form take it
  T* stage = reinterpret_cast<T*>(smem + Lo.ws + warp * Lo.ws_stride);
  RegMsgs<T, GM> ms;
  ms.base = msgs; ms.stride = stride; ms.M = M;
  ms.border = reinterpret_cast<const T*>(smem + Lo.border);

  // The pure error f_s (Algorithm 1) as prefix parities, a warp per row of
  // site checks (x) or column of plaquettes (z).
  for (int r = warp; r < 2 * d; r += NW) {
    const bool row = r < d;
    const uint8_t* src = row ? syn_src + r * (d - 1) : syn_src + d * (d - 1) + (r - d);
    const int step = row ? 1 : d;
    const unsigned b0 = __ballot_sync(kFull, lane < d - 1 && src[lane * step]);
    unsigned b1 = 0;
    if (d > 33) b1 = __ballot_sync(kFull, lane + 32 < d - 1 && src[(lane + 32) * step]);
    if (lane == 0) px[r] = prefix_parity(b0 | ((unsigned long long)b1 << 32));   // pz follows px
  }
  if (tid < 76) misc[tid] = 0;
  if (tid < 4) dsh[tid] = 0.0;
  __syncthreads();
  // Message table in (I, J, dir) order, and each message's rank in its class.
  const int NK = nb * nb * 4;
  auto class_of = [&](int I, int J, int dir) {
    // One direction's code at a time at k = 6, whose blocks have two forms.
    // (Register-form-only kernels have no such messages; without the term
    // their compiled prologue took 0.6 % of the d = 11 decode longer.)
    int c = kClassNone + (K > 4 || kLean ? dir & 1 : 0);
    if (reg) {
      const RegFrame f = reg_frame(g, I, J, dir);
      const int sh = f.shape();
      if (sh != kShapeNone) c = 2 * (sh - 1) + (f.srev() ? 1 : 0);
    }
    return ((I + J) & 1) * kClasses + c;
  };
  for (int key = tid; key < NK; key += NW * 32) {
    const int I = key / 4 / nb, J = (key / 4) % nb, dir = key & 3;
    const bool has = g.has(I, J, dir);
    if (has) {
      const int idx = message_index(nb, I, J, dir);
      if (dev_check(idx >= 0 && idx < M, &misc[4])) {
        meta[idx] = (int16_t)key;
        int r = atomicAdd(&cls_n[class_of(I, J, dir)], 1);
        if constexpr (K == 4 && !kLean) {
          if (!reg) r = colour_rank(nb, I, J) + idx - message_index(nb, I, J, kDirR);
        }
        rank[idx] = (int16_t)r;
      }
      if constexpr (!kLean || kEven) msg_of[key] = (int16_t)idx;
    } else {
      if constexpr (!kLean || kEven) msg_of[key] = -1;
    }
  }
  // Every coset's frame, for the node-by-node path.
  if constexpr (!kLean || kEven) {
    for (int e = tid; e < G * WW; e += NW * 32) {
      const int q = e / WW, ij = e - q * WW;
      const int i = ij / W, j = ij - i * W;
      const int coset = c0 + q;
      const bool bx = coset == 1 || coset == 2, bz = coset == 2 || coset == 3;
      const bool hq = ((i | j) & 1) == 0;
      frames[e] = (uint8_t)(frame_bits(px, pz, i, j) ^ ((bx && hq && i == 0) ? 1 : 0) ^ ((bz && hq && j == 0) ? 2 : 0));
    }
  }
  // The border vectors (the messages of a workspace slot have theirs apart).
  if constexpr (K == 4) {
    for (int e = tid; e < (GM ? 1 : G) * kBorderVecs * kRegVec; e += NW * 32) {
      const int q = e / (kBorderVecs * kRegVec), r = e - q * (kBorderVecs * kRegVec);
      T* v = GM ? reinterpret_cast<T*>(smem + Lo.border) : msgs + q * stride + M * kRegVec;
      v[r] = border_entry(r / kRegVec, r % kRegVec) ? T(1) : T(0);
    }
  }
  __syncthreads();
  if (tid < 2 * kClasses) {
    int at = 0;
    for (int c = 0; c < tid; ++c) at += cls_n[c];
    cls_at[tid] = at;
  }
  __syncthreads();
  // The lists: a register-form message's task and qubit ids at its position,
  // a node-by-node message's index.  The order within a colour does not
  // matter for the results (Remark 8: its messages read only the other
  // colour's).
  for (int idx = tid; idx < M; idx += NW * 32) {
    const int key = meta[idx];
    const int I = key / 4 / nb, J = (key / 4) % nb, dir = key & 3;
    const int cls = class_of(I, J, dir);
    const int pos = cls_at[cls] + rank[idx];
    if (!dev_check(pos >= 0 && pos < M, &misc[4])) continue;
    work[pos] = (int16_t)idx;
    if (cls % kClasses < kClassNone) {
      const RegFrame f = reg_frame(g, I, J, dir);
      RegTask q = reg_task(g, M, I, J, f);
      if (!dev_check((q.in & kTaskIdx) < M + kBorderVecs && (q.up & kTaskIdx) < M + kBorderVecs &&
                         (q.lo & kTaskIdx) < M + kBorderVecs && (q.out & kTaskIdx) == idx,
                     &misc[4]))
        q.in = q.up = q.lo = q.out = 0;
      tasks[pos] = q;
      const RegIds v = reg_ids(f, px, pz);
      for (int c = 0; c < G; ++c) qid[c * M + pos] = (uint16_t)coset_id(v, c0 + c);
    }
  }

  // Remark 2: uniform messages of unit norm, unless initial messages are
  // given (learned warm start): those are renormalised on entry.
  // 1 / sqrt(2^w): a power of two, times the rounded 1 / sqrt 2 for odd w.
  auto uniform_entry = [&](int w) { return ((w & 1) ? T(0.70710678118654752440) : T(1)) * pow2_neg<T>(w >> 1); };
  auto width_of = [&](int idx) {
    const int key = meta[idx];
    return g.side_len(key / 4 / nb, (key / 4) % nb, key & 3);
  };
  if (K <= 4 && a.init_msgs) {
    // A message per half-warp, two per half in flight (the proposals come
    // from HBM); the norm sums over 16 lanes.
    const int sub = lane & 15, hi = lane >> 4;
    for (int b0 = 2 * warp; b0 < G * M; b0 += 4 * NW) {   // the same trip count in both halves (shuffles)
      const int q0 = b0 + hi;
      T v[2];
      int w[2];
      T* x[2];
      bool ok[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int qi = q0 + u * 2 * NW;
        ok[u] = qi < G * M;
        const int qq = ok[u] ? qi : 0;
        const int q = qq / M, idx = qq - q * M;
        w[u] = width_of(idx);
        x[u] = msgs + q * stride + idx * VEC;
        v[u] = (ok[u] && sub < (1 << w[u])) ? (T)a.init_msgs[((syn * 4 + c0 + q) * M + idx) * VEC + sub] : T(0);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        T s = v[u] * v[u];
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) s = radd(s, shx(s, o));
        const T nrm = xsqrt(s);
        const bool uniform = !(nrm > T(0));
        if (ok[u] && sub < VEC)
          x[u][sub] = uniform ? (sub < (1 << w[u]) ? uniform_entry(w[u]) : T(0)) : v[u] * (T(1) / nrm);
      }
    }
  } else {
    for (int e = tid; e < M * (VEC / 4); e += NW * 32) {
      const int idx = e / (VEC / 4), i0 = 4 * (e % (VEC / 4));
      const int w = width_of(idx);
      const T u = uniform_entry(w);
      T v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = i0 + i < (1 << w) ? u : T(0);
      for (int q = 0; q < G; ++q) vstore4(msgs + q * stride + idx * VEC + i0, v);
    }
  }
  __syncthreads();

  Ctx<T, K> c;                                       // for the node-by-node path
  c.g = g; c.D = 0; c.cutoff2 = T(0);
  c.pI = a.pI_w; c.pE = a.pE_w;
  c.frame = frames; c.msg_of = msg_of; c.msg_off = nullptr; c.dims = nullptr;
  c.arena = nullptr; c.e0 = nullptr; c.cta_flags = &misc[4];
  FusedWS<T> ws{};
  if constexpr (!kLean) ws = fused_ws_at<T, K>(smem + Lo.ws + warp * Lo.ws_stride, G, fused_slot<K>(kMode));

  const T pI = a.pI_w, pE = a.pE_w;
  const RegUpd<T> upd{a.eta_w, a.one_m_eta_w, ovl, M};
  unsigned act = (1u << G) - 1;                      // cosets still iterating
  for (int it = 1; it <= a.max_iter && M > 0 && act; ++it) {
    int n = 0;
    unsigned cos_of = 0;
#pragma unroll
    for (int q = 0; q < G; ++q)
      if ((act >> q) & 1u) { cos_of |= (unsigned)q << (2 * n); ++n; }
    for (int color = 0; color < 2; ++color) {       // Remark 8
      if constexpr (K == 4) {
        if (reg) {
          int first = 0;
          const int* cn = cls_n + color * kClasses;
          const int* ca = cls_at + color * kClasses;
          first += reg_updates<T, GM, kShapeQuad, NW>(stage, pI, pE, ms, tasks, qid, M, ca[0], cn[0] + cn[1], cos_of,
                                                      n, first, warp, lane, upd);
          first += reg_updates<T, GM, kShapeRow, NW>(stage, pI, pE, ms, tasks, qid, M, ca[4], cn[4] + cn[5], cos_of,
                                                     n, first, warp, lane, upd);
          first += reg_updates<T, GM, kShapeCol, NW>(stage, pI, pE, ms, tasks, qid, M, ca[2], cn[2] + cn[3], cos_of,
                                                     n, first, warp, lane, upd);
          first += reg_updates<T, GM, kShapeDot, NW>(stage, pI, pE, ms, tasks, qid, M, ca[6], cn[6] + cn[7], cos_of, n,
                                                     first, warp, lane, upd);
          if constexpr (!kLean || kEven) {
            first += reg_updates<T, GM, kShape34, NW>(stage, pI, pE, ms, tasks, qid, M, ca[10], cn[10] + cn[11], cos_of,
                                                      n, first, warp, lane, upd);
            first += reg_updates<T, GM, kShape43, NW>(stage, pI, pE, ms, tasks, qid, M, ca[8], cn[8] + cn[9], cos_of, n,
                                                      first, warp, lane, upd);
            reg_updates<T, GM, kShape33, NW>(stage, pI, pE, ms, tasks, qid, M, ca[12], cn[12] + cn[13], cos_of, n, first,
                                             warp, lane, upd);
          }
        }
      }
      // The node-by-node path: whole messages, every coset at once.
      if constexpr (!kLean) {
        const int cnt = cls_n[color * kClasses + kClassNone] + cls_n[color * kClasses + kClassNone + 1];
        const int at = cls_at[color * kClasses + kClassNone];
        c.frame = frames + (cos_of & 3u) * WW;
        if (tid == 0) misc[color ^ 1] = 0;           // the other colour's counter, idle until the barrier
        for (;;) {
          int item = 0;
          if (lane == 0) item = atomicAdd(&misc[color], 1);
          item = __shfl_sync(kFull, item, 0);
          if (item >= cnt) break;
          const int idx = work[at + item];
          if (!dev_check(idx >= 0 && idx < M, &misc[4])) continue;
          const int key = meta[idx];
          const Frame f = make_frame(c, key / 4 / nb, (key / 4) % nb, key & 3);
          if (K > 4 && f.h == 6 && f.ncols == 6) block6_update(ws, c, msgs, f, lane);
          else fused_sweep(ws, c, msgs, stride, cos_of, n, frames, f, (LogAcc<T>*)nullptr, lane);
          fused_update<T, K>(ws, msgs, stride, cos_of, n, idx, f.h, upd.eta, upd.one_m_eta, ovl, M, lane);
        }
      }
      __syncthreads();
    }
    // Delta = sqrt(sum) / M < delta0 (Remark 4), compared as sum <
    // (delta0 M)^2 by the coset's warp, which sets the coset's bit in
    // misc[3]; the square root is taken once, after the loop.  The sum and
    // the compare run in working precision (FP32 terms, each already rounded
    // to FP32; no FP64 instruction in the loop of an FP32 kernel).
    if (warp < G && ((act >> warp) & 1u)) {
      T acc = T(0);
      for (int i = lane; i < M; i += 32) acc += ovl[warp * M + i];
      acc = warp_sum(acc);
      if (lane == 0) {
        const T d0sq = (T)((a.delta0 * M) * (a.delta0 * M));   // the exit threshold in working precision
        const T sum = acc > T(0) ? acc : T(0);
        dsh[warp] = (double)sum;
        misc[8 + warp] = it;
        if (sum < d0sq) atomicOr(&misc[3], 1 << warp);
      }
    }
    __syncthreads();
    act &= ~(unsigned)misc[3];
  }

  if (a.final_msgs)
    for (int e = tid; e < G * M * VEC; e += NW * 32) {
      const int q = e / (M * VEC), r = e - q * (M * VEC);
      a.final_msgs[((syn * 4 + c0 + q) * M) * VEC + r] = (float)msgs[q * stride + r];
    }

  // Lemma 1 read-out: a record (a factor, or in FP64 its log) per block,
  // then per undirected edge in the order of its rightward / downward message.
  const int nblk = nb * nb, nedge = M / 2, per = nblk + nedge;
  auto record = [&](int q, int at, T v) {
    if constexpr (sizeof(T) == 4) {                  // as mantissa and exponent
      LogAcc<float> l;
      l.mul(fabsf(v));
      reinterpret_cast<float*>(rlog + q * per + at)[0] = l.m;
      reinterpret_cast<int*>(rlog + q * per + at)[1] = l.e;
    } else {
      rlog[q * per + at] = at < nblk ? log(fabs(v)) : -log(fabs(v));
    }
    if (!(v > T(0))) atomicOr(&misc[4 + q], at < nblk ? kFlagBlock : kFlagOverlap);
  };
  // A block contracted node by node: its norms taken out on the way and z.
  auto close_block = [&](LogAcc<T>& l, T z, int q, int at) {
    if (lane == 0) {
      l.mul(z < T(0) ? -z : z);
      if constexpr (sizeof(T) == 4) {
        reinterpret_cast<float*>(rlog + q * per + at)[0] = l.m;
        reinterpret_cast<int*>(rlog + q * per + at)[1] = l.e;
      } else {
        rlog[q * per + at] = l.value();
      }
      if (!(z > T(0))) atomicOr(&misc[4 + q], kFlagBlock);
    }
  };
  int first = 0;                                     // passes dealt to the warps so far
  if constexpr (K == 4) {
    // Z_v: the block's outgoing vector to the right, with every other
    // incoming message, closed against the message from the right.  Blocks
    // with a register form need no per-column rescaling (entries are sums of
    // products of node values and message entries, all at most 1).
    if (reg) {
      const int nf = W / 4, edge = W % 4 == 1 ? nf : 0;   // full blocks and, at odd d, one-wide ones per axis
      auto blocks = [&](auto shape_c, int cnt, auto where) {
        constexpr int SHAPE = decltype(shape_c)::value;
        const int passes = (cnt * G + 7) >> 3;
        int p = warp - first % NW;
        if (p < 0) p += NW;
        first += passes;
        for (; p < passes; p += NW) {
          const int j = p * 8 + (lane >> 2);
          RegJob<T, GM> jb;
          int item = j / G;
          jb.cq = j % G;
          jb.on = item < cnt;
          if (!jb.on) item = cnt - 1;
          int I, J;
          where(item, I, J);
          const RegFrame f = reg_frame(g, I, J, kDirR);
          jb.q = reg_task(g, M, I, J, f);
          RegIds v{0u, 0u, 0u};
          if (SHAPE == kShapeQuad) {                 // a column per lane of the job
            add_quad_column(v, f, lane & 3, f.chk0(), px, pz);
#pragma unroll
            for (int o = 1; o <= 2; o <<= 1) {
              v.id |= shx(v.id, o);
              v.fx |= shx(v.fx, o);
              v.fz |= shx(v.fz, o);
            }
          } else {
            v = reg_ids(f, px, pz);
          }
          jb.id = coset_id(v, c0 + jb.cq);
          reg_pass<T, GM, false, SHAPE>(stage, pI, pE, ms, jb, lane, upd);
          // On the grid border the vector is closed against the product
          // vector of the missing legs.
          const bool open = J + 1 < nb;
          int bi, bj;
          f.node(f.ncols - 1, f.h - 1, &bi, &bj);
          const T* R = ms.at(jb.cq, open ? message_index(nb, I, J + 1, kDirL) : M + (((bi + bj) & 1) ? 0 : 1));
          const RowAt at(false, (lane >> 1) & 1, lane & 1);
          T z[2][2];
#pragma unroll
          for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int y = 0; y < 2; ++y) {
              const int i = at(x, y);
              const T s = stage[(lane >> 2) * 16 + i], m = R[i];
              z[x][y] = i >= (1 << f.h) ? T(0) : (open ? s * m : (m != T(0) ? s : T(0)));
            }
          const T zz = job_sum(z);
          if (jb.on && (lane & 3) == 0) record(jb.cq, I * nb + J, zz);
          __syncwarp();
        }
      };
      blocks(IntC<kShapeQuad>{}, nf * nf, [&](int i, int& I, int& J) { I = i / nf; J = i - I * nf; });
      blocks(IntC<kShapeRow>{}, edge, [&](int i, int& I, int& J) { I = nf; J = i; });
      blocks(IntC<kShapeCol>{}, edge, [&](int i, int& I, int& J) { I = i; J = nf; });
      blocks(IntC<kShapeDot>{}, edge ? 1 : 0, [&](int i, int& I, int& J) { I = J = nf; });
    }
  }
  if constexpr (kEven) {
    // Node by node: the blocks three nodes wide, a coset at a time; no other
    // warp's buffers are in use any more but the passes' above.
    const int nf = W / 4, cnt = W % 4 == 3 ? 2 * nf + 1 : 0;
    __syncthreads();
    ws = fused_ws_at<T, K>(smem + Lo.ws + (warp < kReadWarps ? warp : 0) * fused_ws_bytes<T, K>(1), 1,
                           FusedDim<K>::slot);
    for (int j = warp; warp < kReadWarps && j < cnt * G; j += kReadWarps) {
      const int i = j / G, q = j % G;
      const int I = i < nf ? i : nf, J = i < nf ? nf : i - nf;     // (i, nf), (nf, 0 .. nf)
      c.frame = frames + q * WW;
      const Frame f = make_frame(c, I, J, kDirR);
      LogAcc<T> ls[kFusedMaxG];
      fused_sweep(ws, c, msgs, stride, (unsigned)q, 1, frames, f, ls, lane);
      const int right = J + 1 < nb ? msg_index(c, I, J + 1, kDirL) : -1;
      if (!dev_check(right >= -1 && right < M, &misc[4])) continue;
      close_block(ls[0], right >= 0 ? read_dot(ws.s0, msgs + q * stride + right * VEC, 1 << f.h, lane) : ws.s0[0], q,
                  I * nb + J);
      __syncwarp();
    }
  }
  if constexpr (!kLean) {
    const unsigned all = G == 1 ? 0u : (G == 2 ? 0x4u : 0xE4u);    // slot q holds coset q
    c.frame = frames;
    const int full = fused_ws_bytes<T, K>(G);                   // full-size state buffers
    const int nro = K > 4 && LB > 0 ? imin(NW, NW * Lo.ws_stride / full) : NW;
    if (K > 4 && LB > 0 && warp < nro)
      ws = fused_ws_at<T, K>(smem + Lo.ws + warp * full, G, FusedDim<K>::slot);
    while (warp < nro) {
      int item = 0;
      if (lane == 0) item = atomicAdd(&misc[2], 1);
      item = __shfl_sync(kFull, item, 0);
      if (item >= nblk) break;
      const int I = item / nb, J = item % nb;
      const int shape = reg_frame(g, I, J, kDirR).shape();
      if (reg && shape != kShapeNone && shape <= kShapeDot) continue;   // read out above
      const Frame f = make_frame(c, I, J, kDirR);
      LogAcc<T> ls[kFusedMaxG];
      fused_sweep(ws, c, msgs, stride, all, G, frames, f, ls, lane);
      const int right = J + 1 < nb ? msg_index(c, I, J + 1, kDirL) : -1;
      if (!dev_check(right >= -1 && right < M, &misc[4])) continue;
#pragma unroll
      for (int q = 0; q < G; ++q) {
        // On the grid border the right side has no message: missing legs
        // carry the value 0, so only entry 0 survives.
        const T z = right >= 0 ? read_dot(ws.s0 + (q << f.h), msgs + q * stride + right * VEC, 1 << f.h, lane)
                               : ws.s0[q << f.h];
        close_block(ls[q], z, q, item);
      }
      __syncwarp();
    }
  }
  // Edge overlaps o_e = <m_uv|m_vu>.  Horizontal edges first, then vertical.
  {
    const int nh = nb * (nb - 1);
    auto edge_of = [&](int e, int& idx, int& other, int& at, int& w) {
      int I, J;
      if (e < nh) {
        I = e / (nb - 1); J = e - I * (nb - 1);
        idx = message_index(nb, I, J, kDirR); other = message_index(nb, I, J + 1, kDirL);
        w = g.len(I);
      } else {
        I = (e - nh) / nb; J = e - nh - I * nb;
        idx = message_index(nb, I, J, kDirD); other = message_index(nb, I + 1, J, kDirU);
        w = g.len(J);
      }
      // Its rank among the rightward and downward messages.
      at = nblk + I * (2 * nb - 1) + J + (I + 1 < nb ? J : 0) + (e >= nh && J + 1 < nb ? 1 : 0);
    };
    if constexpr (K <= 4) {                          // eight (edge, coset) jobs a pass, entries beyond 2^w are zero
      const int passes = (nedge * G + 7) >> 3;
      int p = warp - first % NW;
      if (p < 0) p += NW;
      for (; p < passes; p += NW) {
        const int j = p * 8 + (lane >> 2), q = j % G;
        const bool on = j / G < nedge;
        int idx, other, at, w;
        edge_of(on ? j / G : nedge - 1, idx, other, at, w);
        if (!dev_check(idx >= 0 && idx < M && other >= 0 && other < M && at < per, &misc[4])) idx = other = 0;
        const T* x = msgs + q * stride + idx * VEC;
        const T* y = msgs + q * stride + other * VEC;
        const RowAt ra(false, (lane >> 1) & 1, lane & 1);
        T v[2][2];
#pragma unroll
        for (int s = 0; s < 2; ++s)
#pragma unroll
          for (int t = 0; t < 2; ++t) v[s][t] = x[ra(s, t)] * y[ra(s, t)];
        const T o = job_sum(v);
        if (on && (lane & 3) == 0 && at < per) record(q, at, o);
      }
    } else {
      for (int e = warp; e < nedge; e += NW) {
        int idx, other, at, w;
        edge_of(e, idx, other, at, w);
        if (!dev_check(idx >= 0 && idx < M && other >= 0 && other < M && at < per, &misc[4])) continue;
        const T o = read_dot(msgs + idx * VEC, msgs + other * VEC, 1 << w, lane);
        if (lane == 0) record(0, at, o);
      }
    }
  }
  __syncthreads();
  if (warp < G) {
    double acc = 0.0;
    if constexpr (sizeof(T) == 4) {
      // Products of the block values and of the edge overlaps in a fixed
      // order (lane-strided, then a fixed tree), one log each.
      LogAcc<float> pz, po;
      for (int i = lane; i < per; i += 32) {
        LogAcc<float> r;
        r.m = reinterpret_cast<const float*>(rlog + warp * per + i)[0];
        r.e = reinterpret_cast<const int*>(rlog + warp * per + i)[1];
        if (i < nblk) pz.mul(r); else po.mul(r);
      }
#pragma unroll
      for (int msk = 16; msk >= 1; msk >>= 1) {
        LogAcc<float> oz, oo;
        oz.m = __shfl_xor_sync(kFull, pz.m, msk);
        oz.e = __shfl_xor_sync(kFull, pz.e, msk);
        oo.m = __shfl_xor_sync(kFull, po.m, msk);
        oo.e = __shfl_xor_sync(kFull, po.e, msk);
        pz.mul(oz);
        po.mul(oo);
      }
      if (lane == 0) acc = pz.value() - po.value();   // FP64 logs on one lane (2 FP64 lanes a cycle per SM)
    } else {
      for (int i = lane; i < per; i += 32) acc += rlog[warp * per + i];
      acc = warp_sum(acc);
    }
    if (lane == 0) {
      const double dq = M > 0 ? sqrt(dsh[warp]) / M : 0.0;
      const int iq = misc[8 + warp];
      // Capacity and check failures are recorded on the first coset's word
      // and hold for every coset of the item.
      int fl = misc[4 + warp] | (misc[4] & (kFlagCapacity | kFlagCheck));
      if (!isfinite(acc)) fl |= kFlagNonfinite;
      if (!(dq < a.delta1)) fl |= kFlagUntrusted;
      const long long row = syn * 4 + c0 + warp;
      a.logp[row] = acc;
      a.delta[row] = dq;
      a.iters[row] = iq;
      a.flags[row] = fl;
    }
  }
}

// Messages in shared memory: one CTA per (syndrome, group of G cosets).
// Messages in the workspace (GM; always for k = 5, 6): a persistent grid,
// CTA b taking items b, b + gridDim.x, ... with its messages in slot b.
template <typename T, int NW, int G, int K, bool GM = (K > 4), int LB = 0>
__global__ void __launch_bounds__(NW * 32, (FusedMinBlocks<T, NW, G, K, LB>::value)) fused_kernel(KArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int NG = 4 / G;
  const int m = 2 * a.geo.d * (a.geo.d - 1);
  if constexpr (GM) {
    T* gm = a.arena + (long long)blockIdx.x * a.slot_elems;
    for (long long item = blockIdx.x; item < a.n_items; item += gridDim.x) {
      const long long syn = item / NG;
      fused_item<T, NW, G, K, true, LB>(a, a.geo, a.M, a.synd + syn * m, syn, (int)(item % NG) * G, smem, gm);
      __syncthreads();
    }
  } else {
    const long long syn = blockIdx.x / NG;
    const int c0 = (int)(blockIdx.x % NG) * G;
    fused_item<T, NW, G, K, false, LB>(a, a.geo, a.M, a.synd + syn * m, syn, c0, smem, nullptr);
  }
}

// A batch of syndromes of different distances in one persistent launch: CTAs
// take (syndrome, coset group) items from a global counter in the order
// given (largest distance first balances the tail) until the batch is done.
struct MixedArgs {
  const int32_t* d_of;          // distance of each syndrome
  const int64_t* offsets;       // byte offset of each syndrome in the packed buffer
  const int32_t* order;         // syndrome order of the items, or null
  unsigned long long* counter;  // zero before the launch
  long long n_items;            // B * (4 / G)
  long long B;                  // syndromes
  int k, d_max;                 // shared memory is sized for d_max
};

// LB > 0: the register-form-only kernel (every distance of the batch odd).
template <typename T, int NW, int G, int K, bool GM = (K > 4), int LB = 0>
__global__ void __launch_bounds__(NW * 32, (FusedMinBlocks<T, NW, G, K, LB>::value))
    fused_mixed_kernel(KArgs<T> a, MixedArgs mx) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ long long item_sh;
  constexpr int NG = 4 / G;
  for (;;) {
    if (threadIdx.x == 0) item_sh = (long long)atomicAdd(mx.counter, 1ull);
    __syncthreads();
    const long long item = item_sh;
    __syncthreads();
    if (item >= mx.n_items) break;
    const long long shot = mx.order ? (long long)mx.order[item / NG] : (item / NG);
    const int c0 = (int)(item % NG) * G;
    // The batch comes from device buffers the host cannot read: a syndrome
    // index outside the batch is skipped, a distance outside 2..d_max (more
    // than the shared memory holds) gives its rows kFlagCheck and NaN.
    if (shot < 0 || shot >= mx.B) continue;
    const int d = mx.d_of[shot];
    if (d < 2 || d > mx.d_max) {
      if (threadIdx.x < G) {
        const long long row = shot * 4 + c0 + threadIdx.x;
        a.logp[row] = __longlong_as_double(0x7ff8000000000000ll);
        a.delta[row] = __longlong_as_double(0x7ff8000000000000ll);
        a.iters[row] = 0;
        a.flags[row] = kFlagCheck | kFlagNonfinite;
      }
      continue;
    }
    const Geo g = make_geo(d, mx.k);
    int M = 0, ae = 0;
    count_messages(g, 1, &M, &ae);
    fused_item<T, NW, G, K, GM, LB>(a, g, M, a.synd + mx.offsets[shot], shot, c0, smem,
                                    GM ? a.arena + (long long)blockIdx.x * a.slot_elems : nullptr);
    __syncthreads();
  }
}

}  // namespace bbp
