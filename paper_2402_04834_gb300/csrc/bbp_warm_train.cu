// One training step of the warm-start network F -> H -> H -> O with GELU
// (forward, the loss 1 - <u, t>^2 of Remark 4's Delta term, backward, Adam),
// FP32 throughout on the CUDA cores.
//
// A step over N rows is five 256 x 256 x N contractions (two forward, one
// data gradient, two weight gradients: 6.6 GFLOP at N = 8192 with the output
// layer) and the row-wise output layer and head.  Its bound is the FP32 pipe;
// the operands (a few N x 256 matrices) stay in L2.  Seven launches:
//   gemm forward x 2      Z = X W + b and GELU(Z)
//   head_kernel           output layer, loss, dL/dlogits, the gradient at Z2
//                         and the partial sums of gW3, gb3, gb2: one read of
//                         A2 and Z2
//   gemm weight gradient  gW2 = A1^T G2
//   gemm data gradient    G1 = (G2 W2^T) GELU'(Z1), and gb1's partial sums
//   gemm weight gradient  gW1 = X^T G1
//   finish_kernel         sums the partials in a fixed order, Adam
// A weight gradient sums over the N rows into only 16 tiles of 64 x 64, so
// its rows are split over up to kSplits groups of CTAs; unsplit, each of the
// two kept 16 of 152 SMs busy for 2.2 ms at N = 8192.  With that and with
// separate passes for the head, GELU' and the column sums a step took 4314 us
// from call to call; it takes 245 us.
// Every sum has a fixed order: two runs give the same bits.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "../../include/blockbp.h"
#include "bbp_warm_tc.h"

namespace bbp {
namespace warm {
namespace {

constexpr int F = BBP_WARM_FEATURES;   // 256
constexpr int H = BBP_WARM_HIDDEN;     // 256
constexpr int O = BBP_WARM_OUT;        // 16
constexpr int kParams = F * H + H + H * H + H + H * O + O;

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float x) {
  return 0.5f * (1.f + erff(x * 0.70710678118654752f)) + x * expf(-0.5f * x * x) * 0.39894228040143268f;
}

// ---------------------------------------------------------------------------
// C = op(A) op(B) over tiles of 64 x 64 x 16, 128 threads with 8 x 4 outputs
// each: at N = 8192 the forward grid is 512 CTAs, all resident (about 3.4
// per SM), and small N still spreads.  Per k a warp issues 32 multiply-adds
// a lane for three 16-byte shared loads; the next tile's global loads are
// issued before the current tile's arithmetic (two shared buffers, one
// barrier a tile).  The k order is ascending.
enum Epi { kForward, kData, kWeight };

struct GemmArgs {
  int M, Kb, Ke;              // rows of C (kForward, kData), k range of the whole product
  int chunk;                  // kWeight: k per split (blockIdx.z)
  const float* A;
  int lda;
  const float* B;
  int ldb;
  float* C;                   // kWeight: + blockIdx.z * H * H
  const float* bias;          // kForward
  float* Z;                   // kForward: Z out; kData: Z in, at C's own places
  float* colpart;             // kData: column sums of C per row tile, [gridDim.y][H]
  int vec;                    // A, B (and nothing else read through float4) 16-byte aligned
};

constexpr int BM = 64, BN = 64, BK = 16, kLd = BM + 4;

// Four consecutive floats of an operand, zero outside (whole quads are in or
// out: rows and k ranges are tested by the caller).
__device__ __forceinline__ float4 quad(const float* p, bool in, int vec) {
  if (!in) return make_float4(0.f, 0.f, 0.f, 0.f);
  if (vec) return *reinterpret_cast<const float4*>(p);
  return make_float4(p[0], p[1], p[2], p[3]);
}

// TA: A is stored k x m; TB: B is stored n x k (both row-major).
template <bool TA, bool TB, Epi E>
__global__ void __launch_bounds__(128) gemm_kernel(GemmArgs a) {
  __shared__ __align__(16) float As[2][BK][kLd];
  __shared__ __align__(16) float Bs[2][BK][kLd];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  int kb = a.Kb, ke = a.Ke;
  if (E == kWeight) {
    kb = a.Kb + blockIdx.z * a.chunk;
    ke = min(a.Ke, kb + a.chunk);
  }
  float4 ra[2], rb[2];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int f = tid + 128 * u;
      if (TA) {
        const int k = k0 + (f >> 4), m = m0 + 4 * (f & 15);
        ra[u] = quad(a.A + (long long)k * a.lda + m, k < ke, a.vec);
      } else {
        const int m = m0 + (f >> 2), k = k0 + 4 * (f & 3);
        ra[u] = quad(a.A + (long long)m * a.lda + k, m < a.M, a.vec);
      }
      if (TB) {
        const int n = n0 + (f >> 2), k = k0 + 4 * (f & 3);
        rb[u] = quad(a.B + (long long)n * a.ldb + k, true, a.vec);
      } else {
        const int k = k0 + (f >> 4), n = n0 + 4 * (f & 15);
        rb[u] = quad(a.B + (long long)k * a.ldb + n, k < ke, a.vec);
      }
    }
  };
  auto put = [&](int buf) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int f = tid + 128 * u;
      if (TA) {
        *reinterpret_cast<float4*>(&As[buf][f >> 4][4 * (f & 15)]) = ra[u];
      } else {
        const int m = f >> 2, k = 4 * (f & 3);
        As[buf][k][m] = ra[u].x; As[buf][k + 1][m] = ra[u].y;
        As[buf][k + 2][m] = ra[u].z; As[buf][k + 3][m] = ra[u].w;
      }
      if (TB) {
        const int n = f >> 2, k = 4 * (f & 3);
        Bs[buf][k][n] = rb[u].x; Bs[buf][k + 1][n] = rb[u].y;
        Bs[buf][k + 2][n] = rb[u].z; Bs[buf][k + 3][n] = rb[u].w;
      } else {
        *reinterpret_cast<float4*>(&Bs[buf][f >> 4][4 * (f & 15)]) = rb[u];
      }
    }
  };
  float acc[8][4] = {};
  fetch(kb);
  put(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = kb; k0 < ke; k0 += BK, buf ^= 1) {
    const bool more = k0 + BK < ke;
    if (more) fetch(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][kk][8 * ty]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][kk][8 * ty + 4]);
      const float4 b = *reinterpret_cast<const float4*>(&Bs[buf][kk][4 * tx]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
    if (more) put(buf ^ 1);
    __syncthreads();
  }
  float cs[4] = {0.f, 0.f, 0.f, 0.f};
  const int n = n0 + 4 * tx;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = m0 + 8 * ty + i;
    if (E != kWeight && m >= a.M) break;
    if (E == kForward) {
      float z[4], g[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        z[j] = acc[i][j] + a.bias[n + j];
        g[j] = gelu(z[j]);
      }
      *reinterpret_cast<float4*>(a.Z + (long long)m * H + n) = make_float4(z[0], z[1], z[2], z[3]);
      *reinterpret_cast<float4*>(a.C + (long long)m * H + n) = make_float4(g[0], g[1], g[2], g[3]);
    } else if (E == kData) {
      const float4 z = *reinterpret_cast<const float4*>(a.Z + (long long)m * H + n);
      float4 g;
      g.x = acc[i][0] * gelu_grad(z.x); g.y = acc[i][1] * gelu_grad(z.y);
      g.z = acc[i][2] * gelu_grad(z.z); g.w = acc[i][3] * gelu_grad(z.w);
      *reinterpret_cast<float4*>(a.C + (long long)m * H + n) = g;
      cs[0] += g.x; cs[1] += g.y; cs[2] += g.z; cs[3] += g.w;
    } else {
      float* c = a.C + (long long)blockIdx.z * H * H + (long long)m * H + n;   // possibly the caller's gradient
      c[0] = acc[i][0]; c[1] = acc[i][1]; c[2] = acc[i][2]; c[3] = acc[i][3];
    }
  }
  if (E == kData) {            // As is free: every thread is past the last tile's barrier
    float* red = &As[0][0][0];
#pragma unroll
    for (int j = 0; j < 4; ++j) red[ty * BN + 4 * tx + j] = cs[j];
    __syncthreads();
    if (tid < BN) {
      float s = 0.f;
      for (int y = 0; y < 8; ++y) s += red[y * BN + tid];
      a.colpart[(long long)blockIdx.y * H + n0 + tid] = s;
    }
  }
}

// ---------------------------------------------------------------------------
// Output layer and head of kRows rows: logits = A2 W3 + b3, u = masked
// exp(logits - max) / norm, the loss 1 - <u, t>^2 and dL/dlogits (mean over
// N), then dL/dZ2 = (dL/dlogits W3^T) GELU'(Z2) and the rows' partial sums
// of gW3, gb3, gb2 and the loss.  The A2 tile is staged once and serves the
// logits and gW3.
constexpr int kRows = 32;
constexpr int kLdA = H + 4;
constexpr int kPartLoss = H * O + O + H;            // per CTA: gW3, gb3, gb2, loss
constexpr int kPart = kPartLoss + 1;

struct HeadArgs {
  const float *A2, *Z2, *W3, *b3, *targets;
  const int32_t* lens;
  float* G2;
  float* part;                                      // [gridDim.x][kPart]
  long long N;
};

constexpr int kHeadSmem = (kRows * kLdA + H * O + kRows * O) * (int)sizeof(float);

__global__ void __launch_bounds__(256) head_kernel(HeadArgs a) {
  extern __shared__ __align__(16) float sm[];
  float* sA = sm;                                   // [kRows][kLdA]
  float* sW = sA + kRows * kLdA;                    // [H][O]
  float* sG = sW + H * O;                           // [kRows][O]
  __shared__ float sLoss[kRows];
  const int tid = threadIdx.x;
  const long long r0 = (long long)blockIdx.x * kRows;
  const int nr = (int)min((long long)kRows, a.N - r0);
  for (int e = tid; e < kRows * (H / 4); e += 256) {
    const int r = e / (H / 4), q = e % (H / 4);
    const float4 v = r < nr ? *reinterpret_cast<const float4*>(a.A2 + (r0 + r) * H + 4 * q)
                            : make_float4(0.f, 0.f, 0.f, 0.f);
    *reinterpret_cast<float4*>(sA + r * kLdA + 4 * q) = v;
  }
  for (int e = tid; e < H * O; e += 256) sW[e] = a.W3[e];
  __syncthreads();
  {
    // Eight lanes per row, two logits each, k ascending.
    const int r = tid >> 3, o = 2 * (tid & 7);
    float l0 = 0.f, l1 = 0.f;
    for (int k = 0; k < H; k += 4) {
      const float4 x = *reinterpret_cast<const float4*>(sA + r * kLdA + k);
      const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 w = *reinterpret_cast<const float2*>(sW + (k + j) * O + o);
        l0 = fmaf(xv[j], w.x, l0);
        l1 = fmaf(xv[j], w.y, l1);
      }
    }
    l0 += a.b3[o];
    l1 += a.b3[o + 1];
    const bool in = r < nr;
    const int n = in ? a.lens[r0 + r] : 1;
    float mx = fmaxf(o < n ? l0 : -INFINITY, o + 1 < n ? l1 : -INFINITY);
#pragma unroll
    for (int s = 4; s > 0; s >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, s));
    const float m0 = o < n ? expf(l0 - mx) : 0.f, m1 = o + 1 < n ? expf(l1 - mx) : 0.f;
    float s2 = m0 * m0 + m1 * m1;
#pragma unroll
    for (int s = 4; s > 0; s >>= 1) s2 += __shfl_xor_sync(0xffffffffu, s2, s);
    const float inv = 1.f / sqrtf(s2);
    const float t0 = in ? a.targets[(r0 + r) * O + o] : 0.f, t1 = in ? a.targets[(r0 + r) * O + o + 1] : 0.f;
    float c = m0 * inv * t0 + m1 * inv * t1;
#pragma unroll
    for (int s = 4; s > 0; s >>= 1) c += __shfl_xor_sync(0xffffffffu, c, s);
    // dL/du = -2 c t / N; dL/dm = (gu - <gu, u> u) / |m|; dL/do = dL/dm m.
    const float sc = -2.f * c / (float)a.N;
    float gu_u = sc * t0 * m0 * inv + sc * t1 * m1 * inv;
#pragma unroll
    for (int s = 4; s > 0; s >>= 1) gu_u += __shfl_xor_sync(0xffffffffu, gu_u, s);
    sG[r * O + o] = in ? (sc * t0 - gu_u * m0 * inv) * inv * m0 : 0.f;
    sG[r * O + o + 1] = in ? (sc * t1 - gu_u * m1 * inv) * inv * m1 : 0.f;
    if (o == 0) sLoss[r] = in ? 1.f - c * c : 0.f;
  }
  __syncthreads();
  // A thread per hidden unit: its row of W3 and its column of gW3 in registers.
  float w3[O], gw[O];
#pragma unroll
  for (int o = 0; o < O; ++o) { w3[o] = sW[tid * O + o]; gw[o] = 0.f; }
  float gb2 = 0.f;
#pragma unroll 2
  for (int r = 0; r < nr; ++r) {
    const float x = sA[r * kLdA + tid];
    float g = 0.f;
#pragma unroll
    for (int q = 0; q < O; q += 4) {
      const float4 go = *reinterpret_cast<const float4*>(sG + r * O + q);
      const float gv[4] = {go.x, go.y, go.z, go.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        g = fmaf(gv[j], w3[q + j], g);
        gw[q + j] = fmaf(x, gv[j], gw[q + j]);
      }
    }
    g *= gelu_grad(a.Z2[(r0 + r) * H + tid]);
    a.G2[(r0 + r) * H + tid] = g;
    gb2 += g;
  }
  float* part = a.part + (long long)blockIdx.x * kPart;
#pragma unroll
  for (int o = 0; o < O; ++o) part[tid * O + o] = gw[o];
  part[H * O + O + tid] = gb2;
  if (tid < O) {
    float s = 0.f;
    for (int r = 0; r < nr; ++r) s += sG[r * O + tid];
    part[H * O + tid] = s;
  }
  if (tid == 32) {
    float s = 0.f;
    for (int r = 0; r < nr; ++r) s += sLoss[r];
    part[kPartLoss] = s;
  }
}

// ---------------------------------------------------------------------------
// Gradients from their partial sums, and Adam.  A CTA takes 32 consecutive
// parameters, its eight warps the partials p = warp, warp + 8, ...; the
// eight sums are added in order.
struct FinishArgs {
  const float *w1, *b1, *w2, *head;                 // partials (w1 / w2: null, the gradient is in grad already)
  int s1, s2, nb1, nhead;
  float *grad, *loss_sum, *theta, *m, *v;           // m, v null: no update
  float lr, c1, c2;
};

__global__ void __launch_bounds__(256) finish_kernel(FinishArgs a) {
  __shared__ float sh[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int e = blockIdx.x * 32 + lane;
  const float* src = nullptr;                       // element e's partials: src[p * stride]
  int n = 0;
  long long stride = 0;
  int at = e;
  if (e < F * H) {
    src = a.w1; n = a.s1; stride = H * H;
  } else if ((at -= F * H) < H) {
    src = a.b1; n = a.nb1; stride = H;
  } else if ((at -= H) < H * H) {
    src = a.w2; n = a.s2; stride = H * H;
  } else if ((at -= H * H) < H) {
    src = a.head + H * O + O; n = a.nhead; stride = kPart;
  } else if ((at -= H) < H * O + O) {
    src = a.head; n = a.nhead; stride = kPart;      // gW3 then gb3, as in theta
  } else if (e == kParams) {
    src = a.head + kPartLoss; n = a.nhead; stride = kPart;
    at = 0;
  }
  float s = 0.f;
  if (src) {
#pragma unroll 4
    for (int p = warp; p < n; p += 8) s += src[p * stride + at];
  }
  sh[warp][lane] = s;
  __syncthreads();
  if (warp || e > kParams) return;
  float g = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) g += sh[w][lane];
  if (e == kParams) {
    *a.loss_sum = g;
    return;
  }
  if (src) a.grad[e] = g;
  else g = a.grad[e];
  if (!a.m) return;
  const float b1 = 0.9f, b2 = 0.999f;
  const float mm = b1 * a.m[e] + (1.f - b1) * g;
  const float vv = b2 * a.v[e] + (1.f - b2) * g * g;
  a.m[e] = mm;
  a.v[e] = vv;
  a.theta[e] -= a.lr * (mm / a.c1) / (sqrtf(vv / a.c2) + 1e-8f);
}

size_t al256(size_t x) { return (x + 255) / 256 * 256; }

// Row groups of a weight gradient: 16 tiles x kSplits = 608 CTAs, four per
// SM; each group at least 128 rows, so that the partials fit in the two
// activation buffers that are dead by then.
constexpr int kSplits = 38;

struct TrainPlan {
  size_t nh, headp, colp, total;
  int splits, nhead, mt;
};

TrainPlan plan(long long N) {
  TrainPlan p;
  p.nh = al256((size_t)N * H * 4);
  p.nhead = (int)((N + kRows - 1) / kRows);
  p.mt = (int)((N + BM - 1) / BM);
  p.splits = (int)(N / 128 < 1 ? 1 : (N / 128 < kSplits ? N / 128 : kSplits));
  p.headp = al256((size_t)p.nhead * kPart * 4);
  p.colp = al256((size_t)p.mt * H * 4);
  p.total = 5 * p.nh + p.headp + p.colp;
  return p;
}

template <bool TA, bool TB, Epi E>
void gemm(const GemmArgs& a, int mt, int splits, cudaStream_t st) {
  gemm_kernel<TA, TB, E><<<dim3(H / BN, mt, splits), 128, 0, st>>>(a);
}

bool al16(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

}  // namespace

size_t train_workspace_bytes(long long N) { return plan(N).total + 256; }   // the base is rounded up to 256 bytes

cudaError_t train_step(float* theta, float* adam_m, float* adam_v, int32_t step, float lr, const float* feats,
                       const float* targets, const int32_t* lens, long long N, float* grad, float* loss_sum,
                       void* workspace, cudaStream_t st) {
  const TrainPlan p = plan(N);
  const float *W1 = theta, *b1 = W1 + F * H, *W2 = b1 + H, *b2 = W2 + H * H, *W3 = b2 + H, *b3 = W3 + H * O;
  char* w = reinterpret_cast<char*>(al256(reinterpret_cast<uintptr_t>(workspace)));
  float* Z1 = reinterpret_cast<float*>(w);                     // then G1, in place
  float* Z2 = reinterpret_cast<float*>(w + p.nh);              // Z2, A2: then gW2's partials
  float* A2 = reinterpret_cast<float*>(w + 2 * p.nh);
  float* A1 = reinterpret_cast<float*>(w + 3 * p.nh);          // A1, G2: then gW1's partials
  float* G2 = reinterpret_cast<float*>(w + 4 * p.nh);
  float* headp = reinterpret_cast<float*>(w + 5 * p.nh);
  float* colp = reinterpret_cast<float*>(w + 5 * p.nh + p.headp);
  const int n = (int)N, vf = al16(feats), vt = al16(theta);
  const int mt = p.mt, chunk = (n + p.splits - 1) / p.splits;
  cudaError_t e = cudaFuncSetAttribute(head_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kHeadSmem);
  if (e != cudaSuccess) return e;
  GemmArgs g{};
  g.M = n; g.Kb = 0; g.Ke = F; g.A = feats; g.lda = F; g.B = W1; g.ldb = H; g.C = A1; g.bias = b1; g.Z = Z1;
  g.vec = vf && vt;
  gemm<false, false, kForward>(g, mt, 1, st);
  g.Ke = H; g.A = A1; g.lda = H; g.B = W2; g.C = A2; g.bias = b2; g.Z = Z2; g.vec = vt;
  gemm<false, false, kForward>(g, mt, 1, st);
  HeadArgs h{A2, Z2, W3, b3, targets, lens, G2, headp, N};
  head_kernel<<<p.nhead, 256, kHeadSmem, st>>>(h);
  GemmArgs q{};
  q.M = H; q.Kb = 0; q.Ke = n; q.chunk = chunk; q.A = A1; q.lda = H; q.B = G2; q.ldb = H; q.vec = 1;
  q.C = p.splits > 1 ? Z2 : grad + F * H + H;
  gemm<true, false, kWeight>(q, H / BM, p.splits, st);
  GemmArgs d{};
  d.M = n; d.Kb = 0; d.Ke = H; d.A = G2; d.lda = H; d.B = W2; d.ldb = H; d.C = Z1; d.Z = Z1; d.colpart = colp;
  d.vec = vt;
  gemm<false, true, kData>(d, mt, 1, st);
  q.A = feats; q.lda = F; q.B = Z1; q.vec = vf; q.C = p.splits > 1 ? A1 : grad;
  gemm<true, false, kWeight>(q, F / BM, p.splits, st);
  FinishArgs f{};
  f.w1 = p.splits > 1 ? A1 : nullptr; f.w2 = p.splits > 1 ? Z2 : nullptr;
  f.s1 = f.s2 = p.splits; f.b1 = colp; f.nb1 = mt; f.head = headp; f.nhead = p.nhead;
  f.grad = grad; f.loss_sum = loss_sum; f.theta = theta; f.lr = lr;
  if (step > 0 && adam_m && adam_v) {
    f.m = adam_m; f.v = adam_v;
    f.c1 = 1.f - powf(0.9f, (float)step); f.c2 = 1.f - powf(0.999f, (float)step);
  }
  finish_kernel<<<(kParams + 1 + 31) / 32, 256, 0, st>>>(f);
  return cudaGetLastError();
}

}  // namespace warm
}  // namespace bbp
