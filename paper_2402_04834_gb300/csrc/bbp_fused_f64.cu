// FP64 instances of the fused-block kernel (Remark 9) and the table of the
// compiled launch shapes (warps per CTA, cosets per CTA) of both precisions.
#include "bbp_decode_inst.cuh"

namespace bbp {

cudaError_t launch_fused_f64(const LaunchArgs& a, int warps, int cosets, bool gm, int lean, cudaStream_t st) {
  if (lean > 0 && a.geo.k > 4) {           // small state buffers, sized for `lean` CTAs per SM
    switch (warps * 100 + cosets * 10 + lean) {
      case 811: return launch_fused_nw<double, 8, 1, 6, true, 1>(a, st);
      default: return cudaErrorInvalidValue;
    }
  }
  if (lean > 0) {                          // every block update in register form, sized for `lean` CTAs per SM
    switch (warps * 100 + cosets * 10 + lean) {
      case 1611: return launch_fused_nw<double, 16, 1, 4, false, 1>(a, st);
      case 1621: return launch_fused_nw<double, 16, 2, 4, false, 1>(a, st);
      case 841: return launch_fused_nw<double, 8, 4, 4, false, 1>(a, st);
      case 443: return launch_fused_nw<double, 4, 4, 4, false, 3>(a, st);
      case 424: return launch_fused_nw<double, 4, 2, 4, false, 4>(a, st);
      case 822: return launch_fused_nw<double, 8, 2, 4, false, 2>(a, st);
      default: return cudaErrorInvalidValue;
    }
  }
  if (a.geo.k > 4) {
    switch (warps * 10 + cosets) {
      case 21: return launch_fused_nw<double, 2, 1, 6>(a, st);
      case 31: return launch_fused_nw<double, 3, 1, 6>(a, st);
      default: return cudaErrorInvalidValue;
    }
  }
  if (gm) return warps * 10 + cosets == 42 ? launch_fused_nw<double, 4, 2, 4, true>(a, st) : cudaErrorInvalidValue;
  switch (warps * 10 + cosets) {
    case 81: return launch_fused_nw<double, 8, 1, 4>(a, st);
    case 42: return launch_fused_nw<double, 4, 2, 4>(a, st);
    case 82: return launch_fused_nw<double, 8, 2, 4>(a, st);
    case 44: return launch_fused_nw<double, 4, 4, 4>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_fused_mixed_f64(const LaunchArgs& a, const MixedLaunch& m, int warps, int cosets, bool gm,
                                   int lean, cudaStream_t st) {
  if (lean > 0) {                          // every distance odd: every block update in register form
    switch (warps * 100 + cosets * 10 + lean) {
      case 1611: return launch_fused_mixed_nw<double, 16, 1, 4, false, 1>(a, m, st);
      case 1621: return launch_fused_mixed_nw<double, 16, 2, 4, false, 1>(a, m, st);
      case 841: return launch_fused_mixed_nw<double, 8, 4, 4, false, 1>(a, m, st);
      case 443: return launch_fused_mixed_nw<double, 4, 4, 4, false, 3>(a, m, st);
      case 424: return launch_fused_mixed_nw<double, 4, 2, 4, false, 4>(a, m, st);
      case 822: return launch_fused_mixed_nw<double, 8, 2, 4, false, 2>(a, m, st);
      default: return cudaErrorInvalidValue;
    }
  }
  if (a.geo.k > 4) {
    switch (warps * 10 + cosets) {
      case 21: return launch_fused_mixed_nw<double, 2, 1, 6>(a, m, st);
      case 31: return launch_fused_mixed_nw<double, 3, 1, 6>(a, m, st);
      default: return cudaErrorInvalidValue;
    }
  }
  if (gm)
    return warps * 10 + cosets == 42 ? launch_fused_mixed_nw<double, 4, 2, 4, true>(a, m, st) : cudaErrorInvalidValue;
  switch (warps * 10 + cosets) {
    case 81: return launch_fused_mixed_nw<double, 8, 1, 4>(a, m, st);
    case 42: return launch_fused_mixed_nw<double, 4, 2, 4>(a, m, st);
    case 82: return launch_fused_mixed_nw<double, 8, 2, 4>(a, m, st);
    case 44: return launch_fused_mixed_nw<double, 4, 4, 4>(a, m, st);
    default: return cudaErrorInvalidValue;
  }
}

namespace {

struct Shape {
  int warps, cosets;
  bool gm;        // messages in a workspace slot of the CTA instead of shared memory
  int lean = 0;   // > 0: every block update in register form, sized for this many CTAs per SM
};

// The shapes that can be asked for, in order of preference: the
// register-form-only kernels where the geometry allows them, then
// shared-memory messages where they leave room for the CTAs per SM of
// target_blocks, then the same shape with its messages in the workspace.  They
// decide what is accepted and the workspace it needs; a default launch takes its
// kernel from fused_pick, and the first of these that fits where that has none
// (k <= 3 and the geometries it leaves).
constexpr Shape kShapesF32[] = {{8, 4, false, 4}, {8, 4, false, 3}, {8, 2, false, 4}, {8, 4, false}, {8, 4, true}, {8, 2, false},
                                {8, 2, true}, {4, 2, false}, {4, 4, false}, {16, 1, false}, {8, 1, false},
                                {4, 1, false}};
constexpr Shape kShapesF64[] = {{4, 2, false, 4}, {8, 2, false, 2}, {4, 2, false}, {4, 2, true}, {8, 2, false},
                                {8, 1, false}, {4, 4, false}};

// Block sides 5 and 6: states of 2^12 entries, one coset per CTA, messages
// in the workspace; the most warps whose state buffers fit one SM first.
constexpr Shape kShapesF32K6[] = {{6, 1, true}, {4, 1, true}, {2, 1, true}};
constexpr Shape kShapesF64K6[] = {{3, 1, true}, {2, 1, true}};

// Resident CTAs per SM that the register budget of a shape is sized for
// (the host-side value of FusedMinBlocks).
int target_blocks(int precision, int k, const Shape& s) {
  if (s.lean > 0) return s.lean;
  const int warps = k > 4 ? s.warps : (precision == 0 ? 16 : 32) / (s.cosets > 1 ? 2 : 1);
  return warps / s.warps > 1 ? warps / s.warps : 1;
}

}  // namespace

// The shared memory that decides which geometries a shape is accepted for
// and where the default shape keeps its messages (hence the workspace a
// caller provides).  These limits are part of the interface, so they stay
// where they were when they were set; the kernels need no more than this
// (fused_layout).
static int admitted_smem(int precision, const Geo& g, int M, int warps, int cosets, bool gm, bool lean) {
  const int K = g.k > 4 ? 6 : 4, vec = 1 << K, slot = lean ? vec : 1 << (2 * K), sz = precision == 0 ? 8 : 4;
  const int side = K == 4 && cosets < 2 ? 2 : cosets;
  int o = align_up(2 * g.d * (g.d - 1), 16);
  o += align_up(cosets * g.W * g.W, 16) + align_up(8 * g.nb * g.nb, 16) + align_up(2 * M, 16) + align_up(4 * M, 16);
  o += align_up(sz * cosets * M, 16) + align_up(8 * cosets * (g.nb * g.nb + M), 16) + 128;
  if (g.k == 4) o += align_up(10 * M, 16) + align_up(2 * cosets * M, 16);
  if (!gm) o += sz * vec * cosets * M;
  return align_up(o + warps * align_up(sz * (cosets * (2 * slot + 16) + 2 * side * vec), 16), 16);
}

bool fused_shape(int precision, const Geo& g, int M, int* warps, int* cosets, int* messages, bool allow_lean,
                 int* lean_blocks) {
  const bool k6 = g.k > 4;
  const Shape* sh = k6 ? (precision == 0 ? kShapesF64K6 : kShapesF32K6) : (precision == 0 ? kShapesF64 : kShapesF32);
  const int n = k6 ? (precision == 0 ? (int)(sizeof(kShapesF64K6) / sizeof(Shape)) : (int)(sizeof(kShapesF32K6) / sizeof(Shape)))
                   : (precision == 0 ? (int)(sizeof(kShapesF64) / sizeof(Shape)) : (int)(sizeof(kShapesF32) / sizeof(Shape)));
  // Pass 0 keeps only shapes whose shared memory allows their target CTAs
  // per SM; pass 1 any shape that fits.
  for (int pass = 0; pass < 2; ++pass) {
    for (int i = 0; i < n; ++i) {
      if (*warps != 0 && sh[i].warps != *warps) continue;
      if (*cosets != 0 && sh[i].cosets != *cosets) continue;
      const int mem = sh[i].lean > 0 ? 3 : (sh[i].gm ? 2 : 1);
      if (*messages != 0 && *messages != mem) continue;
      if (sh[i].lean > 0 && (!allow_lean || !register_form_only(g))) continue;
      const int smem = admitted_smem(precision, g, M, sh[i].warps, sh[i].cosets, sh[i].gm, sh[i].lean > 0);
      if (smem > kMaxSmemBytes) continue;
      if (pass == 0 && kSmemPerSm / (smem + kSmemReservedPerCta) < target_blocks(precision, g.k, sh[i])) continue;
      *warps = sh[i].warps;
      *cosets = sh[i].cosets;
      *messages = mem;
      if (lean_blocks) *lean_blocks = sh[i].lean;
      return true;
    }
  }
  return false;
}

// The kernel of a default launch at k = 4 where every block has a register
// form, for B syndromes (G = 4 / cosets CTAs each) on sms SMs.  Few
// syndromes: as many CTAs as SMs allow at one per SM, 16 warps each, so that
// a half-round of one coset's messages is a single round of passes (d = 11:
// 1 syndrome 148 us with (8, 4), 74 us with (16, 1); 64 at d = 9: 125 and 78;
// 152 at d = 11: 170 with (8, 4, 4), 137 with (16, 4, 1)).  Then four cosets per
// CTA and as many CTAs as shared memory allows: the more warps per CTA the
// fewer CTAs fit ((8, 4, 4) at d = 11, 3 at 13 and 15, 2 at 17, and from d = 19
// on one CTA of 16 warps: d = 21, 2000 syndromes 4.64 ms against 5.58 for (8,
// 4, 2) and 4.93 for (8, 2, 2)).  Small codes have too few passes per
// half-round for 8 warps: four warps where six such CTAs fit (d <= 9; d = 5,
// 10^4 syndromes 1.58 ms against 1.78), or five and the batch is long enough
// to hide its slower CTAs' tail (d = 11, 10^4 syndromes 4.93 ms against 5.06).
// Where four cosets do not fit (d >= 27), two or one.  Batches that may hold
// even distances take the kernels that know three-wide blocks too, by the
// same rule.  FP64 is bound by its pipe, so at large batches the shape
// matters little (within 7 % at d = 11, 1000 syndromes) but for the smallest
// codes ((4, 4, 3) at d = 5, 1000 syndromes: a quarter less than (8, 2, 2));
// small batches gain most (one syndrome at d = 11: (16, 1) 0.58 of (4, 2)).
// Block sides 5 and 6 (messages in workspace slots, one coset per CTA): the
// kernels with small state buffers, 16 warps per SM (8 in FP64), where every
// block's state fits them (not at k = 6 and d a multiple of 3: small_states).
// In FP32 a half-round of at most six messages (two blocks a side), one network
// per SM, is no more than the full-size kernel's six warps, which have twice the
// registers: k = 5, d = 5, 30 syndromes 230 us against 256 (d = 6, 12 messages: 393
// against 319), k = 6, d = 5: 194 against 227.
bool fused_pick(int precision, const Geo& g, int M, long long B, int sms, bool odd, int* warps, int* cosets,
                int* lean) {
  if (g.k > 4) {
    if (!small_states(g)) return false;
    auto fit6 = [&](int w) {
      const int smem = precision == 0 ? fused_smem_for<double, 6>(g, M, w, 1, true, true)
                                      : fused_smem_for<float, 6>(g, M, w, 1, true, true);
      return smem > kMaxSmemBytes ? 0 : kSmemPerSm / (smem + kSmemReservedPerCta);
    };
    *cosets = 1;
    if (precision == 0) {
      if (fit6(8) < 1) return false;
      *warps = 8; *lean = 1;
      return true;
    }
    if (4 * B > sms && fit6(8) >= 2) {
      *warps = 8; *lean = 2;
      return true;
    }
    if (4 * B <= sms && (M + 1) / 2 <= 6) return false;
    if (fit6(16) < 1) return false;
    *warps = 16; *lean = 1;
    return true;
  }
  auto fit = [&](int w, int c) {
    const int smem = precision == 0 ? fused_smem_for<double, 4>(g, M, w, c, false, odd ? 1 : 2)
                                    : fused_smem_for<float, 4>(g, M, w, c, false, odd ? 1 : 2);
    return smem > kMaxSmemBytes ? 0 : kSmemPerSm / (smem + kSmemReservedPerCta);
  };
  auto take = [&](int w, int c, int l) { *warps = w; *cosets = c; *lean = odd ? l : kEvenLB + l; return true; };
  int c = 4 * B <= sms ? 1 : (2 * B <= sms ? 2 : 4);
  while (c > 1 && fit(16, c) < 1) c /= 2;
  if (fit(16, c) < 1) return false;
  if (precision == 0) {
    if (c < 4) return take(16, c, 1);
    if (B <= sms) return take(8, 4, 1);
    if (odd && fit(4, 4) >= 6) return take(4, 4, 3);
    return fit(8, 2) >= 2 ? take(8, 2, 2) : take(16, 2, 1);
  }
  if (B <= sms || c < 4 || fit(8, 4) < 2) return take(16, c, 1);
  if (B <= 2ll * sms) return take(8, 4, 2);
  if (odd && (fit(4, 4) >= 6 || (fit(4, 4) >= 5 && B >= 16ll * sms))) return take(4, 4, 6);
  const int n = fit(8, 4);
  return take(8, 4, n < 4 ? n : 4);
}

}  // namespace bbp
