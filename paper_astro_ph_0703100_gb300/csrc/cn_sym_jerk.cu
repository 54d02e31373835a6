// Symmetric force-jerk(-potential) form: the pairs of one moving set, each
// evaluated once.
#include "cn_sym.cuh"

namespace cn {
namespace {

// Per pair, with d = x_j - x_i, w = v_j - v_i, s = |d|^2 + eps2, r = s^-1/2
// and b = 3 (d . w) r^2, particle i gets m_j r^3 d, m_j r^3 (w - b d) and m_j
// r, particle j the same with -m_i (the potential with +m_i). The common r^3,
// d and w - b d serve both sides: 31 lane operations per unordered pair with
// equal masses (33 without, 3 more with the potential) against 2 x 27 for the
// ordered pairs. What bounds it: as the force form, with 12 to 14 of the 31
// to 34 packed operations reading three registers, and 14 shuffles per step;
// all the registers of one CTA per SM (up to 255 per thread) go to four or
// eight particles per thread. Sums are folded every 256 records, 128 at sizes
// where the one-sided kernel's chains are as short (512: 6.8e-8 against 5.5e-8
// at N = 8192). Steps per trip and the flush's form as measured for K = 8 (65536,
// 4 / 8 steps, rolled / not: 2267 .. 2330 us, with the potential 2543 .. 2609).
template <int K_, bool POT>
struct SymJerkPolicy {
  static constexpr int K = K_;
  static constexpr int P = K / 2;
  static constexpr int kSumsI = POT ? 7 : 6;
  static constexpr int kSumsJ = kSumsI;
  static constexpr int kRec = 2;
  static constexpr bool kGuard = false;
  static constexpr int kUnroll = K >= 8 && POT ? 4 : 8;
  static constexpr int kFold = 256;
  static constexpr int kStage = 256;
  static constexpr int kMinBlocks = 1;
  static constexpr bool kWide = true;
  static constexpr bool kLow = false;
  static constexpr bool kRolled = K >= 8 && !POT;
  static constexpr bool kSameMass = false;
  // r^-3 is at least 2e-17 there, and r^-3 w a normal number for |w| > 1e-21
  static constexpr float kHeavyReach = 1e5f;
  static constexpr float kHeavySoft = 1e10f;
  static constexpr float kOwnSign = -1.f;
  float2 nx[P][3], nv[P][3], acc[P][kSumsI];

  __device__ __forceinline__ void load(const SymArgs& a, int64_t p, bool valid, int k, float& mass, float& reach,
                                       float& speed) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f), u = v;
    if (valid) {
      v = __ldg(a.pos + p);
      u = __ldg(a.rec2 + p);
    }
    sym_half(nx[k >> 1][0], k) = -v.x;
    sym_half(nx[k >> 1][1], k) = -v.y;
    sym_half(nx[k >> 1][2], k) = -v.z;
    sym_half(nv[k >> 1][0], k) = -u.x;
    sym_half(nv[k >> 1][1], k) = -u.y;
    sym_half(nv[k >> 1][2], k) = -u.z;
    mass = v.w;
    reach = sym_reach(v);
    speed = sym_reach(u);
  }

  template <int MODE, bool BOTH>
  __device__ __forceinline__ void term(const float4 r0, const float4 r1, float2 e2, const float2 (&nm)[P],
                                       float2 (&c)[kSumsJ]) {
    const float2 jx = sym_dup(r0.x), jy = sym_dup(r0.y), jz = sym_dup(r0.z), jm = sym_dup(r0.w);
    const float2 ux = sym_dup(r1.x), uy = sym_dup(r1.y), uz = sym_dup(r1.z), m3 = sym_dup(-3.f);
#pragma unroll
    for (int p = 0; p < P; ++p) {
      const float2 dx = __fadd2_rn(jx, nx[p][0]);
      const float2 dy = __fadd2_rn(jy, nx[p][1]);
      const float2 dz = __fadd2_rn(jz, nx[p][2]);
      const float2 wx = __fadd2_rn(ux, nv[p][0]);
      const float2 wy = __fadd2_rn(uy, nv[p][1]);
      const float2 wz = __fadd2_rn(uz, nv[p][2]);
      float2 s, d2;
      if constexpr (POT) {
        d2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
        s = __fadd2_rn(d2, e2);
      } else {
        s = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, e2)));
      }
      const float2 r = make_float2(rsqrt_mufu(s.x), rsqrt_mufu(s.y));
      const float2 rr = __fmul2_rn(r, r);
      const float2 dw = __ffma2_rn(dx, wx, __ffma2_rn(dy, wy, __fmul2_rn(dz, wz)));
      const float2 nb = __fmul2_rn(__fmul2_rn(m3, rr), dw);  // -b
      const float2 tx = __ffma2_rn(nb, dx, wx);
      const float2 ty = __ffma2_rn(nb, dy, wy);
      const float2 tz = __ffma2_rn(nb, dz, wz);
      float2 qi, qj;
      if constexpr (MODE == kSymUniform) {
        qi = qj = __fmul2_rn(r, rr);
      } else if constexpr (MODE == kSymGeneral) {
        const float2 r3 = __fmul2_rn(r, rr);
        qi = __fmul2_rn(jm, r3);
        if constexpr (BOTH) qj = __fmul2_rn(nm[p], r3);
      } else {
        qi = __fmul2_rn(__fmul2_rn(jm, r), rr);
        if constexpr (BOTH) qj = __fmul2_rn(__fmul2_rn(nm[p], r), rr);
      }
      acc[p][0] = __ffma2_rn(qi, dx, acc[p][0]);
      acc[p][1] = __ffma2_rn(qi, dy, acc[p][1]);
      acc[p][2] = __ffma2_rn(qi, dz, acc[p][2]);
      acc[p][3] = __ffma2_rn(qi, tx, acc[p][3]);
      acc[p][4] = __ffma2_rn(qi, ty, acc[p][4]);
      acc[p][5] = __ffma2_rn(qi, tz, acc[p][5]);
      if constexpr (BOTH) {
        c[0] = __ffma2_rn(qj, dx, c[0]);
        c[1] = __ffma2_rn(qj, dy, c[1]);
        c[2] = __ffma2_rn(qj, dz, c[2]);
        c[3] = __ffma2_rn(qj, tx, c[3]);
        c[4] = __ffma2_rn(qj, ty, c[4]);
        c[5] = __ffma2_rn(qj, tz, c[5]);
      }
      if constexpr (POT) {
        const float2 rp = make_float2(d2.x != 0.f ? r.x : 0.f, d2.y != 0.f ? r.y : 0.f);
        if constexpr (MODE == kSymUniform) {
          acc[p][6] = __fadd2_rn(acc[p][6], rp);
          if constexpr (BOTH) c[6] = __fadd2_rn(c[6], rp);
        } else {
          acc[p][6] = __ffma2_rn(jm, rp, acc[p][6]);
          if constexpr (BOTH) c[6] = __ffma2_rn(nm[p], rp, c[6]);
        }
      }
    }
  }
  template <int MODE>
  __device__ __forceinline__ void pair(const float4* ring, uint32_t off, int chunk, float2 e2, const float2 (&nm)[P],
                                       float2 (&c)[kSumsJ]) {
    const float4* rec = reinterpret_cast<const float4*>(reinterpret_cast<const char*>(ring) + off);
    term<MODE, true>(rec[0], rec[chunk], e2, nm, c);
  }
  template <int MODE>
  __device__ __forceinline__ void one(const float4* js, int chunk, float2 e2, int /*self*/, int /*nt*/) {
    float2 none[kSumsJ], own[P];
    term<MODE, false>(js[0], js[chunk], e2, own, none);
  }
  __device__ static __forceinline__ float weight(int c, float mass) { return c == 6 ? -mass : mass; }
  __device__ static __forceinline__ float back(int /*c*/, int mode, float own) {
    return mode == kSymUniform ? -own : 1.f;
  }
  __device__ static __forceinline__ void output(const SymMerge& m, int64_t p, int c, float v) {
    if (c < 3)
      m.out[0][3 * p + c] = v;
    else if (c < 6)
      m.out[1][3 * p + c - 3] = v;
    else
      m.out[2][p] = v;
  }
};

template <bool POT>
using JerkTable = SymTable<SymJerkPolicy<2, POT>, SymJerkPolicy<4, POT>, SymJerkPolicy<8, POT>, SymJerkPolicy<2, POT>>;

}  // namespace

SymOps sym_jerk_ops(bool pot) { return pot ? JerkTable<true>::ops(8) : JerkTable<false>::ops(8); }

}  // namespace cn
