// Symmetric (Newton's third law) evaluation for an i set equal to the j set:
// every unordered pair is evaluated once and its term is added to both
// particles. The paper's kernel evaluates every ordered pair; this form does
// about half the pair work.
//
// A warp holds 32 x K particles of its CTA's tile (threads x K particles, K
// per thread in packed f32x2 pairs) and sweeps the other particles in blocks
// of 32: at step t lane l takes record l ^ t of the block from shared memory,
// so at every step the lanes hold 32 different j records, and the j-side
// sums travel with their record, exchanged by one shuffle per step (lane
// l's sums at step t belong to record l ^ t; the exchange between steps t
// and t + 1 is the xor with t ^ (t + 1)). After 32 steps lane l holds the
// sums of record l over the warp's particles. No reduction over lanes is
// needed: against summing each record over the warp by a reduce-scatter
// this takes 24 shuffles and 24 additions per 8 records to 48 shuffles and
// none, which leaves the FP32 pipe to the pair terms (inner loop at K = 8 x
// 256 threads, 2.07 GHz: 1.93e12 -> 2.03e12 unordered pairs/s; whole calls at
// N = 131072 with equal masses: 4653 -> 3985 us).
//
// What bounds the loop: the FP32 pipe, and with it the register file. A
// packed multiply-add whose three operands are different registers issues
// every third cycle, against every second one when an operand is repeated
// from the instruction before it (measured: 3.17 and 2.17 cycles), and
// 6 of the 14-16 packed operations of a pair term are of that kind; two CTAs
// of 256 threads per SM (<= 128 registers) run 4% faster than one.
//
// Masses. Where the masses of a staged chunk are all equal, they leave the
// pair term: the sums are formed of r^-3 d and scaled when they are folded
// (14 instead of 16 lane operations per unordered pair: 2.20e12 pairs/s).
// That is decided per chunk and warp from the records themselves (the
// warp's own masses equal too). It needs r^-3 within the FP32 range, as
// does the general term's r^-3 m: beyond coordinates of 1e11 and outside
// softenings of 1e-10 .. 1e12 the term is formed as (m r)(r r), the order of the
// one-sided kernel. The unscaled sums r^-3 d must stay in that range too. They
// cannot overflow there (at most eps^-2 a term); a mass above 1 that would have
// kept a product from underflowing stays in its term unless the softening is
// below 1e6 (kHeavySoft). Sums r^-3 w of a velocity or weight underflow and
// overflow with w: see kHeavyReach and SymArgs::fast.
//
// Shared memory per CTA: a ring of staged chunks (bulk copies), three buffers
// of the j-side sums of a chunk, one row per warp, and the i-side (hi, lo)
// sums of the current row of tiles, folded from registers every kFold
// records by TwoSum, mid-size sets sooner (force: 512 are 0.4% faster at N =
// 131072 and 0.8% at 50001, but leave a larger error than the reduce-scatter form
// did: with the potential 4.8e-8 against 4.1e-8 at 9836, 256 4.0e-8). The warps
// are not held together by a barrier: a warp that has swept chunk k waits for the "done" barrier of chunk k - 1 (long
// complete unless a warp is a whole chunk behind), adds up its share of
// chunk k - 1's rows and arrives on chunk k's barrier. A __syncthreads per
// chunk instead cost 1.4 us per chunk (N = 131072, 64-record chunks).
//
// j-side sums go to one slot per (row, block), i-side sums to one segment
// per (CTA, row), both as planes of one float per particle; a second kernel
// adds them per particle in a fixed order: the result is deterministic,
// with no atomics on data. A part of more than 1024 records is the sum of
// several register chains; in the force forms its segment then keeps the low
// words as well (all segments at all sizes: 4096 .. 24576 2 to 7% slower, for words
// that are zero while a segment is one chain).
#pragma once

#include "cn_device.cuh"
#include "cn_sym.h"

namespace cn {

constexpr float kSymFar = 1e11f;       // |coordinate| up to which r^-3 stays a normal number
constexpr float kSymSoft = 1e-20f;     // eps2 from which it stays finite
constexpr float kSymStiff = 1e24f;     // eps2 up to which it stays a normal number
constexpr float kSymHuge = 3.402823466e38f;  // finite

enum SymMode : int {
  kSymUniform = 0,  // equal masses, factored out of the pair terms
  kSymGeneral = 1,  // r^-3 times either mass
  kSymWide = 2,     // (m r)(r r): any range
};

// of a warp's own particles
enum SymOwn : int {
  kOwnEqual = 1,  // equal masses
  kOwnNear = 2,   // r^-3 in range
  kOwnClose = 4,  // within kHeavyReach and kHeavySoft
  kOwnSlow = 8,   // second records within SymArgs::fast
};

__device__ __forceinline__ float sym_reach(const float4& v) {
  return fmaxf(fabsf(v.x), fmaxf(fabsf(v.y), fabsf(v.z)));
}
__device__ __forceinline__ float2 sym_dup(float v) { return make_float2(v, v); }
__device__ __forceinline__ float& sym_half(float2& v, int k) { return (k & 1) ? v.y : v.x; }

// ------------------------------------------------------------------ policies
// A policy holds K i-particles and their FP32 sums (`acc`), and adds one j
// record's terms to both sides (`pair`) or to the i side alone (`one`):
//   kSumsI, kSumsJ  sums per particle and side
//   kRec            float4 words per record (2: a velocity or a loss weight)
//   kMinBlocks      256-thread CTAs per SM the registers are limited for
//   kUnroll         steps per loop trip (divides 32)
//   kFold           j records summed in FP32 registers between TwoSum folds, at
//                   most (SymArgs::fold, where a stage is one sweep)
//   kStage          records per stage, at most
//   kWide           offers the kSymWide terms
//   kLow            long segments keep their low words (single systems)
//   kRolled         the loop that writes a segment is not unrolled over its
//                   sums: which is the faster one is up to the registers that
//                   the compiler then finds for the sweeps (2%, measured)
//   kSameMass       equal masses factor out only if the warp's and the
//                   chunk's are the same
//   kHeavyReach     |coordinate| (with a second record) and eps2 up to which
//   kHeavySoft      masses above 1 factor out: unscaled sums there are well
//                   above underflow
//   kOwnSign        sign of the warp's own masses handed to `pair`
//   weight          factor of i-side sum c when it is folded (mass: the
//                   chunk's mass where the masses are factored out, else 1)
//   back            factor of j-side sum c at the end of a block (own: the
//                   particle's own mass there, else 1)
//   output          where the merged sum c of a particle goes
//
// Force (and potential): per pair, d = x_j - x_i, s = |d|^2 + eps2, r =
// s^-1/2; i: m_j r^3 d (and m_j r), j: -m_i r^3 d (and -m_i r). The
// potential skips pairs at exactly zero separation.
template <int K_, bool POT, bool GUARD, int UNROLL, int FOLD = 256>
struct SymForcePolicy {
  static constexpr int K = K_;
  static constexpr int P = K / 2;
  static constexpr int kSumsI = POT ? 4 : 3;
  static constexpr int kSumsJ = POT ? 4 : 3;
  static constexpr int kRec = 1;
  static constexpr bool kGuard = GUARD;
  static constexpr int kUnroll = UNROLL;
  static constexpr int kFold = FOLD;
  static constexpr int kStage = FOLD < 256 ? FOLD : 256;
  static constexpr int kMinBlocks = 2;
  static constexpr bool kWide = true;
  static constexpr bool kLow = true;
  static constexpr bool kRolled = (POT && K >= 4) || FOLD < 256;
  static constexpr bool kSameMass = false;
  // r^-3 d is at least 1e-23 where d is the longer one, r^-3 at least 1e-18 where eps is
  static constexpr float kHeavySoft = 1e12f;
  static constexpr float kOwnSign = -1.f;
  float2 nx[P][3], acc[P][kSumsI];

  __device__ __forceinline__ void load(const SymArgs& a, int64_t p, bool valid, int k, float& mass, float& reach,
                                       float& /*speed*/) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (valid) v = __ldg(a.pos + p);
    sym_half(nx[k >> 1][0], k) = -v.x;
    sym_half(nx[k >> 1][1], k) = -v.y;
    sym_half(nx[k >> 1][2], k) = -v.z;
    mass = v.w;
    reach = sym_reach(v);
  }

  template <int MODE, bool BOTH>
  __device__ __forceinline__ void term(const float4 r0, float2 e2, const float2 (&nm)[P], float2 (&c)[kSumsJ]) {
    const float2 jx = sym_dup(r0.x), jy = sym_dup(r0.y), jz = sym_dup(r0.z), jm = sym_dup(r0.w);
#pragma unroll
    for (int p = 0; p < P; ++p) {
      const float2 dx = __fadd2_rn(jx, nx[p][0]);
      const float2 dy = __fadd2_rn(jy, nx[p][1]);
      const float2 dz = __fadd2_rn(jz, nx[p][2]);
      float2 s, d2;
      if constexpr (POT) {
        d2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __fmul2_rn(dz, dz)));
        s = __fadd2_rn(d2, e2);
      } else {
        s = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, e2)));
      }
      float2 r = make_float2(rsqrt_mufu(s.x), rsqrt_mufu(s.y));
      if constexpr (GUARD) {
        r.x = (s.x > 0.f) ? r.x : 0.f;
        r.y = (s.y > 0.f) ? r.y : 0.f;
      }
      const float2 rr = __fmul2_rn(r, r);
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
      if constexpr (BOTH) {
        c[0] = __ffma2_rn(qj, dx, c[0]);
        c[1] = __ffma2_rn(qj, dy, c[1]);
        c[2] = __ffma2_rn(qj, dz, c[2]);
      }
      if constexpr (POT) {
        const float2 rp = make_float2(d2.x != 0.f ? r.x : 0.f, d2.y != 0.f ? r.y : 0.f);
        if constexpr (MODE == kSymUniform) {
          acc[p][3] = __fadd2_rn(acc[p][3], rp);
          if constexpr (BOTH) c[3] = __fadd2_rn(c[3], rp);
        } else {
          acc[p][3] = __ffma2_rn(jm, rp, acc[p][3]);
          if constexpr (BOTH) c[3] = __ffma2_rn(nm[p], rp, c[3]);
        }
      }
    }
  }
  template <int MODE>
  __device__ __forceinline__ void pair(const float4* ring, uint32_t off, int /*chunk*/, float2 e2,
                                       const float2 (&nm)[P], float2 (&c)[kSumsJ]) {
    term<MODE, true>(*reinterpret_cast<const float4*>(reinterpret_cast<const char*>(ring) + off), e2, nm, c);
  }
  template <int MODE>
  __device__ __forceinline__ void one(const float4* js, int /*chunk*/, float2 e2, int /*self*/, int /*nt*/) {
    float2 none[kSumsJ], own[P];
    term<MODE, false>(js[0], e2, own, none);
  }
  __device__ static __forceinline__ float weight(int c, float mass) { return c == 3 ? -mass : mass; }  // phi = -sum m r
  __device__ static __forceinline__ float back(int /*c*/, int mode, float own) {
    return mode == kSymUniform ? -own : 1.f;
  }

  __device__ static __forceinline__ void output(const SymMerge& m, int64_t p, int c, float v) {
    if (c < 3)
      m.out[0][3 * p + c] = v;
    else if (m.out[1])  // a plan with the potential may be run without it
      m.out[1][p] = v;
  }
};

// ------------------------------------------------------------------ sweeps
// The off-diagonal blocks of a chunk against the warp's particles, both
// sides. `off`: byte offset of the chunk in the ring (a multiple of 512), so
// that record l ^ t of a block is at its offset ^ (l ^ t) * 16. The j-side
// sums of each block go to this warp's row; `mass`: the
// thread's own masses in shared memory (mass[k * nt]).
template <class Pol, int MODE>
__device__ __forceinline__ void sym_sweep(Pol& acc, const float4* ring, uint32_t off, int chunk, int blocks, int lane,
                                          float2 e2, const float* mass, int nt, float* row) {
  float2 nm[Pol::P];
#pragma unroll
  for (int k = 0; k < Pol::K; ++k) sym_half(nm[k >> 1], k) = MODE == kSymUniform ? 0.f : Pol::kOwnSign * mass[k * nt];
  const float own = MODE == kSymUniform ? mass[0] : 1.f;
#pragma unroll 1
  for (; blocks > 0; --blocks) {
    float2 c[Pol::kSumsJ];
#pragma unroll
    for (int d = 0; d < Pol::kSumsJ; ++d) c[d] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int u = 0; u < kSymBlock; u += Pol::kUnroll) {
      const uint32_t o = off + (static_cast<uint32_t>(lane ^ u) << 4);
      const int next = ((Pol::kUnroll - 1) ^ u ^ (u + Pol::kUnroll)) & 31;  // exchange into the next trip
#pragma unroll
      for (int s = 0; s < Pol::kUnroll; ++s) {
        acc.template pair<MODE>(ring, o ^ static_cast<uint32_t>(s << 4), chunk, e2, nm, c);
        const int m = s + 1 < Pol::kUnroll ? s ^ (s + 1) : next;
#pragma unroll
        for (int d = 0; d < Pol::kSumsJ; ++d) {
          c[d].x = __shfl_xor_sync(0xffffffffu, c[d].x, m);
          c[d].y = __shfl_xor_sync(0xffffffffu, c[d].y, m);
        }
      }
    }
#pragma unroll
    for (int d = 0; d < Pol::kSumsJ; ++d) row[d * chunk + lane] = Pol::back(d, MODE, own) * (c[d].x + c[d].y);
    off += kSymBlock * 16;
    row += kSymBlock;
  }
}

// Diagonal blocks: every ordered pair, i side only (self: the thread's first
// particle's index relative to js[0]; its others follow nt apart).
template <class Pol, int MODE>
__device__ __forceinline__ void sym_diag(Pol& acc, const float4* js, int chunk, int count, float2 e2, int self, int nt) {
#pragma unroll 1
  for (int j = 0; j < count; j += 8) {
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) acc.template one<MODE>(js + j + jj, chunk, e2, self - (j + jj), nt);
  }
}

// ------------------------------------------------------------------ kernel
// Shared-memory control block. What only thread 0 or the start of a chunk
// needs lives here, not in registers: the sweeps need all 128.
struct SymChunk {
  int32_t row, blk, nb, diag;  // nb = 0: no more chunks
};
struct SymSlot {               // ensembles: a chunk's j-side slots, and their plane
  int64_t at;
  int64_t plane;
};
struct SymControl {
  uint64_t full[8];
  uint64_t done[3];  // a chunk swept by every warp (and the chunk before it added up)
  int32_t abort;
  uint32_t issued;   // chunks staged (thread 0)
  int32_t own[8];    // with a second record: what holds for each warp's own particles (kOwn...)
  SymCursor ahead;   // the next one (thread 0)
  int64_t end;
  SymChunk chunk[16];
  SymSlot slot[16];
};
static_assert(sizeof(SymControl) <= 1024, "control block");

// Stages the next chunk of this CTA (thread 0), or marks the end.
template <class Pol, bool BATCHED>
__device__ __noinline__ void sym_produce(const SymArgs& a, SymControl* ctl, float4* ring) {
  constexpr int JR = Pol::kRec;
  const uint32_t q = ctl->issued;
  SymChunk& ch = ctl->chunk[q & 15u];
  const int slot = static_cast<int>(q % static_cast<uint32_t>(a.stages));
  SymCursor cur = ctl->ahead;
  bool diag = false;
  ch.nb = 0;
  int64_t p0 = 0, n = a.g.n;
  if (cur.s < ctl->end) {
    if constexpr (BATCHED) {
      sym_take_rows(cur, a.rows, a.n_rows, ctl->end, a.chunk / kSymBlock, &ch.row, &ch.blk, &ch.nb, &diag);
      const SymRow r = a.rows[ch.row];
      p0 = r.p0;
      n = r.n;
      ctl->slot[q & 15u] = SymSlot{r.slot + static_cast<int64_t>(ch.blk - r.diag_end) * kSymBlock, r.plane};
    } else {
      cur.take(a.g, ctl->end, a.chunk / kSymBlock, &ch.row, &ch.blk, &ch.nb, &diag);
    }
  }
  ch.diag = diag;
#ifdef CN_DEBUG_BOUNDS
  bool bad = false;
  if (ch.nb != 0) {
    if constexpr (BATCHED)
      bad = ch.row < 0 || ch.row >= a.n_rows || ch.blk < a.rows[ch.row].blk0 ||
            ch.blk + ch.nb > a.rows[ch.row].n_blocks || p0 < 0 || p0 + n > a.g.n;
    else
      bad = ch.row < a.g.row0 || ch.row >= a.g.row1 || ch.blk < ch.row * a.g.tile_blocks ||
            ch.blk + ch.nb > a.g.n_blocks;
    bad = bad || ch.nb < 1 || ch.nb > a.chunk / kSymBlock ||
          static_cast<int64_t>(blockIdx.x) + (ch.row - a.g.row0) >= a.n_seg;
  }
  if (bad) {
    set_status(a.status, kStatusBadSchedule);
    ch.nb = 0;  // the CTA stops here
  }
#endif
  ctl->ahead = cur;
  ctl->issued = q + 1;
  if (ch.nb == 0) {
    ctl->ahead.s = ctl->end;
    mbar_arrive(&ctl->full[slot]);
    return;
  }
  const int64_t left = n - static_cast<int64_t>(ch.blk) * kSymBlock;
  const int64_t first = p0 + static_cast<int64_t>(ch.blk) * kSymBlock;
  const int want = ch.nb * kSymBlock;
  const int cnt = static_cast<int>(left < want ? left : want);
  float4* dst = ring + static_cast<size_t>(slot) * JR * a.chunk;
  for (int z = cnt; z < want; ++z) {  // zero-mass padding of the last block
    dst[z] = make_float4(0.f, 0.f, 0.f, 0.f);
    if constexpr (JR == 2) dst[a.chunk + z] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  mbar_arrive_expect_tx(&ctl->full[slot], static_cast<uint32_t>(cnt) * 16u * JR);
  bulk_copy_g2s(dst, a.pos + first, static_cast<uint32_t>(cnt) * 16u, &ctl->full[slot]);
  if constexpr (JR == 2)
    bulk_copy_g2s(dst + a.chunk, a.rec2 + first, static_cast<uint32_t>(cnt) * 16u, &ctl->full[slot]);
}

template <class Pol, bool BATCHED>
__global__ void __launch_bounds__(256, Pol::kMinBlocks) sym_kernel(const __grid_constant__ SymArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  constexpr int K = Pol::K, P = Pol::P, NI = Pol::kSumsI, NJ = Pol::kSumsJ, JR = Pol::kRec;
  constexpr bool LOW = Pol::kLow && !BATCHED;
  constexpr int NS = LOW ? 2 * NI : NI;  // planes of a segment
  const int NT = blockDim.x;
  const int tid = threadIdx.x;
  const int lane = tid & 31;
  const int warp = tid >> 5;
  const int NW = NT >> 5;
  const int B = NT * K;
  const int CH = a.chunk;
  const uint32_t S = static_cast<uint32_t>(a.stages);
  SymControl* ctl = reinterpret_cast<SymControl*>(smem);
  volatile int32_t* abort = &ctl->abort;
  float4* ring = reinterpret_cast<float4*>(smem + 1024);                             // [S][JR][CH]
  float* rows = reinterpret_cast<float*>(ring + static_cast<size_t>(S) * JR * CH);   // [3][NW][NJ][CH]
  float* sums = rows + static_cast<size_t>(3) * NW * NJ * CH;  // [2][NI][B]: (hi, lo) of the row's i side
  float* mass = sums + static_cast<size_t>(2) * NI * B;        // [B]: the tile's masses

  if (tid == 0) {
    for (uint32_t s = 0; s < S; ++s) mbar_init(&ctl->full[s], 1);
    for (int s = 0; s < 3; ++s) mbar_init(&ctl->done[s], NW);
    ctl->abort = 0;
    ctl->issued = 0;
    mbar_init_fence();
    ctl->end = a.g.part(static_cast<int64_t>(blockIdx.x) + 1);
    if constexpr (BATCHED)  // the plan's table: written when the plan was made
      sym_seek_rows(ctl->ahead, a.rows, a.n_rows, a.g.part(blockIdx.x));
    else
      ctl->ahead.seek(a.g, a.g.part(blockIdx.x));
  }
  __syncthreads();
  // no call's data so far: that only after the previous kernel ends
  grid_dependency_wait();
  if (tid == 0)
    for (uint32_t s = 0; s < S; ++s) sym_produce<Pol, BATCHED>(a, ctl, ring);

  Pol acc;
  float2 e2 = sym_dup(a.eps2);
  int32_t cur_I = -1;
  float scale = 1.f;   // of the sums in registers
  int held = 0;        // j blocks in them

  // the warp's own particles: equal masses that may factor out; r^-3 in range
  bool own_uniform = false, own_near = false;
  // the largest mass that may factor out, by the softening alone
  auto heaviest = [&]() { return e2.x <= Pol::kHeavySoft ? kSymHuge : 1.f; };

  // adds the register sums to the row's (hi, lo) sums (each thread its own
  // particles') and clears them
  auto fold = [&]() {
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int c = 0; c < NI; ++c) {
        float* h = sums + c * B + k * NT + tid;
        float* l = h + NI * B;
        float s, e;
        two_sum(*h, __fmul_rn(Pol::weight(c, scale), sym_half(acc.acc[k >> 1][c], k)), s, e);
        *h = s;
        *l = __fadd_rn(*l, e);
      }
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int c = 0; c < NI; ++c) acc.acc[p][c] = make_float2(0.f, 0.f);
    held = 0;
  };
  // writes the row's i-side sums to this CTA's segment: their totals and, where
  // asked for, what those lack
  auto flush = [&](int32_t I) {
    fold();
    const bool both = LOW && a.both_words;
    float* seg = a.slots_seg + (static_cast<size_t>(blockIdx.x) + static_cast<size_t>(I - a.g.row0)) * NS * B;
#pragma unroll(Pol::kRolled ? 1 : NI)
    for (int c = 0; c < NI; ++c)
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int e = c * B + k * NT + tid;
        seg[e] = pair_total(sums[e], sums[e + NI * B]);
      }
    if (both) {
#pragma unroll 1
      for (int e = tid; e < NI * B; e += NT) {
        const float h = sums[e], l = sums[e + NI * B];
        seg[e + NI * B] = __fadd_rn(__fadd_rn(h, -pair_total(h, l)), l);
      }
    }
  };
  // once every warp has swept chunk q: refills its stage (thread 0) and adds
  // up this warp's share of its j-side sums, over the warps in order
  auto settle = [&](uint32_t q) {
    const uint32_t b = q % 3;
    bool live = !*abort;
    if (live && !mbar_wait(&ctl->done[b], (q / 3) & 1u, a.wait_ns)) {
      set_status(a.status, kStatusTimeoutEmpty);
      *abort = 1;
      live = false;
    }
    live = __all_sync(0xffffffffu, live);
    if (!live) return;
    if (tid == 0) sym_produce<Pol, BATCHED>(a, ctl, ring);
    const SymChunk ch = ctl->chunk[q & 15u];
    if (ch.diag) return;
    const float* row = rows + b * (NW * NJ * CH);
    float* slot = a.slots_j;
    size_t plane = static_cast<size_t>(a.n_pad);
    if constexpr (BATCHED) {
      slot += ctl->slot[q & 15u].at;
      plane = static_cast<size_t>(ctl->slot[q & 15u].plane);
    } else {
      slot += static_cast<size_t>(ch.row - a.g.row0) * NJ * a.n_pad + static_cast<size_t>(ch.blk) * kSymBlock;
    }
    for (int it = warp; it < NJ * ch.nb; it += NW) {
      const int d = it % NJ, j = (it / NJ) * kSymBlock + lane;
      const float* r = row + d * CH + j;
      float v = r[0];
      for (int w = 1; w < NW; ++w) v += r[w * (NJ * CH)];
      slot[static_cast<size_t>(d) * plane + j] = v;
    }
  };

  uint32_t q = 0;
  for (;; ++q) {
    const uint32_t slot = q % S;
    // After a timed-out wait anywhere in the CTA (abort set) every warp
    // leaves: nothing below waits for another warp but with a bound.
    bool live = !*abort;
    if (live && !mbar_wait(&ctl->full[slot], (q / S) & 1u, a.wait_ns)) {
      set_status(a.status, kStatusTimeoutFull);
      *abort = 1;
      live = false;
    }
    live = __all_sync(0xffffffffu, live);
    if (!live) break;
    const SymChunk ch = ctl->chunk[q & 15u];
    if (ch.nb == 0) break;
    if (ch.row != cur_I) {
      if (cur_I >= 0) flush(cur_I);
      cur_I = ch.row;
      bool same = true, near = true, close = true, slow = true;
      float m0 = 0.f;
      int64_t p0 = static_cast<int64_t>(cur_I) * B, pn = a.g.n;
      if constexpr (BATCHED) {
        const SymRow r = a.rows[cur_I];
        p0 = r.p0 + static_cast<int64_t>(r.blk0) * kSymBlock;
        pn = r.p0 + r.n;
        e2 = sym_dup(r.eps2);
      }
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int64_t p = p0 + k * NT + tid;
        float m, reach, speed = 0.f;
        acc.load(a, p, p < pn, k, m, reach, speed);
        mass[k * NT + tid] = m;
        if (k == 0) m0 = __shfl_sync(0xffffffffu, m, 0);
        same = same && m == m0;
        near = near && reach <= kSymFar;
        if constexpr (JR == 2) {
          close = close && reach <= Pol::kHeavyReach;
          slow = slow && speed <= a.fast;
        }
      }
      own_uniform = __all_sync(0xffffffffu, same && fabsf(m0) <= (JR == 2 ? kSymHuge : heaviest()));
      own_near = __all_sync(0xffffffffu, near && e2.x >= kSymSoft && e2.x <= kSymStiff);
      if constexpr (JR == 2) {
        close = __all_sync(0xffffffffu, close && e2.x <= Pol::kHeavySoft);
        slow = __all_sync(0xffffffffu, slow);
        ctl->own[warp] = (own_uniform ? kOwnEqual : 0) | (own_near ? kOwnNear : 0) | (close ? kOwnClose : 0) | (slow ? kOwnSlow : 0);
      }
#pragma unroll
      for (int p = 0; p < P; ++p)
#pragma unroll
        for (int c = 0; c < NI; ++c) acc.acc[p][c] = make_float2(0.f, 0.f);
#pragma unroll
      for (int k = 0; k < K; ++k)
#pragma unroll
        for (int c = 0; c < 2 * NI; ++c) sums[c * B + k * NT + tid] = 0.f;
      held = 0;
      __syncwarp();
    }
    const uint32_t off = slot * static_cast<uint32_t>(JR * CH) * 16u;
    const float4* js = ring + slot * static_cast<uint32_t>(JR * CH);
    const int count = ch.nb * kSymBlock;
    int mode = Pol::kWide ? kSymWide : kSymGeneral;
    float factor = 1.f;
    if constexpr (!Pol::kGuard) {
      const float mj = js[0].w;
      bool own_close = true, own_slow = true;
      if constexpr (JR == 2) {
        const int own = ctl->own[warp];
        own_uniform = own & kOwnEqual;
        own_near = own & kOwnNear;
        own_close = own & kOwnClose;
        own_slow = own & kOwnSlow;
      }
      // with a second record the positions count too where either mass is above 1
      const bool heavy = JR == 2 && (fabsf(mj) > 1.f || (own_uniform && fabsf(mass[tid]) > 1.f));
      bool same = fabsf(mj) <= (JR == 2 ? kSymHuge : heaviest()), near = own_near;
      if constexpr (JR == 2) same = same && own_slow && (!heavy || own_close);
#pragma unroll(JR == 2 ? 1 : 4)
      for (int t = lane; t < count; t += 32) {
        const float4 v = js[t];
        const float reach = sym_reach(v);
        same = same && v.w == mj;
        near = near && reach <= kSymFar;
        if constexpr (JR == 2) same = same && (!heavy || reach <= Pol::kHeavyReach) && sym_reach(js[CH + t]) <= a.fast;
      }
      if (Pol::kSameMass)
        same = same && own_uniform && mass[tid] == mj;
      else
        same = same && (ch.diag || own_uniform);
      if (__all_sync(0xffffffffu, near)) {
        mode = kSymGeneral;
        if (__all_sync(0xffffffffu, same)) {
          mode = kSymUniform;
          factor = mj;
        }
      }
    }
    constexpr int kStep = Pol::kFold / kSymBlock;  // blocks between folds, at most
    // the blocks b0 .. b0 + nb - 1 of the chunk
    auto sweep = [&](int b0, int nb) {
      if (held > 0 && (factor != scale || held + nb > (Pol::kFold >= Pol::kStage ? a.fold : kStep))) fold();
      scale = factor;
      held += nb;
      if (ch.diag) {
        const float4* js0 = js + b0 * kSymBlock;
        const int self = cur_I * B - (ch.blk + b0) * kSymBlock + tid;
        if constexpr (!Pol::kGuard) {
          if (mode == kSymUniform)
            sym_diag<Pol, kSymUniform>(acc, js0, CH, nb * kSymBlock, e2, self, NT);
          else if (mode == kSymGeneral)
            sym_diag<Pol, kSymGeneral>(acc, js0, CH, nb * kSymBlock, e2, self, NT);
        }
        if constexpr (Pol::kWide) {
          if (mode == kSymWide) sym_diag<Pol, kSymWide>(acc, js0, CH, nb * kSymBlock, e2, self, NT);
        }
      } else {
        float* mine = rows + (q % 3) * (NW * NJ * CH) + warp * (NJ * CH) + b0 * kSymBlock;
        const uint32_t off0 = off + static_cast<uint32_t>(b0) * (kSymBlock * 16);
        if constexpr (!Pol::kGuard) {
          if (mode == kSymUniform)
            sym_sweep<Pol, kSymUniform>(acc, ring, off0, CH, nb, lane, e2, mass + tid, NT, mine);
          else if (mode == kSymGeneral)
            sym_sweep<Pol, kSymGeneral>(acc, ring, off0, CH, nb, lane, e2, mass + tid, NT, mine);
        }
        if constexpr (Pol::kWide) {
          if (mode == kSymWide) sym_sweep<Pol, kSymWide>(acc, ring, off0, CH, nb, lane, e2, mass + tid, NT, mine);
        }
      }
    };
    if constexpr (Pol::kFold >= Pol::kStage) {
      sweep(0, ch.nb);
    } else {
      for (int b0 = 0; b0 < ch.nb; b0 += kStep) sweep(b0, ch.nb - b0 < kStep ? ch.nb - b0 : kStep);
    }
    if (q > 0) settle(q - 1);
    __syncwarp();
    if (lane == 0) mbar_arrive(&ctl->done[q % 3]);
  }
  // the merge kernel may be scheduled while this one ends (not earlier: its
  // waiting CTAs would take room beside this one's)
  grid_launch_dependents();
  if (q > 0) settle(q - 1);
  if (cur_I >= 0) flush(cur_I);
  // an aborted run: wait (bounded) for copies that may still be in flight
  __syncthreads();
  if (tid == 0 && *abort) {
    const uint32_t issued = ctl->issued;
    for (uint32_t c = issued > S ? issued - S : 0u; c < issued; ++c) {
      if (!mbar_wait(&ctl->full[c % S], (c / S) & 1u, a.wait_ns)) {
        set_status(a.status, kStatusTimeoutDrain);
        break;
      }
    }
  }
}

// Per-particle merge (see SymMerge): 32 particles per CTA, whose slots and
// segments are dealt out over the 8 warps, in flight together (the chain of
// loads of one thread per particle was the larger part of the time at
// N = 4096 .. 16384); the warps' sums are added in warp order. All sums
// are FP32 (hi, lo) pairs by TwoSum: six FP32 operations, where an FP64
// addition and its conversion take 32 times as long on this GPU.
// An ensemble's particles have few of either: 2 warps there.
template <bool BATCHED>
constexpr int kSymMergeWarps = BATCHED ? 2 : 8;
// LOW: the segments have low words.
template <class Pol, bool BATCHED, bool LOW>
__global__ void __launch_bounds__(32 * kSymMergeWarps<BATCHED>) sym_merge_kernel(const __grid_constant__ SymMerge m) {
  constexpr int NI = Pol::kSumsI, NW = kSymMergeWarps<BATCHED>;
  constexpr int NS = Pol::kLow && !BATCHED ? 2 * NI : NI;  // planes of a segment
  __shared__ float2 part[NW][NI][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t p, jrow = 0;  // the particle; the first row with a slot of it
  bool valid;
  int nj = 0, ns = 0;   // its slots and segments
  const float* seg = nullptr;
  const float* slot = nullptr;
  int32_t blk = static_cast<int32_t>(blockIdx.x);
  if constexpr (BATCHED) {
    const SymMergeBlock mb = m.blocks[blockIdx.x];
    const SymRow r = m.rows[mb.row];
    blk = mb.blk;
    const int32_t local = blk * kSymBlock + lane;
    p = r.p0 + local;
    valid = local < r.n;
    jrow = mb.first;
    nj = mb.row - mb.first;
    const int64_t c0 = m.g.owner(r.cost);
    ns = static_cast<int>(m.g.owner(r.last()) - c0 + 1);
    seg = m.slots_seg + static_cast<size_t>(c0 + mb.row) * NS * m.tile + (local - r.blk0 * kSymBlock);
  } else {
    p = static_cast<int64_t>(blk) * kSymBlock + lane;
    valid = p < m.g.n;
    const int32_t I = static_cast<int32_t>((static_cast<int64_t>(blk) * kSymBlock) / m.tile);  // 32 divides the tile
    const int32_t jend = I < m.g.row1 ? I : m.g.row1;
    nj = jend > m.g.row0 ? jend - m.g.row0 : 0;
    // i-side: the CTAs whose parts hold the units of row I (when it is one of the launch's rows)
    if (I >= m.g.row0 && I < m.g.row1) {
      const int64_t s0 = m.g.row_start(I), s1 = m.g.row_start(static_cast<int64_t>(I) + 1);
      const int64_t last = s1 - (m.g.diag_end(I) < m.g.n_blocks ? kSymCostPair : kSymCostDiag);
      const int64_t c0 = m.g.owner(s0), c1 = m.g.owner(last);
      ns = static_cast<int>(c1 - c0 + 1);
      seg = m.slots_seg + (static_cast<size_t>(c0) + static_cast<size_t>(I - m.g.row0)) * NS * m.tile +
            static_cast<size_t>(p - static_cast<int64_t>(I) * m.tile);
    }
    slot = m.slots_j + static_cast<size_t>(p);
  }
  const int total = nj + ns;
  grid_dependency_wait();  // the slots are complete once the symmetric kernel has ended
  grid_launch_dependents();
  float hi[NI], lo[NI];
#pragma unroll
  for (int c = 0; c < NI; ++c) hi[c] = lo[c] = 0.f;
  constexpr int kAhead = 4;
  for (int q = warp; q < total; q += kAhead * NW) {
    float w[kAhead][NI], v[LOW ? kAhead : 1][NI];  // high words; low words of segments
#pragma unroll
    for (int u = 0; u < kAhead; ++u) {
      const int e = q + u * NW;
      if (e < total && valid) {
        const float* src = seg + static_cast<int64_t>(e - nj) * NS * m.tile;
        int64_t plane = m.tile;
        if constexpr (LOW) {
#pragma unroll
          for (int c = 0; c < NI; ++c) v[u][c] = 0.f;
          if (e >= nj) {
#pragma unroll
            for (int c = 0; c < NI; ++c) v[u][c] = __ldcs(src + (NI + c) * plane);
          }
        }
        if (e < nj) {
          if constexpr (BATCHED) {
            const SymRow& r = m.rows[jrow + e];
            src = m.slots_j + r.slot + static_cast<int64_t>(blk - r.diag_end) * kSymBlock + lane;
            plane = r.plane;
          } else {
            src = slot + static_cast<size_t>(e) * NI * m.n_pad;
            plane = m.n_pad;
          }
        }
#pragma unroll
        for (int c = 0; c < NI; ++c) w[u][c] = __ldcs(src + c * plane);
      }
    }
#pragma unroll
    for (int u = 0; u < kAhead; ++u)
      if (q + u * NW < total && valid) {
#pragma unroll
        for (int c = 0; c < NI; ++c) {
          float e;
          two_sum(hi[c], w[u][c], hi[c], e);
          if constexpr (LOW) e = __fadd_rn(e, v[u][c]);
          lo[c] = __fadd_rn(lo[c], e);
        }
      }
  }
#pragma unroll
  for (int c = 0; c < NI; ++c) part[warp][c][lane] = make_float2(hi[c], lo[c]);
  __syncthreads();
  if (!valid) return;
  for (int c = warp; c < NI; c += NW) {
    float h = 0.f, l = 0.f;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      float e;
      two_sum(h, part[w][c][lane].x, h, e);
      l = __fadd_rn(l, __fadd_rn(e, part[w][c][lane].y));
    }
    if (m.first && m.last) {
      Pol::output(m, p, c, pair_total(h, l));
      continue;
    }
    // bands: few and long, so that their sums can be added in FP64
    double* carry = m.carry + static_cast<size_t>(c) * m.n_pad + p;
    double t = m.first ? 0.0 : *carry;
    t += static_cast<double>(h);
    if (fabsf(h) <= kSymHuge) t += static_cast<double>(l);
    if (m.last)
      Pol::output(m, p, c, static_cast<float>(t));
    else
      *carry = t;
  }
}

// ------------------------------------------------------------------ host side
// The launch functions of a form, over its policies with 2, 4 and 8 particles
// per thread and the guarded one (eps2 = 0).
template <class P2, class P4, class P8, class PG, bool BATCHED = false>
struct SymTable {
  template <class F>
  static auto pick(int k, bool guard, F&& f) {
    if (guard) return f(PG{});
    if (k >= 8) return f(P8{});
    if (k >= 4) return f(P4{});
    return f(P2{});
  }
  static size_t smem(int threads, int k, int chunk, int stages) {
    return pick(k, false, [&](auto pol) {
      using Pol = decltype(pol);
      return 1024 + static_cast<size_t>(stages) * Pol::kRec * chunk * 16 +
             (static_cast<size_t>(3) * (threads / 32) * Pol::kSumsJ * chunk +
              static_cast<size_t>(2 * Pol::kSumsI + 1) * threads * Pol::K) * sizeof(float);
    });
  }
  static cudaError_t occupancy(int k, bool guard, int threads, size_t bytes, int* ctas) {
    return pick(k, guard, [&](auto pol) {
      const void* f = reinterpret_cast<const void*>(&sym_kernel<decltype(pol), BATCHED>);
      const cudaError_t e = prepare_kernel(f, bytes);
      return e != cudaSuccess ? e : cudaOccupancyMaxActiveBlocksPerMultiprocessor(ctas, f, threads, bytes);
    });
  }
  static cudaError_t launch(const SymArgs& a, const SymMerge& m, int k, bool guard, int threads, size_t bytes,
                            cudaStream_t s) {
    return pick(k, guard, [&](auto pol) {
      const void* f = reinterpret_cast<const void*>(&sym_kernel<decltype(pol), BATCHED>);
      cudaError_t e = prepare_kernel(f, bytes);
      if (e != cudaSuccess) return e;
      void* args[] = {const_cast<SymArgs*>(&a)};
      e = launch_pdl(f, dim3(static_cast<unsigned>(a.g.grid)), dim3(threads), args, bytes, s);
      if (e != cudaSuccess) return e;
      void* margs[] = {const_cast<SymMerge*>(&m)};
      const void* merge = reinterpret_cast<const void*>(&sym_merge_kernel<decltype(pol), BATCHED, false>);
      if constexpr (P2::kLow && !BATCHED)
        if (a.both_words) merge = reinterpret_cast<const void*>(&sym_merge_kernel<decltype(pol), BATCHED, true>);
      return launch_pdl(merge, dim3(static_cast<unsigned>(m.n_merge)), dim3(32 * kSymMergeWarps<BATCHED>), margs, 0, s);
    });
  }
  static SymOps ops(int max_k) { return SymOps{P2::kSumsI, P2::kLow && !BATCHED ? 2 * P2::kSumsI : P2::kSumsI, max_k, P2::kStage, &smem, &occupancy, &launch}; }
};

}  // namespace cn
