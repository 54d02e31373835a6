// One-sided kernel for an i set against another j set: every CTA holds a tile
// of i-particles in registers (K per thread, in packed f32x2 pairs) and
// streams its part of the tile's j records.
//
// What bounds it: the FP32 pipe and the register file, as in the symmetric
// kernel (the accumulating multiply-adds read three registers); 12 lane
// operations per pair, 11 where a warp's records of a stage all have one mass,
// which is then factored out of the pair terms. Two CTAs of 256 threads fit
// an SM (<= 128 registers; the running sums live in shared memory).
//
// Against the pair kernel it spreads the i-particles of small sets over the
// lanes (32 K per warp) and their j records over the warps, kRowUnit at a time,
// so that a record is read once per warp by all lanes alike and serves K x
// 32 pairs (the pair kernel's lane groups read as many records as they
// share a warp), cuts the work at any block instead of at whole j-tiles, and
// merges split rows with as many threads as they have sums (there the last
// CTA of a tile adds all its partials alone). With per-particle softening the
// s = 0 guard is taken only by warps that hold one outside kRowSoft .. kRowStiff. Measured
// (us, pair kernel / this one with equal / unequal masses): 1024 x 65536 47.0
// / 33.6 / 35.3, 4000 x 16384 39.6 / 31.8 / 33.6, 2048 x 262144 241 / 193 /
// 211; per-particle softening 16384 x 16384 135.8 / 104.6 / 113.4. Unequal
// masses in large sets of about equal sizes stay with the pair kernel
// (32768 x 32768 392 / 370 / 406).
//
// The rows' blocks lie on one line that is split evenly over the CTAs. A row
// that one CTA holds alone is written to the outputs; the sums of a split row
// go to one segment per (CTA, row), which a second kernel adds per particle
// in CTA order. Register sums are folded into (hi, lo) sums by TwoSum every
// kRowFold records: 128 cost 1% at 2048 x 262144 (208 / 211 us) and keep the
// error below the pair kernel's (8192 x 8192 1.0e-7 of 1.1e-7, 1.3e-7 with 512;
// 2048 x 262144 3.7e-8 of 5.1e-8). Where each warp has particles of its own
// (large sets with per-particle softening) it is every stage of 256: 0.71 of the
// pair kernel's error (24000 to 65536, geometric mean over 36 sets), and 128 cost 4%
// there (65536 x 65536 1499 / 1563 us). Deterministic, no atomics on data.
#pragma once

#include "cn_device.cuh"
#include "cn_rows.h"

namespace cn {

constexpr int kRowFold = 128;        // j records summed in FP32 registers between TwoSum folds; a warp's share of a stage, if more
constexpr int kRowUnit = 16;         // records per loop trip (divides 32)
constexpr int kRowWarps = 8;
constexpr int kRowThreads = 32 * kRowWarps;
constexpr float kRowFar = 1e11f;     // |coordinate| up to which r^-3 stays a normal number
constexpr float kRowSoft = 1e-20f;   // eps2 from which it stays finite
constexpr float kRowStiff = 1e24f;   // eps2 up to which it stays a normal number
constexpr float kRowHeavySoft = 1e12f;  // eps2 up to which the sums r^-3 d of masses above 1 are well above underflow

enum RowMode : int {
  kRowUniform = 0,  // equal masses, factored out
  kRowGeneral = 1,  // (m r)(r r); s > 0
  kRowGuarded = 2,  // the same, pairs with s = 0 give nothing
};

__device__ __forceinline__ float2 row_dup(float v) { return make_float2(v, v); }
__device__ __forceinline__ float& row_half(float2& v, int k) { return (k & 1) ? v.y : v.x; }

template <int K_, bool POT, bool EPSI>
struct RowForce {
  static constexpr int K = K_;
  static constexpr int P = K / 2;
  static constexpr int NS = POT ? 4 : 3;
  float2 nx[P][3], acc[P][NS];
  float2 ei[EPSI ? P : 1];

  template <int MODE>
  __device__ __forceinline__ void one(const float4 r0, float2 e2u) {
    const float2 jx = row_dup(r0.x), jy = row_dup(r0.y), jz = row_dup(r0.z), jm = row_dup(r0.w);
#pragma unroll
    for (int p = 0; p < P; ++p) {
      const float2 e2 = EPSI ? ei[EPSI ? p : 0] : e2u;
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
      if constexpr (MODE == kRowGuarded) {
        r.x = (s.x > 0.f) ? r.x : 0.f;
        r.y = (s.y > 0.f) ? r.y : 0.f;
      }
      const float2 rr = __fmul2_rn(r, r);
      const float2 mr = MODE == kRowUniform ? r : __fmul2_rn(jm, r);
      const float2 q = __fmul2_rn(mr, rr);
      acc[p][0] = __ffma2_rn(q, dx, acc[p][0]);
      acc[p][1] = __ffma2_rn(q, dy, acc[p][1]);
      acc[p][2] = __ffma2_rn(q, dz, acc[p][2]);
      if constexpr (POT)
        acc[p][3] = __fadd2_rn(acc[p][3], make_float2(d2.x != 0.f ? mr.x : 0.f, d2.y != 0.f ? mr.y : 0.f));
    }
  }
  // a stage's units first, first + step, ... < end
  template <int MODE>
  __device__ __forceinline__ void sweep(const float4* js, int first, int end, int step, float2 e2) {
#pragma unroll 1
    for (int u = first; u < end; u += step) {
#pragma unroll
      for (int j = 0; j < kRowUnit; ++j) one<MODE>(js[u * kRowUnit + j], e2);
    }
  }
};

struct RowChunk {
  int32_t row, blk, nb;  // nb = 0: no more
};
struct RowControl {
  uint64_t full[8];
  uint64_t empty[8];
  int32_t abort;
};

// where a CTA's walk stands: the row, its block, blocks left to the end of its part
struct RowCursor {
  int64_t left;
  int32_t row, blk;
  __device__ __forceinline__ RowChunk take(const RowArgs& a, int most) {
    RowChunk c{row, blk, 0};
    if (left <= 0) return c;
    int32_t n = a.blocks - blk;
    if (n > most) n = most;
    if (n > left) n = static_cast<int32_t>(left);
    c.nb = n;
    left -= n;
    blk += n;
    if (blk >= a.blocks) {
      ++row;
      blk = 0;
    }
    return c;
  }
};

template <int K, bool POT, bool EPSI>
__global__ void __launch_bounds__(kRowThreads, 2) rows_kernel(const __grid_constant__ RowArgs a) {
  extern __shared__ __align__(1024) unsigned char smem[];
  using Pol = RowForce<K, POT, EPSI>;
  constexpr int NS = Pol::NS, P = Pol::P;
  constexpr int kPer = 32 * K;             // particles per warp
  constexpr int kAll = kRowWarps * kPer;   // sums of all warps
  RowControl* const ctl = reinterpret_cast<RowControl*>(smem);
  float* const sums = reinterpret_cast<float*>(smem + 256);  // [2][NS][kAll]: (hi, lo) per warp
  float4* const ring = reinterpret_cast<float4*>(smem + 256 + static_cast<size_t>(2) * NS * kAll * sizeof(float));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wi = warp % a.wi, wj = warp / a.wi, nwj = kRowWarps / a.wi;
  const int CH = a.chunk, S = a.stages, most = CH / kRowBlock;
  volatile int32_t* abort = &ctl->abort;

  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&ctl->full[s], 1);
      mbar_init(&ctl->empty[s], kRowWarps);
    }
    ctl->abort = 0;
    mbar_init_fence();
  }
  __syncthreads();
  const int64_t u0 = a.part(blockIdx.x), u1 = a.part(static_cast<int64_t>(blockIdx.x) + 1);
  RowCursor cur;
  cur.left = u1 - u0;
  cur.row = static_cast<int32_t>(u0 / a.blocks);
  cur.blk = static_cast<int32_t>(u0 - static_cast<int64_t>(cur.row) * a.blocks);
  RowCursor ahead = cur;  // the producer's (thread 0)
  uint32_t issued = 0;
  // no call's data so far: that only after the previous kernel ends
  grid_dependency_wait();
  grid_launch_dependents();

  // stages the next chunk by one bulk copy (thread 0); a stage is refilled two
  // chunks after it was read, so that no warp is waited for
  auto produce = [&]() {
    if (ahead.left <= 0 || *abort) return;
    const uint32_t slot = issued % S;
    if (issued >= static_cast<uint32_t>(S) && !mbar_wait(&ctl->empty[slot], ((issued / S) - 1) & 1u, a.wait_ns)) {
      set_status(a.status, kStatusTimeoutEmpty);
      *abort = 1;
      return;
    }
    const RowChunk c = ahead.take(a, most);
    const int64_t first = static_cast<int64_t>(c.blk) * kRowBlock;
    const int64_t rest = a.n_j - first;
    const int want = c.nb * kRowBlock;
    const int cnt = static_cast<int>(rest < want ? rest : want);
#ifdef CN_DEBUG_BOUNDS
    if (c.row < 0 || c.row >= a.n_rows || cnt < 1 || first + cnt > a.n_j) {
      set_status(a.status, kStatusBadSchedule);
      *abort = 1;
      return;
    }
#endif
    float4* dst = ring + slot * static_cast<uint32_t>(CH);
    for (int z = cnt; z < want; ++z) dst[z] = make_float4(0.f, 0.f, 0.f, 0.f);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    mbar_arrive_expect_tx(&ctl->full[slot], static_cast<uint32_t>(cnt) * 16u);
    bulk_copy_g2s(dst, a.pos_j + first, static_cast<uint32_t>(cnt) * 16u, &ctl->full[slot]);
    ++issued;
  };
  if (tid == 0)
    for (int s = 0; s < S - 2; ++s) produce();

  Pol acc;
  int32_t row = -1;
  const float2 e2 = row_dup(a.eps2);
  float scale = 1.f;  // of the sums in registers
  int held = 0;       // j records in them
  float cap = -1.f;   // masses that may factor out with the warp's particles, up to (none: -1)
  float* const mine = sums + warp * kPer + lane;  // the thread's sums: mine[c * kAll + 32 k]

  auto fold = [&]() {
#pragma unroll
    for (int k = 0; k < K; ++k)
#pragma unroll
      for (int c = 0; c < NS; ++c) {
        float* h = mine + c * kAll + 32 * k;
        float* l = h + NS * kAll;
        float s, e;
        two_sum(*h, __fmul_rn(c == 3 ? -scale : scale, row_half(acc.acc[k >> 1][c], k)), s, e);
        *h = s;
        *l = __fadd_rn(*l, e);
      }
#pragma unroll
    for (int p = 0; p < P; ++p)
#pragma unroll
      for (int c = 0; c < NS; ++c) acc.acc[p][c] = row_dup(0.f);
    held = 0;
  };
  // the end of this CTA's blocks of a row: adds the sums of the warps that
  // share particles, in order, and writes the outputs or the segment
  auto flush = [&]() {
    fold();
    __syncthreads();
    const int64_t i0 = static_cast<int64_t>(row) * a.tile, left = a.n_i - i0;
    const int ni = static_cast<int>(left < a.tile ? left : a.tile);
    const int64_t first = static_cast<int64_t>(row) * a.blocks;
    const bool whole = first >= u0 && first + a.blocks <= u1;
    // the segment: the CTA's first if the row began before its part, else its last
    float* seg = a.segs + static_cast<size_t>(2 * blockIdx.x + (first >= u0 ? 1 : 0)) * NS * a.tile;
    for (int e = tid; e < NS * a.tile; e += kRowThreads) {
      const int c = e / a.tile, p = e - c * a.tile;
      const float* h = sums + c * kAll + p;
      float s = h[0], l = h[NS * kAll];
      for (int w = 1; w < nwj; ++w) {
        float t;
        two_sum(s, h[w * a.tile], s, t);
        l = __fadd_rn(l, __fadd_rn(t, h[NS * kAll + w * a.tile]));
      }
      const float v = pair_total(s, l);
      if (!whole)
        seg[e] = v;
      else if (p < ni) {
        if (c < 3)
          a.acc_out[3 * (i0 + p) + c] = v;
        else
          a.pot_out[i0 + p] = v;
      }
    }
    __syncthreads();
  };

  uint32_t q = 0;
  for (; cur.left > 0; ++q) {
    if (tid == 0) produce();
    const RowChunk ch = cur.take(a, most);
    if (ch.row != row) {
      if (row >= 0) flush();
      row = ch.row;
      const int64_t i0 = static_cast<int64_t>(row) * a.tile;
      bool near = EPSI || (a.eps2 >= kRowSoft && a.eps2 <= kRowStiff), heavy = EPSI || a.eps2 <= kRowHeavySoft;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int64_t p = i0 + wi * kPer + 32 * k + lane;
        float4 v = make_float4(0.f, 0.f, 0.f, 1.f);
        if (p < a.n_i) v = __ldg(a.pos_i + p);
        row_half(acc.nx[k >> 1][0], k) = -v.x;
        row_half(acc.nx[k >> 1][1], k) = -v.y;
        row_half(acc.nx[k >> 1][2], k) = -v.z;
        if constexpr (EPSI) {
          row_half(acc.ei[k >> 1], k) = v.w;
          near = near && v.w >= kRowSoft && v.w <= kRowStiff;
          heavy = heavy && v.w <= kRowHeavySoft;
        }
        near = near && fmaxf(fabsf(v.x), fmaxf(fabsf(v.y), fabsf(v.z))) <= kRowFar;
      }
      heavy = __all_sync(0xffffffffu, heavy);
      cap = __all_sync(0xffffffffu, near) ? (heavy ? 3.4e38f : 1.f) : -1.f;
#pragma unroll
      for (int p = 0; p < P; ++p)
#pragma unroll
        for (int c = 0; c < NS; ++c) acc.acc[p][c] = row_dup(0.f);
#pragma unroll
      for (int k = 0; k < K; ++k)
#pragma unroll
        for (int c = 0; c < 2 * NS; ++c) mine[c * kAll + 32 * k] = 0.f;
      held = 0;
      scale = 1.f;
    }
    const uint32_t slot = q % S;
    bool live = !*abort;
    if (live && !mbar_wait(&ctl->full[slot], (q / S) & 1u, a.wait_ns)) {
      set_status(a.status, kStatusTimeoutFull);
      *abort = 1;
      live = false;
    }
    live = __all_sync(0xffffffffu, live);
    const int units = ch.nb * (kRowBlock / kRowUnit);
    if (live && wj < units) {
      // this warp's records of the stage: the units wj, wj + nwj, ...
      const float4* js = ring + slot * static_cast<uint32_t>(CH);
      const int count = ((units - wj + nwj - 1) / nwj) * kRowUnit;
      bool same = true, near = cap >= 0.f;
      const float mj = js[wj * kRowUnit].w;
      for (int t = lane; t < count; t += 32) {
        const float4 v = js[(wj + t / kRowUnit * nwj) * kRowUnit + t % kRowUnit];
        same = same && v.w == mj;
        near = near && fmaxf(fabsf(v.x), fmaxf(fabsf(v.y), fabsf(v.z))) <= kRowFar;
      }
      near = __all_sync(0xffffffffu, near);
      same = __all_sync(0xffffffffu, same && near && fabsf(mj) <= cap);
      const float factor = same ? mj : 1.f;
      if (held > 0 && (factor != scale || held + count > kRowFold)) fold();
      scale = factor;
      held += count;
      if (same)
        acc.template sweep<kRowUniform>(js, wj, units, nwj, e2);
      else if (near || !EPSI)
        acc.template sweep<kRowGeneral>(js, wj, units, nwj, e2);
      else
        acc.template sweep<kRowGuarded>(js, wj, units, nwj, e2);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&ctl->empty[slot]);
  }
  if (row >= 0) flush();
  // an aborted run: wait (bounded) for copies that may still be in flight
  if (tid == 0 && *abort) {
    for (uint32_t c = issued > static_cast<uint32_t>(S) ? issued - S : 0u; c < issued; ++c) {
      if (!mbar_wait(&ctl->full[c % S], (c / S) & 1u, a.wait_ns)) {
        set_status(a.status, kStatusTimeoutDrain);
        break;
      }
    }
  }
}

// Adds the segments of split rows, in CTA order, four loads in flight. Block x
// stands for the start of part x + 1: it takes the row that this cuts, if it
// is the first such cut of the row.
template <int NS>
__global__ void __launch_bounds__(256) rows_merge_kernel(const __grid_constant__ RowArgs a) {
  grid_dependency_wait();
  grid_launch_dependents();
  const int64_t g0 = blockIdx.x;
  const int64_t cut = a.part(g0 + 1);
  const int64_t row = cut / a.blocks, first = row * a.blocks;
  if (cut >= a.units || first == cut || a.owner(first) != g0) return;
  const int n = static_cast<int>(a.owner(first + a.blocks - 1) - g0 + 1);
  const int64_t i0 = row * a.tile;
  const int e = blockIdx.y * 256 + threadIdx.x;
  if (e >= NS * a.tile) return;
  const int c = e / a.tile, p = e - c * a.tile;
  if (i0 + p >= a.n_i) return;
  const size_t seg = static_cast<size_t>(NS) * a.tile;
  const float* src = a.segs + e;
  float h = 0.f, l = 0.f;
  for (int q = 0; q < n; q += 4) {
    float v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (q + u < n) v[u] = __ldcs(src + static_cast<size_t>(2 * (g0 + q + u) + (q + u == 0 ? 1 : 0)) * seg);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (q + u < n) {
        float t;
        two_sum(h, v[u], h, t);
        l = __fadd_rn(l, t);
      }
  }
  const float v = pair_total(h, l);
  if (c < 3)
    a.acc_out[3 * (i0 + p) + c] = v;
  else
    a.pot_out[i0 + p] = v;
}

// ------------------------------------------------------------------ host side
template <bool POT, bool EPSI>
const void* rows_fn(int k) {
  if (k >= 8) return reinterpret_cast<const void*>(&rows_kernel<8, POT, EPSI>);
  return reinterpret_cast<const void*>(&rows_kernel<4, POT, EPSI>);
}

}  // namespace cn
