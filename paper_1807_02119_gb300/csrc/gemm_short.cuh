// Split-precision GEMM steps with a short contraction (K <= 32) in one kernel, included by
// launch.cu after gemm_tc.cuh, whose digits, levels and sums it shares bit for bit (K is below
// one flush group, and a level's sum is exact in whatever order its products are taken).
//
// As two launches (k_digits, k_gemm_tc) such a step took about 23 us however small, and a wide
// one moved 2.5 times its operands through the digit workspace.  Here a CTA takes a block of 128
// rows and a run of its column tiles: it turns its rows of A into digits in shared memory once,
// then for each tile the columns of B, issues the tile's MMAs and stores C from tensor memory.
// A thread owns one (row, part) of A, so that its offsets, exponent and stores need no tables;
// K is laid out by octets of 8 complex k, one K = 16 MMA step [Re | Im] each, so that K = 5 costs
// one step instead of two.  Tiles are the N columns split evenly (25 columns: 13 + 12, not
// 24 + 1).  One accumulator set and at most 110 KB: two CTAs per multiprocessor, one storing
// while the other multiplies.  The epilogue's instructions bound it (about 80 per complex output).
#pragma once

namespace pk {
namespace tcs {

constexpr int kMaxK = kTcShortK;  // four octets: A's digits and a B tile's within half of shared memory
constexpr int kThreads = 256;    // thread (row, part): warps 0-3 real parts, warps 4-7 imaginary
constexpr int kAOct = tc::kMc * 32;   // one digit of an octet of A: 128 rows x 16 BF16

// Octets rounded up to the kernel's variants, and a step's column tiles: W columns each, nw real
// columns per MMA, a multiple of 16.
struct Geom {
  int octs, tiles_n, W, nw;
  long long row_blocks;
};
__host__ __device__ inline Geom geom(const Step& s) {
  Geom g;
  g.octs = s.K <= 8 ? 1 : s.K <= 16 ? 2 : 4;
  g.tiles_n = (int)((s.N + tc::kNc - 1) / tc::kNc);
  g.W = (int)((s.N + g.tiles_n - 1) / g.tiles_n);
  g.nw = 2 * ((g.W + 7) & ~7);
  g.row_blocks = s.Bsz * ((s.M + tc::kMc - 1) / tc::kMc);
  return g;
}
constexpr int smem_bytes(int S, int octs) { return S * octs * (kAOct + 2 * tc::kNc * 32); }

// Column runs per row block: the fewest rounds over the GPU's slots, a round being the conversion
// of A (about a third of a tile's time per octet) and the run's tiles.
inline int col_runs(const Geom& g, long long slots) {
  int best = 1;
  double best_cost = 0;
  for (int r = 1; r <= g.tiles_n && r <= 64; ++r) {
    const long long ctas = g.row_blocks * r;
    const double cost = (double)((ctas + slots - 1) / slots) * (0.3 * g.octs + (g.tiles_n + r - 1) / r);
    if (r == 1 || cost < best_cost) best = r, best_cost = cost;
  }
  return best;
}

// 8 consecutive k of one part: (hi, lo) pairs, zero past K.
__device__ __forceinline__ void load8(float2* v, const Cx<ff>* p, const long long* kt, int k0, int K, int part) {
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    v[u] = make_float2(0.f, 0.f);
    if (k0 + u < K) v[u] = *((const float2*)(p + kt[k0 + u]) + part);
  }
}
__device__ __forceinline__ float max8(const float2* v) {
  float m = 0.f;
#pragma unroll
  for (int u = 0; u < 8; ++u) m = fmaxf(m, fabsf(v[u].x));
  return m;
}
// Offset of (row, part) in one digit of an octet: 8-row groups of two core matrices.
__device__ __forceinline__ uint32_t off8(int row, int part) {
  return (uint32_t)((row >> 3) * 256 + part * 128 + (row & 7) * 16);
}
template <int S>
__device__ __forceinline__ void put8(const float2* v, int e, unsigned char* out, unsigned char* out2, bool neg2, int slice) {
  float f1, f2, xh[8], xl[8];
  tc::pow2_pair(7 - e, f1, f2);
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    xh[u] = v[u].x;
    xl[u] = v[u].y;
  }
  tc::digit_rows8<S>(xh, xl, f1, f2, out, out2, neg2, slice);
}

}  // namespace tcs

template <int S, int OCTS>
__global__ void __launch_bounds__(tcs::kThreads, 2) k_gemm_short(const Step s, Cx<ff>* arena, Meta* meta, int runs,
                                                                  unsigned long long* err) {
  using namespace tcs;
  using tc::kMc;
  using tc::smem_u32;
  constexpr uint32_t kCols = tc::Cfg<S>::kCols;
  constexpr int kBLanes = 2 * OCTS;   // threads per column of B: (part, octet)
  static_assert(tc::kNc * kBLanes <= kThreads && 32 % kBLanes == 0, "columns of B per pass");
  extern __shared__ __align__(16) unsigned char dsm[];   // A: [octet][digit], then B: [octet][digit]
  __shared__ long long ka[kMaxK], kb[kMaxK], cn[tc::kNc];
  __shared__ int ea_s[kMc], eb_s[tc::kNc];
  __shared__ unsigned mx[kMc];
  __shared__ __align__(8) unsigned long long done, drain;
  __shared__ uint32_t tmem_slot;
  __shared__ int bad;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, K = (int)s.K;
  const Geom G = geom(s);
  const long long rb = blockIdx.x / runs;
  const int run = (int)(blockIdx.x - rb * runs);
  const long long tiles_m = (s.M + kMc - 1) / kMc, bb = rb / tiles_m, tm = rb - bb * tiles_m;
  // this thread's row: of A with one part for the digits, of C with half of the columns
  const int row = tid & (kMc - 1), half = tid >> 7;
  const long long m = tm * kMc + row;
  const bool live = m < s.M;
  long long ba, bbs, bc, oa = 0, ob, oc = 0;
  runs4(bb, s.gb, s.ngb, ba, bbs, bc);
  if (live) runs4(m, s.gm, s.ngm, oa, ob, oc);
  if (tid < K) split_runs32((unsigned)tid, s.kr, s.nk, ka[tid], kb[tid]);
  if (tid < kMc) mx[tid] = 0;
  if (tid == 0) {
    bad = 0;
    tc::mbar_init(smem_u32(&done), 1);
    tc::mbar_init(smem_u32(&drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  pdl_wait();   // before the allocation: a CTA of the launch before may still need the tensor memory
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(kCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const float scale = step_scale<float>(s, meta, blockIdx.x == 0 && tid == 0);
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tmem_slot;

  // ---- A: rows past the edge are left as they are (multiplied into rows never stored)
  {
    const Cx<ff>* src = arena + s.off_a + ba + oa;
    float2 v[8 * OCTS];
    float top = 0.f;
#pragma unroll
    for (int o = 0; o < OCTS; ++o) {
      load8(v + 8 * o, src, ka, 8 * o, live ? K : 0, half);
      top = fmaxf(top, max8(v + 8 * o));
    }
    if (live) atomicMax(&mx[row], __float_as_uint(top));
    __syncthreads();
    const int e = bin_exp(__uint_as_float(mx[row]));
    if (half == 0) ea_s[row] = e;
    if (live) {
#pragma unroll
      for (int o = 0; o < OCTS; ++o)
        put8<S>(v + 8 * o, e, dsm + o * S * kAOct + off8(row, half), nullptr, false, kAOct);
    }
  }

  // ---- B: threads (column, octet, part) of a tile; its exponent over kBLanes threads
  unsigned char* bsm = dsm + OCTS * S * kAOct;
  const int slice = G.nw * 32;
  const int col = tid / kBLanes, bo = (tid % kBLanes) >> 1, bpart = tid & 1;
  float2 bv[8];
  auto load_b = [&](int t) {
    const long long n = (long long)t * G.W + col;
    const bool has = col < G.W && n < s.N;
    long long a, b = 0, c = -1;
    if (has) runs4(n, s.gn, s.ngn, a, b, c);
    load8(bv, arena + s.off_b + bbs + b, kb, 8 * bo, has ? K : 0, bpart);
    return has ? c : -1ll;
  };
  auto put_b = [&](long long c) {   // Re: row 2c first half, 2c + 1 second; Im: 2c + 1 first, -Im: 2c second
    float top = max8(bv);
#pragma unroll
    for (int o = kBLanes / 2; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
    const int e = bin_exp(top);
    if (col < G.W) {
      if (tid % kBLanes == 0) {
        cn[col] = c;
        eb_s[col] = e;
      }
      unsigned char* at = bsm + bo * S * slice;
      put8<S>(bv, e, at + off8(2 * col + bpart, 0), at + off8(2 * col + 1 - bpart, 1), bpart != 0, slice);
    }
  };
  const int t0 = (int)((long long)G.tiles_n * run / runs), t1 = (int)((long long)G.tiles_n * (run + 1) / runs);
  const int quarter = warp & 3;
  const int hb = ((G.W + 3) / 4 + 1) / 2;             // blocks of 4 complex columns of the first half
  Cx<ff>* C = arena + s.off_c + bc + oc;
  float vmax = 0;
  bool failed = false;
  long long cc = load_b(t0);
  for (int t = t0; t < t1; ++t) {
    put_b(cc);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0) {   // A digit i meets B digits 0 .. S-1-i: levels i .. S-1 lie one after another
      const uint64_t da0 = tc::smem_desc(smem_u32(dsm), 128, 256), db0 = tc::smem_desc(smem_u32(bsm), 128, 256);
#pragma unroll
      for (int o = 0; o < OCTS; ++o)
#pragma unroll
        for (int i = 0; i < S; ++i)
          tc::mma_bf16(tmem + (uint32_t)(i * G.nw), da0 + (uint64_t)(((o * S + i) * kAOct) >> 4),
                       db0 + (uint64_t)((o * S * slice) >> 4), tc::idesc((S - i) * G.nw), i > 0 || o > 0 ? 1u : 0u);
      tc::commit(smem_u32(&done));
    }
    if (t + 1 < t1) cc = load_b(t + 1);
    if (!tc::mbar_wait(smem_u32(&done), (uint32_t)((t - t0) & 1), err)) {
      if (lane == 0) {
        bad = 1;
        atomicOr(err, 1ull);
      }
      failed = true;
    }
    __syncwarp();
    tc::fence_after();
    // ---- store: as k_gemm_tc, one flush group
    const int ea = live ? ea_s[row] : 0;
    const long long nv = min((long long)G.W, s.N - (long long)t * G.W);
    const int b1 = half ? (int)(nv + 3) / 4 : min(hb, (int)(nv + 3) / 4);
    for (int b = half ? hb : 0; b < b1; ++b) {   // warp-uniform
      const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * 8);
      float hi[8], lo[8];
      __syncwarp();
      tc::tmem_ld8x2(ta, ta + G.nw, hi, lo);   // levels 0 and 1, added exactly
#pragma unroll
      for (int i = 0; i < 8; ++i) two_sum(hi[i], lo[i] * 0.00390625f, hi[i], lo[i]);
#pragma unroll
      for (int lv = 2; lv < S; lv += 2) {
        float v[8], v2[8];
        const float w = __int_as_float((127 - 8 * lv) << 23);
        if (lv + 1 < S) {
          tc::tmem_ld8x2(ta + lv * G.nw, ta + (lv + 1) * G.nw, v, v2);
          const float w2 = w * 0.00390625f;
#pragma unroll
          for (int i = 0; i < 8; ++i) lo[i] = fmaf(v2[i], w2, fmaf(v[i], w, lo[i]));
        } else {
          tc::tmem_ld8(ta + lv * G.nw, v);
#pragma unroll
          for (int i = 0; i < 8; ++i) lo[i] = fmaf(v[i], w, lo[i]);
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = b * 4 + j;
        if (!live || c >= nv) continue;
        float f1, f2;
        tc::pow2_pair(ea - 14 + eb_s[c], f1, f2);
        ff re = ff_norm((hi[2 * j] * f1) * f2, (lo[2 * j] * f1) * f2);
        ff im = ff_norm((hi[2 * j + 1] * f1) * f2, (lo[2 * j + 1] * f1) * f2);
        re.hi *= scale;
        re.lo *= scale;
        im.hi *= scale;
        im.lo *= scale;
        if (failed) re.hi = re.lo = im.hi = im.lo = __int_as_float(0x7fc00000);
        const Cx<ff> out{re, im};
        st(C + cn[c], out);
        vmax = fmaxf(vmax, mag(out));
      }
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (bad) break;   // uniform: written before the barrier above
  }

  // ---- give-up path: the MMAs in flight are waited for (bounded) before their memory is freed;
  // tiles not reached are left to the error word, which turns the result into a timeout
  if (bad) {
    if (tid == 0) {
      tc::commit(smem_u32(&drain));
      tc::mbar_wait(smem_u32(&drain), 0u, nullptr);
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
  }
  block_max_to_meta(vmax, meta + s.c);
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kCols) : "memory");
}

}  // namespace pk
