// Split-precision GEMM steps with a short contraction (K <= 32) in one kernel, included by
// launch.cu after gemm_tc.cuh, whose digits, levels and sums it shares bit for bit (K is below
// one flush group, and a level's sum is exact in whatever order its products are taken).
//
// As two launches (k_digits, k_gemm_tc) such a step took about 23 us however small, and a wide
// one moved 2.5 times its operands through the digit workspace.  Here a CTA takes a block of 128
// rows and a run of its column tiles: it turns its rows of A into digits in shared memory once,
// then for each tile the columns of B, issues the tile's MMAs and stores C from tensor memory.
// The digits of the next tile's columns are made while the tensor cores read the last one's.
// K is laid out by octets of 8 complex k, one K = 16 MMA step [Re | Im] each, so that K = 5 costs
// one step instead of two.  Tiles are the N columns split evenly (25 columns: 13 + 12, not
// 24 + 1).  One accumulator set and at most 110 KB: two CTAs per multiprocessor, one storing
// while the other multiplies.  The epilogue's instructions bound it (about 80 per complex output).
#pragma once

namespace pk {
namespace tcs {

constexpr int kMaxK = kTcShortK;  // four octets: A's digits and a B tile's within half of shared memory
constexpr int kThreads = 256;
constexpr int kAOct = tc::kMc * 32;   // one digit of an octet of A: 128 rows x 16 BF16

// A step as the kernel reads it: 32-bit extents and strides (a tensor has at most 2^31 elements),
// divisions by multiplication where that is exact (mul 0: not), found once on the host.  Read
// from the 4 KB Step with divisions, the offsets alone took 3000 of a CTA's 12,500 cycles.
struct Run3 {
  uint32_t size, mul, s1, s2;
};
struct Args {
  int32_t a, b, c;                    // bookkeeping slots
  int32_t K, W, nw, tiles_n, runs;    // W columns per tile, nw real columns per MMA (a multiple of 16)
  uint32_t M, N, tiles_m;
  int32_t nm, nn, nk, nb;
  int64_t off_a, off_b, off_c;
  Run3 m[kMaxRuns], n[kMaxRuns], k[kMaxRuns], b3[kMaxRuns];   // strides (A, C), (B, C), (A, B), (A, B)
  uint32_t bc[kMaxRuns];              // a batch index's strides in C
};

inline Args args(const Step& s) {
  Args g;
  g.a = s.a, g.b = s.b, g.c = s.c;
  g.K = (int32_t)s.K;
  g.tiles_n = (int32_t)((s.N + tc::kNc - 1) / tc::kNc);
  g.W = (int32_t)((s.N + g.tiles_n - 1) / g.tiles_n);
  g.nw = 2 * ((g.W + 7) & ~7);
  g.M = (uint32_t)s.M, g.N = (uint32_t)s.N, g.tiles_m = (uint32_t)((s.M + tc::kMc - 1) / tc::kMc);
  g.nm = s.ngm, g.nn = s.ngn, g.nk = s.nk, g.nb = s.ngb;
  g.off_a = s.off_a, g.off_b = s.off_b, g.off_c = s.off_c;
  auto run = [](int64_t size, int64_t top, int64_t s1, int64_t s2) {
    return Run3{(uint32_t)size, div_mul(size, top), (uint32_t)s1, (uint32_t)s2};
  };
  for (int i = 0; i < s.ngm; ++i) g.m[i] = run(s.gm[i].size, s.M, s.gm[i].sa, s.gm[i].sc);
  for (int i = 0; i < s.ngn; ++i) g.n[i] = run(s.gn[i].size, s.N, s.gn[i].sb, s.gn[i].sc);
  for (int i = 0; i < s.nk; ++i) g.k[i] = run(s.kr[i].size, s.K, s.kr[i].sa, s.kr[i].sb);
  for (int i = 0; i < s.ngb; ++i) {
    g.b3[i] = run(s.gb[i].size, s.Bsz, s.gb[i].sa, s.gb[i].sb);
    g.bc[i] = (uint32_t)s.gb[i].sc;
  }
  return g;
}
inline int octets(const Step& s) { return s.K <= 8 ? 1 : s.K <= 16 ? 2 : 4; }   // the kernel's variants
constexpr int smem_bytes(int S, int octs) { return S * octs * (kAOct + 2 * tc::kNc * 32); }

// Column runs per row block: the fewest rounds over the GPU's slots, a round being a CTA's start
// and its conversion of A (about a tile's time and a third of one per octet) and the run's tiles.
inline int col_runs(const Args& g, int octs, long long row_blocks, long long slots) {
  int best = 1;
  double best_cost = 0;
  for (int r = 1; r <= g.tiles_n && r <= 64; ++r) {
    const double cost = (double)((row_blocks * r + slots - 1) / slots) * (0.7 + 0.3 * octs + (g.tiles_n + r - 1) / r);
    if (r == 1 || cost < best_cost) best = r, best_cost = cost;
  }
  return best;
}

__device__ __forceinline__ unsigned quot(unsigned y, const Run3& r) { return r.mul ? __umulhi(y, r.mul) : y / r.size; }
// Both strides' offsets of index y.
__device__ __forceinline__ void offsets(unsigned y, const Run3* r, int n, unsigned& o1, unsigned& o2) {
  o1 = o2 = 0;
#pragma unroll 1
  for (int i = 0; i < n; ++i) {
    const Run3 w = r[i];
    const unsigned q = quot(y, w), d = y - q * w.size;
    y = q;
    o1 += d * w.s1;
    o2 += d * w.s2;
  }
}
// cnt (hi, lo) pairs of one part of consecutive k from k0, zero past K.
template <int CNT>
__device__ __forceinline__ void load_k(float2* v, const Cx<ff>* p, const unsigned* kt, int k0, int K, int part) {
#pragma unroll
  for (int u = 0; u < CNT; ++u) {
    v[u] = make_float2(0.f, 0.f);
    if (k0 + u < K) v[u] = *((const float2*)(p + kt[k0 + u]) + part);
  }
}
template <int CNT>
__device__ __forceinline__ float max_k(const float2* v) {
  float m = 0.f;
#pragma unroll
  for (int u = 0; u < CNT; ++u) m = fmaxf(m, fabsf(v[u].x));
  return m;
}
// Offset of (row, part) in one digit of an octet: 8-row groups of two core matrices.
__device__ __forceinline__ uint32_t off8(int row, int part) {
  return (uint32_t)((row >> 3) * 256 + part * 128 + (row & 7) * 16);
}

}  // namespace tcs

template <int S, int OCTS>
__global__ void __launch_bounds__(tcs::kThreads, 2) k_gemm_short(const __grid_constant__ tcs::Args s, Cx<ff>* arena,
                                                                  Meta* meta, unsigned long long* err) {
  using namespace tcs;
  using tc::kMc;
  using tc::smem_u32;
  constexpr uint32_t kCols = tc::Cfg<S>::kCols;
  constexpr int kPairs = OCTS;            // words per digit of a thread of B: 8 threads per column
  constexpr bool kHold = OCTS <= 2;       // A's values stay in registers between exponent and digits
  static_assert(tc::kNc * 8 <= kThreads, "columns of B per pass");
  extern __shared__ __align__(16) unsigned char dsm[];   // A: [octet][digit], then B: [octet][digit]
  __shared__ unsigned ka[kMaxK], kb[kMaxK];
  __shared__ unsigned cn[2][tc::kNc];     // a tile's C offsets and exponents: two tiles in turn
  __shared__ int eb_s[2][tc::kNc], ea_s[kMc];
  __shared__ __align__(8) unsigned long long done, drain;
  __shared__ uint32_t tmem_slot;
  __shared__ int bad;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, K = s.K, runs = s.runs;
  const unsigned bb = blockIdx.x / s.tiles_m, m0 = (blockIdx.x - bb * s.tiles_m) * kMc;
  const int run = blockIdx.y;
  // the thread's row and part of A for the digits: a warp takes both parts of 16 rows, eight
  // threads in a row the same part (stores without bank conflicts)
  const int part = (lane >> 3) & 1, arow = warp * 16 + (lane & 7) + ((lane >> 4) << 3);
  // its row of C (a tensor memory lane of its warp's quarter) and half of the columns
  const int row = (warp & 3) * 32 + lane, half = warp >> 2;
  const bool alive = m0 + arow < s.M, live = m0 + row < s.M;
  unsigned oa = 0, oc = 0, ob = 0;
  {
    unsigned y = bb, ya = alive ? m0 + arow : 0, yc = live ? m0 + row : 0;
#pragma unroll 1
    for (int i = 0; i < s.nb; ++i) {
      const unsigned q = quot(y, s.b3[i]), d = y - q * s.b3[i].size;
      y = q;
      oa += d * s.b3[i].s1;
      ob += d * s.b3[i].s2;
      oc += d * s.bc[i];
    }
#pragma unroll 1
    for (int i = 0; i < s.nm; ++i) {
      const unsigned qa = quot(ya, s.m[i]), qc = quot(yc, s.m[i]);
      oa += (ya - qa * s.m[i].size) * s.m[i].s1;
      oc += (yc - qc * s.m[i].size) * s.m[i].s2;
      ya = qa;
      yc = qc;
    }
  }
  if (tid < K) offsets((unsigned)tid, s.k, s.nk, ka[tid], kb[tid]);
  if (tid == 0) {
    bad = 0;
    tc::mbar_init(smem_u32(&done), 1);
    tc::mbar_init(smem_u32(&drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  // ---- B: eight threads per column, each kPairs pairs of one part of one octet
  unsigned char* bsm = dsm + OCTS * S * kAOct;
  const int slice = s.nw * 32;
  const int col = tid >> 3, bpart = tid & 1, bo = ((tid >> 1) & 3) * OCTS / 4, p0 = ((tid >> 1) & 3) * OCTS & 3;
  const int bk = 8 * bo + 2 * p0;
  const int t0 = s.tiles_n * run / runs, t1 = s.tiles_n * (run + 1) / runs;
  float2 bv[2 * kPairs];   // loaded one tile ahead
  uint32_t bw[S][kPairs];
  unsigned bcn = 0, bwcn = 0;
  int be = 0;
  auto load_b = [&](int t) {
    const unsigned n = (unsigned)(t * s.W + col);
    const bool has = col < s.W && n < s.N;
    unsigned o = 0;
    if (has) offsets(n, s.n, s.nn, o, bcn);
    load_k<2 * kPairs>(bv, arena + s.off_b + ob + o, kb, bk, has ? K : 0, bpart);
  };
  auto conv_b = [&]() {
    float top = max_k<2 * kPairs>(bv);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, o));
    be = bin_exp(top);
    bwcn = bcn;
    tc::digit_pairs<S, kPairs>([&](int u) { return bv[u]; }, col < s.W ? K - bk : 0, be, bw);
  };
  auto put_b = [&](int buf) {   // Re: row 2c first half, 2c + 1 second; Im: 2c + 1 first, -Im: 2c second
    if (col >= s.W) return;
    if ((tid & 7) == 0) {
      cn[buf][col] = bwcn;
      eb_s[buf][col] = be;
    }
    unsigned char* at = bsm + bo * S * slice + p0 * 4;
    tc::store_pairs<S, kPairs>(bw, at + off8(2 * col + bpart, 0), 0u, slice);
    tc::store_pairs<S, kPairs>(bw, at + off8(2 * col + 1 - bpart, 1), bpart ? 0x80008000u : 0u, slice);
  };

  if (gridDim.x * gridDim.y <= 152) pdl_next();
  pdl_wait();   // before the allocation: a CTA of the launch before may still need the tensor memory
  const Meta ma = meta[s.a], mb = meta[s.b];
  load_b(t0);
  // ---- A: rows past the edge are left as they are (multiplied into rows never stored)
  const Cx<ff>* asrc = arena + s.off_a + oa;
  const int rows_k = alive ? K : 0;
  float2 av[kHold ? 8 * OCTS : 8];
  float top = 0.f;
#pragma unroll
  for (int o = 0; o < OCTS; ++o) {
    float2* v = av + (kHold ? 8 * o : 0);
    load_k<8>(v, asrc, ka, 8 * o, rows_k, part);
    top = fmaxf(top, max_k<8>(v));
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)),
                 "r"(kCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  conv_b();
  put_b(0);
  if (t0 + 1 < t1) load_b(t0 + 1);
  top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, 8));
  const int e = bin_exp(top);
  if (part == 0) ea_s[arow] = e;
  if constexpr (kHold) {
#pragma unroll
    for (int o = 0; o < OCTS; ++o)
      if (alive) tc::digit_rows8<S>([&](int u) { return av[8 * o + u]; }, K - 8 * o, e,
                                    dsm + o * S * kAOct + off8(arow, part), nullptr, false, kAOct);
  } else {   // read again, one octet ahead: unrolled, the code of four octets was mostly fetched
    load_k<8>(av, asrc, ka, 0, rows_k, part);
#pragma unroll 1
    for (int o = 0; o < OCTS; ++o) {
      float2 next[8];
      load_k<8>(next, asrc, ka, 8 * o + 8, rows_k, part);
      if (alive) tc::digit_rows8<S>([&](int u) { return av[u]; }, K - 8 * o, e,
                                    dsm + o * S * kAOct + off8(arow, part), nullptr, false, kAOct);
#pragma unroll
      for (int u = 0; u < 8; ++u) av[u] = next[u];
    }
  }
  // the step's normalisation: a power of two, whose exponent joins the rows' and columns'
  const int en = bin_exp(bits_to_val<float>(ma.maxbits)) + bin_exp(bits_to_val<float>(mb.maxbits));
  if (blockIdx.x == 0 && run == 0 && tid == 0) meta[s.c].exp = ma.exp + mb.exp + en;
  const bool plain = en >= -126 && en <= 126;
  const int ex0 = (plain ? -en : 0) - 14 + 127;   // biased as a float's exponent
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tmem_slot;
  const int ea = ea_s[row] + ex0;
  const int hb = ((s.W + 3) / 4 + 1) / 2;   // blocks of 4 complex columns of the first half
  Cx<ff>* C = arena + s.off_c + oc;
  float vmax = 0;
  bool failed = false;
  for (int t = t0; t < t1; ++t) {
    const int buf = (t - t0) & 1;
    if (tid == kThreads - 32) {   // a warp without columns of B.  A digit i meets B digits 0 .. S-1-i: levels i .. S-1 lie one after another
      const uint64_t da0 = tc::smem_desc(smem_u32(dsm), 128, 256), db0 = tc::smem_desc(smem_u32(bsm), 128, 256);
#pragma unroll 1
      for (int o = 0; o < OCTS; ++o)
#pragma unroll
        for (int i = 0; i < S; ++i)
          tc::mma_bf16(tmem + (uint32_t)(i * s.nw), da0 + (uint64_t)(((o * S + i) * kAOct) >> 4),
                       db0 + (uint64_t)((o * S * slice) >> 4), tc::idesc((S - i) * s.nw), i > 0 || o > 0 ? 1u : 0u);
      tc::commit(smem_u32(&done));
    }
    __syncwarp();
    if (t + 1 < t1) {   // the next tile's digits, in registers while the tensor cores read this one's
      conv_b();
      if (t + 2 < t1) load_b(t + 2);
    }
    if (!tc::mbar_wait(smem_u32(&done), (uint32_t)buf, err)) {
      if (lane == 0) {
        bad = 1;
        atomicOr(err, 1ull);
      }
      failed = true;
    }
    __syncwarp();
    tc::fence_after();
    if (t + 1 < t1) put_b(buf ^ 1);
    // ---- store: as k_gemm_tc, one flush group
    const int nv = min(s.W, (int)s.N - t * s.W);
    const int b1 = half ? (nv + 3) / 4 : min(hb, (nv + 3) / 4);
    for (int b = half ? hb : 0; b < b1; ++b) {   // warp-uniform
      const uint32_t ta = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(b * 8);
      float hi[8], lo[8];
      __syncwarp();
      float lv[S][8];
      if constexpr (S == 5)
        tc::tmem_ld8x5(ta, s.nw, lv);
      else {
        tc::tmem_ld8x2(ta, ta + s.nw, lv[0], lv[1]);
        tc::tmem_ld8x2(ta + 2 * s.nw, ta + 3 * s.nw, lv[2], lv[3]);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        two_sum(lv[0][i], lv[1][i], hi[i], lo[i]);   // levels 0 and 1, added exactly
#pragma unroll
        for (int l = 2; l < S; ++l) lo[i] += lv[l][i];
      }
      float f[4];
      bool far = !plain;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        // the row's and the column's exponent and the step's normalisation (a power of two) at once
        const int x = ea + eb_s[buf][b * 4 + j];
        f[j] = __int_as_float(x << 23);
        far |= (unsigned)(x - 1) >= 254u;
      }
      if (__any_sync(0xffffffffu, far)) {   // beyond a float's exponents: factor by factor
        const float scale = plain ? 1.f : (float)ldexp(1.0, -en);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          float f1, f2;
          tc::pow2_pair(ea + eb_s[buf][b * 4 + i / 2] - 127, f1, f2);
          hi[i] = ((hi[i] * f1) * f2) * scale;
          lo[i] = ((lo[i] * f1) * f2) * scale;
        }
        f[0] = f[1] = f[2] = f[3] = 1.f;
      }
      if (failed) f[0] = f[1] = f[2] = f[3] = __int_as_float(0x7fc00000);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = b * 4 + j;
        if (!live || c >= nv) continue;
        const ff re = ff_norm(hi[2 * j] * f[j], lo[2 * j] * f[j]), im = ff_norm(hi[2 * j + 1] * f[j], lo[2 * j + 1] * f[j]);
        const Cx<ff> out{re, im};
        st(C + cn[buf][c], out);
        vmax = fmaxf(vmax, mag(out));
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (bad) break;   // uniform: written before the barrier above
  }

  // ---- give-up path: the MMAs in flight are waited for (bounded) before their memory is freed;
  // tiles not reached are left to the error word, which turns the result into a timeout
  if (bad) {
    if (tid == kThreads - 32) {
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
