// Complex128 GEMM steps on the tensor cores, included by launch.cu after gemm_tc.cuh.
//
// FP64 runs at 2 multiply-adds per cycle and multiprocessor here (1.25 TFLOP/s), BF16
// products on the tensor cores at 4096, so a wide complex128 step is worth 36 BF16 products
// per real multiply-add.  The splitting is that of Ozaki et al. ("Error-free transformations of
// matrix multiplication", Numer. Algorithms 2012) in fixed point: with e(m) the binary exponent
// of row m's largest entry over the whole contracted index (columns of B likewise),
//     F = round(x 2^(62 - e)),  |F| <= 2^62,  F = sum_{i<8} d_i 256^(7-i),  -128 <= d_i < 128,
// a digit per byte of F + 0x8080808080808080.  A digit is exact in BF16, digit products and
// their FP32 sums over one flush group of K are exact integers (below 2^24), and the groups'
// sums are added as 64-bit integers.  What is lost is the rounding of F (2^-63 of the row's
// largest entry), the dropped levels i + j >= 8 (per term up to 2^-59 of the product of the
// row's and the column's largest entries, 2^-62 as a rule) and the final rounding to 53 bits:
// about sqrt(K) 2^-61 of that product P(m, n), whatever the output's own size.
//
// FP64's own rounding is a share of the terms, not of P.  With the standard weights and q <= 4
// every clause matrix is the exponential of a quadratic form (over Z_2, Z_3 or Z_2^2), every
// tensor a Gauss sum, and its nonzero entries have one magnitude: an output has a term as large
// as P or none at all.  Elsewhere (q > 4, general weights) the entries of a row may lie any
// number of powers of two apart.  There an output is kept if it is above 2^-kSure of P, or one of
// its terms is above 2^-(kSure + 2) of P (marks, k_digits64): the loss is then about sqrt(K) 2^-53 of
// that, as FP64's.  Any other is formed again in FP64 (small_outputs), and so is every output of a
// row or column with an infinity or a NaN.  Counted on the CPU over the steps of nine knots at
// q = 5 to 12: 0 to 4 % of a step's outputs are small as a rule (up to 87 %), and 0 to 0.3 % are
// formed again (up to 14 %).  Cost on GB300, 167 crossings at q = 5: 872 -> 886 us per launch
// sequence, 788 -> 806 to 822 us with over / under bits that form outputs again.
//
// The complex product is arranged as in gemm_tc.cuh: a complex row of A is one real row
// [Re | Im], a complex column of B two real columns [Re; -Im] and [Im; Re].
//
//  * k_digits64: a CTA per 8 to 128 rows (8 or 16 complex columns of B), fewer for a longer K:
//    their exponents over all of K, then the digits in the MMA's canonical K-major layout (8-row
//    x 16-byte core matrices).  Only integer and FP32 instructions: a conversion through FP64
//    would take longer than the GEMM.
//  * k_gemm64: persistent, one CTA per multiprocessor, tiles of 128 complex rows x 16 complex
//    columns; warp 0 streams the digit chunks (8 complex k: 32 KB + 8 KB) through a 5-stage
//    ring of bulk copies, warp 1 issues 8 MMAs per chunk (A digit i against B digits 0 .. 7-i
//    stacked along N), 16 epilogue warps fold the 8 level accumulators (two sets in tensor
//    memory, so a group's flush overlaps the next one's products) into 64-bit integers and
//    build the doubles from their bits.  A chunk needs 68 KB of operand reads and 40 KB of
//    copy writes of shared memory, 850 cycles at 128 B per cycle, against 576 of the tensor
//    pipe: 47 complex TFLOP/s at most.
//
// Measured on GB300, per call, this path alone: 167 crossings at q = 5 6070 -> 807 us (without the
// small outputs), 205 crossings at q = 3 1250 -> 214 us, the reverse pass of 300 crossings 3860 ->
// 2147 us; the step of 2.4e8 multiply-adds 2090 -> 94 us and 35 us of conversion.  Error of Z against exact integers,
// 36 knots at q = 3, 4, 5: rms 2.5e-15 -> 1.6e-15, largest 1.2e-14 -> 3.7e-15.
#pragma once

namespace pk {
namespace d64 {

constexpr int kS = 8;                        // digits
constexpr int kNc = kTc64Nc, kKc = kTc64Kc;  // complex columns per tile, complex k per chunk
constexpr int kMc = kTcMc;                   // complex rows per tile
constexpr int kN = 2 * kNc;
constexpr int kABytes = kMc * 2 * kKc * 2, kBBytes = kN * 2 * kKc * 2;   // one digit of a chunk
constexpr int kAChunk = kS * kABytes, kBChunk = kS * kBBytes, kStage = kAChunk + kBChunk;
constexpr int kStages = 5, kSmem = kStages * kStage;
// chunks per flush: 8 pairs x 16 real k x 2^14 per chunk stay below 2^24
constexpr int kFlush = ((1 << 10) - 1) / (kS * 2 * kKc);
constexpr int kEpiWarps = 16, kThreads = 32 * (2 + kEpiWarps);
constexpr int kConvThreads = 128;
constexpr int kBad = 1 << 28;                // exponent of a row with a non-finite entry
constexpr int kSure = 8;
constexpr int kListed = 2048, kListWarp = 24;   // small outputs a CTA leaves to its end, at most; of a warp's 128
// An entry's marks: it reaches 2^-mark(j) of its row's largest entry (a column's: the marks in turn
// from the last); a pair with a common mark has a product above 2^-(kSure + 2) of P.  A last mark
// says that it is not 0 (below 2^-1042: as 0); without a pair of these the output is 0.
constexpr int kMarks = 3;
__device__ __forceinline__ constexpr int mark(int j) { return kSure / (kMarks - 1) * j; }
static_assert(kS * kN <= 256 && kSmem <= 220 * 1024 && kFlush * kS * 2 * kKc < 1024, "tile geometry");
static_assert(kAChunk == kTc64AChunk && kBChunk == kTc64BChunk, "scratch layout");

// F = round(x 2^(62 - e)) + 0x8080808080808080: a digit plus 128 per byte, the leading digit in
// the top byte.
__device__ __forceinline__ unsigned long long fixed_bytes(double x, int e) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = max(1, (int)(b >> 52) & 0x7ff);
  unsigned long long m = b & 0xFFFFFFFFFFFFFull;
  if ((b >> 52) & 0x7ff) m |= 1ull << 52;
  const int s = ex - 1013 - e;   // m 2^(ex - 1075) 2^(62 - e); at most 9
  unsigned long long f;
  if (s >= 0)
    f = m << s;
  else
    f = s < -54 ? 0ull : (m + (1ull << (-s - 1))) >> -s;
  if ((long long)b < 0) f = 0ull - f;
  return f + 0x8080808080808080ull;
}

// BF16 digit i of 8 consecutive k as 16 bytes; flip: negated.
__device__ __forceinline__ uint4 digit_row(const unsigned long long* f, int i, bool flip) {
  uint32_t w[4];
#pragma unroll
  for (int u = 0; u < 8; u += 2) {
    float d[2];
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const uint32_t word = i < 4 ? (uint32_t)(f[u + v] >> 32) : (uint32_t)f[u + v];
      d[v] = __int_as_float(__byte_perm(word, 0x4B000000u, 0x7440 | (3 - (i & 3)))) - 8388736.0f;   // 2^23 + 128
    }
    w[u >> 1] = __byte_perm(__float_as_uint(d[0]), __float_as_uint(d[1]), 0x7632);
    if (flip) w[u >> 1] ^= 0x80008000u;
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

}  // namespace d64

// 8-row groups per CTA (a power of two up to a tile's `parts`): about 16 (group, chunk) items
// for its 16 groups of 8 threads, so that a short K still fills the CTA.
__host__ __device__ inline int d64_groups(long long chunks, int parts) {
  int g = 1;
  while (g < parts && 2 * g * chunks <= 16) g *= 2;
  return g;
}

template <bool IS_A>
__device__ __forceinline__ void digits64_block(const Step& s, const Cx<double>* arena, unsigned char* scratch,
                                               const int* even, long long blk, unsigned* kt, unsigned* mx,
                                               long long* ro) {
  using namespace d64;
  const Tc64Scratch L = tc64_scratch(s.Bsz, s.M, s.N, s.K);
  constexpr int kT = IS_A ? kMc : kNc, kParts = kT / 8;
  const int G = d64_groups(L.chunks, kParts), RB = 8 * G, parts = kParts / G;
  const int part = (int)(blk % parts);
  const long long t = blk / parts, tiles = IS_A ? L.tiles_m : L.tiles_n;
  const long long tile = t % tiles, bb = t / tiles;
  const long long ext = IS_A ? s.M : s.N;
  const long long r0 = tile * kT + part * RB;
  const int tid = threadIdx.x, K = (int)s.K;
  const bool own = *even == 0;
  if (tid < RB) {
    mx[tid] = 0;
    long long a = 0, b = 0, c, ba, bo, bc, off = -1, cc = -1;
    if (r0 + tid < ext) {
      runs4(bb, s.gb, s.ngb, ba, bo, bc);
      if (IS_A)
        runs4(r0 + tid, s.gm, s.ngm, a, b, c);
      else
        runs4(r0 + tid, s.gn, s.ngn, a, b, c);
      off = IS_A ? ba + a : bo + b;
      cc = IS_A ? bc + c : c;
    }
    ro[tid] = off;
    // the row's (column's) C offset for the GEMM's epilogue; columns do not depend on bb
    if (IS_A || bb == 0)
      ((long long*)(scratch + (IS_A ? L.cr_off : L.cc_off)))[(IS_A ? bb * tiles + tile : tile) * kT + part * RB + tid] = cc;
    if (own)
      ((unsigned*)(scratch + (IS_A ? L.oa_off : L.ob_off)))[(bb * tiles + tile) * kT + part * RB + tid] = (unsigned)max(off, 0LL);
  }
  for (int k = tid; k < K; k += kConvThreads) {
    long long ka, kb;
    split_runs32((unsigned)k, s.kr, s.nk, ka, kb);
    kt[k] = (unsigned)(IS_A ? ka : kb);
    if (own && IS_A && blk == 0) ((uint2*)(scratch + L.ok_off))[k] = make_uint2((unsigned)ka, (unsigned)kb);
  }
  __syncthreads();
  if (r0 >= ext) return;   // rows past the edge are multiplied but not stored
  const Cx<double>* src = arena + (IS_A ? s.off_a : s.off_b);
  const bool kin = IS_A ? s.a_kinner != 0 : s.b_kinner != 0;
  const int lanes = kConvThreads / RB;   // threads per row in the exponent pass
  {  // largest high word of each row over all of K; lanes along the operand's unit stride
    const int r = kin ? tid / lanes : tid & (RB - 1), l = kin ? tid & (lanes - 1) : tid / RB;
    unsigned m = 0;
    if (ro[r] >= 0)
      for (int k = l; k < K; k += lanes) {
        const Cx<double> v = ld(src + ro[r] + kt[k]);
        m = max(m, max((unsigned)__double2hiint(v.re) & 0x7fffffffu, (unsigned)__double2hiint(v.im) & 0x7fffffffu));
      }
    atomicMax(&mx[r], m);
  }
  __syncthreads();
  auto exponent = [&](int r) {
    const unsigned top = mx[r];
    return top >= 0x7ff00000u ? kBad : (int)(max(top, 1u << 20) >> 20) - 1022;
  };
  if (tid < RB)
    ((int*)(scratch + (IS_A ? L.ea_off : L.eb_off)))[(bb * tiles + tile) * kT + part * RB + tid] = exponent(tid);
  constexpr int kChunk = IS_A ? kAChunk : kBChunk, kSlice = IS_A ? kABytes : kBBytes;
  unsigned char* dst = scratch + (IS_A ? L.a_off : L.b_off) + (bb * tiles + tile) * L.chunks * (long long)kChunk;
  // items (8-row group, chunk): 8 threads each, a row of 8 k per thread
  for (int it = tid >> 3; it < G * (int)L.chunks; it += kConvThreads / 8) {
    const int g = it & (G - 1), c = it / G, r = g * 8 + (tid & 7);
    const int e = exponent(r);
    const long long off = ro[r];
    unsigned char* ch = dst + (long long)c * kChunk;
    double re[8], im[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      re[u] = im[u] = 0;
      const int k = c * kKc + u;
      if (off >= 0 && k < K && e != kBad) {
        const Cx<double> v = ld(src + off + kt[k]);
        re[u] = v.re;
        im[u] = v.im;
      }
    }
    if (own) {   // the 8 entries' marks, a byte for each threshold
      unsigned m = 0, least[kMarks];   // high words; entries below the normal range have no mark
#pragma unroll
      for (int j = 0; j < kMarks; ++j) least[j] = (unsigned)max(1, min(2047, e + 1022 - mark(IS_A ? j : kMarks - 1 - j))) << 20;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const unsigned top = max((unsigned)__double2hiint(re[u]) & 0x7fffffffu, (unsigned)__double2hiint(im[u]) & 0x7fffffffu);
#pragma unroll
        for (int j = 0; j < kMarks; ++j)
          if (top >= least[j]) m |= 1u << (8 * j + u);
        if (top) m |= 1u << (8 * kMarks + u);
      }
      ((unsigned*)(scratch + (IS_A ? L.xa_off : L.xb_off)))[((bb * tiles + tile) * L.chunks + c) * kT + part * RB + r] = m;
    }
#pragma unroll
    for (int part2 = 0; part2 < 2; ++part2) {   // the real, then the imaginary components
      unsigned long long f[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) f[u] = fixed_bytes(part2 ? im[u] : re[u], e);
      if (IS_A) {   // row [Re | Im]
        unsigned char* o = ch + (part * G + g) * 256 + part2 * 128 + (tid & 7) * 16;
#pragma unroll
        for (int i = 0; i < kS; ++i) *(uint4*)(o + i * kSlice) = digit_row(f, i, false);
      } else {      // complex column n: rows 2n = [Re | -Im], 2n + 1 = [Im | Re]
        const int n = part * RB + r;
        unsigned char* o = ch + (n >> 2) * 256 + ((2 * n) & 7) * 16;
#pragma unroll
        for (int i = 0; i < kS; ++i) {
          const uint4 d = digit_row(f, i, false);
          *(uint4*)(o + i * kSlice + (part2 ? 16 : 0)) = d;
          *(uint4*)(o + i * kSlice + (part2 ? 128 : 128 + 16)) = part2 ? digit_row(f, i, true) : d;
        }
      }
    }
  }
}

// Blocks [0, nA) convert A, the rest B.
__global__ void __launch_bounds__(d64::kConvThreads, 8) k_digits64(const Step s, const Cx<double>* arena,
                                                                unsigned char* scratch, const int* even, long long nA) {
  pdl_wait();
  __shared__ unsigned kt[kTc64MaxK], mx[kTcMc];
  __shared__ long long ro[kTcMc];
  const long long blk = blockIdx.x;
  if (blk < nA)
    digits64_block<true>(s, arena, scratch, even, blk, kt, mx, ro);
  else
    digits64_block<false>(s, arena, scratch, even, blk - nA, kt, mx, ro);
}

namespace d64 {
// T = h 2^32 + l as a double times 2^x, rounded to nearest, from integer instructions.
__device__ __forceinline__ unsigned long long to_double_bits(long long h, long long l, int x) {
  long long th = (h >> 32) + (l >> 63);
  unsigned long long tl = (unsigned long long)h << 32;
  const unsigned long long sum = tl + (unsigned long long)l;
  th += sum < tl ? 1 : 0;
  tl = sum;
  const unsigned long long sign = th < 0 ? 1ull << 63 : 0ull;
  if (th < 0) {
    tl = 0ull - tl;
    th = ~th + (tl == 0 ? 1 : 0);
  }
  unsigned long long u = (unsigned long long)th;
  int p = 127;
  if (u == 0) {
    u = tl;
    tl = 0;
    p = 63;
  }
  if (u == 0) return 0ull;
  const int z = __clzll((long long)u);
  if (z) u = u << z | tl >> (64 - z);
  p -= z;                       // the leading bit's weight
  u = (u >> 11) + ((u >> 10) & 1);   // 53 bits; a carry to 2^53 moves into the exponent below
  const int ef = p + x + 1022;  // the leading bit of u adds 1
  if (ef < 0) return sign;      // below the normal range: 0
  if (ef >= 2046) return sign | 0x7ff0000000000000ull;
  return sign | (((unsigned long long)ef << 52) + u);
}

// A sum over k by eight lanes.
__device__ __forceinline__ Acc<double> eighth_sum(const Cx<double>* A, const Cx<double>* B, const uint2* ok, int K) {
  Acc64 acc;
#pragma unroll 2
  for (int k = threadIdx.x & 7; k < K; k += 8) {
    const uint2 o = ok[k];
    acc.mac(ld(A + o.x), ld(B + o.y));
  }
  Acc<double> sum = acc.sum();
  lanes_sum(sum, 3);
  return sum;
}

// The listed small outputs (tile, row << 4 | column in it) in FP64, by the epilogue warps: four at a
// time, eight lanes each.  Returns the lane's largest magnitude.  This and the next one are out of
// line and not unrolled: inlined, their instructions cost every launch of k_gemm64 2 us.
__device__ __noinline__ unsigned long long listed_outputs(const Step& s, Cx<double>* arena, const unsigned char* scratch,
                                                          const uint2* list, int n, int e) {
  const Tc64Scratch L = tc64_scratch(s.Bsz, s.M, s.N, s.K);
  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) - 2;
  const double scale = ldexp(1.0, e);
  unsigned long long vmax = 0;
#pragma unroll 1
  for (int i0 = 4 * warp; i0 < n; i0 += 4 * kEpiWarps) {
    const int i = i0 + (lane >> 3);
    const uint2 at = list[min(i, n - 1)];
    const bool has = i < n && at.x != ~0u;
    const unsigned t = has ? at.x : 0, tiles_n = (unsigned)L.tiles_n, row = t / tiles_n, tn = t - row * tiles_n;
    const unsigned r = row * kMc + (at.y >> 4), c = tn * kNc + (at.y & 15);
    const unsigned oa = ((const unsigned*)(scratch + L.oa_off))[r];
    const unsigned ob = ((const unsigned*)(scratch + L.ob_off))[row / (unsigned)L.tiles_m * tiles_n * kNc + c];
    const long long out = ((const long long*)(scratch + L.cr_off))[r] + ((const long long*)(scratch + L.cc_off))[c];
    const Acc<double> sum = eighth_sum(arena + s.off_a + oa, arena + s.off_b + ob, (const uint2*)(scratch + L.ok_off),
                                       has ? (int)s.K : 0);
    if (has && (lane & 7) == 0) {
      const Cx<double> v = sum.get(scale);
      vmax = max(vmax, mag_key(v));
      st(arena + s.off_c + out, v);
    }
  }
  return vmax;
}

// A warp's small outputs in FP64 at once: bit j of `again`, column j of the warp's four in the lane's
// row, to crow + cc[j].  Returns the lane's largest magnitude.
__device__ __noinline__ unsigned long long small_outputs(const Step& s, Cx<double>* arena, const unsigned char* scratch,
                                                         long long row, long long tn, long long crow, unsigned again, int e) {
  const Tc64Scratch L = tc64_scratch(s.Bsz, s.M, s.N, s.K);
  const int lane = threadIdx.x & 31, quarter = (threadIdx.x >> 5) & 3, cq = ((threadIdx.x >> 5) - 2) >> 2, K = (int)s.K;
  const unsigned oa = ((const unsigned*)(scratch + L.oa_off))[row * kMc + quarter * 32 + lane];
  const unsigned* ob = (const unsigned*)(scratch + L.ob_off) + (row / L.tiles_m * L.tiles_n + tn) * kNc + cq * 4;
  const long long* cc = (const long long*)(scratch + L.cc_off) + tn * kNc + cq * 4;
  const uint2* ok = (const uint2*)(scratch + L.ok_off);
  const Cx<double>*A0 = arena + s.off_a, *B0 = arena + s.off_b;
  Cx<double>* C = arena + s.off_c;
  const double scale = ldexp(1.0, e);
  unsigned long long vmax = 0;
  auto put = [&](const Acc<double>& sum, long long at) {
    const Cx<double> v = sum.get(scale);
    vmax = max(vmax, mag_key(v));
    st(C + at, v);
  };
  __syncwarp();   // the stores before the call come before those of other lanes here
#pragma unroll 1
  for (int j = 0; j < 4; ++j) {
    const bool mine = again >> j & 1;
    unsigned todo = __ballot_sync(0xffffffffu, mine);
    if (!todo) continue;
    const Cx<double>* B = B0 + ob[j];
    const long long c = cc[j];
    // FP64 instructions: a lane per output, or eight (and their sum) for four outputs at a time
    if (4 * K + 6 < ((__popc(todo) + 3) >> 2) * (4 * ((K + 7) >> 3) + 10)) {
      Acc64 acc;
      if (mine) {
#pragma unroll 4
        for (int k = 0; k < K; ++k) {
          const uint2 o = ok[k];
          acc.mac(ld(A0 + oa + o.x), ld(B + o.y));
        }
        put(acc.sum(), crow + c);
      }
      continue;
    }
#pragma unroll 1
    while (todo) {
      int src = -1;   // this group's lane: of the first four in turn
#pragma unroll 1
      for (int i = 0; i < 4 && todo; ++i, todo &= todo - 1)
        if (i == lane >> 3) src = __ffs(todo) - 1;
      const Cx<double>* A = A0 + __shfl_sync(0xffffffffu, oa, max(src, 0));
      const long long at = __shfl_sync(0xffffffffu, crow, max(src, 0)) + c;
      const Acc<double> sum = eighth_sum(A, B, ok, src < 0 ? 0 : K);
      if (src >= 0 && (lane & 7) == 0) put(sum, at);
    }
  }
  return vmax;
}
}  // namespace d64

// even: a word of the uploaded program, nonzero where no output needs small_outputs.
__global__ void __launch_bounds__(d64::kThreads, 1) k_gemm64(const __grid_constant__ Step s, Cx<double>* arena, Meta* meta,
                                                             const unsigned char* scratch, const int* even,
                                                             unsigned long long* err) {
  pdl_wait();
  using namespace d64;
  using tc::bulk_g2s;
  using tc::commit;
  using tc::mbar_arrive;
  using tc::mbar_expect_tx;
  using tc::mbar_init;
  using tc::mbar_wait;
  using tc::smem_u32;
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ __align__(8) unsigned long long full[kStages], empty[kStages], acc_full[2], acc_empty[2], drain;
  __shared__ unsigned long long red[kEpiWarps + 2];
  __shared__ uint32_t tmem_slot;
  __shared__ int bad, listed;
  __shared__ uint2 list[kListed];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const Tc64Scratch L = tc64_scratch(s.Bsz, s.M, s.N, s.K);
  const int ntiles = (int)(L.tiles_m * L.tiles_n * s.Bsz);
  if (tid == 0) {
    bad = listed = 0;
    for (int i = 0; i < kStages; ++i) {
      mbar_init(smem_u32(&full[i]), 1);
      mbar_init(smem_u32(&empty[i]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&acc_full[i]), 1);
      mbar_init(smem_u32(&acc_empty[i]), kEpiWarps);
    }
    mbar_init(smem_u32(&drain), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  const int ea = bin_exp(bits_to_val<double>(meta[s.a].maxbits)), eb = bin_exp(bits_to_val<double>(meta[s.b].maxbits));
  if (blockIdx.x == 0 && tid == 0) meta[s.c].exp = meta[s.a].exp + meta[s.b].exp + ea + eb;
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tmem_slot, sm0 = smem_u32(dsm);
  const int nchunks = (int)L.chunks, ngroups = (nchunks + kFlush - 1) / kFlush;
  int issued = 0, mmas = 0;   // chunks whose copies / MMAs this CTA started
  unsigned long long vmax = 0;
  // tiles: column blocks fastest, so the tiles in flight share few row blocks of A
  if (warp == 0) {
    if (lane == 0) {
      int gc = 0;
      for (int t = blockIdx.x; t < ntiles && !bad; t += gridDim.x) {
        const long long row = t / L.tiles_n, bb = row / L.tiles_m;
        const unsigned char* a = scratch + L.a_off + row * nchunks * (long long)kAChunk;
        const unsigned char* b = scratch + L.b_off + (bb * L.tiles_n + t % L.tiles_n) * nchunks * (long long)kBChunk;
        for (int c = 0; c < nchunks; ++c, ++gc) {
          const int st = gc % kStages;
          if (gc >= kStages && !mbar_wait(smem_u32(&empty[st]), (uint32_t)((gc / kStages - 1) & 1), err)) {
            bad = 1;
            atomicOr(err, 1ull);
            break;
          }
          const uint32_t dst = sm0 + st * kStage;
          mbar_expect_tx(smem_u32(&full[st]), kStage);
          bulk_g2s(dst, a + (long long)c * kAChunk, kAChunk, smem_u32(&full[st]));
          bulk_g2s(dst + kAChunk, b + (long long)c * kBChunk, kBChunk, smem_u32(&full[st]));
          issued = gc + 1;
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int gc = 0, gg = 0;
      bool stop = false;
      for (int t = blockIdx.x; t < ntiles && !stop; t += gridDim.x)
        for (int c = 0; c < nchunks; ++c, ++gc) {
          const int st = gc % kStages, set = gg & 1, use = gg >> 1;
          const bool first = c % kFlush == 0, last = (c + 1) % kFlush == 0 || c + 1 == nchunks;
          if ((first && use > 0 && !mbar_wait(smem_u32(&acc_empty[set]), (uint32_t)((use - 1) & 1), err)) ||
              !mbar_wait(smem_u32(&full[st]), (uint32_t)((gc / kStages) & 1), err)) {
            bad = 1;
            atomicOr(err, 1ull);
            stop = true;
            break;
          }
          tc::fence_after();
          const uint32_t a0 = sm0 + st * kStage, tacc = tmem + (uint32_t)set * 256u;
          const uint64_t da = tc::smem_desc(a0, 128, 256), db = tc::smem_desc(a0 + kAChunk, 128, 256);
          // A digit i meets B digits 0 .. 7-i in one MMA: levels i .. 7 lie one after another
#pragma unroll
          for (int i = 0; i < kS; ++i)
            tc::mma_bf16(tacc + i * kN, da + (uint64_t)((i * kABytes) >> 4), db, tc::idesc((kS - i) * kN),
                         first && i == 0 ? 0u : 1u);
          commit(smem_u32(&empty[st]));
          if (last) {
            commit(smem_u32(&acc_full[set]));
            ++gg;
          }
          mmas = gc + 1;
        }
    }
  } else {
    const int quarter = warp & 3, cq = (warp - 2) >> 2;   // lanes and 8 real columns of this warp
    const bool check = *even == 0;
    int gg = 0;
    bool failed = false;
    for (int t = blockIdx.x; t < ntiles && !failed; t += gridDim.x) {
      const long long row = t / L.tiles_n, bb = row / L.tiles_m, tn = t % L.tiles_n;
      const long long crow = ((const long long*)(scratch + L.cr_off))[row * kMc + quarter * 32 + lane];
      const int em = ((const int*)(scratch + L.ea_off))[row * kMc + quarter * 32 + lane];
      const long long* ccp = (const long long*)(scratch + L.cc_off) + tn * kNc + cq * 4;
      const int* enp = (const int*)(scratch + L.eb_off) + (bb * L.tiles_n + tn) * kNc + cq * 4;
      const bool any = tn * kNc + cq * 4 < s.N;   // columns of C among this warp's (warp-uniform)
      long long h[8], l[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) h[j] = l[j] = 0;
      for (int g = 0; g < ngroups; ++g, ++gg) {
        const int set = gg & 1;
        if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(&acc_full[set]), (uint32_t)((gg >> 1) & 1), err))) {
          if (lane == 0) {
            bad = 1;
            atomicOr(err, 1ull);
          }
          failed = true;
          break;
        }
        tc::fence_after();
        if (any) {
          // level L's integers (exact, below 2^24 in magnitude) at weight 256^(7-L)
          const uint32_t ta = tmem + (uint32_t)set * 256u + ((uint32_t)(quarter * 32) << 16) + cq * 8;
          float v[4][8];
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            long long* acc = half ? l : h;
            tc::tmem_ld8x2(ta + (4 * half) * kN, ta + (4 * half + 1) * kN, v[0], v[1]);
            tc::tmem_ld8x2(ta + (4 * half + 2) * kN, ta + (4 * half + 3) * kN, v[2], v[3]);
            if (nchunks <= 2) {   // |v| <= 2^22: the integer is the pattern of v + 1.5 2^23 less a constant
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const auto n = [&](int i) { return __float_as_int(v[i][j] + 12582912.0f); };
                acc[j] += ((((long long)n(0) * 256 + n(1)) * 256 + n(2)) * 256 + n(3)) - 0x4B400000ll * 0x01010101ll;
              }
            } else {
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const auto n = [&](int i) { return __float2int_rn(v[i][j]); };
                acc[j] += (((long long)n(0) * 256 + n(1)) * 256 + n(2)) * 256 + n(3);
              }
            }
          }
        }
        tc::fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&acc_empty[set]));
      }
      // the tile, while the next one's products run
      Cx<double>* C = arena + s.off_c;
      unsigned again = 0, bare = 0;   // outputs that are small against P; those without digits
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const long long cc = any ? ccp[j] : -1;
        if (crow < 0 || cc < 0) continue;
        const int en = enp[j];
        unsigned long long re = 0x7ff8000000000000ull, im = re;   // NaN
        bool sure = failed || !check;
        if (!failed && em < kBad && en < kBad) {
          const int x = em + en - 68 - ea - eb;
          re = to_double_bits(h[2 * j], l[2 * j], x);
          im = to_double_bits(h[2 * j + 1], l[2 * j + 1], x);
          const unsigned long long top = max(re & 0x7fffffffffffffffull, im & 0x7fffffffffffffffull);
          const int et = (int)(top >> 52);   // 0: zero, or below the normal range
          sure = sure || (et > 0 && et - 1023 >= x + 68 - kSure);
          vmax = max(vmax, top);
        } else {
          bare |= 1u << j;
        }
        if (!sure) again |= 1u << j;
        st(C + crow + cc, Cx<double>{__longlong_as_double((long long)re), __longlong_as_double((long long)im)});
      }
      if (__any_sync(0xffffffffu, again)) {   // those with two entries that share a mark are kept, and zeros
        const unsigned* xa = (const unsigned*)(scratch + L.xa_off) + row * nchunks * kMc + quarter * 32 + lane;
        const uint4* xb = (const uint4*)(scratch + L.xb_off) + (bb * L.tiles_n + tn) * nchunks * (kNc / 4) + cq;
        uint4 hit = make_uint4(0, 0, 0, 0);
#pragma unroll 4
        for (int c = 0; c < nchunks; ++c) {
          const unsigned a = xa[c * kMc];
          const uint4 b = xb[c * (kNc / 4)];
          hit.x |= a & b.x;
          hit.y |= a & b.y;
          hit.z |= a & b.z;
          hit.w |= a & b.w;
        }
        const auto open = [](unsigned h) { return h >> (8 * kMarks) && !(h << (32 - 8 * kMarks)) ? 1u : 0u; };
        again &= open(hit.x) | open(hit.y) << 1 | open(hit.z) << 2 | open(hit.w) << 3 | bare;
        const int most = (int)__reduce_add_sync(0xffffffffu, (unsigned)__popc(again));
        if (most > 0) {
          // few: left to the end of the CTA's tiles, where their chains of loads run side by side
          // (167 crossings at q = 5 with 0.2 % of one K = 5 step's outputs: 849 -> 822 us)
          int at = kListed;
          if (most <= kListWarp) {
            if (lane == 0) at = atomicAdd(&listed, most);
            at = __shfl_sync(0xffffffffu, at, 0);
          }
          const bool fits = at + most <= kListed;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const unsigned who = __ballot_sync(0xffffffffu, again >> j & 1);
            const int i = at + __popc(who & ((1u << lane) - 1));
            if ((again >> j & 1) && i < kListed)   // where they no longer fit: empty entries
              list[i] = make_uint2(fits ? (unsigned)t : ~0u, (unsigned)((quarter * 32 + lane) << 4 | (cq * 4 + j)));
            at += __popc(who);
          }
          if (!fits) vmax = max(vmax, small_outputs(s, arena, scratch, row, tn, crow, again, -(ea + eb)));
        }
      }
    }
    if (check) {
      asm volatile("bar.sync 1, %0;" ::"n"(32 * kEpiWarps) : "memory");
      const int n = min(listed, kListed);
      if (n > 0 && !failed) vmax = max(vmax, listed_outputs(s, arena, scratch, list, n, -(ea + eb)));
    }
  }
  {  // max-abs of the CTA's outputs
    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(vmax >> 32));
    const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(vmax >> 32) == hi ? (unsigned)vmax : 0u);
    if (lane == 0) red[warp] = (unsigned long long)hi << 32 | lo;
  }
  __syncthreads();
  if (bad) {   // give-up path: wait (bounded) for this CTA's copies and MMAs in flight
    if (warp == 0 && lane == 0)
      for (int c = issued > kStages ? issued - kStages : 0; c < issued; ++c)
        mbar_wait(smem_u32(&full[c % kStages]), (uint32_t)((c / kStages) & 1), nullptr);
    if (warp == 1 && lane == 0 && mmas > 0) {
      commit(smem_u32(&drain));
      mbar_wait(smem_u32(&drain), 0u, nullptr);
    }
  }
  if (tid == 0) {
    unsigned long long m = 0;
    for (int i = 0; i < kEpiWarps + 2; ++i) m = max(m, red[i]);
    if (m) atomicMax(&meta[s.c].maxbits, m);
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

}  // namespace pk
