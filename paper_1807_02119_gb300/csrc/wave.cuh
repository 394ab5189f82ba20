// Level kernels: the light steps of one or more levels of the contraction tree in one
// launch (schedule and records: wave_plan.cpp), included by launch.cu.
//
// What bounds them is latency: a level holds a few hundred to a few ten thousand outputs of
// 1 to 100 terms, so its time is one warp's chain of instructions and memory round trips plus
// the gap to the next level.  Hence the compact records (64 bytes and 16 per stride run, read
// as 16-byte broadcasts), one warp per 32 lanes of outputs without block barriers, index
// divisions by one multiplication, and levels chained inside one cluster.
#pragma once

namespace pk {

// Measured on GB300, whole calls of perf/cases.py against one small step after another in one CTA:
// 330 crossings at q = 3 in complex64 1.17 -> 0.35 ms (0.27 to 0.35 by the over / under bits) and
// 167 crossings at q = 5 in split 1.97 -> 0.47 ms (with gemm_short.cuh); the reverse pass of 99
// crossings at q = 5 in split 2.09 -> 0.37 ms.  A level
// of the cluster kernel takes 1.5 to 2 us: 0.16 us for an operand's round trip to L2, 0.3 us
// for the cluster barrier, the rest one warp's 200 to 300 dependent instructions (FP64
// multiply-adds: 63 cycles each).  A level launched alone takes 0.9 us more.

// How a level's operands are read: written by other CTAs of the same launch (past L1), by
// earlier launches only (L1, once those have ended), or by this CTA only (L1).  kWaveAny besides:
// steps of any size, whose divisions may lack an exact multiplier (mul 0).
enum WaveMode { kWaveL2 = 0, kWaveEarlier = 1, kWaveOwn = 2, kWaveAny = 4 };

// Offsets in A and B of index y of a run class (`r` the class's first run, n >= 1 of them);
// y / size = umulhi(y, ceil(2^32 / size)), exact for the steps the planner gives a multiplier.
template <int M = kWaveL2>
__device__ __forceinline__ void wave_offsets(unsigned y, const uint4* r, int n, unsigned& oa, unsigned& ob) {
  uint4 w = *r;   // size, mul, sa, sb
#pragma unroll 1
  for (; --n > 0; w = *++r) {
    const unsigned t = (M & kWaveAny) && !w.y ? y / w.x : __umulhi(y, w.y), d = y - t * w.x;
    oa += d * w.z;
    ob += d * w.w;
    y = t;
  }
  oa += y * w.z;
  ob += y * w.w;
}

// Operands may have been written by another CTA of the same launch: read past L1.
__device__ __forceinline__ Cx<double> ldl2(const Cx<double>* p) {
  const double2 v = __ldcg(reinterpret_cast<const double2*>(p));
  return {v.x, v.y};
}
__device__ __forceinline__ Cx<float> ldl2(const Cx<float>* p) {
  const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
  return {v.x, v.y};
}
__device__ __forceinline__ Cx<ff> ldl2(const Cx<ff>* p) {
  const float4 v = __ldcg(reinterpret_cast<const float4*>(p));
  return {{v.x, v.y}, {v.z, v.w}};
}

template <int M, typename R>
__device__ __forceinline__ Cx<R> wave_ld(const Cx<R>* p) {
  return M & (kWaveOwn | kWaveEarlier) ? ld(p) : ldl2(p);
}

// FP64 multiply-adds take 63 cycles each, so the four products of a term go to four sums.
struct Acc64 {
  double rr = 0, ii = 0, ri = 0, ir = 0;
  __device__ __forceinline__ void mac(const Cx<double>& a, const Cx<double>& b) {
    rr = fma(a.re, b.re, rr);
    ii = fma(a.im, b.im, ii);
    ri = fma(a.re, b.im, ri);
    ir = fma(a.im, b.re, ir);
  }
  __device__ __forceinline__ void add(const Cx<double>& a) {
    rr += a.re;
    ri += a.im;
  }
  __device__ __forceinline__ Acc<double> sum() const {
    Acc<double> s;
    s.v = {rr - ii, ri + ir};
    return s;
  }
};
template <typename R>
struct WaveAcc : Acc<R> {
  __device__ __forceinline__ Acc<R> sum() const { return *this; }
};
template <>
struct WaveAcc<double> : Acc64 {};

// The sum over the lanes o, o ^ 1, ... of a group of 2^lg lanes.
template <typename R>
__device__ __forceinline__ void lanes_sum(Acc<R>& a, int lg) {
  for (int o = (1 << lg) >> 1; o > 0; o >>= 1) {
    a.v.re += __shfl_xor_sync(0xffffffffu, a.v.re, o);
    a.v.im += __shfl_xor_sync(0xffffffffu, a.v.im, o);
  }
}
__device__ __forceinline__ void lanes_sum(Acc<ff>& a, int lg) {
  for (int o = (1 << lg) >> 1; o > 0; o >>= 1) {
    const float rh = __shfl_xor_sync(0xffffffffu, a.rh, o), rl = __shfl_xor_sync(0xffffffffu, a.rl, o);
    const float ih = __shfl_xor_sync(0xffffffffu, a.ih, o), il = __shfl_xor_sync(0xffffffffu, a.il, o);
    ff_acc(a.rh, a.rl, rh, rl);
    ff_acc(a.ih, a.il, ih, il);
  }
}

// bin_exp of a magnitude given by its bits and 2^n, without FP64 instructions for normal
// numbers (FP64 latency and rate are poor here).
static __device__ __noinline__ int exp_slow(double m) { return bin_exp(m); }
static __device__ __noinline__ double pow2_slow(int n) { return ldexp(1.0, n); }
__device__ __forceinline__ int exp_of_bits(unsigned long long b, double) {
  const int e = (int)(b >> 52);   // non-negative: no sign bit
  return (unsigned)(e - 1) < 2046u ? e - 1022 : exp_slow(bits_to_val<double>(b));
}
__device__ __forceinline__ int exp_of_bits(unsigned long long b, float) {
  const int e = (int)((unsigned)b >> 23);
  return (unsigned)(e - 1) < 254u ? e - 126 : exp_slow((double)bits_to_val<float>(b));
}
__device__ __forceinline__ double pow2_of(int n, double) {
  return (unsigned)(n + 1022) <= 2045u ? __hiloint2double((n + 1023) << 20, 0) : pow2_slow(n);
}
__device__ __forceinline__ float pow2_of(int n, float) {
  return (unsigned)(n + 126) <= 253u ? __int_as_float((n + 127) << 23) : (float)pow2_slow(n);
}

// An output's max-abs: FP64 as bits, without FP64 instructions (0 for NaN, as fmax drops it).
__device__ __forceinline__ unsigned long long mag_key(const Cx<double>& v) {
  const unsigned long long abs = 0x7fffffffffffffffull, inf = 0x7ff0000000000000ull;
  unsigned long long a = (unsigned long long)__double_as_longlong(v.re) & abs,
                     b = (unsigned long long)__double_as_longlong(v.im) & abs;
  a = a > inf ? 0ull : a;
  b = b > inf ? 0ull : b;
  return max(a, b);
}
__device__ __forceinline__ float mag_key(const Cx<float>& v) { return mag(v); }
__device__ __forceinline__ float mag_key(const Cx<ff>& v) { return mag(v); }

// The warp's largest magnitude as bits (integer order = value order; NaN counts as 0, as fmax
// drops it): one or two warp reductions instead of five shuffle steps.
__device__ __forceinline__ unsigned long long warp_max_bits(float v) {
  return __reduce_max_sync(0xffffffffu, v == v ? __float_as_uint(v) : 0u);
}
__device__ __forceinline__ unsigned long long warp_max_bits(unsigned long long b) {
  const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(b >> 32));
  const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(b >> 32) == hi ? (unsigned)b : 0u);
  return (unsigned long long)hi << 32 | lo;
}

// Outputs of lanes [32 chunk, 32 chunk + 32) of the step at `rec`, 2^lanes lanes sharing one
// output's sum over k; returns the warp's max-abs bits.  Warp-synchronous; every k is added in
// order within a lane.  The operands of kWaveK terms are loaded together: one round trip.
template <typename R, int M>
__device__ __forceinline__ unsigned long long wave_outputs(const uint4* rec, unsigned chunk, Cx<R>* arena,
                                                           Meta* meta, int& slot) {
  using S = typename Traits<R>::S;
  const uint4 h0 = rec[0], h1 = rec[1];
  const longlong2 h2 = *(const longlong2*)(rec + 2);
  const long long off_c = *(const long long*)(rec + 3);
  const int sa = (int)h0.x, sb = (int)h0.y;
  slot = (int)h0.z;
  const unsigned Rr = h0.w, N = h1.x, K = h1.y;
  const int nrow = h1.w & 255, nk = (h1.w >> 8) & 255, nn = (h1.w >> 16) & 255, lg = h1.w >> 24;
  const bool hasB = sb >= 0;
  const uint4 *rr = rec + 4, *rk = rr + nrow, *rn = rk + nk;
  const int lane = threadIdx.x & 31;
  // bookkeeping of the operands (read past L1, as they are); a launch of its own first works
  // out its indices, while the launch before it ends
  ulonglong2 ma, mb = make_ulonglong2(0, 0);
  auto load_meta = [&] {
    ma = __ldcg((const ulonglong2*)(meta + sa));
    if (hasB) mb = __ldcg((const ulonglong2*)(meta + sb));
  };
  if (M != kWaveEarlier) load_meta();
  const unsigned q = chunk * 32 + lane, o = q >> lg;
  unsigned k0 = q & ((1u << lg) - 1), kd = 1u << lg;
  bool live = o < Rr * N;
  if (std::is_same<R, float>::value) {   // complex64 keeps its sums in order, bit for bit: one lane each
    live = live && k0 == 0;   // (records made for complex64 alone have one)
    kd = 1;
  }
  WaveAcc<R> part;
  unsigned oa = 0, ob = 0;
  if (live) {
    unsigned r = o, d = 0;
    if (N > 1) {
      const unsigned n = Rr == 1 ? o : (M & kWaveAny) && !h1.z ? o / Rr : __umulhi(o, h1.z);
      r = o - n * Rr;
      wave_offsets<M>(n, rn, nn, d, ob);
    }
    if (nrow) wave_offsets<M>(r, rr, nrow, oa, ob);
  }
  if (M == kWaveEarlier) {
    pdl_wait();
    load_meta();
  }
  if (live) {
    const Cx<R>* A = arena + h2.x + oa;
    const Cx<R>* B = arena + h2.y + ob;
    uint4 w = make_uint4(1, 0, 0, 0);   // one contracted run (or none): constant strides
    if (nk) w = *rk;
#pragma unroll 1
    for (unsigned k = k0; k < K; k += kWaveK * kd) {
      unsigned ka[kWaveK], kb[kWaveK];
#pragma unroll
      for (int u = 0; u < kWaveK; ++u) {
        ka[u] = (k + (unsigned)u * kd) * w.z;
        kb[u] = (k + (unsigned)u * kd) * w.w;
      }
      if (nk > 1) {   // the terms' digits of a run together: one record read, independent chains
        unsigned y[kWaveK];
#pragma unroll
        for (int u = 0; u < kWaveK; ++u) {
          y[u] = min(k + (unsigned)u * kd, K - 1);
          ka[u] = kb[u] = 0;
        }
        uint4 x = w;
#pragma unroll 1
        for (int i = 1; i < nk; x = rk[i++]) {
#pragma unroll
          for (int u = 0; u < kWaveK; ++u) {
            const unsigned t = (M & kWaveAny) && !x.y ? y[u] / x.x : __umulhi(y[u], x.y), d = y[u] - t * x.x;
            ka[u] += d * x.z;
            kb[u] += d * x.w;
            y[u] = t;
          }
        }
#pragma unroll
        for (int u = 0; u < kWaveK; ++u) {
          ka[u] += y[u] * x.z;
          kb[u] += y[u] * x.w;
        }
      }
      Cx<R> a[kWaveK], b[kWaveK];
#pragma unroll
      for (int u = 0; u < kWaveK; ++u)
        if (k + (unsigned)u * kd < K) {
          a[u] = wave_ld<M>(A + ka[u]);
          if (hasB) b[u] = wave_ld<M>(B + kb[u]);
        }
#pragma unroll
      for (int u = 0; u < kWaveK; ++u)
        if (k + (unsigned)u * kd < K) {
          if (hasB)
            part.mac(a[u], b[u]);
          else
            part.add(a[u]);
        }
    }
  }
  Acc<R> acc = part.sum();
  if (kd > 1) lanes_sum(acc, lg);
  const int ea = exp_of_bits(ma.x, S()), eb = hasB ? exp_of_bits(mb.x, S()) : 0;
  if (chunk == 0 && lane == 0)
    meta[slot].exp = (long long)ma.y + (long long)mb.y + ea + eb;
  decltype(mag_key(Cx<R>())) vmax = 0;
  if (live && k0 == 0) {
    const Cx<R> v = acc.get(pow2_of(-(ea + eb), S()));
    st(arena + off_c + o, v);   // C is [n, r] with r innermost: o = r + n R
    vmax = mag_key(v);
  }
  return warp_max_bits(vmax);
}

// The levels of one stage by one cluster of CTAs (its whole grid); the warps of the cluster
// share a level's items, a cluster barrier stands between levels.  Each CTA first copies the
// stage's records, items and level table to shared memory (`smem` bytes; 0: they do not fit
// and are read where they are), so that a level's chain of dependent memory reads is one
// round trip to L2: the operands and their bookkeeping.  Results go to L2 (stores and
// atomics) and are read from there past L1; the barrier's release and acquire order them.
template <class F>   // F(record, chunk): one item by the calling warp
__device__ __forceinline__ void wave_walk(const unsigned char* blob, const WaveRange& rg, int n_lev, int smem, F&& item) {
  extern __shared__ __align__(16) unsigned char wsm[];
  pdl_next();
  const unsigned char *recs = blob, *items = blob + rg.item - rg.item0 * sizeof(WaveItem);
  const unsigned* lev = (const unsigned*)(blob + rg.lev);
  if (smem) {
    const int nr = rg.rec_bytes, ni = rg.item_bytes, nl = rg.lev_bytes;   // multiples of 16
    for (int i = threadIdx.x * 16; i < nr + ni + nl; i += blockDim.x * 16) {
      const unsigned src = i < nr ? rg.rec + i : i < nr + ni ? rg.item + (i - nr) : rg.lev + (i - nr - ni);
      tc::cp_async16(tc::smem_u32(wsm + i), blob + src);
    }
    tc::cp_async_wait();
    __syncthreads();
    recs = wsm - rg.rec;
    items = wsm + nr - rg.item0 * sizeof(WaveItem);
    lev = (const unsigned*)(wsm + nr + ni);
  }
  lev += rg.lev0;
  pdl_wait();   // the records are constant: copied while the launch before ends
  const unsigned w0 = blockIdx.x + gridDim.x * (threadIdx.x >> 5);   // consecutive items on different CTAs
  const unsigned nw = gridDim.x * kWaveCtaWarps;
  for (int l = 0; l < n_lev; ++l) {
    const unsigned end = lev[l + 1];
    for (unsigned i = lev[l] + w0; i < end; i += nw) {
      const uint2 it = ((const uint2*)items)[i];
      item((const uint4*)recs + it.x, it.y);
    }
    if (l + 1 == n_lev) break;
    if (gridDim.x == 1)
      __syncthreads();
    else
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

template <typename R, int M>   // kWaveOwn: a single CTA
__global__ void __launch_bounds__(32 * kWaveCtaWarps)
    k_waves(const unsigned char* __restrict__ blob, WaveRange rg, int n_lev, int smem, Cx<R>* arena, Meta* meta) {
  wave_walk(blob, rg, n_lev, smem, [&](const uint4* rec, unsigned chunk) {
    int slot;
    const unsigned long long v = wave_outputs<R, M>(rec, chunk, arena, meta, slot);
    if ((threadIdx.x & 31) == 0 && v) atomicMax(&meta[slot].maxbits, v);
  });
}

// One level over the whole GPU, a warp per item; one atomic per CTA where its warps work on
// one step (a large step has thousands of warps).
template <typename R>
__global__ void __launch_bounds__(256)
    k_wave_wide(const unsigned char* __restrict__ blob, WaveRange rg, unsigned first, unsigned n_items,
                Cx<R>* arena, Meta* meta) {
  __shared__ unsigned long long red[8];
  __shared__ int slots[8];
  pdl_next();
  const unsigned w = threadIdx.x >> 5, i = blockIdx.x * (blockDim.x >> 5) + w;
  int slot = -1;
  unsigned long long v = 0;
  if (i >= n_items) {
    pdl_wait();
  } else {
    const uint2 it = __ldg((const uint2*)(blob + rg.item) + first + i);
    v = wave_outputs<R, kWaveEarlier>((const uint4*)blob + it.x, it.y, arena, meta, slot);
  }
  if ((threadIdx.x & 31) == 0) {
    red[w] = v;
    slots[w] = slot;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long m = red[0];
    for (unsigned j = 1; j <= blockDim.x >> 5; ++j) {
      if (j < blockDim.x >> 5 && slots[j] == slots[j - 1]) {
        m = max(m, red[j]);
        continue;
      }
      if (m) atomicMax(&meta[slots[j - 1]].maxbits, m);
      if (j < blockDim.x >> 5) m = red[j];
    }
  }
}

// Launches `fn` on `stream`; pdl: it may start while the launch before it still runs (every
// kernel calls pdl_wait); cluster > 1: CTAs per cluster.
template <typename... P, typename... A>
cudaError_t launch_kernel(void (*fn)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t stream, bool pdl,
                          unsigned cluster, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at[2];
  if (pdl) {
    at[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (cluster > 1) {
    at[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    at[cfg.numAttrs].val.clusterDim.x = cluster;
    at[cfg.numAttrs].val.clusterDim.y = 1;
    at[cfg.numAttrs++].val.clusterDim.z = 1;
  }
  cfg.attrs = at;
  return cudaLaunchKernelEx(&cfg, fn, static_cast<P>(args)...);
}

// Launches a FUSED stage as one cluster; fn: a level kernel (blob, range, levels, smem, args).
constexpr uint32_t kWaveSmem = 100 * 1024;   // its records in shared memory: two CTAs per SM
template <typename F, typename... A>
cudaError_t launch_cluster(const WaveStage& g, const unsigned char* blob, cudaStream_t stream, bool pdl, F fn, A... args) {
  const uint32_t prog = g.range.rec_bytes + g.range.item_bytes + g.range.lev_bytes;
  const int smem = prog <= kWaveSmem ? (int)prog : 0;
  return launch_kernel(fn, dim3((unsigned)g.ctas), 32 * kWaveCtaWarps, (size_t)smem, stream, pdl, (unsigned)g.ctas, blob,
                       g.range, (int)g.units, smem, args...);
}

}  // namespace pk
