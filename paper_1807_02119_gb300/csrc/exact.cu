// Exact evaluation: Z(q) modulo word-size primes, on the GPU.
//
// At integer q the Potts t(q) is a root of x^2 - (q - 2) x + 1, and with the standard
// weights every clause entry is an integer polynomial in t (off-diagonal 1, diagonal
// (-1)^mult t^-signsum, t^-1 = (q - 2) - t).  Z(q) is therefore an element a + b t of
// Z[t]/(t^2 - (q - 2) t + 1).  The same plan (network, order, slicing, step records) is
// contracted in F_p[t]/(t^2 - (q - 2) t + 1) for a prime p < 2^31: an element is a pair
// of residues (a, b), stored where a complex64 value would be (8 bytes), and
//     (a + b t)(c + d t) = (ac - bd) + (ad + bc + (q - 2) bd) t.
// Several primes determine Z(q), or quantities derived from it, by the Chinese remainder
// theorem.  No rescaling is needed: the arithmetic is exact.
//
// The kernels mirror the floating-point ones in their indexing only: the initial tensors
// follow their recipes (sum over the vertex spin of products of COPY legs and clause
// entries), every contraction step is C[n R + r] = sum_k A[row r, k] B[k, column n] through
// the step's stride runs, light steps level by level (wave_plan.cpp), and the slice results are
// summed.  What bounded it were 64-bit divisions, four per term, and a thread per output however
// long the sum: products now add up below p 2^31 with one conditional subtraction each and are
// reduced once per output, and a warp or a CTA shares a long sum.  Measured on GB300, 36 crossings
// at q = 10 modulo four primes (perf/cases.py): 4589 -> 340 us per call.
#include <cuda_runtime.h>

#include <algorithm>

#include "exact_ring.h"
#include "handles.h"
#include "pk_internal.h"
#include "kernels.cuh"
#include "gemm_tc.cuh"
#include "wave.cuh"

namespace pk {
namespace exact {

// Initial tensor blockIdx.y of one slice: entry e = sum_s prod_j f_j(s, x_j), with f_j a
// COPY leg [s = x_j] or an absorbed clause matrix (diagonal (-1)^mult t^-signsum when
// s = x_j, off-diagonal 1), x_j the entry's digit at the slot's position or the slice's
// fixed value of a sliced index.
__global__ void __launch_bounds__(256) k_exact_build(const Recipe* rec, const Slot* slots,
                                                     const int64_t* offs, E* arena, int q, Ring ring, long long slice, int n_sliced) {
  const Recipe R = rec[blockIdx.y];
  int sdig[64];
  {
    long long s = slice;
    for (int i = 0; i < n_sliced && i < 64; ++i) {
      sdig[i] = (int)(s % q);
      s /= q;
    }
  }
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < R.elems;
       e += (long long)gridDim.x * blockDim.x) {
    E v{0, 0};
    if (R.kind == 1) {
      v = E{1, 0};
    } else {
      for (int s = 0; s < q; ++s) {
        E pr{1, 0};
        bool zero = false;
        for (int j = 0; j < R.nslot; ++j) {
          const Slot sl = slots[R.slot0 + j];
          int x;
          if (sl.dimpos >= 0) {
            long long t = e;
            for (int d = 0; d < sl.dimpos; ++d) t /= q;
            x = (int)(t % q);
          } else {
            x = sdig[sl.slice_ord];
          }
          if (sl.absorbed) {
            if (s == x) {
              int32_t mult, signsum;
              slot_exact_unpack(sl.pad, mult, signsum);
              E dg = epow_t(-(long long)signsum, ring);
              if (mult & 1) dg = eneg(dg, ring);
              pr = emul(pr, dg, ring);
            }
          } else if (s != x) {
            zero = true;
            break;
          }
        }
        if (!zero) v = eadd(v, pr, ring);
      }
    }
    arena[offs[blockIdx.y] + e] = v;
  }
}

// Sums of products modulo p without a division per term: every sum stays below p 2^31, so a
// product (below p^2 < p 2^31) can be added and the excess subtracted in 63 bits.
struct Sums {
  uint64_t ac = 0, bd = 0, x = 0;   // sum of a c, of b d, of a d + b c
  __device__ __forceinline__ static void add(uint64_t& s, uint64_t t, uint64_t lim) {
    s += t;
    s -= s >= lim ? lim : 0;
  }
  __device__ __forceinline__ void mac(uint2 u, uint2 v, uint64_t lim) {
    add(ac, (uint64_t)u.x * v.x, lim);
    add(bd, (uint64_t)u.y * v.y, lim);
    add(x, (uint64_t)u.x * v.y, lim);
    add(x, (uint64_t)u.y * v.x, lim);
  }
  __device__ __forceinline__ void plus(uint2 u) {   // at most 2^31 terms below 2^31
    ac += u.x;
    x += u.y;
  }
  __device__ __forceinline__ E get(Ring r) const {
    const uint32_t b = redm(bd, r);
    return {subm(redm(ac, r), b, r.p), addm(redm(x, r), redm((uint64_t)r.qm2 * b, r), r.p)};
  }
};

__device__ __forceinline__ E lanes_add(E v, int lanes, Ring r) {
  for (int o = lanes >> 1; o > 0; o >>= 1) {
    const E w{__shfl_xor_sync(0xffffffffu, v.a, o), __shfl_xor_sync(0xffffffffu, v.b, o)};
    v = eadd(v, w, r);
  }
  return v;
}

// Outputs of lanes [32 chunk, 32 chunk + 32) of a light step (record as in wave.cuh): 2^lanes
// lanes share an output's sum.  Bound, as there, by one warp's chain of instructions.
__device__ __forceinline__ void exact_outputs(const uint4* rec, unsigned chunk, E* arena, const Ring& ring) {
  const uint4 h0 = rec[0], h1 = rec[1];
  const longlong2 h2 = *(const longlong2*)(rec + 2);
  const long long off_c = *(const long long*)(rec + 3);
  const unsigned Rr = h0.w, N = h1.x, K = h1.y;
  const int nrow = h1.w & 255, nk = (h1.w >> 8) & 255, nn = (h1.w >> 16) & 255, lg = h1.w >> 24;
  const bool hasB = (int)h0.y >= 0;
  const uint4 *rr = rec + 4, *rk = rr + nrow, *rn = rk + nk;
  const unsigned q = chunk * 32 + (threadIdx.x & 31), o = q >> lg, k0 = q & ((1u << lg) - 1);
  const uint64_t lim = (uint64_t)ring.p << 31;
  Sums acc;
  if (o < Rr * N) {
    unsigned r = o, oa = 0, ob = 0, d = 0;
    if (N > 1) {
      const unsigned n = Rr == 1 ? o : __umulhi(o, h1.z);
      r = o - n * Rr;
      wave_offsets(n, rn, nn, d, ob);
    }
    if (nrow) wave_offsets(r, rr, nrow, oa, ob);
    const uint2* A = (const uint2*)(arena + h2.x) + oa;
    const uint2* B = (const uint2*)(arena + h2.y) + ob;
    uint4 w = make_uint4(1, 0, 0, 0);   // one contracted run (or none): constant strides
    if (nk) w = *rk;
#pragma unroll 1
    for (unsigned k = k0; k < K; k += kWaveK << lg) {
      uint2 a[kWaveK], b[kWaveK];
#pragma unroll
      for (int u = 0; u < kWaveK; ++u) {
        const unsigned ku = k + ((unsigned)u << lg);
        uint2 f = make_uint2(ku * w.z, ku * w.w);
        if (nk > 1) {
          f = make_uint2(0, 0);
          wave_offsets(min(ku, K - 1), rk, nk, f.x, f.y);
        }
        a[u] = make_uint2(0, 0);
        b[u] = make_uint2(1, 0);   // without B: the constant 1
        if (ku < K) {
          a[u] = __ldcg(A + f.x);
          if (hasB) b[u] = __ldcg(B + f.y);
        }
      }
#pragma unroll
      for (int u = 0; u < kWaveK; ++u) acc.mac(a[u], b[u], lim);
    }
  }
  const E v = lanes_add(acc.get(ring), 1 << lg, ring);
  if (o < Rr * N && k0 == 0) arena[off_c + o] = v;
}

__global__ void __launch_bounds__(32 * kWaveCtaWarps)
    k_exact_waves(const unsigned char* __restrict__ blob, WaveRange rg, int n_lev, int smem, E* arena, Ring ring) {
  wave_walk(blob, rg, n_lev, smem, [&](const uint4* rec, unsigned chunk) { exact_outputs(rec, chunk, arena, ring); });
}
__global__ void __launch_bounds__(256)
    k_exact_wide(const unsigned char* __restrict__ blob, WaveRange rg, unsigned first, unsigned n_items, E* arena, Ring ring) {
  pdl_next();
  const unsigned i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  pdl_wait();
  if (i >= n_items) return;
  const uint2 it = __ldg((const uint2*)(blob + rg.item) + first + i);
  exact_outputs((const uint4*)blob + it.x, it.y, arena, ring);
}

// A heavy step: T threads of a CTA of 256 per output o = n R + r; a table of the contracted
// index's offsets in shared memory when it fits (kTab entries), else decoded per term.
constexpr int kTab = 2048;
template <int T>
__global__ void __launch_bounds__(256) k_exact_step(const Step s, E* arena, Ring ring) {
  __shared__ uint2 tab[kTab];
  __shared__ E red[8];
  pdl_wait();
  const bool in_tab = s.K <= kTab;
  if (in_tab)
    for (unsigned k = threadIdx.x; k < (unsigned)s.K; k += 256) {
      long long ka, kb;
      split_runs32(k, s.kr, s.nk, ka, kb);
      tab[k] = make_uint2((unsigned)ka, (unsigned)kb);
    }
  __syncthreads();
  const bool hasB = s.b >= 0;
  const unsigned R = (unsigned)s.R, total = (unsigned)(s.R * s.N), K = (unsigned)s.K, t = threadIdx.x % T;
  const uint64_t lim = (uint64_t)ring.p << 31;
  // CTA-uniform bounds: the reductions below take every thread
  for (unsigned o0 = blockIdx.x * (256 / T); o0 < total; o0 += gridDim.x * (256 / T)) {
    const unsigned o = o0 + threadIdx.x / T;
    Sums acc;
    if (o < total) {
      const unsigned n = o / R, r = o - n * R;
      long long oa, ob, nb = 0, dummy;
      split_runs32(r, s.row, s.nrow, oa, ob);
      split_runs32(n, s.nr, s.nn, dummy, nb);
      const uint2* A = (const uint2*)(arena + s.off_a) + oa;
      const uint2* B = (const uint2*)(arena + s.off_b) + (hasB ? ob + nb : 0);
#pragma unroll 4
      for (unsigned k = t; k < K; k += T) {
        uint2 off;
        if (in_tab) {
          off = tab[k];
        } else {
          long long ka, kb;
          split_runs32(k, s.kr, s.nk, ka, kb);
          off = make_uint2((unsigned)ka, (unsigned)kb);
        }
        if (hasB)
          acc.mac(A[off.x], B[off.y], lim);
        else
          acc.plus(A[off.x]);
      }
    }
    E v = acc.get(ring);
    if (T > 1) v = lanes_add(v, T < 32 ? T : 32, ring);
    if (T == 256) {
      if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
      __syncthreads();
      if (threadIdx.x == 0)
        for (int i = 1; i < 8; ++i) v = eadd(v, red[i], ring);
      __syncthreads();
    }
    if (o < total && t == 0) arena[s.off_c + o] = v;
  }
}

// Slice result: the final (rank-0) tensor added into the running sum.
__global__ void k_exact_accum(const E* arena, long long off_final, E* sum, Ring ring) {
  if (threadIdx.x == 0 && blockIdx.x == 0) *sum = eadd(*sum, arena[off_final], ring);
}

}  // namespace exact

// Z(q) of plan `p` modulo `prime` (before the host's loop factor), left in *d_sum as
// (a, b): every slice's initial tensors, steps and result, in the plan's own order.  The
// program must be uploaded (pk_upload) in `ws`; the arena is the complex64 one.
cudaError_t launch_exact(const Plan& p, uint32_t prime, void* ws, void* arena, void* d_sum,
                         cudaStream_t stream) {
  using namespace exact;
  char* base = (char*)ws;
  E* ar = (E*)arena;
  E* sum = (E*)d_sum;
  const WaveProgram& w = p.wave[kWaveExact];
  const unsigned char* blob = (const unsigned char*)base + p.off_wave[kWaveExact];
  const Ring ring = make_ring(prime, p.q);
  cudaError_t e = cudaMemsetAsync(sum, 0, sizeof(E), stream);
  if (e != cudaSuccess) return e;
  if (p.n_init > 65535) return cudaErrorInvalidValue;
  e = cudaFuncSetAttribute(k_exact_waves, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWaveSmem);
  if (e != cudaSuccess) return e;
  int64_t maxel = 1;
  for (const auto& r : p.recipes) maxel = std::max<int64_t>(maxel, r.elems);
  const unsigned bx = (unsigned)std::min<int64_t>((maxel + 255) / 256, 1024);
  for (long long sl = 0; sl < p.n_slices; ++sl) {
    if (p.n_init > 0)
      k_exact_build<<<dim3(bx, (unsigned)p.n_init), 256, 0, stream>>>(
          (const Recipe*)(base + p.off_recipe), (const Slot*)(base + p.off_slots),
          (const int64_t*)(blob + w.init_off), ar, p.q, ring, sl, (int)p.sliced.size());
    for (const WaveStage& g : w.stages[0]) {
      if (g.kind == WaveStage::FUSED) {
        if ((e = launch_cluster(g, blob, stream, true, k_exact_waves, ar, ring)) != cudaSuccess) return e;
      } else if (g.kind == WaveStage::WIDE) {
        const int64_t wpb = std::max<int64_t>(1, std::min<int64_t>(8, g.items / 304));
        launch_kernel(k_exact_wide, dim3((unsigned)((g.items + wpb - 1) / wpb)), 32 * (unsigned)wpb, 0, stream, true, 1,
                      blob, g.range, g.first, (unsigned)g.items, ar, ring);
      } else {
        Step st = p.steps[g.step];
        st.off_a = w.off[st.a];
        st.off_b = st.b >= 0 ? w.off[st.b] : 0;
        st.off_c = w.off[st.c];
        // threads per output: while the outputs alone leave the GPU short of threads
        const long long outs = st.R * st.N;
        const int T = st.K >= 1024 && outs <= 152 * 32 ? 256 : st.K >= 64 && outs <= 152 * 512 ? 32 : 1;
        const unsigned grid = (unsigned)std::max<long long>(1, std::min<long long>((outs * T + 255) / 256, 152 * 16));
        launch_kernel(T == 256 ? k_exact_step<256> : T == 32 ? k_exact_step<32> : k_exact_step<1>, dim3(grid), 256, 0,
                      stream, true, 1, st, ar, ring);
      }
    }
    k_exact_accum<<<1, 32, 0, stream>>>(ar, w.off[p.final_tensor], sum, ring);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace pk
