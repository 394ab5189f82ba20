// Batched evaluation: many knots (each with its own plan) in one persistent launch.
//
// Every CTA repeatedly takes the next knot from an atomic work counter (the most work first)
// and performs that knot's whole contraction itself: initial tensors (a part of a warp per
// tensor), then the plan's levels with the CTA's warps spread over a level's outputs and a
// block barrier between levels (records and code as in wave.cuh), then the slice scalar.  Clusters
// of eight CTAs take the largest knots so; beyond its cluster no CTA waits for another.  The launch (preceded by a reset of the counter) is recorded
// once into a CUDA graph and replayed.  What bounds it is the chain of levels of the largest
// knots: 10 to 25 levels of about 1.5 us, where one step after another took 120 times 10 us.
// Measured on GB300, per launch: 1024 knots of 20 to 120 crossings at q = 3 in split 1.80 ->
// 0.54 ms, 192 of 20 to 60 at q = 5 in complex128 1.20 -> 0.40 ms (one CTA per knot for all of
// them: 0.71 and 1.40 ms; everything above half a CTA's share in clusters: 0.67 and 0.57 ms).
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "handles.h"
#include "kernels.cuh"
#include "gemm_tc.cuh"
#include "wave.cuh"

namespace pk {

// Per-knot header of the batch image (all offsets relative to the batch arrays).
struct BatchKnot {
  int64_t recipe0, n_recipe;   // recipes of the knot
  int64_t slot_base;           // added to Recipe::slot0
  int64_t blob;                // the knot's level records in the record array (bytes)
  int64_t arena_off;           // first arena element of the knot
  int64_t meta_off;            // first bookkeeping slot of the knot
  int64_t n_slices;
  int64_t final_offset;        // final tensor (arena elements, relative)
  int32_t n_sliced, q, final_tensor, n_meta;
  int32_t n_lev, blob_bytes, item, lev;   // levels; bytes of the records; items and level table in them
};

namespace {

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// The knots order[first .. last), most work first.  CL = 1: each by one CTA (T threads), taken
// from the work counter.  CL > 1: each by a cluster of CL CTAs, for the knots that would keep
// one CTA busy long after the others are done; cluster c takes every (number of clusters)-th.
// A knot's records are copied to shared memory when they fit `smem` bytes.
template <typename R, int T, int CL>
__global__ void __launch_bounds__(T) k_batch(const BatchKnot* __restrict__ knots, const int* __restrict__ order,
                                             int first, int last, const Recipe* recs, const Slot* slots,
                                             const unsigned char* blobs, Cx<R>* arena,
                                             Meta* meta_all, SliceResult* out, unsigned* next, int smem) {
  using S = typename Traits<R>::S;
  constexpr int kMode = (CL == 1 ? kWaveOwn : kWaveL2) | kWaveAny;
  extern __shared__ __align__(16) unsigned char bsm[];
  __shared__ int kn_s;
  const int rank = CL == 1 ? 0 : (int)cluster_rank();
  const int lane = threadIdx.x & 31, tid = rank * T + threadIdx.x, threads = CL * T;
  // consecutive items of a level on different CTAs
  const int warp = rank + CL * (threadIdx.x >> 5), nwarps = threads / 32;
  auto sync = [] {
    if (CL == 1)
      __syncthreads();
    else
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  };
  for (int turn = first + (int)(blockIdx.x / CL);; turn += (int)(gridDim.x / CL)) {
    __syncthreads();
    if (CL == 1) {
      if (threadIdx.x == 0) kn_s = first + (int)atomicAdd(next, 1u);
      __syncthreads();
      turn = kn_s;
    }
    if (turn >= last) return;
    const int kn = order[turn];
    const BatchKnot K = knots[kn];
    const unsigned char* blob = blobs + K.blob;
    if (K.blob_bytes <= smem) {
      for (int i = threadIdx.x * 16; i < K.blob_bytes; i += T * 16) tc::cp_async16(tc::smem_u32(bsm + i), blob + i);
      tc::cp_async_wait();   // read after the barrier below
      blob = bsm;
    }
    Cx<R>* A0 = arena + K.arena_off;
    Meta* meta = meta_all + K.meta_off;
    double tre = 0, tim = 0;
    long long texp = LLONG_MIN;
    for (long long sl = 0; sl < K.n_slices; ++sl) {
      int sdig[64];
      {
        long long t = sl;
        for (int i = 0; i < K.n_sliced && i < 64; ++i) {
          sdig[i] = (int)(t % K.q);
          t /= K.q;
        }
      }
      for (int i = (int)K.n_recipe + tid; i < K.n_meta; i += threads) meta[i].maxbits = 0;
      // initial tensors: `part` lanes (a power of two up to a warp) per tensor
      int part = 1;
      while (part < 32 && part < K.q * K.q) part *= 2;
      for (long long j0 = (long long)warp * (32 / part); j0 < K.n_recipe; j0 += (long long)nwarps * (32 / part)) {
        const long long j = j0 + lane / part;
        S vmax = 0;
        Recipe r;
        if (j < K.n_recipe) {
          r = recs[K.recipe0 + j];
          for (long long e = lane & (part - 1); e < r.elems; e += part) {
            double re, im;
            recipe_value(r, slots + K.slot_base, e, K.q, sdig, re, im);
            const Cx<R> v{from_double<R>(re), from_double<R>(im)};
            st(A0 + r.offset + e, v);
            vmax = fmax(vmax, mag(v));
          }
        }
        for (int o = part >> 1; o > 0; o >>= 1) vmax = fmax(vmax, __shfl_xor_sync(0xffffffffu, vmax, o));
        if (j < K.n_recipe && (lane & (part - 1)) == 0) {
          meta[r.meta].maxbits = max_bits(vmax);
          meta[r.meta].exp = r.exp2;
        }
      }
      sync();
      const unsigned* lev = (const unsigned*)(blob + K.lev);
      for (int l = 0; l < K.n_lev; ++l) {
        const unsigned end = lev[l + 1];
        for (unsigned i = lev[l] + warp; i < end; i += nwarps) {
          const uint2 it = ((const uint2*)(blob + K.item))[i];
          const uint4* rec = (const uint4*)blob + it.x;
          const unsigned per = rec[3].z;   // WaveRec::per
          unsigned long long m = 0;
          int slot = 0;
          for (unsigned c = 0; c < per; ++c)
            m = max(m, wave_outputs<R, kMode>(rec, it.y * per + c, A0, meta, slot));
          if (lane == 0 && m) atomicMax(&meta[slot].maxbits, m);
        }
        sync();
      }
      if (tid == 0) {  // add this slice's scalar at a common exponent
        const Cx<R> v = ldl2(A0 + K.final_offset);
        double vr = to_double(v.re), vi = to_double(v.im);
        long long ve = __ldcg(&meta[K.final_tensor].exp);
        double m = fmax(fabs(vr), fabs(vi));
        if (m > 0) {
          int k;
          frexp(m, &k);
          vr = ldexp(vr, -k);
          vi = ldexp(vi, -k);
          ve += k;
          if (texp == LLONG_MIN) {
            tre = vr;
            tim = vi;
            texp = ve;
          } else {
            const long long e = max(texp, ve);
            const long long da = max(texp - e, -2000LL), db = max(ve - e, -2000LL);
            tre = ldexp(tre, (int)da) + ldexp(vr, (int)db);
            tim = ldexp(tim, (int)da) + ldexp(vi, (int)db);
            texp = e;
          }
        }
      }
      sync();
    }
    if (tid == 0) {
      out[kn].re = tre;
      out[kn].im = tim;
      out[kn].exp = texp == LLONG_MIN ? 0 : texp;
    }
  }
}

constexpr int kCl = 8, kClThreads = 512;   // CTAs of a cluster, threads of each

uint64_t a256(uint64_t x) { return (x + 255) & ~uint64_t(255); }

}  // namespace
}  // namespace pk

struct pk_batch {
  int32_t precision = 0;
  int32_t n = 0;
  std::vector<pk::BatchKnot> knots;
  std::vector<pk::Recipe> recipes;
  std::vector<pk::Slot> slots;
  std::vector<uint8_t> blobs;          // every knot's level records
  std::vector<int32_t> order;          // knots by decreasing work
  std::vector<pk::Knot> kinfo;
  std::vector<pk::Scaled> factor, prefactor;   // of Z (folded loops), and A(q)
  std::vector<int32_t> qs;
  uint64_t off_knots = 0, off_recipes = 0, off_slots = 0, off_order = 0, off_blobs = 0, off_meta = 0,
           off_results = 0, off_counter = 0, off_arena = 0, total = 0, image_bytes = 0;
  std::vector<uint8_t> image;
  uint8_t* pinned = nullptr;
  pk::SliceResult* pinned_results = nullptr;
  void* graph_ws = nullptr;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  int32_t device = -1;
  int32_t n_big = 0;                   // knots run by clusters (the first of `order`)
  int32_t threads = 256, smem = 0;      // launch shape (the context's tuning at creation)
};

namespace {

pk_status bfail(pk_ctx* c, pk_status s, const std::string& m) {
  if (c) c->err = m;
  return s;
}

template <typename R>
void* batch_kernel(int threads, bool cluster) {
  if (cluster) return (void*)pk::k_batch<R, pk::kClThreads, pk::kCl>;
  if (threads == 128) return (void*)pk::k_batch<R, 128, 1>;
  if (threads == 512) return (void*)pk::k_batch<R, 512, 1>;
  return (void*)pk::k_batch<R, 256, 1>;
}
void* batch_kernel(int32_t precision, int threads, bool cluster) {
  return precision == PK_C128 ? batch_kernel<double>(threads, cluster)
         : precision == PK_C64 ? batch_kernel<float>(threads, cluster)
                               : batch_kernel<pk::ff>(threads, cluster);
}

cudaError_t build_graph(pk_batch* b, void* ws, cudaStream_t stream) {
  (void)stream;
  if (b->exec && b->graph_ws == ws) return cudaSuccess;
  if (b->exec) {
    cudaGraphExecDestroy(b->exec);
    b->exec = nullptr;
  }
  if (b->graph) {
    cudaGraphDestroy(b->graph);
    b->graph = nullptr;
  }
  char* base = (char*)ws;
  cudaError_t e = cudaGraphCreate(&b->graph, 0);
  if (e != cudaSuccess) return e;
  cudaMemsetParams mp;
  std::memset(&mp, 0, sizeof(mp));
  mp.dst = base + b->off_counter;
  mp.value = 0;
  mp.elementSize = 4;
  mp.width = 1;
  mp.height = 1;
  cudaGraphNode_t memset_node;
  e = cudaGraphAddMemsetNode(&memset_node, b->graph, nullptr, 0, &mp);
  if (e != cudaSuccess) return e;
  const pk::BatchKnot* knots = (const pk::BatchKnot*)(base + b->off_knots);
  const pk::Recipe* recs = (const pk::Recipe*)(base + b->off_recipes);
  const pk::Slot* slots = (const pk::Slot*)(base + b->off_slots);
  const int* order = (const int*)(base + b->off_order);
  const unsigned char* blobs = (const unsigned char*)(base + b->off_blobs);
  void* arena = base + b->off_arena;
  pk::Meta* meta = (pk::Meta*)(base + b->off_meta);
  pk::SliceResult* res = (pk::SliceResult*)(base + b->off_results);
  unsigned* counter = (unsigned*)(base + b->off_counter);
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, b->device);
  // two independent launches: the knots of the most work by clusters, the others a CTA each
  for (int big = 1; big >= 0; --big) {
    int first = big ? 0 : b->n_big, last = big ? b->n_big : b->n;
    if (last <= first) continue;
    void* func = batch_kernel(b->precision, b->threads, big != 0);
    const size_t smem = (size_t)b->smem;
    e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int records = b->smem, per_sm = 0;
    const int threads = big ? pk::kClThreads : b->threads;
    void* args[] = {&knots, &order, &first, &last, &recs, &slots, &blobs, &arena, &meta, &res, &counter, &records};
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, func, threads, smem);
    if (e != cudaSuccess) return e;
    cudaKernelNodeParams kp;
    std::memset(&kp, 0, sizeof(kp));
    kp.func = func;
    kp.gridDim = dim3((unsigned)(big ? pk::kCl * std::min(sms / pk::kCl, last - first)
                                     : std::max(1, std::min(per_sm * sms, last - first))));
    kp.blockDim = dim3((unsigned)threads);
    kp.sharedMemBytes = (unsigned)smem;
    kp.kernelParams = args;
    cudaGraphNode_t node;
    e = cudaGraphAddKernelNode(&node, b->graph, &memset_node, 1, &kp);
    if (e == cudaSuccess && big) {
      cudaLaunchAttributeValue v;
      std::memset(&v, 0, sizeof(v));
      v.clusterDim.x = pk::kCl;
      v.clusterDim.y = v.clusterDim.z = 1;
      e = cudaGraphKernelNodeSetAttribute(node, cudaLaunchAttributeClusterDimension, &v);
    }
    if (e != cudaSuccess) return e;
  }
  e = cudaGraphInstantiate(&b->exec, b->graph, 0);
  if (e != cudaSuccess) return e;
  b->graph_ws = ws;
  return cudaSuccess;
}

}  // namespace

extern "C" {

pk_status pk_batch_create(pk_ctx* ctx, const pk_plan* const* plans, int32_t n, int32_t precision,
                          pk_batch** out) {
  if (!out || (n > 0 && !plans) || n < 0) return bfail(ctx, PK_EINVAL, "bad argument");
  if (precision != PK_C128 && precision != PK_C64 && precision != PK_SPLIT)
    return bfail(ctx, PK_EINVAL, "bad precision");
  *out = nullptr;
  pk_batch* b = new (std::nothrow) pk_batch();
  if (!b) return bfail(ctx, PK_ENOMEM, "out of host memory");
  b->precision = precision;
  b->n = n;
  b->device = ctx ? ctx->device : -1;
  b->threads = ctx ? ctx->tuning.batch_threads : kTunedDefault.batch_threads;
  b->smem = 32 * (ctx ? ctx->tuning.batch_ktab : kTunedDefault.batch_ktab);
  int64_t arena = 0, meta = 0;
  std::vector<uint8_t> blob;
  std::vector<double> work;
  for (int32_t i = 0; i < n; ++i) {
    if (!plans[i]) {
      delete b;
      return bfail(ctx, PK_EINVAL, "null plan");
    }
    const pk::Plan& P = plans[i]->p;
    pk::BatchKnot k;
    std::memset(&k, 0, sizeof(k));
    k.recipe0 = (int64_t)b->recipes.size();
    k.n_recipe = (int64_t)P.recipes.size();
    k.slot_base = (int64_t)b->slots.size();
    pk::WaveRange rg;
    k.n_lev = pk::wave_batch(P, precision != PK_C64, blob, rg);
    k.blob = (int64_t)b->blobs.size();
    k.blob_bytes = (int32_t)blob.size();
    k.item = (int32_t)rg.item;
    k.lev = (int32_t)rg.lev;
    k.n_meta = (int32_t)P.tensors.size();
    b->blobs.insert(b->blobs.end(), blob.begin(), blob.end());
    work.push_back(P.cmacs);
    k.arena_off = arena;
    k.meta_off = meta;
    k.n_slices = P.n_slices;
    k.final_offset = P.wave[PK_C64].off[P.final_tensor];
    k.n_sliced = (int32_t)P.sliced.size();
    k.q = P.q;
    k.final_tensor = P.final_tensor;
    b->knots.push_back(k);
    for (int32_t j = 0; j < P.n_init; ++j) {
      b->recipes.push_back(P.recipes[j]);
      b->recipes.back().offset = P.wave[PK_C64].off[j];
    }
    b->slots.insert(b->slots.end(), P.slots.begin(), P.slots.end());
    b->kinfo.push_back(P.knot);
    b->factor.push_back(P.factor);
    b->prefactor.push_back(pk::jones_defined(P.knot) ? pk::jones_prefactor(P.knot, P.q) : pk::Scaled());
    b->qs.push_back(P.q);
    arena += (P.wave[PK_C64].arena_elems + 63) / 64 * 64;
    meta += (int64_t)P.tensors.size();
  }
  // the most work first: the launch ends with the small knots
  b->order.resize((size_t)n);
  for (int32_t i = 0; i < n; ++i) b->order[i] = i;
  std::stable_sort(b->order.begin(), b->order.end(), [&](int32_t x, int32_t y) { return work[x] > work[y]; });
  // a knot goes to a cluster when one CTA would need both more than the levels' own latency (about
  // 10^5 cycles) and more than its share of the whole batch; a multiprocessor does 0.5
  // complex multiply-adds per cycle in FP64, 2.7 in float-float, 8 in complex64
  const double rate = precision == PK_C128 ? 0.5 : precision == PK_SPLIT ? 2.7 : 8.0;
  double total = 0;
  for (double w : work) total += w;
  const double share = std::max(1e5, total / rate / 152);
  while (b->n_big < n && work[b->order[b->n_big]] / rate > share) ++b->n_big;
  const uint64_t eb = precision == PK_C64 ? 8 : 16;
  uint64_t off = 0;
  b->off_knots = off;
  off = pk::a256(off + sizeof(pk::BatchKnot) * std::max<size_t>(1, b->knots.size()));
  b->off_recipes = off;
  off = pk::a256(off + sizeof(pk::Recipe) * std::max<size_t>(1, b->recipes.size()));
  b->off_slots = off;
  off = pk::a256(off + sizeof(pk::Slot) * std::max<size_t>(1, b->slots.size()));
  b->off_order = off;
  off = pk::a256(off + 4 * std::max<size_t>(1, b->order.size()));
  b->off_blobs = off;
  off = pk::a256(off + std::max<size_t>(16, b->blobs.size()));
  b->image_bytes = off;
  b->off_meta = off;
  off = pk::a256(off + 16ull * (uint64_t)std::max<int64_t>(1, meta));
  b->off_results = off;
  off = pk::a256(off + sizeof(pk::SliceResult) * (uint64_t)std::max(1, n));
  b->off_counter = off;
  off = pk::a256(off + 256);
  b->off_arena = off;
  b->total = off + eb * (uint64_t)std::max<int64_t>(1, arena);
  b->image.assign(b->image_bytes, 0);
  if (!b->knots.empty())
    std::memcpy(b->image.data() + b->off_knots, b->knots.data(), sizeof(pk::BatchKnot) * b->knots.size());
  if (!b->recipes.empty())
    std::memcpy(b->image.data() + b->off_recipes, b->recipes.data(),
                sizeof(pk::Recipe) * b->recipes.size());
  if (!b->slots.empty())
    std::memcpy(b->image.data() + b->off_slots, b->slots.data(), sizeof(pk::Slot) * b->slots.size());
  if (!b->order.empty()) std::memcpy(b->image.data() + b->off_order, b->order.data(), 4 * b->order.size());
  if (!b->blobs.empty()) std::memcpy(b->image.data() + b->off_blobs, b->blobs.data(), b->blobs.size());
  *out = b;
  return PK_OK;
}

pk_status pk_batch_workspace_bytes(const pk_batch* b, uint64_t* bytes, uint64_t* upload_bytes) {
  if (!b || !bytes) return PK_EINVAL;
  *bytes = b->total;
  if (upload_bytes) *upload_bytes = b->image_bytes;
  return PK_OK;
}

pk_status pk_batch_upload(pk_ctx* ctx, pk_batch* b, void* d_ws, uint64_t bytes) {
  if (!ctx || !b || !d_ws) return bfail(ctx, PK_EINVAL, "bad argument");
  if (ctx->device < 0) return bfail(ctx, PK_ENODEVICE, "host-only context");
  if (bytes < b->total) return bfail(ctx, PK_ENOMEM, "workspace smaller than pk_batch_workspace_bytes");
  if ((uintptr_t)d_ws & 255u) return bfail(ctx, PK_EINVAL, "workspace must be 256-byte aligned");
  if (!b->pinned) {
    if (cudaMallocHost((void**)&b->pinned, std::max<uint64_t>(1, b->image_bytes)) != cudaSuccess)
      return bfail(ctx, PK_ENOMEM, "pinned host allocation failed");
    std::memcpy(b->pinned, b->image.data(), b->image_bytes);
  }
  cudaError_t e = cudaMemcpyAsync(d_ws, b->pinned, b->image_bytes, cudaMemcpyHostToDevice, ctx->stream);
  if (e != cudaSuccess) return bfail(ctx, PK_ECUDA, std::string("batch upload: ") + cudaGetErrorString(e));
  return PK_OK;
}

pk_status pk_batch_upload_inputs(pk_ctx* ctx, pk_batch* b, void* d_ws, uint64_t bytes,
                                 uint64_t* copied) {
  if (!ctx || !b || !d_ws) return bfail(ctx, PK_EINVAL, "bad argument");
  if (ctx->device < 0) return bfail(ctx, PK_ENODEVICE, "host-only context");
  if (bytes < b->total) return bfail(ctx, PK_ENOMEM, "workspace smaller than pk_batch_workspace_bytes");
  if ((uintptr_t)d_ws & 255u) return bfail(ctx, PK_EINVAL, "workspace must be 256-byte aligned");
  if (!b->pinned) {
    if (cudaMallocHost((void**)&b->pinned, std::max<uint64_t>(1, b->image_bytes)) != cudaSuccess)
      return bfail(ctx, PK_ENOMEM, "pinned host allocation failed");
    std::memcpy(b->pinned, b->image.data(), b->image_bytes);
  }
  // knots, recipes and slots lie first in the image, the order and the level records after them
  const uint64_t n = b->off_order - b->off_knots;
  cudaError_t e = cudaMemcpyAsync((char*)d_ws + b->off_knots, b->pinned + b->off_knots, n,
                                  cudaMemcpyHostToDevice, ctx->stream);
  if (e != cudaSuccess) return bfail(ctx, PK_ECUDA, std::string("batch upload: ") + cudaGetErrorString(e));
  if (copied) *copied = n;
  return PK_OK;
}

pk_status pk_batch_launch(pk_ctx* ctx, pk_batch* b, void* d_ws, uint64_t bytes) {
  if (!ctx || !b || !d_ws) return bfail(ctx, PK_EINVAL, "bad argument");
  if (ctx->device < 0) return bfail(ctx, PK_ENODEVICE, "host-only context");
  if (bytes < b->total) return bfail(ctx, PK_ENOMEM, "workspace smaller than pk_batch_workspace_bytes");
  if (b->n == 0) return PK_OK;
  cudaError_t e = build_graph(b, d_ws, ctx->stream);
  if (e == cudaSuccess) e = cudaGraphLaunch(b->exec, ctx->stream);
  if (e != cudaSuccess) return bfail(ctx, PK_ECUDA, std::string("batch launch: ") + cudaGetErrorString(e));
  return PK_OK;
}

pk_status pk_batch_download(pk_ctx* ctx, pk_batch* b, const void* d_ws, pk_scaled* Z, pk_scaled* V) {
  if (!ctx || !b || !d_ws || (!Z && b->n > 0)) return bfail(ctx, PK_EINVAL, "bad argument");
  if (b->n == 0) return PK_OK;
  if (!b->pinned_results &&
      cudaMallocHost((void**)&b->pinned_results, sizeof(pk::SliceResult) * b->n) != cudaSuccess)
    return bfail(ctx, PK_ENOMEM, "pinned host allocation failed");
  cudaError_t e = cudaMemcpyAsync(b->pinned_results, (const char*)d_ws + b->off_results,
                                  sizeof(pk::SliceResult) * b->n, cudaMemcpyDeviceToHost, ctx->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(ctx->stream);
  if (e != cudaSuccess) return bfail(ctx, PK_ECUDA, std::string("batch download: ") + cudaGetErrorString(e));
  pk_status status = PK_OK;
  for (int32_t i = 0; i < b->n; ++i) {
    pk::Scaled z;
    z.re = b->pinned_results[i].re;
    z.im = b->pinned_results[i].im;
    z.e = b->pinned_results[i].exp;
    z.norm();
    z = pk::s_mul(z, b->factor[i]);
    Z[i].re = z.re;
    Z[i].im = z.im;
    Z[i].exp2 = z.e;
    if (V) {
      const pk::Knot& k = b->kinfo[i];
      if (!pk::jones_defined(k)) {
        V[i].re = V[i].im = 0;
        V[i].exp2 = 0;
        status = PK_EINVAL;
        continue;
      }
      pk::Scaled v = pk::s_mul(b->prefactor[i], z);
      V[i].re = v.re;
      V[i].im = v.im;
      V[i].exp2 = v.e;
    }
  }
  if (status != PK_OK) ctx->err = "some batch entries violate the A(q) exponent condition: V left 0";
  return status;
}

pk_status pk_eval_batch(pk_ctx* ctx, const pk_plan* const* plans, int32_t n, int32_t precision,
                        void* d_ws, uint64_t bytes, pk_scaled* Z, pk_scaled* V) {
  pk_batch* b = nullptr;
  pk_status s = pk_batch_create(ctx, plans, n, precision, &b);
  if (s != PK_OK) return s;
  s = pk_batch_upload(ctx, b, d_ws, bytes);
  if (s == PK_OK) s = pk_batch_launch(ctx, b, d_ws, bytes);
  if (s == PK_OK) s = pk_batch_download(ctx, b, d_ws, Z, V);
  pk_batch_destroy(b);
  return s;
}

void pk_batch_destroy(pk_batch* b) {
  if (!b) return;
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  if (b->pinned) cudaFreeHost(b->pinned);
  if (b->pinned_results) cudaFreeHost(b->pinned_results);
  delete b;
}

}  // extern "C"
