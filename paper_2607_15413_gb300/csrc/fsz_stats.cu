// Value-range pass, set-up and planning kernels.
//
// fsz_stats_kernel: min, max and finiteness of every field (Sec. 5.1: eb = REL x (max -
// min)), then the float32-safe quantization step of each field, derived on the device
// (by whichever CTA finishes the field's last chunk or, in a one-field call, by the compression
// kernel), so the host never waits.
// Set-up kernels (one field) and planning kernels (a batch) fill the per-field state and
// the chunk -> field table that every later kernel of the call reads.
#include "fsz_internal.cuh"

namespace fsz {

namespace {

constexpr int kStatsThreads = 256;

__device__ __forceinline__ void finish_field(Ctrl* ctrl, FieldInfo* fi) {
  if (fi->status != 0) return;
  FieldStep p;
  const uint32_t st = derive_step(*fi, &p);
  if (st != FSZ_OK)
    set_error(ctrl, fi, st);
  else
    store_step(fi, p);
}

// n *= dk; false if the product exceeds kMaxElems (n itself does not). Without a 64-bit
// division, which the single thread that plans a field would wait for.
__device__ __forceinline__ bool times_dim(uint64_t* n, uint64_t dk) {
  if (__umul64hi(*n, dk) != 0) return false;
  *n *= dk;
  return *n <= kMaxElems;
}

// Validates one compression descriptor and fills the field's shape (host-visible errors
// of the one-field entry point are checked again here for batches).
__device__ uint32_t plan_cfield(FieldInfo* fi, const fsz_cfield& d) {
  fi->in = d.in;
  fi->out = static_cast<uint8_t*>(d.out);
  fi->cap = d.out_capacity;
  fi->out_bytes = d.out_bytes;
  fi->mode = d.mode;
  fi->eb_req = d.eb;
  fi->ndim = d.dims.ndim;
  fi->nchunks = 0;
  fi->features_off = d.features_off;
  if (d.dims.ndim < 1 || d.dims.ndim > 3 || d.dims.reserved != 0 || !features_valid(d.features_off) ||
      d.mode > 1 || !(d.eb > 0.0) || isinf(d.eb) || d.out == nullptr)
    return FSZ_ERR_INVALID_ARG;
  uint64_t n = 1;
#pragma unroll
  for (uint32_t k = 0; k < 3; ++k) {
    if (k >= d.dims.ndim) continue;
    const uint64_t dk = d.dims.dims[k];
    if (!times_dim(&n, dk)) return FSZ_ERR_INVALID_ARG;
    fi->dims[k] = dk;
  }
  if (n > kMaxElems) return FSZ_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(d.in) & 15) || (reinterpret_cast<uintptr_t>(d.out) & 15))
    return FSZ_ERR_ALIGN;
  if (n > 0 && d.in == nullptr) return FSZ_ERR_INVALID_ARG;
  const uint64_t T = (n + kTile - 1) / kTile;
  fi->n = n;
  fi->T = T;
  if (d.out_capacity < 64 + 8 * T) return FSZ_ERR_CAPACITY;
  fi->nchunks = (T + kCChunkTiles - 1) / kCChunkTiles;
  return FSZ_OK;
}

// The chunk ranges of a batch of up to kStatsPlanned fields, worked out from the descriptors by
// each CTA of the value-range kernel for itself: its loads then run under the planning kernel (4 to
// 5 us of loads that wait for one another in one CTA), which only the publication of the ranges
// waits for. An instance of its own, because 760 CTAs of 48 registers stream at the copy peak only
// while the L1 has room for what they have in flight: with up to 256 fields in one instance with
// the other way, 32 mixed fields of 258 MB took 121.0 us instead of 118.9. Whole calls, behind the
// planning kernel and for themselves: 32 fields of 512 KB 18.4 / 16.5 us, 64 of 256 KB 19.6 / 17.6,
// 64 of 4 MB 108.8 / 106.1. Above 64 fields (this instance with room for 256, 6 KB of shared
// memory) it depends on their size, for better and worse: 65 of 256 KB 20.1 / 18.0, 128 of 64 KB
// 18.3 / 16.7, 128 of 256 KB 26.1 / 26.4, 128 of 1 MB 60.4 / 62.0, 128 of 4 MB 210.5 / 205.9, 256 of
// 64 KB 23.8 / 24.6, 256 of 1 MB 112.2 / 107.9, 256 of 4 MB 413.6 / 407.0; so the rule on the count
// stops where it has been better at every size.
constexpr uint32_t kStatsPlanned = 64;
struct StatsPlan {
  uint64_t total;
  uint64_t first[kStatsPlanned];      // a field's first chunk,
  uint64_t n[kStatsPlanned];          // ... its elements,
  const float* in[kStatsPlanned];
};

// Fills S by the rules of the planning kernel; returns the chunks (none if they exceed the
// workspace's slots, as it does).
__device__ uint64_t stats_plan(StatsPlan& S, const fsz_cfield* d_fields, uint32_t nfields,
                               uint64_t chunk_cap) {
  const uint32_t tid = threadIdx.x;
  uint64_t nch = 0;
  if (tid < nfields) {
    FieldInfo rec = {};
    if (plan_cfield(&rec, d_fields[tid]) == FSZ_OK) nch = rec.nchunks;
    S.n[tid] = rec.n;
    S.in[tid] = rec.in;
  }
  if (tid < kStatsPlanned) {
    uint64_t inc = nch;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if ((tid & 31) >= uint32_t(o)) inc += y;
    }
    S.first[tid] = inc - nch;
    if (tid == 31) S.total = inc;  // (of the first 32)
  }
  __syncthreads();
  if (tid >= 32 && tid < kStatsPlanned) S.first[tid] += S.total;
  __syncthreads();
  if (tid == kStatsPlanned - 1) S.total = S.first[tid] + nch;
  __syncthreads();
  return S.total > chunk_cap ? 0 : S.total;
}

// A CTA's chunks are taken in segments of up to kSegChunks. For a batch, the segment's chunk
// descriptors are read together at its start (two dependent loads for all of them instead
// of two per chunk), and each field's partial range is left in shared memory; at the
// segment's end one thread per field met publishes it. Bound by HBM reads for large fields
// (512^3: 78 us, 6.9 TB/s); for a mix of many small fields by latency: with the descriptor
// loads, barriers and atomics done field by field, a CTA that met a run of small fields
// waited out that chain for each and held the launch (258 MB in 32 log-uniform fields:
// 62 us before, 45 us now).
constexpr int kSegChunks = 64;

struct StatsItem {
  const float* p;
  uint32_t cnt;
  uint32_t f;
};

// kStatsSingle: the field src of n elements. kStatsBatch: the batch that the planning kernel has
// recorded. kStatsBatchOwn: the batch of the nfields descriptors at src, n chunk slots in the
// workspace.
enum StatsKind { kStatsSingle = 0, kStatsBatch = 1, kStatsBatchOwn = 2 };

template <int kKind>
__global__ void __launch_bounds__(kStatsThreads, 5) fsz_stats_kernel(KernelArgs a, const void* src,
                                                                       uint64_t n, uint32_t nfields) {
  constexpr bool kSingle = kKind == kStatsSingle, kOwn = kKind == kStatsBatchOwn;
  constexpr int kStatsWarps = kStatsThreads / 32;
  __shared__ StatsItem s_item[kSegChunks];
  __shared__ float s_lo[kSegChunks][kStatsWarps], s_hi[kSegChunks][kStatsWarps];
  __shared__ uint32_t s_abs[kSegChunks][kStatsWarps];
  __shared__ uint32_t s_f[kSegChunks], s_cnt[kSegChunks];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  float lo = __int_as_float(0x7f800000), hi = __int_as_float(0xff800000);
  uint32_t mabs = 0;
  auto take4 = [&](float4 v) {
    lo = fminf(lo, fminf(fminf(v.x, v.y), fminf(v.z, v.w)));
    hi = fmaxf(hi, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
    uint32_t m0 = max(__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.y) & 0x7fffffffu);
    uint32_t m1 = max(__float_as_uint(v.z) & 0x7fffffffu, __float_as_uint(v.w) & 0x7fffffffu);
    mabs = max(mabs, max(m0, m1));
  };
  // All of a chunk's loads are issued together; in a field's ragged last chunk the pieces
  // past the end read as the chunk's first element.
  auto chunk = [&](const float* p, uint32_t cnt) {
    constexpr int kPer = kCChunkElems / 4 / kStatsThreads;
    const float4* p4 = reinterpret_cast<const float4*>(p);
    float4 v[kPer];
    if (cnt == uint32_t(kCChunkElems)) {
#pragma unroll
      for (int u = 0; u < kPer; ++u) v[u] = __ldcs(p4 + threadIdx.x + u * kStatsThreads);
    } else {
      const uint32_t nv4 = cnt / 4, k = 4 * nv4 + threadIdx.x;
      const float x0 = __ldcs(p);
      const float x = k < cnt ? __ldcs(p + k) : x0;  // the last cnt mod 4 elements
#pragma unroll
      for (int u = 0; u < kPer; ++u) {
        v[u] = make_float4(x0, x0, x0, x);
        if (threadIdx.x + u * kStatsThreads < nv4) v[u] = __ldcs(p4 + threadIdx.x + u * kStatsThreads);
      }
      take4(make_float4(x0, x0, x0, x));
    }
#pragma unroll
    for (int u = 0; u < kPer; ++u) take4(v[u]);
  };
  // Leaves the warp's share of the range of field f (`items` chunks of it) in slot k.
  auto deposit = [&](int k, uint32_t f, uint32_t items) {
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
      lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
      mabs = max(mabs, __shfl_xor_sync(0xffffffffu, mabs, o));
    }
    if (lane == 0) { s_lo[k][warp] = lo; s_hi[k][warp] = hi; s_abs[k][warp] = mabs; }
    if (threadIdx.x == 0) { s_f[k] = f; s_cnt[k] = items; }
    lo = __int_as_float(0x7f800000);
    hi = __int_as_float(0xff800000);
    mabs = 0;
  };
  // Publishes slot k; the CTA that completes a field's count derives the field's step.
  auto publish = [&](int k) {
    float l = s_lo[k][0], h = s_hi[k][0];
    uint32_t m = s_abs[k][0];
    for (int w = 1; w < kStatsWarps; ++w) {
      l = fminf(l, s_lo[k][w]);
      h = fmaxf(h, s_hi[k][w]);
      m = max(m, s_abs[k][w]);
    }
    FieldInfo* fi = a.fields + s_f[k];
    if (l <= h) {
      atomicMax(&fi->min_inv_key, ~float_key(l));
      atomicMax(&fi->max_key, float_key(h));
    }
    atomicMax(&fi->max_abs_bits, m);
    if (kSingle && a.derive) return;  // (the compression kernel behind this one derives the step)
    __threadfence();
    const uint32_t prev = atomicAdd(&fi->done_chunks, s_cnt[k]);
    if (uint64_t(prev) + s_cnt[k] == fi->nchunks) {
      __threadfence();
      finish_field(a.ctrl, fi);
    }
  };

  if constexpr (kSingle) {
    // One field: a stride over the grid, from the field's end to its start, so that what the
    // pass leaves in L2 is what the compression kernel reads first (121 x 251 x 269 field,
    // whole call: 38.0 us upwards, 36.3 us downwards; 512^3: equal).
    // The field is read before grid_wait: the set-up kernel before this one does not write it,
    // and has itself waited for what came before the call.
    const uint64_t total = (n + kCChunkElems - 1) / kCChunkElems;  // >= gridDim.x
    const uint64_t gn = (total - blockIdx.x + gridDim.x - 1) / gridDim.x;
    for (uint64_t k = 0; k < gn; ++k) {
      const uint64_t e0 = (total - 1 - (blockIdx.x + k * gridDim.x)) * uint64_t(kCChunkElems);
      chunk(static_cast<const float*>(src) + e0, uint32_t(min(n - e0, uint64_t(kCChunkElems))));
    }
    deposit(0, 0, uint32_t(gn));
    // (the set-up kernel has completed: the compression kernel may take its first tickets)
    grid_wait();
    grid_release();
    __syncthreads();
    if (threadIdx.x == 0) publish(0);
  } else {
    // A batch: each CTA takes one contiguous range of its chunks and so meets few fields
    // (a batch of 32 mixed fields of 258 MB in all, whole call: 145.5 us with a stride over
    // the grid, 142.4 us with ranges).
    __shared__ StatsPlan plan;
    uint64_t total;
    if constexpr (kOwn) {
      total = stats_plan(plan, static_cast<const fsz_cfield*>(src), nfields, n);
    } else {
      grid_wait();
      total = a.ctrl->total_chunks;
    }
    for (uint64_t k = uint64_t(blockIdx.x) * kStatsThreads + threadIdx.x; k < kFlagStride * total;
         k += uint64_t(gridDim.x) * kStatsThreads)
      a.flags[k] = 0;  // (lookback flags, for the compression kernel)
    const uint64_t g0 = total * blockIdx.x / gridDim.x;
    const uint64_t gn = total * (blockIdx.x + 1) / gridDim.x - g0;
    for (uint64_t k0 = 0; k0 < gn; k0 += kSegChunks) {
      const int seg = int(min(uint64_t(kSegChunks), gn - k0));
      if (int(threadIdx.x) < seg) {
        const uint64_t g = g0 + k0 + threadIdx.x;
        if constexpr (kOwn) {  // the last field that begins at or before the chunk
          uint32_t f = 0;
#pragma unroll
          for (uint32_t s = kStatsPlanned / 2; s > 0; s >>= 1)
            if (f + s < nfields && plan.first[f + s] <= g) f += s;
          const uint64_t e0 = (g - plan.first[f]) * uint64_t(kCChunkElems);
          s_item[threadIdx.x] =
              StatsItem{plan.in[f] + e0, uint32_t(min(plan.n[f] - e0, uint64_t(kCChunkElems))), f};
        } else {
          const uint32_t f = a.chunk_field[g];
          const FieldInfo* fi = a.fields + f;
          const uint64_t e0 = (g - fi->chunk_first) * uint64_t(kCChunkElems);
          s_item[threadIdx.x] = StatsItem{fi->in + e0, uint32_t(min(fi->n - e0, uint64_t(kCChunkElems))), f};
        }
      }
      __syncthreads();
      int parts = 0;
      uint32_t items = 0;
      for (int k = 0; k < seg; ++k) {
        const StatsItem it = s_item[k];
        chunk(it.p, it.cnt);
        ++items;
        if (k + 1 == seg || s_item[k + 1].f != it.f) {
          deposit(parts++, it.f, items);
          items = 0;
        }
      }
      __syncthreads();
      if constexpr (kOwn) grid_wait();  // (the records are there)
      if (k0 + kSegChunks >= gn) grid_release();  // (the compression kernel may take its first tickets)
      if (int(threadIdx.x) < parts) publish(int(threadIdx.x));
      __syncthreads();
    }
    if constexpr (kOwn) grid_wait();
    grid_release();
  }
}

// Parses and checks a stream's preamble (the same rules as the format's definition:
// magic, version, ndim, mode, dims product, positive finite eb and step, sizes).
// kTiled: streams of any tile configuration.
template <bool kTiled>
__device__ uint32_t plan_dfield(FieldInfo* fi, const uint8_t* in, uint64_t in_bytes, float* out,
                                uint64_t cap_elems) {
  fi->sin = in;
  fi->in_bytes = in_bytes;
  fi->dout = out;
  fi->nchunks = 0;
  if (in == nullptr || out == nullptr) return FSZ_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(in) & 15) || (reinterpret_cast<uintptr_t>(out) & 15))
    return FSZ_ERR_ALIGN;
  if (in_bytes < 64) return FSZ_ERR_CORRUPT;
  uint32_t w[16];
  const uint4* p = reinterpret_cast<const uint4*>(in);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint4 v = p[k];
    w[4 * k] = v.x; w[4 * k + 1] = v.y; w[4 * k + 2] = v.z; w[4 * k + 3] = v.w;
  }
  if (w[0] != 0x315A5346u || (w[1] & 0xFFFFu) != 1u) return FSZ_ERR_CORRUPT;
  const uint32_t ndim = (w[1] >> 16) & 0xFFu, mode = w[1] >> 24;
  if (ndim < 1 || ndim > 3 || mode > 1) return FSZ_ERR_CORRUPT;
  const uint64_t n = uint64_t(w[2]) | (uint64_t(w[3]) << 32);
  uint64_t prod = 1;
  for (uint32_t k = 0; k < 3; ++k) {
    const uint64_t dk = uint64_t(w[4 + 2 * k]) | (uint64_t(w[5 + 2 * k]) << 32);
    if (k >= ndim) {
      if (dk != 0) return FSZ_ERR_CORRUPT;
      continue;
    }
    if (!times_dim(&prod, dk)) return FSZ_ERR_CORRUPT;
    fi->dims[k] = dk;
  }
  if (prod != n || n > kMaxElems) return FSZ_ERR_CORRUPT;
  const double eb = __longlong_as_double(static_cast<long long>(uint64_t(w[10]) | (uint64_t(w[11]) << 32)));
  const float sv = __uint_as_float(w[12]);
  if (!(eb > 0.0) || isinf(eb)) return FSZ_ERR_CORRUPT;
  if (!(sv >= 1.5777218104420236e-30f) || isinf(sv)) return FSZ_ERR_CORRUPT;  // 2^-99
  int B = 32, TB = 8;
  if constexpr (kTiled) {
    if (!config_of(w[13], &B, &TB) || !features_valid(w[13] & 7u)) return FSZ_ERR_CORRUPT;
  } else {
    if (w[13] & 0xFF00u) return FSZ_ERR_INVALID_ARG;  // a tile configuration: fsz_decompress_tiled
    if (!features_valid(w[13])) return FSZ_ERR_CORRUPT;
  }
  fi->features_off = w[13];
  const uint64_t db = uint64_t(w[14]) | (uint64_t(w[15]) << 32);
  const uint32_t tile = uint32_t(B * TB);
  const uint64_t T = (n + tile - 1) >> (31 - __clz(int(tile)));  // (a power of two)
  if (in_bytes - 64 < TB * T) return FSZ_ERR_CORRUPT;
  if (db > in_bytes - 64 - TB * T) return FSZ_ERR_CORRUPT;
  fi->n = n;
  fi->T = T;
  fi->ndim = ndim;
  fi->mode = mode;
  fi->eb_req = eb;
  fi->s = sv;
  fi->data_bytes = db;
  if (n > cap_elems) return FSZ_ERR_CAPACITY;
  fi->nchunks = (n + kDChunkElems - 1) / kDChunkElems;
  return FSZ_OK;
}

// A valid field of zero elements: its step, its 64-byte stream and its size.
__device__ void finish_empty_field(Ctrl* ctrl, FieldInfo* fi) {
  finish_field(ctrl, fi);
  if (fi->status == 0) write_preamble(fi, 0, fi->s);
}

// Set-up of a single-field compression, whose descriptor the host has validated: thread 0 of
// CTA 0 clears the control words and the field record and fills them in; every other thread
// clears the lookback flags (nflags words), so that the call needs no separate memset.
constexpr int kSetupThreads = 256;
static_assert(sizeof(Ctrl) <= 256 && sizeof(Ctrl) % 8 == 0 && sizeof(FieldInfo) % 8 == 0,
              "control words and field record clear as 8-byte words");

__device__ __forceinline__ bool setup_clear(const KernelArgs& a, uint64_t nflags) {
  grid_wait();
  grid_release();
  const uint64_t t = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (t == 0) {
    uint64_t* c = reinterpret_cast<uint64_t*>(a.ctrl);
    for (uint32_t k = 0; k < sizeof(Ctrl) / 8; ++k) c[k] = 0;
    uint64_t* f = reinterpret_cast<uint64_t*>(a.fields);
    for (uint32_t k = 0; k < sizeof(FieldInfo) / 8; ++k) f[k] = 0;
    return true;
  }
  const uint64_t nthreads = uint64_t(gridDim.x) * blockDim.x - 1;
  for (uint64_t k = t - 1; k < nflags; k += nthreads) a.flags[k] = 0;
  return false;
}

__global__ void __launch_bounds__(kSetupThreads) fsz_setup_compress_kernel(KernelArgs a, FieldInfo desc,
                                                                           uint64_t nflags) {
  if (!setup_clear(a, nflags)) return;
  FieldInfo* fi = a.fields;
  fi->in = desc.in; fi->out = desc.out; fi->cap = desc.cap; fi->out_bytes = desc.out_bytes;
  fi->n = desc.n; fi->T = desc.T;
  fi->dims[0] = desc.dims[0]; fi->dims[1] = desc.dims[1]; fi->dims[2] = desc.dims[2];
  fi->ndim = desc.ndim; fi->mode = desc.mode; fi->eb_req = desc.eb_req;
  fi->features_off = desc.features_off;
  fi->chunk_first = 0;
  fi->nchunks = desc.nchunks;
  a.ctrl->nfields = 1;
  a.ctrl->total_chunks = desc.nchunks;
  if (desc.n == 0) finish_empty_field(a.ctrl, fi);
}

// Payload sizes of the chunks, from the rate headers alone (8 of them per 32 KiB of output):
// one warp per chunk, one CTA per kSumBlock chunks at a time. A chunk's byte offset is then
// a short sum over these (range_fetch in the decompression kernel), where a decoupled
// lookback during decompression made the first chunk of each CTA wait 5 to 11 us for the
// others. Bound by latency (two loads and two barriers); with the set-up 4.3 us at 512^3
// (4 MB of headers), 3.3 us at 2^20 values, against 3.1 and 2.7 us for the set-up alone.
// 16 warps with two chunks each: 32 warps with one took 7.8 us at 512^3.
constexpr int kSizeWarps = 16;
constexpr int kSizeThreads = 32 * kSizeWarps;
constexpr int kChunksPerWarp = kSumBlock / kSizeWarps;  // of a block: warp, warp + kSizeWarps

// Records the sizes of one block of chunks; bytes[k]: this lane's unit of chunk
// kSumBlock * block + kSizeWarps * k + warp (0 beyond the last one). Returns their sum in thread 0.
__device__ __forceinline__ uint32_t write_chunk_sizes(const KernelArgs& a, uint64_t block, uint64_t total,
                                                  const uint32_t (&bytes)[kChunksPerWarp],
                                                  uint32_t* s_sum) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < kChunksPerWarp; ++k) {
    const uint64_t c = block * kSumBlock + kSizeWarps * k + warp;
    const uint32_t sum = __reduce_add_sync(0xffffffffu, bytes[k]);
    if (lane == 0) {
      s_sum[kSizeWarps * k + warp] = sum;
      if (c < total) a.sums[c] = sum;
    }
  }
  __syncthreads();
  uint32_t all = 0;
  if (warp == 0) {
    all = __reduce_add_sync(0xffffffffu, s_sum[lane]);
    if (lane == 0) a.block_sums[block] = all;
  }
  __syncthreads();
  return all;
}

// One field: sized beside the parsing of its preamble (by one thread of CTA 0) rather than
// after it. The element count is read from the preamble as it stands, bounded by the
// output's capacity, and the headers within the stream's buffer; the sizes of a stream that
// the parsing refuses are not used. kTiled: the headers are checked too, and what each CTA found
// left for the decompression kernel, which writes nothing for a stream whose headers are malformed
// or do not add up to its data.
template <bool kTiled>
__global__ void __launch_bounds__(kSizeThreads) fsz_setup_decompress_kernel(KernelArgs a,
                                                                            uint64_t chunk_cap) {
  const uint8_t* const in = a.sin;
  const uint64_t in_bytes = a.in_bytes, cap_elems = a.cap_elems;
  __shared__ uint32_t s_sum[kSumBlock];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  grid_wait();
  grid_release();
  const unsigned long long* const hdr = reinterpret_cast<const unsigned long long*>(in + 64);
  const uint64_t n = in_bytes >= 64 ? *reinterpret_cast<const uint64_t*>(in + 8) : 0;
  const uint64_t room = in_bytes >= 64 ? in_bytes - 64 : 0;  // bytes after the preamble
  int B = 32, TB = 8;
  uint64_t forbid = 0;
  if constexpr (kTiled) {
    const uint32_t word = in_bytes >= 64 ? *reinterpret_cast<const uint32_t*>(in + 52) : 0u;
    if (!config_of(word, &B, &TB)) B = 32, TB = 8;
    forbid = forbidden_flags(word);
  }
  // rate bytes 8 (u + 0 .. 7), or as many of them as there are before `end`
  auto load_unit = [&](uint64_t u, uint64_t end) -> uint64_t {
    if (8 * u + 8 <= end) return __ldg(hdr + u);
    if (kTiled && 8 * u + 4 <= end) return __ldg(reinterpret_cast<const uint32_t*>(hdr + u));
    return 0;
  };
  const uint32_t units = uint32_t(kDChunkElems / 8) / uint32_t(B);  // of a chunk: 32 or 16
  auto unit = [&](uint64_t b, int k) {
    return (b * kSumBlock + kSizeWarps * k + warp) * units + lane;
  };
  uint64_t h[kChunksPerWarp];
  if constexpr (!kTiled) {
#pragma unroll
    for (int k = 0; k < kChunksPerWarp; ++k)  // (issued with n's load)
      h[k] = load_unit(unit(blockIdx.x, k), room);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    FieldInfo f = {};
    uint32_t st = plan_dfield<kTiled>(&f, in, in_bytes, a.dout, cap_elems);
    if (st == FSZ_OK && f.nchunks > chunk_cap) st = FSZ_ERR_WORKSPACE;
    if (st != FSZ_OK) f.nchunks = 0;
    f.status = st;
    Ctrl c = {};
    c.status = st;
    c.nfields = 1;
    c.total_chunks = f.nchunks;
    *a.fields = f;
    *a.ctrl = c;
  }
  const uint64_t nc = min(n, cap_elems);
  const uint64_t total = (nc + kDChunkElems - 1) / kDChunkElems;  // <= chunk_cap
  const uint64_t hdr_bytes = min(((nc + B * TB - 1) >> (31 - __clz(B * TB))) * TB, room);
  uint64_t sum = 0;
  bool bad = false;
  for (uint64_t b = blockIdx.x; b * kSumBlock < total; b += gridDim.x) {
    uint32_t bytes[kChunksPerWarp];
#pragma unroll
    for (int k = 0; k < kChunksPerWarp; ++k) {
      const uint64_t u = unit(b, k);
      const bool mine = uint32_t(lane) < units && 8 * u < hdr_bytes;
      if (kTiled || b != blockIdx.x) h[k] = mine ? load_unit(u, hdr_bytes) : 0;
      bytes[k] = mine ? unit_bytes(h[k], B, TB, u) : 0u;
      if (kTiled && mine)
        bad |= header_reserved_bits_set(h[k], TB, u) || (h[k] & (forbid * unit_centring_bits(TB, u))) != 0;
    }
    sum += write_chunk_sizes(a, b, total, bytes, s_sum);
  }
  if constexpr (kTiled) {
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) a.found[blockIdx.x] = bad ? kHeadersBad : sum;
  }
}

// The chunk ranges of a batch of up to kSizeThreads fields, worked out from the descriptors by a
// CTA for itself.
struct SelfPlan {
  uint64_t warp_sum[kSizeWarps];
  uint64_t total;
  uint64_t first[kSizeThreads];      // a field's first chunk,
  uint64_t tiles[kSizeThreads];      // ... its tiles,
  const uint8_t* stream[kSizeThreads];
};

// Fills S by the rules of the planning kernel; returns the chunks (none if they exceed the
// workspace's slots, as it does).
__device__ uint64_t self_plan(SelfPlan& S, const fsz_dfield* d_fields, uint32_t nfields, uint64_t chunk_cap) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint64_t nch = 0;
  if (tid < nfields) {
    const fsz_dfield d = d_fields[tid];
    FieldInfo rec = {};
    const uint32_t st = plan_dfield<false>(&rec, static_cast<const uint8_t*>(d.in), d.in_bytes, d.out,
                                           d.out_capacity_elems);
    nch = st == FSZ_OK ? rec.nchunks : 0;
    S.tiles[tid] = rec.T;
    S.stream[tid] = rec.sin;
  }
  uint64_t inc = nch;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= uint32_t(o)) inc += y;
  }
  if (lane == 31) S.warp_sum[warp] = inc;
  __syncthreads();
  uint64_t first = inc - nch;
  for (uint32_t w = 0; w < warp; ++w) first += S.warp_sum[w];
  S.first[tid] = first;
  if (tid == kSizeThreads - 1) S.total = first + nch;
  __syncthreads();
  return S.total > chunk_cap ? 0 : S.total;
}

// The field of chunk c (below the total): the last one that begins at or before it.
__device__ __forceinline__ uint32_t field_of_chunk(const SelfPlan& S, uint32_t nfields, uint64_t c) {
  uint32_t f = 0;
#pragma unroll
  for (uint32_t s = kSizeThreads / 2; s > 0; s >>= 1)
    if (f + s < nfields && S.first[f + s] <= c) f += s;
  return f;
}

// A batch. Its planning kernel is 4 to 5 us of loads that wait for one another in one CTA: with
// up to kSizeThreads fields, a thread each, the sizing CTAs plan for themselves under it instead
// of waiting for its records and its chunk -> field table, unless they are so many that reading
// every field in each costs more (whole calls behind it and for themselves: 32 fields of 258 MB
// 62.8 / 60.5 us; 512 of 256 KB, 128 CTAs: 47.4 / 44.5; 128 of 4 MB, 608 CTAs: 105.6 / 104.6;
// 256 of 4 MB: 193.4 / 196.3).
constexpr uint32_t kSelfPlanReads = 128 * 608;  // fields x CTAs
__global__ void __launch_bounds__(kSizeThreads) fsz_sizes_kernel(KernelArgs a, const fsz_dfield* d_fields,
                                                                 uint32_t nfields, uint64_t chunk_cap) {
  __shared__ uint32_t s_sum[kSumBlock];
  __shared__ SelfPlan plan;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool own = nfields <= uint32_t(kSizeThreads) && nfields * gridDim.x <= kSelfPlanReads;
  uint64_t total;
  if (own) {
    total = self_plan(plan, d_fields, nfields, chunk_cap);
  } else {
    grid_wait();
    total = a.ctrl->total_chunks;
  }
  grid_release();  // (the records may not be there yet: the successor loads nothing early)
  for (uint64_t b = blockIdx.x; b * kSumBlock < total; b += gridDim.x) {
    uint32_t bytes[kChunksPerWarp];
#pragma unroll
    for (int k = 0; k < kChunksPerWarp; ++k) {
      const uint64_t c = b * kSumBlock + kSizeWarps * k + warp;
      bytes[k] = 0;
      if (c < total) {
        const uint32_t f = own ? field_of_chunk(plan, nfields, c) : a.chunk_field[c];
        const FieldInfo* fi = a.fields + f;
        const uint8_t* in = own ? plan.stream[f] : fi->sin;
        const uint64_t first = own ? plan.first[f] : fi->chunk_first, T = own ? plan.tiles[f] : fi->T;
        const uint64_t t = (c - first) * kDChunkTiles + lane;
        if (t < T)
          bytes[k] = unit_bytes(__ldg(reinterpret_cast<const unsigned long long*>(in + 64) + t), 32, 8, t);
      }
    }
    write_chunk_sizes(a, b, total, bytes, s_sum);
  }
  grid_wait();  // (this kernel completes after the planning kernel)
}

// CTAs of a sizing launch: one per kSumBlock chunks, at most four per SM.
int sizes_grid(uint64_t max_chunks) {
  static DeviceCfgCache cache;
  const LaunchCfg c = cache.get([] {
    LaunchCfg cfg = {};
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&cfg.sms, cudaDevAttrMultiProcessorCount, dev);
    cfg.grid = 4 * cfg.sms;
    return cfg;
  });
  const uint64_t g = (max_chunks + kSumBlock - 1) / kSumBlock;
  return g < uint64_t(c.grid) ? int(g > 0 ? g : 1) : c.grid;
}

// CTAs of a set-up launch: one plus one per 2048 flag words, at most 152.
inline int setup_grid(uint64_t nflags) {
  const uint64_t g = 1 + nflags / (8 * kSetupThreads);
  return int(g < 152 ? g : 152);
}

constexpr int kPlanThreads = 1024;

// Batch planning (one CTA): clears the control words and field records, per-field checks, an
// exclusive scan of the fields' chunk counts (their ranges in the field-major ticket order)
// and the chunk -> field table. Bound by latency (a chain of loads and barriers, 4 us for up
// to 1024 fields).
template <bool kCompress>
__global__ void __launch_bounds__(kPlanThreads) fsz_plan_kernel(KernelArgs a, const void* d_fields,
                                                                uint32_t nfields, uint64_t chunk_cap) {
  __shared__ uint64_t s_warp[kPlanThreads / 32];
  __shared__ uint64_t s_first[kPlanThreads], s_count[kPlanThreads];
  __shared__ uint64_t s_carry;
  __shared__ uint32_t s_status;  // the first error met
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    s_carry = 0;
    s_status = 0;
  }
  __syncthreads();
  grid_wait();
  grid_release();
  uint32_t* const map = const_cast<uint32_t*>(a.chunk_field);
  for (uint32_t base = 0; base < nfields; base += kPlanThreads) {
    const uint32_t f = base + tid;
    uint64_t nch = 0;
    if (f < nfields) {
      FieldInfo* fi = a.fields + f;
      FieldInfo rec = {};
      uint32_t st;
      if constexpr (kCompress) {
        st = plan_cfield(&rec, static_cast<const fsz_cfield*>(d_fields)[f]);
      } else {
        const fsz_dfield d = static_cast<const fsz_dfield*>(d_fields)[f];
        st = plan_dfield<false>(&rec, static_cast<const uint8_t*>(d.in), d.in_bytes, d.out,
                                d.out_capacity_elems);
      }
      if (st != FSZ_OK) {
        atomicCAS(&s_status, 0u, st);
        rec.status = st;
        rec.nchunks = 0;
      }
      nch = rec.nchunks;
      *fi = rec;
    }
    // block-wide exclusive scan of nch
    uint64_t inc = nch;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    if (warp == 0) {
      uint64_t v = s_warp[lane];
      uint64_t vi = v;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xffffffffu, vi, o);
        if (lane >= o) vi += y;
      }
      s_warp[lane] = vi - v;
    }
    __syncthreads();
    const uint64_t first = s_carry + s_warp[warp] + inc - nch;
    if (f < nfields) a.fields[f].chunk_first = first;
    s_first[tid] = first;
    s_count[tid] = nch;
    __syncthreads();
    if (tid == kPlanThreads - 1) s_carry = first + nch;
    // These fields' part of the chunk -> field table, one warp per field (their ranges are
    // disjoint); nothing beyond the workspace's slots.
    const uint32_t nb = min(nfields - base, uint32_t(kPlanThreads));
    for (uint32_t k = uint32_t(warp); k < nb; k += uint32_t(kPlanThreads / 32)) {
      const uint64_t c0 = s_first[k], c1 = min(c0 + s_count[k], chunk_cap);
      for (uint64_t c = c0 + uint64_t(lane); c < c1; c += 32) map[c] = base + k;
    }
    __syncthreads();
  }
  const uint64_t total = s_carry;
  if (tid == 0) {
    Ctrl c = {};
    c.status = total > chunk_cap && s_status == 0 ? uint32_t(FSZ_ERR_WORKSPACE) : s_status;
    c.nfields = nfields;
    c.total_chunks = total > chunk_cap ? 0 : total;
    *a.ctrl = c;
  }
  if (total > chunk_cap) return;
  __syncthreads();  // (the control words before an empty field's error)
  if constexpr (kCompress) {
    for (uint32_t f = tid; f < nfields; f += kPlanThreads) {
      FieldInfo* fi = a.fields + f;
      if (fi->status == 0 && fi->n == 0) finish_empty_field(a.ctrl, fi);
    }
  }
}

}  // namespace

LaunchCfg stats_cfg() {
  static DeviceCfgCache cache;
  return cache.get([] {
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fsz_stats_kernel<kStatsSingle>, kStatsThreads, 0);
    LaunchCfg c;
    c.sms = sms;
    c.per = per > 0 ? per : 1;
    c.grid = sms * c.per;
    c.smem = 0;
    return c;
  });
}

void launch_stats(const KernelArgs& a, const float* in, uint64_t n, cudaStream_t st) {
  const uint64_t chunks = (n + kCChunkElems - 1) / kCChunkElems;
  launch_dependent(fsz_stats_kernel<kStatsSingle>, sched_grid(stats_cfg(), kSchedStats, chunks),
                   kStatsThreads, 0, st, a, static_cast<const void*>(in), n, 0u);
}

void launch_stats_batch(const KernelArgs& a, const fsz_cfield* d_fields, uint32_t nfields,
                        uint64_t chunk_cap, uint64_t max_chunks, cudaStream_t st) {
  launch_dependent(nfields <= kStatsPlanned ? fsz_stats_kernel<kStatsBatchOwn> : fsz_stats_kernel<kStatsBatch>,
                   sched_grid(stats_cfg(), kSchedStats, max_chunks), kStatsThreads, 0, st, a,
                   static_cast<const void*>(d_fields), chunk_cap, nfields);
}

void launch_setup_compress(const KernelArgs& a, const FieldInfo& fi, uint64_t chunk_cap, cudaStream_t st) {
  const uint64_t nflags = kFlagStride * chunk_cap;
  launch_dependent(fsz_setup_compress_kernel, setup_grid(nflags), kSetupThreads, 0, st, a, fi, nflags);
}

int setup_decompress_grid(uint64_t cap_elems) {
  return sizes_grid((cap_elems + kDChunkElems - 1) / kDChunkElems);
}

void launch_setup_decompress(const KernelArgs& a, uint64_t chunk_cap, cudaStream_t st, bool tiled) {
  launch_dependent(tiled ? fsz_setup_decompress_kernel<true> : fsz_setup_decompress_kernel<false>,
                   setup_decompress_grid(a.cap_elems), kSizeThreads, 0, st, a, chunk_cap);
}

void launch_sizes(const KernelArgs& a, const fsz_dfield* d_fields, uint32_t nfields, uint64_t chunk_cap,
                  uint64_t max_chunks, cudaStream_t st) {
  launch_dependent(fsz_sizes_kernel, sizes_grid(max_chunks), kSizeThreads, 0, st, a, d_fields, nfields,
                   chunk_cap);
}

void launch_plan_compress(const KernelArgs& a, const fsz_cfield* d_fields, uint32_t nfields,
                          uint64_t chunk_cap, cudaStream_t st) {
  launch_dependent(fsz_plan_kernel<true>, 1, kPlanThreads, 0, st, a, static_cast<const void*>(d_fields),
                   nfields, chunk_cap);
}

void launch_plan_decompress(const KernelArgs& a, const fsz_dfield* d_fields, uint32_t nfields,
                            uint64_t chunk_cap, cudaStream_t st) {
  launch_dependent(fsz_plan_kernel<false>, 1, kPlanThreads, 0, st, a, static_cast<const void*>(d_fields),
                   nfields, chunk_cap);
}

}  // namespace fsz
