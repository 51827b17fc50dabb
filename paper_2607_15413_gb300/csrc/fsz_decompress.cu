// FSZ decompression kernel (Sec. 3.1 "Decompression", steps d1-d5).
//
// Persistent, warp-specialised CTAs; the roles hand chunks to one another through
// mbarriers:
//   header warp   takes a ticket, d1 reads the chunk's rate header, d2 derives the tile
//                 sizes and scans them, d3 sums the sizes of the chunks before (computed
//                 from the headers by the kernel before this one: no CTA waits for another)
//                 and leaves the chunk's record (headers, offsets, field parameters) in a
//                 ring of records, running ahead of decoding;
//   loader warp   takes the chunk's payload bytes (its actual size, not the worst case)
//                 from a byte ring, waiting for the oldest chunks' decoding to release
//                 space, and loads the payload there with a 1-D TMA bulk copy. Compressed
//                 chunks being far below the worst case, several are in flight per CTA;
//   decode warps  (8) each decode a quad of 4 tiles at a time, lane L holding block L & 7
//                 of tile L >> 3 (32 consecutive elements): d4 reads the block's sign map
//                 and planes and undoes the bit shuffle with the register-pair delta swaps
//                 of the compressor, run backwards; d5 inverts the prediction as prefix sums
//                 inside the lane with the carry from the tile's earlier blocks by an 8-lane
//                 scan (once for LZ1, twice for LZ2), adds mu, d' = fl(float(q) s); the
//                 floats go through a per-warp swizzled buffer so that each store of the
//                 warp writes 512 consecutive bytes.
#include "fsz_internal.cuh"

namespace fsz {

namespace {

constexpr int kDecodeWarps = 8;
constexpr int kHeaderWarp = kDecodeWarps;
constexpr int kLoaderWarp = kDecodeWarps + 1;
constexpr int kThreads = (kDecodeWarps + 2) * 32;
#ifndef FSZ_DEC_RING_BYTES
#define FSZ_DEC_RING_BYTES 65536
#endif
constexpr int kMaxRecs = kMaxDecRecords;  // chunk records (fetched .. decoded): up to
constexpr uint32_t kRingBytes = FSZ_DEC_RING_BYTES;  // payload byte ring
constexpr int kQuadElems = 1024;  // elements per decode warp and chunk
static_assert(kDecodeWarps * kQuadElems == kDChunkElems, "a chunk is one quad per decode warp");
// Ring bytes a chunk can take: its payload (header-valid rates go up to 31: 128 bytes per 32
// elements, and up to 64 means) from the 16-byte boundary below its start, rounded up to 16
// bytes.
constexpr uint32_t kMaxChunkRingBytes = kDChunkElems / 32 * 128 + 64 * 4 + 32;
constexpr int kHdrUnits = 32;     // a chunk's rate bytes, 8 at a time (64-element blocks: 16)
static_assert(kRingBytes % 16 == 0 && kRingBytes >= kMaxChunkRingBytes, "the ring holds the largest chunk");

constexpr uint32_t kNoneChunk = 0xffffffffu;
// The schedule's work assignment (kernel arguments): a ticket hands a CTA ticket_chunks
// consecutive chunks (at most kMaxTicketChunks). Their rate headers are read together,
// and the group's byte offset is summed once. A CTA holds `records` chunks
// (2 x ticket_chunks .. kMaxRecs) between ticket and decode.

// Near the launch's end (its last kTailChunks chunks per CTA) tickets are at most kTailTicket
// chunks and a CTA holds at most kTailAhead: what one CTA has taken no other can, and with up
// to 16 chunks (30 us) held each the CTAs finished far apart. 512^3: 112.6 us without, 109.8
// from the last 8 chunks on, 106.9 from 16, 106.2 from 32; batch of 32 fields 69.7, 66.0, 66.5,
// 67.6 us; with kTailAhead 4 or 8: 106.8, 108.9 and 67.9, 67.0 us.
// (A schedule whose min_tickets is 0 keeps its tickets and records to the end.)
constexpr uint32_t kTailChunks = 16, kTailTicket = 2, kTailAhead = 6;

// A chunk's header and parameters, from the header warp to the loader and the decode
// warps through shared memory (keeps dependent global loads off the decode path).
struct ChunkRec {
  uint64_t hdr[kHdrUnits];
  uint64_t boff[kHdrUnits];  // block word offsets inside each unit (block_word_offsets)
  uint32_t toff[kHdrUnits];  // byte offset of each unit's data in the payload
  FieldInfo* fi;
  float* dout;           // the chunk's first output element
  const uint8_t* sin;    // the field's stream
  uint64_t in_bytes;     // its size
  uint64_t data_bytes;   // tile data bytes the preamble declares
  uint64_t data_base;    // start of the tile data, after the rate headers
  uint64_t excl;         // byte offset of the chunk's payload in the tile data
  uint32_t chunk;        // global chunk index, or kNoneChunk
  uint32_t last;         // the field's last chunk
  uint32_t tot;          // payload bytes of the chunk
  uint32_t bad;          // reserved header bits seen
  uint32_t valid;        // payload loaded and decodable
  uint32_t pay;          // payload start inside the ring
  uint32_t ntiles;
  uint32_t cnt;          // valid elements of the chunk
  uint32_t indep;        // the stream's blocks are independent (no carried state)
  float step;
};

struct __align__(16) DecompressSmem {
  uint8_t ring[kRingBytes];
  float out[kDecodeWarps][kQuadElems];  // per-warp re-layout of a quad's floats
  ChunkRec rec[kMaxRecs];
  uint32_t ring_end[kMaxRecs];  // loader only: ring position (mod 2^32) after each chunk's bytes
  // fetched: record in (header -> loader); full: payload in (loader -> decode warps);
  // done: chunk decoded, its record and ring bytes free (decode warps -> header, loader)
  uint64_t fetched[kMaxRecs], full[kMaxRecs], done[kMaxRecs];
};
// two CTAs per SM (228 KiB of shared memory, 1 KiB of it reserved per CTA)
static_assert(sizeof(DecompressSmem) <= 113 * 1024, "shared memory of one CTA");

// Word offsets of a unit's 8 blocks inside its data (means not counted), one per byte: the
// exclusive byte-wise prefix sum of the blocks' word counts (rate + 1, or 0; <= 224).
__device__ __forceinline__ uint64_t block_word_offsets(uint64_t h) {
  const uint64_t R = h & 0x1F1F1F1F1F1F1F1FULL;
  const uint64_t W = R + (((R + 0x7F7F7F7F7F7F7F7FULL) & 0x8080808080808080ULL) >> 7);
  return (W * 0x0101010101010101ULL) << 8;
}

// *p if `in`, else 0, read here: a plain load is moved down to its use by the compiler, past
// the work that it is meant to run under. ld_now32 reads from L2.
__device__ __forceinline__ uint64_t ld_now(const void* p, bool in) {
  uint64_t v;
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\tmov.u64 %0, 0;\n\t"
      "@p ld.global.nc.u64 %0, [%1];\n\t}"
      : "=l"(v)
      : "l"(p), "r"(uint32_t(in)));
  return v;
}
__device__ __forceinline__ uint32_t ld_now32(const uint32_t* p, bool in) {
  uint32_t v;
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\tmov.u32 %0, 0;\n\t"
      "@p ld.global.cg.u32 %0, [%1];\n\t}"
      : "=r"(v)
      : "l"(p), "r"(uint32_t(in)));
  return v;
}

// The payload bytes of chunks lo .. hi - 1 are range_total of what every lane fetched: the
// chunk sizes up to the first and from the last multiple of kSumBlock and the block sums
// between, all loads independent. A CTA's tickets lie about one grid of tickets apart, so a
// launch of 304 CTAs x 4 chunks reads 38 block sums and at most 62 sizes per ticket; only a
// longer stretch needs the loop.
constexpr int kRangeParts = 4;
__device__ __forceinline__ void range_fetch(const uint32_t* sums, const uint32_t* block_sums,
                                            uint32_t lo, uint32_t hi, uint32_t (&part)[kRangeParts],
                                            uint64_t* rest) {
  static_assert(kSumBlock == 32, "one lane per chunk of a block");
  const uint32_t lane = threadIdx.x & 31;
  const uint32_t b0 = (lo + 31) / 32, b1 = hi / 32;  // whole blocks b0 .. b1 - 1
  const bool whole = b0 < b1;                        // (without one: at most 62 chunks)
  const uint32_t k0 = lo + lane, k1 = (whole ? 32 * b1 : lo + 32) + lane;
  part[0] = ld_now32(sums + k0, k0 < (whole ? 32 * b0 : hi));
  part[1] = ld_now32(sums + k1, k1 < hi);
  part[2] = ld_now32(block_sums + b0 + lane, b0 + lane < b1);
  part[3] = ld_now32(block_sums + b0 + 32 + lane, b0 + 32 + lane < b1);
  uint64_t v = 0;
  for (uint32_t b = b0 + 64 + lane; b < b1; b += 32) v += ld_now32(block_sums + b, true);
  *rest = v;
}
__device__ __forceinline__ uint64_t range_total(const uint32_t (&part)[kRangeParts], uint64_t rest) {
  // at most 62 chunks and 64 blocks of 32: below 2^27 bytes
  uint64_t v = __reduce_add_sync(0xffffffffu, part[0] + part[1] + part[2] + part[3]);
  if (__any_sync(0xffffffffu, rest != 0)) v += warp_sum_u64(rest);
  return v;
}

// Byte permute with the generic mode's sign replication (a selector nibble with bit 3 set
// fills the result byte with the top bit of the byte it selects).
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void sts128(uint32_t addr, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y),
               "f"(v.z), "f"(v.w)
               : "memory");
}
__device__ __forceinline__ float4 lds128(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}

// Inclusive prefix sum over a tile of x[0..31] in each lane, a tile's lanes (8 by default)
// carrying from one to the next: the lane's own prefix, then the exclusive scan of the lanes'
// totals, plus `add`. Without the carried state (indep) each block restarts. Lanes with
// `apply` false keep x; every lane of the warp must call this (the scan's shuffles take the
// full warp), and the lanes of a tile agree on `apply`, so the scan segments of applying
// tiles see only their own lanes.
template <bool kAny, typename Cfg>
__device__ __forceinline__ void tile_prefix(uint32_t (&x)[32], const uint32_t add, const bool indep,
                                            const bool apply) {
  // the lane's prefix as four independent 8-element runs (short dependency chains), the
  // runs' offsets folded into the final additions
  uint32_t o1 = 0, o2 = 0, o3 = 0, tot = 0;
  if (apply) {
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int i = 1; i < 8; ++i) x[8 * k + i] += x[8 * k + i - 1];
    o1 = x[7];
    o2 = o1 + x[15];
    o3 = o2 + x[23];
    tot = o3 + x[31];
  }
  uint32_t inc = tot;
#pragma unroll
  for (int o = 1; o < Cfg::kLanes; o <<= 1) inc = scan_step_up<Cfg::kLanes>(inc, o);
  uint32_t ex = inc - tot;
  if (kAny && indep) {
    ex = 0;
    if constexpr (Cfg::kBlockLanes == 2) {  // a 64-element block's second lane follows its first
      const uint32_t before = __shfl_up_sync(0xffffffffu, tot, 1);
      if (threadIdx.x & 1) ex = before;
    }
  }
  ex += add;
  if (apply) {
    const uint32_t e[4] = {ex, ex + o1, ex + o2, ex + o3};
#pragma unroll
    for (int i = 0; i < 32; ++i) x[i] += e[i >> 3];
  }
}

// Decodes one quad (1024 elements) with one warp into o, lane L elements 32 L .. 32 L + 31: a
// block, or half of a 64-element one (whose lanes' words alternate). flags: the first rate
// byte of the lane's tile; Rg: the rate of the lane's block; tp, blk: shared-memory addresses
// of the tile's data and of the lane's first word; live: the tile exists. Returns false if a
// tile's mean slot is malformed. kAny: the instance that also decodes streams without the
// cross-block state (`indep`: every block restarts from zero predecessors).
template <bool kAny, typename Cfg>
__device__ __forceinline__ bool decompress_quad(const uint32_t flags, const int Rg, const uint32_t tp,
                                                const uint32_t blk, const bool live, const float s,
                                                const bool indep, float (&o)[32]) {
  constexpr uint32_t FULL = 0xffffffffu;
  constexpr uint32_t W = Cfg::kWordBytes;
  const bool second = (flags & 0x80u) != 0, centred = (flags & 0x40u) != 0;
  bool good = true;
  int mu = 0;
  if (live && centred) {
    const float muf = __uint_as_float(lds32(tp));
    if (!(fabsf(muf) <= 16777216.0f)) {
      good = false;
    } else {
      mu = __float2int_rn(muf);
      if (__int2float_rn(mu) != muf) good = false;
    }
  }
  // d4: the block's planes (sign map, then the magnitude bits) become the planes of the
  // two's-complement residuals by a bit-sliced negation of the negative elements,
  // x = (m ^ S) + S over all 32 elements at once (S the sign map); the planes above the
  // rate then all equal the result's sign plane. They go back through the plane network,
  // and each element is gathered from its bytes by permutes that replicate the top byte's
  // sign, which sign-extends it.
  const int Rmax = int(__reduce_max_sync(FULL, uint32_t(Rg)));
  const int nch = Rmax > 0 ? (Rmax + 8) >> 3 : 0;
  uint32_t X[4][8];
  {
    const uint32_t S = Rg > 0 ? lds32(blk) : 0u;
    uint32_t carry = S;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (c < nch) {
#pragma unroll
        for (int b = 0; b < 8; ++b) {
          const int j = 8 * c + b;  // plane j of x: magnitude plane j is the block's word j + 1
          const uint32_t M = j < Rg ? lds32(blk + W * uint32_t(j + 1)) : 0u;
          const uint32_t y = M ^ S;
          X[c][b] = y ^ carry;
          carry &= y;
        }
        swap_planes(X[c]);
      }
    }
  }
  // byte m of X[c][k] is byte c of element 8 m + 7 - k
  uint32_t x[32];
  if (nch == 0) {
#pragma unroll
    for (int i = 0; i < 32; ++i) x[i] = 0u;
  } else if (nch == 1) {
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
      for (int m = 0; m < 4; ++m)
        x[8 * m + 7 - k] = prmt(X[0][k], 0u, m | ((8 | m) << 4) | ((8 | m) << 8) | ((8 | m) << 12));
  } else if (nch == 2) {
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
      for (int m = 0; m < 4; ++m)
        x[8 * m + 7 - k] = prmt(X[0][k], X[1][k], m | ((4 + m) << 4) | ((12 + m) << 8) | ((12 + m) << 12));
  } else if (nch == 3) {
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const uint32_t t = prmt(X[0][k], X[1][k], m | ((4 + m) << 4));
        x[8 * m + 7 - k] = prmt(t, X[2][k], 0x0010u | ((4 + m) << 8) | ((12 + m) << 12));
      }
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const uint32_t t = prmt(X[0][k], X[1][k], m | ((4 + m) << 4));
        const uint32_t u = prmt(X[2][k], X[3][k], (m << 8) | ((4 + m) << 12));
        x[8 * m + 7 - k] = prmt(t, u, 0x7610u);
      }
  }
  // d5: inverse prediction. With zero predecessors, LZ1's q_i = l_i + q_{i-1} is an
  // inclusive prefix sum over the tile; LZ2's q_i = l_i + 2 q_{i-1} - q_{i-2} is the prefix
  // sum of the prefix sum (the first sum rebuilds the LZ1 residuals); then + mu. The
  // quad's tiles may differ in their predictor: the first sum runs on the whole warp and
  // applies to the LZ2 tiles only.
  if (__any_sync(FULL, second)) tile_prefix<kAny, Cfg>(x, 0u, indep, second);
  tile_prefix<kAny, Cfg>(x, uint32_t(mu), indep, true);
#pragma unroll
  for (int i = 0; i < 32; ++i) o[i] = __fmul_rn(__int2float_rn(int(x[i])), s);
  return __all_sync(FULL, good);
}

// The CTA's barrier 0, from whichever branch a warp is in.
__device__ __forceinline__ void cta_sync() { asm volatile("barrier.sync 0;" ::: "memory"); }

// What the header warp needs of a field.
struct Field {
  const uint8_t* sin;
  float* dout;
  uint64_t in_bytes, n, T, data_bytes;
  uint64_t first;  // global index of the field's first chunk
  uint32_t features_off;
  float s;
};

__device__ __forceinline__ Field field_of_record(const FieldInfo* fi) {
  return Field{fi->sin, fi->dout, fi->in_bytes, fi->n, fi->T, fi->data_bytes, fi->chunk_first,
               fi->features_off, fi->s};
}

// The field of a one-field call, from the preamble as it stands: within the stream's buffer
// and the output's capacity whatever it says.
template <typename Cfg>
__device__ __forceinline__ Field field_of_stream(const KernelArgs& a) {
  Field f = {};
  f.sin = a.sin;
  f.dout = a.dout;
  f.in_bytes = a.in_bytes;
  if (a.in_bytes < 64) return f;
  const uint4* p = reinterpret_cast<const uint4*>(a.sin);
  const uint4 w0 = p[0], w3 = p[3];
  f.n = min(uint64_t(w0.z) | (uint64_t(w0.w) << 32), a.cap_elems);
  f.T = min((f.n + Cfg::kElems - 1) / Cfg::kElems, (a.in_bytes - 64) / Cfg::kT);
  f.s = __uint_as_float(w3.x);
  f.features_off = w3.y;
  f.data_bytes = uint64_t(w3.z) | (uint64_t(w3.w) << 32);
  return f;
}

// kAny: also decodes streams without the cross-block state. kPrezero: the output already
// holds zeros; tiles whose 8 blocks all have rate 0 and no mean (all +0.0) are neither
// decoded nor written (the adaptive pre-zero of Sec. 3.1 for high compression ratios).
// Cfg: the tile configuration. kChecked: a tiled call, whose set-up kernel has checked every rate
// header; nothing is decoded if it found one malformed, or sizes that do not add up to the data's.
template <bool kAny, bool kPrezero, bool kChecked, typename Cfg>
__device__ __forceinline__ void decompress_cta(const KernelArgs& a) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  DecompressSmem& S = *reinterpret_cast<DecompressSmem*>(smem_raw);
  constexpr uint32_t FULL = 0xffffffffu;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t wait_ns = 4 * a.timeout_ns;
  const uint32_t recs = a.records;

  if (tid == 0) {
    for (int k = 0; k < kMaxRecs; ++k) {
      mbar_init(&S.fetched[k], 1);
      mbar_init(&S.full[k], 1);
      mbar_init(&S.done[k], kDecodeWarps);
    }
    fence_mbar_init();
  }
  // (the header warp reads ahead before it waits)
  if (warp != kHeaderWarp) {
    grid_wait();
    cta_sync();
  } else {
    // ---------------------------------------------------------------- header warp
    // A ticket is a group of up to kMaxTicketChunks consecutive chunks; lane g keeps and writes
    // what concerns chunk g as a whole, all lanes its tiles (lane = tile), the chunks side by
    // side. This warp feeds all the others and shares their issue slots: with the chunks one
    // after another and a ticket's atomic and loads in line it was the slowest stage, and still
    // was for launches of 1-chunk tickets (3 us each) until the scans were packed two to a
    // register and the rest trimmed. Whole calls, at first / chunks side by side / trimmed:
    // 512^3 118.5, 113.8, 112.6 us; 16 M particles 29.5, 25.1, 22.1 us; batch of 32 fields
    // 75.7, 70.0, 69.7 us.
    // (chunk numbers fit 32 bits: at most 2^27 and one per field)
    const bool single = a.sin != nullptr;
    Field f = {};        // lane g: chunk g's field (one field: the same in every lane)
    uint32_t total = 0;  // chunks of the launch
    uint32_t c0 = 0;     // the group's first chunk
    uint32_t group = 1;
    uint64_t h[kMaxTicketChunks];  // the lane's unit of rate bytes in each chunk, 0 beyond the field
    uint32_t nt = 0;               // lane g: tiles of chunk g, 0 if there is none
    uint32_t fidx = 0;             // lane g: chunk g's field
    // the end of the previous group: the chunk after it, its offset in its field
    uint32_t prev_end = 0;
    uint64_t prev_excl = 0;
    uint32_t first0 = 0;  // the first chunk of the group's first field
    uint32_t part[kRangeParts];
    uint64_t part_rest = 0;
    // Tickets 0 .. nbig - 1 are `full` chunks, the launch's last ones at most kTailTicket.
    uint32_t full = 1, nbig = 0;
    auto launch_tickets = [&]() {
      full = launch_ticket_chunks(a.ticket_chunks, a.min_tickets, total, gridDim.x);
      nbig = total > gridDim.x * kTailChunks ? (total - gridDim.x * kTailChunks) / full : 0;
      if (a.min_tickets == 0) nbig = (total + full - 1) / full;
    };
    auto place = [&](uint32_t t) {
      const bool big = t < nbig;
      group = big ? full : min(full, kTailTicket);
      c0 = big ? t * full : nbig * full + (t - nbig) * group;
    };
    auto fetch_headers = [&]() {
      const uint32_t c = c0 + lane;
      const bool mine = uint32_t(lane) < group && c < total;
      if (!single && mine) {
        fidx = a.chunk_field[c];
        f = field_of_record(a.fields + fidx);
      }
      const uint64_t t0 = uint64_t(c - uint32_t(f.first)) * Cfg::kChunkTiles;
      nt = mine ? uint32_t(min(uint64_t(Cfg::kChunkTiles), f.T - t0)) : 0u;
      const uint64_t hp = reinterpret_cast<uint64_t>(f.sin) + 64 + Cfg::kT * t0;
#pragma unroll
      for (int g = 0; g < kMaxTicketChunks; ++g) {
        h[g] = 0;
        if (uint32_t(g) < group) {
          const uint64_t p = __shfl_sync(FULL, hp, g) + 8 * lane;
          const uint32_t end = Cfg::kT * __shfl_sync(FULL, nt, g);  // rate bytes of the chunk
          h[g] = ld_now(reinterpret_cast<const void*>(p), 8u * lane + 8u <= end);
          if (Cfg::kT == 4 && 8u * lane + 4u == end)  // an odd number of 4-block tiles
            h[g] = __ldg(reinterpret_cast<const uint32_t*>(p));
        }
      }
    };
    // d3: a CTA's chunks only go up, so the previous group ended in this one's field if it ended
    // behind the field's first chunk: the offset counts from there, or from the field's start
    auto fetch_sizes = [&]() {
      first0 = __shfl_sync(FULL, uint32_t(f.first), 0);
      const uint32_t from = max(prev_end, first0);
      range_fetch(a.sums, a.block_sums, from, c0 < total ? c0 : from, part, &part_rest);
    };
    if (single) {
      // One field: its preamble and the headers of the CTA's first ticket (its own number) are
      // read under the set-up kernel, which does not write them; what the preamble says counts
      // only once that kernel's verdict (the control words' chunk count) is in.
      f = field_of_stream<Cfg>(a);
      total = uint32_t((f.T + Cfg::kChunkTiles - 1) / Cfg::kChunkTiles);
      launch_tickets();
      place(blockIdx.x);
      fetch_headers();
    }
    grid_wait();
    cta_sync();
    const uint32_t verdict = uint32_t(a.ctrl->total_chunks);
    if (!single) {
      total = verdict;
      launch_tickets();
      place(blockIdx.x);
      fetch_headers();
    }
    fetch_sizes();
    if (verdict == 0) nt = 0;
    total = verdict;
    const uint32_t off_bits = forbidden_flags(f.features_off);
    uint32_t r0 = 0;  // the group's first record: seq % recs
    for (uint32_t seq = 0;;) {
      uint32_t next = 0;
      if (lane == 0) next = gridDim.x + atomicAdd(&a.ctrl->ticket, 1u);
      // the group's records must be free: their previous chunks decoded (the decode warps
      // finish chunks in order, so the last record's tells)
      const uint32_t sl = seq + group - 1;
      const uint32_t ahead = c0 < nbig * full ? recs : min(recs, kTailAhead);
      if (sl >= ahead) {
        const uint32_t w = sl - ahead;
        if (!mbar_wait(&S.done[w % recs], (w / recs) & 1u, wait_ns)) {
          if (lane == 0) set_error(a.ctrl, nullptr, FSZ_ERR_TIMEOUT);
          return;
        }
      }
      // d2: sizes and their scans, two chunks to a register (a chunk is below 2^16 bytes)
      uint32_t mine[kMaxTicketChunks], inc[kMaxTicketChunks / 2];
#pragma unroll
      for (int k = 0; k < kMaxTicketChunks / 2; ++k) {
        mine[2 * k] = unit_bytes(h[2 * k], Cfg::kB, Cfg::kT, lane);
        mine[2 * k + 1] = unit_bytes(h[2 * k + 1], Cfg::kB, Cfg::kT, lane);
        inc[k] = mine[2 * k] | (mine[2 * k + 1] << 16);
      }
#pragma unroll
      for (int o = 1; o < 32; o <<= 1)
#pragma unroll
        for (int k = 0; k < kMaxTicketChunks / 2; ++k) inc[k] = scan_step_up<32>(inc[k], o);
      // a tile may not use a feature the stream has switched off; streams without the
      // cross-block state are decoded by the kAny instance only
      const bool unsupported = !kAny && (f.features_off & kOffCross) && nt > 0;
      if (unsupported) set_error(a.ctrl, a.fields + fidx, FSZ_ERR_INVALID_ARG);
      const uint32_t forbid = single ? off_bits : forbidden_flags(f.features_off);
      const bool any_forbid = __any_sync(FULL, forbid != 0);
      uint32_t bad = 0;
#pragma unroll
      for (int g = 0; g < kMaxTicketChunks; ++g) {
        uint64_t not_allowed = 0;
        if (any_forbid) not_allowed = __shfl_sync(FULL, forbid, g) * unit_centring_bits(Cfg::kT, lane);
        if (header_reserved_bits_set(h[g], Cfg::kT, lane) || (h[g] & not_allowed) != 0) bad |= 1u << g;
      }
      bad = __reduce_or_sync(FULL, bad);
      // offsets: each chunk follows from its predecessor, or starts its field
      const uint32_t starts = __ballot_sync(FULL, c0 + lane == uint32_t(f.first));
      uint64_t excl = range_total(part, part_rest) + (prev_end > first0 ? prev_excl : 0);
      uint64_t my_excl = 0;
      uint32_t my_tot = 0;
      const uint32_t last[2] = {__shfl_sync(FULL, inc[0], 31), __shfl_sync(FULL, inc[1], 31)};
#pragma unroll
      for (int g = 0; g < kMaxTicketChunks; ++g) {
        const uint32_t tot = (last[g / 2] >> (16 * (g & 1))) & 0xffffu;
        if ((starts >> g) & 1u) excl = 0;
        if (lane == g) {
          my_tot = tot;
          my_excl = excl;
        }
        if (uint32_t(g) < group) excl += tot;
      }
      // the records
      uint32_t r = r0, my_r = 0;
#pragma unroll
      for (int g = 0; g < kMaxTicketChunks; ++g) {
        if (uint32_t(g) < group) {
          ChunkRec& q = S.rec[r];
          q.hdr[lane] = h[g];
          q.boff[lane] = block_word_offsets(h[g]);
          q.toff[lane] = ((inc[g / 2] >> (16 * (g & 1))) & 0xffffu) - mine[g];
          if (lane == g) my_r = r;
          if (++r == recs) r = 0;
        }
      }
      r0 = r;
      if (uint32_t(lane) < group) {
        ChunkRec& q = S.rec[my_r];
        const uint64_t lc = c0 + lane - uint32_t(f.first);
        q.chunk = nt > 0 ? c0 + lane : kNoneChunk;
        q.last = (lc + 1) * Cfg::kChunkTiles >= f.T ? 1u : 0u;
        q.tot = my_tot;
        q.bad = unsupported ? 1u : (bad >> lane) & 1u;
        q.fi = a.fields + fidx;
        q.sin = f.sin;
        q.in_bytes = f.in_bytes;
        q.data_bytes = f.data_bytes;
        q.data_base = 64 + Cfg::kT * f.T;
        q.excl = my_excl;
        q.dout = f.dout + lc * kDChunkElems;
        q.ntiles = nt;
        q.cnt = uint32_t(min(f.n - lc * kDChunkElems, uint64_t(kDChunkElems)));
        q.step = f.s;
        q.indep = (f.features_off & kOffCross) ? 1u : 0u;
      }
      __syncwarp();
      // (test hook: the record of skip_chunk is never handed over, nor any after it)
      const bool held = a.skip_chunk >= c0 && a.skip_chunk <= c0 + lane;
      // ... and after the launch's last chunk one record says that there are no more
      const uint32_t live = total > c0 ? min(total - c0, group) : 0u;
      if (uint32_t(lane) < group && !held && uint32_t(lane) <= live) mbar_arrive(&S.fetched[my_r]);
      if (c0 + group > total || __any_sync(FULL, uint32_t(lane) < group && held)) return;
      prev_end = c0 + group;
      prev_excl = excl;
      seq += group;
      place(__shfl_sync(FULL, next, 0));
      fetch_headers();
      fetch_sizes();
    }
  }

  if (warp == kLoaderWarp) {
    // ---------------------------------------------------------------- loader warp
    // Ring positions count bytes modulo 2^32: head = where the next payload goes, freed =
    // how far the decoded chunks have released. Chunks take and release space in ticket
    // order, so the bytes in use are head - freed; pos is head's place in the ring.
    uint32_t head = 0, freed = 0, pos = 0;
    uint32_t oldest = 0;  // the oldest chunk whose bytes are not yet known to be released
    // A tiled call's rate headers as the set-up kernel found them (here, where it costs nothing: the
    // first record is still being made; in the header warp it cost 1 us of 23).
    uint64_t headers = 0;
    if constexpr (kChecked) {
      bool malformed = false;
      for (uint32_t k = lane; k < a.nfound; k += 32) {
        const uint64_t found = __ldcg(reinterpret_cast<const unsigned long long*>(a.found) + k);
        malformed |= found == kHeadersBad;
        headers += found;
      }
      headers = __any_sync(FULL, malformed) ? kHeadersBad : warp_sum_u64(headers);
    }
    for (uint32_t seq = 0;; ++seq) {
      const int r = int(seq % recs);
      if (!mbar_wait(&S.fetched[r], (seq / recs) & 1u, wait_ns)) {
        if (lane == 0) set_error(a.ctrl, nullptr, FSZ_ERR_TIMEOUT);
        return;
      }
      ChunkRec& q = S.rec[r];
      if (q.chunk == kNoneChunk) {
        if (lane == 0) mbar_arrive(&S.full[r]);
        return;
      }
      FieldInfo* fi = q.fi;
      const uint32_t tot = q.tot;
      const uint64_t excl = q.excl;
      bool valid = q.bad == 0;
      if (q.data_base + excl + tot > q.in_bytes) valid = false;
      if (q.last && excl + tot != q.data_bytes) valid = false;
      if (kChecked && headers != q.data_bytes) valid = false;
      const uint64_t base = reinterpret_cast<uint64_t>(q.sin);
      const uint64_t src = base + q.data_base + excl;
      const uint64_t a0 = src & ~uint64_t(15);
      // Round the copy's end up to 16 bytes while that stays inside the stream buffer;
      // otherwise the last few bytes come by plain loads.
      const uint64_t end_up = (src + tot + 15) & ~uint64_t(15);
      const uint64_t a1 = end_up <= base + q.in_bytes ? end_up : ((src + tot) & ~uint64_t(15));
      const uint32_t bulk = (valid && a1 > a0) ? uint32_t(a1 - a0) : 0u;
      // ring space: the payload from a0, rounded up to 16 bytes, in one piece (a payload
      // that would run past the ring's end starts at the ring's start instead)
      const uint32_t need = valid ? (uint32_t(src - a0) + tot + 15u) & ~15u : 0u;
      uint32_t start = head, phys = pos;
      if (pos + need > kRingBytes) {
        start += kRingBytes - pos;
        phys = 0;
      }
      // Chunks seq - recs and older are decoded: the header warp reused their records.
      while (oldest + recs <= seq) freed = S.ring_end[oldest++ % recs];
      bool space = true;
      while (start + need - freed > kRingBytes) {
        if (oldest == seq) {  // nothing in flight: the skipped end of the ring is free too
          freed = start;
          break;
        }
        // wait for the oldest chunk in flight; its record is not reused before it is done
        if (!mbar_wait(&S.done[oldest % recs], (oldest / recs) & 1u, wait_ns)) {
          space = false;
          break;
        }
        freed = S.ring_end[oldest % recs];
        ++oldest;
      }
      if (!space) {
        if (lane == 0) set_error(a.ctrl, nullptr, FSZ_ERR_TIMEOUT);
        return;
      }
      head = start + need;
      pos = phys + need;
      if (lane == 0) S.ring_end[r] = head;
      if (lane == 0) {
        if (!valid) set_error(a.ctrl, fi, FSZ_ERR_CORRUPT);
        q.pay = phys + uint32_t(src - a0);
        q.valid = valid ? 1u : 0u;
        if (bulk) {
          fence_proxy_async();
          mbar_expect_tx(&S.full[r], bulk);
          tma_load_1d(S.ring + phys, reinterpret_cast<const void*>(a0), bulk, &S.full[r]);
        }
      }
      if (valid) {
        // Payload bytes past the last 16-byte boundary of the bulk copy: plain loads.
        const uint32_t lo = uint32_t(max(a1, src) - a0), hi = uint32_t(src + tot - a0);
        const uint8_t* gb = reinterpret_cast<const uint8_t*>(a0);
        for (uint32_t k = lo + 4 * uint32_t(lane); k < hi; k += 128)
          *reinterpret_cast<uint32_t*>(S.ring + phys + k) = *reinterpret_cast<const uint32_t*>(gb + k);
      }
      __threadfence_block();  // every lane's tail bytes before lane 0's arrival
      __syncwarp();
      if (lane == 0) mbar_arrive(&S.full[r]);
    }
  }

  // ------------------------------------------------------------------ decode warps
  const uint32_t obuf = smem_u32(S.out[warp]);
  bool good = true;
  for (uint32_t seq = 0;; ++seq) {
    const int r = int(seq % recs);
    if (!mbar_wait(&S.full[r], (seq / recs) & 1u, wait_ns)) {
      if (lane == 0) set_error(a.ctrl, nullptr, FSZ_ERR_TIMEOUT);
      break;
    }
    const ChunkRec& st = S.rec[r];
    const uint32_t c = st.chunk;
    if (c == kNoneChunk) break;
    FieldInfo* fi = st.fi;
    if (st.valid) {
      const float step = st.step;
      const int ntiles = int(st.ntiles);
      const uint32_t cnt = st.cnt;
      float* dout = st.dout;
      const uint32_t pay = smem_u32(S.ring) + st.pay;
      const int t = Cfg::kQuadTiles * warp + lane / Cfg::kLanes;  // the lane's tile in the chunk
      const bool live = t < ntiles;
      // the lane's block: byte j of header unit u; the unit that begins its tile is uf
      const int u = (Cfg::kB == 32 ? 4 * warp + (lane >> 3) : 2 * warp + (lane >> 4));
      const int j = (Cfg::kB == 32 ? lane : lane >> 1) & 7;
      const int uf = Cfg::kT == 16 ? u & ~1 : u;
      const uint64_t h = live ? st.hdr[u] : 0ull;
      const uint64_t hf = Cfg::kT == 16 ? (live ? st.hdr[uf] : 0ull) : h;
      const uint32_t flags = uint32_t(Cfg::kT == 4 ? h >> (8 * (j & 4)) : hf) & 0xFFu;
      // a pre-zeroed output: a tile whose rates are all 0 and that has no mean is +0.0
      // throughout, neither decoded nor written; a quad of such tiles is skipped
      const bool write_tile = live && (!kPrezero || (h & 0x1F1F1F1F1F1F1F5FULL) != 0);
      const uint32_t tmask = __ballot_sync(FULL, write_tile);
      if (tmask != 0) {
        const uint64_t boff = live ? st.boff[u] : 0ull;
        // d2: the unit's data, the means before the block in it, and the block's word offset
        // (a byte-wise prefix sum by the header warp)
        uint32_t blk = pay + (live ? st.toff[u] : 0u);
        uint32_t tp = Cfg::kT == 16 ? pay + (live ? st.toff[uf] : 0u) : blk;
        blk += Cfg::kWordBytes * uint32_t((boff >> (8 * j)) & 0xFFu) + 4u * uint32_t(lane % Cfg::kBlockLanes);
        if (Cfg::kT == 4) {  // the unit's first tile's mean, then the second's
          if (h & 0x40u) blk += 4u;
          if (j & 4) {
            tp += Cfg::kWordBytes * uint32_t((boff >> 32) & 0xFFu) + ((h & 0x40u) ? 4u : 0u);
            if (flags & 0x40u) blk += 4u;
          }
        } else if (u == uf && (flags & 0x40u)) {
          blk += 4u;  // (a 16-block tile's second unit starts after the mean)
        }
        float o[32];
        good = decompress_quad<kAny, Cfg>(flags, live ? int((h >> (8 * j)) & 31u) : 0, tp, blk, live, step,
                                          st.indep != 0, o);
        // re-layout: lane L's block goes to row L of the buffer, 16-byte piece k at column
        // k ^ (L & 7) (conflict-free); then each piece P = 32 j + lane, read back in order,
        // is stored to the output, the warp writing 512 consecutive bytes per store
        const uint32_t row = obuf + uint32_t(lane) * 128u;
        const uint32_t sw = uint32_t(lane & 7) << 4;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          sts128(row + ((uint32_t(k << 4)) ^ sw), make_float4(o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3]));
        __syncwarp();
        const uint32_t e0 = uint32_t(kQuadElems * warp);  // the quad's first element
        if (tmask == FULL && e0 + kQuadElems <= cnt) {
          // every tile of the quad is written in full: no per-store guards
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint32_t P = uint32_t(32 * j + lane);   // piece: row P >> 3, column P & 7
            const uint32_t rw = P >> 3;
            const float4 val = lds128(obuf + rw * 128u + (((P & 7u) ^ (rw & 7u)) << 4));
            *reinterpret_cast<float4*>(dout + e0 + 4 * P) = val;
          }
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const uint32_t P = uint32_t(32 * j + lane);
            const uint32_t rw = P >> 3;
            const float4 val = lds128(obuf + rw * 128u + (((P & 7u) ^ (rw & 7u)) << 4));
            const uint32_t e = e0 + 4 * P;
            if (!((tmask >> rw) & 1u)) continue;  // (a tile not written)
            if (e + 4 <= cnt) {
              *reinterpret_cast<float4*>(dout + e) = val;
            } else {
              const float vals[4] = {val.x, val.y, val.z, val.w};
#pragma unroll
              for (int i = 0; i < 4; ++i)
                if (e + i < cnt) dout[e + i] = vals[i];
            }
          }
        }
        __syncwarp();  // the buffer is read before the next quad overwrites it
      }
    }
    if (!good && lane == 0) set_error(a.ctrl, fi, FSZ_ERR_CORRUPT);
    good = true;
    __syncwarp();
    if (lane == 0) mbar_arrive(&S.done[r]);
  }
}

template <bool kAny, bool kPrezero>
__global__ void __launch_bounds__(kThreads, 2) fsz_decompress_kernel(KernelArgs a) {
  decompress_cta<kAny, kPrezero, false, DefaultCfg>(a);
}

// Any tile configuration: the stream's own, from its preamble (a configuration that does not
// exist is refused by the set-up kernel; this one then finds no chunks). One kernel that
// branches once, because the host does not know the configuration: with one launch per
// configuration, five of them returning at once, a scan of the tile sizes in three launches
// and one warp per tile, a 256^3 field at 64 x 8 took 93 us; this takes 26 us with its set-up.
__global__ void __launch_bounds__(kThreads, 2) fsz_decompress_tiled_kernel(KernelArgs a) {
  int B = 32, T = 8;
  if (a.in_bytes < 64 || !config_of(*reinterpret_cast<const uint32_t*>(a.sin + 52), &B, &T)) B = 32, T = 8;
  if (B == 32) {
    if (T == 4) decompress_cta<true, false, true, TileCfg<32, 4>>(a);
    else if (T == 8) decompress_cta<true, false, true, TileCfg<32, 8>>(a);
    else decompress_cta<true, false, true, TileCfg<32, 16>>(a);
  } else {
    if (T == 4) decompress_cta<true, false, true, TileCfg<64, 4>>(a);
    else if (T == 8) decompress_cta<true, false, true, TileCfg<64, 8>>(a);
    else decompress_cta<true, false, true, TileCfg<64, 16>>(a);
  }
}

}  // namespace

LaunchCfg decompress_cfg() {
  static DeviceCfgCache cache;
  return cache.get([] {
    LaunchCfg c;
    c.smem = int(sizeof(DecompressSmem));
    auto allow = [&](auto kernel) {
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, c.smem);
    };
    allow(fsz_decompress_kernel<false, false>);
    allow(fsz_decompress_kernel<true, false>);
    allow(fsz_decompress_kernel<false, true>);
    allow(fsz_decompress_tiled_kernel);
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fsz_decompress_kernel<false, false>,
                                                  kThreads, c.smem);
    c.sms = sms;
    c.per = per > 0 ? per : 1;
    c.grid = sms * c.per;
    return c;
  });
}

namespace {
void launch(void (*kernel)(KernelArgs), const KernelArgs& args, uint64_t max_chunks, cudaStream_t st) {
  const LaunchCfg c = decompress_cfg();
  KernelArgs a = args;
  a.ticket_chunks = uint32_t(g_schedule.d_ticket_chunks);
  a.records = uint32_t(g_schedule.d_records);
  a.min_tickets = uint32_t(g_schedule.min_tickets);
  launch_dependent(kernel, sched_grid(c, kSchedDecompress, max_chunks), kThreads, c.smem, st, a);
}
}  // namespace

void launch_decompress(const KernelArgs& a, uint64_t max_chunks, cudaStream_t st, DecompressKind kind) {
  if (kind == kDecompressAny)
    launch(fsz_decompress_kernel<true, false>, a, max_chunks, st);
  else if (kind == kDecompressPrezeroed)
    launch(fsz_decompress_kernel<false, true>, a, max_chunks, st);
  else if (kind == kDecompressTiled)
    launch(fsz_decompress_tiled_kernel, a, max_chunks, st);
  else
    launch(fsz_decompress_kernel<false, false>, a, max_chunks, st);
}

}  // namespace fsz
