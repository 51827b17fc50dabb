// FSZ single-pass compression kernel (Sec. 3.1 steps 1-5, Sec. 4).
//
// Persistent, warp-specialised CTAs (two per SM); the roles hand work to one another
// through mbarriers and shared counters (no CTA-wide barrier in the main loop):
//   compute warps  (kWarps) each stream their own quad (4 tiles) of every chunk into a
//                  private staging buffer with cp.async (16-byte pieces, zero-filled past
//                  the end of the field), one chunk ahead of the one they encode. Lane L of
//                  a warp holds block L & 7 of tile L >> 3 of its quad: 32 consecutive
//                  elements, read from the buffer with conflict-free 128-bit loads (the
//                  pieces sit in a 128-byte swizzled layout). They quantize, predict,
//                  evaluate the four variants, select and size the quad's tiles (steps 1-3;
//                  the input is read from HBM once), write the rate headers, and encode the
//                  quad as one contiguous run into the warp's ring in shared memory
//                  (step 5). The last warp to size a chunk scans the quads' sizes and
//                  publishes the chunk's aggregate flag before any warp has encoded it;
//   resolver warp  looks back for each chunk's exclusive byte offset (step 4, Sec. 4.4),
//                  publishes the inclusive prefix, and copies the runs of the first
//                  kResolverRuns compute warps to the stream before handing the chunk to
//                  the host warp;
//   host warp      takes a ticket per chunk just ahead of its use and leaves the chunk's
//                  parameters in one of kSets chunk slots; and places each chunk, once it
//                  is resolved and encoded, by copying the other compute warps' runs from
//                  their rings to the stream and giving the ring space back.
// The rings decouple encoding from the device-wide scan: chunks finish out of ticket order
// across the grid, and a chunk's offset is known only when every earlier chunk has
// published its size. Keeping the placement out of the compute warps keeps them within 96
// registers, so that 16 of them fit on an SM.
#include "fsz_internal.cuh"

namespace fsz {

namespace {

constexpr uint32_t FULL = 0xffffffffu;
constexpr int kQuadElems = 1024;                   // elements per compute warp and chunk
constexpr int kWarps = kCChunkElems / kQuadElems;  // compute warps per CTA
constexpr int kHostWarp = kWarps;                  // tickets and placement
constexpr int kResolverWarp = kWarps + 1;
constexpr int kThreads = (kWarps + 2) * 32;
#ifndef FSZ_RESOLVER_RUNS
#define FSZ_RESOLVER_RUNS 4
#endif
// Placement split: the resolver copies the runs of compute warps 0 .. kResolverRuns - 1 of
// each chunk it resolves, before handing the chunk to the host, which copies the others.
constexpr int kResolverRuns = FSZ_RESOLVER_RUNS;
#ifndef FSZ_COMPRESS_SETS
#define FSZ_COMPRESS_SETS 12
#endif
#ifndef FSZ_RING_BYTES
#define FSZ_RING_BYTES 6144
#endif
constexpr int kSets = FSZ_COMPRESS_SETS;           // chunk slots per CTA
// The schedule's work assignment (kernel arguments): a ticket hands a CTA ticket_chunks
// consecutive chunks, and a chunk that follows the CTA's previous chunk in the same field
// takes its byte offset from it (the previous offset plus its size) instead of looking
// back; the ticket of chunk seq is taken when the compute warps begin chunk
// seq - ticket_lead.
static_assert(kMaxTicketChunks + kMaxCompressLead <= FSZ_COMPRESS_SETS, "schedule limits");
#ifndef FSZ_COMPRESS_CTAS
#define FSZ_COMPRESS_CTAS 2
#endif
constexpr int kCtasPerSm = FSZ_COMPRESS_CTAS;
constexpr int kQuadBytes = 4 * kQuadElems;         // 4096: a warp's staging buffer
constexpr int kMaxQuadOut = 4 * kMaxTileBytes;
// ... of any tile configuration: 32 blocks (or halves) of at most 24 words, up to 8 means
constexpr int kMaxCfgQuadOut = 32 * 4 * 24 + 8 * 4;
// Ring bytes per compute warp. A run is contiguous: one that would run past the end
// starts at the ring's start instead, and the bytes it skips count as its own until it
// is placed.
constexpr int kRingAlloc = FSZ_RING_BYTES + kMaxQuadOut;
#ifndef FSZ_LOOKBACK_K
#define FSZ_LOOKBACK_K 1
#endif
constexpr int kLookbackPerLane = FSZ_LOOKBACK_K;   // lookback window: 32 K flags (64: +0.5 %)
constexpr uint32_t kNone = 0xffffffffu;
// Polling intervals of waits that sleep between tests (ns): the host warp, the resolver
// waiting for a chunk to be sized, the compute warps waiting for a ticket or ring space.
#ifndef FSZ_HOST_SLEEP_NS
#define FSZ_HOST_SLEEP_NS 100
#endif
#ifndef FSZ_RESOLVER_SLEEP_NS
#define FSZ_RESOLVER_SLEEP_NS 200
#endif
#ifndef FSZ_COMPUTE_SLEEP_NS
#define FSZ_COMPUTE_SLEEP_NS 100
#endif
constexpr uint32_t kHostSleepNs = FSZ_HOST_SLEEP_NS;
constexpr uint32_t kResolverSleepNs = FSZ_RESOLVER_SLEEP_NS;
constexpr uint32_t kComputeSleepNs = FSZ_COMPUTE_SLEEP_NS;
static_assert(kCChunkElems == kWarps * kQuadElems && kCChunkElems == kDChunkElems,
              "a chunk is one quad per compute warp");
static_assert(kRingAlloc >= 2 * kMaxQuadOut && kRingAlloc >= 2 * kMaxCfgQuadOut,
              "worst-case quads fit the ring");
static_assert(kRingAlloc % 16 == 0 && kQuadBytes % 1024 == 0, "alignment of the buffers");
static_assert(kWarps <= 32, "one lane per quad in the chunk scan");

// A chunk's parameters, read once from the field record by the host warp and kept in the
// chunk's slot until the chunk is placed. The compute warps read the first two 16-byte words.
// (What a chunk costs a warp apart from its quad was a third of its instructions: parameters
// worked out beforehand, slot counters instead of divisions and one acquire-release atomic
// instead of two fences around one took the kernel from 147 to 141 us at 512^3.)
constexpr uint32_t kInfoOk = 1u, kInfoLast = 2u, kInfoFirst = 4u, kInfoSkip = 8u, kInfoEnd = 16u;
struct __align__(16) ChunkInfo {
  uint32_t cnt;          // elements to load: the chunk's, or 0 (a field known to be refused, the
                         // end); not changed once the slot is handed over
  uint32_t ntiles;
  float r;
  uint32_t flags;        // kInfo* bits; kInfoEnd: no chunk, the CTA's chunks have run out
  const float* in;       // the chunk's first element
  uint8_t* hdr;          // its first rate-header byte
  uint8_t* out;          // the field's stream
  FieldInfo* fi;
  uint64_t tile0;        // field-local index of the chunk's first tile
  uint64_t data_base;    // start of the field's tile data, after the rate headers
  uint64_t cap;          // the field's output capacity
  uint32_t chunk;        // global chunk index, or kNone
  uint32_t chunk_first;  // global index of the field's first chunk
  uint32_t off;          // the field's switched-off features (kOff* bits)
};

struct __align__(1024) CompressSmem {
  float stage[kWarps][kQuadElems];                // per-warp staging (swizzled pieces)
  uint8_t ring[kWarps][kRingAlloc];               // encoded quads awaiting their offset
  ChunkInfo meta[kSets];
  uint64_t set_excl[kSets];                       // a resolved chunk's exclusive offset
  uint32_t qlen[kSets][kWarps];                   // each warp's quad run: bytes,
  uint32_t qoff[kSets][kWarps];                   // ... offset inside the chunk,
  uint2 qring[kSets][kWarps];                     // ... position in the warp's ring, and ring
                                                  // bytes it holds (run + skipped end)
  uint32_t set_tot[kSets];
  uint32_t done_cnt[kSets];
  uint32_t ring_tail[kWarps];                     // ring bytes given back, per compute warp
  uint64_t info[kSets], computed[kSets], encoded[kSets], resolved[kSets], started[kSets];
};

static_assert(sizeof(CompressSmem) <= 227 * 1024, "shared memory of one CTA");

// Eq. 3: S_b = 0 for r_b = 0, else 4 + 4 r_b; of a 64-element block, each of its two lanes'
// share.
__device__ __forceinline__ uint32_t block_cost(int R) {
  return (uint32_t(R) + (R != 0 ? 1u : 0u)) << 2;
}

// Bit length of a non-negative integer held in a float (Sec. 4.1.2: r_b = ceil(log2(max |l|
// + 1))), from its exponent.
__device__ __forceinline__ int bitlen(float x) {
  return max((__float_as_int(x) >> 23) - 126, 0);
}

// max(|a|, |b|, |c|)
__device__ __forceinline__ float max3_abs(float a, float b, float c) {
  float d;
  asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

// A magnitude m < 2^23 as a float m + 2^23 carries m in its mantissa bits.
constexpr float kMagBase = 8388608.0f;

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
// Copies the first `bytes` (0..16) of the piece and zero-fills the rest of it.
__device__ __forceinline__ void cp_async16_fill(uint32_t dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ void sts32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}

__device__ __forceinline__ void st_release_cta(uint32_t* p, uint32_t v) {
  asm volatile("st.release.cta.shared::cta.u32 [%0], %1;" ::"r"(smem_u32(p)), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t atom_add_acq_rel_cta(uint32_t* p, uint32_t v) {
  uint32_t old;
  asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], %2;"
               : "=r"(old)
               : "r"(smem_u32(p)), "r"(v)
               : "memory");
  return old;
}
__device__ __forceinline__ uint32_t ld_acquire_cta(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.cta.shared::cta.u32 %0, [%1];" : "=r"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}

__device__ __forceinline__ float4 lds128(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(addr));
  return v;
}

// Staging layout of a quad (4 KiB): the 16-byte piece at quad offset o sits at
// o ^ (((o >> 7) & 7) << 4), so piece k of block g (128 bytes) lands in column k ^ g of the
// block's row and the 8 lanes reading piece k of blocks 0..7 hit 8 different bank groups.
//
// Issues the cp.async pieces of this warp's quad of a chunk: lane L copies pieces
// 32 j + L, j = 0..7 (each instruction of the warp reads 512 consecutive bytes). `qv` is
// the quad's count of valid elements (1..1024); pieces past it are zero-filled and read
// nothing beyond the field (their source operand is `safe`, the chunk's first element).
__device__ __forceinline__ void issue_quad(uint32_t buf, const float* src, uint32_t qv, int lane,
                                           const float* safe) {
  // piece 32 j + L is at byte 512 j + 16 L; its block is (4 j + (L >> 3)) & 7
  const uint32_t pe = uint32_t(16 * lane) ^ (uint32_t(lane >> 3) << 4);
  const uint32_t po = pe ^ 64u;
  const char* s = reinterpret_cast<const char*>(src) + 16 * lane;
  if (qv == uint32_t(kQuadElems)) {
#pragma unroll
    for (int j = 0; j < 8; ++j) cp_async16(buf + 512 * j + ((j & 1) ? po : pe), s + 512 * j);
  } else {
    const uint32_t vb = 4 * qv;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t o = uint32_t(512 * j + 16 * lane);
      const uint32_t nb = o >= vb ? 0u : min(16u, vb - o);
      cp_async16_fill(buf + 512 * j + ((j & 1) ? po : pe),
                      nb ? static_cast<const void*>(s + 512 * j) : static_cast<const void*>(safe), nb);
    }
  }
  cp_async_commit();
}

// One byte-slice (magnitude bit-planes 8c .. 8c + 7) of a block's words v[0..31] as the 8
// stream words of those planes (Sec. 4.3: element j at bit 31 - j, most significant byte
// first, so stored little-endian element j sits at bit 8 (j >> 3) + 7 - (j & 7)).
// X[k] gathers byte c of elements 7 - k, 15 - k, 23 - k, 31 - k: bit 8 m + i of X[k] is bit
// i of element 8 m + 7 - k. Three delta swaps between register pairs (k, k ^ 2^t) exchange
// bit t of the register index with bit t of the bit index i, after which register b holds
// bit b of element 8 m + 7 - k at bit 8 m + k: the stream word of plane 8c + b.
template <int c>
__device__ __forceinline__ void planes8(const uint32_t (&v)[32], uint32_t (&X)[8]) {
  constexpr uint32_t sel = uint32_t(c) | (uint32_t(4 + c) << 4);
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const uint32_t a = __byte_perm(v[7 - k], v[15 - k], sel);
    const uint32_t b = __byte_perm(v[23 - k], v[31 - k], sel);
    X[k] = __byte_perm(a, b, 0x5410);
  }
  swap_planes(X);
}

// Compresses one quad (1024 elements: 1 to 8 tiles, 4 in the default configuration) with one
// warp. Lane L holds elements 32 L .. 32 L + 31 in d: a block, or half of a 64-element one;
// g is the lane's number in its tile. `live`: the lane's tile exists. Writes the rate-header
// byte of the lane's block to hdr (the quad's header bytes are consecutive), and returns the
// lane's words' place in the quad's run, with the quad's run length in P.qlen; the words go
// to ring + offset by encode_block(). Switched-off features arrive as `restart` (this lane
// starts from zero predecessors: the tile's first lane, and every block's without the
// cross-block state) and as penalties pen2, pen3 (2^16 for the second-order and the centred
// variants when off). With kGiven the four tile costs come from `given` (this lane's tile,
// stride gT between variants): the multipass evaluation's encoding pass; they are equal, so
// the stream is the same.
struct QuadPlan {
  uint32_t v[32];   // the selected variant's residuals: magnitude in bits 0-22
  uint32_t signs;   // ... and their sign map, as the stream's word
  uint32_t off;     // byte offset of this lane's first word in the quad's run (the words of a
                    // block's lanes alternate)
  int R;            // the block's rate (0 for a dead tile): its planes, after the sign map
  uint32_t mu_off;  // byte offset of the tile's mean slot (lane g = 0 of a centred tile)
  bool mu_slot;
  float mu;
  uint32_t qlen;    // the quad's run length (uniform)
  int Rmax;         // largest live rate of the quad (uniform)
};

template <bool kGiven, typename Cfg>
__device__ __forceinline__ void plan_quad(const float (&d)[32], const float r, const int lane,
                                          const bool live, const bool restart, const int pen2,
                                          const int pen3, const uint32_t* __restrict__ given,
                                          const uint64_t gT, uint8_t* __restrict__ hdr,
                                          QuadPlan& P) {
  constexpr int LT = Cfg::kLanes;
  const int g = lane & (LT - 1);
  // Tile sum for centring (Sec. 4.2.2, variant 3) in the fixed order: the sums of elements
  // 8j..8j+7 left to right (four runs per lane: runs 4g .. 4g + 3), then a butterfly over
  // the run index by half the runs, a quarter, .. 4 (lanes xor LT / 2 .. 1 within the tile),
  // 2 and 1 (in-lane). Float addition is commutative, so both partners of a step get equal
  // sums.
  float R[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    float acc = d[8 * m];
#pragma unroll
    for (int i = 1; i < 8; ++i) acc = __fadd_rn(acc, d[8 * m + i]);
    R[m] = acc;
  }
#pragma unroll
  for (int o = LT / 2; o >= 1; o >>= 1)
#pragma unroll
    for (int m = 0; m < 4; ++m) R[m] = __fadd_rn(R[m], __shfl_xor_sync(FULL, R[m], o));
  const float S = __fadd_rn(__fadd_rn(R[0], R[2]), __fadd_rn(R[1], R[3]));

  // Step 1, quantize (Sec. 4.2.2): t = fl(d r) then the nearest integer, ties to even: Y holds
  // q + M as a float, exactly. Everything up to the magnitudes stays in floats: |q| < 2^21 and
  // every residual is below 2^23, so differences are exact, run on the multiply-add pipe
  // (the integer pipe is the busier one), and take |.| and a three-way maximum for free. The
  // kernel is bound by issue slots; against integers (differences, |.| and ORs, and the sign
  // multiplied into the words): 264 -> 232 warp instructions per tile, 163 -> 147 us at 512^3
  // REL 1e-3.
  float Y[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) Y[i] = __fadd_rn(__fmul_rn(d[i], r), kMagic);
  const float muY = __fadd_rn(__fmul_rn(__fmul_rn(S, 1.0f / float(Cfg::kElems)), r), kMagic);
  const float mu = __fsub_rn(muY, kMagic);

  // Residuals with the state carried across block boundaries (Eq. 2); the tile's first
  // predecessors are zero. LZ2 as the difference of LZ1 residuals:
  // l2_i = (q_i - q_{i-1}) - (q_{i-1} - q_{i-2}).
  float prevY = __shfl_up_sync(FULL, Y[31], 1, LT);
  float prevL = __shfl_up_sync(FULL, __fsub_rn(Y[31], Y[30]), 1, LT);
  if (restart) {
    prevY = kMagic;
    prevL = 0.0f;
  }
  const float l1_0 = __fsub_rn(Y[0], prevY);
  const float l2_0 = __fsub_rn(l1_0, prevL);
  const float l1_1 = __fsub_rn(Y[1], Y[0]);
  const float l2_1 = __fsub_rn(l1_1, l1_0);
  // Block maxima of |l|. rest* leave out the tile's first residual(s), the only ones centring
  // changes (Eq. 4). (three partial maxima each, so that the chains are short)
  float m1[3] = {fabsf(l1_1), 0.0f, 0.0f}, m2[3] = {0.0f, 0.0f, 0.0f};
  float lp = l1_1;
#pragma unroll
  for (int i = 2; i < 32; i += 2) {
    const float la = __fsub_rn(Y[i], Y[i - 1]), lb = __fsub_rn(Y[i + 1], Y[i]);
    m1[(i >> 1) % 3] = max3_abs(m1[(i >> 1) % 3], la, lb);
    m2[(i >> 1) % 3] = max3_abs(m2[(i >> 1) % 3], __fsub_rn(la, lp), __fsub_rn(lb, la));
    lp = lb;
  }
  const float rest1 = max3_abs(m1[0], m1[1], m1[2]);
  const float rest2 = max3_abs(m2[0], m2[1], m2[2]);
  // Centring changes the tile's first residuals (lane g = 0): l1c_0 = q_0 - mu, l2c_0 =
  // q_0 - mu, l2c_1 = q_1 - 2 q_0 + mu = l2_1 + mu; the rest is unchanged (Eq. 4).
  const float c10 = __fsub_rn(Y[0], muY);
  const float c21 = __fadd_rn(l2_1, mu);
  float M1 = fmaxf(rest1, fabsf(l1_0)), M2 = max3_abs(rest2, l2_0, l2_1);
  float M1c = g == 0 ? fmaxf(rest1, fabsf(c10)) : M1;
  float M2c = g == 0 ? max3_abs(rest2, c10, c21) : M2;
  if constexpr (Cfg::kBlockLanes == 2) {  // a block's two lanes
    M1 = fmaxf(M1, __shfl_xor_sync(FULL, M1, 1));
    M2 = fmaxf(M2, __shfl_xor_sync(FULL, M2, 1));
    M1c = fmaxf(M1c, __shfl_xor_sync(FULL, M1c, 1));
    M2c = fmaxf(M2c, __shfl_xor_sync(FULL, M2c, 1));
  }
  const int R1 = bitlen(M1), R2 = bitlen(M2), R1c = bitlen(M1c), R2c = bitlen(M2c);

  // Tile costs (Eq. 3; variants 3 and 4 pay 4 bytes for mu): sums over the tile's lanes of
  // the block costs as 16-bit halves.
  uint32_t A = block_cost(R1) | (block_cost(R2) << 16);
  uint32_t B = block_cost(R1c) | (block_cost(R2c) << 16);
#pragma unroll
  for (int o = 1; o < LT; o <<= 1) {
    A += __shfl_xor_sync(FULL, A, o);
    B += __shfl_xor_sync(FULL, B, o);
  }
  // The partial sums of a tile of more than 256 elements can overflow with both signs (|d| < 2^120.5,
  // by the step's cap), which leaves no mean: the maxima above drop the NaN, and the variant would
  // seem to save block 0's first residual. It is ruled out here. (128 elements' sums are finite, so
  // a smaller tile's mean is a number or infinite, and an infinite one has the highest cost.)
  int penc = pen3;
  if constexpr (Cfg::kElems > 256) penc = fabsf(muY) < 2.0f * kMagBase ? pen3 : 0x10000;
  int C1 = int(A & 0xffffu), C2 = int(A >> 16);
  int C3 = 4 + int(B & 0xffffu) + penc;
  int C4 = 4 + int(B >> 16) + pen2 + penc;
  if constexpr (kGiven) {
    C1 = int(given[0]);
    C2 = int(given[gT]);
    C3 = int(given[2 * gT]);
    C4 = int(given[3 * gT]);
  }
  // Step 3: first strict minimum in the order LZ1, LZ2, LZ1c, LZ2c.
  int v = 0, best = C1;
  if (C2 + pen2 < best) { v = 1; best = C2; }
  if (C3 < best) { v = 2; best = C3; }
  if (C4 < best) { v = 3; best = C4; }
  const bool second = (v & 1) != 0, centred = v >= 2;

  const int Rg = centred ? (second ? R2c : R1c) : (second ? R2 : R1);
  // Rate header (Sec. 3.1): block 0 carries bit 7 = order 2, bit 6 = centred.
  if (live && (Cfg::kBlockLanes == 1 || (lane & 1) == 0)) {
    uint32_t hb = uint32_t(Rg);
    if (g == 0) hb |= (second ? 0x80u : 0u) | (centred ? 0x40u : 0u);
    hdr[lane / Cfg::kBlockLanes] = uint8_t(hb);
  }

  // Offsets: one scan over the quad's 32 lanes in stream order of the lane's bytes (its
  // block's data, preceded in block 0 of a centred tile by the 4-byte mean). The words of a
  // 64-element block alternate between its lanes, starting where the first lane's bytes do.
  const bool slot = live && centred && g == 0;
  const uint32_t mine = live ? block_cost(Rg) + (slot ? 4u : 0u) : 0u;
  uint32_t inc = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) inc = scan_step_up<32>(inc, o);
  const uint32_t excl = inc - mine;
  P.qlen = __shfl_sync(FULL, inc, 31);
  P.mu_slot = slot;
  P.mu_off = excl;
  P.mu = mu;
  P.off = excl + (slot ? 4u : 0u);
  if (Cfg::kBlockLanes == 2 && (lane & 1)) P.off = excl - mine + 4u;
  P.R = live ? Rg : 0;
  P.Rmax = int(__reduce_max_sync(FULL, live ? uint32_t(Rg) : 0u));

  // Step 5: the selected variant's residuals l1_i + m l1_{i-1} with m = 0 (LZ1) or -1 (LZ2),
  // in place over Y from the top (l_i needs Y_i, Y_{i-1}, Y_{i-2}), their magnitudes into the
  // mantissas and their sign bits shifted into one word per 8 elements. (A zero residual is
  // +0: differences of equal floats are, and +0 plus 0 times anything is.)
  const float m = second ? -1.0f : 0.0f;
  const bool first_centred = g == 0 && centred;
  uint32_t sg[4] = {0u, 0u, 0u, 0u};  // bit e of sg[k]: the sign of element 8k + e
  auto put = [&](int i, float l) {
    sg[i >> 3] = __funnelshift_l(__float_as_uint(l), sg[i >> 3], 1);
    P.v[i] = __float_as_uint(__fadd_rn(fabsf(l), kMagBase));
  };
  if (!__any_sync(FULL, second)) {  // (no tile of the quad, as in rough fields: 512^3 -0.8 %)
#pragma unroll
    for (int i = 31; i >= 1; --i) put(i, __fsub_rn(Y[i], Y[i - 1]));
    put(0, first_centred ? c10 : l1_0);
  } else {
    float up = __fsub_rn(Y[31], Y[30]);
#pragma unroll
    for (int i = 31; i >= 2; --i) {
      const float dn = __fsub_rn(Y[i - 1], Y[i - 2]);
      put(i, __fmaf_rn(dn, m, up));
      up = dn;
    }
    put(1, first_centred && second ? c21 : __fmaf_rn(l1_0, m, l1_1));
    put(0, first_centred ? c10 : __fmaf_rn(prevL, m, l1_0));
  }
  // byte k of the sign map: elements 8k .. 8k + 7, the first at the top bit
  P.signs = __byte_perm(__brev(__byte_perm(__byte_perm(sg[0], sg[1], 0x0040),
                                           __byte_perm(sg[2], sg[3], 0x0040), 0x5410)),
                        0u, 0x0123);
}

// Writes this lane's block words (sign map, then bit-planes from the least significant) at
// the shared-memory address blk, for the quad's byte-slices that any lane needs.
template <typename Cfg>
__device__ __forceinline__ void encode_block(const QuadPlan& P, uint32_t blk) {
  constexpr int W = Cfg::kWordBytes;
  uint32_t X[8];
  if (P.Rmax > 0) {
    if (P.R > 0) sts32(blk, P.signs);
    planes8<0>(P.v, X);
#pragma unroll
    for (int b = 0; b < 8; ++b)
      if (b < P.R) sts32(blk + W * (1 + b), X[b]);
  }
  if (P.Rmax > 8) {
    planes8<1>(P.v, X);
#pragma unroll
    for (int b = 0; b < 8; ++b)
      if (8 + b < P.R) sts32(blk + W * (9 + b), X[b]);
  }
  if (P.Rmax > 16) {
    planes8<2>(P.v, X);
#pragma unroll
    for (int b = 0; b < 8; ++b)
      if (16 + b < P.R) sts32(blk + W * (17 + b), X[b]);
  }
}

// Copies the runs of compute warps W0 .. W0 + N - 1 of the chunk in slot b to the stream, base
// being the chunk's place there. The runs' parameters are read side by side (one lane each), then
// the words of all of them, 4 per lane and run at a time: run after run, each waited for its own
// parameters and first words, and a launch of few chunks for that on its way out (2^20 values
// 12.7 -> 12.2 us, 31 MB field 23.3 -> 22.9 us, 512^3 equal; 2 or 8 words: the same, 0.8 % slower
// at 512^3).
template <int W0, int N>
__device__ __forceinline__ void place_runs(CompressSmem& S, int b, uint8_t* base, int lane) {
  if constexpr (N > 0) {
    constexpr int kPer = 4;
    uint32_t nw = 0, src = 0, off = 0;
    if (lane < N) {
      nw = S.qlen[b][W0 + lane] >> 2;
      src = smem_u32(S.ring[W0 + lane]) + S.qring[b][W0 + lane].x;
      off = S.qoff[b][W0 + lane];
    }
    const uint32_t most = __reduce_max_sync(FULL, nw);
    uint32_t n[N], s[N], o[N];
#pragma unroll
    for (int w = 0; w < N; ++w) {
      n[w] = __shfl_sync(FULL, nw, w);
      s[w] = __shfl_sync(FULL, src, w) + 4 * lane;
      o[w] = __shfl_sync(FULL, off, w) + 4 * lane;
    }
    for (uint32_t q0 = uint32_t(lane); q0 < most + uint32_t(lane); q0 += 32 * kPer) {
      uint32_t v[N][kPer];
#pragma unroll
      for (int w = 0; w < N; ++w) {
#pragma unroll
        for (int k = 0; k < kPer; ++k)
          if (q0 + 32 * k < n[w]) v[w][k] = lds32(s[w] + 128 * k);
        s[w] += 128 * kPer;
      }
#pragma unroll
      for (int w = 0; w < N; ++w) {
        uint32_t* dst = reinterpret_cast<uint32_t*>(base + o[w]);
#pragma unroll
        for (int k = 0; k < kPer; ++k)
          if (q0 + 32 * k < n[w]) dst[32 * k] = v[w][k];
        o[w] += 128 * kPer;
      }
    }
  }
}

// kGiven: the multipass evaluation's encoding pass (selection from a.given_costs).
// kFeat: fields' switched-off features honoured; without it the full method is compiled
// with none of that handling. Cfg: the tile configuration. (Every configuration through this
// one kernel: a 256^3 field at 64 x 8 takes 46 us, where a cost pass, a scan of the tile sizes,
// an encoding pass and a preamble kernel, with the field read twice, took 102 us.)
template <bool kGiven, bool kFeat, typename Cfg>
__global__ void __launch_bounds__(kThreads, kCtasPerSm) fsz_compress_kernel(KernelArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  CompressSmem& S = *reinterpret_cast<CompressSmem*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // mbarrier waits outlast the longest lookback wait, so a lookback that runs out is
  // reported as such rather than as a stalled pipeline.
  const uint64_t wait_ns = 4 * a.timeout_ns;

  if (tid == 0) {
    for (int k = 0; k < kSets; ++k) {
      mbar_init(&S.info[k], 1);
      mbar_init(&S.computed[k], 1);
      mbar_init(&S.encoded[k], kWarps);
      mbar_init(&S.resolved[k], 1);
      mbar_init(&S.started[k], 1);
      S.done_cnt[k] = 0;
    }
    for (int w = 0; w < kWarps; ++w) S.ring_tail[w] = 0;
    fence_mbar_init();
  }
  __syncthreads();

  // Tickets (host warp): `group` consecutive chunks each, taken `lead` chunks ahead of the
  // compute warps (one in a launch of a few chunks per CTA: what one CTA has taken no other
  // can; 31 MB field 26.7 -> 26.3 us).
  uint64_t total = 0;
  uint32_t group = 1, lead = 1, seq_t = 0, end_seq = kNone;
  bool single = true;
  float step_s = 0.0f, step_r = 0.0f;  // a.derive: the field's step (lane 0), 0 if it is refused
  auto launch_tickets = [&](uint64_t chunks) {
    total = chunks;
    group = launch_ticket_chunks(a.ticket_chunks, a.min_tickets, total, gridDim.x);
    lead = group < a.ticket_chunks ? 1u : a.ticket_lead;
  };
  // Takes the next ticket and leaves its chunks' parameters in their slots; when `early`, all
  // but the step, which is not in the field record yet.
  auto take_ticket = [&](bool early) {
    uint32_t t = 0;
    if (lane == 0) t = atomicAdd(&a.ctrl->ticket, 1u);
    t = __shfl_sync(FULL, t, 0);
    for (uint32_t g = 0; g < group && end_seq == kNone; ++g) {
      const int b = int((seq_t + g) % kSets);
      const uint32_t c = t * group + g;
      if (lane == 0) {
        ChunkInfo& ci = S.meta[b];
        if (c >= total) {
          ci.chunk = kNone;
          ci.cnt = 0;
          ci.flags = kInfoEnd;
        } else {
          // (early, the value-range pass is still writing other words of the record's lines: from
          // L2, so that no half-written line is in L1)
          const auto get = [&](const auto* p) { return early ? __ldcg(p) : *p; };
          FieldInfo* fi = single ? a.fields : a.fields + get(a.chunk_field + c);
          const uint64_t first = get(&fi->chunk_first), T = get(&fi->T), n = get(&fi->n);
          const uint64_t nchunks = get(&fi->nchunks), cap = get(&fi->cap);
          const uint64_t in = get(reinterpret_cast<const uint64_t*>(&fi->in));
          const uint64_t out = get(reinterpret_cast<const uint64_t*>(&fi->out));
          const uint32_t off = get(&fi->features_off);
          const float s = early ? 1.0f : a.derive ? step_s : fi->s, r = early || a.derive ? step_r : fi->r;
          const uint64_t lc = c - first;
          const uint64_t tile0 = lc * Cfg::kChunkTiles;
          const uint64_t e0 = lc * kCChunkElems;
          const bool ok = s > 0.0f;  // (a field without a step has nothing to load)
          ci.cnt = ok ? uint32_t(min(n - e0, uint64_t(kCChunkElems))) : 0u;
          ci.ntiles = uint32_t(min(uint64_t(Cfg::kChunkTiles), T - tile0));
          ci.r = r;
          ci.flags = (ok ? kInfoOk : 0u) | (lc + 1 == nchunks ? kInfoLast : 0u) |
                     (lc == 0 ? kInfoFirst : 0u) | (uint64_t(c) == a.skip_chunk ? kInfoSkip : 0u);
          ci.in = reinterpret_cast<const float*>(in) + e0;
          ci.out = reinterpret_cast<uint8_t*>(out);
          ci.hdr = ci.out + 64 + Cfg::kT * tile0;
          ci.fi = fi;
          ci.tile0 = tile0;
          ci.data_base = 64 + Cfg::kT * T;
          ci.cap = cap;
          ci.chunk = c;
          ci.chunk_first = uint32_t(first);
          ci.off = off;
        }
        mbar_arrive(&S.info[b]);
      }
      if (c >= total) end_seq = seq_t + g;
    }
    seq_t = end_seq != kNone ? end_seq + 1 : seq_t + group;
  };

  // The compute warps' first quad. Valid elements of this warp's quad in a chunk of cnt:
  const uint32_t e0 = uint32_t(kQuadElems * warp);
  auto quad_valid = [&](uint32_t cnt) { return cnt > e0 ? min(cnt - e0, uint32_t(kQuadElems)) : 0u; };
  const uint32_t buf = smem_u32(S.stage[warp < kWarps ? warp : 0]);
  bool ok_run = true;
  auto load_first = [&]() {
    ok_run = mbar_wait_idle(&S.info[0], 0u, wait_ns, kComputeSleepNs);
    if (!ok_run) {
      if (lane == 0) set_error(a.ctrl, nullptr, FSZ_ERR_TIMEOUT);
    } else {
      const uint32_t qv0 = quad_valid(S.meta[0].cnt);
      if (qv0) issue_quad(buf, S.meta[0].in + e0, qv0, lane, S.meta[0].in);
    }
  };

  // Right behind its value-range pass (a.early): the pass releases this kernel once the set-up or
  // planning kernel before it has completed, so the first ticket is taken and its quads are
  // loaded under the end of that pass; only the step is missing (31 MB field 26.9 -> 25.4 us; a
  // batch of 32 mixed fields of 258 MB 118.7 -> 116.9, of 8 fields of 256 KB 13.2 -> 11.7). A field
  // that turns out to be refused only loses kInfoOk: a warp may still be reading its count, and the
  // main loop waits for what has been loaded before the next chunk (of another field, perhaps) goes
  // into the same buffer.
  if (a.early) {
    if (warp == kHostWarp) {
      single = __ldcg(&a.ctrl->nfields) == 1;
      launch_tickets(__ldcg(&a.ctrl->total_chunks));
      take_ticket(true);
    } else if (warp < kWarps) {
      load_first();
    }
  }
  grid_wait();
  if (a.early && !a.derive && warp == kHostWarp && lane == 0) {
    for (uint32_t k = 0; k < seq_t; ++k) {
      ChunkInfo& ci = S.meta[k];
      if (ci.flags & kInfoEnd) continue;
      ci.r = __ldcg(&ci.fi->r);
      if (!(__ldcg(&ci.fi->s) > 0.0f)) ci.flags &= ~kInfoOk;
    }
  }
  if (a.derive && warp == kHostWarp && lane == 0) {
    // Each CTA derives the step for itself: the value-range pass need not find its last CTA and
    // wait for it, nor this one for the record (31 MB field 24.9 -> 23.7 us, 2^20 values equal). The CTA
    // with the first chunk records it.
    FieldInfo f;
    f.min_inv_key = __ldcg(&a.fields->min_inv_key);
    f.max_key = __ldcg(&a.fields->max_key);
    f.max_abs_bits = __ldcg(&a.fields->max_abs_bits);
    f.n = __ldcg(&a.fields->n);
    f.mode = __ldcg(&a.fields->mode);
    f.eb_req = __ldcg(&a.fields->eb_req);
    FieldStep p = {};
    const uint32_t st = derive_step(f, &p);
    if (st == FSZ_OK) {
      step_s = p.s;
      step_r = p.r;
    }
    for (uint32_t k = 0; k < seq_t; ++k) {
      ChunkInfo& ci = S.meta[k];
      ci.r = step_r;
      if (st != FSZ_OK) ci.flags &= ~kInfoOk;
      if (ci.flags & kInfoFirst) {
        if (st == FSZ_OK)
          store_step(a.fields, p);
        else
          set_error(a.ctrl, a.fields, st);
      }
    }
  }
  __syncthreads();

  if (warp == kHostWarp) {
    // ---------------------------------------------------------------- host
    // Tickets and placement, polled in turn:
    //  * the ticket of chunk seq is taken once the compute warps have begun chunk
    //    seq - lead (so the chunk order across the grid stays close to the ticket
    //    order) and its slot is free (chunk seq - kSets placed); lane 0 reads the field
    //    record and leaves the chunk's parameters in the slot;
    //  * chunk p is placed, in this CTA's order, once its offset is resolved and every
    //    compute warp has encoded its quad: each warp's run is copied from its ring to the
    //    stream and the ring space is given back.
    if (!a.early) {
      single = a.ctrl->nfields == 1;
      launch_tickets(a.ctrl->total_chunks);
    }
    uint32_t p = 0;
    uint64_t deadline = globaltimer_ns() + wait_ns;
    for (;;) {
      bool progress = false;
      if (end_seq == kNone && seq_t + group - p <= uint32_t(kSets) &&
          (seq_t < lead || mbar_test(&S.started[(seq_t - lead) % kSets], ((seq_t - lead) / kSets) & 1u))) {
        take_ticket(false);
        progress = true;
      }
      if (p < seq_t && p != end_seq) {
        const int b = int(p % kSets);
        const uint32_t par = (p / kSets) & 1u;
        if (mbar_test(&S.resolved[b], par) && mbar_test(&S.encoded[b], par)) {
          const ChunkInfo& ci = S.meta[b];
          if ((ci.flags & (kInfoOk | kInfoSkip)) == kInfoOk) {
            const uint64_t excl = S.set_excl[b];
            const uint32_t tot = S.set_tot[b];
            if (ci.data_base + excl + tot > ci.cap) {
              if (lane == 0) set_error(a.ctrl, ci.fi, FSZ_ERR_CAPACITY);
            } else {
              uint8_t* const base = ci.out + ci.data_base + excl;
              place_runs<kResolverRuns, kWarps - kResolverRuns>(S, b, base, lane);
              if (lane == 0 && (ci.flags & kInfoLast))
                write_preamble(ci.fi, excl + tot, a.derive ? step_s : ci.fi->s, Cfg::kT);
            }
          }
          // the runs are read: their ring space goes back to the compute warps
          __syncwarp();
          if (lane >= kResolverRuns && lane < kWarps) {
            __threadfence_block();
            st_release_cta(&S.ring_tail[lane], S.ring_tail[lane] + S.qring[b][lane].y);
          }
          __syncwarp();
          ++p;
          progress = true;
        }
      }
      if (end_seq != kNone && p == end_seq) break;
      if (progress) {
        deadline = globaltimer_ns() + wait_ns;
      } else {
        __nanosleep(kHostSleepNs);
        if (globaltimer_ns() > deadline) {
          if (lane == 0) set_error(a.ctrl, nullptr, FSZ_ERR_TIMEOUT);
          break;
        }
      }
    }
    return;
  }

  if (warp == kResolverWarp) {
    // ---------------------------------------------------------------- resolver
    // Step 4 at device level, one chunk after another in this CTA's ticket order, as soon
    // as the chunk's aggregate is out: the compute warps keep encoding meanwhile.
    uint32_t prev_c = kNone, prev_tot = 0;
    const FieldInfo* prev_fi = nullptr;
    uint64_t prev_excl = 0;
    bool prev_held = true;  // the previous chunk's flags are held back (test hook)
    for (uint32_t seq = 0;; ++seq) {
      const int b = int(seq % kSets);
      if (!mbar_wait_idle(&S.computed[b], (seq / kSets) & 1u, wait_ns, kResolverSleepNs)) {
        if (lane == 0) set_error(a.ctrl, nullptr, FSZ_ERR_TIMEOUT);
        return;
      }
      const ChunkInfo& ci = S.meta[b];
      const uint32_t c = ci.chunk;
      if (c == kNone) return;
      const uint32_t flags = ci.flags;
      uint64_t excl = 0;
      if (!(flags & kInfoFirst)) {
        bool to = false;
        if (c == prev_c + 1 && ci.fi == prev_fi && !prev_held)
          excl = prev_excl + prev_tot;  // the CTA's previous chunk is the one before
        else
          excl = lookback<kLookbackPerLane>(a.flags, int64_t(c), int64_t(ci.chunk_first),
                                            globaltimer_ns() + a.timeout_ns, &to);
        if (lane == 0) {
          if (to) set_error(a.ctrl, ci.fi, FSZ_ERR_TIMEOUT);
          if (!(flags & kInfoSkip))
            st_flag(a.flags + uint64_t(c) * kFlagStride, kFlagIncl | (excl + S.set_tot[b]));
        }
      }
      prev_c = c;
      prev_fi = ci.fi;
      prev_excl = excl;
      prev_tot = S.set_tot[b];
      prev_held = (flags & kInfoSkip) != 0;
      if constexpr (kResolverRuns > 0) {
        // copy this warp's share of the runs once they are all encoded (the host copies
        // the rest after the chunk is handed over)
        if (!mbar_wait_idle(&S.encoded[b], (seq / kSets) & 1u, wait_ns, kResolverSleepNs)) {
          if (lane == 0) set_error(a.ctrl, nullptr, FSZ_ERR_TIMEOUT);
          return;
        }
        const uint32_t tot = S.set_tot[b];
        if ((flags & (kInfoOk | kInfoSkip)) == kInfoOk && ci.data_base + excl + tot <= ci.cap) {
          uint8_t* const base = ci.out + ci.data_base + excl;
          place_runs<0, kResolverRuns>(S, b, base, lane);
        }
        __syncwarp();
        if (lane < kResolverRuns) {
          __threadfence_block();
          st_release_cta(&S.ring_tail[lane], S.ring_tail[lane] + S.qring[b][lane].y);
        }
      }
      __syncwarp();
      if (lane == 0) {
        S.set_excl[b] = excl;
        mbar_arrive(&S.resolved[b]);
      }
    }
  }

  // ------------------------------------------------------------------ compute warps
  const uint32_t ring_u32 = smem_u32(S.ring[warp]);
  uint32_t head = 0;  // bytes this warp has written to its ring (warp-uniform, wrapping)
  uint32_t pos = 0;   // ... the position in the ring where the next run goes
  if (!a.early) load_first();
  int b = 0;           // the chunk's slot and the parity of its phase there
  uint32_t par = 0;
  while (ok_run) {
    if (warp == 0 && lane == 0) mbar_arrive(&S.started[b]);  // the chunk begins
    const ChunkInfo& ci = S.meta[b];
    const uint32_t flags = ci.flags;
    const bool end = (flags & kInfoEnd) != 0;
    // Whatever has been loaded has to be in before the next chunk's pieces go into the buffer, the
    // quad of a refused field too, which is then dropped. (Waited for only where there are pieces,
    // in the same branch as the reads: 224.8 us at 512^3 against 219.7 us.)
    cp_async_wait_all();
    __syncwarp();
    const uint32_t qv = (flags & kInfoOk) ? quad_valid(ci.cnt) : 0u;
    float d[32];
    if (qv) {
      // lane L reads block g = L & 7 of tile L >> 3: piece k at column k ^ g of its row
      const uint32_t row = buf + uint32_t(lane) * 128u;
      const uint32_t base = row | (uint32_t(lane & 7) << 4);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float4 x = lds128(base ^ uint32_t(k << 4));
        d[4 * k] = x.x; d[4 * k + 1] = x.y; d[4 * k + 2] = x.z; d[4 * k + 3] = x.w;
      }
    }
    uint32_t qlen = 0;
    QuadPlan P;
    const int qt0 = Cfg::kQuadTiles * warp;            // the quad's first tile in the chunk
    const bool any = qv != 0;
    if (any) {
      const int t = qt0 + lane / Cfg::kLanes;
      const bool live = t < int(ci.ntiles);
      const uint32_t foff = kFeat ? ci.off : 0u;
      const bool restart = lane % Cfg::kLanes == 0 ||
                           ((foff & kOffCross) && lane % Cfg::kBlockLanes == 0);
      const int pen2 = (foff & kOffLz2) ? 0x10000 : 0;
      const int pen3 = (foff & kOffCenter) ? 0x10000 : 0;
      uint8_t* hdr = ci.hdr + Cfg::kT * qt0;
      // (a lane of a missing tile reads the quad's first tile's given costs)
      plan_quad<kGiven, Cfg>(d, ci.r, lane, live, restart, pen2, pen3,
                        a.given_costs + ci.tile0 + uint64_t(live ? t : qt0), a.given_T, hdr, P);
      qlen = P.qlen;
    }
    // sized: the last warp through the chunk scans the quads' sizes and publishes its
    // aggregate (step 4, warp level), before the quads are encoded; the end marker tells
    // the resolver that the CTA's chunks have run out
    if (lane == 0) S.qlen[b][warp] = qlen;
    uint32_t last = 0;
    if (lane == 0) last = atom_add_acq_rel_cta(&S.done_cnt[b], 1u) == uint32_t(kWarps - 1) ? 1u : 0u;
    last = __shfl_sync(FULL, last, 0);
    if (last) {
      if (!end) {
        __syncwarp();  // lane 0's acquire (the other warps' lengths) before every lane's reads
        const uint32_t ql = lane < kWarps ? S.qlen[b][lane] : 0u;
        uint32_t inc = ql;
#pragma unroll
        for (int o = 1; o < kWarps; o <<= 1) inc = scan_step_up<32>(inc, o);
        if (lane < kWarps) S.qoff[b][lane] = inc - ql;
        const uint32_t tot = __shfl_sync(FULL, inc, kWarps - 1);
        if (lane == 0) {
          S.set_tot[b] = tot;
          if (!(flags & kInfoSkip))
            st_flag(a.flags + uint64_t(ci.chunk) * kFlagStride,
                    ((flags & kInfoFirst) ? kFlagIncl : kFlagAgg) | tot);
        }
      }
      __syncwarp();
      if (lane == 0) {
        S.done_cnt[b] = 0;
        mbar_arrive(&S.computed[b]);
      }
    }
    if (end) break;
    // The next chunk's pieces go into the same buffer once every lane has its values.
    const int b1 = b + 1 == kSets ? 0 : b + 1;
    const uint32_t par1 = b1 == 0 ? par ^ 1u : par;
    if (!mbar_wait_idle(&S.info[b1], par1, wait_ns, kComputeSleepNs)) {
      if (lane == 0) set_error(a.ctrl, nullptr, FSZ_ERR_TIMEOUT);
      ok_run = false;
    } else {
      __syncwarp();  // every lane's loads of this buffer are done
      const ChunkInfo& cn = S.meta[b1];
      const uint32_t qv1 = quad_valid(cn.cnt);
      if (qv1) issue_quad(buf, cn.in + e0, qv1, lane, cn.in);
    }
    // room for the run in the ring (logical bytes), given back by the host as it places
    // the run's place: contiguous, from the ring's start if it would run past the end
    uint32_t skip = 0;
    if (pos + qlen > uint32_t(kRingAlloc)) {
      skip = uint32_t(kRingAlloc) - pos;
      pos = 0;
    }
    const uint32_t alloc = skip + qlen;  // (pos stays head mod kRingAlloc)
    if (any && uint32_t(kRingAlloc) - (head - ld_acquire_cta(&S.ring_tail[warp])) < alloc) {
      const uint64_t deadline = globaltimer_ns() + wait_ns;
      while (uint32_t(kRingAlloc) - (head - ld_acquire_cta(&S.ring_tail[warp])) < alloc) {
        __nanosleep(kComputeSleepNs);
        if (globaltimer_ns() > deadline) {
          if (lane == 0) set_error(a.ctrl, nullptr, FSZ_ERR_TIMEOUT);
          ok_run = false;
          break;
        }
      }
    }
    if (any && ok_run) {
      const uint32_t run = ring_u32 + pos;
      if (P.mu_slot) sts32(run + P.mu_off, __float_as_uint(P.mu));
      encode_block<Cfg>(P, run + P.off);
    }
    if (lane == 0) S.qring[b][warp] = make_uint2(pos, alloc);
    head += alloc;
    pos += qlen;
    __syncwarp();
    if (lane == 0) mbar_arrive(&S.encoded[b]);  // this warp's run of the chunk is in its ring
    b = b1;
    par = par1;
  }
  cp_async_wait_all();
}

}  // namespace

LaunchCfg compress_cfg() {
  static DeviceCfgCache cache;
  return cache.get([] {
    LaunchCfg c;
    c.smem = int(sizeof(CompressSmem));
    auto allow = [&](auto kernel) {
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, c.smem);
    };
    allow(fsz_compress_kernel<false, false, DefaultCfg>);
    allow(fsz_compress_kernel<false, true, DefaultCfg>);
    allow(fsz_compress_kernel<true, false, DefaultCfg>);
    allow(fsz_compress_kernel<false, true, TileCfg<32, 4>>);
    allow(fsz_compress_kernel<false, true, TileCfg<32, 16>>);
    allow(fsz_compress_kernel<false, true, TileCfg<64, 4>>);
    allow(fsz_compress_kernel<false, true, TileCfg<64, 8>>);
    allow(fsz_compress_kernel<false, true, TileCfg<64, 16>>);
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fsz_compress_kernel<false, false, DefaultCfg>,
                                                  kThreads, c.smem);
    c.sms = sms;
    c.per = per > 0 ? per : 1;
    c.grid = sms * c.per;
    return c;
  });
}

namespace {
template <bool kGiven, bool kFeat, typename Cfg>
void launch(const KernelArgs& args, uint64_t max_chunks, cudaStream_t st) {
  const LaunchCfg c = compress_cfg();
  KernelArgs a = args;
  a.ticket_chunks = uint32_t(g_schedule.c_ticket_chunks);
  a.ticket_lead = uint32_t(g_schedule.c_ticket_lead);
  a.min_tickets = uint32_t(g_schedule.min_tickets);
  launch_dependent(fsz_compress_kernel<kGiven, kFeat, Cfg>, sched_grid(c, kSchedCompress, max_chunks),
                   kThreads, c.smem, st, a);
}
}  // namespace

void launch_compress(const KernelArgs& a, uint64_t max_chunks, cudaStream_t st, CompressKind kind) {
  if (kind == kCompressFeatures)
    launch<false, true, DefaultCfg>(a, max_chunks, st);
  else if (kind == kCompressGiven)
    launch<true, false, DefaultCfg>(a, max_chunks, st);
  else
    launch<false, false, DefaultCfg>(a, max_chunks, st);
}

void launch_compress_tiled(const KernelArgs& a, uint64_t max_chunks, int B, int T, cudaStream_t st) {
  if (B == 32 && T == 4) launch<false, true, TileCfg<32, 4>>(a, max_chunks, st);
  else if (B == 32 && T == 8) launch<false, true, DefaultCfg>(a, max_chunks, st);
  else if (B == 32 && T == 16) launch<false, true, TileCfg<32, 16>>(a, max_chunks, st);
  else if (B == 64 && T == 4) launch<false, true, TileCfg<64, 4>>(a, max_chunks, st);
  else if (B == 64 && T == 8) launch<false, true, TileCfg<64, 8>>(a, max_chunks, st);
  else launch<false, true, TileCfg<64, 16>>(a, max_chunks, st);
}

}  // namespace fsz
