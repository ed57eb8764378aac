// Shared declarations of the CUDA library: format constants, workspace layout, launcher prototypes.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/lc.h"

namespace lc {

// ---- stream format, version 1 (docs/FORMAT.md) -------------------------------------------------
constexpr uint32_t kChunkElems = 4096;  // elements per chunk
constexpr uint32_t kLanes = 32;         // lane sub-streams per chunk (one per warp lane)
constexpr uint32_t kGroup = 4;          // consecutive elements a lane takes per step (one float4)
constexpr uint32_t kSteps = kChunkElems / (kLanes * kGroup);  // 32 steps per chunk
constexpr uint32_t kHeaderBytes = 64;
constexpr uint32_t kTableEntryBytes = 16;
constexpr uint32_t kPayloadAlign = 16;
constexpr uint32_t kKeys = 512;  // 256*sign + exponent field
constexpr int kMaxNbits = 9;     // 9 keeps every occupied bucket (at most 508 of them, plus the zero symbol)
constexpr uint32_t kMaxSymbols = 512;

__host__ __device__ constexpr inline uint64_t align_up(uint64_t x, uint64_t a) { return (x + a - 1) / a * a; }

struct StreamLayout {
  uint64_t nchunks, table_off, chunk_index_off, lane_index_off, payload_off;
};

__host__ __device__ inline StreamLayout stream_layout(uint64_t n, uint32_t nsym) {
  StreamLayout L;
  L.nchunks = (n + kChunkElems - 1) / kChunkElems;
  L.table_off = kHeaderBytes;
  L.chunk_index_off = L.table_off + (uint64_t)kTableEntryBytes * nsym;
  L.lane_index_off = L.chunk_index_off + 8 * (L.nchunks + 1);
  L.payload_off = align_up(L.lane_index_off + 64 * L.nchunks, kPayloadAlign);
  return L;
}

// ---- statistics pass -> encode pass hand-over ("key plane") -----------------------------------
// The statistics kernel leaves one byte per element in the workspace so that the encode pass reads
// 1 byte per element instead of 8: (exponent field << 1 | sign) ^ 1, the two signs of an exponent side by side, so that 16 neighbouring
// exponents fall into 32 different banks of a table indexed by this byte. It identifies the bucket of every delta below 2 (exponent
// field below 128). Byte 0 stands for all larger ones (and, which is the zero bucket, for exponent field 0 with the sign set): if the statistics say
// that there are some, the encode pass looks for it and forms the keys of such a chunk from base and cur. (With a byte modulo 256 it did so for
// all chunks: 138 M elements, one of them above 2, 1158 us for the call instead of 331, of which 60 are that chunk.)
// A *unit* is 1024 consecutive elements = 8 steps of one chunk, handled by one warp iteration:
//   unit u: bytes [1024u, 1024u+1024): byte 512*(r/4) + 16*lane + 4*(r%4) + e
// for step r (0..7) of the unit, lane (0..31) and slot e (0..3), i.e. element 1024u + 128r + 4lane + e.
constexpr uint32_t kUnitElems = 1024;
constexpr uint32_t kPlaneFlip = 0x01010101u;  // four bytes' flip
__host__ __device__ constexpr inline uint32_t key_of_byte(uint32_t b) { return ((~b & 1u) << 8) | (b >> 1); }
constexpr uint32_t kUnitsPerChunk = kChunkElems / kUnitElems;

// ---- encode pass ----------------------------------------------------------------------------------
constexpr uint32_t kEncWarps = 8;  // warps per CTA of the encode pass (one chunk per warp at a time)

// Tile descriptor of the scan of the encode pass: flag in the top two bits, bytes below.
constexpr uint64_t kTileFlagShift = 62;
constexpr uint64_t kTileInvalid = 0, kTileAggregate = 1, kTilePrefix = 2, kTileAbort = 3;
constexpr uint64_t kTileValueMask = (1ull << kTileFlagShift) - 1;
// The encode pass for one vector also adds the tiles of kScanGroupChunks chunks up in a word of their own: how many of them have a
// size yet (at most 256) above kGroupCountShift, their bytes below, and from the group's first tile, once it knows its offset, that offset
// and flag kTilePrefix. All of it by atomic additions, so that their order does not matter: a word is complete when all tiles are in it.
constexpr uint32_t kScanGroupChunks = 256;
constexpr uint64_t kGroupCountShift = 53;
constexpr uint64_t kGroupValueMask = (1ull << kGroupCountShift) - 1;

// Entry of the per-key encode table written by the table kernel.
struct EncEntry {
  uint32_t code_lo;  // low 32 bits of the canonical code
  uint32_t len;      // code length in bits (0..63)
  uint32_t code_hi;  // bits 32.. of the code (non-zero only when len > 32)
  uint32_t sym;      // symbol id
};

// Control block at the start of the workspace. Zeroed at the start of every lc_compress.
struct Control {
  int32_t status;         // first device-detected error, 0 if none
  uint32_t ticket;        // next chunk of the encode pass; in a recovery, the rank of the error (set_status_ranked)
  uint32_t nsym;          // written by the table kernel
  uint32_t max_len;       // written by the table kernel
  uint64_t payload_bits;  // written by the table kernel
  uint32_t wide;          // written by the table kernel: some delta has an exponent field >= 128, byte 0 in the key plane
  uint32_t seg_ticket;    // per-layer compress: next tile of the launch
  uint32_t seg_fail;      // per-layer compress: ~number of the first segment that failed, 0 if none
  uint32_t pad32_;
  uint64_t pad_[27];
  unsigned long long count[kKeys];  // elements per key
  uint32_t inv_min[kKeys];          // max over the bucket of ~bits (zero-initialised running minimum)
  uint32_t max_bits[kKeys];         // max over the bucket of bits
  EncEntry enc[kKeys];
  unsigned long long mant_sum[kKeys];  // mean-representative variant only: sum of the bucket's mantissa fields
};
// The bucket statistics as a shard of a split vector hands them out and takes them back (include/lc.h, lc_shard_*):
// the three arrays of Control, in Control's order, so that one copy moves them.
struct ShardStats {
  unsigned long long count[kKeys];
  uint32_t inv_min[kKeys];
  uint32_t max_bits[kKeys];
};
static_assert(sizeof(ShardStats) == LC_STATS_BYTES, "size promised by the header");
static_assert(sizeof(Control) % 256 == 0, "control block must keep the planes 256-byte aligned");

// A region behind the control block whose size does not depend on n. The per-layer compress puts the blocks and scan
// descriptors of a group of segments over it and what follows: without it a workspace for n elements would not hold those
// of one segment of n elements. The passes for one vector keep the group words of their scan at its end, in front of the tiles'
// descriptors, so that one range is cleared.
constexpr uint32_t kSpareRegionBytes = 96 * 1024;
__host__ __device__ constexpr inline uint64_t scan_group_words(uint64_t nchunks) {  // an even number
  return align_up((nchunks + kScanGroupChunks - 1) / kScanGroupChunks, 2);
}
static_assert(8 * scan_group_words(1ull << 20) <= kSpareRegionBytes, "the groups of the largest vector");

struct WorkspaceLayout {
  uint64_t control_off, spare_off, tiles_off, plane_off, total;
  uint64_t nchunks, nunits;
};

__host__ __device__ constexpr inline WorkspaceLayout workspace_layout(uint64_t n) {
  WorkspaceLayout W{};
  W.nchunks = (n + kChunkElems - 1) / kChunkElems;
  W.nunits = W.nchunks * kUnitsPerChunk;
  W.control_off = 0;
  W.spare_off = sizeof(Control);
  W.tiles_off = W.spare_off + kSpareRegionBytes;              // one 8-byte descriptor per chunk
  W.plane_off = align_up(W.tiles_off + 8 * W.nchunks, 256);
  W.total = align_up(W.plane_off + W.nchunks * kChunkElems, 256);  // 1 byte per element, whole chunks
  return W;
}

// ---- device helpers ----------------------------------------------------------------------------
__device__ inline void set_status(int32_t* status, int32_t code) { atomicCAS(status, 0, code); }

// For a launch that does in parallel what is defined as a sequence (the segments of a vector, a chain's streams): of
// several failures the one with the smallest rank stays. The rank stands in the word behind the status word, and means
// something only once the status is set.
static __device__ __noinline__ void set_status_ranked(int32_t* status, uint32_t rank, int32_t code) {
  unsigned long long* w = reinterpret_cast<unsigned long long*>(status);  // the control block is 256-byte aligned
  unsigned long long old = *reinterpret_cast<volatile unsigned long long*>(w);
  while ((uint32_t)old == 0 || (uint32_t)(old >> 32) > rank) {
    const unsigned long long seen = atomicCAS(w, old, (unsigned long long)rank << 32 | (uint32_t)code);
    if (seen == old) return;
    old = seen;
  }
}

// ---- overlapped launches -------------------------------------------------------------------------------
// The kernels of a call follow each other closely and the small ones last as long as a launch. A kernel launched with
// `overlap` may start once every CTA of the one before it in the stream has called begin_next(), and may touch what that
// kernel (and those before it) wrote only behind wait_previous(). Every kernel of such a chain calls wait_previous(), so
// that the guarantee reaches back to the first; the first of a call is launched without `overlap`, i.e. behind everything
// the caller has enqueued (but lc_wait's kernel, its call's only one, which touches nothing ahead of wait_previous()). Without the
// attribute both are no-ops. With a memset and plain launches instead, a compress of 11.7 M elements took 52 us on the GPU, with
// this 45 us. (The first launch of a recovery has a memset ahead of it, beyond kClearChunks chunks; there the launch of a clearing
// kernel costs the host more than the overlap gains.)
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void begin_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
cudaError_t launch_kernel(bool overlap, void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t cs, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = cs;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// ---- per-device launch parameters ---------------------------------------------------------------------
// Occupancy figures, SM counts and the "attributes are set" marks that the launchers cache are properties of a
// device (cudaFuncSetAttribute applies to the current device only), so every such cache is an array indexed by
// the device ordinal. Returns -1 if the ordinal cannot be had or is beyond the arrays.
constexpr int kMaxDevices = 64;
inline int current_device_index() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return -1;
  return dev;
}

// How the encode pass finds the byte offset of a tile of chunks, and the limits of its bounded wait.
struct EncodeOptions {
  bool two_pass_scan = false;     // offsets from a sizes pass and a one-CTA scan: no CTA ever waits for another
  uint32_t spin_limit = 1u << 20; // polls of the look-back before it gives up with LC_ERR_TIMEOUT
  uint32_t ticket_bias = 0;       // added to every tile ticket (test aid: with 1, tile 0 is never coded)
  bool fixed_width = false;       // fixed-width codes (format section 1.5) instead of the Huffman code
  bool mean_rep = false;          // bucket means as representatives (format section 1.8) instead of the midrange
  uint8_t* length_cache = nullptr;  // DEVICE, kLengthCacheBytes: code lengths of earlier calls (format section 1.7)
};

constexpr uint32_t kLengthCacheRow = 512;                            // bytes per row: one row per number of used symbols
constexpr uint64_t kLengthCacheBytes = 512ull * kLengthCacheRow;

// Vectors of at most this many elements take the single-launch compress path: one CTA for one chunk, a cluster of up to
// 16 CTAs (the most that the hardware schedules together) with one or two chunks each beyond that.
constexpr uint64_t kSmallMaxElems = 32 * kChunkElems;

// Zeroes two ranges (16-byte aligned, multiples of 16 bytes; the first word of `a` is kept if keep_first) with a kernel, the
// first of a chain of overlapped launches: unlike a memset it lets the next kernel begin beside it. overlap: the launch ahead is one of this library's, and
// this one goes on as soon as that has ended (lc_merge, 0.3 M elements, two streams: 57.0 -> 53.7 us blocking, 20 M, four: 149.6 -> 147.9 queued).
cudaError_t launch_clear(void* a, uint64_t a_bytes, void* b, uint64_t b_bytes, bool keep_first, cudaStream_t cs, bool overlap = false);

// ---- launchers (each defined next to its kernel) ---------------------------------------------------
// the whole compress pass of a small vector (0 < n <= kSmallMaxElems) in one launch; tracked_out may be null.
// cudaErrorNotSupported, with nothing launched: the device has no room for a cluster of that size.
cudaError_t launch_small_compress(Control* ctl, const float* base, const float* cur, uint64_t n, int nbits,
                                  uint8_t* stream, float* tracked_out, bool keep_status, cudaStream_t cs);
// mean: also accumulate the mantissa sums the mean-representative variant needs (a slower kernel variant)
cudaError_t launch_stats(const float* base, const float* cur, uint64_t n, Control* ctl, uint8_t* plane,
                         cudaStream_t cs, bool mean = false, bool overlap = false);
// wide_ok: false if the encode pass will not be able to read base and cur (the table pass then rejects a vector
// with an exponent field >= 128 with LC_ERR_RANGE)
// fixed: fixed-width codes (format section 1.5) instead of the Huffman code
// whole: nullptr, or the statistics of the whole vector of which this call codes a shard (format section 1.6):
//        kept buckets, representatives and code then come from them, the table's counts from ctl's own
cudaError_t launch_table(Control* ctl, uint64_t n, int nbits, uint8_t* stream, bool wide_ok, bool fixed,
                         const ShardStats* whole, uint8_t* length_cache, cudaStream_t cs, bool mean = false, bool overlap = false);
// tiles: one word per chunk, behind scan_group_words(chunks) others; zero
// tracked_out: nullptr, or where to write base + quantized delta (may be base itself)
cudaError_t launch_encode(Control* ctl, unsigned long long* tiles, const uint8_t* plane, const float* base,
                          const float* cur, uint64_t n, uint8_t* stream, float* tracked_out, const EncodeOptions& opt,
                          cudaStream_t cs, bool overlap = false);

struct DecodeStreams {
  const uint8_t* ptr[4];
  uint64_t bytes[4];
};
// ---- per-layer compress ---------------------------------------------------------------------------------
// A group of segments goes through three launches (statistics, tables, encode). Passed by value, within the 4 KB that
// kernel parameters may take.
constexpr uint32_t kSegGroup = 128;
// Larger segments go through the passes for one vector (four launches, which end the group before them): those write a key
// plane once, the group's encode reads base and cur a second time, and what is much larger than the L2 comes from memory
// again: 16.5 bytes per element against 10.5, or with a tracked state 20.5 against 18.5. So the line lies higher with one.
// Measured (4 bits, us in the group / by itself): without a tracked state 8 segments of 32 M 777 / 711, one of 32 M among
// 120 small ones 171 / 187, of 48 M 263 / 221, 2 of 128 M 783 / 552; with one 8 of 32 M 954 / 1011, 4 of 64 M 963 / 900, one of
// 64 M among small ones 323 / 329, 2 of 128 M 947 / 834.
constexpr uint64_t kSegLarge = 40ull << 20, kSegLargeTracked = 64ull << 20;
struct SegGroup {
  uint32_t nseg;
  uint32_t first;                        // number of the first of them among the segments of the call
  uint32_t cta_begin[kSegGroup + 1];     // statistics CTAs of each segment (filled in by the launcher)
  uint32_t tile_begin[kSegGroup + 1];    // tiles of kEncWarps chunks of each segment (0 for one of a single chunk)
  uint16_t block[kSegGroup];             // its SegBlock, if it has tiles
  uint64_t elem_begin[kSegGroup + 1];
  uint64_t stream_begin[kSegGroup + 1];  // segment i's stream starts there in the streams buffer
};
// What the passes hand each other about one segment of more than one chunk; zero at the start of the group.
struct SegBlock {
  uint32_t nsym;  // 0: no stream (the segment, or one before it, has failed)
  uint32_t max_len, wide, pad_;
  uint64_t payload_bits, pad64_[5];
  union {
    ShardStats stats;     // until the table pass has read them
    EncEntry enc[kKeys];  // after it
  };
};
static_assert(sizeof(SegBlock) == 64 + 8192, "two arrays of the same size share the block");
// `blocks`, then the scan descriptors of the tiles (one u64 each), both zeroed by the caller, lie in the workspace
cudaError_t launch_compress_segments(Control* ctl, SegBlock* blocks, unsigned long long* tiles, const float* base,
                                     const float* cur, SegGroup& group, int nbits, uint8_t* streams, float* tracked_out,
                                     cudaStream_t cs);

// The segments of one launch of the per-layer recovery, passed by value (within the 4 KB that kernel parameters may
// take): where each begins in the vector and in every streams buffer, and which CTAs work on it.
constexpr uint32_t kSegBatch = 160;
struct SegBatch {
  uint32_t nseg;
  uint32_t first;                       // number of the first of them among the segments of the call
  uint32_t cta_begin[kSegBatch + 1];    // filled in by the launcher
  uint64_t elem_begin[kSegBatch + 1];
  uint64_t stream_begin[kSegBatch + 1]; // segment i's stream has the bytes up to stream_begin[i + 1]
};
// Fills in cta_begin for CTAs of `warps` warps, `slots` of which the device holds at once; returns their number.
uint32_t split_segments(SegBatch& batch, uint32_t warps, uint32_t slots);
// Decodes every segment's k <= 4 streams onto its part of base, in one launch; second: later streams of the same chains.
// The streams of segment i start at streams[j] + stream_begin[i].
cudaError_t launch_decode_segments(const float* base, const uint8_t* const* streams, int k, SegBatch& batch, int nbits,
                                   float* out, int32_t* status, bool second, cudaStream_t cs);

// Warps on an SM in a launch with k streams whose chunks have chunk_bytes on average, by a kernel of so many registers a thread.
uint32_t decode_warps(int k, uint64_t chunk_bytes, uint32_t regs);
// How many streams the next launch takes, of `left` that remain of a chain.
int decode_group(int left);
int decode_group_segments(int left, int nbits);  // the same for layers coded with nbits
// Decodes the chunks [chunk_begin, chunk_end) only (clipped to the vector's chunks). second: as above.
// clear: the launch clears the status word itself, for a vector of at most kClearChunks chunks; cudaErrorNotSupported, with nothing launched, if the device
// has no room for its cluster. A memset ahead of it costs more: one stream of 61,706 elements 14.5 us queued instead of 13.0 and 25.2 blocking instead of
// 24.4, of 1000 28.2 blocking instead of 26.9, four streams 18.1 queued instead of 16.1 and as long blocking.
constexpr uint32_t kClearChunks = 32;
cudaError_t launch_decode(const float* base, const DecodeStreams& streams, int k, uint64_t n, float* out,
                          int32_t* status, bool second, cudaStream_t cs, uint64_t chunk_begin = 0, uint64_t chunk_end = ~0ull, bool clear = false);

}  // namespace lc
