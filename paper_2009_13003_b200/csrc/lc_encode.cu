// Encode pass: key plane -> Huffman bitstream with chunk and lane indices.
//
// Paper: Algorithm 1 step 6 and Section 3.1.2 (the quantized delta, i.e. the sequence of bucket
// indices, is Huffman-coded). Element order, bit order and the two indices are those of the stream
// format text, sections 2 and 3.
//
// A CTA takes a tile of 8 consecutive chunks, one per warp; lane t owns lane sub-stream t. Per chunk:
//   A. every lane codes its 128 elements into its own column of a warp-private word matrix in shared
//      memory (word k of lane t at k*32 + t: plain stores, no bank conflicts, no atomics). Two elements are looked up at
//      once in a table of pairs whose index is formed for all four elements of a step together (lc_encode_bits.cuh),
//      and the step's codes are appended as one, so a step of four elements costs two lookups and one append. The table's entries
//      are spread so that lookups meet little in banks (268 M elements 173 -> 166 us);
//   B. a warp shuffle scan of the lane bit counts gives every lane its bit offset in the chunk (the
//      lane index of the stream) and the chunk its size, which is published at once;
//   C. the lanes' words are shifted to their bit offsets and written to the chunk image (shared memory);
//   D. the tile's byte offset comes from an exclusive scan over all tiles, done across CTAs with a
//      decoupled look-back over per-tile descriptors and words that sum up groups of 32 tiles (per-chunk descriptors were tried: with
//      thousands of chunks in flight every look-back walks too far back, and so it does over 592 tiles in flight);
//   E. the chunk image is copied to the payload with coalesced 16-byte stores.
// The loop is software-pipelined: D and E of a tile run after A and B of the CTA's next tile (whose C follows
// once E has freed the image area), and D is done by whichever warp finishes coding first (see the loop). Tiles are handed out by an atomic ticket, so
// every tile a CTA waits for in D has already been started by a running CTA, and coding never waits for
// anything. The wait is bounded all the same: after `spin_limit` polls the CTA records LC_ERR_TIMEOUT, marks
// its tile aborted (successors see that at once and abort too) and moves on.
// A caller that wants no device-side wait at all selects the two-pass scan (EncodeOptions::two_pass_scan):
// encode_sizes_kernel computes every chunk's size, encode_scan_kernel (one CTA) turns the sizes into the chunk
// index, and this kernel takes its offsets from there instead of looking back. Same bytes, one more pass over
// the key plane.
//
// The vector's partial last chunk takes a masked form of A. Rare cases take a compact two-pass path (lengths, then bits
// ORed in place; chunk_slow): codes longer than 32 bits, a lane or chunk that outgrows its shared-memory area, and chunks with an
// exponent field >= 128, for which the one-byte key plane is not enough and keys come from base and cur.
//
// Bound: reads 1 byte and writes about 0.5 bytes per element, so this pass is limited by the integer work per element,
// not by HBM: logic, shifts, permutes and compares issue at 64 lanes per clock and SM, half the rate of multiply-adds. 268 M elements in 5 bits take
// 147 us (Gaussian deltas 143), 62 for the bytes alone; with lookups and appends left out 100. Tried and not kept: warps that wait for each other through
// barriers in shared memory instead of the block's (147), one vote for two rows (148; Gaussian 163), an append of nine instructions instead of ten that
// counts all bits (148), and one of seven that splits a code with a 64-bit multiply-add (174 instead of 169).
#include "lc_encode_bits.cuh"

namespace lc {
namespace {

using namespace enc;

constexpr int kEncThreads = kEncWarps * 32;
// 48 KB of shared memory per CTA for coding (four CTAs per SM, beside 8 KB of tables), split evenly between the warps that work:
// all 8 while an average chunk fits half of a 6 KB share (column matrix + chunk image), else 4, 2 or 1. Up to 5.1 bits per
// element that is all 8; with 44 KB it was up to 4.7, and 134 M elements in codes of a fixed 5 bits took 362 us instead of 322
// (with the tracked state 498 instead of 433).
constexpr uint32_t kEncSmem = 48 * 1024;
constexpr uint32_t kEncDyn = kTablesBytes + kEncSmem;
// bytes of a share's half that an average chunk of `avg` bytes needs: 15 % more, for the lanes and chunks above the average
__host__ __device__ constexpr uint64_t share_need(uint64_t avg) { return avg + avg / 7 + 64; }
static_assert(share_need(kChunkElems * 5 / 8) <= kEncSmem / kEncWarps / 2, "codes of 5 bits throughout are coded by all warps");
constexpr int kUpdRows = 4;  // rows of base in flight per warp in the kernel that also writes the tracked state
constexpr uint32_t kUpdSmem = kEncWarps * kUpdRows * 512;  // its ring, behind the kEncSmem bytes of coding areas
constexpr int kGroupWindows = 2;  // sub-windows of 32 group words that a round of the look-back reads

// UPDATE: the kernel also writes the tracked state of Algorithm 1 step 7, tracked_out = base + quantized delta
// (fp32, the representative of the zero bucket, +0, added like any other): inside the coding loop for the chunks
// whose coding never reads base, otherwise chunk by chunk once a chunk's coding no longer needs base.
// tracked_out may be base itself, hence no __restrict__ on the two. Three CTAs per SM instead of four, for the
// registers the rows of base in flight take.
template <bool UPDATE>
__global__ void __launch_bounds__(kEncThreads, UPDATE ? 3 : 4)
encode_kernel(Control* __restrict__ ctl, unsigned long long* __restrict__ tiles, const uint8_t* __restrict__ plane,
              const float* base, const float* __restrict__ cur, uint64_t n, uint8_t* __restrict__ stream,
              float* tracked_out, uint32_t spin_limit, uint32_t ticket_bias, uint32_t two_pass_scan) {
  extern __shared__ __align__(128) uint32_t s_all[];
  Tables& tb = shared_tables();
  uint32_t* s_dyn = s_all + kTablesBytes / 4;  // rows that straddle lines cost the asynchronous copies of UPDATE 5 %
  // What warps hand each other in iteration i of the loop. A warp may reach the next iteration's barrier while another is still behind this one's, so
  // the words alternate: those read behind the iteration's barrier by i % 2, those that the next iteration reads too by i % 3.
  __shared__ uint32_t s_chunk_bytes[3][kEncWarps];
  __shared__ uint32_t s_arrived[3];  // warps that have coded their chunk
  __shared__ uint32_t s_tile[2];     // the tile to be coded next
  __shared__ unsigned long long s_tile_base[2], s_tile_end[2];  // of the pending tile
  __shared__ int s_abort[2];
  __shared__ uint32_t s_any_wide;               // the vector has elements that the plane does not identify
  __shared__ uint32_t s_rep[UPDATE ? 256 : 1];  // UPDATE: representative (bit pattern) by plane byte

  wait_previous();
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // The table pass may have rejected the vector, or another CTA may already have given up waiting: leave, all
  // threads together (one thread reads the word; a thread-by-thread test could split the CTA if the word changed
  // in between, and the warps that stayed would wait at barriers for the ones that left).
  // What the preparation reads is asked for at once, and a representative, which is where its entry says, used behind the tables (3 M elements 32.7 -> 31.3 us,
  // 11.7 M 46.9 -> 46.3).
  static_assert(kEncThreads == 256, "a thread per plane byte");
  const EncEntry e = ctl->enc[key_of_byte(tid)];
  const uint32_t sym0_len = ctl->enc[0].len, nsym = ctl->nsym;
  const bool long_codes = ctl->max_len > 32;
  const unsigned long long payload_bits = ctl->payload_bits;
  if (tid == 0) {
    s_abort[0] = ctl->status;
    s_any_wide = ctl->wide;
    s_tile[0] = atomicAdd(&ctl->ticket, 1u) + ticket_bias;
    s_arrived[0] = s_arrived[1] = s_arrived[2] = 0;
  }
  if (tid == 0) tb.long_codes = long_codes;
  tb.full[tid] = make_uint2(e.code_lo, e.len);
  __syncthreads();
  if (s_abort[0] != 0) return;
  // the table pass has written the stream's symbol table: entry of symbol s at 64 + 16 s, representative at +4
  uint32_t rep = 0;
  if (UPDATE) rep = *reinterpret_cast<const uint32_t*>(stream + kHeaderBytes + kTableEntryBytes * e.sym + 4);
  build_tables(tb, sym0_len, [&](uint32_t) { return e.sym != 0; });
  if (UPDATE) {
    s_rep[tid] = rep;
    __syncthreads();
  }

  const StreamLayout L = stream_layout(n, nsym);
  const uint32_t nchunks = (uint32_t)L.nchunks, whole = (uint32_t)(n / kChunkElems);  // at most 2^20 chunks
  unsigned long long* chunk_index = reinterpret_cast<unsigned long long*>(stream + L.chunk_index_off);
  uint16_t* lane_index = reinterpret_cast<uint16_t*>(stream + L.lane_index_off);
  uint8_t* payload = stream + L.payload_off;
  // how many warps work: as many as can each hold an average chunk (plus 15 %) twice
  const uint64_t need = share_need(nchunks ? payload_bits / 8 / nchunks : 0);
  uint32_t active = kEncWarps;
  while (active > 1 && need > kEncSmem / active / 2) active >>= 1;
  const uint32_t image_words = kEncSmem / active / 8;  // half of the warp's share, in words
  const uint32_t lane_words = image_words / 32;        // rows of the column matrix
  uint32_t* column = s_dyn + (warp % active) * (2 * image_words);  // word k of lane t at column[k*32 + t]
  uint32_t* image = column + image_words;
  const uint32_t neg_base = (uint32_t)(-tb.base) & 0xffffu, neg_base2 = neg_base << 16 | neg_base;
  const bool use_pair = tb.use_pair != 0;

  // wide_chunk: keys from base and cur. The tracked state of a chunk that is neither that nor long_codes is written while it is coded.
  auto wide_chunk = [&](uint32_t cc) { return s_any_wide != 0 && has_escape(plane, cc, lane); };
  auto keys = [&](bool wide) { return KeySource{plane, base, cur, wide}; };

  const uint32_t ntiles = (nchunks + active - 1) / active;
  const uint32_t group_tiles = kScanGroupChunks / active;
  unsigned long long* groups = tiles - scan_group_words(nchunks);

  // The loop is software-pipelined over tiles: a tile's offset is looked up, and its image copied out, only
  // after the *next* tile has been coded. Every earlier tile needs its size before this one can be placed, and
  // with hundreds of tiles in flight some predecessor is always late; looking back right after coding made the
  // whole CTA wait for that straggler for a third of its time. One coding phase later the predecessors' sizes
  // are there. The pending tile lives in the warps' image areas, which coding (phase A) does not touch.
  // What the pending tile needs later is kept in shared memory (its chunk sizes; the lanes' start bits, in the image area
  // of a chunk that has no image because it is too large) or
  // recomputed from its number: phase A has no registers to spare.
  // There is one barrier an iteration, behind coding: the first warp that gets there takes the next ticket and looks up the pending tile's
  // offset while the others are still coding, the last one publishes the tile's size.
  bool p_have = false;
  uint32_t p_tile = 0, parity = 0, buf = 0, p_buf = 2;
  uint32_t tile = s_tile[0];
  while (true) {
    const bool have = tile < ntiles;
    if (!have && !p_have) break;
    const uint32_t c = tile * active + warp;
    const bool valid = have && warp < active && c < nchunks;
    const bool wide = valid && wide_chunk(c);
    bool fast = valid && c < whole && !long_codes && !wide;

    // ---- A: code the lane's elements into its column. Lookups run one row (4 elements) ahead of the
    // appends, which depend on each other through the bit accumulator.
    uint32_t lane_bits = 0;
    if (fast) {
      const uint4* ep = reinterpret_cast<const uint4*>(plane + (uint64_t)c * kChunkElems) + lane;
      const uint32_t col0 = smem_addr(column) + lane * 4;
      ColumnPacker pk{0u, 0u, col0, col0 + lane_words * 128};
      // UPDATE: the tracked state of this chunk is written here, where its plane bytes are in registers; the
      // memory traffic of the update then runs under the coding, which is bound by instruction issue. A chunk on
      // this path never reads base for its coding (not even when it is coded again the slow way), so base may be
      // overwritten at once. Row j of base is requested while row j - 1 is coded.
      const float4* b4 = reinterpret_cast<const float4*>(base + (uint64_t)c * kChunkElems) + lane;
      float4* o4 = reinterpret_cast<float4*>(tracked_out + (uint64_t)c * kChunkElems) + lane;
      // Rows of base come through a ring of kUpdRows 512-byte slots per warp behind the coding areas, filled by
      // cp.async four rows ahead: that many loads in flight per lane would not fit the registers, and the kernel's
      // L1 is too small to help. A lane reads back only the 16 bytes it copied itself, so no barrier is needed.
      const uint32_t ring = smem_addr(s_dyn) + kEncSmem + warp * (kUpdRows * 512) + lane * 16;
      auto issue_row = [&](int j) {
        if (j < (int)kSteps)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(ring + (j % kUpdRows) * 512), "l"(b4 + 32 * j)
                       : "memory");
        asm volatile("cp.async.commit_group;" ::: "memory");  // also when empty: the wait below counts groups
      };
      if (UPDATE) {
#pragma unroll
        for (int j = 0; j < kUpdRows; ++j) issue_row(j);
      }
      auto update_row = [&](uint32_t word, int j) {
        asm volatile("cp.async.wait_group %0;" ::"n"(kUpdRows - 1) : "memory");  // row j has landed
        float4 b;
        asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];"
                     : "=f"(b.x), "=f"(b.y), "=f"(b.z), "=f"(b.w)
                     : "r"(ring + (j % kUpdRows) * 512));
        float4 x;
        x.x = __fadd_rn(b.x, __uint_as_float(s_rep[__byte_perm(word, 0u, 0x4440)]));
        x.y = __fadd_rn(b.y, __uint_as_float(s_rep[__byte_perm(word, 0u, 0x4441)]));
        x.z = __fadd_rn(b.z, __uint_as_float(s_rep[__byte_perm(word, 0u, 0x4442)]));
        x.w = __fadd_rn(b.w, __uint_as_float(s_rep[__byte_perm(word, 0u, 0x4443)]));
        o4[32 * j] = x;
        issue_row(j + kUpdRows);
      };
      auto load = [&](int q) { return __ldg(ep + 32 * q); };
      auto row = [&](uint32_t word, int j) {
        if (UPDATE) update_row(word, j);
      };
      if (use_pair) code_rows<true>(pk, tb, neg_base2, load, row);
      else code_rows<false>(pk, tb, neg_base2, load, row);
      lane_bits = finish_column(pk, col0);
    } else if (valid && !long_codes && !wide) {
      lane_bits = code_partial(&tb, reinterpret_cast<const uint4*>(plane + (uint64_t)c * kChunkElems) + lane, (uint32_t)(n - (uint64_t)c * kChunkElems),
                               lane, smem_addr(column) + lane * 4, lane_words);
      fast = true;
    }
    if (fast && __any_sync(0xffffffffu, lane_bits == 0xffffffffu)) fast = false;  // some lane outgrew its column: redo the chunk the slow way
    if (!fast && valid) lane_bits = chunk_slow<true>(ctl->enc, keys(wide), c, lane, n, nullptr, 0);

    // ---- B: lane offsets, lane index, chunk size; the tile's size is published as early as possible
    if (valid) lane_index[c * kLanes + lane] = (uint16_t)lane_bits;
    uint32_t incl = lane_bits;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, d);
      if ((int)lane >= d) incl += v;
    }
    const uint32_t lane_start = incl - lane_bits;
    const uint32_t chunk_bits = __shfl_sync(0xffffffffu, incl, 31);
    const uint32_t chunk_bytes = valid ? (uint32_t)align_up((chunk_bits + 7) / 8, kPayloadAlign) : 0u;
    const bool staged = chunk_bytes <= image_words * 4;
    uint32_t arrival = 0;
    if (lane == 0) {
      s_chunk_bytes[buf][warp] = chunk_bytes;
      __threadfence_block();
      arrival = atomicAdd(&s_arrived[buf], 1u);
    }
    arrival = __shfl_sync(0xffffffffu, arrival, 0);
    if (arrival == kEncWarps - 1 && have && !two_pass_scan) {
      __threadfence_block();  // lane 0 has seen the other warps arrive; behind this and the warp's barrier all lanes see their sizes
      __syncwarp();
      uint32_t bytes = 0;
      if (lane < kEncWarps) bytes = *reinterpret_cast<volatile uint32_t*>(&s_chunk_bytes[buf][lane]);
      bytes = __reduce_add_sync(0xffffffffu, bytes);
      if (lane == 0) {
        st_tile(&tiles[tile], (kTileAggregate << kTileFlagShift) | bytes);
        atomicAdd(&groups[tile / group_tiles], (1ull << kGroupCountShift) | bytes);
      }
    }

    // ---- D: the next ticket, and the offset of the pending tile: the sum over the tiles before it. Those of its own group (32 with
    // eight warps) it reads one by one, behind them the group words up to the nearest that knows its offset. (Tiles one by one all the way, 592
    // and more back, took three dependent rounds of 256 words, and the other seven warps waited for them: 268 M elements 164 us, so 158.)
    if (arrival == 0) {
      uint32_t next = 0;
      if (have && lane == 0) next = atomicAdd(&ctl->ticket, 1u) + ticket_bias;
      if (p_have) {
        unsigned long long part = 0;  // this lane's share of the groups before
        uint32_t own_bytes = 0;       // the tiles before it in its group, 256 chunks at most
        bool abort = false;
        const uint32_t group = p_tile / group_tiles, before = p_tile % group_tiles;
        if (two_pass_scan) {
          // the chunk index is already there (encode_scan_kernel): the tile starts where its first chunk starts
          if (lane == 0) part = chunk_index[p_tile * active];
        } else {
          int look = (int)group - 1;
          bool own = before == 0, done = group == 0;
          uint32_t spins = 0;
          while (!abort && !(own && done)) {
            unsigned long long st[kGroupWindows];
#pragma unroll
            for (int u = 0; u < kGroupWindows; ++u) {
              const int idx = look - 32 * u - (int)lane;
              st[u] = kTilePrefix << kTileFlagShift | (unsigned long long)group_tiles << kGroupCountShift;  // before the first: prefix 0
              if (!done && idx >= 0) st[u] = ld_tile(&groups[idx]);
            }
            bool retry = false;
            if (!own) {
              uint32_t sum = 0;
              uint32_t missing = 0;  // 1: a tile without a size, 2: an aborted one
              for (uint32_t i = lane; i < before; i += 32) {
                const unsigned long long t = ld_tile(&tiles[group * group_tiles + i]);
                const uint32_t flag = (uint32_t)(t >> kTileFlagShift);
                sum += (uint32_t)t;
                missing |= flag == kTileAggregate ? 0u : flag == kTileAbort ? 2u : 1u;
              }
              missing = __reduce_or_sync(0xffffffffu, missing);
              if (missing & 2u) abort = true;
              else if (missing) retry = true;
              else own_bytes = __reduce_add_sync(0xffffffffu, sum), own = true;
            }
#pragma unroll
            for (int u = 0; u < kGroupWindows; ++u) {
              if (done || abort || retry) continue;
              const uint32_t flag = (uint32_t)(st[u] >> kTileFlagShift);
              const bool complete = ((uint32_t)(st[u] >> kGroupCountShift) & 511u) == group_tiles && (flag & 1u) == 0;
              const uint32_t m_prefix = __ballot_sync(0xffffffffu, complete && flag == kTilePrefix);
              const uint32_t m_other = __ballot_sync(0xffffffffu, !complete);
              const int first_prefix = m_prefix ? __ffs(m_prefix) - 1 : 32;
              const uint32_t relevant = first_prefix < 32 ? (0xffffffffu >> (31 - first_prefix)) : 0xffffffffu;
              if (m_other & relevant) {
                // a group with a tile that has no size yet, or an aborted one
                if (__ballot_sync(0xffffffffu, (flag & 1u) != 0) & relevant) abort = true;
                else retry = true;  // poll again from `look`, which already skips the complete sub-windows
              } else {
                if ((int)lane <= first_prefix) part += st[u] & kGroupValueMask;
                if (first_prefix < 32) done = true;
                else look -= 32;
              }
            }
            if (retry) {
              if (++spins > spin_limit) abort = true;
              else __nanosleep(40);
            }
          }
        }
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) part += __shfl_xor_sync(0xffffffffu, part, d);
        if (lane == 0) {
          if (abort) {
            set_status(&ctl->status, LC_ERR_TIMEOUT);
            st_tile(&tiles[p_tile], kTileAbort << kTileFlagShift);
            st_tile(&groups[group], kTileAbort << kTileFlagShift);  // what is still added to it leaves the lower flag bit
            s_abort[parity] = 1;
          } else {
            unsigned long long p_tile_bytes = 0;
#pragma unroll
            for (int w = 0; w < (int)kEncWarps; ++w) p_tile_bytes += s_chunk_bytes[p_buf][w];
            // added, not stored: sizes of the group's tiles may still be on their way
            if (before == 0 && !two_pass_scan) atomicAdd(&groups[group], (kTilePrefix << kTileFlagShift) | part);
            s_abort[parity] = 0;
            s_tile_base[parity] = part + own_bytes;
            s_tile_end[parity] = part + own_bytes + p_tile_bytes;
          }
        }
      }
      if (have && lane == 0) s_tile[parity ^ 1] = next;
    }
    __syncthreads();  // the pending tile's offset and the next ticket are known
    if (tid == 0) s_arrived[p_buf] = 0;  // used again behind the next barrier
    const uint32_t next_tile = have ? s_tile[parity ^ 1] : ntiles;
    // The next chunk's plane bytes are asked into the L2, a line per lane (268 M elements 158 -> 147 us; with the tracked state, where rows of base
    // are what counts, 782 either way).
    {
      const uint32_t next_c = next_tile * active + warp;
      if (!UPDATE && warp < active && next_c < nchunks)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(plane + (uint64_t)next_c * kChunkElems + lane * 128));
    }
    const bool p_write = p_have && !s_abort[parity];

    // ---- E: write the pending tile's chunks and their index entries
    if (p_write) {
      unsigned long long chunk_off = s_tile_base[parity];
      for (uint32_t w = 0; w < warp; ++w) chunk_off += s_chunk_bytes[p_buf][w];
      const uint32_t p_c = p_tile * active + warp;
      const uint32_t p_chunk_bytes = s_chunk_bytes[p_buf][warp];
      const bool p_staged = p_chunk_bytes <= image_words * 4;
      if (warp < active && p_c < nchunks) {
        if (lane == 0) chunk_index[p_c] = chunk_off;
        uint4* dst4 = reinterpret_cast<uint4*>(payload + chunk_off);
        if (p_staged) {
          const uint4* im4 = reinterpret_cast<const uint4*>(image);
          for (uint32_t k = lane; k < p_chunk_bytes / 16; k += 32) dst4[k] = im4[k];
        } else {
          // chunk larger than the image area: OR the bits straight into (zeroed) global memory.
          for (uint32_t k = lane; k < p_chunk_bytes / 16; k += 32) dst4[k] = make_uint4(0, 0, 0, 0);
          __threadfence_block();
          __syncwarp();
          chunk_slow<true>(ctl->enc, keys(wide_chunk(p_c)), p_c, lane, n, reinterpret_cast<uint32_t*>(dst4), image[lane]);
        }
      }
      if (p_tile == ntiles - 1 && tid == 0) {
        const unsigned long long payload_bytes = s_tile_end[parity];
        chunk_index[nchunks] = payload_bytes;
        *reinterpret_cast<unsigned long long*>(stream + 48) = L.payload_off + payload_bytes;
      }
    }
    // ---- tracked state of the pending tile's chunks (everything that reads base for coding them is done)
    if (UPDATE && p_write) {
      const uint32_t p_c = p_tile * active + warp;
      const bool p_wide = warp < active && p_c < nchunks && wide_chunk(p_c);
      if (warp < active && p_c < nchunks && (p_c >= whole || long_codes || p_wide)) {  // the others were updated while they were coded
        if (p_c < whole && !p_wide) {
          const uint4* ep = reinterpret_cast<const uint4*>(plane + (uint64_t)p_c * kChunkElems) + lane;
          const float4* b4 = reinterpret_cast<const float4*>(base + (uint64_t)p_c * kChunkElems) + lane;
          float4* o4 = reinterpret_cast<float4*>(tracked_out + (uint64_t)p_c * kChunkElems) + lane;
#pragma unroll 2
          for (int q = 0; q < 8; ++q) {
            const uint4 w4 = __ldg(ep + 32 * q);  // plane bytes of steps 4q .. 4q+3
            const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
            float4 b[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) b[r] = b4[32 * (4 * q + r)];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              float4 x;
              x.x = __fadd_rn(b[r].x, __uint_as_float(s_rep[__byte_perm(w[r], 0u, 0x4440)]));
              x.y = __fadd_rn(b[r].y, __uint_as_float(s_rep[__byte_perm(w[r], 0u, 0x4441)]));
              x.z = __fadd_rn(b[r].z, __uint_as_float(s_rep[__byte_perm(w[r], 0u, 0x4442)]));
              x.w = __fadd_rn(b[r].w, __uint_as_float(s_rep[__byte_perm(w[r], 0u, 0x4443)]));
              o4[32 * (4 * q + r)] = x;
            }
          }
        } else if (p_wide) {
          // exponents the one-byte plane does not hold: element by element
          for (uint32_t j = 0; j < kSteps; ++j) {
            for (uint32_t e = 0; e < kGroup; ++e) {
              const KeySource ks = keys(true);
              const uint64_t i = (uint64_t)p_c * kChunkElems + 128ull * j + 4 * lane + e;
              if (i >= n) continue;
              const uint32_t sym = ctl->enc[ks.key(p_c, j, lane, e)].sym;
              const uint32_t rep = *reinterpret_cast<const uint32_t*>(stream + kHeaderBytes + kTableEntryBytes * sym + 4);
              tracked_out[i] = __fadd_rn(base[i], __uint_as_float(rep));
            }
          }
        }
      }
    }
    // The partial last chunk's, by all warps of the CTA, four rows each: by the one warp that has coded it, it took the launch
    // 10 us longer (11.7 M elements: 35 us instead of 25).
    if (UPDATE && p_write && p_tile == ntiles - 1 && n % kChunkElems != 0 && !wide_chunk(nchunks - 1)) {
      const uint64_t p_c = nchunks - 1;
      const uint32_t rem = (uint32_t)(n - p_c * kChunkElems);
      const float* b1 = base + p_c * kChunkElems;
      float* o1 = tracked_out + p_c * kChunkElems;
      constexpr uint32_t kRows = kSteps / kEncWarps;
      static_assert(kRows == 4, "a lane's plane bytes of four steps are one load");
      const uint4 w4 = __ldg(reinterpret_cast<const uint4*>(plane + p_c * kChunkElems) + 32 * warp + lane);
      const uint32_t w[kRows] = {w4.x, w4.y, w4.z, w4.w};
      float b[kRows][4];
#pragma unroll
      for (uint32_t r = 0; r < kRows; ++r)
#pragma unroll
        for (uint32_t e = 0; e < 4; ++e) {
          const uint32_t i = (kRows * warp + r) * 128 + 4 * lane + e;
          if (i < rem) b[r][e] = b1[i];
        }
#pragma unroll
      for (uint32_t r = 0; r < kRows; ++r)
#pragma unroll
        for (uint32_t e = 0; e < 4; ++e) {
          const uint32_t i = (kRows * warp + r) * 128 + 4 * lane + e;
          if (i < rem) o1[i] = __fadd_rn(b[r][e], __uint_as_float(s_rep[__byte_perm(w[r], 0u, 0x4440 + e)]));
        }
    }
    if (!have) break;
    __syncwarp();  // the warp's image area is free again

    // ---- C: assemble the new tile's chunk image in shared memory
    if (valid && staged) {
      if (fast) {
        assemble_chunk(column, lane, lane_bits, lane_start, image, chunk_bytes);
      } else {
        uint4* im4 = reinterpret_cast<uint4*>(image);
        for (uint32_t k = lane; k < chunk_bytes / 16; k += 32) im4[k] = make_uint4(0, 0, 0, 0);
        __syncwarp();
        chunk_slow<true>(ctl->enc, keys(wide), c, lane, n, image, lane_start);
      }
    } else if (valid) {
      image[lane] = lane_start;
    }
    __syncwarp();
    p_have = true;
    p_tile = tile;
    p_buf = buf;
    buf = buf == 2 ? 0 : buf + 1;
    parity ^= 1;
    tile = next_tile;
  }
}

// ---- two-pass scan: chunk sizes, then their exclusive prefix sum, with no CTA waiting for another ----------

constexpr int kScanThreads = 1024;

// Size in bytes of every chunk (format section 3.3: the chunk's bits rounded up to 16 bytes), one warp per chunk,
// into sizes[c]. Whole chunks whose keys the one-byte plane identifies take their code lengths from a 256-byte
// table in shared memory, 16 plane bytes per load; the vector's partial last chunk and chunks that hold byte 0 while the
// vector has exponent fields >= 128 go through the slow path's counting mode.
__global__ void __launch_bounds__(kEncThreads)
encode_sizes_kernel(const Control* __restrict__ ctl, unsigned long long* __restrict__ sizes,
                    const uint8_t* __restrict__ plane, const float* base, const float* __restrict__ cur, uint64_t n,
                    uint64_t nchunks) {
  __shared__ uint8_t s_len[256];  // code length by plane byte (lengths are at most 63)
  if (ctl->status != 0) return;  // nothing in this kernel writes the word: the same for every thread
  for (uint32_t b = threadIdx.x; b < 256; b += kEncThreads) s_len[b] = (uint8_t)ctl->enc[key_of_byte(b)].len;
  __syncthreads();
  const uint32_t lane = threadIdx.x & 31;
  const bool any_wide = ctl->wide != 0;
  const uint64_t warp0 = (uint64_t)blockIdx.x * kEncWarps + (threadIdx.x >> 5), nwarps = (uint64_t)gridDim.x * kEncWarps;
  for (uint64_t c = warp0; c < nchunks; c += nwarps) {
    uint32_t bits = 0;
    const bool wide = any_wide && has_escape(plane, (uint32_t)c, lane);
    if (!wide && (c + 1) * kChunkElems <= n) {
      const uint4* ep = reinterpret_cast<const uint4*>(plane + (uint64_t)c * kChunkElems) + lane;
      uint4 v[kSteps / 4];
#pragma unroll
      for (uint32_t q = 0; q < kSteps / 4; ++q) v[q] = __ldg(ep + 32 * q);
#pragma unroll
      for (uint32_t q = 0; q < kSteps / 4; ++q) {
        const uint32_t w[4] = {v[q].x, v[q].y, v[q].z, v[q].w};
#pragma unroll
        for (int r = 0; r < 4; ++r)
          bits += s_len[w[r] & 255u] + s_len[(w[r] >> 8) & 255u] + s_len[(w[r] >> 16) & 255u] + s_len[w[r] >> 24];
      }
    } else {
      bits = chunk_slow<false>(ctl->enc, KeySource{plane, base, cur, wide}, c, lane, n, nullptr, 0);
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) bits += __shfl_xor_sync(0xffffffffu, bits, d);
    if (lane == 0) sizes[c] = align_up((bits + 7) / 8, kPayloadAlign);
  }
}

// chunk_off[c] = sum of sizes[0..c) for c = 0..nchunks, and the stream's total size into its header. One CTA:
// each thread sums a contiguous run of chunks, the run totals are scanned in shared memory.
__global__ void __launch_bounds__(kScanThreads)
encode_scan_kernel(const Control* __restrict__ ctl, const unsigned long long* __restrict__ sizes, uint64_t n,
                   uint64_t nchunks, uint8_t* __restrict__ stream) {
  __shared__ unsigned long long run_total[kScanThreads];
  if (ctl->status != 0) return;
  const StreamLayout L = stream_layout(n, ctl->nsym);
  unsigned long long* chunk_index = reinterpret_cast<unsigned long long*>(stream + L.chunk_index_off);
  const uint64_t per = (nchunks + kScanThreads - 1) / kScanThreads;
  const uint64_t lo = min(nchunks, per * threadIdx.x), hi = min(nchunks, lo + per);
  unsigned long long sum = 0;
  for (uint64_t c = lo; c < hi; ++c) sum += sizes[c];
  run_total[threadIdx.x] = sum;
  __syncthreads();
  for (int d = 1; d < kScanThreads; d <<= 1) {  // inclusive scan of the run totals
    const unsigned long long v = (int)threadIdx.x >= d ? run_total[threadIdx.x - d] : 0ull;
    __syncthreads();
    run_total[threadIdx.x] += v;
    __syncthreads();
  }
  unsigned long long off = run_total[threadIdx.x] - sum;
  for (uint64_t c = lo; c < hi; ++c) {
    chunk_index[c] = off;
    off += sizes[c];
  }
  if (threadIdx.x == kScanThreads - 1) {
    chunk_index[nchunks] = run_total[kScanThreads - 1];
    *reinterpret_cast<unsigned long long*>(stream + 48) = L.payload_off + run_total[kScanThreads - 1];
  }
}

}  // namespace

cudaError_t launch_encode(Control* ctl, unsigned long long* tiles, const uint8_t* plane, const float* base,
                          const float* cur, uint64_t n, uint8_t* stream, float* tracked_out, const EncodeOptions& opt,
                          cudaStream_t cs, bool overlap) {
  const WorkspaceLayout W = workspace_layout(n);
  if (W.nchunks == 0) return cudaSuccess;
  static int blocks_per_sm[kMaxDevices][2] = {}, sms[kMaxDevices] = {};  // by device ordinal
  const int dev = current_device_index();
  if (dev < 0) return cudaErrorInvalidDevice;
  const int v = tracked_out ? 1 : 0;
  if (blocks_per_sm[dev][v] == 0) {
    const void* fn = v ? reinterpret_cast<const void*>(encode_kernel<true>) : reinterpret_cast<const void*>(encode_kernel<false>);
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kEncDyn + (v ? kUpdSmem : 0));
    if (e != cudaSuccess) return e;
    int nsm = 0;
    if ((e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    int bps = 0;
    e = v ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, encode_kernel<true>, kEncThreads, kEncDyn + kUpdSmem)
          : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, encode_kernel<false>, kEncThreads, kEncDyn);
    if (e != cudaSuccess) return e;
    sms[dev] = nsm;
    blocks_per_sm[dev][v] = bps > 0 ? bps : 1;
  }
  const uint64_t want = (W.nchunks + kEncWarps - 1) / kEncWarps;
  const uint64_t full = (uint64_t)sms[dev] * blocks_per_sm[dev][v];
  const unsigned grid = (unsigned)(want < full ? want : full);
  if (opt.two_pass_scan) {
    // tiles[] (zeroed by the caller, one entry per chunk) holds the chunk sizes in this mode
    encode_sizes_kernel<<<grid, kEncThreads, 0, cs>>>(ctl, tiles, plane, base, cur, n, W.nchunks);
    encode_scan_kernel<<<1, kScanThreads, 0, cs>>>(ctl, tiles, n, W.nchunks, stream);
    if (cudaGetLastError() != cudaSuccess) return cudaErrorLaunchFailure;
  }
  const uint32_t two = opt.two_pass_scan ? 1u : 0u;
  overlap = overlap && !opt.two_pass_scan;
  if (v)
    return launch_kernel(overlap, encode_kernel<true>, grid, kEncThreads, kEncDyn + kUpdSmem, cs, ctl, tiles, plane, base, cur, n, stream,
                         tracked_out, opt.spin_limit, opt.ticket_bias, two);
  return launch_kernel(overlap, encode_kernel<false>, grid, kEncThreads, kEncDyn, cs, ctl, tiles, plane, base, cur, n, stream,
                       static_cast<float*>(nullptr), opt.spin_limit, opt.ticket_bias, two);
}

}  // namespace lc
