// Per-layer compress: the compress pass (Algorithm 1 steps 4-6, optionally step 7) of many segments of a vector, each
// coded as a stream of its own, in three launches for up to 128 segments.
//
// Segment after segment through the passes for one vector, a model of 62 layers took 62 times a memset and three
// launches, most of them on a handful of SMs: 1540 us (1234 us with the faster table pass) for 11.7 M values that take 22 us
// to move; in this form 117 us, of which the three kernels take 21, 11 and 36 us. Here
//   1. segments_stats_kernel: several CTAs per segment; a segment of at most one chunk is only checked for non-finite
//      deltas (the segments behind a failed one must be left without a stream, so all failures have to be known first);
//   2. segments_table_kernel: one CTA per segment: the table pass, or the whole pass of a segment of one chunk;
//   3. segments_encode_kernel: one CTA per tile of 8 chunks of the larger segments.
// There is no key plane in global memory (the workspace is sized for the longest segment only): the encode kernel forms
// the keys again from base and cur, which for models of this size are still in the L2, and keeps them in shared memory,
// and it writes the tracked state from the registers it has base in. (Segments far larger than the L2 are not brought here:
// kSegLarge.)
#include "lc_encode_bits.cuh"
#include "lc_small.cuh"
#include "lc_stats.cuh"

namespace lc {
namespace {

using namespace enc;
using namespace stats;

// The segment that CTA (or tile) b belongs to: the last one with begin[i] <= b.
__device__ __forceinline__ uint32_t find_segment(const uint32_t* begin, uint32_t nseg, uint32_t b) {
  uint32_t lo = 0, hi = nseg;
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) / 2;
    if (begin[mid] <= b) lo = mid;
    else hi = mid;
  }
  return lo;
}

__global__ void __launch_bounds__(kStatsThreads, 2)
segments_stats_kernel(const float* base, const float* __restrict__ cur, Control* __restrict__ ctl, SegBlock* __restrict__ blocks,
                      const __grid_constant__ SegGroup group) {
  extern __shared__ __align__(16) uint32_t smem[];
  begin_next();
  const uint32_t s = find_segment(group.cta_begin, group.nseg, blockIdx.x);
  const uint64_t lo = group.elem_begin[s], n = group.elem_begin[s + 1] - lo;
  bool bad = false;
  if (n <= kChunkElems) {
    for (uint32_t i = threadIdx.x; i < n; i += kStatsThreads)
      bad |= (__float_as_uint(__fsub_rn(cur[lo + i], base[lo + i])) & 0x7f800000u) == 0x7f800000u;
  } else {
    uint32_t* cnt = smem;
    uint2* mm = reinterpret_cast<uint2*>(smem + kCntWords);
    uint4* clear = reinterpret_cast<uint4*>(smem);
    for (uint32_t i = threadIdx.x; i < (kCntWords + 2 * kKeys) / 4; i += kStatsThreads) clear[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t cta = blockIdx.x - group.cta_begin[s], ctas = group.cta_begin[s + 1] - group.cta_begin[s];
    Acc<false> acc{cnt + lane, mm};
    stats_units<false, false>(acc, base + lo, cur + lo, n, (uint64_t)cta * (kStatsThreads / 32) + warp, (n + kUnitElems - 1) / kUnitElems,
                              (uint64_t)ctas * (kStatsThreads / 32), lane, nullptr);
    wait_previous();  // the blocks are clear
    __syncthreads();
    ShardStats& out = blocks[group.block[s]].stats;
    bad = fold_stats<false>(cnt, mm, out.count, out.inv_min, out.max_bits, nullptr);
  }
  wait_previous();
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicMax(&ctl->seg_fail, ~(group.first + s));
  // a segment before this group that went through the passes for one vector has failed: all of the group are behind it
  if (group.first > 0 && blockIdx.x == 0 && threadIdx.x == 0 && ctl->status != 0) atomicMax(&ctl->seg_fail, ~(group.first - 1));
}

__global__ void __launch_bounds__(kTableThreads)
segments_table_kernel(const float* base, const float* cur, Control* __restrict__ ctl, SegBlock* __restrict__ blocks, int nbits,
                      uint8_t* __restrict__ streams, float* tracked_out, const __grid_constant__ SegGroup group) {
  extern __shared__ __align__(16) unsigned char s_small[];
  small::SmallShared<1>& S = *reinterpret_cast<small::SmallShared<1>*>(s_small);
  begin_next();
  const uint32_t s = blockIdx.x, tid = threadIdx.x;
  const uint64_t lo = group.elem_begin[s], n = group.elem_begin[s + 1] - lo;
  uint8_t* stream = streams + group.stream_begin[s];
  // The first failed segment, and every one behind it, is left without a stream; nothing in this kernel writes the word.
  const auto failed = [&]() {
    wait_previous();
    const uint32_t fail = *reinterpret_cast<volatile uint32_t*>(&ctl->seg_fail);
    if (s == 0 && tid == 0) ctl->seg_ticket = 0;
    if (fail == 0 || group.first + s < ~fail) return false;
    if (tid == 0 && group.first + s == ~fail) set_status_ranked(&ctl->status, ~fail, LC_ERR_NONFINITE);
    return true;
  };
  if (n <= kChunkElems) {
    // Everything up to the first write runs beside the statistics pass, on the SMs that its CTAs leave: a segment of one chunk needs none of
    // its results but which segments have failed. (11.7 M elements in 62 layers 66.9 -> 61.7 us, 2 M in 20 47.9 -> 44.7, with the look-back's 128
    // descriptors a round.)
    bool without = false;
    const int err = small::small_vector<1, false>(S, base + lo, cur + lo, (uint32_t)n, nbits, stream, tracked_out ? tracked_out + lo : nullptr, nullptr,
                                                  [&]() { return !(without = failed()); });
    if (err && !without) failed();  // its own failure, which the statistics pass has found too
    if (err) clear_header(stream);
    return;
  }
  if (failed()) {
    clear_header(stream);
    return;
  }
  SegBlock& B = blocks[group.block[s]];
  const uint32_t key = key_of_position(tid);
  KeyStats my;
  my.count = my.local = B.stats.count[key];
  my.inv_min = B.stats.inv_min[key];
  my.max_bits = B.stats.max_bits[key];
  my.mant_sum = 0;
  if (table_pass(S.T, my, TableArgs{n, nbits, true, false, false, false, nullptr}, stream) != LC_OK) return;
  const uint32_t sym = S.T.sym_of_key[key];
  // the table takes the place of the statistics, which every thread has read before the table pass's barriers
  B.enc[key] = EncEntry{(uint32_t)S.T.code[sym], S.T.len[sym], (uint32_t)(S.T.code[sym] >> 32), sym};
  if (tid == 0) {
    B.nsym = S.T.nsym;
    B.max_len = S.T.max_len;
    B.wide = S.T.wide;
    B.payload_bits = S.T.payload_bits;
  }
}

// ---- encode ------------------------------------------------------------------------------------------------
// A warp's shared memory: the column matrix of phase A (lane_words rows of 32 words), then the chunk's plane bytes, whose
// place the chunk's image takes once it is coded.
constexpr int kSegThreads = kEncWarps * 32;

// Rows of the column matrix: nbits bits per element is the average of a code that saves nothing, and one eighth more is
// left for lanes above their chunk's average; a lane that outgrows its column takes the slow path.
inline uint32_t seg_lane_words(int nbits) { return 4u * (uint32_t)nbits + (uint32_t)nbits / 2 + 2; }
inline uint32_t seg_image_bytes(int nbits) { return nbits <= 7 ? kChunkElems : kChunkElems * (uint32_t)nbits / 8 + 256; }

__device__ __forceinline__ float4 load_group(const float* p, uint32_t have) {
  if (have >= 4) return *reinterpret_cast<const float4*>(p);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (have > 0) v.x = p[0];
  if (have > 1) v.y = p[1];
  if (have > 2) v.z = p[2];
  return v;
}

// One CTA per tile; the tiles are handed out by a ticket, so that every tile a CTA waits for in the look-back is being
// coded by a CTA that already runs. Bound: latency at one tile per CTA (a model of 11.7 M values has 370 tiles, all of
// them resident at once), then the integer work of coding.
__global__ void __launch_bounds__(kSegThreads, 3)
segments_encode_kernel(Control* __restrict__ ctl, const SegBlock* __restrict__ blocks, unsigned long long* __restrict__ tiles,
                       const float* base, const float* cur, uint8_t* __restrict__ streams, float* tracked_out,
                       uint32_t lane_words, uint32_t image_bytes, uint32_t spin_limit, const __grid_constant__ SegGroup group) {
  extern __shared__ __align__(128) unsigned char s_all[];
  Tables& tb = shared_tables();
  unsigned char* s_dyn = s_all + kTablesBytes;
  __shared__ uint32_t s_rep[256];  // representative (bit pattern) by the low byte of a slot, which is plane byte ^ 1
  __shared__ uint32_t s_bytes[kEncWarps];
  __shared__ uint32_t s_tile;
  __shared__ unsigned long long s_prefix;
  __shared__ int s_abort;
  wait_previous();
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    s_tile = atomicAdd(&ctl->seg_ticket, 1u);
    s_abort = 0;
  }
  __syncthreads();
  const uint32_t tile = s_tile;
  const uint32_t s = find_segment(group.tile_begin, group.nseg, tile);
  const SegBlock& B = blocks[group.block[s]];
  static_assert(kSegThreads == 256, "a thread per plane byte");
  const EncEntry e = B.enc[key_of_byte(tid)];
  const uint32_t nsym = B.nsym, sym0_len = B.enc[0].len;
  if (nsym == 0) return;  // failed: the same word for every thread
  const uint64_t lo = group.elem_begin[s], n = group.elem_begin[s + 1] - lo;
  uint8_t* stream = streams + group.stream_begin[s];
  const bool wide = B.wide != 0, long_codes = B.max_len > 32;
  const uint32_t rep = *reinterpret_cast<const uint32_t*>(stream + kHeaderBytes + kTableEntryBytes * e.sym + 4);
  if (tid == 0) tb.long_codes = long_codes;
  tb.full[tid] = make_uint2(e.code_lo, e.len);
  __syncthreads();
  build_tables(tb, sym0_len, [&](uint32_t) { return e.sym != 0; });
  s_rep[tid ^ 1] = rep;
  __syncthreads();

  const StreamLayout L = stream_layout(n, nsym);
  const uint32_t first_tile = group.tile_begin[s], last_tile = group.tile_begin[s + 1] - 1;
  const uint64_t c = (uint64_t)(tile - first_tile) * kEncWarps + warp;
  const bool valid = c < L.nchunks;
  const uint32_t rem = valid ? (uint32_t)min((uint64_t)kChunkElems, n - c * kChunkElems) : 0u;  // elements of the chunk
  uint32_t* column = reinterpret_cast<uint32_t*>(s_dyn + warp * (lane_words * 128 + image_bytes));
  uint8_t* plane = reinterpret_cast<uint8_t*>(column + lane_words * 32);
  uint32_t* image = reinterpret_cast<uint32_t*>(plane);
  const uint32_t col0 = smem_addr(column) + lane * 4;
  // the slow path reads the plane in shared memory, or base and cur if a byte does not identify a bucket
  const KeySource ks{plane - c * kChunkElems, base + lo, cur + lo, wide};

  uint32_t lane_bits = 0;
  bool fast = valid && !wide && !long_codes;
  if (valid && !wide) {
    // ---- delta, plane bytes and tracked state. A lane reads back only the bytes it wrote itself.
    const uint64_t e0 = lo + c * kChunkElems + 4 * lane;
#pragma unroll 1
    for (uint32_t q = 0; q < kSteps / 4; ++q) {
      float4 b4[4], c4[4];
      uint32_t w[4];
#pragma unroll
      for (uint32_t r = 0; r < 4; ++r) {
        const uint32_t i = (4 * q + r) * 128 + 4 * lane, have = i < rem ? rem - i : 0u;
        b4[r] = load_group(base + e0 + (4 * q + r) * 128, have);
        c4[r] = load_group(cur + e0 + (4 * q + r) * 128, have);
      }
#pragma unroll
      for (uint32_t r = 0; r < 4; ++r) {
        const uint32_t k0 = slot_of(__float_as_uint(__fsub_rn(c4[r].x, b4[r].x)));
        const uint32_t k1 = slot_of(__float_as_uint(__fsub_rn(c4[r].y, b4[r].y)));
        const uint32_t k2 = slot_of(__float_as_uint(__fsub_rn(c4[r].z, b4[r].z)));
        const uint32_t k3 = slot_of(__float_as_uint(__fsub_rn(c4[r].w, b4[r].w)));
        w[r] = __byte_perm(__byte_perm(k0, k1, 0x0040), __byte_perm(k2, k3, 0x0040), 0x5410) ^ kPlaneFlip;  // all exponent fields are below 128
        if (tracked_out) {
          const uint32_t i = (4 * q + r) * 128 + 4 * lane, have = i < rem ? rem - i : 0u;
          float4 x;
          x.x = __fadd_rn(b4[r].x, __uint_as_float(s_rep[k0 & 255u]));
          x.y = __fadd_rn(b4[r].y, __uint_as_float(s_rep[k1 & 255u]));
          x.z = __fadd_rn(b4[r].z, __uint_as_float(s_rep[k2 & 255u]));
          x.w = __fadd_rn(b4[r].w, __uint_as_float(s_rep[k3 & 255u]));
          float* o = tracked_out + e0 + (4 * q + r) * 128;
          if (have >= 4) {
            *reinterpret_cast<float4*>(o) = x;
          } else {
            if (have > 0) o[0] = x.x;
            if (have > 1) o[1] = x.y;
            if (have > 2) o[2] = x.z;
          }
        }
      }
      reinterpret_cast<uint4*>(plane)[q * 32 + lane] = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
  // ---- A: code the lane's elements into its column, lookups one row ahead of the appends
  if (fast) {
    const uint4* ep = reinterpret_cast<const uint4*>(plane) + lane;
    if (rem == kChunkElems) {
      ColumnPacker pk{0u, 0u, col0, col0 + lane_words * 128};
      const uint32_t neg_base = (uint32_t)(-tb.base) & 0xffffu, neg_base2 = neg_base << 16 | neg_base;
      auto load = [&](int q) { return ep[32 * q]; };
      auto row = [](uint32_t, int) {};
      if (tb.use_pair) code_rows<true>(pk, tb, neg_base2, load, row);
      else code_rows<false>(pk, tb, neg_base2, load, row);
      lane_bits = finish_column(pk, col0);
    } else {
      lane_bits = code_partial(&tb, ep, rem, lane, col0, lane_words);
    }
    if (__any_sync(0xffffffffu, lane_bits == 0xffffffffu)) fast = false;  // some lane outgrew its column
  }
  if (!fast && valid) lane_bits = chunk_slow<true>(B.enc, ks, c, lane, n, nullptr, 0);

  // ---- B: lane offsets, lane index, chunk size
  if (valid) reinterpret_cast<uint16_t*>(stream + L.lane_index_off)[c * kLanes + lane] = (uint16_t)lane_bits;
  uint32_t incl = lane_bits;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t v = __shfl_up_sync(0xffffffffu, incl, d);
    if ((int)lane >= d) incl += v;
  }
  const uint32_t lane_start = incl - lane_bits;
  const uint32_t chunk_bits = __shfl_sync(0xffffffffu, incl, 31);
  const uint32_t chunk_bytes = valid ? (uint32_t)align_up((chunk_bits + 7) / 8, kPayloadAlign) : 0u;
  const bool staged = fast && chunk_bytes <= image_bytes;
  if (lane == 0) s_bytes[warp] = chunk_bytes;
  __syncthreads();
  unsigned long long before = 0, tile_bytes = 0;
#pragma unroll
  for (uint32_t w = 0; w < kEncWarps; ++w) {
    before += w < warp ? s_bytes[w] : 0u;
    tile_bytes += s_bytes[w];
  }
  if (tid == 0 && tile != last_tile)
    *reinterpret_cast<volatile unsigned long long*>(&tiles[tile]) =
        (tile == first_tile ? kTilePrefix : kTileAggregate) << kTileFlagShift | tile_bytes;

  // ---- C: assemble the chunk's image (in the place of the plane bytes, which have been read)
  if (staged) {
    __syncwarp();
    assemble_chunk(column, lane, lane_bits, lane_start, image, chunk_bytes);
  }

  // ---- D: the tile's offset: exclusive prefix over the segment's tiles by decoupled look-back (bounded), one warp
  if (warp == 0) {
    unsigned long long part = 0;
    bool abort = false;
    long long look = (long long)tile - 1;
    uint32_t spins = 0;
    bool done = tile == first_tile;
    while (!done && !abort) {
      // a round reads the 128 descriptors before `look` at once (a segment of 2.4 M elements has 72 tiles)
      unsigned long long st[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const long long idx = look - 32 * u - lane;
        st[u] = idx >= (long long)first_tile ? ld_tile(&tiles[idx]) : kTilePrefix << kTileFlagShift;
      }
      bool retry = false;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (done || abort || retry) continue;
        const uint32_t flag = (uint32_t)(st[u] >> kTileFlagShift);
        const uint32_t m_prefix = __ballot_sync(0xffffffffu, flag == kTilePrefix);
        const uint32_t m_other = __ballot_sync(0xffffffffu, flag != kTilePrefix && flag != kTileAggregate);
        const int first_prefix = m_prefix ? __ffs(m_prefix) - 1 : 32;
        const uint32_t relevant = first_prefix < 32 ? (0xffffffffu >> (31 - first_prefix)) : 0xffffffffu;
        if (m_other & relevant) {
          if (__ballot_sync(0xffffffffu, flag == kTileAbort) & relevant) abort = true;
          else retry = true;  // poll again from `look`, which already skips the complete windows
        } else {
          if ((int)lane <= first_prefix) part += st[u] & kTileValueMask;
          if (first_prefix < 32) done = true;
          else look -= 32;
        }
      }
      if (retry) {
        if (++spins > spin_limit) abort = true;
        else __nanosleep(40);
      }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) part += __shfl_xor_sync(0xffffffffu, part, d);
    if (lane == 0) {
      if (tile != first_tile && tile != last_tile)
        *reinterpret_cast<volatile unsigned long long*>(&tiles[tile]) =
            abort ? kTileAbort << kTileFlagShift : kTilePrefix << kTileFlagShift | (part + tile_bytes);
      if (abort) {
        // this segment and all behind it are left without a stream: those of later groups by the failure word, those of
        // this one by taking the magic away again, which nobody else writes in this kernel
        s_abort = 1;
        set_status_ranked(&ctl->status, group.first + s, LC_ERR_TIMEOUT);
        atomicMax(&ctl->seg_fail, ~(group.first + s));
        for (uint32_t j = s; j < group.nseg; ++j) *reinterpret_cast<uint32_t*>(streams + group.stream_begin[j]) = 0u;
      }
      s_prefix = part;
    }
  }
  __syncthreads();
  if (s_abort) return;

  // ---- E: the payload, the chunk index, and with the last tile the stream's size
  const unsigned long long off = s_prefix + before;
  unsigned long long* chunk_index = reinterpret_cast<unsigned long long*>(stream + L.chunk_index_off);
  if (valid) {
    if (lane == 0) chunk_index[c] = off;
    uint4* dst4 = reinterpret_cast<uint4*>(stream + L.payload_off + off);
    if (staged) {
      const uint4* im4 = reinterpret_cast<const uint4*>(image);
      for (uint32_t k = lane; k < chunk_bytes / 16; k += 32) dst4[k] = im4[k];
    } else if (fast) {
      // coded, but larger than the image area: OR the column's words into (zeroed) global memory
      for (uint32_t k = lane; k < chunk_bytes / 16; k += 32) dst4[k] = make_uint4(0, 0, 0, 0);
      __threadfence_block();
      __syncwarp();
      or_column(column, lane, lane_bits, lane_start, reinterpret_cast<uint32_t*>(dst4));
    } else {
      for (uint32_t k = lane; k < chunk_bytes / 16; k += 32) dst4[k] = make_uint4(0, 0, 0, 0);
      __threadfence_block();
      __syncwarp();
      chunk_slow<true>(B.enc, ks, c, lane, n, reinterpret_cast<uint32_t*>(dst4), lane_start);
    }
  }
  if (tile == last_tile && tid == 0) {
    const unsigned long long payload_bytes = s_prefix + tile_bytes;
    chunk_index[L.nchunks] = payload_bytes;
    *reinterpret_cast<unsigned long long*>(stream + 48) = L.payload_off + payload_bytes;
  }
  // ---- tracked state of a segment whose keys come from base and cur: only now has its coding read them for the last time
  if (tracked_out && valid && wide) {
    for (uint32_t j = 0; j < kSteps; ++j)
      for (uint32_t e = 0; e < kGroup; ++e) {
        const uint32_t i = 128 * j + 4 * lane + e;
        if (i >= rem) continue;
        const uint64_t at = lo + c * kChunkElems + i;
        const uint32_t sym = B.enc[ks.key(c, j, lane, e)].sym;
        const uint32_t rep = *reinterpret_cast<const uint32_t*>(stream + kHeaderBytes + kTableEntryBytes * sym + 4);
        tracked_out[at] = __fadd_rn(base[at], __uint_as_float(rep));
      }
  }
}

}  // namespace

cudaError_t launch_compress_segments(Control* ctl, SegBlock* blocks, unsigned long long* tiles, const float* base,
                                     const float* cur, SegGroup& group, int nbits, uint8_t* streams, float* tracked_out,
                                     cudaStream_t cs) {
  static int sms_of[kMaxDevices] = {};  // by device ordinal; non-zero once the kernels' attributes are set there
  const int dev = current_device_index();
  if (dev < 0) return cudaErrorInvalidDevice;
  if (sms_of[dev] == 0) {
    int v = 0;
    cudaError_t e = cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(segments_stats_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kStatsSmem);
    // the carve-out that two resident CTAs need, as for the kernel for one vector (the rest serves as L1)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(segments_stats_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 61);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(segments_table_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(small::SmallShared<1>));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(segments_encode_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)(kTablesBytes + kEncWarps * (seg_lane_words(kMaxNbits) * 128 + seg_image_bytes(kMaxNbits))));
    if (e != cudaSuccess) return e;
    sms_of[dev] = v;
  }
  if (group.nseg == 0) return cudaSuccess;
  // Statistics CTAs: one unit per warp while all CTAs fit on the device at once (two per SM), else as many more as that
  // takes; a second wave would only clear and fold its tables again.
  const uint64_t slots = 2ull * (uint64_t)sms_of[dev];
  uint64_t ctas = 0;
  for (uint64_t per_cta = kStatsThreads / 32;; per_cta += kStatsThreads / 32) {
    ctas = 0;
    uint64_t longest = 0;
    for (uint32_t i = 0; i < group.nseg; ++i) {
      const uint64_t n = group.elem_begin[i + 1] - group.elem_begin[i], units = (n + kUnitElems - 1) / kUnitElems;
      group.cta_begin[i] = (uint32_t)ctas;
      ctas += n <= kChunkElems ? (n > 0 ? 1 : 0) : (units + per_cta - 1) / per_cta;
      longest = units > longest ? units : longest;
    }
    if (ctas <= slots || per_cta >= longest) break;
  }
  group.cta_begin[group.nseg] = (uint32_t)ctas;
  // overlapped launches, the first behind the caller's clear kernel; one CTA at least, which looks at the status word
  cudaError_t e = launch_kernel(true, segments_stats_kernel, (unsigned)(ctas > 0 ? ctas : 1), kStatsThreads, kStatsSmem, cs, base, cur,
                                ctl, blocks, group);
  if (e == cudaSuccess)
    e = launch_kernel(true, segments_table_kernel, group.nseg, kTableThreads, sizeof(small::SmallShared<1>), cs, base, cur, ctl, blocks,
                      nbits, streams, tracked_out, group);
  const uint32_t ntiles = group.tile_begin[group.nseg];
  if (e == cudaSuccess && ntiles > 0) {
    const uint32_t lane_words = seg_lane_words(nbits), image_bytes = seg_image_bytes(nbits);
    e = launch_kernel(true, segments_encode_kernel, ntiles, kSegThreads, kTablesBytes + kEncWarps * (lane_words * 128 + image_bytes), cs, ctl, blocks,
                      tiles, base, cur, streams, tracked_out, lane_words, image_bytes, EncodeOptions().spin_limit, group);
  }
  return e;
}

}  // namespace lc
