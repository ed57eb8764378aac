// The compress pass of a vector of at most one chunk in one CTA (see lc_small.cu for the design): shared by the kernel
// for one vector and the kernel for the segments of a vector.
#pragma once
#include "lc_table.cuh"

namespace lc {
namespace small {

constexpr uint32_t kThreadSteps = 2;  // steps per warp: 16 warps cover the 32 steps of a chunk
static_assert(kThreadSteps * (kTableThreads / 32) == kSteps && kSmallMaxElems == kChunkElems, "one chunk per CTA");
constexpr uint32_t kHistCols = 8;     // columns of the histogram: lane % 8 (32 of them take longer to clear and fold)
constexpr uint32_t kImageWords = (kChunkElems * kMaxNbits / 8 + 16) / 4;  // the payload has at most nbits bits per element

struct SmallShared {
  TableShared T;
  union {
    struct {
      uint32_t cnt[kKeys * kHistCols];
      uint2 mm[kKeys];  // running maxima of ~bits and of bits
    } h;
    struct {
      uint4 image[kImageWords / 4];
      uint32_t bits[kTableThreads / 32][32];  // [warp][lane]: bit count, then bit position, of a thread's piece
      uint32_t code[kKeys], len[kKeys], rep[kKeys];
      uint32_t chunk_bytes;
    } c;
  };
};

__device__ __forceinline__ uint32_t key_of_bits(uint32_t bits) { return ((bits >> 31) << 8) | ((bits >> 23) & 255u); }

// One vector of n <= kSmallMaxElems elements; all threads of the CTA. dbg: nullptr, or the control block that receives
// the statistics and the code table (lc_debug_*). Returns 0 or the error that makes the vector unencodable.
__device__ __forceinline__ int small_vector(SmallShared& S, const float* base, const float* cur, uint32_t n, int nbits,
                                            uint8_t* stream, float* tracked_out, Control* dbg) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  // ---- load; delta against the tracked state
  float b[kThreadSteps][4];
  uint32_t d[kThreadSteps][4];
  uint32_t have[kThreadSteps];  // elements of the thread's slot group that exist
#pragma unroll
  for (uint32_t r = 0; r < kThreadSteps; ++r) {
    const uint32_t i = 128 * (kThreadSteps * warp + r) + 4 * lane;
    have[r] = i < n ? min(n - i, 4u) : 0u;
    float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (uint32_t e = 0; e < 4; ++e) b[r][e] = 0.f;
    if (have[r] == 4) {
      const float4 b4 = *reinterpret_cast<const float4*>(base + i), c4 = *reinterpret_cast<const float4*>(cur + i);
      b[r][0] = b4.x; b[r][1] = b4.y; b[r][2] = b4.z; b[r][3] = b4.w;
      c[0] = c4.x; c[1] = c4.y; c[2] = c4.z; c[3] = c4.w;
    } else {
#pragma unroll
      for (uint32_t e = 0; e < 3; ++e)
        if (e < have[r]) b[r][e] = base[i + e], c[e] = cur[i + e];
    }
#pragma unroll
    for (uint32_t e = 0; e < 4; ++e) d[r][e] = __float_as_uint(__fsub_rn(c[e], b[r][e]));
  }

  // ---- statistics (Section 3.1.1): count, and the running maxima of ~bits and bits, per key
  for (uint32_t k = tid; k < kKeys * kHistCols / 4; k += kTableThreads) reinterpret_cast<uint4*>(S.h.cnt)[k] = make_uint4(0u, 0u, 0u, 0u);
  S.h.mm[tid] = make_uint2(0u, 0u);
  __syncthreads();
#pragma unroll
  for (uint32_t r = 0; r < kThreadSteps; ++r)
#pragma unroll
    for (uint32_t e = 0; e < 4; ++e)
      if (e < have[r]) {
        const uint32_t bits = d[r][e], key = key_of_bits(bits);
        atomicAdd(&S.h.cnt[key * kHistCols + lane % kHistCols], 1u);
        const uint2 mm = S.h.mm[key];
        if (~bits > mm.x) atomicMax(&S.h.mm[key].x, ~bits);
        if (bits > mm.y) atomicMax(&S.h.mm[key].y, bits);
      }
  __syncthreads();
  const uint32_t my_key = key_of_position(tid);
  KeyStats my;
  {
    const uint4* row = reinterpret_cast<const uint4*>(&S.h.cnt[my_key * kHistCols]);
    const uint4 x = row[0], y = row[1];
    static_assert(kHistCols == 8, "two 16-byte reads");
    my.count = my.local = x.x + x.y + x.z + x.w + y.x + y.y + y.z + y.w;
    my.inv_min = S.h.mm[my_key].x;
    my.max_bits = S.h.mm[my_key].y;
    my.mant_sum = 0;
  }
  if (dbg) {
    dbg->count[my_key] = my.count;
    dbg->inv_min[my_key] = my.inv_min;
    dbg->max_bits[my_key] = my.max_bits;
    dbg->mant_sum[my_key] = 0;
  }

  // ---- table pass: header, symbol table (its barriers also end the histogram's use)
  const int err = table_pass(S.T, my, TableArgs{n, nbits, true, false, false, false, nullptr}, stream);
  if (err || n == 0) return err;
  {
    const uint32_t sym = S.T.sym_of_key[my_key];
    const unsigned long long code = S.T.code[sym];
    S.c.code[my_key] = (uint32_t)code;
    S.c.len[my_key] = S.T.len[sym];
    S.c.rep[my_key] = S.T.rep[sym];
    if (dbg) dbg->enc[my_key] = EncEntry{(uint32_t)code, S.T.len[sym], (uint32_t)(code >> 32), sym};
  }
  for (uint32_t k = tid; k < kImageWords / 4; k += kTableThreads) S.c.image[k] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();

  // ---- tracked state (Algorithm 1 step 7; tracked_out may be base: a thread reads only its own elements), and the bit
  // count of the thread's piece
  uint32_t piece = 0;
#pragma unroll
  for (uint32_t r = 0; r < kThreadSteps; ++r) {
    float x[4];
#pragma unroll
    for (uint32_t e = 0; e < 4; ++e) {
      const uint32_t key = key_of_bits(d[r][e]);
      if (e < have[r]) piece += S.c.len[key];
      x[e] = __fadd_rn(b[r][e], __uint_as_float(S.c.rep[key]));
    }
    if (tracked_out) {
      const uint32_t i = 128 * (kThreadSteps * warp + r) + 4 * lane;
      if (have[r] == 4) {
        *reinterpret_cast<float4*>(tracked_out + i) = make_float4(x[0], x[1], x[2], x[3]);
      } else {
#pragma unroll
        for (uint32_t e = 0; e < 3; ++e)
          if (e < have[r]) tracked_out[i + e] = x[e];
      }
    }
  }
  S.c.bits[warp][lane] = piece;
  __syncthreads();

  // ---- bit position of every piece: pieces of a lane follow each other by warp, lanes follow each other
  const StreamLayout L = stream_layout(n, S.T.nsym);
  if (warp == 0) {
    uint32_t at[kTableThreads / 32], total = 0;
#pragma unroll
    for (uint32_t w = 0; w < kTableThreads / 32; ++w) {
      at[w] = total;
      total += S.c.bits[w][lane];
    }
    uint32_t incl = total;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, s);
      if ((int)lane >= s) incl += v;
    }
#pragma unroll
    for (uint32_t w = 0; w < kTableThreads / 32; ++w) S.c.bits[w][lane] = incl - total + at[w];
    reinterpret_cast<uint16_t*>(stream + L.lane_index_off)[lane] = (uint16_t)total;
    if (lane == 31) {
      const uint32_t bytes = (uint32_t)align_up((incl + 7) / 8, kPayloadAlign);
      S.c.chunk_bytes = bytes;
      unsigned long long* chunk_index = reinterpret_cast<unsigned long long*>(stream + L.chunk_index_off);
      chunk_index[0] = 0;
      chunk_index[1] = bytes;
      *reinterpret_cast<unsigned long long*>(stream + 48) = L.payload_off + bytes;
    }
  }
  __syncthreads();

  // ---- the codes
  if (piece > 0) {
    uint32_t* image = reinterpret_cast<uint32_t*>(S.c.image);
    const uint32_t pos = S.c.bits[warp][lane];
    uint32_t* dst = image + (pos >> 5);
    unsigned long long acc = 0;  // pending bits in the low `nb` bits; the first word's leading bits belong to others
    uint32_t nb = pos & 31u;
    auto put = [&](uint32_t code, uint32_t len) {  // len <= 32
      acc = (acc << len) | code;
      nb += len;
      if (nb >= 32) {
        nb -= 32;
        atomicOr(dst, (uint32_t)(acc >> nb));
        dst += 1;
      }
    };
#pragma unroll
    for (uint32_t r = 0; r < kThreadSteps; ++r)
#pragma unroll
      for (uint32_t e = 0; e < 4; ++e) {
        if (e >= have[r]) continue;
        const uint32_t key = key_of_bits(d[r][e]), len = S.c.len[key];
        if (len > 32) {
          put((uint32_t)(S.T.code[S.T.sym_of_key[key]] >> 32), len - 32);
          put(S.c.code[key], 32);
        } else {
          put(S.c.code[key], len);
        }
      }
    if (nb > 0) atomicOr(dst, (uint32_t)(acc << (32 - nb)));
  }
  __syncthreads();
  uint4* payload = reinterpret_cast<uint4*>(stream + L.payload_off);
  for (uint32_t k = tid; k < S.c.chunk_bytes / 16; k += kTableThreads) payload[k] = S.c.image[k];
  return LC_OK;
}

}  // namespace small
}  // namespace lc
