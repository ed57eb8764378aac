// The compress pass of a vector of a few chunks without any workspace, in one CTA or one cluster of CTAs (see lc_small.cu
// for the design): shared by the kernels for one vector and the kernel for the segments of a vector.
#pragma once
#include "lc_table.cuh"

namespace lc {
namespace small {

constexpr uint32_t kWarps = kTableThreads / 32;
constexpr uint32_t kThreadSteps = 2;  // steps per warp and chunk: 16 warps cover the 32 steps of a chunk
static_assert(kThreadSteps * kWarps == kSteps, "a chunk per pass over the CTA's warps");
constexpr uint32_t kHistCols = 8;     // columns of the histogram: lane % 8 (32 of them take longer to clear and fold)
// a chunk's image holds nbits bits per element, which the payload of a vector of one chunk cannot exceed; a chunk of a
// larger vector that does is coded in global memory
constexpr uint32_t kImageBytes = kChunkElems * kMaxNbits / 8 + 16;

// M: chunks per CTA
template <int M>
struct SmallShared {
  TableShared T;
  union {
    struct {
      uint32_t cnt[kKeys * kHistCols];
      uint2 mm[kKeys];  // running maxima of ~bits and of bits
    } h;
    struct {
      uint4 image[M][kImageBytes / 16];
      uint32_t bits[M][kWarps][32];  // [chunk][warp][lane]: bit count, then bit position, of a thread's piece
      uint32_t code[kKeys], len[kKeys], rep[kKeys];
    } c;
  };
  uint32_t fold[3][kKeys];   // cluster: count and running maxima of this CTA's elements, by position
  uint32_t whole[3][kKeys];  // cluster: of the vector; the CTAs add to each other's
  uint32_t present[kWarps];  // cluster: which positions have a count in `fold`
  uint32_t chunk_bytes[M];
};

__device__ __forceinline__ uint32_t key_of_bits(uint32_t bits) { return ((bits >> 31) << 8) | ((bits >> 23) & 255u); }

// ---- cluster: shared memory of the other CTAs, and the barrier (it also orders those accesses)
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// address, in the shared memory of CTA `rank`, of what lies at `p` in this CTA's
__device__ __forceinline__ uint32_t cluster_addr(const void* p, uint32_t rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void cluster_add(uint32_t a, uint32_t v) {
  asm volatile("red.relaxed.cluster.shared::cluster.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void cluster_max(uint32_t a, uint32_t v) {
  asm volatile("red.relaxed.cluster.shared::cluster.max.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t cluster_ld(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}

// One vector of n <= (CTAs) * M * kChunkElems elements; all threads of the CTA or cluster. dbg: nullptr, or the control
// block that receives the statistics and the code table (lc_debug_*). Returns 0 or the error that makes the vector
// unencodable, the same everywhere.
// gate: table_pass's; nothing is written to the stream, or to tracked_out, before it.
template <int M, bool CLUSTER, class Gate = NoGate>
__device__ __forceinline__ int small_vector(SmallShared<M>& S, const float* base, const float* cur, uint32_t n, int nbits,
                                            uint8_t* stream, float* tracked_out, Control* dbg, Gate gate = Gate()) {
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = CLUSTER ? cluster_rank() : 0u, ctas = CLUSTER ? cluster_size() : 1u;
  const uint32_t chunk0 = rank * M;  // this CTA's first chunk
  const auto element = [&](uint32_t m, uint32_t r) {  // first element of the thread's slot group
    return (chunk0 + m) * kChunkElems + 128 * (kThreadSteps * warp + r) + 4 * lane;
  };
  const auto held = [&](uint32_t m, uint32_t r) {  // elements of that group that exist
    const uint32_t i = element(m, r);
    return i < n ? min(n - i, 4u) : 0u;
  };

  if (CLUSTER) {
#pragma unroll
    for (int i = 0; i < 3; ++i) S.whole[i][tid] = 0;
    cluster_arrive();
  }
  // ---- load; delta against the tracked state
  float b[M][kThreadSteps][4];
  uint32_t d[M][kThreadSteps][4];
#pragma unroll
  for (uint32_t m = 0; m < M; ++m)
#pragma unroll
    for (uint32_t r = 0; r < kThreadSteps; ++r) {
      const uint32_t i = element(m, r), have = held(m, r);
      float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (uint32_t e = 0; e < 4; ++e) b[m][r][e] = 0.f;
      if (have == 4) {
        const float4 b4 = *reinterpret_cast<const float4*>(base + i), c4 = *reinterpret_cast<const float4*>(cur + i);
        b[m][r][0] = b4.x; b[m][r][1] = b4.y; b[m][r][2] = b4.z; b[m][r][3] = b4.w;
        c[0] = c4.x; c[1] = c4.y; c[2] = c4.z; c[3] = c4.w;
      } else {
#pragma unroll
        for (uint32_t e = 0; e < 3; ++e)
          if (e < have) b[m][r][e] = base[i + e], c[e] = cur[i + e];
      }
#pragma unroll
      for (uint32_t e = 0; e < 4; ++e) d[m][r][e] = __float_as_uint(__fsub_rn(c[e], b[m][r][e]));
    }

  // ---- statistics (Section 3.1.1): count, and the running maxima of ~bits and bits, per key
  for (uint32_t k = tid; k < kKeys * kHistCols / 4; k += kTableThreads) reinterpret_cast<uint4*>(S.h.cnt)[k] = make_uint4(0u, 0u, 0u, 0u);
  S.h.mm[tid] = make_uint2(0u, 0u);
  __syncthreads();
#pragma unroll
  for (uint32_t m = 0; m < M; ++m)
#pragma unroll
    for (uint32_t r = 0; r < kThreadSteps; ++r) {
      // four at once: counts and reads of the running maxima do not wait for each other
      const uint32_t have = held(m, r);
      uint2 mm[4];
#pragma unroll
      for (uint32_t e = 0; e < 4; ++e)
        if (e < have) {
          const uint32_t key = key_of_bits(d[m][r][e]);
          mm[e] = S.h.mm[key];
          atomicAdd(&S.h.cnt[key * kHistCols + lane % kHistCols], 1u);
        }
#pragma unroll
      for (uint32_t e = 0; e < 4; ++e)
        if (e < have) {
          const uint32_t bits = d[m][r][e], key = key_of_bits(bits);
          if (~bits > mm[e].x) atomicMax(&S.h.mm[key].x, ~bits);
          if (bits > mm[e].y) atomicMax(&S.h.mm[key].y, bits);
        }
    }
  __syncthreads();
  const uint32_t my_key = key_of_position(tid);
  uint4 f;
  {
    const uint4* row = reinterpret_cast<const uint4*>(&S.h.cnt[my_key * kHistCols]);
    const uint4 x = row[0], y = row[1];
    static_assert(kHistCols == 8, "two 16-byte reads");
    f = make_uint4(x.x + x.y + x.z + x.w + y.x + y.y + y.z + y.w, S.h.mm[my_key].x, S.h.mm[my_key].y, 0u);
  }
  if (CLUSTER) {
    // Every CTA adds its own to all of them, a warp to one; few of the 512 keys occur, and only those go. (With every CTA reading the others' of the keys that
    // occur, each read waiting for its answer, this took 9000 of the 23,500 cycles of a vector of 61,706 elements; now 5200 of 20,100.)
    S.fold[0][tid] = f.x;
    S.fold[1][tid] = f.y;
    S.fold[2][tid] = f.z;
    const uint32_t present = __ballot_sync(0xffffffffu, f.x != 0);
    if (lane == 0) S.present[warp] = present;
    __syncthreads();
    cluster_wait();  // all CTAs have cleared `whole`
    static_assert(kWarps >= 16, "a warp per CTA of the largest cluster");
    if (warp < ctas) {
      const uint32_t whole = cluster_addr(&S.whole[0][lane], (rank + warp) & (ctas - 1));  // every CTA begins with another one
#pragma unroll 4
      for (uint32_t g = 0; g < kWarps; ++g)
        if ((S.present[g] >> lane) & 1u) {
          const uint32_t at = whole + 128 * g;
          cluster_add(at, S.fold[0][32 * g + lane]);
          cluster_max(at + 4 * kKeys, S.fold[1][32 * g + lane]);
          cluster_max(at + 8 * kKeys, S.fold[2][32 * g + lane]);
        }
    }
    cluster_arrive();
    cluster_wait();
    f = make_uint4(S.whole[0][tid], S.whole[1][tid], S.whole[2][tid], 0u);
  }
  KeyStats my;
  my.count = my.local = f.x;
  my.inv_min = f.y;
  my.max_bits = f.z;
  my.mant_sum = 0;
  if (dbg && rank == 0) {
    dbg->count[my_key] = my.count;
    dbg->inv_min[my_key] = my.inv_min;
    dbg->max_bits[my_key] = my.max_bits;
    dbg->mant_sum[my_key] = 0;
  }

  // ---- table pass, in every CTA (its barriers also end the histogram's use); header and symbol table by the first
  const int err = table_pass(S.T, my, TableArgs{n, nbits, true, false, false, false, nullptr}, stream, rank == 0, gate);
  if (err) return err;
  if (n == 0) return LC_OK;
  {
    const uint32_t sym = S.T.sym_of_key[my_key];
    const unsigned long long code = S.T.code[sym];
    S.c.code[my_key] = (uint32_t)code;
    S.c.len[my_key] = S.T.len[sym];
    S.c.rep[my_key] = S.T.rep[sym];
    if (dbg && rank == 0) dbg->enc[my_key] = EncEntry{(uint32_t)code, S.T.len[sym], (uint32_t)(code >> 32), sym};
  }
  for (uint32_t k = tid; k < M * (kImageBytes / 16); k += kTableThreads) S.c.image[0][k] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();

  // ---- tracked state (Algorithm 1 step 7; tracked_out may be base: a thread reads only its own elements), and the bit
  // count of the thread's pieces
  uint32_t piece[M];
#pragma unroll
  for (uint32_t m = 0; m < M; ++m) {
    piece[m] = 0;
#pragma unroll
    for (uint32_t r = 0; r < kThreadSteps; ++r) {
      const uint32_t have = held(m, r);
      float x[4];
#pragma unroll
      for (uint32_t e = 0; e < 4; ++e) {
        const uint32_t key = key_of_bits(d[m][r][e]);
        if (e < have) piece[m] += S.c.len[key];
        x[e] = __fadd_rn(b[m][r][e], __uint_as_float(S.c.rep[key]));
      }
      if (tracked_out) {
        const uint32_t i = element(m, r);
        if (have == 4) {
          *reinterpret_cast<float4*>(tracked_out + i) = make_float4(x[0], x[1], x[2], x[3]);
        } else {
#pragma unroll
          for (uint32_t e = 0; e < 3; ++e)
            if (e < have) tracked_out[i + e] = x[e];
        }
      }
    }
    S.c.bits[m][warp][lane] = piece[m];
  }
  __syncthreads();

  // ---- bit position of every piece: pieces of a lane follow each other by warp, lanes follow each other; a warp per chunk
  const StreamLayout L = stream_layout(n, S.T.nsym);
  if (warp < M) {
    const uint32_t m = warp, c = chunk0 + m;
    uint32_t at[kWarps], total = 0;
#pragma unroll
    for (uint32_t w = 0; w < kWarps; ++w) {
      at[w] = total;
      total += S.c.bits[m][w][lane];
    }
    uint32_t incl = total;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, s);
      if ((int)lane >= s) incl += v;
    }
#pragma unroll
    for (uint32_t w = 0; w < kWarps; ++w) S.c.bits[m][w][lane] = incl - total + at[w];
    if (c < L.nchunks) reinterpret_cast<uint16_t*>(stream + L.lane_index_off)[c * kLanes + lane] = (uint16_t)total;
    if (lane == 31) S.chunk_bytes[m] = (uint32_t)align_up((incl + 7) / 8, kPayloadAlign);  // 0 for a chunk behind the end
  }
  __syncthreads();
  if (CLUSTER) cluster_arrive();  // the sizes are there for the others

  // ---- the codes
  auto code_piece = [&](uint32_t m, uint32_t* image) {
    const uint32_t pos = S.c.bits[m][warp][lane];
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
        if (e >= held(m, r)) continue;
        const uint32_t key = key_of_bits(d[m][r][e]), len = S.c.len[key];
        if (len > 32) {
          put((uint32_t)(S.T.code[S.T.sym_of_key[key]] >> 32), len - 32);
          put(S.c.code[key], 32);
        } else {
          put(S.c.code[key], len);
        }
      }
    if (nb > 0) atomicOr(dst, (uint32_t)(acc << (32 - nb)));
  };
#pragma unroll
  for (uint32_t m = 0; m < M; ++m)
    if (piece[m] > 0 && S.chunk_bytes[m] <= kImageBytes) code_piece(m, reinterpret_cast<uint32_t*>(S.c.image[m]));
  __syncthreads();

  // ---- where the chunks go: behind those of the CTAs before this one
  uint32_t off = 0, total = 0;
  if (CLUSTER) {
    cluster_wait();
    // one lane per chunk of the vector (at most 32), in every warp
    const uint32_t mine = lane < ctas * M ? cluster_ld(cluster_addr(&S.chunk_bytes[lane % M], lane / M)) : 0u;
    total = __reduce_add_sync(0xffffffffu, mine);
    off = __reduce_add_sync(0xffffffffu, (int)lane < (int)chunk0 ? mine : 0u);
    cluster_arrive();  // nobody leaves before all have read the sizes; waited for at the end
  } else {
#pragma unroll
    for (uint32_t m = 0; m < M; ++m) total += S.chunk_bytes[m];
  }
  unsigned long long* chunk_index = reinterpret_cast<unsigned long long*>(stream + L.chunk_index_off);
  if (rank == 0 && tid == 0) {
    chunk_index[L.nchunks] = total;
    *reinterpret_cast<unsigned long long*>(stream + 48) = L.payload_off + total;
  }
#pragma unroll
  for (uint32_t m = 0; m < M; ++m) {
    if (chunk0 + m < L.nchunks) {
      if (tid == 0) chunk_index[chunk0 + m] = off;
      uint4* payload = reinterpret_cast<uint4*>(stream + L.payload_off + off);
      const uint32_t bytes = S.chunk_bytes[m];
      if (bytes <= kImageBytes) {
        for (uint32_t k = tid; k < bytes / 16; k += kTableThreads) payload[k] = S.c.image[m][k];
      } else {
        for (uint32_t k = tid; k < bytes / 16; k += kTableThreads) payload[k] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();  // the same branch for the whole CTA
        if (piece[m] > 0) code_piece(m, reinterpret_cast<uint32_t*>(payload));
      }
      off += bytes;
    }
  }
  if (CLUSTER) cluster_wait();
  return LC_OK;
}

}  // namespace small
}  // namespace lc
