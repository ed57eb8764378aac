// The table pass as a function of one CTA of kTableThreads threads (Section 3.1.1: priority promotion and
// representatives; Section 3.1.2: Huffman code; format sections 1.2-1.8): shared by table_kernel and by the
// single-CTA kernel for small vectors.
//
// Bound: latency. Every compress call waits for this one CTA, so what counts is the length of its dependent chain: one
// thread per bucket (later per symbol), ten block barriers, and a single serial loop (the Huffman merges, one thread,
// with the fronts of both queues in registers). Ranks, tree depths (pointer jumping), codes
// (a sum over the symbols that come before) and sums are computed by all symbols at once; the stream's header and table
// leave as 16-byte stores. With those steps in one thread, 64-bit shared-memory atomics and byte stores the pass took 10.5 us
// for 8 symbols, 14 us for 16 and 28-36 us for 64; in cycles of the pass alone it now takes 6000 (3 us) for 8, 6600 for 16 and 12,000 for 64.
#pragma once
#include "lc_common.cuh"

namespace lc {

constexpr int kTableThreads = 512;

// Thread `tid` of the pass looks at one key: positions 0..507 are the candidates in priority order (exponent descending,
// + before -), then come the non-finite keys and the two keys of exponent field 0.
__device__ __forceinline__ uint32_t key_of_position(uint32_t tid) {
  if (tid < 508) return 256 * (tid & 1) + 254 - (tid >> 1);
  return tid == 508 ? 255u : tid == 509 ? 511u : tid == 510 ? 0u : 256u;
}

// The statistics of one key.
struct KeyStats {
  unsigned long long count;     // elements, of the vector that decides the table
  unsigned long long local;     // elements of the vector that is coded: the same unless it is a shard
  uint32_t inv_min, max_bits;
  unsigned long long mant_sum;  // mean representatives only
};

struct TableArgs {
  uint64_t n;
  int nbits;
  bool wide_ok;    // false: a vector with an exponent field >= 128 is rejected
  bool fixed;      // fixed-width codes
  bool shard;      // the counts decide the table, the local counts go into it
  bool mean;
  uint8_t* cache;  // nullptr, or the length cache
};

// What the pass leaves in shared memory.
struct TableShared {
  unsigned long long count[kMaxSymbols], local[kMaxSymbols], code[kMaxSymbols];  // by symbol
  unsigned long long leaf_w[kMaxSymbols + 4], node_w[kMaxSymbols + 4];           // the two queues (merge_leaves)
  unsigned long long part[4][kTableThreads / 32];
  uint32_t rep[kMaxSymbols], key[kMaxSymbols], len[kMaxSymbols];                 // by symbol
  uint32_t up[2 * kMaxSymbols];  // by tree node: depth below the node in the low half << 16 | that node
  uint32_t warps[kTableThreads / 32];  // candidates of a warp's keys in the low half, what is wrong with the keys above
  uint16_t sym_of_key[kKeys], place[kMaxSymbols];  // place: by symbol, among the leaves
  uint32_t nsym, max_len, wide;
  unsigned long long payload_bits;
};

__device__ __forceinline__ unsigned long long table_warp_sum(unsigned long long v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}
__device__ __forceinline__ unsigned long long table_part_total(const unsigned long long* part) {
  unsigned long long v = 0;
#pragma unroll
  for (int w = 0; w < kTableThreads / 32; ++w) v += part[w];
  return v;
}

// The two-queue construction over `used` leaves, ascending, by one thread: leaf_w and node_w hold the queues, all ones behind their ends; up[v]
// becomes node v's parent with a depth of one above it. W: what holds the sum of all weights.
// Bound: the dependent chain of a merge. The first four of either queue are in registers; a merge takes two of them, so that what it loads is needed
// only in the next one's second half. (With the first two in registers and 64-bit weights, a compress of
// 61,706 elements in 64 symbols took 21.0 us on the GPU instead of 18.9, one of 11.7 M in 16 symbols 48.5 instead of 47.9.)
template <class W>
__device__ __forceinline__ void merge_leaves(const W* leaf_w, W* node_w, uint32_t* up, uint32_t used) {
  W a0 = leaf_w[0], a1 = leaf_w[1], a2 = leaf_w[2], a3 = leaf_w[3], b0 = (W)~0ull, b1 = b0, b2 = b0, b3 = b0;
  uint32_t fa = 0, fb = 0;  // of a0, b0
  for (uint32_t m = 0; m + 1 < used; ++m) {
    const bool p = a0 <= b0;  // a leaf goes before an internal node of the same weight
    const W x = p ? a0 : b0, ra0 = p ? a1 : a0, ra1 = p ? a2 : a1, ra2 = p ? a3 : a2, rb0 = p ? b0 : b1, rb1 = p ? b1 : b2, rb2 = p ? b2 : b3;
    const bool q = ra0 <= rb0;
    const W sum = x + (q ? ra0 : rb0);
    const uint32_t first = p ? fa : used + fb;
    fa += p ? 1u : 0u;
    fb += p ? 0u : 1u;
    const uint32_t second = q ? fa : used + fb;
    fa += q ? 1u : 0u;
    fb += q ? 0u : 1u;
    node_w[m] = sum;
    a0 = q ? ra1 : ra0;
    a1 = q ? ra2 : ra1;
    b0 = fb == m ? sum : q ? rb0 : rb1;
    b1 = fb + 1 == m ? sum : q ? rb1 : rb2;
    a2 = leaf_w[fa + 2];
    a3 = leaf_w[fa + 3];
    b2 = node_w[fb + 2];
    b3 = node_w[fb + 3];
    up[first] = up[second] = 1u << 16 | (used + m);
  }
}

// No stream is left: its first 64 bytes (the magic among them) become zero.
__device__ __forceinline__ void clear_header(uint8_t* stream) {
  if (threadIdx.x < 4) reinterpret_cast<uint4*>(stream)[threadIdx.x] = make_uint4(0u, 0u, 0u, 0u);
}

struct NoGate {
  __device__ __forceinline__ bool operator()() const { return true; }
};

// gate(): called by all threads before the first write to the stream; false, the same for all, ends the pass with LC_ERR_ARG.
// `my`: the statistics of key_of_position(threadIdx.x). Returns 0, or the error that makes the vector unencodable, the
// same for all threads; on success the stream's header (but for its total size), table and padding are written (unless
// !write), and T is complete and visible to all threads.
template <class Gate = NoGate>
__device__ __forceinline__ int table_pass(TableShared& T, const KeyStats& my, const TableArgs& A, uint8_t* __restrict__ stream,
                                          bool write = true, Gate gate = Gate()) {
  constexpr uint32_t kAll = 0xffffffffu;
  constexpr unsigned long long kNone = ~0ull;  // weight behind the end of a queue
  const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t key = key_of_position(tid);

  // ---- non-finite deltas make the vector unencodable; exponent fields >= 128 are more than the key plane holds
  const bool cand = tid < 508 && my.count != 0;
  const uint32_t ballot = __ballot_sync(kAll, cand);
  const bool bad = (key & 255u) == 255u && my.count != 0;
  const bool big = (key & 255u) >= 128u && (my.count != 0 || my.local != 0);
  const uint32_t flags = (__any_sync(kAll, bad) ? 1u : 0u) | (__any_sync(kAll, big) ? 2u : 0u);
  if (lane == 0) T.warps[warp] = __popc(ballot) | flags << 16;
  T.sym_of_key[tid] = 0;
  T.len[tid] = 0;
  T.code[tid] = 0;
  T.node_w[tid] = kNone;
  T.leaf_w[tid] = kNone;
  if (tid < 4) T.node_w[kMaxSymbols + tid] = T.leaf_w[kMaxSymbols + tid] = kNone;
  if (tid == 0) T.max_len = 0;
  __syncthreads();

  // ---- priority promotion
  uint32_t rank = __popc(ballot & ((1u << lane) - 1)), ncand = 0, all_flags = 0;
#pragma unroll
  for (uint32_t w = 0; w < kTableThreads / 32; ++w) {
    const uint32_t v = T.warps[w];
    if (w < warp) rank += v & 0xffffu;
    ncand += v & 0xffffu;
    all_flags |= v >> 16;
  }
  if (all_flags & 1u) return LC_ERR_NONFINITE;
  const uint32_t wide = all_flags >> 1;
  // the caller has released base and cur, and the one-byte keys do not identify the buckets of this vector
  if (wide && !A.wide_ok) return LC_ERR_RANGE;
  const uint32_t keep = min((1u << A.nbits) - 1u, ncand), nsym = keep + 1;
  const bool kept = cand && rank < keep;
  if (kept) {
    const uint32_t sym = rank + 1;
    T.sym_of_key[key] = (uint16_t)sym;
    T.count[sym] = my.count;
    T.local[sym] = my.local;
    T.key[sym] = key;
    // midrange of two values with the same sign and exponent, rounded to nearest even, on mantissas.
    const uint32_t t = ((~my.inv_min) & 0x7FFFFFu) + (my.max_bits & 0x7FFFFFu);
    uint32_t mr = t >> 1;
    if ((t & 1u) && (mr & 1u)) mr += 1;
    if (A.mean) {
      // variant (format section 1.8): mean of the mantissa fields, rounded to nearest, ties to even; it cannot reach
      // 2^23 because it does not exceed the largest field
      unsigned long long q = my.mant_sum / my.count;
      const unsigned long long r = my.mant_sum - q * my.count;
      if (2 * r > my.count || (2 * r == my.count && (q & 1ull))) q += 1;
      mr = (uint32_t)q;
    }
    T.rep[sym] = (key << 23) | mr;
  }
  {
    // a vector's own counts add up to less than 2^32
    const unsigned long long kept_sum =
        A.shard ? table_warp_sum(kept ? my.count : 0ull) : __reduce_add_sync(kAll, kept ? (uint32_t)my.count : 0u);
    if (lane == 0) T.part[0][warp] = kept_sum;
    if (A.shard) {
      const unsigned long long kept_local = table_warp_sum(kept ? my.local : 0ull), whole = table_warp_sum(my.count);
      if (lane == 0) {
        T.part[1][warp] = kept_local;
        T.part[2][warp] = whole;
      }
    }
  }
  __syncthreads();

  // ---- from here on thread tid looks at symbol tid. Symbol 0 is everything that is not kept.
  const unsigned long long kept_total = table_part_total(T.part[0]);
  const unsigned long long count0 = (A.shard ? table_part_total(T.part[2]) : A.n) - kept_total;
  const unsigned long long local0 = A.n - (A.shard ? table_part_total(T.part[1]) : kept_total);
  const bool is_sym = tid < nsym;
  const unsigned long long my_count = !is_sym ? 0ull : tid == 0 ? count0 : T.count[tid];
  const unsigned long long my_local = !is_sym ? 0ull : tid == 0 ? local0 : T.local[tid];
  const bool used = my_count != 0;  // every kept symbol is
  const uint32_t nused = keep + (count0 != 0 ? 1u : 0u);
  uint32_t my_len = 0;
  bool hit = false;
  uint8_t* row = nullptr;
  if (A.fixed) {
    // fixed-width codes (format section 1.5): every symbol, used or not, takes ceil(log2 nsym) bits; its code is its id
    uint32_t width = 0;
    while ((1u << width) < nsym) width += 1;
    my_len = width;
    if (is_sym) {
      T.len[tid] = width;
      T.code[tid] = tid;
    }
    if (tid == 0) T.max_len = width;
  } else if (nused >= 2) {
    // Place among the used symbols by (count, id) ascending, which is the order of the leaves: a warp per symbol, which compares it with 32 others at
    // a time. (A thread per symbol with a loop over the others took 60 cycles for each of them, and so did the codes below: 20 M elements in 64
    // symbols 68.4 us instead of 66.8, 11.7 M in 32 49.8 instead of 48.9, in 16 47.5 instead of 47.1.) Weights of a vector's own elements fit 32 bits, those of the whole vector of a shard may not.
    uint32_t *leaf32 = reinterpret_cast<uint32_t*>(T.leaf_w), *node32 = reinterpret_cast<uint32_t*>(T.node_w);
    for (uint32_t i = warp; i < nsym; i += kTableThreads / 32) {
      const unsigned long long ci = i == 0 ? count0 : T.count[i];
      if (ci == 0) continue;
      uint32_t place = 0;
      for (uint32_t first = 0; first < nsym; first += 32) {
        const uint32_t j = first + lane;
        const unsigned long long cj = j >= nsym ? 0ull : j == 0 ? count0 : T.count[j];
        place += __popc(__ballot_sync(kAll, cj != 0 && (cj < ci || (cj == ci && j < i))));
      }
      if (lane == 0) {
        T.place[i] = (uint16_t)place;
        if (A.shard) T.leaf_w[place] = ci;
        else leaf32[place] = (uint32_t)ci;
      }
    }
    // ---- code-table caching (Section 3.2; format section 1.7): a valid row for this number of used symbols gives
    // the r-th most frequent symbol its r-th length, if the payload then stays within n * nbits bits
    row = A.cache ? A.cache + (size_t)kLengthCacheRow * (nused - 1) : nullptr;
    if (row && row[0] != 0) {  // read before anything in this kernel writes the row
      uint32_t offered = 0;
      if (used) {
        uint32_t r = 0;  // place by (count descending, id ascending)
        for (uint32_t j = 0; j < nsym; ++j) {
          const unsigned long long cj = j == 0 ? count0 : T.count[j];
          r += cj != 0 && (cj > my_count || (cj == my_count && j < tid)) ? 1u : 0u;
        }
        offered = row[r];
      }
      const unsigned long long bits = table_warp_sum(my_count * offered);
      if (lane == 0) T.part[1][warp] = bits;  // a shard takes no cache
      __syncthreads();
      hit = table_part_total(T.part[1]) <= A.n * (unsigned long long)A.nbits;
      if (hit) my_len = offered;
    }
    if (!hit) {
      // ---- Huffman lengths: two-queue construction over the leaves
      __syncthreads();
      const uint32_t root = 2 * nused - 2;
      if (tid == 0) {
        if (A.shard) merge_leaves(T.leaf_w, T.node_w, T.up, nused);
        else merge_leaves(leaf32, node32, T.up, nused);
        T.up[root] = root;
      }
      // ---- depths: every node jumps to its ancestor's ancestor until all have reached the root
      const auto above = [&](uint32_t v) {
        const uint32_t a = T.up[v], b = T.up[a & 0xffffu];
        return ((a >> 16) + (b >> 16)) << 16 | (b & 0xffffu);
      };
      if (nused <= 32) {
        // two nodes a lane in the warp that has built the tree, without block barriers (sixteen symbols: 670 cycles instead of 1140)
        if (warp == 0) {
          __syncwarp();
          for (uint32_t reach = 1; reach < nused; reach *= 2) {
            const uint32_t v0 = min(lane, root), v1 = min(lane + 32, root), x0 = above(v0), x1 = above(v1);
            __syncwarp();
            T.up[v0] = x0;
            T.up[v1] = x1;
            __syncwarp();
          }
        }
        __syncthreads();
      } else {
        __syncthreads();
        for (uint32_t reach = 1; reach < min(nused, 64u); reach *= 2) {  // no leaf is deeper than nused - 1, nor than 63
          uint32_t x[2];
#pragma unroll
          for (uint32_t h = 0; h < 2; ++h) {
            const uint32_t v = tid + h * kTableThreads;
            if (v <= root) x[h] = above(v);
          }
          __syncthreads();
#pragma unroll
          for (uint32_t h = 0; h < 2; ++h)
            if (tid + h * kTableThreads <= root) T.up[tid + h * kTableThreads] = x[h];
          __syncthreads();
        }
      }
      if (used) my_len = T.up[T.place[tid]] >> 16;
    }
    if (used) T.len[tid] = my_len;
    // ---- canonical codes: used symbols sorted by (len, id); a code is the sum of 2^-len over those before it
    __syncthreads();
    for (uint32_t i = warp; i < nsym; i += kTableThreads / 32) {
      const uint32_t li = T.len[i];
      if (li == 0) continue;
      unsigned long long before = 0;
      uint32_t r = 0;
      for (uint32_t first = 0; first < nsym; first += 32) {
        const uint32_t j = first + lane, lj = j < nsym ? T.len[j] : 0u;
        const bool precedes = lj != 0 && (lj < li || (lj == li && j < i));
        before += precedes ? 1ull << (63 - lj) : 0ull;
        r += __popc(__ballot_sync(kAll, precedes));
      }
      // codes of up to 31 bits leave the lower word empty
      before = li <= 31 ? (unsigned long long)__reduce_add_sync(kAll, (uint32_t)(before >> 32)) << 32 : table_warp_sum(before);
      if (lane == 0) {
        T.code[i] = before >> (63 - li);
        if (row && !hit) row[r] = (uint8_t)li;  // a miss stores the new lengths, ascending
      }
    }
    if (row && !hit && tid >= nused) row[tid] = 0;
    const uint32_t longest = __reduce_max_sync(kAll, my_len);
    if (lane == 0 && longest) atomicMax(&T.max_len, longest);
  }
  // ---- payload size: this vector's own elements, with the lengths just found
  {
    const unsigned long long mine = my_local * my_len;  // below 2^38
    const unsigned long long bits = (unsigned long long)__reduce_add_sync(kAll, (uint32_t)(mine >> 24)) << 24;
    const uint32_t low = __reduce_add_sync(kAll, (uint32_t)mine & 0xffffffu);
    if (lane == 0) T.part[3][warp] = bits + low;
  }
  __syncthreads();
  const unsigned long long payload_bits = table_part_total(T.part[3]);

  // ---- outputs
  if (!gate()) return LC_ERR_ARG;
  if (tid == 0) {
    T.rep[0] = 0;
    T.nsym = nsym;
    T.wide = wide;
    T.payload_bits = payload_bits;
  }
  const StreamLayout L = stream_layout(A.n, nsym);
  if (is_sym && write)
    reinterpret_cast<uint4*>(stream + L.table_off)[tid] =
        make_uint4((tid ? T.key[tid] : 0u) | my_len << 16, tid ? T.rep[tid] : 0u, (uint32_t)my_local, (uint32_t)(my_local >> 32));
  if (tid < 4 && write) {
    const uint32_t flag = (A.fixed ? 1u : 0u) | (A.shard ? 2u : 0u) | (hit ? 4u : 0u) | (A.mean ? 8u : 0u);
    // a vector without chunks leaves nothing for the encode pass to do: its stream ends here
    const unsigned long long total = L.nchunks == 0 ? L.payload_off : 0ull;
    uint4 h;
    if (tid == 0) h = make_uint4(0x3143434Cu /* "LCC1" */, 1u | (uint32_t)A.nbits << 16 | flag << 24, (uint32_t)A.n, (uint32_t)(A.n >> 32));
    else if (tid == 1) h = make_uint4(nsym, T.max_len, kChunkElems, kLanes | kGroup << 16);
    else if (tid == 2) h = make_uint4((uint32_t)L.nchunks, kPayloadAlign, (uint32_t)payload_bits, (uint32_t)(payload_bits >> 32));
    else h = make_uint4((uint32_t)total, (uint32_t)(total >> 32), (uint32_t)L.payload_off, (uint32_t)(L.payload_off >> 32));
    reinterpret_cast<uint4*>(stream)[tid] = h;
  }
  // bytes between the lane index and the payload are zero
  const uint64_t index_end = L.lane_index_off + 64 * L.nchunks;
  if (write && tid < L.payload_off - index_end) stream[index_end + tid] = 0;
  if (write && tid == 0 && L.nchunks == 0) *reinterpret_cast<unsigned long long*>(stream + L.chunk_index_off) = 0;
  __syncthreads();
  return LC_OK;
}

}  // namespace lc
