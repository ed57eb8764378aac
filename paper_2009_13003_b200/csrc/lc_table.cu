// Table pass: one CTA turns the 512 bucket statistics into the symbol table of the stream.
//
// Paper: Section 3.1.1 (priority promotion: keep the 2^x - 1 occupied buckets with the largest
// exponent, merge the rest into one bucket of value 0; representative = average of the bucket's
// minimum and maximum) and Section 3.1.2 (Huffman code over the bucket indices). Tie-breaks and the
// canonical code assignment are those of the stream format text, sections 1.2-1.4.
//
// Latency-only: O(512) work. Writes the stream header and symbol table, and the per-key encode table
// the encode pass looks codes up in.
#include "lc_table.cuh"

namespace lc {
namespace {

__global__ void __launch_bounds__(kTableThreads)
table_kernel(Control* __restrict__ ctl, uint64_t n, int nbits, uint8_t* __restrict__ stream, int wide_ok,
             int fixed, const ShardStats* __restrict__ whole, uint8_t* __restrict__ cache, int mean) {
  __shared__ TableShared T;
  begin_next();
  wait_previous();
  const uint32_t tid = threadIdx.x, key = key_of_position(tid);
  // The statistics that decide the table: this vector's own, or those of the whole vector it is a shard of. (Read together with the status word.)
  const int32_t status = *reinterpret_cast<const volatile int32_t*>(&ctl->status);
  KeyStats my;
  my.local = ctl->count[key];
  my.count = whole ? whole->count[key] : my.local;
  my.inv_min = whole ? whole->inv_min[key] : ctl->inv_min[key];
  my.max_bits = whole ? whole->max_bits[key] : ctl->max_bits[key];
  my.mant_sum = mean ? ctl->mant_sum[key] : 0ull;
  // an earlier pass of the same call has failed (lc_merge: a stream was rejected): leave no stream behind
  if (status != 0) {  // nothing in this kernel has written the word yet: the same for every thread
    clear_header(stream);
    return;
  }
  const int err = table_pass(T, my, TableArgs{n, nbits, wide_ok != 0, fixed != 0, whole != nullptr, mean != 0, cache}, stream);
  if (err) {
    clear_header(stream);
    if (tid == 0) set_status(&ctl->status, err);  // every thread has read the word: there are barriers in between
    return;
  }
  const uint32_t sym = T.sym_of_key[key];
  ctl->enc[key] = EncEntry{(uint32_t)T.code[sym], T.len[sym], (uint32_t)(T.code[sym] >> 32), sym};
  if (tid == 0) {
    ctl->ticket = 0;
    ctl->nsym = T.nsym;
    ctl->wide = T.wide;
    ctl->max_len = T.max_len;
    ctl->payload_bits = T.payload_bits;
  }
}

__device__ __forceinline__ void clear_range(uint4* p, uint64_t count, bool keep_first) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (uint64_t)gridDim.x * blockDim.x) {
    if (i == 0 && keep_first) {
      uint32_t* w = reinterpret_cast<uint32_t*>(p);
      w[1] = w[2] = w[3] = 0;
    } else {
      p[i] = make_uint4(0u, 0u, 0u, 0u);
    }
  }
}

__global__ void __launch_bounds__(256) clear_kernel(uint4* a, uint64_t a_count, uint4* b, uint64_t b_count, uint32_t keep_first) {
  wait_previous();
  begin_next();  // only now: the statistics pass reads what the launch before this one writes
  clear_range(a, a_count, keep_first != 0);
  clear_range(b, b_count, false);
}

}  // namespace

cudaError_t launch_clear(void* a, uint64_t a_bytes, void* b, uint64_t b_bytes, bool keep_first, cudaStream_t cs, bool overlap) {
  const uint64_t items = (a_bytes > b_bytes ? a_bytes : b_bytes) / 16, ctas = (items + 255) / 256;
  return launch_kernel(overlap, clear_kernel, (unsigned)(ctas < 1 ? 1 : ctas > 148 ? 148 : ctas), 256, 0, cs, static_cast<uint4*>(a),
                       a_bytes / 16, static_cast<uint4*>(b), b_bytes / 16, keep_first ? 1u : 0u);
}

cudaError_t launch_table(Control* ctl, uint64_t n, int nbits, uint8_t* stream, bool wide_ok, bool fixed,
                         const ShardStats* whole, uint8_t* cache, cudaStream_t cs, bool mean, bool overlap) {
  return launch_kernel(overlap, table_kernel, 1, kTableThreads, 0, cs, ctl, n, nbits, stream, wide_ok ? 1 : 0, fixed ? 1 : 0, whole,
                       cache, mean ? 1 : 0);
}

}  // namespace lc
