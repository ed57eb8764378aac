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
  const uint32_t tid = threadIdx.x, key = key_of_position(tid);
  // an earlier pass of the same call has failed (lc_merge: a stream was rejected): leave no stream behind
  if (ctl->status != 0) {  // nothing in this kernel has written the word yet: the same for every thread
    clear_header(stream);
    return;
  }
  // The statistics that decide the table: this vector's own, or those of the whole vector it is a shard of.
  KeyStats my;
  my.local = ctl->count[key];
  my.count = whole ? whole->count[key] : my.local;
  my.inv_min = whole ? whole->inv_min[key] : ctl->inv_min[key];
  my.max_bits = whole ? whole->max_bits[key] : ctl->max_bits[key];
  my.mant_sum = mean ? ctl->mant_sum[key] : 0ull;
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

}  // namespace

cudaError_t launch_table(Control* ctl, uint64_t n, int nbits, uint8_t* stream, bool wide_ok, bool fixed,
                         const ShardStats* whole, uint8_t* cache, cudaStream_t cs, bool mean) {
  table_kernel<<<1, kTableThreads, 0, cs>>>(ctl, n, nbits, stream, wide_ok ? 1 : 0, fixed ? 1 : 0, whole, cache,
                                            mean ? 1 : 0);
  return cudaGetLastError();
}

}  // namespace lc
