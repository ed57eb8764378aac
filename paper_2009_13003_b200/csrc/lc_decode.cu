// Recovery pass: chunk-parallel Huffman decode of up to four streams fused with the chain add.
//
// Paper: the reconstruction identity u_t = u_0 + sum of the quantized deltas (Section 3, after
// component C2) and Algorithm 1 step 7 (tracked state += quantized delta), applied k times left to
// right in fp32. Stream layout: format text sections 2-4.
//
// One warp decodes one chunk; lane t walks lane sub-stream t of every stream at once, so at step j
// the warp holds 128 consecutive elements: one coalesced 16-byte load of base and one 16-byte store of
// out per lane, with the k representatives added in registers in between.
//
//  * The chunk's payload of every stream is first copied, coalesced, into a warp-private staging
//    area in shared memory; the lanes then pull their words from there. (Reading them straight from
//    global memory makes every refill touch one cache line per lane.) A chunk that does not fit the
//    staging area takes the streams one after the other with tables of one level, and what then does not fit, or any with two levels, is
//    decoded from global memory by the same code.
//  * Codes are looked up in shared-memory tables whose entries hold the representative itself, 16 copies of each: a 64-bit
//    shared load is served half a warp at a time, so 16 lanes that read copies of their own always hit 16 different bank
//    pairs although their indices are data dependent.
//  * Most streams take a table of one level, indexed by the next 7 bits, or by the number of leading ones of the next bits and three bits
//    behind them (fill_one_level, decode_chunk_one_level); a lane keeps a bit position per stream and reads three words every eighth symbol.
//  * Streams whose codes neither index resolves (by_direct, by_ones) take two levels: the next kL1Bits bits, and for the last of those prefixes,
//    which belong to the longer codes, up to 9 more (decode_chunk_fast); a lane keeps a 64-bit buffer per stream and tops it
//    up with one predicated word load before every fourth symbol.
//    Both resolve codes of up to 15 bits; still longer ones are found by a canonical search behind a warp vote.
//
// Every read of a stream is bounds-checked against the caller's buffer size and every table is
// validated before use, so a damaged stream yields LC_ERR_FORMAT (and unspecified output), never an
// out-of-bounds access.
//
// Bound: HBM at k = 1 and 2 (8 bytes per element + the streams: 1.75 and 1.72 ms for 1.3 G elements in 5 bits); at k = 4 issue slots
// (58 % busy) and shared-memory wavefronts (62 %) side by side, 2.5 to 2.8 ms where the two levels alone took 3.0 to 3.3. A launch of 2^26 elements in
// four streams executes 49 instructions per element and warp, with the two levels 72.
#include "lc_decode_bits.cuh"

namespace lc {
namespace {

using namespace dec;

// Warps per CTA at most, and CTAs per SM that the registers must allow: with one stream 24 warps fit on an SM as two CTAs
// of 12 (80 registers); two streams fit one CTA of 20 (96 registers: 138 M elements 240 -> 220 us against 16 warps, 11.7 M
// elements 46 -> 31 us, because their 19.3 chunks per SM are then one round), and so do three (11.7 M elements 48 -> 31 us, 61,706 22 -> 17); with four
// a thread holds more state and one CTA of 16 takes the SM (18 or 20 warps of 96 registers: 134 M elements 307 us instead of 290, and
// staging areas so small that a vector of layers took 243 us instead of 155). With three streams there is a kernel for 16 warps of 128 registers too,
// for flat vectors whose areas leave no room for 20 (uniform codes of 8 bits, 134 M elements 433 -> 415 us, 0.5 M 28.7 -> 26.7) and for layers
// (62 of 11.7 M elements 48 -> 43 us, 20 of 4 M 28.7 -> 24.7).
template <int KS>
constexpr int kDecWarps = KS == 1 ? 12 : KS == 4 ? 16 : 20;
template <int KS>
constexpr int kDecCtas = KS == 1 ? 2 : 1;
constexpr int kL1Bits = 6;
constexpr int kL1Rep = 16;
// Second level: one sub-table per 6-bit prefix that belongs to longer codes, all of one depth: the next 9 bits if at most
// two prefixes need one (8 KB hold two tables of 512 entries; a Huffman code's long codes usually hang under one
// prefix), down to the next 4 bits if every prefix does (64 tables of 16 entries). Not 10 bits: two codes of 16 are 32,
// and the bit buffer is shifted once per pair, by their sum modulo 32.
constexpr int kSubBitsMax = 9;
constexpr int kSubBitsMin = 4;
constexpr int kL2Bits = kL1Bits + kSubBitsMax;     // longest code the two table levels resolve
static_assert(2 * kL2Bits < 32, "a pair of codes leaves the bit buffer with one shift of a 32-bit word");
static_assert(((1 << kL1Bits) << (kSubBitsMin + 3)) <= 8192, "at the smallest depth every prefix gets a sub-table");
// The tables of one level have 128 entries, 16 copies each. Direct: by the next 7 bits. By leading ones (see fill_one_level): windows of
// kOnesWindow bits in 16 classes by the number of their leading ones, 8 entries a class.
constexpr int kDirectBits = 7;
constexpr int kOnesWindow = 15;
constexpr uint32_t kOneLevelEntries = 128;
constexpr uint32_t kResolved = 64;  // four codes that the table resolves are shorter
static_assert(4 * kOnesWindow < kResolved && 4 * kOnesWindow <= 65 && 4 * kDirectBits < kResolved, "and lie within a window of three words");
static_assert(kOneLevelEntries == 1u << kDirectBits && kOneLevelEntries == (kOnesWindow + 1) * 8, "either index");
static_assert(2 * kOnesWindow < 32, "a pair of codes leaves a 32-bit word with one shift");
// Length field of a table entry that does not resolve its code. As a length it takes the bit count far below zero,
// which is how the hot loop notices: a step subtracts at most four of them per stream, and 1..4 times 2^29 (less a
// few real lengths) leaves the sign bit of the 32-bit count set in every case.
constexpr uint32_t kLongCode = 0x20000000u;
// distance, in steps of 512 bytes per warp, of the L2 prefetch of base: chains of two and more do not care between 4 and 12;
// a single stream of 138 M elements takes 194 us at 4, 207 at 6, 228 at 8 and 247 at 12
template <int KS>
constexpr int kPrefetchRows = KS == 1 ? 4 : 8;
// the same for decode_chunk_one_level, in rows: with one stream 1.3 G elements take 1.75 ms at 4 and 2.06 at 8, with two 1.71, 1.86 at 6 and
// 1.91 at 8; with three and four 2 to 12 make no difference
constexpr int kAskRows = 4;

// The two lookup tables of a stream are 8 KB each; the first starts on a 128-byte boundary of shared memory.
constexpr uint32_t kTableBytes = 8192;
constexpr uint32_t kTablePad = 128;  // the tables start on a 128-byte boundary (a lane's copy of an entry is chosen by OR)
static_assert((1 << kL1Bits) * kL1Rep * 8 == kTableBytes, "table sizes");

// Where device-detected errors go.
struct Status {
  int32_t* word;
  uint32_t rank;
  __device__ __forceinline__ void set(int32_t code) const { set_status_ranked(word, rank, code); }
};

struct alignas(16) StreamState {
  const uint8_t* ptr;  // the stream
  uint32_t l1_addr;    // shared address of the first level: [(1 << kL1Bits) * kL1Rep] {bit pattern of rep, code length}.
                       // The second level follows it at kTableBytes: nsub sub-tables of (1 << sub_bits) entries:
                       // {rep, length} or length kLongCode = longer code
  int32_t err;         // outcome of the validation
  unsigned long long payload_off, payload_size, chunk_index_off, lane_index_off;
  uint32_t max_len, nused, only_rep;
  uint32_t misses;      // first-level prefixes that belong to longer codes: the last ones (codes are canonical)
  uint32_t nsub;        // prefixes looked up in the second level: the most misses among the launch's streams
  uint32_t sub_bits;    // depth of the sub-tables, kSubBitsMin..kSubBitsMax: as many as 8 KB hold at that depth
  uint32_t unresolved;  // windows of 15 bits whose code the table by leading ones does not resolve
  uint32_t end31[20];   // [L], L = 1..16: end of the range that codes of at most L bits fill, left-aligned to 31 bits
  uint32_t sorted_rep[kMaxSymbols];    // representatives in canonical (len, id) order
  unsigned long long first_code[64];   // first canonical code of each length
  unsigned long long last_aligned[64]; // largest left-aligned 64-bit window whose code has at most this length
  uint32_t len_count[64];              // codes of each length
  uint32_t len_offset[64];             // index of the first of them in sorted_rep
  uint32_t len_next[64];               // index of the next of them while sorted_rep is filled
};

static_assert(sizeof(StreamState) % 16 == 0, "the staging areas behind the tables take 16-byte accesses");

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(0xffffffffu, v, d);
  return v;
}

// Parses and validates stream `s` and derives its canonical code, all in one warp: every CTA of the decode kernel runs
// this for its streams at once, a warp each, before it fills its tables. `scratch`: 5 * kMaxSymbols bytes of shared
// memory. Returns 0 or the error to report (the same for all lanes).
// Bound: latency. Two dependent reads of the stream (header, then symbol table and chunk index) and no block barrier;
// 64-bit sums go through shuffles (a 64-bit shared-memory atomic is a compare-and-swap loop) and the per-length
// quantities through one scan over the lengths instead of a serial loop of one thread. As a kernel of its own that built
// the tables once per launch this step took 12 to 20 us, ahead of a decode kernel that takes as long for a small vector.
__device__ __noinline__ int prepare_stream(StreamState& S, unsigned char* scratch, const uint8_t* __restrict__ s,
                                           uint64_t bytes, uint64_t n, uint32_t lane) {
  constexpr uint32_t kAll = 0xffffffffu;
  uint32_t* sym_rep = reinterpret_cast<uint32_t*>(scratch);
  uint8_t* sym_len = scratch + 4 * kMaxSymbols;
  if (bytes < kHeaderBytes) return LC_ERR_FORMAT;
  const uint4 hv = __ldg(reinterpret_cast<const uint4*>(s) + (lane & 3));
  // the entry of symbol `lane`, read with the header, if the buffer holds it
  uint4 entry = make_uint4(0u, 0u, 0u, 0u);
  if (kHeaderBytes + kTableEntryBytes * (lane + 1) <= bytes) entry = __ldg(reinterpret_cast<const uint4*>(s + kHeaderBytes) + lane);
  const auto u32_at = [&](int off) {
    const uint32_t v = (off & 12) == 0 ? hv.x : (off & 12) == 4 ? hv.y : (off & 12) == 8 ? hv.z : hv.w;
    return __shfl_sync(kAll, v, off >> 4);
  };
  const auto u64_at = [&](int off) { return (unsigned long long)u32_at(off + 4) << 32 | u32_at(off); };
  const uint32_t magic = u32_at(0), ver = u32_at(4), nsym = u32_at(16), max_len = u32_at(20);
  const uint32_t nbits = (ver >> 16) & 255u, flags = ver >> 24;
  const unsigned long long hdr_n = u64_at(8), payload_bits = u64_at(40), total_bytes = u64_at(48), payload_off = u64_at(56);
  const uint32_t chunk_elems = u32_at(24), lanes_group = u32_at(28), nchunks = u32_at(32), payload_align = u32_at(36);
  const bool fixed = (flags & 1u) != 0, shared_table = (flags & 2u) != 0;  // format sections 1.5 and 1.6
  if (magic != 0x3143434Cu || (ver & 0xffffu) != 1 || nbits < 1 || nbits > (uint32_t)kMaxNbits || (flags > 4 && flags != 8))
    return LC_ERR_FORMAT;  // flag bits 2 (cached lengths) and 3 (mean) go alone
  if (nsym < 1 || nsym > (1u << nbits) || max_len > 63) return LC_ERR_FORMAT;
  if (chunk_elems != kChunkElems || lanes_group != (kLanes | kGroup << 16) || payload_align != kPayloadAlign) return LC_ERR_FORMAT;
  if (hdr_n != n) return hdr_n < (1ull << 32) ? LC_ERR_MISMATCH : LC_ERR_FORMAT;
  const StreamLayout L = stream_layout(n, nsym);
  if (nchunks != L.nchunks || payload_off != L.payload_off || total_bytes > bytes || total_bytes < payload_off)
    return LC_ERR_FORMAT;
  const unsigned long long payload_size = total_bytes - payload_off;
  // first and last entry of the chunk index, read beside the symbol table
  const unsigned long long index_end =
      __ldg(reinterpret_cast<const unsigned long long*>(s + L.chunk_index_off) + ((lane & 1) ? L.nchunks : 0));

  for (uint32_t l = lane; l < 64; l += 32) S.len_count[l] = 0;
  __syncwarp();
  uint32_t fixed_width = 0;
  while ((1u << fixed_width) < nsym) fixed_width += 1;
  // ---- table entries, 32 symbols at a time
  bool bad = false;
  unsigned long long kraft = 0, count_sum = 0, bit_sum = 0;
  uint32_t nused = 0, seen_max = 0, only_rep = 0;
  for (uint32_t first = 0; first < nsym; first += 32) {
    const uint32_t sym = first + lane;
    const bool have = sym < nsym;
    uint4 e = make_uint4(0u, 0u, 0u, 0u);
    if (have) e = first == 0 ? entry : __ldg(reinterpret_cast<const uint4*>(s + kHeaderBytes) + sym);  // key:16 len:8 pad:8 | rep | count
    const uint32_t len = (e.x >> 16) & 255u;
    const unsigned long long count = ((unsigned long long)e.w << 32) | e.z;
    if (have) {
      bad |= (e.x >> 24) != 0 || len > 63;
      bad |= fixed ? (len != fixed_width) : (!shared_table && count == 0 && len != 0);
      bad |= count != 0 && len == 0 && shared_table && max_len != 0;  // a used symbol needs its code
      sym_len[sym] = (uint8_t)len;
      sym_rep[sym] = e.y;
    }
    seen_max = max(seen_max, len);
    count_sum += count;
    bit_sum += count * len;
    // the symbols that have a code
    const bool coded = have && (fixed ? (fixed_width > 0 || sym == 0) : (shared_table && max_len != 0 ? len != 0 : count != 0));
    if (coded && len > 0 && len <= 63) {
      kraft += 1ull << (63 - len);
      atomicAdd(&S.len_count[len], 1u);
    }
    nused += __popc(__ballot_sync(kAll, coded));
    // meaningful only when no symbol has a code length
    const uint32_t single = __ballot_sync(kAll, fixed ? have && sym == 0 : count != 0);
    const uint32_t rep = __shfl_sync(kAll, e.y, single ? __ffs(single) - 1 : 0);
    if (single) only_rep = rep;
  }
  bad |= index_end != ((lane & 1) ? payload_size : 0ull);
  if (__any_sync(kAll, bad)) return LC_ERR_FORMAT;
  seen_max = __reduce_max_sync(kAll, seen_max);
  if (warp_sum(count_sum) != n || warp_sum(bit_sum) != payload_bits) return LC_ERR_FORMAT;
  if (fixed) {
    if (max_len != fixed_width) return LC_ERR_FORMAT;  // every entry's length was compared with the width above
  } else {
    if (seen_max != max_len) return LC_ERR_FORMAT;
    if (nused >= 2 ? warp_sum(kraft) != (1ull << 63) : max_len != 0) return LC_ERR_FORMAT;
  }
  __syncwarp();  // len_count is complete

  // ---- canonical code: codes of length <= L fill the left-aligned range [0, sum over l <= L of count[l] << (63 - l)) of
  // 2^63, so one inclusive scan over the lengths (two per lane) gives every first code, range end and table offset
  const uint32_t l0 = 2 * lane, l1 = l0 + 1;
  const uint32_t c0 = S.len_count[l0], c1 = S.len_count[l1];  // length 0 counts nothing
  const unsigned long long r0 = (unsigned long long)c0 << (63 - l0), r1 = (unsigned long long)c1 << (63 - l1);
  unsigned long long range = r0 + r1;
  uint32_t offset = c0 + c1;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const unsigned long long rv = __shfl_up_sync(kAll, range, d);
    const uint32_t ov = __shfl_up_sync(kAll, offset, d);
    if ((int)lane >= d) range += rv, offset += ov;
  }
  const unsigned long long end1 = range, end0 = range - r1, begin0 = end0 - r0;
  S.first_code[l0] = begin0 >> (63 - l0);
  S.first_code[l1] = end0 >> (63 - l1);
  S.last_aligned[l0] = (end0 << 1) - 1;
  S.last_aligned[l1] = (end1 << 1) - 1;
  S.len_offset[l0] = S.len_next[l0] = offset - c1 - c0;
  S.len_offset[l1] = S.len_next[l1] = offset - c1;
  if (l0 <= 16) S.end31[l0] = (uint32_t)(end0 >> 32);
  if (l1 <= 16) S.end31[l1] = (uint32_t)(end1 >> 32);
  // first-level prefixes behind the codes of at most kL1Bits bits
  const uint32_t short_end = (uint32_t)(__shfl_sync(kAll, (kL1Bits & 1) ? end1 : end0, kL1Bits / 2) >> (63 - kL1Bits));
  const uint32_t misses = nused >= 2 ? (1u << kL1Bits) - min(short_end, 1u << kL1Bits) : 0u;
  if (lane == 0) {
    S.payload_off = payload_off;
    S.payload_size = payload_size;
    S.chunk_index_off = L.chunk_index_off;
    S.lane_index_off = L.lane_index_off;
    S.max_len = max_len;
    S.nused = nused;
    S.only_rep = only_rep;
    S.misses = misses;
    S.unresolved = 0;
  }
  __syncwarp();

  // ---- representatives in canonical order: a symbol's place among those of its length is by id
  if (nused >= 2) {
    for (uint32_t first = 0; first < nsym; first += 32) {
      const uint32_t sym = first + lane;
      const uint32_t len = sym < nsym ? sym_len[sym] : 0u;  // 0: a symbol without a code (unused, in a Huffman-coded stream)
      const uint32_t same = __match_any_sync(kAll, len);
      const uint32_t place = S.len_next[len] + __popc(same & ((1u << lane) - 1));
      if (len) S.sorted_rep[min(place, kMaxSymbols - 1)] = sym_rep[sym];
      __syncwarp();
      if (len && (int)lane == __ffs(same) - 1) S.len_next[len] += __popc(same);
      __syncwarp();
    }
  } else if (lane == 0) {
    S.sorted_rep[0] = only_rep;
  }
  return 0;
}

// {representative, length} of the code at the top of the 31-bit left-aligned window `v`, length 0 if no code of at most
// `width` (<= 16) bits is there.
__device__ __forceinline__ uint2 canonical_lookup(const StreamState& S, uint32_t v, uint32_t width) {
  uint32_t L = 1;
#pragma unroll
  for (int l = 1; l <= kL2Bits; ++l) L += v >= S.end31[l] ? 1u : 0u;
  if (L > width) return make_uint2(0u, 0u);
  const uint32_t r = (v >> (31 - L)) - (uint32_t)S.first_code[L];
  if (r >= S.len_count[L]) return make_uint2(0u, 0u);  // only with damaged lengths
  return make_uint2(S.sorted_rep[min(S.len_offset[L] + r, kMaxSymbols - 1)], L);
}

// Fills the two table levels of all KS streams; all threads of the CTA.
template <int KS>
__device__ __forceinline__ void fill_tables(const StreamState* S, unsigned char* tables) {
  for (uint32_t k = threadIdx.x; k < KS * (1u << kL1Bits) * (kL1Rep / 2); k += blockDim.x) {  // two copies of an entry each
    const uint32_t s = k / ((1u << kL1Bits) * (kL1Rep / 2)), pair = k % (kL1Rep / 2);
    const uint32_t idx = k / (kL1Rep / 2) % (1u << kL1Bits);
    const StreamState& T = S[s];
    uint2 ent = make_uint2(T.only_rep, 0u);
    if (T.nused >= 2) {
      if (idx >= (1u << kL1Bits) - T.nsub) continue;  // looked up in the second level
      ent = canonical_lookup(T, idx << (31 - kL1Bits), kL1Bits);
      if (ent.y == 0) ent.y = kLongCode;  // only with damaged lengths
    }
    uint4* l1 = reinterpret_cast<uint4*>(tables + s * 2 * kTableBytes);
    l1[idx * (kL1Rep / 2) + pair] = make_uint4(ent.x, ent.y, ent.x, ent.y);
  }
  for (uint32_t k = threadIdx.x; k < KS * (kTableBytes / 8); k += blockDim.x) {
    const uint32_t s = k / (kTableBytes / 8), i = k % (kTableBytes / 8);
    const StreamState& T = S[s];
    const uint32_t sub = i >> T.sub_bits, j = i & ((1u << T.sub_bits) - 1);
    uint2 ent = T.nused >= 2 ? make_uint2(0u, kLongCode) : make_uint2(T.only_rep, 0u);
    if (sub < T.nsub && T.nused >= 2) {
      const uint32_t idx = (1u << kL1Bits) - T.nsub + sub, width = kL1Bits + T.sub_bits;
      const uint2 r = canonical_lookup(T, ((idx << T.sub_bits) | j) << (31 - width), width);
      if (r.y) ent = r;
    }
    reinterpret_cast<uint2*>(tables + s * 2 * kTableBytes + kTableBytes)[i] = ent;
  }
}

// How the codes of a launch's streams are looked up, the same for all of them.
enum class Index { kDirect, kOnes, kTwoLevel };

// The tables of one level. Direct, where no code is longer than 7 bits: entry i has the code that the 7 bits i begin with.
//
// By leading ones: by the number of leading ones of the next 15
// bits and the three bits behind the zero that ends them. Codes are canonical, so a code's length grows with its leading ones, and
// wherever the lengths of neighbouring codes differ by little (a Huffman code of buckets by exponent), three bits behind the zero
// tell the code. That index comes out of a floating-point number: with the complement of the window as its value, the exponent
// counts the leading ones and the top of the mantissa holds the bits behind (lookup_ones). A lookup then has one level: no compare, no
// second address, and no uncopied entries with bank conflicts; and a table of 128 entries is filled in a fraction of the time of
// 64 + 1024. Entry i stands for the windows whose complement v (an integer from 0 to 32767) has v + 1/2 in
// [2^e (1 + q/8), 2^e (1 + (q + 1)/8)), e = i / 8 - 1, q = i % 8; where that is one code, the entry has it.
template <int KS>
__device__ __forceinline__ void fill_one_level(StreamState* S, unsigned char* tables, bool direct) {
  static_assert(kOneLevelEntries * kL1Rep * 8 == 2 * kTableBytes, "in the place of the two levels");
  const uint32_t lane = threadIdx.x & 31;
  for (uint32_t k = threadIdx.x; k < KS * kOneLevelEntries; k += blockDim.x) {  // a warp's entries are of one stream
    const uint32_t s = k / kOneLevelEntries, i = k % kOneLevelEntries;
    StreamState& T = S[s];
    uint2 ent = make_uint2(T.only_rep, 0u);
    uint32_t missed = 0;
    if (T.nused >= 2 && direct) {
      ent = canonical_lookup(T, i << (31 - kDirectBits), kDirectBits);
      if (ent.y == 0) ent.y = kLongCode;  // only with damaged lengths
    } else if (T.nused >= 2) {
      const uint32_t e = i / 8, q = i % 8;  // e: the exponent plus one
      const uint32_t least = ((8 + q) << e) >> 4, end = ((9 + q) << e) >> 4;
      const uint32_t most = end > least ? end - 1 : least;
      const uint32_t first = (0x7fffu - most) << 16, last = (0x7fffu - least) << 16 | 0xffffu;  // windows left-aligned to 31 bits
      const uint2 a = canonical_lookup(T, first, kOnesWindow), b = canonical_lookup(T, last, kOnesWindow);
      const bool one = a.y != 0 && a.y == b.y && first >> (31 - a.y) == last >> (31 - a.y);
      ent = one ? a : make_uint2(0u, kLongCode);
      // (in the lowest classes several entries stand for one window, and one of them is looked up)
      missed = one || ((2 * least + 1) << 3 >> e) != 8 + q ? 0u : most - least + 1;
    }
    missed = __reduce_add_sync(0xffffffffu, missed);
    if (lane == 0 && missed) atomicAdd(&T.unresolved, missed);
    uint4* row = reinterpret_cast<uint4*>(tables + s * 2 * kTableBytes) + i * (kL1Rep / 2);
#pragma unroll
    for (uint32_t j = 0; j < kL1Rep / 2; ++j) row[(j + lane) % (kL1Rep / 2)] = make_uint4(ent.x, ent.y, ent.x, ent.y);  // rotated: no bank conflicts
  }
}

// Direct if no stream has a code of more than 7 bits (134 M elements, four streams: fixed 4 bits 338 us, with the two levels 411; fixed 5 bits 330
// and 372; 20 codes of 4 and 5 bits 287 and 363).
template <int KS>
__device__ __forceinline__ bool by_direct(const StreamState* S) {
  bool direct = true;
#pragma unroll
  for (int s = 0; s < KS; ++s) direct = direct && (S[s].nused < 2 || S[s].max_len <= kDirectBits);
  return direct;
}
// By leading ones unless that leaves more windows of some stream unresolved than the two levels do (codes of one length
// of 8 or 9 bits, say: 200 of them would send every row the long way; with the two levels four streams of 134 M take 545 us). Where both
// resolve the codes, leading ones are the faster: 134 M elements, 5 bits, four streams 289 us and 337, three 236 and 270, two 201 and 226.
template <int KS>
__device__ __forceinline__ bool by_ones(const StreamState* S) {
  bool ones = true;
#pragma unroll
  for (int s = 0; s < KS; ++s) {
    const uint32_t two_level = 0x8000u - (S[s].end31[kL1Bits + S[s].sub_bits] >> 16);  // windows that the two levels leave
    ones = ones && (S[s].nused < 2 || S[s].unresolved <= two_level);
  }
  return ones;
}

// What by_ones would find, known before the table is filled: with more codes than the table has entries some window of a code is left, and none
// by two levels that resolve every code. (Filled all the same, for uniform codes of 8 bits: 0.5 M elements, two streams 24.6 us and 22.7 so; four of
// 5 M 47.2 and 45.9.)
template <int KS>
__device__ __forceinline__ bool too_many_codes(const StreamState* S, uint32_t sub_bits) {
  bool many = false;
#pragma unroll
  for (int s = 0; s < KS; ++s) many = many || (S[s].nused > kOneLevelEntries && S[s].max_len <= kL1Bits + sub_bits);
  return many;
}

// {representative, length} of the code at the top of `hi`, length kLongCode if the table does not resolve it. `table`: shared
// address of this lane's copy of entry 0, less kOnesBias by leading ones. There the float x is 1 + w 2^-23, w the top 15 bits of hi; the
// multiply-add makes it (32767 - w + 1/2 + a bit less than 2^-9) 2^-23: the half keeps it above zero and away from the integers, where
// rounding could matter.
constexpr uint32_t kOnesBias = (127 - 24) * 8 * kL1Rep * 8;  // exponent field of 2^-24, the smallest value there is
template <Index INDEX, int OFFSET>
__device__ __forceinline__ uint2 lookup_one_level(uint32_t hi, uint32_t table) {
  uint32_t v = hi;
  if (INDEX == Index::kOnes) {
    const uint32_t x = __funnelshift_r(hi, 0x3F800000u >> 15, 17);
    v = __float_as_uint(__fmaf_rn(__uint_as_float(x), __uint_as_float(0xBF7FFFFFu) /* -(1 - 2^-24) */, __uint_as_float(0x3F807FFFu) /* 1 + 32767 * 2^-23 */));
  }
  uint2 ent;
  asm("{\n\t"
      ".reg .u32 t, a;\n\t"
      "shr.u32 t, %2, %6;\n\t"
      "mad.lo.u32 a, t, %4, %3;\n\t"
      "ld.shared.v2.u32 {%0,%1}, [a+%5];\n\t"
      "}"
      : "=&r"(ent.x), "=&r"(ent.y)
      : "r"(v), "r"(table), "n"(kL1Rep * 8), "n"(OFFSET), "n"(INDEX == Index::kOnes ? 20 : 32 - kDirectBits));
  return ent;
}
template <Index INDEX, int KS>
__device__ __forceinline__ void lookup_all(uint2 (&e)[KS], const uint32_t (&hi)[KS], uint32_t table) {
  e[0] = lookup_one_level<INDEX, 0>(hi[0], table);
  if (KS > 1) e[1 % KS] = lookup_one_level<INDEX, 2 * kTableBytes>(hi[1 % KS], table);
  if (KS > 2) e[2 % KS] = lookup_one_level<INDEX, 4 * kTableBytes>(hi[2 % KS], table);
  if (KS > 3) e[3 % KS] = lookup_one_level<INDEX, 6 * kTableBytes>(hi[3 % KS], table);
}

// How the lanes address the tables of all streams of a launch; the same for each, so that it takes four registers.
struct Lookup {
  uint32_t l1lane;      // shared address of this lane's copy of first-level entry 0 of the first stream
  uint32_t first_long;  // first-level prefixes from this one on are looked up in the second level
  uint32_t sub_shift;   // their prefix and sub-table bits together: hi >> sub_shift
  uint32_t sub;         // shared address of the second level less what first_long adds to an index (wraps around)
};

// Table lookup of the code at the top of `hi`: {representative, length}, length kLongCode if the tables do not resolve
// it. Codes are canonical, so the prefixes of longer codes are the last ones: a compare tells which level a lane reads, and
// one load serves both. (With the second level's address in the first-level entry, its load waited for the first one in
// nearly every warp. 1.3 G elements and four streams: 3.40 -> 3.31 ms, one chunk and one stream 19.4 -> 17.3 us.)
// Written in PTX so that index scaling and base addition stay multiply-adds (they then run beside the
// shifts and compares instead of competing with them for the integer pipe).
template <int OFFSET>
__device__ __forceinline__ uint2 lookup_code(uint32_t hi, const Lookup& T) {
  uint2 ent;
  asm("{\n\t"
      ".reg .u32 t, a;\n\t"
      ".reg .pred q;\n\t"
      "shr.u32 t, %2, %7;\n\t"
      "setp.ge.u32 q, t, %4;\n\t"
      "mad.lo.u32 a, t, %8, %3;\n\t"
      "@q shr.u32 t, %2, %5;\n\t"
      "@q mad.lo.u32 a, t, 8, %6;\n\t"
      "ld.shared.v2.u32 {%0,%1}, [a+%9];\n\t"
      "}"
      : "=&r"(ent.x), "=&r"(ent.y)
      : "r"(hi), "r"(T.l1lane), "r"(T.first_long), "r"(T.sub_shift), "r"(T.sub), "n"(32 - kL1Bits), "n"(kL1Rep * 8), "n"(OFFSET));
  return ent;
}

// Code the tables did not resolve: canonical search on a 64-bit window read from the chunk, then re-seat
// the lane's bit buffer behind the code. Returns the representative.
template <bool STAGED>
__device__ __forceinline__ uint32_t long_code(LaneBits<STAGED>& B, const StreamState& S, const Source& W,
                                              Status status) {
  const uint32_t pos = B.bitpos(W);
  const uint32_t idx = pos >> 5, sh = pos & 31;
  const uint32_t w0 = B.word(W, idx), w1 = B.word(W, idx + 1), w2 = B.word(W, idx + 2);
  const unsigned long long window =
      ((unsigned long long)__funnelshift_l(w1, w0, sh) << 32) | __funnelshift_l(w2, w1, sh);
  // the first level resolves shorter codes, and so does the prefix's sub-table
  uint32_t L = kL1Bits + 1 + (S.nsub ? S.sub_bits : 0u);
  while (L < S.max_len && (S.len_count[L] == 0 || window > S.last_aligned[L])) L += 1;
  const unsigned long long code = window >> (64 - L);
  uint32_t rep = 0;
  if (L <= S.max_len && code >= S.first_code[L] && code - S.first_code[L] < S.len_count[L]) {
    rep = S.sorted_rep[S.len_offset[L] + (uint32_t)(code - S.first_code[L])];
  } else {
    status.set(LC_ERR_FORMAT);  // no code matches: damaged payload
  }
  B.seek(W, pos + L);
  return rep;
}

// Full chunk: the hot loop. Per step a lane decodes 4 elements x KS streams; the KS streams are independent
// dependency chains and are written interleaved.
//
// The loop body is straight-line code. A lane tops its bit buffers up once per step and then decodes its four
// codes per stream from the upper word alone, two at a time (the second lookup takes the first code's length,
// the buffer is shifted once per pair, by 30 bits at most). Two things can go wrong for a lane in a step, both rare: a code longer
// than the tables resolve, and four codes that take more bits than the buffer held (32 are guaranteed, four
// table-resolved codes can take 60). Both show as a negative bit count at the end of the step: the marker of an
// unresolved code is a huge length, and a lookup on too few valid bits always overdraws, because no code is a
// prefix of another. One warp vote per step finds them, and the flagged lanes decode the step again from where it
// started, one code at a time with a top-up before each (a top-up makes 32 bits valid, a table-resolved code
// takes at most 15). Whatever the quick pass did to their buffers in
// between stays inside the staged chunk (a top-up moves one word per step) and is discarded.
// PARTIAL: the vector's last chunk. Only the steps that hold elements are visited, and of a step's four slots only
// the first `have` are loaded, checked and stored. (The lane's codes end with its last element, so what the quick pass
// decodes behind it are codes of the next lane or the chunk's zero slack; nothing is reported for them.)
template <bool PARTIAL>
__device__ __forceinline__ float4 load_row(const float* p, int have) {
  if (!PARTIAL || have >= 4) return ldg_stream_v4(p);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (have > 0) v.x = p[0];
  if (have > 1) v.y = p[1];
  if (have > 2) v.z = p[2];
  return v;
}

template <bool PARTIAL>
__device__ __forceinline__ void store_row(float* p, float x0, float x1, float x2, float x3, int have) {
  if (!PARTIAL || have >= 4) {
    *reinterpret_cast<float4*>(p) = make_float4(x0, x1, x2, x3);
  } else {
    if (have > 0) p[0] = x0;
    if (have > 1) p[1] = x1;
    if (have > 2) p[2] = x2;
  }
}

template <int KS, bool STAGED, bool PARTIAL>
__device__ __forceinline__ void decode_chunk_fast(const StreamState* S, const Source* W, const uint32_t* start,
                                                    const float* base, float* out, uint64_t c, uint64_t n, uint32_t lane,
                                                    const float* next_rows, Status status) {
  LaneBits<STAGED> bits[KS];
  const uint32_t elems = PARTIAL ? (uint32_t)min(n - c * kChunkElems, (uint64_t)kChunkElems) : kChunkElems;
  const int rem = PARTIAL ? (int)elems - 4 * (int)lane : 0;  // elements from this lane's first slot on
  const uint32_t steps = PARTIAL ? (elems + 127) / 128 : kSteps;
  // the streams' tables follow each other at 2 * kTableBytes: one base address, the rest as immediate offsets
  const Lookup T{S[0].l1_addr | ((lane & (kL1Rep - 1)) * 8u), (1u << kL1Bits) - S[0].nsub, 32 - kL1Bits - S[0].sub_bits,
                 S[0].l1_addr + kTableBytes - ((((1u << kL1Bits) - S[0].nsub) << S[0].sub_bits) << 3)};
#pragma unroll
  for (int s = 0; s < KS; ++s) bits[s].seek(W[s], start[s]);
  const uint64_t e0 = c * kChunkElems + 4 * lane;
  float4 b = load_row<PARTIAL>(base + e0, rem);
  // With one stream a step is short, and one row of base in registers ahead of its use leaves too few bytes in flight
  // for the L2's latency (0.80 of the copy rate); a second row brings that to 0.92. With two or more streams the
  // second row makes the kernel slower (measured for 2, 3 and 4 streams), so they keep one.
  float4 b2 = b;
  if (KS == 1) b2 = load_row<PARTIAL>(base + e0 + 128, rem - 128);
  // Rows of base are asked into the L2 kPrefetchRows steps before they are loaded: a warp has one row in
  // registers ahead of its use, which alone leaves far too few bytes in flight per SM for the DRAM latency.
  // Behind this chunk's last row the requests go on with the first rows of the chunk this warp decodes next
  // (`next_rows`: this lane's part of that chunk's first row, or of this chunk's first row if there is none).
  const float* pf = base + e0 + 128 * kPrefetchRows<KS>;
#pragma unroll 1
  for (uint32_t j = 0; j < steps; ++j) {
    const uint64_t i = e0 + 128ull * j;
    const int have = rem - 128 * (int)j;  // PARTIAL: slots of this step that hold elements, if fewer than four
    float x[4] = {b.x, b.y, b.z, b.w};
    // the 16 bytes of base of a later step, requested one step ahead (one stream: two steps); the last steps
    // re-read their own
    if (KS == 1) {
      b = b2;
      b2 = PARTIAL ? load_row<PARTIAL>(base + i + 256, have - 256) : ldg_stream_v4(base + i + (j + 2 < kSteps ? 256 : 0));
    } else {
      b = PARTIAL ? load_row<PARTIAL>(base + i + 128, have - 128) : ldg_stream_v4(base + i + (j + 1 < kSteps ? 128 : 0));
    }
    if (!PARTIAL) asm volatile("prefetch.global.L2 [%0];" ::"l"(pf));
    pf = (j == kSteps - kPrefetchRows<KS> - 1) ? next_rows : pf + 128;
    int cnt0[KS];
    uint32_t flags = 0;
#pragma unroll
    for (int s = 0; s < KS; ++s) {
      bits[s].refill(W[s]);
      cnt0[s] = bits[s].cnt;  // where the step starts, for the careful pass (`next` does not move within a step)
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint2 ea[KS], eb[KS];
      uint32_t h1[KS];
      ea[0] = lookup_code<0>(bits[0].hi, T);
      if (KS > 1) ea[1 % KS] = lookup_code<2 * kTableBytes>(bits[1 % KS].hi, T);
      if (KS > 2) ea[2 % KS] = lookup_code<4 * kTableBytes>(bits[2 % KS].hi, T);
      if (KS > 3) ea[3 % KS] = lookup_code<6 * kTableBytes>(bits[3 % KS].hi, T);
#pragma unroll
      for (int s = 0; s < KS; ++s) h1[s] = __funnelshift_l(0u, bits[s].hi, ea[s].y);  // hi << length (mod 32)
      eb[0] = lookup_code<0>(h1[0], T);
      if (KS > 1) eb[1 % KS] = lookup_code<2 * kTableBytes>(h1[1 % KS], T);
      if (KS > 2) eb[2 % KS] = lookup_code<4 * kTableBytes>(h1[2 % KS], T);
      if (KS > 3) eb[3 % KS] = lookup_code<6 * kTableBytes>(h1[3 % KS], T);
#pragma unroll
      for (int s = 0; s < KS; ++s) {
        x[2 * h] = __fadd_rn(x[2 * h], __uint_as_float(ea[s].x));
        x[2 * h + 1] = __fadd_rn(x[2 * h + 1], __uint_as_float(eb[s].x));
        const uint32_t len = ea[s].y + eb[s].y;
        bits[s].hi = __funnelshift_l(bits[s].lo, bits[s].hi, len);
        bits[s].lo = __funnelshift_l(0u, bits[s].lo, len);
        bits[s].cnt = (int)((uint32_t)bits[s].cnt - len);
      }
    }
#pragma unroll
    for (int s = 0; s < KS; ++s) flags |= (uint32_t)bits[s].cnt;
    if (PARTIAL && have <= 0) flags = 0;
    if (__builtin_expect(__any_sync(0xffffffffu, (int)flags < 0), 0)) {
      if ((int)flags < 0) {
        const float4 b0 = load_row<PARTIAL>(base + i, have);
        x[0] = b0.x; x[1] = b0.y; x[2] = b0.z; x[3] = b0.w;
#pragma unroll
        for (int s = 0; s < KS; ++s) {
          bits[s].cnt = cnt0[s];
          bits[s].seek(W[s], bits[s].bitpos(W[s]));
        }
        // one element per trip; x is rotated so that the loop needs no indexed register
#pragma unroll 1
        for (int e = 0; e < 4; ++e) {
          float v = x[0];
          if (PARTIAL && e >= have) {
            x[0] = x[1]; x[1] = x[2]; x[2] = x[3];
            continue;
          }
          uint2 ent[KS];
#pragma unroll
          for (int s = 0; s < KS; ++s) bits[s].refill(W[s]);
          ent[0] = lookup_code<0>(bits[0].hi, T);
          if (KS > 1) ent[1 % KS] = lookup_code<2 * kTableBytes>(bits[1 % KS].hi, T);
          if (KS > 2) ent[2 % KS] = lookup_code<4 * kTableBytes>(bits[2 % KS].hi, T);
          if (KS > 3) ent[3 % KS] = lookup_code<6 * kTableBytes>(bits[3 % KS].hi, T);
#pragma unroll
          for (int s = 0; s < KS; ++s) {
            if (ent[s].y > 63u) ent[s] = make_uint2(long_code<STAGED>(bits[s], S[s], W[s], status), 0u);  // consumed
            v = __fadd_rn(v, __uint_as_float(ent[s].x));
            bits[s].consume(ent[s].y);
          }
          x[0] = x[1]; x[1] = x[2]; x[2] = x[3]; x[3] = v;
        }
      }
    }
    store_row<PARTIAL>(out + i, x[0], x[1], x[2], x[3], have);
  }
}
static_assert(kL1Rep * 8 == 128, "first-level entries of one index span 128 bytes");

// Code that a table of one level did not resolve, at bit `pos` of its chunk: canonical search. Returns {representative, length}.
// Where nothing but the codes beyond kOnesWindow bits is left to it, the search begins there: an iteration waits for shared memory, and the first 15 of
// them took most of the row's time (134 M elements in 6 bits, student deltas, four streams, 5 % of a warp's rows with such a code: 346 -> 306 us).
template <bool STAGED>
__device__ __forceinline__ uint2 long_code_at(const StreamState& S, const Words<STAGED>& words, uint32_t pos, Status status) {
  const uint32_t at = words.at(pos), w0 = words.load(at, 0), w1 = words.load(at, 1), w2 = words.load(at, 2);
  const unsigned long long window = ((unsigned long long)__funnelshift_l(w1, w0, pos) << 32) | __funnelshift_l(w2, w1, pos);
  uint32_t L = S.unresolved <= 0x8000u - (S.end31[kOnesWindow] >> 16) ? kOnesWindow + 1 : 1;
  while (L < S.max_len && (S.len_count[L] == 0 || window > S.last_aligned[L])) L += 1;
  const unsigned long long code = window >> (64 - L);
  if (L <= S.max_len && code >= S.first_code[L] && code - S.first_code[L] < S.len_count[L])
    return make_uint2(S.sorted_rep[S.len_offset[L] + (uint32_t)(code - S.first_code[L])], L);
  status.set(LC_ERR_FORMAT);  // no code matches: damaged payload
  return make_uint2(0u, L);
}

// A chunk through the tables of one level. A step is two rows (or one: see R): a lane decodes eight elements x KS
// streams from a window of three words per stream, read anew in every step, so that all it keeps of a stream from step to step is a bit position. (A 64-bit buffer
// that is topped up takes four registers and, with its bookkeeping, 45 instructions for four codes where this form takes 36.)
// The window has at least 65 bits behind the position; four codes of a row that are together shorter than 32 bits leave
// it with one funnel shift, and at least 34 bits are then left for the second row. One vote per row finds the lanes with a longer row or a
// code that the table does not resolve (whose marker is a huge length). Rows of 32 to 60 bits were looked up from valid bits, and stand, if the
// window had as many: always in the first of two rows, behind which the window is read anew; in the second, and with one stream, 64 less
// the position within its word are certain. (A lookup on too few bits always overdraws, because no code is a prefix of another.)
// Only what is left goes through the row again, one code at a time. They are rare on the whole (four streams in 6 bits: 0.3 to 1.4 % of a
// warp's rows), but a chunk of rare exponents has nothing else, and a launch of one round waits for it. With all of them one code at a time, four
// streams of 11.7 M elements in 62 scales took 57 us instead of 41; two of 134 M, 10 % in rare exponents, 311 instead of 226.
// Every code has at most 63 bits, so a lane of a damaged stream reads at most 1013 bytes beyond its chunk (kOverrunBytes).
// PARTIAL: the vector's last chunk, or any chunk larger than the staging area: of each row only the slots that exist are read and written. (A
// lane's codes end with its last element; nothing is reported for what it decodes behind it.)
// next_chunk: floats from this chunk to the one the warp takes next, whose first rows are asked into the L2 behind this one's last; 0 if there is none.
// R: rows a step. Two, but one with a single stream in a launch of many rounds: that is bound by HBM, and it is the steady trickle of single rows, each waited
// for a step before its use, that reaches the copy rate (two_rows).
template <int KS, int R, Index INDEX, bool STAGED, bool PARTIAL>
__device__ __forceinline__ void decode_chunk_one_level(const StreamState* S, const Source* W, uint32_t (&pos)[KS], const float* base,
                                                  float* out, uint32_t c, uint64_t n, uint32_t lane, uint64_t next_chunk,
                                                  Status status) {
  const uint32_t elems = PARTIAL ? (uint32_t)min(n - (uint64_t)c * kChunkElems, (uint64_t)kChunkElems) : kChunkElems;
  int have = (int)elems - 4 * (int)lane;  // PARTIAL: elements from this lane's first slot of the next row on
  const uint32_t steps = PARTIAL ? (elems + 128 * R - 1) / (128 * R) : kSteps / R;
  const uint32_t table = (S[0].l1_addr | ((lane & (kL1Rep - 1)) * 8u)) - (INDEX == Index::kOnes ? kOnesBias : 0u);
  const float* bp = base + (uint64_t)c * kChunkElems + 4 * lane;
  float* op = out + (uint64_t)c * kChunkElems + 4 * lane;
  float4 b[2];  // the next two rows
  b[0] = load_row<PARTIAL>(bp, have);
  b[1] = load_row<PARTIAL>(bp + 128, have - 128);
#pragma unroll 1
  for (uint32_t j = 0; j < steps; ++j) {
    // rows are asked into the L2 kAskRows ahead of the one that is about to be decoded; behind the last row the next chunk's, or again
    // this step's
    const int64_t on = j < steps - kAskRows / R ? 0 : next_chunk ? (int64_t)next_chunk - (int64_t)kChunkElems : -128 * kAskRows;
    uint32_t hi[KS], mid[KS], lo[KS];
    bool reloaded = false;  // the second row's window, anew behind the first row: 64 bits of it are valid
#pragma unroll
    for (int s = 0; s < KS; ++s) {
      const Words<STAGED> words(W[s]);
      const uint32_t at = words.at(pos[s]);
      const uint32_t w0 = words.load(at, 0), w1 = words.load(at, 1), w2 = R > 1 ? words.load(at, 2) : 0u;
      hi[s] = __funnelshift_l(w1, w0, pos[s]);
      mid[s] = __funnelshift_l(w2, w1, pos[s]);
      lo[s] = __funnelshift_l(0u, w2, pos[s]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float4 x = b[r];
      if (R == 1) b[0] = b[1];
      if (j + 2 / R < steps) b[R == 1 ? 1 : r] = load_row<PARTIAL>(bp + 256, have - 256);
      if (!PARTIAL) asm volatile("prefetch.global.L2 [%0];" ::"l"(bp + on + 128 * kAskRows));
      uint2 e[KS];
      uint32_t h[KS], len[KS], flags = 0;
      lookup_all<INDEX>(e, hi, table);
#pragma unroll
      for (int s = 0; s < KS; ++s) {
        x.x = __fadd_rn(x.x, __uint_as_float(e[s].x));
        len[s] = e[s].y;
        h[s] = __funnelshift_l(0u, hi[s], e[s].y);  // hi << length (mod 32)
      }
      lookup_all<INDEX>(e, h, table);
#pragma unroll
      for (int s = 0; s < KS; ++s) {
        x.y = __fadd_rn(x.y, __uint_as_float(e[s].x));
        len[s] += e[s].y;
        h[s] = __funnelshift_l(mid[s], hi[s], len[s]);
      }
      lookup_all<INDEX>(e, h, table);
#pragma unroll
      for (int s = 0; s < KS; ++s) {
        x.z = __fadd_rn(x.z, __uint_as_float(e[s].x));
        len[s] += e[s].y;
        h[s] = __funnelshift_l(0u, h[s], e[s].y);
      }
      lookup_all<INDEX>(e, h, table);
#pragma unroll
      for (int s = 0; s < KS; ++s) {
        x.w = __fadd_rn(x.w, __uint_as_float(e[s].x));
        len[s] += e[s].y;
        flags |= len[s];
      }
      if (PARTIAL && have <= 0) flags = 0;
      const bool wide = flags >= 32u;
      if (r + 1 < R) {
#pragma unroll
        for (int s = 0; s < KS; ++s) {
          hi[s] = __funnelshift_l(mid[s], hi[s], len[s]);
          mid[s] = __funnelshift_l(lo[s], mid[s], len[s]);
        }
      }
      if (__builtin_expect(__any_sync(0xffffffffu, wide), 0)) {
        if (wide) {
          bool stands = flags < kResolved;
          if (R == 1 || r == 1) {  // (the first of two rows has bits enough)
#pragma unroll
            for (int s = 0; s < KS; ++s) stands = stands && (reloaded || len[s] <= 64 - (pos[s] & 31));
          }
          if (!stands) {
            x = load_row<PARTIAL>(bp, have);
            // one element per trip; x is rotated so that the loop needs no indexed register
#pragma unroll 1
            for (int i = 0; i < 4; ++i) {
              float v = x.x;
              if (!PARTIAL || i < have) {
                uint2 ent[KS];
#pragma unroll
                for (int s = 0; s < KS; ++s) {
                  const Words<STAGED> words(W[s]);
                  const uint32_t at = words.at(pos[s]);
                  h[s] = __funnelshift_l(words.load(at, 1), words.load(at, 0), pos[s]);
                }
                lookup_all<INDEX>(ent, h, table);
#pragma unroll
                for (int s = 0; s < KS; ++s) {
                  if (ent[s].y > 63u) ent[s] = long_code_at<STAGED>(S[s], Words<STAGED>(W[s]), pos[s], status);
                  v = __fadd_rn(v, __uint_as_float(ent[s].x));
                  pos[s] += ent[s].y;
                }
              }
              x.x = x.y, x.y = x.z, x.z = x.w, x.w = v;
            }
#pragma unroll
            for (int s = 0; s < KS; ++s) len[s] = 0;
          }
          if (r + 1 < R) {  // the next row's window
#pragma unroll
            for (int s = 0; s < KS; ++s) {
              const Words<STAGED> words(W[s]);
              const uint32_t next = pos[s] + len[s], at = words.at(next), w1 = words.load(at, 1);
              hi[s] = __funnelshift_l(w1, words.load(at, 0), next);
              mid[s] = __funnelshift_l(words.load(at, 2), w1, next);
            }
            reloaded = true;
          }
        }
      }
#pragma unroll
      for (int s = 0; s < KS; ++s) pos[s] += len[s];
      store_row<PARTIAL>(op, x.x, x.y, x.z, x.w, have);
      bp += 128;
      op += 128;
      if (PARTIAL) have -= 128;
    }
  }
}

// Chunk `c` of every stream: where its payload is and the lanes' bit counts. An entry that is not a valid range of the
// payload is reported and taken as empty. The payloads are copied one behind the other into the warp's staging area of
// KS * stage_bytes; returns whether they fit.
// start: the lanes' first bits; ONE_LEVEL: as decode_chunk_one_level counts them, in shared memory if the payloads fit.
//
// ONE_LEVEL: the lanes of decode_chunk_one_level read three words a step, wherever each of them is. Lanes are as many words apart as
// a lane's codes take, give or take a few, and if that is near a multiple of 8 words, they meet in a few banks: codes of 4.05 bits on
// average had 4.9 wavefronts a load instead of 2.1. Such a chunk is copied with 16 bytes of space before every fourth lane (the unit on a
// boundary twice), which makes it 2.9 to 3.4. Not always: the copy then waits for the lane starts, and the space brings lanes together that
// are well apart without it. So a chunk has space from 19 bytes below a multiple of 1024 to 38 above (0.15 and 0.3 words a lane). 134 M elements,
// four streams: chunks about 30 above, log-normal deltas, 323 us with space and 339 without; but 48 above 363 and 287, 32 below (5.9 bits) 382 and
// 353, 74 below 294 and 276.
constexpr uint32_t kSpaceUnit = 16, kSpaceBelow = 19, kSpaceAbove = 38;
constexpr uint32_t kSpaceBytes = 7 * kSpaceUnit;
__host__ __device__ constexpr bool spaced_chunk(uint64_t bytes) { return ((bytes + kSpaceBelow) & 1023u) <= kSpaceBelow + kSpaceAbove; }

template <int KS, bool ONE_LEVEL>
__device__ __forceinline__ bool stage_chunk(const StreamState* S, uint32_t c, uint32_t lane, unsigned char* stage0,
                                            uint32_t stage_bytes, Source* W, uint32_t (&start)[KS], Status status) {
  constexpr uint32_t kUnit = kSpaceUnit;
  uint32_t bytes[KS], filled = 0;
  unsigned long long off0[KS], off1[KS];
  // all index loads of all streams first, so that their latencies overlap
#pragma unroll
  for (int s = 0; s < KS; ++s) {
    const uint8_t* sp = S[s].ptr;
    const unsigned long long* ci = reinterpret_cast<const unsigned long long*>(sp + S[s].chunk_index_off);
    off0[s] = __ldg(ci + c);
    off1[s] = __ldg(ci + c + 1);
    const uint16_t* li = reinterpret_cast<const uint16_t*>(sp + S[s].lane_index_off);
    start[s] = __ldg(li + (uint64_t)c * kLanes + lane);
  }
  const auto spaced = [](uint32_t bytes) { return ONE_LEVEL && spaced_chunk(bytes); };
  // the asynchronous copies of the payloads into the staging areas
#pragma unroll
  for (int s = 0; s < KS; ++s) {
    if (off0[s] > off1[s] || off1[s] > S[s].payload_size || (off0[s] & 15) || (off1[s] & 15)) {
      status.set(LC_ERR_FORMAT);
      off0[s] = off1[s] = 0;
    }
    bytes[s] = (uint32_t)min(off1[s] - off0[s], (unsigned long long)kChunkElems * 8);
    const uint8_t* g = S[s].ptr + S[s].payload_off + off0[s];
    W[s].g = reinterpret_cast<const uint32_t*>(g);
    W[s].nw = bytes[s] >> 2;
    W[s].sbase = smem_addr(stage0) + filled;
    W[s].slim = W[s].sbase + bytes[s] + 12;
    filled += bytes[s] + (spaced(bytes[s]) ? kSpaceBytes : 16);  // 16 bytes of zero slack after the chunk must fit too
    if (filled <= KS * stage_bytes && !spaced(bytes[s])) {
      for (uint32_t k = lane * 16; k < bytes[s]; k += 32 * 16) cp_async_16(W[s].sbase + k, g + k);
      if (lane == 0) asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" ::"r"(W[s].sbase + bytes[s]), "r"(0) : "memory");
    }
  }
  const bool fits = filled <= KS * stage_bytes;
  // lane start offsets (exclusive scan of the lane bit counts) while the copies are in flight
#pragma unroll
  for (int s = 0; s < KS; ++s) {
    const uint32_t lane_bits = start[s];
    uint32_t incl = lane_bits;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, d);
      if ((int)lane >= d) incl += v;
    }
    start[s] = min(incl - lane_bits, bytes[s] * 8u);
    if (spaced(bytes[s]) && fits) {
      // four lanes copy the units that their codes lie in
      const uint32_t group = lane >> 2, units = bytes[s] / kUnit;
      const uint32_t first = __shfl_sync(0xffffffffu, start[s], lane & 28u) >> 7;
      const uint32_t behind = __shfl_sync(0xffffffffu, start[s], (lane & 28u) + 4) >> 7;
      const uint32_t end = group == 7 ? units : min(behind + 1, units);
      const uint8_t* g = reinterpret_cast<const uint8_t*>(W[s].g);
      for (uint32_t u = first + (lane & 3u); u < end; u += 4) cp_async_16(W[s].sbase + (u + group) * kUnit, g + u * kUnit);
      start[s] += group * kUnit * 8;
    }
    if (ONE_LEVEL && fits) start[s] += W[s].sbase * 8;
  }
  cp_async_commit();
  cp_async_wait_all();
  __syncwarp();
  return fits;
}

// A chunk that is partial (the vector's last) or larger than the staging area, out of line: it must not weigh on the registers of
// the main loop. On vectors of a few thousand chunks the whole launch waits for the warp that has it, so it runs the same
// straight-line steps as the others (one code at a time the last chunk took 15 us with one stream and 60 us with four). If the
// area does not hold all streams' payloads, they take it one after the other, each over what the one before has written.
// (All from global memory at once instead, without a copy: 134 M elements with 10 % in rare exponents, four streams, 916 us and 683; only the streams
// that do not fit 1109.) The masked rows ask nothing into the L2, so a whole chunk's are asked for here at once: 637.
template <int KS, Index INDEX>
__device__ __noinline__ void decode_rare_chunk(const StreamState* S, const float* base, float* out, uint32_t c, uint64_t n,
                                               uint32_t lane, unsigned char* stage0, uint32_t stage_bytes, Status status) {
  if (lane == 0 && ((uint64_t)c + 1) * kChunkElems <= n)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(base + (uint64_t)c * kChunkElems), "r"(4 * kChunkElems) : "memory");
  {
    Source W[KS];
    uint32_t pos[KS];
    __syncwarp();  // the previous chunk's reads of the staging area are done
    if (stage_chunk<KS, true>(S, c, lane, stage0, stage_bytes, W, pos, status)) {
      decode_chunk_one_level<KS, 2, INDEX, true, true>(S, W, pos, base, out, c, n, lane, 0, status);
      return;
    }
  }
#pragma unroll 1
  for (int s = 0; s < KS; ++s) {
    Source W[1];
    uint32_t pos[1];
    __syncwarp();
    if (stage_chunk<1, true>(S + s, c, lane, stage0, KS * stage_bytes, W, pos, status))
      decode_chunk_one_level<1, 2, INDEX, true, true>(S + s, W, pos, s ? out : base, out, c, n, lane, 0, status);
    else
      decode_chunk_one_level<1, 2, INDEX, false, true>(S + s, W, pos, s ? out : base, out, c, n, lane, 0, status);
  }
}

// Any chunk through the two-level tables, likewise out of line.
template <int KS>
__device__ __noinline__ void decode_chunk_two_level(const StreamState* S, const float* base, float* out, uint32_t c, uint64_t n,
                                                    uint32_t lane, unsigned char* stage0, uint32_t stage_bytes, const float* next_rows,
                                                    Status status) {
  Source W[KS];
  uint32_t start[KS];
  __syncwarp();
  if (!stage_chunk<KS, false>(S, c, lane, stage0, stage_bytes, W, start, status))
    decode_chunk_fast<KS, false, true>(S, W, start, base, out, c, n, lane, base, status);
  else if (((uint64_t)c + 1) * kChunkElems <= n)
    decode_chunk_fast<KS, true, false>(S, W, start, base, out, c, n, lane, next_rows, status);
  else
    decode_chunk_fast<KS, true, true>(S, W, start, base, out, c, n, lane, base, status);
}

// This warp's chunks, from c on, through the tables of one level.
template <int KS, int R, Index INDEX>
__device__ __forceinline__ void decode_chunks(const StreamState* S, const float* base, float* out, uint32_t c, uint32_t nwarps,
                                              uint32_t whole_end, uint32_t chunk_end, uint64_t n, uint32_t lane, unsigned char* stage0,
                                              uint32_t stage_bytes, Status status) {
  for (; c < whole_end; c += nwarps) {
    Source W[KS];
    uint32_t pos[KS];
    __syncwarp();  // the previous chunk's reads of the staging area are done
    if (stage_chunk<KS, true>(S, c, lane, stage0, stage_bytes, W, pos, status))
      decode_chunk_one_level<KS, R, INDEX, true, false>(S, W, pos, base, out, c, n, lane, c + nwarps < whole_end ? (uint64_t)nwarps * kChunkElems : 0, status);
    else
      decode_rare_chunk<KS, INDEX>(S, base, out, c, n, lane, stage0, stage_bytes, status);
  }
  if (c < chunk_end) decode_rare_chunk<KS, INDEX>(S, base, out, c, n, lane, stage0, stage_bytes, status);
}

// Asks a chunk's first rows into the L2.
__device__ __forceinline__ void prefetch_rows(const float* first, uint32_t lane) {
  if (lane == 0) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(first), "r"(4096u) : "memory");
}

// Chunks [chunk_begin, chunk_end) of one vector, by `ctas` CTAs of which this is number `cta`.
// stage_bytes: bytes of staging area per warp and stream (a multiple of 16, at least 32).
// CLEAR: the CTAs are one cluster, whose first clears the status word; none writes to it before.
template <int KS, int R, bool CLEAR>
__device__ __forceinline__ void decode_vector(const float* base, const DecodeStreams& streams, uint64_t n, float* out,
                                              Status status, uint32_t stage_bytes, uint32_t chunk_begin,
                                              uint32_t chunk_end, uint32_t cta, uint32_t ctas) {
  // dynamic shared memory: [pad to 128 bytes | 2 tables per stream | StreamState per stream | staging areas]
  extern __shared__ __align__(16) unsigned char s_raw[];
  unsigned char* tables = s_raw + ((kTablePad - (smem_addr(s_raw) & (kTablePad - 1))) & (kTablePad - 1));
  StreamState* S = reinterpret_cast<StreamState*>(s_raw + kTablePad + KS * 2 * kTableBytes);
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const uint32_t nwarps = ctas * warps;
  if (CLEAR) {
    if (cta == 0 && threadIdx.x == 0) *status.word = 0;
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  }
  begin_next();  // the next group of a chain may prepare its tables on the SMs that this launch leaves
  const uint32_t whole_end = min(chunk_end, (uint32_t)(n / kChunkElems));  // the chunks that are full; at most 2^20 in all
  uint32_t c = chunk_begin + cta * warps + warp;
  if (c < whole_end) prefetch_rows(base + (uint64_t)c * kChunkElems, lane);
  static_assert(KS <= 4 && 5 * kMaxSymbols <= kTableBytes, "a warp per stream; the second level is the scratch");
  if (warp < KS) {
    const uint8_t* ptr = streams.ptr[0];
    uint64_t bytes = streams.bytes[0];
#pragma unroll
    for (int s = 1; s < KS; ++s)
      if (warp == s) ptr = streams.ptr[s], bytes = streams.bytes[s];
    const int err = prepare_stream(S[warp], tables + warp * 2 * kTableBytes + kTableBytes, ptr, bytes, n, lane);
    if (lane == 0) {
      S[warp].err = err;
      S[warp].ptr = ptr;
      S[warp].l1_addr = smem_addr(tables + warp * 2 * kTableBytes);
    }
  }
  __syncthreads();
  if (CLEAR) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
#pragma unroll
  for (int s = 0; s < KS; ++s) {
    const int err = S[s].err;
    if (err) {  // the same words for every thread
      wait_previous();  // the launch before this one may clear the word; and the order of the launches reaches back to the first
      if (threadIdx.x == 0) status.set(err);
      return;
    }
  }
  // Prefixes that any of the streams resolves in the second level are looked up there in all of them, in sub-tables as
  // deep as their number allows: the lookup's addressing is then the same for all streams.
  uint32_t most = 0;  // this and what follows are the same for every thread
#pragma unroll
  for (int s = 0; s < KS; ++s) most = max(most, S[s].misses);
  static_assert(kTableBytes / 8 == 1u << 10 && kSubBitsMax == 9 && kSubBitsMin == 4, "sub-tables of 10 - ceil(log2 most) bits fill the second level");
  const uint32_t sub_bits = __clz(max(most, 2u) - 1) - 22;  // 9 to 4
  if (threadIdx.x < KS) {
    S[threadIdx.x].nsub = most;
    S[threadIdx.x].sub_bits = sub_bits;
  }
  Index index = by_direct<KS>(S) ? Index::kDirect : too_many_codes<KS>(S, sub_bits) ? Index::kTwoLevel : Index::kOnes;
  if (index != Index::kTwoLevel) fill_one_level<KS>(S, tables, index == Index::kDirect);
  __syncthreads();
  if (index == Index::kOnes && !by_ones<KS>(S)) index = Index::kTwoLevel;
  if (index == Index::kTwoLevel) {
    fill_tables<KS>(S, tables);
    __syncthreads();
  }

  unsigned char* stage0 = reinterpret_cast<unsigned char*>(S + KS) + (size_t)warp * KS * stage_bytes;
  wait_previous();  // the launch before this one, if it is a chain's, has written `base`
  if (index == Index::kDirect) {
    decode_chunks<KS, R, Index::kDirect>(S, base, out, c, nwarps, whole_end, chunk_end, n, lane, stage0, stage_bytes, status);
  } else if (index == Index::kOnes) {
    decode_chunks<KS, R, Index::kOnes>(S, base, out, c, nwarps, whole_end, chunk_end, n, lane, stage0, stage_bytes, status);
  } else {
    for (; c < chunk_end; c += nwarps) {
      // where the L2 prefetch goes on behind this chunk: the next full chunk of this warp, if there is one
      const float* next_rows = base + (uint64_t)(c + nwarps < whole_end ? c + nwarps : c) * kChunkElems + 4 * lane;
      decode_chunk_two_level<KS>(S, base, out, c, n, lane, stage0, stage_bytes, next_rows, status);
    }
  }
}

template <int KS, int WARPS, int R, bool CLEAR>
__global__ void __launch_bounds__(32 * WARPS, kDecCtas<KS>)
decode_kernel(const float* base, DecodeStreams streams, uint64_t n, float* out, int32_t* __restrict__ status, uint32_t rank,
              uint32_t stage_bytes, uint32_t chunk_begin, uint32_t chunk_end) {
  decode_vector<KS, R, CLEAR>(base, streams, n, out, Status{status, rank}, stage_bytes, chunk_begin, chunk_end, blockIdx.x, gridDim.x);
}

// Per-layer recovery: the CTAs [cta_begin[i], cta_begin[i + 1]) decode segment i. One launch instead of one per segment
// (a segment of a few chunks occupies one SM for the 15 us that a chunk takes; 62 of them in a row took 870 us).
template <int KS, int WARPS, int R>
__global__ void __launch_bounds__(32 * WARPS, kDecCtas<KS>)
decode_segments_kernel(const float* base, const __grid_constant__ DecodeStreams buffers, float* out,
                       int32_t* __restrict__ status, uint32_t second, uint32_t stage_bytes,
                       const __grid_constant__ SegBatch batch) {
  uint32_t lo = 0, hi = batch.nseg;  // cta_begin[lo] <= blockIdx.x < cta_begin[hi]
  while (hi - lo > 1) {
    const uint32_t mid = (lo + hi) / 2;
    if (batch.cta_begin[mid] <= blockIdx.x) lo = mid;
    else hi = mid;
  }
  const uint64_t first = batch.elem_begin[lo], n = batch.elem_begin[lo + 1] - first;
  const uint64_t off = batch.stream_begin[lo], bytes = batch.stream_begin[lo + 1] - off;
  DecodeStreams streams;
#pragma unroll
  for (int s = 0; s < KS; ++s) {
    streams.ptr[s] = buffers.ptr[s] + off;
    streams.bytes[s] = bytes;
  }
  decode_vector<KS, R, false>(base + first, streams, n, out + first, Status{status, 2 * (batch.first + lo) + second}, stage_bytes, 0,
                    (uint32_t)((n + kChunkElems - 1) / kChunkElems), blockIdx.x - batch.cta_begin[lo],
                    batch.cta_begin[lo + 1] - batch.cta_begin[lo]);
}

// Launch shape: CTAs of `warps` warps, `per_sm` of them on an SM, `stage` bytes of staging area per warp and stream.
struct Shape {
  uint32_t warps, stage, dyn, per_sm, sms;
};

// What bounds the CTAs on an SM: registers (allocated in units of 256 per warp), shared memory (1 KB per CTA is the
// system's) and 64 warps. Computed here because the occupancy query costs the host about a microsecond a call.
inline uint32_t ctas_on_sm(uint32_t warps, uint32_t dyn, uint32_t regs) {
  const uint32_t per_warp = (regs * 32 + 255) / 256 * 256;
  const uint32_t by_regs = 65536 / per_warp / 4 * 4 / warps;  // warps are spread over four schedulers
  const uint32_t by_smem = 228 * 1024 / (dyn + 1024), by_warps = 64 / warps;
  return min(min(by_regs, by_smem), by_warps);
}

constexpr uint32_t kMaxStage = kChunkElems * 8 + 16;

// Staging bytes a warp and stream that hold a chunk of `avg` bytes with some room (chunks vary, and the streams' areas are one), and its space
// if such chunks are copied with space. Asked for in every case, the space took four of 16 warps from chunks of 2137 to 2206 bytes in
// four streams, which have none: 134 M elements of 4.2 bits a code 325 us instead of 291.
uint32_t wanted_stage(uint64_t avg) {
  return (uint32_t)min(align_up(avg + avg / 32 + (spaced_chunk(avg) ? kSpaceBytes + 16 : 48), 16), (uint64_t)kMaxStage);
}

constexpr uint32_t tables_bytes(int ks) { return kTablePad + ks * (2 * kTableBytes + (uint32_t)sizeof(StreamState)); }
constexpr uint32_t kMaxDyn = kSmemPerSm - 1024 - kOverrunBytes;  // room for static __shared__ and the padding

// Among CTAs of `most` warps and four, eight, ... fewer, down to eight, the shape that puts most warps on an SM (with four streams that is
// one CTA of 16 warps, with one stream several smaller ones), with the staging areas given whatever shared memory that shape leaves.
Shape choose_shape(int ks, uint32_t want_stage, uint32_t regs, uint32_t most) {
  const uint32_t tables = tables_bytes(ks);
  if (want_stage > kMaxStage) want_stage = kMaxStage;
  Shape best{};
  for (uint32_t w = most; w >= 8; w -= 4) {
    uint32_t st = want_stage;
    if (tables + (uint64_t)w * ks * st > kMaxDyn) {
      if (w > 8) continue;                               // try fewer warps first
      st = ((kMaxDyn - tables) / (w * ks)) / 16 * 16;    // last resort: what fits; large chunks decode from global
    }
    const uint32_t d = tables + w * ks * st + kOverrunBytes, bps = ctas_on_sm(w, d, regs);
    if (bps * w > best.per_sm * best.warps) {
      best.warps = w;
      best.stage = st;
      best.dyn = d;
      best.per_sm = bps;
    }
  }
  if (best.per_sm == 0) return best;
  const uint32_t budget = kSmemPerSm / best.per_sm - 1024 - 64;
  if (budget > tables + kOverrunBytes) {
    uint32_t st = ((budget - tables - kOverrunBytes) / (best.warps * ks)) / 16 * 16;
    if (st > kMaxStage) st = kMaxStage;
    const uint32_t d = tables + best.warps * ks * st + kOverrunBytes;
    if (st > best.stage && d <= kMaxDyn + kOverrunBytes && ctas_on_sm(best.warps, d, regs) >= best.per_sm) {
      best.stage = st;
      best.dyn = d;
    }
  }
  return best;
}

template <int KS, int WARPS>
cudaError_t decode_shape(const void* fn, uint32_t want_stage, uint32_t (&regs_of)[kMaxDevices], Shape& best) {
  static int sms_of[kMaxDevices] = {};
  const int dev = current_device_index();
  if (dev < 0) return cudaErrorInvalidDevice;
  if (regs_of[dev] == 0) {  // by device ordinal; non-zero once the kernel's attributes are set there
    int v = 0;
    cudaFuncAttributes at;
    cudaError_t e = cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&at, fn);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(kMaxDyn + kOverrunBytes));
    if (e != cudaSuccess) return e;
    sms_of[dev] = v;
    regs_of[dev] = (uint32_t)at.numRegs;
  }
  best = choose_shape(KS, want_stage, regs_of[dev], WARPS);
  best.sms = (uint32_t)sms_of[dev];
  if (best.per_sm == 0) return cudaErrorLaunchOutOfResources;
  // shared-memory carve-out in percent of the SM's 228 KB: what the resident CTAs use (dynamic, static and the
  // 1 KB per CTA that the system reserves), so that whatever is left serves as L1
  const int carve = (int)(((uint64_t)best.per_sm * (best.dyn + 2048) * 100 + 228 * 1024 - 1) / (228 * 1024)) + 1;
  return cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, carve < 100 ? carve : 100);
}

// One stream: two rows a step while the warps on the device have two and a half chunks each at most. A launch of few rounds waits for its lanes' chains, which
// are shorter that way; one of many rounds for HBM. One row and two: 61,706 elements blocking 26.9 and 25.4 us, 11.7 M 28.0 and 24.8, 21 M (1.4 rounds)
// 47.3 and 42.3, 32 M (2.2) 57.5 and 52.6, 43 M (3.0) 69.5 and 72.1, 87 M 129.5 and 138.0, 1.3 G 1750 and 1870.
constexpr bool two_rows(uint64_t chunks, uint64_t warps) { return 2 * chunks <= 5 * warps; }

// A warp decodes whole chunks, so `chunks` of them take a whole number of rounds over the CTAs that fit on the device.
// With as few warps as do them in the same number of rounds all rounds are equally full; with all warps the last one can
// be nearly empty, and takes nearly as long as the others (11.7 M elements, four streams: 19.3 chunks per SM in rounds of
// 16 and 3.3, or of 10 and 9.3). Four warps at least: fewer take longer over the tables than they save.
uint32_t balanced_warps(uint64_t chunks, uint64_t ctas, uint32_t most) {
  const uint64_t rounds = (chunks + ctas * most - 1) / (ctas * most);
  if (rounds == 0) return 4;
  const uint64_t w = (chunks + ctas * rounds - 1) / (ctas * rounds);
  return w < 4 ? 4 : (uint32_t)w;
}

constexpr unsigned kMaxClearCtas = 8;  // a portable cluster size
static_assert(kClearChunks <= 4 * kMaxClearCtas, "four warps a CTA at least");

// second: this launch goes on from what the one before it recovers, and may begin beside its end: tables and first rows do not wait for it (11.7 M
// elements, eight streams: 81.0 -> 76.0 us).
// CLEAR: see decode_vector; at most kClearChunks chunks. cudaErrorNotSupported, with nothing launched: the device has no room for the cluster.
template <int KS, bool CLEAR, int WARPS = kDecWarps<KS>, int R = 2>
cudaError_t launch_decode_ks(const float* base, const DecodeStreams& streams, uint64_t n, float* out,
                             int32_t* status, bool second, uint64_t chunk_begin, uint64_t chunk_end, cudaStream_t cs) {
  static uint32_t regs_of[kMaxDevices] = {};
  const uint64_t nchunks = (n + kChunkElems - 1) / kChunkElems;
  // the largest average chunk of the streams (from the buffer sizes, which bound the payload)
  uint64_t avg = 0;
  for (int s = 0; s < KS; ++s) {
    const uint64_t index_bytes = 72 * nchunks;  // lane and chunk index entries are not staged
    const uint64_t a = (streams.bytes[s] > index_bytes ? streams.bytes[s] - index_bytes : 0) / (nchunks ? nchunks : 1);
    avg = a > avg ? a : avg;
  }
  // where the areas of 20 warps do not fit, the kernel for 16
  if constexpr (KS == 3 && WARPS == 20)
    if (choose_shape(KS, wanted_stage(avg), 96, WARPS).warps < WARPS)
      return launch_decode_ks<KS, CLEAR, 16>(base, streams, n, out, status, second, chunk_begin, chunk_end, cs);
  Shape sh;
  const auto kernel = decode_kernel<KS, WARPS, R, CLEAR>;
  const cudaError_t e = decode_shape<KS, WARPS>(reinterpret_cast<const void*>(kernel), wanted_stage(avg), regs_of, sh);
  if (e != cudaSuccess) return e;
  const uint64_t chunks = chunk_end - chunk_begin, full = (uint64_t)sh.sms * sh.per_sm;
  if constexpr (KS == 1 && R == 2 && !CLEAR)
    if (!two_rows(chunks, full * sh.warps)) return launch_decode_ks<KS, CLEAR, WARPS, 1>(base, streams, n, out, status, second, chunk_begin, chunk_end, cs);
  const uint32_t warps = balanced_warps(chunks, full, sh.warps);
  uint64_t want = (chunks + warps - 1) / warps;
  if (want == 0) want = 1;  // still reports a rejected stream
  const unsigned grid = (unsigned)(want < full ? want : full);
  // the staging areas of the warps left out go to the others: chunks vary (a layer of rare exponents in a vector of layers
  // takes twice the average), and one that is read from global memory word by word holds up the launch
  const uint32_t stage = min(sh.warps * sh.stage / warps / 16 * 16, kChunkElems * 8 + 16);
  const size_t dyn = sh.dyn - (sh.warps * sh.stage - warps * stage) * KS;
  if constexpr (CLEAR) {
    static int room_of[kMaxDevices] = {};  // by device ordinal: 0 not looked at yet, 1 room, 2 none
    const int dev = current_device_index();
    if (dev < 0) return cudaErrorInvalidDevice;
    unsigned ctas = 1;  // a power of two, so that every size is one the hardware schedules
    while (ctas < grid) ctas *= 2;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    cfg.blockDim = dim3(warps * 32);
    cfg.stream = cs;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (room_of[dev] == 0) {
      int fit = 0;
      at[0].val.clusterDim = {kMaxClearCtas, 1, 1};
      cfg.gridDim = dim3(kMaxClearCtas);
      cfg.dynamicSmemBytes = kMaxDyn;
      room_of[dev] = cudaOccupancyMaxActiveClusters(&fit, kernel, &cfg) == cudaSuccess && fit > 0 ? 1 : 2;
      (void)cudaGetLastError();
    }
    if (room_of[dev] == 2 || ctas > kMaxClearCtas) return cudaErrorNotSupported;
    at[0].val.clusterDim = {ctas, 1, 1};
    cfg.gridDim = dim3(ctas);
    cfg.dynamicSmemBytes = dyn;
    return cudaLaunchKernelEx(&cfg, kernel, base, streams, n, out, status, 0u, stage, (uint32_t)chunk_begin, (uint32_t)chunk_end);
  } else {
    return launch_kernel(second, kernel, grid, warps * 32, dyn, cs, base, streams, n, out, status, second ? 1u : 0u, stage, (uint32_t)chunk_begin,
                         (uint32_t)chunk_end);
  }
}

template <int KS, int WARPS = KS == 3 ? 16 : kDecWarps<KS>, int R = 2>
cudaError_t launch_segments_ks(const float* base, const uint8_t* const* streams, SegBatch& batch, int nbits, float* out,
                               int32_t* status, bool second, cudaStream_t cs) {
  static uint32_t regs_of[kMaxDevices] = {};
  // the buffers are sized for nbits bits per element, which no chunk exceeds by much
  Shape sh;
  const cudaError_t e = decode_shape<KS, WARPS>(reinterpret_cast<const void*>(decode_segments_kernel<KS, WARPS, R>),
                                         (uint32_t)align_up((uint64_t)nbits * (kChunkElems / 8) + 64, 16), regs_of, sh);
  if (e != cudaSuccess) return e;
  if constexpr (KS == 1 && R == 2) {
    const uint64_t chunks = (batch.elem_begin[batch.nseg] - batch.elem_begin[0]) / kChunkElems;  // about
    if (!two_rows(chunks, (uint64_t)sh.sms * sh.per_sm * sh.warps)) return launch_segments_ks<KS, WARPS, 1>(base, streams, batch, nbits, out, status, second, cs);
  }
  DecodeStreams buffers;
  for (int s = 0; s < 4; ++s) buffers.ptr[s] = s < KS ? streams[s] : nullptr, buffers.bytes[s] = 0;
  const uint32_t ctas = split_segments(batch, sh.warps, sh.sms * sh.per_sm);
  return launch_kernel(second, decode_segments_kernel<KS, WARPS, R>, ctas, sh.warps * 32, sh.dyn, cs, base, buffers, out, status, second ? 1u : 0u, sh.stage,
                       batch);
}

}  // namespace

uint32_t decode_warps(int k, uint64_t chunk_bytes, uint32_t regs) {
  if (k < 1 || k > 4 || regs < 16 || regs > 255) return 0;
  const int most = k == 1 ? kDecWarps<1> : k == 2 ? kDecWarps<2> : k == 3 ? kDecWarps<3> : kDecWarps<4>;
  const Shape sh = choose_shape(k, wanted_stage(chunk_bytes), regs, most);
  return sh.per_sm * sh.warps;
}

// How the CTAs are dealt out: every one takes up to r rounds (a chunk per warp) of one segment, the same r for all. While
// all CTAs fit on the device at once, the launch takes as long as the preparation and r rounds, so the smallest such r is
// the best of those. But every segment takes a CTA of its own, however small: with about as many segments as slots that r
// grows to the largest segment's whole length. So the smaller r, which take several waves, are weighed against it by the
// bound for work dealt out in order, (all preparations and rounds) / slots + the longest CTA's. 159 layers of up to 12,000
// values and one of 25 M: 131 us with two streams and 153 with four, with one wave in every case 5177 and 8507; 130 layers,
// 30 of them of 2.5 M: 191 and 256 us, with one wave 516 and 833. One wave that is nearly even stays.
uint32_t split_segments(SegBatch& batch, uint32_t warps, uint32_t slots) {
  constexpr double kPrepare = 0.5;  // of a round's time: 8 to 10 us beside 15 to 20
  uint32_t rounds_of[kSegBatch], longest = 1, all = 0;  // 2^20 chunks a segment at most
  for (uint32_t i = 0; i < batch.nseg; ++i) {
    const uint32_t chunks = (uint32_t)((batch.elem_begin[i + 1] - batch.elem_begin[i] + kChunkElems - 1) / kChunkElems);
    rounds_of[i] = chunks ? (chunks + warps - 1) / warps : 1;  // an empty segment's stream is validated too
    all += rounds_of[i];
    longest = max(longest, rounds_of[i]);
  }
  const auto ctas_with = [&](uint32_t r) {
    uint32_t ctas = 0;
    for (uint32_t i = 0; i < batch.nseg; ++i) ctas += (rounds_of[i] + r - 1) / r;
    return ctas;
  };
  const auto time_of = [&](uint32_t r) {
    const uint32_t ctas = ctas_with(r);
    const double one = kPrepare + r;
    return ctas <= slots ? one : (ctas * kPrepare + all) / slots + one;
  };
  // the smallest r of one wave, or `longest` if there is none; `least` rounds would fill it evenly
  const uint32_t least = min(longest, (all + slots - 1) / slots);
  uint32_t lo = least, fit = least;
  while (fit < longest && ctas_with(fit) > slots) lo = fit + 1, fit = min(longest, 2 * fit);
  while (lo < fit) {
    const uint32_t mid = (lo + fit) / 2;
    if (ctas_with(mid) <= slots) fit = mid;
    else lo = mid + 1;
  }
  uint32_t best = fit;
  if (fit > least + 1) {  // no split takes less than `least` rounds and one more
    double shortest = time_of(fit);
    for (uint32_t r = 1; r < fit; r += (r + 3) / 4) {
      const double t = time_of(r);
      if (t < shortest) shortest = t, best = r;
    }
  }
  uint32_t ctas = 0;
  for (uint32_t i = 0; i < batch.nseg; ++i) {
    batch.cta_begin[i] = ctas;
    ctas += (rounds_of[i] + best - 1) / best;
  }
  batch.cta_begin[batch.nseg] = ctas;
  return ctas;
}

// Four at a time, but five as three and two: a launch with one stream is bound by HBM and takes as long as one with two (1.3 G elements: four
// and one 4602 us, three and two 4023). (Eight as three, three and two, where 16 warps an SM need two rounds and 20 one: 11.7 M elements of 62
// layers 214 us instead of 155, because the smaller staging areas do not hold the chunks of some layers.)
// Layers of up to 4 bits stay four and one: their areas, sized by nbits, let four streams have as many warps as three, and the launch with one ends
// soonest (62 layers, 11.7 M, 3 and 4 bits: 76 and 74 us, three and two 84 and 80; 40 layers, 16 M, 94 and 93, 88 and 91). With 5 and 6 bits four
// streams get fewer (62 layers 83 and 97, three and two 83 and 91; 40 layers 105 and 120, 92 and 101).
int decode_group(int left) { return left <= 4 ? left : left == 5 ? 3 : 4; }
int decode_group_segments(int left, int nbits) { return nbits <= 4 ? (left <= 4 ? left : 4) : decode_group(left); }

cudaError_t launch_decode_segments(const float* base, const uint8_t* const* streams, int k, SegBatch& batch, int nbits,
                                   float* out, int32_t* status, bool second, cudaStream_t cs) {
  switch (k) {
    case 1: return launch_segments_ks<1>(base, streams, batch, nbits, out, status, second, cs);
    case 2: return launch_segments_ks<2>(base, streams, batch, nbits, out, status, second, cs);
    case 3: return launch_segments_ks<3>(base, streams, batch, nbits, out, status, second, cs);
    case 4: return launch_segments_ks<4>(base, streams, batch, nbits, out, status, second, cs);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_decode(const float* base, const DecodeStreams& streams, int k, uint64_t n, float* out,
                          int32_t* status, bool second, cudaStream_t cs, uint64_t chunk_begin, uint64_t chunk_end, bool clear) {
  if (k < 1 || k > 4 || (clear && (second || n > (uint64_t)kClearChunks * kChunkElems))) return cudaErrorInvalidValue;
  const uint64_t all_chunks = (n + kChunkElems - 1) / kChunkElems;
  if (chunk_end > all_chunks) chunk_end = all_chunks;
  if (chunk_begin > chunk_end) chunk_begin = chunk_end;
  switch (k) {
    case 1: return clear ? launch_decode_ks<1, true>(base, streams, n, out, status, second, chunk_begin, chunk_end, cs)
                         : launch_decode_ks<1, false>(base, streams, n, out, status, second, chunk_begin, chunk_end, cs);
    case 2: return clear ? launch_decode_ks<2, true>(base, streams, n, out, status, second, chunk_begin, chunk_end, cs)
                         : launch_decode_ks<2, false>(base, streams, n, out, status, second, chunk_begin, chunk_end, cs);
    case 3: return clear ? launch_decode_ks<3, true>(base, streams, n, out, status, second, chunk_begin, chunk_end, cs)
                         : launch_decode_ks<3, false>(base, streams, n, out, status, second, chunk_begin, chunk_end, cs);
    case 4: return clear ? launch_decode_ks<4, true>(base, streams, n, out, status, second, chunk_begin, chunk_end, cs)
                         : launch_decode_ks<4, false>(base, streams, n, out, status, second, chunk_begin, chunk_end, cs);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lc
