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
//    staging area is decoded from global memory by the same code.
//  * Codes are looked up in shared-memory tables whose entries hold the representative itself. The
//    first level is indexed by the next kL1Bits bits and replicated 16 times (entry for (index, lane)
//    at index*16 + lane%16): a 64-bit shared load is served half a warp at a time, so the 16 lanes of
//    a half-warp always hit 16 different bank pairs although their indices are data dependent.
//    Codes are canonical, so the 6-bit prefixes of longer codes are the last ones; from the first of them on a lane
//    reads the second level instead, indexed by up to 9 more bits (the same load, no branch), which resolves codes of
//    up to 15 bits; still longer codes are found by a canonical search behind a warp vote.
//  * A lane keeps a 64-bit bit buffer per stream and tops it up with one predicated word load before
//    every fourth symbol; a lane whose four codes take more bits than it held does the step again.
//
// Every read of a stream is bounds-checked against the caller's buffer size and every table is
// validated before use, so a damaged stream yields LC_ERR_FORMAT (and unspecified output), never an
// out-of-bounds access.
//
// Bound: HBM at k = 1 (8 bytes per element + the stream); at k = 4 the integer work per symbol is
// the limit.
#include "lc_decode_bits.cuh"

namespace lc {
namespace {

using namespace dec;

// Threads per CTA at most, and CTAs per SM that the registers must allow: with one stream 24 warps fit on an SM as two CTAs
// of 12 (80 registers); two streams fit one CTA of 20 (96 registers: 138 M elements 240 -> 220 us against 16 warps, 11.7 M
// elements 46 -> 31 us, because their 19.3 chunks per SM are then one round); with three and four a thread holds more state
// and one CTA of 16 takes the SM (bounded to 96 registers, four streams spill and take 1.4 times as long).
template <int KS>
constexpr int kDecThreads = KS == 1 ? 384 : KS == 2 ? 640 : 512;
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
// Length field of a table entry that does not resolve its code. As a length it takes the bit count far below zero,
// which is how the hot loop notices: a step subtracts at most four of them per stream, and 1..4 times 2^29 (less a
// few real lengths) leaves the sign bit of the 32-bit count set in every case.
constexpr uint32_t kLongCode = 0x20000000u;
// distance, in steps of 512 bytes per warp, of the L2 prefetch of base: chains of two and more do not care between 4 and 12;
// a single stream of 138 M elements takes 194 us at 4, 207 at 6, 228 at 8 and 247 at 12
template <int KS>
constexpr int kPrefetchRows = KS == 1 ? 4 : 8;

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
  bool bad = index_end != ((lane & 1) ? payload_size : 0ull);
  unsigned long long kraft = 0, count_sum = 0, bit_sum = 0;
  uint32_t nused = 0, seen_max = 0, only_rep = 0;
  for (uint32_t first = 0; first < nsym; first += 32) {
    const uint32_t sym = first + lane;
    const bool have = sym < nsym;
    uint4 e = make_uint4(0u, 0u, 0u, 0u);
    if (have) e = __ldg(reinterpret_cast<const uint4*>(s + kHeaderBytes) + sym);  // key:16 len:8 pad:8 | rep | count
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

template <int KS, bool STAGED, bool PARTIAL>
__device__ __forceinline__ void decode_chunk_fast(const StreamState* S, const Source* W, const uint32_t* start,
                                                    const float* base, float* out, uint64_t c, uint64_t n, uint32_t lane,
                                                    const float* next_rows, Status status) {
  LaneBits<STAGED> bits[KS];
  const int rem = PARTIAL ? (int)(n - c * kChunkElems) - 4 * (int)lane : 0;  // elements from this lane's first slot on
  const uint32_t steps = PARTIAL ? (uint32_t)(n - c * kChunkElems + 127) / 128 : kSteps;
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
    if (!PARTIAL || have >= 4) {
      *reinterpret_cast<float4*>(out + i) = make_float4(x[0], x[1], x[2], x[3]);
    } else {
      if (have > 0) out[i] = x[0];
      if (have > 1) out[i + 1] = x[1];
      if (have > 2) out[i + 2] = x[2];
    }
  }
}
static_assert(kL1Rep * 8 == 128, "first-level entries of one index span 128 bytes");

// Chunk `c` of every stream: where its payload is and the lanes' bit counts. An entry that is not a valid range of the
// payload is reported and taken as empty.
template <int KS>
__device__ __forceinline__ bool stage_chunk(const StreamState* S, uint64_t c, uint32_t lane, unsigned char* stage0,
                                            uint32_t stage_bytes, Source* W, uint32_t* start, Status status) {
  uint32_t bytes[KS];
  unsigned long long off0[KS], off1[KS];
  bool fits = true;
  // all index loads of all streams first, so that their latencies overlap
#pragma unroll
  for (int s = 0; s < KS; ++s) {
    const uint8_t* sp = S[s].ptr;
    const unsigned long long* ci = reinterpret_cast<const unsigned long long*>(sp + S[s].chunk_index_off);
    off0[s] = __ldg(ci + c);
    off1[s] = __ldg(ci + c + 1);
    const uint16_t* li = reinterpret_cast<const uint16_t*>(sp + S[s].lane_index_off);
    start[s] = __ldg(li + c * kLanes + lane);
  }
  // then the asynchronous copies of the payloads into the staging areas
#pragma unroll
  for (int s = 0; s < KS; ++s) {
    if (off0[s] > off1[s] || off1[s] > S[s].payload_size || (off0[s] & 15) || (off1[s] & 15)) {
      status.set(LC_ERR_FORMAT);
      off0[s] = off1[s] = 0;
    }
    bytes[s] = (uint32_t)min(off1[s] - off0[s], (unsigned long long)kChunkElems * 8);
    const uint8_t* g = S[s].ptr + S[s].payload_off + off0[s];
    unsigned char* st = stage0 + (size_t)s * stage_bytes;
    W[s].g = reinterpret_cast<const uint32_t*>(g);
    W[s].nw = bytes[s] >> 2;
    W[s].sbase = smem_addr(st);
    W[s].slim = W[s].sbase + bytes[s] + 12;
    // 16 bytes of zero slack after the chunk must fit too
    if (bytes[s] + 16 <= stage_bytes) {
      for (uint32_t k = lane * 16; k < bytes[s]; k += 32 * 16) cp_async_16(W[s].sbase + k, g + k);
      if (lane == 0) *reinterpret_cast<uint4*>(st + bytes[s]) = make_uint4(0, 0, 0, 0);
    } else {
      fits = false;
    }
  }
  cp_async_commit();
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
  }
  cp_async_wait_all();
  __syncwarp();
  return fits;
}

// The vector's last, partial chunk, out of line and outside the main loop: it runs once per call, in one warp, and must
// not weigh on the registers of the others. On vectors of a few thousand chunks the whole launch waits for that warp, so
// it runs the same straight-line steps as a whole chunk (one code at a time it took 15 us with one stream and 60 us
// with four).
template <int KS>
__device__ __noinline__ void decode_last_chunk(const StreamState* S, const float* base, float* out, uint64_t c, uint64_t n,
                                               uint32_t lane, unsigned char* stage0, uint32_t stage_bytes, Status status) {
  Source W[KS];
  uint32_t start[KS];
  __syncwarp();  // the previous chunk's reads of the staging area are done
  if (stage_chunk<KS>(S, c, lane, stage0, stage_bytes, W, start, status))
    decode_chunk_fast<KS, true, true>(S, W, start, base, out, c, n, lane, base, status);
  else
    decode_chunk_fast<KS, false, true>(S, W, start, base, out, c, n, lane, base, status);
}

// Chunks [chunk_begin, chunk_end) of one vector, by `ctas` CTAs of which this is number `cta`.
// stage_bytes: bytes of staging area per warp and stream (a multiple of 16, at least 32).
template <int KS>
__device__ __forceinline__ void decode_vector(const float* base, const DecodeStreams& streams, uint64_t n, float* out,
                                              Status status, uint32_t stage_bytes, uint64_t chunk_begin,
                                              uint64_t chunk_end, uint32_t cta, uint32_t ctas) {
  // dynamic shared memory: [pad to 128 bytes | 2 tables per stream | StreamState per stream | staging areas]
  extern __shared__ __align__(16) unsigned char s_raw[];
  unsigned char* tables = s_raw + ((kTablePad - (smem_addr(s_raw) & (kTablePad - 1))) & (kTablePad - 1));
  StreamState* S = reinterpret_cast<StreamState*>(s_raw + kTablePad + KS * 2 * kTableBytes);
  const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
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
#pragma unroll
  for (int s = 0; s < KS; ++s) {
    const int err = S[s].err;
    if (err) {  // the same words for every thread
      if (threadIdx.x == 0) status.set(err);
      return;
    }
  }
  // Prefixes that any of the streams resolves in the second level are looked up there in all of them, in sub-tables as
  // deep as their number allows: the lookup's addressing is then the same for all streams.
  if (threadIdx.x < KS) {
    uint32_t most = 0;
#pragma unroll
    for (int s = 0; s < KS; ++s) most = max(most, S[s].misses);
    uint32_t sub_bits = kSubBitsMax;
    while (sub_bits > kSubBitsMin && most > (kTableBytes >> (sub_bits + 3))) sub_bits -= 1;
    S[threadIdx.x].nsub = most;
    S[threadIdx.x].sub_bits = sub_bits;
  }
  __syncthreads();
  fill_tables<KS>(S, tables);
  __syncthreads();

  unsigned char* stage0 = reinterpret_cast<unsigned char*>(S + KS) + (size_t)warp * KS * stage_bytes;
  const uint64_t nwarps = (uint64_t)ctas * warps;
  const uint64_t whole_end = min(chunk_end, n / kChunkElems);  // the chunks that are full
  uint64_t c = chunk_begin + (uint64_t)cta * warps + warp;
  for (; c < whole_end; c += nwarps) {
    Source W[KS];
    uint32_t start[KS];
    __syncwarp();  // the previous chunk's reads of the staging area are done
    const bool fits = stage_chunk<KS>(S, c, lane, stage0, stage_bytes, W, start, status);
    // where the L2 prefetch goes on behind this chunk: the next full chunk of this warp, if there is one
    const float* next_rows = base + (c + nwarps < whole_end ? c + nwarps : c) * kChunkElems + 4 * lane;
    if (fits) decode_chunk_fast<KS, true, false>(S, W, start, base, out, c, n, lane, next_rows, status);
    else decode_chunk_fast<KS, false, false>(S, W, start, base, out, c, n, lane, next_rows, status);
  }
  if (c < chunk_end) decode_last_chunk<KS>(S, base, out, c, n, lane, stage0, stage_bytes, status);
}

template <int KS>
__global__ void __launch_bounds__(kDecThreads<KS>, kDecCtas<KS>)
decode_kernel(const float* base, DecodeStreams streams, uint64_t n, float* out, int32_t* __restrict__ status, uint32_t rank,
              uint32_t stage_bytes, uint64_t chunk_begin, uint64_t chunk_end) {
  decode_vector<KS>(base, streams, n, out, Status{status, rank}, stage_bytes, chunk_begin, chunk_end, blockIdx.x, gridDim.x);
}

// Per-layer recovery: the CTAs [cta_begin[i], cta_begin[i + 1]) decode segment i. One launch instead of one per segment
// (a segment of a few chunks occupies one SM for the 15 us that a chunk takes; 62 of them in a row took 870 us).
template <int KS>
__global__ void __launch_bounds__(kDecThreads<KS>, kDecCtas<KS>)
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
  decode_vector<KS>(base + first, streams, n, out + first, Status{status, 2 * (batch.first + lo) + second}, stage_bytes, 0,
                    (n + kChunkElems - 1) / kChunkElems, blockIdx.x - batch.cta_begin[lo],
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

// want_stage: staging bytes that hold an average chunk with some room. Among CTAs of 20 (two streams only), 16, 12 and 8 warps, takes the shape
// that puts most warps on an SM (with four streams that is one CTA of 16 warps, with one stream several smaller ones),
// then gives the staging areas whatever shared memory that shape leaves (chunk sizes vary around the average).
template <int KS>
cudaError_t decode_shape(const void* fn, uint64_t want_stage, uint32_t (&regs_of)[kMaxDevices], Shape& best) {
  constexpr uint32_t kTables = kTablePad + KS * (2 * kTableBytes + sizeof(StreamState));
  constexpr uint32_t kMaxDyn = kSmemPerSm - 1024 - kOverrunBytes;  // room for static __shared__ and the padding
  constexpr uint32_t kMaxStage = kChunkElems * 8 + 16;
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
  const uint32_t regs = regs_of[dev];
  if (want_stage > kMaxStage) want_stage = kMaxStage;
  best = Shape{0, 0, 0, 0, (uint32_t)sms_of[dev]};
  for (uint32_t w = kDecThreads<KS> / 32; w >= 8; w -= 4) {
    uint32_t st = (uint32_t)want_stage;
    if (kTables + (uint64_t)w * KS * st > kMaxDyn) {
      if (w > 8) continue;                               // try fewer warps first
      st = ((kMaxDyn - kTables) / (w * KS)) / 16 * 16;   // last resort: what fits; large chunks decode from global
    }
    const uint32_t d = kTables + w * KS * st + kOverrunBytes, bps = ctas_on_sm(w, d, regs);
    if (bps * w > best.per_sm * best.warps) {
      best.warps = w;
      best.stage = st;
      best.dyn = d;
      best.per_sm = bps;
    }
  }
  if (best.per_sm == 0) return cudaErrorLaunchOutOfResources;
  const uint32_t budget = kSmemPerSm / best.per_sm - 1024 - 64;
  if (budget > kTables + kOverrunBytes) {
    uint32_t st = ((budget - kTables - kOverrunBytes) / (best.warps * KS)) / 16 * 16;
    if (st > kMaxStage) st = kMaxStage;
    const uint32_t d = kTables + best.warps * KS * st + kOverrunBytes;
    if (st > best.stage && d <= kMaxDyn + kOverrunBytes && ctas_on_sm(best.warps, d, regs) >= best.per_sm) {
      best.stage = st;
      best.dyn = d;
    }
  }
  // shared-memory carve-out in percent of the SM's 228 KB: what the resident CTAs use (dynamic, static and the
  // 1 KB per CTA that the system reserves), so that whatever is left serves as L1
  const int carve = (int)(((uint64_t)best.per_sm * (best.dyn + 2048) * 100 + 228 * 1024 - 1) / (228 * 1024)) + 1;
  return cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, carve < 100 ? carve : 100);
}

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

template <int KS>
cudaError_t launch_decode_ks(const float* base, const DecodeStreams& streams, uint64_t n, float* out,
                             int32_t* status, bool second, uint64_t chunk_begin, uint64_t chunk_end, cudaStream_t cs) {
  static uint32_t regs_of[kMaxDevices] = {};
  const uint64_t nchunks = (n + kChunkElems - 1) / kChunkElems;
  // 1.03 x the largest average chunk of the streams (from the buffer sizes, which bound the payload)
  uint64_t avg = 0;
  for (int s = 0; s < KS; ++s) {
    const uint64_t index_bytes = 72 * nchunks;  // lane and chunk index entries are not staged
    const uint64_t a = (streams.bytes[s] > index_bytes ? streams.bytes[s] - index_bytes : 0) / (nchunks ? nchunks : 1);
    avg = a > avg ? a : avg;
  }
  Shape sh;
  const cudaError_t e = decode_shape<KS>(reinterpret_cast<const void*>(decode_kernel<KS>), align_up(avg + avg / 32 + 48, 16),
                                         regs_of, sh);
  if (e != cudaSuccess) return e;
  const uint64_t chunks = chunk_end - chunk_begin, full = (uint64_t)sh.sms * sh.per_sm;
  const uint32_t warps = balanced_warps(chunks, full, sh.warps);
  uint64_t want = (chunks + warps - 1) / warps;
  if (want == 0) want = 1;  // still reports a rejected stream
  const unsigned grid = (unsigned)(want < full ? want : full);
  decode_kernel<KS><<<grid, warps * 32, sh.dyn - (sh.warps - warps) * KS * sh.stage, cs>>>(base, streams, n, out, status, second ? 1u : 0u, sh.stage, chunk_begin,
                                                         chunk_end);
  return cudaGetLastError();
}

template <int KS>
cudaError_t launch_segments_ks(const float* base, const uint8_t* const* streams, SegBatch& batch, int nbits, float* out,
                               int32_t* status, bool second, cudaStream_t cs) {
  static uint32_t regs_of[kMaxDevices] = {};
  // the buffers are sized for nbits bits per element, which no chunk exceeds by much
  Shape sh;
  const cudaError_t e = decode_shape<KS>(reinterpret_cast<const void*>(decode_segments_kernel<KS>),
                                         align_up((uint64_t)nbits * (kChunkElems / 8) + 64, 16), regs_of, sh);
  if (e != cudaSuccess) return e;
  DecodeStreams buffers;
  for (int s = 0; s < 4; ++s) buffers.ptr[s] = s < KS ? streams[s] : nullptr, buffers.bytes[s] = 0;
  const uint32_t ctas = split_segments(batch, sh.warps, sh.sms * sh.per_sm);
  decode_segments_kernel<KS><<<ctas, sh.warps * 32, sh.dyn, cs>>>(base, buffers, out, status, second ? 1u : 0u, sh.stage,
                                                                           batch);
  return cudaGetLastError();
}

}  // namespace

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
                          int32_t* status, bool second, cudaStream_t cs, uint64_t chunk_begin, uint64_t chunk_end) {
  if (k < 1 || k > 4) return cudaErrorInvalidValue;
  const uint64_t all_chunks = (n + kChunkElems - 1) / kChunkElems;
  if (chunk_end > all_chunks) chunk_end = all_chunks;
  if (chunk_begin > chunk_end) chunk_begin = chunk_end;
  switch (k) {
    case 1: return launch_decode_ks<1>(base, streams, n, out, status, second, chunk_begin, chunk_end, cs);
    case 2: return launch_decode_ks<2>(base, streams, n, out, status, second, chunk_begin, chunk_end, cs);
    case 3: return launch_decode_ks<3>(base, streams, n, out, status, second, chunk_begin, chunk_end, cs);
    case 4: return launch_decode_ks<4>(base, streams, n, out, status, second, chunk_begin, chunk_end, cs);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lc
