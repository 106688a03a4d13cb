// Decoder kernels of the GB300 ZipNN codec (device code, included by one
// translation unit per dtype family, decode_<family>.cu, so that their kernels
// compile in parallel): table-driven Huffman decoding of every byte-group
// stream of a chunk and the merge back to the original dtype (ZipNN Sec. 3.1,
// 3.2 inverse; Sec. 4.2 XOR with the base; Sec. 5.1 map).
//
// Work item = one chunk, or one of `parts` equal ranges of a chunk's
// sub-streams.  A persistent grid pulls items of all tensors of a batch from a
// device ticket (atomicAdd), so one launch decodes many tensors of uneven
// sizes.  Per item
//   1. warp 0 validates the chunk's map entries, requests the coded payloads
//      (table, start offsets, bitstream) into the shared-memory stage with one
//      TMA bulk copy each (cp.async.bulk, completion on an mbarrier; payloads
//      are 16-B aligned and padded by the format) and derives the canonical
//      limits of each coded group with warp scans; the ticket and the map
//      entries were requested while the item before this one was set up (payloads
//      that the stage cannot hold: see Where and stage_slice),
//   2. all warps build, per coded group, a 4096-entry table indexed by the
//      next 12 bits (12 = the longest code): the first code of the window, and
//      both its first codes when they fit in it and the group's code makes
//      such pairs common (see kPairMin),
//   3. all warps decode: thread t owns interleaved sub-streams, i.e. the
//      vectors v = t, t+T, ... of the chunk, so each warp step touches 32
//      consecutive 16-byte vectors: raw-group loads and the 16-B output stores
//      are fully coalesced; the inverse permutation and the XOR with a delta
//      base happen in registers.
// Decoding works on four symbols at a time (one 32-bit word of a byte group):
// two pair lookups, or four single ones, from 32-bit windows that hold 24
// bits for two lookups, so a sub-stream's position is advanced and its words
// refilled once per two lookups.  Entries keep the bits they consume in their
// low five bits: a wrapping funnel shift by the entry itself moves the window,
// and adding entries advances the position.
// The decoder is total: symbol counts are fixed by the map, bit reads past a
// payload return zero bits or bytes of the stage, invalid codes and bad map
// entries set the error word, and every loop is bounded; the wait for a bulk
// copy gives up after 2 s of %globaltimer (error ETIMEOUT, the CTA waits
// again, bounded, then exits).
#pragma once
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>

#include "zipnn_internal.cuh"

namespace zipnn {

namespace {

constexpr uint32_t kSmPerSm = 228u * 1024u;  // shared memory of an SM
constexpr uint32_t kSmReserve = 1024u;       // reserved by the system per CTA
constexpr uint32_t kStaticReserve = 2560u;   // the kernel's static shared memory, at most
constexpr uint32_t kLutBytes = 4u * kLutSize;      // one decode table
constexpr uint64_t kWaitLimitNs = 2000000000ull;
constexpr uint64_t kPfBudget = 16ull << 20;  // L2 bytes the loops' prefetches may hold

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
// Loads and stores through 32-bit shared-window addresses, so that table
// lookups compile to shared-memory instructions even where the table's
// location is only known at run time.
__device__ __forceinline__ uint32_t lds32(uint32_t saddr) {
  uint32_t v;
  asm("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(saddr));
  return v;
}
__device__ __forceinline__ void sts32(uint32_t saddr, uint32_t v) {
  asm volatile("st.shared.u32 [%0], %1;" ::"r"(saddr), "r"(v) : "memory");
}
__device__ __forceinline__ void sts128(uint32_t saddr, uint32_t v) {  // four copies of v
  asm volatile("st.shared.v4.u32 [%0], {%1, %1, %1, %1};" ::"r"(saddr), "r"(v) : "memory");
}
__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes) : "memory");
}
// 1-D TMA bulk copy global -> shared (16-B aligned addresses, size % 16 == 0).
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(dst), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}
// Count `bytes` of the barrier's expected transaction bytes as arrived without
// a copy (cancels bytes that were expected but never requested).
__device__ __forceinline__ void mbar_complete_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.complete_tx.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// Bounded wait for phase `parity`; false if it gave up after limit_ns.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  const uint64_t t0 = globaltimer();
  while (!mbar_try_wait(bar, parity))
    if (globaltimer() - t0 > limit_ns) return false;
  return true;
}


template <int DT> struct Traits;
template <> struct Traits<ZIPNN_BF16> { static constexpr int G = 2, V = 8; };
template <> struct Traits<ZIPNN_FP32> { static constexpr int G = 4, V = 4; };
template <> struct Traits<ZIPNN_U8> { static constexpr int G = 1, V = 16; };
// (FP16 has BF16's byte groups, so the two share code and kernels.)

struct JobRef {
  const Job* table;
  Job one;
  int n;
};

// Per-group canonical tables (shared memory).
struct GroupTab {
  uint32_t lim[kMaxLen + 2];   // left-justified (12-bit) end of the codes of length l
  uint32_t rank[kMaxLen + 2];  // rank of the first code of length l minus that code
  uint32_t words[68];          // raw table bytes (counts + symbols), 272 B
};

struct ChunkInfo {
  uint32_t mode[4];
  uint32_t value[4];
  uint32_t size[4];
  uint64_t payload[4];      // byte offset of the payload within the container
  uint32_t nwords[4];       // bitstream words (coded groups)
  uint32_t bmo[4];          // vector bitmap offset within the payload (SPARSE)
  uint32_t offs[4];         // start-bit table offset within the payload
  uint32_t bs[4];           // bitstream offset within the payload
  // staged payloads, as shared-window addresses (of byte 0 of what may be
  // staged in part: the vector bitmap, the start-bit table, the bitstream)
  uint32_t at_bm[4], at_starts[4], at_words[4];
  uint32_t end[4];          // where readers of the bitstream are clamped,
  uint32_t first[4];        // and the first bit of it in the stage
  uint32_t lut[4];          // shared-window address of the group's table
  uint32_t coded;           // bit g: group g is coded (HUFF or SPARSE)
  uint32_t pairs;           // bit g: its table holds pairs
  uint32_t stage;           // shared-window address of the stage behind the tables,
  uint32_t stage_bytes;     // its size,
  uint32_t sliced;          // whether the payloads only fit it in slices,
  uint32_t direct;          // or stay in global memory
  uint32_t ring_slots;      // kRinged: slots of the readers' rings at `stage`,
  uint32_t ring_threads;    // and the threads that have one
  uint32_t bad;             // 1: bad map entry or table, 2: a bulk copy timed out
};

// A work item: a chunk, or one of `parts` ranges of its sub-streams.
struct Item {
  const uint8_t* src;   // the container
  uint8_t* dst;         // the chunk's bytes in the tensor
  const uint8_t* base;  // the chunk's bytes of the delta base, or null
  uint32_t nb, nvec;    // its bytes and 16-byte vectors (the last one may be partial)
  uint32_t T;           // sub-streams of the chunk
  uint32_t t_lo, t_hi;  // those of the item
  uint32_t kfull;       // steps of whole vectors in every sub-stream
  uint32_t even;        // a whole chunk whose vectors split evenly over its sub-streams
  uint32_t part;
};

struct Smem {
  Item it;
  ChunkInfo ci;
  GroupTab tab[4];
  // the next item: its job, chunk (within the tensor), part and map entries
  Job job;
  uint64_t job_end;      // first global chunk past the job
  uint64_t chunk;
  uint4 entry[4];
  uint32_t jobno, part;
  uint32_t last;         // none left
  uint32_t slice_end;    // sub-stream past the slice being decoded
};

// Groups carried as Huffman sub-streams: HUFF, and SPARSE (the same after a
// bitmap of the vectors that hold a non-zero symbol).
__device__ __forceinline__ bool coded_mode(uint32_t m) { return m == kHuff || m == kSparse; }

__device__ __forceinline__ uint32_t rd_u32(const void* p) {
  return __ldg(reinterpret_cast<const uint32_t*>(p));
}

// Table entry of a 12-bit window:
//   bits 0-4    bits consumed by the entry (1 .. 12; bit 5 is zero, so that a
//               position below 32 plus two entries is exact in bits 0-5)
//   bit 6       kOne: the entry holds one symbol (else two)
//   bit 7       kBad: no code starts the window
//   bits 8-11   length of the first code
//   bits 16-23  first symbol, bits 24-31 second symbol
// Symbols of group 0 are stored rotated right by one bit (but for U8): the
// merge then needs only bit selects, see merge16r.
constexpr uint32_t kOne = 1u << 6;
constexpr uint32_t kBad = 1u << 7;

// Pairs are put in a group's table when at least kPairMin / 2^24 of its
// windows hold two whole codes (the share of lookups that find a pair, since
// windows are as frequent as their codes are short).  A lookup of a warp that
// misses in any lane costs the warp a detour, so pairs pay only when nearly
// every lookup finds one; single lookups take twice as many steps but no
// detours and no second table pass.
constexpr uint32_t kPairMin = (uint32_t)(0.990 * (1 << 24));

// Per-thread asynchronous copies global -> shared (no registers held while in
// flight); groups complete in the order they were committed.  The ring is
// touched only by these volatile statements, whose order the compiler keeps.
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N));
}
__device__ __forceinline__ uint32_t lds32v(uint32_t saddr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(saddr));
  return v;
}


// One sub-stream's reader: w0:w1 hold the 64 bits around the position (bit
// pos & 31 of w0 first), wn the word after them, read one refill ahead so that
// a refill only moves registers; nx is where the word after wn is.
struct Bits {
  uint32_t w0, w1, wn, pos, nx;
};
// Where a group's bitstream is read from, as word indexes or addresses nx:
//   kStaged  in shared memory.  nx: shared-window addresses, clamped to `end`,
//            four words past the last one: inside the stage's slack, and past
//            it by enough that a reader that was clamped fails the end check.
//   kRinged  in global memory through a ring of 16-B pieces in shared memory
//            per thread, filled by asynchronous copies.  nx: word index from
//            the payload's start.  Once per vector (refill) the pieces whose
//            slots' last words were read since are requested; pieces past the
//            payload are zero.  (Requested where the last word of a piece was
//            read, some lane of nearly every lookup pair had one, and the
//            other 31 waited: 27 instructions a symbol.)
//   kDirect  in global memory, word by word; zero bits past the last one.  nx: word
//            index.
enum Where { kStaged, kRinged, kDirect };
template <int WH> struct Source;
template <> struct Source<kStaged> {
  uint32_t base, end;
  __device__ __forceinline__ uint32_t at(uint32_t word) const { return min(base + 4u * word, end); }
  __device__ __forceinline__ uint32_t read(uint32_t& nx) const {
    const uint32_t v = lds32v(nx);
    nx = __viaddmin_u32(nx, 4u, end);
    return v;
  }
  __device__ __forceinline__ uint32_t index(uint32_t nx) const { return (nx - base) >> 2; }
  template <int V> __device__ __forceinline__ void refill(uint32_t) {}
};
template <> struct Source<kRinged> {
  const uint8_t* pay;       // the payload (16-B aligned)
  uint32_t bs, pieces;      // its bitstream's first word, its 16-B pieces
  uint32_t ring, stride;    // this thread's slot 0, bytes from slot to slot
  uint32_t mask;            // slots - 1
  uint32_t rq;              // the piece to request next
  __device__ __forceinline__ void request(uint32_t i) const {
    const uint32_t bytes = i < pieces ? 16u : 0u;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(ring + (i & mask) * stride),
                 "l"(pay + 16ull * min(i, pieces - 1u)), "r"(bytes));
  }
  // requests the pieces from word index `word` of the bitstream on
  __device__ __forceinline__ uint32_t at(uint32_t word) {
    const uint32_t nx = bs + word;
    for (uint32_t i = 0; i <= mask; i++) request((nx >> 2) + i);
    rq = (nx >> 2) + mask + 1u;
    cp_async_commit();
    cp_async_wait<0>();
    return nx;
  }
  __device__ __forceinline__ uint32_t read(uint32_t& nx) const {
    const uint32_t v = lds32v(ring + ((nx >> 2) & mask) * stride + 4u * (nx & 3u));
    nx++;
    return v;
  }
  // a vector's V codes take at most 12 V bits: 16 of them end two pieces at most,
  // 8 or 4 one
  template <int V> __device__ __forceinline__ void refill(uint32_t nx) {
#pragma unroll
    for (int k = 0; k < (V > 8 ? 2 : 1); k++)
      if (rq <= (nx >> 2) + mask) request(rq++);
  }
  __device__ __forceinline__ uint32_t index(uint32_t nx) const { return nx - bs; }
};
template <> struct Source<kDirect> {
  const uint8_t* words;
  uint32_t n;
  __device__ __forceinline__ uint32_t at(uint32_t word) const { return word; }
  __device__ __forceinline__ uint32_t read(uint32_t& nx) const {
    const uint32_t v = nx < n ? rd_u32(words + 4ull * nx) : 0u;
    nx++;
    return v;
  }
  __device__ __forceinline__ uint32_t index(uint32_t nx) const { return nx; }
  template <int V> __device__ __forceinline__ void refill(uint32_t) {}
};
// Ring sizes.  At the start of a vector every piece from the reader's own to
// the one `slots` - 1 further on is requested, and the loops close one copy group
// per vector and wait until at most kRingPending are open.  So what was requested
// by the start of two vectors ago has landed, and a vector reads at most 3 vectors'
// bits beyond the word that was next then: 19 words for 16-symbol vectors, 5
// pieces ahead (8 slots), 10 words or 3 pieces for 8 symbols and less for 4
// (4 slots).
constexpr int kRingPending = 2;
template <int V> constexpr uint32_t ring_slots_min() { return V > 8 ? 8u : 4u; }
constexpr uint32_t kRingSlotsMax = 8;

template <int WH>
__device__ __forceinline__ void bits_init(Bits& r, Source<WH>& s, uint32_t start) {
  r.pos = start & 31u;
  r.nx = s.at(start >> 5);
  r.w0 = s.read(r.nx);
  r.w1 = s.read(r.nx);
  r.wn = s.read(r.nx);
}
// Position after everything consumed so far, in bits.
template <int WH>
__device__ __forceinline__ uint32_t bits_end(const Bits& r, const Source<WH>& s) {
  return (s.index(r.nx) - 3u) * 32u + (r.pos & 31u);
}
__device__ __forceinline__ uint32_t window(const Bits& r) {
  return __funnelshift_l(r.w1, r.w0, r.pos);  // (the shift takes pos mod 32)
}
// Advance by the bits of entries whose sum (plus pos & 31) is p.
template <int WH>
__device__ __forceinline__ void advance(Bits& r, const Source<WH>& s, uint32_t p) {
  r.pos = p;
  if (p & 32u) {
    r.w0 = r.w1;
    r.w1 = r.wn;
    r.wn = s.read(r.nx);
  }
}
__device__ __forceinline__ uint32_t lookup(uint32_t lut, uint32_t win) {
  return lds32(lut + ((win >> (32 - kMaxLen)) << 2));
}

// The rest of a pair quad whose lookups e1, e2 (already consumed) did not
// both give two symbols: one or two more first codes.
template <int WH>
__device__ __forceinline__ uint32_t quad_rest(Bits& r, const Source<WH>& s, uint32_t lut,
                                              uint32_t e1, uint32_t e2, uint32_t& bad) {
  uint32_t y = (e1 & kOne) ? __byte_perm(e1, e2, 0x0762) : __byte_perm(e1, e2, 0x0632);
  const bool two = (e1 & e2 & kOne) != 0;
  uint32_t e = lookup(lut, window(r));
  bad |= e1 | e2 | e;
  advance(r, s, (r.pos & 31u) + ((e >> 8) & 15u));
  if (two) {
    y = __byte_perm(y, e, 0x0610);
    e = lookup(lut, window(r));
    bad |= e;
    advance(r, s, (r.pos & 31u) + ((e >> 8) & 15u));
  }
  return __byte_perm(y, e, 0x6210);
}

// Four symbols (first one in the low byte), by pairs or one by one.
template <int WH>
__device__ __forceinline__ uint32_t quad_pairs(Bits& r, const Source<WH>& s, uint32_t lut,
                                               uint32_t& bad) {
  const uint32_t win = window(r);
  const uint32_t e1 = lookup(lut, win);
  const uint32_t e2 = lookup(lut, __funnelshift_l(0u, win, e1));
  uint32_t y = __byte_perm(e1, e2, 0x7632);
  advance(r, s, (r.pos & 31u) + e1 + e2);
  if ((e1 | e2) & kOne) y = quad_rest(r, s, lut, e1, e2, bad);
  return y;
}
template <int WH>
__device__ __forceinline__ uint32_t duo(Bits& r, const Source<WH>& s, uint32_t lut, uint32_t& bad) {
  const uint32_t win = window(r);
  const uint32_t e1 = lookup(lut, win);
  const uint32_t e2 = lookup(lut, __funnelshift_l(0u, win, e1));
  advance(r, s, (r.pos & 31u) + e1 + e2);
  bad |= e1 | e2;
  return __byte_perm(e1, e2, 0x0062);
}
template <int WH>
__device__ __forceinline__ uint32_t quad_singles(Bits& r, const Source<WH>& s, uint32_t lut,
                                                 uint32_t& bad) {
  const uint32_t a = duo(r, s, lut, bad);
  const uint32_t b = duo(r, s, lut, bad);
  return __byte_perm(a, b, 0x5410);
}

// The inverses of split16 / split32 for exponent bytes stored rotated right by one
// bit (e' = e >> 1 | e << 7 per byte): each output byte is a bit select.
__device__ __forceinline__ void merge16r(uint32_t er, uint32_t r, uint32_t& w0, uint32_t& w1) {
  const uint32_t hi = (r & 0x80808080u) | (er & 0x7F7F7F7Fu);
  const uint32_t lo = (er & 0x80808080u) | (r & 0x7F7F7F7Fu);
  w0 = __byte_perm(lo, hi, 0x5140);
  w1 = __byte_perm(lo, hi, 0x7362);
}
__device__ __forceinline__ void merge32r(uint32_t er, uint32_t g1, uint32_t g2, uint32_t g3,
                                         uint32_t x[4]) {
  const uint32_t b3 = (g1 & 0x80808080u) | (er & 0x7F7F7F7Fu);
  const uint32_t b2 = (er & 0x80808080u) | (g1 & 0x7F7F7F7Fu);
  const uint32_t lo01 = __byte_perm(g3, g2, 0x5140), hi01 = __byte_perm(b2, b3, 0x5140);
  const uint32_t lo23 = __byte_perm(g3, g2, 0x7362), hi23 = __byte_perm(b2, b3, 0x7362);
  x[0] = __byte_perm(lo01, hi01, 0x5410);
  x[1] = __byte_perm(lo01, hi01, 0x7632);
  x[2] = __byte_perm(lo23, hi23, 0x5410);
  x[3] = __byte_perm(lo23, hi23, 0x7632);
}
__device__ __forceinline__ uint32_t rot4(uint32_t e) {  // each byte rotated right by one bit
  return ((e >> 1) & 0x7F7F7F7Fu) | ((e << 7) & 0x80808080u);
}

// Request the 128-B line holding p into L2 (no register, nothing to wait for).
__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// Accesses of the decode loops to element v (of 4, 8 or 16 bytes) of an array
// in global memory.  (The store is assembly on a global address: stores through
// generic pointers make the compiler reload, after every vector, what it holds
// of the item's records in shared memory.)
__device__ __forceinline__ uint8_t* to_global(uint8_t* p) {
  return reinterpret_cast<uint8_t*>(__cvta_generic_to_global(p));
}
__device__ __forceinline__ void store_vec(uint8_t* dst, uint32_t v, uint32_t a, uint32_t b,
                                          uint32_t c, uint32_t d) {
  asm volatile("st.global.v4.u32 [%0], {%1, %2, %3, %4};" ::"l"(dst + 16ull * v), "r"(a), "r"(b),
               "r"(c), "r"(d));
}
__device__ __forceinline__ uint32_t load_at4(const uint8_t* p, uint32_t v) {
  return __ldg(reinterpret_cast<const uint32_t*>(p) + v);
}
__device__ __forceinline__ uint2 load_at8(const uint8_t* p, uint32_t v) {
  return __ldg(reinterpret_cast<const uint2*>(p) + v);
}
__device__ __forceinline__ uint4 load_at16(const uint8_t* p, uint32_t v) {
  return __ldg(reinterpret_cast<const uint4*>(p) + v);
}
template <int BYTES>
__device__ __forceinline__ void prefetch_at(const uint8_t* p, uint32_t v) {
  prefetch_l2(p + (uint64_t)BYTES * v);
}
__device__ __forceinline__ void copy_at4(uint32_t saddr, const uint8_t* p, uint32_t v) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(saddr), "l"(p + 4ull * v));
}

// Bytes of vector v past the chunk's last whole vector.
__device__ __forceinline__ void store_partial(uint8_t* dst, const uint8_t* base, uint32_t v,
                                              uint32_t nb, const uint32_t x[4]) {
  for (uint32_t k = v * 16; k < nb; k++) {
    const uint32_t i = k - v * 16;
    const uint32_t w = i < 8 ? (i < 4 ? x[0] : x[1]) : (i < 12 ? x[2] : x[3]);
    uint32_t byte = (w >> (8 * (i & 3))) & 0xFFu;
    if (base) byte ^= base[k];
    dst[k] = (uint8_t)byte;
  }
}

// The loops read the raw groups (and a delta's base) straight from global
// memory, each thread a few vectors ahead: too few bytes in flight per SM to
// cover DRAM latency.  Step k of an item consumes vectors [kT + t_lo, kT +
// t_hi), a contiguous slice of every raw group and of the base; the slices of
// the first steps, up to the CTA's share (pf_bytes) of an L2 budget, are
// requested into L2 by the warps that have nothing to do while warp 0 sets the
// item up (an item earlier is too early: the output written meanwhile evicts
// them), and the loops keep requesting kAhead steps ahead of themselves.  (Line
// prefetches: a bulk prefetch costs its thread some 500 cycles, which a divided
// chunk's many short slices made the longest phase of a small call.)
constexpr uint32_t kAhead = 8;
template <int NT>
__device__ __forceinline__ void prefetch_slices(const uint8_t* p, uint32_t vec_bytes, uint32_t T,
                                                uint32_t t_lo, uint32_t Tp, uint32_t steps) {
  const uint32_t i0 = threadIdx.x - 32u;  // (warps 1 on)
  if (Tp == T) {  // an undivided chunk's steps are one run of bytes
    const uint32_t n = steps * T * vec_bytes;
    for (uint32_t o = i0 * 128u; o < n; o += (NT - 32u) * 128u) prefetch_l2(p + o);
  } else {
    const uint32_t lines = (Tp * vec_bytes + 127u) / 128u;
    for (uint32_t i = i0; i < steps * lines; i += NT - 32u) {
      const uint32_t k = i / lines, l = i - k * lines;
      prefetch_l2(p + (k * T + t_lo) * vec_bytes + l * 128u);
    }
  }
}
template <int DT, int NT>
__device__ __forceinline__ void prefetch_window(const Smem& S, uint32_t parts, uint32_t pf_bytes) {
  constexpr int G = Traits<DT>::G;
  const Job& J = S.job;
  const uint64_t off0 = S.chunk * J.chunk_bytes;
  const uint32_t nb = (uint32_t)min((uint64_t)J.chunk_bytes, J.nbytes - off0);
  const uint32_t T = J.lanes, kfull = (nb / 16u) / T;
  const uint32_t t_lo = T * S.part / parts, Tp = T * (S.part + 1u) / parts - t_lo;
  const uint64_t P = kHdrBytes + (uint64_t)J.n_chunks * G * kEntryBytes;
  const uint64_t avail = J.stream_bytes > P ? J.stream_bytes - P : 0;
  uint32_t rawm = 0;
#pragma unroll
  for (int g = 0; g < G; g++) {
    const uint4 e = S.entry[g];
    const uint64_t po = (uint64_t)e.x | ((uint64_t)e.y << 32);
    if ((e.w & 0xFFu) == kRaw && po <= avail && e.z <= avail - po &&
        (uint64_t)e.z >= (uint64_t)kfull * T * (16u / G))
      rawm |= 1u << g;
  }
  const uint32_t per_step = ((uint32_t)__popc(rawm) * (16u / G) + (J.base ? 16u : 0u)) * Tp;
  if (per_step == 0) return;
  const uint32_t steps = min(max(pf_bytes / per_step, 2u), kfull);
#pragma unroll
  for (int g = 0; g < G; g++) {
    if (!((rawm >> g) & 1u)) continue;
    const uint64_t po = (uint64_t)S.entry[g].x | ((uint64_t)S.entry[g].y << 32);
    prefetch_slices<NT>(J.src + P + po, 16u / G, T, t_lo, Tp, steps);
  }
  if (J.base) prefetch_slices<NT>(J.base + off0, 16u, T, t_lo, Tp, steps);
}

// Raw-word ring of the FP32 loop: kRingBytes of shared memory per thread hold
// the three raw groups' words of the next kRingSteps steps of its sub-stream,
// so that many steps of loads are in flight per thread without holding
// registers.
constexpr uint32_t kRingBytes = 64;
constexpr uint32_t kRingSteps = 4;

// Loop for the dominant chunk layout: group 0 HUFF and staged, every other
// group raw, zero or constant, no base.  Thread t decodes NS interleaved
// sub-streams in lockstep (t and t + nthr, ...: instruction-level parallelism;
// a thread without a second one decodes its first twice); every vector is 16 B
// of output: V/4 quads, the raw groups' words (16-bit: loaded two steps ahead
// into alternating register sets; FP32: from the thread's ring), bit-select
// merge with the rotated exponent symbols, a 16-B store.  The chunk's whole
// steps carry no bounds tests; the vectors of a ragged chunk past them follow
// as one more step.  In an even chunk each sub-stream must end exactly where
// the next one starts (the last one within the bitstream); a mismatch flags
// the chunk as corrupt.
template <int DT, int NS, int NT>
__device__ __forceinline__ void decode_weights(const Smem& S, uint32_t lut, uint32_t rings,
                                               uint32_t* err, uint32_t t_a, uint32_t t_b) {
  constexpr int G = Traits<DT>::G, V = Traits<DT>::V, VW = V / 4;
  constexpr int RW = DT == ZIPNN_FP32 ? 3 : (DT == ZIPNN_U8 ? 1 : 2);
  constexpr bool RING = DT == ZIPNN_FP32;
  static_assert(!RING || NS == 1, "the raw-word ring serves one sub-stream per thread");
  constexpr uint32_t nthr = NT;
  const uint32_t tid = threadIdx.x;
  const ChunkInfo& CI = S.ci;
  const Item& it = S.it;
  const uint32_t T = it.T, nvec = it.nvec, kfull = it.kfull;
  const uint32_t starts = CI.at_starts[0];
  Source<kStaged> src;
  src.base = CI.at_words[0];
  src.end = CI.end[0];
  const uint32_t nbits = CI.nwords[0] * 32u, first = CI.first[0];
  const bool pairs = CI.pairs & 1u;
  uint32_t rawm = 0;
  uint32_t cw[G];
#pragma unroll
  for (int g = 1; g < G; g++) {
    cw[g] = CI.value[g] * 0x01010101u;  // ZERO groups carry value 0
    if (CI.mode[g] == kRaw) rawm |= 1u << g;
  }
  uint8_t* const dst = to_global(it.dst);
  const uint8_t* rawp[RW];  // 16-bit: the raw group; FP32: the three of them
#pragma unroll
  for (int q = 0; q < RW; q++)
    rawp[q] = it.src + CI.payload[DT == ZIPNN_FP32 ? (q + 1) % G : 1 % G];
  const uint32_t ring = rings + tid * 4u, rstride = nthr * 4u;
  // lanes whose raw words start a 128-B line (of a warp's slice) prefetch it
  const bool pfl = (tid & (DT == ZIPNN_FP32 ? 31u : 15u)) == 0 && rawm;
  uint32_t bad = 0;
  for (uint32_t t0 = t_a + tid; t0 < t_b; t0 += NS * nthr) {
    Bits r[NS];
    uint32_t v[NS];                   // the sub-streams' current vectors
    uint32_t ra[NS][RW], rb[NS][RW];  // 16-bit: raw words of the next two vectors
    auto load16 = [&](uint32_t (&w)[RW], uint32_t vv) {
      if (DT == ZIPNN_BF16) {
        if (rawm) {
          const uint2 x = load_at8(rawp[0], vv);
          w[0] = x.x;
          w[1 % RW] = x.y;
        } else {
          w[0] = w[1 % RW] = cw[1 % G];
        }
      }
    };
    // FP32: raw words of step k (vector vv) into ring slot k mod kRingSteps
    // (always one commit group per step, empty past the end, so that step k
    // has landed when at most kRingSteps - 1 groups are pending)
    auto issue = [&](uint32_t vv, uint32_t k) {
      if (vv < nvec) {
        const uint32_t sl = k & (kRingSteps - 1u);
#pragma unroll
        for (int q = 0; q < 3; q++)
          if ((rawm >> (q + 1)) & 1u) copy_at4(ring + (sl * 3u + q) * rstride, rawp[q % RW], vv);
      }
      cp_async_commit();
    };
#pragma unroll
    for (int j = 0; j < NS; j++) {
      const uint32_t t = t0 + j * nthr < t_b ? t0 + j * nthr : t0;
      v[j] = t;
      uint32_t start = t ? lds32v(starts + 4u * (t - 1)) : 0u;
      if (start - first > nbits - first) {
        bad = kBad;
        start = nbits;
      }
      bits_init(r[j], src, start);
      if constexpr (!RING) {
        if (t < nvec) load16(ra[j], t);
        if (t + T < nvec) load16(rb[j], t + T);
      }
    }
    if constexpr (RING) {
#pragma unroll
      for (uint32_t k = 0; k < kRingSteps; k++) issue(v[0] + k * T, k);
    }
    // the next vector's symbols of every sub-stream
    auto symbols = [&](uint32_t (&ex)[NS][VW]) {
      if (pairs) {
#pragma unroll
        for (int q = 0; q < VW; q++)
#pragma unroll
          for (int j = 0; j < NS; j++) ex[j][q] = quad_pairs(r[j], src, lut, bad);
      } else {
#pragma unroll
        for (int q = 0; q < VW; q++)
#pragma unroll
          for (int j = 0; j < NS; j++) ex[j][q] = quad_singles(r[j], src, lut, bad);
      }
    };
    auto take_ring = [&](uint32_t k, uint32_t (&rw)[RW]) {
      cp_async_wait<kRingSteps - 1>();
      const uint32_t sl = k & (kRingSteps - 1u);
#pragma unroll
      for (int q = 0; q < 3; q++)
        rw[q % RW] = ((rawm >> (q + 1)) & 1u) ? lds32v(ring + (sl * 3u + q) * rstride) : cw[(q + 1) % G];
    };
    auto merge = [&](const uint32_t (&ex)[VW], const uint32_t (&rw)[RW], uint32_t (&x)[4]) {
      if constexpr (DT == ZIPNN_FP32) {
        merge32r(ex[0], rw[0], rw[1], rw[2], x);
      } else if constexpr (DT == ZIPNN_U8) {
        x[0] = ex[0]; x[1] = ex[1]; x[2] = ex[2]; x[3] = ex[3];
      } else {
        merge16r(ex[0], rw[0], x[0], x[1]);
        merge16r(ex[1 % VW], rw[1 % RW], x[2], x[3]);
      }
    };
    auto vec = [&](uint32_t k, uint32_t (&rr)[NS][RW]) {
      uint32_t ex[NS][VW];
      symbols(ex);
      if constexpr (RING) take_ring(k, rr[0]);
#pragma unroll
      for (int j = 0; j < NS; j++) {
        uint32_t x[4];
        merge(ex[j], rr[j], x);
        if constexpr (!RING) {
          if (v[j] + 2u * T < nvec) load16(rr[j], v[j] + 2u * T);
          if (DT == ZIPNN_BF16 && pfl && v[j] + kAhead * T < nvec)
            prefetch_at<8>(rawp[0], v[j] + kAhead * T);
        } else if (pfl && v[j] + kAhead * T < nvec) {
#pragma unroll
          for (int q = 0; q < 3; q++)
            if ((rawm >> (q + 1)) & 1u) prefetch_at<4>(rawp[q % RW], v[j] + kAhead * T);
        }
        store_vec(dst, v[j], x[0], x[1], x[2], x[3]);
        if constexpr (RING) issue(v[j] + kRingSteps * T, k + kRingSteps);  // its slot was consumed
        v[j] += T;
      }
    };
    uint32_t k = 0;
    for (; k + 1 < kfull; k += 2) {
      vec(k, ra);
      vec(k + 1, rb);
    }
    if (k < kfull) {
      vec(k, ra);
#pragma unroll
      for (int j = 0; j < NS; j++)
#pragma unroll
        for (int q = 0; q < RW; q++) ra[j][q] = rb[j][q];
    }
    if (it.even) {
#pragma unroll
      for (int j = 0; j < NS; j++) {
        const uint32_t end = bits_end(r[j], src), t = v[j] - kfull * T;
        if (t + 1u < T ? end != lds32v(starts + 4u * t) : end > nbits) bad = kBad;
      }
    } else if (v[0] < nvec || v[NS - 1] < nvec) {
      // the vectors past the whole steps, at most one per sub-stream
      uint32_t ex[NS][VW];
      symbols(ex);
      if constexpr (RING) take_ring(kfull, ra[0]);
#pragma unroll
      for (int j = 0; j < NS; j++) {
        uint32_t x[4];
        merge(ex[j], ra[j], x);
        if ((v[j] + 1u) * 16u <= it.nb) store_vec(dst, v[j], x[0], x[1], x[2], x[3]);
        else if (v[j] < nvec) store_partial(it.dst, nullptr, v[j], it.nb, x);
      }
    }
    if constexpr (RING) cp_async_wait<0>();
  }
  if (bad & kBad) atomicOr(err, 1u);
}

// Loop for every other layout: any mix of coded (HUFF or SPARSE), raw, zero
// and constant groups, with or without a base, the coded payloads read as WH
// says, one sub-stream per thread at a time.  The mode
// tests are uniform over the chunk.  Raw words and the base arrive one step
// ahead in registers, from L2 when the item's prefetch window covers them.  In
// SPARSE groups only the lanes whose vector's bitmap bit is set decode.
template <int DT, int WH, int NT>
__device__ __forceinline__ void decode_general(const Smem& S, uint32_t* err, uint32_t t_a,
                                               uint32_t t_b) {
  constexpr int G = Traits<DT>::G, V = Traits<DT>::V, VW = V / 4;
  const uint32_t tid = threadIdx.x;
  const ChunkInfo& CI = S.ci;
  const Item& it = S.it;
  const uint32_t nthr = WH == kRinged ? CI.ring_threads : (uint32_t)NT;
  if (WH == kRinged && tid >= nthr) return;
  const uint32_t T = it.T;
  const uint32_t coded = CI.coded, pairs = CI.pairs;
  // (what the loop needs of the records, in registers)
  uint32_t rawm = 0, sparse = 0;
  uint32_t cw[G], lut[G], bmp[G];
  const uint8_t* rawp[G];
#pragma unroll
  for (int g = 0; g < G; g++) {
    if (CI.mode[g] == kRaw) rawm |= 1u << g;
    if (CI.mode[g] == kSparse) sparse |= 1u << g;
    cw[g] = CI.value[g] * 0x01010101u;
    lut[g] = CI.lut[g];
    bmp[g] = WH == kStaged ? CI.at_bm[g] : CI.bmo[g];
    rawp[g] = it.src + CI.payload[g];
  }
  uint8_t* const dst = to_global(it.dst);
  const uint8_t* const base8 = it.base;
  const uint32_t nvec = it.nvec, nb = it.nb;
  // lanes whose raw words / base vectors start a 128-B line prefetch it
  const bool pfr = rawm && (tid & (G == 4 ? 31u : (G == 2 ? 15u : 7u))) == 0;
  const bool pfb = base8 && (tid & 7u) == 0;
  // end positions are checked in even chunks of one coded group in front, or
  // two 16-bit ones
  const bool check = it.even && (G <= 2 || coded == 1u);
  uint32_t bad = 0;
  Source<WH> src[G];
  // words of coded group g's bitmap and start-bit table
  auto word_at = [&](int g, uint32_t at) -> uint32_t {
    if constexpr (WH == kStaged) return lds32v(at);
    else return rd_u32(rawp[g] + at);
  };
  auto start_of = [&](int g, uint32_t t) -> uint32_t {
    return word_at(g, (WH == kStaged ? CI.at_starts[g] : CI.offs[g]) + 4u * (t - 1u));
  };
#pragma unroll
  for (int g = 0; g < G; g++) {
    if (!((coded >> g) & 1u)) continue;
    if constexpr (WH == kStaged) {
      src[g].base = CI.at_words[g];
      src[g].end = CI.end[g];
    } else if constexpr (WH == kDirect) {
      src[g].words = rawp[g] + CI.bs[g];
      src[g].n = CI.nwords[g];
    } else {
      const uint32_t slots = CI.ring_slots;
      src[g].pay = rawp[g];
      src[g].bs = CI.bs[g] / 4u;
      src[g].pieces = (CI.bs[g] + 4u * CI.nwords[g] + 15u) / 16u;
      src[g].stride = nthr * 16u;
      src[g].mask = slots - 1u;
      src[g].ring = CI.stage + __popc(coded & ((1u << g) - 1u)) * slots * nthr * 16u + tid * 16u;
    }
  }
  for (uint32_t t = t_a + tid; t < t_b; t += nthr) {
    Bits r[G];
    uint32_t raw[G][VW];
    uint4 bb = make_uint4(0, 0, 0, 0);
    auto load_raw = [&](uint32_t v) {
#pragma unroll
      for (int g = 0; g < G; g++) {
        if (!((rawm >> g) & 1u)) continue;
        const uint8_t* p = rawp[g];
        if constexpr (V == 8) {
          const uint2 x = load_at8(p, v);
          raw[g][0] = x.x; raw[g][1 % VW] = x.y;
        } else if constexpr (V == 4) {
          raw[g][0] = load_at4(p, v);
        } else {
          const uint4 x = load_at16(p, v);
          raw[g][0] = x.x; raw[g][1 % VW] = x.y; raw[g][2 % VW] = x.z; raw[g][3 % VW] = x.w;
        }
      }
      if (base8 && (v + 1u) * 16u <= nb) bb = load_at16(base8, v);
    };
#pragma unroll
    for (int g = 0; g < G; g++) {
      if (!((coded >> g) & 1u)) continue;
      uint32_t start = t ? start_of(g, t) : 0u;
      if (start > CI.nwords[g] * 32u || (WH == kStaged && start < CI.first[g])) {
        bad = kBad;
        start = CI.nwords[g] * 32u;
      }
      bits_init(r[g], src[g], start);
    }
    if (t < nvec) load_raw(t);
    for (uint32_t v = t; v < nvec; v += T) {
      const uint32_t va = v + kAhead * T;
      if (pfb && va < nvec) prefetch_at<16>(base8, va);
      if (pfr && va < nvec) {
#pragma unroll
        for (int g = 0; g < G; g++)
          if ((rawm >> g) & 1u) prefetch_at<V>(rawp[g], va);
      }
      if constexpr (WH == kRinged) {
#pragma unroll
        for (int g = 0; g < G; g++)
          if ((coded >> g) & 1u) src[g].template refill<V>(r[g].nx);
        cp_async_commit();
        cp_async_wait<kRingPending>();
      }
      uint32_t gw[G][VW];
#pragma unroll
      for (int g = 0; g < G; g++)
#pragma unroll
        for (int q = 0; q < VW; q++)
          gw[g][q] = ((rawm >> g) & 1u) ? raw[g][q] : cw[g];
      const uint4 b = bb;
      if (v + T < nvec) load_raw(v + T);
      if (DT != ZIPNN_U8 && !(coded & 1u)) {
#pragma unroll
        for (int q = 0; q < VW; q++) gw[0][q] = rot4(gw[0][q]);
      }
#pragma unroll
      for (int g = 0; g < G; g++) {
        if (!((coded >> g) & 1u)) continue;
        if (((sparse >> g) & 1u) && !((word_at(g, bmp[g] + 4u * (v >> 5)) >> (v & 31u)) & 1u)) {
#pragma unroll
          for (int q = 0; q < VW; q++) gw[g][q] = 0;
        } else if ((pairs >> g) & 1u) {
#pragma unroll
          for (int q = 0; q < VW; q++) gw[g][q] = quad_pairs(r[g], src[g], lut[g], bad);
        } else {
#pragma unroll
          for (int q = 0; q < VW; q++) gw[g][q] = quad_singles(r[g], src[g], lut[g], bad);
        }
      }
      uint32_t x[4];
      if constexpr (DT == ZIPNN_FP32) {
        merge32r(gw[0][0], gw[1 % G][0], gw[2 % G][0], gw[3 % G][0], x);
      } else if constexpr (DT == ZIPNN_U8) {
        x[0] = gw[0][0]; x[1] = gw[0][1 % VW]; x[2] = gw[0][2 % VW]; x[3] = gw[0][3 % VW];
      } else {
        merge16r(gw[0][0], gw[1 % G][0], x[0], x[1]);
        merge16r(gw[0][1 % VW], gw[1 % G][1 % VW], x[2], x[3]);
      }
      if ((v + 1u) * 16u <= nb) {
        store_vec(dst, v, x[0] ^ b.x, x[1] ^ b.y, x[2] ^ b.z, x[3] ^ b.w);
      } else {
        store_partial(it.dst, base8, v, nb, x);
      }
    }
    if constexpr (WH == kRinged) cp_async_wait<0>();  // before the ring is used again
    if (check) {
#pragma unroll
      for (int g = 0; g < G; g++) {
        if (!((coded >> g) & 1u)) continue;
        const uint32_t end = bits_end(r[g], src[g]);
        if (t + 1u < T ? end != start_of(g, t + 1u) : end > CI.nwords[g] * 32u)
          bad = kBad;
      }
    }
  }
  if (bad & kBad) atomicOr(err, 1u);
}

// Set-up of the next item (S.job, S.chunk, S.part, S.entry) by warp 0: its
// record, placement of tables and payloads, the bulk copies, table bytes and
// canonical limits, into S.it, S.ci and S.tab.
template <int DT, int NT, bool RINGED, bool DIRECT>
__device__ __forceinline__ void setup_item(Smem& S, uint32_t parts, uint32_t lut0, uint32_t ntab,
                                           uint32_t stage_cap, uint32_t ring_bytes, uint64_t* bar,
                                           uint32_t extra_tx) {
  constexpr int G = Traits<DT>::G, V = Traits<DT>::V, ES = 16 / V;
  const uint32_t lane = threadIdx.x & 31u;
  const Job& J = S.job;
  const uint8_t* cont = J.src;
  const uint64_t off0 = S.chunk * J.chunk_bytes;
  const uint32_t nb = (uint32_t)min((uint64_t)J.chunk_bytes, J.nbytes - off0), m = nb / ES;
  const uint32_t T = J.lanes, nvec = (nb + 15u) / 16u, part = S.part;
  const uint64_t P = kHdrBytes + (uint64_t)J.n_chunks * G * kEntryBytes;
  const uint64_t avail = J.stream_bytes > P ? J.stream_bytes - P : 0;
  ChunkInfo& CI = S.ci;
  if (lane == 31) {
    Item& it = S.it;
    it.src = cont;
    it.dst = J.dst + off0;
    it.base = J.base ? J.base + off0 : nullptr;
    it.nb = nb;
    it.nvec = nvec;
    it.T = T;
    it.t_lo = T * part / parts;
    it.t_hi = T * (part + 1u) / parts;
    it.kfull = (nb / 16u) / T;
    it.even = nb == J.chunk_bytes && nvec % T == 0;
    it.part = part;
  }
  // the map entry of group `lane`
  const uint4 e = lane < (uint32_t)G ? S.entry[lane] : make_uint4(0, 0, 0, 0);
  const uint64_t po = (uint64_t)e.x | ((uint64_t)e.y << 32), pay = P + po;
  const uint32_t size = e.z, mode = e.w & 0xFFu;
  bool bad = lane < (uint32_t)G &&
             ((e.w >> 16) != 0 || mode > kSparse || po > avail || align_up(size, 16) > avail - po ||
              (po & 15) || (mode == kRaw && size != m) ||
              ((mode == kZero || mode == kConst) && size != 0) || (coded_mode(mode) && size < 12));
  if (__any_sync(0xffffffffu, bad)) {
    if (lane == 0) {
      CI.coded = 0;
      CI.pairs = 0;
      CI.stage_bytes = 0;
      CI.bad = 1;
    }
    return;
  }
  const bool mine = lane < (uint32_t)G && coded_mode(mode);
  const uint32_t coded = __ballot_sync(0xffffffffu, mine), nhuff = (uint32_t)__popc(coded);
  // placement: the first ntab coded groups' tables in their slots, the others
  // at the start of the stage (with the raw-word rings behind it, which only
  // chunks with one coded group use); behind them the payloads, whole or slice
  // by slice (stage_slice), or the readers' rings
  const uint32_t extra = nhuff > ntab ? (nhuff - ntab) * kLutBytes : 0u;
  const uint32_t cap = stage_cap + (nhuff > 1 ? ring_bytes : 0u), stage0 = lut0 + ntab * kLutBytes;
  const uint32_t room = cap > extra ? cap - extra : 0u;  // (always: the launch sizes the stage so)
  uint64_t before = 0, total = 0;
#pragma unroll
  for (int g = 0; g < G; g++) {
    const uint64_t s = __shfl_sync(0xffffffffu, mine ? align_up(size, 16) : 0ull, g);
    if ((uint32_t)g < lane) before += s;
    total += s;
  }
  const bool fits = total + 32u <= room;
  // (DIRECT: what does not take the weight loop is read from global memory)
  const bool direct = DIRECT && !(coded == 1u && (S.entry[0].w & 0xFFu) == kHuff);
  const uint32_t at = stage0 + extra + (uint32_t)before;
  if (lane < (uint32_t)G) {
    const uint32_t k = (uint32_t)__popc(coded & ((1u << lane) - 1u));
    CI.mode[lane] = mode;
    CI.value[lane] = (e.w >> 8) & 0xFFu;
    CI.size[lane] = size;
    CI.payload[lane] = pay;
    CI.lut[lane] = k < ntab ? lut0 + k * kLutBytes : stage0 + (k - ntab) * kLutBytes;
  }
  const bool copy = !RINGED && fits && nhuff && !direct;
  if (copy) {
    if (lane == 0) mbar_expect_tx(bar, (uint32_t)total + extra_tx);
    __syncwarp();
    if (mine) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bulk_g2s(at, cont + pay, (uint32_t)align_up(size, 16), bar);
    }
  }
  // table bytes (word loads, clamped to the payload) and canonical limits:
  // lane l holds the number of codes of length l; with A(l) = count(l) <<
  // (12 - l), the left-justified end of the codes of length l is the sum of
  // A(1..l) and their first code the sum of A(1..l-1) >> (12 - l)
  uint32_t pairs = 0;
#pragma unroll
  for (int g = 0; g < G; g++) {
    if (!((coded >> g) & 1u)) continue;
    GroupTab& t = S.tab[g];
    const uint32_t sz = __shfl_sync(0xffffffffu, size, g);
    const uint8_t* q = cont + __shfl_sync(0xffffffffu, pay, g);
    const uint32_t i1 = lane + 32u, i2 = lane + 64u;
    const uint32_t b0 = 4u * lane + 4u <= sz ? rd_u32(q + 4u * lane) : 0u;
    const uint32_t b1 = 4u * i1 + 4u <= sz ? rd_u32(q + 4u * i1) : 0u;
    const uint32_t b2 = i2 < 68u && 4u * i2 + 4u <= sz ? rd_u32(q + 4u * i2) : 0u;
    t.words[lane] = b0;
    t.words[i1] = b1;
    if (i2 < 68u) t.words[i2] = b2;
    const uint32_t cword = __shfl_sync(0xffffffffu, b0, ((lane - 1u) >> 2) & 3u);
    const bool is_len = lane >= 1u && lane <= (uint32_t)kMaxLen;
    const uint32_t cl = is_len ? (cword >> (8u * ((lane - 1u) & 3u))) & 0xFFu : 0u;
    const uint32_t A = is_len ? cl << (kMaxLen - lane) : 0u;
    uint32_t lim = A, idx = cl;
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, lim, o), y = __shfl_up_sync(0xffffffffu, idx, o);
      if (lane >= (uint32_t)o) {
        lim += x;
        idx += y;
      }
    }
    if (is_len) {
      t.lim[lane] = lim;
      t.rank[lane] = (idx - cl) - ((lim - A) >> (kMaxLen - lane));
    }
    const uint32_t kraft = __shfl_sync(0xffffffffu, lim, kMaxLen);
    uint32_t nz = __shfl_sync(0xffffffffu, idx, kMaxLen);
    if (nz == 0) {  // 256 codes of 8 bits, whose count is stored as 0? (then the symbols are 0..255)
      auto flat = [](uint32_t i) { return i < 3u ? 0u : 0x03020100u + 0x04040404u * (i - 3u); };
      if (__all_sync(0xffffffffu, b0 == flat(lane) && b1 == flat(i1) && (i2 > 66u || b2 == flat(i2)))) {
        nz = 256;
        if (is_len && lane >= 8u) t.lim[lane] = (uint32_t)kLutSize;
      }
    }
    // windows that hold two whole codes: for a first code of length l, the
    // codes of at most 12 - l bits
    const uint32_t rest = __shfl_sync(0xffffffffu, lim, (kMaxLen - lane) & 31u);
    uint32_t w2 = is_len && lane < (uint32_t)kMaxLen && kraft <= (uint32_t)kLutSize ? A * rest : 0u;
#pragma unroll
    for (int o = 8; o; o >>= 1) w2 += __shfl_xor_sync(0xffffffffu, w2, o);
    if (__shfl_sync(0xffffffffu, w2, 1) >= kPairMin) pairs |= 1u << g;
    const uint32_t h = (uint32_t)align_up(12 + nz, 4);
    // SPARSE: the vector bitmap (one bit per 16-byte vector of the chunk)
    // sits between the table and the start-bit table
    const uint32_t bmb = __shfl_sync(0xffffffffu, mode, g) == kSparse ? 4u * ((nb + 511u) / 512u) : 0u;
    const uint32_t hdr = h + bmb + 4u * (T - 1u);
    if (nz < 2 || nz > 256 || kraft > (uint32_t)kLutSize || sz < hdr || (sz - hdr) % 4) {
      bad = true;
    } else if (lane == (uint32_t)g) {
      const uint32_t nw = (sz - hdr) / 4u;
      CI.bmo[g] = h;
      CI.offs[g] = h + bmb;
      CI.bs[g] = hdr;
      CI.nwords[g] = nw;
      CI.at_bm[g] = at + h;
      CI.at_starts[g] = at + h + bmb;
      CI.at_words[g] = at + hdr;
      CI.end[g] = at + hdr + 4u * (nw + 4u);
      CI.first[g] = 0;
    }
  }
  uint32_t slots = 0, threads = 0;
  if (RINGED && nhuff) {  // rings for as many of the threads as there is room for
    for (uint32_t th = NT; th >= 32u && !slots; th /= 2)
      for (uint32_t sl = kRingSlotsMax; sl >= ring_slots_min<V>() && !slots; sl /= 2)
        if (nhuff * sl * th * 16u <= room) {
          slots = sl;
          threads = th;
        }
    if (!slots) bad = true;  // cannot happen with the launch's sizing
  }
  bad = __any_sync(0xffffffffu, bad);
  if (lane == 0) {
    CI.coded = coded;
    CI.pairs = pairs;
    CI.stage = stage0 + extra;
    CI.stage_bytes = copy ? (uint32_t)total : (RINGED ? 0u : room);
    CI.sliced = !RINGED && nhuff && !fits && !direct;
    if (DIRECT) CI.direct = direct;
    CI.ring_slots = slots;
    CI.ring_threads = nhuff ? threads : (uint32_t)NT;
    CI.bad = bad ? 1u : 0u;
  }
}

// Payloads that do not fit the stage (FP16 holding BF16 values, 1 MiB chunks):
// the sub-streams from t_a on are decoded slice by slice, each with its own
// part of the start-bit tables and bitstreams in the stage (the sub-streams
// follow one another in the bitstream) and with the bitmaps of SPARSE groups.
// Thread 0: picks the slice [t_a, t_b), as many sub-streams as fit of the rest, its
// half, its quarter ..., requests its bytes and sets the addresses; returns t_b, or 0
// if not one fits (a launch has a stage for the longest one that a valid container
// can hold).
template <int DT>
__device__ __noinline__ uint32_t stage_slice(Smem& S, uint32_t t_a, uint64_t* bar) {
  constexpr int G = Traits<DT>::G;
  const Item& it = S.it;
  ChunkInfo& CI = S.ci;
  for (uint32_t n = it.t_hi - t_a;; n = (n + 1u) / 2u) {
    const uint32_t t_b = t_a + n, T = it.T;
    // pass 0 counts the bytes, pass 1 requests them
    uint32_t total = 0;
    for (int pass = 0; pass < 2; pass++) {
      uint32_t to = CI.stage;
      auto piece = [&](int g, uint32_t lo, uint32_t hi) -> uint32_t {  // address of byte 0
        lo &= ~15u;
        hi = min((hi + 15u) & ~15u, (uint32_t)align_up(CI.size[g], 16));
        const uint32_t len = hi > lo ? hi - lo : 0u, at = to - lo;
        if (pass && len) bulk_g2s(to, it.src + CI.payload[g] + lo, len, bar);
        to += len;
        return at;
      };
      for (int g = 0; g < G; g++) {
        if (!((CI.coded >> g) & 1u)) continue;
        const uint8_t* p = it.src + CI.payload[g];
        const uint32_t nbits = CI.nwords[g] * 32u;
        const uint32_t s0 = t_a ? min(rd_u32(p + CI.offs[g] + 4u * (t_a - 1u)), nbits) : 0u;
        const uint32_t s1 = t_b < T ? min(rd_u32(p + CI.offs[g] + 4u * (t_b - 1u)), nbits) : nbits;
        const uint32_t w0 = s0 / 32u, w1 = max(s1 / 32u + 2u, w0 + 2u);
        if (CI.mode[g] == kSparse) CI.at_bm[g] = piece(g, CI.bmo[g], CI.offs[g]) + CI.bmo[g];
        CI.at_starts[g] = piece(g, CI.offs[g] + 4u * (t_a ? t_a - 1u : 0u), CI.offs[g] + 4u * min(t_b, T - 1u)) +
                          CI.offs[g];
        CI.at_words[g] = piece(g, CI.bs[g] + 4u * w0, CI.bs[g] + 4u * w1) + CI.bs[g];
        CI.end[g] = CI.at_words[g] + 4u * (w1 + 3u);
        CI.first[g] = 32u * w0;
      }
      total = to - CI.stage;
      if (pass == 0) {
        if (total + 32u > CI.stage_bytes && n > 1u) break;
        if (total + 32u > CI.stage_bytes) {  // one sub-stream too long: corrupt starts
          return 0;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(bar, total);
      } else {
        return t_b;
      }
    }
  }
}

// Tables of the coded groups, in two passes.  Pass 1, first codes: the length
// of the code at window w is one more than the limits lim[1..11] that w
// reaches.  Codes of at most 8 bits cover aligned runs of 16 windows, so a
// thread finds one code per run and stores its 16 entries as four vectors (in
// an order rotated by lane, which spreads them over the banks); the windows of
// longer codes, from lim[8] on, are few and done one by one.  Pass 2 (groups
// with pairs): the second code is the first code of window (w << l) & 4095
// (the remaining 12 - l bits, zero-filled), kept when it fits in them; loads
// are issued in batches so that their latencies overlap.  Pass 2 reads entries
// that other threads are turning into pairs; a pair keeps the first code's
// symbol and length where pass 2 reads them, so either value serves.
template <int DT, int NT>
__device__ __forceinline__ void first_codes(const Smem& S) {
  constexpr int G = Traits<DT>::G;
  const uint32_t tid = threadIdx.x;
#pragma unroll
  for (int g = 0; g < G; g++) {
    if (!((S.ci.coded >> g) & 1u)) continue;
    const GroupTab& t = S.tab[g];
    const uint8_t* syms = reinterpret_cast<const uint8_t*>(t.words) + 12;
    const uint32_t L = S.ci.lut[g];
    auto entry = [&](uint32_t w, uint32_t l) -> uint32_t {
      uint32_t s = syms[(t.rank[l] + (w >> (kMaxLen - l))) & 255u];
      if (DT != ZIPNN_U8 && g == 0) s = ((s >> 1) | (s << 7)) & 0xFFu;
      return kOne | (s << 16) | (l << 8) | l;
    };
    const uint32_t lim8 = t.lim[8];
    for (uint32_t w = 16u * tid; w < lim8; w += 16u * NT) {
      uint32_t l = 1;
#pragma unroll
      for (int i = 1; i < 8; i++) l += w >= t.lim[i];
      const uint32_t e = entry(w, l);
#pragma unroll
      for (uint32_t q = 0; q < 4; q++)
        sts128(L + 4u * w + 16u * ((q + (tid >> 1)) & 3u), e);
    }
    for (uint32_t w = lim8 + tid; w < (uint32_t)kLutSize; w += NT) {
      uint32_t l = 9;
#pragma unroll
      for (int i = 9; i < kMaxLen; i++) l += w >= t.lim[i];
      sts32(L + 4u * w, w < t.lim[kMaxLen] ? entry(w, l) : kOne | kBad | (12u << 8) | 12u);
    }
  }
}
template <int DT, int NT>
__device__ __forceinline__ void second_codes(const Smem& S) {
  constexpr int G = Traits<DT>::G;
  const uint32_t tid = threadIdx.x;
  constexpr int B = kLutSize / NT < 8 ? kLutSize / NT : 8;
#pragma unroll
  for (int g = 0; g < G; g++) {
    if (!((S.ci.pairs >> g) & 1u)) continue;
    const uint32_t L = S.ci.lut[g];
    for (uint32_t w0 = tid; w0 < (uint32_t)kLutSize; w0 += B * NT) {
      uint32_t e[B], e2[B];
#pragma unroll
      for (int i = 0; i < B; i++) e[i] = lds32v(L + 4u * (w0 + i * NT));
#pragma unroll
      for (int i = 0; i < B; i++)
        e2[i] = lds32v(L + 4u * (((w0 + i * NT) << ((e[i] >> 8) & 15u)) & (kLutSize - 1u)));
#pragma unroll
      for (int i = 0; i < B; i++) {
        const uint32_t l = ((e[i] >> 8) & 15u) + ((e2[i] >> 8) & 15u);
        if (!((e[i] | e2[i]) & kBad) && l <= (uint32_t)kMaxLen)
          sts32(L + 4u * (w0 + i * NT), (e[i] & 0x00FF0F00u) | ((e2[i] << 8) & 0xFF000000u) | l);
      }
    }
  }
}

// Kinds of kernel: kWeights for launches of plain tensors (the loop for model
// weights and the general one), kDeltas for launches that hold deltas (the
// general loop alone: sharing the kernel costs it registers), kRings for
// launches whose payloads do not fit the stage (the general loop over rings).
enum Kind { kWeights, kDeltas, kRings };
// FP32 weights: the tables of four coded groups leave next to no stage where three CTAs
// share an SM, so chunks that do not take the weight loop are read from global
// memory.  (256 MiB of 16 values, all groups coded: 647 us; by slices of a few
// sub-streams 3840.  With both forms of the general loop the kernel spills and this
// takes 967; plans have another kernel for such tensors, see decode_config.)
template <int DT, int KIND> constexpr bool kReadsDirect = DT == ZIPNN_FP32 && KIND == kWeights;

template <int DT, int KIND, int NT>
__device__ __noinline__ void decode_general_ool(const Smem& S, uint32_t* err, uint32_t t_a,
                                                uint32_t t_b) {
  decode_general<DT, kReadsDirect<DT, KIND> ? kDirect : kStaged, NT>(S, err, t_a, t_b);
}

// Decode sub-streams [t_a, t_b) of the current item.
template <int DT, int KIND, int NT>
__device__ __forceinline__ void decode_range(const Smem& S, uint32_t lut0, uint32_t rings,
                                             uint32_t* err, uint32_t t_a, uint32_t t_b) {
  if constexpr (KIND == kRings) {
    decode_general<DT, kRinged, NT>(S, err, t_a, t_b);
  } else {
    if constexpr (KIND == kWeights) {
      if (S.ci.coded == 1u && S.ci.mode[0] == kHuff && !S.it.base) {
        if (DT == ZIPNN_BF16 && t_b - t_a > (uint32_t)NT)
          decode_weights<DT, DT == ZIPNN_BF16 ? 2 : 1, NT>(S, lut0, rings, err, t_a, t_b);
        else
          decode_weights<DT, 1, NT>(S, lut0, rings, err, t_a, t_b);
        return;
      }
    }
    if constexpr (KIND == kWeights) decode_general_ool<DT, KIND, NT>(S, err, t_a, t_b);
    else decode_general<DT, kStaged, NT>(S, err, t_a, t_b);
  }
}

// DT: the dtype family of the launch's jobs (BF16 stands for both 16-bit
// types; a batch of several families takes one launch for each).  REGS: 256-thread
// CTAs per SM that the registers are budgeted for: three (80 registers), or two
// (128) where the stage leaves no room for three, where the general loop over
// four groups would spill (what spills misses the 28 KiB of L1 that the shared
// memory leaves), and in the 128-thread kernels of small launches.  (The tables of
// FP32 weights leave room for three of 128 threads at most.)
template <int DT, int KIND, int NT, int REGS>
__global__ void __launch_bounds__(NT, DT == ZIPNN_FP32 && KIND == kWeights ? 3 : REGS * 256 / NT)
k_decode(JobRef jr, uint64_t nchunks_total, uint32_t* __restrict__ err,
         unsigned long long* __restrict__ ticket, uint32_t debug_flags, uint32_t ntab,
         uint32_t stage_cap, uint32_t ring_bytes, uint32_t pf_bytes, uint32_t parts) {
  constexpr int G = Traits<DT>::G;
  extern __shared__ __align__(128) uint8_t dsm[];  // ntab table slots | stage | raw-word rings
  __shared__ Smem S;
  __shared__ uint64_t bar;
  const uint32_t lut0 = smem_u32(dsm);
  const uint32_t rings = lut0 + ntab * kLutBytes + stage_cap;
  // debug flag 1 (tests only): expect 16 bytes more than the bulk copies send,
  // so the wait can only end by its (shortened) limit -> ETIMEOUT
  const uint32_t extra_tx = (debug_flags & 1u) ? 16u : 0u;
  const uint64_t limit_ns = (debug_flags & 1u) ? 100000000ull : kWaitLimitNs;
  const uint32_t tid = threadIdx.x, lane = tid & 31u;
  if (tid == 0) {
    mbar_init(&bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    S.jobno = 0;
    S.job_end = 0;
  }
  __syncthreads();
  uint32_t parity = 0;
  // Taking a work item.  draw (thread 0): its number, from the device queue or
  // by stride.  take (warp 0): its job -- items come in increasing order, so
  // unless it is the job already at hand it is found by scanning forward from
  // there (a few steps; after eight, a search) -- and the request of the
  // chunk's map entries (lane g: group g).  keep (warp 0): the entries, and
  // L2 prefetches of the table bytes.
  auto draw = [&](uint32_t iter) -> uint64_t {
    return ticket ? atomicAdd(ticket, 1ull) : blockIdx.x + (uint64_t)iter * gridDim.x;
  };
  auto take = [&](uint64_t item) -> uint4 {
    item = __shfl_sync(0xffffffffu, item, 0);
    const uint64_t ch = item >> (__ffs(parts) - 1);  // (parts is a power of two)
    const bool last = ch >= nchunks_total;
    if (!last && ch >= S.job_end) {
      int j = (int)S.jobno;
      if (jr.table && lane == 0) {
        int steps = 0;
        while (j + 1 < jr.n && jr.table[j + 1].chunk_begin <= ch && steps < 8) {
          j++;
          steps++;
        }
        if (steps == 8) j += find_job(jr.table + j, jr.n - j, ch);
      }
      j = __shfl_sync(0xffffffffu, j, 0);
      const uint32_t* from = reinterpret_cast<const uint32_t*>(jr.table ? jr.table + j : &jr.one);
      if (lane < sizeof(Job) / 4) reinterpret_cast<uint32_t*>(&S.job)[lane] = from[lane];
      if (lane == 0) {
        S.jobno = (uint32_t)j;
        S.job_end = jr.table && j + 1 < jr.n ? jr.table[j + 1].chunk_begin : nchunks_total;
      }
      __syncwarp();
    }
    if (lane == 0) {
      S.last = last;
      S.chunk = ch - S.job.chunk_begin + S.job.chunk0;
      S.part = (uint32_t)item & (parts - 1u);
    }
    __syncwarp();
    uint4 e = make_uint4(0, 0, 0, 0);
    if (!last && lane < (uint32_t)G)
      e = __ldg(reinterpret_cast<const uint4*>(S.job.src + kHdrBytes + (S.chunk * G + lane) * kEntryBytes));
    return e;
  };
  auto keep = [&](const uint4& e) {
    if (S.last) return;
    if (lane < (uint32_t)G) S.entry[lane] = e;
    const Job& J = S.job;
    const uint64_t P = kHdrBytes + (uint64_t)J.n_chunks * G * kEntryBytes;
    const uint64_t avail = J.stream_bytes > P ? J.stream_bytes - P : 0;
    const uint64_t po = (uint64_t)e.x | ((uint64_t)e.y << 32);
    if (lane < (uint32_t)G && coded_mode(e.w & 0xFFu) && po <= avail && e.z <= avail - po) {
      prefetch_l2(J.src + P + po);
      if (e.z > 128u) prefetch_l2(J.src + P + po + 128u);
    }
  };
  if (tid < 32) keep(take(tid == 0 ? draw(0) : 0ull));
  __syncthreads();
  bool ok = true;
  for (uint32_t iter = 1;; iter++) {
    if (tid < 32) {
      __syncwarp();
      if (!S.last)
        setup_item<DT, NT, KIND == kRings, kReadsDirect<DT, KIND>>(S, parts, lut0, ntab, stage_cap,
                                                                   ring_bytes, &bar, extra_tx);
    } else if (!S.last) {
      prefetch_window<DT, NT>(S, parts, pf_bytes);
    }
    __syncthreads();
    if (S.last) break;
    const bool rejected = S.ci.bad != 0;
    const bool sliced = KIND != kRings && S.ci.sliced;
    const bool copied = KIND != kRings && S.ci.coded && !sliced &&
                        !(kReadsDirect<DT, KIND> && S.ci.direct);
    uint64_t item = 0;
    if (tid == 0) item = draw(iter);  // (needed after the next barrier)
    if (!rejected && S.ci.coded) first_codes<DT, NT>(S);
    __syncthreads();
    uint4 e;
    if (tid < 32) e = take(item);  // (needed after the next barrier)
    if (!rejected && S.ci.pairs) second_codes<DT, NT>(S);
    if (copied) {  // the staged payloads (every thread; bounded)
      if (!mbar_wait(&bar, parity, limit_ns)) atomicOr(&S.ci.bad, 2u);
      parity ^= 1u;
    }
    __syncthreads();
    if (tid < 32) keep(e);
    ok = !(S.ci.bad & 2u);
    if (rejected) {
      if (tid == 0 && S.it.part == 0) atomicOr(err, 1u);
    } else if (ok) {
      uint32_t t_a = S.it.t_lo;
      const uint32_t t_hi = S.it.t_hi;
      while (t_a < t_hi) {
        uint32_t t_b = t_hi;
        if (sliced) {
          if (tid == 0) S.slice_end = stage_slice<DT>(S, t_a, &bar);
          __syncthreads();
          t_b = S.slice_end;
          if (t_b == 0) {
            if (tid == 0) atomicOr(err, 1u);
            break;
          }
          if (!mbar_wait(&bar, parity, limit_ns)) atomicOr(&S.ci.bad, 2u);
          parity ^= 1u;
          __syncthreads();
          ok = !(S.ci.bad & 2u);
          if (!ok) break;
        }
        decode_range<DT, KIND, NT>(S, lut0, rings, err, t_a, t_b);
        t_a = t_b;
        if (sliced) __syncthreads();
      }
    }
    if (!ok) break;
    __syncthreads();
  }
  if (!ok) {
    // A wait gave up (ETIMEOUT).  Before the CTA leaves, drain the copies it
    // issued, so that none of them can still write into this shared memory:
    // thread 0 first cancels the bytes that were expected but never requested
    // (the test-only fault injection), so the phase completes exactly when the
    // real copies have landed; then every thread waits for it, again bounded.
    // Only copies that themselves never finish end this second wait by its
    // limit, and then the drain is best effort.
    if (tid == 0) {
      atomicOr(err, 4u);
      if (extra_tx && !S.ci.sliced) mbar_complete_tx(&bar, extra_tx);
    }
    __syncthreads();
    mbar_wait(&bar, parity ^ 1u, limit_ns);
  }
  // the last CTA to leave resets the work queue for the next launch on the
  // same buffer (ticket[0]: next work item, ticket[1]: CTAs done)
  if (ticket) {
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      if (atomicAdd(ticket + 1, 1ull) == (unsigned long long)gridDim.x - 1ull) {
        atomicExch(ticket, 0ull);
        atomicExch(ticket + 1, 0ull);
      }
    }
  }
}

// Kernel of a dtype family, kind, CTA size and CTAs per SM (`three`: the shared
// memory lets three of 256 threads share an SM), as the handle the runtime's
// launch and attribute calls take.
template <int DT, int KIND>
const void* kernel_of(int threads, bool three) {
  if (threads != 256) return reinterpret_cast<const void*>(k_decode<DT, KIND, 128, 2>);
  if constexpr (DT != ZIPNN_FP32 || KIND == kWeights)
    if (three || DT != ZIPNN_BF16 || KIND == kRings)
      return reinterpret_cast<const void*>(k_decode<DT, KIND, 256, 3>);
  if constexpr ((DT == ZIPNN_BF16 && KIND != kRings) || (DT == ZIPNN_FP32 && KIND != kWeights))
    return reinterpret_cast<const void*>(k_decode<DT, KIND, 256, 2>);
  return nullptr;
}
template <int DT>
const void* kernel_handle(int kind, int threads, bool three) {
  if constexpr (DT != ZIPNN_U8) {  // (U8 payloads seldom fit a stage)
    if (kind == kWeights) return kernel_of<DT, kWeights>(threads, three);
    if (kind == kDeltas) return kernel_of<DT, kDeltas>(threads, three);
  }
  return kernel_of<DT, kRings>(threads, three);
}

}  // namespace
}  // namespace zipnn
