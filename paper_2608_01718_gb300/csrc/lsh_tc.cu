// The SimHash-indexed key check of larger batches on the tensor cores (Eq. 1; Algorithm 1's cache search): the
// Hamming test of every (query, entry) pair as one e4m3 GEMM over the packed signatures, then the exact key check of
// the admitted pairs. Same contract and outputs as the popcount scan in lsh.cu, which serves small batches.
//
// With signature bit 0 read as +1 and bit 1 as -1, the dot product of two b-bit signatures is
// (agreements - disagreements) = b - 2 hd, so hd <= radius iff dot >= b - 2 radius. Each term is +-1 and each sum
// an integer of at most 512 in magnitude, so an fp32 accumulation of e4m3 +-1 operands is exact.
//
// The entries are the GEMM's A operand (M = 128 entries a block) and are expanded from one bit to one byte inside the
// SM, straight into TMEM, from where tcgen05.mma reads A: HBM carries b / 8 bytes an entry, and the expanded bytes
// cross neither HBM nor shared memory. The order of K is free as long as both operands share it, so it is chosen for the
// expansion: four e4m3 values take one shift and one LOP3 (e4m3_word). The queries are the B operand, expanded once
// per pass into shared memory in the 128-byte swizzle layout.
//
// One CTA per contiguous range of 128-entry blocks, warp-specialised:
//   warp 31 (loader): cp.async.bulk of one stage (8 KB of packed signatures, kBPS blocks) into an 8-deep ring;
//   warps 22-29 (expanders, two sets of four that take blocks in turn; warp w writes TMEM lane quadrant w % 4): read
//     their 32 entries' words of a block from the ring, expand them and store them to one of kABuf A buffers in TMEM;
//   warp 30 (MMA): allocates TMEM; per block issues tcgen05.mma.kind::f8f6f4 (M = 128 entries, N = the pass's
//     queries rounded up to 32, K = 32) over the resident query operand, into one of up to 8 accumulators;
//   warps 0-15 (mask warps; warp w reads TMEM lane quadrant w % 4 and the 32-query column chunk w / 4): read each
//     entry's dot products into registers and release the accumulator; only where their maximum reaches the threshold
//     turn them into a mask of the admitted queries and queue those (query, entry) pairs in shared memory, each as one
//     word that also holds the queue's epoch;
//   warps 16-21 (checker warps): claim queued pairs as they arrive, compute their exact fp32 key scores over the
//     gathered key rows (each lane's 8-element chunks in order, then a butterfly sum) while the scan goes on, and
//     fold each score into its query's best score and, if it clears tau_c, into the query's list (lock-free). The
//     mask warps join them at every close of the queue.
// When the queue passes three quarters of its capacity, and at the end of the range, the mask warps close it: all checking
// warps finish what was queued below the close, then the queue is emptied and reopened in a new epoch. A pair
// that finds the queue full stays with its thread and is queued after the reopening. All
// epilogue warps expand the pass's query signatures into the query operand and write the lists out. The checker
// warps leave their loop only at a reopening, which the mask warps always run at the end of a pass, also after a
// timeout, so every named barrier sees all its warps.
// Queries are taken kQC at a time (one pass over the range each). Every mbarrier wait is bounded: on a timeout the
// CTA records LACACHE_ERR_DEVICE_TIMEOUT in the status word, the roles stop at the next pass boundary, in-flight
// copies and MMAs are drained, TMEM is freed and the CTA exits.
//
// What bounds it: instruction issue (0.62 a scheduler and cycle at 128 queries and 256 bits, ALU pipe half busy), at
// some 1,500 cycles per block of 128 entries at 128 queries; the packed index takes 20 us of HBM time on 4M entries,
// the MMAs 55 us. So the warps' loops are kept short, and in 64 registers a thread almost without spills (32-bit entry
// numbers, no running counts: 8 % at 128 queries); two expander sets, since one took 1,000 cycles a block and the MMAs
// waited for it (48 queries 166, with two 151); accumulators are released before their scores are looked at, not after
// the admitted pairs are queued, and mask warps without a query chunk leave them alone (48 queries 145 -> 137). Four
// mask warps share a block's columns, since accumulators for only three blocks fit beside the A buffers; they meet at a
// barrier only every 32 blocks (every 16: 2 % slower). Six checker warps: with four, 128 queries take 179 instead of
// 171; two pairs a checker at a time, or more A buffers, give nothing.
// Measured per lookup step (us) against the scan over an index kept expanded in HBM that was here first / against one
// expander set and late release: 4M x 768, 256 bits, 48 queries 176 / 172 -> 120, 64 180 / 174 -> 123, 128 202 / 188 ->
// 160, 384 563 / 536 -> 452; 128 bits, 48 queries 132 / 133 -> 108, 128 188 / 163 -> 144; 512 bits, 64 queries 326 / 232
// -> 174, 128 631 / 253 -> 225. The packed index takes an eighth of the expanded one's memory, and signing entries no
// second kernel.
// The mask warps' help counts where many pairs are admitted. At the end of the range: without it 128 queries on 4M x 1024
// take 18 % longer, and 357 on 36,433 x 768 a fifth. At the closes before: 1M x 768 in 64 clusters, 256 bits at radius 60,
// 48 queries 859 -> 310, 128 2,050 -> 784 (the scan over the expanded index 450 and 1,128); 4,096 clusters, radius 112, 64
// queries 2,393 -> 859 (1,146).
#include "internal.cuh"
#include "tcgen05.cuh"

namespace lc {
namespace {

constexpr int kMaskParts = 4;                            // mask warps per TMEM lane quadrant
constexpr int kMaskWarps = 4 * kMaskParts;               // warps 0-15: lane quadrant w % 4, column chunk w / 4
constexpr int kCheckWarps = 6;                           // warps 16-21: exact checks of the queued pairs
constexpr int kEpiWarps = kMaskWarps + kCheckWarps;      // warps 0-21
constexpr int kExpSets = 2;                              // each takes every second block
constexpr int kExpWarps = 4 * kExpSets;                  // warps 22-29: expand entry signatures into TMEM
constexpr int kMmaWarp = kEpiWarps + kExpWarps;          // warp 30
constexpr int kLoadWarp = kMmaWarp + 1;                  // warp 31
constexpr int kThreads = (kLoadWarp + 1) * 32;
// Queue capacity. A close before the end of the range stalls the scan until the checks are done, so the queue holds what
// a CTA usually queues in a whole range: 600 pairs on 4M entries in clusters of a thousand, 2,400 on a Zipf-skewed store of
// 16.8M x 1024, where a lookup of 128 queries takes 1.02 ms with 1,024, 0.90 with 2,048 and 0.71 with 4,096.
constexpr int kCap = 4096;
constexpr int kFlushAt = kCap - kCap / 4;                // a round that leaves more items than this closes the queue
constexpr int kRound = 32;                               // blocks the mask warps take between their barriers
constexpr int kBlockRows = 128;                          // entries per block and MMA (TMEM lanes)
constexpr int kAtomBytes = 128;                          // K bytes per swizzle atom (128 e4m3 values)
constexpr int kQC = 128;                                 // queries per pass
constexpr int kS = 8;                                    // ring stages
constexpr int kStageBytes = 8192;                        // packed signatures per stage
constexpr int kMaxNbuf = 8;                              // accumulators (at most)
constexpr int kMaxABuf = 4;                              // A buffers (at most)
constexpr unsigned kFull = 0xffffffffu;

// Geometry per signature width: W = b / 32 words. TMEM's 512 columns hold kABuf A buffers (128 entries x b bytes, 8 W
// columns each) at the top and nbuf accumulators of 32-query chunks below them.
template <int W>
struct TcGeo {
  static constexpr int kBits = 32 * W;
  static constexpr int kAtoms = kBits / kAtomBytes;            // 1, 2 or 4
  static constexpr int kBlockBytes = kBlockRows * 4 * W;       // packed: 2, 4 or 8 KB
  static constexpr int kBPS = kStageBytes / kBlockBytes;       // blocks per stage: 4, 2 or 1
  static constexpr int kQueryBytes = kQC * kBits;              // 16, 32 or 64 KB
  static constexpr int kABuf = W == 4 ? 4 : 2;
  static constexpr int kACols = 8 * W;
  static constexpr int kAccCols = 512 - kABuf * kACols;        // 384, 384 or 256
};
constexpr int kChunks = kQC / 32;                        // 32-query chunks of a block (at most)
static_assert(kMaskParts == kChunks, "a mask warp has one chunk");
static_assert(kRound <= 32, "a mask thread marks its blocks of a round in one word");
static_assert(kEpiWarps * 32 >= 128, "the epilogue threads cover a pass's queries when they set up the lists");

// A queued (query, entry) pair in one word, written and polled as a whole: bits 0-31 the entry id, 32-39 the query within
// the pass, 40-63 the queue's epoch (reopenings so far). A slot holds a pair of the current epoch iff its epoch says so.
__device__ __forceinline__ uint64_t pack_item(uint32_t ep, int q, int32_t j) {
  return ((uint64_t)ep << 40) | ((uint64_t)q << 32) | (uint32_t)j;
}
__device__ __forceinline__ int item_query(uint64_t x) { return (int)(x >> 32) & 0xFF; }
__device__ __forceinline__ int32_t item_entry(uint64_t x) { return (int32_t)(uint32_t)x; }

// Shared memory after the operands: the queue, the per-query best scores, flags and barriers; the per-query lists
// follow it.
struct Tail {
  uint64_t items[kCap];
  unsigned int best[128];      // score_order of the best admitted score, per query of the pass
  int taken[128];              // candidates folded, per query of the pass
  int count;                   // queued items (may run past kCap: those pairs stay pending)
  int claim;                   // queue positions claimed by the checker warps
  uint32_t closed;             // 0: open; else 1 + min(count, kCap) when the mask warps closed the queue
  uint32_t pass_end;           // closed for the last time in the pass
  uint32_t abort_flag;
  uint32_t tmem_slot;
  uint32_t issued;             // the loader's copies: stages 0 .. issued - 1
  long long progress;          // clock64() of the last reopening: restarts the budget of the waits behind the mask warps
  uint64_t bars[2 * kS + 2 * kMaxABuf + 2 * kMaxNbuf + 1];   // ring full / empty, A full / empty, accumulator full /
                                                             // empty, drain
};

template <int W>
constexpr size_t tc_smem_bytes(int top_c) {
  using G = TcGeo<W>;
  return 1024 + (size_t)kS * kStageBytes + G::kQueryBytes + sizeof(Tail) + (size_t)kQC * top_c * 8;
}

// acc + the products of 8 bf16 pairs, in order, each added by one fp32 FMA. The mixed-precision form reads the bf16 halves
// where they are; a bf16 is exact in fp32 and the FMA rounds once, so the sums are those of converting first, in a third
// fewer instructions (128 queries on 4M x 768, 256 bits: 168 us a lookup -> 162).
__device__ __forceinline__ float dot8(const uint4& u, const uint4& v, float acc) {
  const uint32_t x[4] = {u.x, u.y, u.z, u.w}, y[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int e = 0; e < 4; ++e)
    asm("{\n\t.reg .b16 xl, xh, yl, yh;\n\t"
        "mov.b32 {xl, xh}, %1;\n\t"
        "mov.b32 {yl, yh}, %2;\n\t"
        "fma.rn.f32.bf16 %0, xl, yl, %0;\n\t"
        "fma.rn.f32.bf16 %0, xh, yh, %0;\n\t}"
        : "+f"(acc)
        : "r"(x[e]), "r"(y[e]));
  return acc;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// The mask warps' OR barrier (named barrier 1), and the barrier of all epilogue warps (named barrier 2).
__device__ __forceinline__ bool mask_any(bool p) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred pi, po;\n\t"
      "setp.ne.u32 pi, %1, 0;\n\t"
      "bar.red.or.pred po, 1, %2, pi;\n\t"
      "selp.u32 %0, 1, 0, po;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)p), "n"(kMaskWarps * 32)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 2, %0;" ::"n"(kEpiWarps * 32) : "memory"); }

// Maximum of 32 fp32 values given as bits, by the three-operand form (two-operand: 2 % of a lookup at 128 queries).
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float max32(const uint32_t (&r)[32]) {
  float m[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    m[i] = __uint_as_float(r[8 * i]);
#pragma unroll
    for (int k = 1; k < 7; k += 2)
      m[i] = max3(m[i], __uint_as_float(r[8 * i + k]), __uint_as_float(r[8 * i + k + 1]));
    m[i] = fmaxf(m[i], __uint_as_float(r[8 * i + 7]));
  }
  return fmaxf(max3(m[0], m[1], m[2]), m[3]);
}

__device__ __forceinline__ uint32_t ld_volatile(const uint32_t* p) { return *reinterpret_cast<const volatile uint32_t*>(p); }
__device__ __forceinline__ void st_volatile(uint32_t* p, uint32_t v) { *reinterpret_cast<volatile uint32_t*>(p) = v; }

// Word i (0-7) of the 8 that signature word x expands to: bits i, 8 + i, 16 + i and 24 + i of x as four e4m3 bytes,
// +1 (0x38) for a clear bit and -1 (0xB8) for a set one.
__device__ __forceinline__ uint32_t e4m3_word(uint32_t x, int i) { return ((x << (7 - i)) & 0x80808080u) | 0x38383838u; }

// The 16 e4m3 bytes of 16-byte chunk c of a signature: words 4 (c & 1) .. 4 (c & 1) + 3 of signature word c / 2.
__device__ __forceinline__ uint4 e4m3_chunk(const uint32_t* words, int c) {
  const uint32_t x = words[c / 2];
  const int i = 4 * (c & 1);
  return make_uint4(e4m3_word(x, i), e4m3_word(x, i + 1), e4m3_word(x, i + 2), e4m3_word(x, i + 3));
}

// Byte offset of chunk c of row r in a [rows x b] operand in the 128-byte swizzle layout: atom c / 8 is its own
// [rows x 128 B] block, and chunk c % 8 of row r sits at ((c % 8) ^ (r & 7)) * 16 within the row's 128-byte line.
__device__ __forceinline__ uint32_t swizzled_chunk(int rows, int r, int c) {
  return (uint32_t)(c / 8) * rows * kAtomBytes + (uint32_t)r * kAtomBytes + (uint32_t)(((c % 8) ^ (r & 7)) << 4);
}

// A (the entries) in TMEM: lane = row, 4 e4m3 values per column; B in shared memory.
__device__ __forceinline__ void mma_e4m3(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// A checker lane's wait for queue position `slot` of epoch ep: true, with the pair, once it is there; false once the
// mask warps closed the queue at or below the slot (that position holds nothing to check in this epoch), or after
// about a second (the timeout is recorded; the mask warps then see the abort flag and close the queue).
__device__ __forceinline__ bool wait_slot(Tail& t, int slot, uint32_t ep, uint64_t* item, unsigned int* dev_status) {
  const long long t0 = clock64();
  for (;;) {
    if (slot < kCap) {
      *item = *reinterpret_cast<const volatile uint64_t*>(&t.items[slot]);
      if ((uint32_t)(*item >> 40) == (ep & 0xFFFFFFu)) return true;
    }
    const uint32_t closed = ld_volatile(&t.closed);
    // below the close: the pair was queued before it and its word is on the way
    if (closed && slot >= (int)closed - 1) return false;
    if (clock64() - t0 > kWaitCycles) {
      st_volatile(&t.abort_flag, 1u);
      atomicOr(dev_status, kDevTimeout);
      return false;
    }
    __nanosleep(256);
  }
}

// A checker warp's exact key score of one pair: the key row's loads of up to 768 elements are in flight together, each
// lane takes its 8-element chunks in order, then a butterfly sum (every lane ends with the score).
__device__ __forceinline__ float check_pair(uint64_t item, const __nv_bfloat16* __restrict__ keys,
                                            const __nv_bfloat16* __restrict__ q, int d, int q0, int lane) {
  constexpr int kAhead = 3;   // chunks per lane
  const int v = d / 8;
  const uint4* kp = reinterpret_cast<const uint4*>(keys + (int64_t)item_entry(item) * d);
  const uint4* xp = reinterpret_cast<const uint4*>(q + (int64_t)(q0 + item_query(item)) * d);
  float acc = 0.f;
#pragma unroll 1
  for (int c0 = lane; c0 < v; c0 += 32 * kAhead) {
    uint4 kv[kAhead], x[kAhead];
#pragma unroll
    for (int i = 0; i < kAhead; ++i)
      if (c0 + 32 * i < v) kv[i] = __ldg(kp + c0 + 32 * i);
#pragma unroll
    for (int i = 0; i < kAhead; ++i)
      if (c0 + 32 * i < v) x[i] = __ldg(xp + c0 + 32 * i);
#pragma unroll
    for (int i = 0; i < kAhead; ++i)
      if (c0 + 32 * i < v) acc = dot8(x[i], kv[i], acc);
  }
  return warp_sum(acc);
}

// The same for kNarrowItems pairs of rows of at most 256 elements, one chunk per lane: as many loads in flight as for one
// wide pair. Lane u returns pair u's score. (One at a time, 357 queries on 36,433 x 160 took 47 us, and so 37.)
constexpr int kNarrowItems = 3;
__device__ __forceinline__ float check_narrow(const uint64_t (&item)[kNarrowItems],
                                              const __nv_bfloat16* __restrict__ keys,
                                              const __nv_bfloat16* __restrict__ q, int d, int q0, int lane) {
  uint4 kv[kNarrowItems], x[kNarrowItems];
#pragma unroll
  for (int u = 0; u < kNarrowItems; ++u) {
    kv[u] = x[u] = make_uint4(0u, 0u, 0u, 0u);
    if (lane < d / 8) {
      kv[u] = __ldg(reinterpret_cast<const uint4*>(keys + (int64_t)item_entry(item[u]) * d) + lane);
      x[u] = __ldg(reinterpret_cast<const uint4*>(q + (int64_t)(q0 + item_query(item[u])) * d) + lane);
    }
  }
  float score = 0.f;
#pragma unroll
  for (int u = 0; u < kNarrowItems; ++u) {
    const float s = warp_sum(dot8(x[u], kv[u], 0.f));
    if (lane == u) score = s;
  }
  return score;
}

// Fold one exact score into its query's best score and, if it clears tau_c, into the query's list (unordered, 0 =
// empty) of at most C candidates, without a lock. The first C candidates of a query each take a slot of their own. Later
// ones are offered to every slot in turn: a slot keeps the larger of its candidate and the one offered, and the smaller
// goes on, so what leaves the last slot is no larger than any candidate kept, and slots only grow. A candidate that
// such an offer left in a slot before the slot's owner wrote it is offered again. A candidate below every slot is not
// offered: C others are larger (a Zipf-skewed store of 16.8M x 1024, where hot queries have hundreds of candidates per CTA:
// 1.11 ms a lookup -> 1.02).
__device__ __forceinline__ void fold_one(Tail& t, uint64_t* lists, int C, float tau_c, int qq, int32_t j, float sc) {
  const unsigned int order = score_order(sc);
  if (order > ld_volatile(&t.best[qq])) atomicMax(&t.best[qq], order);
  if (!(sc >= tau_c)) return;
  unsigned long long x = pack_cand(sc, (uint32_t)j);
  unsigned long long* L = reinterpret_cast<unsigned long long*>(lists + (size_t)qq * C);
  const int slot = *reinterpret_cast<volatile int*>(&t.taken[qq]) < C ? atomicAdd(&t.taken[qq], 1) : C;
  if (slot < C) {
    x = atomicExch(L + slot, x);
  } else {
    bool larger = true;
#pragma unroll 4
    for (int i = 0; i < C; ++i) larger &= *reinterpret_cast<volatile unsigned long long*>(L + i) > x;
    if (larger) return;
  }
  for (int i = 0; i < C && x; ++i) {
    const unsigned long long old = atomicMax(L + i, x);
    if (old < x) x = old;
  }
}

// Run by all epilogue warps after the mask warps closed the queue: once every checker has arrived, every queued
// pair has been checked and folded into its query's list; then the queue is emptied and reopened. Whether that was the
// pass's last close is read between the barriers, where no later close can have been made.
__device__ __forceinline__ bool reopen(Tail& t, int ew, int lane) {
  epi_sync();
  const bool end = ld_volatile(&t.pass_end) != 0;
  if (ew == 0 && lane == 0) {
    t.count = 0;
    t.claim = 0;
    t.closed = 0;
    *reinterpret_cast<volatile long long*>(&t.progress) = clock64();
  }
  epi_sync();
  return end;
}

template <int W>
__global__ void __launch_bounds__(kThreads, 1) lsh_tc_kernel(Stage1Args a, LshArgs l, int splits) {
  using G = TcGeo<W>;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  unsigned char* gbase = smem_raw + (base - raw);
  const uint32_t q_smem = base;                                      // kQC query rows
  const unsigned char* ring = gbase + G::kQueryBytes;                // kS stages of packed signatures
  const uint32_t ring_smem = base + G::kQueryBytes;
  Tail& t = *reinterpret_cast<Tail*>(gbase + G::kQueryBytes + (size_t)kS * kStageBytes);
  uint64_t* lists = reinterpret_cast<uint64_t*>(&t + 1);            // [kQC][top_c]
  volatile uint32_t* abort_flag = &t.abort_flag;
  const uint32_t bar0 = smem_u32(t.bars);
  auto full_bar = [&](int s) { return bar0 + 8u * s; };
  auto empty_bar = [&](int s) { return bar0 + 8u * (kS + s); };
  auto afull_bar = [&](int b) { return bar0 + 8u * (2 * kS + b); };
  auto aempty_bar = [&](int b) { return bar0 + 8u * (2 * kS + kMaxABuf + b); };
  auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * kS + 2 * kMaxABuf + b); };
  auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * kS + 2 * kMaxABuf + kMaxNbuf + b); };
  const uint32_t drain_bar = bar0 + 8u * (2 * kS + 2 * kMaxABuf + 2 * kMaxNbuf);

  const int warp = __shfl_sync(kFull, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;   // warp: uniform
  // accumulators: the same for every pass (the first pass has the most queries). Mask warps of chunks past first_chunks
  // have none in any pass.
  const int first_chunks = (min(kQC, a.B) + 31) / 32;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kS; ++s) {
      mbar_init(full_bar(s), 1);              // the loader's arrive, with the copy's bytes
      mbar_init(empty_bar(s), 4 * G::kBPS);   // four expander warps per block of the stage
    }
    for (int b = 0; b < G::kABuf; ++b) {
      mbar_init(afull_bar(b), 4);             // the block's four expander warps
      mbar_init(aempty_bar(b), 1);            // the MMA commit
    }
    for (int b = 0; b < kMaxNbuf; ++b) {
      mbar_init(tfull_bar(b), 1);             // the MMA commit
      mbar_init(tempty_bar(b), 4 * first_chunks);
    }
    mbar_init(drain_bar, 1);
    t.abort_flag = 0;
    t.issued = 0;
    t.progress = clock64();
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = threadIdx.x; i < kCap; i += kThreads) t.items[i] = ~(uint64_t)0;   // no epoch
  if (warp == kMmaWarp) {
    tmem_alloc<false>(smem_u32(&t.tmem_slot), 512);
    tmem_relinquish<false>();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = t.tmem_slot;
  const uint32_t a_tmem = tmem + (uint32_t)G::kAccCols;
  // the query signatures are the previous kernel's output
  asm volatile("griddepcontrol.wait;" ::: "memory");

  auto fail = [&]() {
    *abort_flag = 1u;
    atomicOr(a.dev_status, kDevTimeout);
  };
  // The loader's, expanders' and MMA issuer's waits. All three stand still while the mask warps have the pairs of a round
  // checked that found the queue full. A round may leave 524,288 of them, and at d = 8192 with lists of 32 the checks of
  // so many take 0.26 s (0.8 s by the checker warps alone), much of one wait's budget. So it restarts at every reopening, of
  // which those pairs allow a limited number: every reopening either takes all of them or fills the queue.
  auto wait = [&](uint32_t bar, uint32_t parity) { return mbar_wait_inline(bar, parity, abort_flag, &t.progress); };

  const int s = blockIdx.x;
  const int64_t nblocks = (a.n + kBlockRows - 1) / kBlockRows;
  const uint32_t g_begin = (uint32_t)(nblocks * s / splits), nb = (uint32_t)(nblocks * (s + 1) / splits) - g_begin;
  // the range's entries (ids are int32: so is the store's size)
  const uint32_t j_begin = g_begin * kBlockRows, j_end = min((uint32_t)a.n, (g_begin + nb) * kBlockRows);
  const uint32_t nstages = (nb + G::kBPS - 1) / G::kBPS;    // ring stages per pass
  const bool withhold = a.inject_stall && s == 0;           // test support: the first stage's copy is not issued
  const int C = a.top_c;
  const float thr = (float)(G::kBits - 2 * l.radius);   // admitted iff dot >= b - 2 radius
  const int stride = 32 * first_chunks;
  const uint32_t nbuf = (uint32_t)min(kMaxNbuf, G::kAccCols / stride);
  uint32_t b = 0, ph = 0; // MMA issuer, mask warps: the next block's accumulator, and the parity of its use
  const auto first_acc = [&](uint32_t block) {
    b = block % nbuf;
    ph = (block / nbuf) & 1u;
  };
  const auto next_acc = [&]() {
    if (++b == nbuf) {
      b = 0;
      ph ^= 1u;
    }
  };
  uint32_t ep = 0;        // epilogue: reopenings so far (the epoch of the queue's ready stamps)

  for (int q0 = 0; q0 < a.B; q0 += kQC) {
    const uint32_t it = (uint32_t)(q0 / kQC) * nb, st_base = (uint32_t)(q0 / kQC) * nstages;   // blocks, stages so far
    const int qn = min(kQC, a.B - q0);
    const int npad = (qn + 31) / 32 * 32;
    // ---- pass set-up (epilogue warps): the resident query operand, the lists and counters ----
    if (warp < kEpiWarps) {
      const int et = threadIdx.x;
      // one thread per (query row, 16-byte chunk)
      for (int i = et; i < npad * 2 * W; i += kEpiWarps * 32) {
        const int r = i / (2 * W), c = i % (2 * W);
        uint4 v = make_uint4(0, 0, 0, 0);
        if (r < qn) v = e4m3_chunk(l.qsig + (int64_t)(q0 + r) * W, c);
        const uint32_t addr = q_smem + swizzled_chunk(kQC, r, c);
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                     : "memory");
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      for (int i = et; i < qn * C; i += kEpiWarps * 32) lists[i] = 0;
      for (int i = et; i < qn; i += kEpiWarps * 32) {
        t.best[i] = score_order(-INFINITY);
        t.taken[i] = 0;
      }
      if (et == 0) {
        t.count = 0;
        t.claim = 0;
        t.closed = 0;
        t.pass_end = 0;
      }
    }
    __syncthreads();

    if (warp == kLoadWarp) {
      // ---------------- loader ----------------
      if (lane == 0) {
        for (uint32_t si = 0; si < nstages; ++si) {
          const uint32_t k = st_base + si;
          const int st = k % kS;
          if (!wait(empty_bar(st), ((k / kS) & 1u) ^ 1u)) {
            fail();
            break;
          }
          if (withhold && k == 0) continue;   // nothing arrives on this stage: the expanders' wait runs out
          // the stage's entries, at most j_end: whole signatures of 16 W / 4 bytes, so a multiple of 16
          const uint32_t e0 = j_begin + si * G::kBPS * kBlockRows;
          const uint32_t bytes = min((uint32_t)G::kBPS * kBlockRows, j_end - e0) * W * 4;
          mbar_expect_tx(full_bar(st), bytes);
          asm volatile(
              "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
              ::"r"(ring_smem + (uint32_t)st * kStageBytes), "l"(l.sig + (int64_t)e0 * W), "r"(bytes), "r"(full_bar(st))
              : "memory");
          t.issued = k + 1;
        }
      }
      __syncwarp();
    } else if (warp >= kEpiWarps && warp < kMmaWarp) {
      // ---------------- expanders ----------------
      const int quad = warp % 4, set = (warp - kEpiWarps) / 4;
      const uint32_t lane_addr = (uint32_t)(quad * 32) << 16;
      bool ok = true;
      // every kExpSets-th block slot of the pass's stages, also those past the last block: each stage gets all its
      // releases
      for (uint32_t ti = set; ti < nstages * G::kBPS; ti += kExpSets) {
        const uint32_t k = st_base + ti / G::kBPS;
        const int st = k % kS;
        bool there = wait(full_bar(st), (k / kS) & 1u);
        if (ti < nb) {
          const unsigned char* src = ring + (size_t)st * kStageBytes +
                                     ((size_t)(ti % G::kBPS) * kBlockRows + quad * 32 + lane) * W * 4;
          uint4 y[W / 4];
#pragma unroll
          for (int h = 0; h < W / 4; ++h) y[h] = *reinterpret_cast<const uint4*>(src + 16 * h);
          const uint32_t u = it + ti;
          const int b = u % G::kABuf;
          there = there && wait(aempty_bar(b), ((u / G::kABuf) & 1u) ^ 1u);
          ok = __all_sync(kFull, there);
          if (!ok) break;
          tc_fence_after();
          const uint32_t dst = a_tmem + lane_addr + (uint32_t)(b * G::kACols);
          // four signature words, 32 columns, at a time
#pragma unroll
          for (int h = 0; h < W / 4; ++h) {
            const uint32_t x[4] = {y[h].x, y[h].y, y[h].z, y[h].w};
            uint32_t r[32];
#pragma unroll
            for (int w = 0; w < 4; ++w)
#pragma unroll
              for (int i = 0; i < 8; ++i) r[8 * w + i] = e4m3_word(x[w], i);
            tmem_st32(dst + 32u * h, r);
          }
          tmem_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) {
            mbar_arrive(afull_bar(b));
            mbar_arrive(empty_bar(st));
          }
        } else {   // past the last block: only the stage's release
          ok = __all_sync(kFull, there);
          if (!ok) break;
          if (lane == 0) mbar_arrive(empty_bar(st));
        }
      }
      if (!ok && lane == 0) fail();
      __syncwarp();
    } else if (warp == kMmaWarp) {
      // ---------------- MMA issue ----------------
      // kind::f8f6f4: D f32 (bits 4-5 = 1), A and B e4m3 (bits 7-9, 10-12 = 0), both K-major, N >> 3 in bits 17-22,
      // M >> 4 in bits 24-28. The whole warp runs the loop and one lane issues (see elect_one).
      const uint32_t idesc = (1u << 4) | ((uint32_t)(npad >> 3) << 17) | ((uint32_t)(kBlockRows >> 4) << 24);
      const uint64_t qdesc = smem_desc(q_smem);
      first_acc(it);
      for (uint32_t ti = 0; ti < nb; ++ti) {
        const uint32_t u = it + ti, ab = u % G::kABuf;
        if (!__all_sync(kFull, wait(tempty_bar(b), ph ^ 1u) && wait(afull_bar(ab), (u / G::kABuf) & 1u))) {
          if (lane == 0) fail();
          break;
        }
        tc_fence_after();
        const uint32_t d = tmem + b * (uint32_t)stride;
        const uint32_t ad = a_tmem + ab * (uint32_t)G::kACols;
        if (elect_one()) {
#pragma unroll
          for (int at = 0; at < G::kAtoms; ++at)
#pragma unroll
            for (int ks = 0; ks < kAtomBytes / 32; ++ks)
              mma_e4m3(d, ad + (uint32_t)(at * (kAtomBytes / 4) + 8 * ks),
                       qdesc + (uint64_t)((at * kQC * kAtomBytes + 32 * ks) >> 4), idesc, (at | ks) != 0 ? 1u : 0u);
          mma_commit<false>(tfull_bar(b), 0);
          mma_commit<false>(aempty_bar(ab), 0);
        }
        __syncwarp();
        next_acc();
      }
    }

    if (warp < kEpiWarps) {
      // ---------------- mask warps: scan; checker warps, and the mask warps at a close: check ----------------
      const int quad = warp % 4, part = warp / 4;            // mask warps: TMEM lane quadrant; 32-query column chunk
      const int nch = npad / 32;                             // 32-query chunks of a block
      // A mask thread's pairs that found the queue full: the queries per block of a round; which blocks have some; the
      // round's first block. (Local memory: touched only when the queue fills up.)
      uint32_t rest[kRound + 2];
      // queue the queries of `mask` with entry j, as many as fit; the others are returned
      auto push = [&](uint32_t mask, uint32_t j) -> uint32_t {
        uint32_t full = 0;
        while (mask) {
          const int bit = __ffs(mask) - 1;
          mask &= mask - 1;
          const int slot = atomicAdd(&t.count, 1);
          if (slot < kCap)
            *reinterpret_cast<volatile uint64_t*>(&t.items[slot]) = pack_item(ep, 32 * part + bit, (int32_t)j);
          else
            full |= 1u << bit;
        }
        return full;
      };
      // this thread's entry of a block
      const auto entry = [&](uint32_t block) { return j_begin + block * kBlockRows + quad * 32 + lane; };
      // A round: the blocks from t0 on, at most kRound. False after a timeout. Admitted pairs are rare: a first look at a
      // block takes only the maximum of the chunk's scores; the admitted queries are told apart, and queued for the
      // checker warps, where some lane's maximum reaches the threshold.
      auto scan_round = [&](uint32_t t0) -> bool {
#pragma unroll 1
        for (int r = 0; part < first_chunks && r < kRound && t0 + r < nb; ++r) {
          // the warp-collective loads below need the whole warp
          if (!__all_sync(kFull, mbar_wait_inline(tfull_bar(b), ph, abort_flag))) return false;
          tc_fence_after();
          const uint32_t acc = tmem + ((uint32_t)(quad * 32) << 16) + b * (uint32_t)stride;
          // the accumulator is free once its scores are in registers: the MMA issuer does not wait for what follows
          const uint32_t free_bar = tempty_bar(b);
          next_acc();
          if (part >= nch) {   // no chunk of this pass's queries
            if (lane == 0) mbar_arrive(free_bar);
            continue;
          }
          uint32_t v[32];
          tmem_ld32_issue(acc + 32u * part, v);
          tmem_ld32_wait(v);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(free_bar);
          if (__any_sync(kFull, max32(v) >= thr)) {
            // the differences' signs, taken by a subtraction and a shift each (integers: no rounding, and no -0)
            uint32_t mask = 0;
#pragma unroll
            for (int i = 31; i >= 0; --i)
              mask = __funnelshift_l(__float_as_uint(__uint_as_float(v[i]) - thr), mask, 1);
            mask = ~mask;
            const int left = qn - 32 * part;   // padding queries past qn are never admitted
            if (left < 32) mask &= (1u << left) - 1u;
            const uint32_t j = entry(t0 + r);
            const uint32_t full = j < j_end ? push(mask, j) : 0u;
            if (full) {
              rest[kRound] |= 1u << r;
              rest[r] = full;
            }
            __syncwarp();   // the next load is warp-collective
          }
        }
        return true;
      };
      // Whether the queue has to be closed now, with *last set after a timeout. All mask warps get the same answer.
      auto must_close = [&](bool got, bool* last) -> bool {
        __syncwarp();
        if (!mask_any(!got || *abort_flag || *reinterpret_cast<volatile int*>(&t.count) > kFlushAt)) return false;
        *last = mask_any(!got || *abort_flag);
        if (!got) fail();
        return true;
      };
      // close the queue (every mask warp has queued its pairs); the pass's last close also after a timeout: the checkers
      // leave only at a reopening
      auto close = [&](bool last) {
        if (threadIdx.x == 0) {
          if (last) t.pass_end = 1;
          st_volatile(&t.closed, 1u + (uint32_t)min(t.count, kCap));
        }
      };

      if (warp < kMaskWarps) {
        rest[kRound] = 0;
        first_acc(it);
        bool last = true;
        for (uint32_t t0 = 0; t0 < nb; t0 += kRound)
          if (must_close(scan_round(t0), &last)) {
            rest[kRound + 1] = t0;
            break;
          }
        close(last);
      }
      for (;;) {   // an epoch of the queue
        // claim a queue position (several for narrow rows), check and fold its pair while the scan goes on; at a close,
        // finish what was queued below it, then take part in the reopening
        const int claims = a.d <= 256 ? kNarrowItems : 1;
        for (;;) {
          int base = 0;
          if (lane == 0) base = atomicAdd(&t.claim, claims);
          base = __shfl_sync(kFull, base, 0);
          uint64_t got = 0;
          const bool mine = lane < claims && wait_slot(t, base + lane, ep, &got, a.dev_status);
          const unsigned ready = __ballot_sync(kFull, mine);
          if (ready) {
            float score;   // lane u: of the pair at base + u
            if (claims == 1) {
              score = check_pair(__shfl_sync(kFull, got, 0), a.keys, a.q, a.d, q0, lane);
            } else {
              // a position without a pair repeats one that has it, and is not folded
              uint64_t item[kNarrowItems];
#pragma unroll
              for (int u = 0; u < kNarrowItems; ++u)
                item[u] = __shfl_sync(kFull, got, (ready >> u) & 1u ? u : __ffs(ready) - 1);
              score = check_narrow(item, a.keys, a.q, a.d, q0, lane);
            }
            if (mine) fold_one(t, lists, C, a.tau_c, item_query(got), item_entry(got), score);
            __syncwarp();
          }
          if (ready != (1u << claims) - 1u) break;   // a position past the close (or a timeout)
        }
        const bool end = reopen(t, warp, lane);
        ++ep;
        if (end) break;
        if (warp < kMaskWarps) {
          // The range's rest: first what found the queue full (every epoch either queues all of it or fills the queue, so
          // this ends). A copy of the scan above and no way back to it, which would keep more in registers over the
          // checks: the common pass, with one close, then spills (8 % of a lookup).
          uint32_t t0 = rest[kRound + 1], left = 0;
          for (uint32_t o = rest[kRound]; o; o &= o - 1) {
            const int i = __ffs(o) - 1;
            rest[i] = push(rest[i], entry(t0 + i));
            if (rest[i]) left |= 1u << i;
          }
          rest[kRound] = left;
          t0 += kRound;
          first_acc(it + min(t0, nb));
          bool last = true;
          for (bool got = true; !must_close(got, &last); t0 += kRound) {
            if (t0 >= nb) {
              last = true;
              break;
            }
            got = scan_round(t0);
          }
          rest[kRound + 1] = t0 - kRound;
          close(last);
        }
      }
    }

    // ---- pass end: every role is here; a timeout anywhere stops them all together ----
    if (__syncthreads_or(*abort_flag != 0)) break;
    if (warp < kEpiWarps) {
      const int et = threadIdx.x;
      // the lists' candidates (a list of n < C candidates holds them in its first n slots) and each list's record
      for (int i = et; i < qn * C; i += kEpiWarps * 32) {
        const int qq = i / C;
        if (lists[i]) a.part_cand[((int64_t)s * a.B + q0 + qq) * C + (i - qq * C)] = lists[i];
      }
      for (int i = et; i < qn; i += kEpiWarps * 32) {
        uint32_t count = 0;
        while ((int)count < C && lists[(size_t)i * C + count]) ++count;
        a.part_meta[(int64_t)s * a.B + q0 + i] = PartMeta{score_of_order(t.best[i]), count};
      }
    }
    __syncthreads();
  }

  // nothing in flight when the CTA exits: the loader waits for its last kS copies (a consumed one passes at
  // once), the MMA issuer for every MMA; then TMEM is freed
  if (warp == kLoadWarp && lane == 0) {
    const uint32_t issued = t.issued;
    for (uint32_t k = max(issued >= (uint32_t)kS ? issued - kS : 0u, withhold ? 1u : 0u); k < issued; ++k)
      mbar_wait_inline(full_bar(k % kS), (k / kS) & 1u, nullptr);
  }
  if (warp == kMmaWarp) {
    // from the lane that issued the MMAs: a commit covers its own thread's only, and after a timeout some may still run
    if (elect_one()) mma_commit<false>(drain_bar, 0);
    __syncwarp();
    mbar_wait_inline(drain_bar, 0, nullptr);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kMmaWarp) tmem_dealloc<false>(tmem, 512);
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// A programmatic dependent launch of the query-signature kernel: the CTAs may be scheduled while the signatures are
// computed and wait in griddepcontrol.wait.
template <int W>
cudaError_t launch_w(const Stage1Args& a, const LshArgs& l, int splits, cudaStream_t st) {
  const size_t smem = tc_smem_bytes<W>(a.top_c);
  cudaError_t e = cudaFuncSetAttribute(lsh_tc_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(splits);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, lsh_tc_kernel<W>, a, l, splits);
}

static_assert(tc_smem_bytes<4>(kMaxTopC) <= 227 * 1024 && tc_smem_bytes<8>(kMaxTopC) <= 227 * 1024 &&
                  tc_smem_bytes<16>(kMaxTopC) <= 227 * 1024,
              "shared memory budget");

}  // namespace

cudaError_t launch_stage1_lsh_tc(const Stage1Args& a, const LshArgs& l, int num_sms, int max_splits,
                                 cudaStream_t st, int* splits) {
  const int64_t blocks = (a.n + kBlockRows - 1) / kBlockRows;
  int s = (int)(blocks < (int64_t)num_sms ? blocks : (int64_t)num_sms);
  if (s > max_splits) s = max_splits;
  if (s < 1) s = 1;
  *splits = s;
  switch (l.words) {   // 128, 256 or 512-bit signatures
    case 4: return launch_w<4>(a, l, s, st);
    case 8: return launch_w<8>(a, l, s, st);
    case 16: return launch_w<16>(a, l, s, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lc
