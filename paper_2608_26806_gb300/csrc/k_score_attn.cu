// Criterion B: text-to-visual attention mass per visual token (the per-token form of
// the attention quantity of paper §3.3.2), without materialising the attention matrix:
//   s_t = 1/(Hq*|Q_r|) * sum_h sum_{q in Q_r, pos q >= pos t} exp2(z2(h,q,t) - lse2(h,q)),
//   z2 = softmax_scale * log2(e) * q_h . k_{g(h)},  lse2 = log2 sum_{visible keys} exp2(z2).
//
// Rows: for KV group g, row o*G + j is text query o (in text order over the batch)
// with query head g*G + j. The text queries are first repacked by group into
// Qt[g][row][d] (k_attn_pack), so that both passes read them with TMA boxes. A
// request's rows are cut into blocks of 256.
//
// Pass 1, k_attn_lse (skipped when the caller supplies FlashAttention's LSE): a block's rows
// stay in shared memory as two A operands of 128 rows and the tiles of 128 keys, from the
// request's first token to the block's last query, stream past them as B: two products of
// 128 x 128 x d a tile. A thread owns a row and keeps (reference, sum of exp2) of every other
// tile's logits; one partial per (row, CTA) is left behind.
// Pass 2, k_attn_mass: the same with the roles exchanged: the tiles of 128 visual keys of
// every image that one of the block's queries follows are the A operand, the block's halves
// the B operand. A thread owns a key and sums exp2(z2 - lse2) over 128 rows, leaving out the
// rows whose query precedes the key's image and those of another request; lse2 comes from
// the pass-1 partials of the block (merged when the walk enters it) or from the supplied
// LSE. The per-key sums of all blocks and KV groups meet in a 64-bit fixed-point accumulator
// (integer atomics: the result does not depend on their order).
// k_attn_finalize turns the accumulator into scores and the fixed-point image sums.
//
// Both passes are persistent: the flat list of (KV group, block, key tile) is split into
// equal contiguous runs, one per CTA (one CTA per SM). TMEM holds four accumulators of 128
// columns, one for each half of the block and parity of the step. Warps 0-15 are the
// epilogue, four per accumulator (warp w reads TMEM lanes 32(w%4)..+31 of accumulator w/4),
// so every SM sub-partition has a warp of each; warp 16 issues the TMA loads; warps 17 and
// 18 own a half of the block each and issue its MMAs, so that a half whose epilogue is
// slower (its rows see more) does not hold up the other.
//
// What bounds them: the epilogue's exponentials and sums, 1235 cycles for a tile's 128 x 256
// logits with all sixteen warps busy (measured alone; exp2 alone 1024), against 1024 for the
// MMAs; where causality leaves an epilogue little to do, the key tiles' delivery (24 bytes a
// cycle and SM). Serving batch of 34423 tokens (8 requests, 32 heads, 8 KV heads): pass 1
// 83 -> 62 us, pass 2 86 -> 70 us; one request of 10368 tokens with 256 text tokens: 27 -> 20
// and 26 -> 24 us. Before, eight epilogue warps and two accumulators of 256 columns left the
// MMAs and the epilogue of an accumulator waiting for each other, pass 1 took a maximum per
// 32 logits, one lane behind a lane branch issued the MMAs, and every block began with
// searches in the prefix arrays (AttnBlkInfo).
#include <cudaTypedefs.h>

#include <type_traits>

#include "avtp_tc.cuh"

namespace avtp {
namespace {

constexpr int kM = kAttnTileM;        // 128
constexpr int kBlk = kAttnBlockRows;  // 256
constexpr int kGroupWarps = 4;        // epilogue warps of an accumulator
constexpr int kSetThreads = 2 * 32 * kGroupWarps;  // threads of the two accumulators of a step
constexpr int kTmaWarp = 4 * kGroupWarps;
constexpr int kMmaWarp = kTmaWarp + 1;  // and the next
constexpr int kThreads = 32 * (kMmaWarp + 2);
constexpr uint32_t kTmemCols = 512;  // four accumulators of 128 columns
constexpr int kStages = 4;            // key tiles in flight
constexpr int kMassWindow = 12;       // steps of an epilogue group whose key masses are held in shared memory between flushes
constexpr float kLog2e = 1.4426950408889634f;
// Flag of a key whose mass in some block is not a number in [0, 2^kAttnBlockMassBits]
// (non-finite inputs, or a supplied normaliser far below the row's own). The sum of its finite
// contributions stays below this bit (attn_mass_frac_bits).
constexpr unsigned long long kMassNotFinite = 1ull << 63;

static_assert(kBlk == 2 * kM, "a block is two products of 128 rows");

// Shared memory for head_dim d (1024-byte aligned tiles): the row block and kStages key tiles.
__host__ __device__ constexpr size_t a_bytes(int d) { return static_cast<size_t>(kM) * d * 2; }
__host__ __device__ constexpr size_t b_bytes(int d) { return static_cast<size_t>(kBlk) * d * 2; }
__host__ __device__ constexpr size_t attn_smem_bytes(int d) { return 1024 + b_bytes(d) + kStages * a_bytes(d); }

struct Sync {
  uint64_t k_full[kStages], k_empty[kStages];
  uint64_t b_full[2], b_empty[2];            // halves of the row block
  uint64_t acc_full[2][2], acc_empty[2][2];  // [buffer: step parity][half]
  uint64_t drain[2];
  uint32_t tmem;
  int abort;
};

struct AttnArgs {
  const int32_t* text_idx;
  const int4* blk_info;          // the validation kernel's tables, see AttnBlkInfo
  const int4* tile_info;
  const int4* cta_start;
  const int32_t* meta;           // F1, C1, F2, C2, NB, fraction bits of the mass
  const float* lse_rows;         // [Hkv, rows] (supplied LSE) or nullptr
  float2* p1_part;               // [Hkv * NB][256 rows][kAttnMaxChunks]
  unsigned long long* mass;      // [key tile][128] fixed point, 2^-meta[5]
  int64_t rows;
  int G;
  float c2;                      // softmax_scale * log2(e)
  DevStatus* st;
};

// Barriers of the 256 epilogue threads of step parity b (id 1 + b), of all 512 (id 3), and of
// the 128 of one accumulator (ids 4 .. 7).
__device__ __forceinline__ void bar_set(int b) { asm volatile("bar.sync %0, 256;" ::"r"(1 + b) : "memory"); }
__device__ __forceinline__ void bar_epi() { asm volatile("bar.sync 3, 512;" ::: "memory"); }
__device__ __forceinline__ void bar_acc(int b, int t) {
  asm volatile("bar.sync %0, 128;" ::"r"(4 + 2 * b + t) : "memory");
}

// Diagnostic timeline build (-DAVTP_TIMELINE): clock stamps of each pass's first CTA, per
// step s of its run. Slots: 0 the key tile's load issued (TMA thread); 1 the MMA thread at
// the step, 2 its operands and accumulators ready, 3 its MMAs issued and committed (of the
// block's first half); on even steps 4 that half's accumulator ready for epilogue warp 0, 5
// released by it. Read with avtp_score_timeline().
#ifdef AVTP_TIMELINE
constexpr int kAttnTlSteps = 64;
constexpr int kAttnTlSlots = 6;
__device__ long long g_attn_tl[2][kAttnTlSteps][kAttnTlSlots];
#endif
__device__ __forceinline__ void attn_stamp(int pass, int st, int slot) {
#ifdef AVTP_TIMELINE
  if (blockIdx.x == 0 && st < kAttnTlSteps) g_attn_tl[pass][st][slot] = clock64();
#else
  (void)pass;
  (void)st;
  (void)slot;
#endif
}

// Walks a CTA's run of a pass's flat list (KV group, block, entry): pass 1's entries are
// steps of 128 keys from the request's first key, pass 2's the request's key tiles in order.
template <int PASS>
struct Walk {
  int g, b, j, n;  // KV group, block, entry within the block, entries of the block
  AttnBlkInfo blk;
  const int4* tab;
  int NB;
  __device__ __forceinline__ void load() {
    const int4 lo = tab[2 * b], hi = tab[2 * b + 1];
    blk = AttnBlkInfo{lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, 0};
    n = PASS == 1 ? blk.n1 : blk.n2;
  }
  __device__ __forceinline__ void init(const AttnArgs& a, const int4& start) {
    g = start.x;
    b = start.y;
    j = start.z;
    tab = a.blk_info;
    NB = a.meta[4];
    load();
  }
  // Next entry; returns true when it lies in another block. Only called while another
  // entry exists, so the loop over empty blocks ends.
  __device__ __forceinline__ bool next() {
    if (++j < n) return false;
    j = 0;
    do {
      if (++b == NB) {
        b = 0;
        ++g;
      }
      load();
    } while (n == 0);
    return true;
  }
  __device__ __forceinline__ bool last_of_block() const { return j + 1 == n; }
};

// ---------------------------------------------------------------- epilogue arithmetic
// A warp's slice of an accumulator: its 32 TMEM lanes x kHalf columns, read as 32-column
// chunks.
constexpr int kHalf = kM;
constexpr int kChunks = kHalf / 32;
// A slice's sum above this moves the row's reference, if the slice's maximum exceeds it by
// more than kRescaleTau (log2 units).
constexpr float kRescaleSum = 16384.f;
constexpr float kRescaleTau = 8.f;

// Pass 1: f(chunk values) over the chunks [0, pe) of a row's slice, one at a time (four
// warps a sub-partition hide each other's loads). MASKED: columns past lim (per lane) read
// as -inf.
template <bool MASKED, class F>
__device__ __forceinline__ void p1_chunks(uint32_t taddr, int pe, int lim, F&& f) {
#pragma unroll 1
  for (int p = 0; p < pe; ++p) {
    uint32_t r[32];
    tc::tmem_ld32_async(taddr + p * 32, r);
    tc::tmem_wait(r);
    if (MASKED) {
#pragma unroll
      for (int q = 0; q < 32; ++q) r[q] = (p * 32 + q <= lim) ? r[q] : 0xff800000u;
    }
    f(r);
  }
}
// Sum of exp2(c2 z - m) over the slice, in four partial sums (columns q mod 4).
template <bool MASKED>
__device__ __forceinline__ float p1_sum(uint32_t taddr, int pe, int lim, float c2, float m) {
  const float nm1 = (m == -INFINITY) ? 0.f : -m;
  const float2 cc = make_float2(c2, c2), nm = make_float2(nm1, nm1);
  float2 s01 = make_float2(0.f, 0.f), s23 = s01;
  p1_chunks<MASKED>(taddr, pe, lim, [&](const uint32_t(&r)[32]) {
#pragma unroll
    for (int q = 0; q < 32; q += 4) {
      const float2 a01 = tc::ffma2(make_float2(__uint_as_float(r[q]), __uint_as_float(r[q + 1])), cc, nm);
      const float2 a23 = tc::ffma2(make_float2(__uint_as_float(r[q + 2]), __uint_as_float(r[q + 3])), cc, nm);
      s01 = tc::add2(s01, make_float2(tc::ex2(a01.x), tc::ex2(a01.y)));
      s23 = tc::add2(s23, make_float2(tc::ex2(a23.x), tc::ex2(a23.y)));
    }
  });
  return (s01.x + s01.y) + (s23.x + s23.y);
}
// Pass 1: the slice added to (reference m, sum l of exp2(c2 z - m)) of the row. A row
// without a reference takes the maximum of its first chunk; a slice is then summed against
// the reference as it stands, and only where the sum leaves its range (or is a NaN, or
// there is still no reference) is the slice's maximum taken and the slice summed again.
template <bool MASKED>
__device__ __forceinline__ void p1_slice(uint32_t taddr, int pe, int lim, float c2, float& m, float& l) {
  auto refer = [&](int chunks) {
    float t = -INFINITY;
    p1_chunks<MASKED>(taddr, chunks, lim, [&](const uint32_t(&r)[32]) {
#pragma unroll
      for (int q = 0; q < 32; ++q) t = fmaxf(t, __uint_as_float(r[q]));
    });
    const float mb = t * c2;
    if (mb > m + kRescaleTau) {
      if (m != -INFINITY) l *= tc::ex2(m - mb);
      m = mb;
    }
  };
  if (__any_sync(0xffffffffu, m == -INFINITY && lim >= 0)) refer(1);
  float sum = p1_sum<MASKED>(taddr, pe, lim, c2, m);
  if (__any_sync(0xffffffffu, (m == -INFINITY && lim >= 0) || !(sum <= kRescaleSum))) {
    refer(pe);
    sum = p1_sum<MASKED>(taddr, pe, lim, c2, m);
  }
  l += sum;
}

// Pass 2: sum of exp2(c2 * z - lse2[c]) over the columns c0 <= c < c1 of a key's slice. `nlse`
// holds -lse2. Chunks outside are not looked at; in those that c0 and c1 fall into the
// exponents outside read -inf, whatever logit or normaliser they came from. A slice that is
// live throughout has a loop of its own with a fixed end: with one loop for both, the score
// call over eight requests (34423 tokens) took 150.0 us, so 146.5.
__device__ __forceinline__ float p2_slice(uint32_t taddr, const float* nlse, int c0, int c1, float c2) {
  // four partial sums (columns q mod 4), two per packed register
  float2 m01 = make_float2(0.f, 0.f), m23 = m01;
  const float2 cc = make_float2(c2, c2);
  constexpr uint32_t kAll = 0xffffffffu;
  auto chunk = [&](auto edge, int p, uint32_t live) {
    uint32_t r[32];
    tc::tmem_ld32_async(taddr + p * 32, r);
    const float4* l4 = reinterpret_cast<const float4*>(nlse + p * 32);
    tc::tmem_wait(r);
#pragma unroll
    for (int q4 = 0; q4 < 8; ++q4) {
      const float4 lv = l4[q4];
      float2 a01 = tc::ffma2(make_float2(__uint_as_float(r[4 * q4 + 0]), __uint_as_float(r[4 * q4 + 1])), cc,
                             make_float2(lv.x, lv.y));
      float2 a23 = tc::ffma2(make_float2(__uint_as_float(r[4 * q4 + 2]), __uint_as_float(r[4 * q4 + 3])), cc,
                             make_float2(lv.z, lv.w));
      if (decltype(edge)::value) {
        a01.x = (live >> (4 * q4 + 0)) & 1u ? a01.x : -INFINITY;
        a01.y = (live >> (4 * q4 + 1)) & 1u ? a01.y : -INFINITY;
        a23.x = (live >> (4 * q4 + 2)) & 1u ? a23.x : -INFINITY;
        a23.y = (live >> (4 * q4 + 3)) & 1u ? a23.y : -INFINITY;
      }
      m01 = tc::add2(m01, make_float2(tc::ex2(a01.x), tc::ex2(a01.y)));
      m23 = tc::add2(m23, make_float2(tc::ex2(a23.x), tc::ex2(a23.y)));
    }
  };
  if (c0 <= 0 && c1 >= kHalf) {
#pragma unroll 1
    for (int p = 0; p < kChunks; ++p) chunk(std::false_type{}, p, kAll);
  } else {
    const int pe = min(kChunks, (c1 + 31) >> 5);
#pragma unroll 1
    for (int p = c0 > 0 ? c0 >> 5 : 0; p < pe; ++p) {
      const int lo = c0 - p * 32, hi = c1 - p * 32;
      const uint32_t live = (lo > 0 ? kAll << lo : kAll) & (hi < 32 ? ~(kAll << hi) : kAll);
      if (live != kAll) chunk(std::true_type{}, p, live);
      else chunk(std::false_type{}, p, kAll);
    }
  }
  return (m01.x + m01.y) + (m23.x + m23.y);
}

// 2^e, -126 <= e <= 127.
__device__ __forceinline__ float pow2(int e) { return __int_as_float((127 + e) << 23); }

__device__ __forceinline__ void setup_sync(Sync& sy, int warp) {
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      tc::mbar_init(&sy.k_full[s], 1);
      tc::mbar_init(&sy.k_empty[s], 2);
    }
    for (int t = 0; t < 2; ++t) {
      tc::mbar_init(&sy.b_full[t], 1);
      tc::mbar_init(&sy.b_empty[t], 1);
    }
    for (int b = 0; b < 2; ++b)
      for (int t = 0; t < 2; ++t) {
        tc::mbar_init(&sy.acc_full[b][t], 1);
        tc::mbar_init(&sy.acc_empty[b][t], kGroupWarps);
      }
    tc::mbar_init(&sy.drain[0], 1);
    tc::mbar_init(&sy.drain[1], 1);
    sy.abort = 0;
    tc::fence_mbar_init();
  }
  if (warp == kMmaWarp) {
    tc::tmem_alloc(&sy.tmem, kTmemCols);
    tc::tmem_relinquish();
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
}

__device__ __forceinline__ void teardown(Sync& sy, int warp, uint32_t tmem, DevStatus* st) {
  tc::fence_before_sync();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, kTmemCols);
  }
  if (threadIdx.x == 0 && sy.abort) record_error(st, AVTP_ERR_TIMEOUT, static_cast<int32_t>(blockIdx.x));
}

// ---------------------------------------------------------------- the two passes' common parts
// Accumulator t (rows 128 t .. of the block) of the steps of parity b: 128 columns each.
__device__ __forceinline__ uint32_t acc_col(int b, int t) { return static_cast<uint32_t>(b * 256 + t * 128); }

// The row block of the walk's block, in halves of 128 rows (number nbl of the CTA's blocks):
// a half is loaded as soon as its last product is done.
template <int D>
__device__ __forceinline__ bool load_block(unsigned char* sB, const CUtensorMap* mapQ, int g, int R0, uint32_t nbl,
                                           Sync& sy) {
  for (int t = 0; t < 2; ++t) {
    if (nbl >= 1 && !tc::mbar_wait(&sy.b_empty[t], (nbl - 1) & 1)) return false;
    tc::mbar_arrive_expect_tx(&sy.b_full[t], static_cast<uint32_t>(a_bytes(D)));
    for (int ac = 0; ac < D / 64; ++ac)
      tc::tma_load_3d(sB + ac * (kBlk * 128) + t * (kM * 128), mapQ, ac * 64, R0 + t * kM, g, &sy.b_full[t]);
  }
  return true;
}
// Key tile load number n: 128 keys of group g from packed position key0.
template <int D>
__device__ __forceinline__ bool load_keys(unsigned char* sK, const CUtensorMap* mapK, int g, int key0, uint32_t n,
                                          Sync& sy) {
  const int sk = n % kStages;
  if (n >= kStages && !tc::mbar_wait(&sy.k_empty[sk], (n / kStages - 1) & 1)) return false;
  tc::mbar_arrive_expect_tx(&sy.k_full[sk], static_cast<uint32_t>(a_bytes(D)));
  for (int ac = 0; ac < D / 64; ++ac)
    tc::tma_load_3d(sK + sk * a_bytes(D) + ac * (kM * 128), mapK, ac * 64, g, key0, &sy.k_full[sk]);
  return true;
}
// Lets the copies in flight land before the CTA may exit.
__device__ __forceinline__ void drain_loads(Sync& sy, uint32_t nk, uint32_t nbl) {
  for (int t = 0; t < 2 && nbl >= 1; ++t) tc::mbar_wait(&sy.b_full[t], (nbl - 1) & 1);
  for (uint32_t k = (nk >= kStages ? nk - kStages : 0); k < nk; ++k)
    tc::mbar_wait(&sy.k_full[k % kStages], (k / kStages) & 1);
}

// The MMAs of half t of the block over a CTA's run, by one elected thread (the halves run on
// two warps, each at the pace of its own epilogues, up to kStages key tiles apart). Pass 1
// (the log-sum-exp) takes 128 rows as A and the key tile as B, pass 2 (the mass) the key
// tile as A and 128 rows as B, into the accumulator of the half and the step's parity. The
// next step's barriers are looked at before the commit ahead of them (behind it the look
// outlasts the MMAs queued).
template <int D, int PASS>
__device__ __forceinline__ void issue_steps(int t, Walk<PASS> cur, int n_steps, uint32_t rows, uint32_t keys,
                                            uint32_t tmem, Sync& sy) {
  constexpr uint32_t idesc = tc::idesc_bf16(kM, kM);
  constexpr uint32_t atomK = kM * 128, atomB = kBlk * 128;  // bytes per 64-element atom column
  const uint32_t rt = rows + t * (kM * 128);
  uint32_t nbl = 0;
  bool new_seg = true, bad = false, k_seen = false, acc_seen = false;
  auto wait = [&](uint64_t* bar, uint32_t parity, bool seen) {
    if (!seen && !bad) bad = !tc::mbar_wait(bar, parity);
  };
#pragma unroll 1
  for (int st = 0; st < n_steps && !bad; ++st) {
    const int sk = st % kStages, b = st & 1;
    if (t == 0) attn_stamp(PASS - 1, st, 1);
    if (new_seg) wait(&sy.b_full[t], nbl++ & 1, false);
    wait(&sy.k_full[sk], (st / kStages) & 1, k_seen);
    // its previous use (step st - 2) must have been read out
    if (st >= 2) wait(&sy.acc_empty[b][t], ((st >> 1) - 1) & 1, acc_seen);
    if (t == 0) attn_stamp(PASS - 1, st, 2);
    tc::fence_after_sync();
    const uint32_t kt = keys + sk * static_cast<uint32_t>(a_bytes(D));
    if (PASS == 1) tc::mma_rows<D>(tmem + acc_col(b, t), rt, atomB, kt, atomK, idesc);
    else tc::mma_rows<D>(tmem + acc_col(b, t), kt, atomK, rt, atomB, idesc);
    const bool more = st + 1 < n_steps;
    acc_seen = st >= 1 && tc::mbar_test_wait(&sy.acc_empty[b ^ 1][t], (((st + 1) >> 1) - 1) & 1);
    k_seen = more && tc::mbar_test_wait(&sy.k_full[(st + 1) % kStages], ((st + 1) / kStages) & 1);
    tc::mma_commit(&sy.acc_full[b][t]);
    tc::mma_commit(&sy.k_empty[sk]);
    if (!more || cur.last_of_block()) tc::mma_commit(&sy.b_empty[t]);
    new_seg = more && cur.next();
    if (t == 0) attn_stamp(PASS - 1, st, 3);
  }
  if (bad) *static_cast<volatile int*>(&sy.abort) = 1;
  // every MMA issued has completed once this arrives
  tc::mma_commit(&sy.drain[t]);
  tc::mbar_wait(&sy.drain[t], 0);
}

// ---------------------------------------------------------------- pass 1: log-sum-exp of every row
// mapQ: Qt {d, rows, Hkv}, box 64 x 128 x 1; mapK: keys {d, Hkv, T}, box 64 x 1 x 128.
template <int D>
__global__ void __launch_bounds__(kThreads, 1)
k_attn_lse(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK, AttnArgs a) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ Sync sy;
  __shared__ float2 s_mrg[2][kBlk];  // [segment parity][row]: the odd steps' (reference, sum)
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  unsigned char* sB = smem;                // the block's rows
  unsigned char* sK = smem + b_bytes(D);  // key tile s at sK + s * a_bytes(D)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // TMEM first: the next kernel's CTAs, which also allocate all of it, may start on this SM
  // from the trigger on, and wait for this grid with it
  setup_sync(sy, warp);
  pdl_trigger();
  pdl_wait();
  const uint32_t tmem = sy.tmem;
  volatile int* abort_flag = &sy.abort;
  const int4 start = a.cta_start[blockIdx.x];
  const int n_steps = a.st->layout_ok ? start.w : 0;
  Walk<1> cur{};
  if (n_steps > 0) cur.init(a, start);

  if (n_steps == 0) {
    // nothing to do (or a layout that did not validate)
  } else if (warp == kTmaWarp) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      tc::tma_prefetch_map(&mapQ);
      tc::tma_prefetch_map(&mapK);
      uint32_t nk = 0, nbl = 0;  // key tile loads and block loads issued so far
      bool new_seg = true;
      for (int st = 0; st < n_steps && !*abort_flag; ++st) {
        if (!load_keys<D>(sK, &mapK, cur.g, cur.blk.key0 + cur.j * kM, nk, sy)) { *abort_flag = 1; break; }
        attn_stamp(0, st, 0);
        ++nk;
        if (new_seg) {
          if (!load_block<D>(sB, &mapQ, cur.g, cur.blk.R0, nbl, sy)) { *abort_flag = 1; break; }
          ++nbl;
        }
        new_seg = st + 1 < n_steps && cur.next();
      }
      drain_loads(sy, nk, nbl);
    }
  } else if (warp >= kMmaWarp) {
    // ------------------------------------------------------------ MMA issuers: rows (A) x keys (B)
    if (tc::elect_one())
      issue_steps<D, 1>(warp - kMmaWarp, cur, n_steps, tc::smem_u32(sB), tc::smem_u32(sK), tmem, sy);
  } else {
    // ------------------------------------------------------------ epilogue, 4 warps per accumulator
    // Warp w reads TMEM lanes 32(w%4)..+31 (its rows of A tile t) of the accumulators of the
    // steps of parity b; the two parities of a row meet in shared memory when the row's
    // partial is written.
    const int quad = warp & 3, t = (warp >> 2) & 1, b = warp >> 3;
    const int lrow = t * kM + quad * 32 + lane;  // row of the block
    const uint32_t taddr = tmem + (static_cast<uint32_t>(quad * 32) << 16) + acc_col(b, t);
    const float c2 = a.c2;
    // After a wait that gave up (ok false) the warp keeps walking the same steps, skipping
    // every wait and TMEM read, so that the named barriers still line up.
    const int F1 = a.meta[0], C1 = a.meta[1];
    int qpos = -1, par = 0;
    bool new_seg = true, ok = true;
    float2* dst = nullptr;         // this row's partial of the current block
    float m = -INFINITY, l = 0.f;  // reference and sum, log2 domain
    for (int st = 0; st < n_steps; ++st) {
      if (new_seg) {
        const int64_t F0 = static_cast<int64_t>(cur.g) * F1 + cur.blk.s1;
        const int slot = static_cast<int>(blockIdx.x - F0 / C1);
        const bool live = lrow < cur.blk.rows;
        qpos = live ? a.text_idx[(cur.blk.R0 + lrow) / a.G] : -1;
        dst = live ? a.p1_part + (static_cast<int64_t>(cur.g * cur.NB + cur.b) * kBlk + lrow) * kAttnMaxChunks + slot
                   : nullptr;
        m = -INFINITY;
        l = 0.f;
      }
      if ((st & 1) == b) {
        if (ok && !tc::mbar_wait_warp(&sy.acc_full[b][t], (st >> 1) & 1)) {
          if (lane == 0) *abort_flag = 1;
          ok = false;
        }
        if (warp == 0 && lane == 0) attn_stamp(0, st, 4);
        tc::fence_after_sync();
        // columns 0..lim are visible to the row
        const int lim = qpos - (cur.blk.key0 + cur.j * kM);
        const int lim_max = __reduce_max_sync(0xffffffffu, lim);
        if (ok && lim_max >= 0) {
          if (__all_sync(0xffffffffu, lim >= kM - 1)) {
            p1_slice<false>(taddr, kChunks, lim, c2, m, l);
          } else {
            // 32-column chunks 0 .. pe-1 hold a visible column for some lane
            p1_slice<true>(taddr, min(kChunks, (lim_max >> 5) + 1), lim, c2, m, l);
          }
        }
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&sy.acc_empty[b][t]);
        if (warp == 0 && lane == 0) attn_stamp(0, st, 5);
      }
      const bool more = st + 1 < n_steps;
      if (!more || cur.last_of_block()) {
        // the block ends here for this CTA: merge the step parities and write the partial
        par ^= 1;
        if (b == 1) s_mrg[par][lrow] = make_float2(m, l);
        bar_epi();
        if (b == 0 && dst != nullptr) {
          const float2 o = s_mrg[par][lrow];
          const float M = fmaxf(m, o.x);
          const float L = (M == -INFINITY) ? 0.f : l * tc::ex2(m - M) + o.y * tc::ex2(o.x - M);
          *dst = make_float2(M, L);
        }
      }
      new_seg = more && cur.next();
    }
  }
  teardown(sy, warp, tmem, a.st);
}

// ---------------------------------------------------------------- pass 2: probability mass of every visual key
// mapK: keys {d, Hkv, T}, box 64 x 1 x 128; mapQ: Qt {d, rows, Hkv}, box 64 x 128 x 1.
template <int D>
__global__ void __launch_bounds__(kThreads, 1)
k_attn_mass(const __grid_constant__ CUtensorMap mapK, const __grid_constant__ CUtensorMap mapQ, AttnArgs a) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ Sync sy;
  __shared__ __align__(16) float s_lse[2][2][kBlk];  // -lse2, [step parity][block parity][row of the block]
  // key masses of the last steps of a parity, per row half, flushed to the accumulator every
  // kMassWindow of them (global atomics inside the step loop would be waited for by the
  // next step's TMEM fence)
  __shared__ float s_mass[2][kMassWindow][2][kM];
  __shared__ int s_tile[2][kMassWindow], s_nk[2][kMassWindow];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  unsigned char* sB = smem;                // the block's rows
  unsigned char* sK = smem + b_bytes(D);  // key tile s at sK + s * a_bytes(D)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // TMEM first: the next kernel's CTAs, which also allocate all of it, may start on this SM
  // from the trigger on, and wait for this grid with it
  setup_sync(sy, warp);
  pdl_trigger();
  pdl_wait();
  const uint32_t tmem = sy.tmem;
  volatile int* abort_flag = &sy.abort;
  const int4 start = a.cta_start[gridDim.x + blockIdx.x];
  const int n_steps = a.st->layout_ok ? start.w : 0;
  Walk<2> cur{};
  if (n_steps > 0) cur.init(a, start);

  if (n_steps == 0) {
    // nothing to do (or a layout that did not validate)
  } else if (warp == kTmaWarp) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      tc::tma_prefetch_map(&mapQ);
      tc::tma_prefetch_map(&mapK);
      uint32_t nk = 0, nbl = 0;  // key tile loads and block loads issued so far
      bool new_seg = true;
      int key0 = a.tile_info[cur.blk.tile0 + cur.j].x;
      for (int st = 0; st < n_steps && !*abort_flag; ++st) {
        if (!load_keys<D>(sK, &mapK, cur.g, key0, nk, sy)) { *abort_flag = 1; break; }
        attn_stamp(1, st, 0);
        ++nk;
        const int g = cur.g, R0 = cur.blk.R0;
        const bool load = new_seg;
        new_seg = st + 1 < n_steps && cur.next();
        if (st + 1 < n_steps) key0 = a.tile_info[cur.blk.tile0 + cur.j].x;
        if (load) {
          if (!load_block<D>(sB, &mapQ, g, R0, nbl, sy)) { *abort_flag = 1; break; }
          ++nbl;
        }
      }
      drain_loads(sy, nk, nbl);
    }
  } else if (warp >= kMmaWarp) {
    // ------------------------------------------------------------ MMA issuers: keys (A) x rows (B)
    if (tc::elect_one())
      issue_steps<D, 2>(warp - kMmaWarp, cur, n_steps, tc::smem_u32(sB), tc::smem_u32(sK), tmem, sy);
  } else {
    // ------------------------------------------------------------ epilogue, 4 warps per accumulator
    // Warp w reads TMEM lanes 32(w%4)..+31 (its keys) of the accumulators of row half `half`
    // of the steps of parity t; the halves of a key's mass meet at the flush into the
    // fixed-point accumulator.
    const int quad = warp & 3, half = (warp >> 2) & 1, t = warp >> 3;
    const int klane = quad * 32 + lane;                       // key of the tile = TMEM lane
    const int etid = static_cast<int>(threadIdx.x) - t * kSetThreads;  // 0 .. 255
    const uint32_t taddr = tmem + (static_cast<uint32_t>(quad * 32) << 16) + acc_col(t, half);
    const float c2 = a.c2;
    int par = 0, c1 = 0;
    bool new_seg = true, ok = true;  // ok: see k_attn_lse
    const int F1 = a.meta[0], C1 = a.meta[1];
    int4 tile = make_int4(0, 0, 0, 0);
    if (t == 1 && n_steps > 1) cur.next();
    if (t < n_steps) tile = a.tile_info[cur.blk.tile0 + cur.j];
    for (int st = t, w = 0; st < n_steps; st += 2) {
      if (new_seg) {
        c1 = cur.blk.rows;
        const int g = cur.g;
        float lse_own = INFINITY;  // lse2 of this thread's row of the block (row etid)
        if (etid < c1) {
          const int64_t row = static_cast<int64_t>(cur.blk.R0) + etid;
          if (a.lse_rows != nullptr) {
            lse_own = a.lse_rows[static_cast<int64_t>(g) * a.rows + row];
          } else {
            // merge the row's pass-1 partials, eight loads in flight at a time
            const int64_t F0 = static_cast<int64_t>(g) * F1 + cur.blk.s1;
            const int steps = cur.blk.n1;
            const int n = static_cast<int>((F0 + steps - 1) / C1 - F0 / C1) + 1;
            const float2* src = a.p1_part + (static_cast<int64_t>(g * cur.NB + cur.b) * kBlk + etid) * kAttnMaxChunks;
            float M = -INFINITY, L = 0.f;
            for (int k0 = 0; k0 < n; k0 += 8) {
              float2 pk[8];
#pragma unroll
              for (int k = 0; k < 8; ++k) pk[k] = (k0 + k < n) ? src[k0 + k] : make_float2(-INFINITY, 0.f);
#pragma unroll
              for (int k = 0; k < 8; ++k) {
                const float Mn = fmaxf(M, pk[k].x);
                if (Mn != -INFINITY) {
                  L = L * tc::ex2(M - Mn) + pk[k].y * tc::ex2(pk[k].x - Mn);
                  M = Mn;
                }
              }
            }
            lse_own = M + log2f(L);
          }
        }
        // thread etid's row is one that its own accumulator's threads read; rows past the
        // request's (another request's, or none) are left out by p2_slice
        par ^= 1;
        s_lse[t][par][etid] = -lse_own;
        bar_acc(t, half);
      }
      if (ok && !tc::mbar_wait_warp(&sy.acc_full[t][half], (static_cast<uint32_t>(st) >> 1) & 1)) {
        if (lane == 0) *abort_flag = 1;
        ok = false;
      }
      if (warp == 0 && lane == 0) attn_stamp(1, st, 4);
      tc::fence_after_sync();
      // first row of the block that sees the tile's image: its queries follow it
      const int tile_id = cur.blk.tile0 + cur.j;
      const int c0 = tile.z * a.G - cur.blk.R0;
      // does this warp's row half hold a visible row? (uniform over its group)
      const bool any = c0 < (half + 1) * kHalf && c1 > half * kHalf;
      float mass = 0.f;
      if (ok && any) mass = p2_slice(taddr, &s_lse[t][par][half * kHalf], c0 - half * kHalf, c1 - half * kHalf, c2);
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&sy.acc_empty[t][half]);
      if (warp == 0 && lane == 0) attn_stamp(1, st, 5);
      s_mass[t][w][half][klane] = mass;
      if (etid == 0) {
        s_tile[t][w] = tile_id;
        s_nk[t][w] = tile.y;
      }
      if (++w == kMassWindow || st + 2 >= n_steps) {
        // flush: one fixed-point integer add per (step, key), both column halves summed
        // in fp32 first (integer adds: the result does not depend on their order)
        bar_set(t);
        const float mass_scale = pow2(a.meta[5]);
        for (int e = etid; e < w * kM; e += kSetThreads) {
          const int ws = e / kM, k = e % kM;
          if (k < s_nk[t][ws]) {
            const float m = s_mass[t][ws][0][k] + s_mass[t][ws][1][k];
            unsigned long long* dst = a.mass + static_cast<int64_t>(s_tile[t][ws]) * kM + k;
            if (m <= static_cast<float>(1 << kAttnBlockMassBits)) {
              atomicAdd(dst, static_cast<unsigned long long>(__float2ll_rn(m * mass_scale)));
            } else {
              atomicOr(dst, kMassNotFinite);  // NaN or inf inputs: the key scores NaN (bit 63; finite adds never reach it)
            }
          }
        }
        bar_set(t);
        w = 0;
      }
      // two steps on, past the other parity's
      new_seg = false;
      for (int k = 0; k < 2 && st + 1 + k < n_steps; ++k) new_seg |= cur.next();
      if (st + 2 < n_steps) tile = a.tile_info[cur.blk.tile0 + cur.j];
    }
  }
  teardown(sy, warp, tmem, a.st);
}

// ---------------------------------------------------------------- repacking of the text queries
// Qt[g][o*G + j][:] = q[text_idx[o], g*G + j, :]; with a supplied LSE also
// lse_rows[g][o*G + j] = lse[g*G + j][text_idx[o]] * log2(e). One thread per 16 bytes.
// Also clears the per-key mass accumulator of pass 2.
__global__ void __launch_bounds__(256)
k_attn_pack(const __nv_bfloat16* __restrict__ q, int64_t q_stride, int Hq, int G, int d,
            const int32_t* __restrict__ text_idx, const int32_t* __restrict__ text_cu, int R, int64_t rows,
            __nv_bfloat16* __restrict__ qt, const float* __restrict__ lse, int64_t lse_stride,
            float* __restrict__ lse_rows, unsigned long long* __restrict__ mass, int64_t n_mass, const DevStatus* st) {
  pdl_wait();
  pdl_trigger();
  if (!st->layout_ok) return;
  const int64_t n_text = text_cu[R];
  const int vec = d / 8;
  const int64_t total = n_text * Hq * vec;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t tid0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  for (int64_t u = tid0; u < n_mass; u += stride) mass[u] = 0ull;
  for (int64_t u = tid0; u < total; u += stride) {
    const int c = static_cast<int>(u % vec);
    const int64_t oh = u / vec;
    const int h = static_cast<int>(oh % Hq);
    const int64_t o = oh / Hq;
    const int g = h / G, j = h - g * G;
    const int64_t pos = text_idx[o];
    const int64_t row = o * G + j;
    const uint4 v = *reinterpret_cast<const uint4*>(q + pos * q_stride + static_cast<int64_t>(h) * d + c * 8);
    *reinterpret_cast<uint4*>(qt + (static_cast<int64_t>(g) * rows + row) * d + c * 8) = v;
    if (lse != nullptr && c == 0) lse_rows[static_cast<int64_t>(g) * rows + row] = lse[h * lse_stride + pos] * kLog2e;
  }
}

// ---------------------------------------------------------------- finalize
// One CTA per key tile (128 keys of one image): s_t = mass_t * 2^-bits / (Hq * |Q_r|), and
// the tile's fixed-point score sum added to its image's sum with one atomic.
__global__ void __launch_bounds__(kM)
k_attn_finalize(const unsigned long long* __restrict__ mass, const int32_t* __restrict__ ktile_cu,
                const int32_t* __restrict__ ktile_img, const int4* __restrict__ tile_info, int Hq,
                const int32_t* __restrict__ text_cu, const int32_t* __restrict__ meta, int NI, float* __restrict__ scores,
                int64_t* __restrict__ img_sums, const DevStatus* st) {
  __shared__ long long s_part[kM / 32];
  pdl_wait();
  pdl_trigger();
  if (!st->layout_ok) return;
  for (int tile = blockIdx.x; tile < ktile_cu[NI]; tile += gridDim.x) {
    const int i = ktile_img[tile];
    const int4 info = tile_info[tile];
    const unsigned long long m = mass[static_cast<int64_t>(tile) * kM + threadIdx.x];
    const int nq = text_cu[info.w + 1] - text_cu[info.w];  // the request's queries
    const float unit = pow2(-meta[5]);
    long long fx = 0;
    if (static_cast<int>(threadIdx.x) < info.y) {
      float s = 0.f;
      if (nq > 0) {
        if (m & kMassNotFinite) {
          s = __int_as_float(0x7fc00000);
        } else {
          s = __ll2float_rn(static_cast<long long>(m)) * unit;
          s = s / static_cast<float>(static_cast<int64_t>(Hq) * nq);
        }
      }
      scores[static_cast<int64_t>(info.x) + threadIdx.x] = s;
      fx = fixed_point_score(s);
    }
    fx = warp_sum(fx);
    if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = fx;
    __syncthreads();
    if (threadIdx.x == 0) {
      long long sum = 0;
#pragma unroll
      for (int w = 0; w < kM / 32; ++w) sum += s_part[w];
      atomicAdd(reinterpret_cast<unsigned long long*>(img_sums + i), static_cast<unsigned long long>(sum));
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- host side
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }();
  return fn;
}

// A 3-D bf16 tensor map with 128-byte swizzle and a box of 64 x box1 x box2 elements.
bool make_map(CUtensorMap* m, const void* base, uint64_t d0, uint64_t d1, uint64_t d2, uint64_t stride1_bytes,
              uint64_t stride2_bytes, uint32_t box1, uint32_t box2) {
  auto fn = encode_fn();
  if (fn == nullptr) return false;
  const cuuint64_t dims[3] = {d0, d1, d2};
  const cuuint64_t strides[2] = {stride1_bytes, stride2_bytes};
  const cuuint32_t box[3] = {64, box1, box2};
  const cuuint32_t es[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

cudaError_t launch_score_attn(const avtp_layout_t& L, const avtp_score_args_t& sa, float* scores,
                              int64_t* img_sums, void* ws, const WsPlan& p, cudaStream_t s) {
  if (L.n_images == 0 || L.n_tokens == 0) return cudaSuccess;
  const int d = sa.head_dim, Hq = sa.n_q_heads, Hkv = sa.n_kv_heads;
  const AttnPlan plan = attn_plan(L, sa);
  static PerDevice attrs;
  cudaError_t ae = once_per_device(attrs, [](int, int*) {
    auto allow = [](auto kernel, size_t bytes) {
      return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
    };
    cudaError_t e = allow(k_attn_lse<128>, attn_smem_bytes(128));
    if (e == cudaSuccess) e = allow(k_attn_lse<64>, attn_smem_bytes(64));
    if (e == cudaSuccess) e = allow(k_attn_mass<128>, attn_smem_bytes(128));
    if (e == cudaSuccess) e = allow(k_attn_mass<64>, attn_smem_bytes(64));
    return e;
  });
  if (ae != cudaSuccess) return ae;
  DevStatus* st = ws_at<DevStatus>(ws, p.status);
  AttnArgs a{};
  a.text_idx = ws_at<int32_t>(ws, p.text_idx);
  a.blk_info = ws_at<int4>(ws, p.blk_info);
  a.tile_info = ws_at<int4>(ws, p.tile_info);
  a.cta_start = ws_at<int4>(ws, p.cta_start);
  a.meta = ws_at<int32_t>(ws, p.meta);
  float* lse_rows = sa.lse != nullptr ? ws_at<float>(ws, p.lse_rows) : nullptr;
  a.lse_rows = lse_rows;
  a.p1_part = sa.lse == nullptr ? ws_at<float2>(ws, p.p1_part) : nullptr;
  a.mass = ws_at<unsigned long long>(ws, p.mass);
  a.rows = plan.rows;
  a.G = plan.G;
  a.c2 = sa.softmax_scale * kLog2e;
  a.st = st;
  __nv_bfloat16* qt = ws_at<__nv_bfloat16>(ws, p.qt);

  // tensor maps: keys {d, Hkv, T} (token stride k_stride), packed queries {d, rows, Hkv}
  CUtensorMap mk, mq;
  const uint64_t ks = static_cast<uint64_t>(sa.k_stride) * 2, qs = static_cast<uint64_t>(plan.rows) * d * 2;
  if (!make_map(&mk, sa.k, d, Hkv, L.n_tokens, static_cast<uint64_t>(d) * 2, ks, 1, kM) ||
      !make_map(&mq, qt, d, plan.rows, Hkv, static_cast<uint64_t>(d) * 2, qs, kM, 1))
    return cudaErrorInvalidValue;

  const int sms = plan.grid;
  {
    const int64_t want = (plan.max_text * Hq * (d / 8) + 255) / 256;
    const int64_t cap = static_cast<int64_t>(sms) * 8;
    const int grid = static_cast<int>(want < 1 ? 1 : (want < cap ? want : cap));
    cudaError_t e = launch_kernel(k_attn_pack, dim3(grid), dim3(256), 0, s, /*pdl=*/true,
                                  static_cast<const __nv_bfloat16*>(sa.q), sa.q_stride, Hq, plan.G, d, a.text_idx,
                                  static_cast<const int32_t*>(ws_at<int32_t>(ws, p.text_cu)), L.n_requests, plan.rows, qt, sa.lse, sa.lse_stride, lse_rows, a.mass,
                                  plan.n_ktiles_max * kM, static_cast<const DevStatus*>(st));
    if (e != cudaSuccess) return e;
  }
  if (sa.lse == nullptr) {
    cudaError_t e = launch_kernel(d == 128 ? k_attn_lse<128> : k_attn_lse<64>, dim3(sms), dim3(kThreads),
                                  attn_smem_bytes(d), s, /*pdl=*/true, mq, mk, a);
    if (e != cudaSuccess) return e;
  }
  cudaError_t e =
      launch_kernel(d == 128 ? k_attn_mass<128> : k_attn_mass<64>, dim3(sms), dim3(kThreads), attn_smem_bytes(d), s,
                    /*pdl=*/true, mk, mq, a);
  if (e != cudaSuccess) return e;
  return launch_attn_finalize(L, sa, scores, img_sums, ws, p, plan, s);
}

cudaError_t launch_attn_finalize(const avtp_layout_t& L, const avtp_score_args_t& sa, float* scores,
                                 int64_t* img_sums, void* ws, const WsPlan& p, const AttnPlan& plan, cudaStream_t s) {
  const int64_t cap = static_cast<int64_t>(device_sm_count()) * 8;
  const int grid3 = static_cast<int>(plan.n_ktiles_max < cap ? plan.n_ktiles_max : cap);
  return launch_kernel(k_attn_finalize, dim3(grid3), dim3(kM), 0, s, /*pdl=*/true,
                       static_cast<const unsigned long long*>(ws_at<unsigned long long>(ws, p.mass)),
                       static_cast<const int32_t*>(ws_at<int32_t>(ws, p.ktile_cu)),
                       static_cast<const int32_t*>(ws_at<int32_t>(ws, p.ktile_img)),
                       static_cast<const int4*>(ws_at<int4>(ws, p.tile_info)), sa.n_q_heads,
                       static_cast<const int32_t*>(ws_at<int32_t>(ws, p.text_cu)),
                       static_cast<const int32_t*>(ws_at<int32_t>(ws, p.meta)), L.n_images, scores, img_sums,
                       static_cast<const DevStatus*>(ws_at<DevStatus>(ws, p.status)));
}

}  // namespace avtp

extern "C" avtp_status_t avtp_score_timeline(int32_t pass, int64_t* out, int32_t max_steps) {
#ifdef AVTP_TIMELINE
  if (out == nullptr || max_steps < 1 || (pass != 1 && pass != 2)) return AVTP_ERR_INVALID_ARG;
  const int n = max_steps < avtp::kAttnTlSteps ? max_steps : avtp::kAttnTlSteps;
  const size_t row = static_cast<size_t>(avtp::kAttnTlSteps) * avtp::kAttnTlSlots * sizeof(long long);
  return cudaMemcpyFromSymbol(out, avtp::g_attn_tl, static_cast<size_t>(n) * avtp::kAttnTlSlots * sizeof(long long),
                              (pass - 1) * row) == cudaSuccess
             ? AVTP_OK
             : AVTP_ERR_CUDA;
#else
  (void)pass;
  (void)out;
  (void)max_steps;
  return AVTP_ERR_UNSUPPORTED;
#endif
}
