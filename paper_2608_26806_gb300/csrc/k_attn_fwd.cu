// The pruning layer's causal attention forward (paper §3.2: the FlashAttention-style
// forward whose natural-log normaliser the text-attention criterion reuses), on a
// varlen-packed batch with grouped-query heads g(h) = h / (Hq / Hkv), head_dim 64 or 128:
//   O[t, h]   = sum_{u visible to t} softmax_u(scale * q[t, h] . k[u, g(h)]) v[u, g(h)]
//   lse[h, t] = ln sum_{u visible to t} exp(scale * q[t, h] . k[u, g(h)])
// where u is visible to t when it lies in t's request and u <= t.
//
// A unit of work is two slots of 128 query rows that share a KV group's keys and values: the same
// query tile of two neighbouring heads of the group when the group has an even number of
// heads (both slots then do the same work), else two neighbouring query tiles of one head.
// Query tiles and key blocks of 128 start at the request's first token, so only a slot's
// last block, its diagonal one, is masked.
//
// Per slot and key block j:
//   S_j = Q K_j^T           tcgen05, M = 128 queries, N = 128 keys, both operands from
//                           shared memory
//   P_j = exp2(c2 S_j - m)  softmax: a thread per row; bf16, two per column, over S_j's
//                           first 64 TMEM columns
//   O  += P_j V_j           tcgen05 with A (P) read from TMEM, M = 128, N = d, K = 128 keys;
//                           V is the MN-major operand, so the TMA's [key][channel] rows are
//                           used as they lie and no transposed copy of the values is made
// with c2 = scale * log2(e) and m the row's reference.
//
// What bounds it: the tensor core, and at full load the power limit. A 128 x 128 x 16 step
// takes 64 cycles whatever the operands' place (1024 per slot and block at d = 128), the
// exponentials 512 at 32 a cycle. The MMA thread issues, slot by slot, P_j V_j and then
// S_{j+1}: while one slot's softmax runs (from S ready to P written about 1100 cycles) the
// tensor core has the other slot's 1024 cycles of work, and the keys and values brought to
// the SM serve 256 rows. The MMAs of one thread run in order, so S_{j+1} may overwrite
// P_j's columns right behind P_j V_j. P is handed over in two halves of 64 keys, so P_j V_j
// starts before the second half's exponentials are done.
//
// The softmax takes no maximum of a half it can do without: it computes P against the row's
// reference and sums it, and only a sum above 2^14 (or no reference yet, or a NaN) makes it
// take the maximum, move the reference and start the half again. The reference is then at
// most about 14 (log2 units) below the running maximum, which scales P and O alike and
// costs no precision in either (against 64 bits: O and the LSE are as far off as with a
// maximum of every block).
//
// The kernel is persistent, a CTA per SM, units taken from a counter in the packed order from
// its end, so that within a request those with the most key blocks come first: the next unit's
// queries and first keys arrive while the last block of the one before is under way, and its S
// runs during the rows' way out. Against a CTA per unit: 206 -> 196 us the call over 5960
// tokens (28 heads), 1104 -> 1028 us over eight requests of 34423 tokens.
//
// Measured (32 query heads, 8 KV heads, d = 128, one request of 10368 tokens, this kernel
// alone): 480 us at the full clock, 1830 TFLOP/s; up to 580 us where the power limit lowers
// the clock. One slot per CTA with Q and P in TMEM and an exchange of half maxima had taken
// 900 us. What made the difference: two slots a unit 726 us, no maximum 690, descriptors in
// uniform registers (elect_one) 562, barriers looked at ahead of the commits 500, persistent
// 480. Two issuing warps, one a slot, ran both slots in step and the tensor core idle
// between (+15 %).
//
// Warps 0-3: softmax and epilogue of slot 0, warps 4-7 of slot 1 (warp w owns rows
// 32 (w % 4) .. + 31, the TMEM lanes it can reach). Warp 8 issues the TMA loads: Q once,
// then K_0, V_0, K_1, V_1, ... through a ring of stages. Warp 9 owns TMEM and issues the
// MMAs. TMEM: S and P of slot s in columns 128 s .. + 127, its O in 256 + 128 s .. + d.
// Every wait is bounded; a CTA whose wait gives up records AVTP_ERR_TIMEOUT and returns.
#include <cudaTypedefs.h>

#include <type_traits>

#include "avtp_fwd.cuh"
#include "avtp_tc.cuh"

namespace avtp {
namespace {

constexpr int kQT = 128;  // query rows per slot (MMA M, TMEM lanes)
constexpr int kKB = 128;  // keys per block (MMA N of Q K^T, K of P V)
constexpr int kThreads = 320;
constexpr int kSlotWarps = 4;
constexpr int kTmaWarp = 8;
constexpr int kMmaWarp = 9;
constexpr int kStages = 4;  // key or value blocks in shared memory
constexpr int kNearRequests = 32;  // unit prefixes of up to this many requests are formed here (a lane each)
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kSCol = 0;    // S (and P) of slot s at kSCol + 128 s
constexpr uint32_t kOCol = 256;  // O of slot s at kOCol + 128 s
// A half's sum of P above kRescaleSum moves the row's reference, if its maximum exceeds the
// reference by more than kRescaleTau (log2 units).
constexpr float kRescaleSum = 16384.f;
constexpr float kRescaleTau = 8.f;
constexpr float kLn2 = 0.6931471805599453f;
constexpr float kLog2e = 1.4426950408889634f;

// One slot's queries, and one key or value block: 128 rows of d bf16, as d / 64 panels of
// 128 rows x 128 bytes in the 128-byte swizzle.
__host__ __device__ constexpr uint32_t tile_bytes(int d) { return static_cast<uint32_t>(kQT) * d * 2; }
constexpr uint32_t kPanel = kQT * 128;
constexpr uint32_t kOutStage = 2048;  // a warp's 32 rows x 16 columns of O on their way out, two of them
__host__ __device__ constexpr size_t fwd_smem_bytes(int d) {
  const size_t need = 1024 + static_cast<size_t>(2 + kStages) * tile_bytes(d) + 4 * kSlotWarps * kOutStage;
  // more than half the SM's shared memory, so that no second CTA (and its 512 TMEM
  // columns) shares an SM
  return need > 116 * 1024 ? need : 116 * 1024;
}
static_assert(fwd_smem_bytes(128) <= 226 * 1024, "shared memory of one CTA");

struct FwdSync {
  uint64_t u_full[2], u_empty[2];  // a unit's place in `unit` written / read by everyone
  uint64_t q_full, q_empty;
  uint64_t kv_full[kStages], kv_empty[kStages];
  uint64_t s_full[2];     // S of a slot written by the MMA
  uint64_t p_full[2][2];  // half of a slot's P written by the softmax (and S read out)
  uint64_t pv_done[2][2]; // P V complete up to that half of a block (phase j: block j)
  uint64_t drain;
  // per request, when they are few: units before it, its first token and its end
  int32_t pre[kNearRequests + 1], start[kNearRequests], end[kNearRequests];
  int4 unit[2];           // request's first token and end, unit's first query, head pair or head (-1: no more)
  uint32_t tmem;
  int abort;
};

struct FwdArgs {
  const int32_t* cu;
  int R;
  int64_t T;
  const int32_t* qtile_cu;  // query tiles (pairs of them when a CTA takes two tiles) per request, prefix
  int Hq, G;
  float c2;
  float* o;
  int64_t o_stride;
  float* lse;
  int64_t lse_stride;
  DevStatus* st;
};

// 32 consecutive fp32 columns of this thread's TMEM lane, stored; complete after
// tmem_wait_st().
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
      "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
      "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// Diagnostic timeline build (-DAVTP_TIMELINE): clock stamps of slot 0 of the grid's first CTA
// (the last request's last tile), per key block j. Stamps: 0-4 from softmax warp 0
// (loop top, S ready, P of the first half computed, of the second half, P handed over); 5-9
// from the MMA thread (S_j: entry, issued; P_j V_j: entry, operands ready, issued). Read with
// avtp_forward_timeline().
#ifdef AVTP_TIMELINE
constexpr int kFwdTlBlocks = 256;
constexpr int kFwdTlSlots = 10;
__device__ long long g_fwd_tl[kFwdTlBlocks][kFwdTlSlots];
#endif
__device__ __forceinline__ void fwd_stamp(int j, int slot) {
#ifdef AVTP_TIMELINE
  if (blockIdx.x == 0 && j < kFwdTlBlocks) g_fwd_tl[j][slot] = clock64();
#else
  (void)j;
  (void)slot;
#endif
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  const __nv_bfloat162 b = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&b);
}
// The larger of three (PTX max with three sources, sm_100 and later); NaN only if all are.
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// 16 fp32 columns x 32 rows of shared memory (64-byte swizzle) to the output tensor.
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, const void* src, int x, int y, int z) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(x), "r"(y), "r"(z), "r"(tc::smem_u32(src))
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Until all but the last N stores committed have read their shared memory.
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// A unit of a CTA's work, seen by every role: two slots of 128 query rows on one key stream.
template <bool kHeads>
struct Unit {
  int cu, end, q, x;  // request's first token and end, first query, head pair (kHeads) or head
  __device__ __forceinline__ int q0(int s) const { return kHeads ? q : q + s * kQT; }
  __device__ __forceinline__ int head(int s) const { return kHeads ? 2 * x + s : x; }
  __device__ __forceinline__ int last(int s) const { return min(q0(s) + kQT, end) - 1; }
  // key blocks of slot s (0: an empty slot), and of both
  __device__ __forceinline__ int blocks(int s) const { return q0(s) < end ? (q0(s) - cu) / kKB + 1 : 0; }
  __device__ __forceinline__ int blocks() const { return max(blocks(0), blocks(1)); }
};

// ---------------------------------------------------------------- forward
// mapQ: q {d, Hq, T}, mapK: k {d, Hkv, T}, mapV: v {d, Hkv, T}, box 64 x 1 x 128 each;
// mapO: o {d, Hq, T} fp32, box 16 x 1 x 32. kHeads: a unit's slots are two heads of a tile.
// Persistent: a CTA takes the unit of its index, then units from a counter. The barriers'
// phases run on across units; a unit takes a whole number of turns of the ring of stages
// (one odd pair of stages is passed on empty), so that a step's stages stay constants.
template <int D, bool kHeads>
__global__ void __launch_bounds__(kThreads, 1)
k_attn_fwd(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
           const __grid_constant__ CUtensorMap mapV, const __grid_constant__ CUtensorMap mapO, FwdArgs a) {
  extern __shared__ unsigned char smem_raw[];
  __shared__ FwdSync sy;
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  constexpr uint32_t kTile = tile_bytes(D);
  unsigned char* sQ = smem;                 // slot s at sQ + s * kTile
  unsigned char* sKV = smem + 2 * kTile;    // stage b at sKV + b * kTile
  unsigned char* sO = sKV + kStages * kTile;  // warp w at sO + 2 w * kOutStage
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      tc::mbar_init(&sy.kv_full[s], 1);
      tc::mbar_init(&sy.kv_empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      tc::mbar_init(&sy.u_full[s], 1);
      tc::mbar_init(&sy.u_empty[s], 2 * kSlotWarps + 1);
      tc::mbar_init(&sy.s_full[s], 1);
      for (int h = 0; h < 2; ++h) {
        tc::mbar_init(&sy.p_full[s][h], kSlotWarps);
        tc::mbar_init(&sy.pv_done[s][h], 1);
      }
    }
    tc::mbar_init(&sy.q_full, 1);
    tc::mbar_init(&sy.q_empty, 1);
    tc::mbar_init(&sy.drain, 1);
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
  // TMEM before the trigger: a later kernel that allocates it too may start on this SM then
  pdl_trigger();
  // Batches of up to kNearRequests requests need nothing of the validation kernel to begin:
  // the units follow from cu_seqlens, clamped into the batch, and the kernel runs beside
  // validation, which only the first write of a row (and the unit counter) waits for. 6 to
  // 9 us of a call: a few hundred tokens 16.4 -> 11.4 us.
  const bool near = a.R <= kNearRequests;
  if (!near) pdl_wait();
  const uint32_t tmem = sy.tmem;
  volatile int* abort_flag = &sy.abort;
  auto read_unit = [&](int us) {
    const int4 v = sy.unit[us];
    return Unit<kHeads>{v.x, v.y, v.z, v.w};
  };

  if (warp == kTmaWarp) {
    // ------------------------------------------------------------ units and TMA loads
    constexpr int kUnitRows = kHeads ? kQT : 2 * kQT;
    if (near) {
      const int64_t lo = lane < a.R ? min(max(static_cast<int64_t>(a.cu[lane]), int64_t(0)), a.T) : 0;
      const int64_t hi = lane < a.R ? min(max(static_cast<int64_t>(a.cu[lane + 1]), lo), a.T) : 0;
      int incl = static_cast<int>((hi - lo + kUnitRows - 1) / kUnitRows);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      sy.pre[lane + 1] = incl;
      sy.start[lane] = static_cast<int32_t>(lo);
      sy.end[lane] = static_cast<int32_t>(hi);
      if (lane == 0) sy.pre[0] = 0;
      __syncwarp();
    }
    if (lane == 0) {
      tc::tma_prefetch_map(&mapQ);
      tc::tma_prefetch_map(&mapK);
      tc::tma_prefetch_map(&mapV);
      const int n_sub = kHeads ? a.Hq / 2 : a.Hq;
      const int32_t* pre = near ? sy.pre : a.qtile_cu;
      // units of one head (pair); more than a batch can have: offsets that validation refuses
      int n_rows = near ? pre[a.R] : (a.st->layout_ok ? pre[a.R] : 0);
      if (n_rows > a.T / kUnitRows + a.R) n_rows = 0;
      const int64_t total = static_cast<int64_t>(n_rows) * n_sub;
      int64_t u = blockIdx.x;
      int uc = 0, n = 0;  // units published, ring slots used (K_0, V_0, K_1, V_1, ...)
      bool ok = true;
      for (;; ++uc) {
        const bool more = u < total;
        Unit<kHeads> un{0, 0, 0, -1};
        if (more) {
          const int tu = static_cast<int>(u / n_sub);
          un.x = static_cast<int>(u - static_cast<int64_t>(tu) * n_sub);
          const int tq = n_rows - 1 - tu;  // the last request's tiles first, each request's from its end
          const int r = upper_index(pre, a.R, tq);
          un.cu = near ? sy.start[r] : a.cu[r];
          un.end = near ? sy.end[r] : a.cu[r + 1];
          un.q = un.cu + (tq - pre[r]) * kUnitRows;
        }
        const int us = uc & 1;
        if (uc >= 2) ok = tc::mbar_wait(&sy.u_empty[us], ((uc >> 1) - 1) & 1);
        if (!ok) break;
        sy.unit[us] = make_int4(un.cu, un.end, un.q, un.x);
        tc::mbar_arrive(&sy.u_full[us]);
        if (!more) break;
        if (uc >= 1) ok = tc::mbar_wait(&sy.q_empty, (uc - 1) & 1);
        if (!ok) break;
        const int nq = un.blocks(1) > 0 ? 2 : 1, nmax = un.blocks(), g = un.head(0) / a.G;
        tc::mbar_arrive_expect_tx(&sy.q_full, nq * kTile);
        for (int s = 0; s < nq; ++s)
          for (int ac = 0; ac < D / 64; ++ac)
            tc::tma_load_3d(sQ + s * kTile + ac * kPanel, &mapQ, ac * 64, un.head(s), un.q0(s), &sy.q_full);
        const int slots = (2 * nmax + kStages - 1) / kStages * kStages;
        for (int i = 0; i < slots && !*abort_flag; ++i, ++n) {
          const int sb = n % kStages;
          ok = n < kStages || tc::mbar_wait(&sy.kv_empty[sb], (n / kStages - 1) & 1);
          if (!ok) break;
          if (i >= 2 * nmax) {  // the odd pair of stages
            tc::mbar_arrive(&sy.kv_full[sb]);
            continue;
          }
          tc::mbar_arrive_expect_tx(&sy.kv_full[sb], kTile);
          const CUtensorMap* map = (i & 1) ? &mapV : &mapK;
          for (int ac = 0; ac < D / 64; ++ac)
            tc::tma_load_3d(sKV + sb * kTile + ac * kPanel, map, ac * 64, g, un.cu + (i >> 1) * kKB, &sy.kv_full[sb]);
        }
        if (!ok || *abort_flag) {
          ok = false;
          ++uc;
          break;
        }
        // taken when the unit's last blocks are under way and not before, so that the CTA that
        // is through first takes the next unit, in one request the heaviest left (252 units of 1
        // to 17 blocks on 152 SMs: 48 us when each CTA took its second unit with its first, 42 us so)
        u = total;
        if (total > gridDim.x) {
          pdl_wait();  // the validation kernel resets the counter
          u = static_cast<int64_t>(gridDim.x) + atomicAdd(&a.st->pool, 1u);
        }
      }
      if (!ok) *abort_flag = 1;
      // let the copies in flight land before the CTA may exit
      if (uc >= 1) tc::mbar_wait(&sy.q_full, (uc - 1) & 1);
      for (int k = (n >= kStages ? n - kStages : 0); k < n; ++k)
        tc::mbar_wait(&sy.kv_full[k % kStages], (k / kStages) & 1);
    }
  } else if (warp == kMmaWarp) {
    // ------------------------------------------------------------ MMA issuer
    // One elected lane issues (see elect_one), serving both slots in turn, which keeps their
    // softmaxes half a period apart. The tensor core queues only about two MMAs, and a look
    // at a barrier behind a commit takes longer than they last: every barrier is looked at
    // before the commit ahead of it, and waited for only if it was not complete then.
    if (tc::elect_one()) {
      constexpr uint32_t idS = tc::idesc_bf16(kQT, kKB);
      constexpr uint32_t idO = tc::idesc_bf16(kQT, D) | (1u << 16);  // B (V) MN-major
      const uint32_t q_base = tc::smem_u32(sQ), kv_base = tc::smem_u32(sKV);
      bool bad = false;
      auto wait = [&](uint64_t* bar, uint32_t parity, bool seen) {
        if (!seen && !bad) bad = !tc::mbar_wait(bar, parity);
      };
      // S of slot s = Q K_j^T from stage `stage`: both K-major
      auto s_mmas = [&](int s, int stage) {
        const uint64_t dq = tc::desc_k_sw128(q_base + s * kTile), dk = tc::desc_k_sw128(kv_base + stage * kTile);
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
          const uint32_t off = static_cast<uint32_t>((ks >> 2) * kPanel + (ks & 3) * 32) / 16;  // in 16-byte units
          tc::mma_bf16(tmem + kSCol + s * 128, dq + off, dk + off, idS, ks > 0 ? 1u : 0u);
        }
      };
      // half of O of slot s += P_j V_j, 16 keys an MMA; only the first `steps` of the block's
      // eight in a request's last tile
      auto pv_mmas = [&](int s, int j, int stage, int steps, int half) {
        const uint64_t dv = tc::desc_mn_sw128(kv_base + stage * kTile, kPanel);
        const uint32_t tP = tmem + kSCol + s * 128, tO = tmem + kOCol + s * 128;
        if (steps == kKB / 16) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int ks = half * 4 + k;
            tc::mma_bf16_ts(tO, tP + ks * 8, dv + ks * (2048 / 16), idO, (j > 0 || ks > 0) ? 1u : 0u);
          }
        } else {
#pragma unroll 1
          for (int ks = half * 4; ks < min(half * 4 + 4, steps); ++ks)
            tc::mma_bf16_ts(tO, tP + ks * 8, dv + ks * (2048 / 16), idO, (j > 0 || ks > 0) ? 1u : 0u);
        }
      };
      using std::integral_constant;
      // Step j, odd or even: V_j sits in stage 1 or 3, K_{j + 1} in stage 2 or 0, and the next
      // step's blocks in the other two (kStages is 4); ph: the ring phase of V_j; pb[s]: the
      // phase of slot s's barriers at the unit's block 0. p0, kv, kk: whether the first half
      // of the next P and the next V and K were seen complete.
      static_assert(kStages == 4, "stages of a step are compile-time constants");
      bool p0 = false, kv = false, kk = false;
      uint32_t pb[2] = {0, 0};
      int n0 = 0, n1 = 0, nm = 0, last_steps = 0;
      int stamp0 = 0;  // timeline build: the first unit's blocks are stamped
      auto slot_group = [&](auto odd, auto slot, int j, uint32_t ph, bool more) {
        constexpr int kOdd = decltype(odd)::value, s = decltype(slot)::value;
        constexpr int sv = kOdd ? 3 : 1, sk = kOdd ? 0 : 2, sv1 = kOdd ? 1 : 3, sk1 = kOdd ? 2 : 0;
        const int steps = j == nm - 1 ? last_steps : kKB / 16;
        const uint32_t pp = kOdd ^ pb[s];
        if (s == 0) fwd_stamp(stamp0 + j, 7);
        if (s == 0 || n0 <= j) {  // the first group of the step: V_j and K_{j + 1}
          wait(&sy.kv_full[sv], ph, kv);
          if (j + 1 < nm) wait(&sy.kv_full[sk], kOdd ? ph ^ 1 : ph, kk);
        }
        wait(&sy.p_full[s][0], pp, p0);
        tc::fence_after_sync();
        if (s == 0) fwd_stamp(stamp0 + j, 8);
        pv_mmas(s, j, sv, steps, 0);
        const bool p1 = tc::mbar_test_wait(&sy.p_full[s][1], pp);
        tc::mma_commit(&sy.pv_done[s][0]);
        wait(&sy.p_full[s][1], pp, p1);
        tc::fence_after_sync();
        pv_mmas(s, j, sv, steps, 1);
        tc::mma_commit(&sy.pv_done[s][1]);
        const bool last = s == 1 || n1 <= j;
        if (last) tc::mma_commit(&sy.kv_empty[sv]);
        if (s == 0) fwd_stamp(stamp0 + j, 9);
        if (s == 0) fwd_stamp(stamp0 + j + 1, 5);
        if (more) s_mmas(s, sk);
        // the next group's barriers
        const int s1 = (s == 0 && j < n1) ? 1 : (n0 > j + 1 ? 0 : 1);
        p0 = tc::mbar_test_wait(&sy.p_full[s1][0], (last ? !kOdd : kOdd) ^ (s1 ? pb[1] : pb[0]));
        if (last) {
          kv = tc::mbar_test_wait(&sy.kv_full[sv1], kOdd ? ph ^ 1 : ph);
          kk = tc::mbar_test_wait(&sy.kv_full[sk1], ph ^ 1);
        }
        if (more) {
          tc::mma_commit(&sy.s_full[s]);
          if (s == 1 || n1 <= j + 1) {
            tc::mma_commit(&sy.kv_empty[sk]);
            if (j + 2 == nm) tc::mma_commit(&sy.q_empty);  // the unit's last S
          }
        }
        if (s == 0) fwd_stamp(stamp0 + j + 1, 6);
      };
      auto step = [&](auto odd, int j, uint32_t ph) {
        if (j < n0) slot_group(odd, integral_constant<int, 0>{}, j, ph, j + 1 < n0);
        if (j < n1) slot_group(odd, integral_constant<int, 1>{}, j, ph, j + 1 < n1);
      };
      uint32_t ph = 0;
#pragma unroll 1
      for (int uc = 0; !bad; ++uc) {
        wait(&sy.u_full[uc & 1], (uc >> 1) & 1, false);
        if (bad) break;
        const Unit<kHeads> un = read_unit(uc & 1);
        tc::mbar_arrive(&sy.u_empty[uc & 1]);
        if (un.x < 0) break;
        n0 = un.blocks(0);
        n1 = un.blocks(1);
        nm = max(n0, n1);
        last_steps = (min(kKB, un.end - (un.cu + (nm - 1) * kKB)) + 15) >> 4;
        p0 = kv = kk = false;
        wait(&sy.q_full, uc & 1, false);
        wait(&sy.kv_full[0], ph, false);
        tc::fence_after_sync();
        if (n0 > 0) {
          s_mmas(0, 0);
          tc::mma_commit(&sy.s_full[0]);
        }
        if (n1 > 0) {
          s_mmas(1, 0);
          tc::mma_commit(&sy.s_full[1]);
        }
        tc::mma_commit(&sy.kv_empty[0]);
        if (nm == 1) tc::mma_commit(&sy.q_empty);
#pragma unroll 1
        for (int j = 0; j < nm; j += 2, ph ^= 1) {
          step(integral_constant<int, 0>{}, j, ph);
          if (j + 1 < nm) {
            step(integral_constant<int, 1>{}, j + 1, ph);
          } else {  // the odd pair of stages, passed on
            wait(&sy.kv_full[2], ph, false);
            tc::mbar_arrive(&sy.kv_empty[2]);
            wait(&sy.kv_full[3], ph, false);
            tc::mbar_arrive(&sy.kv_empty[3]);
          }
        }
        stamp0 = 1 << 20;
        pb[0] ^= n0 & 1;
        pb[1] ^= n1 & 1;
      }
      if (bad) *abort_flag = 1;
      // every MMA issued has completed once this arrives
      tc::mma_commit(&sy.drain);
      tc::mbar_wait(&sy.drain, 0);
    }
  } else {
    // ------------------------------------------------------------ softmax and epilogue (warps 0-7)
    const int slot = warp >> 2, quad = warp & 3;
    const int row = quad * 32 + lane;
    const uint32_t tl = tmem + (static_cast<uint32_t>(quad * 32) << 16);  // this warp's TMEM lanes
    const uint32_t tS = tl + kSCol + slot * 128, tO = tl + kOCol + slot * 128;
    const float c2 = a.c2;
    const float2 cc = make_float2(c2, c2);
    unsigned char* stage = sO + 2 * warp * kOutStage;
    bool ok = true;
    int done = 0, turns = 0;  // blocks of this slot and turns of the ring in earlier units
    int writable = -1;        // the validation kernel's verdict, once it has been waited for
#pragma unroll 1
    for (int uc = 0;; ++uc) {
      ok = tc::mbar_wait_warp(&sy.u_full[uc & 1], (uc >> 1) & 1);
      if (!ok) break;
      const Unit<kHeads> un = read_unit(uc & 1);
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&sy.u_empty[uc & 1]);
      if (un.x < 0) break;
      const int nblk = un.blocks(slot), q0 = un.q0(slot), q_last = un.last(slot), h = un.head(slot);
      float m = -INFINITY, l = 0.f;  // row reference (log2 units); sum of exp2(c2 s - m)
      for (int j = 0; j < nblk; ++j) {
        const bool stamp = warp == 0 && lane == 0 && uc == 0;
        if (stamp) fwd_stamp(j, 0);
        ok = tc::mbar_wait_warp(&sy.s_full[slot], (done + j) & 1);
        if (!ok) break;
        if (stamp) fwd_stamp(j, 1);
        tc::fence_after_sync();
        const bool diag = j == nblk - 1;  // key c of the block is visible to rows >= c
        if (diag && quad == 0 && q_last < q0 + kQT - 1) {
          // a request's last tile: the value rows behind its last key that share the last
          // 16-key step belong to another request and are multiplied by P = 0; they are
          // cleared, so that nothing there (an infinity or a NaN) reaches this request
          const int n = 2 * j + 1, valid = q_last - q0 + 1;
          ok = tc::mbar_wait_warp(&sy.kv_full[n % kStages], (turns + n / kStages) & 1);
          if (!ok) break;
          unsigned char* v = sKV + (n % kStages) * kTile;
          const int dead = ((valid + 15) & ~15) - valid;
          for (int e = lane; e < dead * 8 * (D / 64); e += 32) {
            const int ac = e / (dead * 8), w = e - ac * dead * 8;
            *reinterpret_cast<uint4*>(v + ac * kPanel + valid * 128 + w * 16) = make_uint4(0u, 0u, 0u, 0u);
          }
          fence_proxy_async();
        }
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          uint32_t su[64];  // the row's logits of this half
          uint32_t pk[32];
          auto load = [&](int half) {
            tc::tmem_ld64_async(tS + half * 64, su);
            tc::tmem_wait64(su);
            if (diag) {
#pragma unroll
              for (int c = 0; c < 64; ++c) su[c] = (half * 64 + c <= row) ? su[c] : 0xff800000u;
            }
          };
          // P of the half against the reference m, and its sum
          auto exps = [&]() {
            const float nm = (m == -INFINITY) ? 0.f : -m;
            const float2 nn = make_float2(nm, nm);
            float2 acc0 = make_float2(0.f, 0.f), acc1 = acc0;
#pragma unroll
            for (int c = 0; c < 64; c += 4) {
              const float2 z01 = tc::ffma2(make_float2(__uint_as_float(su[c]), __uint_as_float(su[c + 1])), cc, nn);
              const float2 z23 = tc::ffma2(make_float2(__uint_as_float(su[c + 2]), __uint_as_float(su[c + 3])), cc, nn);
              const float p0 = tc::ex2(z01.x), p1 = tc::ex2(z01.y), p2 = tc::ex2(z23.x), p3 = tc::ex2(z23.y);
              acc0 = tc::add2(acc0, make_float2(p0, p1));
              acc1 = tc::add2(acc1, make_float2(p2, p3));
              pk[c / 2] = pack_bf16x2(p0, p1);
              pk[c / 2 + 1] = pack_bf16x2(p2, p3);
            }
            return (acc0.x + acc0.y) + (acc1.x + acc1.y);
          };
          load(hf);
          float sum = exps();
          // no reference yet, a value far above it, or a NaN: take the maximum of what is left
          // of the block as the reference and start the half again (its logits are in TMEM)
          if (__any_sync(0xffffffffu, m == -INFINITY || !(sum <= kRescaleSum))) {
            float t[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll 1
            for (int half = 1; half >= hf; --half) {
              load(half);
#pragma unroll
              for (int c = 0; c < 64; c += 8) {
#pragma unroll
                for (int w = 0; w < 4; ++w)
                  t[w] = max3(t[w], __uint_as_float(su[c + 2 * w]), __uint_as_float(su[c + 2 * w + 1]));
              }
            }
            const float mb = fmaxf(max3(t[0], t[1], t[2]), t[3]) * c2;  // -inf when nothing is visible
            float factor = 1.f;
            if (mb > m + kRescaleTau) {
              if (m != -INFINITY) factor = tc::ex2(m - mb);
              l *= factor;
              m = mb;
            }
            if (__any_sync(0xffffffffu, factor != 1.f)) {
              // O is final up to the previous half once its P V is done
              ok = tc::mbar_wait_warp(&sy.pv_done[slot][hf ^ 1], (done + j + hf + 1) & 1);
              if (!ok) break;
              tc::fence_after_sync();
#pragma unroll 1
              for (int oc = 0; oc < D; oc += 32) {
                uint32_t ov[32];
                tc::tmem_ld32_async(tO + oc, ov);
                tc::tmem_wait(ov);
#pragma unroll
                for (int i = 0; i < 32; ++i) ov[i] = __float_as_uint(__uint_as_float(ov[i]) * factor);
                tmem_st32(tO + oc, ov);
              }
              tmem_wait_st();
            }
            sum = exps();
          }
          l += sum;
          if (stamp) fwd_stamp(j, 2 + hf);
          tmem_st32(tS + hf * 32, pk);
          tmem_wait_st();
          tc::fence_before_sync();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&sy.p_full[slot][hf]);
        }
        if (!ok) break;
        if (stamp) fwd_stamp(j, 4);
      }
      if (ok && nblk > 0) ok = tc::mbar_wait_warp(&sy.pv_done[slot][1], (done + nblk - 1) & 1);
      if (!ok) break;
      done += nblk;
      turns += (2 * un.blocks() + kStages - 1) / kStages;
      if (nblk == 0) continue;
      if (writable < 0) {
        pdl_wait();
        writable = a.st->layout_ok;
      }
      if (!writable) continue;
      // ---- the unit's rows out. The next unit's S may run meanwhile; its P V, which overwrites
      // O, waits for this warp's next P.
      tc::fence_after_sync();
      const float inv = l > 0.f ? 1.f / l : 0.f;
      const int qpos = q0 + row;
      const bool live = qpos <= q_last;
      // Whole rows go out by TMA through this warp's two stages in turn; a request's last rows,
      // when they do not fill the warp, directly.
      const bool whole = q0 + quad * 32 + 31 <= q_last;
      float* orow = a.o + static_cast<int64_t>(qpos) * a.o_stride + static_cast<int64_t>(h) * D;
#pragma unroll 1
      for (int oc = 0; oc < D; oc += 32) {
        float v[32];
        tc::tmem_ld32(tO + oc, v);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          unsigned char* out = stage + b * kOutStage + lane * 64;
          if (whole) {
            if (lane == 0) bulk_wait_read<1>();  // the store before the last has read this stage
            __syncwarp();
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int c = 16 * b + 4 * i;
            const float4 o4 = make_float4(v[c] * inv, v[c + 1] * inv, v[c + 2] * inv, v[c + 3] * inv);
            if (whole) *reinterpret_cast<float4*>(out + ((i ^ ((lane >> 1) & 3)) << 4)) = o4;
            else if (live) *reinterpret_cast<float4*>(orow + oc + c) = o4;
          }
          if (whole) {
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
              tma_store_3d(&mapO, stage + b * kOutStage, oc + 16 * b, h, q0 + quad * 32);
              bulk_commit();
            }
          }
        }
      }
      if (live) a.lse[static_cast<int64_t>(h) * a.lse_stride + qpos] = (m + log2f(l)) * kLn2;
    }
    if (!ok && lane == 0) *abort_flag = 1;
    if (lane == 0) bulk_wait_read<0>();
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem, kTmemCols);
  }
  pdl_wait();  // this grid's end implies the validation kernel's
  if (threadIdx.x == 0 && sy.abort) record_error(a.st, AVTP_ERR_TIMEOUT, static_cast<int32_t>(blockIdx.x));
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

// A 3-D tensor map, box b0 x 1 x b2, swizzled over the b0 elements (128 bytes of bf16, 64 of
// fp32).
bool map3(CUtensorMap* m, CUtensorMapDataType type, const void* base, uint64_t d0, uint64_t d1, uint64_t d2,
          uint64_t stride1_bytes, uint64_t stride2_bytes, uint32_t b0, uint32_t b2) {
  auto fn = encode_fn();
  if (fn == nullptr) return false;
  const cuuint64_t dims[3] = {d0, d1, d2};
  const cuuint64_t strides[2] = {stride1_bytes, stride2_bytes};
  const cuuint32_t box[3] = {b0, 1, b2};
  const cuuint32_t es[3] = {1, 1, 1};
  const auto swizzle = type == CU_TENSOR_MAP_DATA_TYPE_FLOAT32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B;
  return fn(m, type, 3, const_cast<void*>(base), dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int D, bool kHeads>
cudaError_t launch_fwd(int64_t units, const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv,
                       const CUtensorMap& mo, const FwdArgs& a, cudaStream_t s) {
  static PerDevice attrs;
  const cudaError_t e = once_per_device(attrs, [](int, int*) {
    return cudaFuncSetAttribute(k_attn_fwd<D, kHeads>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                static_cast<int>(fwd_smem_bytes(D)));
  });
  if (e != cudaSuccess) return e;
  const int64_t all = units * (kHeads ? a.Hq / 2 : a.Hq), sms = device_sm_count();
  const int64_t grid = all < sms ? all : sms;
  return launch_kernel(k_attn_fwd<D, kHeads>, dim3(static_cast<unsigned>(grid)), dim3(kThreads), fwd_smem_bytes(D), s,
                       /*pdl=*/true, mq, mk, mv, mo, a);
}

}  // namespace

int forward_unit_rows(const avtp_score_args_t& sa) {
  return (sa.n_q_heads / sa.n_kv_heads) % 2 == 0 ? kQT : 2 * kQT;
}

cudaError_t launch_attn_forward(const avtp_layout_t& L, const avtp_score_args_t& sa, const avtp_forward_args_t& fa,
                                void* ws, const WsPlan& p, const FwdWs& f, cudaStream_t s) {
  if (L.n_tokens == 0) return cudaSuccess;
  const int d = sa.head_dim, Hq = sa.n_q_heads, Hkv = sa.n_kv_heads;
  const int64_t T = L.n_tokens;
  CUtensorMap mq, mk, mv, mo;
  const uint64_t row = static_cast<uint64_t>(d) * 2;
  const auto bf16 = CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  if (!map3(&mq, bf16, sa.q, d, Hq, T, row, static_cast<uint64_t>(sa.q_stride) * 2, 64, kQT) ||
      !map3(&mk, bf16, sa.k, d, Hkv, T, row, static_cast<uint64_t>(sa.k_stride) * 2, 64, kKB) ||
      !map3(&mv, bf16, fa.v, d, Hkv, T, row, static_cast<uint64_t>(fa.v_stride) * 2, 64, kKB) ||
      !map3(&mo, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, fa.o, d, Hq, T, 2 * row, static_cast<uint64_t>(fa.o_stride) * 4, 16,
            32))
    return cudaErrorInvalidValue;
  FwdArgs a{};
  a.cu = L.cu_seqlens;
  a.R = L.n_requests;
  a.T = T;
  a.qtile_cu = ws_at<int32_t>(ws, f.qtile_cu);
  a.Hq = Hq;
  a.G = Hq / Hkv;
  a.c2 = sa.softmax_scale * kLog2e;
  a.o = fa.o;
  a.o_stride = fa.o_stride;
  a.lse = fa.lse;
  a.lse_stride = fa.lse_stride;
  a.st = ws_at<DevStatus>(ws, p.status);
  // units: sum_r ceil(T_r / rows) <= T / rows + R
  const int rows = forward_unit_rows(sa);
  const int64_t units = T / rows + L.n_requests;
  const bool heads = rows == kQT;
  auto launch = d == 128 ? (heads ? launch_fwd<128, true> : launch_fwd<128, false>)
                         : (heads ? launch_fwd<64, true> : launch_fwd<64, false>);
  return launch(units, mq, mk, mv, mo, a, s);
}

}  // namespace avtp

extern "C" avtp_status_t avtp_forward_timeline(int64_t* out, int32_t max_blocks) {
#ifdef AVTP_TIMELINE
  if (out == nullptr || max_blocks < 1) return AVTP_ERR_INVALID_ARG;
  const int n = max_blocks < avtp::kFwdTlBlocks ? max_blocks : avtp::kFwdTlBlocks;
  return cudaMemcpyFromSymbol(out, avtp::g_fwd_tl, static_cast<size_t>(n) * avtp::kFwdTlSlots * sizeof(long long)) ==
                 cudaSuccess
             ? AVTP_OK
             : AVTP_ERR_CUDA;
#else
  (void)out;
  (void)max_blocks;
  return AVTP_ERR_UNSUPPORTED;
#endif
}
