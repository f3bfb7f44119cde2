// Windowed attention of one chunk over the KV ring (sm_100a).
//
// Persistent, warp-specialised kernel, one CTA per SM:
//   warps 0-3   softmax of query tile 0, one thread per query row
//   warps 4-7   softmax of query tile 1
//   warp  8     issues S = Q K^T of both query tiles; owns TMEM
//   warp  9     issues O += P V of both query tiles
//   warp  10    TMA producer (one lane)
// A work item is (stream, head, pair of 128-query tiles): both tiles share every K/V
// tile.  S, P (bf16) and O live in TMEM: one S for both query tiles in turn, a P and an O for each.
// A softmax group takes its scores into registers at once and gives S back, so that the tensor core
// computes the other tile's scores, and then this tile's next ones, while the exponentials run; P V
// follows when P is there.  So the next scores are there when a group is done with its tile, and the
// two groups share the MUFU pipe without waiting for the tensor core.  (With an S for each tile and P over
// S, a tile's next Q K^T had to wait for its P V: exponentials, hand-over, P V and Q K^T were one
// chain of ~3500 clk per key tile.  12 heads, 4680 queries, 32760 keys: 1423-1431 -> 1184-1219 thousand
// cycles and 881-884 -> 808-815 us run on end at the power cap, 755-757 -> 694-697 us in runs of 20.)
//
// What a group does per key tile is as long as the period, so it counts how fast it is fetched: its
// loop over the full tiles is kept short and free of taken branches (rare cases are out of line, one
// masked variant takes first and ragged tiles).  The same pipeline with the variants side by side in one loop
// waited 640 clk per key tile for instructions and took 1425 thousand cycles.
//
// The attended frames are at most three runs of consecutive cache slots (sink prefix, ring
// up to its end, ring from its start).  Key tiles are cut from the runs through a flat
// tensor map over cache rows; only the last tile of a run is ragged, and it is fetched
// through a (token, slot) map whose zero fill ends it exactly at the end of its frame, so
// the cache is never copied and slots outside the window may hold anything.  A ragged tile
// runs with a narrower MMA (N and K rounded up to 16).
#include <cuda.h>
#include <cuda_bf16.h>

#include <map>
#include <mutex>
#include <utility>

#include "common.h"
#include "ptx.cuh"
#include "attn_sched.h"
#include "handover.h"

namespace unstep {

using namespace ptx;

__device__ int g_status = 0;

// Optional timeline of CTA 0 (debug builds only): clock64 stamps per role, tile and event.
#ifdef UNSTEP_TRACE
__device__ long long g_trace[12][64][8];
__device__ unsigned long long g_cta_trace[160][16];
__device__ __forceinline__ unsigned long long gtime() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
#define CTRACE(ev)                                                                       \
  do {                                                                                   \
    if (threadIdx.x == 0 && (ev) < 16) g_cta_trace[blockIdx.x][ev] = gtime();            \
  } while (0)
#define TRACE(role, tile, ev)                                                          \
  do {                                                                                 \
    if (blockIdx.x == 0 && (tile) < 64 && (threadIdx.x & 31) == 0) {                   \
      const int w_ = threadIdx.x >> 5;                                                 \
      const int slot_ = (role) < 2 ? (w_ & 3) * 2 + (role) : 8 + (role) - 2;            \
      g_trace[slot_][tile][ev] = clock64();                                            \
    }                                                                                  \
  } while (0)
#else
#define TRACE(role, tile, ev) \
  do {                        \
  } while (0)
#define CTRACE(ev) \
  do {             \
  } while (0)
#endif

constexpr int kHalfBytes = 128 * 64 * 2;    // one TMA box: 128 rows x 64 bf16 (128-byte rows)
constexpr int kTileBytes = 2 * kHalfBytes;  // 128 x 128 bf16
constexpr int kStages = 5;                  // 32 KB buffers shared by the K and V tiles
constexpr int kThreads = 384;
constexpr int kTmemCols = 512;
constexpr int kTmemS = 0, kTmemP = 128, kTmemO = 256;   // S (128 columns) | P0 | P1 (64 each) | O0 | O1 (128 each)
constexpr long long kWaitCycles = 2000000000LL;  // about a second: then give up, never hang

constexpr int kSmemQ = 0;
constexpr int kSmemKV = 2 * kTileBytes;
constexpr int kSmemBar = kSmemKV + kStages * kTileBytes;
constexpr int kAttnSmemBytes = kSmemBar + 256;

// Partial result of one query tile of a split item: O as [col / 4][row][col % 4] (unnormalised,
// relative to the part's own reference maximum; a warp's 16-byte accesses are 512 consecutive
// bytes), then (m, l)[row].  Two tiles per slot, two slots per CTA.
constexpr int kPartTileFloats = 128 * 128 + 2 * 128;
constexpr int kPartFloats = 2 * kPartTileFloats;
struct Waiter {
  volatile int* abort_flag;
  long long limit;   // clock cycles after which a wait gives up
  // Bounded wait: the hardware parks the thread between polls; the clock and the CTA's abort
  // flag are only looked at every 32 polls so that a waiting warp leaves the issue slots alone.
  __device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity) const {
    if (__builtin_expect(mbar_try_wait(bar, parity) != 0, 1)) return true;
    return wait_long(bar, parity);
  }
  __device__ __forceinline__ bool wait_long(uint32_t bar, uint32_t parity) const {
    const long long t0 = clock64();
#pragma unroll 1
    for (uint32_t spin = 1;; ++spin) {
      if (mbar_try_wait_hint(bar, parity, 2000u)) return true;
      if ((spin & 31u) == 0u) {
        if (*abort_flag) return false;
        if (clock64() - t0 > limit) {
          *abort_flag = 1;
          atomicExch(&g_status, UNSTEP_ERR_TIMEOUT);
          return false;
        }
      }
    }
  }
  // The same by all lanes of a warp, with the warp's answer.
  __device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity) const {
    return __all_sync(0xFFFFFFFFu, wait(bar, parity));
  }
};

// The CTA owns 384 x 168 registers; 128 x 72 for the service warps + 256 x 216 for the softmax
// warps uses exactly that (an increase that the pool cannot satisfy would wait forever).  Nothing spills.
constexpr int kRegsService = 72, kRegsSoftmax = 216;
static_assert(128 * kRegsService + 256 * kRegsSoftmax <= 384 * 168, "register redistribution exceeds the CTA's allocation");
static_assert(kRegsService == 72 && kRegsSoftmax == 216, "keep the setmaxnreg literals below in step");
__device__ __forceinline__ void reg_dealloc_service() { asm volatile("setmaxnreg.dec.sync.aligned.u32 72;"); }
__device__ __forceinline__ void reg_alloc_softmax() { asm volatile("setmaxnreg.inc.sync.aligned.u32 216;"); }

// --------------------------------------------------------------------------------------
// Softmax of one 128 x 128 score tile with one thread per query row (a warpgroup per query
// tile); no data crosses threads.
// --------------------------------------------------------------------------------------
__device__ __forceinline__ void group_barrier(int a) {
  asm volatile("bar.sync %0, 128;" ::"r"(kGroupBarrier + a) : "memory");
}
// The group barrier that also counts the threads with a true predicate: the same answer in every
// thread, with nothing in memory that a warp ahead of the others could overwrite.
__device__ __forceinline__ uint32_t group_count(int a, bool pred) {
  uint32_t n;
  asm volatile("{\n.reg .pred q;\nsetp.ne.u32 q, %2, 0;\nbar.red.popc.u32 %0, %1, 128, q;\n}"
               : "=r"(n) : "r"(kGroupBarrier + a), "r"(static_cast<uint32_t>(pred)) : "memory");
  return n;
}

// Hand-over of P to the P V issuer, and of the read S back to the Q K^T issuer, through named barriers.  An mbarrier lives in shared
// memory, whose bandwidth the MMA operands of Q K^T use up: an arrive or a try_wait there took
// 120-270 clk, several times on every key tile's critical path; a named barrier takes 25-60 clk.
// A named barrier has no bounded wait, so every warp keeps meeting them, once per key tile of its
// segments, after it has given up on an mbarrier as well; handover.h says why all of them end.
__device__ __forceinline__ void p_ready_sync(int a, uint32_t tile) {   // P V issuer: P of group a's tile-th key tile is in TMEM
  asm volatile("bar.sync %0, 160;" ::"r"(p_ready_barrier(a, tile)) : "memory");
}
__device__ __forceinline__ void p_ready_pass(int a, uint32_t tile, bool gave_up) {   // a warp of softmax group a
  if (p_ready_waits(gave_up)) p_ready_sync(a, tile);
  else asm volatile("bar.arrive %0, 160;" ::"r"(p_ready_barrier(a, tile)) : "memory");
}
__device__ __forceinline__ void s_free_sync(int a, uint32_t tile) {   // Q K^T issuer: group a has read S of its tile-th key tile
  asm volatile("bar.sync %0, 160;" ::"r"(s_free_barrier(a, tile)) : "memory");
}
__device__ __forceinline__ void s_free_pass(int a, uint32_t tile, bool gave_up) {   // a warp of softmax group a
  if (p_ready_waits(gave_up)) s_free_sync(a, tile);
  else asm volatile("bar.arrive %0, 160;" ::"r"(s_free_barrier(a, tile)) : "memory");
}

// Exponentials of 32 score columns (registers s) into 16 bf16 pairs (p) and the packed sums.
__device__ __forceinline__ void exp_block32(const uint32_t* s, uint32_t* p, uint64_t c2, uint64_t nm2,
                                            uint64_t* acc) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const uint64_t x2 = fma_f32x2(pack_f32x2(__uint_as_float(s[2 * i]), __uint_as_float(s[2 * i + 1])), c2, nm2);
    float x0, x1;
    unpack_f32x2(x2, x0, x1);
    const float p0 = ex2(x0), p1 = ex2(x1);
    acc[i & 3] = add_f32x2(acc[i & 3], pack_f32x2(p0, p1));
    p[i] = pack_bf16x2(p0, p1);
  }
}
__device__ __forceinline__ float max_block32(const uint32_t* s) {
  float m = fmaxf(__uint_as_float(s[0]), __uint_as_float(s[1]));
#pragma unroll
  for (int i = 2; i < 32; i += 2) m = max3(m, __uint_as_float(s[i]), __uint_as_float(s[i + 1]));
  return m;
}
template <bool kMasked>
__device__ __forceinline__ void mask_block32(uint32_t* s, int col0, int nvalid) {
  if (kMasked) {
#pragma unroll
    for (int i = 0; i < 32; ++i)
      if (col0 + i >= nvalid) s[i] = 0xFF800000u;  // -inf
  }
}

// One key tile of a row: scores from TMEM (columns t_S ..) into registers, S given back, exponentials against
// the row's reference maximum, P (bf16 pairs, keys 0.. from column t_P on) handed over.  False if a wait gave up;
// S has been given back then, P has not been passed.
//
// The reference is the maximum of the segment's first key tile, so that the largest weight there is exactly 1 (with
// the maximum of 32 scores the error of peaked rows against float64 grew from 2.17e-3 to 2.32e-3).  It moves
// only where a later tile has a score more than kJump = 57 (log2 units) above it: up to there P (bf16) and the
// float32 sums are as accurate as near 1 (same relative precision), and what was accumulated before such a jump
// is negligible exactly as in the true softmax.  A tile's sum of P is at most 128 * 2^57 = 2^64, the sum of n keys
// at most n * 2^57, and O that times |v|: finite for any window that the entry points take (2^30 keys) up to
// |v| = 2^40, for 32760 keys up to 2^55.  (With kJump = 64, tiles of 128 keys 62 above the reference overflowed with |v| =
// 2^60.)  The scores have left TMEM by the time a sum of P could tell, so the maximum is looked for in front: 64
// three-input maxima in the shadow of the other group's exponentials.
//
// P may be stored, and O rescaled, once the P V of the tile before has run.  That barrier, and the one of the next
// tile's scores, are looked at once, ahead of time: the look takes 100-200 clk under the MMAs' traffic, and
// almost always finds what it looks for.
// Tiles of at most 64 keys (frames of up to 64 tokens, the end of a run) leave the other half of the columns
// alone.
constexpr float kJump = 57.f;

template <bool kMasked, int kCols, bool kTight>   // kCols: score columns that hold keys, 64 or 128; kTight: not a segment's first tile
__device__ __forceinline__ bool softmax_row_tile(uint32_t t_S, uint32_t t_P, uint32_t t_O, float c, int nvalid,
                                                 bool first, float& m_run, float& l_run, int a, uint32_t tile,
                                                 const Waiter& w, uint32_t bar_pv, uint32_t bar_s, uint32_t& s_seen) {
  uint32_t s[kCols], p[kCols / 2];
#pragma unroll
  for (int q = 0; q < kCols / 32; ++q) tmem_ld32(t_S + 32 * q, s + 32 * q);
  tc_wait_ld32(s);
#pragma unroll
  for (int q = 1; q < kCols / 32; ++q) reg_fence32(s + 32 * q);
  tc_fence_before();
  s_free_pass(a, tile, false);
  TRACE(a, tile, 2);
#pragma unroll
  for (int q = 0; q < kCols / 32; ++q) mask_block32<kMasked>(s + 32 * q, 32 * q, nvalid);
  float mx = max_block32(s);
#pragma unroll
  for (int q = 1; q < kCols / 32; ++q) mx = fmaxf(mx, max_block32(s + 32 * q));
  if (!kTight && first) {
    m_run = mx;
  } else if (__builtin_expect(__any_sync(0xFFFFFFFFu, (mx - m_run) * c > kJump), 0)) {
    if (!w.wait_warp(bar_pv, (tile - 1) & 1)) return false;
    tc_fence_after();
    float alpha = 1.f;
    if (mx > m_run) {
      alpha = ex2((m_run - mx) * c);
      m_run = mx;
      l_run *= alpha;
    }
#pragma unroll 1
    for (int q = 0; q < 16; ++q) {
      uint32_t o[8];
      tmem_ld8(t_O + q * 8, o);
      tc_wait_ld8(o);
#pragma unroll
      for (int i = 0; i < 8; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * alpha);
      tmem_st8(t_O + q * 8, o);
    }
  }
  const uint64_t c2 = pack_f32x2(c, c), nm2 = pack_f32x2(-m_run * c, -m_run * c);
  uint64_t acc[4] = {0ull, 0ull, 0ull, 0ull};
  TRACE(a, tile, 3);
#pragma unroll
  for (int q = 0; q < kCols / 32 - 1; ++q) exp_block32(s + 32 * q, p + 16 * q, c2, nm2, acc);
  uint32_t pv_seen = mbar_test(bar_pv, (tile - 1) & 1);
  exp_block32(s + kCols - 32, p + kCols / 2 - 16, c2, nm2, acc);
  if ((kTight || !first) && __builtin_expect(!__all_sync(0xFFFFFFFFu, pv_seen), 0)) {
    if (!w.wait_warp(bar_pv, (tile - 1) & 1)) return false;
  }
  tc_fence_after();
  TRACE(a, tile, 4);
  if (kCols > 64) tmem_st32(t_P, p);
  s_seen = mbar_test(bar_s, (tile + 1) & 1);
  tmem_st32(t_P + kCols / 2 - 32, p + kCols / 2 - 32);
  tc_wait_st();
  tc_fence_before();
  p_ready_pass(a, tile, false);
  TRACE(a, tile, 5);
  const uint64_t t2 = add_f32x2(add_f32x2(acc[0], acc[1]), add_f32x2(acc[2], acc[3]));
  float t0, t1;
  unpack_f32x2(t2, t0, t1);
  l_run += t0 + t1;
  return true;
}

// Real keys of key tile j of a stream, without the divisions of tile_info: only the last tile of a
// run of slots is ragged (frames shorter than a tile: every tile is one frame).
struct ValidKeys {
  int j_last[3], v_last[3], dflt;
  __device__ __forceinline__ ValidKeys(const AttnParams& p, int b) {
    dflt = p.flat ? kTileN : p.T;
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int begin = r == 0 ? 0 : p.run_tile_end[b][r - 1];
      const int end = p.run_tile_end[b][r];
      const bool any = p.flat && end > begin;
      j_last[r] = any ? end - 1 : -1;
      v_last[r] = p.run_rows[b][r] - kTileN * (end - begin - 1);
    }
  }
  // first tile from j on that is ragged, at most `end`
  __device__ __forceinline__ int full_until(int j, int end) const {
    if (dflt < kTileN) return j;
    int k = end;
#pragma unroll
    for (int r = 0; r < 3; ++r)
      if (j_last[r] >= j && j_last[r] < k && v_last[r] < kTileN) k = j_last[r];
    return k;
  }
  __device__ __forceinline__ int operator()(int j) const {
    return j == j_last[0] ? v_last[0] : (j == j_last[1] ? v_last[1] : (j == j_last[2] ? v_last[2] : dflt));
  }
};

// Partial results exchanged inside a cluster: where the K and V tiles were, O of both query tiles as
// [tile][col / 4][row][col % 4], then (m, l) as [tile][row].
constexpr int kSwapTileBytes = 128 * 128 * 4;
constexpr int kSwapMl = 2 * kSwapTileBytes;
static_assert(kSwapMl + 2 * 128 * 8 <= kStages * kTileBytes, "the exchange does not fit the K and V stages");

// kCluster: a launch of one part per block, in which the parts of an item are a cluster and merge through each
// other's shared memory.  The other form merges through global memory, where a part's stores, the fence
// with its count and the last part's loads took 5-10 us one after the other.
template <bool kCluster>
__global__ void __launch_bounds__(kThreads, 1)
window_attn_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                   const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_kf,
                   const __grid_constant__ CUtensorMap tm_vf, const AttnParams p,
                   __nv_bfloat16* __restrict__ out) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const uint32_t smem_base = smem_u32(smem_raw);
  if (smem_base & 1023u) {  // the 128-byte swizzle needs 1024-byte aligned tiles
    if (threadIdx.x == 0) atomicExch(&g_status, UNSTEP_ERR_CUDA);
    return;
  }
  uint8_t* gen = smem_raw;
  const uint32_t sQ = smem_base + kSmemQ;
  const uint32_t sKV = smem_base + kSmemKV;
  const uint32_t sBar = smem_base + kSmemBar;
  // mbarriers (8 bytes each)
  const uint32_t bar_q_full = sBar;                          // [2]  TMA -> Q K^T issuer
  const uint32_t bar_q_empty = sBar + 16;                    // [2]  Q K^T issuer -> TMA
  const uint32_t bar_kv_full = sBar + 32;                    // [kStages] TMA -> the issuer that reads the stage
  const uint32_t bar_kv_empty = sBar + 32 + 8 * kStages;     // [kStages] that issuer -> TMA
  const uint32_t bar_s_full = sBar + 32 + 16 * kStages;      // [2]  Q K^T issuer -> softmax a
  const uint32_t bar_pv_done = bar_s_full + 16;              // [2]  P V issuer -> softmax a
  volatile uint32_t* tmem_slot = reinterpret_cast<volatile uint32_t*>(gen + kSmemBar + 224);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(gen + kSmemBar + 228);

  const int tid = threadIdx.x;
  const int warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0);   // the same in all lanes, and known to be
  const int lane = tid & 31;
  CTRACE(0);

  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar_q_full + 8 * i, 1);
      mbar_init(bar_q_empty + 8 * i, 1);
      mbar_init(bar_s_full + 8 * i, 1);
      mbar_init(bar_pv_done + 8 * i, 1);
    }
    for (int i = 0; i < kStages; ++i) {
      mbar_init(bar_kv_full + 8 * i, 1);
      mbar_init(bar_kv_empty + 8 * i, 1);
    }
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 8) {
    tmem_alloc(smem_u32(const_cast<uint32_t*>(tmem_slot)), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = __shfl_sync(0xFFFFFFFFu, *tmem_slot, 0);
  // What comes before a role's grid_wait may run under the kernel before this one.  Every role waits
  // there, so that no bounded wait counts that kernel's time.
  const Waiter w{abort_flag, kWaitCycles};

  if (warp >= 8) {
    reg_dealloc_service();
    if (warp == 10 && lane == 0) {
      // ------------------------------------------------------------ TMA producer
      prefetch_tensormap(&tm_q);
      prefetch_tensormap(&tm_k);
      prefetch_tensormap(&tm_v);
      prefetch_tensormap(&tm_kf);
      prefetch_tensormap(&tm_vf);
      grid_wait();
      Sched sched(p, static_cast<int>(blockIdx.x));
      Seg s;
      uint32_t kv_it = 0, q_it[2] = {0, 0};
      bool ok = true;
      while (ok && sched.next(s)) {
        auto load_q = [&](int a) {
          if (!ok || a >= s.nq) return;
          ok = w.wait(bar_q_empty + 8 * a, (q_it[a] & 1) ^ 1);
          if (!ok) return;
          const uint32_t dst = sQ + a * kTileBytes, bar = bar_q_full + 8 * a;
          const int n0 = (2 * s.qp + a) * kTileM;
          mbar_expect_tx(bar, kTileBytes);
          tma_load_4d(dst, &tm_q, bar, 0, s.h, n0, s.b);
          tma_load_4d(dst + kHalfBytes, &tm_q, bar, 64, s.h, n0, s.b);
          ++q_it[a];
        };
        auto load_kv = [&](const TileInfo& ti, int kv) {
          const uint32_t st = kv_it % kStages;
          if (ok) ok = w.wait(bar_kv_empty + 8 * st, ((kv_it / kStages) & 1) ^ 1);
          if (!ok) return;
          const uint32_t dst = sKV + st * kTileBytes, bar = bar_kv_full + 8 * st;
          mbar_expect_tx(bar, kTileBytes);
          if (ti.framed) {
            const CUtensorMap* tm = kv == 0 ? &tm_k : &tm_v;
            tma_load_5d(dst, tm, bar, 0, s.h, ti.tok0, ti.slot, s.b);
            tma_load_5d(dst + kHalfBytes, tm, bar, 64, s.h, ti.tok0, ti.slot, s.b);
          } else {
            const CUtensorMap* tm = kv == 0 ? &tm_kf : &tm_vf;
            tma_load_4d(dst, tm, bar, 0, s.h, ti.row, s.b);
            tma_load_4d(dst + kHalfBytes, tm, bar, 64, s.h, ti.row, s.b);
          }
          ++kv_it;
        };
        load_q(0);   // what the first S needs comes first: Q of tile 0, then K
        TileInfo ti = tile_info(p, s.b, s.t0);
        load_kv(ti, 0);
        load_q(1);
        for (int j = s.t0; j < s.t1 && ok; ++j) {
          TileInfo tn = ti;
          if (j + 1 < s.t1) {
            tn = tile_info(p, s.b, j + 1);
            load_kv(tn, 0);
          }
          load_kv(ti, 1);
          ti = tn;
        }
      }
    } else if (warp == 8) {
      // ------------------------------------------------------------ Q K^T issuer
      // The K and V tiles come in the order in which they are used: K of tile 0, then K of tile j + 1 and V
      // of tile j.  The whole warp runs the code (the loops stay rolled: instruction fetch is scarce).
      grid_wait();
      Sched sched(p, static_cast<int>(blockIdx.x));
      Seg s;
      uint32_t kv_base = 0, n0 = 0, n1 = 0, q0 = 0, q1 = 0;   // tiles and items per group
      int before = -1;   // group whose scores are in S
      bool ok = true;
      const uint32_t idesc_full = idesc_bf16_f32(kTileM, kTileN, 0);
      const uint64_t dq = smem_desc_sw128(sQ, 16, 1024);    // Q tile 0, K-major
      const uint64_t dk0 = smem_desc_sw128(sKV, 16, 1024);  // stage 0 as a K tile
      while (sched.next(s)) {
        const int n = s.t1 - s.t0;
        const ValidKeys valid_of(p, s.b);
        for (int j = 0; j < n; ++j) {
          const uint32_t it = kv_base + (j > 0 ? 2 * j - 1 : 0), st = it % kStages;   // K's place in the order
          const int valid = valid_of(s.t0 + j);
          const uint32_t idesc = valid == kTileN ? idesc_full : idesc_bf16_f32(kTileM, (valid + 15) & ~15, 0);
          const uint64_t dk = dk0 + static_cast<uint64_t>((st * kTileBytes) >> 4);
#pragma unroll 1
          for (int a = 0; a < s.nq; ++a) {
            if (ok && j == 0) ok = w.wait_warp(bar_q_full + 8 * a, (a == 0 ? q0 : q1) & 1);
            if (ok && a == 0) ok = w.wait_warp(bar_kv_full + 8 * st, (it / kStages) & 1);
            TRACE(2, n0 + n1, 0);
            if (before >= 0) s_free_sync(before, (before == 0 ? n0 : n1) - 1);
            TRACE(2, n0 + n1, 1);
            if (ok) {
              tc_fence_after();
              mma_ss_k128(tmem_base + kTmemS, dq + static_cast<uint64_t>((a * kTileBytes) >> 4), dk, idesc, 0u);
            }
            if (ok) {
              tc_commit(bar_s_full + 8 * a);
              if (a == s.nq - 1) tc_commit(bar_kv_empty + 8 * st);
              if (j == n - 1) tc_commit(bar_q_empty + 8 * a);
            }
            TRACE(2, n0 + n1, 2);
            if (j == 0) ++(a == 0 ? q0 : q1);
            ++(a == 0 ? n0 : n1);
            before = a;
          }
        }
        kv_base += 2 * n;
      }
      if (before >= 0) s_free_sync(before, (before == 0 ? n0 : n1) - 1);
    } else if (warp == 9) {
      // ------------------------------------------------------------ P V issuer
      // The commits that free a stage come behind those that a softmax group waits for, but for the segment's last one:
      // behind that the kernel may end.
      grid_wait();
      Sched sched(p, static_cast<int>(blockIdx.x));
      Seg s;
      uint32_t kv_base = 0, n0 = 0, n1 = 0;
      bool ok = true;
      const uint32_t idesc_pv = idesc_bf16_f32(kTileM, kHeadDim, 1);
      const uint64_t dv0 = smem_desc_sw128(sKV, kHalfBytes, 1024);          // stage 0 as a V tile (MN-major)
      while (sched.next(s)) {
        const int n = s.t1 - s.t0;
        const ValidKeys valid_of(p, s.b);
        for (int j = 0; j < n; ++j) {
          const uint32_t it = kv_base + (j + 1 < n ? 2 * j + 2 : 2 * n - 1), st = it % kStages;
          const int k_steps = (valid_of(s.t0 + j) + 15) >> 4;
          const uint64_t dv = dv0 + static_cast<uint64_t>((st * kTileBytes) >> 4);
          if (ok) ok = w.wait_warp(bar_kv_full + 8 * st, (it / kStages) & 1);
#pragma unroll 1
          for (int a = 0; a < s.nq; ++a) {
            const uint32_t o_tmem = tmem_base + kTmemO + a * 128, p_tmem = tmem_base + kTmemP + a * 64;
            TRACE(3, n0 + n1, 0);
            p_ready_sync(a, a == 0 ? n0 : n1);   // P of this tile is in TMEM, O rescaled if need be
            TRACE(3, n0 + n1, 1);
            if (ok) {
              tc_fence_after();
              if (k_steps == 8) {
                mma_ts_k64(o_tmem, p_tmem, dv, idesc_pv, j > 0 ? 1u : 0u);
                mma_ts_k64(o_tmem, p_tmem + 32, dv + 512u, idesc_pv, 1u);
              } else {
#pragma unroll 1
                for (int k = 0; k < k_steps; ++k)
                  mma_ts(o_tmem, p_tmem + k * 8, dv + static_cast<uint64_t>(k * 128), idesc_pv, (j > 0 || k > 0) ? 1u : 0u);
              }
            }
            if (ok) {
              const bool last_of_stage = a == s.nq - 1;
              if (last_of_stage && j == n - 1) tc_commit(bar_kv_empty + 8 * st);
              tc_commit(bar_pv_done + 8 * a);
              if (last_of_stage && j < n - 1) tc_commit(bar_kv_empty + 8 * st);
            }
            TRACE(3, n0 + n1, 2);
            ++(a == 0 ? n0 : n1);
          }
        }
        kv_base += 2 * n;
      }
    }
  } else {
    // ---------------------------------------------------------------- softmax warpgroups
    // Warps 0-3 own query tile 0, warps 4-7 query tile 1; a thread owns a row from the scores
    // to the output.
    reg_alloc_softmax();
    grid_wait();
    const int a = warp >> 2;               // query tile of this warpgroup
    const int row = tid & 127;             // row inside the tile = TMEM lane
    const uint32_t t_lane = tmem_base + (static_cast<uint32_t>((warp & 3) * 32) << 16);
    const uint32_t t_S = t_lane + kTmemS, t_P = t_lane + kTmemP + a * 64, t_O = t_lane + kTmemO + a * 128;
    Sched sched(p, static_cast<int>(blockIdx.x));
    Seg s;
    Seg seg = {};        // of a cluster's block: its only one
    uint32_t it = 0, s_seen = 0;
    bool ok = true;
    int seg_no = 0;
    CTRACE(1);
    // After a wait gave up (ok == false) a warp keeps walking its segments without working, so that
    // it still meets its group and its issuer at every named barrier.  ok is the same in all threads
    // of a warp: barriers and TMEM accesses are instructions of the whole warp.
    while (sched.next(s)) {
      if (kCluster) seg = s;
      if (a >= s.nq) continue;             // a lone last query tile: nothing for group 1
      float m_run = -INFINITY, l_run = 0.f;
      const ValidKeys valid_of(p, s.b);
      const uint32_t pv = bar_pv_done + 8 * a, sb = bar_s_full + 8 * a;
      // scores of tile `it`: true unless the wait gave up, in which case the issuers still count on this warp
      auto scores = [&](uint32_t tile) {
        if (ok && __builtin_expect(!__all_sync(0xFFFFFFFFu, s_seen), 0)) ok = w.wait_warp(sb, tile & 1);
        s_seen = 0;
        if (__builtin_expect(!ok, 0)) {
          s_free_pass(a, tile, true);
          p_ready_pass(a, tile, true);
          return false;
        }
        tc_fence_after();
        return true;
      };
      int j = s.t0;
#pragma unroll 1
      while (j < s.t1) {
        {   // the segment's first tile, or a ragged one
          const int valid = valid_of(j);
          TRACE(a, it, 0);
          if (scores(it)) {
            TRACE(a, it, 1);
            const bool first = j == s.t0;
            if (valid <= 64)   // frames of at most half a tile, and the end of a run
              ok = softmax_row_tile<true, 64, false>(t_S, t_P, t_O, p.scale_log2e, valid, first, m_run, l_run, a, it, w, pv, sb, s_seen);
            else
              ok = softmax_row_tile<true, kTileN, false>(t_S, t_P, t_O, p.scale_log2e, valid, first, m_run, l_run, a, it, w, pv, sb, s_seen);
            if (!ok) p_ready_pass(a, it, true);
          }
          ++j;
          ++it;
        }
        const int jf = valid_of.full_until(j, s.t1);
#pragma unroll 1
        for (; j < jf; ++j, ++it) {
          TRACE(a, it, 0);
          if (scores(it)) {
            TRACE(a, it, 1);
            ok = softmax_row_tile<false, kTileN, true>(t_S, t_P, t_O, p.scale_log2e, kTileN, false, m_run, l_run, a, it, w, pv, sb, s_seen);
            if (__builtin_expect(!ok, 0)) p_ready_pass(a, it, true);
          }
        }
      }
      CTRACE(8 + seg_no);
      // ---- epilogue of this group's query tile ----
      const bool whole = (s.t0 == 0 && s.t1 == s.tiles);
      // Part of a split item: the arrival counter, looked at under the wait for the last P V
      auto counter = [&] { return p.counters + 2 * s.item + a; };
      int seen = 0;
      if (!kCluster && !whole && row == 0) {
#ifdef UNSTEP_CHECK
        if (2 * s.item + a >= p.extent_counters) atomicExch(p.status, static_cast<int>(UNSTEP_ERR_BOUNDS));
#endif
        asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(seen) : "l"(counter()) : "memory");
      }
      if (ok) {
        ok = w.wait_warp(bar_pv_done + 8 * a, (it - 1) & 1);
        tc_fence_after();
      }
      const int n = (2 * s.qp + a) * kTileM + row;
      uint4* const out_v = reinterpret_cast<uint4*>(out);
      const int64_t dst = ((static_cast<int64_t>(s.b) * p.L + n) * p.Hn + s.h) * (kHeadDim / 8);   // 16-byte vectors
      auto store_row = [&](int64_t d, const float* v, float inv_l) {   // 32 columns from vector d on
        uint32_t w[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] = pack_bf16x2(v[2 * i] * inv_l, v[2 * i + 1] * inv_l);
        if (p.out_wide) {   // whole 32-byte sectors
          UNSTEP_STORE_32(out_v, d, p.extent_out, w, p.status);
          UNSTEP_STORE_32(out_v, d + 2, p.extent_out, w + 8, p.status);
          return;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
          UNSTEP_STORE(out_v, d + i, p.extent_out, make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]),
                       p.status);
      };
      if (kCluster) {
        // Every block of a cluster holds one part of the same item.  Each puts its part into its own shared memory and
        // then merges a share of the columns of all rows, in part order, reading the others' parts there.
        if (s.nq == 2) asm volatile("bar.sync %0, 256;" ::"r"(kSwapBarrier) : "memory");   // the stages are free behind both P V
        const uint32_t mine = sKV + a * kSwapTileBytes + row * 16;
        if (ok) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint32_t o[32];
            tmem_ld32(t_O + q * 32, o);
            tc_wait_ld32(o);
#pragma unroll
            for (int i = 0; i < 8; ++i) st_shared_16(mine + (q * 8 + i) * 2048, o + 4 * i);
          }
          st_shared_8(sKV + kSwapMl + a * 1024 + row * 8, __float_as_uint(m_run), __float_as_uint(l_run));
        }
      } else if (whole) {
        // O / l -> bf16 -> out[b][n][h][:]: a thread writes its whole 256-byte row
        if (ok) {
          const float inv_l = 1.f / l_run;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float o[32];
            tmem_ld32(t_O + q * 32, reinterpret_cast<uint32_t*>(o));
            tc_wait_ld32(reinterpret_cast<uint32_t*>(o));
            if (n < p.L) store_row(dst + 4 * q, o, inv_l);
          }
        }
      } else {
        // Part of a split item.  The parts of an item's query tile are merged by whichever of
        // them is done last, in part order (a fixed order, so the result does not depend on
        // which one that is); the merging part takes its own accumulator straight from TMEM.
        // A part that finds all others already published merges at once without publishing
        // itself; otherwise it publishes (O, m, l), counts itself in, and merges if that made
        // the count complete.
        const int c_lo = first_part_worker(p, s);
        const int c_hi = last_part_worker(p, s);
        const int others = c_hi - c_lo;
        // one thread says whether all others are in, the others whether their warp gave up (31 or
        // more do then); a group that gave up publishes nothing
        const uint32_t votes = group_count(a, row == 0 ? seen == others : !ok);
        if (votes > 1) ok = false;
        bool last = votes == 1;
        if (ok && !last) {
          const int64_t mine = (static_cast<int64_t>(2 * blockIdx.x + (s.first_in_worker ? 0 : 1)) * kPartFloats +
                                a * kPartTileFloats);   // first float of this part in the scratch
          float4* const part4 = reinterpret_cast<float4*>(p.part);
          const int64_t mine4 = mine / 4 + row;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint32_t o[32];
            tmem_ld32(t_O + q * 32, o);
            tc_wait_ld32(o);
#pragma unroll
            for (int i = 0; i < 8; ++i)
              UNSTEP_STORE(part4, mine4 + (q * 8 + i) * 128, p.extent_part / 4,
                           make_float4(__uint_as_float(o[4 * i]), __uint_as_float(o[4 * i + 1]),
                                       __uint_as_float(o[4 * i + 2]), __uint_as_float(o[4 * i + 3])),
                           p.status);
          }
          UNSTEP_STORE(reinterpret_cast<float2*>(p.part), mine / 2 + 128 * 64 + row, p.extent_part / 2,
                       make_float2(m_run, l_run), p.status);
          group_barrier(a);   // all of this part is stored
          int before = -1;
          if (row == 0) {
            // release: the group's stores (ordered before this thread by the barrier) become visible
            // before the count; acquire: a merging part sees the other parts' stores
            asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;" : "=r"(before) : "l"(counter()) : "memory");
          }
          last = group_count(a, before == others) != 0;
        }
        if (ok && last) {
          __threadfence();   // acquire side for every thread that reads the other parts below
          if (row == 0) UNSTEP_STORE(p.counters, 2 * s.item + a, p.extent_counters, 0, p.status);   // ready for the next launch
          const int me = static_cast<int>(blockIdx.x);
          const int lo_slot = part_slot(p, c_lo, s.item_step0);   // every later part starts its worker's range
          auto part_of = [&](int c) -> const float* {
            return p.part + (static_cast<int64_t>(2 * c + (c == c_lo ? lo_slot : 0)) * kPartFloats + a * kPartTileFloats);
          };
          auto ml_of = [&](int c) -> float2 {
            return c == me ? make_float2(m_run, l_run)
                           : __ldcg(reinterpret_cast<const float2*>(part_of(c) + 128 * 128) + row);
          };
          float m_all = m_run, l_sum = 0.f;
          if (others <= 3) {   // one round trip for all parts
            float2 x[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) x[i] = i <= others ? ml_of(c_lo + i) : make_float2(-INFINITY, 0.f);
#pragma unroll
            for (int i = 0; i < 4; ++i) m_all = fmaxf(m_all, x[i].x);
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (i <= others) l_sum += x[i].y * ex2((x[i].x - m_all) * p.scale_log2e);
          } else {
#pragma unroll 4
            for (int c = c_lo; c <= c_hi; ++c) m_all = fmaxf(m_all, ml_of(c).x);
#pragma unroll 4
            for (int c = c_lo; c <= c_hi; ++c) {
              const float2 x = ml_of(c);
              l_sum += x.y * ex2((x.x - m_all) * p.scale_log2e);
            }
          }
          const float inv_l = 1.f / l_sum;
#pragma unroll 1
          for (int q = 0; q < 2; ++q) {   // 64 output columns at a time
            float acc[64];
#pragma unroll
            for (int i = 0; i < 64; ++i) acc[i] = 0.f;
            for (int c = c_lo; c <= c_hi; ++c) {
              if (c == me) {
                const float sc = ex2((m_run - m_all) * p.scale_log2e);
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  uint32_t o[32];
                  tmem_ld32(t_O + 64 * q + 32 * h, o);
                  tc_wait_ld32(o);
#pragma unroll
                  for (int i = 0; i < 32; ++i) acc[32 * h + i] = fmaf(__uint_as_float(o[i]), sc, acc[32 * h + i]);
                }
              } else {
                const float4* pc = reinterpret_cast<const float4*>(part_of(c)) + q * 16 * 128 + row;
                float4 v[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) v[i] = __ldcg(pc + i * 128);
                const float sc = ex2((ml_of(c).x - m_all) * p.scale_log2e);
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                  acc[4 * i] = fmaf(v[i].x, sc, acc[4 * i]);
                  acc[4 * i + 1] = fmaf(v[i].y, sc, acc[4 * i + 1]);
                  acc[4 * i + 2] = fmaf(v[i].z, sc, acc[4 * i + 2]);
                  acc[4 * i + 3] = fmaf(v[i].w, sc, acc[4 * i + 3]);
                }
              }
            }
            if (n < p.L) {
              store_row(dst + 8 * q, acc, inv_l);
              store_row(dst + 8 * q + 4, acc + 32, inv_l);
            }
          }
        }
      }
      tc_fence_before();
      CTRACE(3 + seg_no);
      ++seg_no;
    }
    if (kCluster) {
      __syncwarp();
      cluster_sync();   // all parts are in place
      const int parts = p.parts, part = static_cast<int>(cluster_rank());
      // a lone query tile is shared out to both groups
      const int tile = seg.nq == 2 ? a : 0, share = seg.nq == 2 ? part : 2 * part + a, shares = seg.nq == 2 ? parts : 2 * parts;
      const int n = (2 * seg.qp + tile) * kTileM + row;
      bool good = seg.nq > 0;
      for (int c = 0; c < parts; ++c)   // a block that gave up has left no part
        good = good && ld_cluster_4(cluster_addr(smem_u32(const_cast<int*>(abort_flag)), c)) == 0;
      if (good && n < p.L) {
        float2 x[kMaxClusterParts];
        float m_all = -INFINITY, l_sum = 0.f;
#pragma unroll
        for (int c = 0; c < kMaxClusterParts; ++c)
          x[c] = c < parts ? ld_cluster_8(cluster_addr(sKV + kSwapMl + tile * 1024 + row * 8, c)) : make_float2(-INFINITY, 0.f);
#pragma unroll
        for (int c = 0; c < kMaxClusterParts; ++c) m_all = fmaxf(m_all, x[c].x);
#pragma unroll
        for (int c = 0; c < kMaxClusterParts; ++c)
          if (c < parts) {
            x[c].x = ex2((x[c].x - m_all) * p.scale_log2e);
            l_sum += x[c].y * x[c].x;
          }
        const float inv_l = 1.f / l_sum;
        uint4* const out_v = reinterpret_cast<uint4*>(out);
        const int64_t dst = ((static_cast<int64_t>(seg.b) * p.L + n) * p.Hn + seg.h) * (kHeadDim / 8);   // 16-byte vectors
        const uint32_t from = sKV + tile * kSwapTileBytes + row * 16;
#pragma unroll 2
        for (int v = 16 * share / shares; v < 16 * (share + 1) / shares; ++v) {
          float acc[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) acc[i] = 0.f;
#pragma unroll
          for (int c = 0; c < kMaxClusterParts; ++c)
            if (c < parts) {
              const uint32_t at = cluster_addr(from + v * 4096, c);
              const float4 u0 = ld_cluster_16(at), u1 = ld_cluster_16(at + 2048);
              acc[0] = fmaf(u0.x, x[c].x, acc[0]);
              acc[1] = fmaf(u0.y, x[c].x, acc[1]);
              acc[2] = fmaf(u0.z, x[c].x, acc[2]);
              acc[3] = fmaf(u0.w, x[c].x, acc[3]);
              acc[4] = fmaf(u1.x, x[c].x, acc[4]);
              acc[5] = fmaf(u1.y, x[c].x, acc[5]);
              acc[6] = fmaf(u1.z, x[c].x, acc[6]);
              acc[7] = fmaf(u1.w, x[c].x, acc[7]);
            }
          UNSTEP_STORE(out_v, dst + v, p.extent_out,
                       make_uint4(pack_bf16x2(acc[0] * inv_l, acc[1] * inv_l), pack_bf16x2(acc[2] * inv_l, acc[3] * inv_l),
                                  pack_bf16x2(acc[4] * inv_l, acc[5] * inv_l), pack_bf16x2(acc[6] * inv_l, acc[7] * inv_l)),
                       p.status);
        }
      }
    }
  }
  // The other roles meet the softmax groups at the cluster's barrier, and no block leaves while another reads its part.
  if (kCluster) {
    if (warp >= 8) {
      __syncwarp();
      cluster_sync();
    }
    __syncwarp();
    cluster_sync();
  }

  // ---- teardown: every role ends here, also after a timed-out wait --------------------
  tc_fence_before();
  __syncthreads();
  if (warp == 10 && lane == 0 && *abort_flag) {
    // gave up: let copies that are still in flight land (bounded) before smem is released
    const long long t0 = clock64();
    while (clock64() - t0 < 4000000LL) {
    }
  }
  __syncthreads();
  if (warp == 8) tmem_dealloc(tmem_base, kTmemCols);
  CTRACE(7);
}

// A wait on a barrier that nothing ever arrives at, with a short limit: exercises the give-up
// path of Waiter (status word, flag, orderly return) without any other work.
__global__ void wait_limit_probe_kernel(long long limit_cycles) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    abort_flag = 0;
    mbar_fence_init();
  }
  __syncthreads();
  const Waiter w{&abort_flag, limit_cycles};
  w.wait(smem_u32(&bar), 0);
  __syncthreads();
}

// --------------------------------------------------------------------------
// Host side
// --------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

static EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* sym = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(sym);
  });
  return fn;
}

// bf16 tensor map with 128-byte swizzle, box = 64 elements x 128 rows of dimension `row_dim`.
static bool make_map(CUtensorMap* m, const void* base, int rank, const uint64_t* dims,
                     const uint64_t* strides_bytes, int row_dim) {
  EncodeTiledFn fn = get_encode_fn();
  if (fn == nullptr) return false;
  cuuint64_t gdim[5], gstride[4];
  cuuint32_t box[5], estr[5];
  for (int i = 0; i < rank; ++i) {
    gdim[i] = dims[i];
    box[i] = 1;
    estr[i] = 1;
    if (i > 0) gstride[i - 1] = strides_bytes[i - 1];
  }
  box[0] = 64;
  box[row_dim] = 128;
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<void*>(base), gdim, gstride, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

struct DeviceInfo {
  bool ok = false;
  int sm_count = 0;
  int32_t clusters[kMaxClusterParts + 1] = {};   // clusters of that many blocks which the device runs at the same time
};

// Set up and queried once per device and process; each thread keeps a copy for the device it uses.
static DeviceInfo query_device(int dev) {
  static std::mutex mutex;
  static std::map<int, DeviceInfo> known;
  std::lock_guard<std::mutex> lock(mutex);
  auto it = known.find(dev);
  if (it != known.end()) return it->second;
  DeviceInfo info;
  info.ok = cudaDeviceGetAttribute(&info.sm_count, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
            cudaFuncSetAttribute(window_attn_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kAttnSmemBytes) == cudaSuccess &&
            cudaFuncSetAttribute(window_attn_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kAttnSmemBytes) == cudaSuccess;
  if (!info.ok) return info;
  for (int parts = 2; parts <= kMaxClusterParts; ++parts) {
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = parts;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(parts);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kAttnSmemBytes;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, window_attn_kernel<true>, &cfg) == cudaSuccess) info.clusters[parts] = n;
    else cudaGetLastError();   // no clusters of that size, then
  }
  return known[dev] = info;
}

static const DeviceInfo& device_info() {
  static thread_local int cached_dev = -1;
  static thread_local DeviceInfo info;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    info.ok = false;
    return info;
  }
  if (dev != cached_dev || !info.ok) {
    info = query_device(dev);
    cached_dev = dev;
  }
  return info;
}

// Scratch for split items, one per (device, stream): calls on one stream run in order and may
// share it; calls on different streams may overlap on the GPU and must not.  Captured graphs hold
// its addresses, so nothing is given back before unstep_shutdown().  The partial results have two
// slots per SM whatever the launch: the workers of a launch go up and down with the start frame (one
// to all SMs), and a buffer sized by them would move under graphs captured before.  The counters
// go by the work items of the shape and at least double when they grow, so the arrays they have
// left behind are together no larger than the one in use.
struct Workspace {
  float* part = nullptr;
  int* counters = nullptr;
  size_t slots = 0, n_counters = 0;
};
constexpr size_t kLeastCounters = 4096;
constexpr int kMaxGrowths = 32;
struct StreamScratch {
  Workspace ws;
  Workspace left[kMaxGrowths];   // counters of former calls; captured graphs may still count in them
  int n_left = 0;
};
static std::mutex g_ws_mutex;
static std::map<std::pair<int, cudaStream_t>, StreamScratch> g_workspaces;

static int get_workspace(cudaStream_t st, size_t slots, size_t n_counters, Workspace* out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return UNSTEP_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_ws_mutex);
  StreamScratch& s = g_workspaces[std::make_pair(dev, st)];
  Workspace& ws = s.ws;
  if (ws.part == nullptr) {
    if (cudaMalloc(&ws.part, slots * kPartFloats * sizeof(float)) != cudaSuccess) {
      ws.part = nullptr;
      return UNSTEP_ERR_CUDA;
    }
    ws.slots = slots;
  }
  if (ws.n_counters < n_counters) {
    size_t n = ws.n_counters > 0 ? 2 * ws.n_counters : kLeastCounters;
    while (n < n_counters) n *= 2;
    int* counters = nullptr;
    if (s.n_left == kMaxGrowths || cudaMalloc(&counters, n * sizeof(int)) != cudaSuccess) return UNSTEP_ERR_CUDA;
    // cleared on the caller's stream, so that the clear is ordered before the kernel that follows
    // (a non-blocking stream is not ordered against the legacy default stream)
    if (cudaMemsetAsync(counters, 0, n * sizeof(int), st) != cudaSuccess) {
      cudaFree(counters);
      return UNSTEP_ERR_CUDA;
    }
    if (ws.counters != nullptr) s.left[s.n_left++] = ws;
    ws.counters = counters;
    ws.n_counters = n;
  }
  *out = ws;
  return UNSTEP_OK;
}

// After a kernel gave up, arrival counters may be left non-zero: clear them all.
static void reset_workspace_counters() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return;
  std::lock_guard<std::mutex> lock(g_ws_mutex);
  for (auto& kv : g_workspaces) {
    if (kv.first.first != dev) continue;
    const StreamScratch& s = kv.second;
    if (s.ws.counters != nullptr) cudaMemset(s.ws.counters, 0, s.ws.n_counters * sizeof(int));
    for (int i = 0; i < s.n_left; ++i) cudaMemset(s.left[i].counters, 0, s.left[i].n_counters * sizeof(int));
  }
}

// Device address of g_status on the current device, looked up once per device.
int* status_word() {
  static std::mutex mutex;
  static int* addr[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lock(mutex);
  if (addr[dev] == nullptr) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_status) != cudaSuccess) return nullptr;
    addr[dev] = static_cast<int*>(ptr);
  }
  return addr[dev];
}

}  // namespace unstep

using namespace unstep;

// Hands out the scratch of one launch: `slots` partial-result slots (two per SM) and at least
// `n_counters` zeroed arrival counters.
typedef int (*ScratchFn)(cudaStream_t st, size_t slots, size_t n_counters, Workspace* out);   // an unstep_status

constexpr int kOverlapSteps = 64;   // key-tile steps per worker below which a launch overlaps the kernel before it

// Validation, work split, tensor maps and launch shared by the attention entry points.
// The cache has `sink_frames` slots in front of the ring (0 for the plain rolling window);
// stream b attends frames [0, min(sink_attend, lo)) and [lo, hi), lo = max(0, hi - window_frames).
static int window_attn_run(const unstep_shape_t* shape, const int32_t* start_frame,
                           int32_t window_frames, const void* q_rot, const void* ring_k,
                           const void* ring_v, void* out, void* cuda_stream, ScratchFn scratch,
                           int32_t sink_frames = 0, int32_t sink_attend = 0) {
  int rc = check_attn_args(shape, start_frame, window_frames, sink_frames, sink_attend);
  if (rc != UNSTEP_OK) return rc;
  const void* ptrs[] = {q_rot, ring_k, ring_v, out};
  for (const void* ptr : ptrs)
    if (ptr == nullptr || !aligned16(ptr)) return UNSTEP_ERR_INVALID_ARG;
  rc = check_device();
  if (rc != UNSTEP_OK) return rc;
  const DeviceInfo& info = device_info();
  if (!info.ok) return UNSTEP_ERR_CUDA;

  const uint64_t Hn = shape->heads;
  const uint64_t C = static_cast<uint64_t>(shape->ring_frames) + sink_frames;  // cache slots per stream
  const uint64_t T = static_cast<uint64_t>(shape->grid_h) * shape->grid_w;
  const uint64_t L = T * shape->chunk_frames;
  const uint64_t row_bytes = Hn * kHeadDim * 2;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);

  AttnParams p;
  plan_shape(p, shape, sink_frames);
  for (int b0 = 0; b0 < shape->batch; b0 += kMaxStreamsPerLaunch) {
    const int nb = shape->batch - b0 < kMaxStreamsPerLaunch ? shape->batch - b0 : kMaxStreamsPerLaunch;
    rc = plan_launch(p, shape, start_frame + b0, nb, window_frames, sink_frames, sink_attend, info.sm_count,
                     info.clusters);
    if (rc != UNSTEP_OK) return rc;
    Workspace ws;
    rc = scratch(st, 2 * static_cast<size_t>(info.sm_count), 2 * static_cast<size_t>(nb) * p.items_per_stream, &ws);
    if (rc != UNSTEP_OK) return rc;
    p.part = ws.part;
    p.counters = ws.counters;
    p.status = status_word();
    p.out_wide = (reinterpret_cast<uintptr_t>(out) & 31u) == 0;   // rows are multiples of 256 bytes
    p.extent_out = static_cast<int64_t>(nb) * p.L * p.Hn * (kHeadDim / 8);
    p.extent_part = static_cast<int64_t>(ws.slots) * kPartFloats;
    p.extent_counters = static_cast<int64_t>(ws.n_counters);
    const char* qb = static_cast<const char*>(q_rot) + static_cast<uint64_t>(b0) * L * row_bytes;
    const char* kb = static_cast<const char*>(ring_k) + static_cast<uint64_t>(b0) * C * T * row_bytes;
    const char* vb = static_cast<const char*>(ring_v) + static_cast<uint64_t>(b0) * C * T * row_bytes;
    __nv_bfloat16* ob = reinterpret_cast<__nv_bfloat16*>(static_cast<char*>(out) +
                                                         static_cast<uint64_t>(b0) * L * row_bytes);
    CUtensorMap tm_q, tm_k, tm_v, tm_kf, tm_vf;
    const uint64_t qdims[4] = {kHeadDim, Hn, L, static_cast<uint64_t>(nb)};
    const uint64_t qstr[3] = {kHeadDim * 2, row_bytes, L * row_bytes};
    const uint64_t rdims[5] = {kHeadDim, Hn, T, C, static_cast<uint64_t>(nb)};
    const uint64_t rstr[4] = {kHeadDim * 2, row_bytes, T * row_bytes, C * T * row_bytes};
    const uint64_t fdims[4] = {kHeadDim, Hn, C * T, static_cast<uint64_t>(nb)};   // ring rows, flat
    const uint64_t fstr[3] = {kHeadDim * 2, row_bytes, C * T * row_bytes};
    if (!make_map(&tm_q, qb, 4, qdims, qstr, 2) || !make_map(&tm_k, kb, 5, rdims, rstr, 2) ||
        !make_map(&tm_v, vb, 5, rdims, rstr, 2) || !make_map(&tm_kf, kb, 4, fdims, fstr, 2) ||
        !make_map(&tm_vf, vb, 4, fdims, fstr, 2))
      return UNSTEP_ERR_CUDA;
    // Set up under the append before it where the launch is short.  Append and attention (with the pipeline of one
    // S per query tile, 10 % slower per step), us not
    // overlapped -> overlapped, by steps per worker: in runs of 20 (full clock) 24: 78.9 -> 76.5, 35:
    // 94.6 -> 92.6, 57: 143.1 -> 142.3, 114: 242.0 -> 240.6, 226: 446.1 -> 445.5, 394: 754.9 -> 763.7; run
    // on end at the power cap 24: 80.2 -> 79.8 (1912 -> 1867 MHz), 57: 155.2 -> 155.8 (1792 -> 1776), 114:
    // 276.7 -> 276.6 (1702 -> 1688), 169: 395.4 -> 398.6 (1680 -> 1652), 394: 880.4 -> 895.9 (1635 -> 1605).
    // The overlap saves 1.5-6 thousand cycles of a launch at any length; at the cap the clock falls for
    // the idling it takes away.  The line lies about where the gain of short runs (0.6 % at 57 steps) has
    // come down to the loss of runs at the cap (0.4 %).
    const bool brief = p.all_steps < static_cast<int64_t>(kOverlapSteps) * p.n_workers;
    const cudaError_t err =
        launch_clusters(brief, p.cluster ? p.parts : 1, p.cluster ? window_attn_kernel<true> : window_attn_kernel<false>,
                        p.n_workers, kThreads, kAttnSmemBytes, st, tm_q, tm_k, tm_v, tm_kf, tm_vf, p, ob);
    g_launches.fetch_add(1);
    if (err != cudaSuccess) return UNSTEP_ERR_CUDA;
  }
  return UNSTEP_OK;
}

#ifdef UNSTEP_TRACE
extern "C" int unstep_debug_read_cta_trace(unsigned long long* host_out) {
  if (cudaDeviceSynchronize() != cudaSuccess) return UNSTEP_ERR_CUDA;
  return cudaMemcpyFromSymbol(host_out, g_cta_trace, sizeof(unsigned long long) * 160 * 16) == cudaSuccess
             ? UNSTEP_OK : UNSTEP_ERR_CUDA;
}
extern "C" int unstep_debug_read_trace(long long* host_out) {
  if (cudaDeviceSynchronize() != cudaSuccess) return UNSTEP_ERR_CUDA;
  return cudaMemcpyFromSymbol(host_out, g_trace, sizeof(long long) * 12 * 64 * 8) == cudaSuccess
             ? UNSTEP_OK : UNSTEP_ERR_CUDA;
}
#endif

extern "C" int unstep_window_attn(const unstep_shape_t* shape, const int32_t* start_frame,
                                  int32_t window_frames, const void* q_rot, const void* ring_k,
                                  const void* ring_v, void* out, void* cuda_stream) {
  return window_attn_run(shape, start_frame, window_frames, q_rot, ring_k, ring_v, out, cuda_stream,
                         get_workspace);
}

extern "C" int unstep_window_attn_sink(const unstep_shape_t* shape, int32_t sink_frames,
                                       const int32_t* start_frame, int32_t recent_frames,
                                       int32_t sink_attend, const void* q_rot, const void* cache_k,
                                       const void* cache_v, void* out, void* cuda_stream) {
  return window_attn_run(shape, start_frame, recent_frames, q_rot, cache_k, cache_v, out, cuda_stream,
                         get_workspace, sink_frames, sink_attend);
}

// --------------------------------------------------------------------------
// Attention without any allocation: the scratch is a fixed array in the library image.
// --------------------------------------------------------------------------
namespace unstep {

constexpr int kStaticMaxCtas = 148;                      // two partial-result slots per CTA
constexpr int kStaticMaxCounters = 2 * 32768;            // a pair of counters per work item
constexpr size_t kStaticCounterBytes = sizeof(int) * kStaticMaxCounters;
constexpr size_t kStaticScratchBytes =
    kStaticCounterBytes + sizeof(float) * 2 * kStaticMaxCtas * static_cast<size_t>(kPartFloats);

// Counters first, partial results after them.  In host code this name is only a handle for
// cudaGetSymbolAddress: it is not a device address and must never be passed to a kernel.
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

constexpr int kMaxDevices = 64;
static std::mutex g_static_mutex;
static unsigned char* g_static_addr[kMaxDevices] = {};

// Device address of the array on the current device (looked up once per device).
static unsigned char* static_scratch_base() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return nullptr;
  std::lock_guard<std::mutex> lock(g_static_mutex);
  if (g_static_addr[dev] == nullptr) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || ptr == nullptr) return nullptr;
    g_static_addr[dev] = static_cast<unsigned char*>(ptr);
  }
  return g_static_addr[dev];
}

// Scratch source of the no-allocation entry point: carve the fixed array, clear the counters
// this launch will use (the array keeps the previous call's contents).
static int static_scratch(cudaStream_t st, size_t slots, size_t n_counters, Workspace* out) {
  if (slots > 2 * static_cast<size_t>(kStaticMaxCtas) || n_counters > static_cast<size_t>(kStaticMaxCounters))
    return UNSTEP_ERR_TOO_LARGE;
  unsigned char* base = static_scratch_base();
  if (base == nullptr) return UNSTEP_ERR_CUDA;
  if (cudaMemsetAsync(base, 0, n_counters * sizeof(int), st) != cudaSuccess) return UNSTEP_ERR_CUDA;
  out->counters = reinterpret_cast<int*>(base);
  out->part = reinterpret_cast<float*>(base + kStaticCounterBytes);
  out->slots = slots;
  out->n_counters = n_counters;
  return UNSTEP_OK;
}

}  // namespace unstep

extern "C" int unstep_window_attn_noalloc(const unstep_shape_t* shape, const int32_t* start_frame,
                                          int32_t window_frames, const void* q_rot, const void* ring_k,
                                          const void* ring_v, void* out, void* cuda_stream) {
  // size limits of the fixed array first, so that an oversized problem gets its own clear answer
  int rc = check_shape(shape, true);
  if (rc != UNSTEP_OK) return rc;
  const int64_t L = static_cast<int64_t>(shape->grid_h) * shape->grid_w * shape->chunk_frames;
  const int64_t q_pairs = ((L + kTileM - 1) / kTileM + 1) / 2;
  const int64_t streams = shape->batch < kMaxStreamsPerLaunch ? shape->batch : kMaxStreamsPerLaunch;
  if (2 * streams * shape->heads * q_pairs > kStaticMaxCounters) return UNSTEP_ERR_TOO_LARGE;
  rc = check_device();
  if (rc != UNSTEP_OK) return rc;
  const DeviceInfo& info = device_info();
  if (!info.ok) return UNSTEP_ERR_CUDA;
  if (info.sm_count > kStaticMaxCtas) return UNSTEP_ERR_TOO_LARGE;
  return window_attn_run(shape, start_frame, window_frames, q_rot, ring_k, ring_v, out, cuda_stream,
                         static_scratch);
}

extern "C" int unstep_attn_workers(int32_t* workers, int32_t* ctas_per_worker) {
  if (workers == nullptr || ctas_per_worker == nullptr) return UNSTEP_ERR_INVALID_ARG;
  const int rc = check_device();
  if (rc != UNSTEP_OK) return rc;
  const DeviceInfo& info = device_info();
  if (!info.ok) return UNSTEP_ERR_CUDA;
  *workers = info.sm_count;
  *ctas_per_worker = 1;
  return UNSTEP_OK;
}

extern "C" int unstep_attn_clusters(int32_t* clusters) {
  if (clusters == nullptr) return UNSTEP_ERR_INVALID_ARG;
  const int rc = check_device();
  if (rc != UNSTEP_OK) return rc;
  const DeviceInfo& info = device_info();
  if (!info.ok) return UNSTEP_ERR_CUDA;
  for (int n = 0; n <= kMaxClusterParts; ++n) clusters[n] = info.clusters[n];
  return UNSTEP_OK;
}

#ifdef UNSTEP_CHECK
namespace unstep {
// One store just past the end of a 4-element buffer: a checking build must skip it and record it.
__global__ void check_probe_kernel(int* buf, int* status) {
  UNSTEP_STORE(buf, threadIdx.x, 4, 7, status);
}
// Two 32-byte stores into three 16-byte vectors: the second one is half outside and must be skipped whole.
__global__ void check_probe_wide_kernel(int* buf, int* status) {
  const uint32_t w[8] = {7, 7, 7, 7, 7, 7, 7, 7};
  UNSTEP_STORE_32(reinterpret_cast<uint4*>(buf), 2 * threadIdx.x, 3, w, status);
}
}  // namespace unstep

extern "C" int unstep_selftest_bounds_check(int32_t* device_buf5, void* cuda_stream) {
  if (device_buf5 == nullptr) return UNSTEP_ERR_INVALID_ARG;
  const int rc = check_device();
  if (rc != UNSTEP_OK) return rc;
  int* st = status_word();
  if (st == nullptr) return UNSTEP_ERR_CUDA;
  check_probe_kernel<<<1, 5, 0, static_cast<cudaStream_t>(cuda_stream)>>>(device_buf5, st);
  g_launches.fetch_add(1);
  return cudaGetLastError() == cudaSuccess ? UNSTEP_OK : UNSTEP_ERR_CUDA;
}

extern "C" int unstep_selftest_bounds_check_wide(int32_t* device_buf16, void* cuda_stream) {
  if (device_buf16 == nullptr || (reinterpret_cast<uintptr_t>(device_buf16) & 31u) != 0) return UNSTEP_ERR_INVALID_ARG;
  const int rc = check_device();
  if (rc != UNSTEP_OK) return rc;
  int* st = status_word();
  if (st == nullptr) return UNSTEP_ERR_CUDA;
  check_probe_wide_kernel<<<1, 2, 0, static_cast<cudaStream_t>(cuda_stream)>>>(device_buf16, st);
  g_launches.fetch_add(1);
  return cudaGetLastError() == cudaSuccess ? UNSTEP_OK : UNSTEP_ERR_CUDA;
}
#endif

extern "C" int unstep_selftest_wait_limit(int64_t limit_cycles, void* cuda_stream) {
  if (limit_cycles < 1 || limit_cycles > 4000000000LL) return UNSTEP_ERR_INVALID_ARG;
  const int rc = check_device();
  if (rc != UNSTEP_OK) return rc;
  wait_limit_probe_kernel<<<1, 64, 0, static_cast<cudaStream_t>(cuda_stream)>>>(limit_cycles);
  g_launches.fetch_add(1);
  return cudaGetLastError() == cudaSuccess ? UNSTEP_OK : UNSTEP_ERR_CUDA;
}

extern "C" void unstep_shutdown(void) {
  // frees the per-stream scratch buffers of every device; the next attention call makes new ones
  cudaDeviceSynchronize();
  int cur = 0;
  if (cudaGetDevice(&cur) != cudaSuccess) return;
  std::lock_guard<std::mutex> lock(g_ws_mutex);
  for (auto& kv : g_workspaces) {
    if (cudaSetDevice(kv.first.first) != cudaSuccess) continue;
    cudaDeviceSynchronize();
    const StreamScratch& s = kv.second;
    if (s.ws.part != nullptr) cudaFree(s.ws.part);
    if (s.ws.counters != nullptr) cudaFree(s.ws.counters);
    for (int i = 0; i < s.n_left; ++i) cudaFree(s.left[i].counters);
  }
  g_workspaces.clear();
  cudaSetDevice(cur);
}

extern "C" int unstep_poll_status(void) {
  if (cudaDeviceSynchronize() != cudaSuccess) return UNSTEP_ERR_CUDA;
  int st = 0, zero = 0;
  if (cudaMemcpyFromSymbol(&st, g_status, sizeof(int)) != cudaSuccess) return UNSTEP_ERR_CUDA;
  if (st != 0) {
    if (cudaMemcpyToSymbol(g_status, &zero, sizeof(int)) != cudaSuccess) return UNSTEP_ERR_CUDA;
    if (st == UNSTEP_ERR_TIMEOUT) reset_workspace_counters();
  }
  return st;
}
