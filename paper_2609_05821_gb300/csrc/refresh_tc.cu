// Tensor-core causal refresh attention for bf16 caches with head_dim up to 128
// (selective recompute, Conduit Sec. 3.1 / 4.3):
//   out[l][i][h] = sum_{j <= p_i} softmax_j(<q[l][i][h], K'[l][h/G][j]> / sqrt(d)) V'[l][h/G][j]
//
// Two kernels; launch_refresh_tc chooses. A query tile is floor(128/G)
// consecutive selected rows times the G query heads that share the KV head,
// 128 rows of one (layer, KV head, request). Keys stream in tiles of 128. Both
// kernels are persistent: one CTA per SM takes items from an atomic counter.
//
// refresh_tc_kernel: two query tiles A and B per work item; B holds the later
// rows. Every K and V tile is copied once for both. Roles (384 threads):
//   warp 0      takes and decodes the items (record and row positions in
//               shared memory, one item ahead) and loads the K tiles
//   warp 2      loads the V tiles
//   warps 1, 3  the query tile and the MMAs of A and of B. The whole warp walks
//               the schedule on uniform values and one lane issues: beside the
//               softmax warps that keeps an MMA at its 64 tensor cycles, where
//               one lane of a diverged warp needs 83
//   warps 4-7   softmax of tile A, warps 8-11 of tile B: each thread owns one
//               row (TMEM lane) and all 128 keys of a key tile. It reads S(t),
//               applies the causal mask j <= p_i, keeps a lazy running max (O
//               and the row sum are rescaled only when the max grows by 2^8;
//               warp-uniform, since tcgen05.ld/st are warp-collective), writes
//               P as bf16 pairs over the upper half of S(t), and at the item's
//               end writes its row of O / rowsum.
// A turn of an MMA warp is P_x(t) V(t) and then S_x(t+1); the warps take turns
// strictly, so the two tiles stay half a period apart and one tile's softmax
// runs beside the other's MMAs (without turns both softmaxes fall into step:
// 1.1 x slower). MMAs of one thread execute in issue order, so S_x(t+1) may
// overwrite P_x(t) without a wait, and S_x(t+1) ready implies that P_x(t) V(t)
// has completed (the softmax may then rescale O_x).
// TMEM: S_A, S_B at columns [0, 256), O_A, O_B at [256, 512).
//
// What bounds it: the chain softmax (about 1 150 cycles for 128 keys a thread)
// -> P V -> next S of a tile, about 3 000 cycles per pair of tiles against 2 048
// of tensor work.
//
// one_refresh_tc_kernel: one query tile per item, three S buffers, and the two
// softmax warps of a lane quarter share each key tile. It takes about 1 650
// cycles per tile, but its items are half as long, so it is the faster one where
// few items reach an SM, and for the head sizes below 128 throughout. Roles:
//   warp 0      items, query tiles (two buffers) and K tiles; warp 10 V tiles
//   warp 1      S(t) = Q K(t)^T into TMEM buffer t % 3; warp 11 O += P(t) V(t).
//               Two warps, because one issuing both, with a wait for each P V
//               before the S that reuses its buffer, took longer per key tile
//               than the softmax; both converged, as above (refresh attention
//               of 16 layers of 4 096 keys 201 -> 196 us)
//   warps 2-9   softmax: a thread owns one row and 64 of the 128 keys; the two
//               halves of a row exchange their maxima through shared memory
// TMEM: S buffers at columns [0, 384) (P in the upper 64 of each), O at
// [384, 512). S(t) is issued once P(t-3) V(t-3) has completed.
//
// In both, rows a box leaves empty (G not a power of two) hold zeros and are
// never masked: as fully masked rows they sent their warps down the masking
// path in every key tile (28 heads, 8 192 tokens: 1 254 -> 970 us).
//
// Rows past a request's last key (the next request's, or a page's rows without a
// token) reach no output: the two-tile kernel's V warp clears them in the last tile,
// the other's P V warp in its last 16-key step, leaving out the steps behind it. A V
// that is not finite at a later position of the same request is kept out of earlier
// rows below 128 dims (redo_rows); at 128 dims it makes rows of its item NaN.
//
// Measured (GB300, the kernel before and this one timed in turn, back to back):
// multi-image prompt 1 413 -> 1 036 us (at the power limit; 1 254 -> 891 one call at a
// time), batched serving 23.2 -> 19.5 ms, long document 18.6 -> 17.5 ms, single image
// 43.5 -> 38.2 us, 16 layers of 4 096 tokens 225 -> 196 us, 2 layers of 1 885 25.2 ->
// 20.6 us.
//
// The staleness estimator (kStale, 128 dims) runs the same schedule with every scoring
// row of a request at its last key: V is the draw z itself, the softmax warps scale
// each V tile by its keys' standard deviations in shared memory while they would
// wait for their next S (in place of a pass that writes xi = scale z to memory),
// and a row ends as ||O / rowsum||^2, summed over its warp's rows, instead of an
// output row. (Scaling P instead costs accuracy: a row's largest weight is then
// no longer exactly 1.)
//
// Rows are sorted by position, so an item needs keys up to its last row's
// position only (tile A often fewer than tile B). Every barrier phase follows
// from per-CTA sequence numbers that all roles advance alike. Every wait is
// bounded by one second; a role that gives up raises an abort flag the others
// watch, the kernel sets CONDUIT_FLAG_TIMEOUT, drains its copies and MMAs, and
// frees TMEM.
#include <cuda.h>
#include <limits.h>

#include "internal.cuh"
#include "tc_common.cuh"

namespace conduit {
namespace {

constexpr int kMaxD = 128;
constexpr int kKT = 128;                         // keys per tile
constexpr int kRows = 128;                       // rows per query tile
constexpr int kMmaWarp = 1, kVWarp = 2, kSoftWarp0 = 4;  // warp 0: items and K; warps 1, 3: MMAs
constexpr int kThreads = 384;
constexpr uint32_t kHalfBytes = 128 * 128;       // 16 KB: one 64-dim half of a 128-row tile
constexpr int kRecReaders = 11;                  // two MMA warps, V warp, eight softmax warps
constexpr uint32_t kBarBytes = 384;             // barriers, TMEM slot, abort flag, counters
constexpr uint32_t kTailBytes = kBarBytes + 2 * (16 + 2 * kRows) * 4;

constexpr uint32_t kTileBytes = 2 * kHalfBytes;  // a query, K or V tile of 128 dims
// K and V tiles in one ring, K(0) V(0) K(1) V(1) ...: tile T may be loaded once tile
// T - kAhead is done (by both streams), and fewer than kDone tiles are undecided.
constexpr int kStages = 5;
constexpr int kAhead = (kStages - 1) / 2;
constexpr int kDone = 2 * kAhead;
constexpr uint32_t kSmem = (2 + kStages) * kTileBytes + kTailBytes;
static_assert(kSmem <= 232448, "shared memory of one CTA");
static_assert((kStages + 2 * kDone + 6 + 4 + 4 + 2 + 1) * 8 + 32 <= kBarBytes, "barriers and counters");
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kSCols = 128;                 // one S buffer
constexpr uint32_t kPCol = 64;                   // P (bf16 pairs) over the upper half of S ...
constexpr uint32_t kPLoCol = 0;                  // ... and its rounding errors over the lower one (kSplit)
constexpr uint32_t kOCol = 2 * kSCols;           // O_A, then O_B
constexpr float kRescaleLog2 = 8.f;
constexpr int kPassEarly = 2;                    // MMAs of a turn still to issue when the other stream's may start

struct RefArgs {
  KvDev kv;
  BatchDev b;
  const int32_t* idx;
  const int32_t* idx_off;
  __nv_bfloat16* out;
  int32_t out32;           // out is 32-byte aligned: rows are written in 32-byte stores
  int32_t n_sel;
  int32_t rows_per_tile;   // selected rows per query tile, floor(128 / G)
  int32_t n_blocks;        // items (blocks) per (layer, KV head)
  int32_t n_items;         // n_blocks * Hkv * L
  int32_t span;            // selected rows per item: of one query tile or of two
  int32_t tail;            // the last `tail` (layer, KV head) pairs come longest block first (see decode_item)
  int32_t* next_item;      // work counter, zero at launch; NULL: CTA c takes items c, c + grid, ...
  float scale_log2;
  int32_t* status;
  // kStale: idx_off holds the requests' query offsets, n_sel the query count
  int32_t draws;           // n_items = draws * n_blocks * Hkv * L
  const float* key_scale;  // [L][Hkv][n_tot]
  double* part;            // [draws][L * Hkv][n_blocks][2 query tiles][4 warps]
  const __nv_bfloat16* q;  // the query rows, laid out as `out` (not kStale)
};

// A work item: block `blk` of (layer l, KV head g), counted from the largest
// positions, and the request, first selected row and row count. A request's
// blocks are cut from its last row down, so only the block of its smallest
// positions may be partly filled.
// Item order: (layer, head)-major up to the last `tail` pairs, so that the CTAs
// in flight work on few K/V prefixes, which L2 then shares; then all blocks of
// the last pairs, longest first (every layer and head of a request has the same
// selected positions). Longest-first is what evens out the end of the launch.
struct Item {
  int l, g, r, i0, cnt, m, blk;
};

template <bool kStale>
__device__ __forceinline__ Item decode_item(const RefArgs& a, int u) {
  Item it;
  const int n_lg = a.kv.Hkv * a.kv.L;
  it.m = 0;
  if (kStale) {  // a (layer, head)'s blocks and draws follow one another: its K stays in L2
    it.m = u / a.n_blocks % a.draws;
    u = u / (a.n_blocks * a.draws) * a.n_blocks + u % a.n_blocks;
  }
  const int v = u - (n_lg - a.tail) * a.n_blocks;
  const int x = v >= 0 ? v / a.tail : u % a.n_blocks;
  const int lg = v >= 0 ? n_lg - a.tail + v % a.tail : u / a.n_blocks;
  it.g = lg % a.kv.Hkv;
  it.l = lg / a.kv.Hkv;
  int blk = a.n_blocks - 1 - x;
  it.blk = blk;
  it.r = 0;
  it.i0 = 0;
  it.cnt = 0;
  const int span = a.span;
  for (int rr = 0; rr < a.b.R; ++rr) {
    const int k0 = a.idx_off[rr], kr = a.idx_off[rr + 1] - k0;
    const int nb = (kr + span - 1) / span;
    if (blk < nb) {
      const int end = kr - (nb - 1 - blk) * span, begin = max(0, end - span);
      it.r = rr;
      it.i0 = k0 + begin;
      it.cnt = end - begin;
      break;
    }
    blk -= nb;
  }
  return it;
}

struct Smem {
  uint8_t* q;        // [2 tiles][halves][128 rows][128 B]
  uint8_t* kv;       // [kStages][halves][128 keys][128 B]: K tile t of the CTA in slot 2t mod kStages, V in 2t + 1
  uint64_t* full;             // [kStages]
  uint64_t* done;             // [kDone] tile T of the CTA: both streams have used K(T) and V(T - 1)
  uint64_t *sfull, *pfull;    // [2] per query tile: S computed / P written
  uint64_t *ofull;            // [2] per query tile, once per item that has rows in it: O complete
  uint64_t* qfull;            // [2] per query tile
  uint64_t* turn;             // [2] the stream's MMA warp may issue its next turn
  uint64_t *recfull, *recempty;  // [2] item records
  uint64_t* mdone;            // [2] per MMA warp: all its MMAs completed
  uint32_t* tmem_slot;
  volatile int* abort;
  uint32_t* counters;  // [0] K tiles, [1] V tiles loaded
  // per item parity, written by the loader: the decoded item {u (-1: no more
  // work), l, g, r, i0, rows of A, rows of B, key tiles of A, of B, N_r, t0, m, block}
  // and the positions of its selected rows, so that the other roles read no
  // global memory between items
  volatile int* rec;   // [2][16]
  volatile int* pos;   // [2][2 tiles][kRows]
  uint64_t* scaled;    // [kDone] (kStale) tile T's V has been scaled
  uint64_t* raw;       // [1] the copy of a V tile that ends past its request's keys
};

__device__ __forceinline__ Smem carve(uint8_t* base) {
  Smem s;
  s.q = base;
  s.kv = s.q + 2 * kTileBytes;
  uint64_t* bar = reinterpret_cast<uint64_t*>(s.kv + kStages * kTileBytes);
  s.full = bar;
  s.done = s.full + kStages;
  s.sfull = s.done + kDone;
  s.pfull = s.sfull + 2;
  s.ofull = s.pfull + 2;
  s.qfull = s.ofull + 2;
  s.turn = s.qfull + 2;
  s.recfull = s.turn + 2;
  s.recempty = s.recfull + 2;
  s.mdone = s.recempty + 2;
  s.scaled = s.mdone + 2;
  s.tmem_slot = reinterpret_cast<uint32_t*>(s.scaled + kDone);
  s.abort = reinterpret_cast<volatile int*>(s.tmem_slot + 1);
  s.counters = reinterpret_cast<uint32_t*>(s.tmem_slot + 2);
  s.raw = reinterpret_cast<uint64_t*>(s.counters + 2);
  s.rec = reinterpret_cast<volatile int*>(reinterpret_cast<uint8_t*>(bar) + kBarBytes);
  s.pos = s.rec + 2 * 16;
  return s;
}
__device__ __forceinline__ bool wait_or_abort(uint64_t* bar, uint32_t parity, volatile int* abort) {
  if (tc::mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = tc::globaltimer_ns();
  for (uint32_t i = 1; i < tc::kSpinLimit; ++i) {
    if (tc::mbar_try_wait(bar, parity)) return true;
    if ((i & 7u) == 0 && (*abort || tc::globaltimer_ns() - t0 > tc::kWaitNs)) return false;
  }
  return false;
}

// The same for a converged warp. The first test is a plain probe by all lanes,
// which costs about 75 cycles when the phase is complete (a suspending
// try_wait about 100, one lane's wait shared with the others about 250).
__device__ __forceinline__ bool wait_warp(uint64_t* bar, uint32_t parity, volatile int* abort) {
  if (__all_sync(0xffffffffu, tc::mbar_probe(bar, parity))) return true;
  return __all_sync(0xffffffffu, wait_or_abort(bar, parity, abort));
}

__device__ __forceinline__ void raise_abort(const RefArgs& a, volatile int* abort, int32_t site) {
  if (!*abort) flag_status(a.status, CONDUIT_FLAG_TIMEOUT | site);
  *abort = 1;
}

// Warp-cooperative TMA of the 128-key tile starting at request-local key j0:
// lane 0 posts the byte count, then copy c is issued by lane c. A copy is one
// 64-dim half of the whole tile (contiguous cache) or of one page (paged
// cache: 128/page copies per half, up to 32), so a paged tile costs one
// round of parallel page-index loads and copy issues instead of a serial loop.
template <int kHalves>
__device__ __forceinline__ void load_tile(const RefArgs& a, const CUtensorMap* map, uint8_t* dst,
                                          uint64_t* bar, int l, int g, int r, int t0, int N, int j0,
                                          int lane) {
  const KvDev& kv = a.kv;
  if (lane == 0) tc::mbar_arrive_expect_tx(bar, kHalves * kHalfBytes);
  __syncwarp();
  const int hf = lane % kHalves;
  if (kv.page_size == 0) {
    if (lane < kHalves) {
      const int32_t y = int32_t((int64_t(l) * kv.Hkv + g) * kv.n_tot + t0 + j0);
      tc::tma_load_2d(dst + hf * kHalfBytes, map, bar, hf * 64, y);
    }
  } else {
    const int ps = kv.page_size;
    const int i = lane / kHalves;  // page of the tile
    if (i < kKT / ps) {
      const int lp = min((j0 + i * ps) / ps, (N - 1) / ps);  // tail pages repeat the last one (masked)
      const int page = kv.page_table[int64_t(r) * kv.max_pages + lp];
      const int32_t y = int32_t(((int64_t(l) * kv.num_pages + page) * kv.Hkv + g) * ps);
      tc::tma_load_2d(dst + hf * kHalfBytes + i * ps * 128, map, bar, hf * 64, y);
    }
  }
}

// The last V tile of a request may end past its keys: in the next request's rows, or
// in rows of a page that no token has, which may hold anything. P is 0 there, but 0 x
// Inf or NaN is not, so rows first .. end - 1 become zeros, by a whole warp, before an
// MMA reads them.
template <int kHalves>
__device__ __forceinline__ void clear_rows(uint8_t* tile, int first, int end, int lane) {
  for (int i = first * 8 + lane; i < end * 8; i += 32)
    for (int h = 0; h < kHalves; ++h)
      *reinterpret_cast<uint4*>(tile + h * kHalfBytes + i * 16) = make_uint4(0, 0, 0, 0);
  tc::fence_proxy_async_smem();
  __syncwarp();
}

template <bool kStale>
__global__ void __launch_bounds__(kThreads, 1)
    refresh_tc_kernel(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap,
                      const __grid_constant__ CUtensorMap qmap, const __grid_constant__ RefArgs a) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  const Smem s = carve(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const KvDev& kv = a.kv;
  const int G = kv.G, Hq = kv.Hq;
  const int span = a.rows_per_tile;               // selected rows of a query tile
  if (tc::smem_u32(smem_raw) & 1023u) {           // the swizzled tiles need 1024-byte atoms
    if (tid == 0) flag_status(a.status, CONDUIT_FLAG_TIMEOUT | tc::kSiteLoad);
    return;
  }

  if (tid == 0) {
    for (int i = 0; i < kStages; ++i) tc::mbar_init(&s.full[i], 1);
    for (int i = 0; i < kDone; ++i) tc::mbar_init(&s.done[i], 2);    // A's MMAs, B's softmax
    for (int i = 0; i < kDone; ++i) tc::mbar_init(&s.scaled[i], 8);  // the softmax warps
    if (!kStale) tc::mbar_init(s.raw, 1);
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&s.sfull[i], 1);
      tc::mbar_init(&s.pfull[i], 4);     // one arrival per softmax warp of the tile
      tc::mbar_init(&s.ofull[i], 1);
      tc::mbar_init(&s.qfull[i], 1);
      tc::mbar_init(&s.turn[i], 1);
      tc::mbar_init(&s.mdone[i], 1);
      tc::mbar_init(&s.recfull[i], 1);
      tc::mbar_init(&s.recempty[i], kRecReaders);
    }
    *s.abort = 0;
    s.counters[0] = s.counters[1] = 0;
    tc::fence_barrier_init();
    tc::prefetch_tensormap(&kmap);
    tc::prefetch_tensormap(&vmap);
    tc::prefetch_tensormap(&qmap);
  }
  if (warp == kMmaWarp) tc::tmem_alloc(s.tmem_slot, kTmemCols);
  // query rows the boxes never fill: zero, so their logits are finite
  for (uint32_t i = span * G * 128 + tid * 16; i < kHalfBytes; i += kThreads * 16)
    for (int h = 0; h < 4; ++h) *reinterpret_cast<uint4*>(s.q + h * kHalfBytes + i) = make_uint4(0, 0, 0, 0);
  tc::fence_proxy_async_smem();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = *s.tmem_slot;

  // Registers: a softmax thread holds a row of S (128 values). The shares add
  // up to 128 x 88 + 256 x 208 = 384 x 168, what the launch has.
  if (warp < kSoftWarp0) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 88;" ::: "memory");
  if (warp == 0) {
    // ------------------------------------------------ items and K (warp 0)
    uint32_t T = 0;
    bool ok = true;
    for (uint32_t n = 0; ok; ++n) {
      int u = 0;
      if (lane == 0) {
        u = n == 0 ? int(blockIdx.x)
                   : a.next_item ? int(gridDim.x) + atomicAdd(a.next_item, 1) : int(blockIdx.x + n * gridDim.x);
        if (u >= a.n_items) u = -1;
      }
      u = __shfl_sync(0xffffffffu, u, 0);
      const Item it = decode_item<kStale>(a, u < 0 ? 0 : u);
      const int cnt_b = min(it.cnt, span), cnt_a = it.cnt - cnt_b;
      const int t0 = a.b.tok_off[it.r], N = a.b.tok_off[it.r + 1] - t0;
      int my_pos[2 * kRows / 32];  // positions of the item's rows, loaded before the record is free
#pragma unroll
      for (int k = 0; k < 2 * kRows / 32; ++k) {
        const int x = k / (kRows / 32), i = lane + 32 * (k % (kRows / 32));
        my_pos[k] = (!kStale && u >= 0 && i < (x ? cnt_b : cnt_a)) ? a.idx[it.i0 + (x ? cnt_a : 0) + i] : -1;
      }
      auto key_tiles = [&](int first, int cnt) {  // up to the last row's position
        if (u < 0 || cnt == 0) return 0;
        if (kStale) return (N - 1) / kKT + 1;
        const int p = min(a.idx[it.i0 + first + cnt - 1], N - 1);
        return p < 0 ? 0 : p / kKT + 1;
      };
      int nt_a = key_tiles(0, cnt_a), nt = key_tiles(cnt_a, cnt_b);
      nt_a = min(nt_a, nt);  // idx ascends, so this changes nothing unless the caller broke that
      const int rs = n & 1;
      if (!wait_warp(&s.recempty[rs], ((n >> 1) & 1) ^ 1, s.abort)) {
        if (lane == 0) raise_abort(a, s.abort, tc::kSiteLoad);
        break;
      }
      if (!kStale) {
#pragma unroll
        for (int k = 0; k < 2 * kRows / 32; ++k) s.pos[rs * 2 * kRows + lane + 32 * k] = my_pos[k];
      }
      if (lane == 0) {
        volatile int* rec = s.rec + rs * 16;
        rec[0] = u;
        rec[1] = it.l;
        rec[2] = it.g;
        rec[3] = it.r;
        rec[4] = it.i0;
        rec[5] = cnt_a;
        rec[6] = cnt_b;
        rec[7] = nt_a;
        rec[8] = nt;
        rec[9] = N;
        rec[10] = t0;
        rec[11] = it.m;
        rec[12] = it.blk;
      }
      __threadfence_block();
      __syncwarp();  // the lanes' positions are ordered before lane 0's release below
      if (lane == 0) tc::mbar_arrive(&s.recfull[rs]);
      if (u < 0) break;
      for (int t = 0; t < nt; ++t, ++T) {
        const uint32_t sl = 2 * T % kStages;
        if (T >= kAhead && !wait_warp(&s.done[(T - kAhead) % kDone], ((T - kAhead) / kDone) & 1, s.abort)) {
          if (lane == 0) raise_abort(a, s.abort, tc::kSiteLoad);
          ok = false;
          break;
        }
        load_tile<2>(a, &kmap, s.kv + sl * kTileBytes, &s.full[sl], it.l, it.g, it.r, t0, N, t * kKT, lane);
      }
    }
    if (lane == 0) s.counters[0] = T;
  } else if (warp == kVWarp) {
    // ----------------------------------------------------- V loads (warp 2)
    uint32_t T = 0, n_raw = 0;
    bool ok = true;
    for (uint32_t n = 0; ok; ++n) {
      const int rs = n & 1;
      if (!wait_warp(&s.recfull[rs], (n >> 1) & 1, s.abort)) {
        if (lane == 0) raise_abort(a, s.abort, tc::kSiteLoad);
        break;
      }
      const volatile int* rec = s.rec + rs * 16;
      const int u = rec[0], l = rec[1], g = rec[2], r = rec[3], nt = rec[8], N = rec[9], t0 = rec[10], m = rec[11];
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&s.recempty[rs]);  // this warp is done with the record
      if (u < 0) break;
      for (int t = 0; t < nt; ++t, ++T) {
        const uint32_t sl = (2 * T + 1) % kStages;
        if (T >= kAhead && !wait_warp(&s.done[(T - kAhead) % kDone], ((T - kAhead) / kDone) & 1, s.abort)) {
          if (lane == 0) raise_abort(a, s.abort, tc::kSiteLoad);
          ok = false;
          break;
        }
        if (kStale) {
          const int64_t row = (int64_t(l) * kv.Hkv + g) * kv.n_tot + t0;  // of the request's first key
          const int64_t z_row = int64_t(m) * kv.L * kv.Hkv * kv.n_tot + row + t * kKT;
          if (lane == 0) tc::mbar_arrive_expect_tx(&s.full[sl], kTileBytes);
          __syncwarp();
          if (lane < 2)
            tc::tma_load_2d(s.kv + sl * kTileBytes + lane * kHalfBytes, &vmap, &s.full[sl], lane * 64, int32_t(z_row));
        } else if ((t + 1) * kKT <= N) {
          load_tile<2>(a, &vmap, s.kv + sl * kTileBytes, &s.full[sl], l, g, r, t0, N, t * kKT, lane);
        } else {  // the copy arrives on a barrier of its own, and the tile is full once it has been cleared
          uint8_t* tile = s.kv + sl * kTileBytes;
          load_tile<2>(a, &vmap, tile, s.raw, l, g, r, t0, N, t * kKT, lane);
          if (!wait_warp(s.raw, n_raw & 1, s.abort)) {
            if (lane == 0) raise_abort(a, s.abort, tc::kSiteLoad);
            tc::mbar_wait(s.raw, n_raw & 1);  // the copy in flight
            ok = false;
            break;
          }
          ++n_raw;
          clear_rows<2>(tile, N - t * kKT, kKT, lane);
          if (lane == 0) tc::mbar_arrive(&s.full[sl]);
        }
      }
    }
    if (lane == 0) s.counters[1] = T;
  } else {
    // --------------------------- query tile and MMAs of one stream (warps 1, 3)
    // the whole warp walks the schedule on uniform values, one lane issues
    const int x = __shfl_sync(0xffffffffu, warp == kMmaWarp ? 0 : 1, 0);
    const uint32_t leader = lane == 0, frees = x == 0 ? leader : 0u;
    uint32_t T = 0, turn = 0, np = 0, nq = 0, cq = 0;  // tiles, turns, P tiles, query tiles loaded / consumed
    const uint32_t idesc_s = tc::idesc_bf16(kRows, kKT);
    const uint32_t idesc_o = tc::idesc_bf16(kRows, kMaxD, /*b_mn_major=*/true);
    const uint32_t kv_addr = tc::smem_u32(s.kv);
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
    const uint32_t s_col = tm + x * kSCols, o_col = tm + kOCol + x * kMaxD;
    const uint64_t dq = tc::desc_sw128(tc::smem_u32(s.q) + x * kTileBytes);
    bool ok = true;
    auto load_q = [&](const volatile int* rec) {
      if (rec[0] < 0 || rec[7 + x] == 0) return;
      if (lane == 0) {
        uint8_t* dst = s.q + x * kTileBytes;
        tc::mbar_arrive_expect_tx(&s.qfull[x], 256u * uint32_t(span * G));
        for (int hf = 0; hf < 2; ++hf)
          if (kStale)
            tc::tma_load_3d(dst + hf * kHalfBytes, &qmap, &s.qfull[x], hf * 64, rec[4] + (x ? rec[5] : 0),
                            rec[1] * Hq + rec[2] * G);
          else
            tc::tma_load_3d(dst + hf * kHalfBytes, &qmap, &s.qfull[x], hf * 64, rec[2] * G,
                            rec[1] * a.n_sel + rec[4] + (x ? rec[5] : 0));
      }
      __syncwarp();
      ++nq;
    };
    for (uint32_t n = 0;; ++n) {
      if (!(ok = wait_warp(&s.recfull[n & 1], (n >> 1) & 1, s.abort))) break;
      const volatile int* rec = s.rec + (n & 1) * 16;
      if (n == 0) load_q(rec);
      const int u = __shfl_sync(0xffffffffu, rec[0], 0), nt_x = __shfl_sync(0xffffffffu, rec[7 + x], 0),
                nt = __shfl_sync(0xffffffffu, rec[8], 0);
      __syncwarp();
      tc::mbar_arrive_if(leader, &s.recempty[n & 1]);
      if (u < 0) break;
      if (nt_x > 0) {
        if (!(ok = wait_warp(&s.qfull[x], cq & 1, s.abort))) break;
        ++cq;
      }
      for (int t = -1; t < nt; ++t, ++turn) {  // a turn: P(t) V(t), then S(t + 1)
        const uint32_t ev = 2 * (T - 1) + 1, slv = ev % kStages, ek = 2 * T, slk = ek % kStages;
        const bool more = t + 1 < nt;
        if (t >= 0 && !(ok = kStale ? wait_warp(&s.scaled[(T - 1) % kDone], ((T - 1) / kDone) & 1, s.abort)
                                    : wait_warp(&s.full[slv], (ev / kStages) & 1, s.abort)))
          break;
        if (more && !(ok = wait_warp(&s.full[slk], (ek / kStages) & 1, s.abort))) break;
        if (!more) {
          if (t < nt_x && !(ok = wait_warp(&s.pfull[x], np & 1, s.abort))) break;
          // every S of this stream's item has completed: load the next item's
          // query tile while the last P V and the output are under way
          if (!(ok = wait_warp(&s.recfull[(n + 1) & 1], ((n + 1) >> 1) & 1, s.abort))) break;
          load_q(s.rec + ((n + 1) & 1) * 16);
        }
        const uint64_t dk = tc::desc_sw128(kv_addr + slk * kTileBytes);
        const uint64_t dv = tc::desc_sw128_mn(kv_addr + slv * kTileBytes, kHalfBytes);
        if ((x == 1 || turn > 0) && !(ok = wait_warp(&s.turn[x], (x ? turn : turn - 1) & 1, s.abort))) break;
        if (t >= 0 && t < nt_x) {
          if (!(ok = wait_warp(&s.pfull[x], np & 1, s.abort))) break;
          ++np;
          tc::tc_fence_after();
#pragma unroll
          for (int kk = 0; kk < kKT / 16; ++kk)  // O += P(t) V(t)
            tc::mma_bf16_ts_if(leader, o_col, s_col + kPCol + kk * 8, dv + kk * (2048 >> 4), idesc_o, t > 0 || kk > 0);
          if (t + 1 == nt_x) tc::mma_commit_if(leader, &s.ofull[x]);
        }
        if (t + 1 < nt_x) {
#pragma unroll
          for (int kk = 0; kk < kMaxD / 16; ++kk) {  // S(t + 1) = Q K(t + 1)^T
            const uint32_t off = ((kk >> 2) * kHalfBytes + (kk & 3) * 32) >> 4;
            if (kk == kMaxD / 16 - kPassEarly) tc::mbar_arrive_if(leader, &s.turn[x ^ 1]);
            tc::mma_bf16_if(leader, s_col, dq + off, dk + off, idesc_s, kk > 0);
          }
          tc::mma_commit_if(leader, &s.sfull[x]);
        } else {
          tc::mbar_arrive_if(leader, &s.turn[x ^ 1]);
        }
        if (more) {
          // A's share of done[T]: S_A(T) and P_A(T - 1) V(T - 1) have completed, or
          // A's last MMAs where it has no rows left
          tc::mma_commit_if(frees, &s.done[T % kDone]);
          ++T;
        }
      }
      if (!ok) break;
    }
    if (!ok && lane == 0) raise_abort(a, s.abort, tc::kSiteMma);
    tc::mma_commit_if(leader, &s.mdone[x]);  // every MMA issued above has completed once this arrives
    tc::mbar_wait(&s.mdone[x], 0);
    if (cq < nq) tc::mbar_wait(&s.qfull[x], cq & 1);  // a copy in flight (only after an abort)
    __syncwarp();
  }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 208;" ::: "memory");
    // -------------------------------------------------------------- softmax
    const int x = (warp - kSoftWarp0) >> 2;              // query tile
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;                 // TMEM lane = query row of the tile
    const uint32_t tl = tmem + (uint32_t(quarter * 32) << 16);
    const uint32_t sb = tl + x * kSCols, ob = tl + kOCol + x * kMaxD;
    const uint32_t leader = lane == 0, releases = x == 1 && quarter == 0 && lane == 0;
    uint32_t Tv = 0;                                     // (kStale) the CTA's V tiles
    // (kStale) this query tile's share of scaling V tile t of the item: thread j
    // scales its half of row j by the key's deviation
    // `ahead`: this stream has not seen an S of the tile before. Then K(T - kAhead),
    // which had V(T)'s slot before it, may still be on its way, and the wait for the
    // slot's phase would take its unfinished phase for the one after it; so wait
    // first, as the loader does, until that tile is done.
    auto scale_v = [&](const float* scale, int t, int N, bool ahead) {
      const int j = t * kKT + row;
      const float sc = j < N ? scale[j] : 0.f;
      const uint32_t e = 2 * Tv + 1, sl = e % kStages;
      if (ahead && Tv >= uint32_t(kAhead) &&
          !wait_warp(&s.done[(Tv - kAhead) % kDone], ((Tv - kAhead) / kDone) & 1, s.abort)) {
        if (lane == 0) raise_abort(a, s.abort, tc::kSiteLoad);
        return false;
      }
      if (!wait_warp(&s.full[sl], (e / kStages) & 1, s.abort)) {
        if (lane == 0) raise_abort(a, s.abort, tc::kSiteLoad);
        return false;
      }
      uint8_t* tile = s.kv + sl * kTileBytes;
#pragma unroll
      for (int i8 = 0; i8 < 8; ++i8) {
        const int c = 8 * x + i8;
        uint4* p = reinterpret_cast<uint4*>(tile + (c >> 3) * kHalfBytes + tc::sw128_offset(row, c & 7));
        uint4 v = *p;
        __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&v);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 f = __bfloat1622float2(h[i]);
          h[i] = __floats2bfloat162_rn(sc * f.x, sc * f.y);
        }
        *p = v;
      }
      if (j >= N) {  // another request's draws, and 0 x Inf or NaN is not 0
#pragma unroll 1
        for (int c = 8 * x; c < 8 * (x + 1); ++c)
          *reinterpret_cast<uint4*>(tile + (c >> 3) * kHalfBytes + tc::sw128_offset(row, c & 7)) = make_uint4(0, 0, 0, 0);
      }
      tc::fence_proxy_async_smem();
      __syncwarp();
      tc::mbar_arrive_if(leader, &s.scaled[Tv % kDone]);
      ++Tv;
      return true;
    };
    uint32_t ns = 0, no = 0;                             // S tiles and O tiles read by this query tile
    bool ok = true;
    for (uint32_t n = 0; ok; ++n) {
      const int rs = n & 1;
      if (!wait_warp(&s.recfull[rs], (n >> 1) & 1, s.abort)) {
        if (lane == 0) raise_abort(a, s.abort, tc::kSiteLoad);
        break;
      }
      const volatile int* rec = s.rec + rs * 16;
      const int u = rec[0], l = rec[1], g = rec[2], cnt = rec[5 + x], nt = rec[7 + x], N = rec[9];
      const int i0 = rec[4] + (x ? rec[5] : 0), nt_all = rec[8], t0 = rec[10];
      bool live;
      int p_row, i_row = 0, h_row = 0;
      if (kStale) {  // a tile's rows are head major; every row sees every key of the request
        live = u >= 0 && row < span * G && row % span < cnt;
        p_row = N - 1;
        i_row = (rec[11] * kv.L + l) * kv.Hkv + g;
        h_row = rec[12];
      } else {
        // Rows without a position (past the tile or the box, or an index outside
        // the request) are computed unmasked and never written: a masked row
        // would send its warp down the masking path on every key tile.
        const bool row_ok = u >= 0 && row < cnt * G;
        i_row = i0 + (row_ok ? row / G : 0);
        h_row = g * G + (row_ok ? row % G : 0);
        p_row = row_ok ? s.pos[(rs * 2 + x) * kRows + row / G] : -1;
        live = p_row >= 0 && p_row < N;
        if (!live) p_row = INT_MAX;
      }
      __syncwarp();
      tc::mbar_arrive_if(leader, &s.recempty[rs]);
      if (u < 0) break;

      const float* key_scale = nullptr;
      if (kStale) {
        key_scale = a.key_scale + (int64_t(l) * kv.Hkv + g) * kv.n_tot + t0;
        // V(0), or every V tile when no rows of the item are in this query tile
        for (int t = 0; t < (nt == 0 ? nt_all : 1) && ok; ++t) ok = scale_v(key_scale, t, N, true);
      }
      float m_ref = -INFINITY, lsum = 0.f;  // running max (scaled, log2 units) and row sum
      for (int t = 0; t < nt && ok; ++t, ++ns) {
        // the tcgen05.ld below is warp-collective: the whole warp goes on or stops
        if (!wait_warp(&s.sfull[x], ns & 1, s.abort)) {
          if (lane == 0) raise_abort(a, s.abort, tc::kSiteMma);
          ok = false;
          break;
        }
        tc::tc_fence_after();
        float sv[kKT];
        tc::tmem_ld128(sb, sv);
        const int j0 = t * kKT;
        if (j0 + kKT - 1 > p_row) {  // part of this tile is past this row's position
#pragma unroll
          for (int i = 0; i < kKT; ++i)
            if (j0 + i > p_row) sv[i] = -INFINITY;
        }
        float tm[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int i = 0; i < kKT / 2; ++i) tm[i & 3] = tc::fmax3(tm[i & 3], sv[2 * i], sv[2 * i + 1]);
        const float tmax = fmaxf(fmaxf(tm[0], tm[1]), fmaxf(tm[2], tm[3])) * a.scale_log2;
        const bool need = tmax > m_ref + kRescaleLog2 || (m_ref == -INFINITY && tmax != -INFINITY);
        const float alpha = need ? tc::ex2(m_ref - tmax) : 1.f;  // 0 when m_ref is -inf
        if (need) {
          lsum *= alpha;
          m_ref = tmax;
        }
        if (__any_sync(0xffffffffu, need) && t > 0) {
          // S(t) is ready, so P(t-1) V(t-1) has completed; P(t) V(t) waits for
          // this warp's arrival below
          for (int c = 0; c < kMaxD; c += 16) {
            float o[16];
            tc::tmem_ld16(ob + c, o);
            uint32_t w[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) w[i] = __float_as_uint(o[i] * alpha);
            tc::tmem_st16_nowait(ob + c, w);
          }
        }
        // P = 2^(S scale - m) in bf16 pairs over S, which this warp has read (one
        // packed FMA per pair for scale and bias, packed adds for the sum). A row
        // with no visible key yet (m = -inf) uses bias 0: its logits are all
        // -inf and its P is 0.
        const float2 sc2 = make_float2(a.scale_log2, a.scale_log2);
        const float2 nb2 = m_ref == -INFINITY ? make_float2(0.f, 0.f) : make_float2(-m_ref, -m_ref);
        float2 ls2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
        for (int c = 0; c < kKT / 32; ++c) {
          uint32_t pw[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const float2 y = tc::ffma2(make_float2(sv[32 * c + 2 * i], sv[32 * c + 2 * i + 1]), sc2, nb2);
            const float2 pp = make_float2(tc::ex2(y.x), tc::ex2(y.y));
            ls2[i & 1] = tc::fadd2(ls2[i & 1], pp);
            const __nv_bfloat162 pr = __floats2bfloat162_rn(pp.x, pp.y);
            pw[i] = *reinterpret_cast<const uint32_t*>(&pr);
          }
          tc::tmem_st16_nowait(sb + kPCol + 16 * c, pw);
        }
        lsum += (ls2[0].x + ls2[0].y) + (ls2[1].x + ls2[1].y);
        tc::tmem_wait_st();
        tc::tc_fence_before();
        __syncwarp();
        tc::mbar_arrive_if(leader, &s.pfull[x]);
        // B's share of done: S_B(t) has completed and, in warp 3's issue order, so has
        // P_B(t-1) V(t-1). Warp 1 commits A's, which this says nothing of: its last
        // MMAs of a turn may be issued after the turn has passed to B.
        tc::mbar_arrive_if(releases, &s.done[ns % kDone]);
        if (kStale && t + 1 < nt && !scale_v(key_scale, t + 1, N, false)) {
          ok = false;
          break;
        }
      }
      double* const part = kStale ? a.part + ((int64_t(i_row) * a.n_blocks + h_row) * 2 + x) * 4 + quarter : nullptr;
      if (kStale && nt == 0 && lane == 0) *part = 0.0;  // no rows in this tile
      if (nt == 0 || !ok) continue;
      if (!wait_warp(&s.ofull[x], no & 1, s.abort)) {
        if (lane == 0) raise_abort(a, s.abort, tc::kSiteFinal);
        ok = false;
        break;
      }
      ++no;
      tc::tc_fence_after();
      // The row of O as bf16. Each lane writes its own row, so a warp's store
      // covers 32 rows: 32-byte stores (whole sectors) when the buffer allows
      // them. The next item's P(0) V(0), which overwrites O, waits for a P this
      // warp writes after these loads.
      const float inv = lsum > 0.f ? 1.f / lsum : 0.f;
      if (kStale) {  // ||O / rowsum||^2 (in the cache's type) over the warp's rows, in a fixed order
        float ss[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < kMaxD; c += 64) {
          float o[64];
          tc::tmem_ld64(ob + c, o);
#pragma unroll
          for (int i = 0; i < 64; ++i) {
            const float x1 = __bfloat162float(__float2bfloat16_rn(o[i] * inv));
            ss[i & 3] = fmaf(x1, x1, ss[i & 3]);
          }
        }
        double row_ss = live ? double((ss[0] + ss[1]) + (ss[2] + ss[3])) : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) row_ss += __shfl_xor_sync(0xffffffffu, row_ss, o);
        if (lane == 0) *part = row_ss;
        tc::tc_fence_before();
        continue;
      }
      __nv_bfloat16* dst = a.out + ((int64_t(l) * a.n_sel + i_row) * Hq + h_row) * kMaxD;
#pragma unroll
      for (int c = 0; c < kMaxD; c += 64) {
        float o[64];
        tc::tmem_ld64(ob + c, o);
        if (live) {
          uint32_t w[32];
#pragma unroll
          for (int k2 = 0; k2 < 32; ++k2) {
            __nv_bfloat162 pr = __floats2bfloat162_rn(o[2 * k2] * inv, o[2 * k2 + 1] * inv);
            w[k2] = *reinterpret_cast<uint32_t*>(&pr);
          }
          if (a.out32) {
#pragma unroll
            for (int u8 = 0; u8 < 4; ++u8)
              asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + c + u8 * 16),
                           "r"(w[8 * u8]), "r"(w[8 * u8 + 1]), "r"(w[8 * u8 + 2]), "r"(w[8 * u8 + 3]),
                           "r"(w[8 * u8 + 4]), "r"(w[8 * u8 + 5]), "r"(w[8 * u8 + 6]), "r"(w[8 * u8 + 7])
                           : "memory");
          } else {
#pragma unroll
            for (int u4 = 0; u4 < 8; ++u4)
              *reinterpret_cast<uint4*>(dst + c + u4 * 8) = make_uint4(w[4 * u4], w[4 * u4 + 1], w[4 * u4 + 2], w[4 * u4 + 3]);
          }
        }
      }
      tc::tc_fence_before();
    }
  }
  __syncthreads();
  if (tid == 0) {  // wait for each ring slot's last copy (all have landed unless a role gave up)
    const int nk = int(s.counters[0]), nv = int(s.counters[1]);
    for (int sl = 0; sl < kStages; ++sl) {
      int e = max(2 * nk - 2, 2 * nv - 1);
      while (e >= 0 && (e % kStages != sl || e / 2 >= ((e & 1) ? nv : nk))) --e;
      if (e >= 0) tc::mbar_wait(&s.full[sl], (e / kStages) & 1);
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) tc::tmem_dealloc(tmem, kTmemCols);
}

// ------------------------------------------------ one query tile per item
constexpr int kSoftThreads = 256;
constexpr int kOneVWarp = 10, kPvWarp = 11;      // after the item/K, MMA and eight softmax warps
constexpr int kKStages = 2, kVStages = 2, kQBufs = 2;
constexpr uint32_t kOneTileBytes = 2 * kHalfBytes;
constexpr uint32_t kQBytes = 2 * kHalfBytes;
constexpr int kRecInts = 9;                      // decoded item record (see OneSmem::rec)
constexpr uint32_t kOneSmem = 1024 + kQBufs * kQBytes + (kKStages + kVStages) * kOneTileBytes + 256 +
                              2 * 2 * 128 * 4 + 2 * 128 * 4 + kQBufs * (kRecInts + kRows) * 4;
constexpr int kSBufs = 3;                        // S runs up to two key tiles ahead of the softmax
constexpr uint32_t kOneOCol = kSBufs * kSCols;

struct OneSmem {
  uint8_t* q;        // [kQBufs][2 halves][128 rows][128 B]
  uint8_t* k;        // [kKStages][2 halves][128 keys][128 B]
  uint8_t* v;        // [kVStages][2 halves][128 keys][128 B]
  uint64_t *kfull, *kempty;   // [kKStages]
  uint64_t *vfull, *vempty;   // [kVStages]
  uint64_t *sfull, *pfull;    // [kSBufs] per S buffer
  uint64_t *pvdone;           // [kSBufs] per S buffer: the P.V that read its P has completed
  uint64_t *qfull, *qempty;   // [kQBufs] query tile (and item index) of one item
  uint64_t *ofull, *oempty;   // once per item: O complete / O read out
  uint64_t *mdone;            // [2] per MMA thread: all its MMAs completed
  uint32_t* tmem_slot;
  volatile int* abort;
  uint32_t* counters;  // [0] K loads, [1] V loads, [2] K consumed, [3] V consumed
  float* xmax;         // [2 tile parities][2 halves][128 rows] half-row maxima
  float* xsum;         // [2 halves][128 rows] half-row sums at the end
  // per query buffer, written by the loader with the query tile: the decoded
  // item {u (-1: no more work), l, g, r, i0, cnt, key tiles, N_r, t0} and the
  // positions of its selected rows, so the other roles read no global memory
  // between items
  volatile int* rec;   // [kQBufs][kRecInts]
  volatile int* pos;   // [kQBufs][kRows]
};

__device__ __forceinline__ OneSmem carve_one(uint8_t* raw) {
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(raw) + 1023) & ~uintptr_t(1023));
  OneSmem s;
  s.q = base;
  s.k = s.q + kQBufs * kQBytes;
  s.v = s.k + kKStages * kOneTileBytes;
  uint64_t* bar = reinterpret_cast<uint64_t*>(s.v + kVStages * kOneTileBytes);
  s.kfull = bar;
  s.kempty = s.kfull + kKStages;
  s.vfull = s.kempty + kKStages;
  s.vempty = s.vfull + kVStages;
  s.sfull = s.vempty + kVStages;
  s.pfull = s.sfull + kSBufs;
  s.pvdone = s.pfull + kSBufs;
  s.qfull = s.pvdone + kSBufs;
  s.qempty = s.qfull + kQBufs;
  s.ofull = s.qempty + kQBufs;
  s.oempty = s.ofull + 1;
  s.mdone = s.oempty + 1;
  s.tmem_slot = reinterpret_cast<uint32_t*>(s.mdone + 2);
  s.abort = reinterpret_cast<volatile int*>(s.tmem_slot + 1);
  s.counters = reinterpret_cast<uint32_t*>(s.tmem_slot + 2);
  s.xmax = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(bar) + 256);
  s.xsum = s.xmax + 2 * 2 * 128;
  s.rec = reinterpret_cast<volatile int*>(s.xsum + 2 * 128);
  s.pos = s.rec + kQBufs * kRecInts;
  return s;
}

// Output rows with values that are not finite although the row's maximum and sum are:
// V holds such a value, in a key of the row or in a later one that shares a key tile
// with the item's rows, where P is 0 but 0 x Inf or NaN is NaN. A warp computes the
// rows of `lanes` again, key by key over the keys they see: columns col0 ... of each.
// The cost is about 100 ns a key and row (64 dims; 112 at 96), so the 32 rows of a warp
// take half a second at kRedoKeys keys: rows that see more, which would keep the other
// roles waiting past their limit, stay as they are.
constexpr int kRedoKeys = 1 << 17;
template <int kCols>
__device__ __noinline__ void redo_rows(const RefArgs& a, uint32_t lanes, int l, int g, int r, int t0, int p_row,
                                       float m_ref, float inv, int64_t row_off, int col0, int lane) {
  const KvDev& kv = a.kv;
  const __nv_bfloat16* kb = static_cast<const __nv_bfloat16*>(kv.k);
  const __nv_bfloat16* vb = static_cast<const __nv_bfloat16*>(kv.v);
  __syncwarp();  // the rows' first values have been written
  for (; lanes; lanes &= lanes - 1) {
    const int src = __ffs(lanes) - 1;
    const int p = __shfl_sync(0xffffffffu, p_row, src);
    const float m = __shfl_sync(0xffffffffu, m_ref, src), w0 = __shfl_sync(0xffffffffu, inv, src);
    const int64_t off = __shfl_sync(0xffffffffu, static_cast<long long>(row_off), src);
    if (p >= kRedoKeys) continue;
    float acc[kCols / 32] = {};
    for (int j0 = 0; j0 <= p; j0 += 32) {
      const int j = j0 + lane;
      int64_t k_off = 0;
      float w = 0.f;
      if (j <= p) {
        k_off = kv.row(l, g, r, int64_t(t0) + j, j);
        float dot = 0.f;
#pragma unroll 4
        for (int c = 0; c < kv.d; c += 8) {
          const uint4 qv = *reinterpret_cast<const uint4*>(a.q + off + c);
          const uint4 kk = *reinterpret_cast<const uint4*>(kb + k_off + c);
          const __nv_bfloat162* q2 = reinterpret_cast<const __nv_bfloat162*>(&qv);
          const __nv_bfloat162* k2 = reinterpret_cast<const __nv_bfloat162*>(&kk);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float2 x = __bfloat1622float2(q2[i]), y = __bfloat1622float2(k2[i]);
            dot = fmaf(x.y, y.y, fmaf(x.x, y.x, dot));
          }
        }
        w = exp2f(fmaf(dot, a.scale_log2, -m)) * w0;
      }
      const int n = min(32, p - j0 + 1);
#pragma unroll 8
      for (int jj = 0; jj < n; ++jj) {
        const float wj = __shfl_sync(0xffffffffu, w, jj);
        const int64_t v_off = __shfl_sync(0xffffffffu, static_cast<long long>(k_off), jj);
#pragma unroll
        for (int c = 0; c < kCols / 32; ++c) {
          const int e = col0 + 32 * c + lane;
          if (e < kv.d) acc[c] = fmaf(wj, __bfloat162float(vb[v_off + e]), acc[c]);
        }
      }
    }
#pragma unroll
    for (int c = 0; c < kCols / 32; ++c) {
      const int e = col0 + 32 * c + lane;
      if (e < kv.d) a.out[off + e] = __float2bfloat16_rn(acc[c]);
    }
  }
}

// Agreement of the 256 softmax threads (named barrier 1 with an AND
// reduction): every thread arrives, so all of them take the same branch.
__device__ __forceinline__ bool softmax_all(bool pred) {
  uint32_t out;
  asm volatile(
      "{\n.reg .pred pi, po;\nsetp.ne.u32 pi, %1, 0;\nbar.red.and.pred po, 1, %2, pi;\nselp.u32 %0, 1, 0, po;\n}\n"
      : "=r"(out)
      : "r"(uint32_t(pred)), "n"(kSoftThreads)
      : "memory");
  return out != 0;
}

// kHalves 64-dim halves of a row (one 128-byte swizzled row each; a smaller head_dim is
// padded with zeros by the copies). kSplit: P goes to the tensor cores as two bf16
// tiles (value and rounding error), which keeps it as precise as fp32 weights for a
// bf16 result.
template <int kHalves, bool kSplit>
__global__ void __launch_bounds__(kThreads, 1)
    one_refresh_tc_kernel(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap,
                      const __grid_constant__ CUtensorMap qmap, const __grid_constant__ RefArgs a) {
  extern __shared__ uint8_t smem_raw[];
  const OneSmem s = carve_one(smem_raw);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const KvDev& kv = a.kv;
  constexpr int kDP = 64 * kHalves, kOW = kDP / 2;  // kOW: columns of O of a softmax thread
  const int G = kv.G, Hq = kv.Hq;
  const int d = kHalves == 2 && !kSplit ? kMaxD : kv.d;
  const int qrows = a.rows_per_tile * G;          // rows the query box fills

  if (tid == 0) {
    for (int i = 0; i < kKStages; ++i) {
      tc::mbar_init(&s.kfull[i], 1);
      tc::mbar_init(&s.kempty[i], 1);
    }
    for (int i = 0; i < kVStages; ++i) {
      tc::mbar_init(&s.vfull[i], 1);
      tc::mbar_init(&s.vempty[i], 1);
    }
    for (int i = 0; i < kSBufs; ++i) {
      tc::mbar_init(&s.sfull[i], 1);
      // per buffer, so the softmax can never be two phases ahead of the MMA's
      // wait: P(t+3) needs S(t+3), issued only after P(t) V(t) has completed
      tc::mbar_init(&s.pfull[i], kSoftThreads);
      tc::mbar_init(&s.pvdone[i], 1);
    }
    for (int i = 0; i < kQBufs; ++i) {
      tc::mbar_init(&s.qfull[i], 1);   // the loader's expect-tx (or plain arrive at the end)
      // the S thread's commit + the P.V thread's, softmax's and V warp's reads of the item
      tc::mbar_init(&s.qempty[i], 4);
    }
    tc::mbar_init(s.ofull, 1);
    tc::mbar_init(s.oempty, kSoftThreads);
    tc::mbar_init(&s.mdone[0], 1);
    tc::mbar_init(&s.mdone[1], 1);
    *s.abort = 0;
    for (int i = 0; i < 4; ++i) s.counters[i] = 0;
    tc::fence_barrier_init();
    tc::prefetch_tensormap(&kmap);
    tc::prefetch_tensormap(&vmap);
    tc::prefetch_tensormap(&qmap);
  }
  if (warp == 1) tc::tmem_alloc(s.tmem_slot, kTmemCols);
  for (uint32_t i = qrows * 128 + tid * 16; i < kHalfBytes; i += kThreads * 16)  // rows the boxes leave empty
    for (int h = 0; h < 2 * kQBufs; ++h) *reinterpret_cast<uint4*>(s.q + h * kHalfBytes + i) = make_uint4(0, 0, 0, 0);
  tc::fence_proxy_async_smem();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = *s.tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------- loads (warp 0)
    uint32_t nk = 0, T = 0;
    bool ok = true;
    for (uint32_t n = 0; ok; ++n) {
      int u = 0;
      if (lane == 0) {
        u = n == 0 ? int(blockIdx.x)
                   : a.next_item ? int(gridDim.x) + atomicAdd(a.next_item, 1) : int(blockIdx.x + n * gridDim.x);
        if (u >= a.n_items) u = -1;
      }
      u = __shfl_sync(0xffffffffu, u, 0);
      const Item it = decode_item<false>(a, u < 0 ? 0 : u);
      const int t0 = a.b.tok_off[it.r], N = a.b.tok_off[it.r + 1] - t0;
      int nt = 0;
      if (u >= 0 && it.cnt > 0) {
        const int p_max = min(a.idx[it.i0 + it.cnt - 1], N - 1);
        nt = p_max < 0 ? 0 : p_max / kKT + 1;
      }
      int my_pos[kRows / 32];  // positions of the item's rows, loaded before the buffer is free
#pragma unroll
      for (int k = 0; k < kRows / 32; ++k) {
        const int i = lane + 32 * k;
        my_pos[k] = (u >= 0 && i < it.cnt) ? a.idx[it.i0 + i] : -1;
      }
      const int qs = n & 1;
      if (!__all_sync(0xffffffffu, wait_or_abort(&s.qempty[qs], ((n >> 1) & 1) ^ 1, s.abort))) {
        if (lane == 0) raise_abort(a, s.abort, tc::kSiteLoad);
        break;
      }
#pragma unroll
      for (int k = 0; k < kRows / 32; ++k) s.pos[qs * kRows + lane + 32 * k] = my_pos[k];
      if (lane == 0) {
        volatile int* rec = s.rec + qs * kRecInts;
        rec[0] = u;
        rec[1] = it.l;
        rec[2] = it.g;
        rec[3] = it.r;
        rec[4] = it.i0;
        rec[5] = it.cnt;
        rec[6] = nt;
        rec[7] = N;
        rec[8] = t0;
      }
      __threadfence_block();
      __syncwarp();  // the lanes' positions are ordered before lane 0's release below
      if (lane == 0) {
        if (u < 0) {
          tc::mbar_arrive(&s.qfull[qs]);  // no more work: the others stop at this buffer
        } else {
          tc::mbar_arrive_expect_tx(&s.qfull[qs], uint32_t(kHalves) * 128u * uint32_t(qrows));
          for (int hf = 0; hf < kHalves; ++hf)
            tc::tma_load_3d(s.q + qs * kQBytes + hf * kHalfBytes, &qmap, &s.qfull[qs], hf * 64,
                            it.g * G, it.l * a.n_sel + it.i0);
        }
      }
      if (u < 0) break;
      for (int t = 0; t < nt; ++t, ++T) {
        const int sk = T % kKStages;
        if (!__all_sync(0xffffffffu, wait_or_abort(&s.kempty[sk], ((T / kKStages) & 1) ^ 1, s.abort))) {
          if (lane == 0) raise_abort(a, s.abort, tc::kSiteLoad);
          ok = false;
          break;
        }
        load_tile<kHalves>(a, &kmap, s.k + sk * kOneTileBytes, &s.kfull[sk], it.l, it.g, it.r, t0, N, t * kKT, lane);
        ++nk;
      }
    }
    if (lane == 0) s.counters[0] = nk;
  } else if (warp == kOneVWarp) {
    // --------------------------------------------------- V loads (warp 10)
    // on a warp of their own: a V stage frees only once its P.V has
    // completed, and waiting for it must not hold back the K tiles and the
    // next item's query tile
    uint32_t nv = 0, T = 0;
    for (uint32_t n = 0;; ++n) {
      const int qs = n & 1;
      if (!__all_sync(0xffffffffu, wait_or_abort(&s.qfull[qs], (n >> 1) & 1, s.abort))) {
        if (lane == 0) raise_abort(a, s.abort, tc::kSiteLoad);
        break;
      }
      const volatile int* rec = s.rec + qs * kRecInts;
      const int u = rec[0], l = rec[1], g = rec[2], r = rec[3], nt = rec[6], N = rec[7], t0 = rec[8];
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&s.qempty[qs]);  // this warp is done with the record
      if (u < 0) break;
      bool ok = true;
      for (int t = 0; t < nt; ++t, ++T) {
        const int sv = T % kVStages;
        if (!__all_sync(0xffffffffu, wait_or_abort(&s.vempty[sv], ((T / kVStages) & 1) ^ 1, s.abort))) {
          if (lane == 0) raise_abort(a, s.abort, tc::kSiteLoad);
          ok = false;
          break;
        }
        load_tile<kHalves>(a, &vmap, s.v + sv * kOneTileBytes, &s.vfull[sv], l, g, r, t0, N, t * kKT, lane);
        ++nv;
      }
      if (!ok) break;
    }
    if (lane == 0) s.counters[1] = nv;
  } else if (warp == 1) {
    // ---------------------------------------------------------- MMA: S = Q K^T
    // S(t) goes to buffer t % kSBufs once P(t-3) V(t-3), which read that
    // buffer's P, has completed (possibly of an earlier item); so this warp
    // runs up to two tiles ahead of the P.V warp
    const uint32_t leader = lane == 0;
    uint32_t T = 0;
    bool ok = true;
    const uint32_t idesc_s = tc::idesc_bf16(kRows, kKT);
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
    for (uint32_t n = 0; ok; ++n) {
      const int qs = n & 1;
      if (!(ok = wait_warp(&s.qfull[qs], (n >> 1) & 1, s.abort))) break;
      const int u = __shfl_sync(0xffffffffu, s.rec[qs * kRecInts], 0);
      const int nt = __shfl_sync(0xffffffffu, s.rec[qs * kRecInts + 6], 0);
      if (u < 0) break;
      const uint64_t dq = tc::desc_sw128(tc::smem_u32(s.q + qs * kQBytes));
      for (int t = 0; t < nt; ++t, ++T) {
        const int b = T % kSBufs, sk = T % kKStages;
        if (T >= uint32_t(kSBufs) && !(ok = wait_warp(&s.pvdone[b], ((T / kSBufs) - 1) & 1, s.abort))) break;
        if (!(ok = wait_warp(&s.kfull[sk], (T / kKStages) & 1, s.abort))) break;
        if (leader) s.counters[2] = T + 1;
        __syncwarp();
        tc::tc_fence_after();
        const uint64_t dk = tc::desc_sw128(tc::smem_u32(s.k + sk * kOneTileBytes));
        const int ksteps = kSplit ? (d + 15) / 16 : kDP / 16;
#pragma unroll
        for (int kk = 0; kk < kDP / 16; ++kk) {
          const uint32_t off = ((kk >> 2) * kHalfBytes + (kk & 3) * 32) >> 4;
          if (kk < ksteps) tc::mma_bf16_if(leader, tm + b * kSCols, dq + off, dk + off, idesc_s, kk > 0);
        }
        tc::mma_commit_if(leader, &s.sfull[b]);
        tc::mma_commit_if(leader, &s.kempty[sk]);
      }
      if (ok) tc::mma_commit_if(leader, &s.qempty[qs]);  // every S of this item is issued
    }
    if (!ok && leader) raise_abort(a, s.abort, tc::kSiteMma);
    tc::mma_commit_if(leader, &s.mdone[0]);  // every MMA issued above has completed once this arrives
    tc::mbar_wait(&s.mdone[0], 0);
    __syncwarp();
  } else if (warp == kPvWarp) {
    // -------------------------------------------------------- MMA: O += P V
    const uint32_t leader = lane == 0;
    uint32_t T = 0;
    bool ok = true;
    const uint32_t idesc_o = tc::idesc_bf16(kRows, kDP, /*b_mn_major=*/true);
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
    for (uint32_t n = 0; ok; ++n) {
      const int qs = n & 1;
      if (!(ok = wait_warp(&s.qfull[qs], (n >> 1) & 1, s.abort))) break;
      const int u = __shfl_sync(0xffffffffu, s.rec[qs * kRecInts], 0);
      const int nt = __shfl_sync(0xffffffffu, s.rec[qs * kRecInts + 6], 0);
      const int N = __shfl_sync(0xffffffffu, s.rec[qs * kRecInts + 7], 0);
      tc::mbar_arrive_if(leader, &s.qempty[qs]);  // this warp is done with the record
      if (u < 0) break;
      // A last tile that ends past the request's keys is taken after the loop: a V stage
      // is waited for at every tile, and a test for it in the loop took 24 layers of
      // 2 916 tokens, 64 dims from 86.2 to 88.1 us.
      const int whole = min(nt, N / kKT);
      for (int t = 0; t < whole; ++t, ++T) {
        const int b = T % kSBufs, sv = T % kVStages;
        if (!(ok = wait_warp(&s.vfull[sv], (T / kVStages) & 1, s.abort))) break;
        if (leader) s.counters[3] = T + 1;
        __syncwarp();
        if (!(ok = wait_warp(&s.pfull[b], (T / kSBufs) & 1, s.abort))) break;
        // O of the previous item must have been read out before P(0) V(0) overwrites it
        if (t == 0 && n > 0 && !(ok = wait_warp(s.oempty, (n - 1) & 1, s.abort))) break;
        tc::tc_fence_after();
        const uint64_t dv = tc::desc_sw128_mn(tc::smem_u32(s.v + sv * kOneTileBytes), kHalfBytes);
        const uint32_t pb = tm + b * kSCols;
#pragma unroll
        for (int kk = 0; kk < kKT / 16; ++kk)  // O += P(t) V(t)
          tc::mma_bf16_ts_if(leader, tm + kOneOCol, pb + kPCol + kk * 8, dv + kk * (2048 >> 4), idesc_o, t > 0 || kk > 0);
        if (kSplit) {
#pragma unroll
          for (int kk = 0; kk < kKT / 16; ++kk)
            tc::mma_bf16_ts_if(leader, tm + kOneOCol, pb + kPLoCol + kk * 8, dv + kk * (2048 >> 4), idesc_o, true);
        }
        tc::mma_commit_if(leader, &s.pvdone[b]);
        tc::mma_commit_if(leader, &s.vempty[sv]);
      }
      if (ok && whole < nt) {  // 16 keys an MMA, as many as hold the tile's keys; P of those left out is 0
        const int b = T % kSBufs, sv = T % kVStages, keys = N - whole * kKT;
        if (!(ok = wait_warp(&s.vfull[sv], (T / kVStages) & 1, s.abort))) break;
        if (leader) s.counters[3] = T + 1;
        __syncwarp();
        clear_rows<kHalves>(s.v + sv * kOneTileBytes, keys, (keys + 15) & ~15, lane);
        if (!(ok = wait_warp(&s.pfull[b], (T / kSBufs) & 1, s.abort))) break;
        if (whole == 0 && n > 0 && !(ok = wait_warp(s.oempty, (n - 1) & 1, s.abort))) break;
        tc::tc_fence_after();
        const uint64_t dv = tc::desc_sw128_mn(tc::smem_u32(s.v + sv * kOneTileBytes), kHalfBytes);
        const uint32_t pb = tm + b * kSCols;
#pragma unroll 1
        for (int kk = 0; kk * 16 < keys; ++kk)
          tc::mma_bf16_ts_if(leader, tm + kOneOCol, pb + kPCol + kk * 8, dv + kk * (2048 >> 4), idesc_o,
                             whole > 0 || kk > 0);
        if (kSplit) {
#pragma unroll 1
          for (int kk = 0; kk * 16 < keys; ++kk)
            tc::mma_bf16_ts_if(leader, tm + kOneOCol, pb + kPLoCol + kk * 8, dv + kk * (2048 >> 4), idesc_o, true);
        }
        tc::mma_commit_if(leader, &s.pvdone[b]);
        tc::mma_commit_if(leader, &s.vempty[sv]);
        ++T;
      }
      if (ok) tc::mma_commit_if(leader, s.ofull);  // O of this item is complete once this arrives
    }
    if (!ok && leader) raise_abort(a, s.abort, tc::kSiteMma);
    tc::mma_commit_if(leader, &s.mdone[1]);
    tc::mbar_wait(&s.mdone[1], 0);
    __syncwarp();
  } else if (warp >= 2 && warp < kOneVWarp) {
    // -------------------------------------------------------------- softmax
    const int et = tid - 64;                             // 0..255
    const int hh = et >> 7;                              // half of the key tile / of O
    const int quarter = warp & 3;
    const int row = quarter * 32 + lane;                 // TMEM lane = query row of the tile
    const uint32_t lane_base = uint32_t(quarter * 32) << 16;
    const uint32_t tl = tmem + lane_base;
    bool ok = true;
    uint32_t T = 0;
    for (uint32_t n = 0;; ++n) {
      const int qs = n & 1;
      // all 256 threads agree to go on, so the named barriers below stay uniform
      const bool got = wait_or_abort(&s.qfull[qs], (n >> 1) & 1, s.abort);
      if (!softmax_all(ok && got)) {
        if (ok) raise_abort(a, s.abort, tc::kSiteLoad);
        break;
      }
      const volatile int* rec = s.rec + qs * kRecInts;
      const int u = rec[0];
      Item it;
      it.l = rec[1];
      it.g = rec[2];
      it.r = rec[3];
      it.i0 = rec[4];
      it.cnt = rec[5];
      const int nt = rec[6], N = rec[7], rec_t0 = rec[8];
      const bool row_ok = u >= 0 && row < it.cnt * G;
      const int i_row = it.i0 + (row_ok ? row / G : 0);
      const int h_row = it.g * G + (row_ok ? row % G : 0);
      int p_row = row_ok ? s.pos[qs * kRows + row / G] : -1;  // rows past the item (or the box) are fully masked
      const bool live = p_row >= 0 && p_row < N;
      if (!live) p_row = 0x7fffffff;
      asm volatile("bar.sync 1, %0;" ::"n"(kSoftThreads) : "memory");  // everyone has read the record
      if (et == 0) tc::mbar_arrive(&s.qempty[qs]);
      if (u < 0) break;

      float m_ref = -INFINITY, lsum = 0.f;  // running max (scaled, log2 units, same in both halves) and half-row sum
      for (int t = 0; t < nt; ++t) {
        const uint32_t Tc = T + t;
        const uint32_t sbuf = Tc % kSBufs;
        const uint32_t sb = tl + sbuf * kSCols;
        // the tcgen05.ld below is warp-collective: the whole warp goes on or stops
        const bool gs = __all_sync(0xffffffffu, ok && (tc::mbar_probe(&s.sfull[sbuf], (Tc / kSBufs) & 1) ||
                                                       wait_or_abort(&s.sfull[sbuf], (Tc / kSBufs) & 1, s.abort)));
        if (!gs) {
          if (ok) raise_abort(a, s.abort, tc::kSiteMma);
          ok = false;
        }
        float sv[64];
        float hmax = -INFINITY;
        const int j0 = t * kKT + hh * 64;
        if (gs) {
          tc::tc_fence_after();
          tc::tmem_ld64(sb + hh * 64, sv);
          if (j0 + 63 > p_row) {  // part of this half is past this row's position
#pragma unroll
            for (int i = 0; i < 64; ++i)
              if (j0 + i > p_row) sv[i] = -INFINITY;
          }
          float tm[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
          for (int i = 0; i < 32; ++i) tm[i & 3] = tc::fmax3(tm[i & 3], sv[2 * i], sv[2 * i + 1]);
          hmax = fmaxf(fmaxf(tm[0], tm[1]), fmaxf(tm[2], tm[3]));
        }
        // exchange the half-row maxima (buffers alternate with the tile, so a
        // half that runs ahead never overwrites a value its partner still reads)
        float* xm = s.xmax + (Tc & 1) * 256;
        xm[hh * 128 + row] = hmax;
        asm volatile("bar.sync 1, %0;" ::"n"(kSoftThreads) : "memory");
        if (!ok) continue;
        const float tmax = fmaxf(hmax, xm[(hh ^ 1) * 128 + row]) * a.scale_log2;
        const bool need = tmax > m_ref + kRescaleLog2 || (m_ref == -INFINITY && tmax != -INFINITY);
        const float alpha = need ? tc::ex2(m_ref - tmax) : 1.f;  // 0 when m_ref is -inf
        if (need) {
          lsum *= alpha;
          m_ref = tmax;
        }
        // this half of P = 2^(S scale - m) in bf16 pairs over the upper half of S
        // (one packed FMA per pair for scale and bias, packed adds for the sum).
        // A row with no visible key yet (m = -inf) uses bias 0: its logits are
        // all -inf and its P is 0. Both halves of S have been read (the barrier
        // above), so either thread may write over the other's half.
        const float2 sc2 = make_float2(a.scale_log2, a.scale_log2);
        const float2 nb2 = m_ref == -INFINITY ? make_float2(0.f, 0.f) : make_float2(-m_ref, -m_ref);
        float2 ls2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        {
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            uint32_t pw[16], lo[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float2 y = tc::ffma2(make_float2(sv[32 * c + 2 * i], sv[32 * c + 2 * i + 1]), sc2, nb2);
              const float2 pp = make_float2(tc::ex2(y.x), tc::ex2(y.y));
              ls2[i & 1] = tc::fadd2(ls2[i & 1], pp);
              __nv_bfloat162 pr = __floats2bfloat162_rn(pp.x, pp.y);
              pw[i] = *reinterpret_cast<uint32_t*>(&pr);
              if (kSplit) {
                const float2 hi = __bfloat1622float2(pr);
                pr = __floats2bfloat162_rn(pp.x - hi.x, pp.y - hi.y);
                lo[i] = *reinterpret_cast<uint32_t*>(&pr);
              }
            }
            tc::tmem_st16_nowait(sb + kPCol + hh * 32 + 16 * c, pw);
            if (kSplit) tc::tmem_st16_nowait(sb + kPLoCol + hh * 32 + 16 * c, lo);
          }
          tc::tmem_wait_st();
        }
        const float ls[4] = {ls2[0].x, ls2[0].y, ls2[1].x, ls2[1].y};
        lsum += (ls[0] + ls[1]) + (ls[2] + ls[3]);
        if (__any_sync(0xffffffffu, need) && t > 0) {
          // P(t-1) V(t-1) must have completed before this warp rescales its half
          // of O. That buffer's next P.V needs a P this softmax has not written
          // yet, so the barrier's parity cannot alias; P(t) V(t) waits for this
          // warp's pfull arrival below.
          if (!__all_sync(0xffffffffu,
                          wait_or_abort(&s.pvdone[(Tc - 1) % kSBufs], ((Tc - 1) / kSBufs) & 1, s.abort))) {
            raise_abort(a, s.abort, tc::kSiteMma);
            ok = false;
            continue;
          }
          tc::tc_fence_after();
          for (int c = hh * kOW; c < hh * kOW + kOW; c += 32) {
            float o[32];
            tc::tmem_ld32(tl + kOneOCol + c, o);
#pragma unroll
            for (int i = 0; i < 32; ++i) o[i] *= alpha;
            tc::tmem_st32(tl + kOneOCol + c, o);
          }
        }
        tc::tc_fence_before();
        tc::mbar_arrive(&s.pfull[sbuf]);
      }
      T += nt;
      // row sum = the two halves' sums (same running max in both)
      s.xsum[hh * 128 + row] = lsum;
      asm volatile("bar.sync 1, %0;" ::"n"(kSoftThreads) : "memory");
      const float total = s.xsum[row] + s.xsum[128 + row];
      // O of this item is complete once the MMA thread's per-item commit has
      // arrived (it cannot run a phase ahead: the next one needs this warp's P)
      const bool fin = __all_sync(0xffffffffu, ok && wait_or_abort(s.ofull, n & 1, s.abort));
      if (!fin && ok) {
        raise_abort(a, s.abort, tc::kSiteFinal);
        ok = false;
      }
      if (fin) {
        tc::tc_fence_after();
        // no weight at all (every logit -inf): NaN below 128 dims, as on CUDA cores
        const float inv = total > 0.f ? 1.f / total : kSplit ? NAN : 0.f;
        const int64_t row_off = ((int64_t(it.l) * a.n_sel + i_row) * Hq + h_row) * d;
        __nv_bfloat16* dst = a.out + row_off;
        float zero = 0.f;  // NaN where a value is not finite
        // This thread's columns of O, 32 at a time, as bf16. Each lane writes its own
        // row, so a warp's store covers 32 rows: 32-byte stores (whole sectors)
        // when the buffer allows them.
#pragma unroll
        for (int c = hh * kOW; c < hh * kOW + kOW; c += 32) {
          float o[32];
          tc::tmem_ld32(tl + kOneOCol + c, o);
          if (!live) continue;
          if (kSplit) {
#pragma unroll
            for (int i = 0; i < 32; ++i) zero = fmaf(o[i], 0.f, zero);
          }
          uint32_t w[16];
#pragma unroll
          for (int k2 = 0; k2 < 16; ++k2) {
            __nv_bfloat162 pr = __floats2bfloat162_rn(o[2 * k2] * inv, o[2 * k2 + 1] * inv);
            w[k2] = *reinterpret_cast<uint32_t*>(&pr);
          }
          if (a.out32) {
#pragma unroll
            for (int u8 = 0; u8 < 2; ++u8)
              if (c + u8 * 16 < d)
                asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + c + u8 * 16),
                             "r"(w[8 * u8]), "r"(w[8 * u8 + 1]), "r"(w[8 * u8 + 2]), "r"(w[8 * u8 + 3]),
                             "r"(w[8 * u8 + 4]), "r"(w[8 * u8 + 5]), "r"(w[8 * u8 + 6]), "r"(w[8 * u8 + 7])
                             : "memory");
          } else {
#pragma unroll
            for (int u4 = 0; u4 < 4; ++u4)
              if (c + u4 * 8 < d)
                *reinterpret_cast<uint4*>(dst + c + u4 * 8) = make_uint4(w[4 * u4], w[4 * u4 + 1], w[4 * u4 + 2], w[4 * u4 + 3]);
          }
        }
        if (kSplit) {
          // (a sum that is NaN comes from Q or K, and the row is NaN as it should be)
          const uint32_t redo = __ballot_sync(0xffffffffu, live && total > 0.f && zero != 0.f);
          if (redo)
            redo_rows<kOW>(a, redo, it.l, it.g, it.r, rec_t0, p_row, m_ref, inv, row_off, hh * kOW, lane);
        }
      }
      tc::tc_fence_before();
      tc::mbar_arrive(s.oempty);  // O may be overwritten by the next item
    }
  }
  __syncthreads();
  if (tid == 0) {  // drain loads issued but never consumed (only after an abort)
    for (uint32_t n = s.counters[2]; n < s.counters[0]; ++n)
      tc::mbar_wait(&s.kfull[n % kKStages], (n / kKStages) & 1);
    for (uint32_t n = s.counters[3]; n < s.counters[1]; ++n)
      tc::mbar_wait(&s.vfull[n % kVStages], (n / kVStages) & 1);
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 1) tc::tmem_dealloc(tmem, kTmemCols);
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

bool make_map(CUtensorMap* m, const KvDev& kv, void* base) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return false;
  cuuint64_t dims[2] = {cuuint64_t(kv.d), 0};
  cuuint64_t strides[1] = {cuuint64_t(kv.d) * 2};
  cuuint32_t box[2] = {64, 0};
  cuuint32_t estr[2] = {1, 1};
  if (kv.page_size == 0) {
    dims[1] = cuuint64_t(kv.L) * kv.Hkv * kv.n_tot;
    box[1] = kKT;
  } else {
    dims[1] = cuuint64_t(kv.L) * kv.num_pages * kv.Hkv * kv.page_size;
    box[1] = kv.page_size;
  }
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Query rows [L * n_sel][Hq][d] as a 3-D map with box (64 dims, G heads,
// rows_per_tile rows): one box fills one 64-dim half of a query tile in the
// tile's row order (selected row major, head minor).
bool make_qmap(CUtensorMap* m, const KvDev& kv, const void* q_rows, int32_t n_sel, int rows_per_tile) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return false;
  cuuint64_t dims[3] = {cuuint64_t(kv.d), cuuint64_t(kv.Hq), cuuint64_t(kv.L) * cuuint64_t(n_sel)};
  cuuint64_t strides[2] = {cuuint64_t(kv.d) * 2, cuuint64_t(kv.Hq) * kv.d * 2};
  cuuint32_t box[3] = {64, cuuint32_t(kv.G), cuuint32_t(rows_per_tile)};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(q_rows), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

// Every bf16 head size the copies can pad to one or two 64-dim halves: a step on
// a 24-layer, 14/2-head, head_dim 64 cache of 2 900 tokens took 8.6 ms with this
// pass and the scoring on CUDA cores and takes 0.22 ms with both here.
bool refresh_tc_supported(const KvDev& kv) {
  if (kv.dtype != CONDUIT_BF16 || kv.d > kMaxD || kv.G > kRows || !tc_rows_ok(kv)) return false;
  if (kv.page_size != 0 && (kv.page_size % 8 != 0 || kKT % kv.page_size != 0)) return false;
  return true;
}

// Blocks of `span` rows of a (layer, KV head), over its requests.
static int query_blocks(const BatchDev& b, const int32_t* off_host, int span) {
  int blocks = 0;
  for (int r = 0; r < b.R; ++r) blocks += (off_host[r + 1] - off_host[r] + span - 1) / span;
  return blocks;
}

// One query tile per item or two. The split P of the smaller head sizes makes a
// tile's softmax and P V longer, and one tile per item is faster throughout (24
// layers, 14/2 heads of 64 dims: 2 916 tokens 93 us / 107 with two, 24 576 tokens
// 4 636 / 4 747; 16 layers, 32/8 heads of 96 dims, 16 384 tokens 3 229 / 3 855).
// For head_dim 128 it goes by the key tiles that two-tile items would bring to an
// SM. Two-tile items are half as many and cost less per tile, which pays once
// the end of the launch no longer shows (one / two tiles per item, us):
// 2 layers x 1 885 tokens 22.6 / 35.0, 28 x 1 024 42.8 / 45.0, 36 x 4 096 (213
// key tiles per SM) 423 / 442, two requests of 4 096 (283) 498 / 511, 28 x 6 144
// (319) 598 / 590, 28 x 8 192 (540) 912 / 896, long document (8 000) 15 400 /
// 15 000. Pages of 16 keys and fewer cost one tile per item more, since each
// page half is a copy of its own: 8 x 2 048 (10) 39.3 / 42.7, 28 x 2 048 (35)
// 108.7 / 106.9, 8 x 4 096 (40) 109.2 / 105.6, four requests of 2 048 (142) 404
// / 381; pages of 32 are as contiguous caches (28 x 2 048 97.3 / 105.2).
constexpr double kOneKeyTilesPerSm = 300., kOneKeyTilesPerSmPaged = 24.;
constexpr int kOneMinPage = 32;
// Items per SM in longest-first order at the end of a launch whose K/V exceeds
// L2: 0 / 2 / 3 / 4 items took 213 / 196 / 196.5 / 199 us on 16 layers of 4 096
// tokens (one tile per item) and 952 / 908 / 896 / 904 us on 28 of 8 192 (two).
constexpr int kTailItemsPerSm = 3;
// Up to this many one-tile items per SM come in a fixed order (they are then
// longest first throughout): a counter costs its reset and an atomic per item, and
// evens out more items than that. Fixed / counter, us: 2 layers of 1 885 tokens (96
// items) 20.5 / 22.6, 28 of 600 (448) 26.7 / 28.3, three requests of 1 024 (576)
// 38.5 / 38.9, 28 of 1 024 (672) 44.5 / 43.0, 14 of 2 000 (672) 58.0 / 54.6.
constexpr int kDealtItemsPerSm = 3;

cudaError_t launch_refresh_tc(const KvDev& kv, const BatchDev& b, const int32_t* idx,
                              const int32_t* idx_off_dev, const int32_t* idx_off_host, int32_t n_sel,
                              const void* q_rows, void* out, int32_t* work_counter, int32_t* status,
                              cudaStream_t stream) {
  if (n_sel == 0) return cudaSuccess;
  CUtensorMap kmap, vmap, qmap;
  if (!make_map(&kmap, kv, kv.k) || !make_map(&vmap, kv, kv.v) ||
      !make_qmap(&qmap, kv, q_rows, n_sel, kRows / kv.G))
    return cudaErrorInvalidValue;
  RefArgs a{};
  a.kv = kv;
  a.b = b;
  a.idx = idx;
  a.idx_off = idx_off_dev;
  a.out = static_cast<__nv_bfloat16*>(out);
  a.q = static_cast<const __nv_bfloat16*>(q_rows);
  a.out32 = (reinterpret_cast<uintptr_t>(out) & 31) == 0 && kv.d % 16 == 0;
  a.n_sel = n_sel;
  a.rows_per_tile = kRows / kv.G;
  int dev = 0, sms = 0, l2 = 0;
  cudaError_t err;
  if ((err = cudaGetDevice(&dev))) return err;
  if ((err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return err;
  if ((err = cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, dev))) return err;
  const int n_lg = kv.Hkv * kv.L;
  a.span = 2 * a.rows_per_tile;
  a.n_blocks = query_blocks(b, idx_off_host, a.span);
  const double key_tiles = double(a.n_blocks) * n_lg * (double(kv.n_tot) / b.R) / (2 * kKT);
  const bool few_copies = kv.page_size == 0 || kv.page_size >= kOneMinPage;
  const bool one = kv.d != kMaxD || key_tiles < sms * (few_copies ? kOneKeyTilesPerSm : kOneKeyTilesPerSmPaged);
  if (one) {
    a.span = a.rows_per_tile;
    a.n_blocks = query_blocks(b, idx_off_host, a.span);
  }
  a.n_items = a.n_blocks * n_lg;
  a.next_item = a.n_items <= (one ? kDealtItemsPerSm * sms : sms) ? nullptr : work_counter;
  a.scale_log2 = kLog2e / sqrtf(float(kv.d));
  a.status = status;
  if (a.n_blocks == 0) return cudaSuccess;
  // longest-first throughout when the whole K/V of the batch fits in half of L2
  // (the rest holds queries and outputs), else for about the last kTailItemsPerSm
  // items of each SM
  const double kv_bytes = 2.0 * double(n_lg) * double(kv.n_tot) * kv.d * 2;
  a.tail = kv_bytes <= 0.5 * double(l2) ? n_lg : std::min(n_lg, (kTailItemsPerSm * sms + a.n_blocks - 1) / a.n_blocks);
  if (a.next_item && (err = cudaMemsetAsync(work_counter, 0, sizeof(int32_t), stream))) return err;
  auto launch = [&](auto* f, uint32_t smem) -> cudaError_t {
    if ((err = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)))) return err;
    f<<<std::min(a.n_items, sms), kThreads, smem, stream>>>(kmap, vmap, qmap, a);
    return cudaGetLastError();
  };
  // head_dim 128 keeps its bf16 P; the smaller sizes ran with fp32 weights on
  // CUDA cores before and keep that precision by a split P
  if (!one)
    err = launch(refresh_tc_kernel<false>, kSmem);
  else if (kv.d == kMaxD)
    err = launch(one_refresh_tc_kernel<2, false>, kOneSmem);
  else if (kv.d > 64)
    err = launch(one_refresh_tc_kernel<2, true>, kOneSmem);
  else
    err = launch(one_refresh_tc_kernel<1, true>, kOneSmem);
  if (err) return err;
  count_launches(1);
  return cudaSuccess;
}

// At 128 dims, where the estimator has always run on tensor cores. They truncate each
// of their sums, which a bf16 output row does not show and a sum of squared rows does;
// with the split P of the smaller head sizes, twice as many sums, it came out low by
// 3e-5 at 8 192 keys and 7e-5 at 16 384 (64 dims), more than the whole error of the
// CUDA-core kernels (0.6e-5 and 1.7e-5 at 16 384). These take 15.7 ms for 0.7 (28
// layers, 28/4 heads of 64 dims, 4 096 keys, five draws).
bool stale_tc_supported(const KvDev& kv) { return kv.d == kMaxD && refresh_tc_supported(kv); }

int stale_tc_blocks(const KvDev& kv, const BatchDev& b, const int32_t* q_off_host) {
  return query_blocks(b, q_off_host, 2 * (kRows / kv.G));
}

cudaError_t launch_stale_tc(const KvDev& kv, const BatchDev& b, const int32_t* q_off_host, int32_t q_tot,
                            const void* q, const void* z, int draws, const float* key_scale, double* part,
                            int32_t* work_counter, int32_t* status, cudaStream_t stream) {
  CUtensorMap kmap, zmap, qmap;
  RefArgs a{};
  a.kv = kv;
  a.b = b;
  a.idx_off = b.q_off;
  a.n_sel = q_tot;
  a.rows_per_tile = kRows / kv.G;
  a.span = 2 * a.rows_per_tile;
  a.n_blocks = query_blocks(b, q_off_host, a.span);
  a.draws = draws;
  a.n_items = draws * a.n_blocks * kv.Hkv * kv.L;
  a.next_item = work_counter;
  a.scale_log2 = kLog2e / sqrtf(float(kv.d));
  a.status = status;
  a.key_scale = key_scale;
  a.part = part;
  if (a.n_items == 0) return cudaSuccess;
  KvDev kz = kv;  // the draws are contiguous whatever the cache is
  kz.page_size = 0;
  kz.L = kv.L * draws;
  EncodeTiledFn enc = encode_fn();
  if (!enc || !make_map(&kmap, kv, kv.k) || !make_map(&zmap, kz, const_cast<void*>(z))) return cudaErrorInvalidValue;
  // the scoring queries [L * Hq][q_tot][d]: box (64 dims, rows_per_tile queries, G heads)
  cuuint64_t dims[3] = {cuuint64_t(kv.d), cuuint64_t(q_tot), cuuint64_t(kv.L) * kv.Hq};
  cuuint64_t strides[2] = {cuuint64_t(kv.d) * 2, cuuint64_t(q_tot) * kv.d * 2};
  cuuint32_t box[3] = {64, cuuint32_t(a.rows_per_tile), cuuint32_t(kv.G)};
  cuuint32_t estr[3] = {1, 1, 1};
  if (enc(&qmap, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(q), dims, strides, box, estr,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  int dev = 0, sms = 0;
  cudaError_t err;
  if ((err = cudaGetDevice(&dev))) return err;
  if ((err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev))) return err;
  if ((err = cudaMemsetAsync(work_counter, 0, sizeof(int32_t), stream))) return err;
  auto launch = [&](auto* f, uint32_t smem) -> cudaError_t {
    if ((err = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)))) return err;
    f<<<std::min(a.n_items, sms), kThreads, smem, stream>>>(kmap, zmap, qmap, a);
    return cudaGetLastError();
  };
  err = launch(refresh_tc_kernel<true>, kSmem);
  if (err) return err;
  count_launches(1);
  return cudaSuccess;
}

}  // namespace conduit
