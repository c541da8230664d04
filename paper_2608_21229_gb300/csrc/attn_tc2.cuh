// attn_tc2.cuh -- the tcgen05 attention kernel on CTA pairs: for every
// (task, head) item, O = softmax(scale * Q K^T) V over the task's visible keys
// (key ranges A then B; see common.cuh), scores, softmax and accumulation in
// fp32 and P rounded to bf16 for P.V, with every MMA issued over two CTAs on
// neighbouring SMs (tcgen05 cta_group::2, M = 256).  Head dim 128 or 64.
//
// Why pairs: with one 128-row query tile per SM, each S/P.V pair of MMAs
// (1024 tensor cycles at 128-key tiles) needs a fresh 32 KB K tile and 32 KB
// V tile in that SM's shared memory.  The tensor core's operand reads (about
// 96 KB per pair) plus those 64 KB of TMA fills exceed what one SM's shared
// memory delivers in 1024 cycles (128 bytes per cycle), so the tensor core
// waits for data.  A CTA pair shares every K/V tile: CTA r holds keys
// [kBN/2 r, kBN/2 (r + 1)) of each K tile and head-dim columns [64 r, 64 r +
// 64) of each V tile (32 of 64 at head dim 64; the B operand of a cta_group::2
// MMA is split along N between the two CTAs), while each CTA keeps its own 128 query rows (A is
// split along M).  Per SM this halves the tile bytes fetched and the
// B-operand bytes read, for the same MMA work.
//
// Key tiles (kBN): 192 keys for the bf16 cache, 128 for the E4M3 cache and
// the 128-key comparison variant.  At 192 keys P is written over the first
// half of its own S buffer, which is what makes two 192-column S buffers and
// the 128-column O fit in the 512 TMEM columns; each handshake then carries
// 1536 tensor cycles of MMAs instead of 1024 (see Cfg).
//
// Cluster of 2 CTAs (rank 0 = leader), 224 threads each:
//   warps 0-3  softmax: thread l of warp w owns row 32 w + l of this CTA's
//              128 rows (its TMEM lane), all kBN score columns of a tile
//   warp 4     TMA producer: this CTA's Q rows and its halves of the K and V
//              tiles; completion is counted on the leader's barriers
//   warp 5     both CTAs: TMEM allocation (a pair operation); leader only:
//              the MMA warp (one elected lane issues every MMA and commit)
//   warp 6     leader only: the gate warp, which does every mbarrier wait
//              the MMAs depend on and hands each group to the MMA warp
//              through a named barrier
// One softmax warp per SM sub-partition leaves the MMA warp's sub-partition
// with a single busy warp beside it, and a row needs no partner thread.
// An item is a task of up to 256 query rows: CTA r takes rows
// [128 r, 128 r + 128).  Items come from a per-item list ordered on the host
// or, head-major, from the task list: with a work counter each CTA pair takes
// its first item by its index and then the next of the list, else pair c takes
// items c, c + n_pairs, ...  The leader's producer chooses them and passes each
// item's Task on through a ring in both CTAs' shared memory.
//
// Work is done item by item (an item = a task of up to 256 rows x one
// head).  An item with n key tiles is a sequence of n + 1 MMA groups:
//   group G               S_1 = Q K_1^T (empty when n = 1)
//   group G + 1 + j       O += P_j V_j, then S_j+2 = Q K_j+2^T when j + 2 < n;
//                         beside P_n-2 V_n-2 (or in group G when n = 1) the
//                         next item's S_0
// numbered g = 0, 1, 2, ... over all items of the cluster; group 0 is the first
// item's S_0 alone.  Tiles are numbered t over all items: K_t and V_t lie in
// slot t % kStages of a K and a V ring (24 KB each per CTA at 192-key tiles, 16
// KB at 128), S_t and P_t in TMEM buffer t % 2.
//
// Between items: an item's Q and first K tiles are loaded, and its S_0 is
// issued, while the item before it still runs, so that only the epilogue (O
// read, normalised and stored) and the next item's first softmax lie between
// the last P.V of one item and the first of the next.  For that the item is
// chosen a few tiles ahead and its Task travels through shared memory: taking
// the item, passing it to the other CTA and reading its Task from global memory
// in every role one after the other took about 5000 cycles per item, and the
// epilogue's uncoalesced stores 2000.  MMA-thread waits around an item's start
// went from 5100 to 2700 cycles, 3 % of a step with 1280 live and 2048 cached
// rows and 24 heads (items of 18 tiles).
//
// Synchronisation is built so that the MMA thread waits on nothing itself: all
// mbarrier waits are done by the gate warp: per group, the gate warp waits for
// what the group needs and then meets the MMA warp at `bar.red.or` (which also
// carries an abort bit: both warps walk the same group sequence and leave
// together, so neither can be left waiting); the MMA thread then issues the group
// and commits once:
//   pair_done[g % 4]   one commit per group (multicast to both CTAs): its S
//                      is in TMEM, its P.V is in O, the ring slots and the P
//                      buffer it read are free.  Four barriers, so that no
//                      waiter can miss a phase: a waiter for group g holds up
//                      group g + 4.
//   p_full[t % 2]      one arrival per softmax warp of both CTAs.  Its phase
//                      for tile t means P_t is in TMEM and every softmax thread
//                      has finished reading O for the previous item.
//   p_half[t % 2]      192-key tiles: the same for P's first 96 keys, whose
//                      P.V MMAs are issued while the softmax works on the rest
//                      (E4M3 kernel: 64 of 128 keys, with them S_t+2, since P has
//                      buffers of its own there and S_t has been read by then)
//   k_full[s] v_full[s]  the producers' TMA bytes of both CTAs (leader's barriers)
//   q_full             per Q buffer, once per item
//   q_empty            per Q buffer: the item's last S has read it, and the
//                      epilogue no longer stages O in it
//   item_full / item_empty  per slot of the item ring
// The MMAs' operands live in uniform registers.  The MMAs are issued under
// elect.sync, from which the compiler knows that one lane runs (under `lane ==
// 0` it has to cope with any set of lanes, and a tile's 20 MMAs took 1507 cycles
// to issue instead of 610, about as long as the tensor core needs for them), and
// the values the operands are computed from (tensor-memory base, warp index, key
// tiles) pass through a shuffle, which makes them the same in all lanes.
//
// P in two pieces (192-key tiles): a tile's P.V and the S that reuses its
// buffer (1536 tensor cycles) cannot start before its softmax is done, and with
// two S buffers that loop -- S ready, softmax, P, MMAs, next S ready -- set the
// period: 1880 cycles per tile at 4608 live and 20480 cached rows, 24 heads, of
// which the MMA thread waited 480 for P.  With the first 96 keys handed over
// early, their handshake and their P.V MMAs leave the loop.  Cycles per tile by
// the size of the first piece: 64 keys 1678, 96 keys 1635, 128 keys 1641 (32 keys,
// with the MMAs under lane == 0, 46 more than 96).
//
// The softmax warps are as long in a tile (about 1550 cycles: loads and maximum
// 215, exponentials and P 1180 of which the exponential unit needs 800, the rest
// the waits and the loop), so they look at the next S while their last stores of
// P drain instead of waiting for it afterwards (130 cycles of latency per tile),
// and find a tile's end from the item's lengths with two instructions.
//
// E4M3 cache (kF8): key range B is the quantised reference cache -- K as
// E4M3 codes [rows_pad, H, 128] and V transposed per head [H, 128, rows_pad],
// both K-major operands, with one fp32 scale (s_K, s_V) per 128-row tile and
// head.  Its tiles run as kind::f8f6f4 MMAs (K = 32 per instruction, half
// the tensor cycles of bf16); range A (the live rows) stays bf16.  At the
// start of an item with cached tiles every softmax thread quantises its own
// query row of this head into an E4M3 Q tile (one scale per row), and the
// first cached tile's S waits for it (q8_full, one arrival per softmax warp
// of both CTAs).  The producer also feeds each CTA a small shared-memory ring
// of the cached tiles' scales (16-byte bulk copies), so that the softmax loop
// touches no global memory.  The scales enter the softmax, so one O
// accumulator serves both ranges: with
// s_ref = s_V of the item's first cached tile, the weights written are
//   live tile:    exp2(u - m) / s_ref                   (bf16, u = scaled score)
//   cached tile:  exp2(u + delta - m), delta = log2(s_V / s_ref)   (E4M3)
// where the running maximum m is taken over u + delta, so E4M3 weights stay
// at most 2^8; each tile adds its unshifted weight sum to l, and
// O = s_ref * acc / l.
#pragma once
#include "attn_tc.cuh"

namespace rc {

namespace tc2 {
using tc::Ctl;
constexpr int kD = 128;
constexpr uint32_t kQTile = 128 * 128 * 2;
// Warp roles: softmax warps first, then the producer, the MMA warp and the gate
// warp.
//
// kBN = keys per tile: 128, or 192 for the bf16 cache.  With 192-key tiles P
// is written over the first half of its own S buffer, so that tensor memory
// holds S_0 [0, 192), S_1 [192, 384) and O [384, 512); an MMA group is then
// 12 P.V MMAs and 8 S MMAs of N = 192 (1536 tensor cycles per handshake
// instead of 1024), and since the S MMAs that reuse a buffer overwrite the P
// that the group's P.V MMAs read, a group issues all its P.V MMAs first.
// With 128-key tiles P has buffers of its own (the groups keep that order).
template <bool kF8, int kBN>
struct Cfg {
  static_assert(kBN == 128 || (kBN == 192 && !kF8), "key tiles of 128 keys, or 192 with the bf16 cache");
  static constexpr int kSoftmaxWarps = 4;
  static constexpr int kProducerWarp = kSoftmaxWarps, kMmaWarp = kSoftmaxWarps + 1, kGateWarp = kSoftmaxWarps + 2;
  static constexpr int kThreads = 32 * (kSoftmaxWarps + 3);
  static constexpr int kWarpArrivals = 2 * kSoftmaxWarps;  // p_full / q8_full: every softmax warp of both CTAs
  // warps that read each item from the ring: the leader's gate and softmax
  // warps, the follower's producer and softmax warps
  static constexpr int kItemTakers = 2 + 2 * kSoftmaxWarps;
  static constexpr int kStages = kBN == 128 ? 4 : 3;     // K and V ring slots (shared memory: 2 Q + slots <= 227 KB)
  static constexpr uint32_t kKBox = (kBN / 2) * 128;     // one K box: kBN / 2 rows x 128 bytes
  static constexpr uint32_t kKHalf = 2 * kKBox;          // this CTA's kBN / 2 keys x 128 d of a K tile
  static constexpr uint32_t kVHalf = kBN * 64 * 2;       // kBN keys x this CTA's 64 d of a V tile (head dim 64: 32)
  static constexpr uint32_t kStage = kKHalf + kVHalf;
  static constexpr bool kPOverS = kBN != 128;
  static constexpr uint32_t kColS = 0;                   // S buffer b at kColS + b * kBN
  static constexpr uint32_t kColP = kPOverS ? 0u : 256u; // P buffer b at kColP + b * kPStride
  static constexpr uint32_t kPStride = kPOverS ? kBN : 64u;
  static constexpr uint32_t kColO = 384;
  // 32-key chunks of P handed over ahead of the rest (0: P in one piece), see
  // the head of the file
  static constexpr int kPSplit = kPOverS ? 3 : kF8 ? 2 : 0;
  static_assert(2 * kBN <= 384 && kColO + kD <= tc::kTmemCols, "tensor-memory layout");
};
constexpr int kPairDoneBars = 4;          // pair_done[g % 4]: a waiter for group g holds up group g + 4
constexpr uint32_t kGateBarrier = 1;  // named barrier of the MMA and gate warps (0 is __syncthreads)
constexpr uint32_t kKHalf8 = 64 * 128;   // 8 KB: this CTA's 64 keys x 128 d of an E4M3 K tile
constexpr uint32_t kVHalf8 = 64 * 128;   // 8 KB: this CTA's 64 d x 128 keys of an E4M3 V^T tile
constexpr uint32_t kQ8Tile = 128 * 128;  // this CTA's 128 query rows as E4M3
constexpr int kScaleSlots = 8;           // ring of per-tile scales of cached tiles (E4M3 kernel)
constexpr int kItemSlots = 8;            // ring of items

template <bool kF8, int kBN>
struct SmemT {
  using C = Cfg<kF8, kBN>;
  static constexpr int kStages = C::kStages;
  static constexpr uint32_t kQ = 0;                // Q buffers 0 and 1 (this CTA's 128 rows)
  static constexpr uint32_t kRing = 2 * kQTile;    // slot s: [K half | V half]
  static constexpr uint32_t kQ8 = kRing + kStages * C::kStage;  // E4M3 Q tile (kF8 only)
  static constexpr uint32_t kScales = kQ8 + (kF8 ? kQ8Tile : 0u);  // ring of kScaleSlots x 16 B (kF8 only)
  static constexpr uint32_t kBars = kScales + (kF8 ? kScaleSlots * 16u : 0u);
  static constexpr int kQFull = 0, kQEmpty = 2, kKFull = 4, kVFull = kKFull + kStages, kPairDone = kVFull + kStages,
                       kPFull = kPairDone + kPairDoneBars, kPHalf = kPFull + 2, kMmaDone = kPHalf + 2, kQ8Full = kMmaDone + 1,
                       kScaleFull = kQ8Full + 1, kScaleEmpty = kScaleFull + kScaleSlots,
                       kItemFull = kScaleEmpty + kScaleSlots, kItemEmpty = kItemFull + kItemSlots,
                       kNumBars = kItemEmpty + kItemSlots;
  static constexpr uint32_t kTmemHolder = kBars + 8 * kNumBars;
  static constexpr uint32_t kAbort = kTmemHolder + 4;
  // load record of each CTA of the pair (leader's copy read at teardown): K
  // tiles, V tiles and Q tiles loaded, whether the last K load of slot s (bit s)
  // and the last V load (bit kStages + s) was of a cached E4M3 tile, and whether
  // K tile 0 was left out (fault injection)
  static constexpr int kRecK = 0, kRecV = 1, kRecQ = 2, kRecLast8 = 3, kRecSkipped = 4;
  static constexpr uint32_t kRecWords = 5;
  static constexpr uint32_t kLoadRec = kAbort + 4;
  // ring of items: slot k % kItemSlots holds item k of this cluster (a Task;
  // head -1: none left); the gate warp passes the MMA warp its item's tiles
  static constexpr uint32_t kItemRing = (kLoadRec + 2 * kRecWords * 4 + 15u) & ~15u;
  static constexpr uint32_t kGateItem = kItemRing + 32 * kItemSlots;  // two of [key tiles, of range A, first S ahead, -]
  static constexpr uint32_t kPeerAbort = kGateItem + 32;  // the other CTA's abort flag, at teardown
  static constexpr uint32_t kUsed = kPeerAbort + 4;
  static constexpr uint32_t kMaxDynamic = 232448;
  static constexpr uint32_t kDynamic = kUsed + 1024 < kMaxDynamic ? kUsed + 1024 : kMaxDynamic;
  static_assert(kUsed <= kMaxDynamic, "shared-memory layout too large");
  static_assert(C::kStage % 1024 == 0 && C::kKBox % 1024 == 0, "swizzle atoms start on 1024-byte boundaries");
};

// Key tiles of kBN keys: tile j of an item (range A first, then range B).
template <int kBN>
__device__ __forceinline__ tc::TileSrc tile_src(const Task& t, int na, int j) {
  tc::TileSrc s;
  if (j < na) {
    s.row = t.a_row0 + j * kBN;
    s.valid = min(kBN, t.a_len - j * kBN);
    s.in_b = false;
  } else {
    const int jj = j - na;
    s.row = t.b_row0 + jj * kBN;
    s.valid = min(kBN, t.b_len - jj * kBN);
    s.in_b = true;
  }
  return s;
}
template <int kBN>
__device__ __forceinline__ int n_key_tiles(const Task& t, int& na) {
  na = (t.a_len + kBN - 1) / kBN;
  return na + (t.b_len + kBN - 1) / kBN;
}

// Phase parity of pair_done[g % 4] for group g.
__device__ __forceinline__ uint32_t group_parity(int g) { return static_cast<uint32_t>(g >> 2) & 1u; }
// Ring slot of tile t and the phase parity of its barrier.
template <int kStages>
__device__ __forceinline__ int slot_of(int t) { return t % kStages; }
template <int kStages>
__device__ __forceinline__ uint32_t slot_parity(int t) { return static_cast<uint32_t>(t / kStages) & 1u; }

// Bounded wait on a barrier that other CTAs arrive on, for TMA bytes and tensor
// memory (ordered by the copies' completion and the tcgen05 fences).
__device__ __forceinline__ bool wait_cl(uint32_t bar, uint32_t parity, const Ctl& c, int where) {
  return tc::wait_one(bar, parity, c, where);
}
__device__ __forceinline__ bool wait_cl_warp(uint32_t bar, uint32_t parity, const Ctl& c, int where) {
  const bool ok = wait_cl(bar, parity, c, where);
  return __all_sync(0xffffffffu, ok);
}
// The same for what the other CTA wrote, or has read, with ordinary loads and
// stores before it arrived (with release at cluster scope): the acquire has to
// be at cluster scope too.  Once per item; the phase is complete after wait_cl.
__device__ __forceinline__ bool wait_cl_acquire(uint32_t bar, uint32_t parity, const Ctl& c, int where) {
  return wait_cl(bar, parity, c, where) && mbar_try_wait_acquire_cluster(bar, parity);
}
// Work counter [next item, clusters done]: this cluster takes no more items; the
// last cluster resets both words for the next launch, which reads them only
// after this grid has completed.
__device__ __forceinline__ void work_done(int* work, int n_clusters) {
  __threadfence();
  if (atomicAdd(work + 1, 1) == n_clusters - 1) {
    __threadfence();
    atomicExch(work, 0);
    atomicExch(work + 1, 0);
  }
}
}  // namespace tc2

// kDG: the head dim.  At 64 a Q or K row is one 64-column box (S = Q K^T takes
// four K = 16 steps) and each CTA of a pair holds 32 of V's 64 columns: 64-byte
// rows with the 64-byte swizzle, P V with N = 64, O in 64 columns of tensor
// memory.  (Padded to 128 columns, with zeros for the second CTA's half, P V did
// twice the work.  The softmax warps bound this head dim, but the MMAs lie on the
// way from P to the next S: unpadded, an in-place build of three requests with 48
// heads, 1614 to 6271 rows, takes 5 % less, a step of 320 live and 256 cached rows
// with 4 heads 2 %.)
template <bool kF8, int kBN, int kDG>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(tc2::Cfg<kF8, kBN>::kThreads, 1)
    attn_tc2_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_ka,
                    const __grid_constant__ CUtensorMap tm_va, const __grid_constant__ CUtensorMap tm_kb,
                    const __grid_constant__ CUtensorMap tm_vb, const AttnArgs args,
                    const __grid_constant__ Spans spans) {
  using namespace tc;
  using tc2::kQTile;
  using Cfg = tc2::Cfg<kF8, kBN>;
  constexpr uint32_t kKBox = Cfg::kKBox;
  constexpr uint32_t kKHalf = Cfg::kKHalf;
  constexpr uint32_t kVHalf = kBN * kDG;  // bytes of this CTA's V half: kBN keys x kDG / 2 columns
  constexpr uint32_t kVStep = 16 * kDG;   // of which 16 keys
  constexpr uint32_t kStage = Cfg::kStage;
  constexpr int kStages = Cfg::kStages;
  constexpr uint32_t kColS = Cfg::kColS, kColP = Cfg::kColP, kPStride = Cfg::kPStride, kColO = Cfg::kColO;
  constexpr int kWarpArrivals = Cfg::kWarpArrivals;
  constexpr int kPSplit = Cfg::kPSplit;
  using tc2::group_parity;
  using tc2::wait_cl;
  using tc2::wait_cl_acquire;
  using tc2::wait_cl_warp;
  using tc2::kKHalf8;
  using tc2::kVHalf8;
  using L = tc2::SmemT<kF8, kBN>;
  constexpr int D = tc2::kD;   // the larger head dim
  constexpr int DG = kDG;      // head dim of the tensors
  static_assert(DG == D || (DG == 64 && !kF8), "head dim 128, or 64 (bf16 cache)");
  constexpr int kQBoxes = DG / 64;  // 64-column boxes of a Q or K row loaded
  auto slot_of = [](int t) -> int { return tc2::slot_of<kStages>(t); };
  auto slot_parity = [](int t) -> uint32_t { return tc2::slot_parity<kStages>(t); };
  constexpr uint32_t kIdescS = idesc_bf16_f32(256, kBN, false);
  constexpr uint32_t kIdescO = idesc_bf16_f32(256, DG, true);
  constexpr uint32_t kIdesc8 = idesc_e4m3_f32(256, 128);  // S and O of cached tiles (N = 128 keys or d)

  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* base_ptr = smem_raw + (base - raw);
  auto bar = [&](int i) -> uint32_t { return base + L::kBars + 8u * static_cast<uint32_t>(i); };
  volatile int* abort_flag = reinterpret_cast<volatile int*>(base_ptr + L::kAbort);
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(base_ptr + L::kTmemHolder);

  const int warp = __shfl_sync(0xffffffffu, static_cast<int>(threadIdx.x >> 5), 0);
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int cluster = static_cast<int>(blockIdx.x >> 1);
  const int n_clusters = static_cast<int>(gridDim.x >> 1);
  // Both CTAs of a pair get the same layout, so both leave here together.
  if (base - raw + L::kUsed > L::kDynamic) {
    if (threadIdx.x == 0) tc::report_timeout(args.status, 99);
    if (threadIdx.x == 0 && leader && args.work != nullptr) tc2::work_done(args.work, n_clusters);
    return;
  }

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(L::kQFull + i), 1);
      mbar_init(bar(L::kQEmpty + i), 1 + Cfg::kSoftmaxWarps);  // its last S, and O staged in it written
      mbar_init(bar(L::kPFull + i), kWarpArrivals);
      mbar_init(bar(L::kPHalf + i), kWarpArrivals);
    }
    for (int s = 0; s < kStages; ++s) {
      mbar_init(bar(L::kKFull + s), 1);
      mbar_init(bar(L::kVFull + s), 1);
    }
    for (int s = 0; s < tc2::kPairDoneBars; ++s) mbar_init(bar(L::kPairDone + s), 1);
    mbar_init(bar(L::kMmaDone), 1);
    mbar_init(bar(L::kQ8Full), kWarpArrivals);
    for (int s = 0; s < tc2::kScaleSlots; ++s) {
      mbar_init(bar(L::kScaleFull + s), 1);
      mbar_init(bar(L::kScaleEmpty + s), Cfg::kSoftmaxWarps);
    }
    for (int s = 0; s < tc2::kItemSlots; ++s) {
      mbar_init(bar(L::kItemFull + s), 1);
      mbar_init(bar(L::kItemEmpty + s), Cfg::kItemTakers);
    }
    *abort_flag = 0;
    fence_barrier_init();
    fence_proxy_async_smem();
  }
  if (warp == Cfg::kProducerWarp && lane == 0) {
    prefetch_tmap(&tm_q);
    prefetch_tmap(&tm_ka);
    prefetch_tmap(&tm_va);
    prefetch_tmap(&tm_kb);
    prefetch_tmap(&tm_vb);
  }
  if (warp == Cfg::kMmaWarp) {
    tmem_alloc_pair(smem_u32(tmem_holder), kTmemCols);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // both CTAs' barriers exist before any cross-CTA arrival
  tc_fence_after();
  const Ctl ctl{abort_flag, args.timeout_ns, args.status};
  auto lbar = [&](int i) -> uint32_t { return mapa_shared(bar(i), 0); };  // leader's barrier i
  // Items reach the warps that walk them through a ring in the shared memory
  // of both CTAs: the leader's producer chooses item k, reads its Task and
  // writes it to slot k % kItemSlots of both, well before the item is needed.
  // Static order: item cluster + k * n_clusters.  With a work counter: item
  // `cluster` first, then the next of the list (atomic increment).  A slot is
  // reused once every taker is done with it (item_empty, on the leader).
  const bool dyn = args.work != nullptr;
  auto ring_slot = [&](int k) -> uint32_t {
    return base + L::kItemRing + 32u * static_cast<uint32_t>(k % tc2::kItemSlots);
  };
  auto ring_read = [&](int k) -> Task {
    const uint4 lo = ld_shared_v4(ring_slot(k)), hi = ld_shared_v4(ring_slot(k) + 16u);
    Task t;
    t.q_row0 = static_cast<int>(lo.x), t.q_rows = static_cast<int>(lo.y);
    t.a_row0 = static_cast<int>(lo.z), t.a_len = static_cast<int>(lo.w);
    t.b_row0 = static_cast<int>(hi.x), t.b_len = static_cast<int>(hi.y);
    t.head = static_cast<int>(hi.z), t.part = static_cast<int>(hi.w);
    return t;
  };
  // wait until item k is in the ring / this warp (one lane) is done with it
  auto ring_wait = [&](int k, int where) -> bool {
    const uint32_t full = bar(L::kItemFull + k % tc2::kItemSlots), parity = static_cast<uint32_t>(k / tc2::kItemSlots) & 1u;
    return leader ? wait_cl(full, parity, ctl, where) : wait_cl_acquire(full, parity, ctl, where);
  };
  // (release: the leader overwrites the slots of both CTAs once all have read them)
  auto ring_done = [&](int k) { mbar_arrive_release_cluster(lbar(L::kItemEmpty + k % tc2::kItemSlots)); };
  // item `it` of the work list
  auto fetch_item = [&](int it, Task& t, int& head) {
    if (spans.n == 0) {
      decode_item(args, it, t, head);
      return;
    }
    head = it / args.n_tasks;
    const int task = it - head * args.n_tasks;
    int i = 0;
    while (i + 1 < spans.n && spans.span[i + 1].task0 <= task) ++i;
    const int r = (task - spans.span[i].task0) * args.rows_per_task;
    t = Task{spans.span[i].row0 + r, min(args.rows_per_task, spans.span[i].len - r), spans.span[i].row0, spans.span[i].len,
             0, 0, head, 0};
  };
  // the leader's producer (one lane): item k, whose head is -1 when none is left
  auto publish = [&](int k, const Task& t, int head, int q_buf) {
    const uint4 lo = make_uint4(t.q_row0, t.q_rows | q_buf << 16, t.a_row0, t.a_len);  // (Q buffer: for the epilogue)
    const uint4 hi = make_uint4(t.b_row0, t.b_len, head, t.part);
    const uint32_t peer = mapa_shared(ring_slot(k), 1);
    st_shared_v4(ring_slot(k), lo);
    st_shared_v4(ring_slot(k) + 16u, hi);
    st_cluster_v4(peer, lo);
    st_cluster_v4(peer + 16u, hi);
    mbar_arrive(bar(L::kItemFull + k % tc2::kItemSlots));
    mbar_arrive_release_cluster(mapa_shared(bar(L::kItemFull + k % tc2::kItemSlots), 1));
  };
  // A cache's lists were written when it was created: the pair's first item need
  // not wait for the kernel before this one (0.7 us of the 2.5 us from the end of
  // that wait to the first MMA).
  if (args.static_list && leader && warp == Cfg::kProducerWarp && lane == 0) {
    Task t;
    int head;
    fetch_item(cluster, t, head);
    publish(0, t, head, 0);
  }
  // launched as a programmatic dependent of the previous kernel on the stream:
  // everything above overlaps its tail, nothing below reads memory before it
  // is complete; and the next kernel may start its CTAs (they wait likewise).
  // The second line must stay behind the first: the cache writes read the static
  // K and V and write the cache without a wait of their own, on the ground that
  // every CTA of the prefill has passed this one.
  grid_dependency_wait();
  if (threadIdx.x == 0) grid_launch_dependents();
  const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_holder, 0);
  if (warp == Cfg::kProducerWarp) {
    // ------------------------------------------------------------ producer (both CTAs)
    // This CTA's halves of the K and V tiles, and an item's Q rows just before
    // its first K tile.  Tiles are numbered t over all items; step t loads V_t
    // and K_t+2, which may belong to the next item, so that an item's first
    // loads are in flight before the item before it ends.
    if (lane == 0) {
      // Q, K and V tiles loaded (scales: si), from which the loads of
      // every slot follow, and the kind of the last load of each slot; the leader
      // arms every phase for both CTAs' bytes right before it issues its own half.
      // (Kept per slot, in arrays, they lay in local memory, at hundreds of cycles
      // an access: the E4M3 kernel's producer took 11000 cycles from its last load
      // to its end and held up the pair's: 21.4 us a step with 256 live and 256
      // cached rows and 4 heads, 9.7 without; 2 % with 4608 and 20480, 24 heads.)
      int nq = 0, nk = 0, nv = 0;
      uint32_t last8 = 0;
      const bool skip = leader && args.dbg_skip_first_load != 0;
      int si = 0;  // cached tiles whose scales went into the ring
      // The leader's choice of the next item, in three steps, each of whose
      // result is first used by the following one: its index, its Task, its
      // publication.
      int n_pub = args.static_list ? 1 : 0, pub_step = 0, pub_item = 0, pub_head = 0;
      bool pub_end = false;
      Task pub_task{};
      auto pub_advance = [&]() -> bool {
        if (pub_step == 0) {
          const int64_t it = !dyn ? static_cast<int64_t>(cluster) + static_cast<int64_t>(n_pub) * n_clusters
                             : n_pub == 0 ? static_cast<int64_t>(cluster)
                                          : static_cast<int64_t>(n_clusters) + atomicAdd(args.work, 1);
          pub_item = static_cast<int>(min(it, static_cast<int64_t>(args.n_items)));
        } else if (pub_step == 1) {
          if (pub_item < args.n_items)
            fetch_item(pub_item, pub_task, pub_head);
          else
            pub_head = -1;
        } else {
          const int k = n_pub, s = k % tc2::kItemSlots;
          if (k >= tc2::kItemSlots &&
              !wait_cl_acquire(bar(L::kItemEmpty + s), static_cast<uint32_t>(k / tc2::kItemSlots - 1) & 1u, ctl, 21))
            return false;
          publish(k, pub_task, pub_head, k & 1);
          pub_end = pub_head < 0;
          ++n_pub;
        }
        pub_step = pub_step == 2 ? 0 : pub_step + 1;
        return true;
      };
      // The K side: item k_item - 1, of which K tiles [0, kj) are loaded.
      Task kt{};
      int k_item = 0, kj = 0, k_na = 0, k_nkv = 0;
      bool k_end = false;
      // The V side: item v_item - 1, tile vj of it is next; G its group of S_1.
      Task vt{};
      int v_item = 0, vj = 0, v_na = 0, v_nkv = 0, G = 0;
      int done = -1;  // groups up to this one are known to be complete
#pragma unroll 1
      for (int t = -2;; ++t) {  // V_t (from t = 0 on), then K_t+2
        if (t >= 0) {
          if (vj == v_nkv) {  // the next item (the K side has passed it, so it is in the ring)
            G += v_nkv + 1;
            vt = ring_read(v_item);
            if (!leader) ring_done(v_item);
            ++v_item;
            if (vt.head < 0) break;
            v_nkv = tc2::n_key_tiles<kBN>(vt, v_na);
            vj = 0;
          }
          // The slots of V_t and K_t+2 are free once the P.V of tile t - kStages
          // and the S of tile t + 2 - kStages are complete.  Both hold after the
          // group below, which lies at most four groups before the first that
          // needs V_t: pair_done's phase of it cannot have passed unseen.
          const int g = kStages == 3 ? (vj == 0 ? G - 3 : G + vj - 2) : (kF8 && vj == 2 ? G : G + vj - 3);
          if (g > done) {
            if (!wait_one(bar(L::kPairDone + (g & 3)), group_parity(g), ctl, 2)) break;
            done = g;
          }
          const int slot = slot_of(t);
          const TileSrc vs = tc2::tile_src<kBN>(vt, v_na, vj);
          const bool v8 = kF8 && vs.in_b;
          const uint32_t vb = v8 ? kVHalf8 : kVHalf;
          const uint32_t dst = base + L::kRing + static_cast<uint32_t>(slot) * kStage + kKHalf;
          const uint32_t full = lbar(L::kVFull + slot);
          if (leader) mbar_arrive_expect_tx(bar(L::kVFull + slot), 2 * vb);
          ++nv;
          if (kF8) last8 = (last8 & ~(1u << (kStages + slot))) | (v8 ? 1u << (kStages + slot) : 0u);
          // head-dim columns [DG/2 r, DG/2 (r + 1)) of all kBN keys (E4M3: these
          // rows of V^T, all 128 keys)
          const int d0 = vt.head * DG + DG / 2 * static_cast<int>(rank);
          tma_load_2d_pair(dst, vs.in_b ? &tm_vb : &tm_va, full, v8 ? vs.row : d0, v8 ? d0 : vs.row);
          ++vj;
        }
        // the K side's next item, once its tiles are loaded; the leader chooses
        // the item after it from its last tiles on, one step per tile
        const bool need = !k_end && kj == k_nkv;
        bool more = leader && !pub_end && n_pub <= k_item && kj + 3 >= k_nkv;
        while (more) {
          if (!pub_advance()) goto producer_done;
          more = need && n_pub <= k_item;
        }
        if (need) {
          if (!ring_wait(k_item, 18)) goto producer_done;
          kt = ring_read(k_item);
          k_end = kt.head < 0;
          if (!k_end) {
            k_nkv = tc2::n_key_tiles<kBN>(kt, k_na);
            kj = 0;
            const int b = k_item & 1;  // its query rows into Q buffer k_item % 2
            const uint32_t n = static_cast<uint32_t>(k_item >> 1);
            ++k_item;
            if (!wait_one(bar(L::kQEmpty + b), (n & 1u) ^ 1u, ctl, 1)) goto producer_done;
            if (leader) mbar_arrive_expect_tx(bar(L::kQFull + b), 2 * kQBoxes * kBoxBytes);
            const uint32_t qfull = lbar(L::kQFull + b);
            for (int ch = 0; ch < kQBoxes; ++ch)
              tma_load_2d_pair(base + L::kQ + b * kQTile + ch * kBoxBytes, &tm_q, qfull, kt.head * DG + ch * 64,
                               kt.q_row0 + 128 * static_cast<int>(rank));
            ++nq;
          }
        }
        if (k_end) continue;
        const int slot = slot_of(t + 2);
        const TileSrc ks = tc2::tile_src<kBN>(kt, k_na, kj);
        const bool k8 = kF8 && ks.in_b;
        const uint32_t kb = k8 ? kKHalf8 : kKBox * kQBoxes;  // each CTA's bytes
        if (k8) {
          // this CTA's softmax warps read the cached tile's scales from ring slot
          // si % kScaleSlots; the slot's previous tile must have been read
          const int sl = si % tc2::kScaleSlots, use = si / tc2::kScaleSlots;
          if (use > 0 && !wait_one(bar(L::kScaleEmpty + sl), static_cast<uint32_t>(use - 1) & 1u, ctl, 16)) break;
          mbar_arrive_expect_tx(bar(L::kScaleFull + sl), 16u);
          bulk_load(base + L::kScales + 16u * static_cast<uint32_t>(sl),
                    args.b_scales + ((kt.b_row0 >> 7) + (kj - k_na)) * args.num_heads + kt.head, 16u,
                    bar(L::kScaleFull + sl));
          ++si;
        }
        ++kj;
        if (nk++ == 0 && skip) continue;  // fault injection: the leader never arms or loads this tile
        const uint32_t dst = base + L::kRing + static_cast<uint32_t>(slot) * kStage;
        const uint32_t full = lbar(L::kKFull + slot);
        if (leader) mbar_arrive_expect_tx(bar(L::kKFull + slot), 2 * kb);
        if (kF8) last8 = (last8 & ~(1u << slot)) | (k8 ? 1u << slot : 0u);
        // E4M3: keys [64 r, 64 r + 64), one box of 64 rows x 128 bytes; bf16: keys
        // [kBN/2 r, kBN/2 (r + 1)) of the tile, a box per 64 head-dim columns
        const void* map = ks.in_b ? &tm_kb : &tm_ka;
        const int row = ks.row + (kBN / 2) * static_cast<int>(rank);
        tma_load_2d_pair(dst, map, full, kt.head * DG, row);
        if (kQBoxes == 2 && !k8) tma_load_2d_pair(dst + kKBox, map, full, kt.head * DG + 64, row);
      }
    producer_done:
      // the scale ring's barriers are this CTA's own: the last load of each slot
#pragma unroll 1
      for (int s = 0; s < min(si, tc2::kScaleSlots); ++s)
        drain_one(bar(L::kScaleFull + s), static_cast<uint32_t>((si - 1 - s) / tc2::kScaleSlots) & 1u, args.timeout_ns);
      // K, V and Q loads of both CTAs complete on the leader's barriers: record
      // this CTA's loads in the leader's shared memory, where the leader
      // settles and drains them after the teardown's first cluster barrier
      const uint32_t rec = mapa_shared(base + L::kLoadRec + rank * (L::kRecWords * 4u), 0);
      st_cluster_u32(rec + 4u * L::kRecK, static_cast<uint32_t>(nk));
      st_cluster_u32(rec + 4u * L::kRecV, static_cast<uint32_t>(nv));
      st_cluster_u32(rec + 4u * L::kRecQ, static_cast<uint32_t>(nq));
      st_cluster_u32(rec + 4u * L::kRecLast8, last8);
      st_cluster_u32(rec + 4u * L::kRecSkipped, skip && nk > 0 ? 1u : 0u);
      // this cluster takes no more items
      if (dyn && leader) tc2::work_done(args.work, n_clusters);
    }
    __syncwarp();
  } else if (warp == Cfg::kMmaWarp) {
    // ------------------------------------------------------------ MMA warp (leader)
    if (leader) {
      // descriptors of ring slot 0 (slot s: + s * kStage / 16) and of Q buffer 0
      const uint64_t kd0 = sdesc_sw128(base + L::kRing, 16, 1024);
      const uint64_t vd0 = DG == 64 ? sdesc_sw64(base + L::kRing + kKHalf, kVHalf, 512)
                                    : sdesc_sw128(base + L::kRing + kKHalf, kVHalf, 1024);
      const uint64_t qdesc0 = sdesc_sw128(base + L::kQ, 16, 1024);
      // E4M3 operands: Q8 (128 rows x 128 B), K8 half (64 rows x 128 B), V^T half (64 d x 128 B); a
      // K = 32 step advances 32 bytes inside the swizzle atom
      const uint64_t q8d = sdesc_sw128(base + L::kQ8, 16, 1024);
      const uint64_t vd80 = sdesc_sw128(base + L::kRing + kKHalf, 16, 1024);
      // S step kk: A = Q (128-row boxes of 16 KB), B = this CTA's kBN / 2 keys (boxes of kBN / 2 rows)
      auto q_off = [](int kk) -> uint64_t {
        return (static_cast<uint32_t>(kk >> 2) * kBoxBytes + static_cast<uint32_t>(kk & 3) * 32u) >> 4;
      };
      auto k_off = [](int kk) -> uint64_t {
        return (static_cast<uint32_t>(kk >> 2) * kKBox + static_cast<uint32_t>(kk & 3) * 32u) >> 4;
      };
      bool issued = false;
      // Groups: the first item's S_0; then per item S_1 (group G), and P_j V_j
      // with S_j+2 (group G + 1 + j), where S_nkv is the next item's S_0 if that
      // may be issued ahead (inside this item).  The gate warp names the next
      // item at the handshake of that group, or of S_1 when nkv = 1 (item q in
      // entry q % 2: key tiles, 0 if none is left, those of range A, whether S_0
      // goes ahead).
      auto slot_k = [&](int t) -> uint64_t { return kd0 + static_cast<uint64_t>(slot_of(t)) * (kStage >> 4); };
      auto issue_s = [&](uint32_t d_s, uint64_t qd, uint64_t kd, bool s8) {
        if (kF8 && s8) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            tc2_mma_ss_f8(d_s, q8d + ((32u * kk) >> 4), kd + ((32u * kk) >> 4), kIdesc8, kk > 0 ? 1u : 0u);
        } else {
#pragma unroll
          for (int kk = 0; kk < DG / 16; ++kk)
            tc2_mma_ss(d_s, qd + q_off(kk), kd + k_off(kk), kIdescS, kk > 0 ? 1u : 0u);
        }
      };
      const volatile int* gate_item = reinterpret_cast<const volatile int*>(base_ptr + L::kGateItem);
      int nkv = 0, na = 0, ahead = 1, nkv_next = 0, na_next = 0, ahead_next = 1;
      int g = 0, t0 = 0, qi = -1;
      auto named = [&]() {
        const volatile int* n = gate_item + 4 * ((qi + 1) & 1);
        nkv_next = __shfl_sync(0xffffffffu, n[0], 0);
        if (kF8) na_next = __shfl_sync(0xffffffffu, n[1], 0), ahead_next = __shfl_sync(0xffffffffu, n[2], 0);
      };
      // steps without P.V: S_j+2 for j = -2 (the first item's S_0) and j = -1
      for (int j = -2;;) {
        if (bar_red_or(tc2::kGateBarrier, 64, false)) goto mma_done;
        issued = true;
        bool s_on = j + 2 < nkv, s_next = false;
        if (j + 2 == nkv) {
          named();
          s_on = s_next = nkv_next > 0 && ahead_next;
        }
        if (elect_one()) {
          tc_fence_after();
          const int q = qi + (s_next ? 1 : 0);
          const uint64_t qd = qdesc0 + ((static_cast<uint32_t>(q & 1) * kQTile) >> 4);
          if (kF8 && j == -1 && !ahead) {  // an S_0 of a cached tile, not issued ahead
            issue_s(tmem + kColS + static_cast<uint32_t>(t0 & 1) * kBN, qd, slot_k(t0), true);
            if (nkv == 1) tc2_commit_mc(bar(L::kQEmpty + (qi & 1)), 3);
          }
          if (s_on) {
            issue_s(tmem + kColS + static_cast<uint32_t>((t0 + j) & 1) * kBN, qd, slot_k(t0 + j + 2),
                    kF8 && !s_next && j + 2 >= na);
            if (s_next ? nkv_next == 1 : j + 3 == nkv) tc2_commit_mc(bar(L::kQEmpty + (q & 1)), 3);
          }
          tc2_commit_mc(bar(L::kPairDone + (g & 3)), 3);
        }
        __syncwarp();
        ++g;
        if (j == -2) goto next_item;
        {
          const uint64_t qd = qdesc0 + ((static_cast<uint32_t>(qi & 1) * kQTile) >> 4);
          // descriptors and buffers of step j, advanced after each step
          uint32_t vslot = static_cast<uint32_t>(slot_of(t0)), odd = static_cast<uint32_t>(t0 & 1);
          uint64_t vd = vd0 + static_cast<uint64_t>(vslot) * (kStage >> 4), kd = slot_k(t0 + 2);
          uint32_t a_p = tmem + kColP + odd * kPStride, d_s = tmem + kColS + odd * kBN, acc0 = 0;
          for (j = 0; j < nkv; ++j, ++g) {
            // P V of 32-key chunks [c0, c1) of P
            auto issue_pv = [&](int c0, int c1) {
              if (kF8 && j >= na) {
                const uint64_t vd8 = vd + (vd80 - vd0);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                  if (kk >= c0 && kk < c1)
                    tc2_mma_ts_f8(tmem + kColO, a_p + 8u * kk, vd8 + ((32u * kk) >> 4), kIdesc8, kk > 0 ? 1u : acc0);
              } else {
#pragma unroll
                for (int kk = 0; kk < kBN / 16; ++kk)
                  if (kk >= 2 * c0 && kk < 2 * c1)
                    tc2_mma_ts(tmem + kColO, a_p + 8u * kk, vd + ((kVStep * kk) >> 4), kIdescO, kk > 0 ? 1u : acc0);
              }
            };
            // S_j+2, of this item or the next
            auto issue_next = [&]() {
              if (!kF8 && j + 2 < nkv) {
                issue_s(d_s, qd, kd, false);
                if (j + 3 == nkv) tc2_commit_mc(bar(L::kQEmpty + (qi & 1)), 3);
                return;
              }
              const bool s_next = j + 2 == nkv;
              if (j + 2 < nkv || (s_next && nkv_next > 0 && ahead_next)) {
                const int q = qi + (s_next ? 1 : 0);
                issue_s(d_s, qdesc0 + ((static_cast<uint32_t>(q & 1) * kQTile) >> 4), kd, kF8 && !s_next && j + 2 >= na);
                if (s_next ? nkv_next == 1 : j + 3 == nkv) tc2_commit_mc(bar(L::kQEmpty + (q & 1)), 3);
              }
            };
            if (kPSplit > 0) {  // P's first chunks
              if (bar_red_or(tc2::kGateBarrier, 64, false)) goto mma_done;
              if (!Cfg::kPOverS && j + 2 == nkv) named();
              if (elect_one()) {
                tc_fence_after();
                issue_pv(0, kPSplit);
                if (!Cfg::kPOverS) issue_next();
              }
              __syncwarp();
            }
            if (bar_red_or(tc2::kGateBarrier, 64, false)) goto mma_done;
            if ((kPSplit == 0 || Cfg::kPOverS) && j + 2 == nkv) named();
            if (elect_one()) {
              tc_fence_after();
              // P.V first: with P over S, the S overwrites P_j
              issue_pv(kPSplit, kBN / 32);
              if (kPSplit == 0 || Cfg::kPOverS) issue_next();
              tc2_commit_mc(bar(L::kPairDone + (g & 3)), 3);
            }
            __syncwarp();
            // K_t+3's slot: kStages 3: V_t's; 4: the one before it
            kd = kStages == 3 ? kd0 + (vd - vd0) : kd == kd0 + 3ull * (kStage >> 4) ? kd0 : kd + (kStage >> 4);
            vd = vslot == kStages - 1 ? vd0 : vd + (kStage >> 4);
            vslot = vslot == kStages - 1 ? 0u : vslot + 1u;
            odd ^= 1u;
            a_p = tmem + kColP + odd * kPStride;
            d_s = tmem + kColS + odd * kBN;
            acc0 = 1;
          }
        }
      next_item:
        if (nkv_next == 0) break;
        t0 += nkv;
        ++qi;
        nkv = nkv_next, na = na_next, ahead = ahead_next;
        j = -1;
      }
    mma_done:
      // Every MMA must finish before TMEM is freed.  A commit covers the MMAs of the
      // thread that executes it, so the lane that elect.sync picks issues it too.
      __syncwarp();
      if (issued && elect_one()) {
        tc2_commit_mc(bar(L::kMmaDone), 1);
        drain_one(bar(L::kMmaDone), 0u, args.timeout_ns);
      }
    }
    __syncwarp();
  } else if (warp == Cfg::kGateWarp) {
    // ------------------------------------------------------------ gate warp (leader)
    // The same group sequence as the MMA warp; every wait is bounded, and a
    // failed wait is passed on through the handshake, after which both leave.
    if (leader) {
      volatile int* gate_item = reinterpret_cast<volatile int*>(base_ptr + L::kGateItem);
      auto wait_k = [&](int t) -> bool { return wait_cl_warp(bar(L::kKFull + slot_of(t)), slot_parity(t), ctl, 4); };
      // the steps of the MMA warp (see there)
      int nkv = -1, na = 0, nkv_next = 0, na_next = 0, q8i = 0;
#pragma unroll 1
      for (int t0 = 0, qi = -1, j = -2;;) {
        const int t = t0 + j;
        bool ok = true;
        bool k_wait = j + 2 < nkv;
        if (j + 2 == max(nkv, 0)) {  // name the next item
          const int k = qi + 1;
          ok = ok && __all_sync(0xffffffffu, ring_wait(k, 19));
          if (ok) {
            const Task tk = ring_read(k);
            __syncwarp();
            if (lane == 0) ring_done(k);
            nkv_next = tk.head < 0 ? 0 : tc2::n_key_tiles<kBN>(tk, na_next);
          }
          if (lane == 0) {
            volatile int* named = gate_item + 4 * ((qi + 1) & 1);
            named[0] = nkv_next;
            named[1] = na_next;
            // on an E4M3 cache an S_0 of a cached tile cannot go ahead: its Q
            // tile is written only after the item before it is done
            named[2] = kF8 && na_next == 0 ? 0 : 1;
          }
          __syncwarp();
          k_wait = nkv_next > 0;
          if (k_wait)
            ok = ok && wait_cl_warp(bar(L::kQFull + ((qi + 1) & 1)), static_cast<uint32_t>((qi + 1) >> 1) & 1u, ctl, 3);
        }
        if (k_wait) ok = ok && wait_k(t + 2);
        // the first cached tile's S also needs the E4M3 Q tile of both CTAs
        if (kF8 && nkv > na && (j + 2 == na || (j == -1 && na == 0))) {
          ok = ok && __all_sync(0xffffffffu, wait_cl_acquire(bar(L::kQ8Full), static_cast<uint32_t>(q8i) & 1u, ctl, 14));
          ++q8i;
        }
        if (j >= 0) {
          ok = ok && wait_cl_warp(bar(L::kVFull + slot_of(t)), slot_parity(t), ctl, 13);
          if constexpr (kPSplit > 0) {
            ok = ok && wait_cl_warp(bar(L::kPHalf + (t & 1)), static_cast<uint32_t>(t >> 1) & 1u, ctl, 22);
            if (bar_red_or(tc2::kGateBarrier, 64, !ok)) goto gate_done;
          }
          ok = ok && wait_cl_warp(bar(L::kPFull + (t & 1)), static_cast<uint32_t>(t >> 1) & 1u, ctl, 7);
        }
        if (bar_red_or(tc2::kGateBarrier, 64, !ok)) goto gate_done;
        if (++j >= nkv) {
          if (nkv_next == 0) break;
          t0 += max(nkv, 0);
          ++qi;
          nkv = nkv_next, na = na_next;
          j = -1;
        }
      }
    gate_done:;
    }
  } else {
    // ------------------------------------------------------------ softmax (both CTAs)
    // Warp w (0-3) owns rows 32 w .. 32 w + 31 of this CTA's 128 rows (its TMEM
    // lanes) and all kBN key columns.  (E4M3 kernel: two warps per row, each with
    // half the columns, took the same time: both read the whole row for its
    // maximum, and the two of a sub-partition take turns rather than overlap.)
    const int trow = warp * 32 + lane;                     // row within this CTA's 128 rows (= TMEM lane)
    const int prow = 128 * static_cast<int>(rank) + trow;  // row within the item
    const uint32_t lane_off = static_cast<uint32_t>(warp * 32) << 16;
    const float sl2 = args.scale_log2;
    const f32x2 sl2x2 = make_f32x2(sl2, sl2);
    const uint32_t lp = lbar(0);  // the leader's barriers (mapped once)
    int t = 0;     // tiles of earlier items
    int G = 1;     // the item's group of S_1 (S_j: ready after group G + j - 1; P_j V_j: group G + 1 + j)
    int si = 0;    // cached tiles read from the scale ring so far
    // wait until group g is complete (both CTAs see the multicast commit)
    auto wait_group = [&](int g, int where) -> bool {
      return wait_cl_warp(bar(L::kPairDone + (g & 3)), group_parity(g), ctl, where);
    };
    for (int k = 0;; ++k) {
      if (!__all_sync(0xffffffffu, ring_wait(k, 20))) goto softmax_done;
      const Task tk = ring_read(k);
      const int head = tk.head;
      if (head < 0) break;
      int na;
      const int nkv = tc2::n_key_tiles<kBN>(tk, na);
      const bool row_ok = prow < (tk.q_rows & 0xFFFF);
      const int64_t grow = static_cast<int64_t>(tk.q_row0) + prow;
      float m_run = 0.f, l_run = 0.f;
      // E4M3 cache: this row's query scale (folded into sl2) and the weight scale s_ref
      float c_row = sl2, s_ref = 1.f, l2_ref = 0.f;
      const int scale_row0 = kF8 ? (tk.b_row0 >> 7) * args.num_heads + head : 0;
      if (kF8 && nkv > na) {
        // quantise this thread's query row of this head into the E4M3 Q tile:
        // s = amax / 448, code = E4M3(x * (448 / amax)), round to nearest even
        uint4 raw[16];
        if (row_ok) {
          const uint4* src = reinterpret_cast<const uint4*>(args.q + grow * args.row_stride + static_cast<int64_t>(head) * D);
#pragma unroll
          for (int c = 0; c < 16; ++c) raw[c] = src[c];
        } else {
#pragma unroll
          for (int c = 0; c < 16; ++c) raw[c] = make_uint4(0, 0, 0, 0);
        }
        float amax = 0.f;
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          const uint32_t w4[4] = {raw[c].x, raw[c].y, raw[c].z, raw[c].w};
#pragma unroll
          for (int e = 0; e < 4; ++e)
            amax = fmax3(amax, fabsf(__uint_as_float(w4[e] << 16)), fabsf(__uint_as_float(w4[e] & 0xFFFF0000u)));
        }
        const float inv = amax > 0.f ? __fdiv_rn(448.f, amax) : 0.f;
        const uint32_t q8_row = base + L::kQ8 + static_cast<uint32_t>(trow) * 128u;
#pragma unroll
        for (int c = 0; c < 8; ++c) {  // 16 codes per 16-byte chunk, 128-byte swizzle
          uint32_t w[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const uint32_t x0 = e < 2 ? (&raw[2 * c].x)[2 * e] : (&raw[2 * c + 1].x)[2 * e - 4];
            const uint32_t x1 = e < 2 ? (&raw[2 * c].x)[2 * e + 1] : (&raw[2 * c + 1].x)[2 * e - 3];
            w[e] = pack_e4m3x4(__fmul_rn(__uint_as_float(x0 << 16), inv), __fmul_rn(__uint_as_float(x0 & 0xFFFF0000u), inv),
                               __fmul_rn(__uint_as_float(x1 << 16), inv), __fmul_rn(__uint_as_float(x1 & 0xFFFF0000u), inv));
          }
          st_shared_v4(q8_row + ((static_cast<uint32_t>(c) ^ static_cast<uint32_t>(trow & 7)) << 4),
                       make_uint4(w[0], w[1], w[2], w[3]));
        }
        // visible to the tensor core, then one arrival per warp of both CTAs
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive_release_cluster(mapa_shared(bar(L::kQ8Full), 0));
        c_row = sl2 * __fdiv_rn(amax, 448.f);
        const float4 sc0 = args.b_scales[scale_row0];
        s_ref = sc0.y > 0.f ? sc0.y : 1.f;
        l2_ref = sc0.y > 0.f ? sc0.z : 0.f;
      }
      bool ready = false;  // this tile's S was seen ready at the end of the tile before
      bool sc_ready = false;  // this cached tile's scales were read during the tile before
      float4 sc_next = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int j = 0; j < nkv; ++j, ++t) {
        const int b = t & 1;
        const int valid = (j < na ? tk.a_len : tk.b_len + na * kBN) - j * kBN;  // keys inside the range (>= kBN: all)
        // per-tile constants: u = c * s + shift is the shifted scaled score, the
        // weight written is exp2(u - m + wshift), the tile adds lscale * sum to l
        const bool t8 = kF8 && j >= na;
        float c_t = sl2, shift = 0.f, wshift = -l2_ref, lscale = s_ref;
        // S_j is ready and P buffer b is free once group G + j - 1 is complete
        // (one later for an S_0 that was not issued ahead)
        if (!ready && !wait_group(G + j - (kF8 && j == 0 && na == 0 ? 0 : 1), 8)) goto softmax_done;
        tc_fence_after();
        const uint32_t t_s = tmem + lane_off + kColS + static_cast<uint32_t>(kBN) * b;
        // Keys past the end of the range: -inf, written over their scores in
        // tensor memory (a tile with such keys is rare; selects over the loaded
        // columns were 8 KB of code inside the loop, see wait_more).
        if (valid < kBN) {
          uint32_t inf[16];
#pragma unroll
          for (int c = 0; c < 16; ++c) inf[c] = 0xFF800000u;
          int c = valid;
#pragma unroll 1
          for (; c & 15; ++c) tmem_st1(t_s + static_cast<uint32_t>(c), 0xFF800000u);
#pragma unroll 1
          for (; c < kBN; c += 16) tmem_st16(t_s + static_cast<uint32_t>(c), inf);
          tmem_wait_st();
        }
        // this thread's columns of S in s[] and the row's maximum in m_raw.  The
        // loads deliver the maximum of each 32 columns (tcgen05.ld.red).  The
        // maximum sits on the latency loop that bounds the kernel (S ready ->
        // softmax -> P -> next S): with 96 max instructions per 192-key tile it
        // took about 190 of 2142 cycles, and the step at 4608 live and 20480 cached
        // rows, 24 heads, 7 % longer (same bits).
        float s[kBN];
        float m_raw;
        {
          constexpr int kChains = kBN / 32;
          uint32_t r[kChains][32];
          float mx[kChains];
#pragma unroll
          for (int k = 0; k < kChains; ++k) tmem_ld32_max(t_s + 32u * k, r[k], mx[k]);
          if (t8) {
            // the producer's ring of tile scales (no global access here: an
            // ordinary load still in flight would hold up the next P arrival)
            const int sl = si % tc2::kScaleSlots;
            if (!sc_ready) {
              if (!wait_warp(bar(L::kScaleFull + sl), static_cast<uint32_t>(si / tc2::kScaleSlots) & 1u, ctl, 17))
                goto softmax_done;
              sc_next = ld_shared_f4(base + L::kScales + 16u * static_cast<uint32_t>(sl));
            }
            const float4 sc = sc_next;
            __syncwarp();
            if (lane == 0) mbar_arrive(bar(L::kScaleEmpty + sl));
            ++si;
            c_t = fmaxf(c_row * sc.x, 1e-30f);
            // delta = log2(s_V / s_ref); an all-zero V tile (s_V = 0) takes delta = 0
            const bool nz = sc.y > 0.f;
            shift = nz ? sc.z - l2_ref : 0.f;
            wshift = 0.f;
            lscale = nz ? s_ref * sc.w : 1.f;  // 2^-delta
          }
#pragma unroll
          for (int k = 0; k < kChains; ++k) tmem_wait_ld(r[k], mx[k]);
#pragma unroll
          for (int k = 0; k < kChains; ++k)
#pragma unroll
            for (int c = 0; c < 32; ++c) s[32 * k + c] = __uint_as_float(r[k][c]);
          if constexpr (kChains == 6)
            m_raw = fmaxf(fmax3(mx[0], mx[1], mx[2]), fmax3(mx[3], mx[4], mx[5]));
          else
            m_raw = fmax3(mx[0], mx[1], fmaxf(mx[2], mx[3]));
        }
        // rescale this row's O columns and l for a new running maximum m_new (O
        // must first hold P_j-1 V_j-1: group G + j complete)
        auto rescale = [&](float m_new) -> bool {
          if (!wait_group(G + j, 9)) return false;
          tc_fence_after();
          const float alpha = ex2_approx(m_run - m_new);
          const f32x2 alpha2 = make_f32x2(alpha, alpha);
          m_run = m_new;
          l_run *= alpha;
          const uint32_t t_o = tmem + lane_off + kColO;
          // (rolled in the E4M3 kernel, whose tile loop holds the code of both kinds
          // of tile; rolled, by two or unrolled, both kernels take the same time within
          // 0.7 %)
          constexpr int kUnroll = kF8 ? 1 : DG / 16;
#pragma unroll kUnroll
          for (int cc = 0; cc < DG / 16; ++cc) {
            uint32_t o[16];
            tmem_ld16(t_o + 16u * cc, o);
            tmem_wait_ld(o);
#pragma unroll
            for (int c = 0; c < 16; c += 2) {
              f32x2 v = mul_f32x2(make_f32x2(__uint_as_float(o[c]), __uint_as_float(o[c + 1])), alpha2);
              float lo, hi;
              split_f32x2(v, lo, hi);
              o[c] = __float_as_uint(lo);
              o[c + 1] = __float_as_uint(hi);
            }
            tmem_st16(t_o + 16u * cc, o);
          }
          return true;
        };
        // P = exp2(c * S + shift - m) into P buffer b: bf16 pairs (32 keys = 16
        // columns at a time), or for a cached tile E4M3 quads (32 keys = 8
        // columns); returns this thread's sum of the weights written
        const uint32_t t_p = tmem + lane_off + kColP + kPStride * b;
        auto p_arrive = [&](int which) {  // this warp's P so far is in TMEM
          tmem_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(lp + 8u * static_cast<uint32_t>(which));
        };
        auto write_p = [&]() -> float {
          const float bias = (kF8 ? shift + wshift : 0.f) - m_run;
          const f32x2 negm = make_f32x2(bias, bias);
          const f32x2 c2 = kF8 ? make_f32x2(c_t, c_t) : sl2x2;
          f32x2 lacc[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) lacc[i] = make_f32x2(0.f, 0.f);
          if (t8) {
            // the next tile's scales are looked for and read on the way (waited for
            // and read at its start they took 345 cycles of a tile's 1490, 5 % of a
            // step)
            const int sl = si % tc2::kScaleSlots;
            bool found = false;
#pragma unroll
            for (int k = 0; k < kBN / 32; ++k) {
              if (k == 0)
                found = j + 1 < nkv &&
                        mbar_test_wait(bar(L::kScaleFull + sl), static_cast<uint32_t>(si / tc2::kScaleSlots) & 1u);
              if (k == 2 && found) sc_next = ld_shared_f4(base + L::kScales + 16u * static_cast<uint32_t>(sl));
              uint32_t pk[8];
#pragma unroll
              for (int c = 0; c < 8; ++c) {
                const f32x2 e01 = fma_f32x2(make_f32x2(s[32 * k + 4 * c], s[32 * k + 4 * c + 1]), c2, negm);
                const f32x2 e23 = fma_f32x2(make_f32x2(s[32 * k + 4 * c + 2], s[32 * k + 4 * c + 3]), c2, negm);
                float e0, e1, e2, e3;
                split_f32x2(e01, e0, e1);
                split_f32x2(e23, e2, e3);
                const float x0 = ex2_approx(e0), x1 = ex2_approx(e1), x2 = ex2_approx(e2), x3 = ex2_approx(e3);
                lacc[(2 * c) & 3] = add_f32x2(lacc[(2 * c) & 3], make_f32x2(x0, x1));
                lacc[(2 * c + 1) & 3] = add_f32x2(lacc[(2 * c + 1) & 3], make_f32x2(x2, x3));
                pk[c] = pack_e4m3x4(x0, x1, x2, x3);
              }
              tmem_st8(t_p + 8u * k, pk);
              if (k == kPSplit - 1) p_arrive(L::kPHalf + b);
            }
            sc_ready = __all_sync(0xffffffffu, found);
          } else {
#pragma unroll
            for (int k = 0; k < kBN / 32; ++k) {
              uint32_t pk[16];
#pragma unroll
              for (int c = 0; c < 16; ++c) {
                const f32x2 e = fma_f32x2(make_f32x2(s[32 * k + 2 * c], s[32 * k + 2 * c + 1]), c2, negm);
                float e0, e1;
                split_f32x2(e, e0, e1);
                const float x = ex2_approx(e0), y = ex2_approx(e1);
                lacc[c & 3] = add_f32x2(lacc[c & 3], make_f32x2(x, y));
                pk[c] = pack_bf16x2(x, y);
              }
              tmem_st16(t_p + 16u * k, pk);
              if (k == kPSplit - 1) p_arrive(L::kPHalf + b);
            }
          }
          const f32x2 l2 = add_f32x2(add_f32x2(lacc[0], lacc[1]), add_f32x2(lacc[2], lacc[3]));
          float lo, hi;
          split_f32x2(l2, lo, hi);
          return lo + hi;
        };
        // running maximum from the row maximum (lazy: moves only when a tile's
        // maximum exceeds it by more than 2^8)
        const float m_tile = fmaf(m_raw, c_t, shift);
        if (j == 0) {
          m_run = m_tile;
        } else if (__any_sync(0xffffffffu, m_tile > m_run + 8.0f)) {
          if (!rescale(fmaxf(m_run, m_tile))) goto softmax_done;
        }
        const float l_tile = write_p();
        l_run += kF8 ? l_tile * lscale : l_tile;
        // a look at the next S, whose latency passes beside the stores of P
        const bool next_done = j + 1 < nkv && mbar_test_wait(bar(L::kPairDone + ((G + j) & 3)), group_parity(G + j));
        p_arrive(L::kPFull + b);
        ready = __all_sync(0xffffffffu, next_done);
      }
      {
        // the row's place is read again from the item ring, so that it is not
        // kept live through the tile loop
        const Task et = ring_read(k);
        const int e_rows = et.q_rows & 0xFFFF, e_qb = et.q_rows >> 16, e_head = et.head, e_part = et.part;
        const bool e_row_ok = prow < e_rows;
        const int64_t e_grow = static_cast<int64_t>(et.q_row0) + prow;
        __syncwarp();
        if (lane == 0) ring_done(k);
        if (!wait_group(G + nkv, 10)) goto softmax_done;  // the item's last group
        tc_fence_after();
        const float inv_l = kF8 ? s_ref / l_run : 1.0f / l_run;
        const uint32_t t_o = tmem + lane_off + kColO;
        if (e_part > 0) {
          // a part of a split item: O / l in fp32 and m + log l to its workspace
          // slot, [D / 4][rows_per_task] float4, so that a warp's 32 rows of four
          // columns are one run of 512 bytes
          const int64_t slot = e_part - 1;
          float4* dst = reinterpret_cast<float4*>(args.part_o) + slot * (DG / 4) * args.rows_per_task + prow;
#pragma unroll
          for (int cc = 0; cc < DG / 32; ++cc) {
            uint32_t o[32];
            tmem_ld32(t_o + 32u * cc, o);
            tmem_wait_ld(o);
            if (e_row_ok) {
#pragma unroll
              for (int c = 0; c < 8; ++c)
                dst[(8 * cc + c) * args.rows_per_task] =
                    make_float4(__uint_as_float(o[4 * c]) * inv_l, __uint_as_float(o[4 * c + 1]) * inv_l,
                                __uint_as_float(o[4 * c + 2]) * inv_l, __uint_as_float(o[4 * c + 3]) * inv_l);
            }
          }
          tc_fence_before();
          if (e_row_ok)
            args.part_lse[slot * args.rows_per_task + prow] = (m_run + log2f(l_run)) * 0.69314718055994530942f;
        } else {
          // O / l as bf16 through the item's Q buffer, which its S no longer
          // reads: this thread's row in 16-byte chunks (swizzled), then whole
          // rows to global memory, kNC lanes each.  Stored straight from the
          // registers a warp's 16 bytes per row touch 32 lines per instruction,
          // 2048 cycles of the SM's load/store unit per item, which the next
          // item's softmax waited for.
          constexpr int kNC = DG / 8;              // chunks of a row
          constexpr uint32_t kPitch = 16u * kNC;  // bytes of a staged row
          const uint32_t stage = base + L::kQ + static_cast<uint32_t>(e_qb) * kQTile + static_cast<uint32_t>(warp * 32) * kPitch;
#pragma unroll
          for (int cc = 0; cc < DG / 32; ++cc) {
            uint32_t o[32];
            tmem_ld32(t_o + 32u * cc, o);
            tmem_wait_ld(o);
#pragma unroll
            for (int c = 0; c < 4; ++c) {
              uint32_t w[4];
#pragma unroll
              for (int e = 0; e < 4; ++e)
                w[e] = pack_bf16x2(__uint_as_float(o[8 * c + 2 * e]) * inv_l, __uint_as_float(o[8 * c + 2 * e + 1]) * inv_l);
              st_shared_v4(stage + static_cast<uint32_t>(lane) * kPitch +
                               ((static_cast<uint32_t>(4 * cc + c) ^ static_cast<uint32_t>(lane & (kNC - 1))) << 4),
                           make_uint4(w[0], w[1], w[2], w[3]));
            }
          }
          // (the next arrival on p_full, after the next tile's P, tells the MMA
          // thread that these O reads are done)
          tc_fence_before();
          __syncwarp();
          constexpr int kRows = 32 / kNC;  // rows per instruction
          const int r0 = lane / kNC, ch = lane % kNC;
          const int first = 128 * static_cast<int>(rank) + warp * 32;  // the warp's first row in the item
          __nv_bfloat16* dst = args.out + (static_cast<int64_t>(et.q_row0) + first) * args.row_stride +
                               static_cast<int64_t>(e_head) * DG + 8 * ch;
#pragma unroll 4
          for (int i = 0; i < kNC; ++i) {
            const int r = i * kRows + r0;
            const uint4 v = ld_shared_v4(stage + static_cast<uint32_t>(r) * kPitch +
                                         (static_cast<uint32_t>(ch ^ (r & (kNC - 1))) << 4));
            if (first + r < e_rows) *reinterpret_cast<uint4*>(dst + r * args.row_stride) = v;
          }
          if (e_row_ok && args.lse)
            args.lse[e_grow * args.num_heads + e_head] = (m_run + log2f(l_run)) * 0.69314718055994530942f;
        }
        // the Q buffer is free for the TMA loads of the item after the next
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar(L::kQEmpty + e_qb));
      }
      G += nkv + 1;
    }
  softmax_done:;
  }

  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) st_cluster_u32(mapa_shared(base + L::kPeerAbort, rank ^ 1u), static_cast<uint32_t>(*abort_flag));
  // the pair's MMAs and TMEM reads are over in both CTAs, both producers' load
  // records are in the leader's shared memory, and each CTA knows whether the
  // other one gave up
  cluster_sync();
  if (warp == Cfg::kMmaWarp) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, kTmemCols);
  }
  // Every load has landed when neither CTA gave up: each was waited for before
  // the MMAs that read it.  (Settling them all the same, with a second barrier
  // behind, and resetting the work counter after it took 1 us of the 3 us
  // between the last MMA and the exit.)
  if (*abort_flag == 0 && *reinterpret_cast<const volatile int*>(base_ptr + L::kPeerAbort) == 0) return;
  if (leader && warp == Cfg::kProducerWarp && lane == 0) {
    // Every K, V and Q load of either CTA must land before that CTA exits.
    // The leader arms a phase for both halves before it issues its own, and
    // each CTA issues its half after the same wait; after an abort the two can
    // differ by one phase.  A phase the follower loaded but the leader never
    // armed is armed now for the follower's bytes; a phase the leader armed
    // whose follower half was never issued has those bytes counted as
    // arrived.  Then the last phase of every barrier is drained (bounded).
    const volatile uint32_t* rec = reinterpret_cast<const volatile uint32_t*>(base_ptr + L::kLoadRec);
    const volatile uint32_t* peer = rec + L::kRecWords;
    // missing: the follower's bytes of the leader's last phase; loaded: the
    // follower's own bytes of its last load
    auto settle = [&](uint32_t b, int mine, int theirs, uint32_t missing, uint32_t loaded) {
      if (theirs == mine + 1) {
        mbar_arrive_expect_tx(b, loaded);
        mine = theirs;
      } else if (mine == theirs + 1 && missing > 0) {
        mbar_complete_tx(b, missing);
      }
      if (mine > 0) drain_one(b, static_cast<uint32_t>(mine - 1) & 1u, args.timeout_ns);
    };
    // loads of slot s of n, among `tiles` tiles
    auto loads = [](uint32_t tiles, int s, int n) { return (static_cast<int>(tiles) - s + n - 1) / n; };
    auto bytes = [&](const volatile uint32_t* r, int i, uint32_t full, uint32_t cached) {
      return kF8 && (r[L::kRecLast8] >> i & 1u) ? cached : full;
    };
#pragma unroll 1
    for (int s = 0; s < kStages; ++s) {
      settle(bar(L::kKFull + s), loads(rec[L::kRecK], s, kStages) - (s == 0 && rec[L::kRecSkipped] ? 1 : 0),
             loads(peer[L::kRecK], s, kStages), bytes(rec, s, kKBox * kQBoxes, kKHalf8),
             bytes(peer, s, kKBox * kQBoxes, kKHalf8));
      settle(bar(L::kVFull + s), loads(rec[L::kRecV], s, kStages), loads(peer[L::kRecV], s, kStages),
             bytes(rec, kStages + s, kVHalf, kVHalf8), bytes(peer, kStages + s, kVHalf, kVHalf8));
    }
    constexpr uint32_t kQCta = kQBoxes * kBoxBytes;  // each CTA's bytes of a Q load
    for (int b = 0; b < 2; ++b)
      settle(bar(L::kQFull + b), loads(rec[L::kRecQ], b, 2), loads(peer[L::kRecQ], b, 2), kQCta, kQCta);
  }
  // the follower leaves only once the leader has seen every load of the pair land
  cluster_sync();
}

}  // namespace rc
