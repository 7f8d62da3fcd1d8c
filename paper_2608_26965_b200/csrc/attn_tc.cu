// Block-sparse attention with striped mean-compensation on the sm_100a tensor
// cores (eq. 2 over the selected clusters; Appendix A: an excluded cluster
// enters through its centroid key/value with weight |c| exp(q . kbar / sqrt(d))).
//
// Persistent CTAs, one per SM, each walking over tiles of 128 query rows (one query
// cluster, half of a 256-row one, or a 64-row one).  Keys are
// consumed in steps of 128:
//     S   = Q K_s^T        tcgen05.mma, Q and K from shared memory (K-major)
//     P   = exp2(S c - m)  one query row per thread; P is written back over S as
//                          packed bf16; row sums in fp32 registers
//     O  += P V_s          tcgen05.mma, P from tensor memory, V from shared memory (MN-major)
// A softmax warp needs about twice the time of its exponentials for a step (latencies of
// tensor-memory loads, barriers, conversions), so the steps go round three groups of
// four softmax warps, each with a score buffer of its own (3 x 128 + D columns of
// tensor memory), and the tensor core works up to three steps ahead: neither the
// products nor the hand-offs between the units are on a softmax warp's path.  Roles:
// warp 0 loads Q and K, warp 3 V (TMA, 128-byte swizzle, 64-column panels), one thread of warp 1
// issues all products, warp 2 walks over tiles and block lists and writes a descriptor
// per step (rows to load, masks, additive terms) into a ring, warps 4-15 are the
// softmax groups.  The roles run ahead of one another across tiles, so that the start
// of a tile hides behind the end of the one before.
// Query clusters of 64 rows go two to a tile, neighbours, one in either half (siblings of the split tree: their lists
// have 64 to 86 % of their entries in common on the inputs measured).  A key cluster that both lists hold is taken once, by all rows;
// one that a single list holds by the rows of that half, next to one of the other list (the other probabilities of a row
// are stored as zeros), so that all four softmax warps of a group have work.  The warp that writes the step
// descriptors has more to do then, and writes four at a time: one by one it was what the others waited for (247 us, and a wait of
// 400 cycles put into each step cost 46 us; now 4).  Where pairs would take no fewer rounds of tiles, the rows of one cluster
// stand in both halves of a tile, which divide the keys of a step between them and merge their outputs (12 heads of
// 16,385 rows, 33 of 257 clusters 345 us in this form, 221 in pairs, 12 heads of 30,592 rows 667 and 454; 4 heads of 512 x 131,072
// rows 188, and 236 in pairs).  Each form has instances of its own: in one kernel with the pairs' code, which a small
// call fetches and walks through once, 2 heads of 1,000 rows with lists of one cluster took 14.2 us at d = 64 and 16.3 at
// d = 128, 8 heads with 12 of 16 clusters 16.8; now 12.2, 13.6 and 15.4.
// (0 x inf is NaN: where a key cluster of one list holds an infinite value, outputs that are not numbers send the
// query cluster to the second pass.)
// All roles run at the same time on one SM and have to fit its instruction cache
// together: with the loops of the single-warp roles unrolled (105 KB of code) the same
// kernel took 1.40 ms where it now takes 0.72 (2 x 16 heads of 20,000 rows, d = 128, 10
// clusters of 256 kept), so loops stay rolled unless a step is shorter for it.
// What bounds it: at d = 128 no unit by itself.  A step brings 64 KB through L2, since every tile
// loads its lists for itself, and takes 0.945 us: 10.2 TB/s over the SMs of the
// 14.6 that plain bulk loads of L2-resident data reach (0.66 us),
// with the tensor pipe 63 % and the exponentials 62 % busy; the rest are hand-offs, and launches in a row
// run at the power limit (717 us alone, 809 behind one another).  At d = 64 the
// exponentials (1,024 of 1,270 cycles per step) and the hand-offs.  Measured against the kernel before (two CTAs per SM at d = 128,
// four at d = 64, half-steps of 64 keys in one chain per CTA): 40 heads of 32,760 rows,
// d = 128, 32 of 256 clusters kept 2.91 -> 2.40 ms; 8 heads of 16,384 x 131,072, d = 64,
// 128 of 1,024 kept 0.88 -> 0.76.
//
// The softmax keeps a reference m per row instead of the exact running maximum: it is
// measured on a row's first step and raised (by an integer) when a sum of 32
// probabilities exceeded 2^32, at the group's next step; the reference of every step is
// handed from group to group through shared memory, and the group that raises it
// rescales O in tensor memory itself.  A climb beyond 2^96 inside the steps in
// flight marks the tile for the second pass of the fp32 kernel.
// After the selected clusters the key centroids are streamed as extra keys, 64 per
// step: their tile holds bf16 hi parts in rows 0-63 and lo parts in rows 64-127, whose
// scores are added when they are read, with an additive term ln|c|, selected clusters
// masked; values are the value centroids.  Block lists may be ragged (a length per
// query cluster); tiles are handed out by a counter.
// Indices that come from the caller (block lists, list lengths, perm_q) are range-
// checked before use: a bad one sets CA_ERR_BAD_INDEX in the status word and the
// access is skipped (the cluster is masked, the row is not written).
#include <type_traits>

#include "kernels.h"
#include "tc_ptx.cuh"

namespace ca {

using namespace ptx;

constexpr int kGroups = 3;                 // softmax groups of 128 threads, score buffers
constexpr int kTcThreads = 128 + kGroups * 128;
constexpr int kTile = 128;                 // query rows per tile, key rows per step
constexpr int kCen = 64;                   // key centroids per step
constexpr int kParts = 6;                  // steps s - 2 .. s + 3 can have row sums on their way while step s ends a tile
constexpr int kQueue = 64;                 // list entries of a pair of 64-row query clusters in waiting
constexpr int kMergeInts = 18;             // row pitch of the hand-over between the halves of a 64-row query cluster
// first rows of a step's boxes (key clusters of 16 rows: eight boxes), of its value centroids, of Q
constexpr int kRowCenV = 8, kRowQ = 9, kRowInts = 12;
// A reference is raised when a sum of 32 probabilities exceeds 2^32: P is bf16, O and l are fp32, so
// probabilities far above 1 cost no precision, and the climbs that remain below the limit
// (nearly all) need no rescaling of O, which stalls all three groups for some 2,000 cycles.
constexpr float kRescaleThreshold = 32.0f;  // log2 units
constexpr float kSumLimit = 4294967296.0f;  // 2^kRescaleThreshold
constexpr float kDangerSum = 7.9228163e28f;  // 2^96

// flags of a step descriptor
constexpr int kFMasked = 1, kFCentroid = 2, kFFirst = 4, kFLast = 8, kFStop = 16;
// pairs of 64-row query clusters: the upper half of the rows takes keys 0-63 of the step and the lower half keys
// 64-127, or only one of the halves takes part
constexpr int kFSplit = 32, kFUpper = 64, kFLower = 128;
constexpr int kFIndexShift = 8, kFRestShift = 12;   // min(15, index in the tile), min(15, steps after it)
constexpr int kFSingle = 1 << 16;          // the tile holds one cluster

// F8: queries, keys and key centroids arrive as E4M3 codes (one byte per element: a 128-byte row
// of a panel holds 128 of them) and Q K^T runs as kind::f8f6f4 products; values stay bf16.
// MODE: how query clusters stand in tiles of 128 rows: a cluster of 128 (half of one of 256) in one; two clusters of 64 in one, or
// in both halves of one
constexpr int kWhole = 0, kPairs = 1, kTwice = 2;
template <int D, bool F8, int MODE>
struct TcCfg {
  static constexpr int RING = MODE != kPairs ? 8 : D == 64 ? 16 : 12;   // step descriptors in flight (pairs: four are written at a time)
  static constexpr int PANELS = D / 64;                      // value panels (bf16: 64 elements per 128-byte row)
  static constexpr int QK_PANELS = F8 ? D / 128 : D / 64;    // query / key panels
  static constexpr int QK_PANEL_COLS = F8 ? 128 : 64;        // elements per panel row
  static constexpr int QK_KSTEP = F8 ? 32 : 16;              // elements per tensor-core instruction (32 bytes)
  static constexpr int PANEL_BYTES = kTile * 128;            // 128 rows x 128 bytes
  static constexpr int QK_BYTES = QK_PANELS * PANEL_BYTES;   // a query tile, a key tile
  static constexpr int V_BYTES = PANELS * PANEL_BYTES;       // a value tile
  static constexpr uint32_t TMEM_COLS = 512;                 // kGroups x 128 score columns (P over 64 of them), D of O
  static constexpr int NK = kGroups;                         // key tiles in shared memory: one per score buffer
  static constexpr int NV = D == 64 ? 4 : F8 ? 3 : 2;        // value tiles
  // Query tiles: two where there is room, so that the scores of a tile do not wait until its queries have come behind the last
  // scores of the one before (with four value tiles for three, 8 heads of 16,384 x 131,072 rows 788 -> 758 us)
  static constexpr int NQ = (D == 64 || F8) ? 2 : 1;
  // shared memory layout (offsets from a 1024-byte aligned base)
  static constexpr int OFF_Q = 0;
  static constexpr int OFF_K = OFF_Q + NQ * QK_BYTES;
  static constexpr int OFF_V = OFF_K + NK * QK_BYTES;
  static constexpr int OFF_BIAS = OFF_V + NV * V_BYTES;                  // [RING][128] floats
  static constexpr int OFF_LPART = OFF_BIAS + RING * kTile * 4;         // [kParts steps][128 rows] {row sum, reference}
  static constexpr int OFF_QUEUE = OFF_LPART + kParts * kTile * 8;       // pairs: [3][kQueue] {first key row, rows, scale of the keys}
  static constexpr int OFF_MERGE = OFF_QUEUE;                            // twice: [64 rows][kMergeInts] 16 columns of O, sum, reference
  static constexpr int OFF_REF = OFF_QUEUE + (MODE == kPairs ? 3 * kQueue * 16 : MODE == kTwice ? 64 * kMergeInts * 4 : 0);   // [128 rows] {reference, step}
  static constexpr int OFF_ROWS = OFF_REF + kTile * 8;                   // [RING][kRowInts]
  static constexpr int OFF_TILE = OFF_ROWS + RING * kRowInts * 4;       // [RING] head, first position, redo word, tile
  static constexpr int OFF_FLAGS = OFF_TILE + RING * 16;
  static constexpr int OFF_SCALE = OFF_FLAGS + RING * 4;                // [RING][2] scales of the keys (F8)
  static constexpr int OFF_BAR = OFF_SCALE + RING * 8;
  static constexpr int NUM_BARS = 1 + NQ + 4 + 2 * kGroups + 2 * RING + NK + 2 * NV + (MODE == kTwice ? 4 : 0);
  static constexpr int OFF_MISC = OFF_BAR + NUM_BARS * 8;                // tmem base, abort flag, redo counts x 4
  static constexpr int OFF_BITMAP = OFF_MISC + 32;
  static_assert(OFF_TILE % 16 == 0 && OFF_BAR % 8 == 0 && OFF_MISC % 8 == 0, "alignment");
};

struct TcParams {
  const int32_t* count_k;
  const int32_t* block_idx;
  const int32_t* keep_count;      // per query cluster list length, or null: every list holds `keep` entries
  const int32_t* perm_q;
  __nv_bfloat16* O;
  float* lse;
  int* status;
  int* next_tile;                 // counter that hands out tiles, zero at the start
  int32_t* redo;                  // [B*H, n_qc, 2] per tile: scores left the range of the fast softmax
  int n_q, n_k, c_q, c_k, keep, list_stride, n_qc, n_kc, cen_tiles, compensate, bitmap_words, n_tiles;
  float scale_log2;
  // quantised Q K^T: de-quantisation scales of the query rows [B*H*n_qc*c_q], of the key clusters
  // [B*H*n_kc] and of the runs of 64 key centroids [B*H*cen_tiles]; null otherwise
  const float* q_scale;
  const float* k_scale;
  const float* c_scale;
  long long wait_limit;           // SM cycles after which a barrier wait gives up (CA_ERR_TIMEOUT)
  int skip_key_load;              // diagnostic hook: the loader leaves out the keys of the step with these 64 (-1: none)
};

constexpr int kErrBadIndex = 6;   // CA_ERR_BAD_INDEX
constexpr int kBitmapWords = 4096;        // of a list: 131,072 key clusters (d = 128 leaves 17 KB)
constexpr int kPairBitmapWords = 2048;    // of each list of a pair

// key rows of the selected clusters are consumed in tiles of 128 rows
__host__ __device__ inline int selected_tiles(int keep, int c_k) {
  return c_k >= kTile ? keep * (c_k / kTile) : (keep * c_k + kTile - 1) / kTile;
}

// A value that all lanes of a (converged) warp hold, made known as such to the compiler: branches on it
// and addresses from it stay in the uniform datapath.
__device__ __forceinline__ int warp_uniform(int x) { return __shfl_sync(0xffffffffu, x, 0); }

template <int D, bool F8, int MODE>
__global__ void __launch_bounds__(kTcThreads, 1)
attn_tc_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
               const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_ck,
               const __grid_constant__ CUtensorMap tm_cv, const TcParams prm) {
  wait_for_previous();
  using C = TcCfg<D, F8, MODE>;
  extern __shared__ unsigned char smem_unaligned[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_unaligned) + 1023) & ~uintptr_t(1023));
  const uint32_t s_base = smem_u32(smem);
  const uint32_t s_q = s_base + C::OFF_Q, s_k = s_base + C::OFF_K, s_v = s_base + C::OFF_V;
  float* bias = reinterpret_cast<float*>(smem + C::OFF_BIAS);
  float2* lpart = reinterpret_cast<float2*>(smem + C::OFF_LPART);
  const uint32_t s_ref = s_base + C::OFF_REF;
  int* st_rows = reinterpret_cast<int*>(smem + C::OFF_ROWS);
  int4* st_tile = reinterpret_cast<int4*>(smem + C::OFF_TILE);
  int* st_flags = reinterpret_cast<int*>(smem + C::OFF_FLAGS);
  float* st_scale = reinterpret_cast<float*>(smem + C::OFF_SCALE);
  const uint32_t bar0 = s_base + C::OFF_BAR;
  const uint32_t b_o_empty = bar0;
  auto b_q_empty = [&](int t) { return bar0 + 8 + 8 * (t % C::NQ); };   // the scores of tile t are complete
  // O of tile t is complete.  With tiles of one step three groups wait for three tiles at a time: a
  // barrier for each, so that no parity stands for two of them.
  auto b_o_full = [&](int t) { return bar0 + 8 + 8 * C::NQ + 8 * (t & 3); };
  const uint32_t bar1 = bar0 + 40 + 8 * C::NQ;
  auto b_s_full = [&](int b) { return bar1 + 8 * b; };
  auto b_p_ready = [&](int b) { return bar1 + 8 * (kGroups + b); };
  auto b_step_full = [&](int s) { return bar1 + 8 * (2 * kGroups + s); };
  auto b_step_empty = [&](int s) { return bar1 + 8 * (2 * kGroups + C::RING + s); };
  auto b_k_full = [&](int s) { return bar1 + 8 * (2 * kGroups + 2 * C::RING + s); };
  auto b_v_full = [&](int s) { return bar1 + 8 * (2 * kGroups + 2 * C::RING + C::NK + s); };
  auto b_v_empty = [&](int s) { return bar1 + 8 * (2 * kGroups + 2 * C::RING + C::NK + C::NV + s); };
  // hand-over between the halves of a cluster whose rows stand in both, by warp of a half
  auto b_m_full = [&](int w) { return bar1 + 8 * (2 * kGroups + 2 * C::RING + C::NK + 2 * C::NV + w); };
  auto b_m_empty = [&](int w) { return b_m_full(2 + w); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::OFF_MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + C::OFF_MISC + 4);
  int* redo_acc = reinterpret_cast<int*>(smem + C::OFF_MISC + 8);
  unsigned* bitmap = reinterpret_cast<unsigned*>(smem + C::OFF_BITMAP);

  const int tid = threadIdx.x, warp = warp_uniform(tid >> 5), lane = tid & 31;
  // a query cluster of 256 rows takes two tiles; two of 64 rows (or one) share one
  const int tiles_per_qc = prm.c_q >= kTile ? prm.c_q / kTile : 1;
  constexpr bool pairs = MODE == kPairs, twice = MODE == kTwice, halves = pairs || twice;
  const int box_rows = min(prm.c_k, pairs ? kTile / 2 : kTile);   // of a load of keys

  if (tid == 0) {
    mbar_init(b_o_empty, 4);
#pragma unroll 1
    for (int w = 0; w < C::NQ; ++w) mbar_init(b_q_empty(w), 1);
#pragma unroll 1
    for (int b = 0; b < kGroups; ++b) { mbar_init(b_s_full(b), 1); mbar_init(b_p_ready(b), 4); }
#pragma unroll 1
    for (int s = 0; s < C::RING; ++s) { mbar_init(b_step_full(s), 1); mbar_init(b_step_empty(s), 6); }
#pragma unroll 1
    for (int s = 0; s < C::NK; ++s) mbar_init(b_k_full(s), 1);
#pragma unroll 1
    for (int s = 0; s < C::NV; ++s) { mbar_init(b_v_full(s), 1); mbar_init(b_v_empty(s), 1); }
#pragma unroll 1
    for (int w = 0; w < 4; ++w) mbar_init(b_o_full(w), 1);
    if (twice)
#pragma unroll 1
      for (int w = 0; w < 4; ++w) mbar_init(b_m_full(w), 1);
    *abort_flag = 0;
    for (int b = 0; b < 4; ++b) redo_acc[b] = 0;
    fence_mbar_init();
  }
  if (tid < kTile) reinterpret_cast<int2*>(smem + C::OFF_REF)[tid] = make_int2(0, -1);
  if (warp == 1) {                       // this warp owns the TMEM allocation
    tmem_alloc(smem_u32(tmem_slot), C::TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = warp_uniform(*tmem_slot);
  const uint32_t tmem_o = tmem_base + kGroups * kTile;

  if (warp < 4) {
    auto relaxed = [&](uint32_t bar, uint32_t phase) {
      return mbar_wait_relaxed(bar, phase & 1, abort_flag, prm.status, prm.wait_limit);
    };
    if (warp == 0 || warp == 3) {
      // ---------------------------------------------------------- TMA producers: Q and K, V
      if (lane == 0) {
        prefetch_tensormap(warp == 0 ? &tm_q : &tm_v);
        prefetch_tensormap(warp == 0 ? &tm_k : &tm_cv);
        const int boxes = kTile / box_rows;
        auto produce = [&](auto is_key) {
          constexpr bool key = decltype(is_key)::value;
          constexpr int panels = key ? C::QK_PANELS : C::PANELS, cols = key ? C::QK_PANEL_COLS : 64;
          constexpr int slots = key ? C::NK : C::NV, bytes = key ? C::QK_BYTES : C::V_BYTES;
          static_assert(!key || slots == kGroups, "a key slot goes with a score buffer");
          int tiles = 0, stops = 0;
          int ring = 0, slot = 0;               // of step i
          uint32_t ph_ring = 0, ph_slot = 1;    // of its descriptor; of the product that read the slot before
#pragma unroll 1
          for (int i = 0;; ++i) {
            if (!relaxed(b_step_full(ring), ph_ring)) return;
            const int fl = st_flags[ring];
            const int* rows = st_rows + ring * kRowInts;
            // A slot is free when the product that read it has completed: for keys the scores of step
            // i - slots, whose barrier takes its next phase behind this load.
            if (i >= slots && !relaxed(key ? b_s_full(slot) : b_v_empty(slot), ph_slot)) return;
            const uint32_t dst = (key ? s_k : s_v) + slot * bytes, bar = key ? b_k_full(slot) : b_v_full(slot);
            if (fl & kFStop) {                             // passed on to the issuer
              if (!key) return;
              mbar_arrive(bar);
              if (++stops == kGroups) return;
            } else {
              if (key && (fl & kFFirst)) {
                if (tiles >= C::NQ && !relaxed(b_q_empty(tiles), tiles / C::NQ - 1)) return;
                const uint32_t q_dst = s_q + tiles % C::NQ * C::QK_BYTES;
                ++tiles;
                // Q arrives with the tile's first keys (scores of a half without a cluster are not read)
                const bool one = pairs && (fl & kFSingle) != 0;
                mbar_expect_more(bar, one ? C::QK_BYTES / 2 : C::QK_BYTES);
#pragma unroll 1
                for (int half = 0; half <= (halves && !one ? 1 : 0); ++half)
#pragma unroll
                  for (int pn = 0; pn < C::QK_PANELS; ++pn)
                    tma_load_2d(q_dst + pn * C::PANEL_BYTES + half * 64 * 128, &tm_q, pn * C::QK_PANEL_COLS, rows[kRowQ] + (twice ? 0 : half * 64), bar);
              }
              if (!(fl & kFCentroid)) {
                // 128 rows: one box, or several boxes
                if (!key || i != (prm.skip_key_load >> 1)) {     // diagnostic: this slot never fills, its waiters time out
                  mbar_expect_tx(bar, bytes);
#pragma unroll 1
                  for (int x = 0; x < boxes; ++x)
#pragma unroll
                    for (int pn = 0; pn < panels; ++pn)
                      tma_load_2d(dst + pn * C::PANEL_BYTES + x * box_rows * 128, key ? &tm_k : &tm_v, pn * cols, rows[x], bar);
                }
              } else {
                // keys as bf16: 64 rows of hi parts and 64 rows of lo parts; as codes, and values: 64 rows
                mbar_expect_tx(bar, panels * ((key && !F8) ? kTile : kCen) * 128);
#pragma unroll
                for (int pn = 0; pn < panels; ++pn)
                  tma_load_2d(dst + pn * C::PANEL_BYTES, key ? &tm_ck : &tm_cv, pn * cols, rows[key ? 0 : kRowCenV], bar);
              }
              mbar_arrive(b_step_empty(ring));
            }
            if (++slot == slots) { slot = 0; ph_slot ^= 1; }
            if (++ring == C::RING) { ring = 0; ph_ring ^= 1; }
          }
        };
        if (warp == 0) produce(std::true_type{});
        else produce(std::false_type{});
      }
    } else if (warp == 1) {
      // ---------------------------------------------------------- MMA issuer
      // One thread issues all products: P V in the order of the steps, scores in the order of the steps and up to three
      // steps ahead, either as soon as what it needs is there.  An instruction is issued when the one before it
      // has been taken in, so that all that this thread does between products leaves the tensor core idle: with a warp that
      // waited for one barrier after the other, voted and read the flags by shuffles 500 to 600 of the 1,600
      // cycles of a step at d = 128.  It looks at all barriers at once and waits for none.  40 heads of 32,760
      // rows, 32 of 256 clusters, d = 128 2,483 -> 2,395 us, 2 x 16 heads of 20,000 rows, 10 clusters of 256 749 -> 717, 12 heads of
      // 16,385 rows, d = 64, clusters of 64 226 -> 221.  (One thread and one barrier after the other: 2,414, 727, 228.)
      if (elect_one()) {
        constexpr uint32_t idesc_qk = F8 ? idesc_e4m3_f32(kTile, kTile) : idesc_bf16_f32(kTile, kTile, 0, 0);
        constexpr uint32_t idesc_qc = F8 ? idesc_e4m3_f32(kTile, kCen) : idesc_qk;      // centroid steps
        constexpr uint32_t idesc_pv = idesc_bf16_f32(kTile, D, 0, 1);
        // descriptors differ from a base one only in the start-address field (units of 16 bytes):
        // the base descriptors are built once, the per-instruction part is an addition
        const uint64_t q_desc0 = smem_desc_sw128(s_q, 16, 1024);
        const uint64_t k_desc0 = smem_desc_sw128(s_k, 16, 1024);
        const uint64_t v_desc0 = smem_desc_sw128(s_v, C::PANEL_BYTES, 1024);
        int o_tiles = 0, q_tiles = 0;
        // scores of step n, into the buffer that P V (n - kGroups) was issued from
        auto scores = [&](int fl, int buf) {
          if (fl & kFStop) {                    // wakes the group of this step, which ends with it
            mbar_arrive(b_s_full(buf));
            return;
          }
          const uint32_t d_cols = tmem_base + buf * kTile;
          const uint64_t kd = k_desc0 + ((buf * C::QK_BYTES) >> 4);
          const uint64_t qd = q_desc0 + (uint64_t)((q_tiles % C::NQ * C::QK_BYTES) >> 4);
          const uint32_t idesc = (fl & kFCentroid) ? idesc_qc : idesc_qk;
  #pragma unroll
          for (int ks = 0; ks < D / C::QK_KSTEP; ++ks) {
            // K-major operands: 32 bytes (16 bf16 or 32 E4M3 elements) per instruction, four per panel
            const uint32_t off = ((ks / 4) * C::PANEL_BYTES + (ks % 4) * 32) >> 4;
            if (F8) mma_ss_f8(d_cols, qd + off, kd + off, idesc, ks > 0 ? 1u : 0u);
            else mma_ss(d_cols, qd + off, kd + off, idesc, ks > 0 ? 1u : 0u);
          }
          mma_commit(b_s_full(buf));
          if (fl & kFLast) mma_commit(b_q_empty(q_tiles));
        };
        static_assert(C::NK == kGroups, "key slots and score buffers go round together");
        bool first = true;                      // P V of step u is the first one of a tile
        int u = 0, n = 0;                       // steps of the next P V, of the next scores
        int buf_u = 0, buf_n = 0, slot_v = 0, ring = 0;
        uint32_t ph_s = 0, ph_p = 0, ph_v = 0;  // phases of the keys of step n, of P and of V of step u
        unsigned long long flags = 0;           // of steps u .. n - 1, 21 bits each
        uint32_t idle = 0;
        long long t0 = 0;
  #pragma unroll 1
        for (;;) {
          const int fl = (int)flags & 0x1fffff;
          if (n == u + kGroups && (fl & kFStop)) break;
          const bool keys = mbar_test_wait(b_k_full(buf_n), ph_s);
          const bool probabilities = mbar_test_wait(b_p_ready(buf_u), ph_p), value_rows = mbar_test_wait(b_v_full(slot_v), ph_v);
          const int fl_n = reinterpret_cast<volatile int*>(st_flags)[ring];    // published when the keys have arrived
          // (behind the first P V of a tile: O of the tile before has been read)
          bool go = n > u && !(fl & kFStop) && probabilities && value_rows;
          if (go && first && o_tiles > 0) go = mbar_test_wait(b_o_empty, (o_tiles - 1) & 1);
          tc_fence_after();
          if (go) {
            // V is MN-major: 16 key rows (2048 bytes) per instruction; panels along d
            const uint64_t vd = v_desc0 + ((slot_v * C::V_BYTES) >> 4);
            const uint32_t p_cols = tmem_base + buf_u * kTile;
  #pragma unroll
            for (int ks = 0; ks < 4; ++ks)
              mma_ts(tmem_o, p_cols + ks * 8, vd + (uint64_t)(ks * (2048 >> 4)), idesc_pv, (ks > 0 || !first) ? 1u : 0u);
            if (!(fl & kFCentroid)) {
  #pragma unroll
              for (int ks = 4; ks < 8; ++ks)
                mma_ts(tmem_o, p_cols + ks * 8, vd + (uint64_t)(ks * (2048 >> 4)), idesc_pv, 1u);
            }
            mma_commit(b_v_empty(slot_v));
            if (fl & kFLast) mma_commit(b_o_full(o_tiles));
            first = (fl & kFLast) != 0;
            if (first) ++o_tiles;
            flags >>= 21;
            ++u;
            if (++buf_u == kGroups) { buf_u = 0; ph_p ^= 1; }
            if (++slot_v == C::NV) { slot_v = 0; ph_v ^= 1; }
          }
          const bool more = keys && n < u + kGroups;
          if (more) {
            scores(fl_n, buf_n);
            flags |= (unsigned long long)fl_n << (21 * (n - u));
            if (C::NQ > 1 && (fl_n & kFLast)) ++q_tiles;
            ++n;
            if (++buf_n == kGroups) { buf_n = 0; ph_s ^= 1; }
            if (++ring == C::RING) ring = 0;
          }
          if (go || more) { idle = 0; continue; }
          if ((idle++ & 255u) == 0) {           // bounded, as every wait
            const long long t = clock64();
            if (idle == 1) t0 = t;
            if (*abort_flag) break;
            if (t - t0 > prm.wait_limit) {
              *abort_flag = 1;
              atomicExch(prm.status, 5 /* CA_ERR_TIMEOUT */);
              break;
            }
          }
        }
      }
      __syncwarp();
    } else {
      // ---------------------------------------------------------- tiles, lists, step descriptors
      const int per_head = pairs ? (prm.n_qc + 1) >> 1 : prm.n_qc * tiles_per_qc;
      const int ck_shift = __ffs(prm.c_k) - 1;
      const int boxes = prm.c_k >= kTile ? 1 : kTile / prm.c_k;      // list entries per step, at most 8
      int s = 0, ord = 0;
      bool ok = true;
      auto claim = [&]() {
        if (s >= C::RING) ok = __all_sync(0xffffffffu, relaxed(b_step_empty(s % C::RING), s / C::RING - 1));
        return ok;
      };
      auto publish = [&]() {
        __syncwarp();
        if (lane == 0) mbar_arrive(b_step_full(s % C::RING));
        ++s;
      };
      // centroids [64 i, 64 i + 64) of a step: additive term log2 of the count, the clusters of a list (of
      // either of two) masked
      auto centroid_bias = [&](float* bz, const unsigned* in0, const unsigned* in1, const int32_t* cnt, int i) {
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          const int j = i * kCen + lane + 32 * g;
          const float w = j < prm.n_kc ? log2f((float)cnt[min(j, prm.n_kc - 1)]) : -INFINITY;
          bz[lane + 32 * g] = (in0[j >> 5] >> (j & 31)) & 1u ? -INFINITY : w;
          if (pairs) bz[kCen + lane + 32 * g] = (in1[j >> 5] >> (j & 31)) & 1u ? -INFINITY : w;
        }
      };
      auto list_length = [&](size_t at) {
        int keep = prm.keep_count ? prm.keep_count[at] : prm.keep;
        if (keep < 0 || keep > prm.list_stride) {            // a list length that does not fit its row
          if (lane == 0) atomicCAS(prm.status, 0, kErrBadIndex);
          keep = keep < 0 ? 0 : prm.list_stride;
        }
        return keep;
      };
#pragma unroll 1
      for (int tile = blockIdx.x; tile < prm.n_tiles && ok; ++ord) {
        int next = 0;
        if (lane == 0) next = (int)gridDim.x + atomicAdd(prm.next_tile, 1);
        const int p = tile / per_head, x = tile % per_head;
        const int32_t* cnt = prm.count_k + (size_t)p * prm.n_kc;
        const int cen_steps = prm.compensate ? prm.cen_tiles : 0;
        if constexpr (pairs) {
          // ---- Two 64-row query clusters, one in either half of the tile, or one in the upper half.  Neighbours in
          // cluster order are siblings of the split tree, and most of their lists are the same: key clusters of both
          // lists are taken by all rows, those of one list two at a time by a half each.  In runs of 64 keys:
          //   shared       two runs of both lists per step
          //   split        a run of the upper list, for the upper half, and one of the lower
          //   one-sided    two runs of the list that is longer than the other
          // which are never more steps than two tiles of one cluster each.  (A list that holds a cluster twice counts it twice: then
          // nothing is shared.)
          const int qc = 2 * x;
          const bool single = qc + 1 == prm.n_qc;
          const size_t at = (size_t)p * prm.n_qc + qc;
          const int32_t* sel0 = prm.block_idx + at * prm.list_stride;
          const int32_t* sel1 = sel0 + prm.list_stride;
          const int keep0 = list_length(at), keep1 = single ? 0 : list_length(at + 1);
          unsigned* in0 = bitmap;
          unsigned* in1 = single ? bitmap : bitmap + prm.bitmap_words;
          __syncwarp();
#pragma unroll 1
          for (int w = lane; w < (single ? 1 : 2) * prm.bitmap_words; w += 32) bitmap[w] = 0u;
          __syncwarp();
          int n0 = 0, n1 = 0, both = 0;                      // entries of the lists that are key clusters, shared ones
          bool again = false;
#pragma unroll 1
          for (int base = 0; base < max(keep0, keep1); base += 32) {
            const int e = base + lane;
            const int j0 = e < keep0 ? sel0[e] : 0, j1 = e < keep1 ? sel1[e] : 0;
            const bool ok0 = e < keep0 && (unsigned)j0 < (unsigned)prm.n_kc, ok1 = e < keep1 && (unsigned)j1 < (unsigned)prm.n_kc;
            // not a key cluster: flagged, left out
            if ((e < keep0 && !ok0) || (e < keep1 && !ok1)) atomicCAS(prm.status, 0, kErrBadIndex);
            const unsigned bit0 = 1u << (j0 & 31), bit1 = 1u << (j1 & 31);
            if (ok0) again |= (atomicOr(&in0[j0 >> 5], bit0) & bit0) != 0;
            if (ok1) again |= (atomicOr(&in1[j1 >> 5], bit1) & bit1) != 0;
            n0 += __popc(__ballot_sync(0xffffffffu, ok0));
            n1 += __popc(__ballot_sync(0xffffffffu, ok1));
          }
          const bool apart = __any_sync(0xffffffffu, again);
          __syncwarp();
          if (!single && !apart) {
#pragma unroll 1
            for (int w = lane; w < prm.bitmap_words; w += 32) both += __popc(in0[w] & in1[w]);
            both = __reduce_add_sync(0xffffffffu, both);
          }
          // Entries of the lists in waiting: `taken` have been looked at, those of `kind` (0: not in the other list,
          // 1: in both, 2: any) are put in, first key row, rows and scale of the keys.
          auto fill = [&](int4* queue, const int32_t* sel, int keep, const unsigned* other, int kind, int& taken, int& filled, int upto) {
#pragma unroll 1
            while (filled < upto && taken < keep) {
              const int e = taken + lane;
              const int j = e < keep ? sel[e] : -1;
              bool in = (unsigned)j < (unsigned)prm.n_kc;
              if (in && kind != 2) in = ((other[j >> 5] >> (j & 31)) & 1u) == (unsigned)kind;
              const unsigned found = __ballot_sync(0xffffffffu, in);
              if (in)
                queue[(filled + __popc(found & ((1u << lane) - 1u))) % kQueue] =
                    make_int4((p * prm.n_kc + j) * prm.c_k, min(max(cnt[j], 0), prm.c_k),
                              F8 ? __float_as_int(prm.k_scale[(size_t)p * prm.n_kc + j]) : 0, 0);
              filled += __popc(found);
              taken += 32;
            }
          };
          // runs of 64 keys: a cluster has 2^parts of them, a run holds 2^each clusters
          const int parts = max(ck_shift - 6, 0), each = max(6 - ck_shift, 0);
          auto through = [&](int run) { return ((run >> parts) + 1) << each; };                    // entries of runs 0 .. run
          auto runs = [&](int entries) { return ((entries + (1 << each) - 1) >> each) << parts; };
          const int all = single ? n0 : both, own0 = single ? 0 : n0 - both, own1 = n1 - both;     // entries
          const int runs0 = runs(own0), runs1 = runs(own1);
          const int end_shared = (runs(all) + 1) >> 1, end_split = end_shared + min(runs0, runs1);
          const int end_runs = end_split + ((abs(runs0 - runs1) + 1) >> 1), n = max(end_runs + cen_steps, 1);
          const int longer = runs1 > runs0 ? 1 : 0;            // list of the one-sided steps
          const int kind = apart ? 2 : 0;
          int4* queue = reinterpret_cast<int4*>(smem + C::OFF_QUEUE);
          int taken_both = 0, filled_both = 0, taken0 = 0, filled0 = 0, taken1 = 0, filled1 = 0;
          // Four steps at a time, eight lanes to a step, one to a box: a step by itself takes this warp longer
          // (1,800 cycles) than the softmax.
          const int k = lane >> 3, box = lane & 7;
          const int h = box * box_rows >= kCen ? 1 : 0;        // the box's run of the step
          const bool a_box = box * box_rows < kTile;
#pragma unroll 1
          for (int u0 = 0; u0 < n && ok; u0 += 4) {
            const int u = u0 + k, last = min(u0 + 3, n - 1);   // this lane's step; the last one of the four
            if (u0 < end_shared)
              fill(queue, sel0, keep0, in1, single ? 2 : 1, taken_both, filled_both, min(all, through(2 * min(last, end_shared - 1) + 1)));
            if (last >= end_shared && u0 < end_runs) {
              // runs of either list up to step `last`
              const int v = min(last, end_runs - 1), far = max(v - end_split + 1, 0);
              const int to = min(v, end_split - 1) - end_shared + 2 * far;
              fill(queue + kQueue, sel0, keep0, in1, kind, taken0, filled0, min(own0, through(longer == 0 ? to : to - 2 * far)));
              fill(queue + 2 * kQueue, sel1, keep1, in0, kind, taken1, filled1, min(own1, through(longer == 1 ? to : to - 2 * far)));
            }
            __syncwarp();
            const bool shared = u < end_shared, split = !shared && u < end_split, one = u >= end_split && u < end_runs;
            const bool cen = u >= end_runs && cen_steps > 0, live = u < n;
            const int which = shared ? 0 : split ? 1 + h : 1 + longer;
            const int run = shared ? 2 * u + h : split ? u - end_shared : 2 * (u - end_split) + end_split - end_shared + h;
            const int entries = shared ? all : !(split || one) ? 0 : which == 2 ? own1 : own0;
            const int entry = ((run >> parts) << each) + (box & ((1 << each) - 1));
            const int first = (run & ((1 << parts) - 1)) * kCen;
            int4 it = make_int4(p * prm.n_kc * prm.c_k, 0, 0, 0);   // (behind the end of a list: rows of the first cluster, masked)
            if (a_box && entry < entries) it = queue[which * kQueue + entry % kQueue];
            const int members = entry < entries ? it.y - first : 0;
            const bool starts = live && box == 0;              // the lane that waits for the step's slot and hands it over
            const int slot = (s + k) % C::RING;
            if (starts && s + k >= C::RING) ok = relaxed(b_step_empty(slot), (s + k) / C::RING - 1);
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            int* rows = st_rows + slot * kRowInts;
            const unsigned cut = __ballot_sync(0xffffffffu, live && !cen && a_box && members < box_rows);
            if (live && !cen && a_box) {
              rows[box] = it.x + first;
              if (F8 && box < 2) st_scale[slot * 2 + box] = __int_as_float(it.z);
            }
            if (live && cen) {
              const int i = u - end_runs;
              if (box == 0) rows[0] = (p * prm.cen_tiles + i) * (F8 ? kCen : kTile);
              if (box == 1) rows[kRowCenV] = (p * prm.cen_tiles + i) * kCen;
              if (F8 && box < 2) st_scale[slot * 2 + box] = prm.c_scale[(size_t)p * prm.cen_tiles + i];
            }
            if (starts) {
              st_flags[slot] = (!single ? 0 : kFSingle | kFUpper) | (u == 0 ? kFFirst : 0) |
                               (u == n - 1 ? kFLast : 0) | (min(u, 15) << kFIndexShift) | (min(n - 1 - u, 15) << kFRestShift) |
                               (split ? kFSplit : one ? (longer ? kFLower : kFUpper) : 0) | (cen ? kFCentroid : 0) |
                               (cen || ((cut >> (lane & 24)) & 255u) ? kFMasked : 0);
              rows[kRowQ] = (int)at * prm.c_q;
              st_tile[slot] = make_int4(p, qc * prm.c_q, (int)at * 2, ord);
            }
            // additive terms of short clusters and of centroids, a step after the other
#pragma unroll 1
            for (int kk = 0; kk < 4; ++kk) {
              float* bz = bias + ((s + kk) % C::RING) * kTile;
              if ((cut >> (8 * kk)) & 255u) {
#pragma unroll 1
                for (int c = lane; c < kTile; c += 32) {
                  const int m = __shfl_sync(0xffffffffu, members, 8 * kk + c / box_rows);
                  bz[c] = (c & (box_rows - 1)) < m ? 0.f : -INFINITY;
                }
              }
              if (cen_steps > 0 && u0 + kk >= end_runs && u0 + kk < n) centroid_bias(bz, in0, in1, cnt, u0 + kk - end_runs);
            }
            __syncwarp();
            if (starts) mbar_arrive(b_step_full(slot));
            s += last - u0 + 1;
          }
          tile = __shfl_sync(0xffffffffu, next, 0);
        } else {
        const int qc = x / tiles_per_qc, half = x % tiles_per_qc;
        const int32_t* sel = prm.block_idx + ((size_t)p * prm.n_qc + qc) * prm.list_stride;
        const int keep = list_length((size_t)p * prm.n_qc + qc);
        const int sel_steps = selected_tiles(keep, prm.c_k);
        const int n = max(sel_steps + cen_steps, 1);      // nothing to attend to: one step with every column masked
        if (prm.compensate) {
#pragma unroll 1
          for (int w = lane; w < prm.bitmap_words; w += 32) bitmap[w] = 0u;
          __syncwarp();
        }
        int base = -32, my_j = 0, my_members = 0;            // list entries [base, base + 32), one per lane
        float my_scale = 0.f;
#pragma unroll 1
        for (int u = 0; u < n && ok; ++u) {
          int fl = (u == 0 ? kFFirst : 0) | (u == n - 1 ? kFLast : 0) | (min(u, 15) << kFIndexShift) |
                   (min(n - 1 - u, 15) << kFRestShift);
          const int e0 = prm.c_k >= kTile ? u >> (ck_shift - 7) : u * boxes;
          if (u < sel_steps && e0 >= base + 32) {
            base = e0 & ~31;
            const int e = base + lane;
            my_members = 0;
            my_j = 0;
            my_scale = 0.f;
            if (e < keep) {
              const int j = sel[e];
              my_j = min(max(j, 0), prm.n_kc - 1);
              if (j != my_j) {                             // not a key cluster: flagged, all of its columns masked
                atomicCAS(prm.status, 0, kErrBadIndex);
              } else {
                my_members = min(max(cnt[j], 0), prm.c_k);
                if (F8) my_scale = prm.k_scale[(size_t)p * prm.n_kc + j];
                if (prm.compensate) atomicOr(&bitmap[j >> 5], 1u << (j & 31));
              }
            }
          }
          if (!claim()) break;
          int* rows = st_rows + (s % C::RING) * kRowInts;
          float* bz = bias + (s % C::RING) * kTile;
          float sc = 0.f;
          if (u < sel_steps) {
            // filler boxes behind the end of the list repeat its last entry, masked
            const int at = e0 - base;
            const int src = prm.c_k >= kTile ? at : min(at + (lane & 7), keep - 1 - base);
            const int j = __shfl_sync(0xffffffffu, my_j, src);
            int members = __shfl_sync(0xffffffffu, my_members, src);
            if (F8) sc = __shfl_sync(0xffffffffu, my_scale, src);
            const int first = prm.c_k >= kTile ? (u << 7) & (prm.c_k - 1) : 0;    // row of the step's first column
            members -= first;
            if (prm.c_k < kTile && e0 + (lane & 7) >= keep) members = 0;
            if (lane < boxes) rows[lane] = (p * prm.n_kc + j) * prm.c_k + first;
            const int width = min(prm.c_k, kTile);
            if (__any_sync(0xffffffffu, lane < boxes && members < width)) {
              fl |= kFMasked;
#pragma unroll 1
              for (int c = lane; c < kTile; c += 32) {
                const int m = __shfl_sync(0xffffffffu, members, c / width);
                bz[c] = (c & (width - 1)) < m ? 0.f : -INFINITY;
              }
            }
          } else {
            fl |= kFMasked;
            if (cen_steps > 0) {
              const int i = u - sel_steps;
              fl |= kFCentroid;
              __syncwarp();
              centroid_bias(bz, bitmap, bitmap, cnt, i);
              if (lane == 0) rows[0] = (p * prm.cen_tiles + i) * (F8 ? kCen : kTile);
              if (lane == 1) rows[kRowCenV] = (p * prm.cen_tiles + i) * kCen;
              if (F8) sc = prm.c_scale[(size_t)p * prm.cen_tiles + i];
            } else {
#pragma unroll 1
              for (int c = lane; c < kTile; c += 32) bz[c] = -INFINITY;
              if (lane < boxes) rows[lane] = p * prm.n_kc * prm.c_k;
            }
          }
          if (F8 && lane < 2) st_scale[(s % C::RING) * 2 + lane] = sc;
          if (lane == 0) {
            st_flags[s % C::RING] = fl;
            rows[kRowQ] = (p * prm.n_qc + qc) * prm.c_q + half * kTile;
            st_tile[s % C::RING] = make_int4(p, qc * prm.c_q + half * kTile, (p * prm.n_qc + qc) * 2 + half, ord);
          }
          publish();
        }
        tile = __shfl_sync(0xffffffffu, next, 0);
        }
      }
#pragma unroll 1
      for (int g = 0; g < kGroups && ok; ++g) {
        if (!claim()) break;
        if (lane == 0) st_flags[s % C::RING] = kFStop;
        publish();
      }
    }
  } else {
    // ------------------------------------------------------------ softmax groups and epilogue
    const int group = (warp >> 2) - 1;
    const int quarter = warp & 3;                  // TMEM lanes this warp may touch
    const int row = quarter * 32 + lane;           // row within the tile
    const int half = quarter >> 1;                 // of the tile
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const uint32_t t_s = tmem_base + group * kTile + lane_addr;
    auto wait = [&](uint32_t bar, uint32_t phase) {
      return __all_sync(0xffffffffu, mbar_wait(bar, phase & 1, abort_flag, prm.status, prm.wait_limit));
    };
    float m_own = -INFINITY, l_run = 0.f, pend = 0.f;
    // factor from a raw score to log2 units: the softmax scale, and with quantised Q K^T the scale
    // of this thread's query row (times, per 64 keys, the scale of the key cluster or centroid run)
    float row_sc = prm.scale_log2;
    uint32_t ph_s = 0;
#pragma unroll 1
    for (int s = group;; s += kGroups) {
      const int ring = s % C::RING;
      if (!wait(b_s_full(group), ph_s)) break;
      ph_s ^= 1;
      tc_fence_after();
      const int fl = warp_uniform(st_flags[ring]);
      if (fl & kFStop) break;
      const int index = (fl >> kFIndexShift) & 15, rest = (fl >> kFRestShift) & 15;
      const bool cen = (fl & kFCentroid) != 0, masked = (fl & kFMasked) != 0;
      if (index < kGroups) {                       // this group's first step of the tile
        m_own = -INFINITY;
        l_run = 0.f;
        pend = 0.f;
        if (F8) {
          const int4 tl = st_tile[ring];
          row_sc = prm.scale_log2 * prm.q_scale[(size_t)tl.x * prm.n_qc * prm.c_q + tl.y + (twice || (pairs && (fl & kFSingle)) ? row & 63 : row)];
        }
      }
      // scales of this step's scores, per run of 64 columns.  A zero scale (an all-zero query row or
      // key group) makes every logit 0: the raw scores are then dropped and the additive terms
      // enter with scale 1.
      float sc_h[2] = {prm.scale_log2, prm.scale_log2};
      float raw_h[2] = {1.f, 1.f};
      if (F8) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float sc_eff = row_sc * st_scale[ring * 2 + h];
          raw_h[h] = sc_eff > 0.f ? 1.f : 0.f;
          sc_h[h] = sc_eff > 0.f ? sc_eff : (masked ? 1.f : 0.f);
        }
      }
      // (the two lists of a tile of 64-row query clusters leave out different centroids)
      const float* bz = bias + ring * kTile + (pairs && cen ? half * kCen : 0);
      // chunks [c_begin, c_end) of 32 columns
      const bool idle = pairs ? (fl & (half == 0 ? kFLower : kFUpper)) != 0 : twice && cen && half == 1;
      const bool split = pairs ? (fl & kFSplit) != 0 : twice && !cen;
      // (kept from the compiler that it is 0 in the instances for 128 rows: with the loops below arranged for
      // that, they are 3 % slower, 807 -> 835 us for 8 heads of 16,384 x 131,072 rows)
      int c_begin = split ? 2 * half : 0;
      asm volatile("" : "+r"(c_begin));
      const int c_end = idle ? 0 : split ? c_begin + 2 : (cen ? 2 : 4);
      // ---- masked or weighted steps: scores of hi and lo parts of centroids are added and the additive
      // term is folded into the scores in tensor memory first, so that the common path below has
      // no bias
      if (masked) {
#pragma unroll 1
        for (int c4 = c_begin; c4 < c_end; ++c4) {
          const float inv = __fdividef(1.f, F8 && c4 >= 2 ? sc_h[1] : sc_h[0]);
          const float raw = F8 && c4 >= 2 ? raw_h[1] : raw_h[0];
          uint32_t r[32];
          tmem_ld32(t_s + c4 * 32, r);
          if (!F8 && cen) {
            uint32_t lo[32];
            tmem_ld32(t_s + kCen + c4 * 32, lo);
            tmem_wait_ld32(r);
            tmem_wait_ld32(lo);
#pragma unroll
            for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) + __uint_as_float(lo[j]));
          } else {
            tmem_wait_ld32(r);
          }
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const float x = F8 ? __uint_as_float(r[j]) * raw : __uint_as_float(r[j]);
            r[j] = __float_as_uint(fmaf(bz[c4 * 32 + j], inv, x));
          }
          tmem_st32(t_s + c4 * 32, r);
        }
        tmem_wait_st();
      }
      // ---- reference.  The softmax needs no exact row maximum, only a reference m that keeps
      // exp2(x - m) in range.  The first step of a row (and any later one while the row has seen only
      // masked columns) measures the maximum of its scores; afterwards a row whose probabilities
      // exceeded 2^threshold (seen in the sum of 32 of them) moves its reference up at its group's
      // NEXT step (`pend`).  Values between 2^threshold and 2^96 are exact all the same: P is
      // bf16, which has the exponent range of fp32, and O and l are fp32.  A sum beyond 2^96 may
      // overflow: the row sum then becomes NaN, which marks the tile in `redo`, and the launcher's
      // second pass recomputes marked tiles with the fp32 kernel (exact row maxima).
      // The reference of step s - 1 comes from the group before through shared memory.
      float m_prev;
      {
        int at;
        bool got = true;
        long long t0 = 0;
#pragma unroll 1
        for (uint32_t it = 0;; ++it) {
          asm volatile("ld.volatile.shared.v2.b32 {%0, %1}, [%2];" : "=f"(m_prev), "=r"(at) : "r"(s_ref + row * 8) : "memory");
          if (__all_sync(0xffffffffu, at >= s - 1)) break;
          if ((it & 255u) == 255u) {
            if (t0 == 0) t0 = clock64();
            const bool late = *abort_flag != 0 || clock64() - t0 > prm.wait_limit;
            if (__any_sync(0xffffffffu, late)) {
              *abort_flag = 1;
              if (lane == 0) atomicCAS(prm.status, 0, 5 /* CA_ERR_TIMEOUT */);
              got = false;
              break;
            }
          }
        }
        if (!got) break;
      }
      if (index == 0) m_prev = -INFINITY;
      float m_ref = m_prev;
      if (__any_sync(0xffffffffu, m_prev == -INFINITY || m_prev != m_own || pend > 0.f)) {
        if (pend > 0.f) m_ref = fmaxf(m_ref, m_own + pend);
        if (c_end > 0 && __any_sync(0xffffffffu, m_ref == -INFINITY)) {
          float tmax = -INFINITY;
#pragma unroll 1
          for (int c4 = c_begin; c4 < c_end; ++c4) {
            uint32_t r[32];
            tmem_ld32(t_s + c4 * 32, r);
            tmem_wait_ld32(r);
            float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY, mx3 = -INFINITY;
#pragma unroll
            for (int j = 0; j < 32; j += 8) {
              mx0 = max3(mx0, __uint_as_float(r[j]), __uint_as_float(r[j + 1]));
              mx1 = max3(mx1, __uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]));
              mx2 = max3(mx2, __uint_as_float(r[j + 4]), __uint_as_float(r[j + 5]));
              mx3 = max3(mx3, __uint_as_float(r[j + 6]), __uint_as_float(r[j + 7]));
            }
            tmax = fmaxf(tmax, fmaxf(fmaxf(mx0, mx1), fmaxf(mx2, mx3)) * (F8 && c4 >= 2 ? sc_h[1] : sc_h[0]));
          }
          if (tmax > m_ref + kRescaleThreshold || m_ref == -INFINITY) m_ref = fmaxf(m_ref, tmax);
        }
        if (m_own > -INFINITY) l_run *= ex2_approx(m_own - m_ref);
        if (index > 0 && __any_sync(0xffffffffu, m_ref != m_prev)) {
          // P V (s - 1) is complete when its value slot is free again; P V (s) waits for this warp
          if (!wait(b_v_empty((s - 1) % C::NV), (s - 1) / C::NV)) break;
          tc_fence_after();
          const float alpha = m_prev == -INFINITY ? 0.f : ex2_approx(m_prev - m_ref);
#pragma unroll 1
          for (int c4 = 0; c4 < D / 32; ++c4) {
            uint32_t o[32];
            tmem_ld32(tmem_o + lane_addr + c4 * 32, o);
            tmem_wait_ld32(o);
#pragma unroll
            for (int j = 0; j < 32; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * alpha);
            tmem_st32(tmem_o + lane_addr + c4 * 32, o);
          }
          tmem_wait_st();
        }
        pend = 0.f;
      }
      m_own = m_ref;
      asm volatile("st.volatile.shared.v2.b32 [%0], {%1, %2};" ::"r"(s_ref + row * 8), "f"(m_ref), "r"(s) : "memory");

      // ---- P = exp2(x - m), packed to bf16: the 32 columns of chunk c go to columns [16 c, 16 c + 16),
      // which have been read by then.  A chunk is loaded while the one before it is computed.
      const float neg_m = (m_ref == -INFINITY) ? 0.f : -m_ref;
      const f32x2 nm2 = pack2(neg_m, neg_m);
      float big = 0.f;                                   // largest sum of a chunk
      auto chunk = [&](uint32_t (&r)[32], f32x2 sc2, uint32_t dst) {
        // The special-function unit takes one exponential per 8 cycles and sub-core: scaling and
        // sums use two-value fp32 instructions, and the other work of the chunk is interleaved
        // with the exponentials in groups of four, two groups behind, so that it issues in the
        // shadow of that unit.
        float x[32];
        uint32_t pk[16];
        f32x2 s01 = pack2(0.f, 0.f), s23 = s01;
        auto scale4 = [&](int j) {
          unpack2(fma2(pack2(__uint_as_float(r[j]), __uint_as_float(r[j + 1])), sc2, nm2), x[j], x[j + 1]);
          unpack2(fma2(pack2(__uint_as_float(r[j + 2]), __uint_as_float(r[j + 3])), sc2, nm2), x[j + 2], x[j + 3]);
        };
        scale4(0);
        scale4(4);
#pragma unroll
        for (int g = 0; g < 10; ++g) {
          if (g < 8) {
#pragma unroll
            for (int e = 4 * g; e < 4 * g + 4; ++e) x[e] = ex2_approx(x[e]);
          }
          if (g + 2 < 8) scale4(4 * (g + 2));
          if (g >= 2) {
            const int j = 4 * (g - 2);
            s01 = add2(s01, pack2(x[j], x[j + 1]));
            s23 = add2(s23, pack2(x[j + 2], x[j + 3]));
            pk[j / 2] = pack_bf16x2(x[j], x[j + 1]);
            pk[j / 2 + 1] = pack_bf16x2(x[j + 2], x[j + 3]);
          }
        }
        float sa, sb, sc, sd;
        unpack2(s01, sa, sb);
        unpack2(s23, sc, sd);
        const float sum = (sa + sb) + (sc + sd);
        l_run += sum;
        big = fmaxf(big, sum);
        if (!(sum < kDangerSum)) l_run = __int_as_float(0x7fffffff);
        tmem_st16(dst, pk);
      };
      uint32_t ra[32], rb[32];
      tmem_ld32(t_s + c_begin * 32, ra);
      tmem_wait_ld32(ra);
#pragma unroll 1
      for (int h = c_begin >> 1; 2 * h < c_end; ++h) {
        const float sc = F8 && h > 0 ? sc_h[1] : sc_h[0];
        const f32x2 sc2 = pack2(sc, sc);
        tmem_ld32(t_s + h * 64 + 32, rb);
        chunk(ra, sc2, t_s + h * 32);
        tmem_wait_ld32(rb);
        if (2 * h + 2 < c_end) tmem_ld32(t_s + h * 64 + 64, ra);
        chunk(rb, sc2, t_s + h * 32 + 16);
        tmem_wait_ld32(ra);
      }
      if (split || idle) {                                 // the other half's keys
#pragma unroll
        for (int j = 0; j < 32; ++j) ra[j] = 0u;
        tmem_st32(t_s + (split && half == 0 ? 32 : 0), ra);
        if (idle && !cen) tmem_st32(t_s + 32, ra);
      }
      if (big > kSumLimit) pend = ceilf(log2f(big));
      // the group's last step of the tile: its row sums go to the group that ends the tile
      if (rest > 0 && rest < kGroups) lpart[s % kParts * kTile + row] = make_float2(l_run, m_ref);
      const int4 tl = st_tile[ring];
      // one arrival per warp: 128 arrivals on one barrier word would be serialised in shared memory
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) { mbar_arrive(b_p_ready(group)); mbar_arrive(b_step_empty(ring)); }
      if (rest > 0) continue;

      // ---- epilogue: O / l, rows back to their original positions
      const int pos = tl.y + (twice ? row & 63 : row);
      // rows of the padding are not written, nor those of a half without a cluster of its own
      bool live = pos < prm.n_q && !((twice || (pairs && (fl & kFSingle))) && half == 1);
      int orig = live ? prm.perm_q[(size_t)tl.x * prm.n_q + pos] : 0;
      if (orig < 0 || orig >= prm.n_q) {                // not a row of O: flagged, nothing written
        atomicCAS(prm.status, 0, kErrBadIndex);
        live = false;
        orig = 0;
      }
      // products complete in order, and the sums were written before the probabilities were handed over
      if (!wait(b_o_full(tl.w), tl.w >> 2)) break;
      tc_fence_after();
#pragma unroll
      for (int g = 1; g < kGroups; ++g) {
        if (g <= index) {
          const float2 other = lpart[(s - g) % kParts * kTile + row];
          if (other.y > -INFINITY) l_run += other.x * ex2_approx(other.y - m_ref);
        }
      }
      // Rows that stand in both halves: the lower one hands over its sum and reference and 16 columns of O at a time, which
      // the upper one scales to the larger reference.
      float* merge = reinterpret_cast<float*>(smem + C::OFF_MERGE) + (row & 63) * kMergeInts;
      const int pair = quarter & 1, uses = tl.w * (D / 16);
      bool got = true;
      if (twice && half == 1) {
#pragma unroll 1
        for (int c = 0; c < D / 16 && got; ++c) {
          const int use = uses + c;
          uint32_t o[16];
          tmem_ld16(tmem_o + lane_addr + c * 16, o);
          tmem_wait_ld();
          if (use > 0) got = wait(b_m_empty(pair), use - 1);
          if (!got) break;
#pragma unroll
          for (int j = 0; j < 16; ++j) merge[j] = __uint_as_float(o[j]);
          merge[16] = l_run;
          merge[17] = m_ref;
          __syncwarp();
          if (lane == 0) mbar_arrive(b_m_full(pair));
        }
        if (!got) break;
      }
      float l_all = l_run, m_all = m_ref, w_own = 1.f, w_other = 0.f;
      if (twice && half == 0) {
        got = wait(b_m_full(pair), uses);
        if (!got) break;
        const float l_other = merge[16], m_other = merge[17];
        m_all = fmaxf(m_ref, m_other);
        w_own = m_ref > -INFINITY ? ex2_approx(m_ref - m_all) : 0.f;
        w_other = m_other > -INFINITY ? ex2_approx(m_other - m_all) : 0.f;
        l_all = l_run * w_own + l_other * w_other;
      }
      // a row without a single live entry (an empty list without compensation): zeros, lse = -inf
      const bool empty = !(l_all > 0.f);
      const float inv = empty ? 0.f : 1.f / l_all;
      __nv_bfloat16* out = prm.O + ((size_t)tl.x * prm.n_q + orig) * D;
      const float inv_own = inv * w_own, inv_other = inv * w_other;
#pragma unroll 1
      for (int c = 0; c < (twice && half == 1 ? 0 : D / 16); ++c) {
        uint32_t o[16];
        tmem_ld16(tmem_o + lane_addr + c * 16, o);
        tmem_wait_ld();
#pragma unroll
        for (int j = 0; j < 16; ++j) o[j] = __float_as_uint(__uint_as_float(o[j]) * inv_own);
        if (twice) {
          if (c > 0) got = wait(b_m_full(pair), uses + c);
          if (!got) break;
#pragma unroll
          for (int j = 0; j < 16; ++j) o[j] = __float_as_uint(fmaf(merge[j], inv_other, __uint_as_float(o[j])));
          __syncwarp();
          if (lane == 0) mbar_arrive(b_m_empty(pair));
        }
        if (halves) {                                      // 0 x inf, mostly an infinite value among the other half's keys: for the second pass
          f32x2 any2 = pack2(0.f, 0.f);
#pragma unroll
          for (int j = 0; j < 16; j += 2) any2 = add2(any2, pack2(__uint_as_float(o[j]), __uint_as_float(o[j + 1])));
          float any, any_odd;
          unpack2(any2, any, any_odd);
          any += any_odd;
          if (any != any) l_all = any;
        }
        if (live) {
          uint4* dst = reinterpret_cast<uint4*>(out + c * 16);
#pragma unroll
          for (int v = 0; v < 2; ++v) {
            uint4 w;
            w.x = pack_bf16x2(__uint_as_float(o[8 * v + 0]), __uint_as_float(o[8 * v + 1]));
            w.y = pack_bf16x2(__uint_as_float(o[8 * v + 2]), __uint_as_float(o[8 * v + 3]));
            w.z = pack_bf16x2(__uint_as_float(o[8 * v + 4]), __uint_as_float(o[8 * v + 5]));
            w.w = pack_bf16x2(__uint_as_float(o[8 * v + 6]), __uint_as_float(o[8 * v + 7]));
            if (empty) w = make_uint4(0u, 0u, 0u, 0u);   // every column masked: the accumulator may hold 0 x inf
            dst[v] = w;
          }
        }
      }
      if (!got) break;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(b_o_empty);
      if (live && prm.lse)
        prm.lse[(size_t)tl.x * prm.n_q + orig] = empty ? -INFINITY : (m_all + log2f(l_all)) * 0.6931471805599453f;
      // one word per tile or 64-row query cluster, written on every launch by the last of its four warps: 1 = recompute
      // (a row left the range)
      const bool redo = __any_sync(0xffffffffu, live && !(l_all < INFINITY));
      if (lane == 0) {
        int* acc = &redo_acc[tl.w & 3];
        const int mine = redo ? (pairs && half == 1 ? 65537 : 257) : 1;
        if ((atomicAdd(acc, mine) & 255) == 3) {
          const int all = atomicExch(acc, 0);
          prm.redo[tl.z] = (all >> 8) & 255 ? 1 : 0;
          if (pairs && !(fl & kFSingle)) prm.redo[tl.z + 2] = all >> 16 ? 1 : 0;
        }
      }
    }
  }

  let_next_start();
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, C::TMEM_COLS);
}

// ---------------------------------------------------------------------------
// Centroids for the tensor-core path, 64 per tile: key tile = 64 rows of bf16 hi
// parts followed by 64 rows of lo parts; value centroids as bf16.  Rows beyond
// the last centroid are zero.  The first CTA clears the status block (the kernels before the attention
// kernel write no status).
// ---------------------------------------------------------------------------
__global__ void centroid_prep_kernel(const float* __restrict__ ck, const float* __restrict__ cv, int n_kc,
                                     int cen_tiles, int D, __nv_bfloat16* __restrict__ kmix,
                                     __nv_bfloat16* __restrict__ vb, int* __restrict__ status) {
  wait_for_previous();
  let_next_start();
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < kStatusClearBytes / sizeof(int)) status[threadIdx.x] = 0;
  const int p = blockIdx.y;
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= cen_tiles * kCen * D) return;
  const int j = e / D, col = e % D;
  float k = 0.f, v = 0.f;
  if (j < n_kc) {
    k = ck[(size_t)p * n_kc * D + e];
    v = cv[(size_t)p * n_kc * D + e];
  }
  const __nv_bfloat16 h = __float2bfloat16_rn(k);
  const size_t tile = (size_t)p * cen_tiles + j / kCen;
  kmix[(tile * kTile + (j % kCen)) * D + col] = h;
  kmix[(tile * kTile + kCen + (j % kCen)) * D + col] = __float2bfloat16_rn(k - __bfloat162float(h));
  vb[((size_t)p * cen_tiles * kCen + j) * D + col] = __float2bfloat16_rn(v);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

// matrix [rows, D] row-major of bf16 (or of one-byte codes); box = one 128-byte panel row (64 bf16
// or 128 codes) x box_rows rows, 128-byte swizzle
static bool make_map(CUtensorMap* map, const void* base, size_t rows, int D, int box_rows, bool bytes = false) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)D, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)D * (bytes ? 1 : 2)};
  cuuint32_t box[2] = {bytes ? 128u : 64u, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return fn(map, bytes ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool attn_tc_supported(const ca_problem_t& pr) {
  if (pr.dtype != CA_DTYPE_BF16 || (pr.flags & CA_ATTN_FP32)) return false;
  if (pr.cluster_q != 64 && pr.cluster_q != 128 && pr.cluster_q != 256) return false;
  if (pr.cluster_k < 16 || pr.cluster_k > 256) return false;
  const int n_kc = ceil_div(pr.n_k, pr.cluster_k);
  if ((n_kc + 31) / 32 > kBitmapWords) return false;       // selected-cluster bitmap in shared memory
  return true;
}

// quantised Q K^T: head dimension 128 (one 128-byte panel row of codes), key clusters of at least
// 64 rows (one scale per 64 columns)
bool attn_tc_fp8_supported(const ca_problem_t& pr) {
  return attn_tc_supported(pr) && pr.head_dim == 128 && pr.cluster_k >= kCen;
}

size_t attn_tc_workspace_bytes(const ca_problem_t& pr) {
  const size_t P = (size_t)pr.batch * pr.heads;
  const size_t cen_tiles = (size_t)ceil_div(ceil_div(pr.n_k, pr.cluster_k), kCen);
  const size_t n_qc = (size_t)ceil_div(pr.n_q, pr.cluster_q);
  size_t bytes = kStatusBytes + align_up(P * cen_tiles * kTile * pr.head_dim * sizeof(__nv_bfloat16), 256) +
                 align_up(P * cen_tiles * kCen * pr.head_dim * sizeof(__nv_bfloat16), 256) +
                 align_up(P * n_qc * 2 * sizeof(int32_t), 256);
  if (pr.flags & CA_ATTN_FP8_QK) {
    const size_t n_kc = (size_t)ceil_div(pr.n_k, pr.cluster_k), D = pr.head_dim;
    const size_t q_rows = P * n_qc * pr.cluster_q, k_rows = P * n_kc * pr.cluster_k;
    bytes += align_up(q_rows * D, 256) + align_up(q_rows * 4, 256) + align_up(k_rows * D, 256) +
             align_up(P * n_kc * 4, 256) + align_up(P * cen_tiles * kCen * D, 256) + align_up(P * cen_tiles * 4, 256);
  }
  return bytes;
}

template <int D, bool F8, int MODE>
static int launch_tc_d(const CUtensorMap* maps, const TcParams& prm, int grid, LaunchStream st) {
  using C = TcCfg<D, F8, MODE>;
  static_assert(1024 + C::OFF_BITMAP + 4 * (MODE == kPairs ? 2 * kPairBitmapWords : kBitmapWords) <= 227 * 1024, "bitmaps of the largest number of key clusters");
  const size_t smem = 1024 + C::OFF_BITMAP + (size_t)prm.bitmap_words * 4 * (MODE == kPairs ? 2 : 1);
  auto k = attn_tc_kernel<D, F8, MODE>;
  CA_RETURN_IF_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  launch_chained(k, grid, kTcThreads, smem, st, maps[0], maps[1], maps[2], maps[3], maps[4], prm);
  CA_LAUNCH_CHECK();
  return CA_OK;
}

namespace {
long long g_wait_limit = kWaitLimitCycles;   // host-side settings of the diagnostic hook
int g_skip_key_load = -1;
}  // namespace
void attn_tc_set_debug(long long wait_limit_cycles, int skip_key_load) {
  g_wait_limit = wait_limit_cycles > 0 ? wait_limit_cycles : kWaitLimitCycles;
  g_skip_key_load = skip_key_load;
}

int launch_attn_tc(const ca_problem_t& pr, const void* Qp, const void* Kp, const void* Vp, const float* ck,
                   const float* cv, const int32_t* count_k, const int32_t* block_idx, const int32_t* keep_count,
                   int list_stride, const int32_t* perm_q, float scale, void* O, float* lse, void* ws,
                   LaunchStream st) {
  const int P = pr.batch * pr.heads, D = pr.head_dim;
  const int n_qc = ceil_div(pr.n_q, pr.cluster_q), n_kc = ceil_div(pr.n_k, pr.cluster_k);
  const int cen_tiles = ceil_div(n_kc, kCen);
  Carver c(ws);
  int* status = c.take<int>(kStatusBytes / sizeof(int));
  __nv_bfloat16* kmix = c.take<__nv_bfloat16>((size_t)P * cen_tiles * kTile * D);
  __nv_bfloat16* vb = c.take<__nv_bfloat16>((size_t)P * cen_tiles * kCen * D);
  int32_t* redo = c.take<int32_t>((size_t)P * n_qc * 2);
  const bool f8 = (pr.flags & CA_ATTN_FP8_QK) != 0;
  unsigned char *q8 = nullptr, *k8 = nullptr, *c8 = nullptr;
  float *sq = nullptr, *sk = nullptr, *sc = nullptr;
  if (f8) {
    // queries, keys and key centroids as E4M3 codes with their scales (quantize.cu)
    const size_t q_rows = (size_t)P * n_qc * pr.cluster_q, k_rows = (size_t)P * n_kc * pr.cluster_k;
    q8 = c.take<unsigned char>(q_rows * D);  sq = c.take<float>(q_rows);
    k8 = c.take<unsigned char>(k_rows * D);  sk = c.take<float>((size_t)P * n_kc);
    c8 = c.take<unsigned char>((size_t)P * cen_tiles * kCen * D);  sc = c.take<float>((size_t)P * cen_tiles);
    ProfScope ps(kProfAttnPrep, st);
    const int rq = launch_quantize_qk(Qp, Kp, pr.compensate ? ck : nullptr, P, n_qc, pr.cluster_q, n_kc, pr.cluster_k,
                                      cen_tiles, D, q8, sq, k8, sk, c8, sc, st);
    if (rq != CA_OK) return rq;
  }
  if (pr.compensate) {
    ProfScope ps(kProfAttnPrep, st);
    launch_chained(centroid_prep_kernel, dim3(ceil_div(cen_tiles * kCen * D, 256), P), 256, 0, st, ck, cv, n_kc, cen_tiles,
                   D, kmix, vb, status);
    CA_LAUNCH_CHECK();
  }
  const int bitmap_words = (cen_tiles * kCen + 31) / 32;
  int sms = 0, dev = 0;
  CA_RETURN_IF_CUDA(cudaGetDevice(&dev));
  CA_RETURN_IF_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // A pair takes about 1.4 times the steps of one cluster (less the more their lists share), and tiles go in rounds of one per SM:
  // pairs where their rounds are shorter by that, which they are not up to a cluster per SM, nor up to two where odd counts per
  // head leave more than one tile per SM (54 heads of 5 clusters, 32 of 256 clusters of 64, d = 64 42 us by ones, 55 in pairs); and by
  // ones where the bitmaps of two lists do not fit.  At d = 64 three rounds against two are worth it from four steps on, since a
  // pair's tile takes 2 us longer to start (9 heads of 35 clusters, us by ones / in pairs, lists of 2 clusters of 64 17.1 / 20.4,
  // 6 of 64 21.6 / 22.9, 6 of 128 27.0 / 25.3; at d = 128 1 of 64 22.6 / 21.2, 6 of 128 41 / 34).
  const int rounds_of_pairs = ceil_div(P * ((n_qc + 1) / 2), sms), rounds_of_ones = ceil_div(P * n_qc, sms);
  const bool long_lists = D == 128 || keep_count || (long long)pr.keep * pr.cluster_k >= 4 * kTile;    // (of lengths not known here: taken as long)
  const bool pairs = pr.cluster_q < kTile && (long_lists ? 7LL : 8LL) * rounds_of_pairs < 5LL * rounds_of_ones && bitmap_words <= kPairBitmapWords;
  CUtensorMap maps[5];
  const int qbox = pr.cluster_q < kTile ? pr.cluster_q : kTile;
  const int kbox = min(pr.cluster_k, pairs ? kTile / 2 : kTile);  // pairs: keys in runs of 64
  bool ok = make_map(&maps[2], Vp, (size_t)P * n_kc * pr.cluster_k, D, kbox) &&
            make_map(&maps[4], vb, (size_t)P * cen_tiles * kCen, D, kCen);
  if (f8)
    ok = ok && make_map(&maps[0], q8, (size_t)P * n_qc * pr.cluster_q, D, qbox, true) &&
         make_map(&maps[1], k8, (size_t)P * n_kc * pr.cluster_k, D, kbox, true) &&
         make_map(&maps[3], c8, (size_t)P * cen_tiles * kCen, D, kCen, true);
  else
    ok = ok && make_map(&maps[0], Qp, (size_t)P * n_qc * pr.cluster_q, D, qbox) &&
         make_map(&maps[1], Kp, (size_t)P * n_kc * pr.cluster_k, D, kbox) &&
         make_map(&maps[3], kmix, (size_t)P * cen_tiles * kTile, D, kTile);
  if (!ok) return CA_ERR_CUDA;
  TcParams prm;
  prm.count_k = count_k; prm.block_idx = block_idx; prm.keep_count = keep_count; prm.perm_q = perm_q;
  prm.list_stride = list_stride;
  prm.O = static_cast<__nv_bfloat16*>(O); prm.lse = lse; prm.status = status; prm.redo = redo;
  prm.n_q = pr.n_q; prm.n_k = pr.n_k; prm.c_q = pr.cluster_q; prm.c_k = pr.cluster_k; prm.keep = pr.keep;
  prm.n_qc = n_qc; prm.n_kc = n_kc; prm.cen_tiles = cen_tiles; prm.compensate = pr.compensate;
  prm.bitmap_words = bitmap_words;
  prm.scale_log2 = scale * 1.4426950408889634f;
  prm.wait_limit = g_wait_limit;
  prm.skip_key_load = g_skip_key_load;
  prm.q_scale = sq; prm.k_scale = sk; prm.c_scale = sc;
  const int tiles_per_qc = pr.cluster_q >= kTile ? pr.cluster_q / kTile : 1;
  prm.next_tile = status + kTileWord;
  prm.n_tiles = P * (pairs ? (n_qc + 1) / 2 : n_qc * tiles_per_qc);
  const int grid = prm.n_tiles < sms ? prm.n_tiles : sms;
  int rc;
  {
    ProfScope ps(kProfAttn, st);
    auto go = [&](auto mode) {
      constexpr int M = decltype(mode)::value;
      if (f8) return launch_tc_d<128, true, M>(maps, prm, grid, st);
      return D == 64 ? launch_tc_d<64, false, M>(maps, prm, grid, st) : launch_tc_d<128, false, M>(maps, prm, grid, st);
    };
    if (pairs) rc = go(std::integral_constant<int, kPairs>{});
    else rc = pr.cluster_q < kTile ? go(std::integral_constant<int, kTwice>{}) : go(std::integral_constant<int, kWhole>{});
  }
  if (rc != CA_OK) return rc;
  ProfScope ps(kProfAttnSecond, st);
  // second pass: query tiles whose scores left the range of the fast softmax (a climb of more than
  // 2^96 within the steps that the reference lags behind) are recomputed by the fp32 kernel; its CTAs
  // return at once for the others
  return launch_attn_ref(pr, Qp, Kp, Vp, ck, cv, count_k, block_idx, keep_count, list_stride, perm_q, scale, O, lse,
                         status, st, redo, tiles_per_qc, status + kRecomputedWord);
}

}  // namespace ca
