// Dense convolution with many input channels as an implicit GEMM over PIXEL ROWS fed straight from
// TMA tiles (see KOrder, "rows" order): stride 1, and stride 2 with a plane held as four sub-tiles
// (S2 below).  1x1 layers see their pixels as one run, whatever image or row they lie in.
//
// A shared-memory line (128 bytes) holds 64 channels of one pixel; the input channels are cut into
// planes of 64 (the last one zero filled by the TMA unit), and a GEMM row is a pixel of the haloed
// patch.  Tap (r, s) of plane g is the plane's tile read (r * patch width + s) lines further on, so
// one 4-D TMA load per (tile, plane) -- box 64 channels x patch width x patch rows x images, 128-byte
// swizzle, zero fill outside the image -- feeds every instruction of that plane.  Small feature
// maps are tiled several images at a time (the box's image extent), so that the 128 rows of a
// block are not mostly halo and the weights, which are far larger than the activations in these
// layers, are streamed once per group of images instead of once per image.
//
// The reduction runs over (plane g, tap row r) steps.  Each step needs k * nsl(g) * 2 chunk planes
// of weights ([n_tile rows][8] bf16, no swizzle), which stream through their own ring: a layer such
// as 160 -> 960, 3x3 has 2.8 MB of weights, 40x the activations of an image.  Output channels go in
// passes of n_tile <= 128 (256 for deep wide 1x1 layers and stride 2); accumulators (blocks of 128 rows x n_tile columns) live in tensor memory,
// two sets when they fit so that the epilogue of one work item overlaps the MMAs of the next.
//
// Roles (352 threads): warp 0 producer (issues TMA / bulk loads in consumption order),
// warps 1-2 MMA issue (blocks alternate between them), warps 3-10 epilogue (two per tensor-memory
// lane quadrant, blocks alternate).  A work item is (tile, output-channel pass); CTAs (one per SM)
// take contiguous runs of items, or a cluster of them shares one item (SPLITK below).  All waits are bounded (tc::mbar_wait).
#include <type_traits>
#include "tc_ptx.cuh"

namespace {
using namespace tc;

constexpr int kMaxA = 8;                         // activation plane stages
constexpr int kMaxB = 12;                        // weight stages
constexpr int kFirstA = 3, kFirstB = 4;          // depths reached first (weights, then activations), before the rings deepen in turn
constexpr int kMmaWarp = 1;
constexpr int kMmaWarps = 2;
constexpr int kFirstEpiWarp = kMmaWarp + kMmaWarps;
constexpr int kEpiWarps = 8;
constexpr int kConsumerThreads = (kMmaWarps + kEpiWarps) * 32;
constexpr int kThreads = 32 + kConsumerThreads;
constexpr int kBarConsumers = 7;                 // named barrier of all consumer warps
constexpr int kMaxSplit = 8;                     // CTAs that share an item
constexpr int kMaxBlocks = 2;                    // 128-row blocks per tile
constexpr int kStagePitch = 64;                  // bytes per pixel in an epilogue warp's turn-around buffer (pieces XOR-swizzled)

struct RowsParams {
  int n_img, h, w, ho, wo, c_in, c_out;
  int k, stride, pad, planes;  // planes of 64 input channels
  int tw, th, nxt, wbox, rbox, ni;   // tile: outputs per row, rows, strips per row, patch width / rows, images
  int tiles_y, img_groups;
  int grid, items_per, items_rem;    // CTAs; CTA b takes items_per (+1 if b < items_rem) work items
  int split;                         // the counts above are 128-row blocks instead: a CTA's run may begin and end inside an item
  int n_tile, nnt, n_pad;      // output channels per pass, passes, nnt * n_tile
  int planes_all;              // chunk planes of the packed weights (all 64-channel planes and taps)
  int mb;                      // blocks per tile
  int lines_img;               // rbox * wbox: GEMM rows per image of a tile
  int share;                   // halo columns (and, between images, rows) stand once: see rows_plan
  int front, tail;             // bytes of zeros in front of and behind a stage's patch (share)
  uint32_t inv_lines, inv_wbox; // ceil(2^20 / lines_img), ceil(2^20 / wbox)
  int partial;                       // weight stages of one tap column instead of a whole (plane, tap row) step
  int a_stage_bytes, a_box_bytes, b_stage_bytes;
  int sa, sb, nacc, act;
  int b_resident;              // all weights stay in shared memory (one copy per CTA)
  int ksplit, part_pitch;      // CTAs that share an item's reduction; floats between rows of their partial sums
  int off_bias, off_stage, off_b, off_a, smem_bytes;
  int tmem_cols;
};

struct Shared {
  uint64_t a_full[kMaxA], a_empty[kMaxA];
  uint64_t b_full[kMaxB], b_empty[kMaxB];
  uint64_t b_all;              // resident weights have landed
  uint64_t acc_full[2], acc_empty[2];
  uint32_t tmem_base;
  uint32_t abort;
};

// 16-channel K steps of plane g
__device__ __forceinline__ int plane_steps(const RowsParams &p, int g) {
  const int left = p.c_in - 64 * g;
  return left >= 64 ? 4 : (left + 15) >> 4;
}

// Activation plane v of an item: 64 channels of the patch, or for stride 2 one of the four sub-tiles of those, with the
// taps that read it: kr rows x kc columns, the first at position tap0 of the plane's taps in the packed weights.
struct Plane {
  int g, py, px, kr, kc, tap0;
  __device__ __forceinline__ Plane(const RowsParams &p, int v, bool s2) {
    g = v; py = 0; px = 0; kr = p.k; kc = p.k; tap0 = 0;
    if (s2) {
      g = v >> 2;
      py = (v >> 1) & 1;
      px = v & 1;
      kr = (p.k + 1 - py) >> 1;
      kc = (p.k + 1 - px) >> 1;
      tap0 = dc_s2_base(p.k, py, px);
    }
  }
};

// work item -> (pass, image group, column strip, row tile); items are ordered (tile, pass)
struct Item {
  int nt, img0, xt, ty;
  __device__ __forceinline__ void of(const RowsParams &p, int item) {
    const int tile = item / p.nnt;
    nt = item - tile * p.nnt;
    const int strip = tile / p.tiles_y;
    ty = tile - strip * p.tiles_y;
    const int ig = strip / p.nxt;
    xt = strip - ig * p.nxt;
    img0 = ig * p.ni;
  }
};

// RESIDENT: all weights of the layer (a single output-channel pass, at most 128 KB) stay in shared memory:
// one copy per CTA instead of one stream per work item.  Compile-time, so that the streaming version's
// loops carry no switches.  PARTIAL (streamed weights only): a weight stage holds one tap column of a (plane, tap row)
// step instead of all of them, for layers whose whole step does not fit twice beside the activation planes (5x5 with
// 128 outputs per pass: 82 KB).  Where it fits, the whole step is faster: half as many waits, and longer stretches of
// instructions (160 -> 960 3x3: 26.0 us whole and two deep, 30.2 us by tap columns six deep).
//
// SPLITK: a cluster of p.ksplit CTAs shares one work item, each taking a run of its (plane, tap row) steps, for layers
// with fewer items than SMs whose reduction is long (384 -> 64 3x3 on one 14 x 14 image is one item of 432
// instructions per block).  The partial sums meet in distributed shared memory -- in the rings' place, which nothing
// reads any more -- and are added in rank order; every CTA finishes its share of the outputs.  What bounds it is a chain:
// of the 11000 cycles of 960 -> 160 1x1 on one 7 x 7 image 1300 went into bias rows before the first instruction, 3000 into
// the sums of the other CTAs (a lane read 16 of every 32 bytes of theirs, twice) and 1300 into a last meeting that waited for
// the results to be stored.  Now one CTA fetches the bias, and only of its pass; a stage's first use waits for nothing;
// lanes read neighbouring 16-byte pieces, all CTAs' before the first is added; the last meeting orders only reads.
// 960 -> 160 6.3 -> 4.6 us, 960 -> 1280 9.9 -> 6.6, 384 -> 64 3x3 at 14 x 14 6.5 -> 5.4, 96 -> 144 5x5 of stride 2 at 56 x 56
// 9.6 -> 7.6, 960 -> 160 on 20 images 9.5 -> 6.1 (shared only now).  The unsplit forms are faster without these (up to 8 %).
//
// S2: stride 2.  A plane of 64 channels is four sub-tiles of every second row and column of the patch (tensor map with
// element strides 2, one load each), and tap (r, s) reads sub-tile (r & 1, s & 1) at row r >> 1, column s >> 1: each
// sub-tile is a plane of its own with a smaller kernel, and GEMM rows are output pixels as before.  Gathered by 16-byte
// cp.async (conv_tc.cu, which had these layers before), an SM took in 16 KB of patch per microsecond: 96 -> 144 5x5 to
// 28 x 28, 128 images 77 us there, 70 here; 20 images of 50 x 50 53 and 15.5; 40 -> 32 3x3, 64 images of 28 x 28, 14.0
// and 6.0; 160 -> 96 3x3, 64 images of 14 x 14, 23.6 and 11.0.
template <bool RESIDENT, bool PARTIAL, bool SPLITK, bool S2>
__device__ __forceinline__ void rows_body(const CUtensorMap &map_a, const RowsParams &p,
                                          const void *__restrict__ w_packed, const float *__restrict__ bias,
                                          const __nv_bfloat16 *__restrict__ residual, __nv_bfloat16 *__restrict__ y,
                                          DcWsHeader *ws) {
  extern __shared__ __align__(1024) uint8_t smem_raw_base[];
  __shared__ __align__(8) Shared sh;

  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw_base) + 1023) & ~uintptr_t(1023));
  uint8_t *smem_b = smem + p.off_b;
  uint8_t *smem_a = smem + p.off_a;              // 1024-byte aligned stages (the swizzle pattern repeats every 1024 bytes)
  uint8_t *smem_ones = smem + p.off_bias;        // 8 lines of the constant operand (1024-byte aligned)
  uint8_t *smem_bias = smem_ones + 1024;         // [n_pad][16 bytes]: bias as three bf16 terms, then n_tile zero rows

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile uint32_t *abort_flag = &sh.abort;

  const int bid = (int)blockIdx.x;
  // This CTA's run of work items.  When the plan balances by blocks (split), the run is counted in 128-row
  // blocks: its first item starts at block blk_first and its last one ends before blk_end; the tile and the
  // weights of such an item are still staged whole.
  int nitems = p.items_per + (bid < p.items_rem ? 1 : 0);
  int item0 = bid * p.items_per + (bid < p.items_rem ? bid : p.items_rem);
  int blk_first = 0, blk_end = p.mb;
  // Activation planes (S2: four sub-tiles of each), and this CTA's share of the item: a run of (plane, weight stage)
  // steps -- whole sub-tiles for S2, whose stages are not all alike.
  const int nv = p.planes * (S2 ? 4 : 1);
  const int unit = S2 ? 1 : (PARTIAL ? p.k * p.k : p.k);
  const int rank = SPLITK ? bid % p.ksplit : 0;
  const int st0 = SPLITK ? nv * unit * rank / p.ksplit : 0;
  const int st1 = SPLITK ? nv * unit * (rank + 1) / p.ksplit : nv * unit;
  const int v_lo = SPLITK ? st0 / unit : 0, v_hi = SPLITK ? (st1 + unit - 1) / unit : nv;
  if (SPLITK) {
    item0 = bid / p.ksplit;
    nitems = 1;
  } else if (p.split) {
    const int u0 = item0, u1 = item0 + nitems - 1;           // first and last block of the run
    item0 = u0 / p.mb;
    const int item1 = u1 / p.mb;
    nitems = item1 - item0 + 1;
    blk_first = u0 - item0 * p.mb;
    blk_end = u1 - item1 * p.mb + 1;
  }

  {
    const int t = (int)threadIdx.x;
    bool did = false;
    if (t < p.sa) { mbar_init(&sh.a_full[t], 1); mbar_init(&sh.a_empty[t], kMmaWarps); did = true; }
    else if (t >= 32 && t < 32 + p.sb) { mbar_init(&sh.b_full[t - 32], 1); mbar_init(&sh.b_empty[t - 32], kMmaWarps); did = true; }
    else if (t >= 64 && t < 66) { mbar_init(&sh.acc_full[t - 64], kMmaWarps); mbar_init(&sh.acc_empty[t - 64], kEpiWarps); did = true; }
    else if (t == 96) { sh.abort = 0; mbar_init(&sh.b_all, 1); prefetch_tensormap(&map_a); did = true; }
    if (did) asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  Item first;                                    // SPLITK: the CTA's item, worked out while the previous kernel ends
  if (SPLITK) first.of(p, item0);
  dc_pdl_enter();                                // nothing above touched global memory; everything below may
  __syncthreads();

  if (warp == 0) {
    // ================================================================== producer
    // The whole warp walks the loop (every lane observes the barriers itself); lane 0 announces the
    // bytes and issues the activation tile, the weight planes of a step are issued one per lane.
    {
      const uint32_t a_base0 = smem_u32(smem_a), b_base0 = smem_u32(smem_b);
      const char *wsrc = reinterpret_cast<const char *>(w_packed);
      int sa = 0, sb = 0;
      uint32_t pa = 0, pb = 0;
      bool a_used = false, b_used = false;       // the rings have been filled once
      bool ok = true;
      if (RESIDENT && lane == 0) {               // the whole packed buffer once
        const uint32_t all = (uint32_t)(p.planes_all * p.n_tile * 16);
        mbar_arrive_expect_tx(&sh.b_all, all);
        bulk_load(b_base0, wsrc, all, &sh.b_all);
      }
#pragma unroll 1
      for (int it = 0; it < nitems && ok; ++it) {
        Item q;
        if (SPLITK) q = first; else q.of(p, item0 + it);
#pragma unroll 1
        for (int v = v_lo; v < v_hi && ok; ++v) {
          const Plane pl(p, v, S2);
          // (SPLITK: a stage's first use, often its only one, waits for nothing)
          if ((!SPLITK || a_used) && !warp_wait(&sh.a_empty[sa], pa ^ 1, abort_flag, ws, 0x10000u | sa)) { ok = false; break; }
          if (lane == 0) {
            // channels past c_in, pixels outside the image and images past the batch arrive as zeros
            mbar_arrive_expect_tx(&sh.a_full[sa], (uint32_t)p.a_box_bytes);
            tma_load_4d(a_base0 + (uint32_t)(sa * p.a_stage_bytes + p.front), &map_a, &sh.a_full[sa], 64 * pl.g,
                        (S2 ? 2 : 1) * q.xt * p.tw - (p.share ? 0 : p.pad) + pl.px, (S2 ? 2 : 1) * q.ty * p.th - p.pad + pl.py, q.img0);
          }
          if (++sa == p.sa) { sa = 0; pa ^= 1; a_used = true; }
          const int nsl = plane_steps(p, pl.g);
          const int nplanes = (PARTIAL ? 1 : pl.kc) * nsl * 2;     // chunk planes of one weight stage
          const int nstages = PARTIAL ? pl.kr * pl.kc : pl.kr;
          const int r_lo = SPLITK && !S2 && st0 > v * unit ? st0 - v * unit : 0;
          const int r_hi = SPLITK && !S2 && st1 < (v + 1) * unit ? st1 - v * unit : nstages;
          size_t plane0 = (size_t)pl.g * p.k * p.k * 8 + (size_t)(pl.tap0 * nsl * 2) + (size_t)r_lo * nplanes;
#pragma unroll 1
          for (int r = r_lo; r < r_hi && !RESIDENT; ++r, plane0 += nplanes) {
            if ((!SPLITK || b_used) && !warp_wait(&sh.b_empty[sb], pb ^ 1, abort_flag, ws, 0x20000u | sb)) { ok = false; break; }
            // the planes of a stage are contiguous in the packed weights, with several passes too (there a
            // pass's rows of all planes are stored together): one bulk copy
            if (lane == 0) {
              const uint32_t bytes = (uint32_t)(nplanes * p.n_tile * 16);
              mbar_arrive_expect_tx(&sh.b_full[sb], bytes);
              bulk_load(b_base0 + (uint32_t)sb * (uint32_t)p.b_stage_bytes,
                        wsrc + ((size_t)q.nt * p.planes_all + plane0) * p.n_tile * 16, bytes, &sh.b_full[sb]);
            }
            if (++sb == p.sb) { sb = 0; pb ^= 1; b_used = true; }
          }
        }
      }
    }
    __syncwarp();
    if (SPLITK) { cluster_sync(); cluster_meet_relaxed(); }
  } else {
    // ---- consumer preparation
    if (warp == kMmaWarp) {
      tmem_alloc(&sh.tmem_base, (uint32_t)p.tmem_cols);
      tmem_relinquish();
    } else if (warp >= kFirstEpiWarp) {
      // The bias is added by the tensor core: one instruction per block multiplies a constant operand
      // (1.0 in the first three K elements of every line) with the bias of each output channel as three bf16
      // terms before the block's other instructions accumulate.
      // The constant operand is one 8-line group read sixteen times (group stride 0); with the 128-byte
      // swizzle the first 16-byte chunk of line r sits at chunk r.
      const int t0 = (int)threadIdx.x - kFirstEpiWarp * 32;
      for (int t = t0; t < 64; t += kEpiWarps * 32) {
        const int r = t >> 3, c = t & 7;
        reinterpret_cast<uint4 *>(smem_ones)[t] = c == r ? bias_ones() : make_uint4(0u, 0u, 0u, 0u);
      }
      if (SPLITK) {                              // the item's pass where it is added, and the zero rows
        if (rank == 0)
          for (int t = first.nt * p.n_tile + t0; t < (first.nt + 1) * p.n_tile; t += kEpiWarps * 32)
            reinterpret_cast<uint4 *>(smem_bias)[t] = bias_terms(bias && t < p.c_out ? bias[t] : 0.f);
        for (int t = t0; t < p.n_tile; t += kEpiWarps * 32) reinterpret_cast<uint4 *>(smem_bias)[p.n_pad + t] = make_uint4(0u, 0u, 0u, 0u);
      } else {
        for (int t = t0; t < p.n_pad + p.n_tile; t += kEpiWarps * 32)
          reinterpret_cast<uint4 *>(smem_bias)[t] = bias_terms(bias && t < p.c_out ? bias[t] : 0.f);
      }
      // zeros around the patches, which the loads never touch, in the stages that this CTA fills
      if (p.share) {
        const int per = (p.front + p.tail) >> 4, fills = nitems * (v_hi - v_lo), used = fills < p.sa ? fills : p.sa;
        for (int st = 0; st < used; ++st)
          for (int e = t0; e < per; e += kEpiWarps * 32) {
            uint8_t *at = smem_a + st * p.a_stage_bytes + (e * 16 < p.front ? e * 16 : p.a_box_bytes + e * 16);
            *reinterpret_cast<uint4 *>(at) = make_uint4(0u, 0u, 0u, 0u);
          }
      }
      fence_proxy_async();                       // all are read by the tensor core (async proxy)
    }
    tc_fence_before();
    bar_sync(kBarConsumers, kConsumerThreads);
    tc_fence_after();
    const uint32_t tmem_base = sh.tmem_base;

    if (warp < kFirstEpiWarp) {
      // ================================================================== MMA issue
      const int mw = warp - kMmaWarp;
      // one election for the whole role: the warp stays converged and the same lane issues every instruction
      const bool leader = elect_one();
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(p.n_tile >> 3) << 17) | (8u << 24);
      const uint32_t b_hi = (128u >> 4) | (1u << 14);                 // no swizzle: 128 bytes between 8-row groups
      const uint32_t a_hi = (1024u >> 4) | (1u << 14) | (2u << 29);   // 128-byte swizzle: 1024 bytes between 8-row groups
      const uint32_t a_row0 = (smem_u32(smem_a) + (uint32_t)(p.front - (p.share ? p.pad * 128 : 0))) >> 4, b_row0 = smem_u32(smem_b) >> 4;
      const uint32_t bias_row0 = smem_u32(smem_bias) >> 4, zero_row = bias_row0 + (uint32_t)p.n_pad;
      const uint64_t ones_desc = ((uint64_t)((1u << 14) | (2u << 29)) << 32) | (uint64_t)(((smem_u32(smem_ones) >> 4) & 0x3FFFu) | (1u << 16));
      int sa = 0, sb = 0;
      uint32_t pa = 0, pb = 0;
      uint32_t acc_ph[2] = {1u, 1u};             // parity this warp waits for on acc_empty (first use passes)
      bool ok = true;
      if (RESIDENT) {
        ok = warp_wait(&sh.b_all, 0, abort_flag, ws, 0x70000u);
        tc_fence_after();
      }
#pragma unroll 1
      for (int it = 0; it < nitems && ok; ++it) {
        const int set = p.nacc == 2 ? (it & 1) : 0;
        const int blk_lo = it == 0 ? blk_first : 0, blk_hi = it == nitems - 1 ? blk_end : p.mb;   // this run's blocks of the item
        if (!warp_wait(&sh.acc_empty[set], acc_ph[set], abort_flag, ws, 0x30000u | set)) break;
        acc_ph[set] ^= 1u;
        tc_fence_after();
        {
          // bias first (needs no load): it also initialises the accumulators of this warp's blocks
          Item iq;
          if (SPLITK) iq = first; else iq.of(p, item0 + it);
          // (with the reduction split, one CTA adds the bias and the others start from zero rows)
          const uint32_t bias_row = SPLITK && rank > 0 ? zero_row : bias_row0 + (uint32_t)(iq.nt * p.n_tile);
          const uint64_t bd = ((uint64_t)b_hi << 32) | (uint64_t)((bias_row & 0x3FFFu) | ((zero_row - bias_row) << 16));
#pragma unroll 1
          for (int b = blk_lo + mw; b < blk_hi; b += kMmaWarps)
            if (leader) umma_bf16(tmem_base + (uint32_t)((set * p.mb + b) * p.n_tile), ones_desc, bd, idesc, 0u);
        }
#pragma unroll 1
        for (int v = v_lo; v < v_hi && ok; ++v) {
          const Plane pl(p, v, S2);
          if (!warp_wait(&sh.a_full[sa], pa, abort_flag, ws, 0x40000u | sa)) { ok = false; break; }
          tc_fence_after();
          const uint32_t a_stage = a_row0 + (uint32_t)sa * ((uint32_t)p.a_stage_bytes >> 4);
          const int nsl = plane_steps(p, pl.g);
          const int nstages = PARTIAL ? pl.kr * pl.kc : pl.kr;
          const int r_lo = SPLITK && !S2 && st0 > v * unit ? st0 - v * unit : 0;
          const int r_hi = SPLITK && !S2 && st1 < (v + 1) * unit ? st1 - v * unit : nstages;
          int col = PARTIAL && SPLITK ? r_lo % pl.kc : 0;          // PARTIAL: tap column of the stage
          uint32_t tap_off = (uint32_t)(((PARTIAL ? r_lo / pl.kc : r_lo) * p.wbox + col) * 8);   // of the stage's first tap, in 16-byte units
#pragma unroll 1
          for (int r = r_lo; r < r_hi; ++r) {
            uint32_t b_stage;
            if (RESIDENT) {
              b_stage = b_row0 + (uint32_t)((pl.g * p.k * p.k * 8 + (pl.tap0 + r * pl.kc) * nsl * 2) * p.n_tile);   // planes before this step
            } else {
              if (!warp_wait(&sh.b_full[sb], pb, abort_flag, ws, 0x50000u | sb)) { ok = false; break; }
              tc_fence_after();
              b_stage = b_row0 + (uint32_t)sb * ((uint32_t)p.b_stage_bytes >> 4);
            }
            // One lane issues the step's instructions in one stretch and the warp meets again behind it: with a
            // branch around every single instruction the warp diverged and met again each time, ~130 cycles per
            // instruction where the instruction itself takes ~50.  (Measured the same: every lane executing the
            // instruction under the leader's predicate, no branch at all.)
            if (leader) {
#pragma unroll 1
              for (int b = blk_lo + mw; b < blk_hi; b += kMmaWarps) {
                const uint32_t d = tmem_base + (uint32_t)((set * p.mb + b) * p.n_tile);
                // descriptors advance by adds only: +8 (one line) per tap column, +2 (32 bytes) per K step on
                // the activation side, two chunk planes per instruction on the weight side
                uint32_t a_lo = ((a_stage + (uint32_t)(b * 1024) + tap_off) & 0x3FFFu) | (1u << 16);
                uint32_t b_lo = (b_stage & 0x3FFFu) | ((uint32_t)p.n_tile << 16);
                const uint32_t b_inc = 2u * (uint32_t)p.n_tile;
                if (nsl == 4) {                  // a full plane of 64 channels
#pragma unroll 1
                  for (int s = 0; s < (PARTIAL ? 1 : pl.kc); ++s, a_lo += 8u) {
#pragma unroll
                    for (int sl = 0; sl < 4; ++sl) {
                      umma_bf16(d, ((uint64_t)a_hi << 32) | (uint64_t)(a_lo + 2u * sl), ((uint64_t)b_hi << 32) | (uint64_t)b_lo, idesc, 1u);
                      b_lo += b_inc;
                    }
                  }
                } else {
#pragma unroll 1
                  for (int s = 0; s < (PARTIAL ? 1 : pl.kc); ++s, a_lo += 8u) {
#pragma unroll 1
                    for (int sl = 0; sl < nsl; ++sl) {
                      umma_bf16(d, ((uint64_t)a_hi << 32) | (uint64_t)(a_lo + 2u * sl), ((uint64_t)b_hi << 32) | (uint64_t)b_lo, idesc, 1u);
                      b_lo += b_inc;
                    }
                  }
                }
              }
            }
            __syncwarp();
            if (!RESIDENT) {
              if (leader) umma_commit(&sh.b_empty[sb]);    // this warp is done with the weight stage
              if (++sb == p.sb) { sb = 0; pb ^= 1; }
            }
            if (!PARTIAL) {
              tap_off += (uint32_t)(p.wbox * 8);
            } else if (++col == pl.kc) {
              col = 0;
              tap_off += (uint32_t)((p.wbox - pl.kc + 1) * 8);
            } else {
              tap_off += 8u;
            }
          }
          if (ok && leader) umma_commit(&sh.a_empty[sa]);  // ... and with the plane
          if (++sa == p.sa) { sa = 0; pa ^= 1; }
        }
        if (ok && leader) umma_commit(&sh.acc_full[set]);  // this warp's blocks of the item are complete
      }
    } else {
      // ================================================================== epilogue
      // Two warps per tensor-memory lane quadrant; blocks alternate between them.  A thread owns a
      // GEMM row = one pixel of the patch; valid ones store their n_tile channels 16 bytes at a time.
      const int ew = warp - kFirstEpiWarp;
      const int q = warp & 3, par = ew >> 2;
      const uint32_t tmem_row = tmem_base + ((uint32_t)(q * 32) << 16);
      // this warp's turn-around buffer, as 32-bit shared addresses: where this lane writes its pixel, and where it
      // reads the piece it stores of pixel lane / 4 (the three other pixels lie 8 * kStagePitch bytes apart)
      const uint32_t stage = smem_u32(smem + p.off_stage + ew * (32 * kStagePitch));
      // 16-byte piece g of pixel px sits at piece g ^ ((px >> 1) & 3) of the pixel's 64 bytes: the eight lanes of a
      // quarter warp then touch eight different 16-byte bank groups both when every lane writes piece g of its own
      // pixel and when four lanes read the four pieces of each of two neighbouring pixels
      const uint32_t stage_wr = stage + (uint32_t)lane * kStagePitch, swz_wr = (uint32_t)((lane >> 1) & 3);
      const uint32_t stage_rd = stage + (uint32_t)(lane >> 2) * kStagePitch +
                                (uint32_t)((lane & 3) ^ ((lane >> 3) & 3)) * 16u;
      uint32_t acc_ph[2] = {0u, 0u};
      const bool relu6 = p.act == DC_ACT_RELU6;
      if (SPLITK && warp_wait(&sh.acc_full[0], 0u, abort_flag, ws, 0x60000u)) {
        // all of this CTA's instructions are done, so its rings hold nothing any more: the partial sums go there
        tc_fence_after();
        const uint32_t part = smem_u32(smem_a);
#pragma unroll 1
        for (int b = p.mb == 1 ? 0 : par; b < p.mb; b += 2) {   // one block: the two warps of a quadrant take its columns in turn
          const uint32_t row = part + (uint32_t)(b * 128 + q * 32 + lane) * (uint32_t)(p.part_pitch * 4);
          const uint32_t taddr = tmem_row + (uint32_t)(b * p.n_tile);
#pragma unroll 1
          for (int ch = p.mb == 1 ? par * 16 : 0; ch < p.n_tile; ch += p.mb == 1 ? 32 : 16) {
            uint32_t v[16];
            tmem_ld16(taddr + (uint32_t)ch, v);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; i += 4) sts_u4(row + (uint32_t)(ch + i) * 4u, make_uint4(v[i], v[i + 1], v[i + 2], v[i + 3]));
          }
        }
      }
#pragma unroll 1
      for (int it = 0; it < nitems && !SPLITK; ++it) {
        const int set = p.nacc == 2 ? (it & 1) : 0;
        Item iq;
        iq.of(p, item0 + it);
        if (!warp_wait(&sh.acc_full[set], acc_ph[set], abort_flag, ws, 0x60000u | set)) break;
        acc_ph[set] ^= 1u;
        tc_fence_after();
        const int x0 = iq.xt * p.tw, y0 = iq.ty * p.th;
        const int tw_valid = p.wo - x0 < p.tw ? p.wo - x0 : p.tw;
        const int th_valid = p.ho - y0 < p.th ? p.ho - y0 : p.th;
        const int ch0 = iq.nt * p.n_tile;
        const int nch = p.c_out - ch0 < p.n_tile ? p.c_out - ch0 : p.n_tile;   // multiple of 8
        const int blk_lo = it == 0 ? blk_first : 0, blk_hi = it == nitems - 1 ? blk_end : p.mb;   // this run's blocks of the item
#pragma unroll 1
        for (int b = blk_lo + par; b < blk_hi; b += 2) {
          const int pos = b * 128 + q * 32 + lane;
          // pos < 256 and the divisors are below 2^12: multiplying by the rounded-up reciprocal is exact
          const int il = (int)(((uint32_t)pos * p.inv_lines) >> 20), rem = pos - il * p.lines_img;
          const int yy = (int)(((uint32_t)rem * p.inv_wbox) >> 20), xx = rem - yy * p.wbox;
          const bool valid = il < p.ni && iq.img0 + il < p.n_img && yy < th_valid && xx < tw_valid;
          // (the plan keeps the pixel count of the output below 2^31)
          const int pix = ((iq.img0 + il) * p.ho + (y0 + yy)) * p.wo + (x0 + xx);
          __nv_bfloat16 *dst = y + (size_t)pix * p.c_out + ch0;
          const __nv_bfloat16 *rp = residual ? residual + (size_t)pix * p.c_out + ch0 : nullptr;
          const uint32_t taddr = tmem_row + (uint32_t)((set * p.mb + b) * p.n_tile);
          // eight channels of this thread's pixel: skip input, activation -> eight bf16
          // (RELU and RES are compile-time: the per-pixel code carries no run-time switches)
          auto cook8 = [&](auto RELU, auto RES, const uint32_t *v, int ch) {
            float f[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) f[i] = __uint_as_float(v[i]);     // the bias is in the accumulator already
            if (decltype(RES)::value && valid) {
              const uint4 rv = *reinterpret_cast<const uint4 *>(rp + ch);
              const __nv_bfloat162 *rb = reinterpret_cast<const __nv_bfloat162 *>(&rv);
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const float2 rf = __bfloat1622float2(rb[i]);
                f[2 * i] += rf.x; f[2 * i + 1] += rf.y;
              }
            }
            uint4 ov;
            uint32_t *ow = reinterpret_cast<uint32_t *>(&ov);
#pragma unroll
            for (int i = 0; i < 4; ++i)
              ow[i] = decltype(RELU)::value ? relu6_bf16x2(f[2 * i], f[2 * i + 1]) : pack_bf16x2(f[2 * i], f[2 * i + 1]);
            return ov;
          };
          // 32 accumulator columns per read while they last.  A thread owns a pixel, so stored directly
          // its 16-byte pieces would land c_out * 2 bytes apart from its neighbours' (half-filled
          // sectors, 32 lines per instruction).  The warp instead turns the 32 pixels x 64 bytes around
          // in its staging buffer (64-byte pitch, pieces XOR-swizzled: conflict-free both ways) and writes them four lanes to a
          // pixel: every store instruction then fills eight whole 64-byte segments.
          const uint32_t vmask = __ballot_sync(0xffffffffu, valid);
          // the four pixels this lane helps to store (pixel i * 8 + lane / 4 of the warp's 32): their addresses
          // come from the lanes that own them, once per block
          uint8_t *px_ptr[4];                              // + 16 bytes per lane of the four that share a pixel
          bool px_on[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            px_ptr[i] = reinterpret_cast<uint8_t *>((uintptr_t)__shfl_sync(0xffffffffu, (unsigned long long)(uintptr_t)dst, i * 8 + (lane >> 2))) + (lane & 3) * 16;
            px_on[i] = (vmask >> (i * 8 + (lane >> 2))) & 1u;
          }
          auto emit32 = [&](auto RELU, auto RES, const uint32_t *v, int c0) {
#pragma unroll
            for (int g8 = 0; g8 < 4; ++g8) sts_u4(stage_wr + (((uint32_t)g8 ^ swz_wr) << 4), cook8(RELU, RES, v + 8 * g8, c0 + 8 * g8));
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const uint4 piece = lds_u4(stage_rd + (uint32_t)(i * 8 * kStagePitch));
              if (px_on[i]) *reinterpret_cast<uint4 *>(px_ptr[i] + (size_t)c0 * 2) = piece;
            }
            __syncwarp();
          };
          auto channels = [&](auto RELU, auto RES) {
            int ch = 0;
#pragma unroll 1
            for (; ch + 32 <= nch; ch += 32) {
              uint32_t v[32];
              tmem_ld32(taddr + (uint32_t)ch, v);
              tmem_ld_wait();
              emit32(RELU, RES, v, ch);
            }
#pragma unroll 1
            for (; ch < nch; ch += 8) {
              uint32_t v[8];
              tmem_ld8(taddr + (uint32_t)ch, v);
              tmem_ld_wait();
              const uint4 ov = cook8(RELU, RES, v, ch);
              if (valid) *reinterpret_cast<uint4 *>(dst + ch) = ov;
            }
          };
          using T = std::true_type;
          using F = std::false_type;
          if (relu6) { if (rp) channels(T{}, T{}); else channels(T{}, F{}); }
          else { if (rp) channels(F{}, T{}); else channels(F{}, F{}); }
        }
        // this warp has read what it needs of the accumulator set
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.acc_empty[set]);
      }
    }
    if (SPLITK) {
      cluster_sync();                              // every CTA's partial sums are written
      if (warp >= kFirstEpiWarp && !*abort_flag) {
        const Item iq = first;
        const int x0 = iq.xt * p.tw, y0 = iq.ty * p.th;
        const int tw_valid = p.wo - x0 < p.tw ? p.wo - x0 : p.tw;
        const int th_valid = p.ho - y0 < p.th ? p.ho - y0 : p.th;
        const int ch0 = iq.nt * p.n_tile;
        const int quads = (p.c_out - ch0 < p.n_tile ? p.c_out - ch0 : p.n_tile) >> 2;
        const uint32_t part = smem_u32(smem_a);
        const bool relu6 = p.act == DC_ACT_RELU6;
        // 4 channels of a pixel at a time, dealt out over the threads of the whole cluster: lanes read 16 neighbouring bytes
#pragma unroll 1
        for (int u = rank * (kEpiWarps * 32) + (int)threadIdx.x - kFirstEpiWarp * 32; u < p.mb * 128 * quads; u += p.ksplit * kEpiWarps * 32) {
          const int pos = u / quads, ch = (u - pos * quads) * 4;
          const int il = (int)(((uint32_t)pos * p.inv_lines) >> 20), rem = pos - il * p.lines_img;
          const int yy = (int)(((uint32_t)rem * p.inv_wbox) >> 20), xx = rem - yy * p.wbox;
          if (il >= p.ni || iq.img0 + il >= p.n_img || yy >= th_valid || xx >= tw_valid) continue;
          const uint32_t at = part + (uint32_t)(pos * p.part_pitch + ch) * 4u;
          uint4 v[kMaxSplit];                      // all are asked for before the first is added
#pragma unroll
          for (int r = 0; r < kMaxSplit; ++r)
            if (r < p.ksplit) v[r] = lds_cluster_u4(map_cluster(at, (uint32_t)r));
          float f[4] = {};
#pragma unroll
          for (int r = 0; r < kMaxSplit; ++r)
            if (r < p.ksplit) {
              f[0] += __uint_as_float(v[r].x); f[1] += __uint_as_float(v[r].y);
              f[2] += __uint_as_float(v[r].z); f[3] += __uint_as_float(v[r].w);
            }
          const size_t o = ((size_t)((iq.img0 + il) * p.ho + (y0 + yy)) * p.wo + (x0 + xx)) * p.c_out + ch0 + ch;
          if (residual) {
            const uint2 rv = *reinterpret_cast<const uint2 *>(residual + o);
            const __nv_bfloat162 *rb = reinterpret_cast<const __nv_bfloat162 *>(&rv);
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              const float2 rf = __bfloat1622float2(rb[i]);
              f[2 * i] += rf.x; f[2 * i + 1] += rf.y;
            }
          }
          uint2 ov;
          ov.x = relu6 ? relu6_bf16x2(f[0], f[1]) : pack_bf16x2(f[0], f[1]);
          ov.y = relu6 ? relu6_bf16x2(f[2], f[3]) : pack_bf16x2(f[2], f[3]);
          *reinterpret_cast<uint2 *>(y + o) = ov;
        }
      }
      cluster_meet_relaxed();                      // nobody leaves while its sums may still be read
    }
    // ---- consumer teardown
    if (*abort_flag) {
      const unsigned long long t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    tc_fence_before();
    bar_sync(kBarConsumers, kConsumerThreads);
    if (warp == kMmaWarp) {
      tc_fence_after();
      tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
    }
  }
}

template <bool RESIDENT, bool PARTIAL, bool SPLITK>
__global__ void __launch_bounds__(kThreads, 1)
k_conv_tc_rows(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ RowsParams p,
               const void *__restrict__ w_packed, const float *__restrict__ bias,
               const __nv_bfloat16 *__restrict__ residual, __nv_bfloat16 *__restrict__ y, DcWsHeader *ws) {
  rows_body<RESIDENT, PARTIAL, SPLITK, false>(map_a, p, w_packed, bias, residual, y, ws);
}
// stride 2
template <bool RESIDENT, bool PARTIAL, bool SPLITK>
__global__ void __launch_bounds__(kThreads, 1)
k_conv_tc_rows_s2(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ RowsParams p,
                  const void *__restrict__ w_packed, const float *__restrict__ bias,
                  const __nv_bfloat16 *__restrict__ residual, __nv_bfloat16 *__restrict__ y, DcWsHeader *ws) {
  rows_body<RESIDENT, PARTIAL, SPLITK, true>(map_a, p, w_packed, bias, residual, y, ws);
}

// ------------------------------------------------------------------------------------------ host
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void *ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

constexpr int kSmemBudget = 220 * 1024;
constexpr int kSlack = 1024;

// Shared memory in front of the rings: constant operand, bias rows and zero rows, the epilogue warps' buffers.
int rows_fixed_bytes(const KOrder &ko, int *off_stage) {
  *off_stage = (int)dc_round_up((size_t)1024 + (size_t)(ko.n_pad + ko.n_tile) * 16, 128);
  return (int)dc_round_up((size_t)*off_stage + kEpiWarps * 32 * kStagePitch, 1024);
}

// Clusters of `size` CTAs (an SM's shared memory each) the current device runs at once: a property of its GPCs, asked for
// once per device.  Without a device (planning on the host): a B200's.
int max_clusters(int size) {
  static constexpr int kB200[kMaxSplit + 1] = {0, 148, 74, 45, 33, 26, 22, 15, 15};
  static int cached[kDcMaxDevices][kMaxSplit + 1];
  const int dev = dc_current_device();
  if (dev < 0) { (void)cudaGetLastError(); return kB200[size]; }
  if (cached[dev][size] == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)size * 64);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBudget;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)size;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    static unsigned char attr_done[kDcMaxDevices];
    if (dc_set_max_smem_once(k_conv_tc_rows<false, false, true>, kSmemBudget, attr_done) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, k_conv_tc_rows<false, false, true>, &cfg) != cudaSuccess || n <= 0) {
      (void)cudaGetLastError();
      n = kB200[size];
    }
    cached[dev][size] = n;
  }
  return cached[dev][size];
}

bool make_rows_plan(int n, int h, int w, const dc_geom *g, int n_sm, RowsParams *p) {
  KOrder ko;
  dc_korder_init(&ko, g);
  if (!ko.rows) return false;
  if ((long long)n * h * w * g->c_in >= (1ll << 40) || (long long)n * h * w >= (1ll << 31)) return false;
  // a 1x1 layer does not know rows or images: its pixels are one run, which tiles cut without a remainder per row
  if (g->k == 1 && g->pad == 0) { w *= n * h; n = 1; h = 1; }
  const int S = g->stride, ho = dc_out_extent(h, g->k, S, g->pad), wo = dc_out_extent(w, g->k, S, g->pad);
  const int halo = S == 2 ? (g->k - 1) / 2 : g->k - 1, subs = S == 2 ? 4 : 1;      // of a plane (sub-tile); sub-tiles per plane
  if (ho <= 0 || wo <= 0 || (long long)n * ho * wo >= (1ll << 31)) return false;
  p->n_img = n; p->h = h; p->w = w; p->ho = ho; p->wo = wo;
  p->c_in = g->c_in; p->c_out = g->c_out;
  p->k = g->k; p->stride = S; p->pad = g->pad;
  p->planes = dc_div_up(g->c_in, 64);
  p->n_tile = ko.n_tile; p->nnt = ko.nnt; p->n_pad = ko.n_pad;
  p->planes_all = ko.e_pad;
  p->off_bias = 0;
  p->off_a = rows_fixed_bytes(ko, &p->off_stage);
  // A tile's GEMM rows are the patch pixels from its first to its last output, halo columns included: at most two
  // 128-row blocks.  Its patch (rows and halo) must fit the activation ring twice beside three weight stages.
  // weights of one tap column of a (plane, tap row) step: two chunk planes for each 16 channels of the widest plane.
  // (Counted as eight for every plane, the steps of 16 to 48 channels seemed not to fit and ran by tap columns of one to
  // three instructions: 32 -> 224 5x5, 10 images of 23 x 23 10.8 us, now 6.8.)
  const long long tap_bytes = (g->c_in >= 64 ? 8ll : 2ll * dc_div_up(g->c_in, 16)) * p->n_tile * 16;
  const long long max_a = (kSmemBudget - 1024 - p->off_a - kSlack - (3 * tap_bytes > 26 * 1024 ? 3 * tap_bytes : 26 * 1024)) / 2;
  // Tile and split of the reduction: the least estimated time of the CTA with the most work, in cycles.  An item costs
  // its tensor-core instructions (a 128 x N x 16 takes max(36 + N/4, N/2)) and the bytes it takes in from L2, which
  // overlap in part, and a chain of waits; a shared item costs the meeting of its partial sums, which grows with the
  // CTAs and the bytes.  The constants are fitted to 41 layers timed in every tile and split considered here (1 to 128
  // images of 49 to 12544 pixels).  Timed again on 32 layers: the choice is 2 % above the best on
  // average, 21 % at worst (160 -> 96 3x3 of stride 2, 64 images of 14 x 14).  Whether a split beats the best tile by itself is
  // asked with terms of its own, fitted to 237 layers of 1 to 128 images (20 to 6272 pixels) in up to nine tiles and splits:
  // 1.2 % above the best of those on average, 1.19 times at worst, none more than 3 % slower than unsplit; with the one
  // estimate that both shared before, fitted to a meeting of twice the time, 4.9 % and 1.64 times.
  // Candidates: every strip count that leaves rows of at most 256 pixels, with as many rows as give two blocks or
  // one, evened out over the height; whole small images several at a time.
  const int cyc = 36 + p->n_tile / 4 > p->n_tile / 2 ? 36 + p->n_tile / 4 : p->n_tile / 2;
  const double per_block = (double)g->k * g->k * dc_div_up(g->c_in, 16) * cyc;
  const double w_item = (double)ko.e_pad * p->n_tile * 16;
  double best = 0.0, best_shared = 0.0;          // of the best tile by itself; the same tile beside the shared ones
  struct { double cost; int nxt, tw, th, ni, ksplit; bool halos; } sp = {0.0, 0, 0, 0, 0, 1, false};   // the best shared one
  p->nxt = 0;
  p->ksplit = 1;
  p->share = 0;
  const int fixed_part = kSmemBudget - 1024 - p->off_a;     // bytes of the rings, where partial sums would go
  // Tiles of whole rows: the halo column right of a row is the one left of the next row (a load starts at column 0 and ends
  // pad columns past the last), and in tiles of several images the halo rows below one image are those above the next; the
  // zeros in front of the first and behind the last stand in shared memory and are never loaded over.  Of the 128 rows
  // that an instruction multiplies more are outputs, 98 instead of 74 for 3x3 at 7 x 7 (two images in 128 rows, before
  // three in 256): 160 -> 960, 128 images 28.9 -> 20.8 us.  Taken where the estimate is 8 % lower than that of the best tile with
  // both halos.  Of two tiles alike but for that the shared one is up to 5 % slower (zeros to write, patches that no longer start on
  // a swizzle's boundary), and where few blocks are saved the estimate cannot tell (160 -> 144 3x3, 16 images of 106 x
  // 106: 89.4 us by 106 x 2 shared, 80.4 by 18 x 12; 144 -> 144 5x5, 41 of 41 x 41: 90.0 by 41 x 3, 79.8 by 14 x 14).  Of 180 layers
  // timed in up to ten tiles the choice is 1.5 % above the best on average, none more than 2 % slower than without sharing; any line from 6
  // to 10 % gives the same; without one 1.7 % and three.
  const bool may_share = S == 1 && g->pad > 0 && 2 * g->pad == g->k - 1 && g->pad <= 8;
  auto stage_bytes = [&](int lines, int ni, int wbox, bool share) {
    return (long long)dc_round_up((size_t)ni * lines * 128 + (share ? 1024 + (ni > 1 ? g->pad * wbox * 128 : 0) : 0), 1024);
  };
  auto consider_form = [&](int tw, int th, int ni, bool share) {
    const int wbox = share ? tw + g->pad : tw + halo, rbox = share && ni > 1 ? th + g->pad : th + halo;
    if (S * wbox > 256 || S * rbox > 256) return;
    const int lines = rbox * wbox;
    if (stage_bytes(lines, ni, wbox, share) > max_a) return;
    const int mb = dc_div_up((ni - 1) * lines + (th - 1) * wbox + tw, 128);
    if (mb > kMaxBlocks) return;
    const int nxt = dc_div_up(wo, tw);
    const long long items = (long long)dc_div_up(n, ni) * nxt * dc_div_up(ho, th) * p->nnt;
    const long long per_cta = (items + n_sm - 1) / n_sm, blocks = (items * mb + n_sm - 1) / n_sm;
    const double mma = 1.7 * (double)(blocks < per_cta * mb ? blocks : per_cta * mb) * per_block;
    const double bytes = (double)ni * lines * 128 * p->planes * subs + w_item;
    const double all = (double)items * bytes / 8000.0;               // what L2 gives all SMs together
    // Where a whole step does not fit twice beside two planes the weights come by tap columns, each with a wait of its own
    // behind a handful of instructions: 150 cycles a column.  Of 1500 random 3x3, 5x5 and 7x7 layers 33 became 1.06 to 1.5
    // times as fast (72 -> 64 7x7, 29 images of 28 x 55: 51.3 -> 34.4 us), three 1.08 times slower.  Not at stride 2, whose
    // steps are short and where five became slower (176 -> 104 7x7, 6 images of 76 x 76: 24.5 -> 30.9 us) and none faster.
    const long long whole = (long long)dc_round_up((size_t)(g->k * tap_bytes), 1024);
    const bool columns = S == 1 && g->k > 1 && 2048 + p->off_a + 2 * whole + 2 * stage_bytes(lines, ni, wbox, share) > kSmemBudget;
    const double waits = columns ? 150.0 * (double)per_cta * p->planes * g->k * g->k : 0.0;
    const double line = share ? 1.08 : 1.0;
    auto estimate = [&](int split, double more) {
      const double m = mma / split, one = (double)per_cta * bytes / split / 67.0, l = one > all ? one : all;
      const double ctas = (double)(items * split < n_sm ? items * split : n_sm);
      return line * ((m > l ? m + 0.77 * l : l + 0.77 * m) + waits / split + 1700.0 * (double)per_cta + 1.1 * lines * ni + 30.0 * ctas + more);
    };
    // Beside the shared items a step and a plane have a price of their own, and a shared one pays for the meeting: the CTAs
    // that meet, the sums that each writes and reads and the results.
    // (At stride 2, items that three CTAs or more share take a quarter less than these terms say.  Of 158 layers at stride 2 the
    // choice takes 0.986 of the time that it takes without this, none more: 72 -> 216 3x3, 20 images of 17 x 12, 9.8 us unsplit, 7.4
    // by six CTAs; 64 -> 696, two of 12 x 7, 7.7 and 5.9 by four.)
    auto shared = [&](int split) {
      const double s2 = S == 2 && split > 2 ? 0.72 : 1.0;
      const int steps = dc_div_up(p->planes * g->k * S, split), pl = dc_div_up(p->planes, split);
      const double sums = p->n_tile * (0.5 * ni * th * tw + mb * 128 * (0.2 + 0.5 / split));
      return s2 * estimate(split, (double)per_cta * (600.0 * steps + 800.0 * pl) + 3.9 * lines * ni + (split > 1 ? 500.0 + 200.0 * split + sums : 0.0));
    };
    const double alone = estimate(1, 0.0);
    if (p->nxt == 0 || alone < best) { best = alone; best_shared = shared(1); p->nxt = nxt; p->tw = tw; p->th = th; p->ni = ni; p->share = share; }
    for (int split = 2; split <= kMaxSplit; ++split) {
      // A shared item: all clusters at once, at least one (plane, tap row) step per CTA, partial sums in the rings' place.
      if (split == 7) continue;                  // no more clusters of seven than of eight run at once (15 each)
      if (items * split > n_sm || items > max_clusters(split) || p->planes * (S == 2 ? 4 : g->k) < split ||
          mb * 128 * (p->n_tile + 4) * 4 > fixed_part)
        break;
      const double cost = shared(split);
      if (sp.ksplit == 1 || cost < sp.cost) sp = {cost, nxt, tw, th, ni, split, share};
    }
  };
  auto consider = [&](int tw, int th, int ni) {
    consider_form(tw, th, ni, false);
    if (may_share && tw == wo) consider_form(tw, th, ni, true);
  };
  // The fewest strips whose tile of one output row is within the tensor map's box (256 pixels) and the activation ring
  // (max_a, in whole kilobytes).  The ring is the tighter bound for 5x5 and 7x7 kernels, whose weight stages leave it
  // less room and whose patches have more rows: 128 -> 128 7x7 has strips of at most 78 outputs, not 250.
  const long long ring = max_a / 1024 * 8 / (1 + halo) - halo, box = 256 / S - halo;
  const int strip = (int)(ring < box ? ring : box);
  if (strip < 1) return false;
  const int nxt0 = dc_div_up(wo, strip);
  if (ho == 1 && g->k == 1) {
    // one run of pixels: full tiles, or as many as there are CTAs to take them
    consider(wo < 256 ? wo : 256, 1, 1);
    consider(wo < 128 ? wo : 128, 1, 1);
    for (int r = 1; r <= 4; ++r) {
      const long long tiles = (long long)r * n_sm / p->nnt;
      const long long tw = tiles > 0 ? (wo + tiles - 1) / tiles : 0;
      if (tw >= 1 && tw <= 256) consider((int)tw, 1, 1);
    }
  } else {
    for (int cand = nxt0; cand <= nxt0 + 5 && cand <= wo; ++cand) {
      const int tw = dc_div_up(wo, cand);
      for (int share = 0; share <= (may_share && tw == wo ? 1 : 0); ++share) {
        int last_th = 0;
        for (int mb = kMaxBlocks; mb >= 1; --mb) {
          if (mb * 128 < tw) break;
          int th = (mb * 128 - tw) / (tw + (share ? g->pad : halo)) + 1;
          if (th > ho) th = ho;
          if (th != last_th) consider_form(tw, th, 1, share != 0);
          last_th = th;
          const int even = dc_div_up(ho, dc_div_up(ho, th));
          if (even != th) consider_form(tw, even, 1, share != 0);
        }
      }
      if (p->nxt == 0) consider(tw, 1, 1);
    }
    if (nxt0 == 1)
      for (int ni = 2; ni <= 8 && ni <= n; ++ni) consider(wo, ho, ni);
  }
  if (p->nxt == 0) return false;
  // (a hundredth less: 144 -> 144 5x5, two images of 53 x 53, was split in two for a tenth of that, 15.7 us, 13.5 unsplit)
  if (sp.ksplit > 1 && sp.cost < 0.99 * best_shared) {
    p->nxt = sp.nxt; p->tw = sp.tw; p->th = sp.th; p->ni = sp.ni; p->ksplit = sp.ksplit; p->share = sp.halos;
  }
  const int th = p->th;
  p->wbox = p->share ? p->tw + g->pad : p->tw + halo;
  p->rbox = p->share && p->ni > 1 ? th + g->pad : th + halo;
  p->front = p->share ? 1024 : 0;
  p->tail = p->share && p->ni > 1 ? g->pad * p->wbox * 128 : 0;
  p->lines_img = p->rbox * p->wbox;
  p->inv_lines = ((1u << 20) + (uint32_t)p->lines_img - 1) / (uint32_t)p->lines_img;
  p->inv_wbox = ((1u << 20) + (uint32_t)p->wbox - 1) / (uint32_t)p->wbox;
  p->tiles_y = dc_div_up(ho, th);
  p->img_groups = dc_div_up(n, p->ni);
  const int last = (p->ni - 1) * p->lines_img + (th - 1) * p->wbox + p->tw;    // GEMM rows up to the last valid one
  p->mb = dc_div_up(last, 128);
  if (p->mb > kMaxBlocks) return false;
  p->nacc = (2 * p->mb * p->n_tile <= 512) ? 2 : 1;
  if (p->nacc * p->mb * p->n_tile > 512) return false;
  int cols = 32;
  while (cols < p->nacc * p->mb * p->n_tile) cols *= 2;
  p->tmem_cols = cols;
  const long long items = (long long)p->img_groups * p->nxt * p->tiles_y * p->nnt;
  if (items >= (1ll << 30)) return false;
  p->grid = items < n_sm ? (int)items : n_sm;
  p->items_per = (int)(items / p->grid);
  p->items_rem = (int)(items % p->grid);
  // Where whole items leave some CTAs a block more than an even split would (160 -> 960, 3 x 3 at 7 x 7: 344
  // items of two blocks on 148 SMs, three items = six blocks on 48 of them against five by blocks), the runs are
  // cut by blocks: an item at a run's end is then shared by two CTAs, each staging its tile and weights.
  p->split = 0;
  if (p->mb > 1 && p->ksplit == 1) {
    const long long units = items * p->mb;
    const int grid_u = units < n_sm ? (int)units : n_sm;
    const long long whole = (items / p->grid + (items % p->grid ? 1 : 0)) * p->mb, cut = units / grid_u + (units % grid_u ? 1 : 0);
    if (cut * 8 <= whole * 7 && units < (1ll << 30)) {     // worth it from an eighth less (a shared item is staged twice)
      p->split = 1;
      p->grid = grid_u;
      p->items_per = (int)(units / grid_u);
      p->items_rem = (int)(units % grid_u);
    }
  }
  p->a_box_bytes = p->ni * p->lines_img * 128;
  p->a_stage_bytes = (int)dc_round_up((size_t)(p->front + p->a_box_bytes + p->tail), 1024);
  // Layout: bias, activation stages, weight stages.  The last block's 128 GEMM rows plus the tap shift reach at most 127
  // lines (16 KB) past its stage, because the patch holds the halo of its last output; behind the last activation stage
  // that lands in the weight stages or in room kept free for it (what is read there only feeds rows that are dropped).
  // (26 KB are kept: the constants of the estimate above were fitted with that.)
  // rings: weights first (they are the larger stream), then activation planes
  int sa = 2, sb = 2;
  // Small weights of a single pass stay resident where a work item would otherwise stream more weight than
  // activation bytes (many input planes, or a k x k kernel on few): then it streams its activation planes only.
  // (For 1 x 1 layers of one or two planes the weight stream is small beside the activations and the resident
  // version measured no faster.)
  const long long b_all = (long long)dc_round_up((size_t)ko.e_pad * p->n_tile * 16, 1024);
  p->b_resident = (p->ksplit == 1 && p->nnt == 1 && b_all <= 128 * 1024 && (p->planes >= 3 || b_all >= 2ll * p->a_stage_bytes)) ? 1 : 0;
  // a weight stage is a whole (plane, tap row) step where that fits twice
  p->partial = 0;
  p->b_stage_bytes = (int)dc_round_up((size_t)((S == 2 ? (g->k + 1) / 2 : g->k) * tap_bytes), 1024);
  auto total = [&](int a, int b) {
    const long long wbytes = p->b_resident ? b_all : (long long)b * p->b_stage_bytes;
    const long long tail = wbytes >= 26 * 1024 ? kSlack : 26 * 1024 - wbytes + kSlack;   // room for the overrun
    return 1024ll + p->off_a + wbytes + (long long)a * p->a_stage_bytes + tail;
  };
  if (p->b_resident && total(sa, sb) > kSmemBudget) p->b_resident = 0;
  if (!p->b_resident && total(sa, sb) > kSmemBudget) {
    p->partial = 1;
    p->b_stage_bytes = (int)dc_round_up((size_t)tap_bytes, 1024);
  }
  if (total(sa, sb) > kSmemBudget) return false;
  while (!p->b_resident && sb < kFirstB && total(sa, sb + 1) <= kSmemBudget) ++sb;
  while (sa < kFirstA && total(sa + 1, sb) <= kSmemBudget) ++sa;
  // Layers of many input planes with small stages (deep 1 x 1 layers: 10-30 KB per step) are bound by the
  // bytes in flight (a stage comes back ~1 us after it was asked for), so what shared memory is left deepens
  // both rings in turn.
  for (bool grew = true; grew;) {
    grew = false;
    if (!p->b_resident && sb < kMaxB && total(sa, sb + 1) <= kSmemBudget) { ++sb; grew = true; }
    if (sa < kMaxA && total(sa + 1, sb) <= kSmemBudget) { ++sa; grew = true; }
  }
  p->sa = sa; p->sb = sb;
  p->off_b = p->off_a + sa * p->a_stage_bytes;
  p->smem_bytes = (int)total(sa, sb);
  p->part_pitch = p->n_tile + 4;                 // lanes of a quarter warp 16 bytes apart in the banks
  if (p->ksplit > 1) {
    const int need = 1024 + p->off_a + p->mb * 128 * p->part_pitch * 4;
    if (p->smem_bytes < need) p->smem_bytes = need;
  }
  return true;
}

bool rows_plan(int n, int h, int w, const dc_geom *g, int n_sm, RowsParams *p) {
  static thread_local DcPlans<RowsParams> plans;
  return plans.get(DC_PLAN_KEY(n, h, w, g, n_sm), p, [&](RowsParams *q) { return make_rows_plan(n, h, w, g, n_sm, q); });
}

}  // namespace

bool dc_conv_rows_supported(int n, int h, int w, const dc_geom *g) {
  RowsParams p;
  return rows_plan(n, h, w, g, dc_sm_count(), &p);
}

dc_status dc_launch_conv_rows(const void *x, int n, int h, int w, const dc_geom *g, const void *w_packed,
                              const float *bias, dc_act act, const void *residual, void *y, void *workspace,
                              cudaStream_t stream) {
  RowsParams p;
  const int n_sm = dc_sm_count();
  if (!rows_plan(n, h, w, g, n_sm, &p)) return DC_ERR_UNSUPPORTED;
  p.act = (int)act;
  EncodeTiledFn encode = get_encode_fn();
  if (!encode) return DC_ERR_CUDA;
  CUtensorMap map_a;
  {
    const cuuint64_t C = (cuuint64_t)g->c_in;
    cuuint64_t gdim[4] = {C, (cuuint64_t)p.w, (cuuint64_t)p.h, (cuuint64_t)p.n_img};
    cuuint64_t gstr[3] = {2 * C, (cuuint64_t)p.w * C * 2, (cuuint64_t)p.h * p.w * C * 2};
    // stride 2: the box spans 2 wbox x 2 rbox pixels and takes every second column and row
    const cuuint32_t S = (cuuint32_t)p.stride;
    cuuint32_t box[4] = {64, S * (cuuint32_t)p.wbox, S * (cuuint32_t)p.rbox, (cuuint32_t)p.ni};
    cuuint32_t es[4] = {1, S, S, 1};
    CUresult r = encode(&map_a, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(x), gdim, gstr, box, es,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return DC_ERR_CUDA;
  }
  using Kernel = decltype(&k_conv_tc_rows<false, false, false>);
  static constexpr Kernel kernels[10] = {
      k_conv_tc_rows<false, false, false>,    k_conv_tc_rows<true, false, false>,    k_conv_tc_rows<false, true, false>,
      k_conv_tc_rows<false, false, true>,     k_conv_tc_rows<false, true, true>,     k_conv_tc_rows_s2<false, false, false>,
      k_conv_tc_rows_s2<true, false, false>,  k_conv_tc_rows_s2<false, true, false>, k_conv_tc_rows_s2<false, false, true>,
      k_conv_tc_rows_s2<false, true, true>};
  static unsigned char attr_done[10][kDcMaxDevices];
  const int which = (p.stride == 2 ? 5 : 0) + (p.b_resident ? 1 : (p.partial ? 2 : 0) + (p.ksplit > 1 ? (p.partial ? 2 : 3) : 0));
  DC_CUDA_OK(dc_set_max_smem_once(kernels[which], kSmemBudget, attr_done[which]));
  const cudaError_t le = dc_launch_pdl_cluster(kernels[which], dim3(p.grid * p.ksplit), dim3(kThreads), (size_t)p.smem_bytes, stream,
                                               p.ksplit, map_a, p, w_packed, bias, (const __nv_bfloat16 *)residual,
                                               (__nv_bfloat16 *)y, (DcWsHeader *)workspace);
  return le == cudaSuccess && cudaGetLastError() == cudaSuccess ? DC_OK : DC_ERR_CUDA;
}
