// What a 1x1 layer is composed with, as one product on the tensor core, by operands cut into bf16 terms (bf16_terms2):
//   an inverted-residual block    W'[o][i][t] = g3[o] sum_c (W3[o][c] D~[c][t]) W1[c][i]       D~ = D g1 g2, rows (o, t)
//   two 1x1 layers                W'[o][i]    = g2[o] sum_c W2[o][c] W1~[c][i]
//
// A value is three bf16 terms, exactly; six products of them are above 2^-24 and take three instructions a step of 16 channels (A_h x
// [h m l], A_m x [h m], A_l x [h], sums in column groups of their own, as in conv_f32_tc.cu).  The rows of a block are made on the
// way: nine taps times a weight cost less than reading them would.
//
// A tile is 14 output channels x nine taps (126 of 128 rows), or 128 output channels, by NT input channels.  A cluster of CTAs shares
// the reduction of a tile where there are few of them.  Two teams of warps cut the steps in turn, 8 channels of a row or a column
// to a thread, the next step's weights on their way meanwhile; what is cut stays where it is for all of a CTA's steps where it fits
// (a slot is written twice at most), so there is next to nothing to wait for.  Two warps issue.  Then all add up the sums, send
// each CTA of the cluster its share of the tile, and finish it: parts in rank order, scale, identities, result, packed copy.
// The bias is summed with the channels a CTA has anyway.
//
// An infinity or a NaN among the weights makes NaN of results: such a result is computed again by FMAs.
//
// 160 -> 960 -> 160 19.7 us by FMAs (k_merge_block33), here 14.3; 200 -> 928 -> 200 39.4 -> 17.4; 960 -> 320 -> 1280 30.4 us (k_merge_11) ->
// 22.0; 320 -> 1280 -> 320 25.4 -> 14.3; small ones are left to the FMAs (24 -> 144 -> 24 6.1, here 8.2).  Of 160 channels' 20 thousand
// cycles the first weights and scales take 3, the twelve steps 8, their instructions 2 more, the meeting 3 and the shares 2 (with two
// sums of the products of the high terms, 13.9).
// Everything that runs once costs its instructions' way from memory: a third of the warps' time goes to that and to
// branches.  On the way: shares of a step dealt out over the warps by number 16.2, the same rows for each warp 14.3, one team (two steps at a time) 13.9,
// the others' sums read from their shared memory instead of sent 14.3; terms by packed subtractions the same.
#include "merge_parts.cuh"
#include "tc_ptx.cuh"

namespace {
using namespace tc;

__device__ unsigned int g_product_status;        // DC_ERR_TIMEOUT once a wait of this kernel ran out in a launch without a workspace header

constexpr int kPitchA = 128 * 16;                // bytes between the halves of a step's 16 channels
constexpr int kStepA = 6 * kPitchA;
constexpr int kMaxSlots = 16, kMaxSplit = 8;
constexpr int kSmemMax = 225 * 1024;             // asked for always: a CTA holds all of its SM's tensor memory, and clusters that did so
                                                 // beside one another on an SM could wait for each other's

// sums of the products of the high terms in the fine form: what tensor memory holds beside those of the other products
__host__ __device__ constexpr int sums_of(int nt) { return 512 / nt - 2; }
__host__ __device__ constexpr int threads_of(int nt) { return 2 * (8 + nt / 16) * 32 + 64; }      // two teams that cut, two warps that issue

// The waits of a step on its slot, which a plan uses twice at most.  A barrier's wait tells two neighbouring phases apart and no more, so
// every phase but the last must be known to be over where a wait begins.  (On the host as well: a test walks them through every order of
// events.)
//
// Terms of a second use are the second phase of their barrier, and a wait for that one returns at once while the first is still open.
// The warp that issues need not have met the first one: with an odd number of slots and two sums that was the other warp's step, and
// the teams that cut are not ordered against each other.  So it waits first until the first use is multiplied, as those that cut do.  Of
// that barrier no second phase can be over before this warp has issued the step.
#pragma nv_exec_check_disable
template <typename Wait>
__host__ __device__ __forceinline__ bool cut_waits(int step, int slots, Wait wait) {
  return step < slots || wait(kMaxSlots + step - slots, 0u);
}
#pragma nv_exec_check_disable
template <typename Wait>
__host__ __device__ __forceinline__ bool issue_waits(int step, int slots, Wait wait) {
  return step < slots ? wait(step, 0u) : wait(kMaxSlots + step - slots, 0u) && wait(step - slots, 1u);
}

template <int KIND>
struct Shape {
  static constexpr int T = KIND == kProductPair ? 1 : 9, OT = KIND == kProductPair ? 128 : 14, ROWS = OT * T;
  static constexpr int UNIT = 8 * T;             // floats of 8 input channels of an output channel
};

struct Plan {
  int n_tiles, split, steps, total_steps, slots; // a CTA's steps of 16 channels, all steps
  int off_d, off_q, off_parts;
  int fine;                                      // the products of the high terms in sums_of() sums instead of two
};

// one result by FMAs, before the last layer's scale: where the terms gave NaN
template <int KIND>
__device__ __noinline__ float sum_by_fma(const Product &a, int o, int i, int t) {
  float s = 0.f;
#pragma unroll 1
  for (int c = 0; c < a.c1; ++c) {
    const float w1 = a.l1.w[(size_t)c * a.c0 + i], g1 = raw_scale(a.l1, c);
    if (KIND == kProductBlock)
      s = fmaf((a.l2.w[(size_t)o * a.c1 + c] * (g1 * raw_scale(a.mid, c))) * w1, a.mid.w[(size_t)c * 9 + t], s);
    else
      s = fmaf(a.l2.w[(size_t)o * a.c1 + c], w1 * g1, s);
  }
  return s;
}

// the identities that ride on the layers, or on the whole, added to a scaled result
template <int KIND>
__device__ __forceinline__ float add_ident(const Product &a, bool whole, float g2, float s, int o, int i, int t) {
  if (KIND == kProductBlock) return s + (whole && t == 4 && o == i ? 1.f : 0.f);
  if (a.ident1) s = fmaf(g2, a.l2.w[(size_t)o * a.c1 + i], s);                                                 // W2 o I
  if (a.ident2) s = fmaf(raw_scale(a.l1, o), a.l1.w[(size_t)o * a.c0 + i], s);                                 // I o W1
  if (o == i) s += (a.ident1 && a.ident2 ? 1.f : 0.f) + (whole ? 1.f : 0.f);
  return s;
}

template <int KIND, int NT>
__global__ void __launch_bounds__(threads_of(NT), 1)
k_merge_product_tc(const __grid_constant__ Product a, const __grid_constant__ BlockDelivery dv, const __grid_constant__ Plan p, DcWsHeader *ws) {
  using S = Shape<KIND>;
  constexpr int T = S::T, OT = S::OT, UNIT = S::UNIT, kStep = kStepA + NT * 96;
  constexpr int kSums = sums_of(NT);
  constexpr int kTeam = 8 + NT / 16, kWarpsCut = 2 * kTeam, kIssue = kWarpsCut, kCutThreads = kWarpsCut * 32, kThreads = threads_of(NT);
  static_assert(NT % 16 == 0 && 6 * NT <= 512, "tile");
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ uint64_t bar[2 * kMaxSlots + 2];    // [slot] terms are there; [kMaxSlots + slot] they are multiplied; all sums are there; the others' parts are
  __shared__ uint32_t tmem_s, abort_s;
  __shared__ float bias_s[OT], g_last[OT], b_last[OT];
  volatile uint32_t *abort_flag = &abort_s;
  const int tid = (int)threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t sm = smem_u32(smem);
  const int c0 = a.c0, c1 = a.c1, c2 = a.c2;
  const int rank = (int)blockIdx.x % p.split, tile = (int)blockIdx.x / p.split, mt = tile / p.n_tiles, nt = tile - mt * p.n_tiles;
  const int o0 = mt * OT, i0 = nt * NT;
  const int steps = p.total_steps - rank * p.steps < p.steps ? p.total_steps - rank * p.steps : p.steps;    // at least one
  const int cb = rank * p.steps * 16, kc = c1 - cb < steps * 16 ? c1 - cb : steps * 16;
  float *z = reinterpret_cast<float *>(smem);    // the tile's sums, where the terms were: [8 input channels][o][i][t]
  if (warp == kIssue) {
    for (int b = lane; b < 2 * kMaxSlots + 2; b += 32) mbar_init(&bar[b], b < kMaxSlots ? kTeam : b < 2 * kMaxSlots ? (p.fine ? 2 : 1) : b == 2 * kMaxSlots && (p.fine || steps > 1) ? 2 : 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
    if (lane == 0) {
      abort_s = 0;
      const int all = OT * (NT / 8), per = (all + p.split - 1) / p.split, left = all - rank * per;
      if (left > 0) mbar_arrive_expect_tx(&bar[2 * kMaxSlots + 1], (uint32_t)((p.split - 1) * (left < per ? left : per) * UNIT * 4));
    }
  }
  dc_pdl_enter();                                // global memory and tensor memory only behind this
  // ---------------------------------------------------------------- cut: a warp takes 8 channels of the same 32 rows, or columns, of every step
  const int team = warp >= kTeam ? 1 : 0, cw = warp - team * kTeam;              // two teams take the steps in turn
  const bool rows = cw < 8;
  const int e = (cw - 8) * 32 + lane, half = rows ? cw >> 2 : (e >= NT ? 1 : 0);
  const int line = rows ? (cw & 3) * 32 + lane : e - half * NT, tap = line % T;
  const float *w;                                // the next step's first weight
  int rem;                                       // channels from there on
  if (rows) {
    const int o = o0 + line / T;
    const bool in = line < S::ROWS && o < c2;
    w = a.l2.w + (in ? (size_t)o * c1 + cb + team * 16 + half * 8 : 0);
    rem = in ? c1 - cb - team * 16 - half * 8 : 0;
  } else {
    const bool in = i0 + line < c0;
    w = a.l1.w + (in ? (size_t)(cb + team * 16 + half * 8) * c0 + i0 + line : 0);
    rem = in ? c1 - cb - team * 16 - half * 8 : 0;
  }
  const size_t next = rows ? 32 : (size_t)c0 * 32;
  auto load = [&](float *f) {                    // c1 is a multiple of 4
    if (rows) {
      const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
      *reinterpret_cast<float4 *>(f) = rem > 0 ? *reinterpret_cast<const float4 *>(w) : none;
      *reinterpret_cast<float4 *>(f + 4) = rem > 4 ? *reinterpret_cast<const float4 *>(w + 4) : none;
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) f[j] = rem > (j & 4) ? w[(size_t)j * c0] : 0.f;
    }
    w += next;
    rem -= 32;
  };
  float v[8];
  float *ds = reinterpret_cast<float *>(smem + p.off_d), *qs = reinterpret_cast<float *>(smem + p.off_q);
  if (warp < kWarpsCut) {
    // A thread to a channel: the scale of its taps, or of the first layer, and what its bias is multiplied by.  All that is read is
    // asked for first.
    const bool in = tid < kc;
    const int c = in ? cb + tid : 0;
    const RawNumbers n1(a.l1, c), nm(KIND == kProductBlock ? a.mid : a.l1, c);
    float dw[9], sum = 0.f;
    if (KIND == kProductBlock)
#pragma unroll
      for (int t = 0; t < 9; ++t) dw[t] = a.mid.w[(size_t)c * 9 + t];
    const int ow = kCutThreads - 1 - tid, o = ow < OT && o0 + ow < c2 ? o0 + ow : 0;
    const RawNumbers n2(a.l2, o);
    load(v);
    const float g1 = in ? n1.scale(a.l1) : 0.f;
    if (tid < steps * 16) {
      float q = n1.bias(a.l1, g1);
      if (KIND == kProductBlock) {
        const float gm = in ? nm.scale(a.mid) : 0.f, g = g1 * gm;
#pragma unroll
        for (int t = 0; t < 9; ++t) {
          ds[tid * 9 + t] = in ? dw[t] * g : 0.f;
          sum += gm * dw[t];
        }
        q = fmaf(sum, q, nm.bias(a.mid, gm));
      } else {
        ds[tid] = g1;
      }
      qs[tid] = q;
    }
    if (ow < OT) {
      const float g = n2.scale(a.l2);
      g_last[ow] = g;
      b_last[ow] = n2.bias(a.l2, g);
    }
  } else if (warp == kIssue) {
    tmem_alloc(&tmem_s, 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_s;
  bool ok = true;
  if (warp < kWarpsCut) {
    const uint32_t to = rows ? (uint32_t)(half * kPitchA + line * 16) : (uint32_t)(kStepA + half * (NT * 48) + line * 16);
    const uint32_t plane = rows ? 2 * kPitchA : NT * 16;
    const float *x = ds + (KIND == kProductBlock ? (team * 16 + half * 8) * 9 + tap : team * 16 + half * 8);
#pragma unroll 1
    for (int s = team; s < steps; s += 2) {      // a step's weights become terms while the next one's are on their way
      float n[8];
      load(n);
      if (KIND == kProductBlock ? rows : !rows) {
        constexpr int kNext = KIND == kProductBlock ? 9 : 1;
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] *= x[q * kNext];
        x += 32 * kNext;
      }
      uint4 h, mi, l;
      bf16_terms8(v, h, mi, l);
      const int slot = s < p.slots ? s : s - p.slots;
      ok = cut_waits(s, p.slots, [&](int b, uint32_t parity) { return warp_wait(&bar[b], parity, abort_flag, ws, 0x220000u | (uint32_t)b); });
      if (!ok) break;
      const uint32_t d = sm + to + (uint32_t)(slot * kStep);
      sts_u4(d, h);
      sts_u4(d + plane, mi);
      sts_u4(d + 2 * plane, l);
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar[slot]);
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = n[q];
    }
    // ---- the bias: the tiles beside one another deal out their output channels, a warp takes one; and the packed chunks without weights
    for (int ow = warp * p.n_tiles + nt; ow < OT; ow += kWarpsCut * p.n_tiles) {
      float sum = 0.f;
      const float *wo = a.l2.w + (size_t)(o0 + ow < c2 ? o0 + ow : 0) * c1 + cb;
#pragma unroll 1
      for (int c = lane; c < kc; c += 256) {
        float y[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) y[j] = c + 32 * j < kc ? wo[c + 32 * j] : 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (c + 32 * j < kc) sum = fmaf(y[j], qs[c + 32 * j], sum);
      }
      for (int dlt = 16; dlt > 0; dlt >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, dlt);
      if (lane == 0) bias_s[ow] = sum;
    }
    if (dv.mode == 2) zero_dead_chunks_by(dv, c2, (int)blockIdx.x * kCutThreads + tid, (int)gridDim.x * kCutThreads);
  } else {
    // ---------------------------------------------------------------- issue, by two warps, the barriers of some steps waited for side by side
    constexpr uint32_t id0 = (1u << 4) | (1u << 7) | (1u << 10) | (8u << 24);
    constexpr uint32_t i3 = id0 | (3 * NT / 8) << 17, i2 = id0 | (2 * NT / 8) << 17, i1 = id0 | (NT / 8) << 17;
    const uint64_t hi = (uint64_t)((128u >> 4) | (1u << 14)) << 32;
    const uint64_t a_hi = hi | ((uint64_t)(kPitchA >> 4) << 16), b_hi = hi | ((uint64_t)(3 * NT) << 16);
    const uint32_t sm16 = (sm >> 4) & 0x3FFFu;   // a CTA's own addresses name its rank in a cluster
    const int odd = warp - kIssue;
    auto ready = [&](int mine) {
      ok = issue_waits(mine, p.slots, [&](int b, uint32_t parity) { return mbar_wait(&bar[b], parity, abort_flag, ws, 0x230000u | (uint32_t)b); });
      __syncwarp();
      ok = __all_sync(0xffffffffu, ok) != 0;
      tc_fence_after();
      return ok;
    };
    if (!p.fine) {                               // a warp takes every second step, into sums of its own: h h; h m + m h; the others
      const uint32_t d = tmem + (uint32_t)(odd * 3 * NT);
#pragma unroll 1
      for (int s = odd; s < steps; s += 4) {
        const int mine = s + (lane & 1) * 2;
        if (!ready(mine < steps ? mine : s)) break;
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int st = s + 2 * q, slot = st < p.slots ? st : st - p.slots;
          if (st >= steps) break;
          const uint32_t at = sm16 + (uint32_t)(slot * (kStep >> 4));
          const uint64_t ad = a_hi | at, bd = b_hi | (at + (kStepA >> 4));
          if (elect_one()) {
            umma_bf16(d, ad, bd, i3, st > 1);
            umma_bf16(d + NT, ad + (2 * kPitchA >> 4), bd, i2, 1u);
            umma_bf16(d + 2 * NT, ad + (4 * kPitchA >> 4), bd, i1, 1u);
            umma_commit(&bar[kMaxSlots + slot]);
            if (st + 2 >= steps) umma_commit(&bar[2 * kMaxSlots]);
          }
        }
        __syncwarp();
      }
    } else {                                     // one warp issues h h, every kSums-th step into the same sums, the other the rest
#pragma unroll 1
      for (int s = 0; s < steps; s += 4) {
        const int mine = s + (lane & 3);
        if (!ready(mine < steps ? mine : s)) break;
#pragma unroll 1
        for (int st = s; st < s + 4 && st < steps; ++st) {
          const int slot = st < p.slots ? st : st - p.slots;
          const uint32_t at = sm16 + (uint32_t)(slot * (kStep >> 4));
          const uint64_t ad = a_hi | at, bd = b_hi | (at + (kStepA >> 4));
          if (elect_one()) {
            if (odd == 0) {
              umma_bf16(tmem + (uint32_t)(st % kSums * NT), ad, bd, i1, st >= kSums);
            } else {
              umma_bf16(tmem + kSums * NT, ad, bd + NT, i2, st > 0);
              umma_bf16(tmem + kSums * NT, ad + (2 * kPitchA >> 4), bd, i2, 1u);
              umma_bf16(tmem + (kSums + 1) * NT, ad + (4 * kPitchA >> 4), bd, i1, 1u);
            }
            umma_commit(&bar[kMaxSlots + slot]);
            if (st + 1 == steps) umma_commit(&bar[2 * kMaxSlots]);
          }
        }
        __syncwarp();
      }
    }
  }
  // ---------------------------------------------------------------- sums: the warps that can read the same 32 rows take 8 columns in turn
  if (warp < kWarpsCut) {
    ok = warp_wait(&bar[2 * kMaxSlots], 0u, abort_flag, ws, 0x240000u) && ok;
    tc_fence_after();
    const int quarter = warp & 3, m = quarter * 32 + lane, ow = m / T;
    const uint32_t drow = tmem + ((uint32_t)(quarter * 32) << 16);
    float *to = z + ow * UNIT + (m - ow * T);
#pragma unroll 1
    for (int col = (warp >> 2) * 8; col < NT && ok; col += (kWarpsCut - quarter + 3) / 4 * 8) {
      float sum[8] = {};
      if (p.fine) {
#pragma unroll
        for (int h = 0; h < kSums + 2; h += 2) {
          uint32_t x[2][8];
          tmem_ld8(drow + (uint32_t)(h * NT + col), x[0]);
          tmem_ld8(drow + (uint32_t)((h + 1) * NT + col), x[1]);
          tmem_ld_wait();
#pragma unroll
          for (int g = 0; g < 2; ++g)            // a sum of no step holds anything
            if (h + g < kSums && h + g >= steps)
#pragma unroll
              for (int j = 0; j < 8; ++j) x[g][j] = 0u;
#pragma unroll
          for (int j = 0; j < 8; ++j) sum[j] += __uint_as_float(x[0][j]) + __uint_as_float(x[1][j]);
        }
      } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t x[3][8];
#pragma unroll
          for (int g = 0; g < 3; ++g) tmem_ld8(drow + (uint32_t)((3 * h + g) * NT + col), x[g]);
          tmem_ld_wait();
          if (h > 0 && steps == 1) break;        // nor has the second warp any here
#pragma unroll
          for (int j = 0; j < 8; ++j) sum[j] += __uint_as_float(x[0][j]) + (__uint_as_float(x[1][j]) + __uint_as_float(x[2][j]));
        }
      }
      if (m < S::ROWS) {
        float *unit = to + col / 8 * (OT * UNIT);
        if (T == 1) {
          *reinterpret_cast<float4 *>(unit) = make_float4(sum[0], sum[1], sum[2], sum[3]);
          *reinterpret_cast<float4 *>(unit + 4) = make_float4(sum[4], sum[5], sum[6], sum[7]);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) unit[j * T] = sum[j];
        }
      }
    }
    tc_fence_before();
  }
  if (!ok && !ws) atomicExch(&g_product_status, (unsigned int)DC_ERR_TIMEOUT);
  // ---------------------------------------------------------------- each CTA takes a share of the tile: units of 8 input channels of an output channel
  constexpr int kPieces = 2 * T, kAll = OT * (NT / 8);
  const int per = (kAll + p.split - 1) / p.split, u0 = rank * per, left = kAll - u0, cnt = left < 0 ? 0 : (left < per ? left : per);
  const float *parts = reinterpret_cast<const float *>(smem + p.off_parts);      // the others' sums of it, by rank
  if (p.split > 1) {
    fence_proxy_async();
    cluster_sync();                              // everybody's terms are multiplied, and its sums and its part of the bias written
    if (tid == 0)                                // to each of the others its share, into its shared memory
#pragma unroll 1
      for (int q = 0; q < p.split; ++q) {
        const int v0 = q * per, n = kAll - v0 < per ? kAll - v0 : per;
        if (q == rank || n <= 0) continue;
        bulk_send(map_cluster(sm + (uint32_t)(p.off_parts + rank * per * UNIT * 4), (uint32_t)q), sm + (uint32_t)(v0 * UNIT * 4),
                  (uint32_t)(n * UNIT * 4), map_cluster(smem_u32(&bar[2 * kMaxSlots + 1]), (uint32_t)q));
      }
    __syncwarp();
    if (cnt > 0 && !warp_wait(&bar[2 * kMaxSlots + 1], 0u, abort_flag, ws, 0x250000u) && !ws)
      atomicExch(&g_product_status, (unsigned int)DC_ERR_TIMEOUT);
  } else {
    __syncthreads();
  }
  if (warp == kIssue) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  {
    const bool whole = dv.mode >= 0 && dv.ident, ident = KIND != kProductBlock && (a.ident1 || a.ident2);
    // the bias, by the threads behind the others
    if (rank == 0)
      for (int ow = (kThreads - 1 - tid) * p.n_tiles + nt; ow < OT; ow += kThreads * p.n_tiles) {
        const int o = o0 + ow;
        if (o >= c2) continue;
        float sum = bias_s[ow], r[kMaxSplit];
#pragma unroll
        for (int q = 1; q < kMaxSplit; ++q)
          if (q < p.split) r[q] = lds_cluster_f(map_cluster(smem_u32(bias_s + ow), (uint32_t)q));
#pragma unroll
        for (int q = 1; q < kMaxSplit; ++q)
          if (q < p.split) sum += r[q];
        float b = fmaf(g_last[ow], sum, b_last[ow]);
        if (KIND != kProductBlock && a.ident2) b += raw_bias(a.l1, o, raw_scale(a.l1, o));
        a.b_out[o] = b;
      }
#pragma unroll 1
    for (int e = tid; e < cnt * kPieces; e += kThreads) {
      const int ul = e / kPieces, x = (e - ul * kPieces) * 4, u = u0 + ul, ig = u / OT, ow = u - ig * OT;
      const int o = o0 + ow, i = i0 + ig * 8;
      if (o >= c2 || i + x / T >= c0) continue;
      float4 *zp = reinterpret_cast<float4 *>(z + u * UNIT + x);
      const float4 own = *zp;
      const float *part = parts + ul * UNIT + x;
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);                  // in rank order
#pragma unroll 4
      for (int q = 0; q < p.split; ++q) {
        const float4 r = q == rank ? own : *reinterpret_cast<const float4 *>(part + q * per * UNIT);
        s.x += r.x; s.y += r.y; s.z += r.z; s.w += r.w;
      }
      const float g = g_last[ow], sum = (s.x + s.y) + (s.z + s.w);
      s.x *= g; s.y *= g; s.z *= g; s.w *= g;
      if (ident || (whole && o >= i && o < i + 8) || sum != sum) {
        float f[4] = {s.x, s.y, s.z, s.w};
#pragma unroll 1
        for (int j = 0; j < 4; ++j) {
          const int ii = i + (x + j) / T, t = (x + j) % T;
          float y = j == 0 ? s.x : j == 1 ? s.y : j == 2 ? s.z : s.w;
          if (!(y - y == 0.f)) y = g * sum_by_fma<KIND>(a, o, ii, t);
          y = add_ident<KIND>(a, whole, g, y, o, ii, t);
          if (j == 0) f[0] = y;
          else if (j == 1) f[1] = y;
          else if (j == 2) f[2] = y;
          else f[3] = y;
        }
        s = make_float4(f[0], f[1], f[2], f[3]);
      }
      *reinterpret_cast<float4 *>(a.w_out + ((size_t)o * c0 + i) * T + x) = s;
      *zp = s;                                   // which no other thread reads; nor has it been sent
    }
    if (dv.mode > 0) {
      __syncthreads();
#pragma unroll 1
      for (int e = tid; e < cnt * T; e += kThreads) {
        const int t = e / cnt, u = u0 + e - t * cnt, ig = u / OT, ow = u - ig * OT, o = o0 + ow, i = i0 + ig * 8;
        if (o < c2 && i < c0) deliver_chunk<T>(dv, z + u * UNIT + t, o, i, t, c0, c2);
      }
    }
  }
  if (p.split > 1) cluster_meet_relaxed();       // nobody leaves while its sums, or its bias, may still be read
}

// ------------------------------------------------------------------------------------------ host
// Clusters of `size` CTAs (an SM's shared memory each) the current device runs at once, asked for once per device.
int max_clusters(int size) {
  static int cached[kDcMaxDevices][kMaxSplit + 1];
  const int dev = dc_current_device();
  if (dev < 0) { (void)cudaGetLastError(); return 1; }
  if (cached[dev][size] == 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)size * 64);
    cfg.blockDim = dim3(threads_of(80));
    cfg.dynamicSmemBytes = kSmemMax;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)size;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    static unsigned char attr_done[kDcMaxDevices];
    if (dc_set_max_smem_once(k_merge_product_tc<kProductBlock, 80>, kSmemMax, attr_done) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&n, k_merge_product_tc<kProductBlock, 80>, &cfg) != cudaSuccess || n <= 0) {
      (void)cudaGetLastError();
      n = 1;
    }
    cached[dev][size] = n;
  }
  return cached[dev][size];
}

// In microseconds, `rounds` tiles (clusters) one after another on an SM, `busy` of the SMs at work.  Fitted to 1538 plans of 110 blocks and
// pairs (blocks 2.7 % off in the root mean square, pairs 7.4 %); the plan with the smallest is 0.3 % slower than the best on average.
template <int KIND>
double estimate_us(int nt, int split, int steps, int fine, int rounds, double busy) {
  const double work = (double)rounds * steps;
  if (KIND == kProductPair) return 5.9 + 4.47 * (rounds - 1) + 0.041 * rounds * nt + work * (0.296 + 0.0026 * nt);
  return 6.25 + (split > 1 ? 4.8 * (rounds - 1) : 0.0) + rounds * (0.034 * nt + 0.49 * busy) + work * (0.173 + 0.0023 * nt + (fine ? 0.053 : 0.0));
}

// The columns of a tile and the parts of its reduction with the smallest estimate, in us; 0: outside the range.  `run`: channels that
// one sum of the FMA kernel goes through.  The tensor core cuts its sums instead of rounding them, so a sum of products of high terms
// takes a tenth as many steps at most, and from five steps on there are as many sums as tensor memory holds (0.3 to 0.8 us for 0.6 to
// 0.9 of the error).  Against 64 bits (2-norm), of 166 drawn blocks and 57 pairs the 102 and 29 that go there: weights of both
// signs 0.73 of the FMAs' error on average and 0.87 at most, pairs 0.42 and 0.60; weights of one sign, where what is cut off adds up, 1.19 and
// 1.79 (1.56e-7 at most; FMAs have up to 2.5e-7 for weights of both signs), pairs 0.66 and 0.90.  At most three steps a sum would be 1.44
// instead of 1.79, for 0.757 instead of 0.716 of the FMAs' time.
template <int KIND>
double make_plan(int c0, int c1, int c2, int run, Plan *best, int *best_nt) {
  using S = Shape<KIND>;
  if (c0 % 4 || c1 % 4 || c1 < 16) return 0.0;
  const int total = dc_div_up(c1, 16), n_sm = dc_sm_count();
  const int widths[3] = {48, 64, 80};
  double us = 0.0;
  for (int nt : widths)
    for (int split = 1; split <= kMaxSplit; ++split) {
      const int steps = dc_div_up(total, split), step_bytes = kStepA + nt * 96;
      if ((split - 1) * steps >= total || steps > 2 * (8 + nt / 16)) continue;                     // a thread to a channel
      const int fine = steps > 4;
      if (dc_div_up(steps, fine ? sums_of(nt) : 2) * 10 > run) continue;
      const int scales = steps * 16 * 4 * (KIND == kProductBlock ? 9 : 1), sums = S::ROWS * nt * 4;
      const int parts = split > 1 ? split * dc_div_up(S::OT * (nt / 8), split) * S::UNIT * 4 : 0;
      int slots = (kSmemMax - 256 - scales - steps * 64) / step_bytes;
      if (slots > kMaxSlots) slots = kMaxSlots;
      if (slots > steps) slots = steps;
      if (steps > 2 * slots) continue;
      const long long tiles = (long long)dc_div_up(c2, S::OT) * dc_div_up(c0, nt);
      if (tiles * split >= (1ll << 24)) continue;
      const int at_once = split == 1 ? n_sm : max_clusters(split), rounds = (int)((tiles + at_once - 1) / at_once);
      const double t = estimate_us<KIND>(nt, split, steps, fine, rounds, tiles * split < n_sm ? (double)(tiles * split) / n_sm : 1.0);
      if (us != 0.0 && t >= us) continue;
      us = t;
      *best_nt = nt;
      const int off_parts = (int)dc_round_up((size_t)sums, 128), end = off_parts + parts;
      const int ring = (int)dc_round_up((size_t)(slots * step_bytes > end ? slots * step_bytes : end), 128);
      *best = Plan{dc_div_up(c0, nt), split, steps, total, slots, ring, ring + scales, off_parts, fine};
    }
  return us;
}

template <int KIND, int NT>
dc_status launch(const Product &a, const BlockDelivery &dv, const Plan &p, DcWsHeader *ws, cudaStream_t st) {
  static unsigned char attr_done[kDcMaxDevices];
  DC_CUDA_OK(dc_set_max_smem_once(k_merge_product_tc<KIND, NT>, kSmemMax, attr_done));
  const int grid = dc_div_up(a.c2, Shape<KIND>::OT) * p.n_tiles * p.split;
  const cudaError_t e = dc_launch_pdl_cluster(k_merge_product_tc<KIND, NT>, dim3((unsigned)grid), dim3(threads_of(NT)), (size_t)kSmemMax, st, p.split, a, dv, p, ws);
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? DC_OK : DC_ERR_CUDA;
}

template <int KIND>
dc_status launch_kind(const Product &a, const BlockDelivery &dv, int run, DcWsHeader *ws, cudaStream_t st) {
  Plan p{};
  int nt = 0;
  if (make_plan<KIND>(a.c0, a.c1, a.c2, run, &p, &nt) == 0.0) return DC_ERR_UNSUPPORTED;
  if (nt == 48) return launch<KIND, 48>(a, dv, p, ws, st);
  if (nt == 64) return launch<KIND, 64>(a, dv, p, ws, st);
  return launch<KIND, 80>(a, dv, p, ws, st);
}

}  // namespace

dc_status dc_launch_merge_product_tc(int kind, const Product &a, const BlockDelivery &dv, int run, DcWsHeader *ws, cudaStream_t st) {
  return kind == kProductBlock ? launch_kind<kProductBlock>(a, dv, run, ws, st) : launch_kind<kProductPair>(a, dv, run, ws, st);
}

double dc_merge_product_tc_us(int kind, int c0, int c1, int c2, int run) {
  Plan p{};
  int nt = 0;
  return kind == kProductBlock ? make_plan<kProductBlock>(c0, c1, c2, run, &p, &nt) : make_plan<kProductPair>(c0, c1, c2, run, &p, &nt);
}

cudaError_t dc_merge_product_tc_flag(unsigned int **flag) { return cudaGetSymbolAddress((void **)flag, g_product_status); }

extern "C" int dc_selftest_product_waits(int step, int slots, unsigned int waits[8]) {
  if (slots < 1 || slots > kMaxSlots || step < 0 || step >= 2 * slots) return 0;
  int n = 0;
  auto note = [&](int at, uint32_t parity) {
    waits[2 + 2 * n] = (unsigned int)at;
    waits[3 + 2 * n] = parity;
    ++n;
    return true;
  };
  cut_waits(step, slots, note);
  waits[0] = (unsigned int)n;
  issue_waits(step, slots, note);
  waits[1] = (unsigned int)kMaxSlots;
  return n;
}
