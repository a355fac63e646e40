// A dense 3x3 layer after a dense 3x3 one (stride 1) on the tensor core, by operands cut into bf16 terms (bf16_terms2).
//
// W'[o][i][t] = sum_c sum_{t1 + t2 = t} W2[o][c][t2] W1~[c][i][t1]: the product Z of the matrix W2 with rows (o, t2) and the matrix W1
// with columns (i, t1), reduction over c, has none of the structural zeros that a gathered product has, and the 25 taps of a pair
// are sums of its 81 elements Z[o, t2][i, t1].  A tile is 14 output channels (126 of 128 rows) x 8 input channels (72 columns).
// A value is three bf16 terms, six products of them are above 2^-24, and they are four instructions a step of 16 channels: A_h x h into
// sums of hh, A_h x [m l], A_m x [h m] and A_l x h into sums of hm + mh and of the rest.  The tensor core cuts its sums instead of
// rounding them, so those of hh are read out every four steps and added in fp32; the others, 2^8 times smaller, every sixteen.
// Error against 64 bits (2-norm), 256 channels between: weights of both signs 1.2e-7, by FMAs 2.3e-7; of one sign, where what is cut off adds up,
// 1.2e-7 and 0.96e-7.  (512 channels 1.3e-7 and 3.2e-7, 1.2e-7 and 1.2e-7.)
//
// Warps: one loads the second layer by TMA, eight cut operands into terms, in four pairs that take the steps in turn (a pair has four
// steps' time for one: a warp alone on its scheduler needs it), one issues, four add up, take the 25 taps together through shared
// memory and deliver the result while the next tile is multiplied: the four sums of hh hold sixteen steps.  The terms of a tile's columns stay in
// shared memory for all tiles below one another where they fit (256 channels between); CTAs own runs of such tiles.  The warps that cut
// compute the bias behind their last tile.  What bounds it is no unit (the counters are in profiles/) but the way of a step through its
// pair of warps: operands there, read, cut, slot free, written, multiplied, 2.7 thousand cycles with four on their way at once, and a
// slot of operands and terms more has no room beside the columns' terms.
//
// An infinity or a NaN among the weights makes NaN of results: such a result is computed again by FMAs.
//
// 256 -> 256 -> 256 75.6 us by FMAs (k_compose33), here 47; 512 551 -> 289; 104 -> 208 -> 136 21.0 -> 16.1; 64 6.7 -> 9.0 (left to FMAs).
// The taps, the scale, the result and its packed copy take 9 thousand cycles a tile in the adding warps (they run once a tile, from a cold
// instruction cache).  On the way: cut by nine warps together 76, by pairs 54, operands asked for again before they are cut 47 (not sound, see
// there; without, no slower any more), one issuing warp that waits for two steps side by side 45.  80 columns a term instead of 72 0.5 to
// 0.9 % more; eight adding warps 44.6, but 512 channels 296; steps cut by four warps 51, by two teams with two slots each 53.  All sums read
// out every eight steps, two sets of them: 45.0, 512 channels 279, but errors of 1.6e-7 and, for weights of one sign, 2.0e-7; those of
// hh every two steps: 53.2 and 298, errors of 1.1e-7 and 0.9e-7 (the adding warps then fall behind: four such sums hold half a tile).
#include "merge_parts.cuh"
#include "tc_ptx.cuh"

namespace {
using namespace tc;

__device__ unsigned int g_merge_status;          // DC_ERR_TIMEOUT once a wait of this kernel ran out in a launch without a workspace header

constexpr int kO = 14, kI = 8, kRows = kO * 9, kCols = kI * 9;
constexpr int kRowsB = 3 * kCols;                // of the columns' terms of 8 channels
constexpr int kWarpsAcc = 4, kPairs = 4, kWarpsCut = 2 * kPairs, kLoad = kWarpsAcc + kWarpsCut, kIssue = kLoad + 1, kThreads = (kIssue + 1) * 32;
constexpr int kChunk = 4, kLong = 16;            // steps of 16 channels between two read-outs of the sums of hh, and of the others
constexpr int kSums = 4, kPitchSum = 80;         // sums of hh and their columns (8 of them only make up an instruction); then those of the others
constexpr int kColM = kSums * kPitchSum, kColR = kColM + kCols;
constexpr int kPitchA = 128 * 16;                // bytes between the halves of a step's 16 channels
constexpr int kStepA = 6 * kPitchA, kStepB = 2 * kRowsB * 16, kRawA = kO * 144 * 4;
constexpr int kPitchZ = kCols / 2 + 1;           // floats of a row of Z, four input channels at a time
constexpr int kZ = (kRows * kPitchZ * 4 + 127) / 128 * 128;
constexpr int kMaxB = 16;                        // steps whose columns' terms are there at once
constexpr int kSmemMax = 226 * 1024;
static_assert(kRawA % 128 == 0 && kO * kI * 25 * 4 <= kZ, "slots; the taps' sums lie where Z was");

struct Params33 {
  int m_tiles, n_tiles, items, steps;
  int resident, ring_b;                          // columns' terms stay for a column of tiles; slots of them
  int off_raw, off_b, off_z, off_scale, smem_bytes;
};

// A pair of warps owns a slot of operands (R), of terms (A) and, of the columns' terms (B), every fourth; D are the sums of hh, M those of
// the other products.  Every role waits for every phase of its barriers in order, so a phase's bit tells it from the one before.
enum { kRFull = 0, kREmpty = kPairs, kAFull = 2 * kPairs, kAEmpty = 3 * kPairs, kBFull = 4 * kPairs, kBEmpty = kBFull + kMaxB,
       kDFull = kBEmpty + kMaxB, kMFull = kDFull + kSums, kDEmpty = kMFull + 1, kMEmpty = kDEmpty + kSums, kBars = kMEmpty + 1 };

// a load that stays where it is written
__device__ __forceinline__ float ask(const float *p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}

// one result by FMAs, before the second layer's scale: where the terms gave NaN
__device__ __noinline__ float sum_by_fma(const Compose33 &a, int o, int i, int t) {
  const RawLayer &l1 = a.first.l, &l2 = a.second.l;
  const int y = t / 5, x = t - 5 * y;
  float s = 0.f;
#pragma unroll 1
  for (int c = 0; c < a.c1; ++c) {
    const float g = raw_scale(l1, c);
#pragma unroll 1
    for (int t2 = 0; t2 < 9; ++t2) {
      const int u = y - t2 / 3, v = x - t2 % 3;
      if (u < 0 || u > 2 || v < 0 || v > 2) continue;
      s = fmaf(l2.w[((size_t)o * a.c1 + c) * 9 + t2], l1.w[((size_t)c * a.c0 + i) * 9 + u * 3 + v] * g, s);
    }
  }
  return s;
}

__global__ void __launch_bounds__(kThreads, 1)
k_compose33_tc(const __grid_constant__ CUtensorMap map_w2, const __grid_constant__ Compose33 a,
               const __grid_constant__ BlockDelivery dv, const __grid_constant__ Params33 p, DcWsHeader *ws) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ uint64_t bar[kBars];
  __shared__ size_t row_s[kO];                   // where the tile's output channels, and its taps, are in the packed copy
  __shared__ int plane_s[25];
  __shared__ uint32_t tmem_s, abort_s;
  volatile uint32_t *abort_flag = &abort_s;
  const int tid = (int)threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t sm = smem_u32(smem);
  const int c0 = a.c0, c1 = a.c1, c2 = a.c2;
  const int begin = (int)((long long)p.items * blockIdx.x / gridDim.x), end = (int)((long long)p.items * (blockIdx.x + 1) / gridDim.x);
  if (tid < kBars) {
    uint32_t count = 1;
    if ((tid >= kREmpty && tid < kAEmpty) || (tid >= kBFull && tid < kBEmpty)) count = 2;  // a pair of warps
    else if (tid >= kDEmpty) count = kWarpsAcc;
    mbar_init(&bar[tid], count);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  } else if (tid == 96) {
    abort_s = 0;
    prefetch_tensormap(&map_w2);
  }
  __syncthreads();
  dc_pdl_enter();                                // global memory and tensor memory only behind this
  if (warp < kWarpsAcc || warp == kIssue) {
    if (warp == kIssue) {
      tmem_alloc(&tmem_s, 512);
      tmem_relinquish();
    }
    tc_fence_before();
    bar_sync(1, (kWarpsAcc + 1) * 32);
    tc_fence_after();
  }
  const uint32_t tmem = tmem_s;
  auto wait = [&](int b, uint32_t parity) { return warp_wait(&bar[b], parity, abort_flag, ws, 0x200000u | (uint32_t)b); };
  // the first and the last of a CTA's tiles that use the same columns' terms
  auto first_of = [&](int item) { return !p.resident || item == begin || item % p.m_tiles == 0; };
  auto last_of = [&](int item) { return !p.resident || item + 1 == end || (item + 1) % p.m_tiles == 0; };

  if (warp < kWarpsAcc) {
    // ---------------------------------------------------------------- sums, taps, delivery
    const uint32_t drow = tmem + ((uint32_t)(warp * 32) << 16);
    float *z = reinterpret_cast<float *>(smem + p.off_z);
    const bool last = dv.mode >= 0, special = a.first.ident || a.second.ident || (last && dv.ident);
    // where a bf16 chunk goes: rows of a tap's chunk plane, except in orders that hold taps or pixels in the rows
    const bool rows = dv.mode == 2 && !dv.ko.fold && !dv.ko.pair;
    const int po = (tid & 63) >> 2, pi = tid & 3, side = tid >> 6;               // this thread's pair of channels, when taps are summed
    uint32_t fl = 0, ml = 0;
    bool ok = true;
#pragma unroll 1
    for (int item = begin; item < end && ok; ++item) {
      const int nt = item / p.m_tiles, o0 = (item - nt * p.m_tiles) * kO, i0 = nt * kI, m = tid;
      const int o = o0 + po, iw = side * 4 + pi, i = i0 + iw;
      const bool live = po < kO && o < c2 && i < c0;
      const bool scaled = live && a.second.l.gamma != nullptr;
      float gamma = 1.f, var = 0.f;              // asked for here, first touched when the sums are there
      if (scaled) { gamma = ask(a.second.l.gamma + o); var = ask(a.second.l.var + o); }
      float acc[kCols];
#pragma unroll
      for (int j = 0; j < kCols; ++j) acc[j] = 0.f;
#pragma unroll 1
      for (int s = 0; s < p.steps; s += kChunk, ++fl) {
        const uint32_t b = fl % kSums;
        if (!(ok = wait(kDFull + (int)b, (fl / kSums) & 1u))) break;
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < kCols; c += 24) {
          uint32_t v0[8], v1[8], v2[8];
          const uint32_t at = drow + b * kPitchSum + c;
          tmem_ld8(at, v0);
          tmem_ld8(at + 8, v1);
          tmem_ld8(at + 16, v2);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            acc[c + j] += __uint_as_float(v0[j]);
            acc[c + 8 + j] += __uint_as_float(v1[j]);
            acc[c + 16 + j] += __uint_as_float(v2[j]);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar[kDEmpty + b]);
        if (s % kLong != kLong - kChunk && s + kChunk < p.steps) continue;
        if (!(ok = wait(kMFull, ml & 1u))) break;
        ++ml;
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < kCols; c += 8) {
          uint32_t v0[8], v1[8];
          tmem_ld8(drow + kColM + c, v0);
          tmem_ld8(drow + kColR + c, v1);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[c + j] += __uint_as_float(v0[j]) + __uint_as_float(v1[j]);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar[kMEmpty]);
      }
      if (!(ok = bar_all(3, 128, ok))) break;    // the four warps agree before they meet below
      if (rows) {                                // read behind the barriers below
        if (first_of(item) && tid < 25) plane_s[tid] = dc_korder_encode(dv.ko, nt, tid / 5, tid % 5);
        if (tid >= 32 && tid < 32 + kO) row_s[tid - 32] = dc_packed_chunk(dv.ko, 0, o0 + tid - 32);
      }
      // four input channels at a time: row (o, t2) of Z; then two warps take a pair (o, i) to a thread, 81 elements of Z to its 25 taps
      float t5[25];
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {              // one copy of this code: what runs once a tile comes from far away each time
        if (m < kRows)
#pragma unroll
          for (int j = 0; j < kCols / 2; ++j) z[m * kPitchZ + j] = h ? acc[kCols / 2 + j] : acc[j];
        bar_sync(3, 128);
        if (side == h && po < kO) {
#pragma unroll
          for (int t = 0; t < 25; ++t) t5[t] = 0.f;
          const float *zp = z + po * 9 * kPitchZ + pi * 9;
#pragma unroll
          for (int t2 = 0; t2 < 9; ++t2)
#pragma unroll
            for (int t1 = 0; t1 < 9; ++t1) t5[(t2 / 3 + t1 / 3) * 5 + t2 % 3 + t1 % 3] += zp[t2 * kPitchZ + t1];
        }
        bar_sync(3, 128);
      }
      if (live) {
        float *to = z + (po * kI + iw) * 25;
        const float g2 = scaled ? gamma / sqrtf(var + a.second.l.eps) : 1.f;
#pragma unroll
        for (int t = 0; t < 25; ++t) to[t] = g2 * t5[t];
        if (special)
#pragma unroll 1
          for (int t = 0; t < 25; ++t) to[t] = compose33_ident(a, last && dv.ident, g2, to[t], o, i, t);
      }
      bar_sync(3, 128);
      // [o][i][tap]: rows of 200 neighbouring elements of the result, three reads at a time
      constexpr int kPieces = kO * kI * 25 / 4;
#pragma unroll 1
      for (int e0 = tid; e0 < kPieces; e0 += 384) {
        float4 s4[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) s4[q] = reinterpret_cast<const float4 *>(z)[e0 + q * 128 < kPieces ? e0 + q * 128 : e0];
        uint32_t bad = 0;                        // pieces that hold a NaN, or infinities of both signs
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const int e = e0 + q * 128, oi = e / (kI * 25 / 4), x = (e - oi * (kI * 25 / 4)) * 4, oo = o0 + oi;
          if (e >= kPieces || oo >= c2 || i0 + x / 25 >= c0) continue;
          const float sum = (s4[q].x + s4[q].y) + (s4[q].z + s4[q].w);
          if (sum != sum) bad |= 1u << q;
          *reinterpret_cast<float4 *>(a.w_out + ((size_t)oo * c0 + i0) * 25 + x) = s4[q];
        }
        if (bad)
#pragma unroll 1
          for (int f = 0; f < 12; ++f)
            if ((bad >> (f / 4)) & 1u) {
              const int e = (e0 + f / 4 * 128) * 4 + f % 4, oi = e / (kI * 25), r = e - oi * (kI * 25), ii = r / 25, t = r - ii * 25;
              const float g = raw_scale(a.second.l, o0 + oi);
              float v = g * sum_by_fma(a, o0 + oi, i0 + ii, t);
              if (special) v = compose33_ident(a, last && dv.ident, g, v, o0 + oi, i0 + ii, t);
              z[e] = v;
              a.w_out[((size_t)(o0 + oi) * c0 + i0) * 25 + r] = v;
            }
      }
      bar_sync(3, 128);
      if (last && dv.mode > 0) {
        if (rows) {
          const int per = dv.ko.rows && dv.ko.nnt > 1 ? dv.ko.n_tile : dv.ko.n_pad;
          uint4 *out = reinterpret_cast<uint4 *>(dv.packed);
#pragma unroll 1
          for (int e = tid; e < kO * 25; e += 128) {
            const int t = e / kO, ow = e - t * kO;
            const float *f = z + ow * (kI * 25) + t;
            const uint4 v = make_uint4(pack_bf16x2(f[0], f[25]), pack_bf16x2(f[50], f[75]), pack_bf16x2(f[100], f[125]), pack_bf16x2(f[150], f[175]));
            if (o0 + ow < c2) out[row_s[ow] + (size_t)plane_s[t] * per] = v;
          }
        } else {
          deliver_tile<kO, kI, 5>(dv, z, o0, i0, c0, c2, tid, 128);
        }
      }
      bar_sync(3, 128);
    }
    if (!ok && !ws && tid == 0) atomicExch(&g_merge_status, (unsigned int)DC_ERR_TIMEOUT);
  } else if (warp < kLoad) {
    // ---------------------------------------------------------------- operands into terms: a pair of warps takes every fourth step
    const int cw = warp - kWarpsAcc, ct = tid - kWarpsAcc * 32, pair = cw >> 1, w1 = cw & 1;
    float *g1s = reinterpret_cast<float *>(smem + p.off_scale);
    for (int c = ct; c < p.steps * 16; c += kWarpsCut * 32) g1s[c] = c < c1 ? raw_scale(a.first.l, c) : 0.f;
    bar_sync(2, kWarpsCut * 32);
    const uint32_t raw = sm + (uint32_t)(p.off_raw + pair * kRawA), to_a = sm + (uint32_t)(pair * kStepA);
    // a warp's four turns of a step: 8 channels (of its half of the 16) of 32 rows (o, t2)
    uint32_t f[4];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int row = t * 32 + lane, r = row < kRows ? row : kRows - 1, o = r / 9;
      f[t] = raw + (uint32_t)((o * 144 + w1 * 72 + r - o * 9) * 4);
    }
    const uint32_t d0 = to_a + (uint32_t)(w1 * kPitchA + lane * 16);
    uint32_t pr = 0, pa = 1, pb = 1;             // phases of the pair's operands, terms and column terms
    int bs = pair;                               // the slot of the column terms of its next step
    bool ok = true;
    int at = pair;                               // its next step, counted over the items' steps
#pragma unroll 1
    for (int item = begin; item < end && ok; ++item, at -= p.steps) {
      const bool first = first_of(item);
      const int n0 = item / p.m_tiles * kCols;
#pragma unroll 1
      for (; at < p.steps; at += kPairs) {
        if (first) {
          // 8 channels of a column to a thread: five turns, three of the first warp's
          uint32_t db[3];
          float vb[3][8];
#pragma unroll
          for (int t = 0; t < 3; ++t) {
            const int e = (t * 2 + w1) * 32 + lane, half = e >= kCols ? 1 : 0, n = e - half * kCols, c = at * 16 + half * 8;
            const bool in = e < 2 * kCols && n0 + n < c0 * 9;
            db[t] = (uint32_t)(half * (kRowsB * 16) + n * 16);
#pragma unroll
            for (int j = 0; j < 8; ++j) vb[t][j] = in && c + j < c1 ? a.first.l.w[(size_t)(c + j) * c0 * 9 + n0 + n] : 0.f;
          }
          const int slot = p.resident ? at : bs;
          if (!(ok = wait(kBEmpty + slot, pb))) break;
#pragma unroll
          for (int t = 0; t < 3; ++t) {
            const int e = (t * 2 + w1) * 32 + lane, half = e >= kCols ? 1 : 0, c = at * 16 + half * 8;
            if (e >= 2 * kCols) continue;
#pragma unroll
            for (int j = 0; j < 8; ++j) vb[t][j] *= g1s[c + j];
            uint4 h, mi, l;
            bf16_terms8(vb[t], h, mi, l);
            const uint32_t d = sm + (uint32_t)(p.off_b + slot * kStepB) + db[t];
            sts_u4(d, h);
            sts_u4(d + kCols * 16u, mi);
            sts_u4(d + kCols * 32u, l);
          }
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bar[kBFull + slot]);
          bs += kPairs;
          if (!p.resident && bs >= p.ring_b) { bs -= p.ring_b; pb ^= 1u; }
        }
        if (!(ok = wait(kRFull + pair, pr))) break;
        float v[4][8];
#pragma unroll
        for (int t = 0; t < 4; ++t)
#pragma unroll
          for (int j = 0; j < 8; ++j) v[t][j] = lds_f(f[t] + (uint32_t)(j * 36));
        // half is cut before the slot is free (all of it would spill): what is behind the wait stands between two steps' instructions
        uint4 h[2], mi[2], l[2];
        bf16_terms8(v[0], h[0], mi[0], l[0]);
        bf16_terms8(v[1], h[1], mi[1], l[1]);
        if (!(ok = wait(kAEmpty + pair, pa))) break;
        pr ^= 1u;
        pa ^= 1u;
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          if (t == 2) bf16_terms8(v[2], h[0], mi[0], l[0]);
          if (t == 3) bf16_terms8(v[3], h[1], mi[1], l[1]);
          const uint32_t d = d0 + (uint32_t)(t * 512);
          sts_u4(d, h[t & 1]);
          sts_u4(d + 2 * kPitchA, mi[t & 1]);
          sts_u4(d + 4 * kPitchA, l[t & 1]);
        }
        fence_proxy_async();
        __syncwarp();
        // The operands' slot is given back here, behind the stores that need what was read from it.  Given back before the cut, with
        // the values in registers, it was read too late: the compiler reads shared memory again where a value is used, or moves a
        // read behind the arrival, __syncwarp() or not (single channels of the next step in some rows, of a CTA's later tiles).
        if (lane < 2) mbar_arrive(&bar[lane ? kREmpty + pair : kAFull + pair]);
      }
      if (p.resident && last_of(item)) pb ^= 1u;
    }
    // ---- beside the last tiles: the bias, a warp to an output channel, and the packed chunks without weights
    for (int o = (int)blockIdx.x * kWarpsCut + cw; o < c2; o += (int)gridDim.x * kWarpsCut) compose33_bias(a, o, lane);
    if (dv.mode == 2) zero_dead_chunks_by(dv, c2, (int)blockIdx.x * kWarpsCut * 32 + ct, (int)gridDim.x * kWarpsCut * 32);
  } else if (warp == kLoad) {
    // ---------------------------------------------------------------- loads of the second layer: [o][channel][tap], 16 channels of 14 o
    int rs = 0;
    uint32_t pr = 1;
    bool ok = true;
#pragma unroll 1
    for (int item = begin; item < end && ok; ++item) {
      const int o0 = item % p.m_tiles * kO;
#pragma unroll 1
      for (int s = 0; s < p.steps; ++s) {
        if (!(ok = wait(kREmpty + rs, pr))) break;
        if (lane == 0) {
          mbar_arrive_expect_tx(&bar[kRFull + rs], kRawA);
          tma_load_2d(sm + (uint32_t)(p.off_raw + rs * kRawA), &map_w2, &bar[kRFull + rs], s * 144, o0);
        }
        __syncwarp();
        if (++rs == kPairs) { rs = 0; pr ^= 1u; }
      }
    }
    if (!ok) {                                   // copies may still be in flight: give them time to land
      const unsigned long long t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    }
  } else {
    // ---------------------------------------------------------------- issue: two steps at a time, their barriers waited for side by side
    const uint32_t id0 = (1u << 4) | (1u << 7) | (1u << 10) | (8u << 24);
    constexpr uint32_t i2 = (2 * kCols / 8) << 17, i1 = (kPitchSum / 8) << 17;
    const uint64_t hi = (uint64_t)((128u >> 4) | (1u << 14)) << 32;
    const uint64_t a_hi = hi | ((uint64_t)(kPitchA >> 4) << 16), b_hi = hi | ((uint64_t)kRowsB << 16);
    const uint32_t sm16 = sm >> 4, b16 = (sm + (uint32_t)p.off_b) >> 4;
    int as = 0, bs = 0;
    uint32_t pa = 0, pb = 0, fl = 0, ml = 0;
    bool ok = true;
#pragma unroll 1
    for (int item = begin; item < end && ok; ++item) {
      const bool first = first_of(item), last = last_of(item);
#pragma unroll 1
      for (int s = 0; s < p.steps; s += 2) {
        const bool opens_h = s % kChunk == 0, closes_h = s % kChunk == kChunk - 2;
        const bool opens = s % kLong == 0, closes = s % kLong == kLong - 2 || s + 2 == p.steps;
        const uint32_t buf = fl % kSums, d = tmem + buf * kPitchSum;
        int b = kAFull + as + (lane & 1);
        uint32_t parity = pa;
        if (first && (lane & 2)) { b = kBFull + bs + (lane & 1); parity = pb; }
        if (opens_h && lane == 4) { b = kDEmpty + (int)buf; parity = ((fl / kSums) & 1u) ^ 1u; }
        if (opens && lane == 5) { b = kMEmpty; parity = (ml & 1u) ^ 1u; }
        ok = mbar_wait(&bar[b], parity, abort_flag, ws, 0x210000u | (uint32_t)b);
        __syncwarp();
        if (!(ok = __all_sync(0xffffffffu, ok) != 0)) break;
        tc_fence_after();
        const uint32_t at = sm16 + (uint32_t)(as * (kStepA >> 4)), bt = b16 + (uint32_t)(bs * (kStepB >> 4));
        if (elect_one()) {
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const uint64_t bd = b_hi | (uint64_t)((bt + q * (kStepB >> 4)) & 0x3FFFu);
            const uint32_t aq = at + q * (kStepA >> 4);
            const uint64_t bm = b_hi | (uint64_t)((bt + q * (kStepB >> 4) + kCols) & 0x3FFFu);       // from the middle terms on
            umma_bf16(d, a_hi | (uint64_t)(aq & 0x3FFFu), bd, id0 | i1, opens_h && q == 0 ? 0u : 1u);
            umma_bf16(tmem + kColM, a_hi | (uint64_t)(aq & 0x3FFFu), bm, id0 | i2, opens && q == 0 ? 0u : 1u);
            umma_bf16(tmem + kColM, a_hi | (uint64_t)((aq + (2 * kPitchA >> 4)) & 0x3FFFu), bd, id0 | i2, 1u);
            umma_bf16(tmem + kColR, a_hi | (uint64_t)((aq + (4 * kPitchA >> 4)) & 0x3FFFu), bd, id0 | i1, 1u);
            umma_commit(&bar[kAEmpty + as + q]);
            if (last) umma_commit(&bar[kBEmpty + bs + q]);
          }
          if (closes_h) umma_commit(&bar[kDFull + buf]);
          if (closes) umma_commit(&bar[kMFull]);
        }
        __syncwarp();
        if (closes_h) ++fl;
        if (closes) ++ml;
        as += 2;
        if (as == kPairs) { as = 0; pa ^= 1u; }
        bs += 2;
        if (bs == p.ring_b) { bs = 0; if (!p.resident) pb ^= 1u; }
      }
      if (p.resident && last) pb ^= 1u;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kIssue) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// ------------------------------------------------------------------------------------------ host
bool plan33(int c0, int c1, int c2, Params33 *p) {
  if (c0 % 4 || c1 % 4) return false;
  p->m_tiles = dc_div_up(c2, kO);
  p->n_tiles = dc_div_up(c0, kI);
  if ((long long)p->m_tiles * p->n_tiles >= (1 << 24) || c1 > 4096) return false;
  p->items = p->m_tiles * p->n_tiles;
  // a multiple of the pairs: each slot then belongs to one pair for good, whose waits on it are in order (a wait tells a phase from
  // the one before it by a bit)
  p->steps = dc_div_up(c1, 16 * kPairs) * kPairs;
  const int scale = (int)dc_round_up((size_t)p->steps * 64, 128), fixed = kPairs * (kStepA + kRawA) + kZ + scale;
  p->resident = p->steps <= kMaxB && fixed + p->steps * kStepB <= kSmemMax;
  p->ring_b = p->resident ? p->steps : 2 * kPairs;
  p->off_raw = kPairs * kStepA;
  p->off_b = p->off_raw + kPairs * kRawA;
  p->off_z = p->off_b + p->ring_b * kStepB;
  p->off_scale = p->off_z + kZ;
  p->smem_bytes = p->off_scale + scale;
  return p->smem_bytes <= kSmemMax;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *, const cuuint64_t *,
                                  const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

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

// a matrix of fp32 rows, loaded in boxes of `across` x `down`
bool matrix_map(CUtensorMap *map, EncodeTiledFn encode, const float *w, long long rows, long long columns, int across, int down) {
  const cuuint64_t dim[2] = {(cuuint64_t)columns, (cuuint64_t)rows}, str[1] = {4 * (cuuint64_t)columns};
  const cuuint32_t box[2] = {(cuuint32_t)across, (cuuint32_t)down}, es[2] = {1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float *>(w), dim, str, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

dc_status dc_launch_compose33_tc(const Compose33 &a, const BlockDelivery &dv, DcWsHeader *ws, cudaStream_t st) {
  Params33 p{};
  if (!plan33(a.c0, a.c1, a.c2, &p)) return DC_ERR_UNSUPPORTED;
  EncodeTiledFn encode = get_encode_fn();
  CUtensorMap map_w2;
  if (!encode || !matrix_map(&map_w2, encode, a.second.l.w, a.c2, 9ll * a.c1, 144, kO)) return DC_ERR_CUDA;
  static unsigned char attr_done[kDcMaxDevices];
  DC_CUDA_OK(dc_set_max_smem_once(k_compose33_tc, kSmemMax, attr_done));
  const int n_sm = dc_sm_count();
  const cudaError_t e = dc_launch_pdl(k_compose33_tc, dim3((unsigned)(p.items < n_sm ? p.items : n_sm)), dim3(kThreads),
                                      (size_t)p.smem_bytes, st, map_w2, a, dv, p, ws);
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? DC_OK : DC_ERR_CUDA;
}

cudaError_t dc_merge_tc_flag(unsigned int **flag) { return cudaGetSymbolAddress((void **)flag, g_merge_status); }
