// Dense convolution in fp32 on the tensor core, by operands cut into bf16 terms.
//
// An fp32 value of 2^-110 or more is exactly three bf16 terms of 8 significant bits each (smaller ones are to within 2^-133: the smallest
// bf16 ends there), so a product of two values is nine products of terms, of which six are above 2^-24: hh, hm, mh, hl, mm, lh.
// tcgen05.mma multiplies bf16 terms exactly; its fp32 sums are cut instead of rounded, which over a long reduction would cost
// more than fp32 FMAs do (2.7e-6 of the result after 800 products).  So the sums are kept short and apart: hh, hm + mh and
// hl + mm + lh have accumulators of their own, and after at most kFlush steps of 16 products they are read out and added to the
// outputs' sums in registers by ordinary fp32 additions.  Measured against 64 bits on normal values (2-norm): 288 products
// 0.8e-7, 800 1.0e-7, 2400 1.35e-7, where one chain of FMAs has 3.0e-7, 5.1e-7 and 8.7e-7, eight chains 1.2e-7, 1.9e-7, 3.2e-7.  Where all
// products have one sign, what is cut off adds up: maps behind ReLU6 under weights of one sign, 19 layers, 0.6 to 0.9e-7, 0.28 to 0.84 of
// k_conv_dense_f32's error, one of them 1.06 of it (20 -> 36 5x5, 0.72e-7).
//
// The three groups cost no instruction of their own: the B operand of a step holds the terms of NT output channels one behind
// the other, [h | m | l], and A_h x [h m l], A_m x [h m], A_l x [h] are three instructions of 3 NT, 2 NT and NT columns whose
// results start at the accumulator columns of hh, mh and lh.  NT is at most 80 (256 columns an instruction, and two sets of 3 NT of
// the 512 columns).
//
// GEMM rows are the lines of one long raster: the images' padded rows one behind the other, the zeros right of a row being those
// left of the next one and the zeros below an image those above the next one (stride 1; at stride 2 one such raster for
// each parity of row and column).  A tile is any 128 lines of it; tap (u, v) reads the same lines u rows and v lines further
// on.  Lines lie 16 bytes apart for each 8 channels (no swizzle), so a tap is a start address, and a group of 16
// channels is cut into terms once for all its taps.
//
// Warps: one asks for fp32 operands by TMA (zeros outside the image come with them), nine cut them into terms (some of them
// activations, the others weights, whose 8 channels of an output become one 16-byte piece on the way), two issue in turn, a set
// of accumulators each (an issuing warp is never far ahead of the tensor core, so what it does between two runs of
// instructions would stand in the open), four add the accumulators up, each thread one pixel x NT outputs, and store.  Few tiles: a cluster of up to eight CTAs shares the channel
// groups of a tile, and the parts are added in rank order through distributed shared memory.
//
// An infinity or a NaN makes NaN of the outputs that read it (its difference from its first term is one): an output that is
// NaN is computed again by FMAs, so infinities and NaN come out as they do there.
//
// What bounds it.  NT = 32: an instruction is bound by fetching its 128 x 16 operand, a step of 128 lines takes 190 cycles
// (3 x 32 of them that fetch); at NT = 80 256, for 2.5 times the products.  With two runs of 128 lines to a step of weights (NT <= 32)
// the cuts stay behind that; with one the weights' cuts take about as long.  Before the first instruction 3.5 us: setup,
// TMA, first cuts, every role's instructions cold.  So small layers stay with k_conv_dense_f32 (the rule is at make_plan).  32 -> 32
// 5x5, 32 images of 28 x 28 45.5 -> 19.5 us; 208 -> 96 3x3, one 96 x 97 140 -> 42; 56 -> 128 5x5, one 94 x 96 114 -> 39; 328 -> 56
// 1x1, 78 of 15 x 15 36 -> 19.
//
// On the way (first layer): weights and activations through cp.async slots and a wait for each step of weights 41.7 us; by TMA the same; waits
// and commits by chunks 27.8; two issuing warps 24.4; two runs of lines 19.8; terms by integer rounding the same.
#include "tc_ptx.cuh"

namespace {
using namespace tc;

constexpr int kWarpsAcc = 4, kWarpsCut = 9;
constexpr int kLoad = kWarpsAcc + kWarpsCut, kIssue = kLoad + 1;     // the loading warp and the first of two issuing ones
constexpr int kThreads = (kIssue + 2) * 32;      // sixteen warps: 128 registers a thread
constexpr int kFlush = 4;                        // steps of 16 products between two read-outs, at most: a chunk
constexpr int kMaxStages = 6;                    // of a ring
constexpr int kMaxTaps = 49, kMaxChunks = 16, kMaxSplit = 8;
constexpr int kSmemMax = 225 * 1024;

struct Params {
  int n, h, w, ho, wo, c_in, c_out, k, stride, pad, act;
  int hv, wv;                  // rows of an image and lines of a row in the raster
  int tiles, passes, items;
  int groups, planes, taps;    // groups of 16 channels; parities that have taps; k * k
  int per_stage, units;        // groups of an activation stage; stages of a plane: a chunk is part of one
  int chunk_steps;             // steps of the longest chunk
  int lines;                   // raster lines that a tile reads
  int pitch;                   // lines between the two halves of a group: 4 more than a multiple of 8 (stores without bank conflicts)
  int flat;                    // 1x1: all pixels are one run
  int boxes, box_lines, box_rows;            // loads of a tile's lines: raster rows, or whole images of small maps
  int stages_a, stages_w, raw_a, raw_w;      // of the rings of terms and of fp32 operands
  int warps_a;                 // of those that cut
  int w_boxes;                 // loads of a chunk's weights: one, or one to a step
  int split, units_per;        // CTAs that share an item, units of each
  int off_raw_a, off_raw_w, off_a, off_w, off_out;
  int tmem_cols;
  unsigned char plane_q[4];    // parity (row * 2 + column) of a plane
  unsigned char plane_first[5];              // its first chunk
  unsigned char chunk_tap[kMaxChunks + 1];   // first tap of a chunk
  unsigned char tap_uv[kMaxTaps + 32];         // tap row * k + tap column, by planes
  unsigned short tap_line[kMaxTaps + kFlush];       // lines that the tap is further on
};

__device__ __forceinline__ void store4(const Params &p, const float *bias, const float *residual, float *y, int pix, int o, float4 s) {
  if (bias) {
    const float4 b = *reinterpret_cast<const float4 *>(bias + o);
    s.x += b.x; s.y += b.y; s.z += b.z; s.w += b.w;
  }
  const size_t at = (size_t)pix * p.c_out + o;
  if (residual) {
    const float4 r = *reinterpret_cast<const float4 *>(residual + at);
    s.x += r.x; s.y += r.y; s.z += r.z; s.w += r.w;
  }
  if (p.act == DC_ACT_RELU6) {
    s.x = dc_act_apply(s.x, DC_ACT_RELU6); s.y = dc_act_apply(s.y, DC_ACT_RELU6);
    s.z = dc_act_apply(s.z, DC_ACT_RELU6); s.w = dc_act_apply(s.w, DC_ACT_RELU6);
  }
  *reinterpret_cast<float4 *>(y + at) = s;
}
// Four outputs by FMAs over (tap row, tap column, channel): where the terms gave NaN; four sums that are all NaN stay so.  A thread to four
// outputs is slow: 32 -> 32 5x5, 32 images of 28 x 28, 20 us, with a NaN in one pixel 238, in all of one image 200, in all of them 320
// (without the way out behind a tap, and channel by channel, 443, 2330 and 2390; k_conv_dense_f32 47 in any case).  More loads at once (eight
// channels: 168 and 229) cost the kernel registers, 5 % where there is no NaN.
__device__ __noinline__ void outputs_by_fma(const Params &p, const float *x, const float *w, const float *bias, const float *residual, float *y,
                                            int pix, int o) {
  const int t = pix / p.wo, X = pix - t * p.wo, img = t / p.ho, Y = t - img * p.ho;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
  for (int tap = 0; tap < p.taps; ++tap) {
    const int u = tap / p.k, iy = Y * p.stride + u - p.pad, ix = X * p.stride + tap - u * p.k - p.pad;
    const bool in = (unsigned)iy < (unsigned)p.h && (unsigned)ix < (unsigned)p.w;     // the padding's zeros are multiplied as well
    const float *xp = x + (in ? ((size_t)(img * p.h + iy) * p.w + ix) * p.c_in : 0);
    const float *wp = w + (size_t)tap * p.c_in * p.c_out + o;
#pragma unroll 2
    for (int c = 0; c < p.c_in; ++c) {
      const float a = in ? xp[c] : 0.f;
      const float4 b = *reinterpret_cast<const float4 *>(wp + (size_t)c * p.c_out);
      s.x = fmaf(a, b.x, s.x); s.y = fmaf(a, b.y, s.y); s.z = fmaf(a, b.z, s.z); s.w = fmaf(a, b.w, s.w);
    }
    if (s.x != s.x && s.y != s.y && s.z != s.z && s.w != s.w) break;
  }
  store4(p, bias, residual, y, pix, o, s);
}

// the barriers of a CTA: operands as they come (RA, RW) and their terms (A, W), full and empty; accumulators
enum { kRaFull = 0, kRaEmpty = kMaxStages, kRwFull = 2 * kMaxStages, kRwEmpty = 3 * kMaxStages, kAFull = 4 * kMaxStages,
       kAEmpty = 5 * kMaxStages, kWFull = 6 * kMaxStages, kWEmpty = 7 * kMaxStages, kDFull = 8 * kMaxStages, kDEmpty = kDFull + 2,
       kBars = kDEmpty + 2 };

template <int NT, int T>
__global__ void __launch_bounds__(kThreads, 1)
k_conv_f32_tc(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w, const float *__restrict__ x,
              const float *__restrict__ w, const float *__restrict__ bias, const float *residual, float *y,
              const __grid_constant__ Params p, DcWsHeader *ws) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ uint64_t bar[kBars];
  __shared__ uint4 chunk_s[kMaxChunks];          // steps, first and last of its parity, first tap; operand lines that each step is further on
  __shared__ uint32_t tmem_s, abort_s;
  volatile uint32_t *abort_flag = &abort_s;
  const int tid = (int)threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t sm = smem_u32(smem);
  const uint32_t raw_group = (uint32_t)(p.boxes * p.box_lines) * 64u, raw_a_bytes = raw_group * (uint32_t)p.per_stage;
  const uint32_t chunk_a = (uint32_t)p.pitch * 16u, stage_a = chunk_a * 6u * (uint32_t)p.per_stage;
  constexpr uint32_t kRawStep = NT * 64u, kStep = NT * 96u, kHalf = NT * 48u;              // a step's weights, in fp32 and in terms
  const uint32_t raw_w_bytes = kRawStep * (uint32_t)p.chunk_steps, stage_w = kStep * (uint32_t)p.chunk_steps;
  const int rank = p.split > 1 ? (int)blockIdx.x % p.split : 0;
  const int first_item = (int)blockIdx.x / p.split, step_item = (int)gridDim.x / p.split;
  const int u_begin = rank * p.units_per, u_end = u_begin + p.units_per < p.units ? u_begin + p.units_per : p.units;
  const int n_chunks = p.plane_first[p.planes], warps_w = kWarpsCut - p.warps_a;
  // steps of a chunk: some taps of a 3x3 kernel or larger, or a unit's channel groups
  auto steps_of = [&](int unit, uint4 ch) {
    const int n = (int)(ch.x & 0xFFu), left = p.groups - unit * p.per_stage;
    return p.taps > 1 || left >= n ? n : left;
  };
  if (tid < kBars) {
    const int kind = tid / kMaxStages;
    uint32_t count = 1;
    if (tid >= kDEmpty) count = kWarpsAcc;
    else if (kind == kRaEmpty / kMaxStages || kind == kAFull / kMaxStages) count = (uint32_t)p.warps_a;
    else if (kind == kRwEmpty / kMaxStages || kind == kWFull / kMaxStages) count = (uint32_t)warps_w;
    else if (kind == kAEmpty / kMaxStages) count = 2;
    mbar_init(&bar[tid], count);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  } else if (tid >= 64 && tid < 64 + n_chunks) {
    const int c = tid - 64;
    uint4 e = make_uint4((uint32_t)p.chunk_tap[c] << 16, 0u, 0u, 0u);
    if (p.taps > 1) {
      const unsigned short *l = p.tap_line + p.chunk_tap[c];
      e.x |= (uint32_t)(p.chunk_tap[c + 1] - p.chunk_tap[c]);
      e.y = (uint32_t)l[0] | ((uint32_t)l[1] << 16);
      e.z = (uint32_t)l[2] | ((uint32_t)l[3] << 16);
    } else {
      e.x |= (uint32_t)p.per_stage;
      e.y = (uint32_t)(6 * p.pitch) << 16;
    }
#pragma unroll 1
    for (int pl = 0; pl < p.planes; ++pl) e.x |= (c == p.plane_first[pl] ? 0x100u : 0u) | (c + 1 == p.plane_first[pl + 1] ? 0x200u : 0u);
    chunk_s[c] = e;
  } else if (tid == 96) {
    abort_s = 0;
    prefetch_tensormap(&map_x);
    prefetch_tensormap(&map_w);
  }
  __syncthreads();
  dc_pdl_enter();                                // global memory and tensor memory only behind this
  if (warp < kWarpsAcc || warp >= kIssue) {      // the others start at once
    if (warp == kIssue) {
      tmem_alloc(&tmem_s, (uint32_t)p.tmem_cols);
      tmem_relinquish();
    }
    tc_fence_before();
    bar_sync(1, (kWarpsAcc + 2) * 32);
    tc_fence_after();
  }
  const uint32_t tmem = tmem_s;

  auto wait = [&](int b, uint32_t parity, uint32_t site) { return warp_wait(&bar[b], parity, abort_flag, ws, site); };
  // two barriers at once, by the even and the odd lanes; `tid`'s warp meets behind them
  auto wait2 = [&](int b0, uint32_t par0, int b1, uint32_t par1, uint32_t site) {
    const bool ok = mbar_wait(&bar[lane & 1 ? b1 : b0], lane & 1 ? par1 : par0, abort_flag, ws, site + (uint32_t)(lane & 1));
    __syncwarp();
    return __all_sync(0xffffffffu, ok) != 0;
  };
  auto locate = [&](int line, int &img, int &row, int &col) {
    const int q = line / p.wv;
    col = line - q * p.wv;
    img = q / p.hv;
    row = q - img * p.hv;
  };
  // 16-byte piece `pc` of a pixel's NT sums in shared memory, without bank conflicts between pixels
  auto piece = [](int row, int pc) {
    return (uint32_t)(row * NT * 4 + ((NT / 16) % 2 ? (pc ^ ((row >> 1) & 3)) : (pc ^ (row & 7))) * 16);
  };

  if (warp < kWarpsAcc) {
    // ---------------------------------------------------------------- accumulators: T pixels x NT outputs to a thread
    const uint32_t drow = tmem + ((uint32_t)(warp * 32) << 16);
    const uint32_t out_s = sm + (p.split > 1 ? 0u : (uint32_t)p.off_out) + (uint32_t)(warp * 32 * NT * 4);
    const int chunks = (u_end - u_begin) * n_chunks;
    uint32_t fl = 0;
    bool ok = true;
#pragma unroll 1
    for (int item = first_item; item < p.items && ok; item += step_item) {
      float acc[T][NT];
#pragma unroll
      for (int j = 0; j < T * NT; ++j) acc[j / NT][j % NT] = 0.f;
#pragma unroll 1
      for (int s = 0; s < chunks; ++s, ++fl) {
        const uint32_t b = fl & 1u;
        if (!(ok = wait(kDFull + (int)b, (fl >> 1) & 1u, 0x100000u))) break;
        tc_fence_after();
        constexpr int V = NT >= 64 ? 8 : 16;       // columns at a time (registers)
#pragma unroll
        for (int c = 0; c < T * NT; c += V) {
          uint32_t v0[V], v1[V], v2[V];
          const uint32_t at = drow + b * (3 * NT * T) + (c / NT) * (3 * NT) + c % NT;
          tmem_ld_cols<V>(at, v0);
          tmem_ld_cols<V>(at + NT, v1);
          tmem_ld_cols<V>(at + 2 * NT, v2);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < V; ++j)
            acc[c / NT][c % NT + j] += __uint_as_float(v0[j]) + (__uint_as_float(v1[j]) + __uint_as_float(v2[j]));
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bar[kDEmpty + b]);
      }
      if (!ok) break;
      const int pass = item / p.tiles, line0 = (item - pass * p.tiles) * (128 * T);
      if (p.split > 1) __syncthreads();          // the rings are no longer in use: the parts go there (with the other roles, below)
#pragma unroll
      for (int t = 0; t < T; ++t) {
#pragma unroll
        for (int q = 0; q < NT / 4; ++q)
          sts_u4(out_s + piece(lane, q), make_uint4(__float_as_uint(acc[t][4 * q]), __float_as_uint(acc[t][4 * q + 1]), __float_as_uint(acc[t][4 * q + 2]), __float_as_uint(acc[t][4 * q + 3])));
        if (p.split > 1) break;
        __syncwarp();
        int img, Y, X;
        locate(line0 + t * 128 + warp * 32 + lane, img, Y, X);
        const int pix = img < p.n && Y < p.ho && X < p.wo ? (img * p.ho + Y) * p.wo + X : -1;
#pragma unroll 1
        for (int i = 0; i < NT / 4; i += 4) {    // neighbouring lanes store neighbouring pieces, four each
          float4 v[4];
          int px[4], o[4];
          uint32_t bad = 0;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int e = (i + q) * 32 + lane, r = e / (NT / 4), pc = e - r * (NT / 4);
            o[q] = pass * NT + pc * 4;
            px[q] = __shfl_sync(0xffffffffu, pix, r);
            if (o[q] >= p.c_out) px[q] = -1;
            const uint4 u = lds_u4(out_s + piece(r, pc));
            v[q] = make_float4(__uint_as_float(u.x), __uint_as_float(u.y), __uint_as_float(u.z), __uint_as_float(u.w));
            const float sum = (v[q].x + v[q].y) + (v[q].z + v[q].w);        // NaN where one of them is
            if (px[q] >= 0 && sum != sum) bad |= 1u << q;
          }
          if (bias)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float4 a = px[q] >= 0 ? *reinterpret_cast<const float4 *>(bias + o[q]) : make_float4(0.f, 0.f, 0.f, 0.f);
              v[q].x += a.x; v[q].y += a.y; v[q].z += a.z; v[q].w += a.w;
            }
          if (residual)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float4 a = px[q] >= 0 ? *reinterpret_cast<const float4 *>(residual + (size_t)px[q] * p.c_out + o[q]) : make_float4(0.f, 0.f, 0.f, 0.f);
              v[q].x += a.x; v[q].y += a.y; v[q].z += a.z; v[q].w += a.w;
            }
          if (p.act == DC_ACT_RELU6)
#pragma unroll
            for (int q = 0; q < 4; ++q)
              v[q] = make_float4(dc_act_apply(v[q].x, DC_ACT_RELU6), dc_act_apply(v[q].y, DC_ACT_RELU6), dc_act_apply(v[q].z, DC_ACT_RELU6), dc_act_apply(v[q].w, DC_ACT_RELU6));
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (px[q] >= 0 && !((bad >> q) & 1u)) *reinterpret_cast<float4 *>(y + (size_t)px[q] * p.c_out + o[q]) = v[q];
          if (bad)
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if ((bad >> q) & 1u) outputs_by_fma(p, x, w, bias, residual, y, px[q], o[q]);
        }
        __syncwarp();
      }
      if (p.split > 1) break;
    }
    if (p.split > 1 && !ok) __syncthreads();
  } else if (warp < kWarpsAcc + p.warps_a) {
    // ---------------------------------------------------------------- activations into terms: 8 channels of a line to a thread
    const int half = lane & 1, first = (warp - kWarpsAcc) * 16 + (lane >> 1), step = p.warps_a * 16;
    const int stages = (u_end - u_begin) * p.planes;
    int sr = 0, st = 0;
    uint32_t pr = 0, ph = 1;
    bool ok = true;
#pragma unroll 1
    for (int item = first_item; item < p.items && ok; item += step_item) {
      const int line0 = item % p.tiles * (128 * T);
      const uint32_t src = sm + (uint32_t)p.off_raw_a + (uint32_t)(line0 % p.box_lines) * 64u + (uint32_t)half * 32u;
#pragma unroll 1
      for (int s = 0; s < stages; ++s) {
        if (!(ok = wait2(kRaFull + sr, pr, kAEmpty + st, ph, 0x110000u))) break;
#pragma unroll 1
        for (int g = 0; g < p.per_stage; ++g) {  // groups past the last channel come as zeros and are not used
          const uint32_t from = src + (uint32_t)sr * raw_a_bytes + (uint32_t)g * raw_group;
          const uint32_t to = sm + (uint32_t)p.off_a + (uint32_t)st * stage_a + (uint32_t)(g * 6 + half) * chunk_a;
          // two lines at a time: their reads, then the arithmetic, then the stores
#pragma unroll 1
          for (int i = first; i < p.lines; i += 2 * step) {
            const bool two = i + step < p.lines;
            const uint32_t r0 = from + (uint32_t)i * 64u, r1 = two ? r0 + (uint32_t)step * 64u : r0, d0 = to + (uint32_t)i * 16u, d1 = d0 + (uint32_t)step * 16u;
            const uint4 u0 = lds_u4(r0), u1 = lds_u4(r0 + 16u), u2 = lds_u4(r1), u3 = lds_u4(r1 + 16u);
            const float v0[8] = {__uint_as_float(u0.x), __uint_as_float(u0.y), __uint_as_float(u0.z), __uint_as_float(u0.w),
                                 __uint_as_float(u1.x), __uint_as_float(u1.y), __uint_as_float(u1.z), __uint_as_float(u1.w)};
            const float v1[8] = {__uint_as_float(u2.x), __uint_as_float(u2.y), __uint_as_float(u2.z), __uint_as_float(u2.w),
                                 __uint_as_float(u3.x), __uint_as_float(u3.y), __uint_as_float(u3.z), __uint_as_float(u3.w)};
            uint4 h0, m0, l0, h1, m1, l1;
            bf16_terms8(v0, h0, m0, l0);
            bf16_terms8(v1, h1, m1, l1);
            sts_u4(d0, h0);
            sts_u4(d0 + 2 * chunk_a, m0);
            sts_u4(d0 + 4 * chunk_a, l0);
            if (two) {
              sts_u4(d1, h1);
              sts_u4(d1 + 2 * chunk_a, m1);
              sts_u4(d1 + 4 * chunk_a, l1);
            }
          }
        }
        fence_proxy_async();
        __syncwarp();
        if (lane < 2) mbar_arrive(&bar[lane ? kRaEmpty + sr : kAFull + st]);
        if (++st == p.stages_a) { st = 0; ph ^= 1u; }
        if (++sr == p.raw_a) { sr = 0; pr ^= 1u; }
      }
    }
  } else if (warp < kLoad) {
    // ---------------------------------------------------------------- weights into terms: 8 channels of an output to a thread
    const int wi = warp - kWarpsAcc - p.warps_a, hf = lane >> 4;
    int st = 0, sr = 0;
    uint32_t ph = 1, pr = 0;
    bool ok = true;
#pragma unroll 1
    for (int item = first_item; item < p.items && ok; item += step_item)
#pragma unroll 1
      for (int u = u_begin; u < u_end && ok; ++u)
#pragma unroll 1
        for (int c = 0; c < n_chunks; ++c) {
          const int turns = steps_of(u, chunk_s[c]) * (NT / 16);
          const uint32_t from = sm + (uint32_t)p.off_raw_w + (uint32_t)sr * raw_w_bytes, to = sm + (uint32_t)p.off_w + (uint32_t)st * stage_w;
          // the places of turn e0 (32 times 8 channels of an output): where its weights lie, and where their terms go
          auto place = [&](int e0, uint32_t &f, uint32_t &d) {
            const int q = e0 / (NT / 16), e = (e0 - q * (NT / 16)) * 32 + hf * 16, chunk = e >= NT ? 1 : 0, o = e - chunk * NT + (lane & 15);
            f = from + (uint32_t)q * kRawStep + (uint32_t)((chunk * 8 * NT + o) * 4);
            d = to + (uint32_t)q * kStep + (uint32_t)chunk * kHalf + (uint32_t)o * 16u;
          };
          if (!(ok = wait2(kRwFull + sr, pr, kWEmpty + st, ph, 0x120000u))) break;
#pragma unroll 1
          for (int e0 = wi; e0 < turns; e0 += 2 * warps_w) {
            const bool two = e0 + warps_w < turns;
            uint32_t f0, d0, f1, d1;
            place(e0, f0, d0);
            place(two ? e0 + warps_w : e0, f1, d1);
            float v0[8], v1[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) v0[j] = lds_f(f0 + (uint32_t)(j * NT * 4));
#pragma unroll
            for (int j = 0; j < 8; ++j) v1[j] = lds_f(f1 + (uint32_t)(j * NT * 4));
            uint4 h0, m0, l0, h1, m1, l1;
            bf16_terms8(v0, h0, m0, l0);
            bf16_terms8(v1, h1, m1, l1);
            sts_u4(d0, h0);
            sts_u4(d0 + NT * 16u, m0);
            sts_u4(d0 + NT * 32u, l0);
            if (two) {
              sts_u4(d1, h1);
              sts_u4(d1 + NT * 16u, m1);
              sts_u4(d1 + NT * 32u, l1);
            }
          }
          fence_proxy_async();
          __syncwarp();
          if (lane < 2) mbar_arrive(&bar[lane ? kRwEmpty + sr : kWFull + st]);
          if (++st == p.stages_w) { st = 0; ph ^= 1u; }
          if (++sr == p.raw_w) { sr = 0; pr ^= 1u; }
        }
  } else if (warp == kLoad) {
    // ---------------------------------------------------------------- loads, in the order in which they are used
    int sa = 0, sw = 0;
    uint32_t pa = 1, pw = 1;
    bool ok = true;
    const int boxes = p.boxes * p.per_stage;
#pragma unroll 1
    for (int item = first_item; item < p.items && ok; item += step_item) {
      const int pass = item / p.tiles, box0 = (item - pass * p.tiles) * (128 * T) / p.box_lines;
#pragma unroll 1
      for (int u = u_begin; u < u_end && ok; ++u)
#pragma unroll 1
        for (int pl = 0; pl < p.planes && ok; ++pl) {
          if (!(ok = wait(kRaEmpty + sa, pa, 0x160000u))) break;
          if (lane == 0) mbar_arrive_expect_tx(&bar[kRaFull + sa], raw_a_bytes);
          __syncwarp();
          const int y0 = (p.plane_q[pl] >> 1) - p.pad, x0 = (p.plane_q[pl] & 1) - p.pad;
#pragma unroll 1
          for (int e = lane; e < boxes; e += 32) {
            const int g = e / p.boxes, b = e - g * p.boxes, ch = (u * p.per_stage + g) * 16;
            const uint32_t to = sm + (uint32_t)p.off_raw_a + (uint32_t)sa * raw_a_bytes + (uint32_t)g * raw_group + (uint32_t)(b * p.box_lines) * 64u;
            int cx = x0, cy = y0, img = 0;
            if (p.flat) {
              cx = (box0 + b) * p.box_lines;
            } else {
              const int row = (box0 + b) * p.box_rows;
              img = row / p.hv;
              cy += p.stride * (row - img * p.hv);
            }
            tma_load_4d(to, &map_x, &bar[kRaFull + sa], ch, cx, cy, img);
          }
          __syncwarp();
          if (++sa == p.raw_a) { sa = 0; pa ^= 1u; }
#pragma unroll 1
          for (int c = p.plane_first[pl]; c < p.plane_first[pl + 1]; ++c) {
            const uint4 ch = chunk_s[c];
            const int n = p.w_boxes > 1 ? steps_of(u, ch) : 1;
            const uint32_t to = sm + (uint32_t)p.off_raw_w + (uint32_t)sw * raw_w_bytes + (uint32_t)lane * kRawStep;
            const int tap = p.w_boxes > 1 ? p.tap_uv[(ch.x >> 16) + lane] : (int)(ch.x >> 16);
            if (!(ok = wait(kRwEmpty + sw, pw, 0x170000u))) break;
            if (lane == 0) mbar_arrive_expect_tx(&bar[kRwFull + sw], p.w_boxes > 1 ? kRawStep * (uint32_t)n : raw_w_bytes);
            __syncwarp();
            if (lane < n) tma_load_3d(to, &map_w, &bar[kRwFull + sw], pass * NT, u * p.per_stage * 16, tap);
            __syncwarp();
            if (++sw == p.raw_w) { sw = 0; pw ^= 1u; }
          }
        }
    }
    if (!ok) {                                   // copies may still be in flight: give them time to land
      const unsigned long long t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    }
  } else {
    // ---------------------------------------------------------------- issue
    const uint32_t id0 = (1u << 4) | (1u << 7) | (1u << 10) | (8u << 24);
    const uint32_t i3 = id0 | ((3 * NT / 8) << 17), i2 = id0 | ((2 * NT / 8) << 17), i1 = id0 | ((NT / 8) << 17);
    const uint64_t hi = (uint64_t)((128u >> 4) | (1u << 14)) << 32;
    const uint64_t a_hi = hi | ((uint64_t)p.pitch << 16), b_hi = hi | ((uint64_t)(3 * NT) << 16);
    const uint32_t term_a = chunk_a >> 3;        // 16-byte units between terms
    const uint32_t mine = (uint32_t)(warp - kIssue), d = tmem + mine * (3 * NT * T);
    int sa = 0, sw = 0;
    uint32_t pa = 0, pw = 0, pd = 1, fl = 0;
    bool ok = true;
#pragma unroll 1
    for (int item = first_item; item < p.items && ok; item += step_item)
#pragma unroll 1
      for (int u = u_begin; u < u_end && ok; ++u)
#pragma unroll 1
        for (int c = 0; c < n_chunks; ++c, ++fl) {
          const uint4 ch = chunk_s[c];
          const bool my = (fl & 1u) == mine, last = (ch.x & 0x200u) != 0;
          if ((ch.x & 0x100u) && !(ok = wait(kAFull + sa, pa, 0x130000u))) break;
          if (my) {
            const int n = steps_of(u, ch);
            const uint32_t a0 = (sm + (uint32_t)p.off_a + (uint32_t)sa * stage_a) >> 4, b0 = (sm + (uint32_t)p.off_w + (uint32_t)sw * stage_w) >> 4;
            const uint32_t a[kFlush] = {a0 + (ch.y & 0xFFFFu), a0 + (ch.y >> 16), a0 + (ch.z & 0xFFFFu), a0 + (ch.z >> 16)};
            if (!(ok = wait2(kDEmpty + (int)mine, pd, kWFull + sw, pw, 0x140000u))) break;
            pd ^= 1u;
            tc_fence_after();
            if (elect_one()) {
#pragma unroll
              for (int q = 0; q < kFlush; ++q)
                if (q < n) {
                  const uint64_t bd = b_hi | (uint64_t)((b0 + q * (kStep >> 4)) & 0x3FFFu);
#pragma unroll
                  for (int t = 0; t < T; ++t) {
                    const uint32_t dt = d + t * (3 * NT), at = a[q] + t * 128;
                    umma_bf16(dt, a_hi | (uint64_t)(at & 0x3FFFu), bd, i3, q == 0 ? 0u : 1u);
                    umma_bf16(dt + NT, a_hi | (uint64_t)((at + term_a) & 0x3FFFu), bd, i2, 1u);
                    umma_bf16(dt + 2 * NT, a_hi | (uint64_t)((at + 2 * term_a) & 0x3FFFu), bd, i1, 1u);
                  }
                }
              umma_commit(&bar[kDFull + mine]);
              umma_commit(&bar[kWEmpty + sw]);
              if (last) umma_commit(&bar[kAEmpty + sa]);
            }
            __syncwarp();
          } else if (last) {                     // the other warp's run ends the stage: this one's instructions on it count as well
            if (elect_one()) umma_commit(&bar[kAEmpty + sa]);
            __syncwarp();
          }
          if (++sw == p.stages_w) { sw = 0; pw ^= 1u; }
          if (last && ++sa == p.stages_a) { sa = 0; pa ^= 1u; }
        }
  }
  if (p.split > 1) {
    // ---- the parts of the cluster's CTAs, [pixel][NT], added in rank order; each CTA stores its share
    if (warp >= kWarpsAcc) __syncthreads();      // the accumulating warps wait for this above
    cluster_sync();
    const int pass = first_item / p.tiles, tile = first_item - pass * p.tiles;
    if (*abort_flag == 0)
#pragma unroll 1
      for (int e = rank * kThreads + tid; e < 128 * (NT / 4); e += p.split * kThreads) {
        const int m = e / (NT / 4), pc = e - m * (NT / 4), o = pass * NT + pc * 4;
        int img, Y, X;
        locate(tile * 128 + m, img, Y, X);
        if (img >= p.n || Y >= p.ho || X >= p.wo || o >= p.c_out) continue;
        const uint32_t at = sm + (uint32_t)(m & ~31) * (NT * 4) + piece(m & 31, pc);
        float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
        for (int r = 0; r < p.split; ++r) {
          const uint4 v = lds_cluster_u4(map_cluster(at, (uint32_t)r));
          s.x += __uint_as_float(v.x); s.y += __uint_as_float(v.y); s.z += __uint_as_float(v.z); s.w += __uint_as_float(v.w);
        }
        const int pix = (img * p.ho + Y) * p.wo + X;
        if (s.x != s.x || s.y != s.y || s.z != s.z || s.w != s.w) outputs_by_fma(p, x, w, bias, residual, y, pix, o);
        else store4(p, bias, residual, y, pix, o, s);
      }
    cluster_sync();                              // nobody leaves while its part may still be read
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kIssue) {
    tc_fence_after();
    tmem_dealloc(tmem, (uint32_t)p.tmem_cols);
  }
}

// ------------------------------------------------------------------------------------------ host
// one shape in tiles of 128 tn lines x nt outputs, shared by `split` CTAs each; false: it does not apply
bool grid_of(int n, int h, int w, const dc_geom *g, int nt, int tn, int split, Params *p) {
  if (tn > 1 && (split > 1 || 6 * nt * tn > 512)) return false;
  if (g->groups != 1 || g->c_in % 4 || g->c_out % 4 || g->stride > 2 || g->k > 7 || g->pad >= g->k) return false;
  const int k = g->k, s = g->stride, ho = dc_out_extent(h, k, s, g->pad), wo = dc_out_extent(w, k, s, g->pad);
  if (ho <= 0 || wo <= 0) return false;
  *p = Params{};
  p->n = n; p->h = h; p->w = w; p->ho = ho; p->wo = wo;
  p->c_in = g->c_in; p->c_out = g->c_out; p->k = k; p->stride = s; p->pad = g->pad;
  // lines of a raster row are an even number: a row is loaded to a multiple of 128 bytes
  p->flat = k == 1 && s == 1 && g->pad == 0;
  if ((long long)n * (h + g->pad + k) * (w + g->pad + k + 1) >= (1ll << 29)) return false;
  if (p->flat) {
    p->w = p->wo = p->wv = n * h * w;
    p->n = p->h = p->ho = p->hv = 1;
    p->box_lines = 128 * tn;
    p->box_rows = 1;
  } else {
    p->hv = s == 1 ? h + g->pad : ho + (k - 1) / 2;
    p->wv = ((s == 1 ? w + g->pad : wo + (k - 1) / 2) + 1) & ~1;
    if (p->wv * s > 256) return false;           // a tensor map's box
    // a load takes rows that divide an image's: few loads, few lines beside the tile's
    p->box_rows = 1;
    for (int r = 2; r <= p->hv && r * p->wv <= 64 && r * s <= 256; ++r)
      if (p->hv % r == 0) p->box_rows = r;
    if (p->hv * p->wv <= 160 && p->hv * s <= 256) p->box_rows = p->hv;
    p->box_lines = p->box_rows * p->wv;
  }
  const long long last = ((long long)(p->n - 1) * p->hv + p->ho - 1) * p->wv + p->wo;
  p->tiles = (int)((last + 128 * tn - 1) / (128 * tn));
  p->passes = dc_div_up(g->c_out, nt);
  if ((long long)p->tiles * p->passes >= (1ll << 24)) return false;
  p->items = p->tiles * p->passes;
  p->groups = dc_div_up(g->c_in, 16);
  p->taps = k * k;
  // 1x1: two channel groups to a stage, one chunk; else the taps of a parity, cut evenly into chunks
  p->per_stage = k == 1 ? 2 : 1;
  p->units = dc_div_up(p->groups, p->per_stage);
  p->chunk_steps = p->per_stage;
  int tap = 0, reach = 0, chunks = 0;
  for (int q = 0; q < (s == 1 ? 1 : 4); ++q) {
    const int first = tap;
    for (int u = q >> 1; u < k; u += s)
      for (int v = q & 1; v < k; v += s) {
        const int line = (u / s) * p->wv + v / s;
        if (line > 16000) return false;
        p->tap_uv[tap] = (unsigned char)(u * k + v);
        p->tap_line[tap++] = (unsigned short)line;
        if (line > reach) reach = line;
      }
    if (tap == first) continue;
    p->plane_q[p->planes] = (unsigned char)q;
    p->plane_first[p->planes++] = (unsigned char)chunks;
    const int n = tap - first, nc = dc_div_up(n, kFlush);
    for (int c = 0; c < nc; ++c) {
      p->chunk_tap[chunks++] = (unsigned char)(first + (int)((long long)n * c / nc));
      const int steps = (int)((long long)n * (c + 1) / nc) - (int)((long long)n * c / nc);
      if (steps > p->chunk_steps) p->chunk_steps = steps;
    }
  }
  p->plane_first[p->planes] = (unsigned char)chunks;
  p->chunk_tap[chunks] = (unsigned char)tap;
  p->lines = 128 * tn + reach;
  p->pitch = (p->lines + 3) / 8 * 8 + 4;
  p->split = split;
  if (split > p->units) return false;
  p->units_per = dc_div_up(p->units, split);
  if (p->units_per * (split - 1) >= p->units) return false;          // no CTA without one
  p->w_boxes = s == 1 || k == 1 ? 1 : p->chunk_steps;
  p->boxes = p->flat ? 1 : dc_div_up(p->box_lines - 2 + p->lines, p->box_lines);
  // The warps that cut, as the work is (activations that all taps share against weights).
  const double cut_a = 2.0 * p->lines * p->planes * (k == 1 ? 2 : 1), cut_w = 2.0 * nt * p->taps * (tn == 1 ? 1 : 0.5);
  const int wa = (int)(kWarpsCut * cut_a / (cut_a + cut_w) + 0.5);
  p->warps_a = wa < 2 ? 2 : (wa > kWarpsCut - 2 ? kWarpsCut - 2 : wa);
  // the rings: what keeps loads, cuts and instructions apart, then deeper while there is room
  const long long ra = 64ll * p->boxes * p->box_lines * p->per_stage, a = 96ll * p->pitch * p->per_stage, rb = 64ll * nt * p->chunk_steps,
                  b = 96ll * nt * p->chunk_steps, out = 512ll * nt, room = kSmemMax - out - 256;
  static constexpr int kRings[3][4] = {{2, 2, 2, 2}, {1, 2, 2, 2}, {1, 1, 2, 2}};          // fp32 and terms of activations, of weights
  long long r[4] = {0, 0, 0, 0};
  auto bytes = [&]() { return r[0] * ra + r[1] * a + r[2] * rb + r[3] * b; };
  for (int i = 0; i < 3; ++i) {
    for (int j = 0; j < 4; ++j) r[j] = kRings[i][j];
    if (bytes() <= room) break;
  }
  if (bytes() > room) return false;
  for (bool grew = true; grew;) {
    grew = false;
    for (int j = 3; j >= 0; --j) {
      if (r[j] >= (j < 2 ? 4 : kMaxStages)) continue;
      ++r[j];
      if (bytes() <= room) grew = true;
      else --r[j];
    }
  }
  p->raw_a = (int)r[0]; p->stages_a = (int)r[1]; p->raw_w = (int)r[2]; p->stages_w = (int)r[3];
  p->off_raw_a = 0;
  p->off_raw_w = (int)(r[0] * ra);
  p->off_out = p->off_raw_w + (int)(r[2] * rb);
  p->off_w = p->off_out + (int)out;
  p->off_a = p->off_w + (int)(r[3] * b);
  p->tmem_cols = 32;
  while (p->tmem_cols < 6 * nt * tn) p->tmem_cols *= 2;
  return true;
}
int smem_bytes(const Params &p) { return p.off_a + p.stages_a * p.pitch * 96 * p.per_stage; }

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

struct Plan {
  Params p;
  int nt, tn;                  // outputs of a tile, runs of 128 lines
};

// Estimated time of a plan in microseconds, fitted to 300 layers (16 to 960 channels, 1x1 to 5x5, both strides, 4 MFLOP to 4
// GFLOP) timed in all their plans: 11 % off, its choice 1.7 % above the best on average.  A tile costs its instructions, its cuts of weights or
// its cuts of activations, whichever is most, and its read-out beside the next one's; shallow rings make them wait for one
// another.  Of the start-up, 3.5 us, most is a cold instruction cache in every role.
double estimate_us(const Params &p, int nt, int tn, int n_sm) {
  static constexpr int kClusters[kMaxSplit + 1] = {0, 148, 74, 45, 33, 26, 22, 15, 15};    // of that many CTAs that run at once, on 148 SMs
  const double steps = p.units_per * (p.taps > 1 ? p.taps : p.per_stage), chunks = p.units_per * p.plane_first[p.planes],
               stages = p.units_per * p.planes, turns = steps * nt / 16 / (kWarpsCut - p.warps_a);
  const double issue = steps * tn * (20 + 5.75 * nt) + chunks * 690, cut_w = chunks * 710 + (chunks > turns ? chunks : turns) * 390,
               cut_a = stages * (1000 + p.boxes * p.per_stage * 130 + dc_div_up(p.lines, 16 * p.warps_a) * p.per_stage * 230);
  double main = issue > cut_w ? issue : cut_w;
  if (cut_a > main) main = cut_a;
  main += ((p.raw_a < 2 ? 0.5 : 0.0) + (p.stages_a < 2 ? 0.5 : 0.0) + (p.raw_w < 3 || p.stages_w < 3 ? 0.45 : 0.0)) * cut_a;
  const double out = 850 + 90.0 * nt * tn;
  const double cycles = p.split > 1 ? dc_div_up(p.items, kClusters[p.split]) * (9950 + main + out / 2 + 240 * p.split)
                                    : 6650 + dc_div_up(p.items, n_sm) * (main > out ? main : out) + (main > out ? out : main);
  return cycles / 1900;
}

bool make_plan(int n, int h, int w, const dc_geom *g, int n_sm, Plan *pl) {
  // Taken from 0.85 of what the FMA kernel is estimated to need: of the 300 layers 161, together 0.756 of the time on (geometric) average,
  // one of them slower (5 %); a line at 0.8 leaves 0.758, at 0.95 it takes five that are slower, by up to 12 %.
  double best = 0.85 * dc_conv_f32_estimate_us(n, h, w, g);
  int best_nt = 0, best_tn = 0, best_split = 0;
  for (int nt = 16; nt <= 80 && nt < g->c_out + 16; nt += 16)
    for (int tn = 1; tn <= 2; ++tn)
      for (int split = 1; split <= kMaxSplit; ++split) {
        Params &p = pl->p;
        if (split == 5 || split == 7 || !grid_of(n, h, w, g, nt, tn, split, &p) || (split > 1 && p.items * split > n_sm)) continue;
        const double us = estimate_us(p, nt, tn, n_sm);
        if (us < best) { best = us; best_nt = nt; best_tn = tn; best_split = split; }
      }
  pl->nt = best_nt;
  pl->tn = best_tn;
  return best_nt != 0 && grid_of(n, h, w, g, best_nt, best_tn, best_split, &pl->p);
}
bool plan_of(int n, int h, int w, const dc_geom *g, int n_sm, Plan *pl) {
  static thread_local DcPlans<Plan> plans;
  return plans.get(DC_PLAN_KEY(n, h, w, g, n_sm), pl, [&](Plan *q) { return make_plan(n, h, w, g, n_sm, q); });
}

template <int NT, int T>
cudaError_t launch(const Params &p, const float *x, const float *w, const float *bias, const float *residual, float *y, DcWsHeader *ws,
                   int n_sm, cudaStream_t st) {
  static unsigned char attr_done[kDcMaxDevices];
  const cudaError_t e = dc_set_max_smem_once(k_conv_f32_tc<NT, T>, kSmemMax, attr_done);
  if (e != cudaSuccess) return e;
  EncodeTiledFn encode = get_encode_fn();
  if (!encode) return cudaErrorNotSupported;
  CUtensorMap map_x, map_w;
  {
    const cuuint64_t C = (cuuint64_t)p.c_in, W = (cuuint64_t)p.w, H = (cuuint64_t)p.h;
    const cuuint64_t dim[4] = {C, W, H, (cuuint64_t)p.n}, str[3] = {4 * C, 4 * C * W, 4 * C * W * H};
    const cuuint32_t S = (cuuint32_t)p.stride, box[4] = {16, S * (cuuint32_t)(p.flat ? 128 * T : p.wv), S * (cuuint32_t)p.box_rows, 1}, es[4] = {1, S, S, 1};
    if (encode(&map_x, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float *>(x), dim, str, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorNotSupported;
  }
  {
    const cuuint64_t I = (cuuint64_t)p.c_in, O = (cuuint64_t)p.c_out, dim[3] = {O, I, (cuuint64_t)p.taps}, str[2] = {4 * O, 4 * O * I};
    // a chunk's weights in one box where they lie so: both channel groups of a 1x1 layer, neighbouring taps at stride 1
    const cuuint32_t box[3] = {NT, 16u * (cuuint32_t)p.per_stage, p.w_boxes > 1 ? 1u : (cuuint32_t)(p.taps > 1 ? p.chunk_steps : 1)}, es[3] = {1, 1, 1};
    if (encode(&map_w, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float *>(w), dim, str, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return cudaErrorNotSupported;
  }
  const int grid = p.split > 1 ? p.items * p.split : (p.items < n_sm ? p.items : n_sm);
  return dc_launch_pdl_cluster(k_conv_f32_tc<NT, T>, dim3((unsigned)grid), dim3(kThreads), (size_t)smem_bytes(p), st, p.split, map_x, map_w, x, w, bias, residual, y, p, ws);
}

}  // namespace

bool dc_conv_f32_tc_supported(int n, int h, int w, const dc_geom *g) {
  Plan pl;
  return plan_of(n, h, w, g, dc_sm_count(), &pl);
}

dc_status dc_launch_conv_f32_tc(const void *x, int n, int h, int w, const dc_geom *g, const void *w_packed, const float *bias, dc_act act,
                                const void *residual, void *y, void *workspace, cudaStream_t st) {
  Plan pl;
  const int n_sm = dc_sm_count();
  if (!plan_of(n, h, w, g, n_sm, &pl)) return DC_ERR_UNSUPPORTED;
  pl.p.act = (int)act;
  const float *xf = (const float *)x, *wf = (const float *)w_packed, *rf = (const float *)residual;
  float *yf = (float *)y;
  DcWsHeader *ws = (DcWsHeader *)workspace;
  cudaError_t e;
  switch (pl.nt * 10 + pl.tn) {
    case 161: e = launch<16, 1>(pl.p, xf, wf, bias, rf, yf, ws, n_sm, st); break;
    case 162: e = launch<16, 2>(pl.p, xf, wf, bias, rf, yf, ws, n_sm, st); break;
    case 321: e = launch<32, 1>(pl.p, xf, wf, bias, rf, yf, ws, n_sm, st); break;
    case 322: e = launch<32, 2>(pl.p, xf, wf, bias, rf, yf, ws, n_sm, st); break;
    case 481: e = launch<48, 1>(pl.p, xf, wf, bias, rf, yf, ws, n_sm, st); break;
    case 641: e = launch<64, 1>(pl.p, xf, wf, bias, rf, yf, ws, n_sm, st); break;
    default: e = launch<80, 1>(pl.p, xf, wf, bias, rf, yf, ws, n_sm, st); break;
  }
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? DC_OK : DC_ERR_CUDA;
}
