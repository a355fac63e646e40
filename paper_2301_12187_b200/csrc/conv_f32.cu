// Dense convolution in fp32 (the accuracy path): an implicit GEMM on the FMA pipes.
//
// M = output pixels (all images in one run), N = output channels, K = (tap row, tap column, input
// channel) in the order of the packed weights [k][k][c_in][c_out], whose rows are therefore simply
// rows of B.  Tensor cores are out: tf32 and bf16 operands lose the precision this path is for.
//
// What bounds it is the FMA pipes (148 SMs x 128 x 2 x 1.965 GHz = 74 TFLOP/s) and the shared-memory
// reads that feed them, so the tile is built around those:
//  * a thread owns TM pixels x TN channels; four K of a pixel are one 16-byte read, four (or two)
//    channels of a K another: TM + TN reads for 4 TM TN FMAs, and no operand is turned around on its
//    way in;
//  * slices of 16 K are staged by cp.async several deep in 16-byte pieces, straight from the feature
//    map (zero filled outside it) and the weights.  With 4-byte pieces (weights turned to [channel][K],
//    so that packed FMAs could take pairs of K) the copies cost as many shared-memory cycles as the
//    reads: 30 instead of 38 TFLOP/s with the chip full and the best tile;
//  * TN follows the output channels (16 to 64 per tile), so that 24 or 40 of them do not run as 32 or 64;
//  * K is split over a cluster of up to eight CTAs where the tiles alone would leave SMs idle (one
//    image of a deep layer): the partial tiles meet in distributed shared memory and are added in rank
//    order, so the result does not depend on timing.
//
// Before, with four outputs per thread and both operands from L1: 32 -> 32, 5x5, 32 images of 28 x 28
// 162 us, here 46 (28 TFLOP/s; 33 on 256 images with the plan below, 38 with the best one); 160 -> 160, 3x3, one
// 7 x 7 image 255, here 7.8; 960 -> 160, 1x1, the same image 175, here 5.8.
#include <cooperative_groups.h>

#include "tc_ptx.cuh"

namespace {
namespace cg = cooperative_groups;

constexpr int kF32Threads = 128;
constexpr int kBK = 16;                          // K per slice
constexpr int kMaxSplit = 8;

struct F32Params {
  int h, w, ho, wo, c_in, c_out, k, stride, pad, act;
  int pixels;                                    // n * ho * wo
  int kdim, slices, slices_per;                  // K, slices of 16 K, slices of one CTA of the cluster
  int m_tiles, n_tiles, split;
};

template <int VW>
__device__ __forceinline__ void load_run(float *d, const float *s) {
  if (VW == 4) {
    const float4 v = *reinterpret_cast<const float4 *>(s);
    d[0] = v.x; d[1] = v.y; d[2] = v.z; d[3] = v.w;
  } else {
    const float2 v = *reinterpret_cast<const float2 *>(s);
    d[0] = v.x; d[1] = v.y;
  }
}

// CTAs on an SM, by the outputs of a thread (registers)
constexpr int f32_resident(int area) { return area > 48 ? 3 : (area > 20 ? 4 : 5); }

// A warp is 32 / CL pixel lanes x CL channel lanes; pixel i of a thread lies one CTA's worth of pixel lanes
// after pixel i - 1; its channels are runs of VW, CL runs apart.
template <int TM, int TN, int CL>
struct F32Tile {
  static constexpr int PL = kF32Threads / CL;            // pixel lanes of the CTA
  static constexpr int BM = PL * TM, BN = CL * TN;
  static constexpr int A_FLOATS = BM * kBK, STAGE = A_FLOATS + kBK * BN;   // a stage: [BM pixels][16 K], [16 K][BN channels]
  static constexpr int VW = TN % 4 == 0 ? 4 : 2;         // channels per shared-memory read: a thread owns TN / VW runs of VW
  // a slice comes back from L2 after 700 cycles or more: small tiles, which multiply one in 300, keep more in flight
  static constexpr int STAGES = STAGE <= 2048 ? 6 : (STAGE <= 3072 ? 4 : 3);
  static constexpr int SMEM = BM * 16 + STAGES * STAGE * 4;
  static_assert(STAGES * STAGE >= BM * BN, "the partial tile reuses the stages");
  static_assert(BN % 8 == 0 && BM % 32 == 0 && TN % 2 == 0, "staging");
};

template <int TM, int TN, int CL>
__global__ void __launch_bounds__(kF32Threads, f32_resident(TM * TN))
k_conv_dense_f32(const float *__restrict__ x, const float *__restrict__ w, const float *__restrict__ bias,
                 const float *__restrict__ residual, float *__restrict__ y, const __grid_constant__ F32Params p) {
  using T = F32Tile<TM, TN, CL>;
  constexpr int BM = T::BM, BN = T::BN, A_FLOATS = T::A_FLOATS, STAGE = T::STAGE, STAGES = T::STAGES;
  extern __shared__ __align__(16) uint8_t sm_f32[];
  int4 *pix = reinterpret_cast<int4 *>(sm_f32);          // per pixel: row and column of its tap (0, 0), element offset of that
  float *sm = reinterpret_cast<float *>(sm_f32 + BM * 16);
  const int t = (int)threadIdx.x, lane = t & 31, warp = t >> 5;
  const int rank = p.split > 1 ? (int)blockIdx.x % p.split : 0;
  const int tile = (int)blockIdx.x / p.split;
  const int mt = tile / p.n_tiles, nt = tile - mt * p.n_tiles;
  const int m0 = mt * BM, n0 = nt * BN;
  const int s_begin = rank * p.slices_per;
  const int s_end = s_begin + p.slices_per < p.slices ? s_begin + p.slices_per : p.slices;
  // Programmatic dependent launch, but the next kernel is let in only when this CTA's arithmetic is done: let in at
  // once, the next kernel's CTAs take the slots this one leaves open, which spreads them unevenly over the SMs
  asm volatile("griddepcontrol.wait;" ::: "memory");

  for (int i = t; i < BM; i += kF32Threads) {
    const int m = m0 + i;
    int4 e = make_int4(-0x20000000, 0, 0, 0);            // past the last pixel: never inside the image
    if (m < p.pixels) {
      const int q = m / p.wo, X = m - q * p.wo, img = q / p.ho, Y = q - img * p.ho;
      const int iy = Y * p.stride - p.pad, ix = X * p.stride - p.pad;
      const long long off = ((long long)(img * p.h + iy) * p.w + ix) * p.c_in;
      e = make_int4(iy, ix, (int)(unsigned)off, (int)(off >> 32));
    }
    pix[i] = e;
  }
  __syncthreads();
  // ---- staging, in 16-byte pieces: four channels (t & 3) of the pixels (t >> 2) + 32 i, and pieces t + 128 i of the
  // slice's 16 weight rows
  const uint32_t sm0 = tc::smem_u32(sm);
  const uint32_t a_dst = sm0 + (uint32_t)(t * 16);
  constexpr int NB = (kBK * BN / 4 + kF32Threads - 1) / kF32Threads;
  const uint32_t w_dst = sm0 + (uint32_t)((A_FLOATS + t * 4) * 4);
  int w_row0 = s_begin * kBK;
  // this thread's position in K: (tap row u, tap column v, channel c) of its piece in slice s_begin
  int kpos = s_begin * kBK + (t & 3) * 4;
  int u, v, c;
  {
    const int tap = kpos / p.c_in;
    c = kpos - tap * p.c_in;
    u = tap / p.k;
    v = tap - u * p.k;
  }
  auto fetch = [&](int buf) {
    const uint32_t base = (uint32_t)(buf * STAGE * 4);
    const bool k_ok = kpos < p.kdim;
    const long long shift = (long long)(u * p.w + v) * p.c_in + c;
#pragma unroll
    for (int i = 0; i < BM / 32; ++i) {
      const int4 e = pix[(t >> 2) + 32 * i];
      const bool ok = k_ok && (unsigned)(e.x + u) < (unsigned)p.h && (unsigned)(e.y + v) < (unsigned)p.w;
      const long long off = (long long)(((unsigned long long)(unsigned)e.w << 32) | (unsigned)e.z) + shift;
      tc::cp_async16(a_dst + base + (uint32_t)(32 * i * kBK * 4), ok ? x + off : x, ok ? 16u : 0u);
    }
    kpos += kBK;
    c += kBK;
    while (c >= p.c_in) {
      c -= p.c_in;
      if (++v == p.k) { v = 0; ++u; }
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int e = t + kF32Threads * i, r = e / (BN / 4), o = n0 + (e - r * (BN / 4)) * 4, row = w_row0 + r;
      const bool ok = row < p.kdim && o < p.c_out;       // c_out is a multiple of 4: a piece is whole or absent
      if (e < kBK * BN / 4)
        tc::cp_async16(w_dst + base + (uint32_t)(kF32Threads * i * 16), ok ? w + (size_t)row * p.c_out + o : w, ok ? 16u : 0u);
    }
    w_row0 += kBK;
  };

  float acc[TM][TN] = {};

  const int pg = warp * (32 / CL) + lane / CL, ch = lane % CL;
  auto channel = [&](int j) { return ch * T::VW + CL * (j / T::VW) * T::VW + j % T::VW; };   // of the tile's BN
  const int nsl = s_end - s_begin;
#pragma unroll
  for (int s = 0; s < STAGES - 1; ++s) {
    if (s < nsl) fetch(s);
    tc::cp_async_commit();
  }
  int buf = 0, fbuf = STAGES - 1;
#pragma unroll 1
  for (int s = 0; s < nsl; ++s) {
    asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
    __syncthreads();                             // slice s has landed for everyone; slice s - 1 is read by no one any more
    if (s + STAGES - 1 < nsl) fetch(fbuf);
    tc::cp_async_commit();
    const float *as = sm + buf * STAGE + pg * kBK, *bs = sm + buf * STAGE + A_FLOATS + ch * T::VW;
#pragma unroll
    for (int kk = 0; kk < kBK; kk += 4) {
      float b[4][TN];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int j = 0; j < TN; j += T::VW) load_run<T::VW>(&b[q][j], bs + (kk + q) * BN + CL * j);
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const float4 a = *reinterpret_cast<const float4 *>(as + T::PL * i * kBK + kk);
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a.x, b[0][j], acc[i][j]);
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a.y, b[1][j], acc[i][j]);
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a.z, b[2][j], acc[i][j]);
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a.w, b[3][j], acc[i][j]);
      }
    }
    buf = buf + 1 == STAGES ? 0 : buf + 1;
    fbuf = fbuf + 1 == STAGES ? 0 : fbuf + 1;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  auto finish = [&](int m, int o, float s) {
    const size_t at = (size_t)m * p.c_out + o;
    float r = s + (bias ? bias[o] : 0.f);
    if (residual) r += residual[at];
    y[at] = dc_act_apply(r, p.act);
  };
  if (p.split == 1) {
#pragma unroll
    for (int i = 0; i < TM; ++i) {
      const int m = m0 + pg + T::PL * i;
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int o = n0 + channel(j);
        if (m < p.pixels && o < p.c_out) finish(m, o, acc[i][j]);
      }
    }
    return;
  }
  // ---- K split over the cluster: partial tiles [BM][BN] in shared memory, each CTA adds up its share of them
  cg::cluster_group cluster = cg::this_cluster();
  __syncthreads();
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) sm[(pg + T::PL * i) * BN + channel(j)] = acc[i][j];
  cluster.sync();
  for (int e = rank * kF32Threads + t; e < BM * BN; e += p.split * kF32Threads) {
    float s = 0.f;
    for (int r = 0; r < p.split; ++r) s += cluster.map_shared_rank(sm, r)[e];
    const int m = m0 + e / BN, o = n0 + e % BN;
    if (m < p.pixels && o < p.c_out) finish(m, o, s);
  }
  cluster.sync();                                // nobody leaves while its tile may still be read
}

// ------------------------------------------------------------------------------------------ host
struct F32Plan {
  F32Params p;
  int config;
};

template <int TM, int TN, int CL>
cudaError_t launch_f32(const F32Plan &pl, const float *x, const float *w, const float *bias, const float *residual,
                       float *y, cudaStream_t st) {
  using T = F32Tile<TM, TN, CL>;
  static unsigned char attr_done[kDcMaxDevices];
  const cudaError_t e = dc_set_max_smem_once(k_conv_dense_f32<TM, TN, CL>, T::SMEM, attr_done);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((long long)pl.p.m_tiles * pl.p.n_tiles * pl.p.split));
  cfg.blockDim = dim3(kF32Threads);
  cfg.dynamicSmemBytes = T::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)pl.p.split;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pl.p.split > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, k_conv_dense_f32<TM, TN, CL>, x, w, bias, residual, y, pl.p);
}

struct F32Config {
  int tm, tn, bm, bn;
  cudaError_t (*launch)(const F32Plan &, const float *, const float *, const float *, const float *, float *, cudaStream_t);
};
template <int TM, int TN, int CL>
constexpr F32Config f32_config() {
  return {TM, TN, F32Tile<TM, TN, CL>::BM, F32Tile<TM, TN, CL>::BN, launch_f32<TM, TN, CL>};
}
constexpr F32Config kF32Configs[] = {
    f32_config<8, 8, 8>(), f32_config<8, 8, 4>(),  f32_config<8, 6, 8>(), f32_config<8, 6, 4>(), f32_config<8, 4, 4>(),
    f32_config<8, 4, 8>(), f32_config<8, 10, 4>(), f32_config<4, 8, 8>(), f32_config<4, 8, 4>(), f32_config<4, 6, 4>(),
    f32_config<4, 10, 4>(), f32_config<4, 4, 4>(), f32_config<4, 4, 8>(), f32_config<4, 2, 8>(), f32_config<8, 2, 8>(),
};

bool f32_shape(int n, int h, int w, const dc_geom *g, F32Params *p) {
  if (g->groups != 1 || g->c_in % 4 || g->c_out % 4) return false;       // 16-byte pieces of four channels
  const int ho = dc_out_extent(h, g->k, g->stride, g->pad), wo = dc_out_extent(w, g->k, g->stride, g->pad);
  if (ho <= 0 || wo <= 0) return false;
  const long long pixels = (long long)n * ho * wo, kdim = (long long)g->k * g->k * g->c_in;
  if (pixels >= (1ll << 30) || (long long)n * (h + 2ll * g->pad) * (w + 2ll * g->pad) >= (1ll << 30) || kdim >= (1ll << 30))
    return false;
  p->h = h; p->w = w; p->ho = ho; p->wo = wo;
  p->c_in = g->c_in; p->c_out = g->c_out; p->k = g->k; p->stride = g->stride; p->pad = g->pad;
  p->pixels = (int)pixels;
  p->kdim = (int)kdim;
  p->slices = (int)((kdim + kBK - 1) / kBK);
  return true;
}

// the grid of one configuration and split; false when it does not apply
bool f32_grid(F32Plan *pl, int config, int split) {
  const F32Config &c = kF32Configs[config];
  F32Params &p = pl->p;
  if (split > 1 && p.slices < 4 * split) return false;   // at least four slices for each CTA of a cluster
  const long long mt = ((long long)p.pixels + c.bm - 1) / c.bm, nt = (p.c_out + c.bn - 1) / c.bn;
  if (mt * nt * split >= (1ll << 31)) return false;
  pl->config = config;
  p.m_tiles = (int)mt; p.n_tiles = (int)nt;
  p.split = split;
  p.slices_per = (p.slices + split - 1) / split;
  return true;
}

bool make_f32_plan(int n, int h, int w, const dc_geom *g, int n_sm, F32Plan *pl) {
  if (!f32_shape(n, h, w, g, &pl->p)) return false;
  // Least estimated time, in cycles of the SM with the most CTAs.  Per slice an SM needs the FMAs of its CTAs (16 x
  // TM x TN cycles of a CTA at full rate) but never less than a slice's own chain; a round of resident CTAs costs a
  // start-up, a cluster its meeting.  The constants are fitted to 15 layers (one pixel tile to eight rounds of them)
  // timed in every configuration and split.  Timed again on 15 layers: the choice is 10 % above the
  // best on average, 43 % at worst (24 -> 32 3x3 of stride 2, 16 images of 56 x 56).
  int best_config = -1, best_split = 0;
  double best = 0.0;
  for (int cfg = 0; cfg < (int)(sizeof(kF32Configs) / sizeof(kF32Configs[0])); ++cfg)
    for (int split = 1; split <= kMaxSplit; split *= 2) {
      if (!f32_grid(pl, cfg, split)) continue;
      const F32Config &c = kF32Configs[cfg];
      const double on_sm = (double)(((long long)pl->p.m_tiles * pl->p.n_tiles * split + n_sm - 1) / n_sm);
      const int area = c.tm * c.tn, resident = f32_resident(area);
      const double rounds = (double)((long long)(on_sm + resident - 1) / resident);
      const double fma = on_sm * (14.7 * area + 100.0), chain = rounds * (16.0 * area + 1380.0);
      const double cost = pl->p.slices_per * (fma > chain ? fma : chain) + 4000.0 * rounds + on_sm * c.bm * c.bn / 64 +
                          (split > 1 ? 5300.0 + 800.0 * split : 0.0);
      if (best_config < 0 || cost < best) { best = cost; best_config = cfg; best_split = split; }
    }
  return best_config >= 0 && f32_grid(pl, best_config, best_split);
}

bool f32_plan(int n, int h, int w, const dc_geom *g, int n_sm, F32Plan *p) {
  static thread_local DcPlans<F32Plan> plans;
  return plans.get(DC_PLAN_KEY(n, h, w, g, n_sm), p, [&](F32Plan *q) { return make_f32_plan(n, h, w, g, n_sm, q); });
}

}  // namespace

// Estimated time, fitted to 300 layers as this plan runs them (13 % off; the plan's own cost ranks tiles and splits of one layer and is up
// to three times off from one layer to another).  0: outside the kernel's range.
double dc_conv_f32_estimate_us(int n, int h, int w, const dc_geom *g) {
  F32Plan pl;
  const int n_sm = dc_sm_count();
  if (!f32_plan(n, h, w, g, n_sm, &pl)) return 0.0;
  const F32Config &c = kF32Configs[pl.config];
  const int area = c.tm * c.tn, resident = f32_resident(area);
  const double on_sm = (double)(((long long)pl.p.m_tiles * pl.p.n_tiles * pl.p.split + n_sm - 1) / n_sm);
  const double rounds = (double)((long long)(on_sm + resident - 1) / resident);
  const double fma = on_sm * (28.6 * area + 180.0), chain = rounds * (16.4 * area + 560.0);
  return (4000.0 + pl.p.slices_per * (fma > chain ? fma : chain) + on_sm * c.bm * (0.33 * c.bn + 3.5) + (pl.p.split > 1 ? 3500.0 : 0.0)) / 1900.0;
}

bool dc_conv_f32_supported(int n, int h, int w, const dc_geom *g) {
  F32Plan pl;
  return f32_plan(n, h, w, g, dc_sm_count(), &pl);
}

dc_status dc_launch_conv_f32(const void *x, int n, int h, int w, const dc_geom *g, const void *w_packed,
                             const float *bias, dc_act act, const void *residual, void *y, cudaStream_t stream) {
  F32Plan pl;
  if (!f32_plan(n, h, w, g, dc_sm_count(), &pl)) return DC_ERR_UNSUPPORTED;
  pl.p.act = (int)act;
  const cudaError_t e = kF32Configs[pl.config].launch(pl, (const float *)x, (const float *)w_packed, bias,
                                                      (const float *)residual, (float *)y, stream);
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? DC_OK : DC_ERR_CUDA;
}
