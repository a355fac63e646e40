// Depthwise convolution (bf16, k = 3 or 5, stride 1 or 2) as a shared-memory stencil on CUDA cores.
//
// A CTA owns a tile of output rows x the whole output width x a group of channels (x several
// images for small maps).  One 4-D TMA load brings the haloed input patch of the tile into shared
// memory as [image][row][column][channel]; the TMA unit writes zeros for everything outside the image,
// so the stencil itself has no border cases.  Threads then compute from shared memory: a thread owns
// 4 channels of TX neighbouring outputs of R rows (two where the tiles give every thread enough, one otherwise), so that an
// input is read and unpacked once for all the outputs it feeds -- 9 instructions per output value of a 3x3 layer with 7 x
// 2 outputs, 13 with the 8 channels x 7 x 1 of before -- with fp32 weights and fp32 accumulation, and writes 8-byte pieces
// (neighbouring threads write neighbouring pieces of a pixel: whole 32-byte sectors).  Depthwise layers are bound by HBM (1.8-4.5
// FLOP/B):
// the tile is read from HBM once (neighbouring tiles share only their halo rows), and several CTAs
// per SM overlap one tile's load with another's arithmetic and stores.  No tensor cores.
//
// Channels come in tiles of 32, 16 or 8, the last one of a pixel partly filled where that is cheaper than narrow tiles (with 8
// channels a line the load unit moves half as many bytes).  All three are compile-time: every shared-memory offset of the
// stencil is an immediate.  Inputs from HBM, against the 8 channels x 7 x 1: 144 channels, 64 images of 56 x 56 28.8 -> 25.6 us, of
// stride 2 23.1 -> 16.3, one image 4.9 -> 3.0; 40 channels, 32 images 14.3 -> 6.8; 96 channels of stride 2, 20 images of 100 x 100
// 14.6 -> 12.0; 240 channels 5x5, 64 images of 28 x 28 27.6 -> 24.6.
//
// The one wait (for the tile to land) is bounded like every wait of the library; a wait that runs
// out sets a library-wide flag that dc_async_status reports, and the CTA returns.
#include "tc_ptx.cuh"

namespace {
using namespace tc;

constexpr int kThreads = 128;
constexpr int kV = 4;                            // channels per thread (8 bytes of bf16)
constexpr int kTileBytes = 48 * 1024;            // patch size limit: four CTAs per SM, so that three loads are in flight
                                                 // while one tile is computed (measured: 256 threads x 2 CTAs x 64 KB
                                                 // took 76 / 100 us on the 112 x 112 layers of cfg4, this 68 / 81 us)

struct StencilParams {
  int n_img, h, w, c, ho, wo, pad, act;
  int ct, cgroups;             // channels per tile, tiles per pixel's channels
  int rows;                    // output rows per thread
  int rt, ytiles;              // output rows per tile, tiles per image column
  int ni, igroups;             // images per tile, tiles over the batch
  int in_rows, in_w;           // patch rows and columns (with halo)
  int box_bytes, patch_bytes;  // bytes the TMA load delivers; the same rounded up to 128
};

// Outputs of one row that a thread computes together (the kernel's register tile and the patch width depend on
// it).  Stride 1: an ODD count.  The two items of a half warp (8 lanes = the 64 bytes of a 32-channel pixel
// each) then read pixels of different parity, i.e. the two halves of the 128 bytes that the 32 banks span; with
// 8 outputs per item all items of a warp read from the same 16 banks and every load took two
// wavefronts (112 x 112 x 32: 49 us with 8, 42 us with 7; 5x5 at 28 x 28 x 240: 96 us with 4, 48 us with 5).
// Stride 2 moves an item by an even number of pixels whatever the count.
__host__ __device__ constexpr int outputs_per_item(int k, int stride) {
  return stride == 1 ? (k == 3 ? 7 : 5) : 4;
}

__device__ unsigned int g_dw_status;             // DC_ERR_TIMEOUT once a wait of these kernels ran out

__device__ __forceinline__ uint2 lds_u2(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float4 lds_f4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}

template <int K, int S, int ACT, int CT, int R>
__global__ void __launch_bounds__(kThreads, 4)
k_dwconv_stencil(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ StencilParams p,
                 const float *__restrict__ w, const float *__restrict__ bias, __nv_bfloat16 *__restrict__ y) {
  constexpr int TX = outputs_per_item(K, S);
  constexpr int NJ = (TX - 1) * S + K;           // input columns they read
  constexpr int ct = CT;                         // channels per tile: every shared-memory offset of the stencil is an immediate
  extern __shared__ __align__(128) uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t abort_word;
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  float *w_s = reinterpret_cast<float *>(smem + p.patch_bytes);          // [K*K][ct] weights, then [ct] bias

  // tile of this CTA: (image group, row tile, channel group), channel groups fastest
  int t = (int)blockIdx.x;
  const int cg = t % p.cgroups; t /= p.cgroups;
  const int ty = t % p.ytiles;
  const int ig = t / p.ytiles;
  const int c0 = cg * ct, y0 = ty * p.rt, img0 = ig * p.ni;

  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_word = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  dc_pdl_enter();                                // nothing above touched global memory; everything below may
  if (threadIdx.x == 0) {
    mbar_arrive_expect_tx(&bar, (uint32_t)p.box_bytes);
    // coordinates may be negative or reach past the tensor: those elements arrive as zeros
    tma_load_4d(smem_u32(smem), &map_x, &bar, c0, -p.pad, y0 * S - p.pad, img0);
  }
  for (int i = (int)threadIdx.x; i < (K * K + 1) * ct; i += kThreads) {
    const int tap = i / ct, ch = i - tap * ct;
    const bool on = c0 + ch < p.c;               // the last tile of a pixel may be partly filled
    w_s[i] = !on ? 0.f : (tap < K * K ? w[(size_t)tap * p.c + c0 + ch] : (bias ? bias[c0 + ch] : 0.f));
  }
  __syncthreads();
  if (!mbar_wait(&bar, 0, &abort_word, nullptr, 0xA0000u)) {
    atomicExch(&g_dw_status, (unsigned int)DC_ERR_TIMEOUT);
    return;
  }

  constexpr int cvt = CT / kV;                   // threads per pixel of this tile: divides kThreads
  const int cv = (int)threadIdx.x % cvt;         // this thread's channels, the same for all its items
  const int xtiles = (p.wo + TX - 1) / TX;
  const int rows_valid = p.ho - y0 < p.rt ? p.ho - y0 : p.rt, pairs = (rows_valid + R - 1) / R;
  const int imgs_valid = p.n_img - img0 < p.ni ? p.n_img - img0 : p.ni;
  // shared-memory addresses as 32-bit offsets (the loop below is bound by its instruction stream)
  constexpr uint32_t ct2 = (uint32_t)CT * 2u, ct4 = (uint32_t)CT * 4u;
  const uint32_t w_sa = smem_u32(w_s) + (uint32_t)(cv * kV) * 4u;         // this thread's channels of tap 0
  const uint32_t row_pitch = (uint32_t)p.in_w * ct2, img_pitch = (uint32_t)p.in_rows * row_pitch;   // bytes
  const uint32_t patch_sa = smem_u32(smem) + (uint32_t)(cv * kV) * 2u;
  const size_t c2 = (size_t)p.c * 2;             // bytes from one output pixel to the next
  // items (image, rows, group of TX outputs) of this thread: the first one by division, the following ones by
  // adding the decomposed step with carries (two divisions per item cost more than the rest of its index work)
  constexpr int step = kThreads / cvt;
  const int d_il = step / (pairs * xtiles), d_rem = step - d_il * pairs * xtiles;
  const int d_ry = d_rem / xtiles, d_xt = d_rem - d_ry * xtiles;
  int il, ry, xt;
  {
    const int item = (int)threadIdx.x / cvt;
    il = item / (pairs * xtiles);
    const int rem = item - il * pairs * xtiles;
    ry = rem / xtiles;
    xt = rem - ry * xtiles;
    if (c0 + cv * kV >= p.c) il = imgs_valid;    // channels past the last one
  }
#pragma unroll 1
  while (il < imgs_valid) {
    const int X0 = xt * TX;
    // packed fp32 arithmetic (two multiply-adds per instruction): the layer has 4.5 FLOP per byte
    // moved, which one scalar FMA per instruction would not keep up with
    float2 acc[R][TX][kV / 2];
    {
      const float4 bz = lds_f4(w_sa + (uint32_t)(K * K) * ct4);
#pragma unroll
      for (int q = 0; q < R; ++q)
#pragma unroll
        for (int o = 0; o < TX; ++o) { acc[q][o][0] = make_float2(bz.x, bz.y); acc[q][o][1] = make_float2(bz.z, bz.w); }
    }
    uint32_t prow = patch_sa + (uint32_t)il * img_pitch + (uint32_t)(ry * (R * S)) * row_pitch + (uint32_t)(X0 * S) * ct2;
    float2 wr[K][K][kV / 2];                     // rows of taps, each read when the first input row needs it
#pragma unroll
    for (int r = 0; r < (R - 1) * S + K; ++r, prow += row_pitch) {
      if (r < K) {
#pragma unroll
        for (int sx = 0; sx < K; ++sx) {
          const float4 w0 = lds_f4(w_sa + (uint32_t)(r * K + sx) * ct4);
          wr[r][sx][0] = make_float2(w0.x, w0.y); wr[r][sx][1] = make_float2(w0.z, w0.w);
        }
      }
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const uint2 raw = lds_u2(prow + (uint32_t)j * ct2);
        // bf16 -> fp32: the 16 bits moved to the top of a word
        const float2 x0 = make_float2(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xFFFF0000u));
        const float2 x1 = make_float2(__uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xFFFF0000u));
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const int tr = r - q * S;                // tap row with which this input row feeds output row q
          if (tr < 0 || tr >= K) continue;
#pragma unroll
          for (int o = 0; o < TX; ++o) {
            const int sx = j - o * S;              // tap column with which input j feeds output o
            if (sx >= 0 && sx < K) {
              acc[q][o][0] = __ffma2_rn(x0, wr[tr][sx][0], acc[q][o][0]);
              acc[q][o][1] = __ffma2_rn(x1, wr[tr][sx][1], acc[q][o][1]);
            }
          }
        }
      }
    }
    const int n_out = p.wo - X0;                 // outputs of this item inside the row (the last item may hang over)
    uint8_t *yrow = reinterpret_cast<uint8_t *>(y + (((size_t)(img0 + il) * p.ho + (size_t)(y0 + ry * R)) * p.wo + (size_t)X0) * p.c + c0 + cv * kV);
#pragma unroll
    for (int q = 0; q < R; ++q, yrow += (size_t)p.wo * c2) {
      uint8_t *yp = yrow;
      const bool on = q == 0 || ry * R + q < rows_valid;
#pragma unroll
      for (int o = 0; o < TX; ++o, yp += c2) {
        uint2 ov;
        // ReLU6 (compile-time): the conversion clamps at zero itself, one packed minimum against (6, 6) does
        // the rest -- the same values as clamping before rounding, since 0 and 6 are bf16 values
        ov.x = ACT ? min_bf16x2(pack_bf16x2_relu(acc[q][o][0].x, acc[q][o][0].y), 0x40C040C0u) : pack_bf16x2(acc[q][o][0].x, acc[q][o][0].y);
        ov.y = ACT ? min_bf16x2(pack_bf16x2_relu(acc[q][o][1].x, acc[q][o][1].y), 0x40C040C0u) : pack_bf16x2(acc[q][o][1].x, acc[q][o][1].y);
        if (on && o < n_out) *reinterpret_cast<uint2 *>(yp) = ov;
      }
    }
    xt += d_xt;
    if (xt >= xtiles) { xt -= xtiles; ++ry; }
    ry += d_ry;
    if (ry >= pairs) { ry -= pairs; ++il; }
    il += d_il;
  }
}

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

bool make_stencil_plan(int n, int h, int w, int c, int k, int stride, int pad, StencilParams *p) {
  if ((k != 3 && k != 5) || (stride != 1 && stride != 2) || c % 8) return false;
  const int ho = dc_out_extent(h, k, stride, pad), wo = dc_out_extent(w, k, stride, pad);
  if (ho <= 0 || wo <= 0) return false;
  p->n_img = n; p->h = h; p->w = w; p->c = c; p->ho = ho; p->wo = wo; p->pad = pad;
  // patch columns: up to the last input column of the last thread item of a row (an item is tx outputs wide;
  // what lies past the image is zero-filled by the TMA unit), so that the stencil needs no column clamp
  const int tx = outputs_per_item(k, stride), xtiles = dc_div_up(wo, tx);
  p->in_w = (xtiles * tx - 1) * stride + k;
  // A TMA box is at most 256 elements wide.  Without room for the last item's overhang it reads on into the next row, or
  // behind the patch into the weights, for outputs that are not stored.
  if (p->in_w > 256) p->in_w = (wo - 1) * stride + k;
  if (p->in_w > 256) return false;
  const int n_sm = dc_sm_count(), nj = (tx - 1) * stride + k;
  double best = 0.0;
  p->ct = 0;
  // Channels per tile (the last tile of a pixel may be partly filled), output rows per tile and per thread, images per tile:
  // the least estimated time, which is what the CTAs of the SM with most of them issue and what a CTA's chain takes (rounds of
  // thread items, its patch's way in, of which the load unit moves fewer bytes at a time in narrow tiles, its weights, read 128
  // at a time) as often as one follows the other in the four places of an SM.  Fitted to 303 layers (8 to 960 channels, 3x3 and
  // 5x5, maps of 7 to 112, 1 to 128 images) timed in up to 24 tiles each, 6324 timings, for the choice: 3.4 % above the best on
  // average, 27 % at worst (80 channels of stride 2, 31 maps of 13 x 13).  A product of powers of the two, without the weights and the
  // places, fitted to 26 layers, chose tiles 8.8 % above the best, 64 % at worst: 304 channels 5x5, 35 maps of 7 x 7 5.6 us, now 4.4;
  // 88 channels 5x5 of stride 2, 4 of 21 x 20 3.1, now 2.4; 192 channels, 121 of 9 x 10 5.8, now 5.0.
  auto consider = [&](int r, int ct, int rt, int ni) {
    const int rows = dc_div_up(rt, r) * r, in_rows = (rows - 1) * stride + k;
    const long long bytes = (long long)ni * in_rows * p->in_w * ct * 2;
    if (bytes > kTileBytes || in_rows > 256) return false;
    const int items = ni * dc_div_up(rt, r) * xtiles * (ct / kV);
    const long long ctas = (long long)dc_div_up(c, ct) * dc_div_up(ho, rt) * dc_div_up(n, ni);
    const int instructions = 40 + k * k + ((r - 1) * stride + k) * nj * 5 + (2 * k * k + 7) * tx * r;
    const double item = instructions * (r == 1 ? 1.35 : 1.0) * (stride == 2 ? 2.3 : 1.0);
    const double moved = (double)bytes * (ct == 32 ? 1.0 : (stride == 2 ? (ct == 16 ? 3.1 : 5.0) : (ct == 16 ? 1.6 : 3.2)));
    const double per_sm = (double)ctas / n_sm, most = 0.77 * (double)((ctas + n_sm - 1) / n_sm) + 0.23 * per_sm;
    const double places = 0.46 * (double)((ctas + 4 * n_sm - 1) / (4 * n_sm)) + 0.54 * (per_sm > 4.0 ? per_sm / 4.0 : 1.0);
    const double chain = dc_div_up(items, kThreads) * item + moved / 10.3 + 635.0 * dc_div_up((k * k + 1) * ct, kThreads);
    const double cost = most * (0.5 * dc_div_up(items, 32) * item + 45.0) + places * chain;
    if (p->ct == 0 || cost < best) { best = cost; p->rows = r; p->ct = ct; p->rt = rt; p->ni = ni; }
    return true;
  };
  for (int r = 2; r >= 1; --r)
    for (int ct = 32; ct >= 8; ct /= 2) {
      if (ct > 8 && ct / 2 >= c) continue;
      bool whole = false;
      int last = 0;
      for (int yt = 1; yt <= ho; ++yt) {
        const int rt = dc_div_up(ho, yt);
        if (rt == last) continue;
        last = rt;
        if (consider(r, ct, rt, 1) && yt == 1) whole = true;
        if (rt <= r) break;
      }
      for (int ni = 2; whole && ni <= 8 && ni <= n; ni *= 2) consider(r, ct, ho, ni);   // small maps: several images per tile
    }
  if (p->ct == 0) return false;
  p->cgroups = dc_div_up(c, p->ct);
  p->ytiles = dc_div_up(ho, p->rt);
  p->in_rows = (dc_div_up(p->rt, p->rows) * p->rows - 1) * stride + k;
  p->igroups = dc_div_up(n, p->ni);
  p->box_bytes = p->ni * p->in_rows * p->in_w * p->ct * 2;
  p->patch_bytes = (int)dc_round_up((size_t)p->box_bytes, 128);
  if ((long long)p->igroups * p->ytiles * p->cgroups >= (1ll << 31)) return false;
  return true;
}

bool stencil_plan(int n, int h, int w, int c, int k, int stride, int pad, StencilParams *p) {
  static thread_local DcPlans<StencilParams> plans;
  return plans.get({n, h, w, c, k, stride, pad, dc_plan_device(), 0, 0, 0, 0}, p,
                   [&](StencilParams *q) { return make_stencil_plan(n, h, w, c, k, stride, pad, q); });
}

}  // namespace

bool dc_dwconv_stencil_supported(int n, int h, int w, int c, int k, int stride, int pad) {
  StencilParams p;
  return stencil_plan(n, h, w, c, k, stride, pad, &p);
}

dc_status dc_launch_dwconv_stencil(const void *x, int n, int h, int w, int c, int k, int stride, int pad, const float *wp,
                                   const float *bias, dc_act act, void *y, cudaStream_t st) {
  StencilParams p;
  if (!stencil_plan(n, h, w, c, k, stride, pad, &p)) return DC_ERR_UNSUPPORTED;
  p.act = (int)act;
  EncodeTiledFn encode = get_encode_fn();
  if (!encode) return DC_ERR_CUDA;
  CUtensorMap map_x;
  {
    const cuuint64_t C = (cuuint64_t)c;
    cuuint64_t gdim[4] = {C, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)n};
    cuuint64_t gstr[3] = {2 * C, (cuuint64_t)w * C * 2, (cuuint64_t)h * w * C * 2};
    cuuint32_t box[4] = {(cuuint32_t)p.ct, (cuuint32_t)p.in_w, (cuuint32_t)p.in_rows, (cuuint32_t)p.ni};
    cuuint32_t es[4] = {1, 1, 1, 1};
    CUresult r = encode(&map_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(x), gdim, gstr, box, es,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return DC_ERR_CUDA;
  }
  const int smem = p.patch_bytes + (k * k + 1) * p.ct * 4 + 256;
  const int grid = p.igroups * p.ytiles * p.cgroups;
  __nv_bfloat16 *yp = (__nv_bfloat16 *)y;
#define DC_DW_LAUNCH3(KK, SS, AA, CC, RR)                                                                    \
  do {                                                                                                    \
    static unsigned char attr_done[kDcMaxDevices];                                                        \
    DC_CUDA_OK(dc_set_max_smem_once(k_dwconv_stencil<KK, SS, AA, CC, RR>, kTileBytes + 8 * 1024, attr_done));     \
    if (dc_launch_pdl(k_dwconv_stencil<KK, SS, AA, CC, RR>, dim3(grid), dim3(kThreads), (size_t)smem, st, map_x, p, wp, bias, yp) != cudaSuccess) \
      return DC_ERR_CUDA;                                                                                 \
  } while (0)
#define DC_DW_LAUNCH2(KK, SS, AA, CC)                                                                        \
  do {                                                                                                    \
    if (p.rows == 2) DC_DW_LAUNCH3(KK, SS, AA, CC, 2);                                                    \
    else DC_DW_LAUNCH3(KK, SS, AA, CC, 1);                                                                \
  } while (0)
#define DC_DW_LAUNCH1(KK, SS, AA)                                                                         \
  do {                                                                                                    \
    if (p.ct == 32) DC_DW_LAUNCH2(KK, SS, AA, 32);                                                        \
    else if (p.ct == 16) DC_DW_LAUNCH2(KK, SS, AA, 16);                                                   \
    else DC_DW_LAUNCH2(KK, SS, AA, 8);                                                                    \
  } while (0)
#define DC_DW_LAUNCH(KK, SS)                                                                              \
  do {                                                                                                    \
    if (act == DC_ACT_RELU6) DC_DW_LAUNCH1(KK, SS, 1);                                                    \
    else DC_DW_LAUNCH1(KK, SS, 0);                                                                        \
  } while (0)
  if (k == 3 && stride == 1) DC_DW_LAUNCH(3, 1);
  else if (k == 3) DC_DW_LAUNCH(3, 2);
  else if (stride == 1) DC_DW_LAUNCH(5, 1);
  else DC_DW_LAUNCH(5, 2);
#undef DC_DW_LAUNCH3
#undef DC_DW_LAUNCH2
#undef DC_DW_LAUNCH1
#undef DC_DW_LAUNCH
  return cudaGetLastError() == cudaSuccess ? DC_OK : DC_ERR_CUDA;
}

cudaError_t dc_dwconv_flag(unsigned int **flag) { return cudaGetSymbolAddress((void **)flag, g_dw_status); }
