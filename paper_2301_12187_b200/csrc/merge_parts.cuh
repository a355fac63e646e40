// What the merge kernels of merge.cu and merge_tc.cu share: layers as they are, and the delivery of a merged run.
#pragma once

#include "common.cuh"

struct RawLayer {
  const float *w, *b, *gamma, *beta, *mean, *var;
  float eps;
};
__device__ __forceinline__ float raw_scale(const RawLayer &L, int o) {
  return L.gamma ? L.gamma[o] / sqrtf(L.var[o] + L.eps) : 1.f;
}
__device__ __forceinline__ float raw_bias(const RawLayer &L, int o, float g) {
  const float b = L.b ? L.b[o] : 0.f;
  return L.gamma ? fmaf(b - L.mean[o], g, L.beta[o]) : b;
}

static __device__ __noinline__ float bn_scale(float gamma, float var) { return gamma / sqrtf(var); }
// BN and bias of a channel as they are read: asked for at once, used later
struct RawNumbers {
  float gamma, var, mean, beta, b;
  __device__ __forceinline__ RawNumbers(const RawLayer &l, int c) {
    gamma = 1.f; var = mean = beta = b = 0.f;
    if (l.gamma) { gamma = l.gamma[c]; var = l.var[c]; mean = l.mean[c]; beta = l.beta[c]; }
    if (l.b) b = l.b[c];
  }
  __device__ __forceinline__ float scale(const RawLayer &l) const { return l.gamma ? bn_scale(gamma, var + l.eps) : 1.f; }
  __device__ __forceinline__ float bias(const RawLayer &l, float g) const { return l.gamma ? fmaf(b - mean, g, beta) : b; }
};

struct BlockDelivery {           // of a run that is one block; mode < 0: the block is a piece of a longer run
  void *packed;
  int mode;                      // 0: no packed copy, 1: fp32, 2: bf16 chunks
  int ident;
  KOrder ko;
};

__device__ __forceinline__ void mb_cp16(float *dst, const float *src, bool ok) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst), n = ok ? 16u : 0u;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n));
}

// true when chunk `idx8` of the packed bf16 copy holds weights (c_in is a multiple of 8: all of them or none)
__device__ __forceinline__ bool packed_chunk_live(const KOrder &ko, int idx8, int c_out) {
  int plane, o, pc, ccg, r, s;
  dc_packed_unchunk(ko, idx8, &plane, &o);
  const int grp = plane / ko.e_pad, e = plane - grp * ko.e_pad;
  if (!dc_korder_decode(ko, e, &pc, &ccg, &r, &s)) return false;
  if (ko.fold) {
    s = o / ko.co8;
    return s < ko.k && o - s * ko.co8 < c_out;
  }
  if (ko.pair >= 2) {
    int px = 0;
    if (ko.pair == 2) { px = o / ko.co8; o -= px * ko.co8; }
    s = 2 * s + (ccg >= ko.cch ? 1 : 0) - (ko.pair == 2 ? px : (ko.pad & 1));
    return px < 2 && o < c_out && s >= 0 && s < ko.k;
  }
  return o < c_out && (grp * ko.cg + ccg) * 8 < ko.c_in;
}

// Tap t of KK of 8 input channels i .. i + 7 of output channel o, which lie STRIDE floats apart, in the packed copy.  fp32: [tap][i][o].  bf16: one
// chunk, written where the forward kernels' K order wants it; pair rows hold every chunk twice, the second copy one pixel
// further on.
template <int KK, int STRIDE = KK>
__device__ __forceinline__ void deliver_chunk(const BlockDelivery &dv, const float *f, int o, int i, int t, int c0, int c2) {
  constexpr int K = KK == 1 ? 1 : KK == 9 ? 3 : 5;
  if (dv.mode == 1) {
    float *out = reinterpret_cast<float *>(dv.packed);
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (i + q < c0) out[((size_t)t * c0 + i + q) * c2 + o] = f[q * STRIDE];
    return;
  }
  uint4 *out = reinterpret_cast<uint4 *>(dv.packed);
  __align__(16) __nv_bfloat16 v8[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) v8[q] = __float2bfloat16_rn(f[q * STRIDE]);
  const uint4 v = *reinterpret_cast<const uint4 *>(v8);
  const int r = t / K, sx = t - K * r;
  out[dc_packed_chunk(dv.ko, dc_korder_encode(dv.ko, i >> 3, r, sx), dc_korder_row(dv.ko, sx, o))] = v;
  if (dv.ko.pair == 2) {
    const int plane = (r * dv.ko.ns[0] + ((sx + 1) >> 1)) * 2 * dv.ko.cch + ((sx + 1) & 1) * dv.ko.cch + (i >> 3);
    out[dc_packed_chunk(dv.ko, plane, dv.ko.co8 + o)] = v;
  }
}

// The packed copy of a tile of OT output x IT input channels whose K x K kernels lie in shared memory as [o][i][tap].
template <int OT, int IT, int K>
__device__ __forceinline__ void deliver_tile(const BlockDelivery &dv, const float *sums, int o0, int i0, int c0, int c2,
                                             int tid, int threads) {
  constexpr int KK = K * K;
  if (dv.mode == 1) {
    float *out = reinterpret_cast<float *>(dv.packed);
    for (int e = tid; e < OT * IT * KK; e += threads) {
      const int ow = e % OT, rest = e / OT, iw = rest % IT, t = rest / IT;
      if (o0 + ow < c2 && i0 + iw < c0) out[((size_t)t * c0 + i0 + iw) * c2 + o0 + ow] = sums[(ow * IT + iw) * KK + t];
    }
    return;
  }
  for (int e = tid; e < OT * (IT / 8) * KK; e += threads) {
    const int ow = e % OT, rest = e / OT, hf = rest % (IT / 8), t = rest / (IT / 8), o = o0 + ow, ch = i0 + hf * 8;
    if (o >= c2 || ch >= c0) continue;
    deliver_chunk<KK>(dv, sums + (ow * IT + hf * 8) * KK + t, o, ch, t, c0, c2);
  }
}

// zeroes the chunks of the packed bf16 copy that hold no weight; thread `thread` of `threads`, CTA `cta` of `ctas`
__device__ __forceinline__ void zero_dead_chunks_by(const BlockDelivery &dv, int c_out, int thread, int threads) {
  const int total8 = dv.ko.ng * dv.ko.e_pad * dv.ko.n_pad;
  for (int e = thread; e < total8; e += threads)
    if (!packed_chunk_live(dv.ko, e, c_out)) reinterpret_cast<uint4 *>(dv.packed)[e] = make_uint4(0u, 0u, 0u, 0u);
}
__device__ __forceinline__ void zero_dead_chunks(const BlockDelivery &dv, int c_out, int cta, int ctas) {
  zero_dead_chunks_by(dv, c_out, cta * (int)blockDim.x + (int)threadIdx.x, ctas * (int)blockDim.x);
}

struct Operand33 {
  RawLayer l;                    // weights, bias, BN (none for a piece)
  int ident;                     // the identity kernel is added
};
struct Compose33 {
  Operand33 first, second;
  int c0, c1, c2;
  float *w_out, *b_out;
  int gi, go;                    // tiles
};

// Bias of output channel o, by one warp: b2~[o] + sum_c (g2 sum of W2[o][c] (+ 1 where c == o and an identity rides)) b1~[c]
__device__ __forceinline__ void compose33_bias(const Compose33 &a, int o, int lane) {
  const RawLayer &l1 = a.first.l, &l2 = a.second.l;
  const int c1 = a.c1;
  const float g2 = raw_scale(l2, o);
  float s = 0.f;
#pragma unroll 2
  for (int c = lane; c < c1; c += 32) {
    const float b1 = raw_bias(l1, c, raw_scale(l1, c));
    float ws = (a.second.ident && c == o) ? 1.f : 0.f;
    float wt = 0.f;
#pragma unroll
    for (int t = 0; t < 9; ++t) wt += l2.w[((size_t)o * c1 + c) * 9 + t];
    s = fmaf(fmaf(g2, wt, ws), b1, s);
  }
  for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
  if (lane == 0) a.b_out[o] = raw_bias(l2, o, g2) + s;
}

// Tap t of the scaled sums of (o, i): the identities are added (`whole`: the run's)
__device__ __forceinline__ float compose33_ident(const Compose33 &a, bool whole, float g2, float s, int o, int i, int t) {
  const RawLayer &l1 = a.first.l, &l2 = a.second.l;
  const int u = t / 5 - 1, v = t - (t / 5) * 5 - 1;                  // tap of the 3x3 kernel centred in the 5x5 one
  if (u >= 0 && u < 3 && v >= 0 && v < 3) {
    if (a.first.ident) s = fmaf(g2, l2.w[((size_t)o * a.c1 + i) * 9 + u * 3 + v], s);                 // W2 o I
    if (a.second.ident) s = fmaf(raw_scale(l1, o), l1.w[((size_t)o * a.c0 + i) * 9 + u * 3 + v], s);  // I o W1
  }
  if (t == 12 && o == i) s += (a.first.ident && a.second.ident ? 1.f : 0.f) + (whole ? 1.f : 0.f);
  return s;
}

// The same composition on the tensor core (merge_tc.cu); DC_ERR_UNSUPPORTED: outside its range, nothing was launched.  A wait that runs
// out is latched in `ws` where there is one, else in the device's flag of these kernels.
dc_status dc_launch_compose33_tc(const Compose33 &a, const BlockDelivery &dv, DcWsHeader *ws, cudaStream_t st);

// What a dense 1x1 layer l1 is composed with, as one product on the tensor core (merge_product_tc.cu): the rest of an inverted-residual
// block (mid: the 3x3 depthwise layer, l2: the last one), or a 1x1 layer l2.  c0 and c1 are multiples of 4.
enum { kProductBlock, kProductPair };
struct Product {
  RawLayer l1, mid, l2;
  int ident1, ident2;            // identity kernels riding on l1 and l2 (not of a block)
  int c0, c1, c2;
  float *w_out, *b_out;
};
// DC_ERR_UNSUPPORTED: outside its range, nothing was launched.  `run`: see make_plan there; `ws` as above
dc_status dc_launch_merge_product_tc(int kind, const Product &a, const BlockDelivery &dv, int run, DcWsHeader *ws, cudaStream_t st);
// its estimated time; 0: outside its range
double dc_merge_product_tc_us(int kind, int c0, int c1, int c2, int run);
