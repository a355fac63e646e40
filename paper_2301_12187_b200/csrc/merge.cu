// BN folding, composition of a run of convolutions into one convolution, and weight repacking.
// fp32 arithmetic (the merged weights must match an fp64 evaluation of the same formula to 1e-5 relative): FMAs on CUDA cores here; large 3x3
// pairs (merge_tc.cu), blocks and 1x1 pairs (merge_product_tc.cu) as products on the tensor core, operands in exact bf16 terms.
#include <vector>

#include "merge_parts.cuh"

// ----------------------------------------------------------------------------------------------
// kernels
// ----------------------------------------------------------------------------------------------

#define DC_FOLD_MAX 16
struct FoldTable {
  const float *w[DC_FOLD_MAX], *b[DC_FOLD_MAX], *gamma[DC_FOLD_MAX], *beta[DC_FOLD_MAX],
      *mean[DC_FOLD_MAX], *var[DC_FOLD_MAX];
  float *w_out[DC_FOLD_MAX], *b_out[DC_FOLD_MAX];
  float eps[DC_FOLD_MAX];
  int c_out[DC_FOLD_MAX], per_out[DC_FOLD_MAX];
  int n;
};

// blockIdx.y = layer; grid-stride over that layer's weights.  g = gamma / sqrt(var + eps).
__global__ void k_fold_bn(const __grid_constant__ FoldTable t) {
  const int l = blockIdx.y;
  const int per = t.per_out[l];
  const int total = t.c_out[l] * per;
  const bool has_bn = t.gamma[l] != nullptr;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int o = i / per;
    float g = 1.f;
    if (has_bn) g = t.gamma[l][o] / sqrtf(t.var[l][o] + t.eps[l]);
    t.w_out[l][i] = g * t.w[l][i];
    if (i - o * per == 0) {
      float b = t.b[l] ? t.b[l][o] : 0.f;
      t.b_out[l][o] = has_bn ? fmaf(b - t.mean[l][o], g, t.beta[l][o]) : b;
    }
  }
}

// One piece of a run while it is being merged: a dense kernel [c_out][c_in][k][k] or a diagonal
// (depthwise) one [c][k][k], with its bias and accumulated stride.
struct Piece {
  const float *w;
  const float *b;
  int c_in, c_out, k, stride, diag;
  int ident;   // 1: the piece stands for w + I (identity kernel of a skip addition: +1 on the centre
               // tap of every (c, c) pair), added where the weights are read instead of by a launch
};

__device__ __forceinline__ float piece_dense_at(const Piece &p, int o, int i, int u, int v) {
  float w = p.w[(((size_t)o * p.c_in + i) * p.k + u) * p.k + v];
  const int ctr = (p.k - 1) / 2;
  if (p.ident && o == i && u == ctr && v == ctr) w += 1.f;
  return w;
}
__device__ __forceinline__ float piece_diag_at(const Piece &p, int c, int u, int v) {
  float w = p.w[((size_t)c * p.k + u) * p.k + v];
  const int ctr = (p.k - 1) / 2;
  if (p.ident && u == ctr && v == ctr) w += 1.f;
  return w;
}

// b'[o] = b2[o] + sum_c (sum_taps W2[o,c]) * b1[c]; one warp per output channel.  Runs in the
// tail blocks of the composition kernels (block index `blk` counted from the first bias block).
__device__ __forceinline__ void compose_bias_block(const Piece &first, const Piece &second, float *out, int blk) {
  const int warp = (blk * (int)blockDim.x + (int)threadIdx.x) / 32, lane = threadIdx.x % 32;
  if (warp >= second.c_out) return;
  const int o = warp, t2 = second.k * second.k;
  float acc = 0.f;
  if (second.diag) {
    if (lane == 0) {
      float ws = second.ident ? 1.f : 0.f;
      for (int t = 0; t < t2; ++t) ws += second.w[(size_t)o * t2 + t];
      acc = ws * first.b[o];
    }
  } else {
    for (int c = lane; c < second.c_in; c += 32) {
      float ws = (second.ident && c == o) ? 1.f : 0.f;
      for (int t = 0; t < t2; ++t) ws += second.w[((size_t)o * second.c_in + c) * t2 + t];
      acc = fmaf(ws, first.b[c], acc);
    }
  }
  for (int d = 16; d > 0; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
  if (lane == 0) out[o] = second.b[o] + acc;
}
static int bias_blocks(int c_out, int threads) { return dc_div_up(c_out * 32, threads); }

// dense (second) o dense (first) for large results:  out[o][j] = sum_r A[o][r] * B[r][j] with
//   r = (c, u2, v2),  j = (i, u', v'),  A = W2 as stored,
//   B[r][j] = W1[c][i][u' - s1*u2][v' - s1*v2]  (0 when the tap falls outside W1):
// a gathered-operand SGEMM with register-staged double buffering.  Tile (16 * TM) x 64 outputs, 256 threads, TM x 4 outputs per thread, reduction slices of
// 16 rows: while a slice is multiplied from shared memory the next one's operands are already on
// their way into registers, so the loads' round trips to L2 hide behind the arithmetic instead of
// alternating with it.  Same reduction order (c, u2, v2) as the other composition kernels.
constexpr int kDtK = 16;                         // reduction rows per slice
template <int TM>
__global__ void __launch_bounds__(256) k_compose_dd_tiled(Piece first, Piece second, float *out, float *b_out,
                                                          int kk, int gx, int gy) {
  constexpr int BM = 16 * TM, PA = BM + 4, PB = 64 + 4;
  __shared__ __align__(16) float As[2][kDtK][PA];
  __shared__ __align__(16) float Bs[2][kDtK][PB];
  if ((int)blockIdx.x >= gx * gy) {
    compose_bias_block(first, second, b_out, (int)blockIdx.x - gx * gy);
    return;
  }
  const int ctr1 = (first.k - 1) / 2, ctr2 = (second.k - 1) / 2;
  const int k1 = first.k, k2 = second.k, s1 = first.stride, t2sz = k2 * k2;
  const int c0 = first.c_in, c1 = first.c_out, c2 = second.c_out;
  const int R = c1 * t2sz, J = c0 * kk * kk;
  const int o0 = ((int)blockIdx.x / gx) * BM, j0 = ((int)blockIdx.x % gx) * 64;
  const int t = threadIdx.x, ty = t >> 4, tx = t & 15;
  // loads: A element (o = o0 + (t >> 4) + 16 q, r = t & 15), B element (r = (t >> 6) + 4 u, j = j0 + (t & 63))
  const int ar = t & 15, ao = t >> 4;
  const int jj = t & 63, j = j0 + jj, br = t >> 6;
  const int bi = j / (kk * kk), btp = j - bi * kk * kk, bup = btp / kk, bvp = btp - bup * kk;
  // fetch() only issues the loads (from a safe address where the element is structurally zero) and keeps what
  // decides the element's value as two bit masks; the values are first touched in stage(), behind the
  // arithmetic on the current slice, so the loads' round trips hide behind it.  (With the selects in fetch()
  // every warp waited for its loads before it started on the slice.)
  float av[TM], bv[4];
  uint32_t a_ok, a_id, b_ok, b_id;
  auto fetch = [&](int r0) {
    const int ra = r0 + ar;
    a_ok = a_id = b_ok = b_id = 0u;
#pragma unroll
    for (int q = 0; q < TM; ++q) {
      const int o = o0 + ao + 16 * q;
      const bool ok = o < c2 && ra < R;
      av[q] = second.w[ok ? (size_t)o * R + ra : 0];
      a_ok |= (ok ? 1u : 0u) << q;
      a_id |= ((ok && second.ident && ra == (o * k2 + ctr2) * k2 + ctr2) ? 1u : 0u) << q;
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = r0 + br + 4 * u;
      int c = r, u2 = 0, v2 = 0;
      if (t2sz != 1) {
        c = r / t2sz;
        const int t2 = r - c * t2sz;
        u2 = t2 / k2;
        v2 = t2 - u2 * k2;
      }
      const int u1 = bup - s1 * u2, v1 = bvp - s1 * v2;
      const bool ok = r < R && j < J && u1 >= 0 && u1 < k1 && v1 >= 0 && v1 < k1;
      bv[u] = first.w[ok ? (((size_t)c * c0 + bi) * k1 + u1) * k1 + v1 : 0];
      b_ok |= (ok ? 1u : 0u) << u;
      b_id |= ((ok && first.ident && c == bi && u1 == ctr1 && v1 == ctr1) ? 1u : 0u) << u;
    }
  };
  auto stage = [&](int buf) {
#pragma unroll
    for (int q = 0; q < TM; ++q)
      As[buf][ar][ao + 16 * q] = ((a_ok >> q) & 1u) ? (((a_id >> q) & 1u) ? av[q] + 1.f : av[q]) : 0.f;
#pragma unroll
    for (int u = 0; u < 4; ++u)
      Bs[buf][br + 4 * u][jj] = ((b_ok >> u) & 1u) ? (((b_id >> u) & 1u) ? bv[u] + 1.f : bv[u]) : 0.f;
  };
  float acc[TM][4] = {};
  fetch(0);
  stage(0);
  __syncthreads();
  int buf = 0;
  for (int r0 = 0; r0 < R; r0 += kDtK) {
    const bool more = r0 + kDtK < R;
    if (more) fetch(r0 + kDtK);
#pragma unroll
    for (int rr = 0; rr < kDtK; ++rr) {
      float a[TM];
#pragma unroll
      for (int q = 0; q < TM; q += 4) {
        const float4 a4 = *reinterpret_cast<const float4 *>(&As[buf][rr][ty * TM + q]);
        a[q] = a4.x; a[q + 1] = a4.y; a[q + 2] = a4.z; a[q + 3] = a4.w;
      }
      const float4 b4 = *reinterpret_cast<const float4 *>(&Bs[buf][rr][tx * 4]);
      const float b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int p = 0; p < TM; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(a[p], b[q], acc[p][q]);
    }
    if (more) stage(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
#pragma unroll
  for (int p = 0; p < TM; ++p) {
    const int o = o0 + ty * TM + p;
    if (o >= c2) continue;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int jo = j0 + tx * 4 + q;
      if (jo < J) out[(size_t)o * J + jo] = acc[p][q];
    }
  }
}

// dense o dense for small results (the usual case: a merged kernel has a few thousand elements):
// 8 x 32 output tile, one output per thread, so that even a 24 x 216 result spreads over 21 CTAs;
// operands staged in shared memory a slice of up to kDdSmallSlice reduction rows at a time, all of
// a slice's loads in flight together.  Same reduction order (c, u2, v2) as the large-tile kernel.
// Blocks [0, gx*gy) are the tiles (x fastest); the blocks after them compute the bias.
constexpr int kDdSmallSlice = 256;
__global__ void __launch_bounds__(256) k_compose_dd_small(Piece first, Piece second, float *out, float *b_out,
                                                          int kk, int gx, int gy) {
  __shared__ float As[kDdSmallSlice][8];
  __shared__ float Bs[kDdSmallSlice][32];
  __shared__ unsigned char tap_u[64], tap_v[64];     // (u2, v2) of tap t2 of the second kernel
  if ((int)blockIdx.x >= gx * gy) {
    compose_bias_block(first, second, b_out, (int)blockIdx.x - gx * gy);
    return;
  }
  const int ctr1 = (first.k - 1) / 2, ctr2 = (second.k - 1) / 2;
  const int k1 = first.k, k2 = second.k, s1 = first.stride, t2sz = k2 * k2;
  const int c0 = first.c_in, c1 = first.c_out, c2 = second.c_out;
  const int R = c1 * t2sz, J = c0 * kk * kk;
  const int o0 = ((int)blockIdx.x / gx) * 8, j0 = ((int)blockIdx.x % gx) * 32;
  const int t = threadIdx.x, ol = t >> 5, jl = t & 31;
  if (t < t2sz) { tap_u[t] = (unsigned char)(t / k2); tap_v[t] = (unsigned char)(t % k2); }
  __syncthreads();
  const int j = j0 + jl, o = o0 + ol;
  const int bi = j / (kk * kk), btp = j - bi * kk * kk, bup = btp / kk, bvp = btp - bup * kk;
  float acc = 0.f;
  for (int r0 = 0; r0 < R; r0 += kDdSmallSlice) {
    const int rows = R - r0 < kDdSmallSlice ? R - r0 : kDdSmallSlice;
    // Operand loads go out in batches with no branch between them (an element outside the operand
    // reads element 0 and is zeroed afterwards: a load behind a branch waits for the one before it).
    // A[o][r]: a warp reads 32 consecutive r of one output channel
    {
      float av[kDdSmallSlice / 32];
#pragma unroll
      for (int u = 0; u < kDdSmallSlice / 32; ++u) {
        const int rr = jl + 32 * u, r = r0 + (rr < rows ? rr : rows - 1);
        const bool ok = o < c2 && rr < rows;
        const float x = second.w[ok ? (size_t)o * R + r : 0];
        av[u] = ok ? ((second.ident && r == (o * k2 + ctr2) * k2 + ctr2) ? x + 1.f : x) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < kDdSmallSlice / 32; ++u)
        if (jl + 32 * u < rows) As[jl + 32 * u][ol] = av[u];
    }
    // B[r][j]: a warp reads one row r, 32 consecutive j
    for (int rb = ol; rb < rows; rb += 64) {
      float bv[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int rr = rb + 8 * u, r = r0 + (rr < rows ? rr : rows - 1);
        int c = r, t2 = 0;
        if (t2sz != 1) { c = r / t2sz; t2 = r - c * t2sz; }
        const int u1 = bup - s1 * tap_u[t2], v1 = bvp - s1 * tap_v[t2];
        const bool ok = j < J && u1 >= 0 && u1 < k1 && v1 >= 0 && v1 < k1;
        const float x = first.w[ok ? (((size_t)c * c0 + bi) * k1 + u1) * k1 + v1 : 0];
        bv[u] = ok ? ((first.ident && c == bi && u1 == ctr1 && v1 == ctr1) ? x + 1.f : x) : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (rb + 8 * u < rows) Bs[rb + 8 * u][jl] = bv[u];
    }
    __syncthreads();
#pragma unroll 8
    for (int rr = 0; rr < rows; ++rr) acc = fmaf(As[rr][ol], Bs[rr][jl], acc);
    __syncthreads();
  }
  if (o < c2 && j < J) out[(size_t)o * J + j] = acc;
}

// dense k x k (second) after a dense 1x1 with stride 1 (first): every tap sum has one term,
//   out[o][i][t] = sum_c W2[o][c][t] * W1[c][i],
// so the general gather would multiply k*k - 1 zeros per product.  blockIdx.y = o; the CTA stages
// W2[o] ([c1][k*k], at most kAfter1x1MaxFloats) in shared memory, a thread owns one (i, t) and
// walks c.  Blocks with blockIdx.y == c_out compute the bias.
constexpr int kAfter1x1MaxFloats = 11264;
__global__ void __launch_bounds__(256) k_compose_after_1x1(Piece first, Piece second, float *out, float *b_out) {
  __shared__ float Ws[kAfter1x1MaxFloats];
  const int c0 = first.c_in, c1 = first.c_out, c2 = second.c_out, kk = second.k * second.k, J = c0 * kk;
  if ((int)blockIdx.y >= c2) {
    compose_bias_block(first, second, b_out, (int)blockIdx.x);
    return;
  }
  const int o = blockIdx.y, ctr = ((second.k - 1) / 2) * (second.k + 1);
  for (int e = threadIdx.x; e < c1 * kk; e += blockDim.x) {
    float w = second.w[(size_t)o * c1 * kk + e];
    if (second.ident && e == o * kk + ctr) w += 1.f;
    Ws[e] = w;
  }
  __syncthreads();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= J) return;
  const int i = j / kk, t = j - i * kk;
  const float *w1 = first.w + i, *w2 = Ws + t;
  float acc0 = 0.f, acc1 = 0.f, acc2 = 0.f, acc3 = 0.f;
  int c = 0;
  for (; c + 4 <= c1; c += 4) {
    const float b0 = w1[(size_t)(c + 0) * c0], b1 = w1[(size_t)(c + 1) * c0];
    const float b2 = w1[(size_t)(c + 2) * c0], b3 = w1[(size_t)(c + 3) * c0];
    acc0 = fmaf(w2[(c + 0) * kk], b0, acc0);
    acc1 = fmaf(w2[(c + 1) * kk], b1, acc1);
    acc2 = fmaf(w2[(c + 2) * kk], b2, acc2);
    acc3 = fmaf(w2[(c + 3) * kk], b3, acc3);
  }
  for (; c < c1; ++c) acc0 = fmaf(w2[c * kk], w1[(size_t)c * c0], acc0);
  float acc = (acc0 + acc1) + (acc2 + acc3);
  if (first.ident && i < c1) acc += w2[i * kk];      // first + I: the c == i term once more
  out[(size_t)o * J + j] = acc;
}

// Compositions in which at least one operand is diagonal: one thread per output element.
//   second diag, first dense: out[o,i,u',v'] = sum_{u2,v2} W2[o,u2,v2] * W1[o,i,u1,v1]
//   second dense, first diag: out[o,i,u',v'] = sum_{u2,v2} W2[o,i,u2,v2] * W1[i,u1,v1]
//   both diag:                out[c,u',v']   = sum_{u2,v2} W2[c,u2,v2]   * W1[c,u1,v1]
// Blocks [0, nb) walk the elements; the blocks after them compute the bias.
// Depthwise K2 x K2 after a dense 1x1 with stride 1 (expand -> depthwise): the tap sums have one
// term, out[o][i][t] = W2[o][t] * W1[o][i].
template <int K2>
__device__ __forceinline__ void compose_diag_after_1x1(const Piece &first, const Piece &second, float *out, int total,
                                                       int nb) {
  constexpr int KK = K2 * K2, CTR = (K2 / 2) * (K2 + 1);
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += nb * blockDim.x) {
    const int t = idx % KK, rest = idx / KK;
    const int o = rest / first.c_in, i = rest - o * first.c_in;
    float w2 = second.w[(size_t)o * KK + t];
    if (second.ident && t == CTR) w2 += 1.f;
    float w1 = first.w[rest];
    if (first.ident && o == i) w1 += 1.f;
    out[idx] = fmaf(w2, w1, 0.f);
  }
}

__global__ void k_compose_diag(Piece first, Piece second, float *out, float *b_out, int kk, int total, int nb) {
  if ((int)blockIdx.x >= nb) {
    compose_bias_block(first, second, b_out, (int)blockIdx.x - nb);
    return;
  }
  if (second.diag && !first.diag && first.k == 1 && first.stride == 1) {
    if (second.k == 3) { compose_diag_after_1x1<3>(first, second, out, total, nb); return; }
    if (second.k == 5) { compose_diag_after_1x1<5>(first, second, out, total, nb); return; }
  }
  const int k1 = first.k, k2 = second.k, s1 = first.stride;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += nb * blockDim.x) {
    int vp = idx % kk, up = (idx / kk) % kk, rest = idx / (kk * kk);
    int o, i;
    if (first.diag && second.diag) { o = rest; i = rest; }
    else { i = rest % first.c_in; o = rest / first.c_in; }
    float acc = 0.f;
    for (int u2 = 0; u2 < k2; ++u2) {
      int u1 = up - s1 * u2;
      if (u1 < 0 || u1 >= k1) continue;
      for (int v2 = 0; v2 < k2; ++v2) {
        int v1 = vp - s1 * v2;
        if (v1 < 0 || v1 >= k1) continue;
        float w2 = second.diag ? piece_diag_at(second, o, u2, v2) : piece_dense_at(second, o, i, u2, v2);
        float w1 = first.diag ? piece_diag_at(first, i, u1, v1) : piece_dense_at(first, o, i, u1, v1);
        acc = fmaf(w2, w1, acc);
      }
    }
    out[idx] = acc;
  }
}

// ----------------------------------------------------------------------------------------------
// A 3x3 depthwise layer as the last one of a longer run, after a dense 3x3 piece with stride 1: composition and delivery in one launch.
// A CTA owns 8 output x 16 input channels, a thread a pair's 25 results (18 weights, 81 FMAs, in the order of k_compose_diag); they
// meet in shared memory and leave as the result and the packed copy.  Small kernels of a chain: launches and their starts bound it.
// 96 -> 24 -> (144) -> 24 -> 144 -> depthwise: six launches 33.0 us, the last two (a thread per result, found out of its index by divisions, and a
// delivery that read them again) 17 of them; now five, 19.5 us, the same bits.
// ----------------------------------------------------------------------------------------------
constexpr int kDwO = 8, kDwI = 16, kDwThreads = kDwO * kDwI;
__global__ void __launch_bounds__(kDwThreads)
k_compose_dw33(const Piece first, const Piece second, float *w_out, float *b_out, const __grid_constant__ BlockDelivery dv, int gi, int tiles) {
  __shared__ __align__(16) float out[kDwThreads * 25];
  __shared__ size_t row_s[kDwO], plane_s[kDwI / 8 * 25];
  const int tid = (int)threadIdx.x, c0 = first.c_in, c2 = second.c_out;
  dc_pdl_enter();
  if ((int)blockIdx.x >= tiles) {
    zero_dead_chunks(dv, c2, (int)blockIdx.x - tiles, (int)gridDim.x - tiles);
    return;
  }
  const int o0 = (int)blockIdx.x / gi * kDwO, i0 = (int)blockIdx.x % gi * kDwI, o = o0 + tid / kDwI, i = i0 + tid % kDwI;
  if (o < c2 && i < c0) {
    float w1[9], w2[9], r[25] = {};
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      w1[t] = piece_dense_at(first, o, i, t / 3, t % 3);
      w2[t] = piece_diag_at(second, o, t / 3, t % 3);
    }
#pragma unroll
    for (int t2 = 0; t2 < 9; ++t2)
#pragma unroll
      for (int t1 = 0; t1 < 9; ++t1) {
        float &x = r[(t2 / 3 + t1 / 3) * 5 + t2 % 3 + t1 % 3];
        x = fmaf(w2[t2], w1[t1], x);
      }
#pragma unroll
    for (int t = 0; t < 25; ++t) out[tid * 25 + t] = r[t];
    if (i == 0) {                                  // b2~ + (sum of the taps) b1~
      float ws = second.ident ? 1.f : 0.f;
#pragma unroll
      for (int t = 0; t < 9; ++t) ws += second.w[(size_t)o * 9 + t];
      b_out[o] = second.b[o] + __fmul_rn(ws, first.b[o]);
    }
  }
  const bool by_rows = dv.mode == 2 && !dv.ko.fold && !dv.ko.pair;
  const int per = dv.ko.rows && dv.ko.nnt > 1 ? dv.ko.n_tile : dv.ko.n_pad;
  if (by_rows) {                                   // as in k_merge_outer33
    const int e = tid - (kDwThreads - kDwI / 8 * 25);
    if (e >= 0) plane_s[e] = (size_t)dc_korder_encode(dv.ko, (i0 >> 3) + e / 25, e % 25 / 5, e % 5) * per;
    if (tid < kDwO) row_s[tid] = dc_packed_chunk(dv.ko, 0, o0 + tid);
  }
  __syncthreads();
  for (int e = tid; e < kDwThreads * 25 / 4; e += kDwThreads) {
    const int ow = e / (kDwI * 25 / 4), x = (e - ow * (kDwI * 25 / 4)) * 4;
    if (o0 + ow >= c2) continue;
    float *to = w_out + ((size_t)(o0 + ow) * c0 + i0) * 25 + x;
    const float *from = out + ow * (kDwI * 25) + x;
    if (c0 % 4 == 0) {
      if (i0 + x / 25 < c0) *reinterpret_cast<float4 *>(to) = *reinterpret_cast<const float4 *>(from);
    } else {
      for (int j = 0; j < 4; ++j)
        if (i0 + (x + j) / 25 < c0) to[j] = from[j];
    }
  }
  if (dv.mode == 0) return;
  if (!by_rows) {
    deliver_tile<kDwO, kDwI, 5>(dv, out, o0, i0, c0, c2, tid, kDwThreads);
    return;
  }
  auto two = [](float lo, float hi) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&p);
  };
  for (int e = tid; e < kDwO * (kDwI / 8) * 25; e += kDwThreads) {
    const int ow = e % kDwO, rest = e / kDwO, hf = rest % (kDwI / 8), t = rest / (kDwI / 8);
    if (o0 + ow >= c2 || i0 + hf * 8 >= c0) continue;
    const float *f = out + (ow * kDwI + hf * 8) * 25 + t;
    reinterpret_cast<uint4 *>(dv.packed)[row_s[ow] + plane_s[hf * 25 + t]] = make_uint4(two(f[0], f[25]), two(f[50], f[75]), two(f[100], f[125]), two(f[150], f[175]));
  }
}

// fp32 [o][i][u][v] -> fp32 [u][v][i][o]
__global__ void k_pack_f32(const float *w, float *out, int c_out, int c_in, int k) {
  int total = c_out * c_in * k * k;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
    int o = idx % c_out, i = (idx / c_out) % c_in, t = idx / (c_out * c_in);
    out[idx] = w[((size_t)o * c_in + i) * k * k + t];
  }
}

// depthwise fp32 [c][1][k][k] -> fp32 [k][k][c]
__global__ void k_pack_dw(const float *w, float *out, int c, int k) {
  int total = c * k * k;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
    int ch = idx % c, t = idx / c;
    out[idx] = w[(size_t)ch * k * k + t];
  }
}

// fp32 [o][i][u][v] -> bf16 chunk planes [group][entry][n_pad][8] in the K order of KOrder
__global__ void k_pack_bf16(const float *w, __nv_bfloat16 *out, int c_out, KOrder ko) {
  const int total = ko.ng * ko.e_pad * ko.n_pad * 8;
  for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += gridDim.x * blockDim.x) {
    int c8 = idx % 8, o, plane;
    dc_packed_unchunk(ko, idx / 8, &plane, &o);
    int grp = plane / ko.e_pad, e = plane - grp * ko.e_pad;
    int pc, ccg, r, s;
    float v = 0.f;
    if (dc_korder_decode(ko, e, &pc, &ccg, &r, &s)) {
      if (ko.fold) {                       // row = (tap column, output channel)
        s = o / ko.co8;
        o -= s * ko.co8;
        if (s >= ko.k) o = c_out;          // padding rows
      } else if (ko.pair == 2) {           // row = (pixel of the pair, output channel); ccg = chunk of the pair row, s = shift
        const int elem = ccg * 8 + c8, ipx = elem / ko.c_in;
        const int px = o / ko.co8;
        o -= px * ko.co8;
        s = 2 * s + ipx - px;
        ccg = 0;
        c8 = elem - ipx * ko.c_in;         // channel (grp is 0 and cg irrelevant once ccg = 0)
        if (px >= 2 || s < 0 || s >= ko.k) o = c_out;
      } else if (ko.pair == 3) {           // stride 2: row = output channel; tap column = 2 * shift + pixel - (pad & 1)
        const int elem = ccg * 8 + c8, ipx = elem / ko.c_in;
        s = 2 * s + ipx - (ko.pad & 1);
        ccg = 0;
        c8 = elem - ipx * ko.c_in;
        if (s < 0 || s >= ko.k) o = c_out;
      }
      int c = (grp * ko.cg + ccg) * 8 + c8;
      if (o < c_out && c < ko.c_in) v = w[(((size_t)o * ko.c_in + c) * ko.k + r) * ko.k + s];
    }
    out[idx] = __float2bfloat16_rn(v);
  }
}

// Element (o, i, tap t) of the finished run as a dense kernel: a diagonal result is lifted, a
// pending identity is added.
__device__ __forceinline__ float merged_at(const Piece &p, int o, int i, int t) {
  const int kk = p.k * p.k, ctr = ((p.k - 1) / 2) * (p.k + 1);
  float w;
  if (p.diag) w = (o == i) ? p.w[(size_t)o * kk + t] : 0.f;
  else w = p.w[((size_t)o * p.c_in + i) * kk + t];
  if (p.ident && o == i && t == ctr) w += 1.f;
  return w;
}

// The bf16 packed copy with one thread per 16-byte chunk (8 input channels of one operand row),
// for large kernels (a thread walks eight elements, so small ones are faster element by element): the
// entry and row are decoded once per chunk, the eight weights are fetched by eight independent
// loads (an element that is padding reads element 0 and is then zeroed, so that no load sits behind
// a branch) and the chunk is written by one store.
__device__ __forceinline__ void deliver_packed_bf16_chunks(const Piece &acc, __nv_bfloat16 *out, const KOrder &ko,
                                                           int start, int stride) {
  const int c_out = acc.c_out, kk = acc.k * acc.k, ctr = ((acc.k - 1) / 2) * (acc.k + 1);
  const int total8 = ko.ng * ko.e_pad * ko.n_pad;
  for (int idx8 = start; idx8 < total8; idx8 += stride) {
    int plane, o_row;
    dc_packed_unchunk(ko, idx8, &plane, &o_row);
    const int grp = plane / ko.e_pad, e = plane - grp * ko.e_pad;
    int pc, ccg0, r, s0;
    bool live = dc_korder_decode(ko, e, &pc, &ccg0, &r, &s0);
    int o = o_row, px = 0;
    if (live) {
      if (ko.fold) {
        s0 = o / ko.co8;
        o -= s0 * ko.co8;
        if (s0 >= ko.k) live = false;
      } else if (ko.pair == 2) {
        px = o / ko.co8;
        o -= px * ko.co8;
        if (px >= 2) live = false;
      }
    }
    live = live && o < c_out;
    int ch[8], tap[8];
    bool ok[8];
#pragma unroll
    for (int c8 = 0; c8 < 8; ++c8) {
      int sx = s0, c;
      if (ko.pair >= 2) {
        const int elem = ccg0 * 8 + c8, ipx = elem / ko.c_in;
        sx = 2 * s0 + ipx - (ko.pair == 2 ? px : (ko.pad & 1));
        c = grp * ko.cg * 8 + elem - ipx * ko.c_in;
      } else {
        c = (grp * ko.cg + ccg0) * 8 + c8;
      }
      ok[c8] = live && sx >= 0 && sx < ko.k && c >= 0 && c < ko.c_in;
      ch[c8] = c;
      tap[c8] = r * ko.k + sx;
    }
    float w[8];
#pragma unroll
    for (int c8 = 0; c8 < 8; ++c8) {
      size_t off = 0;
      if (ok[c8]) off = acc.diag ? (size_t)o * kk + tap[c8] : ((size_t)o * acc.c_in + ch[c8]) * kk + tap[c8];
      w[c8] = acc.w[off];
    }
    __align__(16) __nv_bfloat16 v8[8];
#pragma unroll
    for (int c8 = 0; c8 < 8; ++c8) {
      float v = w[c8];
      if (acc.diag && o != ch[c8]) v = 0.f;
      if (acc.ident && o == ch[c8] && tap[c8] == ctr) v += 1.f;
      v8[c8] = __float2bfloat16_rn(ok[c8] ? v : 0.f);
    }
    *reinterpret_cast<uint4 *>(out + (size_t)idx8 * 8) = *reinterpret_cast<const uint4 *>(v8);
  }
}

// Last launch of a merge: writes the dense fp32 kernel (blocks [0, nb_w)), the bias (block nb_w)
// and, when asked for, the packed copy for the forward kernels (blocks after that; mode 1: fp32
// [u][v][i][o], mode 2: bf16 chunk planes in the K order of KOrder), all straight from the
// accumulated piece.
__global__ void k_deliver(Piece acc, float *w_merged, float *b_merged, void *packed, int mode, KOrder ko,
                          int nb_w, int nb_p, int chunked) {
  const int c_out = acc.c_out, c_in = acc.c_in, kk = acc.k * acc.k;
  int blk = (int)blockIdx.x;
  if (blk < nb_w) {
    const int total = c_out * c_in * kk;
    for (int idx = blk * blockDim.x + threadIdx.x; idx < total; idx += nb_w * blockDim.x) {
      const int t = idx % kk, i = (idx / kk) % c_in, o = idx / (kk * c_in);
      w_merged[idx] = merged_at(acc, o, i, t);
    }
    return;
  }
  blk -= nb_w;
  if (blk == 0) {
    for (int o = threadIdx.x; o < c_out; o += blockDim.x) b_merged[o] = acc.b[o];
    return;
  }
  blk -= 1;
  if (mode == 1) {
    float *out = reinterpret_cast<float *>(packed);
    const int total = c_out * c_in * kk;
    for (int idx = blk * blockDim.x + threadIdx.x; idx < total; idx += nb_p * blockDim.x) {
      const int o = idx % c_out, i = (idx / c_out) % c_in, t = idx / (c_out * c_in);
      out[idx] = merged_at(acc, o, i, t);
    }
  } else if (mode == 2 && chunked) {
    deliver_packed_bf16_chunks(acc, reinterpret_cast<__nv_bfloat16 *>(packed), ko, blk * blockDim.x + threadIdx.x,
                               nb_p * blockDim.x);
  } else if (mode == 2) {
    __nv_bfloat16 *out = reinterpret_cast<__nv_bfloat16 *>(packed);
    const int total = ko.ng * ko.e_pad * ko.n_pad * 8;
    for (int idx = blk * blockDim.x + threadIdx.x; idx < total; idx += nb_p * blockDim.x) {
      int c8 = idx % 8, o, plane;
      dc_packed_unchunk(ko, idx / 8, &plane, &o);
      int grp = plane / ko.e_pad, e = plane - grp * ko.e_pad;
      int pc, ccg, r, sx;
      float v = 0.f;
      if (dc_korder_decode(ko, e, &pc, &ccg, &r, &sx)) {
        if (ko.fold) {
          sx = o / ko.co8;
          o -= sx * ko.co8;
          if (sx >= ko.k) o = c_out;
        } else if (ko.pair == 2) {
          const int elem = ccg * 8 + c8, ipx = elem / ko.c_in;
          const int px = o / ko.co8;
          o -= px * ko.co8;
          sx = 2 * sx + ipx - px;
          ccg = 0;
          c8 = elem - ipx * ko.c_in;
          if (px >= 2 || sx < 0 || sx >= ko.k) o = c_out;
        } else if (ko.pair == 3) {
          const int elem = ccg * 8 + c8, ipx = elem / ko.c_in;
          sx = 2 * sx + ipx - (ko.pad & 1);
          ccg = 0;
          c8 = elem - ipx * ko.c_in;
          if (sx < 0 || sx >= ko.k) o = c_out;
        }
        const int c = (grp * ko.cg + ccg) * 8 + c8;
        if (o < c_out && c < ko.c_in) v = merged_at(acc, o, c, r * ko.k + sx);
      }
      out[idx] = __float2bfloat16_rn(v);
    }
  }
}

// ----------------------------------------------------------------------------------------------
// An inverted-residual block in one step: dense 1x1 (stride 1) -> depthwise k x k -> dense 1x1.
//
//   W'[o][i][t] = sum_c W3~[o][c] * D~[c][t] * W1~[c][i],   ~ = BN folded (scale g = gamma / sqrt(var + eps))
//   b'[o]       = b3~[o] + sum_c W3~[o][c] * (b2~[c] + (sum_t D~[c][t]) * b1~[c])
//
// which is what folding the three layers and composing them pairwise gives (Eq. 1 applied twice),
// without the folded copies and the 6x wider intermediate kernel ever going through global memory:
// each step of the pairwise walk waits for the one before, and for kernels of a few thousand
// elements those waits are the whole cost.  One CTA per output channel o; the raw layer weights are
// read once per CTA (they sit in L2), `chunk` hidden channels at a time.
// ----------------------------------------------------------------------------------------------
struct BlockArgs {
  RawLayer l1, l2, l3;
  int c0, c1, c2, k;      // input, hidden, output channels; depthwise kernel size
  int chunk;              // hidden channels staged per pass
  float *w_out, *b_out;   // [c2][c0][k][k], [c2]
};
constexpr int kBlockThreads = 256;
constexpr int kBlockMaxPerThread = 8;       // outputs per thread: c0 * k * k <= 2048

// Up to kBlockBatch blocks of one run go out in one launch (blockIdx.y picks the block): they depend
// on the raw layers only, not on one another.
constexpr int kBlockBatch = 4;
struct BlockBatch {
  BlockArgs blk[kBlockBatch];
};

__global__ void __launch_bounds__(kBlockThreads) k_merge_block(const __grid_constant__ BlockBatch batch) {
  extern __shared__ __align__(16) float blk_smem[];
  const BlockArgs &a = batch.blk[blockIdx.y];
  if ((int)blockIdx.x >= a.c2) return;
  const int c0 = a.c0, c1 = a.c1, kk = a.k * a.k, J = c0 * kk, CH = a.chunk;
  float *Ms = blk_smem;                 // [CH][c0]  raw W1 rows
  float *Ds = Ms + CH * c0;             // [CH][kk]  raw D rows, then W3~[o][c] * D~[c][t] * g1[c]
  float *sc = Ds + CH * kk;             // [CH]      W3~[o][c] * g2[c] * g1[c]
  __shared__ float bias_part[kBlockThreads / 32];
  const int o = blockIdx.x, tid = threadIdx.x;
  const float g3 = raw_scale(a.l3, o);
  float acc[kBlockMaxPerThread];
  int oi[kBlockMaxPerThread], ot[kBlockMaxPerThread];
#pragma unroll
  for (int q = 0; q < kBlockMaxPerThread; ++q) {
    const int j = tid + q * kBlockThreads;
    acc[q] = 0.f;
    oi[q] = j / kk;
    ot[q] = j - oi[q] * kk;
  }
  float bsum = 0.f;
  for (int cb = 0; cb < c1; cb += CH) {
    const int rows = c1 - cb < CH ? c1 - cb : CH;
    // all loads of the pass go out together: W1 rows, D rows, and the per-channel scalars
    for (int e = tid; e < rows * c0; e += kBlockThreads) Ms[e] = a.l1.w[(size_t)cb * c0 + e];
    for (int e = tid; e < rows * kk; e += kBlockThreads) Ds[e] = a.l2.w[(size_t)cb * kk + e];
    for (int cl = tid; cl < rows; cl += kBlockThreads) {
      const int c = cb + cl;
      const float g1 = raw_scale(a.l1, c), g2 = raw_scale(a.l2, c);
      const float w3 = g3 * a.l3.w[(size_t)o * c1 + c];
      float dsum = 0.f;
      for (int t = 0; t < kk; ++t) dsum += g2 * a.l2.w[(size_t)c * kk + t];
      bsum = fmaf(w3, fmaf(dsum, raw_bias(a.l1, c, g1), raw_bias(a.l2, c, g2)), bsum);
      sc[cl] = (w3 * g2) * g1;
    }
    __syncthreads();
    for (int e = tid; e < rows * kk; e += kBlockThreads) Ds[e] *= sc[e / kk];
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kBlockMaxPerThread; ++q) {
      if (tid + q * kBlockThreads < J) {
        const float *m = Ms + oi[q], *d = Ds + ot[q];
        float s = acc[q];
#pragma unroll 4
        for (int cl = 0; cl < rows; ++cl) s = fmaf(d[cl * kk], m[cl * c0], s);
        acc[q] = s;
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < kBlockMaxPerThread; ++q) {
    const int j = tid + q * kBlockThreads;
    if (j < J) a.w_out[(size_t)o * J + j] = acc[q];
  }
  // bias: the per-thread terms meet through warp shuffles and one shared-memory hop
  for (int d = 16; d > 0; d >>= 1) bsum += __shfl_xor_sync(0xffffffffu, bsum, d);
  if ((tid & 31) == 0) bias_part[tid >> 5] = bsum;
  __syncthreads();
  if (tid == 0) {
    float b = 0.f;
    for (int w = 0; w < kBlockThreads / 32; ++w) b += bias_part[w];
    a.b_out[o] = raw_bias(a.l3, o, g3) + b;
  }
}

// ----------------------------------------------------------------------------------------------
// The same block step for 3x3 depthwise layers, tiled over (output, input) channels and split over the
// hidden channels inside the CTA, and -- for a run that is one block -- with the delivery in the same
// launch.
//
// For one hidden channel c the 3x3 kernel of a pair (o, i) grows by p = (W3[o][c] s[c]) W1[c][i] times
// the nine taps D[c][.]: one multiplication and nine FMAs per pair, and W', with its 9 x c_hidden terms,
// never exists in between.  A CTA owns 8 x IT pairs, a thread of a warp 2 x IT/8 of them (36 or 54 sums);
// its W warps take an equal part of the hidden channels each, stage their own operands by cp.async four
// slices of 16 channels deep (no CTA barrier until the sums meet in shared memory, in warp order), so
// that narrow blocks are short chains and wide ones fill the chip.  8 x 16 pairs by eight warps; for long
// reductions sixteen warps, in tiles of 8 x 16 or 8 x 24 (see the rule at the launch): 160 -> 960 -> 160 has 140 tiles of
// 8 x 24.  BN scales s = g1 g2 ride on W3, g3 on the result.
//
// Blocks behind the tiles compute the bias (8 output channels each); behind those, for a packed
// result, the chunks of the packed copy that hold no weight are zeroed.
//
// Before, with one CTA per output channel that read every operand, then a delivery launch: 24 -> 144 -> 24 9.4 us, 64 -> 384 -> 64
// 29.5 us; 160 -> 960 -> 160, step by step, 103 us.  With eight warps 6.5, 9.0 and 25.9 us (200 tiles of 8 x 16 on 148 SMs: 52 of
// them had two, the others eight warps with no second tile to hide their latency); by sixteen warps in 140 tiles of 8 x 24 20.7
// us, 120 -> 720 -> 120 (120 tiles) 19.0 -> 12.9, 88 -> 528 -> 88 15.0 -> 11.3.  With the sums added 16 bytes at a time and the
// third layer's scales asked for in front (behind the sums they were a chain of their own) 24 -> 144 -> 24 6.4 -> 6.0, 160 -> 960
// -> 160 19.7.  Halved runs of the sums are nearer to 64 bits as well (160 channels: 1.6e-7 -> 1.35e-7).
// ----------------------------------------------------------------------------------------------
constexpr int kMbO = 8, kMbI = 16, kMbSlice = 16, kMbStages = 4;
constexpr int kMbThreads = 256;
// A form of the kernel: IT input channels of a tile, W warps that share the hidden channels.
template <int IT, int W>
struct MbForm {
  static constexpr int W1 = kMbSlice * IT, W3 = kMbO * kMbSlice, D = kMbSlice * 9;   // floats of a slice's operands
  static constexpr int STAGE = W1 + W3 + D, TILE = kMbO * IT * 9;
  static constexpr int RING = W * kMbStages * STAGE * 4;                             // bytes of the operand rings
  static_assert(RING >= W * TILE * 4, "the warps' sums reuse the rings");
};
constexpr int kMbRing = MbForm<kMbI, 8>::RING;                    // the smallest form's

struct TiledBlocks {
  BlockArgs blk[kBlockBatch];
  int first[kBlockBatch + 1];    // first CTA of each block's tiles and bias groups
  int n;
};
template <int IT, int W>
__global__ void __launch_bounds__(W * 32, W == 8 ? 2 : 1)
k_merge_block33(const __grid_constant__ TiledBlocks tb, const __grid_constant__ BlockDelivery dv) {
  using F = MbForm<IT, W>;
  constexpr int NI = IT / 8;                       // input channels of a thread
  extern __shared__ __align__(16) float mb_smem[];
  const int tid = (int)threadIdx.x, warp = tid >> 5, lane = tid & 31;
  dc_pdl_enter();
  if ((int)blockIdx.x >= tb.first[tb.n]) {
    zero_dead_chunks(dv, tb.blk[0].c2, (int)blockIdx.x - tb.first[tb.n], (int)gridDim.x - tb.first[tb.n]);
    return;
  }
  int bi = 0;
  while ((int)blockIdx.x >= tb.first[bi + 1]) ++bi;
  const BlockArgs &a = tb.blk[bi];
  const int c0 = a.c0, c1 = a.c1, c2 = a.c2;
  const int gi = dc_div_up(c0, IT), go = dc_div_up(c2, kMbO);
  const int blk = (int)blockIdx.x - tb.first[bi];
  if (blk >= gi * go) {
    // ---- bias of 8 output channels: q[c] = b2~ + (sum of D~) b1~, then one dot product per warp
    const int o = (blk - gi * go) * kMbO + warp;
    float *q = mb_smem;                            // the host keeps c1 within the rings
    for (int c = tid; c < c1; c += W * 32) {
      const float g1 = raw_scale(a.l1, c), g2 = raw_scale(a.l2, c);
      float dsum = 0.f;
#pragma unroll
      for (int t = 0; t < 9; ++t) dsum += g2 * a.l2.w[(size_t)c * 9 + t];
      q[c] = fmaf(dsum, raw_bias(a.l1, c, g1), raw_bias(a.l2, c, g2));
    }
    __syncthreads();
    if (warp < kMbO && o < c2) {
      const float g3 = raw_scale(a.l3, o);
      float s = 0.f;
#pragma unroll 4
      for (int c = lane; c < c1; c += 32) s = fmaf(g3 * a.l3.w[(size_t)o * c1 + c], q[c], s);
      for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
      if (lane == 0) a.b_out[o] = raw_bias(a.l3, o, g3) + s;
    }
    return;
  }
  // ---- 8 x IT pairs
  const int o0 = (blk / gi) * kMbO, i0 = (blk % gi) * IT;
  __shared__ float g3s[kMbO];                      // BN scales of the tile's output channels
  if (tid < kMbO) g3s[tid] = o0 + tid < c2 ? raw_scale(a.l3, o0 + tid) : 0.f;
  const int per = ((c1 + W - 1) / W + 3) & ~3;       // hidden channels of a warp
  const int cb = warp * per, ce = cb + per < c1 ? cb + per : c1;
  const int nsl = ce > cb ? (ce - cb + kMbSlice - 1) / kMbSlice : 0;
  float *ring = mb_smem + warp * (kMbStages * F::STAGE);
  auto fetch = [&](int sl, int buf) {
    float *st = ring + buf * F::STAGE;
    const int c = cb + sl * kMbSlice;
    // W1[c..c+15][i0..i0+IT-1]: 64 or 96 pieces; W3[o0..o0+7][c..c+15]: 32; D[c..c+15][9]: 36 (channels and c1 are multiples of 4)
#pragma unroll
    for (int h = 0; h < NI; ++h) {
      const int e = lane + 32 * h, r = e / (IT / 4), ii = i0 + (e % (IT / 4)) * 4;
      const bool ok = c + r < ce && ii < c0;
      mb_cp16(st + e * 4, ok ? a.l1.w + (size_t)(c + r) * c0 + ii : a.l1.w, ok);
    }
    {
      const int o = o0 + (lane >> 2), cc = c + (lane & 3) * 4;
      const bool ok = o < c2 && cc < ce;
      mb_cp16(st + F::W1 + lane * 4, ok ? a.l3.w + (size_t)o * c1 + cc : a.l3.w, ok);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int e = lane + 32 * h;
      const bool ok = e * 4 < (ce - c) * 9;
      if (e < F::D / 4) mb_cp16(st + F::W1 + F::W3 + e * 4, ok ? a.l2.w + (size_t)c * 9 + e * 4 : a.l2.w, ok);
    }
  };
#pragma unroll
  for (int sl = 0; sl < kMbStages - 1; ++sl) {
    if (sl < nsl) fetch(sl, sl);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  const int ol = (lane >> 3) * 2, il = (lane & 7) * NI;            // this thread's pairs: o0 + ol + {0, 1}, i0 + il + {0 .. NI - 1}
  float acc[2][NI][9] = {};
  int buf = 0, fbuf = kMbStages - 1;
  // BN scales of a slice's channels: lane l holds channel l & 15's.  Their operands are asked for a slice ahead and
  // first touched behind the slice's arithmetic.
  float bn[4] = {1.f, 1.f, 1.f, 1.f};
  auto ask = [&](int sl) {
    const int cs = cb + sl * kMbSlice + (lane & 15), c = cs < ce ? cs : cb;
    if (a.l1.gamma) { bn[0] = a.l1.gamma[c]; bn[1] = a.l1.var[c]; }
    if (a.l2.gamma) { bn[2] = a.l2.gamma[c]; bn[3] = a.l2.var[c]; }
  };
  auto scale = [&]() {
    return (a.l1.gamma ? bn[0] / sqrtf(bn[1] + a.l1.eps) : 1.f) * (a.l2.gamma ? bn[2] / sqrtf(bn[3] + a.l2.eps) : 1.f);
  };
  float sc = 1.f;
  if (nsl > 0) { ask(0); sc = scale(); }
#pragma unroll 1
  for (int sl = 0; sl < nsl; ++sl) {
    ask(sl + 1);                                   // past the end: the warp's first channel, not used
    asm volatile("cp.async.wait_group %0;" ::"n"(kMbStages - 2) : "memory");
    __syncwarp();
    if (sl + kMbStages - 1 < nsl) fetch(sl + kMbStages - 1, fbuf);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float *st = ring + buf * F::STAGE;
    auto four = [&](int q) {                       // channels q .. q + 3 of the slice
      float w3[2][4], d[36];
#pragma unroll
      for (int h = 0; h < 2; ++h)
        *reinterpret_cast<float4 *>(w3[h]) = *reinterpret_cast<const float4 *>(st + F::W1 + (ol + h) * kMbSlice + q);
#pragma unroll
      for (int e = 0; e < 9; ++e)
        *reinterpret_cast<float4 *>(d + 4 * e) = *reinterpret_cast<const float4 *>(st + F::W1 + F::W3 + q * 9 + 4 * e);
#pragma unroll
      for (int cl = 0; cl < 4; ++cl) {
        const float s = __shfl_sync(0xffffffffu, sc, q + cl);
        float w1[NI];
        if (NI == 2) *reinterpret_cast<float2 *>(w1) = *reinterpret_cast<const float2 *>(st + (q + cl) * IT + il);
        else
#pragma unroll
          for (int v = 0; v < NI; ++v) w1[v] = st[(q + cl) * IT + il + v];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float ws = w3[h][cl] * s;
          float pr[NI];
#pragma unroll
          for (int v = 0; v < NI; ++v) pr[v] = ws * w1[v];
#pragma unroll
          for (int t = 0; t < 9; ++t)
#pragma unroll
            for (int v = 0; v < NI; ++v) acc[h][v][t] = fmaf(pr[v], d[cl * 9 + t], acc[h][v][t]);
        }
      }
    };
    const int left = ce - (cb + sl * kMbSlice);    // channels of the slice: a multiple of 4
    if (left >= kMbSlice) {
#pragma unroll
      for (int q = 0; q < kMbSlice; q += 4) four(q);
    } else {
#pragma unroll 1
      for (int q = 0; q < left; q += 4) four(q);
    }
    sc = scale();
    __syncwarp();                                  // the slice's buffer may be refilled
    buf = buf + 1 == kMbStages ? 0 : buf + 1;
    fbuf = fbuf + 1 == kMbStages ? 0 : fbuf + 1;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // ---- the warps' sums meet: [warp][o][i][tap]
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int v = 0; v < NI; ++v)
#pragma unroll
      for (int t = 0; t < 9; ++t) mb_smem[warp * F::TILE + ((ol + h) * IT + il + v) * 9 + t] = acc[h][v][t];
  __syncthreads();
  const bool last = dv.mode >= 0;
  // four elements of the warps' sums at a time: rows of IT input channels are whole pieces, and so are 4 channels of them
  for (int e = tid; e < F::TILE / 4; e += W * 32) {
    float4 *p = reinterpret_cast<float4 *>(mb_smem) + e;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const float4 q = p[w * (F::TILE / 4)];
      s.x += q.x; s.y += q.y; s.z += q.z; s.w += q.w;
    }
    const int oi = e / (IT * 9 / 4), x = (e - oi * (IT * 9 / 4)) * 4, o = o0 + oi;
    if (o < c2 && i0 + x / 9 < c0) {
      const float g3 = g3s[oi];
      s.x *= g3; s.y *= g3; s.z *= g3; s.w *= g3;
      if (last && dv.ident) {                      // 1 at tap 4 of channel o
        const int at = (o - i0) * 9 + 4 - x;
        if (at == 0) s.x += 1.f;
        if (at == 1) s.y += 1.f;
        if (at == 2) s.z += 1.f;
        if (at == 3) s.w += 1.f;
      }
      *reinterpret_cast<float4 *>(a.w_out + ((size_t)o * c0 + i0) * 9 + x) = s;
    }
    if (last && dv.mode > 0) *p = s;               // these elements of warp 0's sums are read by this thread alone
  }
  if (!last || dv.mode == 0) return;
  __syncthreads();
  deliver_tile<kMbO, IT, 3>(dv, mb_smem, o0, i0, c0, c2, tid, W * 32);
}

// ----------------------------------------------------------------------------------------------
// dense 3x3 (stride 1) followed by dense 3x3: the result's 5x5 kernel of a pair (o, i) is the sum over the
// intermediate channels c of the full 2-D product of W2[o][c] and W1[c][i], 81 multiply-adds per c and none of
// them with a structural zero (a gathered GEMM multiplies all 9 x 25 tap/position pairs, 64 % of which are).
//
// What bounds it is the FMA pipes, so nothing else may: a CTA owns 8 x 8 pairs, a thread of a warp 2 x 1 of them
// (50 sums, 162 FMAs per c for 27 shared-memory reads, conflict-free because nine floats apart).  The reduction
// is cut into eight parts, one for each of eight warps or two for each of four (see the rule at the launch); a warp
// stages its own operands by cp.async in slices of 4 channels (whole 16-byte pieces: the taps of neighbouring channels
// are contiguous in both operands), three deep, without a CTA barrier until the parts' sums meet in shared memory, in
// the order of the channels.  Small results therefore spread over the chip as well (32 -> 32 -> 32: 16 CTAs, four
// channels a warp).
//
// BN of layers taken as they are: the first's scale rides on its taps, the second's on the sums.  An identity
// riding on a piece adds W2 or W1 itself (and 1) to the sums.  Blocks behind the tiles compute the bias (8 output
// channels each); behind those, for a packed result, the chunks without weights are zeroed.
//
// Tiles of 16 x 32 pairs with CTA barriers per slice, a fold launch before and a delivery after: c = 64 50 us,
// 256 141 us, 512 859 us.  Here 5.9, 76 and 551 us (39 useful fp32 TFLOP/s: two thirds of the issue slots are taken, a
// third of those by what is not an FMA; what holds the rest is the register file, whose banks the compiler cannot
// keep apart for 50 sums).  With eight warps everywhere, sums added element by element, the second layer's scale asked
// for behind them and 64-bit source pointers per copy: 7.6, 86 and 584 us, c = 32 6.4 (now 4.7); a fifth of the
// instructions were those.  Packed FMAs over the two output channels measured 106 us at c = 256, 80 registers and
// three CTAs per SM 98, the taps of two channels by 8-byte reads 1 % (and spills).
// ----------------------------------------------------------------------------------------------
constexpr int kP3O = 8, kP3I = 8, kP3Parts = 8, kP3Slice = 4, kP3Stages = 3;
constexpr int kP3Op = kP3O * kP3Slice * 9;                        // floats of one operand's slice: [o][c][9] or [c][i][9]
constexpr int kP3Stage = 2 * kP3Op;
constexpr int kP3Tile = kP3O * kP3I * 25;
static_assert(kP3Stages * kP3Stage >= kP3Tile, "the warps' sums reuse the rings");
// Floats of the rings of W warps, and with them the sums of the first of two parts of each warp
template <int W>
struct P3Form {
  static constexpr int RING = W * kP3Stages * kP3Stage, BYTES = (RING + (W < kP3Parts ? W * kP3Tile : 0)) * 4;
};

template <int W>
__global__ void __launch_bounds__(W * 32, 16 / W)
k_compose33(const __grid_constant__ Compose33 a, const __grid_constant__ BlockDelivery dv) {
  constexpr int V = kP3Parts / W;                  // parts of the reduction that a warp takes, one after the other
  static_assert(V == 1 || V == 2, "");
  extern __shared__ __align__(16) float p3_smem[];
  const int tid = (int)threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int c0 = a.c0, c1 = a.c1, c2 = a.c2;
  const RawLayer &l1 = a.first.l, &l2 = a.second.l;
  int blk = (int)blockIdx.x;
  dc_pdl_enter();
  if (blk >= a.gi * a.go) {
    blk -= a.gi * a.go;
    if (blk >= a.go) {
      zero_dead_chunks(dv, c2, blk - a.go, (int)gridDim.x - a.gi * a.go - a.go);
      return;
    }
    // ---- bias: b'[o] = b2~[o] + sum_c (g2 sum of W2[o][c] (+ 1 where c == o and an identity rides)) b1~[c]; a warp per o
    for (int o = blk * kP3O + warp; o < c2 && o < (blk + 1) * kP3O; o += W) {
      compose33_bias(a, o, lane);
    }
    return;
  }
  const int o0 = (blk / a.gi) * kP3O, i0 = (blk % a.gi) * kP3I;
  __shared__ float g2s[kP3O];                      // BN scales of the tile's output channels
  if (tid < kP3O) g2s[tid] = o0 + tid < c2 ? raw_scale(l2, o0 + tid) : 0.f;
  const int per = ((c1 + kP3Parts - 1) / kP3Parts + 3) & ~3;        // channels of a part
  const int cb = warp * V * per, ce = cb + V * per < c1 ? cb + V * per : c1;
  const int nsl = ce > cb ? (ce - cb) / kP3Slice : 0;               // c1 is a multiple of 4
  float *ring = p3_smem + warp * (kP3Stages * kP3Stage);
  // 72 pieces of each operand per slice: W2 rows of 36 floats (4 channels of one o), W1 rows of 72 (8 i of one channel).
  // A lane's places in a slice stay the same, what moves is where the slice begins.
  int off[5];
  bool ok[5];
#pragma unroll
  for (int h = 0; h < 5; ++h) {
    const int e = lane + 32 * h;
    if (h < 2 || (h == 2 && e < 72)) {
      const int o = e / 9, x = e - o * 9;
      off[h] = o * c1 * 9 + x * 4;
      ok[h] = o0 + o < c2;
    } else {
      const int f = e - 72, c = f / 18, x = f - c * 18;             // a piece lies inside one channel's 8 i: c0 is a multiple of 4
      off[h] = c * c0 * 9 + x * 4;
      ok[h] = i0 * 9 + x * 4 < c0 * 9;
    }
  }
  const float *w2g = l2.w + ((size_t)o0 * c1 + cb) * 9, *w1g = l1.w + ((size_t)cb * c0 + i0) * 9;
  const int step1 = kP3Slice * c0 * 9;
  auto fetch = [&](int buf) {
    float *st = ring + buf * kP3Stage + lane * 4;
#pragma unroll
    for (int h = 0; h < 5; ++h) {
      const float *g = h < 2 || (h == 2 && lane < 8) ? w2g : w1g;
      if (h < 4 || lane < 16) mb_cp16(st + h * 128, ok[h] ? g + off[h] : l2.w, ok[h]);
    }
    w2g += kP3Slice * 9;
    w1g += step1;
  };
#pragma unroll
  for (int sl = 0; sl < kP3Stages - 1; ++sl) {
    if (sl < nsl) fetch(sl);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  // BN scale of the first layer: lane l holds channel l's of 32, asked for a slice ahead of the first that uses it
  constexpr int kScaled = 32 / kP3Slice;         // slices that one set of scales covers
  float bn_g = 1.f, bn_v = 1.f;
  auto ask = [&](int set) {
    const int cs = cb + set * 32 + lane, c = cs < ce ? cs : cb;
    if (l1.gamma) { bn_g = l1.gamma[c]; bn_v = l1.var[c]; }
  };
  auto scale = [&]() { return l1.gamma ? bn_g / sqrtf(bn_v + l1.eps) : 1.f; };
  float sc = 1.f;
  if (nsl > 0) { ask(0); sc = scale(); }
  const int ol = (lane >> 3) * 2, il = lane & 7;
  float acc[2][25] = {};
  float *mine = p3_smem + (warp * kP3O + ol) * kP3I * 25 + il * 25;  // where this thread leaves its sums
  auto leave = [&](float *at) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int t = 0; t < 25; ++t) at[h * kP3I * 25 + t] = acc[h][t];
  };
  int buf = 0, fbuf = kP3Stages - 1;
#pragma unroll 1
  for (int sl = 0; sl < nsl; ++sl) {
    const int at = sl % kScaled;
    if (at == kScaled - 1) ask(sl / kScaled + 1);  // past the end: the warp's first channel, not used
    asm volatile("cp.async.wait_group %0;" ::"n"(kP3Stages - 2) : "memory");
    __syncwarp();
    if (sl + kP3Stages - 1 < nsl) fetch(fbuf);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float *w2 = ring + buf * kP3Stage + ol * (kP3Slice * 9), *w1 = ring + buf * kP3Stage + kP3Op + il * 9;
#pragma unroll
    for (int c = 0; c < kP3Slice; ++c) {
      const float s = __shfl_sync(0xffffffffu, sc, at * kP3Slice + c);
      float b[9], x[2][9];
#pragma unroll
      for (int t = 0; t < 9; ++t) {
        b[t] = w1[c * (kP3I * 9) + t] * s;
        x[0][t] = w2[c * 9 + t];
        x[1][t] = w2[kP3Slice * 9 + c * 9 + t];
      }
#pragma unroll
      for (int u2 = 0; u2 < 3; ++u2)
#pragma unroll
        for (int v2 = 0; v2 < 3; ++v2)
#pragma unroll
          for (int u1 = 0; u1 < 3; ++u1)
#pragma unroll
            for (int v1 = 0; v1 < 3; ++v1) {
              acc[0][(u1 + u2) * 5 + v1 + v2] = fmaf(x[0][u2 * 3 + v2], b[u1 * 3 + v1], acc[0][(u1 + u2) * 5 + v1 + v2]);
              acc[1][(u1 + u2) * 5 + v1 + v2] = fmaf(x[1][u2 * 3 + v2], b[u1 * 3 + v1], acc[1][(u1 + u2) * 5 + v1 + v2]);
            }
    }
    if (at == kScaled - 1) sc = scale();
    if (V == 2 && sl == per / kP3Slice - 1) {      // the end of the warp's first part: its sums wait behind the rings
      leave(mine + P3Form<W>::RING);
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int t = 0; t < 25; ++t) acc[h][t] = 0.f;
    }
    __syncwarp();                                  // the slice's buffer may be refilled
    buf = buf + 1 == kP3Stages ? 0 : buf + 1;
    fbuf = fbuf + 1 == kP3Stages ? 0 : fbuf + 1;
  }
  if (V == 2 && nsl < per / kP3Slice) {            // the reduction ends inside that part
    leave(mine + P3Form<W>::RING);
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int t = 0; t < 25; ++t) acc[h][t] = 0.f;
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  leave(mine);
  __syncthreads();
  const bool last = dv.mode >= 0, special = a.first.ident || a.second.ident || (last && dv.ident);
  // four elements of the warps' sums at a time: 50 pieces to a row of 8 input channels, 25 to each 4 of them that exist
  for (int e = tid; e < kP3Tile / 4; e += W * 32) {
    float4 *p = reinterpret_cast<float4 *>(p3_smem) + e;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int v = 0; v < kP3Parts; ++v) {           // in the order of the channels, whichever warp had them
      const float4 q = p[v / V * (kP3Tile / 4) + (V == 2 && v % 2 == 0 ? P3Form<W>::RING / 4 : 0)];
      s.x += q.x; s.y += q.y; s.z += q.z; s.w += q.w;
    }
    const int oi = e / (kP3I * 25 / 4), x = (e - oi * (kP3I * 25 / 4)) * 4, o = o0 + oi;
    if (o < c2 && i0 + x / 25 < c0) {
      const float g2 = g2s[oi];
      s.x *= g2; s.y *= g2; s.z *= g2; s.w *= g2;
      if (special) {                               // of a tile with identities to add
        float v4[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) v4[q] = compose33_ident(a, last && dv.ident, g2, v4[q], o, i0 + (x + q) / 25, (x + q) % 25);
        s = make_float4(v4[0], v4[1], v4[2], v4[3]);
      }
      *reinterpret_cast<float4 *>(a.w_out + ((size_t)o * c0 + i0) * 25 + x) = s;
    }
    if (last && dv.mode > 0) *p = s;               // these elements are read by this thread alone
  }
  if (!last || dv.mode == 0) return;
  __syncthreads();
  deliver_tile<kP3O, kP3I, 5>(dv, p3_smem, o0, i0, c0, c2, tid, W * 32);
}

// ----------------------------------------------------------------------------------------------
// A dense 1x1 and a 3x3 depthwise layer, in either order, as a run of its own: every element of the result is one
// product, W'[o][i][t] = W~[o][i] D~[c][t] with c = o (1x1 first) or c = i (depthwise first), so the run is bound by
// writing its result (160 -> 960: 5.5 MB and its packed copy) and by its launches.  One launch reads the layers as they
// are and delivers tiles of 8 x 16 channel pairs, or of 8 x 32 or 8 x 64 where those are two to an SM; blocks behind the tiles compute the
// bias (a warp per output channel) and zero the packed chunks without weights.  As fold, composition and delivery, three launches with the
// result written and read in between: 160 -> 960 then depthwise 27.6 us, depthwise then 576 -> 96 27.1, 384 -> 64 17.3; here 7.3, 4.6 and
// 3.9 us.
//
// Before: 9.3, 7.2 and 5.1 us; 320 -> 1920 20.2, now 13.7, depthwise then 1152 -> 192 16.9, now 8.9.  After a depthwise layer the bias
// blocks were the longest: each warp worked out every channel's factor for itself.  Then each chunk's place in the packed copy,
// divisions all, and in large results the tiles' starts.  (The smallest, 2.7 us, take 0.1 more.)
// ----------------------------------------------------------------------------------------------
struct Outer33 {
  RawLayer dense, dw;
  int ident_dense, ident_dw;     // identity kernels riding on the layers
  int dw_first;
  int c0, c2;                    // input and output channels of the run
  float *w_out, *b_out;
  int gi, go;
};

template <int IT>
__global__ void __launch_bounds__(kMbThreads)
k_merge_outer33(const __grid_constant__ Outer33 a, const __grid_constant__ BlockDelivery dv) {
  constexpr int kBias = 1024;                      // channels whose bias factors a CTA holds at a time
  __shared__ float wv[kMbO * IT > kBias ? kMbO * IT : kBias], dd[IT * 9], out[IT == 16 ? kMbO * IT * 9 : 1];
  __shared__ size_t row_s[kMbO], plane_s[IT / 8 * 9];              // where channels and taps are in the packed copy
  const int tid = (int)threadIdx.x, lane = tid & 31;
  const int c0 = a.c0, c2 = a.c2;
  int blk = (int)blockIdx.x;
  dc_pdl_enter();
  if (blk >= a.gi * a.go) {
    blk -= a.gi * a.go;
    if (blk >= a.go) {
      zero_dead_chunks(dv, c2, blk - a.go, (int)gridDim.x - a.gi * a.go - a.go);
      return;
    }
    const int o = blk * kMbO + (tid >> 5);
    float s = 0.f;
    if (a.dw_first) {                              // b2~ + sum_c W~[o][c] b1~[c], b1~ by all of the CTA
      const int ol = o < c2 ? o : 0;
      const RawNumbers n2(a.dense, ol);
      const float *w = a.dense.w + (size_t)ol * c0;
      const float g2 = n2.scale(a.dense);
      float *b1 = wv;
#pragma unroll 1
      for (int cs = 0; cs < c0; cs += kBias) {
        const int n = c0 - cs < kBias ? c0 - cs : kBias;
        __syncthreads();
        for (int c = tid; c < n; c += kMbThreads) {
          const RawNumbers n1(a.dw, cs + c);
          b1[c] = n1.bias(a.dw, n1.scale(a.dw));
        }
        __syncthreads();
#pragma unroll 1
        for (int c = lane; c < n; c += 256) {      // eight weights on their way at once
          float x[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) x[q] = c + 32 * q < n ? w[cs + c + 32 * q] : 0.f;
#pragma unroll
          for (int q = 0; q < 8; ++q)
            if (c + 32 * q < n) s = fmaf(fmaf(g2, x[q], a.ident_dense && cs + c + 32 * q == o ? 1.f : 0.f), b1[c + 32 * q], s);
        }
      }
      for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
      if (lane == 0 && o < c2) a.b_out[o] = n2.bias(a.dense, g2) + s;
    } else if (o < c2) {                           // b2~ + (sum_t D~[o][t]) b1~[o]
      const float g2 = raw_scale(a.dw, o);
      s = lane < 9 ? g2 * a.dw.w[(size_t)o * 9 + lane] : 0.f;
      for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
      if (lane == 0)
        a.b_out[o] = fmaf(s + (a.ident_dw ? 1.f : 0.f), raw_bias(a.dense, o, raw_scale(a.dense, o)), raw_bias(a.dw, o, g2));
    }
    return;
  }
  const int o0 = (blk / a.gi) * kMbO, i0 = (blk % a.gi) * IT;
  for (int e = tid; e < kMbO * IT; e += kMbThreads) {
    const int o = o0 + e / IT, i = i0 + e % IT;
    wv[e] = o < c2 && i < c0 ? fmaf(raw_scale(a.dense, o), a.dense.w[(size_t)o * c0 + i], a.ident_dense && o == i ? 1.f : 0.f) : 0.f;
  }
  const int d0 = a.dw_first ? i0 : o0, nd = a.dw_first ? IT : kMbO, cd = a.dw_first ? c0 : c2;
  for (int e = tid; e < nd * 9; e += kMbThreads) {
    const int c = d0 + e / 9, t = e % 9;
    dd[e] = c < cd ? fmaf(raw_scale(a.dw, c), a.dw.w[(size_t)c * 9 + t], a.ident_dw && t == 4 ? 1.f : 0.f) : 0.f;
  }
  // Where a bf16 chunk goes: rows of a tap's chunk plane, except in orders that hold taps or pixels in the rows.  Worked out once a
  // CTA: the divisions are most of what a chunk costs.
  const bool by_rows = dv.mode == 2 && !dv.ko.fold && !dv.ko.pair;
  const int per = dv.ko.rows && dv.ko.nnt > 1 ? dv.ko.n_tile : dv.ko.n_pad;
  if (by_rows) {
    const int e = tid - (kMbThreads - IT / 8 * 9), r = tid - 32;
    if (e >= 0) plane_s[e] = (size_t)dc_korder_encode(dv.ko, (i0 >> 3) + e / 9, e % 9 / 3, e % 3) * per;
    if (r >= 0 && r < kMbO) row_s[r] = dc_packed_chunk(dv.ko, 0, o0 + r);
  }
  __syncthreads();
  auto value = [&](int ow, int iw, int t) {
    const float v = wv[ow * IT + iw] * dd[(a.dw_first ? iw : ow) * 9 + t];
    return dv.ident && t == 4 && o0 + ow == i0 + iw ? v + 1.f : v;
  };
  if (IT == 16) {                                  // small results: each once, for the result and its packed copy
    for (int e = tid; e < kMbO * IT * 9; e += kMbThreads) {
      const int ow = e / (IT * 9), x = e - ow * (IT * 9);
      const float v = value(ow, x / 9, x % 9);
      if (o0 + ow < c2 && i0 + x / 9 < c0) a.w_out[((size_t)(o0 + ow) * c0 + i0) * 9 + x] = v;
      out[e] = v;
    }
    if (dv.mode == 0) return;
    __syncthreads();
    if (!by_rows) {
      deliver_tile<kMbO, IT, 3>(dv, out, o0, i0, c0, c2, tid, kMbThreads);
      return;
    }
  } else if (c0 % 4 == 0) {                        // four neighbouring results at a time: rows are whole pieces then
    for (int e = tid; e < kMbO * IT * 9 / 4; e += kMbThreads) {
      const int ow = e / (IT * 9 / 4), x = (e - ow * (IT * 9 / 4)) * 4;
      if (o0 + ow >= c2 || i0 + x / 9 >= c0) continue;
      float v[4];
      int iw = x / 9, t = x - iw * 9;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        v[j] = value(ow, iw, t);
        if (++t == 9) { t = 0; ++iw; }
      }
      *reinterpret_cast<float4 *>(a.w_out + ((size_t)(o0 + ow) * c0 + i0) * 9 + x) = make_float4(v[0], v[1], v[2], v[3]);
    }
  } else {
    for (int e = tid; e < kMbO * IT * 9; e += kMbThreads) {
      const int ow = e / (IT * 9), x = e - ow * (IT * 9);
      if (o0 + ow < c2 && i0 + x / 9 < c0) a.w_out[((size_t)(o0 + ow) * c0 + i0) * 9 + x] = value(ow, x / 9, x % 9);
    }
  }
  if (dv.mode == 0) return;
  if (dv.mode == 1) {
    float *to = reinterpret_cast<float *>(dv.packed);
    for (int e = tid; e < kMbO * IT * 9; e += kMbThreads) {
      const int ow = e % kMbO, rest = e / kMbO, iw = rest % IT, t = rest / IT;
      if (o0 + ow < c2 && i0 + iw < c0) to[((size_t)t * c0 + i0 + iw) * c2 + o0 + ow] = value(ow, iw, t);
    }
    return;
  }
  auto two = [](float lo, float hi) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t *>(&p);
  };
  // a thread to three taps of a chunk's channels, whose weights it reads once; in small results to one
  constexpr int TAPS = IT == 16 ? 1 : 3;
  for (int e = tid; e < kMbO * (IT / 8) * (9 / TAPS); e += kMbThreads) {
    const int ow = e % kMbO, rest = e / kMbO, hf = rest % (IT / 8), o = o0 + ow, i = i0 + hf * 8;
    int t = rest / (IT / 8) * TAPS;
    if (o >= c2 || i >= c0) continue;
#pragma unroll
    for (int n = 0; n < TAPS; ++n, ++t) {
      float v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = IT == 16 ? out[(ow * IT + hf * 8 + q) * 9 + t] : value(ow, hf * 8 + q, t);
      if (by_rows)
        reinterpret_cast<uint4 *>(dv.packed)[row_s[ow] + plane_s[hf * 9 + t]] =
            make_uint4(two(v[0], v[1]), two(v[2], v[3]), two(v[4], v[5]), two(v[6], v[7]));
      else
        deliver_chunk<9, 1>(dv, v, o, i, t, c0, c2);
    }
  }
}

// ----------------------------------------------------------------------------------------------
// Two dense 1x1 layers as a run of their own: W' = (g2 W2 + I2) (g1 W1 + I1), a plain matrix product [c2][c1] x [c1][c0], from
// the layers as they are to the delivered result in one launch.
//
// A CTA owns BO x BI results; its 256 threads are G groups that take the 16-channel slices of the reduction in turn, each
// with operands of its own in shared memory (double buffered through registers, where W2 is turned to [channel][output] and
// W1 gets its BN scale) and a barrier of its own; a thread owns TO x 4 results, TO / 4 + 1 16-byte reads for 4 TO FMAs.  The
// groups' sums meet in shared memory in group order.  Tiles of 64 or 48 x 64 where they give the chip enough of them,
// otherwise 32 x 32 by four groups, whose reductions are shorter chains.  Blocks behind the tiles compute the bias (a warp per
// output) and zero the packed chunks without weights.
//
// As fold, product, bias and delivery, four launches with the product written and read in between: 960 -> 320 -> 1280 60.7 us,
// now 30.1 (35.3 with the sums added element by element and the second layer's scales asked for
// behind them); 32 -> 16 -> 96 7.5, now 3.2; 160 -> 160 -> 160 15.0, now 5.9.
// ----------------------------------------------------------------------------------------------
struct Merge11 {
  RawLayer l1, l2;
  int ident1, ident2;            // identity kernels riding on the layers
  int c0, c1, c2;
  float *w_out, *b_out;
  int gi, go;
};

template <int BO, int BI, int TO, int G>
__global__ void __launch_bounds__(256, 3)
k_merge_11(const __grid_constant__ Merge11 a, const __grid_constant__ BlockDelivery dv) {
  constexpr int VA = TO % 4 == 0 ? 4 : 2;          // channels of W2 per read
  constexpr int T = 256 / G, KS = 16, PA = BO + 4, PB = BI + 4, STAGE = KS * (PA + PB);
  constexpr int PIECES = BO * KS / 4, NA = (PIECES + T - 1) / T, NB = BI * KS / 4 / T;     // 16-byte pieces a thread stages
  static_assert(T == (BO / TO) * (BI / 4) && NA >= 1 && NB >= 1 && G * 2 * STAGE >= G * BO * BI / 2, "tile");
  __shared__ __align__(16) float sm[G * 2 * STAGE < G * BO * BI ? G * BO * BI : G * 2 * STAGE];
  const int tid = (int)threadIdx.x, lane = tid & 31, g = tid / T, t = tid % T;
  const int c0 = a.c0, c1 = a.c1, c2 = a.c2;
  int blk = (int)blockIdx.x;
  dc_pdl_enter();
  if (blk >= a.gi * a.go) {
    blk -= a.gi * a.go;
    const int nb = dc_div_up(c2, 8);
    if (blk >= nb) {
      zero_dead_chunks(dv, c2, blk - nb, (int)gridDim.x - a.gi * a.go - nb);
      return;
    }
    const int o = blk * 8 + (tid >> 5);            // b2~ + sum_c (g2 W2[o][c] + I2) b1~[c]
    if (o >= c2) return;
    const float g2 = raw_scale(a.l2, o);
    float s = 0.f;
#pragma unroll 4
    for (int c = lane; c < c1; c += 32)
      s = fmaf(fmaf(g2, a.l2.w[(size_t)o * c1 + c], a.ident2 && c == o ? 1.f : 0.f), raw_bias(a.l1, c, raw_scale(a.l1, c)), s);
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if (lane == 0) a.b_out[o] = raw_bias(a.l2, o, g2) + s;
    return;
  }
  const int o0 = (blk / a.gi) * BO, i0 = (blk % a.gi) * BI;
  const bool special = a.ident1 || a.ident2 || dv.ident;
  __shared__ float g2s[BO];                        // BN scales of the tile's output channels
  if (tid < BO) g2s[tid] = o0 + tid < c2 ? raw_scale(a.l2, o0 + tid) : 0.f;
  float *mine = sm + g * 2 * STAGE;
  const int slices = (c1 + KS - 1) / KS, my = (slices - g + G - 1) / G;      // slices g, g + G, ...
  float4 va[NA], vb[NB];
  float gm[NB], vr[NB];                            // BN of W1's channels; first touched when staged, like the weights
  auto fetch = [&](int sl) {                       // out-of-range pieces read element 0 and are zeroed when staged
    const int cs = (g + sl * G) * KS;
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int e = t + q * T, o = o0 + e / 4, c = cs + (e & 3) * 4;
      va[q] = *reinterpret_cast<const float4 *>(a.l2.w + (e < PIECES && o < c2 && c < c1 ? (size_t)o * c1 + c : 0));
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int e = t + q * T, c = cs + e / (BI / 4), i = i0 + (e % (BI / 4)) * 4;
      const bool ok = c < c1 && i < c0;
      vb[q] = *reinterpret_cast<const float4 *>(a.l1.w + (ok ? (size_t)c * c0 + i : 0));
      gm[q] = a.l1.gamma ? a.l1.gamma[ok ? c : 0] : 1.f;
      vr[q] = a.l1.gamma ? a.l1.var[ok ? c : 0] : 1.f;
    }
  };
  auto stage = [&](int sl, int buf) {
    float *A = mine + buf * STAGE, *B = A + KS * PA;
    const int cs = (g + sl * G) * KS;
#pragma unroll
    for (int q = 0; q < NA; ++q) {
      const int e = t + q * T, o = o0 + e / 4, c = (e & 3) * 4;
      const bool ok = o < c2 && cs + c < c1;
      if (e >= PIECES) continue;
      A[(c + 0) * PA + e / 4] = ok ? va[q].x : 0.f;
      A[(c + 1) * PA + e / 4] = ok ? va[q].y : 0.f;
      A[(c + 2) * PA + e / 4] = ok ? va[q].z : 0.f;
      A[(c + 3) * PA + e / 4] = ok ? va[q].w : 0.f;
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int e = t + q * T, c = cs + e / (BI / 4), i = i0 + (e % (BI / 4)) * 4;
      const bool ok = c < c1 && i < c0;
      const float sc = a.l1.gamma ? gm[q] / sqrtf(vr[q] + a.l1.eps) : 1.f;
      *reinterpret_cast<float4 *>(B + (e / (BI / 4)) * PB + (e % (BI / 4)) * 4) =
          ok ? make_float4(vb[q].x * sc, vb[q].y * sc, vb[q].z * sc, vb[q].w * sc) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  const int ty = t / (BI / 4), tx = t % (BI / 4);
  float acc[TO][4] = {};
  if (my > 0) { fetch(0); stage(0, 0); }
  asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(T) : "memory");
#pragma unroll 1
  for (int sl = 0; sl < my; ++sl) {
    if (sl + 1 < my) fetch(sl + 1);
    const float *A = mine + (sl & 1) * STAGE + ty * TO, *B = mine + (sl & 1) * STAGE + KS * PA + tx * 4;
#pragma unroll
    for (int k = 0; k < KS; ++k) {
      float x[TO];
#pragma unroll
      for (int q = 0; q < TO; q += VA) {
        if (VA == 4) *reinterpret_cast<float4 *>(x + q) = *reinterpret_cast<const float4 *>(A + k * PA + q);
        else *reinterpret_cast<float2 *>(x + q) = *reinterpret_cast<const float2 *>(A + k * PA + q);
      }
      const float4 b = *reinterpret_cast<const float4 *>(B + k * PB);
#pragma unroll
      for (int q = 0; q < TO; ++q) {
        acc[q][0] = fmaf(x[q], b.x, acc[q][0]);
        acc[q][1] = fmaf(x[q], b.y, acc[q][1]);
        acc[q][2] = fmaf(x[q], b.z, acc[q][2]);
        acc[q][3] = fmaf(x[q], b.w, acc[q][3]);
      }
    }
    if (sl + 1 < my) stage(sl + 1, (sl + 1) & 1);
    asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(T) : "memory");
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < TO; ++q)
    *reinterpret_cast<float4 *>(sm + (g * BO + ty * TO + q) * BI + tx * 4) = make_float4(acc[q][0], acc[q][1], acc[q][2], acc[q][3]);
  __syncthreads();
  for (int e = tid; e < BO * BI / 4; e += 256) {   // four elements of the groups' sums at a time; c0 is a multiple of 4
    float4 *p = reinterpret_cast<float4 *>(sm) + e;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int q = 0; q < G; ++q) {
      const float4 f = p[q * (BO * BI / 4)];
      s.x += f.x; s.y += f.y; s.z += f.z; s.w += f.w;
    }
    const int oi = e / (BI / 4), o = o0 + oi, i = i0 + e % (BI / 4) * 4;
    if (o < c2 && i < c0) {
      const float g2 = g2s[oi];
      s.x *= g2; s.y *= g2; s.z *= g2; s.w *= g2;
      if (special) {                               // of a tile with identities to add
        float v4[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (a.ident1) v4[q] = fmaf(g2, a.l2.w[(size_t)o * c1 + i + q], v4[q]);                      // g2 W2 I1: c0 == c1
          if (a.ident2) v4[q] = fmaf(raw_scale(a.l1, o), a.l1.w[(size_t)o * c0 + i + q], v4[q]);      // I2 g1 W1: c1 == c2
          if (o == i + q) v4[q] += (a.ident1 && a.ident2 ? 1.f : 0.f) + (dv.ident ? 1.f : 0.f);
        }
        s = make_float4(v4[0], v4[1], v4[2], v4[3]);
      }
      *reinterpret_cast<float4 *>(a.w_out + (size_t)o * c0 + i) = s;
    }
    *p = s;                                        // these elements of group 0's sums are read by this thread alone
  }
  if (dv.mode == 0) return;
  __syncthreads();
  deliver_tile<BO, BI, 1>(dv, sm, o0, i0, c0, c2, tid, 256);
}

// ----------------------------------------------------------------------------------------------
// A dense 3x3 piece after a dense 1x1 one with stride 1: every tap sum has one term,
//   W'[o][i][t] = sum_c (W2[o][c][t] + I2) (W1[c][i] + I1),
// a product of [o, t][c] with [c][i].  A CTA owns 8 output channels x nine taps x 32 input channels; a thread the taps of one
// output channel for four of the input channels (nine broadcast values of W2 with four of W1: 36 FMAs for ten reads), and
// the 256 threads are four groups that share the channels of every slice of 32.  Slices come in by cp.async, two deep.  The sums
// meet in shared memory in group order and leave as the piece or, for a run's last composition, delivered.  Blocks
// behind the tiles compute the bias, and zero the packed chunks without weights.
//
// With a thread per result that walked the channels from L2, and a delivery launch behind it, the merge 384 -> 96 -> (576) -> 96
// took 38.0 us, now 21.8; 144 -> 32 -> (192) -> 32 13.9, now 13.3.  (The same for 5x5 pieces, two input channels a thread, was
// faster from 64 channels on but took 9.6 us instead of 7.4 at 24 -> 8 -> 80, and its longer sums were further from 64 bits.)
// ----------------------------------------------------------------------------------------------
struct After11 {
  Piece first, second;
  float *w_out, *b_out;
  int gi, go;
};
constexpr int kA1O = 8, kA1I = 32, kA1C = 32;    // results of a CTA: output and input channels; channels of a slice
constexpr int kA1N = 4, kA1G = 256 / (kA1O * kA1I / kA1N);        // input channels of a thread, groups
constexpr int kA1P = kA1C * 9 + 4;               // floats between output channels of a slice
constexpr int kA1Stage = kA1O * kA1P + kA1C * kA1I, kA1Tile = kA1O * kA1I * 9;
constexpr int kA1Smem = 4 * (2 * kA1Stage > kA1G * kA1Tile ? 2 * kA1Stage : kA1G * kA1Tile);

__global__ void __launch_bounds__(256, 2)
k_compose_after_11(const __grid_constant__ After11 a, const __grid_constant__ BlockDelivery dv) {
  constexpr int K = 3, KK = 9, NI = kA1N, T = kA1O * kA1I / NI, G = kA1G, CTR = 4, PO = kA1P, STAGE = kA1Stage, TILE = kA1Tile;
  extern __shared__ __align__(16) float a1_smem[];
  const int tid = (int)threadIdx.x, g = tid / T, t = tid % T;
  const Piece &p1 = a.first, &p2 = a.second;
  const int c0 = p1.c_in, c1 = p1.c_out, c2 = p2.c_out;
  int blk = (int)blockIdx.x;
  dc_pdl_enter();
  if (blk >= a.gi * a.go) {
    blk -= a.gi * a.go;
    if (blk >= a.go) {
      zero_dead_chunks(dv, c2, blk - a.go, (int)gridDim.x - a.gi * a.go - a.go);
      return;
    }
    compose_bias_block(p1, p2, a.b_out, blk);      // eight warps, eight output channels
    return;
  }
  const int o0 = (blk / a.gi) * kA1O, i0 = (blk % a.gi) * kA1I;
  const int slices = (c1 + kA1C - 1) / kA1C;
  auto fetch = [&](int sl) {
    float *A = a1_smem + (sl & 1) * STAGE, *B = A + kA1O * PO;
    const int cs = sl * kA1C, left = c1 - cs < kA1C ? c1 - cs : kA1C;      // a multiple of 4
    for (int e = tid; e < kA1O * (kA1C * KK / 4); e += 256) {
      const int o = e / (kA1C * KK / 4), x = e - o * (kA1C * KK / 4);
      const bool ok = o0 + o < c2 && x * 4 < left * KK;
      mb_cp16(A + o * PO + x * 4, ok ? p2.w + ((size_t)(o0 + o) * c1 + cs) * KK + x * 4 : p2.w, ok);
    }
    for (int e = tid; e < kA1C * kA1I / 4; e += 256) {
      const int c = e / (kA1I / 4), i = i0 + (e % (kA1I / 4)) * 4;
      const bool ok = c < left && i < c0;
      mb_cp16(B + e * 4, ok ? p1.w + (size_t)(cs + c) * c0 + i : p1.w, ok);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int ol = t / (kA1I / NI), il = (t % (kA1I / NI)) * NI;
  float acc[NI][KK] = {};
  fetch(0);
#pragma unroll 1
  for (int sl = 0; sl < slices; ++sl) {
    if (sl + 1 < slices) {
      fetch(sl + 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const float *A = a1_smem + (sl & 1) * STAGE + ol * PO, *B = a1_smem + (sl & 1) * STAGE + kA1O * PO + il;
#pragma unroll 4
    for (int c = g; c < kA1C; c += G) {            // channels dealt in turn: short runs keep their sums in parts too
      float b[NI];
#pragma unroll
      for (int q = 0; q < NI; ++q) b[q] = B[c * kA1I + q];
#pragma unroll
      for (int u = 0; u < KK; ++u) {
        const float w = A[c * KK + u];
#pragma unroll
        for (int q = 0; q < NI; ++q) acc[q][u] = fmaf(w, b[q], acc[q][u]);
      }
    }
    __syncthreads();                               // the slice's buffer is refilled in the next turn
  }
#pragma unroll
  for (int q = 0; q < NI; ++q)
#pragma unroll
    for (int u = 0; u < KK; ++u) a1_smem[g * TILE + (ol * kA1I + il + q) * KK + u] = acc[q][u];
  __syncthreads();
  const bool last = dv.mode >= 0;
  for (int e = tid; e < TILE; e += 256) {
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < G; ++q) s += a1_smem[q * TILE + e];
    const int oi = e / KK, u = e - oi * KK, o = o0 + oi / kA1I, i = i0 + oi % kA1I;
    if (o < c2 && i < c0) {
      if (p1.ident) s += p2.w[((size_t)o * c1 + i) * KK + u];                          // W2 o I: c0 == c1
      if (p2.ident && u == CTR) s += p1.w[(size_t)o * c0 + i];                         // I o W1: c1 == c2
      if (u == CTR && o == i) s += (p1.ident && p2.ident ? 1.f : 0.f) + (last && dv.ident ? 1.f : 0.f);
      a.w_out[((size_t)o * c0 + i) * KK + u] = s;
    }
    if (last && dv.mode > 0) a1_smem[e] = s;       // element e of group 0's sums is read by this thread alone
  }
  if (!last || dv.mode == 0) return;
  __syncthreads();
  deliver_tile<kA1O, kA1I, K>(dv, a1_smem, o0, i0, c0, c2, tid, 256);
}
// the bias of a composition on its own
__global__ void k_compose_bias(Piece first, Piece second, float *b_out) { compose_bias_block(first, second, b_out, (int)blockIdx.x); }

// ----------------------------------------------------------------------------------------------
// host: validation and geometry
// ----------------------------------------------------------------------------------------------

dc_status dc_validate_geom(const dc_geom *g) {
  if (!g) return DC_ERR_INVALID_ARG;
  if (g->c_in <= 0 || g->c_out <= 0 || g->k <= 0 || g->stride <= 0 || g->pad < 0 || g->groups <= 0)
    return DC_ERR_INVALID_ARG;
  if (g->k % 2 == 0) return DC_ERR_UNSUPPORTED;
  if (!(g->groups == 1 || (g->groups == g->c_in && g->c_in == g->c_out))) return DC_ERR_UNSUPPORTED;
  return DC_OK;
}

static dc_status validate_layer(const dc_layer *L) {
  dc_geom g = {L->c_in, L->c_out, L->groups, L->k, L->stride, L->pad};
  dc_status st = dc_validate_geom(&g);
  if (st != DC_OK) return st;
  if (!L->weight) return DC_ERR_INVALID_ARG;
  int nbn = (L->bn_gamma != nullptr) + (L->bn_beta != nullptr) + (L->bn_mean != nullptr) + (L->bn_var != nullptr);
  if (nbn != 0 && nbn != 4) return DC_ERR_INVALID_ARG;
  return DC_OK;
}

static size_t piece_elems(int c_in, int c_out, int k, int diag) {
  return diag ? (size_t)c_out * k * k : (size_t)c_out * c_in * k * k;
}

static int find_group(const dc_residual *res, int n_res, int first) {
  for (int i = 0; i < n_res; ++i)
    if (res[i].first == first) return i;
  return -1;
}

static dc_status check_chain(const dc_layer *layers, int n, const dc_residual *res, int n_res,
                             dc_geom *merged) {
  if (!layers || n <= 0 || n_res < 0 || (n_res > 0 && !res)) return DC_ERR_INVALID_ARG;
  for (int i = 0; i < n; ++i) {
    dc_status st = validate_layer(&layers[i]);
    if (st != DC_OK) return st;
    if (i > 0 && layers[i].c_in != layers[i - 1].c_out) return DC_ERR_SHAPE;
  }
  int prev_last = -1;
  for (int gi = 0; gi < n_res; ++gi) {
    if (res[gi].first < 0 || res[gi].last >= n || res[gi].first > res[gi].last) return DC_ERR_INVALID_ARG;
    if (res[gi].first <= prev_last) return DC_ERR_INVALID_ARG;
    prev_last = res[gi].last;
    int k = 1, s = 1, p = 0;
    for (int i = res[gi].first; i <= res[gi].last; ++i) {
      k += (layers[i].k - 1) * s;
      p += layers[i].pad * s;
      s *= layers[i].stride;
    }
    if (s != 1 || layers[res[gi].first].c_in != layers[res[gi].last].c_out || 2 * p != k - 1)
      return DC_ERR_NOT_MERGEABLE;
  }
  int k = 1, s = 1, p = 0;
  for (int i = 0; i < n; ++i) {
    k += (layers[i].k - 1) * s;
    p += layers[i].pad * s;
    s *= layers[i].stride;
  }
  if (merged) {
    merged->c_in = layers[0].c_in;
    merged->c_out = layers[n - 1].c_out;
    merged->groups = 1;
    merged->k = k; merged->stride = s; merged->pad = p;
  }
  return DC_OK;
}

// Bump allocator over the caller's workspace (256-byte granules); with base == nullptr it only counts.
struct Bump {
  char *base; size_t off;
  float *take(size_t elems) {
    size_t bytes = dc_round_up(elems * sizeof(float), 256);
    float *p = base ? reinterpret_cast<float *>(base + off) : nullptr;
    off += bytes;
    return p;
  }
};

static inline int blocks_for(size_t total, int threads) {
  size_t b = (total + threads - 1) / threads;
  return (int)(b > 65535 ? 65535 : (b == 0 ? 1 : b));
}

// CTAs that zero the chunks of a packed copy that hold no weight
static int zero_ctas(const BlockDelivery &dv, const dc_geom &mg, int threads) {
  const KOrder &ko = dv.ko;
  if (dv.mode != 2) return 0;
  const bool full = ko.fold == 0 && ko.pair == 0 && ko.n_pad == mg.c_out && ko.e == ko.e_pad && (!ko.rows || mg.c_in % 16 == 0);
  return full ? 0 : dc_div_up(ko.ng * ko.e_pad * ko.n_pad, threads * 4);
}

// 3x3 after 3x3, 16-byte pieces of both operands
static bool compose33_ok(int c_in, int c_mid, int k1, int s1, int k2) {
  return k1 == 3 && s1 == 1 && k2 == 3 && c_in % 4 == 0 && c_mid % 4 == 0;
}
// The first status of a merge's launches that is not DC_OK.  A launch in <<<>>> form leaves its error with
// cudaGetLastError, and it is asked for behind each of them: asked once at the end of the merge it may be gone (the fp32
// convolution asks, and clears, it too; a run whose refused launch was followed by one of those returned DC_OK).
struct MergeStatus {
  dc_status s = DC_OK;
  DcWsHeader *ws = nullptr;      // where a bounded wait of its launches is latched (null: in the device's flags)
  void note(dc_status t) { if (s == DC_OK) s = t; }
  void note(cudaError_t e) { note(e == cudaSuccess ? DC_OK : DC_ERR_CUDA); }
  void launched() { note(cudaGetLastError()); }
};

template <int W>
static void launch_compose33_form(const Compose33 &a, const BlockDelivery &dv, const dc_geom &mg, cudaStream_t st, MergeStatus &status) {
  static unsigned char attr_done[kDcMaxDevices];
  status.note(dc_set_max_smem_once(k_compose33<W>, P3Form<W>::BYTES, attr_done));
  status.note(dc_launch_pdl(k_compose33<W>, dim3(a.gi * a.go + a.go + zero_ctas(dv, mg, W * 32)), dim3(W * 32), P3Form<W>::BYTES, st, a, dv));
  status.launched();
}
// By estimates of both in microseconds, fitted to 93 pairs of 32 to 1024 channels timed on either side (on the tensor core 4 % off, by
// FMAs 13 %): of the 93 this line sends 35 there, together 0.891 of the time on (geometric) average over all (always the faster one:
// 0.881), none slower; a line at 1.0 sends 40, two of them up to 8 % slower.  There a CTA's first tile takes 6.5 us and 0.6 for every 16
// channels between, a further one 4.9 us or more: many output and input channels, and enough between them, go there.  64 channels between
// and fewer stay: chains of FMAs so short are nearer to 64 bits for weights of one sign (0.76e-7, there up to 1.17e-7; the one pair of the 93
// that loses time by it: 144 -> 64 -> 200, 13.6 us there and 15.2 here).
static bool compose33_on_tensor_core(int c0, int c1, int c2) {
  const int n_sm = dc_sm_count(), steps = dc_div_up(c1, 64) * 4, tiles = dc_div_up(c0, 8) * dc_div_up(c2, 8), most = dc_div_up(tiles, n_sm);
  const double further = steps > 16 ? 0.58 * steps : (steps > 7 ? 2.4 + 0.33 * steps : 4.9);
  const double tc = 6.5 + 0.585 * steps + (dc_div_up(dc_div_up(c2, 14) * dc_div_up(c0, 8), n_sm) - 1) * further;
  const double fma = 4.0 + most * c1 * (most > 1 || 2 * tiles <= n_sm ? 0.042 : 0.063);
  return c1 > 64 && tc < 0.95 * fma;
}

// Four warps a tile, four tiles to an SM at once, except where the tiles of the SM with the most of them fill whole rounds of two
// better than of four: one or two of them (136 -> 136 -> 136: 25.6 us by four warps, 17.8 by eight), or three or five with a
// reduction long enough to matter (160 -> 160 -> 160, three: 29.1 and 24.1, with 48 channels between 12.7 and 13.2; 208 -> 208 ->
// 208, five: 55.0 and 49.0, with 48 20.9 and 21.3).  Timed in both forms at 1 to 16 tiles, 48 or as many channels between as
// outside: four tiles and from six on four warps are the faster ones, by up to 30 % with 48 channels between, or within 1.5 %.
static void launch_compose33(const Operand33 &first, const Operand33 &second, int c0, int c1, int c2, float *w, float *b,
                             const BlockDelivery &dv, const dc_geom &mg, cudaStream_t st, MergeStatus &status) {
  const Compose33 a{first, second, c0, c1, c2, w, b, dc_div_up(c0, kP3I), dc_div_up(c2, kP3O)};
  if (compose33_on_tensor_core(c0, c1, c2)) {
    const dc_status s = dc_launch_compose33_tc(a, dv, status.ws, st);
    if (s != DC_ERR_UNSUPPORTED) { status.note(s); return; }       // beyond its range (4096 channels between): the FMAs have none
  }
  const int most = dc_div_up(a.gi * a.go, dc_sm_count());
  if (most <= 2 || ((most == 3 || most == 5) && c1 >= 128)) launch_compose33_form<8>(a, dv, mg, st, status);
  else launch_compose33_form<4>(a, dv, mg, st, status);
}

template <int IT>
static void launch_outer33(Outer33 a, const BlockDelivery &dv, int zero, cudaStream_t st, MergeStatus &status) {
  a.gi = dc_div_up(a.c0, IT);
  status.note(dc_launch_pdl(k_merge_outer33<IT>, dim3(a.gi * a.go + a.go + zero), dim3(kMbThreads), 0, st, a, dv));
  status.launched();
}

template <int IT, int W>
static void launch_block33_form(TiledBlocks &tb, const BlockDelivery &dv, const dc_geom &mg, cudaStream_t st, MergeStatus &status) {
  tb.first[0] = 0;
  for (int i = 0; i < tb.n; ++i) {
    const int go = dc_div_up(tb.blk[i].c2, kMbO);
    tb.first[i + 1] = tb.first[i] + (dc_div_up(tb.blk[i].c0, IT) + 1) * go;       // tiles and bias groups
  }
  // Where every CTA can have an SM of its own it asks for more than half of one's shared memory.  Let in while the previous
  // kernel ends, the CTAs would otherwise gather two to an SM on the SMs that are free first.
  // 24 -> 144 -> 24 and the forward of the result, 64 images of 56 x 56, queued: 15.8 -> 14.5 us a step (13.8 where the forward lets
  // nothing in before its end, which costs 0.2 us where forwards follow one another); 160 -> 960 -> 160, more CTAs than SMs: 25.4.
  constexpr int ring = MbForm<IT, W>::RING, alone = ring > 116 * 1024 ? ring : 116 * 1024;
  const int grid = tb.first[tb.n] + zero_ctas(dv, mg, W * 32);
  static unsigned char attr_done[kDcMaxDevices];
  status.note(dc_set_max_smem_once(k_merge_block33<IT, W>, alone, attr_done));
  status.note(dc_launch_pdl(k_merge_block33<IT, W>, dim3(grid), dim3(W * 32), grid <= dc_sm_count() ? alone : ring, st, tb, dv));
  status.launched();
}
// A single block goes to the tensor core where an estimate says so: of 166 drawn blocks of 40 to 320 channels in and 160 to 1280 hidden
// ones 102, in 0.72 of the time on (geometric) average, two slower, by 2 and 5 %.  160 -> 960 -> 160 20.0 us and
// 14.3, 200 -> 928 -> 200 39.4 and 17.4, 64 -> 1168 -> 64 17.5 and 11.5, 96 -> 576 -> 96 11.2 and 10.5; what 24 -> 144 -> 24 takes there,
// 8.2 us, most of it the start and the end of a launch, is more than here, 6.1.  These are merges repeated; a run's first one finds
// neither weights nor code in L2.  Timed so, between events (5 us more each), 160 -> 960 -> 160 25.5 and 19.4, 200 -> 928 -> 200 45.0 and 23.5,
// 64 -> 1168 -> 64 22.4 and 16.5, 96 -> 576 -> 96 15.9 and 16.4, 120 -> 720 -> 120 17.4 and 18.4: what is near the line loses a little.
static bool block33_on_tensor_core(int c0, int c1, int c2, int run, int most16, int most24, int form) {
  const double fma = form == 0   ? 4.07 + 1.69 * (most16 - 1) + c1 / 8.0 * (0.0692 * most16 + 0.0306 * dc_div_up(most16, 2))
                     : form == 1 ? 4.6 + 0.1757 * c1 / 16.0
                                 : 5.69 + 0.248 * most24 * c1 / 16.0;
  const double tc = dc_merge_product_tc_us(kProductBlock, c0, c1, c2, run);
  return tc != 0.0 && tc < 0.95 * fma;
}
// Tiles of 8 x 16 pairs by eight warps; by sixteen, one CTA to an SM, for long reductions: of 8 x 16 where that gives no SM a
// second tile, of 8 x 24 where it leaves the SM with the most pairs fewer of them.
static void launch_block33(TiledBlocks &tb, const BlockDelivery &dv, const dc_geom &mg, cudaStream_t st, MergeStatus &status) {
  int tiles16 = 0, tiles24 = 0, hidden = 0;
  for (int i = 0; i < tb.n; ++i) {
    tiles16 += dc_div_up(tb.blk[i].c0, 16) * dc_div_up(tb.blk[i].c2, kMbO);
    tiles24 += dc_div_up(tb.blk[i].c0, 24) * dc_div_up(tb.blk[i].c2, kMbO);
    if (tb.blk[i].c1 > hidden) hidden = tb.blk[i].c1;
  }
  const int n_sm = dc_sm_count(), most16 = dc_div_up(tiles16, n_sm), most24 = dc_div_up(tiles24, n_sm);
  const int form = hidden < 320 ? 0 : tiles16 <= n_sm ? 1 : most24 * 24 < most16 * 16 ? 2 : 0;
  const BlockArgs &b = tb.blk[0];
  const int run = hidden / (hidden < 320 ? 8 : 16);          // channels of a warp's sums, at least
  if (tb.n == 1 && block33_on_tensor_core(b.c0, b.c1, b.c2, run, most16, most24, form)) {
    status.note(dc_launch_merge_product_tc(kProductBlock, Product{b.l1, b.l2, b.l3, 0, 0, b.c0, b.c1, b.c2, b.w_out, b.b_out}, dv, run, status.ws, st));
    return;
  }
  if (form == 1) launch_block33_form<16, 16>(tb, dv, mg, st, status);
  else if (form == 2) launch_block33_form<24, 16>(tb, dv, mg, st, status);
  else launch_block33_form<16, 8>(tb, dv, mg, st, status);
}

// A 1x1 after a large dense kernel is a plain matrix product: the fp32 convolution's kernel runs it as a 1x1 layer whose
// pixels are the second layer's rows and whose weights are the first layer as stored (960 -> 320 -> 1280: 81 us with the
// gathered product, 59.9 us).  False: a shape outside that kernel's range, nothing was launched.
static bool compose_as_product(const Piece &first, const Piece &second, float *out, cudaStream_t st, MergeStatus &status) {
  const dc_geom g = {first.c_out, first.c_in * first.k * first.k, 1, 1, 1, 0};
  const dc_status s = dc_launch_conv_f32(second.w, 1, 1, second.c_out, &g, first.w, nullptr, DC_ACT_IDENTITY, nullptr, out, st);
  if (s == DC_ERR_UNSUPPORTED) return false;
  status.note(s);
  return true;
}

// Composes second o first into a new piece; launches when `go`.  With `dv`, the piece is the run's result: where the
// kernel can deliver it itself it goes to w_final / b_final (and the packed copy) and *delivered is set.
static Piece compose(const Piece &first, const Piece &second, Bump &bump, bool go, cudaStream_t st, MergeStatus &status,
                     const BlockDelivery *dv = nullptr, const dc_geom *mg = nullptr, float *w_final = nullptr,
                     float *b_final = nullptr, bool *delivered = nullptr) {
  Piece out;
  out.c_in = first.c_in; out.c_out = second.c_out;
  out.k = first.k + (second.k - 1) * first.stride;
  out.stride = first.stride * second.stride;
  out.diag = first.diag && second.diag;
  out.ident = 0;
  size_t elems = piece_elems(out.c_in, out.c_out, out.k, out.diag);
  float *w = bump.take(elems);
  float *b = bump.take(out.c_out);
  out.w = w; out.b = b;
  if (go) {
    const int nbias = bias_blocks(out.c_out, 256);
    if (!first.diag && !second.diag && compose33_ok(first.c_in, first.c_out, first.k, first.stride, second.k)) {
      auto operand = [](const Piece &p) { return Operand33{RawLayer{p.w, p.b, nullptr, nullptr, nullptr, nullptr, 0.f}, p.ident}; };
      BlockDelivery piece{nullptr, -1, 0, KOrder{}};
      if (dv) { out.w = w = w_final; out.b = b = b_final; *delivered = true; }
      launch_compose33(operand(first), operand(second), first.c_in, first.c_out, second.c_out, w, b, dv ? *dv : piece,
                       mg ? *mg : dc_geom{}, st, status);
    } else if (dv && !first.diag && second.diag && first.k == 3 && first.stride == 1 && second.k == 3) {
      const int gi = dc_div_up(first.c_in, kDwI), tiles = gi * dc_div_up(second.c_out, kDwO);
      out.w = w_final; out.b = b_final; *delivered = true;
      status.note(dc_launch_pdl(k_compose_dw33, dim3(tiles + zero_ctas(*dv, *mg, kDwThreads)), dim3(kDwThreads), 0, st, first, second, w_final, b_final, *dv, gi, tiles));
    } else if (!first.diag && !second.diag && first.k == 1 && first.stride == 1 && second.k == 3 && first.c_in % 4 == 0 &&
               first.c_out % 4 == 0 && first.c_out >= 32) {
      // From 32 intermediate channels on, a whole slice (96 -> 24 -> 24 inside a longer run took 2.3 us more here).
      After11 a{first, second, w, b, dc_div_up(first.c_in, kA1I), dc_div_up(second.c_out, kA1O)};
      BlockDelivery piece{nullptr, -1, 0, KOrder{}};
      if (dv) { out.w = a.w_out = w_final; out.b = a.b_out = b_final; *delivered = true; piece = *dv; }
      static unsigned char attr_done[kDcMaxDevices];
      status.note(dc_set_max_smem_once(k_compose_after_11, kA1Smem, attr_done));
      status.note(dc_launch_pdl(k_compose_after_11, dim3(a.gi * a.go + a.go + zero_ctas(piece, mg ? *mg : dc_geom{}, 256)), dim3(256), kA1Smem, st, a, piece));
    } else if (!first.diag && !second.diag && first.k == 1 && first.stride == 1 && second.k > 1 &&
        first.c_out * second.k * second.k <= kAfter1x1MaxFloats) {
      dim3 grid(dc_div_up(out.c_in * out.k * out.k, 256), out.c_out + 1);
      if ((int)grid.x < nbias) grid.x = nbias;
      k_compose_after_1x1<<<grid, 256, 0, st>>>(first, second, w, b);
    } else if (!first.diag && !second.diag && elems <= (size_t)200000 && second.k <= 7) {
      const int gx = dc_div_up(out.c_in * out.k * out.k, 32), gy = dc_div_up(out.c_out, 8);
      k_compose_dd_small<<<gx * gy + nbias, 256, 0, st>>>(first, second, w, b, out.k, gx, gy);
    } else if (!first.diag && !second.diag && second.k == 1 && !first.ident && !second.ident &&
               compose_as_product(first, second, w, st, status)) {
      k_compose_bias<<<nbias, 256, 0, st>>>(first, second, b);
    } else if (!first.diag && !second.diag) {
      // 128 x 64 tiles when they still give every SM two tiles, 64 x 64 otherwise
      const int gx = dc_div_up(out.c_in * out.k * out.k, 64);
      const int gy8 = dc_div_up(out.c_out, 128), gy4 = dc_div_up(out.c_out, 64);
      if (gx * gy8 >= 2 * dc_sm_count())
        k_compose_dd_tiled<8><<<gx * gy8 + nbias, 256, 0, st>>>(first, second, w, b, out.k, gx, gy8);
      else
        k_compose_dd_tiled<4><<<gx * gy4 + nbias, 256, 0, st>>>(first, second, w, b, out.k, gx, gy4);
    } else {
      const int nb = blocks_for(elems, 256);
      k_compose_diag<<<nb + nbias, 256, 0, st>>>(first, second, w, b, out.k, (int)elems, nb);
    }
    status.launched();
  }
  return out;
}

// Index of the skip group that contains layer idx, or -1.
static int group_of(const dc_residual *res, int n_res, int idx) {
  for (int i = 0; i < n_res; ++i)
    if (res[i].first <= idx && idx <= res[i].last) return i;
  return -1;
}

// How the block that starts at layer i is merged: kTiledBlock by k_merge_block33, a positive number by k_merge_block
// (hidden channels it stages per pass), 0: the layers are no such block.
constexpr int kTiledBlock = -1;
static int block_chunk(const dc_layer *L, int n, const dc_residual *res, int n_res, int i) {
  if (i + 2 >= n) return 0;
  const dc_layer &e = L[i], &d = L[i + 1], &p = L[i + 2];
  if (e.groups != 1 || e.k != 1 || e.stride != 1 || e.pad != 0) return 0;
  if (d.groups == 1 || d.groups != d.c_in) return 0;
  if (p.groups != 1 || p.k != 1 || p.stride != 1 || p.pad != 0) return 0;
  const int g0 = group_of(res, n_res, i), g1 = group_of(res, n_res, i + 1), g2 = group_of(res, n_res, i + 2);
  const bool whole = g0 >= 0 && g0 == g1 && g1 == g2 && res[g0].first == i && res[g0].last == i + 2;
  if (!whole && (g0 >= 0 || g1 >= 0 || g2 >= 0)) return 0;
  // 16-byte pieces of every operand; the bias blocks hold one float per hidden channel where the operand rings lie
  if (d.k == 3 && e.c_in % 4 == 0 && e.c_out % 4 == 0 && e.c_out <= kMbRing / 4) return kTiledBlock;
  if (e.c_in * d.k * d.k > kBlockThreads * kBlockMaxPerThread) return 0;
  // wide blocks of other kernel sizes are faster step by step: their compositions fill the GPU, one CTA per output
  // channel does not
  if ((long)e.c_out * e.c_in * d.k * d.k > 150000) return 0;
  const int per = e.c_in + d.k * d.k + 1;
  int ch = (200 * 1024 / 4) / per;
  if (ch > e.c_out) ch = e.c_out;
  return ch >= 32 || ch == e.c_out ? ch : 0;
}

static RawLayer raw_of(const dc_layer &L) {
  return RawLayer{L.weight, L.bias, L.bn_gamma, L.bn_beta, L.bn_mean, L.bn_var, L.bn_eps};
}

// True when an output of the merge shares memory with an array of its layers.  The kernels that merge and deliver in one
// launch write the result while other CTAs still read the layers, so such a merge goes through the workspace and delivers in
// a launch behind them.
static bool writes_into_layers(const dc_layer *layers, int n, const float *w, size_t w_bytes, const float *b, size_t b_bytes,
                               const void *packed, size_t packed_bytes) {
  auto shares = [](const void *p, size_t np, const void *q, size_t nq) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(p), c = reinterpret_cast<uintptr_t>(q);
    return p && q && a < c + nq && c < a + np;
  };
  for (int i = 0; i < n; ++i) {
    const dc_layer &L = layers[i];
    const size_t per_channel = (size_t)L.c_out * sizeof(float);
    const void *arr[6] = {L.weight, L.bias, L.bn_gamma, L.bn_beta, L.bn_mean, L.bn_var};
    for (int j = 0; j < 6; ++j) {
      const size_t bytes = j == 0 ? piece_elems(L.c_in, L.c_out, L.k, L.groups != 1) * sizeof(float) : per_channel;
      if (shares(arr[j], bytes, w, w_bytes) || shares(arr[j], bytes, b, b_bytes) || shares(arr[j], bytes, packed, packed_bytes)) return true;
    }
  }
  return false;
}

// One walk drives both the size query (go == false: nothing is dereferenced or launched) and the
// launches (go == true: the caller has already checked workspace_bytes against the query).
static dc_status merge_walk(const dc_layer *layers, int n, const dc_residual *res, int n_res,
                            float *w_merged, float *b_merged, void *w_packed, dc_dtype packed_dtype,
                            void *workspace, cudaStream_t st, bool go, dc_geom *merged, size_t *need,
                            dc_merge_algo algo = DC_MERGE_AUTO, DcWsHeader *ws = nullptr) {
  dc_geom mg;
  dc_status s = check_chain(layers, n, res, n_res, &mg);
  if (s != DC_OK) return s;
  if (merged) *merged = mg;
  Bump bump{go ? (char *)workspace : nullptr, 0};
  MergeStatus status;
  status.ws = ws;

  // What the last launch delivers.  A run that is one block of the tiled kind, or two dense 3x3 layers, needs no launch of
  // its own for that (nor, in the second case, for the BN): the kernel that merges it reads the layers as they are and
  // writes the result and the packed copy (a chunk of which is 8 input channels).
  const size_t elems = (size_t)mg.c_out * mg.c_in * mg.k * mg.k;
  KOrder ko;
  dc_korder_init(&ko, &mg);
  const int mode = !w_packed ? 0 : (packed_dtype == DC_F32 ? 1 : 2);
  if (go && !dc_aligned16(w_packed)) return DC_ERR_ALIGNMENT;
  const bool can_pack = mode != 2 || mg.c_in % 8 == 0;
  const size_t p_bytes = mode == 2 ? (size_t)ko.ng * ko.e_pad * ko.n_pad * 16 : elems * sizeof(float);
  const bool direct = go && n <= 3 && algo != DC_MERGE_STEPS && can_pack &&
                      !writes_into_layers(layers, n, w_merged, elems * sizeof(float), b_merged, mg.c_out * sizeof(float), w_packed, p_bytes);
  if (direct && n == 2 && layers[0].groups == 1 && layers[1].groups == 1 &&
      compose33_ok(layers[0].c_in, layers[0].c_out, layers[0].k, layers[0].stride, layers[1].k)) {
    int id[2] = {0, 0}, whole = 0;
    for (int g = 0; g < n_res; ++g) {
      if (res[g].first != res[g].last) whole = 1;
      else id[res[g].first] = 1;
    }
    launch_compose33(Operand33{raw_of(layers[0]), id[0]}, Operand33{raw_of(layers[1]), id[1]}, mg.c_in, layers[0].c_out, mg.c_out,
                     w_merged, b_merged, BlockDelivery{w_packed, mode, whole, ko}, mg, st, status);
    return status.s;
  }

  if (direct && n == 2) {
    const dc_layer &l1 = layers[0], &l2 = layers[1];
    const bool dw_first = l1.groups != 1;
    const dc_layer &de = dw_first ? l2 : l1, &dw = dw_first ? l1 : l2;
    if (de.groups == 1 && de.k == 1 && dw.groups != 1 && dw.k == 3 && (dw_first || de.stride == 1)) {
      int id[2] = {0, 0}, whole = 0;
      for (int g = 0; g < n_res; ++g) {
        if (res[g].first != res[g].last) whole = 1;
        else id[res[g].first] = 1;
      }
      Outer33 a{raw_of(de), raw_of(dw), id[dw_first ? 1 : 0], id[dw_first ? 0 : 1], dw_first ? 1 : 0, mg.c_in, mg.c_out,
                      w_merged, b_merged, 0, dc_div_up(mg.c_out, kMbO)};
      const BlockDelivery dv{w_packed, mode, whole, ko};
      const int n_sm = dc_sm_count(), zero = zero_ctas(dv, mg, kMbThreads);
      if (a.go * dc_div_up(mg.c_in, 64) >= 2 * n_sm) launch_outer33<64>(a, dv, zero, st, status);
      else if (a.go * dc_div_up(mg.c_in, 32) >= 2 * n_sm) launch_outer33<32>(a, dv, zero, st, status);
      else launch_outer33<16>(a, dv, zero, st, status);
      return status.s;
    }
  }

  if (direct && n == 2 && layers[0].groups == 1 && layers[1].groups == 1 && layers[0].k == 1 && layers[1].k == 1 &&
      layers[0].stride == 1 && layers[0].c_in % 4 == 0 && layers[0].c_out % 4 == 0) {
    int id[2] = {0, 0}, whole = 0;
    for (int g = 0; g < n_res; ++g) {
      if (res[g].first != res[g].last) whole = 1;
      else id[res[g].first] = 1;
    }
    Merge11 a{raw_of(layers[0]), raw_of(layers[1]), id[0], id[1], mg.c_in, layers[0].c_out, mg.c_out, w_merged, b_merged, 0, 0};
    const BlockDelivery dv{w_packed, mode, whole, ko};
    // 32 x 32 until tiles of 64 columns give most SMs one; of those the height that leaves the SM with the most tiles the least
    // (960 -> 320 -> 1280: 300 tiles of 64 x 64 are three on four SMs and two on the others, 45.9 us)
    const int n_sm = dc_sm_count(), wide[2] = {64, 48};
    int bo = 32, bi = 32;
    if (dc_div_up(a.c2, 64) * dc_div_up(a.c0, 64) >= 100) {
      bi = 64;
      long long best = 0;
      for (int h : wide) {
        const long long rows = (long long)dc_div_up(dc_div_up(a.c2, h) * dc_div_up(a.c0, 64), n_sm) * h;
        if (bo == 32 || rows < best) { best = rows; bo = h; }
      }
    }
    a.gi = dc_div_up(a.c0, bi);
    a.go = dc_div_up(a.c2, bo);
    // The tensor core by estimates as well: of 57 drawn pairs of 40 to 1280 channels 29, in 0.63 of the time on (geometric) average, none
    // slower.  960 -> 320 -> 1280 30.5 us here and 22.0 there, 320 -> 1280 -> 320 24.9 and 14.3, 1024 -> 256 -> 1024 30.9 and 17.7.
    const int most = dc_div_up(a.gi * a.go, n_sm), run = a.c1 / 4;           // channels of a group's sums, at most half of them
    const double fma = bo == 64   ? 4.82 + a.c1 * (0.0185 * most + 0.0705 * dc_div_up(most, 3))
                       : bo == 48 ? 5.2 + a.c1 * (0.0072 * most + 0.06 * dc_div_up(most, 3))
                                  : 3.07 + a.c1 * (0.0136 * most + 0.0023 * dc_div_up(most, 3));
    const double tc = dc_merge_product_tc_us(kProductPair, a.c0, a.c1, a.c2, run);
    if (tc != 0.0 && tc < 0.95 * fma) {
      status.note(dc_launch_merge_product_tc(kProductPair, Product{a.l1, RawLayer{}, a.l2, a.ident1, a.ident2, a.c0, a.c1, a.c2, a.w_out, a.b_out}, dv, run, status.ws, st));
      return status.s;
    }
    const dim3 grid(a.gi * a.go + dc_div_up(a.c2, 8) + zero_ctas(dv, mg, 256));
    if (bo == 64) status.note(dc_launch_pdl(k_merge_11<64, 64, 8, 2>, grid, dim3(256), 0, st, a, dv));
    else if (bo == 48) status.note(dc_launch_pdl(k_merge_11<48, 64, 6, 2>, grid, dim3(256), 0, st, a, dv));
    else status.note(dc_launch_pdl(k_merge_11<32, 32, 4, 4>, grid, dim3(256), 0, st, a, dv));
    status.launched();
    return status.s;
  }

  // 0. inverted-residual blocks (1x1, depthwise, 1x1) are merged in one step from the raw layers
  std::vector<int> chunk_at(n, 0), covered(n, 0);
  if (algo != DC_MERGE_STEPS)
    for (int i = 0; i + 2 < n;) {
      const int ch = block_chunk(layers, n, res, n_res, i);
      if (ch != 0) { chunk_at[i] = ch; covered[i] = covered[i + 1] = covered[i + 2] = 1; i += 3; }
      else ++i;
    }

  // 1. fold every other layer
  std::vector<Piece> folded(n);
  {
    FoldTable t;
    int cnt = 0;
    size_t max_total = 1;
    auto flush = [&]() {
      if (cnt == 0) return;
      t.n = cnt;
      if (go) {
        int bx = blocks_for(max_total, 256);
        dim3 grid(bx > 1024 ? 1024 : bx, cnt);       // a few elements per thread: the launch is short beside its chain
        k_fold_bn<<<grid, 256, 0, st>>>(t);
        status.launched();
      }
      cnt = 0;
      max_total = 1;
    };
    for (int l = 0; l < n; ++l) {
      if (covered[l]) continue;
      const dc_layer &L = layers[l];
      int diag = L.groups != 1;
      size_t elems = piece_elems(L.c_in, L.c_out, L.k, diag);
      float *w = bump.take(elems), *b = bump.take(L.c_out);
      t.w[cnt] = L.weight; t.b[cnt] = L.bias; t.gamma[cnt] = L.bn_gamma; t.beta[cnt] = L.bn_beta;
      t.mean[cnt] = L.bn_mean; t.var[cnt] = L.bn_var; t.eps[cnt] = L.bn_eps;
      t.w_out[cnt] = w; t.b_out[cnt] = b;
      t.c_out[cnt] = L.c_out; t.per_out[cnt] = (int)(elems / L.c_out);
      if (elems > max_total) max_total = elems;
      folded[l] = Piece{w, b, L.c_in, L.c_out, L.k, L.stride, diag, 0};
      if (++cnt == DC_FOLD_MAX) flush();
    }
    flush();
  }

  const bool at_once = direct && n == 3 && chunk_at[0] == kTiledBlock;

  // 2. compose: blocks and skip groups first (with their identity tap), then left to right
  BlockBatch batch;
  int n_batch = 0, batch_grid = 0;
  size_t batch_smem = 0;
  TiledBlocks tiled;
  tiled.n = 0;
  tiled.first[0] = 0;
  BlockDelivery dv{nullptr, -1, 0, ko};
  bool delivered = false;
  auto flush_tiled = [&]() {
    if (tiled.n == 0) return;
    launch_block33(tiled, dv, mg, st, status);
    tiled.n = 0;
  };
  auto flush_blocks = [&]() {
    flush_tiled();
    if (n_batch == 0) return;
    static unsigned char attr_done[kDcMaxDevices];
    status.note(dc_set_max_smem_once(k_merge_block, 200 * 1024, attr_done));
    k_merge_block<<<dim3(batch_grid, n_batch), kBlockThreads, batch_smem, st>>>(batch);
    status.launched();
    n_batch = 0; batch_grid = 0; batch_smem = 0;
  };
  Piece acc{};
  bool have = false;
  int i = 0;
  while (i < n) {
    Piece piece;
    int gi = find_group(res, n_res, i);
    if (chunk_at[i] != 0) {
      const dc_layer &e = layers[i], &d = layers[i + 1], &p = layers[i + 2];
      piece = Piece{nullptr, nullptr, e.c_in, p.c_out, d.k, d.stride, 0, gi >= 0 ? 1 : 0};
      float *w = bump.take(piece_elems(piece.c_in, piece.c_out, piece.k, 0));
      float *b = bump.take(piece.c_out);
      if (at_once) {
        w = w_merged; b = b_merged;
        dv.packed = w_packed; dv.mode = mode; dv.ident = piece.ident;
      }
      piece.w = w; piece.b = b;
      if (go && chunk_at[i] == kTiledBlock) {
        const int t = tiled.n++;
        tiled.blk[t] = BlockArgs{raw_of(e), raw_of(d), raw_of(p), e.c_in, e.c_out, p.c_out, d.k, 0, w, b};
        if (tiled.n == kBlockBatch) flush_tiled();
      } else if (go) {
        batch.blk[n_batch] = BlockArgs{raw_of(e), raw_of(d), raw_of(p), e.c_in, e.c_out, p.c_out, d.k, chunk_at[i], w, b};
        const size_t smem = (size_t)chunk_at[i] * (e.c_in + d.k * d.k + 1) * sizeof(float);
        if (smem > batch_smem) batch_smem = smem;
        if (p.c_out > batch_grid) batch_grid = p.c_out;
        // the blocks read raw layers only: hold the launch until the batch is full or a composition
        // needs one of its pieces
        if (++n_batch == kBlockBatch) flush_blocks();
      }
      i += 3;
    } else if (gi < 0) {
      piece = folded[i];
      ++i;
    } else {
      piece = folded[res[gi].first];
      if (go) flush_blocks();
      for (int j = res[gi].first + 1; j <= res[gi].last; ++j) piece = compose(piece, folded[j], bump, go, st, status);
      piece.ident = 1;          // f(x) + x: the identity kernel rides along as a flag
      i = res[gi].last + 1;
    }
    if (!have) { acc = piece; have = true; }
    else {
      if (go) flush_blocks();
      // the run's last composition: piece.ident is the second operand's, the result carries none
      const BlockDelivery fin{w_packed, mode, 0, ko};
      const bool last = i == n && go && can_pack;
      acc = compose(acc, piece, bump, go, st, status, last ? &fin : nullptr, &mg, w_merged, b_merged, &delivered);
    }
  }
  if (need) *need = bump.off + 256;
  if (!go) return DC_OK;
  flush_blocks();

  if (at_once || delivered) return status.s;

  // 3. deliver: dense fp32 result, bias, optional packed copy, in one launch
  const size_t p_elems = mode == 2 ? (size_t)ko.ng * ko.e_pad * ko.n_pad * 8 : elems;
  const int chunked = mode == 2 && p_elems >= (size_t)262144;
  const int nb_w = blocks_for(elems, 256), nb_p = mode ? blocks_for(chunked ? p_elems / 8 : p_elems, 256) : 0;
  k_deliver<<<nb_w + 1 + nb_p, 256, 0, st>>>(acc, w_merged, b_merged, w_packed, mode, ko, nb_w, nb_p, chunked);
  status.launched();
  return status.s;
}

// Workspace bytes that cover either launch form.
static dc_status merge_need(const dc_layer *layers, int n, const dc_residual *res, int n_res, dc_geom *merged,
                            size_t *need) {
  size_t a = 0, b = 0;
  dc_status s = merge_walk(layers, n, res, n_res, nullptr, nullptr, nullptr, DC_F32, nullptr, nullptr, false, merged,
                           &a, DC_MERGE_AUTO);
  if (s != DC_OK) return s;
  s = merge_walk(layers, n, res, n_res, nullptr, nullptr, nullptr, DC_F32, nullptr, nullptr, false, nullptr, &b,
                 DC_MERGE_STEPS);
  if (s != DC_OK) return s;
  if (need) *need = a > b ? a : b;
  return DC_OK;
}

// ----------------------------------------------------------------------------------------------
// exported
// ----------------------------------------------------------------------------------------------

extern "C" dc_status dc_fold_bn(const dc_layer *layer, float *w_out, float *b_out, dc_stream stream) {
  if (!layer || !w_out || !b_out) return DC_ERR_INVALID_ARG;
  dc_status s = validate_layer(layer);
  if (s != DC_OK) return s;
  if (!dc_aligned16(layer->weight) || !dc_aligned16(w_out) || !dc_aligned16(b_out)) return DC_ERR_ALIGNMENT;
  FoldTable t;
  t.n = 1;
  size_t elems = piece_elems(layer->c_in, layer->c_out, layer->k, layer->groups != 1);
  t.w[0] = layer->weight; t.b[0] = layer->bias; t.gamma[0] = layer->bn_gamma; t.beta[0] = layer->bn_beta;
  t.mean[0] = layer->bn_mean; t.var[0] = layer->bn_var; t.eps[0] = layer->bn_eps;
  t.w_out[0] = w_out; t.b_out[0] = b_out; t.c_out[0] = layer->c_out; t.per_out[0] = (int)(elems / layer->c_out);
  int bx = blocks_for(elems, 256);
  dim3 grid(bx > 256 ? 256 : bx, 1);
  k_fold_bn<<<grid, 256, 0, (cudaStream_t)stream>>>(t);
  return cudaGetLastError() == cudaSuccess ? DC_OK : DC_ERR_CUDA;
}

extern "C" dc_status dc_merge_query(const dc_layer *layers, int n_layers, const dc_residual *res, int n_res,
                                    dc_geom *merged, size_t *workspace_bytes) {
  return merge_need(layers, n_layers, res, n_res, merged, workspace_bytes);
}

dc_status dc_merge_chain_ws(const dc_layer *layers, int n_layers, const dc_residual *res, int n_res, float *w_merged, float *b_merged,
                            void *w_packed, dc_dtype packed_dtype, void *workspace, size_t workspace_bytes, dc_stream stream,
                            dc_merge_algo algo, DcWsHeader *ws) {
  if (!w_merged || !b_merged) return DC_ERR_INVALID_ARG;
  if (packed_dtype != DC_F32 && packed_dtype != DC_BF16) return DC_ERR_INVALID_ARG;
  if (algo != DC_MERGE_AUTO && algo != DC_MERGE_STEPS) return DC_ERR_INVALID_ARG;
  size_t need = 0;
  dc_status s = merge_need(layers, n_layers, res, n_res, nullptr, &need);
  if (s != DC_OK) return s;
  if (!workspace || workspace_bytes < need) return DC_ERR_WORKSPACE;
  if (!dc_aligned16(w_merged) || !dc_aligned16(b_merged) || !dc_aligned16(workspace) ||
      (w_packed && !dc_aligned16(w_packed)))
    return DC_ERR_ALIGNMENT;
  for (int i = 0; i < n_layers; ++i)
    if (!dc_aligned16(layers[i].weight)) return DC_ERR_ALIGNMENT;
  return merge_walk(layers, n_layers, res, n_res, w_merged, b_merged, w_packed, packed_dtype, workspace,
                    (cudaStream_t)stream, true, nullptr, nullptr, algo, ws);
}

extern "C" dc_status dc_merge_chain_algo(const dc_layer *layers, int n_layers, const dc_residual *res, int n_res,
                                         float *w_merged, float *b_merged, void *w_packed, dc_dtype packed_dtype,
                                         void *workspace, size_t workspace_bytes, dc_stream stream,
                                         dc_merge_algo algo) {
  return dc_merge_chain_ws(layers, n_layers, res, n_res, w_merged, b_merged, w_packed, packed_dtype, workspace, workspace_bytes, stream, algo,
                           nullptr);
}

extern "C" dc_status dc_merge_chain(const dc_layer *layers, int n_layers, const dc_residual *res, int n_res,
                                    float *w_merged, float *b_merged, void *w_packed, dc_dtype packed_dtype,
                                    void *workspace, size_t workspace_bytes, dc_stream stream) {
  return dc_merge_chain_algo(layers, n_layers, res, n_res, w_merged, b_merged, w_packed, packed_dtype, workspace,
                             workspace_bytes, stream, DC_MERGE_AUTO);
}

extern "C" dc_status dc_packed_bytes(const dc_geom *g, dc_dtype dtype, size_t *bytes) {
  dc_status s = dc_validate_geom(g);
  if (s != DC_OK) return s;
  if (!bytes || (dtype != DC_F32 && dtype != DC_BF16)) return DC_ERR_INVALID_ARG;
  if (g->groups != 1) { *bytes = (size_t)g->c_out * g->k * g->k * sizeof(float); return DC_OK; }
  if (dtype == DC_F32) { *bytes = (size_t)g->c_out * g->c_in * g->k * g->k * sizeof(float); return DC_OK; }
  KOrder ko;
  dc_korder_init(&ko, g);
  *bytes = (size_t)ko.ng * ko.e_pad * ko.n_pad * 8 * sizeof(__nv_bfloat16);
  return DC_OK;
}

extern "C" dc_status dc_pack_weights(const float *w, const dc_geom *g, dc_dtype dtype, void *w_packed,
                                     dc_stream stream) {
  dc_status s = dc_validate_geom(g);
  if (s != DC_OK) return s;
  if (!w || !w_packed || (dtype != DC_F32 && dtype != DC_BF16)) return DC_ERR_INVALID_ARG;
  if (!dc_aligned16(w) || !dc_aligned16(w_packed)) return DC_ERR_ALIGNMENT;
  cudaStream_t st = (cudaStream_t)stream;
  if (g->groups != 1) {
    size_t total = (size_t)g->c_out * g->k * g->k;
    k_pack_dw<<<blocks_for(total, 256), 256, 0, st>>>(w, (float *)w_packed, g->c_out, g->k);
  } else if (dtype == DC_F32) {
    size_t total = (size_t)g->c_out * g->c_in * g->k * g->k;
    k_pack_f32<<<blocks_for(total, 256), 256, 0, st>>>(w, (float *)w_packed, g->c_out, g->c_in, g->k);
  } else {
    KOrder ko;
    dc_korder_init(&ko, g);
    size_t total = (size_t)ko.ng * ko.e_pad * ko.n_pad * 8;
    k_pack_bf16<<<blocks_for(total, 256), 256, 0, st>>>(w, (__nv_bfloat16 *)w_packed, g->c_out, ko);
  }
  return cudaGetLastError() == cudaSuccess ? DC_OK : DC_ERR_CUDA;
}

// ----------------------------------------------------------------------------------------------
// Merge without any caller-provided or allocated scratch memory.
//
// Some callers cannot allocate device memory at the point where they merge: code running inside a
// memory-pool or allocator callback, a plug-in whose host forbids allocation calls after
// initialisation, or a process that has handed the whole GPU to another allocator.  For them the
// intermediate kernels of the merge live in a fixed array that is part of the library image: every
// GPU that loads the library holds these bytes until the process exits.
// ----------------------------------------------------------------------------------------------
#define DC_STATIC_SCRATCH_BYTES (4u << 20)
static __device__ __align__(256) unsigned char g_merge_scratch[DC_STATIC_SCRATCH_BYTES];

// In host code the symbol above is only a handle; the device address is looked up once per device.
#define DC_MAX_DEVICES 64
static void *g_merge_scratch_addr[DC_MAX_DEVICES];

extern "C" size_t dc_merge_chain_static_capacity(void) { return (size_t)DC_STATIC_SCRATCH_BYTES; }

extern "C" dc_status dc_merge_chain_static(const dc_layer *layers, int n_layers, const dc_residual *res, int n_res,
                                           float *w_merged, float *b_merged, void *w_packed,
                                           dc_dtype packed_dtype, dc_stream stream) {
  if (!w_merged || !b_merged) return DC_ERR_INVALID_ARG;
  if (packed_dtype != DC_F32 && packed_dtype != DC_BF16) return DC_ERR_INVALID_ARG;
  size_t need = 0;
  dc_status s = merge_need(layers, n_layers, res, n_res, nullptr, &need);
  if (s != DC_OK) return s;
  if (need > (size_t)DC_STATIC_SCRATCH_BYTES) return DC_ERR_WORKSPACE;   // run too large for the built-in scratch
  if (!dc_aligned16(w_merged) || !dc_aligned16(b_merged) || (w_packed && !dc_aligned16(w_packed)))
    return DC_ERR_ALIGNMENT;
  for (int i = 0; i < n_layers; ++i)
    if (!dc_aligned16(layers[i].weight)) return DC_ERR_ALIGNMENT;
  int dev = -1;
  DC_CUDA_OK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= DC_MAX_DEVICES) return DC_ERR_UNSUPPORTED;
  if (!g_merge_scratch_addr[dev]) {
    // first call on this device (with that device current): resolve the array's device address
    void *ptr = nullptr;
    DC_CUDA_OK(cudaGetSymbolAddress(&ptr, g_merge_scratch));
    if (!ptr) return DC_ERR_CUDA;
    g_merge_scratch_addr[dev] = ptr;
  }
  // Nothing in the scratch has to start at zero: every intermediate is written in full before it
  // is read, so the contents a previous call left behind are simply overwritten.
  return merge_walk(layers, n_layers, res, n_res, w_merged, b_merged, w_packed, packed_dtype,
                    g_merge_scratch_addr[dev], (cudaStream_t)stream, true, nullptr, nullptr);
}
