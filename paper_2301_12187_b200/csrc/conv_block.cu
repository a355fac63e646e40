// An unmerged inverted-residual block (bf16: 1x1 expansion, ReLU6, 3x3 depthwise, ReLU6, 1x1 projection, skip input) as
// one kernel: the hidden map, six times as wide as the block's input and output, never leaves the SM.
//
// As three launches (the rows kernel, the depthwise stencil, the rows kernel) the hidden map is written and read twice
// through L2 or HBM, and each launch is a chain of its own of load, arithmetic and store.  Here a CTA owns a tile of
// output pixels (rows x columns x images) and walks the hidden channels in chunks of at most 64:
//
//   expand    H = relu6(X W1 + b1) of the tile's haloed patch: X, the patch's input channels, is brought in once per tile by
//             TMA in planes of 64 channels (128-byte swizzle, zeros outside the image); GEMM rows are patch pixels, at
//             most four 128-row blocks; accumulators in tensor memory
//   convert   tensor memory -> ReLU6 -> bf16 -> shared memory [pixel][64 channels], 144-byte pitch (16-byte stores of
//             neighbouring pixels and 8-byte reads along a pixel are both conflict-free); zero outside the image, which
//             is the padding that the depthwise layer sees
//   depthwise 16 warps, a thread owns TX neighbouring outputs of a row x 4 channels; packed fp32 FMAs; ReLU6 -> bf16
//             -> shared memory as the projection's A operand (128-byte swizzled lines of an output pixel)
//   project   accumulated over the chunks in tensor memory
//
// so the tensor core works on the next chunk's expansion while the warps are at this chunk's stencil.  The roundings are
// those of the three launches: hidden maps to bf16 after their ReLU6, everything else in fp32.
//
// What bounds it is a chunk's chain in a group of warps: its accumulators, their way out of tensor memory, conversion, a barrier,
// the stencil, the hand-over.  Half of the cycles issue nothing (64 -> 384 -> 64, 128 images of 14 x 14: issue slots 48 % taken,
// FMA pipe 19 %, the largest stall is on what memory returns), and of the 11.8 thousand warp instructions of a chunk the stencil,
// 4.5 packed FMAs and 7 others per hidden value, has 4.5.  That block takes 20.2 us, 25.1 as three launches; one image 9.4 and
// 10.1; 24 -> 144 -> 24, 64 images of 56 x 56 60 and 111; 16 -> 96 -> 16, 20 images of 9 x 9 6.4 and 13.9.  Measured and not kept:
// two rows of outputs per thread (fewer instructions, but more than the 96 registers that 19 warps leave: 10 % slower), both
// products issued by one warp, a bulk copy for every 8-channel chunk of the weights (80 cycles each to issue: 3 us a chunk of
// hidden channels).
//
// Roles (608 threads): warp 0 loads (a chunk's weights, several stages ahead), warps 1 and 2 issue the tensor-core
// instructions of the two products, warps 3-18 convert, run the stencil and read out.  All waits are bounded
// (tc::mbar_wait); a warp whose wait ran out goes on through the barriers without working.
#include <math.h>

#include "tc_ptx.cuh"

namespace {
using namespace tc;

constexpr int kMathWarps = 16;
constexpr int kMathThreads = kMathWarps * 32;
constexpr int kFirstMathWarp = 3;
constexpr int kThreads = (kFirstMathWarp + kMathWarps) * 32;
constexpr int kBarMath = 1, kBarTmem = 3;        // named barriers: each group of working warps; all of them and the issuing warps
constexpr int kHPitch = 144;                     // bytes per pixel of a hidden chunk in shared memory
constexpr int kMaxE = 4;                         // 128-row blocks of the patch
constexpr int kMaxW = 4;                         // weight stages

// Forms of the kernel: outputs of a row that a thread computes together (few for tiles that would otherwise leave warps
// without work), and groups of working warps.
constexpr int kForms = 4;
constexpr int kTx[2][kForms] = {{7, 4, 7, 4}, {4, 2, 4, 2}};      // [stride - 1][form]
constexpr int kGroups[kForms] = {1, 1, 2, 2};

struct BlockParams {
  int n_img, h, w, ho, wo, c_in, c_mid, c_out, stride, residual;
  int tw, th, ni;              // output columns, rows and images of a tile
  int nxt, tiles_y, tiles;     // column strips, row tiles, tiles in all
  int wbox, rbox, lines_img, patch;     // patch columns, rows, pixels per image and in all
  int mbe, mbp;                // 128-row blocks of the patch and of the outputs
  int planes, ksteps;          // 64-channel planes and 16-channel steps of the input
  int ch, nch;                 // hidden channels of the widest chunk, chunks
  int npass, last_rows, chp, chl;       // passes of the packed expansion weights, rows of the last; channels per chunk, in the last pass
  int n3, pass3;               // rows of the packed projection weights, passes of them
  int form, tx, groups, strips;         // form of the kernel, its outputs per thread and groups of warps; groups of outputs in a tile's row
  int nt1, e1;                 // packed expansion weights: rows per pass, chunk planes per pass
  int nt3, e3;                 // packed projection weights: the same
  int np, nw;                  // buffers of the projection's operand, weight stages
  int h_bytes, p_bytes, w1_bytes, wd_bytes, w3_bytes;
  int off_bias, off_x, off_p, off_w1, off_wd, off_w3, off_h, smem_bytes;
  int tmem_cols;
  uint32_t inv_lines, inv_wbox, inv_th, inv_strips, inv_outs, inv_tw, inv_mbe, inv_mbp, inv_ncg[4];   // ceil(2^20 / .)
};

struct BlockShared {
  uint64_t x_full, x_empty, w1_full[kMaxW], w1_empty[kMaxW], w3_full[kMaxW], w3_empty[kMaxW];
  uint64_t e_full[2], e_empty[2], p_full[2], p_empty[2], y_full, y_empty;
  uint32_t tmem_base, abort;
};

__device__ __forceinline__ uint2 lds_u2(uint32_t a) {
  uint2 v;
  asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts_u2(uint32_t a, uint32_t x, uint32_t y) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ float4 lds_f4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}
// v / d for inv = ceil(2^20 / d), exact while v * d < 2^20
__device__ __forceinline__ int div20(int v, uint32_t inv) { return (int)(((uint32_t)v * inv) >> 20); }

// Walks the chunks of hidden channels: h0 .. h0 + n, each inside one pass of the packed expansion weights.  (By additions:
// with divisions this took a few hundred cycles of every role's chain per chunk.)
struct Chunks {
  int h0 = 0, n, pass = 0, o = 0;                // o: first channel within the pass
  __device__ __forceinline__ explicit Chunks(const BlockParams &p) { size(p); }
  __device__ __forceinline__ void size(const BlockParams &p) {
    const bool last = pass == p.npass - 1;
    const int left = (last ? p.last_rows : p.nt1) - o, per = last ? p.chl : p.chp;
    n = left < per ? left : per;
  }
  __device__ __forceinline__ void next(const BlockParams &p) {
    o += n;
    if (o >= p.nt1) { o = 0; ++pass; }
    h0 = pass * p.nt1 + o;
    size(p);
  }
};
// a ring of stages: index and the parity of its present use
struct Ring {
  int s = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ void next(int n) { if (++s == n) { s = 0; ph ^= 1u; } }
};

// The waits in front of a chunk's stencil, in their order.  `use` counts the CTA's chunks, s and ph are its weight stage and the
// parity of that stage's present use.  A barrier's wait tells two neighbouring phases apart and no more, so every phase
// but the last must be known to be over where a wait begins.  (On the host as well: a test walks them through every order of events.)
//
// p_full and p_empty alternate between two barriers also where one buffer takes every chunk: the chunk three back, whose phase
// comes before that of the chunk that the wait is for, is then one that the same group has waited for.  On one
// barrier it would be the group's own last chunk, which nobody has waited for, and a wait that finds its phase still open
// would return at once.
//
// The operand comes first: with an odd number of weight stages a group meets a stage every second round only, and has not
// waited for the round between.  But a free operand means that the chunk two back (with one buffer: the last one) is projected, which takes all
// weights up to its own, and the round between has those of a chunk no later than that: there are two stages at least.
enum : uint32_t { kOperandFree, kWeightsIn };
struct StencilOperand {
  uint32_t buffer, barrier, parity;              // where the chunk's result goes, its p_full and p_empty and their phase
  __host__ __device__ __forceinline__ StencilOperand(uint32_t use, uint32_t np)
      : buffer(np == 2 ? use & 1u : 0u), barrier(use & 1u), parity((use >> 1) & 1u) {}
};
#pragma nv_exec_check_disable
template <typename Wait>
__host__ __device__ __forceinline__ bool stencil_waits(uint32_t use, uint32_t np, uint32_t s, uint32_t ph, Wait wait) {
  const StencilOperand last(use - np, np);       // the chunk that had the buffer (before the first ones: the phase before a barrier's first)
  return wait(kOperandFree, last.barrier, last.parity) && wait(kWeightsIn, s, ph);
}

struct Tile {
  int img0, x0, y0;
  __device__ __forceinline__ Tile(const BlockParams &p, int t) {
    const int strip = t / p.tiles_y;
    y0 = (t - strip * p.tiles_y) * p.th;
    const int ig = strip / p.nxt;
    x0 = (strip - ig * p.nxt) * p.tw;
    img0 = ig * p.ni;
  }
};

template <int S, int TX, int G>
__global__ void __launch_bounds__(kThreads, 1)
k_block_tc(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w1,
           const __grid_constant__ CUtensorMap map_wd, const __grid_constant__ BlockParams p, const float *__restrict__ b1,
           const float *__restrict__ bd, const void *__restrict__ w3, const float *__restrict__ b3,
           const __nv_bfloat16 *__restrict__ x, __nv_bfloat16 *__restrict__ y, DcWsHeader *ws) {
  constexpr int NJ = (TX - 1) * S + 3, kGroupWarps = kMathWarps / G, kGroupThreads = kGroupWarps * 32;
  extern __shared__ __align__(1024) uint8_t smem_raw_base[];
  __shared__ __align__(8) BlockShared sh;
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw_base) + 1023) & ~uintptr_t(1023));
  const uint32_t sm = smem_u32(smem);
  const int warp = (int)threadIdx.x >> 5, lane = (int)threadIdx.x & 31;
  volatile uint32_t *abort_flag = &sh.abort;
  const int zero_rows = p.ch > p.n3 ? p.ch : p.n3;

  if (threadIdx.x == 0) {
    mbar_init(&sh.x_full, 1); mbar_init(&sh.x_empty, 1);
    for (int i = 0; i < kMaxW; ++i) {
      mbar_init(&sh.w1_full[i], 1); mbar_init(&sh.w1_empty[i], 1);
      mbar_init(&sh.w3_full[i], 1); mbar_init(&sh.w3_empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sh.p_full[i], kGroupWarps); mbar_init(&sh.p_empty[i], 1);
      mbar_init(&sh.e_full[i], 1); mbar_init(&sh.e_empty[i], kGroupWarps);
    }
    mbar_init(&sh.y_full, 1); mbar_init(&sh.y_empty, kMathWarps);
    sh.abort = 0;
    prefetch_tensormap(&map_x);
    prefetch_tensormap(&map_w1);
    prefetch_tensormap(&map_wd);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  dc_pdl_enter();                                // nothing above touched global memory; everything below may
  __syncthreads();

  if (warp == 0) {
    // ================================================================== loads
    Ring wr;
    uint32_t ph_x = 0;
    bool ok = true;
#pragma unroll 1
    for (int t = (int)blockIdx.x; t < p.tiles && ok; t += (int)gridDim.x) {
      const Tile q(p, t);
      ok = warp_wait(&sh.x_empty, ph_x ^ 1, abort_flag, ws, 0x10000u);
      if (!ok) break;
      ph_x ^= 1;
      if (lane == 0) {
        mbar_arrive_expect_tx(&sh.x_full, (uint32_t)(p.planes * p.patch * 128));
        for (int g = 0; g < p.planes; ++g)
          tma_load_4d(sm + (uint32_t)(p.off_x + g * p.mbe * 16384), &map_x, &sh.x_full, 64 * g, q.x0 * S - 1, q.y0 * S - 1, q.img0);
      }
      __syncwarp();
#pragma unroll 1
      for (Chunks c(p); c.pass < p.npass && c.n > 0 && ok; c.next(p), wr.next(p.nw)) {
        const int s = wr.s;
        // Few and large copies: a bulk copy takes about 80 cycles to issue, and one for every 8-channel chunk and tap (20 to
        // 46 of them) made a chunk of hidden channels cost 1.8 to 3 us whatever its arithmetic.  The expansion's weights
        // have a ring of their own, free again when the instructions that read them are done, long before the others.
        ok = warp_wait(&sh.w1_empty[s], wr.ph ^ 1, abort_flag, ws, 0x20000u | s);
        if (!ok) break;
        if (lane == 0) {
          mbar_arrive_expect_tx(&sh.w1_full[s], (uint32_t)p.w1_bytes);
          tma_load_2d(sm + (uint32_t)(p.off_w1 + s * p.w1_bytes), &map_w1, &sh.w1_full[s], 2 * c.o, c.pass * p.e1);
        }
        __syncwarp();
        ok = warp_wait(&sh.w3_empty[s], wr.ph ^ 1, abort_flag, ws, 0x21000u | s);
        if (!ok) break;
        if (lane == 0) {
          // projection: the planes of a pass are contiguous
          const uint32_t bytes = (uint32_t)((c.n >> 3) * p.nt3 * 16);
          mbar_arrive_expect_tx(&sh.w3_full[s], bytes * (uint32_t)p.pass3 + (uint32_t)(9 * p.ch * 4 + (bd ? c.n * 4 : 0)));
          tma_load_2d(sm + (uint32_t)(p.off_wd + s * p.wd_bytes), &map_wd, &sh.w3_full[s], c.h0, 0);
          if (bd) bulk_load(sm + (uint32_t)(p.off_wd + s * p.wd_bytes + 9 * p.ch * 4), bd + c.h0, (uint32_t)c.n * 4u, &sh.w3_full[s]);
          for (int ps = 0; ps < p.pass3; ++ps)
            bulk_load(sm + (uint32_t)(p.off_w3 + s * p.w3_bytes) + (uint32_t)ps * bytes,
                      reinterpret_cast<const char *>(w3) + ((size_t)ps * p.e3 + (c.h0 >> 3)) * p.nt3 * 16, bytes, &sh.w3_full[s]);
        }
        __syncwarp();
      }
    }
  } else {
    // ---- preparation
    if (warp == 1) {
      tmem_alloc(&sh.tmem_base, (uint32_t)p.tmem_cols);
      tmem_relinquish();
    } else if (warp >= kFirstMathWarp) {
      // constant operand and the biases as three bf16 terms, added by the tensor core (see tc::bias_terms)
      const int t0 = (int)threadIdx.x - kFirstMathWarp * 32;
      if (t0 < 64) reinterpret_cast<uint4 *>(smem)[t0] = (t0 & 7) == (t0 >> 3) ? bias_ones() : make_uint4(0u, 0u, 0u, 0u);
      uint4 *rows = reinterpret_cast<uint4 *>(smem + p.off_bias);
      for (int t = t0; t < p.c_mid + p.n3 + zero_rows; t += kMathThreads) {
        float b = 0.f;
        if (t < p.c_mid) { if (b1) b = b1[t]; }
        else if (t < p.c_mid + p.c_out) { if (b3) b = b3[t - p.c_mid]; }
        rows[t] = bias_terms(b);
      }
      if (!bd && t0 < p.nw * p.ch) {             // no depthwise bias: its row stays zero
        const int s = t0 / p.ch;
        reinterpret_cast<float *>(smem + p.off_wd + s * p.wd_bytes)[9 * p.ch + t0 - s * p.ch] = 0.f;
      }
      fence_proxy_async();
    }
    tc_fence_before();
    bar_sync(kBarTmem, kMathThreads + 64);
    tc_fence_after();
    const uint32_t tmem_e = sh.tmem_base, tmem_y = sh.tmem_base + (uint32_t)(G * p.mbe * p.ch);

    if (warp < kFirstMathWarp) {
      // ================================================================== tensor-core instructions
      // Two warps, so that neither product waits behind the other's barriers (with one, its chain of waits was as long as
      // the working warps' chunk).
      const bool leader = elect_one();
      const uint32_t b_hi = (128u >> 4) | (1u << 14);
      const uint32_t a_hi = (1024u >> 4) | (1u << 14) | (2u << 29);
      const uint32_t id0 = (1u << 4) | (1u << 7) | (1u << 10) | (8u << 24);
      const uint64_t ones = ((uint64_t)((1u << 14) | (2u << 29)) << 32) | (uint64_t)(((sm >> 4) & 0x3FFFu) | (1u << 16));
      const uint32_t bias_row = (sm + (uint32_t)p.off_bias) >> 4, zero_row = bias_row + (uint32_t)(p.c_mid + p.n3);
      auto bias_desc = [&](uint32_t row) { return ((uint64_t)b_hi << 32) | (uint64_t)((row & 0x3FFFu) | ((zero_row - row) << 16)); };
      // `steps` (at most four) instructions of 16 channels each: along a 128-byte line of A, two chunk planes of `pitch` rows of B
      auto multiply = [&](uint32_t d, uint32_t a, uint32_t b, uint32_t pitch, int steps, uint32_t idesc) {
        a = (a & 0x3FFFu) | (1u << 16);
        b = (b & 0x3FFFu) | (pitch << 16);
        if (steps == 4) {
#pragma unroll
          for (uint32_t k = 0; k < 4; ++k)
            umma_bf16(d, ((uint64_t)a_hi << 32) | (uint64_t)(a + 2u * k), ((uint64_t)b_hi << 32) | (uint64_t)(b + 2u * k * pitch), idesc, 1u);
        } else {
#pragma unroll 1
          for (int k = 0; k < steps; ++k, a += 2u, b += 2u * pitch)
            umma_bf16(d, ((uint64_t)a_hi << 32) | (uint64_t)a, ((uint64_t)b_hi << 32) | (uint64_t)b, idesc, 1u);
        }
      };
      Ring ring;
      bool ok = true;
      if (warp == 1) {
        // ---- X W1 of every chunk into the expansion's accumulators
        uint32_t ph_x = 0, use = 0;
        const uint32_t x_row = (sm + (uint32_t)p.off_x) >> 4, w_row = (sm + (uint32_t)p.off_w1) >> 4, ch = (uint32_t)p.ch;
#pragma unroll 1
        for (int t = (int)blockIdx.x; t < p.tiles && ok; t += (int)gridDim.x) {
          ok = warp_wait(&sh.x_full, ph_x, abort_flag, ws, 0x32000u);
          ph_x ^= 1;
          int i = 0;
#pragma unroll 1
          for (Chunks c(p); i < p.nch && ok; ++i, c.next(p), ring.next(p.nw), ++use) {
            const int s = ring.s;
            const uint32_t eb = use % G;
            ok = warp_wait(&sh.w1_full[s], ring.ph, abort_flag, ws, 0x30000u | s) && warp_wait(&sh.e_empty[eb], ((use / G) & 1u) ^ 1u, abort_flag, ws, 0x31000u | eb);
            if (!ok) break;
            tc_fence_after();
            if (leader) {
              const uint32_t idesc = id0 | ((uint32_t)(c.n >> 3) << 17);
              const uint64_t bd = bias_desc(bias_row + (uint32_t)c.h0);
              const uint32_t w = w_row + (uint32_t)(s * (p.w1_bytes >> 4));
#pragma unroll 1
              for (int b = 0; b < p.mbe; ++b) {
                const uint32_t d = tmem_e + (eb * (uint32_t)p.mbe + (uint32_t)b) * ch;
                umma_bf16(d, ones, bd, idesc, 0u);
                uint32_t a = x_row + (uint32_t)(b * 1024), bw = w;
#pragma unroll 1
                for (int left = p.ksteps; left > 0; left -= 4, a += (uint32_t)(p.mbe * 1024), bw += 8u * ch) multiply(d, a, bw, ch, left < 4 ? left : 4, idesc);
              }
            }
            __syncwarp();                        // (commits behind the meeting of the warp: inside the stretch they cost 10 % and more)
            if (leader) {
              umma_commit(&sh.e_full[eb]);
              umma_commit(&sh.w1_empty[s]);
              if (i == p.nch - 1) umma_commit(&sh.x_empty);
            }
          }
        }
      } else {
        // ---- the projection of every chunk whose stencil is done
        uint32_t ph_y = 1, p_use = 0;
        const uint32_t p_row = (sm + (uint32_t)p.off_p) >> 4, w_row = (sm + (uint32_t)p.off_w3) >> 4, nt3 = (uint32_t)p.nt3;
        const uint32_t idesc = id0 | ((nt3 >> 3) << 17);
#pragma unroll 1
        for (int t = (int)blockIdx.x; t < p.tiles && ok; t += (int)gridDim.x) {
          ok = warp_wait(&sh.y_empty, ph_y, abort_flag, ws, 0x35000u);
          ph_y ^= 1;
          if (!ok) break;
          tc_fence_after();
          if (leader)                            // the bias initialises the accumulators
            for (int b = 0; b < p.mbp; ++b)
              for (int ps = 0; ps < p.pass3; ++ps)
                umma_bf16(tmem_y + (uint32_t)(b * p.n3 + ps * p.nt3), ones, bias_desc(bias_row + (uint32_t)(p.c_mid + ps * p.nt3)), idesc, 0u);
          __syncwarp();
          int i = 0;
#pragma unroll 1
          for (Chunks c(p); i < p.nch && ok; ++i, c.next(p), ring.next(p.nw), ++p_use) {
            const int s = ring.s;
            const StencilOperand o(p_use, (uint32_t)p.np);
            ok = warp_wait(&sh.w3_full[s], ring.ph, abort_flag, ws, 0x33000u | s) && warp_wait(&sh.p_full[o.barrier], o.parity, abort_flag, ws, 0x34000u | o.barrier);
            if (!ok) break;
            tc_fence_after();
            if (leader) {
              const uint32_t a0 = p_row + o.buffer * (uint32_t)(p.p_bytes >> 4), w = w_row + (uint32_t)(s * (p.w3_bytes >> 4));
#pragma unroll 1
              for (int b = 0; b < p.mbp; ++b)
#pragma unroll 1
                for (int ps = 0; ps < p.pass3; ++ps)
                  multiply(tmem_y + (uint32_t)(b * p.n3 + ps * p.nt3), a0 + (uint32_t)(b * 1024), w + (uint32_t)(ps * (c.n >> 3)) * nt3, nt3, c.n >> 4, idesc);
            }
            __syncwarp();
            if (leader) {
              umma_commit(&sh.w3_empty[s]);
              umma_commit(&sh.p_empty[o.barrier]);
              if (i == p.nch - 1) umma_commit(&sh.y_full);
            }
          }
        }
      }
    } else {
      // ================================================================== convert, stencil, read-out
      const int mw = warp - kFirstMathWarp, q = warp & 3, j0 = mw >> 2;   // tensor-memory lane quadrant; this warp's turn in it
      // Two groups of eight warps take the chunks in turn, so that one's barriers, tensor-memory reads and conversions lie under
      // the other's stencil; or, where two buffers of the hidden chunk would make the tile smaller, all sixteen each.
      const uint32_t grp = (uint32_t)(mw / kGroupWarps);
      const int mt = (mw % kGroupWarps) * 32 + lane, jg = j0 % (4 / G);
      const uint32_t hb = sm + (uint32_t)p.off_h + grp * (uint32_t)p.h_bytes;
      const uint32_t tm_row = (uint32_t)(q * 32) << 16;
      Ring r3;
      uint32_t y_ph = 0, use = 0;                // use: chunks so far, of all tiles
      bool ok = true;
#pragma unroll 1
      for (int t = (int)blockIdx.x; t < p.tiles; t += (int)gridDim.x) {
        const Tile tl(p, t);
        // which of this lane's patch pixels (one per block) lie inside the image and the batch
        uint32_t inside = 0;
#pragma unroll
        for (int b = 0; b < kMaxE; ++b) {
          const int pos = b * 128 + q * 32 + lane;
          if (pos < p.patch) {
            const int il = div20(pos, p.inv_lines), rem = pos - il * p.lines_img, r = div20(rem, p.inv_wbox), c = rem - r * p.wbox;
            const int iy = tl.y0 * S - 1 + r, ix = tl.x0 * S - 1 + c;
            if ((unsigned)iy < (unsigned)p.h && (unsigned)ix < (unsigned)p.w) inside |= 1u << b;
          }
        }
        const int th_valid = p.ho - tl.y0 < p.th ? p.ho - tl.y0 : p.th;
        int i = 0;
#pragma unroll 1
        for (Chunks c(p); i < p.nch; ++i, c.next(p), r3.next(p.nw), ++use) {
          if (use % G != grp) continue;
          const int chv = c.n;
          // ---- convert: 16 columns of a block at a time
          ok = ok && warp_wait(&sh.e_full[grp], (use / G) & 1u, abort_flag, ws, 0x40000u | grp);
          bar_sync(kBarMath + (int)grp, kGroupThreads);        // the group's buffer is read by no one any more
          const uint32_t s = (uint32_t)r3.s;
          const StencilOperand po(use, (uint32_t)p.np);
          if (ok) {
            tc_fence_after();
            const uint32_t te = tmem_e + tm_row + grp * (uint32_t)(p.mbe * p.ch);
            const int tasks = p.mbe * (chv >> 4);
#pragma unroll 1
            for (int u = jg; u < tasks; u += 8 / G) {
              const bool two = u + 4 / G < tasks;
              const int u2 = two ? u + 4 / G : u;
              const int cq = div20(u, p.inv_mbe), b = u - cq * p.mbe, cq2 = div20(u2, p.inv_mbe), b2 = u2 - cq2 * p.mbe;
              uint32_t v[32];
              tmem_ld16(te + (uint32_t)(b * p.ch + cq * 16), v);
              tmem_ld16(te + (uint32_t)(b2 * p.ch + cq2 * 16), v + 16);
              tmem_ld_wait();
#pragma unroll
              for (int hh = 0; hh < 2; ++hh) {
                const int bb = hh ? b2 : b, pos = bb * 128 + q * 32 + lane;
                if (pos < p.patch && (hh == 0 || two)) {
                  const bool in = (inside >> bb) & 1u;
                  uint32_t o[8];
#pragma unroll
                  for (int e = 0; e < 8; ++e)
                    o[e] = in ? relu6_bf16x2(__uint_as_float(v[hh * 16 + 2 * e]), __uint_as_float(v[hh * 16 + 2 * e + 1])) : 0u;
                  const uint32_t at = hb + (uint32_t)(pos * kHPitch + (hh ? cq2 : cq) * 32);
                  sts_u4(at, make_uint4(o[0], o[1], o[2], o[3]));
                  sts_u4(at + 16u, make_uint4(o[4], o[5], o[6], o[7]));
                }
              }
            }
            tc_fence_before();
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&sh.e_empty[grp]);
          bar_sync(kBarMath + (int)grp, kGroupThreads);
          // ---- depthwise
          ok = ok && stencil_waits(use, (uint32_t)p.np, s, r3.ph, [&](uint32_t kind, uint32_t at, uint32_t parity) {
            return kind == kWeightsIn ? warp_wait(&sh.w3_full[at], parity, abort_flag, ws, 0x41000u | at)
                                      : warp_wait(&sh.p_empty[at], parity, abort_flag, ws, 0x42000u | at);
          });
          if (ok) {
            const uint32_t wdb = sm + (uint32_t)p.off_wd + s * (uint32_t)p.wd_bytes, ch4 = (uint32_t)p.ch * 4u;
            const uint32_t pbuf = sm + (uint32_t)p.off_p + po.buffer * (uint32_t)p.p_bytes;
            const int ncg = chv >> 2;
            const uint32_t inv_ncg = p.inv_ncg[(chv >> 4) - 1];
            const int items = p.ni * p.th * p.strips * ncg;
#pragma unroll 1
            for (int it = mt; it < items; it += kGroupThreads) {
              const int sp = div20(it, inv_ncg), cg = it - sp * ncg;
              const int row = div20(sp, p.inv_strips), X0 = (sp - row * p.strips) * TX;
              const int il = div20(row, p.inv_th), yy = row - il * p.th;
              if (yy >= th_valid) continue;
              uint32_t src = hb + (uint32_t)((il * p.lines_img + yy * S * p.wbox + X0 * S) * kHPitch + cg * 8);
              const uint32_t row_pitch = (uint32_t)(p.wbox * kHPitch);
              const uint32_t wa = wdb + (uint32_t)cg * 16u;
              float2 acc[TX][2];
              {
                const float4 bz = lds_f4(wa + 9u * ch4);
#pragma unroll
                for (int o = 0; o < TX; ++o) { acc[o][0] = make_float2(bz.x, bz.y); acc[o][1] = make_float2(bz.z, bz.w); }
              }
#pragma unroll
              for (int r = 0; r < 3; ++r, src += row_pitch) {
                float2 wr[3][2];
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                  const float4 wv = lds_f4(wa + (uint32_t)(r * 3 + c) * ch4);
                  wr[c][0] = make_float2(wv.x, wv.y);
                  wr[c][1] = make_float2(wv.z, wv.w);
                }
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                  const uint2 raw = lds_u2(src + (uint32_t)(j * kHPitch));
                  const float2 x0 = make_float2(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xFFFF0000u));
                  const float2 x1 = make_float2(__uint_as_float(raw.y << 16), __uint_as_float(raw.y & 0xFFFF0000u));
#pragma unroll
                  for (int o = 0; o < TX; ++o) {
                    const int c = j - o * S;
                    if (c >= 0 && c < 3) {
                      acc[o][0] = __ffma2_rn(x0, wr[c][0], acc[o][0]);
                      acc[o][1] = __ffma2_rn(x1, wr[c][1], acc[o][1]);
                    }
                  }
                }
              }
              const int line0 = (il * p.th + yy) * p.tw + X0, n_out = p.tw - X0;
#pragma unroll
              for (int o = 0; o < TX; ++o) {
                const int line = line0 + o;
                // a NaN becomes 6, as in the depthwise kernel of the three launches
                const uint32_t v0 = min_bf16x2(pack_bf16x2_relu(acc[o][0].x, acc[o][0].y), 0x40C040C0u);
                const uint32_t v1 = min_bf16x2(pack_bf16x2_relu(acc[o][1].x, acc[o][1].y), 0x40C040C0u);
                if (o < n_out) sts_u2(pbuf + (uint32_t)(line * 128 + (((cg >> 1) ^ (line & 7)) << 4) + (cg & 1) * 8), v0, v1);
              }
            }
            fence_proxy_async();
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&sh.p_full[po.barrier]);
        }
        // ---- read-out: 16 channels of 32 outputs at a time, turned around in the place of the group's hidden chunk (every
        // stencil of the tile is done when the sums are) so that two lanes store a pixel's 32 bytes
        ok = ok && warp_wait(&sh.y_full, y_ph, abort_flag, ws, 0x43000u);
        y_ph ^= 1;
        if (ok) {
          tc_fence_after();
          const uint32_t stage = hb + (uint32_t)((mw % kGroupWarps) * 1024);
          const uint32_t st_wr = stage + (uint32_t)(lane * 32), sw = (uint32_t)((lane >> 2) & 1);
          const uint32_t st_rd = stage + (uint32_t)((lane >> 1) * 32 + (((lane & 1) ^ ((lane >> 3) & 1)) * 16));
          const int outs_img = p.th * p.tw, tasks = p.mbp * (p.n3 >> 4);
          const int tw_valid = p.wo - tl.x0 < p.tw ? p.wo - tl.x0 : p.tw;
#pragma unroll 1
          for (int u = j0; u < tasks; u += 4) {
            const int cq = div20(u, p.inv_mbp), b = u - cq * p.mbp;
            uint32_t v[16];
            tmem_ld16(tmem_y + tm_row + (uint32_t)(b * p.n3 + cq * 16), v);
            tmem_ld_wait();
            __syncwarp();
#pragma unroll
            for (int g = 0; g < 2; ++g) {
              // fp32 sums wait for the skip input: two 16-byte pieces of 4 channels would not fit, so the pixel's own lane adds it
              const int line = b * 128 + q * 32 + lane;
              const int il = div20(line, p.inv_outs), rem = line - il * outs_img, r = div20(rem, p.inv_tw), c = rem - r * p.tw;
              float f[8];
#pragma unroll
              for (int e = 0; e < 8; ++e) f[e] = __uint_as_float(v[8 * g + e]);
              const int ch0 = cq * 16 + 8 * g;
              if (p.residual && ch0 < p.c_out && il < p.ni && tl.img0 + il < p.n_img && r < th_valid && c < tw_valid) {
                const uint4 rv = *reinterpret_cast<const uint4 *>(
                    x + ((size_t)((tl.img0 + il) * p.ho + tl.y0 + r) * p.wo + tl.x0 + c) * p.c_out + ch0);
                const __nv_bfloat162 *rb = reinterpret_cast<const __nv_bfloat162 *>(&rv);
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const float2 rf = __bfloat1622float2(rb[e]);
                  f[2 * e] += rf.x;
                  f[2 * e + 1] += rf.y;
                }
              }
              sts_u4(st_wr + (((uint32_t)g ^ sw) << 4),
                     make_uint4(pack_bf16x2(f[0], f[1]), pack_bf16x2(f[2], f[3]), pack_bf16x2(f[4], f[5]), pack_bf16x2(f[6], f[7])));
            }
            __syncwarp();
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
              const int line = b * 128 + q * 32 + hf * 16 + (lane >> 1);
              const int il = div20(line, p.inv_outs), rem = line - il * outs_img, r = div20(rem, p.inv_tw), c = rem - r * p.tw;
              const uint4 piece = lds_u4(st_rd + (uint32_t)(hf * 512));
              const int ch0 = cq * 16 + 8 * (lane & 1);
              if (ch0 < p.c_out && il < p.ni && tl.img0 + il < p.n_img && r < th_valid && c < tw_valid)
                *reinterpret_cast<uint4 *>(y + ((size_t)((tl.img0 + il) * p.ho + tl.y0 + r) * p.wo + tl.x0 + c) * p.c_out + ch0) = piece;
            }
          }
          tc_fence_before();
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&sh.y_empty);
      }
    }
    // ---- teardown
    if (*abort_flag) {
      const unsigned long long t0 = globaltimer_ns();
      while (globaltimer_ns() - t0 < 200000ull) __nanosleep(1000);
    }
    tc_fence_before();
    bar_sync(kBarTmem, kMathThreads + 64);
    if (warp == 1) {
      tc_fence_after();
      tmem_dealloc(sh.tmem_base, (uint32_t)p.tmem_cols);
    }
  }
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

constexpr int kSmemBudget = 224 * 1024;

uint32_t inv20(int d) { return ((1u << 20) + (uint32_t)d - 1) / (uint32_t)d; }

// Lays out the shared memory of a plan whose tile is set; false when it does not fit.
bool block_layout(BlockParams *p) {
  p->p_bytes = p->mbp * 16384;
  p->w1_bytes = 2 * p->ksteps * p->ch * 16;
  p->wd_bytes = (int)dc_round_up((size_t)10 * p->ch * 4, 128);
  p->w3_bytes = (p->ch >> 3) * p->n3 * 16;
  const size_t h_bytes = dc_round_up((size_t)(p->patch + p->tx * p->stride) * kHPitch, 128);   // the last group of a row may hang over
  const int readout = kMathWarps / p->groups * 1024;
  p->h_bytes = (int)h_bytes > readout ? (int)h_bytes : readout;   // room for the read-out
  p->off_bias = 1024;
  p->off_x = (int)dc_round_up((size_t)p->off_bias + (size_t)(p->c_mid + p->n3 + (p->ch > p->n3 ? p->ch : p->n3)) * 16, 1024);
  p->off_p = p->off_x + p->planes * p->mbe * 16384;
  // a buffer of the hidden chunk for each group; two of the projection's operand where they fit, then more weight stages
  const int stage = p->w1_bytes + p->wd_bytes + p->w3_bytes;
  for (p->np = 2; p->np >= 1; --p->np) {
    const int fixed = 1024 + p->off_p + p->np * p->p_bytes + p->groups * p->h_bytes;
    if (fixed + 2 * stage > kSmemBudget) continue;
    p->nw = (kSmemBudget - fixed) / stage;
    if (p->nw > kMaxW) p->nw = kMaxW;
    if (p->nw > p->nch && p->nch >= 2) p->nw = p->nch;
    p->off_w1 = p->off_p + p->np * p->p_bytes;
    p->off_wd = p->off_w1 + p->nw * p->w1_bytes;
    p->off_w3 = p->off_wd + p->nw * p->wd_bytes;
    p->off_h = p->off_w3 + p->nw * p->w3_bytes;
    p->smem_bytes = 1024 + p->off_h + p->groups * p->h_bytes;
    return true;
  }
  return false;
}

// Estimated time of a plan, in cycles.  A chunk of hidden channels costs what its conversions and the stencil's thread items
// need of the SM's schedulers and shared memory, or its chain of waits in a group of warps (two groups run side by side),
// or its weights' way in from L2; a tile its patch's way in and the read-out.  The constants are fitted to 25 blocks (16 to 160
// channels, maps of 7 to 112, 1 to 128 images) timed in every tile and form considered below, 5400 in all: 8 % off in the
// root mean square; the choice is 2 % above the best on average, 10 % at worst (24 -> 144 -> 24, 64 images of 56 x 56).
double chunk_cycles(const BlockParams &p) {
  const int warps = dc_div_up(p.ni * p.th * p.strips * (p.ch >> 2), 32), tasks = p.mbe * (p.ch >> 4);
  const double issue = (158.0 + 80.0 * p.tx) * warps / 4 + 211.0 * tasks;
  const double chain = (835.0 + 718.0 * dc_div_up(tasks * p.groups, 8) + 147.0 * p.tx * dc_div_up(warps * p.groups, kMathWarps)) / p.groups;
  const double weights = (double)(p.w1_bytes + p.wd_bytes + p.w3_bytes) / 24.4;
  return sqrt(sqrt(issue * issue * issue * issue + chain * chain * chain * chain + weights * weights * weights * weights));
}
double plan_cycles(const BlockParams &p, int n_sm) {
  const int out = p.mbp * (p.n3 >> 4);
  return 6234.0 + dc_div_up(p.tiles, n_sm) * (3080.0 + 390.0 * out + 1.35 * p.planes * p.patch + p.nch * chunk_cycles(p));
}

// What the chosen plan takes beside three launches, in cycles: the same terms fitted to the plans that are chosen for 499 blocks (16 to
// 160 channels in, 8 to 320 out, maps of 3 to 112, 1 to 320 images), 6.5 % off in the root mean square (the estimate above,
// fitted to good and bad plans alike, 7.4 %, and up to 26 % too high for wide outputs).
double one_launch_cycles(const BlockParams &p, int n_sm) {
  const int out = p.mbp * (p.n3 >> 4);
  return 5239.0 + dc_div_up(p.tiles, n_sm) * (3207.0 + 239.0 * out + 2.75 * p.planes * p.patch + p.nch * (309.0 + 0.907 * chunk_cycles(p)));
}

// The three launches' time, in cycles: a start, the hidden maps written and read, the products.  The terms of narrow projections are
// those of the general kernel, a chain over the hidden channels.  Fitted to the same blocks: 7 % off in the root mean square (19 %
// without the terms of the products and of narrow projections).  Projections to 16 and 24 channels, by rows, no longer cost that much,
// but the choice is right with them all the same: over 60 blocks one launch takes 0.78 of the three's time, seven of them more, by up
// to 9 % (16 -> 96 -> 24 on 23 maps of 103 x 103 51.6 us here, 47.3 in three; 24 -> 144 -> 24 on 9 maps of 12 x 12 7.4 and 10.4).
double three_launches_cycles(const BlockParams &p, bool narrow) {
  const double hidden = (double)p.n_img * p.h * p.w * p.c_mid * 2e-6, thinned = (double)p.n_img * p.ho * p.wo * p.c_mid * 2e-6;
  const double expand = hidden * 8e-3 * p.ksteps, project = thinned * 5e-4 * p.n3;
  return 1900.0 * (8.97 + 0.393 * hidden + 0.352 * thinned + 4.58e-3 * p.c_mid + 0.25 * expand + 3.18 * project +
                   (narrow ? 0.71 * thinned + 27e-3 * p.c_mid : 0.0));
}

bool make_block_plan(int n, int h, int w, const dc_block *b, int n_sm, BlockParams *p) {
  if (!b->has_expand || b->dw_k != 3 || b->dw_pad != 1 || (b->dw_stride != 1 && b->dw_stride != 2)) return false;
  if (b->act_expand != DC_ACT_RELU6 || b->act_dw != DC_ACT_RELU6) return false;
  if (b->c_in % 8 || b->c_out % 8 || b->c_hidden % 16) return false;
  const int S = b->dw_stride, ho = dc_out_extent(h, 3, S, 1), wo = dc_out_extent(w, 3, S, 1);
  if (ho <= 0 || wo <= 0 || (long long)n * h * w >= (1ll << 31)) return false;
  const dc_geom g1 = {b->c_in, b->c_hidden, 1, 1, 1, 0}, g3 = {b->c_hidden, b->c_out, 1, 1, 1, 0};
  KOrder k1, k3;
  dc_korder_init(&k1, &g1);
  dc_korder_init(&k3, &g3);
  if (!k1.rows || k3.pair || k3.fold) return false;
  p->n_img = n; p->h = h; p->w = w; p->ho = ho; p->wo = wo;
  p->c_in = b->c_in; p->c_mid = b->c_hidden; p->c_out = b->c_out; p->stride = S; p->residual = b->has_residual;
  p->planes = dc_div_up(b->c_in, 64);
  p->ksteps = dc_div_up(b->c_in, 16);
  p->nt1 = k1.n_tile; p->e1 = k1.e_pad;
  p->nt3 = k3.rows ? k3.n_tile : k3.n_pad; p->e3 = k3.e_pad;
  p->n3 = k3.n_pad; p->pass3 = p->n3 / p->nt3;
  if (p->n3 > 256 || (!k3.rows && k3.ng > 1 && k3.e != k3.e_pad)) return false;
  // chunks: the passes of the expansion's weights in equal parts of at most 64
  const int last = b->c_hidden - (k1.nnt - 1) * p->nt1;
  if (last <= 0) return false;
  const int cpl = dc_div_up(last, 64);
  const int cpp = dc_div_up(p->nt1, 64);
  p->npass = k1.nnt;
  p->last_rows = last;
  p->chp = (int)dc_round_up((size_t)dc_div_up(p->nt1, cpp), 16);
  p->chl = (int)dc_round_up((size_t)dc_div_up(last, cpl), 16);
  p->ch = p->chl > p->chp ? p->chl : p->chp;
  if (k1.nnt == 1) p->ch = p->chp = p->chl;
  p->nch = (k1.nnt - 1) * dc_div_up(p->nt1, p->chp) + dc_div_up(last, p->chl);
  BlockParams best;
  double best_cost = 0.0;
  bool any = false;
  auto consider_form = [&](int tw, int th, int ni, int form) {
    p->form = form;
    p->tx = kTx[S - 1][form];
    p->groups = kGroups[form];
    p->tw = tw; p->th = th; p->ni = ni;
    p->wbox = (tw - 1) * S + 3; p->rbox = (th - 1) * S + 3;
    if (p->wbox > 256 || p->rbox > 256) return;
    p->lines_img = p->wbox * p->rbox;
    p->patch = ni * p->lines_img;
    p->mbe = dc_div_up(p->patch, 128);
    p->mbp = dc_div_up(ni * th * tw, 128);
    if (p->mbe > kMaxE || p->groups * p->mbe * p->ch + p->mbp * p->n3 > 512) return;
    p->strips = dc_div_up(tw, p->tx);
    if (!block_layout(p)) return;
    p->nxt = dc_div_up(wo, tw);
    p->tiles_y = dc_div_up(ho, th);
    const long long tiles = (long long)dc_div_up(n, ni) * p->nxt * p->tiles_y;
    if (tiles >= (1ll << 30)) return;
    p->tiles = (int)tiles;
    const double cost = plan_cycles(*p, n_sm);
    if (!any || cost < best_cost) { any = true; best = *p; best_cost = cost; }
  };
  auto consider = [&](int tw, int th, int ni) {
    for (int form = 0; form < kForms; ++form) consider_form(tw, th, ni, form);
  };
  for (int nxt = 1; nxt <= 8 && nxt <= wo; ++nxt) {
    const int tw = dc_div_up(wo, nxt);
    for (int ty = 1; ty <= ho; ++ty) {
      const int th = dc_div_up(ho, ty);
      if (ty > 1 && th == dc_div_up(ho, ty - 1)) continue;
      if (((tw - 1) * S + 3) * ((th - 1) * S + 3) <= kMaxE * 128) consider(tw, th, 1);
    }
  }
  for (int ni = 2; ni <= 8 && ni <= n; ++ni) consider(wo, ho, ni);
  if (!any) return false;
  *p = best;
  // Taken where it is estimated to be faster than the three launches.  The line lies where the 499 blocks together take least: at
  // 1.03 where each tile has an SM of its own (0.756 of the three launches' time on average, as if the faster were always known to
  // 0.3 %; five of 373 are more than 3 % slower than three launches, by 8 % at most), at 0.9 where a CTA has several tiles in turn
  // (0.888; two of 126 by up to 5 %; at 0.95 0.886 but nine by up to 21 %: 32 -> 192 -> 32 on 30 maps of 51 x 48 37.1 us here,
  // 30.7 in three).  Long reductions of few pixels stay with the launches, whose reductions clusters share: 160 -> 960 -> 160 on
  // one 7 x 7 map 22.4 us here, 11.0 there.
  if (one_launch_cycles(*p, n_sm) > (p->tiles > n_sm ? 0.9 : 1.03) * three_launches_cycles(*p, !k3.rows || b->c_out < 32)) return false;
  p->inv_lines = inv20(p->lines_img); p->inv_wbox = inv20(p->wbox); p->inv_th = inv20(p->th);
  p->inv_strips = inv20(p->strips); p->inv_outs = inv20(p->th * p->tw); p->inv_tw = inv20(p->tw);
  p->inv_mbe = inv20(p->mbe); p->inv_mbp = inv20(p->mbp);
  for (int q = 0; q < 4; ++q) p->inv_ncg[q] = inv20(4 * (q + 1));
  int cols = 32;
  while (cols < p->groups * p->mbe * p->ch + p->mbp * p->n3) cols *= 2;
  p->tmem_cols = cols;
  return true;
}

bool block_plan(int n, int h, int w, const dc_block *b, int n_sm, BlockParams *p) {
  static thread_local DcPlans<BlockParams> plans;
  // (the rest of what the plan looks at, in one word)
  const bool plain = b->has_expand && b->dw_k == 3 && b->dw_pad == 1 && b->act_expand == DC_ACT_RELU6 && b->act_dw == DC_ACT_RELU6;
  return plans.get({n, h, w, b->c_in, b->c_hidden, b->c_out, b->dw_stride, b->has_residual != 0, plain, n_sm, dc_plan_device(), 0}, p,
                   [&](BlockParams *q) { return make_block_plan(n, h, w, b, n_sm, q); });
}

}  // namespace

dc_status dc_launch_block_tc(const void *x, int n, int h, int w, const dc_block *b, void *y, void *workspace,
                             cudaStream_t stream) {
  BlockParams p;
  const int n_sm = dc_sm_count();
  if (!block_plan(n, h, w, b, n_sm, &p)) return DC_ERR_UNSUPPORTED;
  EncodeTiledFn encode = get_encode_fn();
  if (!encode) return DC_ERR_CUDA;
  CUtensorMap map_x;
  {
    const cuuint64_t C = (cuuint64_t)p.c_in;
    cuuint64_t gdim[4] = {C, (cuuint64_t)w, (cuuint64_t)h, (cuuint64_t)n};
    cuuint64_t gstr[3] = {2 * C, (cuuint64_t)w * C * 2, (cuuint64_t)h * w * C * 2};
    cuuint32_t box[4] = {64, (cuuint32_t)p.wbox, (cuuint32_t)p.rbox, (cuuint32_t)p.ni};
    cuuint32_t es[4] = {1, 1, 1, 1};
    CUresult r = encode(&map_x, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(x), gdim, gstr, box, es,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return DC_ERR_CUDA;
  }
  CUtensorMap map_w1, map_wd;
  {
    // expansion weights: 16-byte rows (8 input channels) of the hidden channels, as pairs of 8-byte elements
    cuuint64_t gdim[2] = {2 * (cuuint64_t)p.nt1, (cuuint64_t)p.e1 * (cuuint64_t)dc_div_up(p.c_mid, p.nt1)}, gstr[1] = {(cuuint64_t)p.nt1 * 16};
    cuuint32_t box[2] = {2 * (cuuint32_t)p.ch, 2 * (cuuint32_t)p.ksteps}, es[2] = {1, 1};
    if (encode(&map_w1, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, const_cast<void *>(b->w_expand), gdim, gstr, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return DC_ERR_CUDA;
    cuuint64_t ddim[2] = {(cuuint64_t)p.c_mid, 9}, dstr[1] = {(cuuint64_t)p.c_mid * 4};
    cuuint32_t dbox[2] = {(cuuint32_t)p.ch, 9};
    if (encode(&map_wd, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float *>(b->w_dw), ddim, dstr, dbox, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return DC_ERR_CUDA;
  }
  static unsigned char attr_done[2 * kForms][kDcMaxDevices];
  const int which = kForms * (p.stride - 1) + p.form;
  using Kernel = decltype(&k_block_tc<1, 7, 1>);
  static constexpr Kernel kernels[2 * kForms] = {
      k_block_tc<1, kTx[0][0], 1>, k_block_tc<1, kTx[0][1], 1>, k_block_tc<1, kTx[0][2], 2>, k_block_tc<1, kTx[0][3], 2>,
      k_block_tc<2, kTx[1][0], 1>, k_block_tc<2, kTx[1][1], 1>, k_block_tc<2, kTx[1][2], 2>, k_block_tc<2, kTx[1][3], 2>};
  const Kernel kernel = kernels[which];
  DC_CUDA_OK(dc_set_max_smem_once(kernel, kSmemBudget, attr_done[which]));
  const cudaError_t e = dc_launch_pdl(kernel, dim3(p.tiles < n_sm ? p.tiles : n_sm), dim3(kThreads), (size_t)p.smem_bytes, stream,
                                      map_x, map_w1, map_wd, p, b->b_expand, b->b_dw, b->w_project, b->b_project,
                                      (const __nv_bfloat16 *)x, (__nv_bfloat16 *)y, (DcWsHeader *)workspace);
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? DC_OK : DC_ERR_CUDA;
}

dc_status dc_block_tc_plan(int n, int h, int w, const dc_block *b, dc_block_plan *plan) {
  BlockParams p;
  if (!block_plan(n, h, w, b, dc_sm_count(), &p)) return DC_ERR_UNSUPPORTED;
  *plan = {p.tw, p.th, p.ni, p.tiles, p.nch, p.form, p.groups, p.np, p.nw};
  return DC_OK;
}

extern "C" int dc_selftest_block_waits(unsigned int chunk, int operands, int stages, unsigned int waits[12]) {
  if (operands < 1 || operands > 2 || stages < 2 || stages > kMaxW) return 0;
  int n = 0;
  auto note = [&](uint32_t kind, uint32_t at, uint32_t parity) {
    waits[3 + 3 * n] = kind; waits[4 + 3 * n] = at; waits[5 + 3 * n] = parity;
    ++n;
    return true;
  };
  const StencilOperand o(chunk, (uint32_t)operands);
  waits[0] = o.buffer; waits[1] = o.barrier; waits[2] = o.parity;
  stencil_waits(chunk, (uint32_t)operands, chunk % (unsigned)stages, (chunk / (unsigned)stages) & 1u, note);
  return n;
}
