// Learned warm start: a small convolutional network on the nodal image of a 2D structured mesh
// that predicts the next time step's state, used as the initial guess of FGMRES.
//
// Network (3 layers, 3x3 convolutions, "same" zero padding, stride 1):
//   z1 = W1 * x + b1 (12 -> C), a1 = relu(z1)
//   z2 = W2 * a1 + b2 (C -> C), a2 = relu(z2)
//   y  = W3 * a2 + b3 (C -> 4)
// From the last three states s = s_k, q = s_{k-1}, q2 = s_{k-2} (phi_p, phi_n, mu_p, mu_n) the
// prediction is a learned second-order extrapolation,
//   pred = s + d + theta * D,  d = s - q,  D = s - 2 q + q2,  theta = y * out_scale,
// so the zero network is linear and theta = 1 quadratic extrapolation, and the network only scales
// the (smooth) second difference pixel by pixel.  x holds the fields normalised per channel, d in
// units of its RMS over the image and D in units of its RMS (12 of 16 input channels): the map
// does not depend on how fast the state moves.  Activations are NHWC BF16
// with FP32 accumulation; weights are kept as FP32 master copies (Adam) and BF16 copies for the
// tensor cores, the latter also in tap-flipped, channel-transposed form for the backward pass
// through the data.
//
// Convolutions are implicit GEMMs on the tensor cores, BF16 in, FP32 accumulate, M = pixels,
// N = output channels, K = 9 taps x input channels: by default on tcgen05 (k_conv3x3_tc: tensor
// memory accumulators, operands staged in shared memory as row bands), or on mma.sync m16n8k16
// (k_conv3x3: 16 pixels per warp, 8 channels per tile; each lane gathers its A-fragment elements
// straight from the shifted input, zero outside the image, the B fragments from the weights
// staged in shared memory).
// Weight gradients are GEMMs over the pixels on mma.sync, per strip of image rows, the strips' partial
// sums added in order (deterministic).
#include <cuda_bf16.h>

#include <cmath>
#include <vector>

#include <algorithm>
#include <initializer_list>

#include "ch_internal.cuh"

namespace ch {

constexpr int WS_C = 32;       // hidden channels
constexpr int WS_CIN = 16;     // input channels padded for the k16 MMA (12 used)
constexpr int WS_COUT = 8;     // output channels padded for the n8 MMA (4 used)

struct WsParams {  // FP32 master parameters, contiguous
  float* w1;  // [9][WS_CIN][WS_C]
  float* b1;  // [WS_C]
  float* w2;  // [9][WS_C][WS_C]
  float* b2;  // [WS_C]
  float* w3;  // [9][WS_C][WS_COUT]
  float* b3;  // [WS_COUT]
};

constexpr int WS_N1 = 9 * WS_CIN * WS_C, WS_N2 = 9 * WS_C * WS_C, WS_N3 = 9 * WS_C * WS_COUT;
constexpr int WS_NPARAM = WS_N1 + WS_C + WS_N2 + WS_C + WS_N3 + WS_COUT;

// ---------------------------------------------------------------- BF16 helpers
__device__ __forceinline__ uint32_t pack_bf16(__nv_bfloat16 lo, __nv_bfloat16 hi) {
  return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

// D = A (16x16, row) * B (16x8, col) + C, BF16 inputs, FP32 accumulate
__device__ __forceinline__ void mma_bf16(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
      "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// two consecutive BF16 channels (c, c+1) of pixel (r, q) of an NHWC image, zero outside
__device__ __forceinline__ uint32_t load_pair(const __nv_bfloat16* X, int H, int W, int C, int r, int q,
                                              int c) {
  if (r < 0 || r >= H || q < 0 || q >= W) return 0u;
  return *reinterpret_cast<const uint32_t*>(X + ((size_t)r * W + q) * C + c);
}

// ---------------------------------------------------------------- tcgen05 primitives (inline PTX)
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor of a K-major operand without swizzle: the canonical layout of
// 8-row x 16-byte core matrices, lbo = byte distance between core matrices adjacent along K, sbo =
// between core matrices adjacent along M (or N); bits 46-47 hold the descriptor version (1).
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo & 0x3FFFFu) >> 4) << 16) |
         ((uint64_t)((sbo & 0x3FFFFu) >> 4) << 32) | ((uint64_t)1 << 46);
}

// Instruction descriptor of kind::f16: D in FP32, A and B BF16, both K-major, dense, M x N.
__host__ __device__ constexpr uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

// Bounded wait for the phase of parity `parity` of an mbarrier: false after `limit` polls.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int limit) {
  for (int i = 0; i < limit; ++i) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// 8 consecutive FP32 accumulator columns of the warp's 32 TMEM lanes (one lane per thread); the
// wait carries the registers so that nothing reads them before the load has completed
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7])
               :
               : "memory");
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = __uint_as_float(r[j]);
}

// 16-byte asynchronous copy global -> shared; with valid = false the 16 bytes are zero-filled and
// nothing is read (src must still be a mapped address)
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

// ---------------------------------------------------------------- 3x3 convolution (implicit GEMM)
// Y[p][co] = sum_{tap, ci} X[p + off(tap)][ci] Wt[tap][ci][co] (+ bias[co]), p = r W + q, then
//   MODE 0: Yb = bf16(relu(.))                          (hidden layer forward)
//   MODE 1: Yf = float(.)                               (output layer forward)
//   MODE 2: Yb = bf16(. * (mask[p][co] > 0))            (backward through the data: mask = a)
// One warp computes 16 pixels x COUT; 8 warps per block; blockIdx.y = sample.
template <int CIN, int COUT, int MODE>
__global__ void __launch_bounds__(256) k_conv3x3(const __nv_bfloat16* __restrict__ X,
                                                 const __nv_bfloat16* __restrict__ Wt,
                                                 const float* __restrict__ bias, int H, int W,
                                                 __nv_bfloat16* __restrict__ Yb, float* __restrict__ Yf,
                                                 const __nv_bfloat16* __restrict__ mask) {
  __shared__ __nv_bfloat16 ws[9 * CIN * COUT];
  const int P = H * W;
  const size_t xo = (size_t)blockIdx.y * P * CIN, yo = (size_t)blockIdx.y * P * COUT;
  X += xo;
  for (int i = threadIdx.x; i < 9 * CIN * COUT; i += blockDim.x) ws[i] = Wt[i];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int p0 = (blockIdx.x * 8 + warp) * 16;
  if (p0 >= P) return;  // whole warp leaves together
  const int pa = p0 + g, pb = p0 + g + 8;  // the two pixel rows this lane feeds
  const int ra = pa / W, qa = pa % W, rb = pb / W, qb = pb % W;
  const bool va = pa < P, vb = pb < P;
  float acc[COUT / 8][4];
#pragma unroll
  for (int n = 0; n < COUT / 8; ++n)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[n][e] = 0.f;
#pragma unroll 1
  for (int tap = 0; tap < 9; ++tap) {
    const int dy = tap / 3 - 1, dx = tap % 3 - 1;
#pragma unroll
    for (int c0 = 0; c0 < CIN; c0 += 16) {
      uint32_t a[4];
      a[0] = va ? load_pair(X, H, W, CIN, ra + dy, qa + dx, c0 + 2 * t) : 0u;
      a[1] = vb ? load_pair(X, H, W, CIN, rb + dy, qb + dx, c0 + 2 * t) : 0u;
      a[2] = va ? load_pair(X, H, W, CIN, ra + dy, qa + dx, c0 + 2 * t + 8) : 0u;
      a[3] = vb ? load_pair(X, H, W, CIN, rb + dy, qb + dx, c0 + 2 * t + 8) : 0u;
      const __nv_bfloat16* wk = ws + (tap * CIN + c0) * COUT;
#pragma unroll
      for (int n = 0; n < COUT / 8; ++n) {
        const int co = n * 8 + g;
        uint32_t b[2];
        b[0] = pack_bf16(wk[(2 * t) * COUT + co], wk[(2 * t + 1) * COUT + co]);
        b[1] = pack_bf16(wk[(2 * t + 8) * COUT + co], wk[(2 * t + 9) * COUT + co]);
        mma_bf16(acc[n], a, b);
      }
    }
  }
#pragma unroll
  for (int n = 0; n < COUT / 8; ++n) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int p = (e < 2) ? pa : pb;
      if (p >= P) continue;
      const int co = n * 8 + 2 * t + (e & 1);
      float v = acc[n][e] + (bias ? bias[co] : 0.f);
      if (MODE == 0) {
        Yb[yo + (size_t)p * COUT + co] = __float2bfloat16_rn(v > 0.f ? v : 0.f);
      } else if (MODE == 1) {
        Yf[yo + (size_t)p * COUT + co] = v;
      } else {
        const float m = __bfloat162float(mask[yo + (size_t)p * COUT + co]);
        Yb[yo + (size_t)p * COUT + co] = __float2bfloat16_rn(m > 0.f ? v : 0.f);
      }
    }
  }
}

// ---------------------------------------------------------------- 3x3 convolution on tcgen05
// The same implicit GEMM and epilogues as k_conv3x3 on the fifth-generation tensor cores.  A tile is
// a segment of at most 128 pixels of one image row (M = 128 accumulator rows, one per pixel) x N
// output channels (N = COUT, at least 16 as the M = 128 shape requires; padded rows of B are zero)
// over K = 9 taps x CIN channels.  No im2col tile is built: the block stages the three input row
// bands the tile's taps read -- rows r - 1, r, r + 1, from one pixel left of the segment to one
// right of it, zero outside the image -- in shared memory as arrays of 16-byte pixel rows, one
// array per group of 8 channels (the K-major canonical layout without swizzle: 8 consecutive
// pixel rows form a core matrix).  Tap (dy, dx) is then the same arrays read from band dy, one
// pixel row further for each step of dx: each MMA's A operand is a descriptor into the bands, and
// the bands are contiguous in the NHWC image, so the block reads them with coalesced 16-byte
// loads.  Blocks are persistent over tiles: they stage the weights B (N x K) and allocate the
// tensor-memory accumulator once; per tile one thread issues the 9 CIN / 16 MMAs (M = 128, N,
// K = 16) and commits them to an mbarrier (phase = tile parity), and each warp reads its 32
// accumulator lanes back with tcgen05.ld for a vectorised epilogue.  A wait that runs out records
// the failure in *err, waits once more (bounded) for the MMAs, and ends the block's tiles; the
// block always frees its tensor memory.  With `withhold` (a host-set test of that path) no MMA is
// issued or committed, so the wait (then of wait_limit = 256 polls) runs out in every block.
constexpr int TC_M = 128;
constexpr int TC_WAIT = 1 << 20;
constexpr int TC_ROWS = TC_M + 2;             // pixel rows of a band: the segment and one each side
constexpr int TC_CGS = (TC_ROWS + 7) * 16;    // bytes per 8-channel array of a band (2192: not a
                                              // multiple of 128, so the staging stores spread over banks)

template <int CIN, int COUT>
constexpr int tc_smem_bytes() {
  return (COUT < 16 ? 16 : COUT) * 9 * CIN * 2 + 3 * (CIN / 8) * TC_CGS + 16;
}

// tiles of an H x W image: each row split into nseg segments of at most seg <= TC_M pixels
struct TcTiles {
  int nseg, seg;
};
inline TcTiles tc_tiles(int W) {
  const int nseg = (W + TC_M - 1) / TC_M;
  return {nseg, (W + nseg - 1) / nseg};
}

template <int CIN, int COUT, int MODE>
__global__ void __launch_bounds__(TC_M) k_conv3x3_tc(const __nv_bfloat16* __restrict__ X,
                                                     const __nv_bfloat16* __restrict__ Wt,
                                                     const float* __restrict__ bias, int H, int W, int nseg,
                                                     int seg, int B, __nv_bfloat16* __restrict__ Yb,
                                                     float* __restrict__ Yf, const __nv_bfloat16* __restrict__ mask,
                                                     int* __restrict__ err, int wait_limit, int withhold) {
  constexpr int N = COUT < 16 ? 16 : COUT;
  constexpr int CG = CIN / 8, K = 9 * CIN, KB = K / 8, NB = N / 8;
  constexpr uint32_t TMEM_COLS = 32;  // a power of two >= 32 holding the N FP32 columns
  static_assert(CIN % 16 == 0 && COUT % 8 == 0 && N % 16 == 0 && N <= 32, "tile shape");
  extern __shared__ __align__(1024) unsigned char tc_smem[];
  unsigned char* sB = tc_smem;                // B: core matrix (kb, nb) at (kb NB + nb) x 128 bytes
  unsigned char* sX = tc_smem + N * K * 2;    // bands: array (band, cg) at (band CG + cg) x TC_CGS
  uint64_t* bar = reinterpret_cast<uint64_t*>(sX + 3 * CG * TC_CGS);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 1);
  const int P = H * W;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int ntiles = B * H * nseg;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tslot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(bar)));
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  // B: Wt is already in the canonical layout (k_ws_tc_layout): copied as it is
  for (int c = tid; c < KB * N; c += TC_M) cp_async16(smem_u32(sB) + c * 16, Wt + c * 8, true);  // N K / 8 chunks
  cp_async_wait_all();
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = *tslot;
  constexpr uint32_t idesc = tc_idesc(TC_M, N);
  int it = 0;
  for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++it) {
    const int smp = t / (H * nseg), rt = t - smp * (H * nseg);
    const int r = rt / nseg, c0 = (rt - r * nseg) * seg, len = min(seg, W - c0);
    const __nv_bfloat16* Xs = X + (size_t)smp * P * CIN;
    // bands: row j of array (band, cg) = channels 8 cg .. 8 cg + 7 of pixel (r + band - 1, c0 - 1 + j)
    for (int f = tid; f < 3 * TC_ROWS * CG; f += TC_M) {
      const int cg = f % CG, j = (f / CG) % TC_ROWS, band = f / (CG * TC_ROWS);
      const int rr = r + band - 1, qq = c0 - 1 + j;
      const bool in = j < len + 2 && rr >= 0 && rr < H && qq >= 0 && qq < W;
      cp_async16(smem_u32(sX + (band * CG + cg) * TC_CGS + j * 16),
                 in ? Xs + ((size_t)rr * W + qq) * CIN + cg * 8 : Xs, in);  // zero outside the image
    }
    cp_async_wait_all();
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");  // shared writes -> tensor core reads
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (tid == 0 && !withhold) {  // withhold: a test of the timeout path (nothing arrives)
#pragma unroll 1
      for (int tap = 0; tap < 9; ++tap) {
        const int band = tap / 3, dx = tap % 3;  // input row r + band - 1, column offset dx - 1
#pragma unroll
        for (int kp = 0; kp < CG / 2; ++kp) {
          const uint64_t ad = tc_desc(smem_u32(sX) + (band * CG + 2 * kp) * TC_CGS + dx * 16, TC_CGS, 128);
          const uint64_t bd = tc_desc(smem_u32(sB) + (tap * CG + 2 * kp) * NB * 128, NB * 128, 128);
          tc_mma(tmem, ad, bd, idesc, (tap | kp) != 0);
        }
      }
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                       smem_u32(bar))
                   : "memory");
    }
    const bool ok = mbar_wait(smem_u32(bar), it & 1, wait_limit);
    if (__syncthreads_or(!ok)) {
      if (tid == 0) atomicExch(err, 1);
      mbar_wait(smem_u32(bar), it & 1, wait_limit);  // the MMAs may still be running: a last bound
      break;
    }
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    float acc[N];
#pragma unroll
    for (int c8 = 0; c8 < NB; ++c8) {
      float v[8];
      tmem_ld8(tmem + ((uint32_t)(warp * 32) << 16) + c8 * 8, v);
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[c8 * 8 + j] = v[j];
    }
    if (tid < len) {  // accumulator lane tid = pixel c0 + tid of row r
      const size_t o = ((size_t)smp * P + (size_t)r * W + c0 + tid) * COUT;
      if (MODE == 1) {
#pragma unroll
        for (int c4 = 0; c4 < COUT / 4; ++c4) {
          float4 v;
          v.x = acc[4 * c4 + 0] + (bias ? bias[4 * c4 + 0] : 0.f);
          v.y = acc[4 * c4 + 1] + (bias ? bias[4 * c4 + 1] : 0.f);
          v.z = acc[4 * c4 + 2] + (bias ? bias[4 * c4 + 2] : 0.f);
          v.w = acc[4 * c4 + 3] + (bias ? bias[4 * c4 + 3] : 0.f);
          *reinterpret_cast<float4*>(Yf + o + 4 * c4) = v;
        }
      } else {
#pragma unroll
        for (int c8 = 0; c8 < COUT / 8; ++c8) {
          uint4 m4 = make_uint4(0u, 0u, 0u, 0u);
          if (MODE == 2) m4 = *reinterpret_cast<const uint4*>(mask + o + 8 * c8);
          const uint32_t mw[4] = {m4.x, m4.y, m4.z, m4.w};
          uint32_t packed[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const int co = 8 * c8 + 2 * j;
            float a = acc[co] + (bias ? bias[co] : 0.f), b = acc[co + 1] + (bias ? bias[co + 1] : 0.f);
            if (MODE == 0) {
              a = a > 0.f ? a : 0.f;
              b = b > 0.f ? b : 0.f;
            } else {
              a = __uint_as_float(mw[j] << 16) > 0.f ? a : 0.f;           // bf16 (low half) -> fp32
              b = __uint_as_float(mw[j] & 0xFFFF0000u) > 0.f ? b : 0.f;  // bf16 (high half)
            }
            packed[j] = pack_bf16(__float2bfloat16_rn(a), __float2bfloat16_rn(b));
          }
          *reinterpret_cast<uint4*>(Yb + o + 8 * c8) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
        }
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();  // the next tile's staging and MMAs come after every read of this one
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(TMEM_COLS));
}

// ---------------------------------------------------------------- data movement
// Per-sample scales: dscale[smp][c] = RMS over the image of channel c of d = s - q, and
// dscale[smp][4 + c] that of D = s - 2 q + q2 (1 when q2 is null); at least 1e-30.  Two passes,
// both in a fixed order (deterministic): block (b, smp) of k_ws_rms_part sums the squares of
// pixels [b chunk, (b + 1) chunk) in FP64, thread-strided and then by a tree over its threads, into
// part[smp][b][8]; k_ws_rms_fin adds a sample's block partials in block order.
constexpr int WS_RMS_BLOCKS = 256;  // most blocks per sample of the first pass
constexpr int RN_BLOCKS = 152;      // most blocks of a residual norm (k_ws_resnorm)

// The four channels of pixel i (N x 4 node-major arrays): one vector load where the caller's array is
// aligned for it (al: 32 bytes for fp64, 16 for fp32), four scalar loads otherwise.
template <typename T> struct Quad { T x, y, z, w; };
__device__ __forceinline__ Quad<double> ld4(const double* p, size_t i, bool al) {
  if (al) {
    const double4_32a v = reinterpret_cast<const double4_32a*>(p)[i];
    return {v.x, v.y, v.z, v.w};
  }
  return {p[4 * i], p[4 * i + 1], p[4 * i + 2], p[4 * i + 3]};
}
__device__ __forceinline__ Quad<float> ld4(const float* p, size_t i, bool al) {
  if (al) {
    const float4 v = reinterpret_cast<const float4*>(p)[i];
    return {v.x, v.y, v.z, v.w};
  }
  return {p[4 * i], p[4 * i + 1], p[4 * i + 2], p[4 * i + 3]};
}
static bool aligned4(size_t elem, std::initializer_list<const void*> ps) {
  uintptr_t u = 0;
  for (const void* p : ps) u |= reinterpret_cast<uintptr_t>(p);
  return (u & (4 * elem - 1)) == 0;
}

template <typename T>
__global__ void k_ws_rms_part(const T* __restrict__ s, const T* __restrict__ q, const T* __restrict__ q2, int P,
                              int chunk, bool al, double* __restrict__ part) {
  __shared__ double red[8][256];
  const int smp = blockIdx.y, b = blockIdx.x;
  const int i0 = b * chunk, i1 = min(P, i0 + chunk);
  double acc[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (int i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    const size_t o = (size_t)smp * P + i;
    const Quad<T> sv = ld4(s, o, al), qv = ld4(q, o, al), q2v = q2 ? ld4(q2, o, al) : Quad<T>{};
    const T sc[4] = {sv.x, sv.y, sv.z, sv.w}, qc[4] = {qv.x, qv.y, qv.z, qv.w}, q2c[4] = {q2v.x, q2v.y, q2v.z, q2v.w};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const double a = sc[c], bq = qc[c];
      const double d = a - bq;
      acc[c] = fma(d, d, acc[c]);
      if (q2) {
        const double D = a - 2.0 * bq + (double)q2c[c];
        acc[4 + c] = fma(D, D, acc[4 + c]);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) red[c][threadIdx.x] = acc[c];
  __syncthreads();
  for (int h = 128; h > 0; h >>= 1) {
    if (threadIdx.x < h) {
#pragma unroll
      for (int c = 0; c < 8; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + h];
    }
    __syncthreads();
  }
  if (threadIdx.x < 8) part[((size_t)smp * gridDim.x + b) * 8 + threadIdx.x] = red[threadIdx.x][0];
}

__global__ void k_ws_rms_fin(const double* __restrict__ part, int nblk, int P, int has_q2, float* __restrict__ dscale,
                             double* __restrict__ dinv) {
  const int smp = blockIdx.x, c = threadIdx.x;
  if (c >= 8) return;
  double sum = 0.0;
  for (int b = 0; b < nblk; ++b) sum += part[((size_t)smp * nblk + b) * 8 + c];
  const float d = (c >= 4 && !has_q2) ? 1.f : (float)fmax(sqrt(sum / (double)P), 1e-30);
  dscale[smp * 8 + c] = d;
  dinv[smp * 8 + c] = 1.0 / (double)d;
}

// dinv = 1 / dscale in FP64: the per-pixel kernels multiply by it (an FP64 division per channel and
// pixel bound them: packing 8 x 257 x 257 pixels took 100 us).
// Input image of the network from the states s, q, q2 (N x 4 each, fp64 node major or fp32
// sample-major): channels 0-3 = (s - mean[0:4]) * inv_std[0:4] (the fields at step k), channels
// 4-7 = ((s - q) / r1 - mean[4:8]) * inv_std[4:8] (the last change in units of its RMS), channels
// 8-11 = (s - 2 q + q2) / r2 (the second difference in units of its RMS), channels 12-15 zero.
template <typename T>
__global__ void k_ws_pack(const T* __restrict__ s, const T* __restrict__ q, const T* __restrict__ q2, int P, bool al,
                          const float* __restrict__ mean, const float* __restrict__ inv_std,
                          const double* __restrict__ dinv, __nv_bfloat16* __restrict__ x) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;  // pixel; blockIdx.y = sample
  const int smp = blockIdx.y;
  if (i >= (size_t)P) return;
  const size_t o = (size_t)smp * P + i;
  const Quad<T> sv = ld4(s, o, al), qv = ld4(q, o, al), q2v = ld4(q2, o, al);
  const T a[4] = {sv.x, sv.y, sv.z, sv.w}, b[4] = {qv.x, qv.y, qv.z, qv.w}, b2[4] = {q2v.x, q2v.y, q2v.z, q2v.w};
  const double* sc = dinv + smp * 8;
  float v[12];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    v[c] = ((float)a[c] - mean[c]) * inv_std[c];
    const double d = ((double)a[c] - (double)b[c]) * sc[c];
    v[4 + c] = ((float)d - mean[4 + c]) * inv_std[4 + c];
    const double D = (double)a[c] - 2.0 * (double)b[c] + (double)b2[c];
    v[8 + c] = (float)(D * sc[4 + c]);
  }
  uint32_t w[8] = {};
#pragma unroll
  for (int c = 0; c < 6; ++c) w[c] = pack_bf16(__float2bfloat16_rn(v[2 * c]), __float2bfloat16_rn(v[2 * c + 1]));
  uint4* dst = reinterpret_cast<uint4*>(x + o * WS_CIN);
  dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
  dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
}

// State-space error of the prediction in units of the change's RMS, E = (theta D - e) / r1 with
// theta = y out_scale, D = s - 2 q + q2 and e = n - 2 s + q (the linear extrapolation's error), and
// the factor dE/dy = out_scale D / r1 (fp32 inputs, sample-major B x N x 4).
__global__ void k_ws_err_theta(const float* __restrict__ y, const float* __restrict__ s, const float* __restrict__ q,
                               const float* __restrict__ q2, const float* __restrict__ n, int P,
                               const float* __restrict__ out_scale, const double* __restrict__ dinv,
                               float* __restrict__ e, float* __restrict__ fac) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int smp = blockIdx.y;
  if (i >= (size_t)P) return;
  const size_t o = ((size_t)smp * P + i) * 4;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const double a = s[o + c], b = q[o + c];
    const double D = a - 2.0 * b + (double)q2[o + c];
    const double err = (double)n[o + c] - 2.0 * a + b;
    const double r1i = dinv[smp * 8 + c], os = out_scale[c];
    const double th = (double)y[((size_t)smp * P + i) * WS_COUT + c] * os;
    e[o + c] = (float)((th * D - err) * r1i);
    fac[o + c] = (float)(os * D * r1i);
  }
}

// pred = s + (s - q) + y * out_scale * (s - 2 q + q2) (fp64, N x 4): the learned second-order
// extrapolation
__global__ void k_ws_unpack(const double* __restrict__ s, const double* __restrict__ q, const double* __restrict__ q2,
                            const float* __restrict__ y, int P, bool al, const float* __restrict__ out_scale,
                            double* __restrict__ pred) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P) return;
  const Quad<double> a = ld4(s, i, al), b = ld4(q, i, al), b2 = ld4(q2, i, al);
  const float4 yv = *reinterpret_cast<const float4*>(y + (size_t)i * WS_COUT);
  const double p0 = a.x + (a.x - b.x) + (double)yv.x * (double)out_scale[0] * (a.x - 2.0 * b.x + b2.x);
  const double p1 = a.y + (a.y - b.y) + (double)yv.y * (double)out_scale[1] * (a.y - 2.0 * b.y + b2.y);
  const double p2 = a.z + (a.z - b.z) + (double)yv.z * (double)out_scale[2] * (a.z - 2.0 * b.z + b2.z);
  const double p3 = a.w + (a.w - b.w) + (double)yv.w * (double)out_scale[3] * (a.w - 2.0 * b.w + b2.w);
  if (al) {
    reinterpret_cast<double4_32a*>(pred)[i] = make_double4_32a(p0, p1, p2, p3);
  } else {
    double* o = pred + (size_t)i * 4;
    o[0] = p0;
    o[1] = p1;
    o[2] = p2;
    o[3] = p3;
  }
}

// Loss on the 4 used output channels, L = (sum E^2 + lap * sum (G E)^2) / count with E the error
// above and G the graph Laplacian of the pixel grid, (G E)_p = sum over the 4-neighbours q of p
// inside the image of (E_q - E_p).  The second term weighs errors the way the stiffness rows of
// the step's residual do.  Two passes after E: G E with the per-block partial losses (summed in
// block order), then dy = 2 (E + lap G (G E)) / count * dE/dy as a bf16 NHWC image with 16
// channels.
__device__ __forceinline__ float4 grid_laplacian(const float* __restrict__ e, int H, int W, size_t base, int r, int q) {
  const float4 c = *reinterpret_cast<const float4*>(e + (base + (size_t)r * W + q) * 4);
  float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
  const int dr[4] = {-1, 1, 0, 0}, dq[4] = {0, 0, -1, 1};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int rr = r + dr[k], qq = q + dq[k];
    if (rr < 0 || rr >= H || qq < 0 || qq >= W) continue;
    const float4 n = *reinterpret_cast<const float4*>(e + (base + (size_t)rr * W + qq) * 4);
    g.x += n.x - c.x;
    g.y += n.y - c.y;
    g.z += n.z - c.z;
    g.w += n.w - c.w;
  }
  return g;
}

__global__ void k_ws_lap_loss(const float* __restrict__ e, int H, int W, int B, float lap,
                              float* __restrict__ ge, float* __restrict__ loss_part) {
  __shared__ float sm[256];
  const size_t P = (size_t)H * W, total = (size_t)B * P;
  float acc = 0.f;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const size_t smp = i / P, p = i % P;
    const float4 c = *reinterpret_cast<const float4*>(e + i * 4);
    acc = fmaf(c.x, c.x, fmaf(c.y, c.y, fmaf(c.z, c.z, fmaf(c.w, c.w, acc))));
    if (lap != 0.f) {
      const float4 g = grid_laplacian(e, H, W, smp * P, (int)(p / W), (int)(p % W));
      *reinterpret_cast<float4*>(ge + i * 4) = g;
      acc = fmaf(lap, g.x * g.x + g.y * g.y + g.z * g.z + g.w * g.w, acc);
    }
  }
  sm[threadIdx.x] = acc;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sm[threadIdx.x] += sm[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) loss_part[blockIdx.x] = sm[0];
}

__global__ void k_ws_dy(const float* __restrict__ e, const float* __restrict__ ge, const float* __restrict__ fac,
                        int H, int W, int B, float lap, __nv_bfloat16* __restrict__ dy) {
  const size_t P = (size_t)H * W, total = (size_t)B * P;
  const float scale = 2.f / (float)(total * 4);
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const size_t smp = i / P, p = i % P;
    float4 v = *reinterpret_cast<const float4*>(e + i * 4);
    if (lap != 0.f) {
      const float4 g = grid_laplacian(ge, H, W, smp * P, (int)(p / W), (int)(p % W));
      v.x = fmaf(lap, g.x, v.x);
      v.y = fmaf(lap, g.y, v.y);
      v.z = fmaf(lap, g.z, v.z);
      v.w = fmaf(lap, g.w, v.w);
    }
    const float vals[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int c = 0; c < 16; ++c) dy[i * 16 + c] = __float2bfloat16_rn(c < 4 ? scale * vals[c] * fac[i * 4 + c] : 0.f);
  }
}

// ---------------------------------------------------------------- weight gradients
// dW[tap][ci][co] = sum_p X[p + off(tap)][ci] dY[p][co], db[co] = sum_p dY[p][co]: per tap a GEMM with
// M = input channels, N = output channels and K = pixels, both operands stored pixel-major (K x M and
// K x N), which is what ldmatrix.trans turns into mma.sync fragments.  A block takes a strip of image
// rows of one column segment of one sample; per row it needs the input rows r - 1, r, r + 1 (a ring of
// four bands in shared memory, one new band and one dY row copied by cp.async while the row before
// is multiplied) and warp t < 9 multiplies tap t, whose A operand is the band (tap / 3) shifted by
// tap % 3 pixels.  Warp 9 adds the bias gradient.  A row's MMAs (FP32 accumulate) start from zero and
// are added to the strip's FP32 sums, so no accumulation chain is longer than a row or a strip.
// Each strip writes its own partial gradient; k_ws_reduce adds them in order (deterministic).
//
// Pixel rows are padded by 16 bytes (80 or 48 bytes: 8 consecutive pixels hit distinct banks).  The
// FP32-FMA form before it (one thread per (tap, ci), X read through L1 for every pixel) was bound by
// its loads: batch of 8 at 257 x 257, us per layer 664 / 873 / 469.
constexpr int WG_SEG = 160;     // most pixels of a segment
constexpr int WG_BLOCKS = 304;  // strips aimed at: two blocks on each of the 152 SMs
constexpr int WG_WARPS = 10;
struct WgTiles {
  int nseg, seg, rows, nstrip;  // column segments, pixels of one, image rows per strip, strips per segment
};
inline WgTiles wg_tiles(int H, int W, int B) {
  WgTiles t;
  t.nseg = (W + WG_SEG - 1) / WG_SEG;
  t.seg = (W + t.nseg - 1) / t.nseg;
  const int64_t rows = ((int64_t)H * t.nseg * B + WG_BLOCKS - 1) / WG_BLOCKS;
  t.rows = (int)(rows < 2 ? 2 : rows);
  t.nstrip = (H + t.rows - 1) / t.rows;
  return t;
}
template <int CIN, int COUTG>
constexpr int wg_smem(int kp) {
  return 4 * (kp + 2) * (2 * CIN + 16) + 2 * kp * (2 * COUTG + 16);
}

__device__ __forceinline__ void ldsm4_t(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

template <int CIN, int COUTG, int COUTW>  // COUTG: channels stored in dY; COUTW: channels of dW
__global__ void __launch_bounds__(32 * WG_WARPS) k_ws_wgrad(const __nv_bfloat16* __restrict__ X,
                                                            const __nv_bfloat16* __restrict__ dY, int H, int W,
                                                            int nseg, int seg, int rows, int kp,
                                                            float* __restrict__ partials) {
  constexpr int XS = 2 * CIN + 16, DS = 2 * COUTG + 16;  // bytes per pixel in shared memory
  constexpr int MT = CIN / 16, NT = COUTW / 8;
  extern __shared__ __align__(16) unsigned char wg_smem_raw[];
  const int P = H * W, smp = blockIdx.z, c0 = blockIdx.y * seg, len = min(seg, W - c0);
  const int r0 = blockIdx.x * rows, r1 = min(H, r0 + rows);
  const __nv_bfloat16* Xs = X + (size_t)smp * P * CIN;
  const __nv_bfloat16* Ds = dY + (size_t)smp * P * COUTG;
  const uint32_t sx = smem_u32(wg_smem_raw), sd = sx + 4 * (kp + 2) * XS;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // band of image row r: slot (r + 1) & 3, pixel j = column c0 - 1 + j, zero outside the image
  const auto load_band = [&](int r) {
    constexpr int CH = CIN / 8;  // 16-byte chunks per pixel
    const bool in_r = r >= 0 && r < H;
    for (int f = tid; f < (kp + 2) * CH; f += 32 * WG_WARPS) {
      const int j = f / CH, ch = f % CH, q = c0 - 1 + j;
      const bool in = in_r && q >= 0 && q < W && j < len + 2;
      cp_async16(sx + ((r + 1) & 3) * (kp + 2) * XS + j * XS + ch * 16,
                 in ? Xs + ((size_t)r * W + q) * CIN + ch * 8 : Xs, in);
    }
  };
  const auto load_dy = [&](int r) {
    constexpr int CH = COUTG / 8;
    for (int f = tid; f < kp * CH; f += 32 * WG_WARPS) {
      const int j = f / CH, ch = f % CH;
      const bool in = j < len && r < r1;
      cp_async16(sd + (r & 1) * kp * DS + j * DS + ch * 16,
                 in ? Ds + ((size_t)r * W + c0 + j) * COUTG + ch * 8 : Ds, in);
    }
  };
  const auto commit = [] { asm volatile("cp.async.commit_group;\n" ::: "memory"); };
  load_band(r0 - 1);
  load_band(r0);
  load_band(r0 + 1);
  load_dy(r0);
  commit();
  float sum[MT][NT][4] = {};
  float bsum[2] = {0.f, 0.f};
  constexpr int NPAIR = COUTW / 2, PAR = 32 / NPAIR;  // bias warp: lane = channel pair + NPAIR x pixel class
  for (int r = r0; r < r1; ++r) {
    load_band(r + 2);  // the next row's new band and dY, in flight while this row is multiplied
    load_dy(r + 1);
    commit();
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();
    const uint32_t dy = sd + (r & 1) * kp * DS;
    if (warp < 9) {
      const int band = r + warp / 3 - 1, dx = warp % 3;
      const uint32_t xb = sx + ((band + 1) & 3) * (kp + 2) * XS + dx * XS;
      float acc[MT][NT][4] = {};
      const int q = lane >> 3, l8 = lane & 7;
      for (int k0 = 0; k0 < kp; k0 += 16) {
        uint32_t a[MT][4], b[(NT + 1) / 2][4];
#pragma unroll
        for (int m = 0; m < MT; ++m)  // matrices (k half, m half): q >> 1, q & 1
          ldsm4_t(a[m], xb + (k0 + (q >> 1) * 8 + l8) * XS + (m * 16 + (q & 1) * 8) * 2);
#pragma unroll
        for (int n = 0; n < (NT + 1) / 2; ++n) {  // matrices (k half, n half): q & 1, q >> 1 (one n tile: q >> 1 = 0)
          const int nh = NT > 1 ? q >> 1 : 0;
          ldsm4_t(b[n], dy + (k0 + (q & 1) * 8 + l8) * DS + (n * 16 + nh * 8) * 2);
        }
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
          for (int n = 0; n < NT; ++n) {
            const uint32_t bb[2] = {b[n / 2][2 * (n & 1)], b[n / 2][2 * (n & 1) + 1]};
            mma_bf16(acc[m][n], a[m], bb);
          }
      }
#pragma unroll
      for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int e = 0; e < 4; ++e) sum[m][n][e] += acc[m][n][e];
    } else {
      const unsigned char* row = wg_smem_raw + (dy - sx) + (lane % NPAIR) * 4;
      float t0 = 0.f, t1 = 0.f;
      for (int j = lane / NPAIR; j < len; j += PAR) {
        const uint32_t v = *reinterpret_cast<const uint32_t*>(row + j * DS);
        t0 += __uint_as_float(v << 16);
        t1 += __uint_as_float(v & 0xFFFF0000u);
      }
      bsum[0] += t0;
      bsum[1] += t1;
    }
    __syncthreads();  // every read of band r - 1 and of this dY row precedes the next copies into them
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");  // the last prefetch
  float* out = partials + (((size_t)smp * nseg + blockIdx.y) * gridDim.x + blockIdx.x) * (9 * CIN * COUTW + COUTW);
  if (warp < 9) {
    const int g = lane >> 2, t = lane & 3;
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int n = 0; n < NT; ++n)
#pragma unroll
        for (int e = 0; e < 4; ++e)
          out[(warp * CIN + m * 16 + g + (e >> 1) * 8) * COUTW + n * 8 + 2 * t + (e & 1)] = sum[m][n][e];
  } else {
#pragma unroll
    for (int o = NPAIR; o < 32; o <<= 1) {
      bsum[0] += __shfl_xor_sync(0xffffffffu, bsum[0], o);
      bsum[1] += __shfl_xor_sync(0xffffffffu, bsum[1], o);
    }
    if (lane < NPAIR) {
      out[9 * CIN * COUTW + 2 * lane] = bsum[0];
      out[9 * CIN * COUTW + 2 * lane + 1] = bsum[1];
    }
  }
}

// sum of nparts partial gradient vectors of length len: eight threads per value take a contiguous
// eighth of the parts each, in part order, and their sums are added in order
__global__ void __launch_bounds__(256) k_ws_reduce(const float* __restrict__ partials, int nparts, int len,
                                                   float* __restrict__ g) {
  __shared__ float sm[8][32];
  const int i = blockIdx.x * 32 + threadIdx.x, y = threadIdx.y;
  const int per = (nparts + 7) / 8, k0 = y * per, k1 = min(nparts, k0 + per);
  float s = 0.f;
  if (i < len) {
#pragma unroll 8
    for (int k = k0; k < k1; ++k) s += partials[(size_t)k * len + i];
  }
  sm[y][threadIdx.x] = s;
  __syncthreads();
  if (y == 0 && i < len) {
    float t = sm[0][threadIdx.x];
#pragma unroll
    for (int q = 1; q < 8; ++q) t += sm[q][threadIdx.x];
    g[i] = t;
  }
}

// Adam (Kingma & Ba 2015) on the FP32 master parameters
__global__ void k_ws_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                          float* __restrict__ v, int n, float lr, float b1, float b2, float eps,
                          float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// The weights of one convolution (Wt[k][co], k = tap CIN + ci) as the tcgen05 path's B operand:
// N x K (N >= COUT output channels, padded rows zero) in the K-major canonical layout of 8-row x
// 16-byte core matrices, core matrix (kb, nb) at element (kb N/8 + nb) x 64, row n % 8 of it at
// (n % 8) x 8; a block copies it to shared memory as it is.
__global__ void k_ws_tc_layout(const __nv_bfloat16* __restrict__ Wt, int K, int cout, int N,
                               __nv_bfloat16* __restrict__ out) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= N * K) return;
  const int NB = N / 8, c = idx / 8, e = idx % 8;
  const int kb = c / (NB * 8), rem = c % (NB * 8), n = (rem / 8) * 8 + rem % 8;
  const int k = kb * 8 + e;
  out[idx] = n < cout ? Wt[k * cout + n] : __float2bfloat16_rn(0.f);
}

// BF16 copies of the weights: forward [tap][ci][co] and, for the backward pass through the data,
// flipped [8 - tap][co][ci] with the channel counts of that pass (co padded to CPAD rows).
__global__ void k_ws_bf16(const float* __restrict__ w, int cin, int cout, int cout_used, int cpad,
                          __nv_bfloat16* __restrict__ fwd, __nv_bfloat16* __restrict__ flip) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < 9 * cin * cout) {
    const int co = i % cout;
    fwd[i] = __float2bfloat16_rn(co < cout_used ? w[i] : 0.f);
  }
  if (flip && i < 9 * cpad * cin) {  // flip[tap'][c][ci], c < cpad
    const int ci = i % cin, c = (i / cin) % cpad, tp = i / (cin * cpad);
    const float val = c < cout_used ? w[((8 - tp) * cin + ci) * cout + c] : 0.f;
    flip[i] = __float2bfloat16_rn(val);
  }
}

}  // namespace ch

// ---------------------------------------------------------------- handle
struct ch_ws_s {
  int H = 0, W = 0, P = 0, Bmax = 0;
  float* params = nullptr;  // FP32 master, WS_NPARAM
  float* grads = nullptr;
  float* adam_m = nullptr;
  float* adam_v = nullptr;
  int adam_t = 0;
  __nv_bfloat16 *w1 = nullptr, *w2 = nullptr, *w3 = nullptr;     // forward copies
  __nv_bfloat16 *w2f = nullptr, *w3f = nullptr;                    // flipped copies (backward)
  __nv_bfloat16 *c1 = nullptr, *c2 = nullptr, *c3 = nullptr;       // the same as tcgen05 B operands
  __nv_bfloat16 *c2f = nullptr, *c3f = nullptr;
  float* norm = nullptr;  // mean[8], inv_std[8], out_scale[4]
  double* dinv = nullptr;   // 1 / dscale
  float* dscale = nullptr;  // Bmax x 8: RMS of the last change and of the second difference per sample and channel
  float* t = nullptr;       // Bmax x P x 4: dE/dy of the state-space loss
  float* e = nullptr;       // Bmax x P x 4 output errors y - t
  float* ge = nullptr;      // Bmax x P x 4 their grid Laplacian
  double* rex = nullptr;    // Bmax x P x 4 residuals of the extrapolation (residual loss)
  double* rres = nullptr;   // Bmax x P x 4 residuals of the prediction
  double *tmp1 = nullptr, *tmp2 = nullptr;  // P x 4
  double* nrm = nullptr;    // Bmax x 8 squared residual norms per channel
  double* rn_part = nullptr;          // the residual norms' block partials
  unsigned int* rn_ticket = nullptr;  // ... and their last-block counter
  double *zex = nullptr, *zr = nullptr;  // preconditioned residuals: P x 4, Bmax x P x 4
  __nv_bfloat16 *x0 = nullptr, *a1 = nullptr, *a2 = nullptr;      // Bmax x P x {16, 32, 32}
  __nv_bfloat16 *dy = nullptr, *dz2 = nullptr, *dz1 = nullptr;    // Bmax x P x {16, 32, 32}
  float* y = nullptr;                                              // Bmax x P x 8
  float* part = nullptr;                                           // weight-gradient partials
  float* loss_part = nullptr;
  double* rms_part = nullptr;  // Bmax x WS_RMS_BLOCKS x 8: first-pass partials of the RMS scales
  bool fresh = false;  // bf16 copies up to date
  int engine = 1;      // convolutions: 0 mma.sync (warp-level), 1 tcgen05 (tensor memory)
  int withhold = 0;    // test of the timeout path: tcgen05 blocks issue no MMA, so their wait runs out
  int* err_host = nullptr;  // pinned, device-mapped: set by a tcgen05 block whose MMA wait ran out
  int* err_dev = nullptr;
  ch::Alloc mem;
  ~ch_ws_s() {
    if (err_host) cudaFreeHost(err_host);
  }
};

namespace ch {

static WsParams ws_views(float* base) {
  WsParams v;
  v.w1 = base;
  v.b1 = v.w1 + WS_N1;
  v.w2 = v.b1 + WS_C;
  v.b2 = v.w2 + WS_N2;
  v.w3 = v.b2 + WS_C;
  v.b3 = v.w3 + WS_N3;
  return v;
}

static ch_status ws_refresh(ch_ws_s* w, cudaStream_t st) {
  const WsParams p = ws_views(w->params);
  k_ws_bf16<<<blocks_for(9 * WS_CIN * WS_C), TPB, 0, st>>>(p.w1, WS_CIN, WS_C, WS_C, 0, w->w1, nullptr);
  k_ws_bf16<<<blocks_for(9 * WS_C * WS_C), TPB, 0, st>>>(p.w2, WS_C, WS_C, WS_C, WS_C, w->w2, w->w2f);
  k_ws_bf16<<<blocks_for(9 * 16 * WS_C), TPB, 0, st>>>(p.w3, WS_C, WS_COUT, 4, 16, w->w3, w->w3f);
  k_ws_tc_layout<<<blocks_for(9 * WS_CIN * WS_C), TPB, 0, st>>>(w->w1, 9 * WS_CIN, WS_C, WS_C, w->c1);
  k_ws_tc_layout<<<blocks_for(9 * WS_C * WS_C), TPB, 0, st>>>(w->w2, 9 * WS_C, WS_C, WS_C, w->c2);
  k_ws_tc_layout<<<blocks_for(9 * WS_C * 16), TPB, 0, st>>>(w->w3, 9 * WS_C, WS_COUT, 16, w->c3);
  k_ws_tc_layout<<<blocks_for(9 * WS_C * WS_C), TPB, 0, st>>>(w->w2f, 9 * WS_C, WS_C, WS_C, w->c2f);
  k_ws_tc_layout<<<blocks_for(9 * 16 * WS_C), TPB, 0, st>>>(w->w3f, 9 * 16, WS_C, WS_C, w->c3f);
  CH_LAUNCHED();
  w->fresh = true;
  return CH_OK;
}

// The convolutions' shared-memory limits on the tcgen05 path (above the 48 KB default).
static ch_status ws_tc_setup() {
  CH_CUDA(cudaFuncSetAttribute(k_conv3x3_tc<WS_CIN, WS_C, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               tc_smem_bytes<WS_CIN, WS_C>()));
  CH_CUDA(cudaFuncSetAttribute(k_conv3x3_tc<WS_C, WS_C, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               tc_smem_bytes<WS_C, WS_C>()));
  CH_CUDA(cudaFuncSetAttribute(k_conv3x3_tc<WS_C, WS_COUT, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               tc_smem_bytes<WS_C, WS_COUT>()));
  CH_CUDA(cudaFuncSetAttribute(k_conv3x3_tc<16, WS_C, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               tc_smem_bytes<16, WS_C>()));
  CH_CUDA(cudaFuncSetAttribute(k_conv3x3_tc<WS_C, WS_C, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               tc_smem_bytes<WS_C, WS_C>()));
  const int kp = (WG_SEG + 15) / 16 * 16;
  CH_CUDA(cudaFuncSetAttribute(k_ws_wgrad<WS_C, 16, WS_COUT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               wg_smem<WS_C, 16>(kp)));
  CH_CUDA(cudaFuncSetAttribute(k_ws_wgrad<WS_C, WS_C, WS_C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               wg_smem<WS_C, WS_C>(kp)));
  CH_CUDA(cudaFuncSetAttribute(k_ws_wgrad<WS_CIN, WS_C, WS_C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               wg_smem<WS_CIN, WS_C>(kp)));
  return CH_OK;
}

// The per-sample RMS scales of B samples into w->dscale (two fixed-order passes).
template <typename T>
static void ws_rms(ch_ws_s* w, const T* s, const T* q, const T* q2, int B, cudaStream_t st) {
  const int P = w->P;
  const int chunk = std::max(1024, (P + WS_RMS_BLOCKS - 1) / WS_RMS_BLOCKS);
  const int nblk = (P + chunk - 1) / chunk;
  k_ws_rms_part<T><<<dim3(nblk, B), 256, 0, st>>>(s, q, q2, P, chunk, aligned4(sizeof(T), {s, q, q2}), w->rms_part);
  k_ws_rms_fin<<<B, 32, 0, st>>>(w->rms_part, nblk, P, q2 != nullptr, w->dscale, w->dinv);
}

// One convolution of B samples on the handle's engine.
template <int CIN, int COUT, int MODE>
static void ws_conv(ch_ws_s* w, const __nv_bfloat16* X, const __nv_bfloat16* Wt, const __nv_bfloat16* Bc,
                    const float* bias, __nv_bfloat16* Yb, float* Yf, const __nv_bfloat16* mask, int B,
                    cudaStream_t st) {
  if (w->engine == 1) {
    const TcTiles tt = tc_tiles(w->W);
    const int ntiles = B * w->H * tt.nseg;
    k_conv3x3_tc<CIN, COUT, MODE><<<std::min(ntiles, 4 * 152), TC_M, tc_smem_bytes<CIN, COUT>(), st>>>(
        X, Bc, bias, w->H, w->W, tt.nseg, tt.seg, B, Yb, Yf, mask, w->err_dev, w->withhold ? 256 : TC_WAIT,
        w->withhold);
  } else {
    k_conv3x3<CIN, COUT, MODE><<<dim3(blocks_for(w->P, 128), B), 256, 0, st>>>(X, Wt, bias, w->H, w->W, Yb, Yf,
                                                                                 mask);
  }
}

// The flag a tcgen05 convolution block sets when its MMA wait ran out (read after the host has
// synchronised with the work that could set it).
ch_status ws_check(const ch_ws_s* w) {
  if (w->err_host && *reinterpret_cast<volatile int*>(w->err_host)) {
    *reinterpret_cast<volatile int*>(w->err_host) = 0;  // reported once; later calls start clean
    set_error("warm start: a tcgen05 convolution block timed out waiting for its MMAs");
    return CH_ERR_INTERNAL;
  }
  return CH_OK;
}

ch_status ws_withhold_mma(ch_ws_s* w, int on) {
  w->withhold = on;
  return CH_OK;
}

ch_status ws_set_engine(ch_ws_s* w, int engine) {
  w->engine = engine;
  return CH_OK;
}

// forward pass of B samples whose inputs are already packed in w->x0
static ch_status ws_forward_packed(ch_ws_s* w, int B, cudaStream_t st) {
  if (!w->fresh) CH_TRY(ws_refresh(w, st));
  const WsParams p = ws_views(w->params);
  {
    ProfScope ps(st, K_WS_CONV, 1, (double)B * w->P * (16 + 32) * 2, (double)B * w->P * 9 * 16 * 32);
    ws_conv<WS_CIN, WS_C, 0>(w, w->x0, w->w1, w->c1, p.b1, w->a1, nullptr, nullptr, B, st);
  }
  {
    ProfScope ps(st, K_WS_CONV, 1, (double)B * w->P * (32 + 32) * 2, (double)B * w->P * 9 * 32 * 32);
    ws_conv<WS_C, WS_C, 0>(w, w->a1, w->w2, w->c2, p.b2, w->a2, nullptr, nullptr, B, st);
  }
  {
    ProfScope ps(st, K_WS_CONV, 1, (double)B * w->P * (32 * 2 + 8 * 4), (double)B * w->P * 9 * 32 * 8);
    ws_conv<WS_C, WS_COUT, 1>(w, w->a2, w->w3, w->c3, p.b3, nullptr, w->y, nullptr, B, st);
  }
  CH_LAUNCHED();
  return CH_OK;
}

ch_status ws_create(int H, int W, int Bmax, ch_ws_s** out) {
  ch_ws_s* w = new ch_ws_s();
  w->H = H;
  w->W = W;
  w->P = H * W;
  w->Bmax = Bmax;
  const size_t P = (size_t)w->P * Bmax;
  // weight-gradient partials: at most WG_BLOCKS strips and one more per segment and sample
  const size_t nparts = WG_BLOCKS + (size_t)Bmax * ((W + WG_SEG - 1) / WG_SEG);
  ch_status r = CH_OK;
  if (r == CH_OK) r = w->mem.get(&w->params, WS_NPARAM);
  if (r == CH_OK) r = w->mem.get(&w->grads, WS_NPARAM);
  if (r == CH_OK) r = w->mem.get(&w->adam_m, WS_NPARAM);
  if (r == CH_OK) r = w->mem.get(&w->adam_v, WS_NPARAM);
  if (r == CH_OK) r = w->mem.get(&w->w1, 9 * WS_CIN * WS_C);
  if (r == CH_OK) r = w->mem.get(&w->w2, 9 * WS_C * WS_C);
  if (r == CH_OK) r = w->mem.get(&w->w3, 9 * WS_C * WS_COUT);
  if (r == CH_OK) r = w->mem.get(&w->w2f, 9 * WS_C * WS_C);
  if (r == CH_OK) r = w->mem.get(&w->w3f, 9 * 16 * WS_C);
  if (r == CH_OK) r = w->mem.get(&w->c1, 9 * WS_CIN * WS_C);
  if (r == CH_OK) r = w->mem.get(&w->c2, 9 * WS_C * WS_C);
  if (r == CH_OK) r = w->mem.get(&w->c3, 9 * WS_C * 16);
  if (r == CH_OK) r = w->mem.get(&w->c2f, 9 * WS_C * WS_C);
  if (r == CH_OK) r = w->mem.get(&w->c3f, 9 * 16 * WS_C);
  if (r == CH_OK) r = w->mem.get(&w->norm, 20);
  if (r == CH_OK) r = w->mem.get(&w->dscale, (size_t)Bmax * 8);
  if (r == CH_OK) r = w->mem.get(&w->dinv, (size_t)Bmax * 8);
  if (r == CH_OK) r = w->mem.get(&w->t, P * 4);
  if (r == CH_OK) r = w->mem.get(&w->e, P * 4);
  if (r == CH_OK) r = w->mem.get(&w->ge, P * 4);
  if (r == CH_OK) r = w->mem.get(&w->x0, P * WS_CIN);
  if (r == CH_OK) r = w->mem.get(&w->a1, P * WS_C);
  if (r == CH_OK) r = w->mem.get(&w->a2, P * WS_C);
  if (r == CH_OK) r = w->mem.get(&w->dy, P * 16);
  if (r == CH_OK) r = w->mem.get(&w->dz2, P * WS_C);
  if (r == CH_OK) r = w->mem.get(&w->dz1, P * WS_C);
  if (r == CH_OK) r = w->mem.get(&w->y, P * WS_COUT);
  if (r == CH_OK) r = w->mem.get(&w->part, nparts * (9 * WS_C * WS_C + WS_C));
  if (r == CH_OK) r = w->mem.get(&w->loss_part, 1024);
  if (r == CH_OK) r = w->mem.get(&w->rms_part, (size_t)Bmax * WS_RMS_BLOCKS * 8);
  if (r == CH_OK) r = w->mem.get(&w->rn_part, (size_t)RN_BLOCKS * 8);
  if (r == CH_OK) r = w->mem.get(&w->rn_ticket, 1);
  if (r == CH_OK) {
    if (cudaHostAlloc(&w->err_host, sizeof(int), cudaHostAllocMapped) != cudaSuccess ||
        cudaHostGetDevicePointer(&w->err_dev, w->err_host, 0) != cudaSuccess) {
      cudaGetLastError();
      w->err_host = nullptr;
      set_error("warm-start error flag allocation failed");
      r = CH_ERR_CUDA;
    } else {
      *w->err_host = 0;
    }
  }
  if (r == CH_OK) r = ws_tc_setup();
  if (r == CH_OK) {
    cudaMemset(w->params, 0, sizeof(float) * WS_NPARAM);
    cudaMemset(w->adam_m, 0, sizeof(float) * WS_NPARAM);
    cudaMemset(w->adam_v, 0, sizeof(float) * WS_NPARAM);
    cudaMemset(w->rn_ticket, 0, sizeof(unsigned int));
    const float nrm[20] = {0, 0, 0, 0, 0, 0, 0, 0, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1, 1};
    if (cudaMemcpy(w->norm, nrm, sizeof(nrm), cudaMemcpyHostToDevice) != cudaSuccess) {
      set_error("warm-start initialisation failed");
      r = CH_ERR_CUDA;
    }
  }
  if (r != CH_OK) {
    delete w;
    return r;
  }
  *out = w;
  return CH_OK;
}

void ws_destroy(ch_ws_s* w) { delete w; }

ch_status ws_set_params(ch_ws_s* w, const float* host, cudaStream_t st) {
  CH_CUDA(cudaMemcpyAsync(w->params, host, sizeof(float) * WS_NPARAM, cudaMemcpyHostToDevice, st));
  CH_CUDA(cudaStreamSynchronize(st));
  w->fresh = false;
  w->adam_t = 0;
  CH_CUDA(cudaMemsetAsync(w->adam_m, 0, sizeof(float) * WS_NPARAM, st));
  CH_CUDA(cudaMemsetAsync(w->adam_v, 0, sizeof(float) * WS_NPARAM, st));
  return CH_OK;
}

ch_status ws_get_params(const ch_ws_s* w, float* host, float* host_grads, cudaStream_t st) {
  if (host) CH_CUDA(cudaMemcpyAsync(host, w->params, sizeof(float) * WS_NPARAM, cudaMemcpyDeviceToHost, st));
  if (host_grads)
    CH_CUDA(cudaMemcpyAsync(host_grads, w->grads, sizeof(float) * WS_NPARAM, cudaMemcpyDeviceToHost, st));
  CH_CUDA(cudaStreamSynchronize(st));
  return CH_OK;
}

ch_status ws_set_norm(ch_ws_s* w, const float* host20, cudaStream_t st) {
  CH_CUDA(cudaMemcpyAsync(w->norm, host20, sizeof(float) * 20, cudaMemcpyHostToDevice, st));
  CH_CUDA(cudaStreamSynchronize(st));
  return CH_OK;
}

// The weight and bias gradients of one convolution of B samples into g (weights, then biases).
template <int CIN, int COUTG, int COUTW>
static void ws_wgrad(ch_ws_s* w, const __nv_bfloat16* X, const __nv_bfloat16* dY, int B, float* g, cudaStream_t st) {
  const WgTiles t = wg_tiles(w->H, w->W, B);
  const int kp = (t.seg + 15) / 16 * 16, len = 9 * CIN * COUTW + COUTW;
  k_ws_wgrad<CIN, COUTG, COUTW><<<dim3(t.nstrip, t.nseg, B), 32 * WG_WARPS, wg_smem<CIN, COUTG>(kp), st>>>(
      X, dY, w->H, w->W, t.nseg, t.seg, t.rows, kp, w->part);
  k_ws_reduce<<<(len + 31) / 32, dim3(32, 8), 0, st>>>(w->part, t.nstrip * t.nseg * B, len, g);
}

// Backward pass from dy (already in w->dy) and, if lr > 0, an Adam step.
static ch_status ws_backward_update(ch_ws_s* w, int B, float lr, cudaStream_t st) {
  // backward through the data: dz2 = (W3 flipped * dy) . [a2 > 0];  dz1 = (W2 flipped * dz2) . [a1 > 0]
  ws_conv<16, WS_C, 2>(w, w->dy, w->w3f, w->c3f, nullptr, w->dz2, nullptr, w->a2, B, st);
  ws_conv<WS_C, WS_C, 2>(w, w->dz2, w->w2f, w->c2f, nullptr, w->dz1, nullptr, w->a1, B, st);
  CH_LAUNCHED();
  // weight gradients, per strip of image rows, then summed in order
  WsParams g = ws_views(w->grads);
  ws_wgrad<WS_C, 16, WS_COUT>(w, w->a2, w->dy, B, g.w3, st);
  ws_wgrad<WS_C, WS_C, WS_C>(w, w->a1, w->dz2, B, g.w2, st);
  ws_wgrad<WS_CIN, WS_C, WS_C>(w, w->x0, w->dz1, B, g.w1, st);
  CH_LAUNCHED();
  if (lr > 0.f) {
    w->adam_t += 1;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.f - powf(b1, (float)w->adam_t), c2 = 1.f - powf(b2, (float)w->adam_t);
    k_ws_adam<<<blocks_for(WS_NPARAM), TPB, 0, st>>>(w->params, w->grads, w->adam_m, w->adam_v, WS_NPARAM,
                                                      lr, b1, b2, 1e-8f, c1, c2);
    CH_LAUNCHED();
    w->fresh = false;
  }
  return CH_OK;
}

// inference: pred = s + d + (net(...) * out_scale) * D for one state s and its two predecessors
// q, q2 (d = s - q, D = s - 2 q + q2)
ch_status ws_predict(ch_ws_s* w, const double* state, const double* prev, const double* prev2, double* pred,
                     cudaStream_t st) {
  {
    ProfScope ps(st, K_WS_IO, 0, w->P * (32.0 * 3 + 32.0), 0.0);
    ws_rms<double>(w, state, prev, prev2, 1, st);
    k_ws_pack<double><<<dim3(blocks_for(w->P), 1), TPB, 0, st>>>(state, prev, prev2, w->P,
                                                                  aligned4(8, {state, prev, prev2}), w->norm,
                                                                  w->norm + 8, w->dinv, w->x0);
  }
  CH_LAUNCHED();
  CH_TRY(ws_forward_packed(w, 1, st));
  {
    ProfScope ps(st, K_WS_IO, 0, w->P * (32.0 * 3 + 32.0 + 32.0), 0.0);
    k_ws_unpack<<<blocks_for(w->P), TPB, 0, st>>>(state, prev, prev2, w->y, w->P,
                                                      aligned4(8, {state, prev, prev2, pred}), w->norm + 16, pred);
  }
  CH_LAUNCHED();
  return CH_OK;
}

// one training step on B samples (fp32, B x N x 4 each): states x, their two predecessors q, q2
// and successors n.  Computes the state-space loss (with the grid-Laplacian term weighted by lap)
// and the gradients; if lr > 0 also takes an Adam step.
ch_status ws_train_step(ch_ws_s* w, const float* x, const float* q, const float* q2, const float* n, int B,
                        float lap, float lr, float* loss, cudaStream_t st) {
  if (B < 1 || B > w->Bmax) {
    set_error("batch of %d samples outside [1, %d]", B, w->Bmax);
    return CH_ERR_ARG;
  }
  if (!(lap >= 0.f) || !std::isfinite(lap)) {
    set_error("Laplacian loss weight %g must be finite and >= 0", (double)lap);
    return CH_ERR_ARG;
  }
  const int P = w->P;
  ws_rms<float>(w, x, q, q2, B, st);
  k_ws_pack<float><<<dim3(blocks_for(P), B), TPB, 0, st>>>(x, q, q2, P, aligned4(4, {x, q, q2}), w->norm,
                                                            w->norm + 8, w->dinv, w->x0);
  CH_LAUNCHED();
  CH_TRY(ws_forward_packed(w, B, st));
  const int lb = 304;
  k_ws_err_theta<<<dim3(blocks_for(P), B), TPB, 0, st>>>(w->y, x, q, q2, n, P, w->norm + 16, w->dinv, w->e, w->t);
  k_ws_lap_loss<<<lb, 256, 0, st>>>(w->e, w->H, w->W, B, lap, w->ge, w->loss_part);
  k_ws_dy<<<lb, 256, 0, st>>>(w->e, w->ge, w->t, w->H, w->W, B, lap, w->dy);
  CH_TRY(ws_backward_update(w, B, lr, st));
  if (loss) {
    float parts[lb];
    CH_CUDA(cudaMemcpyAsync(parts, w->loss_part, sizeof(parts), cudaMemcpyDeviceToHost, st));
    CH_CUDA(cudaStreamSynchronize(st));
    CH_TRY(ws_check(w));
    double s = 0.0;
    for (int i = 0; i < lb; ++i) s += parts[i];
    *loss = (float)(s / ((double)B * P * 4));
  }
  return CH_OK;
}

// ---------------------------------------------------------------- residual-loss training
// The correction c = y * out_scale * D (fp64, N x 4, D = s - 2 q + q2) of one sample, or the
// linear extrapolation 2 s - q (mode 0).
__global__ void k_ws_guess_part(int P, int mode, bool al, const double* __restrict__ s, const double* __restrict__ q,
                                const double* __restrict__ q2, const float* __restrict__ y,
                                const float* __restrict__ out_scale, double4_32a* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P) return;
  const Quad<double> a = ld4(s, i, al), b = ld4(q, i, al);
  if (mode == 0) {
    out[i] = make_double4_32a(2.0 * a.x - b.x, 2.0 * a.y - b.y, 2.0 * a.z - b.z, 2.0 * a.w - b.w);
  } else {
    const Quad<double> c = ld4(q2, i, al);
    const float4 yv = *reinterpret_cast<const float4*>(y + (size_t)i * WS_COUT);
    out[i] = make_double4_32a((double)yv.x * (double)out_scale[0] * (a.x - 2.0 * b.x + c.x),
                              (double)yv.y * (double)out_scale[1] * (a.y - 2.0 * b.y + c.y),
                              (double)yv.z * (double)out_scale[2] * (a.z - 2.0 * b.z + c.z),
                              (double)yv.w * (double)out_scale[3] * (a.w - 2.0 * b.w + c.w));
  }
}

// out = a - b (N x 4)
__global__ void k_ws_sub(int P, const double4_32a* __restrict__ a, const double4_32a* b, double4_32a* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P) return;
  const double4_32a u = a[i], v = b[i];
  out[i] = make_double4_32a(u.x - v.x, u.y - v.y, u.z - v.z, u.w - v.w);
}

// nrm[0..3] = per channel sum of rex * zex, nrm[4..7] = per channel sum of r * z, where z = P^-1 r
// (or z = r for the plain norm), in a fixed order: block b adds its chunk of pixels into part[b][8]
// and the last block to finish adds the blocks' sums in block order.  (One block over the whole
// image took 222 us at 257 x 257, latency alone.)
__global__ void __launch_bounds__(256) k_ws_resnorm(int P, const double4_32a* __restrict__ rex,
                                                    const double4_32a* __restrict__ zex,
                                                    const double4_32a* __restrict__ r,
                                                    const double4_32a* __restrict__ z, double* __restrict__ part,
                                                    unsigned int* __restrict__ ticket, double* __restrict__ nrm) {
  __shared__ double red[8][8];
  __shared__ bool last;
  double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  const int chunk = (P + gridDim.x - 1) / gridDim.x, i1 = min(P, ((int)blockIdx.x + 1) * chunk);
  for (int i = blockIdx.x * chunk + threadIdx.x; i < i1; i += blockDim.x) {
    const double4_32a a = rex[i], b = zex[i], c = r[i], d = z[i];
    acc[0] = fma(a.x, b.x, acc[0]);
    acc[1] = fma(a.y, b.y, acc[1]);
    acc[2] = fma(a.z, b.z, acc[2]);
    acc[3] = fma(a.w, b.w, acc[3]);
    acc[4] = fma(c.x, d.x, acc[4]);
    acc[5] = fma(c.y, d.y, acc[5]);
    acc[6] = fma(c.z, d.z, acc[6]);
    acc[7] = fma(c.w, d.w, acc[7]);
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
    if (lane == 0) red[w][c] = acc[c];
  }
  __syncthreads();
  if (threadIdx.x < 8) {
    double t = 0.0;
    for (int q = 0; q < 8; ++q) t += red[q][threadIdx.x];
    part[blockIdx.x * 8 + threadIdx.x] = t;
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  // warp w: value w, lanes over blocks (lane, lane + 32, ...), then the lanes' sums
  double t = 0.0;
  for (int b = lane; b < (int)gridDim.x; b += 32) t += __ldcg(part + b * 8 + w);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) nrm[w] = t;
  if (threadIdx.x == 0) *ticket = 0;
}

// dy of one sample from g = A z: L = sum_species ln(<r, z>_sp / <rex, zex>_sp) / (2B) with
// z = P^-1 r (P^-1 symmetric, or the identity), r = rex - A c, so dL/dc = -2 A z / <r, z>_sp / (2B)
// and dL/dy_c = dL/dc_c * out_scale_c * D_c (c = y out_scale D).
// Channel c belongs to species c % 2 (channels phi_p, phi_n, mu_p, mu_n).
__global__ void k_ws_res_dy(int P, int B, const double4_32a* __restrict__ g, const double* __restrict__ nrm,
                            const float* __restrict__ out_scale, const double* __restrict__ s,
                            const double* __restrict__ q, const double* __restrict__ q2, bool al,
                            __nv_bfloat16* __restrict__ dy) {
  __shared__ double wsp[2];
  if (threadIdx.x < 2) {  // once per block: an FP64 division per pixel would cost more than the rest
    const int sp = threadIdx.x;
    const double den = nrm[sp] + nrm[sp + 2], num = nrm[4 + sp] + nrm[6 + sp];
    wsp[sp] = (den > 0.0 && num > 0.0) ? 1.0 / (num * (double)B) : 0.0;
  }
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P) return;
  const double4_32a gv = g[i];
  const Quad<double> sv = ld4(s, i, al), qv = ld4(q, i, al), q2v = ld4(q2, i, al);
  const float v0 = (float)(-gv.x * wsp[0] * ((double)out_scale[0] * (sv.x - 2.0 * qv.x + q2v.x)));
  const float v1 = (float)(-gv.y * wsp[1] * ((double)out_scale[1] * (sv.y - 2.0 * qv.y + q2v.y)));
  const float v2 = (float)(-gv.z * wsp[0] * ((double)out_scale[2] * (sv.z - 2.0 * qv.z + q2v.z)));
  const float v3 = (float)(-gv.w * wsp[1] * ((double)out_scale[3] * (sv.w - 2.0 * qv.w + q2v.w)));
  uint4* o = reinterpret_cast<uint4*>(dy + (size_t)i * 16);
  o[0] = make_uint4(pack_bf16(__float2bfloat16_rn(v0), __float2bfloat16_rn(v1)),
                    pack_bf16(__float2bfloat16_rn(v2), __float2bfloat16_rn(v3)), 0u, 0u);
  o[1] = make_uint4(0u, 0u, 0u, 0u);
}

ch_status ws_train_residual(ch_ws_s* w, const ch_system_s* sys, ch_precond_s* pc, const double* x,
                            const double* q, const double* q2, int B, float lr, float* loss, cudaStream_t st) {
  if (B < 1 || B > w->Bmax) {
    set_error("batch of %d samples outside [1, %d]", B, w->Bmax);
    return CH_ERR_ARG;
  }
  const ch_params& mp = sys->mesh->p;
  if (mp.dim != 2 || sys->mesh->runs.size() != 1 || mp.nx + 1 != w->W || mp.ny + 1 != w->H) {
    set_error("the system must be a single-run 2D mesh of %d x %d nodes", w->W, w->H);
    return CH_ERR_ARG;
  }
  if (pc != nullptr && pc->sys != sys) {
    set_error("the preconditioner was built for another system");
    return CH_ERR_ARG;
  }
  const int P = w->P;
  // each buffer by itself: a call after one that ran out of memory allocates what is missing
  const auto once = [&](double** buf, size_t n) { return *buf ? CH_OK : w->mem.get(buf, n); };
  if (pc != nullptr) {
    CH_TRY(once(&w->zex, (size_t)P * 4));
    CH_TRY(once(&w->zr, (size_t)w->Bmax * P * 4));
  }
  CH_TRY(once(&w->rex, (size_t)w->Bmax * P * 4));
  CH_TRY(once(&w->rres, (size_t)w->Bmax * P * 4));
  CH_TRY(once(&w->tmp1, (size_t)P * 4));
  CH_TRY(once(&w->tmp2, (size_t)P * 4));
  CH_TRY(once(&w->nrm, (size_t)w->Bmax * 8));
  ws_rms<double>(w, x, q, q2, B, st);
  const bool al = aligned4(8, {x, q, q2});  // (a sample is a multiple of 32 bytes)
  k_ws_pack<double><<<dim3(blocks_for(P), B), TPB, 0, st>>>(x, q, q2, P, al, w->norm, w->norm + 8, w->dinv, w->x0);
  CH_LAUNCHED();
  CH_TRY(ws_forward_packed(w, B, st));
  const int nb = blocks_for(P), rnb = std::min(RN_BLOCKS, nb);
  const auto v4 = [](const double* p) { return reinterpret_cast<const double4_32a*>(p); };
  const auto m4 = [](double* p) { return reinterpret_cast<double4_32a*>(p); };
  for (int b = 0; b < B; ++b) {
    const double* xs = x + (size_t)b * P * 4;
    const double* qs = q + (size_t)b * P * 4;
    const double* q2s = q2 + (size_t)b * P * 4;
    double* rex = w->rex + (size_t)b * P * 4;
    double* r = w->rres + (size_t)b * P * 4;
    // rex = b(s) - A (2 s - q)
    CH_TRY(rhs_strided(sys, xs, xs + 1, 4, w->tmp1, st));
    k_ws_guess_part<<<nb, TPB, 0, st>>>(P, 0, al, xs, qs, q2s, nullptr, nullptr, m4(w->tmp2));
    CH_LAUNCHED();
    CH_TRY(apply_A(sys, w->tmp2, rex, st));
    k_ws_sub<<<nb, TPB, 0, st>>>(P, v4(w->tmp1), v4(rex), m4(rex));
    // r = rex - A c
    k_ws_guess_part<<<nb, TPB, 0, st>>>(P, 1, al, xs, qs, q2s, w->y + (size_t)b * P * WS_COUT, w->norm + 16,
                                        m4(w->tmp2));
    CH_LAUNCHED();
    CH_TRY(apply_A(sys, w->tmp2, w->tmp1, st));
    k_ws_sub<<<nb, TPB, 0, st>>>(P, v4(rex), v4(w->tmp1), m4(r));
    // z = P^-1 r, zex = P^-1 rex (Algorithm 1), or the residuals themselves
    const double* zex = rex;
    const double* z = r;
    if (pc != nullptr) {
      CH_TRY(precond_apply(pc, rex, w->zex, st));
      CH_TRY(precond_apply(pc, r, w->zr + (size_t)b * P * 4, st));
      zex = w->zex;
      z = w->zr + (size_t)b * P * 4;
    }
    k_ws_resnorm<<<rnb, 256, 0, st>>>(P, v4(rex), v4(zex), v4(r), v4(z), w->rn_part, w->rn_ticket, w->nrm + 8 * b);
    // g = A z (A is symmetric) -> dy of this sample
    CH_TRY(apply_A(sys, z, w->tmp1, st));
    k_ws_res_dy<<<nb, TPB, 0, st>>>(P, B, v4(w->tmp1), w->nrm + 8 * b, w->norm + 16, xs, qs, q2s, al,
                                    w->dy + (size_t)b * P * 16);
    CH_LAUNCHED();
  }
  CH_TRY(ws_backward_update(w, B, lr, st));
  if (loss) {
    std::vector<double> h((size_t)B * 8);
    CH_CUDA(cudaMemcpyAsync(h.data(), w->nrm, sizeof(double) * 8 * B, cudaMemcpyDeviceToHost, st));
    CH_CUDA(cudaStreamSynchronize(st));
    CH_TRY(ws_check(w));
    double L = 0.0;
    for (int b = 0; b < B; ++b)
      for (int sp = 0; sp < 2; ++sp) {
        const double den = h[8 * b + sp] + h[8 * b + sp + 2], num = h[8 * b + 4 + sp] + h[8 * b + 6 + sp];
        if (den > 0.0 && num > 0.0) L += std::log(num / den);
      }
    *loss = (float)(L / (2.0 * B));
  }
  return CH_OK;
}

// ---------------------------------------------------------------- normalisation of a training set
// S samples of P x 4 states x = s_k (fp64, or fp32 with F = float).  The network's inputs are the
// fields, normalised by their mean and standard deviation over the set (n - 1 divisor), and the
// change and the second difference in units of their per-sample RMS (mean 0, scale 1 as they are);
// its output is theta itself (out_scale = 1).  Sums run in a fixed order (per-block partials, then
// one block in block order), so the statistics are reproducible.
constexpr int FIT_BLOCKS = 152 * 4;

// PASS 0: per channel sums of x; PASS 1: of (x - mean)^2
template <typename F, int PASS>
__global__ void k_fit_sums(const F* __restrict__ x, int64_t total, const double* __restrict__ mean,
                           double* __restrict__ part) {
  __shared__ double sm[TPB / 32][4];
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < total; v += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const double xv = x[v * 4 + c];
      if (PASS == 0) {
        acc[c] += xv;
      } else {
        const double dx = xv - mean[c];
        acc[c] = fma(dx, dx, acc[c]);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    double t = acc[k];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5][k] = t;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    double t = 0.0;
    for (int w = 0; w < TPB / 32; ++w) t += sm[w][threadIdx.x];
    part[blockIdx.x * 4 + threadIdx.x] = t;
  }
}

// one block: out[c] = (sum over the blocks' partials, in block order) / div
__global__ void k_fit_reduce(const double* __restrict__ part, int nparts, double div, double* __restrict__ out) {
  if (threadIdx.x >= 4) return;
  double t = 0.0;
  for (int b = 0; b < nparts; ++b) t += part[b * 4 + threadIdx.x];
  out[threadIdx.x] = t / div;
}

// norm[20] = (mean of the fields, 0 x 4; 1/std of the fields, 1 x 4; 1 x 4) from the means
// (stats[0..4)) and variances (stats[4..8))
__global__ void k_fit_norm(const double* __restrict__ stats, float* __restrict__ norm, double* __restrict__ out20) {
  const int c = threadIdx.x;
  if (c >= 4) return;
  const double vals[5] = {stats[c], 0.0, 1.0 / fmax(sqrt(stats[4 + c]), 1e-30), 1.0, 1.0};
  for (int k = 0; k < 5; ++k) {
    norm[4 * k + c] = (float)vals[k];
    out20[4 * k + c] = vals[k];
  }
}

template <typename F>
static ch_status fit_norm_t(ch_ws_s* w, const F* x, int S, double* host20, cudaStream_t st) {
  const int64_t total = (int64_t)S * w->P;
  if (total < 2) {
    set_error("the normalisation needs at least two pixels of data");
    return CH_ERR_ARG;
  }
  Alloc tmp;
  double *part = nullptr, *stats = nullptr, *out20 = nullptr;
  CH_TRY(tmp.get(&part, (size_t)FIT_BLOCKS * 4));
  CH_TRY(tmp.get(&stats, 8));  // the fields' means [0, 4), variances [4, 8)
  CH_TRY(tmp.get(&out20, 20));
  const int nb = (int)std::min<int64_t>(FIT_BLOCKS, (total + TPB - 1) / TPB);
  k_fit_sums<F, 0><<<nb, TPB, 0, st>>>(x, total, nullptr, part);
  k_fit_reduce<<<1, 32, 0, st>>>(part, nb, (double)total, stats);
  k_fit_sums<F, 1><<<nb, TPB, 0, st>>>(x, total, stats, part);
  k_fit_reduce<<<1, 32, 0, st>>>(part, nb, (double)(total - 1), stats + 4);
  k_fit_norm<<<1, 32, 0, st>>>(stats, w->norm, out20);
  CH_LAUNCHED();
  CH_CUDA(cudaMemcpyAsync(host20, out20, sizeof(double) * 20, cudaMemcpyDeviceToHost, st));
  CH_CUDA(cudaStreamSynchronize(st));
  return CH_OK;
}

ch_status ws_fit_norm(ch_ws_s* w, const void* x, int S, int fp32, double* host20, cudaStream_t st) {
  if (fp32) return fit_norm_t<float>(w, static_cast<const float*>(x), S, host20, st);
  return fit_norm_t<double>(w, static_cast<const double*>(x), S, host20, st);
}

int ws_nparam() { return WS_NPARAM; }

void ws_dims(const ch_ws_s* w, int* H, int* W) {
  *H = w->H;
  *W = w->W;
}

}  // namespace ch
