// Learned correction stage of the preconditioner: a small convolutional
// network on the 2D Cartesian grid, its training on the device, the
// solver-generated training pairs, and the stage inside the flexible PCG.
// The paper has no learned component; this extends its AMG-PCG (Algorithm 1
// step 4).  Definitions (network, pairs, loss, stage) are those of include/eb.h.
//
// Storage: hidden activations BF16 NHWC (32 channels = 64 bytes per pixel);
// FP32 master parameters, BF16 copies of the 32 -> 32 weights; every sum in
// FP32.  The four 32 -> 32 layers (99.6 % of the FLOPs) are implicit GEMMs on
// the 5th-generation tensor cores (tcgen05.mma, accumulators in tensor memory),
// fed by tensor copies (TMA) in a warp-specialised pipeline: a job is 128
// pixels of one image row and all 32 output channels; its three input rows
// (130 pixels x 32 channels) and the 9 x 32 x 32 weights sit in shared memory;
// K = 9 taps x 32 channels.  Data gradients run through
// the same kernel with flipped, transposed weights and the ReLU mask of the
// layer input applied in its epilogue; weight gradients are tcgen05 GEMMs over
// pixels (k_conv32_wgrad) with per-CTA partials summed in a fixed order.  The
// 2 -> 32 and 32 -> 1 layers run on the CUDA cores.  Inference (nn_forward,
// the stage in the PCG) runs all six layers in one launch instead
// (k_net_fwd), with the hidden activations kept in shared memory and tensor
// memory and results identical to the layer-by-layer launches.
#include "eb_solver.cuh"
#include "tma.cuh"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <utility>
#include <vector>

namespace ebk {

using bf16 = __nv_bfloat16;

constexpr int NC = 32;    // hidden channels
constexpr int NMID = 4;   // 32 -> 32 layers
constexpr int TPX = 128;  // pixels per CTA job (one row segment)

// flat parameter vector
constexpr int W1_N = NC * 9 * 2, B1_N = NC;
constexpr int WM_N = NC * 9 * NC, BM_N = NC;
constexpr int W6_N = 9 * NC, B6_N = 1;
constexpr int OFF_W1 = 0;
constexpr int OFF_WM = OFF_W1 + W1_N + B1_N;  // middle layer l at OFF_WM + l (WM_N + BM_N)
constexpr int OFF_W6 = OFF_WM + NMID * (WM_N + BM_N);
constexpr int NPARAM = OFF_W6 + W6_N + B6_N;
static_assert(NPARAM == 37889, "parameter layout");

__host__ __device__ constexpr int off_wm(int l) { return OFF_WM + l * (WM_N + BM_N); }

// A stack of images: H rows of W pixels, image boundaries every R rows.
struct Image {
  int W, H, R;
  __device__ int64_t npx() const { return (int64_t)W * H; }
};

// Packed FP32 pairs: fma.rn.f32x2 is two round-to-nearest FMAs in one
// instruction, so each lane's result is the scalar __fmaf_rn's at half the FMA
// instructions.
__device__ __forceinline__ uint64_t fz_pk(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void fz_upk(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ void fz_fma2(uint64_t& acc, uint64_t w, uint64_t x) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(w), "l"(x));
}
// (max(a, 0), max(b, 0)) in bf16: rounding keeps the sign and the order, so the
// packed maximum after it equals the two FP32 ones before it (NaN gives 0 in both)
__device__ __forceinline__ uint32_t fz_relu2(float a, float b) {
  const __nv_bfloat162 h = __hmax2(__floats2bfloat162_rn(a, b), __floats2bfloat162_rn(0.0f, 0.0f));
  return *reinterpret_cast<const uint32_t*>(&h);
}

// ------------------------------------------------------------ forward
// layer 1 (2 -> 32) + ReLU; in: (s_hat, m) per pixel.  A thread computes two
// x-adjacent pixels of two rows: the 4 x 4 input window is loaded once and every
// weight read from shared memory serves the four, in packed FMAs over channel
// pairs; each output is one FMA chain b, then (tap, input channel) in order.
// Bounded by the FMA pipe and the issue slots.  16 x 512^2: 116 us; 173 us
// with two pixels of one row, scalar FMAs and a channel's weights at a time.
__global__ void __launch_bounds__(128) k_l1_fwd(Image im, const float2* __restrict__ in, const float* __restrict__ P,
                                                bf16* __restrict__ y) {
  __shared__ __align__(16) float w[18 * NC + NC];  // weight (tap, input) of the 32 outputs contiguous, then b
  for (int i = threadIdx.x; i < 18 * NC; i += blockDim.x) w[i] = P[OFF_W1 + (i % NC) * 18 + i / NC];
  for (int i = threadIdx.x; i < NC; i += blockDim.x) w[18 * NC + i] = P[OFF_W1 + W1_N + i];
  __syncthreads();
  const int half = (im.W + 1) >> 1, rp = (im.R + 1) >> 1;
  const int64_t pp = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t q = pp / half;
  const int img = (int)(q / rp);
  const int lo = img * im.R, hi = lo + im.R;
  if (lo >= im.H) return;
  const int x = 2 * (int)(pp - q * half), r = lo + 2 * (int)(q - (int64_t)img * rp);
  float2 v[4][4];
#pragma unroll
  for (int dy = 0; dy < 4; ++dy) {
    const int rr = r + dy - 1;
#pragma unroll
    for (int dx = 0; dx < 4; ++dx) {
      const int xx = x + dx - 1;
      v[dy][dx] = (xx >= 0 && xx < im.W && rr >= lo && rr < hi) ? in[(int64_t)rr * im.W + xx] : make_float2(0.f, 0.f);
    }
  }
  bf16* const y0 = y + ((int64_t)r * im.W + x) * NC;
  const bool okx = x + 1 < im.W, oky = r + 1 < hi;
#pragma unroll 1
  for (int c16 = 0; c16 < NC; c16 += 16) {
    uint32_t o[4][8];
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const int cg = c16 + 8 * g;
      uint64_t acc[4][4];  // [pixel 2 row + column][channel pair]
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[k][c] = *reinterpret_cast<const uint64_t*>(w + 18 * NC + cg + 2 * c);
#pragma unroll
      for (int e = 0; e < 18; ++e) {
        const float4 wa = *reinterpret_cast<const float4*>(w + e * NC + cg);
        const float4 wb = *reinterpret_cast<const float4*>(w + e * NC + cg + 4);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float2 t = v[(e >> 1) / 3 + (k >> 1)][(e >> 1) % 3 + (k & 1)];
          const float xv = (e & 1) ? t.y : t.x;
          const uint64_t x2 = fz_pk(xv, xv);
          fz_fma2(acc[k][0], fz_pk(wa.x, wa.y), x2);
          fz_fma2(acc[k][1], fz_pk(wa.z, wa.w), x2);
          fz_fma2(acc[k][2], fz_pk(wb.x, wb.y), x2);
          fz_fma2(acc[k][3], fz_pk(wb.z, wb.w), x2);
        }
      }
#pragma unroll
      for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          float a0, a1;
          fz_upk(acc[k][c], a0, a1);
          o[k][4 * g + c] = fz_relu2(a0, a1);
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if ((k & 1) && !okx) continue;
      if ((k >> 1) && !oky) continue;
      int4* dst = reinterpret_cast<int4*>(y0 + ((int64_t)(k >> 1) * im.W + (k & 1)) * NC + c16);
      dst[0] = make_int4(o[k][0], o[k][1], o[k][2], o[k][3]);
      dst[1] = make_int4(o[k][4], o[k][5], o[k][6], o[k][7]);
    }
  }
}

// ------------------------------------------- 32 -> 32 convolution (tcgen05)
// Implicit GEMM on the 5th-generation tensor cores (kernel k_conv32_tma below).
// The B operand, the weights, sits in shared memory in the no-swizzle K-major
// layout of "core matrices" (8 rows x 16 bytes stored contiguously):
// [dx][channel group g][dy 32 + n][8 k] (SBO = 128 B between 8-row blocks of n,
// LBO = 96 x 16 B between channel groups).  The A operand (activations) uses the
// 64-byte swizzled layout written by the tensor copies (tc_desc_sw64).
constexpr int TC_PIX = TPX + 2;                  // pixels of a job's rows with their two halo pixels
constexpr int TC_W = 9 * 4 * NC * 16;            // weights of a layer: 18,432 bytes
constexpr uint32_t TC_SPIN = 1u << 22;           // bounded mbarrier polls (~0.1 s)

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor: start, LBO, SBO (bytes), version 1, no swizzle
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}

// shared-memory matrix descriptor of a K-major operand in the 64-byte swizzled
// layout: rows of 64 bytes (32 bf16 along K), the 16-byte chunks of a row
// permuted by the address bits 7-8 as the tensor copies write them, 8-row
// groups 512 bytes apart (SBO); LBO unused (the K extent of one MMA, 32 bytes,
// lies inside a row); swizzle mode 4 (64 bytes) in bits 61-63
__device__ __forceinline__ uint64_t tc_desc_sw64(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)1 << 16) | ((uint64_t)(512 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}

// instruction descriptor of kind::f16: D f32, A and B bf16, both K-major, N, M
__device__ __forceinline__ constexpr uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// ------------------------- 32 -> 32 convolution, TMA-fed warp-specialised pipeline
// y = conv(x; wk) + bias (if bias), then ReLU (if relu), then 0 where
// mask_ref <= 0 (if mask_ref: the ReLU derivative of a data gradient).
// wk: bf16 [9][32 (n)][32 (k)].  A job is 128 pixels of rb <= 4 rows of an image
// and all 32 output channels; its rb + 2 input rows x 130 pixels x 32 channels
// arrive in one 4D tensor copy (cp.async.bulk.tensor) in the 64-byte swizzled
// K-major layout (a pixel's 32 channels are one 64-byte row).  The MMAs are
// input-row stationary: input row j, shifted by dx = 0, 1, 2 pixels (an offset
// of 64 dx bytes) and split in two channel halves, times the weights of the tap
// rows that lead from it into the job, N = 32 per output row: rows j + 1, j, j -
// 1 with dy = 0, 1, 2, at increasing TMEM columns.  Four rows take 39 MMAs, where
// one output row at a time takes 72; issuing one costs its thread some 190
// cycles whatever N, so that count and not the tensor cores bounded the earlier
// form: 172 us a layer at 16 x 512^2 pixels on average over forward and data
// gradient (which also reads the masks), 127 us now, 5.3 TB/s.  An output row receives its taps in
// (dy, dx, kh) order, the first without accumulating.
// Four MMA warps take the jobs in turn, each with a stage and a TMEM region (128
// columns) of its own; eight epilogue warps drain a region (warp w: TMEM lanes 32
// (w % 4) .., rows (w / 4) rb / 2 ..), the ReLU masks of a data gradient loaded
// while the MMAs run.  One CTA per SM.  The tensor map views the activations as
// (32 channels, pixel, row in image, image), so the rows outside an image and the
// pixels outside a row are filled with zeros by the copy.
// Barriers, per stage: full (copy, transaction bytes), empty (MMA commit ->
// copy), tfull (MMA commit -> epilogue), tempty (8 epilogue warps -> MMA).  Every
// wait is bounded; a wait that gives up raises a shared abort flag that ends
// every role's loop, sets *err, and the CTA waits (bounded) for its copies and
// MMAs in flight before freeing TMEM.
constexpr int CP_ROWS = 4;                             // rows of a job at most
constexpr int CP_STAGES = 4;
constexpr int CP_STAGE = 50176;                        // 6 x 130 x 64 bytes rounded up to 1 KB (swizzle atoms stay aligned)
constexpr int CP_W = CP_STAGES * CP_STAGE;             // weights after the stages: [dx][channel group][dy 32 + n][8 k]
constexpr int CP_WDX = 4 * 96 * 16;
constexpr int CP_BAR = CP_W + TC_W;                    // barriers after the weights
constexpr int CP_NBAR = 4 * CP_STAGES;
constexpr int CP_SMEM = CP_BAR + 8 * CP_NBAR + 16;     // + TMEM slot and abort flag
constexpr int CP_THREADS = 13 * 32;                    // warps 0-7 epilogue, 8 copies, 9-12 MMAs
static_assert((CP_ROWS + 2) * TC_PIX * NC * 2 <= CP_STAGE && CP_STAGE % 1024 == 0 && CP_SMEM <= 227 * 1024, "conv stage");

__device__ __forceinline__ bool cp_wait(uint32_t bar, uint32_t parity, volatile int* abort) {
  for (uint32_t it = 0; it < TC_SPIN; ++it) {
    uint32_t ok = 0;
    asm volatile(
        "{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\n\tselp.u32 %0, 1, 0, q;\n\t}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((it & 63) == 63 && *abort) return false;
  }
  *abort = 1;
  return false;
}

__global__ void __launch_bounds__(CP_THREADS, 1) k_conv32_tma(const __grid_constant__ CUtensorMap xmap, Image im,
                                                               int rb, const bf16* __restrict__ wk,
                                                               const float* __restrict__ bias, bf16* __restrict__ y,
                                                               int relu, const bf16* __restrict__ mask_ref,
                                                               int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t base = smem_addr(smem_raw);
  const uint32_t w0 = base + CP_W, bars = base + CP_BAR;
  auto full = [&](int st) { return bars + 8 * st; };
  auto empty = [&](int st) { return bars + 8 * (CP_STAGES + st); };
  auto tfull = [&](int st) { return bars + 8 * (2 * CP_STAGES + st); };
  auto tempty = [&](int st) { return bars + 8 * (3 * CP_STAGES + st); };
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem_raw + CP_BAR + 8 * CP_NBAR);
  volatile int* abort = reinterpret_cast<volatile int*>(smem_raw + CP_BAR + 8 * CP_NBAR + 8);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int i = tid; i < 9 * NC * 4; i += CP_THREADS) {  // weights once per CTA
    const int g = i & 3, n = (i >> 2) % NC, d = (i >> 2) / NC;
    *reinterpret_cast<int4*>(smem_raw + CP_W + (d % 3) * CP_WDX + g * (96 * 16) + ((d / 3) * NC + n) * 16) =
        *reinterpret_cast<const int4*>(wk + (d * NC + n) * NC + g * 8);
  }
  if (tid == 0) {
    for (int b = 0; b < CP_NBAR; ++b) {
      const uint32_t cnt = b >= 3 * CP_STAGES ? 8u : 1u;  // tempty: one arrive per epilogue warp
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bars + 8 * b), "r"(cnt));
    }
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_addr(tslot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("fence.proxy.async.shared::cta;");  // weights (generic stores) are read by the tensor cores
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tslot;
  const int segs = (im.W + TPX - 1) / TPX, chunks = (im.R + rb - 1) / rb;
  const int64_t jobs = (int64_t)segs * chunks * (im.H / im.R);
  const int64_t njob = jobs > (int64_t)blockIdx.x ? (jobs - 1 - blockIdx.x) / gridDim.x + 1 : 0;  // this CTA's jobs
  if (warp == 8) {
    // copies: stage s = k mod S, its u-th use waits for the MMAs of use u - 1
    if (lane == 0) {
      const uint64_t map = reinterpret_cast<uint64_t>(&xmap);
      const uint32_t bytes = (uint32_t)((rb + 2) * TC_PIX * NC * 2);
      asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
      int64_t k = 0;
      for (; k < njob; ++k) {
        const int st = (int)(k % CP_STAGES);
        const uint32_t u = (uint32_t)(k / CP_STAGES);
        if (u > 0 && !cp_wait(empty(st), (u - 1) & 1u, abort)) break;
        const int64_t job = blockIdx.x + k * gridDim.x;
        const int x0 = (int)(job % segs) * TPX, r0 = (int)((job / segs) % chunks) * rb;
        const int img = (int)(job / ((int64_t)segs * chunks));
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full(st)), "r"(bytes) : "memory");
        asm volatile(
            "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
            "%5}], [%6];" ::"r"(base + st * CP_STAGE),
            "l"(map), "r"(0), "r"(x0 - 1), "r"(r0 - 1), "r"(img), "r"(full(st))
            : "memory");
      }
      // copies still in flight (an aborted run) land before the CTA ends
      for (int64_t q = k > CP_STAGES ? k - CP_STAGES : 0; q < k; ++q) {
        volatile int never = 0;
        cp_wait(full((int)(q % CP_STAGES)), (uint32_t)(q / CP_STAGES) & 1u, &never);
      }
    }
  } else if (warp > 8) {
    if (lane == 0) {
      const int st = warp - 9;  // this warp's stage and TMEM region: jobs st, st + 4, ...
      uint32_t u = 0;
      for (int64_t k = st; k < njob; k += CP_STAGES, ++u) {
        if (!cp_wait(full(st), u & 1u, abort)) break;
        if (u > 0 && !cp_wait(tempty(st), (u - 1) & 1u, abort)) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t sa = base + st * CP_STAGE, region = tmem + (uint32_t)(128 * st);
        auto mma = [&](uint32_t dst, uint64_t da, uint32_t sb, int n, uint32_t acc) {
          const uint64_t db = tc_desc(sb, 96 * 16, 128);
          asm volatile(
              "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
              "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(dst),
              "l"(da), "l"(db), "r"(tc_idesc(128, n)), "r"(acc));
        };
#pragma unroll 1
        for (int j = -1; j <= rb; ++j) {
          // tap rows dl .. dh lead from input row j to the job's rows j + 1 - dy;
          // row r accumulates at columns 32 (rb - 1 - r)
          const int dl = j + 1 > rb - 1 ? j + 2 - rb : 0, dh = j + 1 < 2 ? j + 1 : 2;
          const uint32_t dst = region + (uint32_t)(32 * (rb - 2 - j + dl));
#pragma unroll 1
          for (int q = 0; q < 6; ++q) {
            const int dx = q >> 1, kh = q & 1;
            const uint64_t da = tc_desc_sw64(sa + ((j + 1) * TC_PIX + dx) * 64 + kh * 32);
            const uint32_t sb = w0 + dx * CP_WDX + (2 * kh) * (96 * 16) + dl * (NC * 16);
            if (q == 0 && dl == 0) {  // row j + 1 starts here
              mma(dst, da, sb, NC, 0u);
              if (dh > 0) mma(dst + 32, da, sb + NC * 16, NC * dh, 1u);
            } else {
              mma(dst, da, sb, NC * (dh - dl + 1), 1u);
            }
          }
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(empty(st))
                     : "memory");
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tfull(st))
                     : "memory");
      }
      if (u > 0) {  // the last MMAs complete before TMEM is freed
        volatile int never = 0;
        cp_wait(tfull(st), (u - 1) & 1u, &never);
      }
    }
  } else {
    // epilogue: warp w drains TMEM lanes 32 (w % 4) .. (pixels x0 + 32 (w % 4) +
    // lane) of rows (w / 4) half .. of each job
    const int half = (rb + 1) >> 1, q0 = (warp >> 2) * half, q1 = min(q0 + half, rb);
    float bv[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) bv[c] = bias ? bias[c] : 0.0f;
    for (int64_t k = 0; k < njob; ++k) {
      const int st = (int)(k % CP_STAGES);
      const int64_t job = blockIdx.x + k * gridDim.x;
      const int gx = (int)(job % segs) * TPX + (warp & 3) * 32 + lane, r0 = (int)((job / segs) % chunks) * rb;
      const int img = (int)(job / ((int64_t)segs * chunks));
      const int64_t p0 = ((int64_t)img * im.R + r0) * im.W + gx;
      uint4 mr[2][4];  // the masks of this warp's rows (at most two), on their way during the MMAs
      if (mask_ref)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const bool on = q0 + h < q1 && r0 + q0 + h < im.R && gx < im.W;
          const uint4* src = reinterpret_cast<const uint4*>(mask_ref + (on ? p0 + (int64_t)(q0 + h) * im.W : 0) * NC);
#pragma unroll
          for (int c = 0; c < 4; ++c) mr[h][c] = __ldg(src + c);
        }
      // the warp leaves together or not at all (tcgen05.ld is warp-collective)
      const bool okl = cp_wait(tfull(st), (uint32_t)(k / CP_STAGES) & 1u, abort);
      if (!__all_sync(0xffffffffu, okl)) {
        *abort = 1;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = q0 + h;
        if (r >= q1) break;
        uint32_t v[NC];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
            "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
              "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
              "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
              "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
            : "r"(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(128 * st + 32 * (rb - 1 - r))));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (r + 1 == q1) {  // this warp's last read of the region
          asm volatile("tcgen05.fence::before_thread_sync;");
          __syncwarp();
          if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tempty(st)) : "memory");
        }
        if (gx < im.W && r0 + r < im.R) {
          uint32_t o[NC / 2];
          const uint32_t* m = reinterpret_cast<const uint32_t*>(mr[h]);
#pragma unroll
          for (int c = 0; c < NC; c += 2) {
            float f0 = __uint_as_float(v[c]) + bv[c], f1 = __uint_as_float(v[c + 1]) + bv[c + 1];
            if (relu) {
              f0 = fmaxf(f0, 0.0f);
              f1 = fmaxf(f1, 0.0f);
            }
            if (mask_ref) {
              const uint32_t w = m[c / 2];
              if (!(__uint_as_float(w << 16) > 0.0f)) f0 = 0.0f;
              if (!(__uint_as_float(w & 0xFFFF0000u) > 0.0f)) f1 = 0.0f;
            }
            const __nv_bfloat162 hv = __floats2bfloat162_rn(f0, f1);
            o[c / 2] = *reinterpret_cast<const uint32_t*>(&hv);
          }
          uint4* dst = reinterpret_cast<uint4*>(y + (p0 + (int64_t)r * im.W) * NC);
#pragma unroll
          for (int c = 0; c < 4; ++c) dst[c] = make_uint4(o[4 * c], o[4 * c + 1], o[4 * c + 2], o[4 * c + 3]);
        }
      }
      if (q0 >= q1) {  // rb = 1: the second half of the warps has no row
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tempty(st)) : "memory");
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (tid == 0 && *abort) atomicExch(err, 1);
  if (warp == 9) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  }
}

// layer 6 (32 -> 1); out = m * (conv + b6).  Each tap's 32-channel sum is
// formed on its own (one FMA chain from 0) and the nine are added to b6 in tap
// order: the order of k_net_fwd, whose results this kernel reproduces bit for
// bit.
__global__ void k_l6_fwd(Image im, const bf16* __restrict__ y5, const float* __restrict__ P,
                         const float2* __restrict__ in, float* __restrict__ out) {
  __shared__ float w[W6_N + B6_N];
  for (int i = threadIdx.x; i < W6_N + B6_N; i += blockDim.x) w[i] = P[OFF_W6 + i];
  __syncthreads();
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= im.npx()) return;
  const int x = (int)(p % im.W), r = (int)(p / im.W);
  const int lo = (r / im.R) * im.R, hi = lo + im.R;
  float a = w[W6_N];
  for (int d = 0; d < 9; ++d) {
    const int xx = x + d % 3 - 1, rr = r + d / 3 - 1;
    if (xx < 0 || xx >= im.W || rr < lo || rr >= hi) continue;
    const int4* src = reinterpret_cast<const int4*>(y5 + ((int64_t)rr * im.W + xx) * NC);
    float t = 0.0f;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int4 v = src[q];
      const bf16* e = reinterpret_cast<const bf16*>(&v);
#pragma unroll
      for (int c = 0; c < 8; ++c) t = __fmaf_rn(w[d * NC + q * 8 + c], __bfloat162float(e[c]), t);
    }
    a = __fadd_rn(a, t);
  }
  out[p] = in[p].y * a;
}

// --------------------------------------------- fused forward: all six layers
// One launch computes N(in) with every hidden activation kept on chip.  A CTA
// owns a strip of FZ_OUT = 116 output columns and a run of rows of one image
// and walks down it one step at a time; step tau computes layer 1 at row tau,
// layer l (2..5) at row tau - 2 (l - 1) and layer 6 at row tau - 10, so the
// rows a step reads were all finished in earlier steps and the layers of one
// step are independent.  Every layer computes 128 columns (the tensor cores'
// M), the strip's 116 plus 6 on each side: layer l is exact on 128 - 2 (l - 1)
// of them, which leaves layer 6 exact on the strip.
//   * layer 1 (2 -> 32, CUDA cores, warps 20-27): one pixel of two rows per
//     thread, eight output channels' FMA chains side by side, each in
//     k_l1_fwd's order; bf16 result into ring 0.  Two groups of four warps take
//     the pairs of rows in turn.
//   * layers 2-5 (tcgen05, lane 0 of warp 8 + l - 2): the MMAs are input-row
//     stationary.  At step tau layer l takes its newest input row, rho + 1
//     (rho = the output row it finishes), from ring l - 2 (64-byte swizzled
//     K-major rows of 64 bytes, one per pixel, as k_conv32_tma's tensor
//     copies lay them out) and multiplies it, shifted by dx = 0, 1, 2 pixels
//     and split in two channel halves, by the weights of the three tap rows
//     at once: N = 96 = (dy, n), contributions to output rows rho + 2 - dy.
//     Each output row accumulates in one of 16 TMEM slots of 32 columns, a
//     ring shared by the four layers (fz_col): rows rho + 2, rho + 1, rho lie
//     at increasing columns, and a layer issues 6 MMAs per step (12 in the two
//     steps of 16 in which its three slots wrap).  The slot of row rho receives
//     its taps in (dy, dx, kh) order, as in k_conv32_tma, from zero.
//   * epilogues of layers 2-4 (warps 0-7, one TMEM lane = one pixel per
//     thread): read the finished slot of row rho and zero it, bias, ReLU,
//     bf16, 0 outside the image (the next layer's zero padding), into ring
//     l - 1 (the swizzle applied by hand).  Two groups of four warps take the
//     steps in turn.
//   * layers 5-6 (warps 12-19, in turn as well): layer 5's epilogue forms the
//     nine tap partials of layer 6 (a float per tap and pixel, ring T) from its
//     bf16-rounded values, nine FMA chains side by side; layer 6 adds them up:
//     out = m (b6 + sum).
// Ring 0 holds 8 rows (of step k in slot k & 7), rings 1-3 hold 2 (row rho in
// slot rho & 1): a step reads the row that the step before wrote.  T holds 4.
// Every layer's arithmetic is that of the layer-by-layer path (k_l1_fwd,
// k_conv32_tma, k_l6_fwd), so the two give identical outputs.
// Barriers (mbarriers; k counts the steps of the CTA over all its units):
// rdy0 / rdy[j] (ring j row of step k written and, for j >= 1, the slot that
// layer j + 2 enters next zeroed: 4 warp arrivals -> MMA of layer j + 2 at step
// k + 1), mdone[j] (commit of layer j + 2's MMAs at step k -> epilogue; frees
// the ring rows they read: ring 0's for layer 1 six steps on, the others' for
// the epilogue of the next step), tempty[j] (slot read and zeroed: 4 warp
// arrivals -> MMAs at a unit's first step, whose last step before cleared the
// rows begun; layer 5's -> layer 2's MMAs five steps on, which enter its slot),
// tdone (T row of step k written and read: layers 5-6 take turns).  A parity
// wait is sound while its barrier is neither two phases ahead nor one behind:
// eight barriers per layer for mdone, tempty and rdy0 and two for rdy and tdone
// give that, whatever the warps' relative speeds (with four for mdone a slow
// epilogue warp can miss a phase).  Every wait is
// bounded; one that gives up raises a shared abort flag, after which every role
// runs its remaining steps without waiting or computing, the CTA waits
// (bounded) for its MMAs in flight, frees TMEM and sets *err.
// Bound by the issue slots and the shared-memory pipe together (70 % and 75 %
// busy; the tensor pipe 38 %).  At 2048^2: 440 us; 561 us with one group of
// warps per role, whose epilogue (3200 cycles of work in a step of 4280) paced
// the others, and four slots per layer (9 MMAs per step instead of 6.75); with
// one row per thread in layer 1 and 24 warps 451 us.
constexpr int FZ_OUT = TPX - 12;                       // 116
constexpr int FZ_ROW = TC_PIX * NC * 2;                // 8320 bytes: one activation row, 130 pixel slots
constexpr int FZ_RINGB = 2 * FZ_ROW;                   // 16,640: rings 1-3, two rows
constexpr int FZ_RING0 = 8 * FZ_ROW;                   // 66,560: ring 0, eight rows
constexpr int FZ_W = 114 * 1024;                       // weights of layers 2-5: 116,736
constexpr int FZ_WDX = 4 * 96 * 16;                    // B bytes of one horizontal tap: 6144
constexpr int FZ_TRING = 4;                            // rows of the tap-partial ring
constexpr int FZ_TROW = 9 * TC_PIX;                    // floats of a T row: 9 taps x 130 slots
constexpr int FZ_T = FZ_W + NMID * TC_W;               // 190,464
constexpr int FZ_W1 = FZ_T + FZ_TRING * FZ_TROW * 4;   // 209,184: layer-1 weights [d][ci][co], then b1
constexpr int FZ_W6 = FZ_W1 + (NC * 20 + NC) * 4;      // 211,872: W6 as [c][12 taps], then b6
constexpr int FZ_BM = FZ_W6 + 1552;                    // 213,424: biases of layers 2-5
constexpr int FZ_BAR = FZ_BM + NMID * NC * 4;          // 213,936
constexpr int FZ_NBAR = 80;
constexpr int FZ_SMEM = FZ_BAR + 8 * FZ_NBAR + 16;     // 214,592
constexpr int FZ_THREADS = 896;  // warps 0-7 epilogues 2-4, 8-11 MMAs, 12-19 layers 5-6, 20-27 layer 1
static_assert(FZ_SMEM <= 232448, "fused forward: shared memory");
static_assert(FZ_W % 1024 == 0 && FZ_T % 16 == 0 && FZ_BAR % 8 == 0, "fused forward: alignment");

struct FzArgs {
  Image im;
  const float2* in;
  float* out;
  const float* P;
  const bf16* wf;  // [4][9][32 n][32 k] bf16
  int strips, segs, seg_rows;
  int64_t units;
  int* err;
};

// 64 bytes (32 bf16 = 16 words) into the pixel row at shared address row (a
// multiple of 64) in the 64-byte swizzled layout: 16-byte chunk c of the row
// lands at chunk c ^ (address bits 7-8)
__device__ __forceinline__ void fz_st_chunk(uint32_t row, int c, uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(row + ((c ^ ((row >> 7) & 3u)) << 4)), "r"(w0), "r"(w1),
               "r"(w2), "r"(w3)
               : "memory");
}
__device__ __forceinline__ void fz_st_row(uint32_t row, const uint32_t (&w)[NC / 2]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) fz_st_chunk(row, c, w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
}

// Bounded wait of the fused kernel: the waiting thread asks to be suspended
// (up to 20 us per try) until the phase completes, so that spinning warps do
// not take issue slots from the working ones on the same scheduler; gives up
// after FZ_WAIT_NS of wall time (global timer) or when *abort is raised,
// raising it itself on the time limit.
constexpr uint64_t FZ_WAIT_NS = 200000000ull;  // 0.2 s
__device__ __forceinline__ uint64_t fz_now() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ bool fz_wait(uint32_t bar, uint32_t parity, volatile int* abort) {
  uint64_t t0 = 0;
  for (uint32_t it = 0; it < (1u << 26); ++it) {  // the iteration bound backs up the time limit
    uint32_t ok = 0;
    asm volatile(
        "{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2, 20000;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if (it == 0) t0 = fz_now();
    if ((it & 15) == 15) {
      if (*abort) return false;
      if (fz_now() - t0 > FZ_WAIT_NS) break;
    }
  }
  *abort = 1;
  return false;
}

// Tensor-memory column of the accumulator of layer j + 2's output row that is
// finished at step kf.  The 16 slots of 32 columns form one ring for the four
// layers: at step k layer j + 2 holds the rows finished at k + 2, k + 1 and k
// (which one input row feeds) at increasing slots, and every step moves all
// layers one slot down.  The slot a layer enters is the one that the layer below
// it finished the step before; layer 2 enters the one that layer 5 finished five
// steps before.
__device__ __forceinline__ int fz_col(int j, int64_t kf) { return 32 * ((3 * j - (int)kf) & 15); }

// 32 zero columns of tensor memory at taddr for this warp's 32 lanes
__device__ __forceinline__ void fz_tmem_zero32(uint32_t taddr) {
  const uint32_t z = 0u;
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,"
      "%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(taddr),
      "r"(z)
      : "memory");
}

// Reads the accumulator that layer j + 2 finished at step k (32 columns, this
// warp's lanes; tlane = TMEM address of lane 32 (warp % 4), column 0) into v,
// then starts zeroing its slot (at a unit's last step also the two slots of the
// rows begun, which leaves no partial sums to the next unit); fz_release
// completes it.  okw (warp-uniform) false: nothing is read, v = 0.
__device__ __forceinline__ void fz_take(uint32_t tlane, int j, int64_t k, bool okw, bool last, uint32_t (&v)[NC]) {
  const uint32_t tacc = tlane + (uint32_t)fz_col(j, k);
  if (okw) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
        "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(tacc));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
    fz_tmem_zero32(tacc);
    if (last) {
      fz_tmem_zero32(tlane + (uint32_t)fz_col(j, k + 1));
      fz_tmem_zero32(tlane + (uint32_t)fz_col(j, k + 2));
    }
  } else {
#pragma unroll
    for (int c = 0; c < NC; ++c) v[c] = 0u;
  }
}

// after fz_take: the zeroing stores are complete and the slot is released to
// the MMAs (layer j + 3's write it two steps on)
__device__ __forceinline__ void fz_release(uint32_t tempty) {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncwarp();
  if ((threadIdx.x & 31) == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tempty) : "memory");
}

// (a0 + b0, a1 + b1), each rounded to nearest as a scalar addition
__device__ __forceinline__ void fz_add2(float a0, float a1, float b0, float b1, float& r0, float& r1) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(fz_pk(a0, a1)), "l"(fz_pk(b0, b1)));
  fz_upk(r, r0, r1);
}

__device__ __forceinline__ void fz_unit(const FzArgs& a, int64_t u, int& img, int& r0, int& r1, int& x0) {
  const int strip = (int)(u % a.strips);
  const int64_t q = u / a.strips;
  const int seg = (int)(q % a.segs);
  img = (int)(q / a.segs);
  x0 = strip * FZ_OUT;
  r0 = seg * a.seg_rows;
  r1 = min(r0 + a.seg_rows, a.im.R);
}

__global__ void __launch_bounds__(FZ_THREADS, 1) k_net_fwd(const __grid_constant__ FzArgs a) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t base = smem_addr(smem_raw);
  const uint32_t bars = base + FZ_BAR;
  auto rdy0 = [&](int64_t k) { return bars + 8 * (int)(k & 7); };                          // ring 0
  auto rdy = [&](int j, int64_t k) { return bars + 8 * (6 + 2 * j + (int)(k & 1)); };  // rings 1-3
  auto mdone = [&](int j, int64_t k) { return bars + 8 * (14 + 8 * j + (int)(k & 7)); };
  auto tempty = [&](int j, int64_t k) { return bars + 8 * (46 + 8 * j + (int)(k & 7)); };
  auto tdone = [&](int b) { return bars + 8 * (78 + b); };
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem_raw + FZ_BAR + 8 * FZ_NBAR);
  volatile int* abort = reinterpret_cast<volatile int*>(smem_raw + FZ_BAR + 8 * FZ_NBAR + 8);
  float* sT = reinterpret_cast<float*>(smem_raw + FZ_T);
  float* sW1 = reinterpret_cast<float*>(smem_raw + FZ_W1);
  float* sW6 = reinterpret_cast<float*>(smem_raw + FZ_W6);
  float* sBM = reinterpret_cast<float*>(smem_raw + FZ_BM);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const Image& im = a.im;

  // rings and T start at 0 (slots 0 and 129 of every ring row stay 0)
  for (int i = tid; i < FZ_W / 16; i += FZ_THREADS) reinterpret_cast<int4*>(smem_raw)[i] = make_int4(0, 0, 0, 0);
  for (int i = tid; i < FZ_TRING * FZ_TROW; i += FZ_THREADS) sT[i] = 0.0f;
  for (int i = tid; i < NMID * 9 * NC * 4; i += FZ_THREADS) {  // B operands, as in k_conv32_tma
    // [dx][channel group g][dy * 32 + n][8 k]: one horizontal tap's three tap rows side by side in N
    const int g = i & 3, n = (i >> 2) % NC, d = ((i >> 2) / NC) % 9, l = (i >> 2) / (NC * 9);
    const int dy = d / 3, dx = d % 3;
    *reinterpret_cast<int4*>(smem_raw + FZ_W + l * TC_W + dx * FZ_WDX + g * (96 * 16) + (dy * NC + n) * 16) =
        *reinterpret_cast<const int4*>(a.wf + (int64_t)l * WM_N + (d * NC + n) * NC + g * 8);
  }
  // layer 1: weight (tap d, input ci) of the 32 outputs contiguous, so that a
  // thread feeds eight output channels' FMA chains from two float4 loads
  for (int i = tid; i < 18 * NC; i += FZ_THREADS) {
    const int co = i % NC, q = i / NC;
    sW1[i] = a.P[OFF_W1 + co * 18 + q];
  }
  for (int i = tid; i < NC; i += FZ_THREADS) sW1[18 * NC + i] = a.P[OFF_W1 + W1_N + i];
  // layer 6: the nine taps of input channel c contiguous (padded to 12)
  for (int i = tid; i < NC * 12; i += FZ_THREADS) {
    const int c = i / 12, d = i % 12;
    sW6[i] = d < 9 ? a.P[OFF_W6 + d * NC + c] : 0.0f;
  }
  if (tid == 0) sW6[NC * 12] = a.P[OFF_W6 + W6_N];
  for (int i = tid; i < NMID * NC; i += FZ_THREADS) sBM[i] = a.P[off_wm(i / NC) + WM_N + i % NC];
  if (tid == 0) {
    for (int b = 0; b < FZ_NBAR; ++b) {
      const uint32_t cnt = (b >= 14 && b < 46) ? 1u : 4u;  // mdone: one commit; rdy, tempty: four warps
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bars + 8 * b), "r"(cnt));
    }
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 8) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_addr(tslot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("fence.proxy.async.shared::cta;");  // zeroed rings and weights are read by the tensor cores
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tslot;
  // every MMA accumulates: the output-row slots of tensor memory start at 0
  if (warp < 4) {
    for (int c = 0; c < 512; c += 32) fz_tmem_zero32(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c);
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");

  if (warp >= 20) {
    // layer 1, two rows at a time (each weight read from shared memory serves
    // both): warps 20-23 and 24-27 take the pairs of steps in turn; thread t of
    // a group = pixel slot t + 1 of ring 0
    const int t = tid & 127;
    int grp = (warp - 20) >> 2;
    int64_t k = 0;
    for (int64_t u = blockIdx.x; u < a.units; u += gridDim.x) {
      int img, r0, r1, x0;
      fz_unit(a, u, img, r0, r1, x0);
      const int nsteps = r1 - r0 + 15;
      const int x = x0 - 6 + t;
      for (int st = 0; st < nsteps; st += 2, grp ^= 1) {
        const int np = min(2, nsteps - st), tau = r0 - 5 + st;
        if (grp) {
          k += np;
          continue;
        }
        float2 v[12];  // rows tau - 1 .. tau + 2, columns x - 1 .. x + 1
#pragma unroll
        for (int d = 0; d < 12; ++d) {
          const int xx = x + d % 3 - 1, rr = tau + d / 3 - 1;
          v[d] = (xx >= 0 && xx < im.W && rr >= 0 && rr < im.R)
                     ? __ldg(a.in + ((int64_t)img * im.R + rr) * im.W + xx)
                     : make_float2(0.f, 0.f);
        }
        const bool in_x = x >= 0 && x < im.W;
        const bool in0 = in_x && tau >= 0 && tau < im.R, in1 = in_x && tau + 1 >= 0 && tau + 1 < im.R;
        // the rows overwritten here were read by layer 2's MMAs of steps k - 7 and k - 6
        if (k >= 6) fz_wait(mdone(0, k - 6), (uint32_t)((k - 6) >> 3) & 1u, abort);
        const uint32_t row0 = base + (uint32_t)((int)(k & 7) * FZ_ROW + (t + 1) * 64);
        const uint32_t row1 = base + (uint32_t)((int)((k + 1) & 7) * FZ_ROW + (t + 1) * 64);
        // eight output channels at a time, each one FMA chain in k_l1_fwd's order
#pragma unroll
        for (int cg = 0; cg < NC; cg += 8) {
          uint64_t acc[2][4];  // channel pairs (cg + 2q, cg + 2q + 1) of the two rows
#pragma unroll
          for (int q = 0; q < 4; ++q)
            acc[0][q] = acc[1][q] = *reinterpret_cast<const uint64_t*>(sW1 + 18 * NC + cg + 2 * q);
#pragma unroll
          for (int e = 0; e < 18; ++e) {
            const float4 wa = *reinterpret_cast<const float4*>(sW1 + e * NC + cg);
            const float4 wb = *reinterpret_cast<const float4*>(sW1 + e * NC + cg + 4);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const float xv = (e & 1) ? v[(e >> 1) + 3 * h].y : v[(e >> 1) + 3 * h].x;
              const uint64_t x2 = fz_pk(xv, xv);
              fz_fma2(acc[h][0], fz_pk(wa.x, wa.y), x2);
              fz_fma2(acc[h][1], fz_pk(wa.z, wa.w), x2);
              fz_fma2(acc[h][2], fz_pk(wb.x, wb.y), x2);
              fz_fma2(acc[h][3], fz_pk(wb.z, wb.w), x2);
            }
          }
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t o[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              float a0, a1;
              fz_upk(acc[h][q], a0, a1);
              o[q] = (h ? in1 : in0) ? fz_relu2(a0, a1) : 0u;
            }
            const uint32_t row = h ? row1 : row0;
            if (h < np) fz_st_chunk(row, cg / 8, o[0], o[1], o[2], o[3]);
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(rdy0(k)) : "memory");
          if (np == 2) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(rdy0(k + 1)) : "memory");
        }
        k += np;
      }
    }
  } else if (warp >= 12) {
    // layer 5's epilogue, the tap partials and layer 6: warps 12-15 take the
    // even steps, 16-19 the odd ones; thread t of a group = TMEM lane t = pixel
    // slot t + 1
    const int t = tid & 127, grp = (warp - 12) >> 2;
    const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    constexpr int j = NMID - 1;
    int64_t k = 0;
    for (int64_t u = blockIdx.x; u < a.units; u += gridDim.x) {
      int img, r0, r1, x0;
      fz_unit(a, u, img, r0, r1, x0);
      const int nsteps = r1 - r0 + 15;
      const int x = x0 - 6 + t;
      for (int st = 0; st < nsteps; ++st, ++k) {
        const int tau = r0 - 5 + st, b = (int)(k & 1);
        if (b != grp) continue;
        const bool last = st == nsteps - 1;
        // layer 6 writes row tau - 10 at the end of the step: its mask value now
        const int r6 = tau - 10;
        const bool out6 = r6 >= r0 && r6 < r1 && t >= 6 && t < 6 + FZ_OUT && x < im.W;
        const int64_t p6 = ((int64_t)img * im.R + r6) * im.W + x;
        const float m6 = out6 ? __ldg(a.in + p6).y : 0.0f;
        // layer 5 (row tau - 8): its values, bf16-rounded as layer 6 reads them
        bool okl = fz_wait(mdone(j, k), (uint32_t)(k >> 3) & 1u, abort);
        okl = okl && !*abort;
        const bool okw = __all_sync(0xffffffffu, okl);  // tcgen05.ld is warp-collective
        const int rho = tau - 2 * (j + 1);
        uint32_t v5[NC];
        fz_take(tlane, j, k, okw, last, v5);
        const bool in_img = okw && rho >= 0 && rho < im.R && x >= 0 && x < im.W;
        fz_release(tempty(j, k));
        // tap partials of row rho: nine chains over c = 0 .. 31, side by side (taps in pairs)
        const float4* bj = reinterpret_cast<const float4*>(sBM + j * NC);
        uint64_t tp[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) tp[q] = fz_pk(0.0f, 0.0f);
        float t8 = 0.0f;
#pragma unroll
        for (int c = 0; c < NC; c += 4) {
          const float4 bb = bj[c / 4];
          float s0, s1, s2, s3;
          fz_add2(__uint_as_float(v5[c]), __uint_as_float(v5[c + 1]), bb.x, bb.y, s0, s1);
          fz_add2(__uint_as_float(v5[c + 2]), __uint_as_float(v5[c + 3]), bb.z, bb.w, s2, s3);
          const uint32_t h0 = in_img ? fz_relu2(s0, s1) : 0u, h1 = in_img ? fz_relu2(s2, s3) : 0u;
          const float f[4] = {__uint_as_float(h0 << 16), __uint_as_float(h0 & 0xFFFF0000u), __uint_as_float(h1 << 16),
                              __uint_as_float(h1 & 0xFFFF0000u)};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float4 wa = *reinterpret_cast<const float4*>(sW6 + (c + e) * 12);
            const float4 wb = *reinterpret_cast<const float4*>(sW6 + (c + e) * 12 + 4);
            const float wc = sW6[(c + e) * 12 + 8];
            const uint64_t f2 = fz_pk(f[e], f[e]);
            fz_fma2(tp[0], fz_pk(wa.x, wa.y), f2);
            fz_fma2(tp[1], fz_pk(wa.z, wa.w), f2);
            fz_fma2(tp[2], fz_pk(wb.x, wb.y), f2);
            fz_fma2(tp[3], fz_pk(wb.z, wb.w), f2);
            t8 = __fmaf_rn(wc, f[e], t8);
          }
        }
        // T holds the rows of the steps up to k - 1, and the slot written below
        // was last read at step k - 1
        if (k >= 1) fz_wait(tdone(b ^ 1), (uint32_t)((k - 1) >> 1) & 1u, abort);
        // layer 6 at row tau - 10 from the tap partials of earlier steps
        if (!*abort && out6) {
          float acc = sW6[NC * 12];
#pragma unroll
          for (int d = 0; d < 9; ++d) {
            const int dy = d / 3, dx = d % 3;
            acc = __fadd_rn(acc, sT[((r6 - 1 + dy) & 3) * FZ_TROW + d * TC_PIX + t + dx]);
          }
          a.out[p6] = m6 * acc;
        }
        float* tr = sT + (rho & 3) * FZ_TROW + t + 1;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float ta, tb;
          fz_upk(tp[q], ta, tb);
          tr[(2 * q) * TC_PIX] = ta;
          tr[(2 * q + 1) * TC_PIX] = tb;
        }
        tr[8 * TC_PIX] = t8;
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tdone(b)) : "memory");
      }
    }
  } else if (warp >= 8) {
    // warp 8 + j issues the MMAs of layer j + 2 (ring j in): one issuing thread
    // per layer, so that the four layers' MMAs of a step overlap on the tensor
    // cores (an issuing thread waits out each MMA's operand fetch)
    if (lane == 0) {
      const int j = warp - 8;
      int64_t k = 0;
      uint32_t last_bar = 0, last_par = 0;
      bool ok = true;
      for (int64_t u = blockIdx.x; u < a.units && ok; u += gridDim.x) {
        int img, r0, r1, x0;
        fz_unit(a, u, img, r0, r1, x0);
        const int nsteps = r1 - r0 + 15;
        for (int st = 0; st < nsteps && ok; ++st, ++k) {
          const int tau = r0 - 5 + st;
          {
            if (k >= 1 && !(j == 0 ? fz_wait(rdy0(k - 1), (uint32_t)((k - 1) >> 3) & 1u, abort)
                                   : fz_wait(rdy(j, k - 1), (uint32_t)((k - 1) >> 1) & 1u, abort))) {
              ok = false;
              break;
            }
            // the slot written first here has been read and zeroed: by the epilogue
            // that wrote the input row waited for above (layer 5's of step k - 5 for
            // layer 2); the first step of a unit also waits for the step before,
            // whose epilogue cleared the rows that the previous unit had begun
            if ((st == 0 && k >= 1 && !fz_wait(tempty(j, k - 1), (uint32_t)((k - 1) >> 3) & 1u, abort)) ||
                (j == 0 && k >= 5 && !fz_wait(tempty(NMID - 1, k - 5), (uint32_t)((k - 5) >> 3) & 1u, abort))) {
              ok = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
            // input row rho + 1 (the newest) enters output rows rho + 2, rho + 1 and
            // rho (tap rows dy = 0, 1, 2): runs of those whose slots are adjacent
            // in tensor memory take one MMA per (dx, kh), N = 32 x run length
            const int rho = tau - 2 * (j + 1);
            const uint32_t row = base + (uint32_t)(j == 0 ? (int)((k + 7) & 7) * FZ_ROW
                                                          : FZ_RING0 + (j - 1) * FZ_RINGB + ((rho + 1) & 1) * FZ_ROW);
            const uint32_t wl = base + (uint32_t)(FZ_W + j * TC_W);
            for (int dy = 0; dy < 3;) {
              const int c0 = fz_col(j, k + 2 - dy);
              const int n = min(3 - dy, (512 - c0) / 32);
              const uint32_t idesc = tc_idesc(128, 32 * n);
#pragma unroll 1
              for (int q = 0; q < 6; ++q) {
                const int dx = q >> 1, kh = q & 1;
                const uint64_t da = tc_desc_sw64(row + dx * 64 + kh * 32);
                const uint64_t db =
                    tc_desc(wl + (uint32_t)(dx * FZ_WDX + (2 * kh) * (96 * 16) + dy * NC * 16), 96 * 16, 128);
                asm volatile(
                    "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                    "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(
                        tmem + (uint32_t)c0),
                    "l"(da), "l"(db), "r"(idesc), "r"(1u));
              }
              dy += n;
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             mdone(j, k))
                         : "memory");
            last_bar = mdone(j, k);
            last_par = (uint32_t)(k >> 3) & 1u;
          }
        }
      }
      if (last_bar) {  // the last commit covers every MMA this thread issued: they finish before TMEM is freed
        volatile int never = 0;
        fz_wait(last_bar, last_par, &never);
      }
    }
  } else {
    // epilogues of layers 2-4: warps 0-3 take the even steps, 4-7 the odd ones;
    // thread i of a group = TMEM lane i = pixel slot i + 1
    const int i = tid & 127, grp = warp >> 2;
    const uint32_t tlane = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    int64_t k = 0;
    for (int64_t u = blockIdx.x; u < a.units; u += gridDim.x) {
      int img, r0, r1, x0;
      fz_unit(a, u, img, r0, r1, x0);
      const int nsteps = r1 - r0 + 15;
      const int x = x0 - 6 + i;
      for (int st = 0; st < nsteps; ++st, ++k) {
        const int tau = r0 - 5 + st, b = (int)(k & 1);
        if (b != grp) continue;
        const bool last = st == nsteps - 1;
#pragma unroll 1
        for (int j = 0; j < NMID - 1; ++j) {
          bool okl = fz_wait(mdone(j, k), (uint32_t)(k >> 3) & 1u, abort);
          okl = okl && !*abort;
          const bool okw = __all_sync(0xffffffffu, okl);  // tcgen05.ld is warp-collective
          const int rho = tau - 2 * (j + 1);
          uint32_t v[NC];
          fz_take(tlane, j, k, okw, last, v);
          const bool in_img = okw && rho >= 0 && rho < im.R && x >= 0 && x < im.W;
          const float4* bj = reinterpret_cast<const float4*>(sBM + j * NC);
          uint32_t o[NC / 2];
#pragma unroll
          for (int c = 0; c < NC; c += 4) {
            const float4 bb = bj[c / 4];
            float s0, s1, s2, s3;
            fz_add2(__uint_as_float(v[c]), __uint_as_float(v[c + 1]), bb.x, bb.y, s0, s1);
            fz_add2(__uint_as_float(v[c + 2]), __uint_as_float(v[c + 3]), bb.z, bb.w, s2, s3);
            o[c / 2] = in_img ? fz_relu2(s0, s1) : 0u;
            o[c / 2 + 1] = in_img ? fz_relu2(s2, s3) : 0u;
          }
          // the row overwritten here was read by layer j + 3's MMAs of the step before
          if (k >= 1) fz_wait(mdone(j + 1, k - 1), (uint32_t)((k - 1) >> 3) & 1u, abort);
          fz_release(tempty(j, k));
          fz_st_row(base + (uint32_t)(FZ_RING0 + j * FZ_RINGB + (rho & 1) * FZ_ROW + (i + 1) * 64), o);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          __syncwarp();
          if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(rdy(j + 1, b)) : "memory");
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (tid == 0 && *abort) atomicExch(a.err, 1);
  if (warp == 8) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  }
}

// ----------------------------------------------------------- backward
// g6 = dout * m
__global__ void __launch_bounds__(256) k_l6_gate(int64_t npx, const float* __restrict__ dout,
                                                 const float2* __restrict__ in, float* __restrict__ g6) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p < npx) g6[p] = dout[p] * in[p].y;
}

// The gradients of layers 1 and 6 on the CUDA cores walk the image the same
// way: a warp takes a run of BW_RUN pixels of one row in four segments; lane
// (seg, cg) walks its segment left to right for channels 4 cg .. 4 cg + 3 (8
// lanes read a pixel's 64 bytes), keeping the 3 x 3 window of the other
// operand in registers (three new values a pixel) and BW_PF pixels' loads in
// flight, and its share of the weight gradient in registers to the end.  The
// lanes' and warps' shares are added in a fixed order.  Bounded by the
// packed FMAs (fma.rn.f32x2) and the one pass over the 32-channel operand.
// At 16 x 512^2: k_l6_back 161 us and k_l1_wgrad 147 us; one pixel per warp
// (lane = channel, every tap gathered anew) took 1668 + 197 us (weight and data
// gradient apart) and 1481 us.
constexpr int BW_THREADS = 128;
constexpr int BW_SEG = 32;           // pixels per lane and run
constexpr int BW_RUN = 4 * BW_SEG;
constexpr int BW_CTAS = 3;           // per SM

// sum over the four segments (lanes that share cg)
__device__ __forceinline__ float seg_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 8);
  return v + __shfl_xor_sync(0xffffffffu, v, 16);
}

__device__ __forceinline__ float2 fz_unpk(uint64_t v) {
  return make_float2(__uint_as_float((uint32_t)v), __uint_as_float((uint32_t)(v >> 32)));
}

// the four BF16 of v as two packed FP32 pairs
__device__ __forceinline__ void bf4_pairs(uint2 v, uint64_t& a, uint64_t& b) {
  a = fz_pk(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xFFFF0000u));
  b = fz_pk(__uint_as_float(v.y << 16), __uint_as_float(v.y & 0xFFFF0000u));
}

// Layer 6 backward in one pass over y5: the data gradient
//   dy5[p][ci] = (sum_d W6[d][ci] g6[p - off(d)]) (y5[p][ci] > 0)
// and the weight-gradient partials, slot d * 32 + ci: sum_p g6[p - off(d)]
// y5[p][ci]; slot 288: sum g6.  Both need the same 3 x 3 window of g6.
__global__ void __launch_bounds__(BW_THREADS, BW_CTAS) k_l6_back(Image im, const float* __restrict__ g6,
                                                                 const bf16* __restrict__ y5,
                                                                 const float* __restrict__ P, bf16* __restrict__ dy5,
                                                                 float* __restrict__ part) {
  constexpr int PF = 8;
  __shared__ float sm[BW_THREADS / 32][W6_N + B6_N];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, cg = lane & 7, seg = lane >> 3;
  uint64_t wt[9][2], acc[9][2];
#pragma unroll
  for (int d = 0; d < 9; ++d) {
    const float* q = P + OFF_W6 + d * NC + 4 * cg;
    wt[d][0] = fz_pk(q[0], q[1]);
    wt[d][1] = fz_pk(q[2], q[3]);
    acc[d][0] = acc[d][1] = 0;
  }
  float bacc = 0.0f;
  const int runs = (im.W + BW_RUN - 1) / BW_RUN;
  const int64_t tasks = (int64_t)runs * im.H;
  for (int64_t t = (int64_t)blockIdx.x * (BW_THREADS / 32) + w; t < tasks; t += (int64_t)gridDim.x * (BW_THREADS / 32)) {
    const int r = (int)(t / runs), xs = (int)(t - (int64_t)r * runs) * BW_RUN + seg * BW_SEG;
    const int lo = (r / im.R) * im.R, hi = lo + im.R;
    const bool rv[3] = {r - 1 >= lo, true, r + 1 < hi};
    const float* gr = g6 + (int64_t)r * im.W;
    auto g_at = [&](int k, int x) {  // g6 at row r + k - 1, column x
      return (rv[k] && x >= 0 && x < im.W) ? __ldg(gr + (int64_t)(k - 1) * im.W + x) : 0.0f;
    };
    float g0[3], g1[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      g0[k] = g_at(k, xs - 1);
      g1[k] = g_at(k, xs);
    }
    const int64_t px0 = (int64_t)r * im.W;
    for (int x0 = xs; x0 < xs + BW_SEG && x0 < im.W; x0 += PF) {
      uint2 yv[PF];
      float gn[3][PF];
#pragma unroll
      for (int j = 0; j < PF; ++j)
        yv[j] = x0 + j < im.W ? __ldg(reinterpret_cast<const uint2*>(y5 + (px0 + x0 + j) * NC + 4 * cg))
                              : make_uint2(0u, 0u);
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < PF; ++j) gn[k][j] = g_at(k, x0 + j + 1);
#pragma unroll
      for (int j = 0; j < PF; ++j) {
        uint64_t ya, yb, da = 0, db = 0;
        bf4_pairs(yv[j], ya, yb);
#pragma unroll
        for (int d = 0; d < 9; ++d) {  // g6 at p - off(d): row 2 - d / 3, column 2 - d % 3 of the window
          const int k = 2 - d / 3, c = 2 - d % 3;
          const float g = c == 0 ? g0[k] : (c == 1 ? g1[k] : gn[k][j]);
          const uint64_t gg = fz_pk(g, g);
          fz_fma2(acc[d][0], ya, gg);
          fz_fma2(acc[d][1], yb, gg);
          fz_fma2(da, wt[d][0], gg);
          fz_fma2(db, wt[d][1], gg);
        }
        if (x0 + j < im.W) {
          bacc += g1[1];
          const float2 a = fz_unpk(da), b = fz_unpk(db), p = fz_unpk(ya), q = fz_unpk(yb);
          const __nv_bfloat162 h0 = __floats2bfloat162_rn(p.x > 0.0f ? a.x : 0.0f, p.y > 0.0f ? a.y : 0.0f);
          const __nv_bfloat162 h1 = __floats2bfloat162_rn(q.x > 0.0f ? b.x : 0.0f, q.y > 0.0f ? b.y : 0.0f);
          *reinterpret_cast<uint2*>(dy5 + (px0 + x0 + j) * NC + 4 * cg) =
              make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          g0[k] = g1[k];
          g1[k] = gn[k][j];
        }
      }
    }
  }
#pragma unroll
  for (int d = 0; d < 9; ++d)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 v = fz_unpk(acc[d][h]);
      const float a = seg_sum(v.x), b = seg_sum(v.y);
      if (seg == 0) {
        sm[w][d * NC + 4 * cg + 2 * h] = a;
        sm[w][d * NC + 4 * cg + 2 * h + 1] = b;
      }
    }
  bacc = seg_sum(bacc);
  if (lane == 0) sm[w][W6_N] = bacc;
  __syncthreads();
  for (int i = threadIdx.x; i < W6_N + B6_N; i += BW_THREADS) {
    float t = 0.0f;
#pragma unroll
    for (int k = 0; k < BW_THREADS / 32; ++k) t += sm[k][i];
    part[(int64_t)blockIdx.x * (W6_N + B6_N) + i] = t;
  }
}

// Layer 1 gradient partials: slot (co * 9 + d) * 2 + ci: sum dy1[p][co] in[p + off(d)][ci];
// slot 576 + co: sum dy1[p][co].  The packed pairs are the two input channels.
__global__ void __launch_bounds__(BW_THREADS, BW_CTAS) k_l1_wgrad(Image im, const bf16* __restrict__ dy1,
                                                                  const float2* __restrict__ in,
                                                                  float* __restrict__ part) {
  constexpr int PF = 4;
  __shared__ float sm[BW_THREADS / 32][W1_N + B1_N];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, cg = lane & 7, seg = lane >> 3;
  uint64_t acc[9][4];
  float bacc[4];
#pragma unroll
  for (int d = 0; d < 9; ++d)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[d][c] = 0;
#pragma unroll
  for (int c = 0; c < 4; ++c) bacc[c] = 0.0f;
  const int runs = (im.W + BW_RUN - 1) / BW_RUN;
  const int64_t tasks = (int64_t)runs * im.H;
  for (int64_t t = (int64_t)blockIdx.x * (BW_THREADS / 32) + w; t < tasks; t += (int64_t)gridDim.x * (BW_THREADS / 32)) {
    const int r = (int)(t / runs), xs = (int)(t - (int64_t)r * runs) * BW_RUN + seg * BW_SEG;
    const int lo = (r / im.R) * im.R, hi = lo + im.R;
    const bool rv[3] = {r - 1 >= lo, true, r + 1 < hi};
    const unsigned long long* ir = reinterpret_cast<const unsigned long long*>(in) + (int64_t)r * im.W;
    auto v_at = [&](int k, int x) -> uint64_t {  // in at row r + k - 1, column x
      return (rv[k] && x >= 0 && x < im.W) ? __ldg(ir + (int64_t)(k - 1) * im.W + x) : 0ull;
    };
    uint64_t v0[3], v1[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      v0[k] = v_at(k, xs - 1);
      v1[k] = v_at(k, xs);
    }
    const int64_t px0 = (int64_t)r * im.W;
    for (int x0 = xs; x0 < xs + BW_SEG && x0 < im.W; x0 += PF) {
      uint2 dv[PF];
      uint64_t vn[3][PF];
#pragma unroll
      for (int j = 0; j < PF; ++j)
        dv[j] = x0 + j < im.W ? __ldg(reinterpret_cast<const uint2*>(dy1 + (px0 + x0 + j) * NC + 4 * cg))
                              : make_uint2(0u, 0u);
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int j = 0; j < PF; ++j) vn[k][j] = v_at(k, x0 + j + 1);
#pragma unroll
      for (int j = 0; j < PF; ++j) {
        const float g[4] = {__uint_as_float(dv[j].x << 16), __uint_as_float(dv[j].x & 0xFFFF0000u),
                            __uint_as_float(dv[j].y << 16), __uint_as_float(dv[j].y & 0xFFFF0000u)};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          bacc[c] += g[c];
          const uint64_t gg = fz_pk(g[c], g[c]);
#pragma unroll
          for (int d = 0; d < 9; ++d) {
            const int k = d / 3;
            fz_fma2(acc[d][c], d % 3 == 0 ? v0[k] : (d % 3 == 1 ? v1[k] : vn[k][j]), gg);
          }
        }
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          v0[k] = v1[k];
          v1[k] = vn[k][j];
        }
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int co = 4 * cg + c;
#pragma unroll
    for (int d = 0; d < 9; ++d) {
      const float2 v = fz_unpk(acc[d][c]);
      const float a = seg_sum(v.x), b = seg_sum(v.y);
      if (seg == 0) {
        sm[w][(co * 9 + d) * 2] = a;
        sm[w][(co * 9 + d) * 2 + 1] = b;
      }
    }
    const float bs = seg_sum(bacc[c]);
    if (seg == 0) sm[w][W1_N + co] = bs;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < W1_N + B1_N; i += BW_THREADS) {
    float t = 0.0f;
#pragma unroll
    for (int k = 0; k < BW_THREADS / 32; ++k) t += sm[k][i];
    part[(int64_t)blockIdx.x * (W1_N + B1_N) + i] = t;
  }
}

// Weight and bias gradients of a 32 -> 32 layer on the tensor cores:
//   dW[d][ci][co] = sum_p x[p + off(d)][ci] dy[p][co],  db[co] = sum_p dy[p][co].
// With q = p + off(d), a tap's row offset is a row of dy and its column offset
// a shift of x, so one MMA over 16 pixels of a row forms all nine taps at once:
// M = four column shifts of x times 32 channels (three used), N = three rows of
// dy times 32 channels, K = 16 pixels, 128 x 96 x 16.  Both operands are
// "MN-major": a pixel's 32 channels are one 64-byte row of the tensor copy's
// 64-byte swizzled layout, eight pixels along K make a 512-byte atom (SBO), and
// the stride between atoms along M is one pixel (LBO 64 bytes: the shifts) and
// along N one row of dy.  A job is WG_ROWS rows x 128 pixels: two tensor copies
// (x with its halo columns, dy with its halo rows), zero outside the image.
// Warps 5-8 issue the MMAs of one row of the job each (one thread's issue takes
// some 190 cycles whatever N, see k_net_fwd; four overlap) into accumulators of
// their own (128 x 96, TMEM columns 128 apart); every WG_FLUSH jobs warps 0-3
// add the accumulators to FP32 sums in registers, so no chain in the tensor
// core is longer than 8 WG_FLUSH MMAs.  Warps 0-3 also sum dy for the bias from
// the staged rows.  One CTA per SM; part[cta]: 9 x 32 x 32 sums ([d][ci][co]),
// then 32 bias sums.  Bounded by the two passes over HBM: 99 us per layer at 16
// x 512^2 (537 MB, 5.4 TB/s); the mma.sync form, staged by the threads, took
// 607 us and its separate bias pass 66 us.
// Barriers: full[s] (copies), empty[s] (4 commits + 4 sum warps), tfull (4
// commits), tempty (4 sum warps), drain[w] (warp 5 + w's last commit).  Waits
// are bounded as in k_conv32_tma.
constexpr int WG_ROWS = 4;
constexpr int WG_STAGES = 2;
constexpr int WG_FLUSH = 16;
constexpr int WG_X_BYTES = WG_ROWS * TC_PIX * NC * 2;        // 33,280
constexpr int WG_DY_BYTES = (WG_ROWS + 2) * TPX * NC * 2;    // 49,152
constexpr int WG_DY = (WG_X_BYTES + 64 + 1023) / 1024 * 1024;  // dy after x (whose fourth shift reads one row past it)
constexpr int WG_STAGE = WG_DY + WG_DY_BYTES;
constexpr int WG_BAR = WG_STAGES * WG_STAGE;
constexpr int WG_NBAR = 2 * WG_STAGES + 2 + 4;
constexpr int WG_SB = WG_BAR + 8 * WG_NBAR + 16;             // after the TMEM slot and the abort flag: bias sums
constexpr int WG_SMEM = WG_SB + 4 * NC * 4;
constexpr int WG_THREADS = 288;  // warps 0-3 sums, 4 copies, 5-8 MMAs
constexpr int WG_PART = WM_N + BM_N;
static_assert(WG_DY % 1024 == 0 && WG_STAGE % 1024 == 0 && WG_SMEM <= 227 * 1024, "wgrad shared memory");

// descriptor of an MN-major operand in the 64-byte swizzled layout: atoms of 32
// channels x 8 pixels, lbo bytes between atoms along M / N, 512 along K
__device__ __forceinline__ uint64_t tc_desc_mn64(uint32_t saddr, uint32_t lbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)(512 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}

__global__ void __launch_bounds__(WG_THREADS, 1) k_conv32_wgrad(const __grid_constant__ CUtensorMap xmap,
                                                                const __grid_constant__ CUtensorMap dmap, Image im,
                                                                float* __restrict__ part, int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t base = smem_addr(smem_raw), bars = base + WG_BAR;
  auto full = [&](int st) { return bars + 8 * st; };
  auto empty = [&](int st) { return bars + 8 * (WG_STAGES + st); };
  const uint32_t tfull = bars + 8 * (2 * WG_STAGES), tempty = tfull + 8;
  auto drain = [&](int w) { return tempty + 8 + 8 * w; };
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem_raw + WG_BAR + 8 * WG_NBAR);
  volatile int* abort = reinterpret_cast<volatile int*>(smem_raw + WG_BAR + 8 * WG_NBAR + 8);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int b = 0; b < WG_NBAR; ++b) {
      const uint32_t cnt = b < WG_STAGES ? 1u : (b < 2 * WG_STAGES ? 8u : (b < 2 * WG_STAGES + 2 ? 4u : 1u));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bars + 8 * b), "r"(cnt));
    }
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;");
  }
  if (warp == 5) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_addr(tslot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = *tslot;
  const int segs = (im.W + TPX - 1) / TPX, chunks = (im.R + WG_ROWS - 1) / WG_ROWS;
  const int64_t jobs = (int64_t)segs * chunks * (im.H / im.R);
  const int64_t njob = jobs > (int64_t)blockIdx.x ? (jobs - 1 - blockIdx.x) / gridDim.x + 1 : 0;
  if (warp == 4) {
    if (lane == 0) {
      int64_t k = 0;
      for (; k < njob; ++k) {
        const int st = (int)(k % WG_STAGES);
        const uint32_t u = (uint32_t)(k / WG_STAGES);
        if (u > 0 && !cp_wait(empty(st), (u - 1) & 1u, abort)) break;
        const int64_t job = blockIdx.x + k * gridDim.x;
        const int x0 = (int)(job % segs) * TPX, c = (int)((job / segs) % chunks);
        const int img = (int)(job / ((int64_t)segs * chunks)), r0 = c * WG_ROWS;
        const uint32_t sa = base + st * WG_STAGE;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(full(st)),
                     "r"((uint32_t)(WG_X_BYTES + WG_DY_BYTES))
                     : "memory");
        asm volatile(
            "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
            "%5}], [%6];" ::"r"(sa),
            "l"(reinterpret_cast<uint64_t>(&xmap)), "r"(0), "r"(x0 - 1), "r"(r0), "r"(img), "r"(full(st))
            : "memory");
        asm volatile(
            "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
            "%5}], [%6];" ::"r"(sa + WG_DY),
            "l"(reinterpret_cast<uint64_t>(&dmap)), "r"(0), "r"(x0), "r"(r0 - 1), "r"(img), "r"(full(st))
            : "memory");
      }
      // copies still in flight (an aborted run) land before the CTA ends
      for (int64_t q = k > WG_STAGES ? k - WG_STAGES : 0; q < k; ++q) {
        volatile int never = 0;
        cp_wait(full((int)(q % WG_STAGES)), (uint32_t)(q / WG_STAGES) & 1u, &never);
      }
    }
  } else if (warp >= 5) {
    if (lane == 0) {
      const int row = warp - 5;  // of every job
      // bf16 operands, f32 accumulators, both MN-major (bits 15, 16)
      constexpr uint32_t idesc = tc_idesc(128, 96) | (1u << 15) | (1u << 16);
      const uint32_t dst = tmem + (uint32_t)(128 * row);
      uint32_t nf = 0;  // flushes so far
      bool fresh = true;
      for (int64_t k = 0; k < njob; ++k) {
        const int st = (int)(k % WG_STAGES);
        if (!cp_wait(full(st), (uint32_t)(k / WG_STAGES) & 1u, abort)) break;
        if (fresh && nf > 0 && !cp_wait(tempty, (nf - 1) & 1u, abort)) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
        const uint32_t sx = base + st * WG_STAGE + row * TC_PIX * 64;
        const uint32_t sd = base + st * WG_STAGE + WG_DY + row * TPX * 64;
#pragma unroll 1
        for (int q = 0; q < TPX / 16; ++q) {
          const uint64_t da = tc_desc_mn64(sx + q * 1024, 64);
          const uint64_t db = tc_desc_mn64(sd + q * 1024, TPX * 64);
          asm volatile(
              "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
              "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(dst),
              "l"(da), "l"(db), "r"(idesc), "r"((uint32_t)(!fresh || q > 0)));
        }
        fresh = false;
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(empty(st))
                     : "memory");
        if ((k + 1) % WG_FLUSH == 0 || k + 1 == njob) {
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tfull)
                       : "memory");
          ++nf;
          fresh = true;
        }
      }
      // the last MMAs complete before TMEM is freed
      asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(drain(row))
                   : "memory");
      volatile int never = 0;
      cp_wait(drain(row), 0u, &never);
    }
  } else {
    // sums: thread t = TMEM lane t = x's shift t / 32, channel ci = t % 32, 96 columns (dy's row, co)
    float sum[96], bsum[8];
#pragma unroll
    for (int c = 0; c < 96; ++c) sum[c] = 0.0f;
#pragma unroll
    for (int c = 0; c < 8; ++c) bsum[c] = 0.0f;
    const int ch = tid & 3;  // the 8-channel chunk this thread sums for the bias
    uint32_t nf = 0;
    for (int64_t k = 0; k < njob; ++k) {
      const int st = (int)(k % WG_STAGES);
      bool ok = cp_wait(full(st), (uint32_t)(k / WG_STAGES) & 1u, abort);
      if (!__all_sync(0xffffffffu, ok)) {
        *abort = 1;
        break;
      }
      const unsigned char* sd = smem_raw + st * WG_STAGE + WG_DY + TPX * 64;  // without the halo row above
#pragma unroll 4
      for (int q = 0; q < WG_ROWS * TPX / 32; ++q) {
        const uint32_t off = (uint32_t)(32 * q + (tid >> 2)) * 64;
        const uint32_t sw = (off >> 7) & 3u;  // 64-byte swizzle: chunk index xor address bits 7-8
        const uint4 v = *reinterpret_cast<const uint4*>(sd + off + (((uint32_t)ch ^ sw) << 4));
        const uint32_t e[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          bsum[2 * c] += __uint_as_float(e[c] << 16);
          bsum[2 * c + 1] += __uint_as_float(e[c] & 0xFFFF0000u);
        }
      }
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(empty(st)) : "memory");
      if ((k + 1) % WG_FLUSH != 0 && k + 1 != njob) continue;
      ok = cp_wait(tfull, nf & 1u, abort);
      if (!__all_sync(0xffffffffu, ok)) {
        *abort = 1;
        break;
      }
      ++nf;
      asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int h = 0; h < 3; ++h) {
          uint32_t v[NC];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,"
              "%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
              : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]),
                "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]),
                "=r"(v[30]), "=r"(v[31])
              : "r"(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(128 * a + NC * h)));
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int c = 0; c < NC; ++c) sum[NC * h + c] += __uint_as_float(v[c]);
        }
      asm volatile("tcgen05.fence::before_thread_sync;");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tempty) : "memory");
    }
    float* out = part + (int64_t)blockIdx.x * WG_PART;
    if (warp < 3) {  // shift = tap column; dy's row n belongs to tap row 2 - n
#pragma unroll
      for (int h = 0; h < 3; ++h)
#pragma unroll
        for (int c = 0; c < NC; c += 4)
          *reinterpret_cast<float4*>(out + (((2 - h) * 3 + warp) * NC + lane) * NC + c) =
              make_float4(sum[NC * h + c], sum[NC * h + c + 1], sum[NC * h + c + 2], sum[NC * h + c + 3]);
    }
    // bias: lanes of equal chunk within the warp, then the four warps through shared memory
#pragma unroll
    for (int c = 0; c < 8; ++c)
      for (int o = 4; o < 32; o <<= 1) bsum[c] += __shfl_xor_sync(0xffffffffu, bsum[c], o);
    float* sb = reinterpret_cast<float*>(smem_raw + WG_SB);
    if (lane < 4)
#pragma unroll
      for (int c = 0; c < 8; ++c) sb[warp * NC + lane * 8 + c] = bsum[c];
    asm volatile("bar.sync 1, 128;" ::: "memory");
    if (tid < NC) out[WM_N + tid] = ((sb[tid] + sb[NC + tid]) + sb[2 * NC + tid]) + sb[3 * NC + tid];
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (tid == 0 && *abort) atomicExch(err, 1);
  if (warp == 5) {
    asm volatile("tcgen05.fence::after_thread_sync;");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  }
}

// out[place(i)] = sum over parts of part[c][i], i < n: 32 outputs per CTA, 32
// threads per output take every 32nd part, their sums added in a fixed order.
// wm >= 0: the first wm outputs are a middle layer's weights, (d 32 + ci) 32 +
// co -> (co 9 + d) 32 + ci.
constexpr int SP_THREADS = 1024;
__global__ void __launch_bounds__(SP_THREADS) k_sum_parts(const float* __restrict__ part, int nparts, int n, int wm,
                                                          float* __restrict__ out) {
  __shared__ float sm[32][33];
  const int o = threadIdx.x & 31, g = threadIdx.x >> 5, i = blockIdx.x * 32 + o;
  float s = 0.0f;
  if (i < n)
    for (int c = g; c < nparts; c += 32) s += part[(int64_t)c * n + i];
  sm[g][o] = s;
  __syncthreads();
  if (g != 0 || i >= n) return;
  s = 0.0f;
#pragma unroll
  for (int k = 0; k < 32; ++k) s += sm[k][o];
  const int co = i % NC, ci = (i / NC) % NC, d = i / (NC * NC);
  out[i < wm ? (co * 9 + d) * NC + ci : i] = s;
}

// ------------------------------------------------------------- weights
// B operands of k_conv32_tma, [tap][n][k]:
// forward: wf[l][d][n = co][k = ci] = W_l[co][d][ci]
// data gradient: wb[l][8 - d][n = ci][k = co] = W_l[co][d][ci]
__global__ void k_pack_weights(const float* __restrict__ P, bf16* __restrict__ wf, bf16* __restrict__ wb) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= NMID * WM_N) return;
  const int l = i / WM_N, rem = i % WM_N;
  const int co = rem / (9 * NC), d = (rem / NC) % 9, ci = rem % NC;
  const bf16 w = __float2bfloat16_rn(P[off_wm(l) + rem]);
  wf[(int64_t)l * WM_N + (d * NC + co) * NC + ci] = w;
  wb[(int64_t)l * WM_N + ((8 - d) * NC + ci) * NC + co] = w;
}

__global__ void k_adam(int n, float* __restrict__ P, const float* __restrict__ G, float* __restrict__ m,
                       float* __restrict__ v, float lr, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float g = G[i];
  const float mi = b1 * m[i] + (1.0f - b1) * g;
  const float vi = b2 * v[i] + (1.0f - b2) * g * g;
  m[i] = mi;
  v[i] = vi;
  P[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// ----------------------------------------------------------------- loss
// Gathers batch image k from the pair store: input (s_hat, m), node codes,
// diagonal and c.
__global__ void k_gather(Image im, const float* __restrict__ s_store, const double* __restrict__ c_store,
                         const int32_t* __restrict__ geo_of, const uint8_t* __restrict__ code_store,
                         const float* __restrict__ diag_store, const int32_t* __restrict__ pick,
                         float2* __restrict__ in, uint8_t* __restrict__ code, float* __restrict__ diag,
                         double* __restrict__ cimg) {
  const int64_t per = (int64_t)im.W * im.R;
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= im.npx()) return;
  const int k = (int)(p / per);
  const int64_t q = p - (int64_t)k * per;
  const int64_t s = pick[k];
  const int64_t g = geo_of[s];
  const uint8_t c = code_store[g * per + q];
  const bool cp = (c & CODE_CP) != 0;
  in[p] = make_float2(cp ? s_store[s * per + q] : 0.0f, cp ? 1.0f : 0.0f);
  code[p] = c;
  diag[p] = diag_store[g * per + q];
  if (q == 0) cimg[k] = c_store[s];
}

// Per image k (grid.y): per-CTA sums of o'A~o - 2 o's_hat (double);
// dout = (2 / batch) (A~ o - s_hat) / c_k at the CPs, 0 elsewhere.
__global__ void __launch_bounds__(256) k_loss(Image im, const uint8_t* __restrict__ code,
                                              const float* __restrict__ diag, const float2* __restrict__ in,
                                              const float* __restrict__ o, const double* __restrict__ cimg,
                                              float inv_batch, float* __restrict__ dout, double* __restrict__ part) {
  const int k = blockIdx.y;
  const int64_t per = (int64_t)im.W * im.R;
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double contrib = 0.0;
  if (q < per) {
    const int64_t p = (int64_t)k * per + q;
    const uint8_t c = code[p];
    float g = 0.0f;
    if (c & CODE_CP) {
      const int x = (int)(q % im.W), r = (int)(q / im.W);
      const float oc = o[p];
      float sum = 0.0f;
      if (!(c & 1) && x > 0) sum += o[p - 1];
      if (!(c & 2) && x + 1 < im.W) sum += o[p + 1];
      if (!(c & 4) && r > 0) sum += o[p - im.W];
      if (!(c & 8) && r + 1 < im.R) sum += o[p + im.W];
      const float Ao = diag[p] * oc - sum;
      const float sh = in[p].x;
      contrib = (double)oc * Ao - 2.0 * (double)oc * sh;
      g = 2.0f * inv_batch * (Ao - sh) / (float)cimg[k];
    }
    dout[p] = g;
  }
  __shared__ double sm[256];
  sm[threadIdx.x] = contrib;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sm[threadIdx.x] += sm[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[(int64_t)k * gridDim.x + blockIdx.x] = sm[0];
}

// loss[k] = (sum of part[k][*] + c_k) / c_k; loss[batch] = their mean
__global__ void k_loss_reduce(const double* __restrict__ part, int nblk, int batch, const double* __restrict__ cimg,
                              float* __restrict__ loss) {
  __shared__ double sl[256];
  double acc = 0.0;
  for (int k = threadIdx.x; k < batch; k += blockDim.x) {
    double s = 0.0;
    for (int b = 0; b < nblk; ++b) s += part[(int64_t)k * nblk + b];
    const double L = (s + cimg[k]) / cimg[k];
    loss[k] = (float)L;
    acc += L;
  }
  sl[threadIdx.x] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int i = 0; i < (int)blockDim.x; ++i) t += sl[i];
    loss[batch] = (float)(t / batch);
  }
}

// ------------------------------------------------ full-grid operator helpers
// (sigma I + A) x at the CP node p; only CP neighbours are read (mask bits of the code)
struct GridOp {
  int dim;
  int64_t st[3];
  double inv_h2, sigma;
};

template <class T>
__device__ __forceinline__ double op_at(const GridOp& G, const uint8_t c, const double* diag, const T* x, int64_t p) {
  double sum = 0.0;
  for (int s = 0; s < 2 * G.dim; ++s)
    if (!(c & (1u << s))) sum += (double)x[p + ((s & 1) ? G.st[s >> 1] : -G.st[s >> 1])];
  return (G.sigma + diag[p] * G.inv_h2) * (double)x[p] - sum * G.inv_h2;
}

// per-CTA sums of a and b into out2[0..1] (blockDim.x = 256)
__device__ __forceinline__ void block_sum2(double a, double b, double* out2) {
  __shared__ double s0[256], s1[256];
  s0[threadIdx.x] = a;
  s1[threadIdx.x] = b;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      s0[threadIdx.x] += s0[threadIdx.x + w];
      s1[threadIdx.x] += s1[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out2[0] = s0[0];
    out2[1] = s1[0];
  }
}

// r = b - (sigma I + A) x at the CPs, 0 elsewhere
__global__ void __launch_bounds__(256) k_pr_resid(GridOp G, int64_t nn, const uint8_t* __restrict__ code,
                                                  const double* __restrict__ diag, const double* __restrict__ b,
                                                  const double* __restrict__ x, double* __restrict__ r) {
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nn; p += (int64_t)gridDim.x * blockDim.x) {
    const uint8_t c = code[p];
    r[p] = (c & CODE_CP) ? b[p] - op_at(G, c, diag, x, p) : 0.0;
  }
}

// x += z; e = x* - x at the CPs (e = 0 elsewhere)
__global__ void k_pr_update(int64_t nn, const uint8_t* __restrict__ code, const double* __restrict__ z,
                            const double* __restrict__ xs, double* __restrict__ x, double* __restrict__ e) {
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nn; p += (int64_t)gridDim.x * blockDim.x) {
    if (code[p] & CODE_CP) {
      const double xv = x[p] + z[p];
      x[p] = xv;
      e[p] = xs[p] - xv;
    } else {
      e[p] = 0.0;
    }
  }
}

// t = h^2 (sigma I + A) e at the CPs; per-CTA partials (sum t^2, sum e t)
__global__ void __launch_bounds__(256) k_pr_unit(GridOp G, double h2, int64_t nn, const uint8_t* __restrict__ code,
                                                 const double* __restrict__ diag, const double* __restrict__ e,
                                                 double* __restrict__ t, double* __restrict__ part) {
  double a = 0.0, b = 0.0;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nn; p += (int64_t)gridDim.x * blockDim.x) {
    const uint8_t c = code[p];
    double tv = 0.0;
    if (c & CODE_CP) {
      tv = h2 * op_at(G, c, diag, e, p);
      a += tv * tv;
      b += e[p] * tv;
    }
    t[p] = tv;
  }
  block_sum2(a, b, part + 2 * blockIdx.x);
}

// rho = rms(t) over the CPs; scal = (1 / rho, c = sum e t / rho^2), c also into c_out
__global__ void k_pr_norm(const double* __restrict__ part, int nblk, double ncp, double* __restrict__ scal,
                          double* __restrict__ c_out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double a = 0.0, b = 0.0;
  for (int i = 0; i < nblk; ++i) {
    a += part[2 * i];
    b += part[2 * i + 1];
  }
  const double rho = sqrt(a / ncp);
  const double inv = rho > 0.0 ? 1.0 / rho : 0.0;
  scal[0] = inv;
  scal[1] = b * inv * inv;
  *c_out = b * inv * inv;
}

__global__ void k_pr_write(int64_t nn, const double* __restrict__ t, const double* __restrict__ e,
                           const double* __restrict__ scal, float* __restrict__ s_out, double* __restrict__ e_out) {
  const double inv = scal[0];
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nn; p += (int64_t)gridDim.x * blockDim.x) {
    s_out[p] = (float)(t[p] * inv);
    if (e_out) e_out[p] = e[p] * inv;
  }
}

// ------------------------------------------------------ stage in the PCG
// s = r - (sigma I + A) z at the CPs; per-CTA sums of s^2
__global__ void __launch_bounds__(256) k_st_resid(GridOp G, int64_t nn, const uint8_t* __restrict__ code,
                                                  const double* __restrict__ diag, const double* __restrict__ r,
                                                  const double* __restrict__ z, double* __restrict__ s,
                                                  double* __restrict__ part) {
  double a = 0.0;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nn; p += (int64_t)gridDim.x * blockDim.x) {
    const uint8_t c = code[p];
    double v = 0.0;
    if (c & CODE_CP) {
      v = r[p] - op_at(G, c, diag, z, p);
      a += v * v;
    }
    s[p] = v;
  }
  block_sum2(a, 0.0, part + 2 * blockIdx.x);
}

// scal = (1 / rms(s), or 0 when s = 0; h^2 rms(s))
__global__ void k_st_norm(const double* __restrict__ part, int nblk, double ncp, double h2,
                          double* __restrict__ scal) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double a = 0.0;
  for (int i = 0; i < nblk; ++i) a += part[2 * i];
  const double rms = sqrt(a / ncp);
  scal[0] = rms > 0.0 ? 1.0 / rms : 0.0;
  scal[1] = h2 * rms;
}

__global__ void k_st_input(int64_t nn, const uint8_t* __restrict__ code, const double* __restrict__ s,
                           const double* __restrict__ scal, float2* __restrict__ in) {
  const double inv = scal[0];
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nn; p += (int64_t)gridDim.x * blockDim.x) {
    const bool cp = (code[p] & CODE_CP) != 0;
    in[p] = make_float2(cp ? (float)(s[p] * inv) : 0.0f, cp ? 1.0f : 0.0f);
  }
}

// energy-optimal step: per-CTA sums of o's_hat and o'A~o, A~ = h^2 (sigma I + A)
__global__ void __launch_bounds__(256) k_st_energy(GridOp G, double h2, int64_t nn, const uint8_t* __restrict__ code,
                                                   const double* __restrict__ diag, const float2* __restrict__ in,
                                                   const float* __restrict__ o, double* __restrict__ part) {
  double a = 0.0, b = 0.0;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nn; p += (int64_t)gridDim.x * blockDim.x) {
    const uint8_t c = code[p];
    if (c & CODE_CP) {
      const double ov = (double)o[p];
      a += ov * (double)in[p].x;
      b += ov * h2 * op_at(G, c, diag, o, p);
    }
  }
  block_sum2(a, b, part + 2 * blockIdx.x);
}

// scal[1] *= omega = (o's_hat) / (o'A~o), 0 when o'A~o <= 0
__global__ void k_st_omega(const double* __restrict__ part, int nblk, double* __restrict__ scal) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double a = 0.0, b = 0.0;
  for (int i = 0; i < nblk; ++i) {
    a += part[2 * i];
    b += part[2 * i + 1];
  }
  scal[1] *= b > 0.0 ? a / b : 0.0;
}

__global__ void k_st_correct(int64_t nn, const uint8_t* __restrict__ code, const float* __restrict__ o,
                             const double* __restrict__ scal, double* __restrict__ z) {
  const double a = scal[1];
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < nn; p += (int64_t)gridDim.x * blockDim.x)
    if (code[p] & CODE_CP) z[p] += a * (double)o[p];
}

// ---------------------------------------------------------------- host
static uint64_t next_state() {
  static std::atomic<uint64_t> n{0};
  return ++n;
}

struct NN {
  // of the buffers and the route that a captured stage holds (nn_stage_state):
  // renewed when one is reallocated or the forward path changes
  uint64_t state = next_state();
  float* P = nullptr;  // FP32 master parameters
  float* G = nullptr;  // gradient
  float* m = nullptr;  // Adam moments
  float* v = nullptr;
  int* err = nullptr;  // set by a convolution whose tensor-core wait gave up
  // optional CUDA-event timing of the 32 -> 32 convolution launches of forward()
  bool prof = false;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> prof_ev;
  int prof_n = 0;
  bf16* wf = nullptr;  // packed forward weights of the middle layers
  bf16* wb = nullptr;  // packed data-gradient weights
  int64_t steps = 0;
  cudaStream_t home = 0;
  bool fused = true;  // nn_forward and the PCG stage: k_net_fwd (else the layer-by-layer launches)
  // activations (grown to the largest stack seen)
  int64_t cap_px = 0;
  bf16* act[6] = {};  // act[1..5]: outputs of layers 1..5
  bf16* gA = nullptr;
  bf16* gB = nullptr;
  float* out = nullptr;
  float* dout = nullptr;
  float2* in = nullptr;     // gathered / staged input
  uint8_t* code = nullptr;  // gathered batch geometry
  float* diag = nullptr;
  // reductions
  float* part = nullptr;
  int64_t cap_part = 0;
  double* lpart = nullptr;
  int64_t cap_lpart = 0;
  double* cimg = nullptr;
  float* loss = nullptr;
  int cap_batch = 0;
  // stage in the PCG
  int64_t cap_nodes = 0;
  double* s64 = nullptr;
  double* spart = nullptr;
  double* scal = nullptr;
  int snblk = 0;
};

static void set_attrs() {
  static bool done = false;
  if (done) return;
  EB_CUDA(cudaFuncSetAttribute(k_conv32_tma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CP_SMEM));
  EB_CUDA(cudaFuncSetAttribute(k_conv32_wgrad, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)WG_SMEM));
  EB_CUDA(cudaFuncSetAttribute(k_net_fwd, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FZ_SMEM));
  done = true;
}

// Tensor map of a BF16 NHWC activation stack: dimensions (32 channels, pixel,
// row in image, image), strides 64 B, W * 64 B, R * W * 64 B; box (32, px,
// rows, 1) written in the 64-byte swizzled layout;
// out-of-range elements read as zero.
static CUtensorMap conv_map(const bf16* x, const Image& im, int px, int rows) {
  EB_REQUIRE(((uintptr_t)x & 15) == 0, EB_ERR_INVALID, "conv: activations not 16-byte aligned");
  EB_REQUIRE(im.R > 0 && im.H % im.R == 0, EB_ERR_INVALID, "conv: rows are not whole images");
  CUtensorMap m;
  const cuuint64_t dims[4] = {(cuuint64_t)NC, (cuuint64_t)im.W, (cuuint64_t)im.R, (cuuint64_t)(im.H / im.R)};
  const cuuint64_t strides[3] = {(cuuint64_t)NC * 2, (cuuint64_t)im.W * NC * 2, (cuuint64_t)im.R * im.W * NC * 2};
  const cuuint32_t box[4] = {(cuuint32_t)NC, (cuuint32_t)px, (cuuint32_t)rows, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUresult r = tensor_map_encoder()(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<bf16*>(x), dims,
                                          strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                                          CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  EB_REQUIRE(r == CUDA_SUCCESS, EB_ERR_CUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
  return m;
}

// y = conv(x; wk) (+ bias, ReLU, mask) through k_conv32_tma: jobs of four rows,
// or of two or one where four would not give every SM two of them
static void conv32(const Image& im, const bf16* x, const bf16* wk, const float* bias, bf16* y, int relu,
                   const bf16* mask_ref, int* err, cudaStream_t s) {
  auto jobs = [&](int rb) { return (int64_t)((im.W + TPX - 1) / TPX) * ((im.R + rb - 1) / rb) * (im.H / im.R); };
  const int rb = jobs(4) >= 2 * num_sms() ? 4 : (jobs(2) >= 2 * num_sms() ? 2 : 1);
  const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(jobs(rb), num_sms()));
  k_conv32_tma<<<grid, CP_THREADS, CP_SMEM, s>>>(conv_map(x, im, TC_PIX, rb + 2), im, rb, wk, bias, y, relu, mask_ref,
                                                 err);
}

static void ensure_act(NN& N, int64_t px, cudaStream_t s) {
  if (px <= N.cap_px) return;
  N.state = next_state();
  for (int l = 1; l <= 5; ++l) dfree(N.act[l], s);
  dfree(N.gA, s); dfree(N.gB, s); dfree(N.out, s); dfree(N.dout, s); dfree(N.in, s); dfree(N.code, s);
  dfree(N.diag, s);
  N.cap_px = 0;
  for (int l = 1; l <= 5; ++l) N.act[l] = dalloc<bf16>((size_t)px * NC, s, false);
  N.gA = dalloc<bf16>((size_t)px * NC, s, false);
  N.gB = dalloc<bf16>((size_t)px * NC, s, false);
  N.out = dalloc<float>(px, s, false);
  N.dout = dalloc<float>(px, s, false);
  N.in = dalloc<float2>(px, s, false);
  N.code = dalloc<uint8_t>(px, s, false);
  N.diag = dalloc<float>(px, s, false);
  N.cap_px = px;
}

static float* ensure_part(NN& N, int64_t n, cudaStream_t s) {
  if (n > N.cap_part) {
    dfree(N.part, s);
    N.cap_part = 0;
    N.part = dalloc<float>(n, s, false);
    N.cap_part = n;
  }
  return N.part;
}

static int64_t npx_of(const Image& im) { return (int64_t)im.W * im.H; }

static void pack(NN& N, cudaStream_t s, int64_t& nl) {
  k_pack_weights<<<blocks_for(NMID * WM_N, 256), 256, 0, s>>>(N.P, N.wf, N.wb);
  ++nl;
}

// out = N(in) over the stack (out NULL: only the activations that backward
// reads, layer 6 is not needed).  prof (may be NULL): a solver timing the
// 32 -> 32 convolution launches.
static void forward(NN& N, const Image& im, const float2* in, float* out, cudaStream_t s, int64_t& nl,
                    Solver* prof = nullptr) {
  const int64_t npx = npx_of(im);
  // layer 1: two pixels of two rows per thread
  const int64_t nquads = (int64_t)((im.W + 1) / 2) * ((im.R + 1) / 2) * (im.H / im.R);
  k_l1_fwd<<<blocks_for(nquads, 128), 128, 0, s>>>(im, in, N.P, N.act[1]);
  for (int l = 0; l < NMID; ++l) {
    const bool own = N.prof && !prof;  // events of the handle (not inside a solver's graph)
    if (own) {
      if (N.prof_n >= (int)N.prof_ev.size()) {
        cudaEvent_t a, b;
        EB_CUDA(cudaEventCreate(&a));
        EB_CUDA(cudaEventCreate(&b));
        N.prof_ev.push_back({a, b});
      }
      EB_CUDA(cudaEventRecord(N.prof_ev[N.prof_n].first, s));
    }
    if (prof) prof->prof_mark(s, true, PROF_CONV);
    conv32(im, N.act[l + 1], N.wf + (int64_t)l * WM_N, N.P + off_wm(l) + WM_N, N.act[l + 2], 1, nullptr, N.err, s);
    if (prof) prof->prof_mark(s, false, PROF_CONV);
    if (own) EB_CUDA(cudaEventRecord(N.prof_ev[N.prof_n++].second, s));
  }
  nl += 1 + NMID;
  if (out) {
    k_l6_fwd<<<blocks_for(npx, 128), 128, 0, s>>>(im, N.act[5], N.P, in, out);
    nl += 1;
  }
  EB_CUDA(cudaGetLastError());
}

// The work units of k_net_fwd: strips of FZ_OUT columns x runs of rows of
// one image.  A run of n rows takes n + 15 steps; the run length minimises
// (waves of units over the SMs) x (steps per unit).
static FzArgs fz_plan(const Image& im) {
  FzArgs a{};
  a.im = im;
  a.strips = (im.W + FZ_OUT - 1) / FZ_OUT;
  const int64_t nimg = im.H / im.R;
  const int64_t nsm = num_sms();
  int64_t best = -1;
  for (int sg = 1; sg <= im.R; ++sg) {
    const int rows = (im.R + sg - 1) / sg;
    const int segs = (im.R + rows - 1) / rows;
    const int64_t units = (int64_t)a.strips * nimg * segs;
    const int64_t cost = ((units + nsm - 1) / nsm) * (rows + 15);
    if (best < 0 || cost < best) {
      best = cost;
      a.segs = segs;
      a.seg_rows = rows;
      a.units = units;
    }
    if (units > 4 * nsm) break;
  }
  return a;
}

// out = N(in) in one launch of k_net_fwd
static void forward_fused(NN& N, const Image& im, const float2* in, float* out, cudaStream_t s, int64_t& nl,
                          Solver* prof = nullptr) {
  EB_REQUIRE(im.R > 0 && im.H % im.R == 0, EB_ERR_INVALID, "forward: rows are not whole images");
  FzArgs a = fz_plan(im);
  a.in = in;
  a.out = out;
  a.P = N.P;
  a.wf = N.wf;
  a.err = N.err;
  const bool own = N.prof && !prof;
  if (own) {
    if (N.prof_n >= (int)N.prof_ev.size()) {
      cudaEvent_t e0, e1;
      EB_CUDA(cudaEventCreate(&e0));
      EB_CUDA(cudaEventCreate(&e1));
      N.prof_ev.push_back({e0, e1});
    }
    EB_CUDA(cudaEventRecord(N.prof_ev[N.prof_n].first, s));
  }
  if (prof) prof->prof_mark(s, true, PROF_CONV);
  const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(a.units, num_sms()));
  k_net_fwd<<<grid, FZ_THREADS, FZ_SMEM, s>>>(a);
  if (prof) prof->prof_mark(s, false, PROF_CONV);
  if (own) EB_CUDA(cudaEventRecord(N.prof_ev[N.prof_n++].second, s));
  nl += 1;
  EB_CUDA(cudaGetLastError());
}

// the inference forward: fused unless the handle asks for the layer-by-layer path
static void forward_infer(NN& N, const Image& im, const float2* in, float* out, cudaStream_t s, int64_t& nl,
                          Solver* prof = nullptr) {
  if (N.fused) forward_fused(N, im, in, out, s, nl, prof);
  else forward(N, im, in, out, s, nl, prof);
}

static void sum_parts(const float* part, int nparts, int n, int wm, float* out, cudaStream_t s) {
  k_sum_parts<<<blocks_for(n, 32), SP_THREADS, 0, s>>>(part, nparts, n, wm, out);
}

// gradient of sum(dout * out) into N.G (the activations of a forward on the
// same input are in N.act); N.out is overwritten
static void backward(NN& N, const Image& im, const float2* in, const float* dout, cudaStream_t s, int64_t& nl) {
  const int64_t npx = npx_of(im);
  const int64_t tasks = (int64_t)((im.W + BW_RUN - 1) / BW_RUN) * im.H, per = BW_THREADS / 32;
  const int nb = (int)std::max<int64_t>(1, std::min<int64_t>((tasks + per - 1) / per, (int64_t)num_sms() * BW_CTAS));
  const int64_t jobs = (int64_t)((im.W + TPX - 1) / TPX) * ((im.R + WG_ROWS - 1) / WG_ROWS) * (im.H / im.R);
  const int gw = (int)std::max<int64_t>(1, std::min<int64_t>(jobs, num_sms()));
  float* part = ensure_part(N, std::max<int64_t>((int64_t)nb * (W1_N + B1_N), (int64_t)gw * WG_PART), s);
  k_l6_gate<<<blocks_for(npx, 256), 256, 0, s>>>(npx, dout, in, N.out);
  k_l6_back<<<nb, BW_THREADS, 0, s>>>(im, N.out, N.act[5], N.P, N.gA, part);
  sum_parts(part, nb, W6_N + B6_N, 0, N.G + OFF_W6, s);
  bf16* cur = N.gA;
  bf16* nxt = N.gB;
  for (int l = NMID - 1; l >= 0; --l) {
    k_conv32_wgrad<<<gw, WG_THREADS, WG_SMEM, s>>>(conv_map(N.act[l + 1], im, TC_PIX, WG_ROWS),
                                                   conv_map(cur, im, TPX, WG_ROWS + 2), im, part, N.err);
    sum_parts(part, gw, WG_PART, WM_N, N.G + off_wm(l), s);
    conv32(im, cur, N.wb + (int64_t)l * WM_N, nullptr, nxt, 0, N.act[l + 1], N.err, s);
    std::swap(cur, nxt);
  }
  k_l1_wgrad<<<nb, BW_THREADS, 0, s>>>(im, cur, in, part);
  sum_parts(part, nb, W1_N + B1_N, 0, N.G + OFF_W1, s);
  nl += 5 + 3 * NMID;
  EB_CUDA(cudaGetLastError());
}

static GridOp grid_op(const EBHandle& eb, double sigma) {
  GridOp G;
  G.dim = eb.g.dim;
  G.st[0] = 1;
  G.st[1] = eb.g.n0;
  G.st[2] = (int64_t)eb.g.n0 * eb.g.n1;
  G.inv_h2 = 1.0 / (eb.g.h * eb.g.h);
  G.sigma = sigma;
  return G;
}

static unsigned grid_blocks(int64_t nn) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((nn + 255) / 256, (int64_t)num_sms() * 8));
}

}  // namespace ebk

struct nn_handle {
  ebk::NN n;
};

namespace ebk {

uint64_t nn_stage_state(const nn_handle* h) { return h ? h->n.state : 0; }

void nn_stage_prepare(nn_handle* h, const EBHandle& eb, cudaStream_t s) {
  NN& N = h->n;
  EB_REQUIRE(eb.g.dim == 2, EB_ERR_INVALID, "learned stage: 2D grids only");
  const int64_t nn = eb.g.num_nodes;
  ensure_act(N, nn, s);
  if (nn > N.cap_nodes) {
    N.state = next_state();
    dfree(N.s64, s);
    dfree(N.spart, s);
    N.cap_nodes = 0;
    N.snblk = (int)grid_blocks(nn);
    N.s64 = dalloc<double>(nn, s, false);
    N.spart = dalloc<double>(2 * (int64_t)N.snblk, s, false);
    N.cap_nodes = nn;
  }
  if (!N.scal) N.scal = dalloc<double>(2, s);
}

// z = z1 + omega h^2 rms(s) N(s / rms(s), m) with s = r - (sigma I + A) z1 and z1 = z on
// entry; omega = 1 (EB_NN_PLAIN) or the energy-optimal step (EB_NN_ENERGY)
void nn_stage_apply(nn_handle* h, const EBHandle& eb, double shift, int mode, const double* r, double* z,
                    int64_t& nl, Solver* prof, cudaStream_t s) {
  NN& N = h->n;
  const int64_t nn = eb.g.num_nodes;
  const unsigned nb = grid_blocks(nn);
  EB_REQUIRE(nn <= N.cap_nodes && (int)nb <= N.snblk && N.scal, EB_ERR_INVALID, "learned stage: not prepared");
  const GridOp G = grid_op(eb, shift);
  k_st_resid<<<nb, 256, 0, s>>>(G, nn, eb.code, eb.diag, r, z, N.s64, N.spart);
  k_st_norm<<<1, 32, 0, s>>>(N.spart, (int)nb, (double)eb.num_cp, eb.g.h * eb.g.h, N.scal);
  k_st_input<<<nb, 256, 0, s>>>(nn, eb.code, N.s64, N.scal, N.in);
  const Image im{eb.g.n0, eb.g.n1, eb.g.n1};
  forward_infer(N, im, N.in, N.out, s, nl, prof);
  if (mode == EB_NN_ENERGY) {
    k_st_energy<<<nb, 256, 0, s>>>(G, eb.g.h * eb.g.h, nn, eb.code, eb.diag, N.in, N.out, N.spart);
    k_st_omega<<<1, 32, 0, s>>>(N.spart, (int)nb, N.scal);
    nl += 2;
  }
  k_st_correct<<<nb, 256, 0, s>>>(nn, eb.code, N.out, N.scal, z);
  nl += 4;
}

}  // namespace ebk

using namespace ebk;

static int check_shape(int width, int height, int images) {
  if (width < 1 || height < 1 || images < 1 || (int64_t)height * images >= ((int64_t)1 << 30)) {
    set_error("nn: width, height and images must be >= 1 and height x images < 2^30");
    return EB_ERR_INVALID;
  }
  return EB_OK;
}

extern "C" {

int nn_create(nn_handle** out, cudaStream_t stream) {
  if (!out) {
    set_error("nn_create: NULL argument");
    return EB_ERR_INVALID;
  }
  *out = nullptr;
  nn_handle* h = new (std::nothrow) nn_handle();
  if (!h) {
    set_error("nn_create: host allocation failed");
    return EB_ERR_OOM;
  }
  h->n.home = stream;
  int st = guarded([&] {
    NN& N = h->n;
    set_attrs();
    N.P = dalloc<float>(NPARAM, stream);
    N.G = dalloc<float>(NPARAM, stream);
    N.m = dalloc<float>(NPARAM, stream);
    N.v = dalloc<float>(NPARAM, stream);
    N.wf = dalloc<bf16>(NMID * WM_N, stream);
    N.wb = dalloc<bf16>(NMID * WM_N, stream);
    N.err = dalloc<int>(1, stream);
    EB_CUDA(cudaStreamSynchronize(stream));
  });
  if (st != EB_OK) {
    nn_destroy(h);
    return st;
  }
  *out = h;
  return EB_OK;
}

void nn_destroy(nn_handle* h) {
  if (!h) return;
  NN& N = h->n;
  cudaStream_t s = N.home;
  dfree(N.P, s); dfree(N.G, s); dfree(N.m, s); dfree(N.v, s); dfree(N.wf, s); dfree(N.wb, s); dfree(N.err, s);
  for (int l = 1; l <= 5; ++l) dfree(N.act[l], s);
  dfree(N.gA, s); dfree(N.gB, s); dfree(N.out, s); dfree(N.dout, s); dfree(N.in, s); dfree(N.code, s);
  dfree(N.diag, s); dfree(N.part, s); dfree(N.lpart, s); dfree(N.cimg, s); dfree(N.loss, s);
  dfree(N.s64, s); dfree(N.spart, s); dfree(N.scal, s);
  cudaStreamSynchronize(s);
  for (auto& e : N.prof_ev) {
    cudaEventDestroy(e.first);
    cudaEventDestroy(e.second);
  }
  delete h;
}

int nn_num_params(void) { return NPARAM; }

int nn_set_profile(nn_handle* h, int on) {
  if (!h) {
    set_error("nn_set_profile: NULL handle");
    return EB_ERR_INVALID;
  }
  h->n.prof = on != 0;
  h->n.prof_n = 0;
  return EB_OK;
}

int nn_set_fused(nn_handle* h, int on) {
  if (!h) {
    set_error("nn_set_fused: NULL handle");
    return EB_ERR_INVALID;
  }
  if (h->n.fused != (on != 0)) h->n.state = next_state();
  h->n.fused = on != 0;
  return EB_OK;
}

int nn_profile(nn_handle* h, double* ms, int* launches, cudaStream_t stream) {
  if (!h || !ms || !launches) {
    set_error("nn_profile: NULL argument");
    return EB_ERR_INVALID;
  }
  return guarded([&] {
    NN& N = h->n;
    EB_CUDA(cudaStreamSynchronize(stream));
    double t = 0.0;
    for (int i = 0; i < N.prof_n; ++i) {
      float m = 0.0f;
      EB_CUDA(cudaEventElapsedTime(&m, N.prof_ev[i].first, N.prof_ev[i].second));
      t += m;
    }
    *ms = t;
    *launches = N.prof_n;
    N.prof_n = 0;
  });
}

int nn_status(nn_handle* h, cudaStream_t stream) {
  if (!h) {
    set_error("nn_status: NULL handle");
    return EB_ERR_INVALID;
  }
  int flag = 0;
  int st = guarded([&] {
    EB_CUDA(cudaMemcpyAsync(&flag, h->n.err, sizeof(int), cudaMemcpyDeviceToHost, stream));
    EB_CUDA(cudaMemsetAsync(h->n.err, 0, sizeof(int), stream));
    EB_CUDA(cudaStreamSynchronize(stream));
  });
  if (st != EB_OK) return st;
  if (flag) {
    set_error("nn: a tensor-core wait in a convolution gave up (results of that call are invalid)");
    return EB_ERR_TIMEOUT;
  }
  return EB_OK;
}

int nn_set_params(nn_handle* h, const float* params_host, cudaStream_t stream) {
  if (!h || !params_host) {
    set_error("nn_set_params: NULL argument");
    return EB_ERR_INVALID;
  }
  return guarded([&] {
    NN& N = h->n;
    int64_t nl = 0;
    EB_CUDA(cudaMemcpyAsync(N.P, params_host, sizeof(float) * NPARAM, cudaMemcpyHostToDevice, stream));
    EB_CUDA(cudaMemsetAsync(N.m, 0, sizeof(float) * NPARAM, stream));
    EB_CUDA(cudaMemsetAsync(N.v, 0, sizeof(float) * NPARAM, stream));
    pack(N, stream, nl);
    N.steps = 0;
    EB_CUDA(cudaStreamSynchronize(stream));
  });
}

int nn_get_params(const nn_handle* h, float* params_host, float* grad_host, cudaStream_t stream) {
  if (!h) {
    set_error("nn_get_params: NULL handle");
    return EB_ERR_INVALID;
  }
  if (int ns = nn_status(const_cast<nn_handle*>(h), stream)) return ns;
  return guarded([&] {
    const NN& N = h->n;
    if (params_host)
      EB_CUDA(cudaMemcpyAsync(params_host, N.P, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, stream));
    if (grad_host) EB_CUDA(cudaMemcpyAsync(grad_host, N.G, sizeof(float) * NPARAM, cudaMemcpyDeviceToHost, stream));
    EB_CUDA(cudaStreamSynchronize(stream));
  });
}

int nn_forward(nn_handle* h, int width, int height, int images, const float* in_dev, float* out_dev,
               cudaStream_t stream) {
  if (!h || !in_dev || !out_dev) {
    set_error("nn_forward: NULL argument");
    return EB_ERR_INVALID;
  }
  if (int st = check_shape(width, height, images)) return st;
  if (reinterpret_cast<uintptr_t>(in_dev) % 8) {
    set_error("nn_forward: in must be 8-byte aligned");
    return EB_ERR_INVALID;
  }
  return guarded([&] {
    NN& N = h->n;
    const Image im{width, height * images, height};
    if (!N.fused) ensure_act(N, npx_of(im), stream);
    int64_t nl = 0;
    forward_infer(N, im, reinterpret_cast<const float2*>(in_dev), out_dev, stream, nl);
  });
}

int nn_backward(nn_handle* h, int width, int height, int images, const float* in_dev, const float* dout_dev,
                cudaStream_t stream) {
  if (!h || !in_dev || !dout_dev) {
    set_error("nn_backward: NULL argument");
    return EB_ERR_INVALID;
  }
  if (int st = check_shape(width, height, images)) return st;
  if (reinterpret_cast<uintptr_t>(in_dev) % 8) {
    set_error("nn_backward: in must be 8-byte aligned");
    return EB_ERR_INVALID;
  }
  return guarded([&] {
    NN& N = h->n;
    const Image im{width, height * images, height};
    ensure_act(N, npx_of(im), stream);
    int64_t nl = 0;
    const float2* in = reinterpret_cast<const float2*>(in_dev);
    forward(N, im, in, nullptr, stream, nl);
    backward(N, im, in, dout_dev, stream, nl);
  });
}

int nn_geometry(const eb_handle* eb, uint8_t* code_dev, float* diag_dev, cudaStream_t stream) {
  if (!eb || !code_dev || !diag_dev) {
    set_error("nn_geometry: NULL argument");
    return EB_ERR_INVALID;
  }
  return guarded([&] {
    const EBHandle& E = eb->h;
    EB_REQUIRE(!E.has_beta(), EB_ERR_NOT_IMPLEMENTED, "nn_geometry: the learned stage needs beta = 1");
    EB_CUDA(cudaMemcpyAsync(code_dev, E.code, (size_t)E.g.num_nodes, cudaMemcpyDeviceToDevice, stream));
    EB_CUDA(cudaMemcpyAsync(diag_dev, E.diag32, sizeof(float) * E.g.num_nodes, cudaMemcpyDeviceToDevice, stream));
  });
}

int nn_pairs(const amg_handle* amg, const double* b_dev, const double* xstar_dev, int count, float* s_hat_dev,
             double* c_dev, double* e_hat_dev, cudaStream_t stream) {
  if (!amg || !b_dev || !xstar_dev || !s_hat_dev || !c_dev || count < 0) {
    set_error("nn_pairs: NULL argument or count < 0");
    return EB_ERR_INVALID;
  }
  return guarded([&] {
    Solver& S = const_cast<Solver&>(amg->s);
    EB_REQUIRE(S.H != nullptr, EB_ERR_INVALID, "nn_pairs: handle has no hierarchy");
    EB_REQUIRE(!S.eb->has_beta(), EB_ERR_NOT_IMPLEMENTED, "nn_pairs: the learned stage needs beta = 1");
    const EBHandle& eb = *S.eb;
    const int64_t nn = eb.g.num_nodes;
    const unsigned nb = grid_blocks(nn);
    const GridOp G = grid_op(eb, S.shift);
    double *x = nullptr, *r = nullptr, *z = nullptr, *e = nullptr, *t = nullptr, *part = nullptr, *scal = nullptr;
    auto release = [&] {
      dfree(x, stream); dfree(r, stream); dfree(z, stream); dfree(e, stream); dfree(t, stream);
      dfree(part, stream); dfree(scal, stream);
    };
    try {
      x = dalloc<double>(nn, stream);
      r = dalloc<double>(nn, stream);
      z = dalloc<double>(nn, stream);
      e = dalloc<double>(nn, stream);
      t = dalloc<double>(nn, stream);
      part = dalloc<double>(2 * (int64_t)nb, stream);
      scal = dalloc<double>(2, stream);
      for (int k = 0; k < count; ++k) {
        k_pr_resid<<<nb, 256, 0, stream>>>(G, nn, eb.code, eb.diag, b_dev, x, r);
        amg_vcycle_grid(S, r, z, stream);
        k_pr_update<<<nb, 256, 0, stream>>>(nn, eb.code, z, xstar_dev, x, e);
        k_pr_unit<<<nb, 256, 0, stream>>>(G, eb.g.h * eb.g.h, nn, eb.code, eb.diag, e, t, part);
        k_pr_norm<<<1, 32, 0, stream>>>(part, (int)nb, (double)eb.num_cp, scal, c_dev + k);
        k_pr_write<<<nb, 256, 0, stream>>>(nn, t, e, scal, s_hat_dev + (int64_t)k * nn,
                                           e_hat_dev ? e_hat_dev + (int64_t)k * nn : nullptr);
        EB_CUDA(cudaGetLastError());
      }
      EB_CUDA(cudaStreamSynchronize(stream));
    } catch (...) {
      release();
      throw;
    }
    release();
  });
}

int nn_train_step(nn_handle* h, int width, int height, int batch, const float* s_hat_dev, const double* c_dev,
                  const int32_t* geo_of_dev, const uint8_t* code_dev, const float* diag_dev, const int32_t* pick_dev,
                  float lr, float* loss_dev, cudaStream_t stream) {
  if (!h || !s_hat_dev || !c_dev || !geo_of_dev || !code_dev || !diag_dev || !pick_dev) {
    set_error("nn_train_step: NULL argument");
    return EB_ERR_INVALID;
  }
  if (int st = check_shape(width, height, batch)) return st;
  if (!(lr > 0.0f)) {
    set_error("nn_train_step: lr must be > 0");
    return EB_ERR_INVALID;
  }
  return guarded([&] {
    NN& N = h->n;
    const Image im{width, height * batch, height};
    const int64_t npx = npx_of(im);
    ensure_act(N, npx, stream);
    const int64_t per = (int64_t)width * height;
    const int lnb = (int)((per + 255) / 256);
    if ((int64_t)batch * lnb > N.cap_lpart) {
      dfree(N.lpart, stream);
      N.cap_lpart = 0;
      N.lpart = dalloc<double>((int64_t)batch * lnb, stream, false);
      N.cap_lpart = (int64_t)batch * lnb;
    }
    if (batch > N.cap_batch) {
      dfree(N.cimg, stream);
      dfree(N.loss, stream);
      N.cap_batch = 0;
      N.cimg = dalloc<double>(batch, stream);
      N.loss = dalloc<float>(batch + 1, stream);
      N.cap_batch = batch;
    }
    int64_t nl = 0;
    k_gather<<<blocks_for(npx, 256), 256, 0, stream>>>(im, s_hat_dev, c_dev, geo_of_dev, code_dev, diag_dev,
                                                       pick_dev, N.in, N.code, N.diag, N.cimg);
    forward(N, im, N.in, N.out, stream, nl);
    k_loss<<<dim3((unsigned)lnb, (unsigned)batch), 256, 0, stream>>>(im, N.code, N.diag, N.in, N.out, N.cimg,
                                                                      1.0f / (float)batch, N.dout, N.lpart);
    k_loss_reduce<<<1, 256, 0, stream>>>(N.lpart, lnb, batch, N.cimg, loss_dev ? loss_dev : N.loss);
    backward(N, im, N.in, N.dout, stream, nl);
    N.steps += 1;
    const float c1 = (float)(1.0 - std::pow(0.9, (double)N.steps));
    const float c2 = (float)(1.0 - std::pow(0.999, (double)N.steps));
    k_adam<<<blocks_for(NPARAM, 256), 256, 0, stream>>>(NPARAM, N.P, N.G, N.m, N.v, lr, c1, c2);
    pack(N, stream, nl);
    EB_CUDA(cudaGetLastError());
  });
}

int nn_precondition(const amg_handle* amg, nn_handle* nn, int mode, const double* r_dev, double* z_dev,
                    cudaStream_t stream) {
  if (!amg || !nn || !r_dev || !z_dev) {
    set_error("nn_precondition: NULL argument");
    return EB_ERR_INVALID;
  }
  if (mode != EB_NN_PLAIN && mode != EB_NN_ENERGY) {
    set_error("nn_precondition: mode must be EB_NN_PLAIN or EB_NN_ENERGY");
    return EB_ERR_INVALID;
  }
  return guarded([&] {
    Solver& S = const_cast<Solver&>(amg->s);
    EB_REQUIRE(S.H != nullptr, EB_ERR_INVALID, "nn_precondition: handle has no hierarchy");
    EB_REQUIRE(!S.eb->has_beta(), EB_ERR_NOT_IMPLEMENTED, "nn_precondition: the learned stage needs beta = 1");
    nn_stage_prepare(nn, *S.eb, stream);
    int64_t nl = 0;
    amg_vcycle_grid(S, r_dev, z_dev, stream);
    nn_stage_apply(nn, *S.eb, S.shift, mode, r_dev, z_dev, nl, nullptr, stream);
    EB_CUDA(cudaGetLastError());
  });
}

int pcg_solve_nn(const amg_handle* amg, nn_handle* nn, int mode, const double* b_dev, double* x_dev, double rtol,
                 int maxit, const pcg_opts* opts, pcg_stats* stats, cudaStream_t stream) {
  if (!amg || !nn || !b_dev || !x_dev) {
    set_error("pcg_solve_nn: NULL argument");
    return EB_ERR_INVALID;
  }
  if (mode != EB_NN_PLAIN && mode != EB_NN_ENERGY) {
    set_error("pcg_solve_nn: mode must be EB_NN_PLAIN or EB_NN_ENERGY");
    return EB_ERR_INVALID;
  }
  pcg_opts o{EB_PC_AMG_NN, 1, 1, 0};
  if (opts) o = *opts;
  o.precond = EB_PC_AMG_NN;
  int rc = EB_OK;
  int st = guarded([&] {
    Solver& S = const_cast<Solver&>(amg->s);
    EB_REQUIRE(S.H != nullptr, EB_ERR_INVALID, "pcg_solve_nn: handle has no hierarchy");
    EB_REQUIRE(!S.eb->has_beta(), EB_ERR_NOT_IMPLEMENTED, "pcg_solve_nn: the learned stage needs beta = 1");
    nn_stage_prepare(nn, *S.eb, stream);
    S.nn = nn;
    S.nn_mode = mode;
    try {
      rc = S.pcg(b_dev, x_dev, rtol, maxit, o, stats, stream);
    } catch (...) {
      S.nn = nullptr;
      throw;
    }
    S.nn = nullptr;
  });
  if (st != EB_OK) return st;
  const int ns = nn_status(nn, stream);
  return ns != EB_OK ? ns : rc;
}

}  // extern "C"
