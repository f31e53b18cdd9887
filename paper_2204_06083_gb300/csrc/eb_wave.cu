// Several FP32 leapfrog steps per launch on a 2D grid (theta-scheme of Sec.
// 3.5 at theta = 0, beta = 1).
//
// One step per launch moves 13 bytes per DOF and step and waits for the launch
// boundary; here a warp carries a strip of the fields through TT steps in
// registers before it writes them back.  A strip is 128 columns (four adjacent
// ones per lane), of which the middle WV_CORE are written; the warp walks down
// the rows of its task, and when row y of u^n arrives, it forms u^{n+1} at row
// y - 1, u^{n+2} at row y - 2, ..., u^{n+TT} at row y - TT, each from the three
// newest rows of the level before (x neighbours by shuffles).  The columns
// within TT of the strip's edges and the TT rows above and below a task are
// computed by the neighbouring tasks too, from the old fields; so a pass reads
// one pair of fields and writes another, and an even number of passes ends in
// the caller's.  Rows arrive through a ring of asynchronous copies (each lane
// copies and reads its own columns), no barrier.
//
// The arithmetic of a node is k_leapfrog's, operation for operation, so the
// fields are the same bit for bit (up to the sign of a zero): two columns per
// packed instruction (fma.rn.f32x2, each lane the scalar round-to-nearest
// result), and some levels held negated so that no operand needs a negation.
//
// What bounds it is instruction issue: some 200 warp instructions per row of
// a strip for the eight levels, at half an instruction per clock and scheduler
// with three warps each; the fields stay in L2.  Eight levels per launch share
// the work of a row (copies, addresses, the ring), and their 16 halo rows cost
// less than the second pass that four levels need.  4096^2 star (3.3 M CPs),
// per step: 3.9 us with TT = 8 (4.3 with 6, 5.2 with 4), 7.9 us one step per
// launch; 2000^2: 2.4 against 3.9; 1302^2: 2.3 against 2.7; 128^2: 1.7 against
// 1.8.
#include "eb_internal.cuh"
#include "stencil.cuh"

#include <algorithm>
#include <mutex>

namespace ebk {

constexpr int WV_THREADS = 128;
constexpr int WV_COLS = 128;               // columns of a strip: four per lane
constexpr int WV_MAXT = 8;                 // steps per launch at most
constexpr int WV_HALO = 8;                 // columns on either side that are not written
constexpr int WV_CORE = WV_COLS - 2 * WV_HALO;
constexpr int WV_AHEAD = 4;                // rows in flight
constexpr int WV_RING = WV_AHEAD + 1;      // rows of a warp's ring of u^n and u^{n-1}
constexpr int WV_DRING = 16;               // rows of its ring of D: those of y, ..., y - WV_MAXT stay readable
constexpr int WV_ROWF = 2 * WV_COLS;       // floats of a ring row: u^n, u^{n-1}
constexpr int WV_WARPF = WV_RING * WV_ROWF + WV_DRING * WV_COLS;
constexpr int WV_SMEM = WV_THREADS / 32 * WV_WARPF * 4;
constexpr int WV_MAXROWS = 64 - 3 * WV_MAXT;  // rows of a task: a bit of its mask each, with the halo rows
// The plan is made by the call that brings a handle's steps to this many: it
// takes 20 us and the allocation of the second pair of fields (4096^2: 180 us),
// which a program of a few steps does not earn back.  First call of a handle,
// 4096^2: 8 steps 260 us with the plan and 127 without, 64 steps 465 against 649
constexpr int WV_FIRST_STEPS = 32;
constexpr int WV_WARPS = 8;                // warps per SM that the tasks are cut for (12 fit)
static_assert(WV_MAXT <= WV_HALO && WV_HALO % 4 == 0 && WV_DRING >= WV_AHEAD + WV_MAXT + 1, "strip");

// first written column (low 24 bits) and number of rows (above), first written
// row, and, bit k, whether the strip's 128 columns are all interior CPs (D = 4)
// at row y - WV_MAXT + k (all bits set: at every row the task reads)
struct WvTask {
  int x_rows, y;
  uint64_t inner;
};
constexpr int WV_MAXX = 1 << 24;

struct WvArgs {
  int n0, n1;
  const float* diag;         // D_k at the CPs, 0 elsewhere
  const float *cur, *prev;   // u^n, u^{n-1}
  float *ocur, *oprev;       // u^{n+TT}, u^{n+TT-1}
  float c2;                  // dt^2 / h^2
  const WvTask* task;
  const int* ntask;
  bool wide;                 // rows start on 16-byte boundaries (n0 a multiple of 4)
};

__device__ __forceinline__ uint64_t wv_pk(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 wv_up(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ uint64_t wv_add(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t wv_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// whether level l (u^{n+l}) is held negated.  With x = u^{n+l} and po =
// u^{n+l-1} held with equal signs, fma(-c2, s - D x, fma(-2, x, po)) is u^{n+l+1}
// with the opposite sign; with opposite signs, fma(c2, s - D x, fma(2, x, po))
// is u^{n+l+1} with x's sign.
__host__ __device__ constexpr bool wv_neg(int l) {
  bool a = false, b = false;  // levels l - 1 and l, from l = 0
  for (int k = 0; k < l; ++k) {
    const bool c = a == b ? !b : b;
    a = b;
    b = c;
  }
  return b;
}

template <int TT>
struct WvState {
  uint64_t lev[TT][3][2];  // rows of u^n .. u^{n+TT-1}: [level][row slot][column pair]
};

// Row y arrives: u = u^n there, p = u^{n-1} at row y - 1.  INNER: every lane's
// columns at rows y, ..., y - TT are interior CPs (D = 4); else drow(k) is this
// lane's D at row y - k (0 off the CPs).  out = u^{n+TT} at row y - TT (as held).
template <int TT, int PH, bool INNER, class DRow>
__device__ __forceinline__ void wv_row(WvState<TT>& s, const uint64_t (&u)[2], const uint64_t (&p)[2], DRow drow,
                                       float c2, int valid, uint64_t (&out)[2]) {
  constexpr int N = PH, M = (PH + 2) % 3, O = (PH + 1) % 3;  // newest, middle and oldest row slots
  uint64_t f[2] = {u[0], u[1]};
#pragma unroll
  for (int l = 0; l < TT; ++l) {
    uint64_t old[2];  // level l - 1 at the row computed now
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      old[c] = l == 0 ? p[c] : s.lev[l > 0 ? l - 1 : 0][O][c];
      s.lev[l][N][c] = f[c];
    }
    if (l < valid) {
      const bool same = (l == 0 ? false : wv_neg(l - 1)) == wv_neg(l);
      const uint64_t two = same ? wv_pk(-2.0f, -2.0f) : wv_pk(2.0f, 2.0f), cc = same ? wv_pk(-c2, -c2) : wv_pk(c2, c2);
      const float2 a = wv_up(s.lev[l][M][0]), b = wv_up(s.lev[l][M][1]);
      const float left = __shfl_up_sync(0xffffffffu, b.y, 1), right = __shfl_down_sync(0xffffffffu, a.x, 1);
      const uint64_t v0 = wv_add(s.lev[l][O][0], s.lev[l][N][0]), v1 = wv_add(s.lev[l][O][1], s.lev[l][N][1]);
      const uint64_t t0 = wv_fma(two, s.lev[l][M][0], old[0]), t1 = wv_fma(two, s.lev[l][M][1], old[1]);
      const uint64_t m12 = wv_pk(a.y, b.x);
      const uint64_t s0 = wv_add(wv_add(wv_pk(left, a.x), m12), v0);
      const uint64_t s1 = wv_add(wv_add(m12, wv_pk(b.y, right)), v1);
      if (INNER) {
        const uint64_t d = wv_pk(-4.0f, -4.0f);
        f[0] = wv_fma(cc, wv_fma(d, s.lev[l][M][0], s0), t0);
        f[1] = wv_fma(cc, wv_fma(d, s.lev[l][M][1], s1), t1);
      } else {
        const float4 d = drow(l + 1);
        const float2 w0 = wv_up(wv_fma(cc, wv_fma(wv_pk(-d.x, -d.y), s.lev[l][M][0], s0), t0));
        const float2 w1 = wv_up(wv_fma(cc, wv_fma(wv_pk(-d.z, -d.w), s.lev[l][M][1], s1), t1));
        f[0] = wv_pk(d.x > 0.0f ? w0.x : 0.0f, d.y > 0.0f ? w0.y : 0.0f);
        f[1] = wv_pk(d.z > 0.0f ? w1.x : 0.0f, d.w > 0.0f ? w1.y : 0.0f);
      }
    }
  }
  out[0] = f[0];
  out[1] = f[1];
}

// asynchronous copies of 16 or 8 bytes to shared memory
__device__ __forceinline__ void wv_cp16(uint32_t dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void wv_cp8(uint32_t dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}

template <int TT, bool WIDE>
__global__ void __launch_bounds__(WV_THREADS) k_leapfrog_block(WvArgs a) {
  extern __shared__ __align__(16) float wv_smem[];
  const int lane = threadIdx.x & 31;
  float* ringp = wv_smem + (threadIdx.x >> 5) * WV_WARPF + lane * 4;
  float* dringp = ringp + WV_RING * WV_ROWF;
  const uint32_t ring = (uint32_t)__cvta_generic_to_shared(ringp), dring = (uint32_t)__cvta_generic_to_shared(dringp);
  const int nt = __ldg(a.ntask);
  const int nw = (int)gridDim.x * (WV_THREADS / 32);
  static_assert(TT <= WV_MAXT, "levels");
  for (int t = (int)blockIdx.x * (WV_THREADS / 32) + (threadIdx.x >> 5); t < nt; t += nw) {
    const int4 tk = __ldg(reinterpret_cast<const int4*>(a.task + t));
    const int x = (tk.x & (WV_MAXX - 1)) - WV_HALO + 4 * lane;
    const int y0 = tk.y, y1 = min(y0 + (tk.x >> 24), a.n1);
    // written columns (the strip may reach beyond the grid)
    const bool core = lane >= WV_HALO / 4 && lane < 32 - WV_HALO / 4 && x < a.n0, core2 = core && x + 2 < a.n0;
    const int yl = y0 - TT, yh = y1 + TT;  // rows read
    // tasks that read D: bit TT: whether row y is interior as a whole; below:
    // rows y - 1, ...; above: rows to come
    uint64_t inner = (((uint64_t)(uint32_t)tk.w << 32 | (uint32_t)tk.z) >> (WV_MAXT - TT)) << TT;
    const bool cut = tk.w != -1 || tk.z != -1;  // D differs from 4 somewhere
    // Rows and columns beyond the grid are clamped to it.  The outermost rows
    // and columns hold no CP (D = 0), so a clamped row is masked as a whole, and
    // whatever a clamped column holds reaches no CP.
    const int xa = min(max(x, 0), WIDE ? a.n0 - 4 : a.n0 - 2), xb = min(max(x + 2, 0), a.n0 - 2);
    int fy = yl;  // next row to fetch, and its ring rows
    uint32_t fu = ring;
    auto fetch1 = [&](uint32_t dst, const float* src, int y) {
      const float* row = src + min(max(y, 0), a.n1 - 1) * a.n0;
      if (WIDE) {
        wv_cp16(dst, row + xa);
      } else {
        wv_cp8(dst, row + xa);
        wv_cp8(dst + 8, row + xb);
      }
    };
    auto fetch = [&] {
      if (fy < yh) {
        fetch1(fu, a.cur, fy);
        fetch1(fu + WV_COLS * 4, a.prev, fy - 1);
        if (cut) fetch1(dring + (uint32_t)((fy - yl) % WV_DRING) * (WV_COLS * 4), a.diag, fy);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      ++fy;
      fu = fu == ring + (WV_RING - 1) * WV_ROWF * 4 ? ring : fu + WV_ROWF * 4;
    };
    for (int k = 0; k < WV_AHEAD; ++k) fetch();
    WvState<TT> s;
#pragma unroll
    for (int l = 0; l < TT; ++l)
#pragma unroll
      for (int k = 0; k < 3; ++k) s.lev[l][k][0] = s.lev[l][k][1] = 0;
    int rs = 0;  // ring row of row y
    auto row = [&](auto ph, int y) {
      asm volatile("cp.async.wait_group %0;" ::"n"(WV_AHEAD - 1) : "memory");
      const float* st = ringp + rs * WV_ROWF;
      const float4 u4 = *reinterpret_cast<const float4*>(st);
      const float4 p4 = *reinterpret_cast<const float4*>(st + WV_COLS);
      auto drow = [&](int k) {  // D at row y - k
        return *reinterpret_cast<const float4*>(dringp + ((y - yl - k) & (WV_DRING - 1)) * WV_COLS);
      };
      uint64_t u[2] = {wv_pk(u4.x, u4.y), wv_pk(u4.z, u4.w)}, p[2] = {wv_pk(p4.x, p4.y), wv_pk(p4.z, p4.w)}, o[2];
      constexpr uint32_t ALL = (2u << TT) - 1u;  // rows y ... y - TT
      const bool in = !cut || ((uint32_t)inner & ALL) == ALL;
      if (!in) {  // entries off the CPs are ignored
        const float4 d = drow(0), e = drow(1);
        u[0] = wv_pk(d.x > 0.0f ? u4.x : 0.0f, d.y > 0.0f ? u4.y : 0.0f);
        u[1] = wv_pk(d.z > 0.0f ? u4.z : 0.0f, d.w > 0.0f ? u4.w : 0.0f);
        p[0] = wv_pk(e.x > 0.0f ? p4.x : 0.0f, e.y > 0.0f ? p4.y : 0.0f);
        p[1] = wv_pk(e.z > 0.0f ? p4.z : 0.0f, e.w > 0.0f ? p4.w : 0.0f);
      }
      fetch();
      // level l + 1 is needed from row yl + l + 1 on: computed once y >= yl + 2 (l + 1)
      const int valid = (y - yl) >> 1;
      if (in) wv_row<TT, decltype(ph)::value, true>(s, u, p, drow, a.c2, valid, o);
      else wv_row<TT, decltype(ph)::value, false>(s, u, p, drow, a.c2, valid, o);
      const int r = y - TT;
      if (r >= y0 && core) {
        constexpr int M = (decltype(ph)::value + 2) % 3;
        float2 c[2], q[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          c[h] = wv_up(o[h]);
          q[h] = wv_up(s.lev[TT - 1][M][h]);
          if (wv_neg(TT)) c[h] = make_float2(-c[h].x, -c[h].y);
          if (wv_neg(TT - 1)) q[h] = make_float2(-q[h].x, -q[h].y);
        }
        const int at = r * a.n0 + x;
        float *oc = a.ocur + at, *op = a.oprev + at;
        if (WIDE && in) {
          *reinterpret_cast<float4*>(oc) = make_float4(c[0].x, c[0].y, c[1].x, c[1].y);
          *reinterpret_cast<float4*>(op) = make_float4(q[0].x, q[0].y, q[1].x, q[1].y);
        } else {  // the pairs that hold a CP
          const float4 d = in ? make_float4(4.0f, 4.0f, 4.0f, 4.0f) : drow(TT);
          if (d.x > 0.0f || d.y > 0.0f) {
            *reinterpret_cast<float2*>(oc) = c[0];
            *reinterpret_cast<float2*>(op) = q[0];
          }
          if (core2 && (d.z > 0.0f || d.w > 0.0f)) {
            *reinterpret_cast<float2*>(oc + 2) = c[1];
            *reinterpret_cast<float2*>(op + 2) = q[1];
          }
        }
      }
      inner >>= 1;
      rs = rs + 1 == WV_RING ? 0 : rs + 1;
    };
    for (int y = yl; y < yh; y += 3) {
      row(std::integral_constant<int, 0>{}, y);
      if (y + 1 < yh) row(std::integral_constant<int, 1>{}, y + 1);
      if (y + 2 < yh) row(std::integral_constant<int, 2>{}, y + 2);
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  }
}

// the tasks (strip x chunk of rows) that hold a CP, in any order; one warp per
// candidate, a lane per four columns of the strip.  A chunk with cut cells,
// whose rows take about twice the instructions, is cut in two.
__global__ void __launch_bounds__(256) k_wave_tasks(int n0, int n1, const uint8_t* __restrict__ code, int rows,
                                                    int strips, int chunks, WvTask* task, int* ntask) {
  const int lane = threadIdx.x & 31;
  const int w = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (w >= strips * chunks) return;
  const int x0 = (w % strips) * WV_CORE, y0 = (w / strips) * rows;
  uint64_t has = 0, inner = 0;  // bit k: row y0 - WV_MAXT + k holds a CP in the written columns / is interior
  for (int k = 0; k < rows + 2 * WV_MAXT; ++k) {
    const int y = y0 - WV_MAXT + k;
    if (y < 0 || y >= n1) continue;
    bool cp = false, in = true;
    for (int c = 0; c < 4; ++c) {
      const int x = x0 - WV_HALO + 4 * lane + c;
      const uint32_t v = x >= 0 && x < n0 ? code[(int64_t)y * n0 + x] : 0u;
      in = in && v == CODE_CP;
      cp = cp || ((v & CODE_CP) && x >= x0 && x < x0 + WV_CORE);
    }
    if (__any_sync(0xffffffffu, cp)) has |= 1ull << k;
    if (__all_sync(0xffffffffu, in)) inner |= 1ull << k;
  }
  if (lane != 0) return;
  // the bits of a task of r rows from its first row's bit on; all set: no D is read
  const uint64_t whole = (1ull << (rows + 2 * WV_MAXT)) - 1;
  const int parts = (inner & whole) == whole ? 1 : 2;
  for (int q = 0; q < parts; ++q) {
    const int f = rows * q / parts, r = rows * (q + 1) / parts - f;
    if (r == 0 || !((has >> (f + WV_MAXT)) & ((1ull << r) - 1))) continue;
    const uint64_t m = (1ull << (r + 2 * WV_MAXT)) - 1, in = (inner >> f) & m;
    task[atomicAdd(ntask, 1)] = WvTask{x0 | r << 24, y0 + f, in == m ? ~0ull : in};
  }
}

// A handle has one second pair of fields.  A call that finds it in use -- by a
// run still in flight on another stream, or by a call that another thread is
// enqueuing -- takes the in-place steps instead, which need none, so that calls
// of one handle on several streams overlap.
struct WavePlan {
  std::mutex mu;                 // held while a call enqueues
  cudaEvent_t done = nullptr;    // recorded at the end of each use, one that fails half way included
  cudaStream_t stream = nullptr; // of the last use
  int64_t steps = 0;             // taken while the rest is not there
  bool ready = false;            // the rest is there, the task list written before done
  float* buf = nullptr;          // second pair of fields
  WvTask* task = nullptr;        // strips x chunks of rows that hold a CP
  int* ntask = nullptr;
};

static WavePlan& wave_plan(const EBHandle& eb) {
  static std::mutex m;  // of the creation of plans
  std::lock_guard<std::mutex> lock(m);
  if (!eb.wave) eb.wave = new WavePlan();
  return *eb.wave;
}

void wave_plan_free(WavePlan*& W, cudaStream_t s) {
  if (!W) return;
  if (W->done) {
    cudaStreamWaitEvent(s, W->done, 0);
    cudaEventDestroy(W->done);
  }
  dfree(W->buf, s);
  dfree(W->task, s);
  dfree(W->ntask, s);
  delete W;
  W = nullptr;
}

template <int TT>
static void wave_launch(const WvArgs& a, unsigned blocks, cudaStream_t s) {
  auto go = [&](auto wide) {
    const auto fn = k_leapfrog_block<TT, decltype(wide)::value>;
    EB_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, WV_SMEM));
    fn<<<blocks, WV_THREADS, WV_SMEM, s>>>(a);
  };
  if (a.wide) go(std::true_type{});
  else go(std::false_type{});
}

// Tasks: as many as the resident warps, so that a pass is one wave (WV_WARPS
// of the 12 that fit: tasks with cut cells are cut in two, and the domain does
// not fill its strips).  At least four rows -- below that the halo rows cost
// more than the parallelism gives -- or two on grids of a few dozen tasks.
static int wave_rows(int64_t num_cp) {
  const int64_t warps = (int64_t)num_sms() * WV_WARPS;
  const int64_t least = num_cp < 8000 ? 2 : 4;
  return (int)std::min<int64_t>(WV_MAXROWS, std::max<int64_t>(least, (num_cp / WV_CORE + warps - 1) / warps));
}

bool launch_leapfrog_blocked(const EBHandle& eb, float* ua, float* ub, int nsteps, float c2, cudaStream_t s) {
  const Geometry& G = eb.g;
  if (G.n0 >= WV_MAXX) return false;
  WavePlan& W = wave_plan(eb);
  std::unique_lock<std::mutex> lock(W.mu, std::try_to_lock);
  if (!lock) return false;
  if (!W.ready && (W.steps += nsteps) < WV_FIRST_STEPS) return false;
  if (W.done && W.stream != s) {
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;  // a query may meet another stream's capture
    cudaThreadExchangeStreamCaptureMode(&mode);
    const cudaError_t e = cudaEventQuery(W.done);
    cudaThreadExchangeStreamCaptureMode(&mode);
    if (e == cudaErrorNotReady) {
      cudaGetLastError();
      return false;
    }
    EB_CUDA(e);
  }
  const int rows = wave_rows(eb.num_cp);
  const int strips = (G.n0 + WV_CORE - 1) / WV_CORE, chunks = (G.n1 + rows - 1) / rows;
  if (!W.done) EB_CUDA(cudaEventCreateWithFlags(&W.done, cudaEventDisableTiming));
  EB_CUDA(cudaStreamWaitEvent(s, W.done, 0));
  W.stream = s;
  // marks what has been enqueued below, also when a later launch fails
  struct Mark {
    cudaEvent_t e;
    cudaStream_t s;
    ~Mark() { cudaEventRecord(e, s); }
  } mark{W.done, s};
  if (!W.ready) {
    try {
      if (!W.buf) W.buf = dalloc<float>(2 * (size_t)G.num_nodes, s, false);
      if (!W.task) W.task = dalloc<WvTask>(2 * (size_t)strips * chunks, s, false);
      if (!W.ntask) W.ntask = dalloc<int>(1, s);
    } catch (const Failure& f) {
      if (f.code == EB_ERR_OOM) return false;  // the in-place steps need no second pair of fields
      throw;
    }
    EB_CUDA(cudaMemsetAsync(W.ntask, 0, sizeof(int), s));
    k_wave_tasks<<<blocks_for((int64_t)strips * chunks * 32, 256), 256, 0, s>>>(G.n0, G.n1, eb.code, rows, strips,
                                                                                chunks, W.task, W.ntask);
    EB_CUDA(cudaGetLastError());
    W.ready = true;
  }
  float *b0 = W.buf, *b1 = W.buf + G.num_nodes;
  WvArgs a{};
  a.n0 = G.n0;
  a.n1 = G.n1;
  a.diag = eb.diag32;
  a.c2 = c2;
  a.task = W.task;
  a.ntask = W.ntask;
  a.wide = G.n0 % 4 == 0 &&
           (((uintptr_t)ua | (uintptr_t)ub | (uintptr_t)b0 | (uintptr_t)b1 | (uintptr_t)eb.diag32) & 15) == 0;
  const int64_t most = 2 * (int64_t)strips * chunks;
  const unsigned blocks = (unsigned)std::min<int64_t>((most * 32 + WV_THREADS - 1) / WV_THREADS, (int64_t)num_sms() * 3);
  // an even number of passes of as equal lengths as possible
  int np = (nsteps + WV_MAXT - 1) / WV_MAXT;
  np += np & 1;
  a.cur = ub;
  a.prev = ua;
  a.ocur = b1;
  a.oprev = b0;
  for (int i = 0; i < np; ++i) {
    switch (nsteps / np + (i < nsteps % np ? 1 : 0)) {
      case 1: wave_launch<1>(a, blocks, s); break;
      case 2: wave_launch<2>(a, blocks, s); break;
      case 3: wave_launch<3>(a, blocks, s); break;
      case 4: wave_launch<4>(a, blocks, s); break;
      case 5: wave_launch<5>(a, blocks, s); break;
      case 6: wave_launch<6>(a, blocks, s); break;
      case 7: wave_launch<7>(a, blocks, s); break;
      default: wave_launch<8>(a, blocks, s); break;
    }
    float *oc = a.ocur, *op = a.oprev;
    a.ocur = const_cast<float*>(a.cur);
    a.oprev = const_cast<float*>(a.prev);
    a.cur = oc;
    a.prev = op;
  }
  EB_CUDA(cudaGetLastError());
  return true;
}

}  // namespace ebk
