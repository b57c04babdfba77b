// ph.cu -- the particle-hole term P(ij)P(ab) t_ik^ac <kb|chi|cj> of Eq. (ccd3) through the
// cross-coupled channels of Sec. "Developing a CCD code": per channel
//   C[(k,c)][(j,b)] = <kb|v|cj> + 1/2 sum_(e,l) <kl|v|ce> t_lj^eb,   Q[(a,i)][(j,b)] = T C,
// in FP32 (the mixed iteration) and with FP64 accuracy (the FP64 iteration, the refinement sweeps,
// the third-order ring and the operators).
//
// Global spin flip: Q is formed for the cross channels with S_z > 0 and for the spin-up rows of
// the S_z = 0 channels; the update reads every other position at its flip (same value for
// flip-symmetric amplitudes; qmap holds the formed positions only).  In an
// S_z = 0 channel, with rows ordered (spin-up rows u, their flips F u) and columns alike,
// every matrix of the term has the block form [[A, B], [B, A]] (A = M[u][v], B = M[u][F v]);
// products of such matrices are formed from the half-size sums A + B and differences A - B,
//   (A_1 + B_1)(A_2 + B_2) = A_3 + B_3,  (A_1 - B_1)(A_2 - B_2) = A_3 - B_3,
// which is a quarter of the flops of the full channel.  T, W, V1 and Q are held in formed layout
// (pnm_internal.cuh): exactly these elements, the blocks A and B contiguous with 16-byte rows.
#include <algorithm>

#include "dig.cuh"
#include "pnm_context.cuh"

constexpr int PH_WARPS = PH_THREADS / 32;
// Channels of at most PH_WARP_DIM rows and columns per problem take one warp, the others a CTA; of at
// most PH_TINY_DIM (FP32, FP32-pair results) or PH_TINY_FP64 (FP64 results beside larger channels) a
// part of a warp or a warp of the tiny kernels.
constexpr int PH_WARP_DIM = 16, PH_TINY_DIM = 8, PH_TINY_FP64 = 5;

// One cross channel of the term: a problem (S_z > 0) or two of half size (S_z = 0).
struct __align__(16) PhItem {
  int x, sys;               // cross channel, its system
  unsigned short R, H, nm;  // rows, columns of a problem; problems (1: S_z > 0, 2: S_z = 0)
  unsigned short pad;
  // offsets: formed T, Q, W; formed V1; and of the digit term the source indices, the W fragments
  // (uint4), <kb|v|cj> as integers, and of the smallest channels W and <kb|v|cj> as element values
  unsigned to, vo, src, wf, v1, fx;
};

template <int GT>
__device__ __forceinline__ void group_sync() {
  if constexpr (GT == 32) __syncwarp();
  else __syncthreads();
}

__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// ------------------------------------------------------------------------------ FP32
// Shared memory of a group: T, W and C of every problem, rows padded to the 4 x 4 register tiles.
__host__ __device__ __forceinline__ constexpr size_t ph32_smem(int R, int H, int nm) {
  const int R4 = (R + 3) & ~3, H4 = formed_width(H);
  return sizeof(float) * nm * ((size_t)2 * R4 * H4 + (size_t)H4 * H4);
}

__device__ __forceinline__ void fma4(float (&acc)[4], float a, const float4& b) {
  acc[0] = fmaf(a, b.x, acc[0]);
  acc[1] = fmaf(a, b.y, acc[1]);
  acc[2] = fmaf(a, b.z, acc[2]);
  acc[3] = fmaf(a, b.w, acc[3]);
}

// A group of GT threads per channel.  W and V1 (sums and differences of S_z = 0 formed once per
// context) go to shared memory by 16-byte asynchronous copies, T too for S_z > 0; for S_z = 0 the
// blocks A and B are read and stored as sum and difference.  Then C += 1/2 W^T T in place and Q = T C
// in 4 x 4 register tiles; the second product reads four k steps of T's rows at a time, so T is
// staged once and never transposed.
template <int GT, int NM>
__device__ __forceinline__ void ph32_group(const PhItem& it, float* __restrict__ sm, const float* __restrict__ xt,
                                           const float* __restrict__ xw, const float* __restrict__ xv1,
                                           float* __restrict__ xq) {
  const int tid = GT == 32 ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
  const int R = it.R, H = it.H, R4 = (R + 3) & ~3, H4 = formed_width(H);
  const int RH = R4 * H4, HH = H4 * H4, vec = R * H4 / 4, vecc = H * H4 / 4;
  float* Ts = sm;
  float* Ws = Ts + NM * RH;
  float* Cs = Ws + NM * RH;
  const float4* __restrict__ t4 = reinterpret_cast<const float4*>(xt + it.to);
#pragma unroll
  for (int m = 0; m < NM; m++) {
    for (int f = tid; f < vec; f += GT) copy16(Ws + m * RH + 4 * f, xw + it.to + 4 * (m * vec + f));
    for (int f = tid; f < vecc; f += GT) copy16(Cs + m * HH + 4 * f, xv1 + it.vo + 4 * (m * vecc + f));
    // rows of C past H: read against T's zero columns
    for (int f = tid; f < HH - H * H4; f += GT) Cs[m * HH + H * H4 + f] = 0.0f;
  }
  if constexpr (NM == 1) {
    for (int f = tid; f < vec; f += GT) copy16(Ts + 4 * f, t4 + f);
  } else {
#pragma unroll 4
    for (int f = tid; f < vec; f += GT) {
      const float4 a = t4[f], b = t4[vec + f];
      *reinterpret_cast<float4*>(Ts + 4 * f) = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
      *reinterpret_cast<float4*>(Ts + RH + 4 * f) = make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  group_sync<GT>();
  const int th = H4 / 4;
  for (int tile = tid; tile < NM * th * th; tile += GT) {
    const int m = NM == 1 ? 0 : tile >= th * th, tt = tile - m * th * th;
    const int r0 = (tt / th) * 4, s0 = (tt % th) * 4;
    const float* W = Ws + m * RH + r0;
    const float* T = Ts + m * RH + s0;
    float acc[4][4] = {};
#pragma unroll 4
    for (int u = 0; u < R; u++) {
      const float4 a = *reinterpret_cast<const float4*>(W + u * H4), b = *reinterpret_cast<const float4*>(T + u * H4);
      fma4(acc[0], a.x, b);
      fma4(acc[1], a.y, b);
      fma4(acc[2], a.z, b);
      fma4(acc[3], a.w, b);
    }
    float* C = Cs + m * HH + r0 * H4 + s0;
#pragma unroll
    for (int i = 0; i < 4; i++) {
      float4 c = *reinterpret_cast<float4*>(C + i * H4);
      c = make_float4(c.x + 0.5f * acc[i][0], c.y + 0.5f * acc[i][1], c.z + 0.5f * acc[i][2], c.w + 0.5f * acc[i][3]);
      if (r0 + i < H) *reinterpret_cast<float4*>(C + i * H4) = c;
    }
  }
  group_sync<GT>();
  const int tr = R4 / 4;
  for (int tile = tid; tile < tr * th; tile += GT) {
    const int r0 = (tile / th) * 4, s0 = (tile % th) * 4;
    float acc[NM][4][4] = {};
#pragma unroll
    for (int m = 0; m < NM; m++) {
      const float* T = Ts + m * RH + r0 * H4;
      const float* C = Cs + m * HH + s0;
#pragma unroll 2
      for (int u = 0; u < H4; u += 4) {
        float4 a[4], b[4];
#pragma unroll
        for (int i = 0; i < 4; i++) a[i] = *reinterpret_cast<const float4*>(T + i * H4 + u);
#pragma unroll
        for (int i = 0; i < 4; i++) b[i] = *reinterpret_cast<const float4*>(C + (u + i) * H4);
#pragma unroll
        for (int i = 0; i < 4; i++) {
          fma4(acc[m][i], a[i].x, b[0]);
          fma4(acc[m][i], a[i].y, b[1]);
          fma4(acc[m][i], a[i].z, b[2]);
          fma4(acc[m][i], a[i].w, b[3]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {
      if (r0 + i >= R) break;
      float* q = xq + it.to + (r0 + i) * H4 + s0;
      if constexpr (NM == 1) {
        *reinterpret_cast<float4*>(q) = make_float4(acc[0][i][0], acc[0][i][1], acc[0][i][2], acc[0][i][3]);
      } else {
        float p[4], d[4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
          p[j] = 0.5f * (acc[0][i][j] + acc[NM - 1][i][j]);
          d[j] = 0.5f * (acc[0][i][j] - acc[NM - 1][i][j]);
        }
        *reinterpret_cast<float4*>(q) = make_float4(p[0], p[1], p[2], p[3]);
        *reinterpret_cast<float4*>(q + R * H4) = make_float4(d[0], d[1], d[2], d[3]);
      }
    }
  }
}

// The first nblk CTAs take one channel each (the costliest first), the others PH_WARPS channels of at
// most PH_WARP_DIM rows and columns, one per warp (warp_smem bytes of shared memory each).
// What bounds it: latency of the staging (channels are small, 17 to 33 rows for N = 66), then the
// shared-memory reads of the tiles.  Three densities of N = 66, n^2 <= 36: 59 us per launch (with
// k_ph32_tiny) against 97 us with T, W and V1 in full matrices, read through index tables, W and V1
// added and subtracted in every launch and T transposed in shared memory between the products.
__global__ void __launch_bounds__(PH_THREADS) k_ph32(DevState D, const LoopCtl* __restrict__ ctl,
                                                     const PhItem* __restrict__ items, int nblk, int nwarp,
                                                     int warp_smem, const float* __restrict__ xt,
                                                     const float* __restrict__ xw, const float* __restrict__ xv1,
                                                     float* __restrict__ xq) {
  extern __shared__ __align__(16) unsigned char smraw[];
  if ((int)blockIdx.x < nblk) {
    const PhItem it = items[blockIdx.x];
    if (sys_done(D, ctl, it.sys)) return;  // CTA-uniform
    float* sm = reinterpret_cast<float*>(smraw);
    if (it.nm == 2) ph32_group<PH_THREADS, 2>(it, sm, xt, xw, xv1, xq);
    else ph32_group<PH_THREADS, 1>(it, sm, xt, xw, xv1, xq);
    return;
  }
  const int w = threadIdx.x >> 5, idx = ((int)blockIdx.x - nblk) * PH_WARPS + w;
  if (idx >= nwarp) return;  // whole warps leave; the warp path never synchronises the block
  const PhItem it = items[nblk + idx];
  if (sys_done(D, ctl, it.sys)) return;  // warp-uniform
  float* sm = reinterpret_cast<float*>(smraw + (size_t)w * warp_smem);
  if (it.nm == 2) ph32_group<32, 2>(it, sm, xt, xw, xv1, xq);
  else ph32_group<32, 1>(it, sm, xt, xw, xv1, xq);
}

// Channels of at most PH_TINY_DIM rows and columns per problem: eight lanes each, a lane per column.
// T and W in shared memory (rows read as broadcasts), the lane's column of C in registers.
// 120 systems of N = 14 (152 thousand channels of at most 7 rows): 46 us per launch against 159 us with
// a warp per channel and one element of the result per lane and step.
constexpr int PH32_TINY_PER_CTA = PH_THREADS / 8;
__global__ void __launch_bounds__(PH_THREADS) k_ph32_tiny(DevState D, const LoopCtl* __restrict__ ctl,
                                                          const PhItem* __restrict__ items, int n,
                                                          const float* __restrict__ xt, const float* __restrict__ xw,
                                                          const float* __restrict__ xv1, float* __restrict__ xq) {
  constexpr int S = PH_TINY_DIM;
  __shared__ __align__(16) float sm[PH32_TINY_PER_CTA][4 * S * S];  // per channel T and W, two problems each
  const int grp = threadIdx.x >> 3, c = threadIdx.x & 7, idx = blockIdx.x * PH32_TINY_PER_CTA + grp;
  PhItem it;
  int nm = 0;
  if (idx < n) {
    it = items[idx];
    if (!sys_done(D, ctl, it.sys)) nm = it.nm;
  }
  const int R = nm ? it.R : 0, H = nm ? it.H : 0, H4 = formed_width(H), q4 = H4 / 4, vec = R * q4;
  float* Ts = sm[grp];
  float* Ws = Ts + 2 * S * S;
  float v[2][S];
#pragma unroll
  for (int m = 0; m < 2; m++)
#pragma unroll
    for (int r = 0; r < S; r++) v[m][r] = m < nm && r < H && c < H ? __ldg(xv1 + it.vo + (m * H + r) * H4 + c) : 0.0f;
  const float4* __restrict__ t4 = reinterpret_cast<const float4*>(xt + it.to);
  const float4* __restrict__ w4 = reinterpret_cast<const float4*>(xw + it.to);
  // rows of 8 floats; a row of four columns leaves the upper half zero
  for (int f = c; f < R * 2; f += 8) {
    const int u = f >> 1, h = f & 1;
    const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float4 a = zero, b = zero, w0 = zero, w1 = zero;
    if (h < q4) {
      const int g = u * q4 + h;
      a = t4[g];
      w0 = w4[g];
      if (nm == 2) {
        b = t4[vec + g];
        w1 = w4[vec + g];
      }
    }
    float* t = Ts + u * S + 4 * h;
    float* w = Ws + u * S + 4 * h;
    if (nm == 2) {
      *reinterpret_cast<float4*>(t) = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
      *reinterpret_cast<float4*>(t + S * S) = make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
    } else {
      *reinterpret_cast<float4*>(t) = a;
    }
    *reinterpret_cast<float4*>(w) = w0;
    *reinterpret_cast<float4*>(w + S * S) = w1;
  }
  __syncwarp();
  auto row = [&](const float* p, float (&x)[S]) {
    const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
    x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
  };
#pragma unroll
  for (int m = 0; m < 2; m++) {
    if (m >= nm) break;
    float acc[S] = {};
    for (int u = 0; u < R; u++) {
      const float t = Ts[m * S * S + u * S + c];
      float w[S];
      row(Ws + m * S * S + u * S, w);
#pragma unroll
      for (int r = 0; r < S; r++) acc[r] = fmaf(w[r], t, acc[r]);
    }
#pragma unroll
    for (int r = 0; r < S; r++) v[m][r] = r < H ? v[m][r] + 0.5f * acc[r] : 0.0f;
  }
  for (int r = 0; r < R; r++) {
    float q[2] = {0.0f, 0.0f};
#pragma unroll
    for (int m = 0; m < 2; m++) {
      if (m >= nm) break;
      float t[S];
      row(Ts + m * S * S + r * S, t);
#pragma unroll
      for (int u = 0; u < S; u++) q[m] = fmaf(t[u], v[m][u], q[m]);
    }
    if (c < H) {
      float* o = xq + it.to + r * H4 + c;
      if (nm == 2) {
        *o = 0.5f * (q[0] + q[1]);
        o[R * H4] = 0.5f * (q[0] - q[1]);
      } else {
        *o = q[0];
      }
    }
  }
}

// FP32 copies of W and V1 in formed layout, sums and differences of S_z = 0 (one CTA per item).
__global__ void __launch_bounds__(128) k_ph_pack32(DevState D, const PhItem* __restrict__ items, float* __restrict__ xw,
                                                   float* __restrict__ xv1) {
  const PhItem it = items[blockIdx.x];
  auto pack = [&](const double* __restrict__ a, float* __restrict__ o, int n) {
    for (int f = threadIdx.x; f < n; f += blockDim.x) {
      const float x = (float)a[f];
      if (it.nm == 2) {
        const float y = (float)a[n + f];
        o[f] = x + y;
        o[n + f] = x - y;
      } else {
        o[f] = x;
      }
    }
  };
  const int H4 = formed_width(it.H);
  pack(D.x_w + it.to, xw + it.to, it.R * H4);
  pack(D.x_v1 + it.vo, xv1 + it.vo, it.H * H4);
}

void pnm_ph_pack32(pnm_ctx* ctx, float* xw, float* xv1) {
  pnm_need_ph_items(ctx);
  if (ctx->n_ph_items > 0) k_ph_pack32<<<ctx->n_ph_items, 128, 0, ctx->stream>>>(ctx->d, ctx->ph_items, xw, xv1);
  CUDA_TRY(cudaGetLastError());
}

// Mixed ph: T read from the FP32 formed copy the update scatters, Q in FP32 at its formed positions
// (the update gathers the four terms of each amplitude).  s_tiny: the stream of the smallest channels.
void launch_ph_mix(pnm_ctx* ctx, const float* xt, const float* xw, const float* xv1, float* xq, cudaStream_t s,
                   cudaStream_t s_tiny) {
  const int nblk = ctx->n_ph_large + ctx->n_ph_cta, ntiny = ctx->n_ph_tiny, nw = ctx->n_ph_warp - ntiny;
  const int nwb = (nw + PH_WARPS - 1) / PH_WARPS;
  if (nblk + nwb > 0) {
    const size_t smem = std::max(ctx->ph32_smem, PH_WARPS * ctx->ph32_warp_smem);
    k_ph32<<<nblk + nwb, PH_THREADS, smem, s>>>(ctx->d, ctx->ctl, ctx->ph_items, nblk, nw, (int)ctx->ph32_warp_smem, xt,
                                                xw, xv1, xq);
  } else {
    s_tiny = s;
  }
  if (ntiny > 0)
    k_ph32_tiny<<<(ntiny + PH32_TINY_PER_CTA - 1) / PH32_TINY_PER_CTA, PH_THREADS, 0, s_tiny>>>(
        ctx->d, ctx->ctl, ctx->ph_items + nblk + nw, ntiny, xt, xw, xv1, xq);
}

// ------------------------------------------------------------- ph term, FP64 accuracy (digits)
// The FP64 and FP32-pair ph term as digit products on the tensor cores (dig.cuh), mma.sync because
// the matrices are small (N = 66: 17 to 33 rows and columns): per problem (a S_z > 0 channel, or
// the sum and the difference problem of an S_z = 0 channel)
//   C[(k,c)][(j,b)] = <kb|v|cj> + 1/2 sum_(e,l) <kl|v|ce> t_lj^eb,   Q[(a,i)][(j,b)] = T C.
// Operands are integers and their digits from end to end, each with an exponent of its own per channel:
//   - W as digits in fragment order, <kb|v|cj> as integers, and the signed amplitude index of every
//     staged element, fixed per context (k_ph_pack; sums and differences of S_z = 0 formed there);
//   - T gathered as FP64 and converted in place to words of the channel's exponent (sums and
//     differences of S_z = 0 as exact integer sums), two neighbouring columns interleaved: the k index
//     of the second product; the first reads its k pairs across rows;
//   - C as integers, the two terms rounded to the coarser of their units: <kb|v|cj> 2^-61 of its largest,
//     the product 2^-60 of what its sum of R products can reach.  Its digits are stored interleaved by row
//     pairs straight from the first product's registers.
// An integer holds an element within PH_SPAN octaves of its operand's largest one to its last bit, and a
// smaller one to 2^-61 of that largest.  FP64 sums round at 2^-53 of the products they add, so the digits
// stand in for them only where no row or column of T, W or <kb|v|cj> lies wholly further down: a channel
// with such a row or column (one amplitude far above the others, say) is summed in FP64 (ph_values), and
// so is one whose product's unit is more than PH_SPAN octaves above that of <kb|v|cj> (amplitudes above
// about 10) while T has an empty column, where <kb|v|cj> stands alone.
// MBPT2 amplitudes and the Minnesota interaction stay within it (N = 14 to 66, densities 0.02 to 0.3:
// rows of T within 6 octaves of their channel's largest, rows of W within 5, of <kb|v|cj> 0).
// Only the results leave as floating point.  A group of 32 threads (channels of at most PH_WARP_DIM
// rows and columns) or of 128 (the others) takes a channel; a warp forms 16 x 8 blocks.
// What bounds it: instruction issue and its latencies around the products (operand expansion,
// drains, staging) at twelve warps per SM; without the MMAs it takes 6% less time.  Per launch: N = 66,
// n^2 <= 42, FP64 149 us against 405 us on the FP64 pipe; three densities of N = 66, n^2 <= 36, pairs, 298
// against 356 us on the FP32 pipe; symmetric matter, 28 nucleons, n^2 <= 20, FP64 40 against 52 us.  One
// exponent for all amplitudes of a system, their words made in two passes ahead of this kernel, took 153, 298
// and 48 us and left a channel far below the system's largest amplitude few bits (errors of 5e-6 of
// an element's own sum of products beside one amplitude 2^20 above the others).  Nothing of the staging may
// take the FP64 pipe: the signs of the gathered amplitudes as negations made it 160, 337 and 41 us.
__host__ __device__ __forceinline__ constexpr int ph_h8(int H) { return (H + 7) & ~7; }
// Row strides in 16-byte pairs: T's odd, C's 2 modulo 8, so that the fragment loads of the first
// product (two rows per thread) and of the second spread over the banks.
__host__ __device__ __forceinline__ constexpr int ph_ts(int H) { return ph_h8(H) / 2 + 1; }
__host__ __device__ __forceinline__ constexpr int ph_cs(int H) { return ph_h8(H) + 2; }
__host__ __device__ __forceinline__ constexpr size_t ph_dig_smem(int R, int H, int nm) {
  return sizeof(uint4) * nm * ((size_t)ph_h8(R) * ph_ts(H) + (size_t)(ph_h8(H) / 2) * ph_cs(H));
}
// beside the static shared memory of the kernels
constexpr size_t PH_SMEM = 227 * 1024 - 2048;
static_assert(ph_dig_smem(PH_LIMIT_ONE, PH_LIMIT_ONE, 1) <= PH_SMEM && ph_dig_smem(PH_LIMIT_TWO, PH_LIMIT_TWO, 2) <= PH_SMEM &&
                  ph32_smem(PH_LIMIT_ONE, PH_LIMIT_ONE, 1) <= PH_SMEM && ph32_smem(PH_LIMIT_TWO, PH_LIMIT_TWO, 2) <= PH_SMEM,
              "a channel's tiles would not fit an SM");

constexpr int PH_SPAN = 8;
constexpr int PH_MAX_DIM = DIG_FLUSH;  // rows or columns of a problem: the products drain once, at their end
static_assert(PH_LIMIT_ONE <= PH_MAX_DIM && PH_LIMIT_TWO <= PH_MAX_DIM, "digit sums would not be exact");

// Which rows and columns of a matrix hold an element within PH_SPAN octaves of the largest (big), which a
// smaller one other than zero (some): bytes that any thread may set, rows [0, n), columns [n, 2 n).
struct PhMarks {
  unsigned char* at;
  int n;
  __device__ void set(int k, int size, int least) const {
    if (size > 0) at[size >= least ? k : 2 * n + k] = 1;
  }
  __device__ bool empty(int k) const { return !at[k] && !at[2 * n + k]; }
  // whether one of four rows or columns holds small elements only
  __device__ bool low(int k4) const {
    const unsigned* m = reinterpret_cast<const unsigned*>(at);
    return (m[n / 2 + k4] & ~m[k4]) != 0;
  }
};
// The size of an element in integers (no comparison on the FP64 pipe): its bits above the fraction's
// low word, 0 for zero alone; and the least size within PH_SPAN octaves of exponent e.
__device__ __forceinline__ int size_of(double x) {
  return (__double2hiint(x) & 0x7fffffff) | (__double2loint(x) != 0);
}
__device__ __forceinline__ int least_size(int e) { return e > PH_SPAN + 1 ? (e - PH_SPAN) << 20 : 1; }

template <int GT>
__device__ __forceinline__ int group_max(int v, int* sh) {
  v = __reduce_max_sync(0xffffffffu, v);
  if constexpr (GT > 32) {
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < GT / 32; w++) v = max(v, sh[w]);
  }
  return v;
}
template <int GT>
__device__ __forceinline__ bool group_any(bool b) {
  if constexpr (GT == 32) return __any_sync(0xffffffffu, b);
  else return __syncthreads_or(b);
}

// The term of one channel in FP64 arithmetic (infinities, NaN, values so large that intermediate
// results might overflow, rows or columns far below the largest element): the sums of the same
// expressions in order.
template <typename Out, int GT>
__device__ __noinline__ void ph_values(const DevState& D, const PhItem& it, int tid, uint4* Ts, uint4* Cs,
                                       const double* __restrict__ t, bool quad, Out* __restrict__ xq) {
  const int R = it.R, H = it.H, nm = it.nm, TS = ph_ts(H), CS = ph_cs(H), H4 = formed_width(H);
  const long TP = (long)ph_h8(R) * TS, CP = (long)(ph_h8(H) / 2) * CS;
  auto T = [&](int m, int u, int s) -> double& { return reinterpret_cast<double*>(Ts + m * TP + u * TS + (s >> 1))[s & 1]; };
  auto C = [&](int m, int r, int c) -> double& { return reinterpret_cast<double*>(Cs + m * CP + (r >> 1) * CS + c)[r & 1]; };
  auto amp = [&](long e) {
    const int c = D.xmap[e];
    return c == 0 ? 0.0 : (c > 0 ? t[c - 1] : -t[-c - 1]);
  };
  auto pick = [&](const double* __restrict__ M, int m, int o, int n) {  // element o of problem m
    return nm == 1 ? M[o] : (m == 0 ? M[o] + M[n + o] : M[o] - M[n + o]);
  };
  for (int e = tid; e < R * H; e += GT) {
    const int u = e / H, s = e % H;
    const double a = amp(it.to + (long)u * H4 + s);
    if (nm == 1) T(0, u, s) = a;
    else {
      const double b = amp(it.to + (long)(R + u) * H4 + s);
      T(0, u, s) = a + b;
      T(1, u, s) = a - b;
    }
  }
  group_sync<GT>();
  for (int e = tid; e < nm * H * H; e += GT) {
    const int m = e / (H * H), r = (e % (H * H)) / H, c = e % H;
    double acc = 0.0;
    for (int u = 0; u < R && quad; u++) acc += pick(D.x_w + it.to, m, u * H4 + r, R * H4) * T(m, u, c);
    C(m, r, c) = pick(D.x_v1 + it.vo, m, r * H4 + c, H * H4) + 0.5 * acc;
  }
  group_sync<GT>();
  for (int e = tid; e < R * H; e += GT) {
    const int r = e / H, c = e % H;
    double acc[2] = {0.0, 0.0};
    for (int m = 0; m < nm; m++)
      for (int u = 0; u < H; u++) acc[m] += T(m, r, u) * C(m, u, c);
    Out* q = xq + it.to + r * H4 + c;
    if (nm == 1) *q = Arith<Out>::from_double(acc[0]);
    else {
      *q = Arith<Out>::from_double(0.5 * (acc[0] + acc[1]));
      q[R * H4] = Arith<Out>::from_double(0.5 * (acc[0] - acc[1]));
    }
  }
}

// Largest exponent of the amplitudes plus that of W beyond which ph_values is used: C and Q stay
// finite below.
constexpr int PH_MAX_EXP = 2900;

// ex: exponents of W and of <kb|v|cj>; marks: 4 PH_MAX_DIM bytes for a CTA's channel, 64 for a warp's.
template <typename Out, int GT, int NM>
__device__ __forceinline__ void ph_dig(const DevState& D, const PhItem& it, int2 ex, unsigned char* smraw,
                                       const double* __restrict__ t, const int* __restrict__ src,
                                       const uint4* __restrict__ wf, const long long* __restrict__ v1, bool quad,
                                       Out* __restrict__ xq, unsigned char* marks, int* sh_max) {
  const int tid = GT == 32 ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3, wid = tid >> 5;
  constexpr int NW = GT / 32;
  const int R = it.R, H = it.H, R8 = ph_h8(R), H8 = ph_h8(H), TS = ph_ts(H), CS = ph_cs(H);
  const int TP = R8 * TS, CP = (H8 / 2) * CS;
  uint4* Ts = reinterpret_cast<uint4*>(smraw);  // [problem][row][column pair]
  uint4* Cs = Ts + NM * TP;                     // [problem][row pair][column]
  const PhMarks mark{marks, GT == 32 ? PH_WARP_DIM : PH_MAX_DIM};  // of T: of both blocks of S_z = 0
  for (int k = tid; k < mark.n; k += GT) reinterpret_cast<int*>(marks)[k] = 0;
  // T: two neighbouring columns per step (index rows are padded to H8, rows past R read none), the
  // amplitudes and their largest exponent first, then their words, each thread its own elements
  const int wide = H8 / 2, total = R8 * wide, live = R * wide, du = GT / wide, ds = GT % wide;
  auto amp = [&](int c) {  // the sign on its bit: a negation would take the FP64 pipe
    if (c == 0) return 0.0;
    const double v = t[abs(c) - 1];
    return __hiloint2double(__double2hiint(v) ^ (c & (int)0x80000000), __double2loint(v));
  };
  int et = 1;
  {
    int u = tid / wide, s = tid % wide;
#pragma unroll 4
    for (int f = tid; f < total; f += GT) {
      double2* pa = reinterpret_cast<double2*>(Ts + u * TS + s);
      if constexpr (NM == 1) {
        const int2 c = f < live ? reinterpret_cast<const int2*>(src + it.src)[f] : make_int2(0, 0);
        const double2 a = make_double2(amp(c.x), amp(c.y));
        et = max(et, max(dig_exp(a.x), dig_exp(a.y)));
        *pa = a;
      } else {
        const int4 c = f < live ? reinterpret_cast<const int4*>(src + it.src)[f] : make_int4(0, 0, 0, 0);
        const double2 a = make_double2(amp(c.x), amp(c.z)), b = make_double2(amp(c.y), amp(c.w));
        et = max(et, max(max(dig_exp(a.x), dig_exp(a.y)), max(dig_exp(b.x), dig_exp(b.y))));
        *pa = a;
        pa[TP] = b;
      }
      u += du;
      s += ds;
      if (s >= wide) {
        s -= wide;
        u++;
      }
    }
  }
  et = group_max<GT>(et, sh_max);
  if constexpr (GT == 32) __syncwarp();  // the marks are clear
  if (et >= DIG_NONFINITE || ex.x >= DIG_NONFINITE || ex.y >= DIG_NONFINITE || et + ex.x > PH_MAX_EXP) {
    ph_values<Out, GT>(D, it, tid, Ts, Cs, t, quad, xq);  // group-uniform branch
    return;
  }
  {
    const int least = least_size(et);
    int u = tid / wide, s = tid % wide;
#pragma unroll 2
    for (int f = tid; f < total; f += GT) {
      uint4* pa = Ts + u * TS + s;
      const double2 a = *reinterpret_cast<const double2*>(pa);
      int m0 = size_of(a.x), m1 = size_of(a.y);
      const long long a0 = dig_fixed(a.x, et), a1 = dig_fixed(a.y, et);
      if constexpr (NM == 1) {
        *pa = dig_interleave(dig_word(a0), dig_word(a1));
      } else {
        const double2 b = *reinterpret_cast<const double2*>(pa + TP);
        m0 = max(m0, size_of(b.x));
        m1 = max(m1, size_of(b.y));
        const long long b0 = dig_fixed(b.x, et), b1 = dig_fixed(b.y, et);
        *pa = dig_interleave(dig_word(a0 + b0), dig_word(a1 + b1));
        pa[TP] = dig_interleave(dig_word(a0 - b0), dig_word(a1 - b1));
      }
      mark.set(u, max(m0, m1), least);
      mark.set(mark.n + 2 * s, m0, least);
      mark.set(mark.n + 2 * s + 1, m1, least);
      u += du;
      s += ds;
      if (s >= wide) {
        s -= wide;
        u++;
      }
    }
  }
  // units of C's terms (p1 with the factor 1/2), head bits finer than the product's digits allow for any R:
  // sums of R products of 61-bit (62 bits each for sums and differences) integers within 2^60, <kb|v|cj>
  // within 2^62, so that the leading digit of C stays within 82
  const int head = max(0, __clz(R - 1) - 24 - 2 * (NM - 1));
  const int p1 = dig_power(ex.x, et) + 14 - head - 1, pv = ex.y - 1022 - 61;
  const int pc = quad ? max(p1, pv) : pv, sx = min(pc - p1, 63), sv = min(pc - pv, 63);
  const long long rx = (1ll << sx) >> 1, rv = (1ll << sv) >> 1;  // half a unit
  const int rl = (1 << (14 - head)) >> 1;
  group_sync<GT>();
  bool low = tid < mark.n / 2 && mark.low(tid);  // known to the group after the first product
  if (sv > PH_SPAN)
    for (int k = tid; k < H; k += GT) low = low || mark.empty(mark.n + k);
  // C: 16 x 8 blocks of every problem; the fragments of W are requested one step ahead, across
  // blocks too
  const int nt = H8 / 8, sc = (H + 15) >> 4, kr = (R + 15) >> 4, blocks = NM * sc * nt;
  const bool small_r = R <= DIG_SMALL_K, small_h = H <= DIG_SMALL_K;
  uint4 w[4];
  auto load_w = [&](int b, int ks) {  // block b is strip b / nt of the problems' strips in turn
    const uint4* __restrict__ wp = wf + it.wf + ((long)(b / nt) * kr + ks) * 128 + lane;
#pragma unroll
    for (int r = 0; r < 4; r++) w[r] = __ldg(wp + r * 32);
  };
  if (quad && wid < blocks) load_w(wid, 0);
  for (int b = wid; b < blocks; b += NW) {
    const int ms = b / nt, m = ms / sc, strip = ms - m * sc, n0 = (b - ms * nt) * 8;
    const longlong2* __restrict__ vp =
        reinterpret_cast<const longlong2*>(v1 + it.v1) + (((long)ms * 16 + g) * H8 + n0) / 2 + q;
    const longlong2 va = __ldg(vp), vb = __ldg(vp + 4 * H8);
    dig_t c[4] = {(dig_t)((va.x + rv) >> sv), (dig_t)((va.y + rv) >> sv), (dig_t)((vb.x + rv) >> sv),
                  (dig_t)((vb.y + rv) >> sv)};
    if (quad) {
      float acc[DIG_LEVELS][4] = {};
      const uint4* tb = Ts + m * TP + (2 * q) * TS + ((n0 + g) >> 1);
      for (int ks = 0; ks < kr; ks++) {
        uint32_t a[4][DIG_LEVELS], bb[2][DIG_LEVELS];
        const bool half = R - ks * 16 <= 8;
#pragma unroll
        for (int r = 0; r < 4; r++) dig_expand<DIG_LEVELS>(w[r], a[r]);
        if (ks + 1 < kr) load_w(b, ks + 1);
        else if (b + NW < blocks) load_w(b + NW, 0);
        const uint4* tk = tb + ks * 16 * TS;
        dig_expand_across(tk[0], tk[TS], g & 1, bb[0]);
        if (!half) dig_expand_across(tk[8 * TS], tk[9 * TS], g & 1, bb[1]);
        dig_block(acc, a, bb, half);
      }
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const DigSum x = small_r ? dig_drain_small(acc, k) : dig_drain(acc, k);
        c[k] += (dig_t)(((x.hi << (18 + head)) + ((x.lo + rl) >> (14 - head)) + rx) >> sx);
      }
    }
    // digits of the row pairs (g, g ^ 1): the lanes of even g take the block's even columns
    const bool odd = g & 1;
    const dig_t r0 = __shfl_xor_sync(0xffffffffu, odd ? c[0] : c[1], 4);
    const dig_t r1 = __shfl_xor_sync(0xffffffffu, odd ? c[2] : c[3], 4);
    const dig_t o0 = odd ? c[1] : c[0], o1 = odd ? c[3] : c[2];
    uint4* pc0 = Cs + m * CP + ((strip * 16 + g) >> 1) * CS + n0 + 2 * q + (odd ? 1 : 0);
    if (strip * 16 + g < H8)
      *pc0 = dig_interleave(DIG_BIAS + (odd ? r0 : o0), DIG_BIAS + (odd ? o0 : r0));
    if (strip * 16 + g + 8 < H8)
      pc0[4 * CS] = dig_interleave(DIG_BIAS + (odd ? r1 : o1), DIG_BIAS + (odd ? o1 : r1));
  }
  if constexpr (GT == 32) __syncwarp();
  if (group_any<GT>(low)) {
    ph_values<Out, GT>(D, it, tid, Ts, Cs, t, quad, xq);
    return;
  }
  // Q
  const int sr = (R + 15) >> 4, kh = (H + 15) >> 4;
  const int p2 = 56 + (et - 1022 - 61) + pc - (NM == 2 ? 1 : 0);  // the half of sum and difference
  for (int b = wid; b < sr * nt; b += NW) {
    const int m0 = (b / nt) * 16, n0 = (b % nt) * 8;
    const bool low = m0 + 8 < R;  // rows m0 + 8 ... are stored
    DigSum x[4] = {}, x0[4];  // the last problem's sums, and those of the one before
#pragma unroll 1
    for (int m = 0; m < NM; m++) {
      float acc[DIG_LEVELS][4] = {};
      for (int ks = 0; ks < kh; ks++) {
        uint32_t a[4][DIG_LEVELS], bb[2][DIG_LEVELS];
        const bool half = H - ks * 16 <= 8;
        const uint4* ta = Ts + m * TP + (m0 + g) * TS + ks * 8 + q;
        const uint4* cb = Cs + m * CP + (ks * 8 + q) * CS + n0 + g;
        const uint4 zero = make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
        dig_expand<DIG_LEVELS>(ta[0], a[0]);
        dig_expand<DIG_LEVELS>(low ? ta[8 * TS] : zero, a[1]);
        dig_expand<DIG_LEVELS>(cb[0], bb[0]);
        if (!half) {
          dig_expand<DIG_LEVELS>(ta[4], a[2]);
          dig_expand<DIG_LEVELS>(low ? ta[8 * TS + 4] : zero, a[3]);
          dig_expand<DIG_LEVELS>(cb[4 * CS], bb[1]);
        }
        dig_block(acc, a, bb, half);
      }
#pragma unroll
      for (int k = 0; k < 4; k++) {
        x0[k] = x[k];
        x[k] = small_h ? dig_drain_small(acc, k) : dig_drain(acc, k);
      }
    }
    // pairs of neighbouring columns (results of T's padded columns are zero, as the layout's padding)
    const int c = n0 + 2 * q, H4 = formed_width(H);
    auto put = [&](Out* o, const DigSum& y, const DigSum& z) {
      struct __align__(16) Two {
        Out a, b;
      };
      *reinterpret_cast<Two*>(o) = Two{dig_result<Out>(y, p2), dig_result<Out>(z, p2)};
    };
#pragma unroll
    for (int k = 0; k < 4; k += 2) {
      const int r = m0 + g + 4 * k;
      if (r >= R || c >= H4) continue;
      Out* o = xq + it.to + r * H4 + c;
      if constexpr (NM == 1) {
        put(o, x[k], x[k + 1]);
      } else {
        auto sum = [&](int e) { return DigSum{x0[e].hi + x[e].hi, x0[e].lo + x[e].lo}; };
        auto dif = [&](int e) { return DigSum{x0[e].hi - x[e].hi, x0[e].lo - x[e].lo}; };
        put(o, sum(k), sum(k + 1));
        put(o + R * H4, dif(k), dif(k + 1));
      }
    }
  }
}

// Channels of at most PH_TINY_DIM (FP32-pair results) or PH_TINY_FP64 (FP64 results) rows and
// columns per problem, one warp each, in the element arithmetic of the results, the pairs from the
// pair copy of the amplitudes: a 7 x 7 problem would fill a fifth of a 16 x 8 x 8 block.  120 systems
// of N = 14, all of whose channels are of this size: 695 us per launch in digits, 145 here (355 with
// one gather loop per channel in the kernel of the larger channels, at its registers).  In FP64 the
// line lies lower where larger channels take the digit kernel anyway, the products then share the
// slow pipe: 28 nucleons, n^2 <= 20, take 94 us per update with a line at 5 and 99 with one at 8.
// fixed: W [problem][row][column] then <kb|v|cj> [problem][row][column] of the channel.
template <typename T_>
__device__ __forceinline__ void ph_tiny(const DevState& D, const PhItem& it, T_* Ts,
                                        const T_* __restrict__ t, const int* __restrict__ src,
                                        const T_* __restrict__ fixed, bool quad, T_* __restrict__ xq) {
  using A = Arith<T_>;
  constexpr int S = PH_TINY_DIM;
  const int lane = threadIdx.x & 31, R = it.R, H = it.H, nm = it.nm;
  T_* Ws = Ts + 2 * S * S;  // [problem][row][column], as Ts
  T_* Cs = Ws + 2 * S * S;
  const T_* __restrict__ W = fixed + it.fx;
  const T_* __restrict__ V1 = W + nm * R * H;
  const int* __restrict__ sp = src + it.src;
  auto read = [&](int c) {
    if (c == 0) return A::zero();
    const T_ v = t[c > 0 ? c - 1 : -c - 1];
    return c < 0 ? A::neg(v) : v;
  };
  for (int e = lane; e < R * H; e += 32) {
    const int u = e / H, c = e - u * H, k8 = u * ph_h8(H) + c;
    if (nm == 2) {
      const int2 k = reinterpret_cast<const int2*>(sp)[k8];
      const T_ x = read(k.x), y = read(k.y);
      Ts[u * S + c] = A::add(x, y);
      Ts[S * S + u * S + c] = A::sub(x, y);
      if (quad) Ws[S * S + u * S + c] = W[R * H + e];
    } else {
      Ts[u * S + c] = read(sp[k8]);
    }
    if (quad) Ws[u * S + c] = W[e];
  }
  __syncwarp();
  for (int e = lane; e < nm * H * H; e += 32) {
    const int m = e >= H * H, f = e - m * H * H, r = f / H, c = f - r * H;
    T_ acc = A::zero();
    for (int u = 0; u < R && quad; u++) A::mac(acc, Ws[m * S * S + u * S + r], Ts[m * S * S + u * S + c]);
    Cs[m * S * S + r * S + c] = A::add(V1[e], A::half(acc));
  }
  __syncwarp();
  for (int e = lane; e < R * H; e += 32) {
    const int r = e / H, c = e - r * H;
    T_ acc[2] = {A::zero(), A::zero()};
    for (int m = 0; m < nm; m++)
      for (int u = 0; u < H; u++) A::mac(acc[m], Ts[m * S * S + r * S + u], Cs[m * S * S + u * S + c]);
    T_* q = xq + it.to + r * formed_width(H) + c;
    if (nm == 2) {
      *q = A::half(A::add(acc[0], acc[1]));
      q[R * formed_width(H)] = A::half(A::sub(acc[0], acc[1]));
    } else {
      *q = acc[0];
    }
  }
}

// The first nblk CTAs take one channel each (the costliest first), the others PH_WARPS small
// channels each, one per warp (stride warp_smem bytes of shared memory).
template <typename Out>
__global__ void __launch_bounds__(PH_THREADS, 3) k_ph_dig(DevState D, const LoopCtl* __restrict__ ctl,
                                                          const PhItem* __restrict__ items, const int2* __restrict__ exps,
                                                          int nblk, int nwarp, int warp_smem, const int* __restrict__ src,
                                                          const uint4* __restrict__ wf, const long long* __restrict__ v1,
                                                          int quad, Out* __restrict__ xq) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ __align__(4) unsigned char marks[4 * PH_MAX_DIM];
  __shared__ int sh_max[PH_WARPS];
  const double* __restrict__ t = cur_t(D, ctl);
  if ((int)blockIdx.x < nblk) {
    const PhItem it = items[blockIdx.x];
    if (sys_done(D, ctl, it.sys)) return;  // CTA-uniform
    const int2 ex = exps[blockIdx.x];
    if (it.nm == 2) ph_dig<Out, PH_THREADS, 2>(D, it, ex, smraw, t, src, wf, v1, quad != 0, xq, marks, sh_max);
    else ph_dig<Out, PH_THREADS, 1>(D, it, ex, smraw, t, src, wf, v1, quad != 0, xq, marks, sh_max);
    return;
  }
  const int w = threadIdx.x >> 5, idx = ((int)blockIdx.x - nblk) * PH_WARPS + w;
  if (idx >= nwarp) return;  // whole warps; the warp path never synchronises the block
  const PhItem it = items[nblk + idx];
  if (sys_done(D, ctl, it.sys)) return;
  const int2 ex = exps[nblk + idx];
  unsigned char* sm = smraw + (size_t)w * warp_smem;
  unsigned char* mk = marks + w * 4 * PH_WARP_DIM;
  if (it.nm == 2) ph_dig<Out, 32, 2>(D, it, ex, sm, t, src, wf, v1, quad != 0, xq, mk, sh_max);
  else ph_dig<Out, 32, 1>(D, it, ex, sm, t, src, wf, v1, quad != 0, xq, mk, sh_max);
}

// The smallest channels, one warp each, in a kernel of their own: it needs a third of the registers.
template <typename T_>
__global__ void __launch_bounds__(PH_THREADS) k_ph_tiny(DevState D, const LoopCtl* __restrict__ ctl,
                                                        const PhItem* __restrict__ items, int n,
                                                        const int* __restrict__ src, const T_* __restrict__ fixed,
                                                        const f2* __restrict__ tpair, int quad, T_* __restrict__ xq) {
  __shared__ __align__(16) T_ sm[PH_WARPS][6 * PH_TINY_DIM * PH_TINY_DIM];
  const int w = threadIdx.x >> 5, idx = blockIdx.x * PH_WARPS + w;
  if (idx >= n) return;  // whole warps; no block barrier
  const PhItem it = items[idx];
  if (sys_done(D, ctl, it.sys)) return;
  const T_* __restrict__ t;
  if constexpr (std::is_same<T_, f2>::value) t = tpair;
  else t = cur_t(D, ctl);
  ph_tiny<T_>(D, it, sm[w], t, src, fixed, quad != 0, xq);
}

// The fixed operands of the items (one CTA each): source indices (rows padded to H8), <kb|v|cj> of
// the problems as integers (padded to whole blocks) and the digits of W, with their exponents
// (DIG_NONFINITE where a row or column lies too far below the largest element).
__global__ void __launch_bounds__(128) k_ph_pack(DevState D, const PhItem* __restrict__ items, int2* __restrict__ exps,
                                                 int* __restrict__ src, uint4* __restrict__ wf, long long* __restrict__ v1,
                                                 double* __restrict__ fixed64, f2* __restrict__ fixed_f2) {
  __shared__ int top[2];
  __shared__ __align__(4) unsigned char marks[2][4 * PH_MAX_DIM];
  const PhItem it = items[blockIdx.x];
  const int R = it.R, H = it.H, H8 = ph_h8(H), H4 = formed_width(H), RW = R * H4, HW = H * H4;
  const double* __restrict__ W = D.x_w + it.to;
  const double* __restrict__ V = D.x_v1 + it.vo;
  const int* __restrict__ map = D.xmap + it.to;
  const bool two = it.nm == 2;
  const bool tiny = max(R, H) <= PH_TINY_DIM;  // element values too
  auto put = [&](long o, double v) {
    fixed64[it.fx + o] = v;
    fixed_f2[it.fx + o] = Arith<f2>::from_double(v);
  };
  const PhMarks mw{marks[0], PH_MAX_DIM}, mv{marks[1], PH_MAX_DIM};
  for (int k = threadIdx.x; k < 8 * PH_MAX_DIM; k += blockDim.x) marks[0][k] = 0;
  if (threadIdx.x < 2) top[threadIdx.x] = 1;
  __syncthreads();
  int e = 1;
  for (int f = threadIdx.x; f < R * H8; f += blockDim.x) {
    const int u = f / H8, s = f % H8, o = u * H4 + s;
    const bool in = s < H;
    if (two) reinterpret_cast<int2*>(src + it.src)[f] = in ? make_int2(map[o], map[RW + o]) : make_int2(0, 0);
    else src[it.src + f] = in ? map[o] : 0;
    if (!in) continue;
    const double a = W[o], b = two ? W[RW + o] : 0.0;
    e = max(e, max(dig_exp(a), dig_exp(b)));
    if (tiny) {
      put(u * H + s, a + b);
      if (two) put(R * H + u * H + s, a - b);
    }
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) atomicMax(&top[0], e);
  e = 1;
  for (int f = threadIdx.x; f < H * H; f += blockDim.x) {
    const int o = (f / H) * H4 + f % H;
    const double a = V[o], b = two ? V[HW + o] : 0.0;
    e = max(e, max(dig_exp(a), dig_exp(b)));
    if (tiny) {
      put(it.nm * R * H + f, a + b);
      if (two) put(2 * R * H + H * H + f, a - b);
    }
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) atomicMax(&top[1], e);
  __syncthreads();
  const int ew = top[0], ev = top[1];
  auto span = [&](const PhMarks& m, const double* __restrict__ M, int rows, int n, int least) {
    for (int f = threadIdx.x; f < rows * H; f += blockDim.x) {
      const int u = f / H, s = f % H, o = u * H4 + s, x = max(size_of(M[o]), two ? size_of(M[n + o]) : 0);
      m.set(u, x, least);
      m.set(m.n + s, x, least);
    }
  };
  span(mw, W, R, RW, least_size(ew));
  span(mv, V, H, HW, least_size(ev));
  __syncthreads();
  const bool low = __syncthreads_or((int)threadIdx.x < PH_MAX_DIM / 2 && (mw.low(threadIdx.x) || mv.low(threadIdx.x)));
  if (threadIdx.x == 0) exps[blockIdx.x] = low ? make_int2(DIG_NONFINITE, DIG_NONFINITE) : make_int2(ew, ev);
  if (low || ew >= DIG_NONFINITE || ev >= DIG_NONFINITE) return;
  const int sc = (H + 15) >> 4, kr = (R + 15) >> 4;
  for (int f = threadIdx.x; f < sc * 16 * H8; f += blockDim.x) {
    const int r = f / H8, c = f % H8;
    long long a = 0, b = 0;
    if (r < H && c < H) {
      a = dig_fixed(V[r * H4 + c], ev);
      if (two) b = dig_fixed(V[HW + r * H4 + c], ev);
    }
    v1[it.v1 + f] = a + b;
    if (two) v1[it.v1 + (long)sc * 16 * H8 + f] = a - b;
  }
  // fragment order of W as the first operand: rows (k,c), columns (e,l); stored transposed in x_w
  for (int f = threadIdx.x; f < sc * kr * 128; f += blockDim.x) {
    const int lane = f & 31, grp = (f >> 5) & 3, ks = (f >> 7) % kr, strip = (f >> 7) / kr;
    const int r = strip * 16 + (lane >> 2) + (grp & 1) * 8, u0 = ks * 16 + (lane & 3) * 2 + (grp >> 1) * 8;
    long long a[2] = {0, 0}, b[2] = {0, 0};
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const int u = u0 + k;
      if (r >= H || u >= R) continue;
      a[k] = dig_fixed(W[u * H4 + r], ew);
      if (two) b[k] = dig_fixed(W[RW + u * H4 + r], ew);
    }
    wf[it.wf + f] = dig_interleave(dig_word(a[0] + b[0]), dig_word(a[1] + b[1]));
    if (two) wf[it.wf + (long)sc * kr * 128 + f] = dig_interleave(dig_word(a[0] - b[0]), dig_word(a[1] - b[1]));
  }
}

// Items of the ph launches (once per context, on first use): the channels that take a CTA, costliest
// first, those whose digit tiles need more than PH_DIG_SMEM bytes before the others (a launch of their
// own, so that the others keep three CTAs per SM); then the warp path by decreasing dimension, so that
// the tiny channels of every result type are its end.
constexpr size_t PH_DIG_SMEM = 72 * 1024;
void pnm_need_ph_items(pnm_ctx* ctx) {
  if (ctx->ph_items) return;
  cudaStream_t s = ctx->stream;
  // by cost in quarter octaves (a sort by the exact cost of 2500 channels took longer than the launch)
  constexpr int COSTS = 4 * 64;
  std::vector<int> by_dim[PH_WARP_DIM + 1], by_cost[2][COSTS];  // large channels first
  auto problems = [&](int x) { return ctx->h_x_cls[x] == 0 ? 2 : 1; };
  bool larger = false;  // than the tiny kernels take
  for (int x = 0; x < ctx->nx; x++) {
    if (ctx->h_x_cls[x] < 0) continue;
    const int nm = problems(x), R = ctx->h_x_nph[x] / nm, H = ctx->h_x_nhp[x] / nm, dim = std::max(R, H);
    larger = larger || dim > PH_TINY_DIM;
    if (dim <= PH_WARP_DIM) {
      by_dim[dim].push_back(x);
    } else {
      const unsigned long cost = 4UL * nm * R * H * H;  // at least 4: two bits below the leading one
      const int top = 63 - __builtin_clzl(cost);
      by_cost[ph_dig_smem(R, H, nm) > PH_DIG_SMEM ? 0 : 1][4 * top + (int)((cost >> (top - 2)) & 3)].push_back(x);
    }
  }
  std::vector<PhItem> items;
  items.reserve(ctx->nx);
  unsigned long wf = 0, v1 = 0, src = 0, fixed = 0;
  size_t dig = 0, f32 = 0;  // shared memory of the last item
  auto add = [&](int x) {
    PhItem it{};
    const int nm = problems(x), R = ctx->h_x_nph[x] / nm, H = ctx->h_x_nhp[x] / nm;
    it.x = x;
    it.sys = ctx->h_x_sys[x];
    it.nm = (unsigned short)nm;
    it.R = (unsigned short)R;
    it.H = (unsigned short)H;
    it.to = (unsigned)ctx->h_x_t_off[x];
    it.vo = (unsigned)ctx->h_x_c_off[x];
    it.src = (unsigned)src;
    it.wf = (unsigned)wf;
    it.v1 = (unsigned)v1;
    it.fx = (unsigned)fixed;
    src += (unsigned long)nm * R * ph_h8(H);
    wf += (unsigned long)nm * ((H + 15) / 16) * ((R + 15) / 16) * 128;
    v1 += (unsigned long)nm * ((H + 15) / 16) * 16 * ph_h8(H);
    if (std::max(R, H) <= PH_TINY_DIM) fixed += (unsigned long)nm * H * (R + H);
    items.push_back(it);
    dig = (ph_dig_smem(R, H, nm) + 15) / 16 * 16;
    f32 = (ph32_smem(R, H, nm) + 15) / 16 * 16;
  };
  ctx->n_ph_large = ctx->n_ph_cta = ctx->n_ph_warp = ctx->n_ph_tiny = ctx->n_ph_tiny64 = 0;
  ctx->ph_large_smem = ctx->ph_dig_smem = ctx->ph_warp_smem = ctx->ph32_smem = ctx->ph32_warp_smem = 0;
  for (int small = 0; small < 2; small++) {
    size_t& most = small ? ctx->ph_dig_smem : ctx->ph_large_smem;
    for (int k = COSTS - 1; k >= 0; k--)
      for (int x : by_cost[small][k]) {
        add(x);
        (small ? ctx->n_ph_cta : ctx->n_ph_large)++;
        most = std::max(most, dig);
        ctx->ph32_smem = std::max(ctx->ph32_smem, f32);
      }
  }
  // FP64 results: where no channel is larger than PH_TINY_DIM all take the tiny kernel, which saves
  // the passes that make the digits (N = 14: the operator call 96 -> 73 us, a solve of one
  // n^2 <= 24 system 955 -> 852 us, of sixteen 4.82 -> 4.22 ms); beside larger channels the digit
  // kernel is the faster one from PH_TINY_FP64 + 1 on.
  const int tiny64 = larger ? PH_TINY_FP64 : PH_TINY_DIM;
  for (int d = PH_WARP_DIM; d >= 0; d--) {
    const int n = (int)by_dim[d].size();
    for (int x : by_dim[d]) {
      add(x);
      if (d > tiny64) ctx->ph_warp_smem = std::max(ctx->ph_warp_smem, dig);
      if (d > PH_TINY_DIM) ctx->ph32_warp_smem = std::max(ctx->ph32_warp_smem, f32);
    }
    ctx->n_ph_warp += n;
    if (d <= PH_TINY_DIM) ctx->n_ph_tiny += n;
    if (d <= tiny64) ctx->n_ph_tiny64 += n;
  }
  if (std::max(std::max(wf, v1), std::max(src, fixed)) >= (1UL << 32))
    throw PnmError{PNM_EINVAL, "problem too large for 32-bit element maps"};
  ctx->ph_dig_smem = std::max(ctx->ph_dig_smem, PH_WARPS * ctx->ph_warp_smem);
  ctx->ph_sizes[0] = (long)src;
  ctx->ph_sizes[1] = (long)wf;
  ctx->ph_sizes[2] = (long)v1;
  ctx->ph_sizes[3] = (long)fixed;
  ctx->n_ph_items = (int)items.size();
  PhItem* d = ctx_alloc<PhItem>(ctx, items.size());
  if (!items.empty())
    CUDA_TRY(cudaMemcpyAsync(d, items.data(), sizeof(PhItem) * items.size(), cudaMemcpyHostToDevice, s));
  smem_at_least(k_ph32, std::max(ctx->ph32_smem, PH_WARPS * ctx->ph32_warp_smem));
  ctx->ph_items = d;
}

// Fixed operands of the digit ph term (once per context, on first use).
void pnm_need_phdig(pnm_ctx* ctx) {
  if (ctx->ph_exps) return;
  pnm_need_ph_items(ctx);
  cudaStream_t s = ctx->stream;
  ctx->ph_src = ctx_alloc<int>(ctx, ctx->ph_sizes[0]);
  ctx->ph_wf = ctx_alloc<uint4>(ctx, ctx->ph_sizes[1]);
  ctx->ph_v1 = ctx_alloc<long long>(ctx, ctx->ph_sizes[2]);
  ctx->ph_fixed64 = ctx_alloc<double>(ctx, ctx->ph_sizes[3]);
  ctx->ph_fixed_f2 = ctx_alloc<f2>(ctx, ctx->ph_sizes[3]);
  int2* exps = ctx_alloc<int2>(ctx, ctx->n_ph_items);
  if (ctx->n_ph_items > 0)
    k_ph_pack<<<ctx->n_ph_items, 128, 0, s>>>(ctx->d, ctx->ph_items, exps, ctx->ph_src, ctx->ph_wf, ctx->ph_v1,
                                              ctx->ph_fixed64, ctx->ph_fixed_f2);
  CUDA_TRY(cudaGetLastError());
  const size_t most = std::max(ctx->ph_large_smem, ctx->ph_dig_smem);
  smem_at_least(k_ph_dig<double>, most);
  smem_at_least(k_ph_dig<f2>, most);
  ctx->ph_exps = exps;
}

template <typename Out>
static void launch_ph_dig(pnm_ctx* ctx, bool linear, cudaStream_t s, cudaStream_t s_tiny) {
  // made before any capture by the host-side callers
  if (!ctx->ph_exps) throw PnmError{PNM_EINVAL, "the ph term's operands have not been built"};
  constexpr bool pair = std::is_same<Out, f2>::value;
  const int nl = ctx->n_ph_large, n = ctx->n_ph_cta, ntiny = pair ? ctx->n_ph_tiny : ctx->n_ph_tiny64, nw = ctx->n_ph_warp - ntiny;
  const int nwb = (nw + PH_WARPS - 1) / PH_WARPS, quad = linear ? 0 : 1;
  Out* xq = reinterpret_cast<Out*>(ctx->d.xq);
  const PhItem* items = ctx->ph_items;
  if (nl + n + nw == 0) s_tiny = s;
  if (nl > 0)
    k_ph_dig<Out><<<nl, PH_THREADS, ctx->ph_large_smem, s>>>(ctx->d, ctx->ctl, items, ctx->ph_exps, nl, 0, 0, ctx->ph_src,
                                                             ctx->ph_wf, ctx->ph_v1, quad, xq);
  if (n + nwb > 0)
    k_ph_dig<Out><<<n + nwb, PH_THREADS, ctx->ph_dig_smem, s>>>(ctx->d, ctx->ctl, items + nl, ctx->ph_exps + nl, n, nw,
                                                                (int)ctx->ph_warp_smem, ctx->ph_src, ctx->ph_wf,
                                                                ctx->ph_v1, quad, xq);
  if (ntiny > 0) {
    const Out* fixed;
    if constexpr (pair) fixed = ctx->ph_fixed_f2;
    else fixed = ctx->ph_fixed64;
    k_ph_tiny<Out><<<(ntiny + PH_WARPS - 1) / PH_WARPS, PH_THREADS, 0, s_tiny>>>(
        ctx->d, ctx->ctl, items + nl + n + nw, ntiny, ctx->ph_src, fixed, ctx->t_pair, quad, xq);
  }
}

// FP64 ph term (linear: without the quadratic part), and the same with its results as FP32 pairs
// in the 8-byte slots of the FP64 Q (the refinement sweeps with FP32-pair contractions).
// s_tiny: the stream of the smallest channels (beside larger ones a stream of their own; in a context
// without larger channels they keep s).
void launch_ph64(pnm_ctx* ctx, cudaStream_t s, cudaStream_t s_tiny, bool linear) {
  launch_ph_dig<double>(ctx, linear, s, s_tiny);
}
void launch_ph_f2(pnm_ctx* ctx, cudaStream_t s, cudaStream_t s_tiny) { launch_ph_dig<f2>(ctx, false, s, s_tiny); }

// The kernels of the term, for the priorities of a captured update's nodes.
bool pnm_is_ph_kernel(const void* f) {
  return f == (const void*)k_ph32 || f == (const void*)k_ph32_tiny || f == (const void*)k_ph_dig<double> ||
         f == (const void*)k_ph_dig<f2> || f == (const void*)k_ph_tiny<double> || f == (const void*)k_ph_tiny<f2>;
}
