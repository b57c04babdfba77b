// iterate.cu -- one CCD update, Eq. (ccd3) of arXiv:1611.06765 written with the
// intermediates of Sec. "Developing a CCD code":
//
//   0 = v_ab^ij + P(ab) chi_b^c t_ac^ij - P(ij) chi_k^j t_ab^ik + 1/2 <ab|chi|cd> t_cd^ij
//       + 1/2 t_ab^kl <kl|chi|ij> + P(ij)P(ab) t_ik^ac <kb|chi|cj>
//
// with chi_b^c, chi_k^j diagonal here (momentum and S_z conservation), blocked per direct
// channel (restricted pairs) and per cross channel (ordered ph/hp pairs).  Kernels:
//   k_tstats   row and column sums of t o v (one-body intermediates) and
//              <kl|chi|ij> = <kl|v|ij> + 1/2 <kl|v|cd> t_ij^cd per direct channel
//   k_dchi     chi_p - eps_p per state, gathered over the pairs holding p
//   k_tdig, k_pp   1/2 sum_cd <ab|v|cd> t_cd^ij, grouped over all channels with a V_pppp block (FP64
//              accuracy from digit products on the tensor cores)
//   k_update, k_update_mix   Jacobi step t_new = (v + rest) / eps_ij^ab, mixing, energy/residual
//              partials, and by the last block of each system its end (Eq. ccdcorr energy, |dE| test)
//              and the device-side loop condition
//   k_mbpt2, k_mbpt3   start amplitudes and MBPT2 energy, third-order sums
// The ph term is in ph.cu, the tensor-core ladder and the FP32 copies of the mixed iteration in mixed.cu.
#include <cmath>
#include <cstdio>
#include <map>
#include <algorithm>
#include <chrono>
#include <mutex>
#include <type_traits>

#include "dig.cuh"
#include "pnm_context.cuh"

#ifndef PNM_UPD_HH_UNROLL
#define PNM_UPD_HH_UNROLL 4
#endif
constexpr int UPD_MIX_UNROLL = 2;  // chunks of a warp of the mixed update in flight
constexpr int UPD_HH_UNROLL = PNM_UPD_HH_UNROLL;  // loads of the mixed update's hh-ladder pass in flight


// ----------------------------------------------------------------------------- stats
// Element type T_: double for the FP64 iteration (t, v_pphh, v_hhhh, chi_hh, sij, sab), float
// for the mixed-precision one (their FP32 copies).
template <typename T_>
struct StatsIO {
  const T_ *t, *v, *vhh;
  T_ *chi, *sij, *sab;
  __device__ StatsIO(const DevState& D, const LoopCtl* ctl) {
    if constexpr (std::is_same<T_, double>::value) {
      t = cur_t(D, ctl); v = D.v_pphh; vhh = D.v_hhhh; chi = D.chi_hh; sij = D.sij; sab = D.sab;
    } else {
      t = cur_t32(D, ctl); v = D.v32; vhh = D.vhh32; chi = D.chi32; sij = D.sij32; sab = D.sab32;
    }
  }
};

// One warp per item (channel, row kl, first column, 0): up to STAT_COLS sums over the row v_kl, read
// once for all of them: column 0 is sij[kl] = sum_ab t_kl v_kl, column j > 0 chi[kl][ij] of the j-th hole
// pair ij the updates compute.  Items (channel, -1, ab0, 0): sab[ab] = sum_ij t v of 32 columns.
// Bound by latency (a CTA per row and per 128 columns, most of whose threads idled in small channels,
// took 38 us for 120 N=14 systems in FP32, 28 so) and in FP64 by the slow pipe: the four sums of
// a warp share the exchanges, six additions instead of twenty (N=66, N_max=42: 47, 45 us).
// PAIR (FP64 only): the contractions in FP32-pair arithmetic from the pair copies tp of t and vp
// of v_pphh (the refinement sweeps): chi_hh, and the one-body sums as per-thread pair partials
// added in FP64.
constexpr int STAT_COLS = 4;
template <typename T_, bool PAIR = false>
__global__ void __launch_bounds__(128) k_tstats(DevState D, const LoopCtl* __restrict__ ctl,
                                                const int4* __restrict__ items, int n,
                                                const f2* __restrict__ tp = nullptr,
                                                const f2* __restrict__ vp = nullptr) {
  using E = std::conditional_t<PAIR, f2, T_>;
  using A = Arith<E>;
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (w >= n) return;  // whole warps; no block barrier
  const int4 it = items[w];
  const int c = it.x, kl = it.y;
  if (sys_done(D, ctl, D.ch_sys[c])) return;
  StatsIO<T_> io(D, ctl);
  const int npp = D.ch_npp[c], nh = D.ch_nhh[c];
  const long base = D.ch_t_off[c];
  const E *t, *v;
  if constexpr (PAIR) {
    t = tp + base;
    v = vp + base;
  } else {
    t = io.t + base;
    v = io.v + base;
  }
  if (kl < 0) {
    const int ab = it.z + lane;
    if (ab >= npp) return;
    E s = A::zero();
#pragma unroll 4
    for (int ij = 0; ij < nh; ij++) A::mac(s, t[ab + (long)ij * npp], v[ab + (long)ij * npp]);
    if constexpr (PAIR) io.sab[D.ch_pp_off[c] + ab] = A::to_double(s);
    else io.sab[D.ch_pp_off[c] + ab] = s;
    return;
  }
  const int* __restrict__ rl = D.upd_row + D.ch_uoff[c];
  const int m = min(STAT_COLS, D.ch_uoff[c + 1] - D.ch_uoff[c] + 1 - it.z);
  const E* __restrict__ vr = v + (long)kl * npp;
  const E* col[STAT_COLS];
#pragma unroll
  for (int q = 0; q < STAT_COLS; q++) {
    const int k = it.z + min(q, m - 1);
    col[q] = t + (long)(k == 0 ? kl : rl[k - 1]) * npp;
  }
  E acc[STAT_COLS];
#pragma unroll
  for (int q = 0; q < STAT_COLS; q++) acc[q] = A::zero();
#pragma unroll 2
  for (int cd = lane; cd < npp; cd += 32) {
    const E x = vr[cd];
#pragma unroll
    for (int q = 0; q < STAT_COLS; q++)
      if (q < m) A::mac(acc[q], x, col[q][cd]);
  }
  if (PAIR && it.z == 0) {
    const double s = warp_sum((double)A::to_double(acc[0]));
    if (lane == 0) io.sij[D.ch_hh_off[c] + kl] = s;
  }
  // the sums of columns 0 ... 3 end in lanes 0-7, 8-15, 16-23, 24-31
  auto exchange = [&](E keep, E give, int o) {
    E got;
    if constexpr (PAIR) got = f2{__shfl_xor_sync(0xffffffffu, give.hi, o), __shfl_xor_sync(0xffffffffu, give.lo, o)};
    else got = __shfl_xor_sync(0xffffffffu, give, o);
    return A::add(keep, got);
  };
  const bool h16 = lane & 16, h8 = lane & 8;
  const E x0 = exchange(h16 ? acc[2] : acc[0], h16 ? acc[0] : acc[2], 16);
  const E x1 = exchange(h16 ? acc[3] : acc[1], h16 ? acc[1] : acc[3], 16);
  E x = exchange(h8 ? x1 : x0, h8 ? x0 : x1, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) x = exchange(x, x, o);
  const int q = lane >> 3, k = it.z + q;
  if ((lane & 7) != 0 || q >= m) return;
  if (k == 0) {
    if constexpr (!PAIR) io.sij[D.ch_hh_off[c] + kl] = x;
    return;
  }
  const long e = D.ch_vhh_off[c] + (long)kl * nh + rl[k - 1];
  // the pair update reads chi as pairs, in the same 8-byte slots
  if constexpr (PAIR) reinterpret_cast<f2*>(io.chi)[e] = A::from_double(io.vhh[e] + A::to_double(x));
  else io.chi[e] = io.vhh[e] + x;
}

// chi_b - eps_b = -sum_d sum_{k<l} t_kl^bd v_kl^bd   (particles)
// chi_j - eps_j = +sum_l sum_{c<d} v_jl^cd t_jl^cd   (holes)
template <typename T_>
__global__ void k_dchi(DevState D, int nsp_total) {
  int p = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  int lane = threadIdx.x & 31;
  if (p >= nsp_total) return;
  constexpr bool F64 = std::is_same<T_, double>::value;
  int lo = D.occ_off[p], hi = D.occ_off[p + 1];
  bool hole = D.sp_hole[p] != 0;
  const T_* src;
  if constexpr (F64) src = hole ? D.sij : D.sab;
  else src = hole ? D.sij32 : D.sab32;
  T_ s = 0;
  for (int k = lo + lane; k < hi; k += 32) s += src[D.occ_idx[k]];
  s = warp_sum(s);
  if (lane == 0) {
    if constexpr (F64) D.dchi[p] = hole ? s : -s;
    else D.dchi32[p] = hole ? s : -s;
  }
}

// ------------------------------------------------------------------------ ladder basis
// s(ij, q) = sum over the (one or two) pairs of vector q of sign * t(ij, pair) from the current
// FP64 amplitudes, as digit words of the row's common exponent (dig.cuh), zero words in the
// padding.  One CTA per (channel, ij) row of a channel with V_pppp.  A row that holds an infinity
// or a NaN has the exponent DIG_NONFINITE (the ladder kernel then sums it in FP64).  s64: s itself too,
// in the ladder layout, where the ladder checks its results (else null).
constexpr int TDIG_THREADS = 128;
__global__ void __launch_bounds__(TDIG_THREADS) k_tdig(DevState D, const LoopCtl* __restrict__ ctl,
                                                       const int2* __restrict__ rows, double* __restrict__ s64) {
  extern __shared__ double ssum[];
  __shared__ int warp_max[TDIG_THREADS / 32];
  __shared__ unsigned sh_top;
  const int2 it = rows[blockIdx.x];
  const int c = it.x, ij = it.y;
  if (sys_done(D, ctl, D.ch_sys[c])) return;
  const int npp = D.ch_npp[c], nl = D.ch_nlad[c], off = D.ch_pp_off[c];
  const double* __restrict__ tr = cur_t(D, ctl) + D.ch_t_off[c] + (long)ij * npp;
  int e = 1;
  for (int q = threadIdx.x; q < nl; q += TDIG_THREADS) {
    const int2 m = D.lad_mem[off + q];
    const double a = tr[(m.x > 0 ? m.x : -m.x) - 1];
    double v = m.x > 0 ? a : -a;
    if (m.y != 0) {
      const double b = tr[(m.y > 0 ? m.y : -m.y) - 1];
      v += m.y > 0 ? b : -b;
    }
    ssum[q] = v;
    if (s64) s64[D.ch_s_off[c] + (long)ij * nl + q] = v;
    e = max(e, dig_exp(v));
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = e;
  if (threadIdx.x == 0) sh_top = 0;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < TDIG_THREADS / 32; w++) e = max(e, warp_max[w]);
  unsigned top = 0;
  const int steps = (nl + 15) >> 4;
  uint4* o = reinterpret_cast<uint4*>(D.tdig + D.ch_td_off[c]) + (long)ij * steps * 16;
  if (threadIdx.x == 0) D.texp[D.ch_hh_off[c] + ij] = e;
  // per 16-element step and quarter t the elements 2t, 2t + 1, 2t + 8, 2t + 9: the two registers
  // of the product's column operand for every digit, 64 bytes
  for (int f = threadIdx.x; f < steps * 4; f += TDIG_THREADS) {
    const int k0 = (f >> 2) * 16 + (f & 3) * 2;
    double v[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const int q = k0 + (u & 1) + (u >> 1) * 8;
      v[u] = q < nl ? ssum[q] : 0.0;
    }
    long long x[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      x[u] = dig_fixed(v[u], e);
      top = max(top, dig_top(x[u]));
    }
    uint32_t b0[8], b1[8];
    dig_expand<8>(dig_interleave(dig_word(x[0]), dig_word(x[1])), b0);
    dig_expand<8>(dig_interleave(dig_word(x[2]), dig_word(x[3])), b1);
#pragma unroll
    for (int u = 0; u < 4; u++) o[f * 4 + u] = make_uint4(b0[2 * u], b1[2 * u], b0[2 * u + 1], b1[2 * u + 1]);
  }
  top = __reduce_max_sync(0xffffffffu, top);
  if ((threadIdx.x & 31) == 0) atomicMax(&sh_top, top);
  __syncthreads();
  if (threadIdx.x == 0) D.ttop[D.ch_hh_off[c] + ij] = sh_top;
}

// FP32-pair copy of the current amplitudes (the start of a sweep with FP32-pair contractions).
__global__ void k_split_cur(DevState D, const LoopCtl* __restrict__ ctl, f2* __restrict__ tp, long n) {
  long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) tp[i] = Arith<f2>::from_double(cur_t(D, ctl)[i]);
}

void pnm_split_cur(pnm_ctx* ctx, cudaStream_t s) {
  if (ctx->nt > 0)
    k_split_cur<<<(unsigned)((ctx->nt + 255) / 256), 256, 0, s>>>(ctx->d, ctx->ctl, ctx->t_pair, ctx->nt);
}

// The pp ladder in the amplitude layout, from its ladder-layout value (planes summed): zero in
// channels without V_pppp.  One CTA per (channel, ij) row.
template <typename T_>
__global__ void __launch_bounds__(128) k_lad_expand(DevState D, const T_* __restrict__ rs, int planes,
                                                    long pstride, double* __restrict__ out) {
  using A = Arith<T_>;
  int2 it = D.row_item[blockIdx.x];
  int c = it.x, ij = it.y;
  int npp = D.ch_npp[c];
  bool vpp = D.ch_vpp[c] != 0;
  double* o = out + D.ch_t_off[c] + (long)ij * npp;
  for (int ab = threadIdx.x; ab < npp; ab += blockDim.x) {
    double v = 0.0;
    if (vpp) {
      int sg;
      long z = lad_index(D, c, ij, ab, sg);
      T_ a = A::zero();
      for (int p = 0; p < planes; p++) a = A::add(a, rs[p * pstride + z]);
      v = sg > 0 ? A::to_double(a) : -A::to_double(a);
    }
    o[ab] = v;
  }
}

// ------------------------------------------------------------------- pp ladder, FP64 accuracy
// R^T(ij, ab) = sum_cd t(ij, cd) <cd|v|ab>, restricted pairs (1/2 sum over ordered cd of a
// pair-antisymmetric product = sum over c<d), in the ladder basis, as digit products on the
// tensor cores (dig.cuh), with FP64 results or FP32-pair ones (the refinement sweeps).
// An item (PPItem) is a strip of 16 rows ab with up to 8 rows ij; wk warps share its columns cd (a
// step of 16 each in turn) and add their integer sums, exactly, through shared memory: strips of
// large channels would otherwise leave most SMs idle at the end (63% of the time busy with one warp
// per strip), and a small system has too few strips to fill the GPU.  V streams in fragment order
// (8 bytes per element); the amplitudes of the rows ij are the eight columns of the product, read
// as FP16 digits.  Every lane copies the operands it reads itself asynchronously into its own part
// of a PP_DEPTH-step ring in shared memory, so that a warp has PP_DEPTH - 1 steps (6 to 12 KB) in
// flight without a barrier (one step ahead in registers held the stream to 2.8 TB/s).
// Most channels have fewer than eight rows to compute (N = 66: 58% of V in channels of at most
// four, symmetric matter 96%), so the columns hold SLOTS digits of 8 / SLOTS rows: slot s of a
// column holds the digits from 8 / SLOTS * s on, and one MMA forms SLOTS levels; 36, 26 and 15
// MMAs per 16 x 16 block of V for up to 8, 4 and 2 rows.
// What bounds it: the V stream for few rows, the tensor pipe (1024 multiply-adds per clock and SM
// through mma.sync) for many.  Per launch with k_tdig (N = 66, n^2 <= 42, FP64): 76 us (V 250 MB in
// 60 us, 4.2 TB/s) against 291 us on the FP64 pipe; symmetric matter, 28 nucleons, n^2 <= 20: 43
// against 119 us; three densities of N = 66, n^2 <= 36, pairs: 125 against 190 us on the FP32 pipe.
constexpr int PP_WARPS = 4, PP_CTAS = 3, PP_DEPTH = 4;  // warps per CTA, CTAs per SM, ring steps
constexpr size_t PP_SMEM = sizeof(uint4) * 256 * PP_DEPTH * PP_WARPS;  // 64 KB: three CTAs per SM
constexpr int PP_MAX_NLAD = 3376;  // ladder basis of a channel (the amplitudes of a row in shared memory)

// The digits leave an error of 2^-59 or so of the product of V's and the row's largest values in every term,
// mostly of the digit products left out, which add up rather than average in channels of high symmetry (P = 0,
// N = 14: to 2^-52).  In ordinary rows that is less than FP64 sums leave, but V and t fall off
// exponentially, and a result all of whose products are small keeps little of them (two neutrons at density
// 0.3, n^2 <= 36, where V falls by 390 octaves: results off by 1e-3 of themselves).  So results PP_FAR
// octaves below the product of the strip's and the row's largest values are summed in FP64 for amplitudes
// given by the caller, where the diagonal term is as small (a tenth of a percent of the results of random
// amplitudes cancel that far: 217 instead of 236 us for the operator of N = 66, n^2 <= 36), and PP_FAR_STEEP below it where the interaction falls by more than PP_STEEP octaves
// over the model space, with V held in FP64 for them (CHECK).  Elsewhere the errors from MBPT2 amplitudes
// are those of FP64 sums (N = 2 to 66, densities 0.02 to 0.3: at most 8e-15 of the sum of absolute products,
// FP64 sums 7e-15), and looking at every result would cost 3% of an update.  Rows or interactions with
// infinities or NaN are summed in FP64 always.  N = 14, density 0.3, n^2 <= 24, FP64: 0.66 ms a solve without
// the check, 0.68 at 8 octaves and 1.1 at 4 (1.4 on the FP64 pipe), errors 1.6e-14, 1.6e-14 and 6.8e-15
// (4.5e-15).
constexpr int PP_FAR = 12, PP_FAR_STEEP = 4;

// Element q of row ab of the ladder-basis V, from the states as every FP64 kernel forms it: mr, ra, rb are
// the row's representative and its states.
__device__ __forceinline__ double lad_v(const DevState& D, const double* __restrict__ lut, int2 pair, int m, int mr,
                                        char4 ra, char4 rb) {
  const double y = v_minnesota_as(D.nvec[pair.x], D.nvec[pair.y], ra, rb, lut);
  return __hiloint2double(__double2hiint(y) ^ ((m ^ mr) & (int)0x80000000), __double2loint(y));
}

// sum_cd t(ij, cd) V(cd, ab) of one result in FP64, by one thread (rows with infinities or NaN in a solve,
// which ends with them); tr: the row's amplitudes.
__device__ __noinline__ double pp_direct(const DevState& D, const double* __restrict__ lut,
                                         const double* __restrict__ tr, int off, int nl, int ab) {
  const int2* __restrict__ mem = D.lad_mem + off;
  const int2* __restrict__ pair = D.pp_pair + off;
  const int mr = mem[ab].x;
  const int2 pr = pair[abs(mr) - 1];
  const char4 ra = D.nvec[pr.x], rb = D.nvec[pr.y];
  double s = 0.0;
  for (int q = 0; q < nl; q++) {
    const int2 m = mem[q];
    double x = tr[abs(m.x) - 1];
    if (m.x < 0) x = -x;
    if (m.y != 0) x += m.y > 0 ? tr[m.y - 1] : -tr[-m.y - 1];
    s = fma(x, lad_v(D, lut, pair[abs(m.x) - 1], m.x, mr, ra, rb), s);
  }
  return s;
}

// Up to four of an item's results, listed in far, by a warp: the rows from the ladder basis (s64), V stored
// where the interaction is steep and many results are taken so (two neutrons, density 0.3, n^2 <= 36: most of
// them), else from the states.  Four share the loads, which are a chain of round trips (one at a time took
// 6 us a result).
template <typename Out>
__device__ __forceinline__ void pp_far(const DevState& D, const PPItem& it, const int* __restrict__ rows,
                                       const double* __restrict__ lut, const double* __restrict__ s64, bool steep,
                                       const unsigned char* __restrict__ far, int n) {
  const int lane = threadIdx.x & 31, nl = it.nl, off = D.ch_pp_off[it.c];
  const int2* __restrict__ mem = D.lad_mem + off;
  const int2* __restrict__ pair = D.pp_pair + off;
  const long base = D.ch_s_off[it.c];
  int ab[4], ij[4];
  double v[4] = {};
#pragma unroll
  for (int u = 0; u < 4; u++) {
    const int f = far[min(u, n - 1)], r = it.n0 + f % 8;
    ab[u] = it.strip * 16 + f / 8;
    ij[u] = rows ? rows[r] : r;
  }
  const double* __restrict__ sc = s64 + base;
  if (steep) {
    const double* __restrict__ vc = D.v64 + D.ch_vd_off[it.c];
    const int wide = (nl + 15) & ~15;
#pragma unroll 2
    for (int q = lane; q < nl; q += 32)
#pragma unroll
      for (int u = 0; u < 4; u++) v[u] = fma(sc[(long)ij[u] * nl + q], vc[(long)ab[u] * wide + q], v[u]);
  } else {
    int mr[4];
    char4 ra[4], rb[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
      mr[u] = mem[ab[u]].x;
      const int2 p = pair[abs(mr[u]) - 1];
      ra[u] = D.nvec[p.x];
      rb[u] = D.nvec[p.y];
    }
#pragma unroll 2
    for (int q = lane; q < nl; q += 32) {
      const int m = mem[q].x;
      const int2 p = pair[abs(m) - 1];
#pragma unroll
      for (int u = 0; u < 4; u++)
        if (u < n) v[u] = fma(sc[(long)ij[u] * nl + q], lad_v(D, lut, p, m, mr[u], ra[u], rb[u]), v[u]);
    }
  }
#pragma unroll
  for (int u = 0; u < 4; u++) {
    const double y = warp_sum(v[u]);
    if (lane == u && u < n) reinterpret_cast<Out*>(D.rpp)[base + (long)ij[u] * nl + ab[u]] = Arith<Out>::from_double(y);
  }
}

// One step of an item's operands into this lane's ring slots: V's four 16-byte groups and the
// Q / 2 groups of FP16 digits.
template <int Q>
__device__ __forceinline__ void pp_copy(uint4* __restrict__ slot, const uint4* __restrict__ vp,
                                        const uint4* __restrict__ tp, int ks) {
  auto cp = [](uint4* dst, const uint4* src) {  // V is read once: L2 only
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
  };
#pragma unroll
  for (int r = 0; r < 4; r++) cp(slot + r * 32, vp + (long)ks * 128 + r * 32);
#pragma unroll
  for (int r = 0; r < Q / 2; r++)  // the amplitudes are shared by the warps of an SM: L1 too
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(slot + (4 + r) * 32)),
                 "l"(tp + (long)ks * 16 + r)
                 : "memory");
}

// part: this warp's place among the wk warps of the item; ring: this warp's steps; red: the sums
// of the item's warps (4 per lane and warp).  t: the channel's amplitudes.  CHECK: returns in the warp of
// part 0 the number of results left to FP64 sums, listed in far (8 row + column).
template <int SLOTS, typename Out, bool CHECK>
__device__ __forceinline__ int pp_pass(const DevState& D, const PPItem& it, const int* __restrict__ rows, int part,
                                       int wk, uint4* __restrict__ ring, DigSum* __restrict__ red,
                                       const double* __restrict__ lut, const double* __restrict__ t0,
                                       const double* __restrict__ s64, bool steep, unsigned char* __restrict__ far) {
  constexpr int Q = 8 / SLOTS;  // rows ij of this pass, and digits per slot
  const int c = it.c, strip = it.strip, nl = it.nl, n0 = it.n0, nr = it.nr;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int steps = (nl + 15) >> 4;
  const uint4* __restrict__ vp = reinterpret_cast<const uint4*>(D.vdig + it.voff) + lane;
  const int rg = min(n0 + g % Q, nr - 1), ijg = rows ? rows[rg] : rg;
  const uint4* __restrict__ tch = reinterpret_cast<const uint4*>(D.tdig + D.ch_td_off[c]);
  const uint4* __restrict__ tp = tch + ((long)ijg * steps * 4 + t) * 4 + (g / Q) * (Q / 2);
  ring += lane;
  const int mine = part < steps ? (steps - 1 - part) / wk + 1 : 0;  // this warp's steps
#pragma unroll
  for (int d = 0; d < PP_DEPTH - 1; d++) {
    if (d < mine) pp_copy<Q>(ring + d * 256, vp, tp, part + d * wk);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  float acc[DIG_LEVELS][4];
#pragma unroll
  for (int l = 0; l < DIG_LEVELS; l++)
#pragma unroll
    for (int e = 0; e < 4; e++) acc[l][e] = 0.0f;
  DigSum sum[4] = {};
  for (int k = 0; k < mine; k++) {
    asm volatile("cp.async.wait_group %0;" ::"n"(PP_DEPTH - 2) : "memory");
    const uint4* cur = ring + (k % PP_DEPTH) * 256;
    uint32_t a[4][DIG_LEVELS], b[2][Q];
#pragma unroll
    for (int r = 0; r < 4; r++) dig_expand<DIG_LEVELS>(cur[r * 32], a[r]);
#pragma unroll
    for (int r = 0; r < Q / 2; r++) {
      const uint4 v = cur[(4 + r) * 32];
      b[0][2 * r] = v.x; b[1][2 * r] = v.y;
      b[0][2 * r + 1] = v.z; b[1][2 * r + 1] = v.w;
    }
    // the slot of the step before, read in full, takes the step PP_DEPTH - 1 ahead
    if (k + PP_DEPTH - 1 < mine)
      pp_copy<Q>(ring + ((k + PP_DEPTH - 1) % PP_DEPTH) * 256, vp, tp, part + (k + PP_DEPTH - 1) * wk);
    asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll
    for (int i = 0; i < DIG_LEVELS; i++)
#pragma unroll
      for (int j = 0; j < Q; j++)
        if (i + j < DIG_LEVELS) dig_mma16(acc[i + j], a[0][i], a[1][i], a[2][i], a[3][i], b[0][j], b[1][j]);
    if ((k & (DIG_FLUSH / 16 - 1)) == DIG_FLUSH / 16 - 1 || k + 1 == mine) {
#pragma unroll
      for (int e = 0; e < 4; e++) {
        const DigSum x = dig_drain(acc, e);
        sum[e].hi += x.hi;
        sum[e].lo += x.lo;
#pragma unroll
        for (int l = 0; l < DIG_LEVELS; l++) acc[l][e] = 0.0f;
      }
    }
  }
  if (part != 0) {
#pragma unroll
    for (int e = 0; e < 4; e++) red[(part * 4 + e) * 32 + lane] = sum[e];
  }
  __syncthreads();
  if (part != 0) return 0;
  for (int p = 1; p < wk; p++)
#pragma unroll
    for (int e = 0; e < 4; e++) {
      sum[e].hi += red[(p * 4 + e) * 32 + lane].hi;
      sum[e].lo += red[(p * 4 + e) * 32 + lane].lo;
    }
  // accumulator columns 2t, 2t + 1: slot s counts 256^(-Q s); the slots of a row added up
  const int vexp = D.ch_vexp[c];
  const unsigned vtop = CHECK ? D.vtop[it.voff / 256] : 0;
  int nfar = 0;
#pragma unroll
  for (int e = 0; e < 4; e++) {
    const int s = (2 * t + (e & 1)) / Q;
    DigSum x = sum[e];
    if (s) {  // 16 s, 32 or 48 bits down
      const int down = 8 * Q * s;
      x = dig_add_low(DigSum{0, 0}, down < 32 ? (x.hi << (32 - down)) + (x.lo >> down) : (x.hi + (x.lo >> 32)) >> (down - 32));
    }
    if constexpr (SLOTS >= 2) {
      x.hi += __shfl_xor_sync(0xffffffffu, x.hi, 2);
      x.lo += __shfl_xor_sync(0xffffffffu, x.lo, 2);
    }
    if constexpr (SLOTS >= 4) {
      x.hi += __shfl_xor_sync(0xffffffffu, x.hi, 1);
      x.lo += __shfl_xor_sync(0xffffffffu, x.lo, 1);
    }
    const int col = 2 * t + (e & 1), row = g + 8 * (e >> 1), ab = strip * 16 + row;
    bool direct = false;
    if (col < Q && n0 + col < nr && ab < nl) {
      const int ij = rows ? rows[n0 + col] : n0 + col;
      const int te = D.texp[D.ch_hh_off[c] + ij];
      direct = te >= DIG_NONFINITE || vexp >= DIG_NONFINITE;
      if constexpr (CHECK) {
        // the largest V of the strip times the largest amplitude of the row: 2^92 vtop ttop, the sum counts
        // in 2^56 and its part top in 2^88
        const long long top = x.hi + (x.lo >> 32);
        // (nothing is less than 0: in a solve the systems beside a steep one)
        const long long least = steep  ? (long long)vtop * D.ttop[D.ch_hh_off[c] + ij] >> (PP_FAR_STEEP - 4)
                                : rows ? 0
                                       : (long long)vtop * D.ttop[D.ch_hh_off[c] + ij] >> (PP_FAR - 4);
        if (!direct && top < least && top >= -least) {
          direct = true;
          if (!steep) {  // small by cancellation only where the diagonal term is not (random amplitudes)
            const int off = D.ch_pp_off[c];
            const int2 p = D.pp_pair[off + abs(D.lad_mem[off + ab].x) - 1];
            const char4 a = D.nvec[p.x], b = D.nvec[p.y];
            const double diag = v_minnesota_as(a, b, a, b, lut) * s64[D.ch_s_off[c] + (long)ij * nl + ab];
            direct = !(fabs(diag) >= scalbn((double)least, 88 - 122 + vexp + te - 2044));
          }
        }
      }
      Out* o = reinterpret_cast<Out*>(D.rpp) + D.ch_s_off[c] + (long)ij * nl + ab;
      if (!direct) *o = dig_result<Out>(x, dig_power(vexp, te));
      else if (!CHECK)
        *o = Arith<Out>::from_double(pp_direct(D, lut, t0 + (long)ij * D.ch_npp[c], D.ch_pp_off[c], nl, ab));
    }
    if constexpr (CHECK) {
      const unsigned b = __ballot_sync(0xffffffffu, direct);
      if (direct) far[nfar + __popc(b & ((1u << lane) - 1u))] = (unsigned char)(8 * row + col);
      nfar += __popc(b);
    }
  }
  return nfar;
}

// rep_only: the rows ij of the items count the list upd_row of the channel, else every hole pair (the
// operator: amplitudes given by the caller).
// wk (2 or 4) divides PP_WARPS: PP_WARPS / wk items per CTA.  slots: ring steps per warp, PP_DEPTH or
// as many as a warp has.  lut_off: interaction table of every system.  s64: the rows in the
// ladder basis (CHECK).
template <typename Out, bool CHECK>
__global__ void __launch_bounds__(PP_WARPS * 32, PP_CTAS) k_pp(DevState D, const LoopCtl* __restrict__ ctl,
                                                               const PPItem* __restrict__ items, int nitems, int rep_only,
                                                               int wk, int slots, const int* __restrict__ lut_off,
                                                               const double* __restrict__ s64) {
  extern __shared__ __align__(16) uint4 pp_ring[];
  __shared__ DigSum red[PP_WARPS * 128];
  __shared__ unsigned char far[CHECK ? PP_WARPS : 1][128];
  __shared__ int nfar[CHECK ? PP_WARPS : 1];
  const int warp = threadIdx.x >> 5, part = warp % wk, first = warp - part;
  const int item = blockIdx.x * (PP_WARPS / wk) + warp / wk;
  PPItem it;
  if (item < nitems) it = items[item];
  // warps without work join the barriers of pp_pass and after it here
  if (item >= nitems || sys_done(D, ctl, it.sys)) {
    __syncthreads();
    if (CHECK) __syncthreads();
    return;
  }
  const int* __restrict__ rows = rep_only ? D.upd_row + D.ch_uoff[it.c] : nullptr;
  DigSum* mine = red + first * 128;
  uint4* ring = pp_ring + warp * slots * 256;
  const int n = it.nr - it.n0;
  const int c = it.c;
  const double* __restrict__ lut = D.lut + lut_off[it.sys];
  const double* __restrict__ t = cur_t(D, ctl) + D.ch_t_off[c];
  const bool steep = CHECK && D.sys_steep && D.sys_steep[it.sys];
  unsigned char* list = far[CHECK ? first : 0];
  int left;
  if (n > 4) left = pp_pass<1, Out, CHECK>(D, it, rows, part, wk, ring, mine, lut, t, s64, steep, list);
  else if (n > 2) left = pp_pass<2, Out, CHECK>(D, it, rows, part, wk, ring, mine, lut, t, s64, steep, list);
  else left = pp_pass<4, Out, CHECK>(D, it, rows, part, wk, ring, mine, lut, t, s64, steep, list);
  if (!CHECK) return;
  if (part == 0 && (threadIdx.x & 31) == 0) nfar[CHECK ? first : 0] = left;
  __syncthreads();
  left = nfar[CHECK ? first : 0];
  if (left == 0) return;
  // the item's warps take the results left in turn, four at a time
  for (int k = 4 * part; k < left; k += 4 * wk) pp_far<Out>(D, it, rows, lut, s64, steep, list + k, min(4, left - k));
}

// FP32-pair copy of an FP64 array.
__global__ void k_split_f2(const double* __restrict__ a, f2* __restrict__ b, long n) {
  long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = Arith<f2>::from_double(a[i]);
}

void pnm_split_f2(const double* a, f2* b, long n, cudaStream_t s) {
  if (n > 0) k_split_f2<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, b, n);
}

// ----------------------------------------------------------------------- finalize
// End of one update: energy (Eq. ccdcorr, sum of v t over restricted amplitudes) and
// residual norm per system from the block partials in a fixed order, the |dE| test, the
// energy history, and the loop condition of the device-side loop.
// The last CTA of a system closes that system, the last of these the update: a chain of dependent
// round trips, not bandwidth, that adds to every update, so the systems of a batch go side by side
// (one CTA closing all 120 systems of 22 partials each, a warp per system, left the GPU idle for half
// of the update: 141 us, 79 us so).  FIN_UNROLL partial pairs are requested before the first
// is added; up to 32 times as many take one warp without barriers.
constexpr int FIN_UNROLL = 8;

// Sums of a and b over a warp, in lanes 0 and 16: the first exchange leaves the a in one half of the
// warp and the b in the other, so that both take five additions of the slow FP64 pipe instead of ten.
__device__ __forceinline__ double warp_sum_two(double a, double b) {
  const bool low = (threadIdx.x & 16) == 0;
  double x = (low ? a : b) + __shfl_xor_sync(0xffffffffu, low ? b : a, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

__device__ __forceinline__ void sum_partials(const FinArgs& f, int s, int first, int step, double& e, double& r) {
  const int hi = f.hi[s];
  e = 0.0;
  r = 0.0;
  int k = f.lo[s] + first;
  for (; k + (FIN_UNROLL - 1) * step < hi; k += FIN_UNROLL * step) {
    double a[FIN_UNROLL], b[FIN_UNROLL];
#pragma unroll
    for (int j = 0; j < FIN_UNROLL; j++) {
      a[j] = __ldcg(f.eparts + k + j * step);
      b[j] = __ldcg(f.rparts + k + j * step);
    }
#pragma unroll
    for (int j = 0; j < FIN_UNROLL; j++) {
      e += a[j];
      r += b[j];
    }
  }
  for (; k < hi; k += step) {
    e += __ldcg(f.eparts + k);
    r += __ldcg(f.rparts + k);
  }
}

// One system's control block from its energy and squared residual (one thread).  S and the loop
// control c are copies read before the sums, so that their loads overlap the partials'.  Returns
// whether the system has diverged.
__device__ __forceinline__ bool finalize_one(const FinArgs& f, SysCtl& S, const LoopCtl& c, int s, double e, double r) {
  bool bad = false;
  if (!S.done) {
    S.iters += 1;
    S.e_new = e;
    S.resid = sqrt(r);
    if (S.iters < f.hist_cap) f.hist[(long)s * f.hist_cap + S.iters] = e;
    const double diff = fabs(e - S.e_old);
    S.e_old = e;
    S.grow = (diff > 2.0 * S.d_old && diff > S.tol) ? S.grow + 1 : 0;
    S.d_old = diff;
    bad = !isfinite(e) || !isfinite(r) || S.grow >= PNM_DIVERGE_STEPS;
    if (diff < S.tol && c.iter + 1 >= c.min_iter) {
      S.done = 1;
      S.frozen_at = c.iter;
    }
    f.sc[s] = S;
  }
  return bad;
}

// The last of system s's CTAs to finish closes it, and the last system the update (no waiting: CTAs and
// systems count themselves out with atomics after a fence, as in the CUDA threadfence reduction).
// Every counter is left at zero for the next update.
__device__ void finalize_system(const FinArgs& f, LoopCtl* ctl, int s, int ctas) {
  __shared__ int is_last;
  __shared__ double sh32f[32];
  __syncthreads();
  if (threadIdx.x == 0) {
    // only thread 0 wrote the block's partials: its fence orders them before the count
    __threadfence();
    is_last = atomicAdd(f.blocks_done + s, 1) == ctas - 1;
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  const LoopCtl c = *ctl;
  SysCtl S;
  if (threadIdx.x == 0) S = f.sc[s];
  double e, r;
  if (ctas <= 32 * FIN_UNROLL) {  // one warp, without barriers
    if (threadIdx.x >= 32) return;
    const int k0 = f.lo[s] + threadIdx.x, hi = f.hi[s];
    double a[FIN_UNROLL], b[FIN_UNROLL];
#pragma unroll
    for (int j = 0; j < FIN_UNROLL; j++) {
      a[j] = k0 + 32 * j < hi ? __ldcg(f.eparts + k0 + 32 * j) : 0.0;
      b[j] = k0 + 32 * j < hi ? __ldcg(f.rparts + k0 + 32 * j) : 0.0;
    }
    e = a[0];
    r = b[0];
#pragma unroll
    for (int j = 1; j < FIN_UNROLL; j++) {
      if (32 * j >= ctas) break;
      e += a[j];
      r += b[j];
    }
    const double x = warp_sum_two(e, r);
    e = x;
    r = __shfl_sync(0xffffffffu, x, 16);
  } else {
    sum_partials(f, s, threadIdx.x, blockDim.x, e, r);
    block_sum2(e, r, sh32f);
  }
  if (threadIdx.x != 0) return;
  f.blocks_done[s] = 0;
  bool bad = finalize_one(f, S, c, s, e, r), all_done = S.done;
  if (f.nsys > 1) {
    if (bad) {  // before this system is counted
      atomicExch(&ctl->bad, 1);
      __threadfence();
    }
    const unsigned long long one = UpdCount::one(S.done != 0);
    const UpdCount now{atomicAdd(&ctl->closed, one) + one};
    if (now.finished() != (unsigned)f.nsys) return;
    ctl->closed = 0;
    all_done = now.converged() == (unsigned)f.nsys;
    __threadfence();
    bad = atomicExch(&ctl->bad, 0) != 0;
  }
  ctl->iter = c.iter + 1;
  int cont = 1;
  if (c.dev_error) {
    ctl->status = PNM_ETIMEOUT;
    cont = 0;
  } else if (bad) {
    ctl->status = PNM_EDIVERGED;
    cont = 0;
  } else if (all_done) {
    ctl->status = 1;
    cont = 0;
  } else if (c.iter + 1 >= c.max_iter) {
    ctl->status = PNM_ENOTCONV;
    cont = 0;
  }
  if (f.use_cond) cudaGraphSetConditional(f.handle, cont ? 1u : 0u);
}

// ---------------------------------------------------------------------------- update
// Jacobi step of Eq. (ccd3): the bracket collects v, the non-eps parts of the one-body terms, the pp
// and hh ladders and P(ij)P(ab) Q; then t_new = bracket / eps_ij^ab and t = alpha t_new + (1 - alpha)
// t_old.  The residual of the amplitude equation is R = bracket - eps_ij^ab t.
// One amplitude of each spin-flip pair is computed (the one with the smaller index) and written to
// both; the pair counts twice in the energy and the residual norm.
//
// One thread per amplitude of the rows the updates compute, in the order of the list upd_z (chunks of
// 32 in one channel, UpdItem; a CTA's chunks in one system), U chunks per warp.  What bounds an update
// is a chain of dependent round trips, so the chain is three long: the amplitude's index and the
// chunk's metadata; the streams (t, v, eps, maps), the pair's states and the hh ladder's column; the Q,
// ladder and one-body values behind them.  A thread per column that goes through eight rows of a
// channel, as before, has the hh ladder's t column once for eight rows, but idles where a channel has
// less than 128 columns and walks the chain once for every row or two; the column is a coalesced load
// that L1 and L2 serve.  A warp's first chunk is requested before the loop control and the system's
// state are looked at, which takes two round trips off an update of a small system (39 updates of
// N=14, N_max=4: 0.77 -> 0.70 ms).
struct UpdSums {  // energy and residual norm, amplitudes with and without a flip of their own
  double e2 = 0.0, e1 = 0.0, r2 = 0.0, r1 = 0.0;
  __device__ __forceinline__ void add(bool flip, double v, double out, double R) {
    if (flip) {
      e2 = fma(v, out, e2);
      r2 = fma(R, R, r2);
    } else {
      e1 = fma(v, out, e1);
      r1 = fma(R, R, r1);
    }
  }
};

// Block sums of the energy and the residual norm into the CTA's partials.
__device__ __forceinline__ void upd_partials(const DevState& D, const UpdSums& S) {
  __shared__ double red[UPD_THREADS / 32][2];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const double x = warp_sum_two(fma(2.0, S.e2, S.e1), fma(2.0, S.r2, S.r1));
  if ((lane & 15) == 0) red[w][lane >> 4] = x;
  __syncthreads();
  if (threadIdx.x == 0) {
    D.eparts[blockIdx.x] = (red[0][0] + red[1][0]) + (red[2][0] + red[3][0]);
    D.rparts[blockIdx.x] = (red[0][1] + red[1][1]) + (red[2][1] + red[3][1]);
  }
}

// FP64 update, or (T_ = f2) the update of the sweeps with FP32-pair contractions: the pp ladder, the
// hh ladder (from the pair copy of the amplitudes) and the ph term are pairs then (the 8-byte slots of
// rpp and xq) and their sum is formed on the FP32 pipe and converted to FP64 once; the denominator,
// residual, step (alpha / eps_ij^ab prepared per solve, aw) and energy stay FP64.
// One FP64 update with the thread-per-column layout and here: N=66, N_max=42 93, 69 us (the FP64 pipe
// busy for 72% of the time the SMs are); 28 nucleons, N_max=20 27.8, 18.4; N=14, N_max=4 16.4, 12.3.
// Pair sweeps of three N=66, N_max=36 systems: 117, 105.
template <typename T_, int U>
__global__ void __launch_bounds__(UPD_THREADS) k_update(DevState D, LoopCtl* __restrict__ ctl,
                                                        const UpdItem* __restrict__ items,
                                                        const int* __restrict__ upd_z, FinArgs fa,
                                                        const T_* __restrict__ tpair, const double* __restrict__ aw) {
  constexpr bool PAIR = std::is_same<T_, f2>::value;
  using A = Arith<T_>;
  struct Amp {
    UpdItem it;
    long z;
    double tz, v, den, step;
    int4 q;
    int2 p, h;
    int fc, ij, ab, m;
  };
  const double* __restrict__ t = cur_t(D, ctl);
  const long chunk0 = (long)blockIdx.x * (U * UPD_THREADS / 32) + (threadIdx.x >> 5);
  // the amplitude's streams and pair data: its place in the channel, then everything indexed by it
  auto load = [&](int u) {
    Amp a;
    const long chunk = chunk0 + u * (UPD_THREADS / 32);
    a.it = items[chunk];
    a.z = upd_z[chunk * 32 + (threadIdx.x & 31)];
    if (a.z < 0) return a;  // padding
    const int e = (int)(a.z - a.it.base);
    a.ij = e / a.it.npp;
    a.ab = e - a.ij * a.it.npp;
    a.fc = D.fmap[a.z];
    a.tz = t[a.z];
    a.v = D.v_pphh[a.z];
    a.q = D.qmap[a.z];
    a.den = D.den[a.z];
    a.step = PAIR ? aw[a.z] : D.inv_den[a.z];
    a.p = D.pp_pair[a.it.pp_off + a.ab];
    a.h = D.hh_pair[a.it.hh_off + a.ij];
    a.m = a.it.nl ? D.lad_map[a.it.pp_off + a.ab] : 0;
    return a;
  };
  // the first chunk is requested before the loop control and the system's state are looked at
  Amp a = load(0);
  if (ctl->status != 0) return;  // the loop has ended within its body (see pnm_enqueue_loop_body)
  const int sys = a.it.sys, ctas = fa.hi[sys] - fa.lo[sys];
  UpdSums S;
  // converged at least two steps ago: both amplitude buffers already hold its values, and its sums
  // are not read any more
  if (!sys_settled(fa.sc[sys], ctl)) {
    const bool frozen = fa.sc[sys].done != 0;
    const double alpha = ctl->alpha;
    double* __restrict__ tn = next_t(D, ctl);
    const T_* __restrict__ tc;
    if constexpr (PAIR) tc = tpair;
    else tc = t;
    const T_* __restrict__ rp = reinterpret_cast<const T_*>(D.rpp);
    const T_* __restrict__ xq = reinterpret_cast<const T_*>(D.xq);
#pragma unroll
    for (int u = 0; u < U; u++) {
      if (u > 0) a = load(u);
      const long z = a.z;
      if (z < 0) continue;
      const long f = (long)(a.fc > 0 ? a.fc : -a.fc) - 1;
      if (f < z) continue;
      const double tz = a.tz, v = a.v;
      double out = tz, R = 0.0;
      if (!frozen) {
        const int4 q = a.q;
        T_ rl = A::zero();
        if (a.m != 0) {
          rl = rp[a.it.s_off + (long)a.ij * a.it.nl + ((a.m > 0 ? a.m : -a.m) - 1)];
          if (a.m < 0) rl = A::neg(rl);
        }
        const T_ q0 = q.x >= 0 ? xq[q.x] : A::zero(), q1 = q.y >= 0 ? xq[q.y] : A::zero();
        const T_ q2 = q.z >= 0 ? xq[q.z] : A::zero(), q3 = q.w >= 0 ? xq[q.w] : A::zero();
        // one-body part of the bracket: (d_a + d_b - d_i - d_j) t with d_p = chi_p - eps_p
        const double d = (D.dchi[a.p.x] + D.dchi[a.p.y]) - (D.dchi[a.h.x] + D.dchi[a.h.y]);
        // hh ladder sum_kl t_ab^kl chi_kl^ij
        T_ hs = A::zero();
        const int nh = a.it.nh, npp = a.it.npp;
        const T_* __restrict__ col = tc + a.it.base + a.ab;
        const T_* __restrict__ chi = reinterpret_cast<const T_*>(D.chi_hh) + a.it.vhh_off + a.ij;
#pragma unroll 4
        for (int kl = 0; kl < nh; kl++) A::mac(hs, col[(long)kl * npp], chi[(long)kl * nh]);
        if constexpr (PAIR) {
          // pp ladder + hh ladder + P(ij)P(ab) Q in FP32 pairs, converted once
          const f2 corr = A::add(A::sub(A::sub(A::add(A::add(hs, rl), q0), q1), q2), q3);
          const double num = fma(d, tz, v) + A::to_double(corr);
          R = fma(-a.den, tz, num);  // bracket - eps_ij^ab t
          out = fma(R, a.step, tz);  // t + alpha R / eps_ij^ab
        } else {
          const double num = ((fma(d, tz, v) + rl) + hs) + (((q0 - q1) - q2) + q3);
          R = fma(-a.den, tz, num);
          out = fma(alpha, num * a.step, (1.0 - alpha) * tz);
        }
      }
      tn[z] = out;
      if (f != z) tn[f] = a.fc > 0 ? out : -out;
      S.add(f != z, v, out, R);
    }
    upd_partials(D, S);
  }
  finalize_system(fa, ctl, sys, ctas);
}

template <typename T_>
static void launch_update(pnm_ctx* ctx, const FinArgs& fa, const T_* tpair, const double* aw) {
  auto go = [&](auto k) {
    k<<<ctx->n_upd_ctas, UPD_THREADS, 0, ctx->stream>>>(ctx->d, ctx->ctl, ctx->upd_chunks, ctx->upd_z, fa, tpair, aw);
  };
  if (ctx->upd_per_warp == 1) go(k_update<T_, 1>);
  else if (ctx->upd_per_warp == 2) go(k_update<T_, 2>);
  else go(k_update<T_, 4>);
}

void launch_update64(pnm_ctx* ctx, int use_cond, cudaGraphConditionalHandle h, bool pair) {
  const FinArgs fa = fin_args(ctx, use_cond, h);
  if (pair) launch_update<f2>(ctx, fa, ctx->t_pair, pnm_mixed_aw(ctx));
  else launch_update<double>(ctx, fa, nullptr, nullptr);
}

// Mixed-precision update, in the same layout:
//   hh ladder   sum_kl t_ab^kl chi_kl^ij in FP32 from the FP32 copies
//   bracket     corrections in FP32: one-body (d_a + d_b - d_i - d_j) t, pp ladder (ladder
//               layout, k-split planes summed), hh ladder, and the ph term
//               Q_ij^ab - Q_ji^ab - Q_ij^ba + Q_ji^ba gathered from the cross-channel Q (qmap)
//   T scatter   the new FP32 amplitude to its four places in the ph term's T (the positions of
//               the four Q terms, qmap; formed positions only, so the same for the amplitude
//               and its spin flip), which the next ph kernel reads row by row
//   FP64        residual R = v + bracket - eps_ij^ab t, step t + alpha R / eps_ij^ab (alpha / eps_ij^ab
//               prepared per solve), energy and residual partial sums
// Arrays read once per update (t, v, eps, alpha / eps, flip and Q maps) and the FP64 amplitudes
// written for the next update are streamed with the evict-first policy, so that the ph term's T and Q
// (25 MB each for the held-out batch, read and written at random) and the FP32 amplitudes the
// next update's contractions read stay in L2.
// The FP64 unit of a GB300 runs at about 1/64 of its FP32 rate, so the FP64 work is held to
// six instructions and two conversions per amplitude (v and eps are read: forming them from the
// states took three more and two more round trips); the new amplitude goes to t (FP64) for itself and
// to t32 for itself and, sign applied, for its spin flip.  The FP64 flips are not read before the mixed
// iteration ends (the update reads t at the amplitudes it computes only); one flip copy of the
// current buffer fills them then (pnm_flip_copy_current).
// One update with the thread-per-column layout and here: three N=66, N_max=36 systems 113, 90 us; 120
// twisted N=14, N_max=20 systems 190, 79; one of these 14.3, 12.3.
template <int U>
__global__ void __launch_bounds__(UPD_THREADS, UPD_MIN_BLOCKS) k_update_mix(
    DevState D, LoopCtl* __restrict__ ctl, const UpdItem* __restrict__ items, const int* __restrict__ upd_z, FinArgs fa,
    const float* __restrict__ rpp, const float* __restrict__ xq, const double* __restrict__ aw, float* __restrict__ xt,
    int nplanes, long pstride) {
  struct Amp {
    UpdItem it;
    long z;
    double tz, wz, v, den;
    int4 qm;
    int2 p, h;
    float t32z;
    int fc, ij, ab, m;
  };
  const double* __restrict__ t = cur_t(D, ctl);
  const float* __restrict__ t32 = cur_t32(D, ctl);
  const long chunk0 = (long)blockIdx.x * (U * UPD_THREADS / 32) + (threadIdx.x >> 5);
  // the amplitude's streams and pair data: its place in the channel, then everything indexed by it
  auto load = [&](int u) {
    Amp a;
    const long chunk = chunk0 + u * (UPD_THREADS / 32);
    a.it = items[chunk];
    a.z = upd_z[chunk * 32 + (threadIdx.x & 31)];
    if (a.z < 0) return a;  // padding
    const int e = (int)(a.z - a.it.base);
    a.ij = e / a.it.npp;
    a.ab = e - a.ij * a.it.npp;
    a.tz = __ldcs(t + a.z);
    a.wz = __ldcs(aw + a.z);
    a.v = __ldcs(D.v_pphh + a.z);
    a.den = __ldcs(D.den + a.z);
    a.fc = __ldcs(D.fmap + a.z);
    a.qm = __ldcs(D.qmap + a.z);
    a.t32z = t32[a.z];
    a.p = D.pp_pair[a.it.pp_off + a.ab];
    a.h = D.hh_pair[a.it.hh_off + a.ij];
    a.m = a.it.nl ? D.lad_map[a.it.pp_off + a.ab] : 0;
    return a;
  };
  // the first chunk is requested before the loop control and the system's state are looked at
  Amp a = load(0);
  if (ctl->status != 0) return;  // the loop has ended within its body (see pnm_enqueue_loop_body)
  const int sys = a.it.sys, ctas = fa.hi[sys] - fa.lo[sys];
  UpdSums S;
  // converged at least two steps ago: both amplitude buffers already hold its values, and its sums
  // are not read any more
  if (!sys_settled(fa.sc[sys], ctl)) {
    const bool frozen = fa.sc[sys].done != 0;
    double* __restrict__ tn = next_t(D, ctl);
    float* __restrict__ t32n = next_t32(D, ctl);
#pragma unroll (U < UPD_MIX_UNROLL ? U : UPD_MIX_UNROLL)
    for (int u = 0; u < U; u++) {
      if (u > 0) a = load(u);
      const long z = a.z;
      if (z < 0) continue;
      const int4 qm = a.qm;
      float rl = 0.0f;
      if (a.m != 0) {
        const long zl = a.it.s_off + (long)a.ij * a.it.nl + ((a.m > 0 ? a.m : -a.m) - 1);
        for (int pl = 0; pl < nplanes; pl++) rl += rpp[pl * pstride + zl];
        if (a.m < 0) rl = -rl;
      }
      // P(ij)P(ab) Q: Q_ij^ab - Q_ji^ab - Q_ij^ba + Q_ji^ba from the cross-channel layout
      const float a0 = qm.x >= 0 ? xq[qm.x] : 0.0f, a1 = qm.y >= 0 ? xq[qm.y] : 0.0f;
      const float a2 = qm.z >= 0 ? xq[qm.z] : 0.0f, a3 = qm.w >= 0 ? xq[qm.w] : 0.0f;
      const float d = (D.dchi32[a.p.x] + D.dchi32[a.p.y]) - (D.dchi32[a.h.x] + D.dchi32[a.h.y]);
      float hh = 0.0f;
      if (!frozen) {
        const int nh = a.it.nh, npp = a.it.npp;
        const float* __restrict__ col = t32 + a.it.base + a.ab;
        const float* __restrict__ chi = D.chi32 + a.it.vhh_off + a.ij;
#pragma unroll UPD_HH_UNROLL
        for (int kl = 0; kl < nh; kl++) hh = fmaf(col[(long)kl * npp], chi[(long)kl * nh], hh);
      }
      // one amplitude of each spin-flip pair is computed (the smaller index) and written to both
      const long f = (long)(a.fc > 0 ? a.fc : -a.fc) - 1;
      if (f < z) continue;
      double out = a.tz, R = 0.0;
      if (!frozen) {
        const float corr = d * a.t32z + (rl + hh) + ((a0 - a1) - (a2 - a3));
        R = fma(-a.den, a.tz, a.v) + (double)corr;  // bracket - eps_ij^ab t
        out = fma(R, a.wz, a.tz);
      }
      const float o32 = (float)out;
      __stcs(tn + z, out);
      t32n[z] = o32;
      if (f != z) t32n[f] = a.fc < 0 ? -o32 : o32;
      S.add(f != z, a.v, out, R);
      if (!frozen) {
        // the T positions of t_ij^ab, t_ji^ab, t_ij^ba, t_ji^ba (the Q positions of the same
        // amplitude; stores only, nothing waits on them)
        if (qm.x >= 0) xt[qm.x] = o32;
        if (qm.y >= 0) xt[qm.y] = -o32;
        if (qm.z >= 0) xt[qm.z] = -o32;
        if (qm.w >= 0) xt[qm.w] = o32;
      }
    }
    upd_partials(D, S);
  }
  finalize_system(fa, ctl, sys, ctas);
}

void launch_update_mix(pnm_ctx* ctx, const float* rpp, const float* xq, const double* aw, float* xt, int use_cond,
                       cudaGraphConditionalHandle h, int nplanes, long pstride) {
  const FinArgs fa = fin_args(ctx, use_cond, h);
  auto go = [&](auto k) {
    k<<<ctx->n_upd_ctas, UPD_THREADS, 0, ctx->stream>>>(ctx->d, ctx->ctl, ctx->upd_chunks, ctx->upd_z, fa, rpp, xq, aw, xt,
                                                        nplanes, pstride);
  };
  if (ctx->upd_per_warp == 1) go(k_update_mix<1>);
  else if (ctx->upd_per_warp == 2) go(k_update_mix<2>);
  else go(k_update_mix<4>);
}

// alpha / eps_ij^ab per amplitude (the step of the mixed update).
__global__ void k_alpha_inv(const double* __restrict__ inv_den, double alpha, long n, double* __restrict__ aw) {
  long z = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (z < n) aw[z] = alpha * inv_den[z];
}

void pnm_alpha_inv(pnm_ctx* ctx, double alpha, double* aw) {
  if (ctx->nt > 0)
    k_alpha_inv<<<(unsigned)((ctx->nt + 255) / 256), 256, 0, ctx->stream>>>(ctx->d.inv_den, alpha, ctx->nt, aw);
  CUDA_TRY(cudaGetLastError());
}

// t <- (t + F t) / 2 under the global spin flip F (fmap).  The solution is flip-symmetric
// and the ph term is formed for flip-symmetric amplitudes, so kept and learned starts are
// symmetrised first (MBPT2 and zero starts are symmetric already).  A pair (z, F z) is handled
// by the thread of its smaller index; fmap is an involution.
__global__ void k_flip_sym(const int* __restrict__ fmap, double* __restrict__ t, long n) {
  long z = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (z >= n) return;
  int cd = fmap[z];
  long f = (long)(cd > 0 ? cd : -cd) - 1;
  if (f < z) return;
  double v = 0.5 * (t[z] + (cd > 0 ? t[f] : -t[f]));
  t[z] = v;
  if (f != z) t[f] = cd > 0 ? v : -v;
}

// t(F z) <- sign * t(z) for every z that comes before its flip (a start computed on the rows
// the updates compute, made flip-symmetric).
__global__ void k_flip_copy(const int* __restrict__ fmap, double* __restrict__ t, long n) {
  long z = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (z >= n) return;
  int cd = fmap[z];
  long f = (long)(cd > 0 ? cd : -cd) - 1;
  if (f > z) t[f] = cd > 0 ? t[z] : -t[z];
}

void pnm_flip_copy(pnm_ctx* ctx, double* t, cudaStream_t s) {
  if (ctx->nt > 0)
    k_flip_copy<<<(unsigned)((ctx->nt + 255) / 256), 256, 0, s>>>(ctx->d.fmap, t, ctx->nt);
}

// The spin flips of the current FP64 amplitudes (t[iter & 1]) from the amplitudes the updates
// compute, after a mixed-precision iteration (whose updates write the FP64 values of the
// computed amplitudes only).
void pnm_flip_copy_current(pnm_ctx* ctx, int iter) {
  pnm_flip_copy(ctx, (iter & 1) ? ctx->d.t1 : ctx->d.t0, ctx->stream);
  CUDA_TRY(cudaGetLastError());
}

void pnm_flip_symmetrise(pnm_ctx* ctx, double* t, cudaStream_t s) {
  if (ctx->nt > 0)
    k_flip_sym<<<(unsigned)((ctx->nt + 255) / 256), 256, 0, s>>>(ctx->d.fmap, t, ctx->nt);
}

// v / eps from the reciprocal held beside eps: one product and Markstein's correction step (IBM J.
// Res. Dev. 34 (1990) 111: with y = 1 / eps correctly rounded and q = v y, q + y (v - q eps) is the
// correctly rounded quotient whenever q is within one last place of it), three FP64 instructions
// where a division takes a dozen.
__device__ __forceinline__ double div_by_eps(double v, double den, double inv) {
  if (!isfinite(inv)) return v / den;
  const double q = v * inv;
  return fma(fma(-q, den, v), inv, q);
}

// MBPT2 energy partials sum v t over restricted amplitudes per row (channel, ij), and with WRITE the
// start amplitudes (MBPT2 guess, zero, or as they are) into t0.  One amplitude of each spin-flip pair
// is formed, written to both and counted twice; the rows that the flip maps onto earlier ones are
// theirs.  Bound by the FP64 pipe when every amplitude was formed from its states and divided (122 us
// for three N=66, N_max=36 systems; 33 so).
template <bool WRITE>
__global__ void __launch_bounds__(128) k_mbpt2(DevState D, int init) {
  __shared__ double sh32[32];
  const int2 it = D.row_item[blockIdx.x];
  const int npp = D.ch_npp[it.x];
  const long row = D.ch_t_off[it.x] + (long)it.y * npp;
  const int first = D.fmap[row];
  double e2 = 0.0, e1 = 0.0;
  if (abs(first) - 1 >= row) {
#pragma unroll 4
    for (int ab = threadIdx.x; ab < npp; ab += 128) {
      const long z = row + ab;
      const int fc = D.fmap[z];
      const double v = D.v_pphh[z];
      const long f = (long)(fc > 0 ? fc : -fc) - 1;
      double t = 0.0;
      if (init == PNM_INIT_MBPT2) t = div_by_eps(v, D.den[z], D.inv_den[z]);
      else if (init != PNM_INIT_ZERO) t = D.t0[z];
      if (f < z) continue;
      if (WRITE && (init == PNM_INIT_MBPT2 || init == PNM_INIT_ZERO)) {
        D.t0[z] = t;
        if (f != z) D.t0[f] = fc > 0 ? t : -t;
      }
      if (f != z) e2 = fma(v, t, e2);
      else e1 = fma(v, t, e1);
    }
    e1 = block_sum(fma(2.0, e2, e1), sh32);
  }
  if (threadIdx.x == 0) {
    D.eparts[blockIdx.x] = e1;
    if (WRITE) D.rparts[blockIdx.x] = 0.0;
  }
}

// Sums of row or CTA partials per system (fixed order): out[plane * nsys + sys], planes of n partials.
__global__ void k_reduce_rows(const double* __restrict__ parts, long n, const int* __restrict__ row_lo,
                              const int* __restrict__ row_hi, double* __restrict__ out) {
  __shared__ double sh32[32];
  const int s = blockIdx.x;
  parts += blockIdx.y * n;
  double acc = 0.0;
#pragma unroll 4
  for (int r = row_lo[s] + threadIdx.x; r < row_hi[s]; r += blockDim.x) acc += parts[r];
  acc = block_sum(acc, sh32);
  if (threadIdx.x == 0) out[blockIdx.y * gridDim.x + s] = acc;
}

// Energy of the start amplitudes: history[0] per system, reset of the loop state.
__global__ void k_start(const double* __restrict__ parts, const int* __restrict__ row_lo,
                        const int* __restrict__ row_hi, int nsys, SysCtl* __restrict__ sc,
                        LoopCtl* __restrict__ ctl, double* __restrict__ hist, int hist_cap) {
  // one warp per system in batches, else the whole block
  __shared__ double sh32[32];
  const bool by_warp = nsys >= 4;
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int s = by_warp ? threadIdx.x >> 5 : 0; s < nsys; s += by_warp ? nw : 1) {
    double acc = 0.0;
    for (int r = row_lo[s] + (by_warp ? lane : threadIdx.x); r < row_hi[s]; r += by_warp ? 32 : blockDim.x)
      acc += parts[r];
    acc = by_warp ? warp_sum(acc) : block_sum(acc, sh32);
    if (by_warp ? lane == 0 : threadIdx.x == 0) {
      sc[s].e_old = acc;
      sc[s].e_new = acc;
      sc[s].resid = 0.0;
      sc[s].done = 0;
      sc[s].iters = 0;
      hist[(long)s * hist_cap] = acc;
    }
  }
  if (threadIdx.x == 0) {
    ctl->iter = 0;
    ctl->status = 0;
    ctl->dev_error = 0;
  }
}

// ------------------------------------------------------------------------- host side

static void* dmalloc(pnm_ctx* ctx, size_t bytes) { return pnm_ctx_alloc(ctx, bytes); }

__host__ __device__ __forceinline__ int stat_groups(int nrows) { return (nrows + STAT_COLS) / STAT_COLS; }

// The update chunks and their amplitudes: rows of the channel's run of upd_row one after the other, 32
// amplitudes per chunk; a channel per CTA (its chunks start at first[c].x, its items of the stats kernel
// at first[c].y), then a system per CTA for the
// padding up to whole CTAs of the updates.
__global__ void __launch_bounds__(128) k_upd_chunks(DevState D, int nch, const int2* __restrict__ first,
                                                    const int2* __restrict__ pad, UpdItem* __restrict__ items,
                                                    int* __restrict__ upd_z, int4* __restrict__ stat) {
  UpdItem it{};
  if ((int)blockIdx.x >= nch) {
    const int2 p = pad[blockIdx.x - nch];
    it.npp = 1;
    it.sys = blockIdx.x - nch;
    for (int k = p.x * 32 + threadIdx.x; k < p.y * 32; k += blockDim.x) {
      upd_z[k] = -1;
      if ((k & 31) == 0) items[k >> 5] = it;
    }
    return;
  }
  const int c = blockIdx.x;
  it.npp = D.ch_npp[c];
  it.nh = D.ch_nhh[c];
  it.sys = D.ch_sys[c];
  it.nl = D.ch_vpp[c] ? D.ch_nlad[c] : 0;
  it.pp_off = D.ch_pp_off[c];
  it.hh_off = D.ch_hh_off[c];
  it.base = D.ch_t_off[c];
  it.vhh_off = D.ch_vhh_off[c];
  it.s_off = D.ch_s_off[c];
  const int r0 = D.ch_uoff[c], n = (D.ch_uoff[c + 1] - r0) * it.npp;
  const long k0 = 32L * first[c].x;
  for (int e = threadIdx.x; e < ((n + 31) & ~31); e += blockDim.x) {
    const int r = e / it.npp;
    upd_z[k0 + e] = e < n ? (int)(it.base + (long)D.upd_row[r0 + r] * it.npp + (e - r * it.npp)) : -1;
    if ((e & 31) == 0) items[(k0 + e) >> 5] = it;
  }
  // items of the stats kernel: per row its groups of columns, then the channel's columns by 32
  int4* so = stat + first[c].y;
  const int groups = stat_groups(D.ch_uoff[c + 1] - r0), rows = it.nh * groups;
  for (int k = threadIdx.x; k < rows + (it.npp + 31) / 32; k += blockDim.x)
    so[k] = k < rows ? make_int4(c, k / groups, k % groups * STAT_COLS, 0) : make_int4(c, -1, (k - rows) * 32, 0);
}

// pp items of nr[c] rows per channel in the order of decreasing work, so that the last CTAs are
// short ones; the list goes to *dst.  Returns its length.
static int pp_work_list(pnm_ctx* ctx, const std::vector<int>& nr, PPItem** dst) {
  struct Pass {
    long work;
    int c, n0;
  };
  std::vector<Pass> passes;
  size_t n = 0;
  for (int c = 0; c < ctx->nch; c++) {
    if (!ctx->h_vpp[c]) continue;
    for (int n0 = 0; n0 < nr[c]; n0 += 8) {
      passes.push_back({(long)ctx->h_nlad[c] * (nr[c] - n0 > 4 ? 36 : (nr[c] - n0 > 2 ? 26 : 15)), c, n0});
      n += (ctx->h_nlad[c] + 15) / 16;
    }
  }
  std::stable_sort(passes.begin(), passes.end(), [](const Pass& a, const Pass& b) { return a.work > b.work; });
  std::vector<PPItem> items;
  items.reserve(n);
  for (const Pass& p : passes) {
    const int nl = ctx->h_nlad[p.c], steps = (nl + 15) / 16;
    for (int q = 0; q < steps; q++)
      items.push_back(PPItem{p.c, q, p.n0, nr[p.c], nl, ctx->h_ch_sys[p.c], ctx->h_vd_off[p.c] + (long)q * steps * 256});
  }
  *dst = (PPItem*)dmalloc(ctx, sizeof(PPItem) * std::max<size_t>(1, n));
  if (n) CUDA_TRY(cudaMemcpyAsync(*dst, items.data(), sizeof(PPItem) * n, cudaMemcpyHostToDevice, ctx->stream));
  return (int)n;
}

// Work lists of the pp ladder (on first use): ladder rows (channel, ij), those the updates compute
// first, and the items of the computed rows.
void pnm_need_pp_lists(pnm_ctx* ctx) {
  if (ctx->pp_items) return;
  std::vector<int2> rows;
  rows.reserve(ctx->nrows);
  for (int part = 0; part < 2; part++) {
    for (int r = 0; r < ctx->nrows; r++)
      if (ctx->h_vpp[ctx->h_rows[r].x] && (ctx->h_row_mode[r] == 0) == (part == 1)) rows.push_back(ctx->h_rows[r]);
    if (part == 0) ctx->n_lad_rep = (int)rows.size();
  }
  ctx->n_lad_rows = (int)rows.size();
  ctx->lad_rows = (int2*)dmalloc(ctx, sizeof(int2) * std::max<size_t>(1, rows.size()));
  if (!rows.empty())
    CUDA_TRY(cudaMemcpyAsync(ctx->lad_rows, rows.data(), sizeof(int2) * rows.size(), cudaMemcpyHostToDevice, ctx->stream));
  ctx->n_pp_items = pp_work_list(ctx, ctx->h_n_urow, &ctx->pp_items);
}

void pnm_prepare_iteration(pnm_ctx* ctx) {
  cudaStream_t s = ctx->stream;
  int nsys = (int)ctx->sys.size();
  // per-system row ranges and LUT offsets
  std::vector<int> lo(nsys), hi(nsys), lut(nsys);
  for (int k = 0; k < nsys; k++) {
    lo[k] = ctx->sys[k].row_begin;
    hi[k] = ctx->sys[k].row_end;
    lut[k] = ctx->sys[k].lut_off;
  }
  int* d = (int*)dmalloc(ctx, sizeof(int) * 3 * nsys);
  CUDA_TRY(cudaMemcpyAsync(d, lo.data(), sizeof(int) * nsys, cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemcpyAsync(d + nsys, hi.data(), sizeof(int) * nsys, cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemcpyAsync(d + 2 * nsys, lut.data(), sizeof(int) * nsys, cudaMemcpyHostToDevice, s));
  ctx->row_lo_d = d;
  ctx->row_hi_d = d + nsys;
  ctx->lut_off_d = d + 2 * nsys;
  std::vector<int4> upd;
  std::vector<int> ulo(nsys), uhi(nsys);
  int max_npp = 0, max_nlad = 0;
  for (int c = 0; c < ctx->nch; c++) {
    int npp = ctx->h_npp[c];
    max_npp = std::max(max_npp, npp);
    if (!ctx->h_vpp[c]) continue;
    int nl = ctx->h_nlad[c];
    max_nlad = std::max(max_nlad, nl);
  }
  // per-row items (channel, ij, first column), 128 columns each, grouped by system (the
  // learned-start kernels)
  for (int k = 0; k < nsys; k++) {
    ulo[k] = (int)upd.size();
    for (int r = ctx->sys[k].row_begin; r < ctx->sys[k].row_end; r++) {
      int2 row = ctx->h_rows[r];
      for (int ab0 = 0; ab0 < ctx->h_npp[row.x]; ab0 += 128) upd.push_back(make_int4(row.x, row.y, ab0, 0));
    }
    uhi[k] = (int)upd.size();
  }
  int dev = 0, nsm = 148;
  CUDA_TRY(cudaGetDevice(&dev));
  CUDA_TRY(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  // rows the updates compute: of two rows that the spin flip maps onto each other the one
  // whose amplitudes come first, and the rows it maps onto themselves (half of their
  // columns); per channel a run of the list upd_row, which update items index
  const std::vector<int>& rmode = ctx->h_row_mode;
  std::vector<int> urow, uoff(ctx->nch + 1, 0), ucnt(ctx->nch, 0);
  for (int r = 0; r < ctx->nrows; r++)
    if (rmode[r]) ucnt[ctx->h_rows[r].x]++;
  for (int c = 0; c < ctx->nch; c++) uoff[c + 1] = uoff[c] + ucnt[c];
  urow.resize(uoff[ctx->nch]);
  std::fill(ucnt.begin(), ucnt.end(), 0);
  for (int r = 0; r < ctx->nrows; r++)
    if (rmode[r]) {
      int c = ctx->h_rows[r].x;
      urow[uoff[c] + ucnt[c]++] = ctx->h_rows[r].y;
    }
  ctx->h_n_urow.resize(ctx->nch);
  for (int c = 0; c < ctx->nch; c++) ctx->h_n_urow[c] = uoff[c + 1] - uoff[c];
  ctx->nsm = nsm;
  ctx->d.upd_row = (int*)dmalloc(ctx, sizeof(int) * std::max<size_t>(1, urow.size()));
  if (!urow.empty())
    CUDA_TRY(cudaMemcpyAsync(ctx->d.upd_row, urow.data(), sizeof(int) * urow.size(), cudaMemcpyHostToDevice, s));
  ctx->d.ch_uoff = (int*)dmalloc(ctx, sizeof(int) * (ctx->nch + 1));
  CUDA_TRY(cudaMemcpyAsync(ctx->d.ch_uoff, uoff.data(), sizeof(int) * (ctx->nch + 1), cudaMemcpyHostToDevice, s));
  // Chunks of the updates: 32 amplitudes of one channel each (its last is padded), a CTA's in one
  // system (padded chunks past its end).  A warp takes more than one where the GPU stays full: fewer
  // partial sums for the last CTA to add, and the block sums' FP64 additions count for more amplitudes.
  std::vector<int> glo(nsys), ghi(nsys);
  std::vector<int2> first(ctx->nch);
  std::vector<int2> pad(nsys);
  long n_chunks = 0;
  for (int c = 0; c < ctx->nch; c++) n_chunks += ((long)(uoff[c + 1] - uoff[c]) * ctx->h_npp[c] + 31) / 32;
  const int warps = UPD_THREADS / 32;
  ctx->upd_per_warp = 4;
  while (ctx->upd_per_warp > 1 && n_chunks < (long)UPD_FULL * nsm * warps * ctx->upd_per_warp) ctx->upd_per_warp >>= 1;
  const int per_cta = warps * ctx->upd_per_warp;
  n_chunks = 0;
  for (int k = 0; k < nsys; k++) {
    glo[k] = (int)(n_chunks / per_cta);
    for (int c = ctx->sys[k].ch_begin; c < ctx->sys[k].ch_end; c++) {
      first[c] = make_int2((int)n_chunks, ctx->n_stat);
      ctx->n_stat += ctx->h_nhh[c] * stat_groups(uoff[c + 1] - uoff[c]) + (ctx->h_npp[c] + 31) / 32;
      n_chunks += ((long)(uoff[c + 1] - uoff[c]) * ctx->h_npp[c] + 31) / 32;
    }
    pad[k].x = (int)n_chunks;
    // at least one CTA per system: it closes the system's update
    n_chunks = std::max<long>(glo[k] + 1, (n_chunks + per_cta - 1) / per_cta) * per_cta;
    pad[k].y = (int)n_chunks;
    ghi[k] = (int)(n_chunks / per_cta);
  }
  ctx->n_upd_ctas = (int)(n_chunks / per_cta);
  ctx->max_npp = max_npp;
  ctx->max_nlad = max_nlad;
  int max_nhh = 1;
  for (int c = 0; c < ctx->nch; c++) max_nhh = std::max(max_nhh, ctx->h_nhh[c]);
  ctx->max_nhh = max_nhh;
  if (max_nhh > UPD_MAX_NHH) throw PnmError{PNM_EINVAL, "more hole pairs in one channel than the update supports"};
  ctx->n_upd_items = (int)upd.size();
  ctx->upd_items = (int4*)dmalloc(ctx, sizeof(int4) * std::max<size_t>(1, upd.size()));
  if (!upd.empty())
    CUDA_TRY(cudaMemcpyAsync(ctx->upd_items, upd.data(), sizeof(int4) * upd.size(),
                             cudaMemcpyHostToDevice, s));
  int* ud = (int*)dmalloc(ctx, sizeof(int) * 2 * nsys);
  CUDA_TRY(cudaMemcpyAsync(ud, ulo.data(), sizeof(int) * nsys, cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemcpyAsync(ud + nsys, uhi.data(), sizeof(int) * nsys, cudaMemcpyHostToDevice, s));
  ctx->upd_lo_d = ud;
  ctx->upd_hi_d = ud + nsys;
  ctx->upd_chunks = (UpdItem*)dmalloc(ctx, sizeof(UpdItem) * std::max<long>(1, n_chunks));
  ctx->upd_z = (int*)dmalloc(ctx, sizeof(int) * 32 * std::max<long>(1, n_chunks));
  ctx->stat_items = (int4*)dmalloc(ctx, sizeof(int4) * std::max(1, ctx->n_stat));
  int2* dfirst = (int2*)dmalloc(ctx, sizeof(int2) * std::max(1, ctx->nch));
  int2* dpad = (int2*)dmalloc(ctx, sizeof(int2) * nsys);
  if (ctx->nch) CUDA_TRY(cudaMemcpyAsync(dfirst, first.data(), sizeof(int2) * ctx->nch, cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemcpyAsync(dpad, pad.data(), sizeof(int2) * nsys, cudaMemcpyHostToDevice, s));
  k_upd_chunks<<<ctx->nch + nsys, 128, 0, s>>>(ctx->d, ctx->nch, dfirst, dpad, ctx->upd_chunks, ctx->upd_z,
                                                  ctx->stat_items);
  CUDA_TRY(cudaGetLastError());
  int* gd = (int*)dmalloc(ctx, sizeof(int) * 2 * nsys);
  CUDA_TRY(cudaMemcpyAsync(gd, glo.data(), sizeof(int) * nsys, cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemcpyAsync(gd + nsys, ghi.data(), sizeof(int) * nsys, cudaMemcpyHostToDevice, s));
  ctx->grp_lo_d = gd;
  ctx->grp_hi_d = gd + nsys;
  // partial sums: one per update item (at least one per row for init/MBPT2)
  size_t nparts = std::max<size_t>(std::max<size_t>(upd.size(), ctx->n_upd_ctas), (size_t)ctx->nrows);
  ctx->d.eparts = (double*)dmalloc(ctx, sizeof(double) * nparts);
  ctx->d.rparts = (double*)dmalloc(ctx, sizeof(double) * nparts);
  ctx->ctl = (LoopCtl*)dmalloc(ctx, sizeof(LoopCtl));
  CUDA_TRY(cudaMemsetAsync(ctx->ctl, 0, sizeof(LoopCtl), s));
  ctx->blocks_done = (int*)dmalloc(ctx, sizeof(int) * nsys);
  CUDA_TRY(cudaMemsetAsync(ctx->blocks_done, 0, sizeof(int) * nsys, s));
  ctx->small = (double*)dmalloc(ctx, sizeof(double) * 8);
  ctx->sysctl = (SysCtl*)dmalloc(ctx, sizeof(SysCtl) * nsys);
  CUDA_TRY(cudaMemsetAsync(ctx->sysctl, 0, sizeof(SysCtl) * nsys, s));
  ctx->d.sysctl = ctx->sysctl;
  bool fits = max_nlad <= PP_MAX_NLAD;
  for (int x = 0; x < ctx->nx; x++) fits = fits && ph_fits(ctx->h_x_nph[x], ctx->h_x_nhp[x], ctx->h_x_cls[x]);
  if (!fits)
    throw PnmError{PNM_EINVAL, "channel too large for the shared-memory tiles"};
  for (int k = 0; k < 2; k++) {
    CUDA_TRY(cudaStreamCreateWithFlags(&ctx->side[k], cudaStreamNonBlocking));
    CUDA_TRY(cudaEventCreateWithFlags(&ctx->ev_join[k], cudaEventDisableTiming));
  }
  CUDA_TRY(cudaEventCreateWithFlags(&ctx->ev_fork, cudaEventDisableTiming));
  smem_at_least(k_tdig, sizeof(double) * max_nlad);
  smem_at_least(k_pp<double, false>, PP_SMEM);
  smem_at_least(k_pp<double, true>, PP_SMEM);
  smem_at_least(k_pp<f2, false>, PP_SMEM);
  smem_at_least(k_pp<f2, true>, PP_SMEM);
  CUDA_TRY(cudaStreamSynchronize(s));
}

void pnm_eref_all(pnm_ctx* ctx) {
  // E_ref = sum_i h0_ii + 1/2 sum_ij <ij|v|ij>, from the HF energies:
  // sum_i eps_i = sum_i h0_ii + sum_ij <ij|v|ij>, so E_ref = 1/2 (sum_i h0_ii + sum_i eps_i).
  cudaStream_t s = ctx->stream;
  std::vector<double> ekin(ctx->nsp_total), eps(ctx->nsp_total);
  CUDA_TRY(cudaMemcpyAsync(ekin.data(), ctx->d.ekin, sizeof(double) * ctx->nsp_total,
                           cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaMemcpyAsync(eps.data(), ctx->d.eps, sizeof(double) * ctx->nsp_total,
                           cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  for (auto& S : ctx->sys) {
    double a = 0, b = 0;
    for (int i = 0; i < S.N; i++) {
      a += ekin[S.sp_off + i];
      b += eps[S.sp_off + i];
    }
    S.eref = 0.5 * (a + b);
  }
}

void pnm_mbpt2_all(pnm_ctx* ctx, double* out) {
  cudaStream_t s = ctx->stream;
  int nsys = (int)ctx->sys.size();
  CUDA_TRY(cudaEventRecord(ctx->ev[0], s));
  k_mbpt2<false><<<ctx->nrows, 128, 0, s>>>(ctx->d, PNM_INIT_MBPT2);
  k_reduce_rows<<<nsys, 256, 0, s>>>(ctx->d.eparts, 0, ctx->row_lo_d, ctx->row_hi_d, ctx->d.rparts);
  CUDA_TRY(cudaGetLastError());
  CUDA_TRY(cudaEventRecord(ctx->ev[1], s));
  CUDA_TRY(cudaMemcpyAsync(out, ctx->d.rparts, sizeof(double) * nsys, cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  float ms = 0;
  cudaEventElapsedTime(&ms, ctx->ev[0], ctx->ev[1]);
  ctx->t_mbpt2 = ms;
}

// Third-order diagrams (Fig. goldstone, Eqs. diag3-diag5) from the MBPT2 amplitudes t0 held in
// D.t0, the pp ladder of t0 in D.rpp (channels with a V_pppp block) and the linear ph term of t0 in D.xq:
// the sums over the amplitudes of
//   (4)  t0_ab^ij sum_{c<d} <ab|v|cd> t0_cd^ij,
//   (5)  t0_ab^ij sum_{k<l} t0_ab^kl <kl|v|ij>,
//   (3)  t0_ab^ij [P(ij)P(ab) sum_kc <kb|v|cj> t0_ik^ac],
// a thread per amplitude of the update chunks (one of each spin-flip pair, counted twice), into
// parts[0..3) x CTAs.  Bound by the FP64 pipe (the hh sum); a CTA per row, most of whose block sums and
// threads idled in small channels, took 122 us for three N=66, N_max=36 systems, 87 so.
__global__ void __launch_bounds__(UPD_THREADS) k_mbpt3(DevState D, const UpdItem* __restrict__ items,
                                                       const int* __restrict__ upd_z, int per_warp,
                                                       double* __restrict__ parts) {
  __shared__ double red[UPD_THREADS / 32][3];
  const double* __restrict__ t = D.t0;
  double e4 = 0.0, e5 = 0.0, e3 = 0.0;
  for (int u = 0; u < per_warp; u++) {
    const long chunk = ((long)blockIdx.x * per_warp + u) * (UPD_THREADS / 32) + (threadIdx.x >> 5);
    const UpdItem it = items[chunk];
    const int zi = upd_z[chunk * 32 + (threadIdx.x & 31)];
    if (zi < 0) continue;  // padding
    const long z = zi;
    const int fc = D.fmap[z];
    const long f = (long)(fc > 0 ? fc : -fc) - 1;
    if (f < z) continue;
    const int e = (int)(z - it.base), ij = e / it.npp, ab = e - ij * it.npp, nh = it.nh, npp = it.npp;
    const double tz = (f == z ? 1.0 : 2.0) * t[z];
    const int4 q = D.qmap[z];
    double rl = 0.0;
    if (it.nl) {
      const int m = D.lad_map[it.pp_off + ab];
      rl = D.rpp[it.s_off + (long)ij * it.nl + ((m > 0 ? m : -m) - 1)];
      if (m < 0) rl = -rl;
    }
    const double q0 = q.x >= 0 ? D.xq[q.x] : 0.0, q1 = q.y >= 0 ? D.xq[q.y] : 0.0;
    const double q2 = q.z >= 0 ? D.xq[q.z] : 0.0, q3 = q.w >= 0 ? D.xq[q.w] : 0.0;
    const double* __restrict__ col = t + it.base + ab;
    const double* __restrict__ vh = D.v_hhhh + it.vhh_off + ij;
    double hh = 0.0;
#pragma unroll 4
    for (int kl = 0; kl < nh; kl++) hh = fma(col[(long)kl * npp], vh[(long)kl * nh], hh);
    e4 = fma(tz, rl, e4);
    e5 = fma(tz, hh, e5);
    e3 = fma(tz, ((q0 - q1) - q2) + q3, e3);
  }
  e4 = warp_sum(e4);
  e5 = warp_sum(e5);
  e3 = warp_sum(e3);
  if ((threadIdx.x & 31) == 0) {
    red[threadIdx.x >> 5][0] = e4;
    red[threadIdx.x >> 5][1] = e5;
    red[threadIdx.x >> 5][2] = e3;
  }
  __syncthreads();
  if (threadIdx.x < 3)
    parts[(long)threadIdx.x * gridDim.x + blockIdx.x] =
        (red[0][threadIdx.x] + red[1][threadIdx.x]) + (red[2][threadIdx.x] + red[3][threadIdx.x]);
}

// out[3 s + {0, 1, 2}] = diagrams (4), (5), (3) of system s.  Replaces the context's
// amplitudes by the MBPT2 guess.
void pnm_mbpt3_all(pnm_ctx* ctx, double* out) {
  cudaStream_t s = ctx->stream;
  pnm_need_digits(ctx);
  int nsys = (int)ctx->sys.size();
  const int n = ctx->n_upd_ctas;
  if (!ctx->mbpt3_buf) ctx->mbpt3_buf = (double*)dmalloc(ctx, sizeof(double) * (3 * (size_t)n + 3 * nsys));
  double* parts = ctx->mbpt3_buf;
  double* res = parts + 3 * (size_t)n;
  CUDA_TRY(cudaEventRecord(ctx->ev[0], s));
  // amplitudes of the start in t0, read by the contraction kernels (iteration parity 0, no
  // system frozen)
  CUDA_TRY(cudaMemsetAsync(&ctx->ctl->iter, 0, sizeof(int), s));
  CUDA_TRY(cudaMemsetAsync(&ctx->ctl->skip_done, 0, sizeof(int), s));
  k_mbpt2<true><<<ctx->nrows, 128, 0, s>>>(ctx->d, PNM_INIT_MBPT2);
  // the two terms side by side, as in an update: 485 instead of 510 us for three N=66, N_max=36 systems
  const bool side = pnm_concurrent(ctx);
  pnm_fork(ctx);
  pnm_launch_pp(ctx, side ? ctx->side[1] : s, true, false);
  if (ctx->nx > 0) launch_ph64(ctx, side ? ctx->side[0] : s, s, true);  // without cross channels no Q is read
  pnm_join(ctx);
  k_mbpt3<<<n, UPD_THREADS, 0, s>>>(ctx->d, ctx->upd_chunks, ctx->upd_z, ctx->upd_per_warp, parts);
  k_reduce_rows<<<dim3(nsys, 3), 256, 0, s>>>(parts, n, ctx->grp_lo_d, ctx->grp_hi_d, res);
  CUDA_TRY(cudaGetLastError());
  CUDA_TRY(cudaEventRecord(ctx->ev[1], s));
  std::vector<double> h(3 * (size_t)nsys);
  CUDA_TRY(cudaMemcpyAsync(h.data(), res, sizeof(double) * 3 * nsys, cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  for (int k = 0; k < 3; k++)
    for (int y = 0; y < nsys; y++) out[3 * y + k] = h[(size_t)k * nsys + y];
  float ms = 0;
  cudaEventElapsedTime(&ms, ctx->ev[0], ctx->ev[1]);
  ctx->t_mbpt3 = ms;
}

// The MBPT2 kernels of pnm_mbpt2_all with caller-chosen device buffers for the per-row
// partial sums (nrows doubles) and the per-system results (nsys doubles).
void pnm_launch_mbpt2_into(const pnm_ctx* ctx, double* partials, double* results) {
  DevState d = ctx->d;
  d.eparts = partials;
  k_mbpt2<false><<<ctx->nrows, 128, 0, ctx->stream>>>(d, PNM_INIT_MBPT2);
  k_reduce_rows<<<(int)ctx->sys.size(), 256, 0, ctx->stream>>>(partials, 0, ctx->row_lo_d, ctx->row_hi_d, results);
}

// The body of one update, enqueued on the context stream (FP64 path).
FinArgs fin_args(pnm_ctx* ctx, int use_cond, cudaGraphConditionalHandle h) {
  FinArgs f;
  f.eparts = ctx->d.eparts;
  f.rparts = ctx->d.rparts;
  f.lo = ctx->grp_lo_d;
  f.hi = ctx->grp_hi_d;
  f.nsys = (int)ctx->sys.size();
  f.blocks_done = ctx->blocks_done;
  f.sc = ctx->sysctl;
  f.hist = ctx->hist;
  f.hist_cap = ctx->hist_cap;
  f.use_cond = use_cond;
  f.handle = h;
  return f;
}

template <typename T_>
static void lad_expand(pnm_ctx* ctx, const T_* rs, int planes, long pstride) {
  cudaStream_t s = ctx->stream;
  if (!ctx->expand_buf) ctx->expand_buf = (double*)dmalloc(ctx, sizeof(double) * std::max<long>(ctx->nt, 1));
  if (ctx->nrows > 0)
    k_lad_expand<T_><<<ctx->nrows, 128, 0, s>>>(ctx->d, rs, planes, pstride, ctx->expand_buf);
  CUDA_TRY(cudaGetLastError());
}

void pnm_lad_expand(pnm_ctx* ctx, const float* rs, int planes, long pstride) {
  lad_expand(ctx, rs, planes, pstride);
}

void pnm_lad_expand(pnm_ctx* ctx, const double* rs, int planes, long pstride) {
  lad_expand(ctx, rs, planes, pstride);
}

void pnm_lad_expand(pnm_ctx* ctx, const f2* rs, int planes, long pstride) {
  lad_expand(ctx, rs, planes, pstride);
}

// The pp ladder in the ladder basis: the digits of the amplitudes, then the digit products
// (pair: results stored as FP32 pairs); the result stays in the ladder layout
// (consumers read it through lad_index).  rep_only: only the rows the updates compute (one of
// each spin-flip pair of rows); the ladder operator of pnm_apply_pp_ladder takes every row.
void pnm_launch_pp(pnm_ctx* ctx, cudaStream_t s, bool rep_only, bool pair) {
  // the digits of V are built before any capture by the host-side callers (pnm_need_vdig)
  if (!ctx->d.vdig) throw PnmError{PNM_EINVAL, "the ladder V has not been built"};
  if (ctx->n_lad_rows == 0) return;
  const int nrow = rep_only ? ctx->n_lad_rep : ctx->n_lad_rows;
  // the operator takes any amplitudes (it is not captured); in a solve the interaction decides
  const bool check = !rep_only || ctx->d.v64;
  if (check && !ctx->s64) ctx->s64 = (double*)dmalloc(ctx, sizeof(double) * std::max<long>(ctx->ns, 1));
  k_tdig<<<nrow, TDIG_THREADS, sizeof(double) * ctx->max_nlad, s>>>(ctx->d, ctx->ctl, ctx->lad_rows, check ? ctx->s64 : nullptr);
  if (!rep_only && !ctx->pp_items_all) ctx->n_pp_all = pp_work_list(ctx, ctx->h_nhh, &ctx->pp_items_all);
  const PPItem* items = rep_only ? ctx->pp_items : ctx->pp_items_all;
  const int n = rep_only ? ctx->n_pp_items : ctx->n_pp_all;
  // four warps per item where two would not fill the GPU twice over
  const int wk = (long)n * 2 < 2L * PP_WARPS * PP_CTAS * ctx->nsm ? 4 : 2;
  const unsigned nb = (unsigned)((n + PP_WARPS / wk - 1) / (PP_WARPS / wk));
  // no more ring than a warp has steps: a small system's CTAs then leave the SMs' split between L1
  // and shared memory as the neighbouring kernels need it
  const int steps = (ctx->max_nlad + 15) / 16;
  const int slots = std::min(PP_DEPTH, std::max(1, (steps + wk - 1) / wk));
  const size_t smem = PP_SMEM / PP_DEPTH * slots;
  auto go = [&](auto k) {
    k<<<nb, PP_WARPS * 32, smem, s>>>(ctx->d, ctx->ctl, items, n, rep_only ? 1 : 0, wk, slots, ctx->lut_off_d, ctx->s64);
  };
  if (check) {
    if (pair) go(k_pp<f2, true>);
    else go(k_pp<double, true>);
  } else {
    if (pair) go(k_pp<f2, false>);
    else go(k_pp<double, false>);
  }
}

// The ph term and the pp ladder do not depend on each other nor on the one-body sums: in a
// captured update they run on two side streams next to the stats kernels.  While kernels are
// being profiled one by one everything stays on the context stream.
bool pnm_concurrent(const pnm_ctx* ctx) {
  return !ctx->prof_live && !ctx->serial_sched[ctx->cur_mode];
}

void pnm_fork(pnm_ctx* ctx) {
  if (!pnm_concurrent(ctx)) return;
  CUDA_TRY(cudaEventRecord(ctx->ev_fork, ctx->stream));
  for (int k = 0; k < 2; k++) CUDA_TRY(cudaStreamWaitEvent(ctx->side[k], ctx->ev_fork, 0));
}

void pnm_join(pnm_ctx* ctx) {
  if (!pnm_concurrent(ctx)) return;
  for (int k = 0; k < 2; k++) {
    CUDA_TRY(cudaEventRecord(ctx->ev_join[k], ctx->side[k]));
    CUDA_TRY(cudaStreamWaitEvent(ctx->stream, ctx->ev_join[k], 0));
  }
}

// One-body intermediates and <kl|chi|ij> (shared by both precision modes, FP64).
// One-body sums, chi_hh and the one-body terms: FP64 (mixed = false) or from the FP32
// copies of the mixed-precision iteration.
void pnm_enqueue_stats(pnm_ctx* ctx, bool mixed, bool pair) {
  cudaStream_t s = ctx->stream;
  DevState& D = ctx->d;
  const int n = ctx->n_stat;
  unsigned nb = (unsigned)((n + 3) / 4);
  unsigned nd = (unsigned)((ctx->nsp_total * 32 + 255) / 256);
  prof_begin(ctx, mixed ? KID_TSTATS32 : KID_TSTATS);
  if (n == 0) {
  } else if (mixed) k_tstats<float><<<nb, 128, 0, s>>>(D, ctx->ctl, ctx->stat_items, n);
  else if (pair) k_tstats<double, true><<<nb, 128, 0, s>>>(D, ctx->ctl, ctx->stat_items, n, ctx->t_pair, ctx->vpphh_f2);
  else k_tstats<double><<<nb, 128, 0, s>>>(D, ctx->ctl, ctx->stat_items, n);
  prof_end(ctx);
  prof_begin(ctx, mixed ? KID_DCHI32 : KID_DCHI);
  if (mixed) k_dchi<float><<<nd, 256, 0, s>>>(D, ctx->nsp_total);
  else k_dchi<double><<<nd, 256, 0, s>>>(D, ctx->nsp_total);
  prof_end(ctx);
}

// One FP64 update.  terms (PNM_TERMS_*): the full Eq. (ccd3), or a truncation whose
// intermediates were fixed by pnm_prepare_terms (one-body terms zero, chi_kl^ij = <kl|v|ij>
// or zero, the ph term zero unless the linear ph term is launched here).
// pair: the ph and pp contractions with FP32-pair arithmetic (full Eq. ccd3 only).
static void enqueue_body_fp64(pnm_ctx* ctx, int use_cond, cudaGraphConditionalHandle h, int terms, bool pair) {
  cudaStream_t s_ph = pnm_concurrent(ctx) ? ctx->side[0] : ctx->stream;
  cudaStream_t s_pp = pnm_concurrent(ctx) ? ctx->side[1] : ctx->stream;
  bool ph_on = terms == PNM_TERMS_FULL || terms == PNM_TERMS_LINEAR;
  if (pair) pnm_split_cur(ctx, ctx->stream);  // before the fork: both branches read it
  pnm_fork(ctx);
  // the one-body kernels first beside the digit kernels: they are the shortest branch, and behind the
  // others they ended last (per update: N=66, N_max=42 303 -> 299 us, 28 nucleons 83 -> 80); last where
  // the tiny kernel takes every channel, whose FP64 work is then the longest branch (N=14, N_max=20: 32
  // us, first 39)
  const bool digits = ctx->n_ph_large + ctx->n_ph_cta + ctx->n_ph_warp > (pair ? ctx->n_ph_tiny : ctx->n_ph_tiny64);
  if (terms == PNM_TERMS_FULL && digits) pnm_enqueue_stats(ctx, false, pair);
  if (ctx->nx > 0 && ph_on) {
    prof_begin(ctx, pair ? KID_PH_F2 : KID_PH64);
    if (pair) launch_ph_f2(ctx, s_ph, ctx->stream);
    else launch_ph64(ctx, s_ph, ctx->stream, terms == PNM_TERMS_LINEAR);
    prof_end(ctx);
  }
  if (ctx->n_lad_rows > 0) {
    prof_begin(ctx, pair ? KID_PP_F2 : KID_PP64);
    pnm_launch_pp(ctx, s_pp, true, pair);
    prof_end(ctx);
  }
  if (terms == PNM_TERMS_FULL && !digits) pnm_enqueue_stats(ctx, false, pair);
  pnm_join(ctx);
  prof_begin(ctx, KID_UPDATE);
  launch_update64(ctx, use_cond, h, pair);
  prof_end(ctx);
}

const char* const pnm_kernel_names[PNM_NKERNELS] = {
    "k_tstats", "k_dchi", "k_ph64", "k_pp64", "k_update", "k_finalize(unused)",
    "k_pp_tc", "k_ph32", "k_tstats32", "k_update_mix", "k_pack", "k_dchi32", "k_ph_f2", "k_pp_f2"};

void prof_begin(pnm_ctx* ctx, int kid) {
  if (!ctx->prof_live) return;
  size_t k = ctx->prof_pending.size();
  if (k >= ctx->prof_ev.size()) {
    cudaEvent_t a, b;
    CUDA_TRY(cudaEventCreate(&a));
    CUDA_TRY(cudaEventCreate(&b));
    ctx->prof_ev.push_back({a, b});
  }
  ctx->prof_pending.push_back(kid);
  CUDA_TRY(cudaEventRecord(ctx->prof_ev[k].first, ctx->stream));
}

void prof_end(pnm_ctx* ctx) {
  if (!ctx->prof_live) return;
  CUDA_TRY(cudaEventRecord(ctx->prof_ev[ctx->prof_pending.size() - 1].second, ctx->stream));
}

void prof_collect(pnm_ctx* ctx) {
  for (size_t k = 0; k < ctx->prof_pending.size(); k++) {
    float ms = 0;
    CUDA_TRY(cudaEventSynchronize(ctx->prof_ev[k].second));
    CUDA_TRY(cudaEventElapsedTime(&ms, ctx->prof_ev[k].first, ctx->prof_ev[k].second));
    ctx->prof_ms[ctx->prof_pending[k]] += ms;
    ctx->prof_n[ctx->prof_pending[k]] += 1;
  }
  ctx->prof_pending.clear();
}

// mode = precision | (terms << 4) | (pair << 8); truncations (terms != 0) are FP64 only; pair
// selects the FP32-pair contractions for an FP64 update (the refinement sweeps).
void pnm_enqueue_body(pnm_ctx* ctx, int mode, int use_cond, cudaGraphConditionalHandle h) {
  int prec = mode & 15, terms = (mode >> 4) & 15;
  bool pair = ((mode >> 8) & 1) != 0;
  ctx->cur_mode = prec == PNM_PREC_FP64 ? (pair ? 2 : 0) : 1;
  if (prec == PNM_PREC_FP64) enqueue_body_fp64(ctx, use_cond, h, terms, pair);
  else pnm_enqueue_body_mixed(ctx, use_cond, h);
}

// The body of a device-side loop: several updates per evaluation of the loop condition, which costs
// about 5 us between two updates (N = 14, n^2 <= 20, mixed: 26.2 us per update with one update per
// body, 23.5 with two, 22.1 with four).  An update after the loop's end does nothing: its kernels see
// the loop status (sys_done and the updates themselves) and leave, about 8 us in all, so the
// refinement loop, usually two updates, takes two.
constexpr int LOOP_UPDATES = 4, LOOP_REFINE_UPDATES = 2;
void pnm_enqueue_loop_body(pnm_ctx* ctx, int mode, bool refine, cudaGraphConditionalHandle h) {
  for (int k = 0; k < (refine ? LOOP_REFINE_UPDATES : LOOP_UPDATES); k++) pnm_enqueue_body(ctx, mode, 1, h);
}

// The digits of both contractions: V_pppp and the ph term's fixed operands (once per context).
void pnm_need_digits(pnm_ctx* ctx) {
  pnm_need_vdig(ctx);
  pnm_need_phdig(ctx);
}

// What the sweeps with FP32-pair contractions add (once per context): the pair copy of V_pphh.
void pnm_prepare_f2(pnm_ctx* ctx) {
  if (ctx->t_pair) return;
  cudaStream_t s = ctx->stream;
  pnm_need_digits(ctx);
  ctx->t_pair = ctx_alloc<f2>(ctx, ctx->nt);
  ctx->vpphh_f2 = ctx_alloc<f2>(ctx, ctx->nt);
  pnm_split_f2(ctx->d.v_pphh, ctx->vpphh_f2, ctx->nt, s);
  CUDA_TRY(cudaGetLastError());
  CUDA_TRY(cudaStreamSynchronize(s));
}

// Fixed intermediates of a truncated iteration: no one-body terms, chi_kl^ij = <kl|v|ij>
// (hh ladder with the bare interaction) or zero (no hh ladder), and no ph term unless the
// linear one is recomputed every step.
void pnm_prepare_terms(pnm_ctx* ctx, int terms) {
  if (terms == PNM_TERMS_FULL) return;
  cudaStream_t s = ctx->stream;
  CUDA_TRY(cudaMemsetAsync(ctx->d.dchi, 0, sizeof(double) * ctx->nsp_total, s));
  if (terms == PNM_TERMS_PP) CUDA_TRY(cudaMemsetAsync(ctx->d.chi_hh, 0, sizeof(double) * ctx->nvhh, s));
  else CUDA_TRY(cudaMemcpyAsync(ctx->d.chi_hh, ctx->d.v_hhhh, sizeof(double) * ctx->nvhh,
                                cudaMemcpyDeviceToDevice, s));
  if (terms != PNM_TERMS_LINEAR && ctx->nxt > 0)
    CUDA_TRY(cudaMemsetAsync(ctx->d.xq, 0, sizeof(double) * ctx->nxt, s));
}

// Kernel nodes of a captured update: the ph term at the lowest priority, every other kernel at
// the highest, so that the shorter branches (pp ladder, one-body sums) are dispatched ahead of
// the many ph CTAs and run beside them instead of after them.
void pnm_set_node_priorities(cudaGraph_t body) {
  int least = 0, greatest = 0;
  CUDA_TRY(cudaDeviceGetStreamPriorityRange(&least, &greatest));
  size_t n = 0;
  CUDA_TRY(cudaGraphGetNodes(body, nullptr, &n));
  std::vector<cudaGraphNode_t> nodes(n);
  if (n) CUDA_TRY(cudaGraphGetNodes(body, nodes.data(), &n));
  for (cudaGraphNode_t nd : nodes) {
    cudaGraphNodeType t;
    CUDA_TRY(cudaGraphNodeGetType(nd, &t));
    if (t != cudaGraphNodeTypeKernel) continue;
    cudaKernelNodeParams kp = {};
    CUDA_TRY(cudaGraphKernelNodeGetParams(nd, &kp));
    cudaKernelNodeAttrValue v = {};
    v.priority = pnm_is_ph_kernel(kp.func) ? least : greatest;
    CUDA_TRY(cudaGraphKernelNodeSetAttribute(nd, cudaKernelNodeAttributePriority, &v));
  }
}

// Build (once per mode) a graph whose single node is a WHILE conditional looping the body.
static cudaGraphExec_t graph_for(pnm_ctx* ctx, int mode) {
  auto f = ctx->graphs.find(mode);
  if (f != ctx->graphs.end()) return f->second;
  const auto w0 = std::chrono::steady_clock::now();
  cudaGraph_t g;
  CUDA_TRY(cudaGraphCreate(&g, 0));
  cudaGraphConditionalHandle h;
  CUDA_TRY(cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault));
  cudaGraphNodeParams cp = {};
  cp.type = cudaGraphNodeTypeConditional;
  cp.conditional.handle = h;
  cp.conditional.type = cudaGraphCondTypeWhile;
  cp.conditional.size = 1;
  cudaGraphNode_t node;
  CUDA_TRY(cudaGraphAddNode(&node, g, nullptr, nullptr, 0, &cp));
  cudaGraph_t body = cp.conditional.phGraph_out[0];
  CUDA_TRY(cudaStreamBeginCaptureToGraph(ctx->stream, body, nullptr, nullptr, 0,
                                         cudaStreamCaptureModeThreadLocal));
  try {
    pnm_enqueue_loop_body(ctx, mode, false, h);
  } catch (...) {
    cudaGraph_t dummy;
    cudaStreamEndCapture(ctx->stream, &dummy);
    throw;
  }
  cudaGraph_t captured;
  CUDA_TRY(cudaStreamEndCapture(ctx->stream, &captured));
  pnm_set_node_priorities(body);
  cudaGraphExec_t ge;
  CUDA_TRY(cudaGraphInstantiate(&ge, g, cudaGraphInstantiateFlagUseNodePriority));
  ctx->graphs[mode] = ge;
  ctx->graph_defs[mode] = g;
  ctx->t_graph_host += std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - w0).count();
  return ge;
}

// Runs updates until every system meets its tolerance or the cap is hit.  Returns the
// loop status (1 converged, PNM_ENOTCONV, PNM_EDIVERGED).
int pnm_run_loop(pnm_ctx* ctx, int mode, int max_iter, int min_iter, int host_loop, double alpha, int* iter_out) {
  cudaStream_t s = ctx->stream;
  LoopCtl hc{};
  // keep iteration parity: ctl->iter is reset by k_start; only the limits, alpha and mode
  // are set here
  CUDA_TRY(cudaMemcpyAsync(&ctx->ctl->max_iter, &max_iter, sizeof(int), cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemcpyAsync(&ctx->ctl->min_iter, &min_iter, sizeof(int), cudaMemcpyHostToDevice, s));
  static const int kOne = 1, kZero = 0;
  CUDA_TRY(cudaMemcpyAsync(&ctx->ctl->alpha, &alpha, sizeof(double), cudaMemcpyHostToDevice, s));
  static const int kMode[2] = {0, 1};
  CUDA_TRY(cudaMemcpyAsync(&ctx->ctl->mode, &kMode[(mode & 15) == PNM_PREC_FP64 ? 0 : 1], sizeof(int),
                           cudaMemcpyHostToDevice, s));
  if (max_iter <= 0) return PNM_ENOTCONV;
  CUDA_TRY(cudaMemcpyAsync(&ctx->ctl->skip_done, &kOne, sizeof(int), cudaMemcpyHostToDevice, s));
  if (!host_loop) {
    cudaGraphExec_t ge = graph_for(ctx, mode);
    CUDA_TRY(cudaGraphLaunch(ge, s));
  } else {
    ctx->prof_live = ctx->prof_on;
    for (;;) {
      pnm_enqueue_body(ctx, mode, 0, 0);
      CUDA_TRY(cudaGetLastError());
      CUDA_TRY(cudaMemcpyAsync(&hc, ctx->ctl, sizeof(LoopCtl), cudaMemcpyDeviceToHost, s));
      CUDA_TRY(cudaStreamSynchronize(s));
      if (ctx->prof_live) prof_collect(ctx);
      if (hc.status != 0) break;
    }
    ctx->prof_live = false;
  }
  CUDA_TRY(cudaGetLastError());
  CUDA_TRY(cudaMemcpyAsync(&ctx->ctl->skip_done, &kZero, sizeof(int), cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemcpyAsync(&hc, ctx->ctl, sizeof(LoopCtl), cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
  if (iter_out) *iter_out = hc.iter;
  return hc.status;
}

// Initial amplitudes and their energy; resets iteration counters.
void pnm_start(pnm_ctx* ctx, int init, const std::vector<double>& tol) {
  cudaStream_t s = ctx->stream;
  int nsys = (int)ctx->sys.size();
  std::vector<SysCtl> hs(nsys);
  for (int k = 0; k < nsys; k++) {
    hs[k] = SysCtl{};
    hs[k].tol = tol[k];
  }
  CUDA_TRY(cudaMemcpyAsync(ctx->sysctl, hs.data(), sizeof(SysCtl) * nsys, cudaMemcpyHostToDevice, s));
  if (init == PNM_INIT_KEEP) pnm_flip_symmetrise(ctx, ctx->d.t0, s);
  k_mbpt2<true><<<ctx->nrows, 128, 0, s>>>(ctx->d, init);
  k_start<<<1, 256, 0, s>>>(ctx->d.eparts, ctx->row_lo_d, ctx->row_hi_d, nsys, ctx->sysctl,
                            ctx->ctl, ctx->hist, ctx->hist_cap);
  CUDA_TRY(cudaGetLastError());
}

// Reopen the convergence test of every system for a further phase (refinement), keeping
// amplitudes, energies and iteration counts.
__global__ void k_reopen(SysCtl* sc, int nsys, LoopCtl* ctl) {
  for (int s = 0; s < nsys; s++) {
    sc[s].done = 0;
    sc[s].grow = 0;
  }
  ctl->status = 0;
}

void pnm_reopen(pnm_ctx* ctx) {
  k_reopen<<<1, 1, 0, ctx->stream>>>(ctx->sysctl, (int)ctx->sys.size(), ctx->ctl);
  CUDA_TRY(cudaGetLastError());
}

// Make t0 hold the latest amplitudes (the loop leaves them in t[iter & 1]).
void pnm_settle_amplitudes(pnm_ctx* ctx) {
  int it = 0;
  CUDA_TRY(cudaMemcpyAsync(&it, &ctx->ctl->iter, sizeof(int), cudaMemcpyDeviceToHost, ctx->stream));
  CUDA_TRY(cudaStreamSynchronize(ctx->stream));
  if (it & 1) {
    CUDA_TRY(cudaMemcpyAsync(ctx->d.t0, ctx->d.t1, sizeof(double) * ctx->nt,
                             cudaMemcpyDeviceToDevice, ctx->stream));
    int zero = 0;
    CUDA_TRY(cudaMemcpyAsync(&ctx->ctl->iter, &zero, sizeof(int), cudaMemcpyHostToDevice, ctx->stream));
  }
  ctx->last_iters_host = it;
}

// ------------------------------------------------- device-side steps of a whole-solve graph
// Start of a solve: every system's control block cleared with its tolerance; kernels do not
// skip converged systems until the loop begins.
__global__ void k_solve_begin(SysCtl* __restrict__ sc, const double* __restrict__ tol, int nsys,
                              LoopCtl* __restrict__ ctl) {
  for (int k = threadIdx.x; k < nsys; k += blockDim.x) {
    SysCtl z = {};
    z.tol = tol[k];
    sc[k] = z;
  }
  if (threadIdx.x == 0) ctl->skip_done = 0;
}

// Parameters of the first iteration loop (what pnm_run_loop sets from the host).
__global__ void k_loop_begin(LoopCtl* __restrict__ ctl, const SolveParams* __restrict__ par, int mode) {
  ctl->max_iter = par->max_iter;
  ctl->min_iter = 0;
  ctl->alpha = par->alpha;
  ctl->mode = mode;
  ctl->skip_done = 1;
}

// After the mixed loop: if it converged, reopen every system for exactly refine_sweeps FP64
// updates and then the FP64 test (within max_iter more) and run the refinement loop; else
// skip it (the loop status stays the mixed loop's).
__global__ void k_refine_gate(LoopCtl* __restrict__ ctl, SysCtl* __restrict__ sc, int nsys,
                              const SolveParams* __restrict__ par, cudaGraphConditionalHandle h) {
  const bool go = ctl->status == 1;
  if (go) {
    for (int k = 0; k < nsys; k++) {
      sc[k].done = 0;
      sc[k].grow = 0;
    }
    const int it0 = ctl->iter;
    ctl->status = 0;
    ctl->max_iter = it0 + par->refine_sweeps + par->max_iter;
    ctl->min_iter = it0 + par->refine_sweeps;
    ctl->mode = 0;
  }
  cudaGraphSetConditional(h, go ? 1u : 0u);
}

__global__ void k_loop_end(LoopCtl* __restrict__ ctl) { ctl->skip_done = 0; }

// t0 = the latest amplitudes (the loop leaves them in t[iter & 1]); the iteration parity is
// reset by k_settle_reset once every block has copied.
__global__ void k_settle_copy(DevState D, const LoopCtl* __restrict__ ctl, long n) {
  if (!(ctl->iter & 1)) return;
  for (long z = (long)blockIdx.x * blockDim.x + threadIdx.x; z < n; z += (long)gridDim.x * blockDim.x)
    D.t0[z] = D.t1[z];
}
__global__ void k_settle_reset(LoopCtl* __restrict__ ctl) {
  if (ctl->iter & 1) ctl->iter = 0;
}

// The spin flips of the current FP64 amplitudes, the buffer chosen on the device.
__global__ void k_flip_copy_cur(DevState D, const LoopCtl* __restrict__ ctl, long n) {
  long z = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (z >= n) return;
  double* t = (ctl->iter & 1) ? D.t1 : D.t0;
  int cd = D.fmap[z];
  long f = (long)(cd > 0 ? cd : -cd) - 1;
  if (f > z) t[f] = cd > 0 ? t[z] : -t[z];
}

void pnm_solve_begin(pnm_ctx* ctx) {
  k_solve_begin<<<1, 256, 0, ctx->stream>>>(ctx->sysctl, ctx->d_tol, (int)ctx->sys.size(), ctx->ctl);
  CUDA_TRY(cudaGetLastError());
}

// Initial amplitudes and their energy (the device-side pnm_start: control blocks from
// k_solve_begin).
void pnm_start_device(pnm_ctx* ctx, int init) {
  cudaStream_t s = ctx->stream;
  if (init == PNM_INIT_KEEP) pnm_flip_symmetrise(ctx, ctx->d.t0, s);
  k_mbpt2<true><<<ctx->nrows, 128, 0, s>>>(ctx->d, init);
  k_start<<<1, 256, 0, s>>>(ctx->d.eparts, ctx->row_lo_d, ctx->row_hi_d, (int)ctx->sys.size(), ctx->sysctl,
                            ctx->ctl, ctx->hist, ctx->hist_cap);
  CUDA_TRY(cudaGetLastError());
}

void pnm_loop_begin(pnm_ctx* ctx, int mode) {
  k_loop_begin<<<1, 1, 0, ctx->stream>>>(ctx->ctl, ctx->d_par, (mode & 15) == PNM_PREC_FP64 ? 0 : 1);
  CUDA_TRY(cudaGetLastError());
}

void pnm_refine_gate(pnm_ctx* ctx, cudaGraphConditionalHandle h) {
  k_refine_gate<<<1, 1, 0, ctx->stream>>>(ctx->ctl, ctx->sysctl, (int)ctx->sys.size(), ctx->d_par, h);
  CUDA_TRY(cudaGetLastError());
}

void pnm_loop_end_settle(pnm_ctx* ctx) {
  cudaStream_t s = ctx->stream;
  k_loop_end<<<1, 1, 0, s>>>(ctx->ctl);
  if (ctx->nt > 0) {
    const long blocks = std::min<long>((ctx->nt + 255) / 256, 4096);
    k_settle_copy<<<(unsigned)blocks, 256, 0, s>>>(ctx->d, ctx->ctl, ctx->nt);
  }
  k_settle_reset<<<1, 1, 0, s>>>(ctx->ctl);
  CUDA_TRY(cudaGetLastError());
}

void pnm_flip_copy_device(pnm_ctx* ctx) {
  if (ctx->nt > 0)
    k_flip_copy_cur<<<(unsigned)((ctx->nt + 255) / 256), 256, 0, ctx->stream>>>(ctx->d, ctx->ctl, ctx->nt);
  CUDA_TRY(cudaGetLastError());
}

// Schedule tuning: time a few updates with the ph term and the pp ladder on side streams
// (concurrent with the one-body kernels) and a few with everything on one stream; keep the
// faster for this precision mode.  Where concurrent mixed updates take SCHED_ORDER_US or more, the
// orders of pnm_enqueue_body_mixed are timed too, as a graph with the priorities of the solve's (shorter
// updates gain nothing, and launches from the host would blur the difference).  The updates start from
// MBPT2, whatever is held (saved and restored): kernels skip their work once an iteration has ended, so the
// times of updates that diverge at once say nothing.  Where they do so from MBPT2 too (an interaction
// without a solution) the context keeps the concurrent schedule, untuned, and nothing is kept for the shape.
constexpr float SCHED_ORDER_US = 150.0f;
static std::mutex g_sched_mu;
static std::map<std::string, int> g_sched_cache;  // (shape key, mode) -> one stream (-1), or the order

// Milliseconds of four mixed updates as one graph.
static float time_body_graph(pnm_ctx* ctx, int mode, cudaEvent_t e0, cudaEvent_t e1) {
  cudaStream_t s = ctx->stream;
  cudaGraph_t g;
  CUDA_TRY(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
  try {
    for (int k = 0; k < 4; k++) pnm_enqueue_body(ctx, mode, 0, 0);
  } catch (...) {
    cudaGraph_t dummy;
    cudaStreamEndCapture(s, &dummy);
    throw;
  }
  CUDA_TRY(cudaStreamEndCapture(s, &g));
  cudaGraphExec_t ge = nullptr;
  float ms = 0;
  try {
    pnm_set_node_priorities(g);
    CUDA_TRY(cudaGraphInstantiate(&ge, g, cudaGraphInstantiateFlagUseNodePriority));
    CUDA_TRY(cudaGraphLaunch(ge, s));
    CUDA_TRY(cudaEventRecord(e0, s));
    CUDA_TRY(cudaGraphLaunch(ge, s));
    CUDA_TRY(cudaEventRecord(e1, s));
    CUDA_TRY(cudaEventSynchronize(e1));
    CUDA_TRY(cudaEventElapsedTime(&ms, e0, e1));
  } catch (...) {
    if (ge) cudaGraphExecDestroy(ge);
    cudaGraphDestroy(g);
    throw;
  }
  cudaGraphExecDestroy(ge);
  cudaGraphDestroy(g);
  return ms;
}

void pnm_tune_schedule(pnm_ctx* ctx, int mode, double alpha) {
  const bool pair = ((mode >> 8) & 1) != 0;
  int m = (mode & 15) == PNM_PREC_FP64 ? (pair ? 2 : 0) : 1;
  if (ctx->sched_tuned[m] || ctx->sched_ended[m]) return;
  if (m == 0) pnm_need_digits(ctx);
  const std::string key = pnm_shape_key(ctx) + (m == 1 ? "|mixed" : m == 2 ? "|pair" : "|fp64");
  {
    std::lock_guard<std::mutex> lock(g_sched_mu);
    auto f = g_sched_cache.find(key);
    if (f != g_sched_cache.end()) {
      ctx->serial_sched[m] = f->second < 0;
      if (m == 1) ctx->mixed_order = std::max(0, f->second);
      ctx->sched_tuned[m] = true;
      return;
    }
  }
  cudaStream_t s = ctx->stream;
  double* save = (double*)dmalloc(ctx, sizeof(double) * std::max<long>(ctx->nt, 1));
  CUDA_TRY(cudaMemcpyAsync(save, ctx->d.t0, sizeof(double) * ctx->nt, cudaMemcpyDeviceToDevice, s));
  std::vector<double> never(ctx->sys.size(), 0.0);
  int big = 1 << 30;
  CUDA_TRY(cudaMemcpyAsync(&ctx->ctl->max_iter, &big, sizeof(int), cudaMemcpyHostToDevice, s));
  cudaEvent_t e0, e1;
  CUDA_TRY(cudaEventCreate(&e0));
  CUDA_TRY(cudaEventCreate(&e1));
  float best = 1e30f;
  int best_serial = 0;
  bool ended = false;
  auto start = [&] {
    pnm_start(ctx, PNM_INIT_MBPT2, never);
    if (m == 1) pnm_mixed_pack_initial(ctx, alpha);
  };
  auto check = [&] {  // after a measurement
    int status = 0;
    CUDA_TRY(cudaMemcpyAsync(&status, &ctx->ctl->status, sizeof(int), cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
    ended = ended || status != 0;
  };
  for (int serial = 0; serial < 2; serial++) {
    ctx->serial_sched[m] = serial != 0;
    start();
    pnm_enqueue_body(ctx, mode, 0, 0);
    CUDA_TRY(cudaEventRecord(e0, s));
    for (int k = 0; k < 4; k++) pnm_enqueue_body(ctx, mode, 0, 0);
    CUDA_TRY(cudaEventRecord(e1, s));
    CUDA_TRY(cudaEventSynchronize(e1));
    float ms = 0;
    CUDA_TRY(cudaEventElapsedTime(&ms, e0, e1));
    check();
    if (ms < best) {
      best = ms;
      best_serial = serial;
    }
  }
  ctx->serial_sched[m] = best_serial != 0;
  if (m == 1 && !best_serial && best * 1e3f >= 4 * SCHED_ORDER_US) {
    float fastest = 1e30f;
    int order = 0;
    for (int k = 0; k < 3; k++) {
      ctx->mixed_order = k;
      start();
      const float ms = time_body_graph(ctx, mode, e0, e1);
      check();
      if (ms < 0.98f * fastest) {
        fastest = ms;
        order = k;
      }
    }
    ctx->mixed_order = order;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  ctx->sched_ended[m] = ended;
  if (ended) {
    ctx->serial_sched[m] = false;
    if (m == 1) ctx->mixed_order = 0;
  } else {
    ctx->sched_tuned[m] = true;
    std::lock_guard<std::mutex> lock(g_sched_mu);
    g_sched_cache[key] = ctx->serial_sched[m] ? -1 : (m == 1 ? ctx->mixed_order : 0);
  }
  CUDA_TRY(cudaMemcpyAsync(ctx->d.t0, save, sizeof(double) * ctx->nt, cudaMemcpyDeviceToDevice, s));
  CUDA_TRY(cudaGetLastError());
  CUDA_TRY(cudaStreamSynchronize(s));
}
