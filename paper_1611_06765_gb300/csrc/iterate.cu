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
//   k_ph       T_x = remap(t); C_x = V1_x + 1/2 W_x T_x; Q_x = T_x C_x per cross channel
//   k_pp       1/2 sum_cd <ab|v|cd> t_cd^ij, grouped over all channels with a V_pppp block (FP64
//              accuracy from digit products on the tensor cores)
//   k_update   Jacobi step t_new = (v + rest) / eps_ij^ab, mixing, energy/residual partials
//   finalize   (last block of k_update) Eq. (ccdcorr) energy per system, |dE| test,
//              device-side loop condition
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

// Blocks [0, nrows): row (c, kl): sij[kl] = sum_ab t v; chi_hh[kl][ij] for the ij the updates
// compute.
// Blocks [nrows, ...): column chunk (c, ab0): sab[ab] = sum_ij t v.
// PAIR (FP64 only): the contractions in FP32-pair arithmetic from the pair copies tp of t and vp
// of v_pphh (the refinement sweeps): chi_hh, and the one-body sums as per-thread pair partials
// added in FP64.
template <typename T_, bool PAIR = false>
__global__ void __launch_bounds__(128) k_tstats(DevState D, const LoopCtl* __restrict__ ctl,
                                                int nrows, const int2* __restrict__ ab_items,
                                                const f2* __restrict__ tp = nullptr,
                                                const f2* __restrict__ vp = nullptr) {
  __shared__ T_ sh32[32];
  StatsIO<T_> io(D, ctl);
  const T_* __restrict__ t = io.t;
  if ((int)blockIdx.x < nrows) {
    int2 it = D.row_item[blockIdx.x];
    int c = it.x, kl = it.y;
    if (sys_done(D, ctl, D.ch_sys[c])) return;
    int npp = D.ch_npp[c], nh = D.ch_nhh[c];
    long base = D.ch_t_off[c];
    const T_* tr = t + base + (long)kl * npp;
    const T_* vr = io.v + base + (long)kl * npp;
    T_ s = 0;
    if constexpr (PAIR) {
      // per-thread partial sums in FP32 pairs, the block sum in FP64
      const f2* __restrict__ tpr = tp + base + (long)kl * npp;
      const f2* __restrict__ vpr = vp + base + (long)kl * npp;
      f2 a2 = Arith<f2>::zero();
      for (int ab = threadIdx.x; ab < npp; ab += blockDim.x) Arith<f2>::mac(a2, tpr[ab], vpr[ab]);
      s = Arith<f2>::to_double(a2);
    } else {
      for (int ab = threadIdx.x; ab < npp; ab += blockDim.x) s += tr[ab] * vr[ab];
    }
    s = block_sum(s, sh32);
    if (threadIdx.x == 0) io.sij[D.ch_hh_off[c] + kl] = s;
    // chi is read only in the columns ij of the rows the updates compute (the list upd_row)
    int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int* __restrict__ rl = D.upd_row + D.ch_uoff[c];
    const int nr = D.ch_uoff[c + 1] - D.ch_uoff[c];
    for (int k = warp; k < nr; k += blockDim.x >> 5) {
      const int ij = rl[k];
      T_ acc = 0;
      if constexpr (PAIR) {
        const f2* __restrict__ vk = vp + base + (long)kl * npp;
        const f2* __restrict__ tj = tp + base + (long)ij * npp;
        f2 a2 = Arith<f2>::zero();
        for (int cd = lane; cd < npp; cd += 32) Arith<f2>::mac(a2, vk[cd], tj[cd]);
        for (int o = 16; o; o >>= 1)
          a2 = Arith<f2>::add(a2, f2{__shfl_xor_sync(0xffffffffu, a2.hi, o),
                                     __shfl_xor_sync(0xffffffffu, a2.lo, o)});
        acc = Arith<f2>::to_double(a2);
      } else {
        const T_* tj = t + base + (long)ij * npp;
        for (int cd = lane; cd < npp; cd += 32) acc += vr[cd] * tj[cd];
        acc = warp_sum(acc);
      }
      if (lane == 0) {
        long e = D.ch_vhh_off[c] + (long)kl * nh + ij;
        io.chi[e] = io.vhh[e] + acc;
      }
    }
  } else {
    int2 it = ab_items[blockIdx.x - nrows];
    int c = it.x, ab = it.y + threadIdx.x;
    if (sys_done(D, ctl, D.ch_sys[c])) return;
    int npp = D.ch_npp[c], nh = D.ch_nhh[c];
    if (ab < npp) {
      long base = D.ch_t_off[c] + ab;
      T_ s = 0;
      if constexpr (PAIR) {
        f2 a2 = Arith<f2>::zero();
        for (int ij = 0; ij < nh; ij++) Arith<f2>::mac(a2, tp[base + (long)ij * npp], vp[base + (long)ij * npp]);
        s = Arith<f2>::to_double(a2);
      } else {
        for (int ij = 0; ij < nh; ij++) s += t[base + (long)ij * npp] * io.v[base + (long)ij * npp];
      }
      io.sab[D.ch_pp_off[c] + ab] = s;
    }
  }
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

// ----------------------------------------------------------------------------- ph term
// Global spin flip: Q is formed for the cross channels with S_z > 0 and for the spin-up rows of
// the S_z = 0 channels; the update reads every other position at its flip (same value for
// flip-symmetric amplitudes; qmap holds the formed positions only).  In an
// S_z = 0 channel, with rows ordered (spin-up rows u, their flips F u) and columns alike,
// every matrix of the term has the block form [[A, B], [B, A]] (A = M[u][v], B = M[u][F v]);
// products of such matrices are formed from the half-size sums A + B and differences A - B,
//   (A_1 + B_1)(A_2 + B_2) = A_3 + B_3,  (A_1 - B_1)(A_2 - B_2) = A_3 - B_3,
// which is a quarter of the flops of the full channel.
template <typename T_, int TS>
struct VecT;
template <>
struct VecT<float, 2> {
  __device__ __forceinline__ static void ld(const float* p, float (&v)[2]) {
    float2 a = *reinterpret_cast<const float2*>(p);
    v[0] = a.x; v[1] = a.y;
  }
};
template <>
struct VecT<float, 4> {
  __device__ __forceinline__ static void ld(const float* p, float (&v)[4]) {
    float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  }
};
// Bytes reserved for the index tables at the start of a k_ph CTA's shared memory (R4 + 2 H4
// ints are used; 2 (R4 + H4) with R4, H4 even keeps the reservation a multiple of 16 bytes).
__host__ __device__ __forceinline__ size_t ph_index_bytes(int R4, int H4) { return sizeof(int) * 2 * (size_t)(R4 + H4); }

// One CTA (NT threads) per cross channel.  NM = 1: a channel with S_z > 0.  NM = 2: an S_z = 0
// channel as the pair (sum, difference) of half-size problems, Q written on its spin-up rows.
// Per problem, in shared memory zero-padded to multiples of TS (R rows (a,i), H columns (k,c)):
//   Ts = T (R x H), Xt = W^T staged as W (R x H), then T^T (H x R), Cs = C (H x H);
//   C[(k,c)][(j,b)] = <kb|v|cj> + 1/2 sum_(e,l) <kl|v|ce> t_lj^eb
//   Q[(a,i)][(j,b)] = sum_(k,c) t_ik^ac C[(k,c)][(j,b)]
// Each thread accumulates TS x TS outputs of every problem per tile.  Element arithmetic is
// that of Arith<T_> (FP64, FP32, or FP32 pairs with FP64 results).
template <typename T_, int NT, int TS, int NM>
__device__ __forceinline__ void ph_block(const DevState& D, int x, unsigned char* smraw,
                                         const T_* __restrict__ xt, const T_* __restrict__ xw,
                                         const T_* __restrict__ xv1, typename Arith<T_>::Out* __restrict__ xq) {
  using A = Arith<T_>;
  const int nph = D.x_nph[x], nhp = D.x_nhp[x];
  const int R = NM == 2 ? nph >> 1 : nph, H = NM == 2 ? nhp >> 1 : nhp;
  // padded to multiples of the register tile (zeros): the padding costs FMAs in the tiles
  const int R4 = (R + TS - 1) & ~(TS - 1), H4 = (H + TS - 1) & ~(TS - 1);
  const int RH = R4 * H4, HH = H4 * H4;
  // NM = 2: index tables in shared memory first (no chains of dependent global loads below):
  // sra[u] = spin-up row, sca[v] = spin-up column, scb[v] = its flip
  int* sra = reinterpret_cast<int*>(smraw);
  int* sca = sra + R4;
  int* scb = sca + H4;
  T_* Ts = reinterpret_cast<T_*>(smraw + ph_index_bytes(R4, H4));
  T_* Xt = Ts + NM * RH;
  T_* Cs = Xt + NM * RH;
  const long to = D.x_t_off[x], wo = D.x_w_off[x], co = D.x_c_off[x];
  if constexpr (NM == 2) {
    const int* __restrict__ fcol = D.x_fcol + D.x_hp_off[x];
    const int* __restrict__ rrow = D.x_rrow + D.x_ph_off[x];
    const int* __restrict__ rcol = D.x_rcol + D.x_hp_off[x];
    for (int k = threadIdx.x; k < R4; k += NT) sra[k] = k < R ? rrow[k] : 0;
    for (int k = threadIdx.x; k < H4; k += NT) {
      int a = k < H ? rcol[k] : 0;
      sca[k] = a;
      scb[k] = k < H ? fcol[a] : 0;
    }
    __syncthreads();
  }
  // element e = u H4 + s of the staging loops: (u, s) advanced by NT per step without a division
  const int du = NT / H4, ds = NT % H4;
  int u = threadIdx.x / H4, s = threadIdx.x % H4;
#pragma unroll 4
  for (int e = threadIdx.x; e < RH; e += NT) {
    T_ t0 = A::zero(), t1 = A::zero(), w0 = A::zero(), w1 = A::zero();
    if (u < R && s < H) {
      if constexpr (NM == 1) {
        long o = (long)u * nhp + s;
        t0 = xt[to + o];
        w0 = xw[wo + o];
      } else {
        int row = sra[u], ca = sca[s], cb = scb[s];
        long oa = (long)row * nhp + ca, ob = (long)row * nhp + cb;
        T_ ta = xt[to + oa], tb = xt[to + ob];
        t0 = A::add(ta, tb);
        t1 = A::sub(ta, tb);
        T_ wa = xw[wo + oa], wb = xw[wo + ob];
        w0 = A::add(wa, wb);
        w1 = A::sub(wa, wb);
      }
    }
    Ts[e] = t0;
    Xt[e] = w0;
    if constexpr (NM == 2) {
      Ts[RH + e] = t1;
      Xt[RH + e] = w1;
    }
    u += du;
    s += ds;
    if (s >= H4) {
      s -= H4;
      u++;
    }
  }
  int r = threadIdx.x / H4, c = threadIdx.x % H4;
#pragma unroll 4
  for (int e = threadIdx.x; e < HH; e += NT) {
    T_ v0 = A::zero(), v1 = A::zero();
    if (r < H && c < H) {
      if constexpr (NM == 1) {
        v0 = xv1[co + (long)r * nhp + c];
      } else {
        const long ra = co + (long)sca[r] * nhp;
        T_ va = xv1[ra + sca[c]], vb = xv1[ra + scb[c]];
        v0 = A::add(va, vb);
        v1 = A::sub(va, vb);
      }
    }
    Cs[e] = v0;
    if constexpr (NM == 2) Cs[HH + e] = v1;
    r += du;
    c += ds;
    if (c >= H4) {
      c -= H4;
      r++;
    }
  }
  __syncthreads();
  const int th = H4 / TS;
  {
    // C += 1/2 W^T T (padded rows and columns stay zero)
    for (int tile = threadIdx.x; tile < NM * th * th; tile += NT) {
      const int mtx = tile / (th * th), tt = tile % (th * th);
      const int r0 = (tt / th) * TS, s0 = (tt % th) * TS;
      const T_* X = Xt + mtx * RH;
      const T_* Tm = Ts + mtx * RH;
      T_ acc[TS][TS];
#pragma unroll
      for (int i = 0; i < TS; i++)
#pragma unroll
        for (int j = 0; j < TS; j++) acc[i][j] = A::zero();
      for (int u = 0; u < R; u++) {
        T_ a[TS], b[TS];
        VecT<T_, TS>::ld(X + u * H4 + r0, a);
        VecT<T_, TS>::ld(Tm + u * H4 + s0, b);
#pragma unroll
        for (int i = 0; i < TS; i++)
#pragma unroll
          for (int j = 0; j < TS; j++) A::mac(acc[i][j], a[i], b[j]);
      }
      T_* Cm = Cs + mtx * HH;
#pragma unroll
      for (int i = 0; i < TS; i++)
#pragma unroll
        for (int j = 0; j < TS; j++) {
          T_& cv = Cm[(r0 + i) * H4 + s0 + j];
          cv = A::add(cv, A::half(acc[i][j]));
        }
    }
    __syncthreads();
  }
  // T transposed into Xt: Xt[s][u] = T[u][s]
  for (int e = threadIdx.x; e < NM * RH; e += NT) {
    const int mtx = e / RH, f = e % RH;
    Xt[mtx * RH + (f % H4) * R4 + f / H4] = Ts[e];
  }
  __syncthreads();
  const int tr = R4 / TS;
  for (int tile = threadIdx.x; tile < tr * th; tile += NT) {
    const int r0 = (tile / th) * TS, s0 = (tile % th) * TS;
    T_ acc[NM][TS][TS];
#pragma unroll
    for (int m = 0; m < NM; m++)
#pragma unroll
      for (int i = 0; i < TS; i++)
#pragma unroll
        for (int j = 0; j < TS; j++) acc[m][i][j] = A::zero();
    for (int u = 0; u < H; u++) {
#pragma unroll
      for (int mtx = 0; mtx < NM; mtx++) {
        T_ a[TS], b[TS];
        VecT<T_, TS>::ld(Xt + mtx * RH + u * R4 + r0, a);
        VecT<T_, TS>::ld(Cs + mtx * HH + u * H4 + s0, b);
#pragma unroll
        for (int i = 0; i < TS; i++)
#pragma unroll
          for (int j = 0; j < TS; j++) A::mac(acc[mtx][i][j], a[i], b[j]);
      }
    }
#pragma unroll
    for (int i = 0; i < TS; i++) {
      const int r = r0 + i;
      if (r >= R) continue;
      if constexpr (NM == 1) {
        const long qr = to + (long)r * nhp;
#pragma unroll
        for (int j = 0; j < TS; j++)
          if (s0 + j < H) xq[qr + s0 + j] = A::out(acc[0][i][j]);
      } else {
        // the spin-up row's two blocks; the flipped rows are never read (see qpos)
        const long qa = to + (long)sra[r] * nhp;
#pragma unroll
        for (int j = 0; j < TS; j++) {
          const int s = s0 + j;
          if (s < H) {
            xq[qa + sca[s]] = A::out(A::half(A::add(acc[0][i][j], acc[1][i][j])));
            xq[qa + scb[s]] = A::out(A::half(A::sub(acc[0][i][j], acc[1][i][j])));
          }
        }
      }
    }
  }
}

// Cross channels of at most PH_WARP_DIM rows and columns (of their halves for S_z = 0): one
// warp per channel with its own shared buffers (stride PH_WARP_DIM), no block-wide
// synchronisation; the same two bodies as the CTA path, one output element per lane and step.
constexpr int PH_WARPS = PH_THREADS / 32;
template <typename T_>
__device__ __forceinline__ void ph_warp_body(const DevState& D, int x, int w, int lane, unsigned char* smraw,
                                             const T_* __restrict__ xt, const T_* __restrict__ xw,
                                             const T_* __restrict__ xv1, typename Arith<T_>::Out* __restrict__ xq) {
  using A = Arith<T_>;
  constexpr int S = PH_WARP_DIM;
  const int nph = D.x_nph[x], nhp = D.x_nhp[x];
  const bool two = D.x_cls[x] == 0;
  const int nm = two ? 2 : 1;
  const int R = two ? nph >> 1 : nph, H = two ? nhp >> 1 : nhp;
  const long to = D.x_t_off[x], wo = D.x_w_off[x], co = D.x_c_off[x];
  T_* Ts = reinterpret_cast<T_*>(smraw) + (size_t)w * 6 * S * S;  // [m][u][s]
  T_* Ws = Ts + 2 * S * S;                                         // [m][u][r] = W[u][r]
  T_* Cs = Ws + 2 * S * S;                                         // [m][r][s]
  int* sra = reinterpret_cast<int*>(reinterpret_cast<T_*>(smraw) + (size_t)PH_WARPS * 6 * S * S) + w * 3 * S;
  int* sca = sra + S;
  int* scb = sca + S;
  if (two) {
    const int* __restrict__ fcol = D.x_fcol + D.x_hp_off[x];
    const int* __restrict__ rrow = D.x_rrow + D.x_ph_off[x];
    const int* __restrict__ rcol = D.x_rcol + D.x_hp_off[x];
    if (lane < R) sra[lane] = rrow[lane];
    if (lane < H) {
      int a = rcol[lane];
      sca[lane] = a;
      scb[lane] = fcol[a];
    }
  }
  __syncwarp();
  for (int e = lane; e < R * H; e += 32) {
    int u = e / H, c = e % H;
    if (two) {
      long oa = (long)sra[u] * nhp + sca[c], ob = (long)sra[u] * nhp + scb[c];
      T_ ta = xt[to + oa], tb = xt[to + ob];
      Ts[u * S + c] = A::add(ta, tb);
      Ts[S * S + u * S + c] = A::sub(ta, tb);
      T_ wa = xw[wo + oa], wb = xw[wo + ob];
      Ws[u * S + c] = A::add(wa, wb);
      Ws[S * S + u * S + c] = A::sub(wa, wb);
    } else {
      long o = (long)u * nhp + c;
      Ts[u * S + c] = xt[to + o];
      Ws[u * S + c] = xw[wo + o];
    }
  }
  __syncwarp();
  for (int e = lane; e < H * H; e += 32) {
    int r = e / H, c = e % H;
    for (int m = 0; m < nm; m++) {
      T_ v;
      if (two) {
        const long ra = co + (long)sca[r] * nhp;
        T_ va = xv1[ra + sca[c]], vb = xv1[ra + scb[c]];
        v = m == 0 ? A::add(va, vb) : A::sub(va, vb);
      } else {
        v = xv1[co + (long)r * nhp + c];
      }
      T_ acc = A::zero();
      for (int u = 0; u < R; u++) A::mac(acc, Ws[m * S * S + u * S + r], Ts[m * S * S + u * S + c]);
      Cs[m * S * S + r * S + c] = A::add(v, A::half(acc));
    }
  }
  __syncwarp();
  for (int e = lane; e < R * H; e += 32) {
    int r = e / H, c = e % H;
    T_ acc[2] = {A::zero(), A::zero()};
    for (int m = 0; m < nm; m++)
      for (int u = 0; u < H; u++) A::mac(acc[m], Ts[m * S * S + r * S + u], Cs[m * S * S + u * S + c]);
    if (two) {
      const long qa = to + (long)sra[r] * nhp;
      xq[qa + sca[c]] = A::out(A::half(A::add(acc[0], acc[1])));
      xq[qa + scb[c]] = A::out(A::half(A::sub(acc[0], acc[1])));
    } else {
      xq[to + (long)r * nhp + c] = A::out(acc[0]);
    }
  }
}

// The ph term over the S_z >= 0 cross channels (xlist): the first nblk CTAs take one channel
// each (the costliest first), with the S_z > 0 or the S_z = 0 body chosen per channel; the
// remaining CTAs take PH_WARPS small channels each, one per warp.  (FP32, the mixed iteration.)
template <typename T_, int NT, int TS>
__global__ void __launch_bounds__(NT) k_ph(DevState D, const LoopCtl* __restrict__ ctl,
                                           const int* __restrict__ xlist, int nblk, int nwarp,
                                           const T_* __restrict__ xt, const T_* __restrict__ xw,
                                           const T_* __restrict__ xv1, typename Arith<T_>::Out* __restrict__ xq) {
  static_assert(NT == PH_WARPS * 32, "one warp per small channel");
  extern __shared__ __align__(16) unsigned char smraw[];
  if ((int)blockIdx.x < nblk) {
    const int x = xlist[blockIdx.x];
    if (sys_done(D, ctl, D.x_sys[x])) return;  // CTA-uniform
    if (D.x_cls[x] == 0)
      ph_block<T_, NT, TS, 2>(D, x, smraw, xt, xw, xv1, xq);
    else
      ph_block<T_, NT, TS, 1>(D, x, smraw, xt, xw, xv1, xq);
    return;
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int idx = ((int)blockIdx.x - nblk) * PH_WARPS + w;
  if (idx >= nwarp) return;  // whole warps leave; the warp path never synchronises the block
  const int x = xlist[nblk + idx];
  if (sys_done(D, ctl, D.x_sys[x])) return;  // warp-uniform
  ph_warp_body<T_>(D, x, w, lane, smraw, xt, xw, xv1, xq);
}

static size_t ph_warp_smem(size_t elem) {
  return (size_t)PH_WARPS * (6 * PH_WARP_DIM * PH_WARP_DIM * elem + 3 * PH_WARP_DIM * sizeof(int));
}

// Shared memory of a k_ph CTA for channels of at most max_dim (NM = 1) or 2 max_dim (NM = 2)
// rows and columns: the index tables, then NM problems of Ts, Xt (R x H) and Cs (H x H).
size_t ph_smem_bytes(int max_dim, int nm, size_t elem) {
  int m4 = (max_dim + 3) & ~3;
  return ph_index_bytes(m4, m4) + elem * 3 * (size_t)nm * m4 * m4;
}

static size_t ph32_smem(const pnm_ctx* ctx) {
  const size_t b = std::max(std::max(ctx->ph_smem32, ctx->ph_mid_smem32), ctx->ph_big_smem32);
  return ctx->n_ph_warp > 0 ? std::max(b, ph_warp_smem(sizeof(float))) : b;
}

// Register tile of the FP32 ph kernel (4 x 4: few shared-memory loads per FMA).
#ifndef PNM_PH32_TILE
#define PNM_PH32_TILE 4
#endif

// Mixed ph: T read from the FP32 cross-channel copy the update scatters, Q in FP32 at its
// cross-channel positions (the update gathers the four terms of each amplitude).
void launch_ph_mix(pnm_ctx* ctx, const float* xt, const float* xw, const float* xv1, float* xq, cudaStream_t s) {
  // one launch over the S_z >= 0 cross channels, the costliest first (limited by registers)
  const int nwb = (ctx->n_ph_warp + PH_WARPS - 1) / PH_WARPS;
  const int nblk = ctx->n_ph_big + ctx->n_ph_mid + ctx->n_ph;
  if (nblk + nwb > 0)
    k_ph<float, PH_THREADS, PNM_PH32_TILE><<<nblk + nwb, PH_THREADS, ph32_smem(ctx), s>>>(
        ctx->d, ctx->ctl, ctx->ph_list, nblk, ctx->n_ph_warp, xt, xw, xv1, xq);
}

// ------------------------------------------------------------- ph term, FP64 accuracy (digits)
// The FP64 and FP32-pair ph term as digit products on the tensor cores (dig.cuh), mma.sync because
// the matrices are small (N = 66: 17 to 33 rows and columns): per problem (a S_z > 0 channel, or
// the sum and the difference problem of an S_z = 0 channel)
//   C[(k,c)][(j,b)] = <kb|v|cj> + 1/2 sum_(e,l) <kl|v|ce> t_lj^eb,   Q[(a,i)][(j,b)] = T C.
// Operands are integers and their digits from end to end:
//   - the amplitudes as digit words of one exponent per system (k_tmax, k_twords: two passes over
//     them per update, where converting at the gather repeated the work for each of the three or
//     four places of an amplitude and cost two more passes over shared memory);
//   - W as digits in fragment order, <kb|v|cj> as integers, and the signed amplitude index of every
//     staged element, fixed per context (k_ph_pack; sums and differences of S_z = 0 formed there);
//   - T staged as words (sums and differences of S_z = 0 as exact integer sums), two neighbouring
//     columns interleaved: the k index of the second product; the first reads its k pairs across
//     rows;
//   - C as integers, the two terms aligned to the coarser of their units (2^-60 of their bounds or
//     finer), its digits stored interleaved by row pairs straight from the first product's registers.
// Only the results leave as floating point.  A group of 32 threads (channels of at most PH_WARP_DIM
// rows and columns) or of 128 (the others) takes a channel; a warp forms 16 x 8 blocks.
// What bounds it: instruction issue and its latencies around the products (operand expansion,
// drains, staging) at twelve warps per SM; without the MMAs it takes 6% less time.  Per launch with
// the two passes over the amplitudes: N = 66, n^2 <= 42, FP64 149 us against 405 us on the FP64
// pipe; three densities of N = 66, n^2 <= 36, pairs, 290 against 356 us on the FP32 pipe; symmetric
// matter, 28 nucleons, n^2 <= 20, FP64 50 against 52 us launched one by one, and shorter beside the
// ladder in a captured update (no FP64 pipe work to share).
struct __align__(16) PhItem {
  int x, sys;                    // cross channel, its system
  unsigned short R, H, nm, nhp;  // rows, columns of a problem; problems (1: S_z > 0, 2: S_z = 0); channel columns
  int po, ho;                    // pair offsets
  // offsets: Q, source indices, W fragments (uint4), <kb|v|cj>, and of the smallest channels W and
  // <kb|v|cj> as element values
  unsigned to, src, wf, v1, fx, pad;
};

__host__ __device__ __forceinline__ int ph_h8(int H) { return (H + 7) & ~7; }
// Row strides in 16-byte pairs: T's odd, C's 2 modulo 8, so that the fragment loads of the first
// product (two rows per thread) and of the second spread over the banks.
__host__ __device__ __forceinline__ int ph_ts(int H) { return ph_h8(H) / 2 + 1; }
__host__ __device__ __forceinline__ int ph_cs(int H) { return ph_h8(H) + 2; }
__host__ __device__ __forceinline__ size_t ph_dig_smem(int R, int H, int nm) {
  return sizeof(uint4) * nm * ((size_t)ph_h8(R) * ph_ts(H) + (size_t)(ph_h8(H) / 2) * ph_cs(H)) +
         sizeof(int) * ((size_t)ph_h8(R) + 2 * ph_h8(H));
}

template <int GT>
__device__ __forceinline__ void group_sync() {
  if constexpr (GT == 32) __syncwarp();
  else __syncthreads();
}

// The term of one channel in FP64 arithmetic (infinities, NaN, or values so large that intermediate
// results might overflow): the sums of the same expressions in order.
template <typename Out, int GT>
__device__ __noinline__ void ph_values(const DevState& D, const PhItem& it, int tid, uint4* Ts, uint4* Cs,
                                       const int* sra, const int* sca, const int* scb, const double* __restrict__ t,
                                       const int* __restrict__ src, bool quad, Out* __restrict__ xq) {
  const int R = it.R, H = it.H, nm = it.nm, H8 = ph_h8(H), TS = ph_ts(H), CS = ph_cs(H);
  const long TP = (long)ph_h8(R) * TS, CP = (long)(H8 / 2) * CS;
  auto T = [&](int m, int u, int s) -> double& { return reinterpret_cast<double*>(Ts + m * TP + u * TS + (s >> 1))[s & 1]; };
  auto C = [&](int m, int r, int c) -> double& { return reinterpret_cast<double*>(Cs + m * CP + (r >> 1) * CS + c)[r & 1]; };
  auto amp = [&](int c) { return c == 0 ? 0.0 : (c > 0 ? t[c - 1] : -t[-c - 1]); };
  const double* __restrict__ W = D.x_w + D.x_w_off[it.x];
  const double* __restrict__ V = D.x_v1 + D.x_c_off[it.x];
  for (int e = tid; e < R * H; e += GT) {
    const int u = e / H, s = e % H;
    if (nm == 1) T(0, u, s) = amp(src[it.src + u * H8 + s]);
    else {
      const int2 k = reinterpret_cast<const int2*>(src + it.src)[u * H8 + s];
      const double a = amp(k.x), b = amp(k.y);
      T(0, u, s) = a + b;
      T(1, u, s) = a - b;
    }
  }
  group_sync<GT>();
  for (int e = tid; e < nm * H * H; e += GT) {
    const int m = e / (H * H), r = (e % (H * H)) / H, c = e % H;
    auto pick = [&](const double* __restrict__ M, long row, int col) {  // element of problem m
      if (nm == 1) return M[row + col];
      const double a = M[row + sca[col]], b = M[row + scb[col]];
      return m == 0 ? a + b : a - b;
    };
    double acc = 0.0;
    for (int u = 0; u < R && quad; u++) acc += pick(W, (long)(nm == 1 ? u : sra[u]) * it.nhp, r) * T(m, u, c);
    C(m, r, c) = pick(V, (long)(nm == 1 ? r : sca[r]) * it.nhp, c) + 0.5 * acc;
  }
  group_sync<GT>();
  for (int e = tid; e < R * H; e += GT) {
    const int r = e / H, c = e % H;
    double acc[2] = {0.0, 0.0};
    for (int m = 0; m < nm; m++)
      for (int u = 0; u < H; u++) acc[m] += T(m, r, u) * C(m, u, c);
    if (nm == 1) xq[it.to + (long)r * it.nhp + c] = Arith<Out>::from_double(acc[0]);
    else {
      const long q = it.to + (long)sra[r] * it.nhp;
      xq[q + sca[c]] = Arith<Out>::from_double(0.5 * (acc[0] + acc[1]));
      xq[q + scb[c]] = Arith<Out>::from_double(0.5 * (acc[0] - acc[1]));
    }
  }
}

// Largest exponent of the amplitudes plus that of W beyond which ph_values is used: C and Q stay
// finite below.
constexpr int PH_MAX_EXP = 2900;

// ex: exponents of W and of <kb|v|cj>.
template <typename Out, int GT, int NM>
__device__ __forceinline__ void ph_dig(const DevState& D, const PhItem& it, int2 ex, unsigned char* smraw,
                                       const double* __restrict__ t, const int* __restrict__ src,
                                       const uint4* __restrict__ wf, const long long* __restrict__ v1, bool quad,
                                       Out* __restrict__ xq) {
  const int tid = GT == 32 ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3, wid = tid >> 5;
  constexpr int NW = GT / 32;
  const int R = it.R, H = it.H, R8 = ph_h8(R), H8 = ph_h8(H), TS = ph_ts(H), CS = ph_cs(H);
  const int TP = R8 * TS, CP = (H8 / 2) * CS;
  uint4* Ts = reinterpret_cast<uint4*>(smraw);  // [problem][row][column pair]
  uint4* Cs = Ts + NM * TP;                     // [problem][row pair][column]
  int* sra = reinterpret_cast<int*>(Cs + NM * CP);
  int* sca = sra + R8;
  int* scb = sca + H8;
  const int et = D.sys_texp[it.sys];
  if constexpr (NM == 2) {
    for (int k = tid; k < R; k += GT) sra[k] = D.x_rrow[it.po + k];
    for (int k = tid; k < H; k += GT) {
      const int a = D.x_rcol[it.ho + k];
      sca[k] = a;
      scb[k] = D.x_fcol[it.ho + a];
    }
  }
  if (et >= DIG_NONFINITE || ex.x >= DIG_NONFINITE || ex.y >= DIG_NONFINITE || et + ex.x > PH_MAX_EXP) {
    group_sync<GT>();  // the tables; group-uniform branch
    ph_values<Out, GT>(D, it, tid, Ts, Cs, sra, sca, scb, t, src, quad, xq);
    return;
  }
  // T: two neighbouring columns per step (index rows are padded to H8, rows past R read none)
  {
    const dig_t* __restrict__ tw = D.twords;
    auto word = [&](int c) {
      if (c == 0) return DIG_BIAS;
      const dig_t w = tw[c > 0 ? c - 1 : -c - 1];
      return c < 0 ? dig_neg(w) : w;
    };
    const int half = H8 / 2, total = R8 * half, live = R * half, du = GT / half, ds = GT % half;
    int u = tid / half, s = tid % half;
#pragma unroll 4
    for (int f = tid; f < total; f += GT) {
      uint4* pa = Ts + u * TS + s;
      if constexpr (NM == 1) {
        const int2 c = f < live ? reinterpret_cast<const int2*>(src + it.src)[f] : make_int2(0, 0);
        *pa = dig_interleave(word(c.x), word(c.y));
      } else {
        const int4 c = f < live ? reinterpret_cast<const int4*>(src + it.src)[f] : make_int4(0, 0, 0, 0);
        const dig_t a0 = word(c.x), b0 = word(c.y), a1 = word(c.z), b1 = word(c.w);
        *pa = dig_interleave(dig_sum(a0, b0), dig_sum(a1, b1));
        pa[TP] = dig_interleave(dig_diff(a0, b0), dig_diff(a1, b1));
      }
      u += du;
      s += ds;
      if (s >= half) {
        s -= half;
        u++;
      }
    }
  }
  group_sync<GT>();
  // C: 16 x 8 blocks of every problem; the fragments of W are requested one step ahead, across
  // blocks too
  const int nt = H8 / 8, sc = (H + 15) >> 4, kr = (R + 15) >> 4, blocks = NM * sc * nt;
  const int p1 = dig_power(ex.x, et) + 14 - 1, pv = ex.y - 1022 - 61;  // units of the two terms (factor 1/2)
  const int pc = quad ? max(p1, pv) : pv, sx = min(pc - p1, 63), sv = min(pc - pv, 63);
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
    dig_t c[4] = {(dig_t)(va.x >> sv), (dig_t)(va.y >> sv), (dig_t)(vb.x >> sv), (dig_t)(vb.y >> sv)};
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
        c[k] += (dig_t)(((x.hi << 18) + (x.lo >> 14)) >> sx);  // 2^-54 of the maxima's product or finer
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
  group_sync<GT>();
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
#pragma unroll
    for (int k = 0; k < 4; k++) {
      const int r = m0 + g + 8 * (k >> 1), c = n0 + 2 * q + (k & 1);
      if (r >= R || c >= H) continue;
      if constexpr (NM == 1) {
        xq[it.to + (long)r * it.nhp + c] = dig_result<Out>(x[k], p2);
      } else {
        // the spin-up row's two blocks; the flipped rows are never read (see qpos)
        const long o = it.to + (long)sra[r] * it.nhp;
        xq[o + sca[c]] = dig_result<Out>(DigSum{x0[k].hi + x[k].hi, x0[k].lo + x[k].lo}, p2);
        xq[o + scb[c]] = dig_result<Out>(DigSum{x0[k].hi - x[k].hi, x0[k].lo - x[k].lo}, p2);
      }
    }
  }
}

// Digit words of the current amplitudes of every system, of one exponent per system.  TW_PARTS CTAs
// per system find the largest exponents of their parts (k_tmax); k_twords reduces them (again in
// every CTA) and converts; part 0 publishes the system's exponent.
constexpr int TW_THREADS = 256, TW_PARTS = 512;
__global__ void __launch_bounds__(TW_THREADS) k_tmax(DevState D, const LoopCtl* __restrict__ ctl,
                                                     const long* __restrict__ t_lo, int* __restrict__ parts) {
  const int sys = blockIdx.y;
  if (sys_done(D, ctl, sys)) return;
  const double* __restrict__ t = cur_t(D, ctl);
  const long hi = t_lo[sys + 1];
  int e = 1;
#pragma unroll 4
  for (long z = t_lo[sys] + blockIdx.x * TW_THREADS + threadIdx.x; z < hi; z += gridDim.x * TW_THREADS)
    e = max(e, dig_exp(t[z]));
  e = __reduce_max_sync(0xffffffffu, e);
  __shared__ int top;
  if (threadIdx.x == 0) top = 1;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) atomicMax(&top, e);
  __syncthreads();
  if (threadIdx.x == 0) parts[sys * TW_PARTS + blockIdx.x] = top;
}

__global__ void __launch_bounds__(TW_THREADS) k_twords(DevState D, const LoopCtl* __restrict__ ctl,
                                                       const long* __restrict__ t_lo, const int* __restrict__ parts,
                                                       int nparts) {
  const int sys = blockIdx.y;
  if (sys_done(D, ctl, sys)) return;
  int e = 1;
  for (int k = threadIdx.x & 31; k < nparts; k += 32) e = max(e, parts[sys * TW_PARTS + k]);
  e = __reduce_max_sync(0xffffffffu, e);
  if (blockIdx.x == 0 && threadIdx.x == 0) D.sys_texp[sys] = e;
  if (e >= DIG_NONFINITE) return;  // the term is then formed from the FP64 values
  const double* __restrict__ t = cur_t(D, ctl);
  const long hi = t_lo[sys + 1];
#pragma unroll 4
  for (long z = t_lo[sys] + blockIdx.x * TW_THREADS + threadIdx.x; z < hi; z += gridDim.x * TW_THREADS)
    D.twords[z] = dig_word(dig_fixed(t[z], e));
}

// Channels of at most PH_TINY_DIM (FP32-pair results) or PH_TINY_FP64 (FP64 results) rows and
// columns per problem, one warp each, in the element arithmetic of the results, the pairs from the
// pair copy of the amplitudes: a 7 x 7 problem would fill a fifth of a 16 x 8 x 8 block.  120 systems
// of N = 14, all of whose channels are of this size: 695 us per launch in digits, 145 here (355 with
// one gather loop per channel in the kernel of the larger channels, at its registers).  In FP64 the
// line lies lower, the products then share the slow pipe: 28 nucleons, n^2 <= 20, take 94 us per
// update with a line at 5 and 99 with one at 8; N = 14, n^2 <= 20, whose channels have up to 7 rows,
// 34.8 and 36.0; n^2 <= 4 (up to 5 rows) 28.5, and in digits 30.
// fixed: W [problem][row][column] then <kb|v|cj> [problem][row][column] of the channel.
constexpr int PH_TINY_DIM = 8, PH_TINY_FP64 = 5;
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
    if (nm == 2) {
      const long q = it.to + (long)D.x_rrow[it.po + r] * it.nhp;
      const int ca = D.x_rcol[it.ho + c], cb = D.x_fcol[it.ho + ca];
      xq[q + ca] = A::half(A::add(acc[0], acc[1]));
      xq[q + cb] = A::half(A::sub(acc[0], acc[1]));
    } else {
      xq[it.to + (long)r * it.nhp + c] = acc[0];
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
  const double* __restrict__ t = cur_t(D, ctl);
  if ((int)blockIdx.x < nblk) {
    const PhItem it = items[blockIdx.x];
    if (sys_done(D, ctl, it.sys)) return;  // CTA-uniform
    const int2 ex = exps[blockIdx.x];
    if (it.nm == 2) ph_dig<Out, PH_THREADS, 2>(D, it, ex, smraw, t, src, wf, v1, quad != 0, xq);
    else ph_dig<Out, PH_THREADS, 1>(D, it, ex, smraw, t, src, wf, v1, quad != 0, xq);
    return;
  }
  const int w = threadIdx.x >> 5, idx = ((int)blockIdx.x - nblk) * PH_WARPS + w;
  if (idx >= nwarp) return;  // whole warps; the warp path never synchronises the block
  const PhItem it = items[nblk + idx];
  if (sys_done(D, ctl, it.sys)) return;
  const int2 ex = exps[nblk + idx];
  unsigned char* sm = smraw + (size_t)w * warp_smem;
  if (it.nm == 2) ph_dig<Out, 32, 2>(D, it, ex, sm, t, src, wf, v1, quad != 0, xq);
  else ph_dig<Out, 32, 1>(D, it, ex, sm, t, src, wf, v1, quad != 0, xq);
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
// the problems as integers (padded to whole blocks) and the digits of W, with their exponents.
__global__ void __launch_bounds__(128) k_ph_pack(DevState D, const PhItem* __restrict__ items, int2* __restrict__ exps,
                                                 int* __restrict__ src, uint4* __restrict__ wf, long long* __restrict__ v1,
                                                 double* __restrict__ fixed64, f2* __restrict__ fixed_f2) {
  __shared__ int top[2];
  const PhItem it = items[blockIdx.x];
  const int R = it.R, H = it.H, H8 = ph_h8(H);
  const int* __restrict__ rr = D.x_rrow + it.po;
  const int* __restrict__ rc = D.x_rcol + it.ho;
  const int* __restrict__ fc = D.x_fcol + it.ho;
  const double* __restrict__ W = D.x_w + D.x_w_off[it.x];
  const double* __restrict__ V = D.x_v1 + D.x_c_off[it.x];
  const bool two = it.nm == 2;
  const bool tiny = max(R, H) <= PH_TINY_DIM;  // element values too
  auto put = [&](long o, double v) {
    fixed64[it.fx + o] = v;
    fixed_f2[it.fx + o] = Arith<f2>::from_double(v);
  };
  if (threadIdx.x < 2) top[threadIdx.x] = 1;
  __syncthreads();
  int e = 1;
  for (int f = threadIdx.x; f < R * H8; f += blockDim.x) {
    const int u = f / H8, s = f % H8, o = u * H + s;
    if (two) {
      int2 c = make_int2(0, 0);
      if (s < H) {
        const long oa = (long)rr[u] * it.nhp + rc[s], ob = (long)rr[u] * it.nhp + fc[rc[s]];
        c = make_int2(D.xmap[it.to + oa], D.xmap[it.to + ob]);
        e = max(e, max(dig_exp(W[oa]), dig_exp(W[ob])));
        if (tiny) {
          put(o, W[oa] + W[ob]);
          put(R * H + o, W[oa] - W[ob]);
        }
      }
      reinterpret_cast<int2*>(src + it.src)[f] = c;
    } else {
      src[it.src + f] = s < H ? D.xmap[it.to + o] : 0;
      if (s < H) {
        e = max(e, dig_exp(W[o]));
        if (tiny) put(o, W[o]);
      }
    }
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) atomicMax(&top[0], e);
  e = 1;
  for (int f = threadIdx.x; f < H * H; f += blockDim.x) {
    const int r = f / H, c = f % H;
    if (two) {
      const double a = V[(long)rc[r] * it.nhp + rc[c]], b = V[(long)rc[r] * it.nhp + fc[rc[c]]];
      e = max(e, max(dig_exp(a), dig_exp(b)));
      if (tiny) {
        put(2 * R * H + f, a + b);
        put(2 * R * H + H * H + f, a - b);
      }
    } else {
      const double a = V[(long)r * it.nhp + c];
      e = max(e, dig_exp(a));
      if (tiny) put(R * H + f, a);
    }
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) atomicMax(&top[1], e);
  __syncthreads();
  const int ew = top[0], ev = top[1];
  if (threadIdx.x == 0) exps[blockIdx.x] = make_int2(ew, ev);
  if (ew >= DIG_NONFINITE || ev >= DIG_NONFINITE) return;
  const int sc = (H + 15) >> 4, kr = (R + 15) >> 4;
  for (int f = threadIdx.x; f < sc * 16 * H8; f += blockDim.x) {
    const int r = f / H8, c = f % H8;
    long long sum = 0, dif = 0;
    if (r < H && c < H) {
      if (two) {
        const long long a = dig_fixed(V[(long)rc[r] * it.nhp + rc[c]], ev);
        const long long b = dig_fixed(V[(long)rc[r] * it.nhp + fc[rc[c]]], ev);
        sum = a + b;
        dif = a - b;
      } else {
        sum = dig_fixed(V[(long)r * it.nhp + c], ev);
      }
    }
    v1[it.v1 + f] = sum;
    if (two) v1[it.v1 + (long)sc * 16 * H8 + f] = dif;
  }
  // fragment order of W as the first operand: rows (k,c), columns (e,l); stored transposed in x_w
  for (int f = threadIdx.x; f < sc * kr * 128; f += blockDim.x) {
    const int lane = f & 31, grp = (f >> 5) & 3, ks = (f >> 7) % kr, strip = (f >> 7) / kr;
    const int r = strip * 16 + (lane >> 2) + (grp & 1) * 8, u0 = ks * 16 + (lane & 3) * 2 + (grp >> 1) * 8;
    long long sum[2] = {0, 0}, dif[2] = {0, 0};
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const int u = u0 + k;
      if (r >= H || u >= R) continue;
      if (two) {
        const long o = (long)rr[u] * it.nhp;
        const long long a = dig_fixed(W[o + rc[r]], ew), b = dig_fixed(W[o + fc[rc[r]]], ew);
        sum[k] = a + b;
        dif[k] = a - b;
      } else {
        sum[k] = dig_fixed(W[(long)u * it.nhp + r], ew);
      }
    }
    wf[it.wf + f] = dig_interleave(dig_word(sum[0]), dig_word(sum[1]));
    if (two) wf[it.wf + (long)sc * kr * 128 + f] = dig_interleave(dig_word(dif[0]), dig_word(dif[1]));
  }
}

// Items and fixed operands of the digit ph term (once per context, on first use): the costliest
// channels first, in ph_list's order; channels whose tiles need more than PH_DIG_SMEM bytes get a
// launch of their own so that the others keep three CTAs per SM.
constexpr size_t PH_DIG_SMEM = 72 * 1024;
void pnm_need_phdig(pnm_ctx* ctx) {
  if (ctx->ph_items) return;
  cudaStream_t s = ctx->stream;
  const int n = ctx->n_ph_big + ctx->n_ph_mid + ctx->n_ph, nw = ctx->n_ph_warp;
  std::vector<PhItem> items;
  items.reserve(n + nw);
  long wf = 0, v1 = 0, src = 0, fixed = 0;
  ctx->ph_warp_smem = 0;
  ctx->n_ph_large = 0;
  ctx->ph_large_smem = ctx->ph_dig_smem = 0;
  auto add = [&](int x) {
    PhItem it{};
    it.x = x;
    it.sys = ctx->h_x_sys[x];
    it.nm = ctx->h_x_cls[x] == 0 ? 2 : 1;
    it.R = ctx->h_x_nph[x] / it.nm;
    it.H = ctx->h_x_nhp[x] / it.nm;
    it.nhp = ctx->h_x_nhp[x];
    it.po = ctx->h_x_ph_off[x];
    it.ho = ctx->h_x_hp_off[x];
    it.to = (unsigned)ctx->h_x_t_off[x];
    it.src = (unsigned)src;
    src += (long)it.nm * it.R * ph_h8(it.H);
    it.wf = (unsigned)wf;
    it.v1 = (unsigned)v1;
    it.fx = (unsigned)fixed;
    wf += (long)it.nm * ((it.H + 15) / 16) * ((it.R + 15) / 16) * 128;
    v1 += (long)it.nm * ((it.H + 15) / 16) * 16 * ph_h8(it.H);
    const bool tiny = std::max(it.R, it.H) <= PH_TINY_DIM;
    if (tiny) fixed += (long)it.nm * it.H * (it.R + it.H);
    items.push_back(it);
    return ph_dig_smem(it.R, it.H, it.nm);
  };
  for (int part = 0; part < 2; part++)
    for (int k = 0; k < n; k++) {
      const int x = ctx->h_ph_list[k], nm = ctx->h_x_cls[x] == 0 ? 2 : 1;
      if ((ph_dig_smem(ctx->h_x_nph[x] / nm, ctx->h_x_nhp[x] / nm, nm) > PH_DIG_SMEM) != (part == 0)) continue;
      const size_t b = add(x);
      size_t& most = part == 0 ? ctx->ph_large_smem : ctx->ph_dig_smem;
      most = std::max(most, b);
      if (part == 0) ctx->n_ph_large++;
    }
  // the warp path by decreasing dimension: the tiny channels of either result type are its end
  std::vector<int> by_dim[PH_WARP_DIM + 1];
  for (int k = 0; k < nw; k++) {
    const int x = ctx->h_ph_list[n + k];
    by_dim[std::max(ctx->h_x_nph[x], ctx->h_x_nhp[x]) / (ctx->h_x_cls[x] == 0 ? 2 : 1)].push_back(x);
  }
  ctx->n_ph_tiny64 = ctx->n_ph_tiny_f2 = 0;
  for (int d = PH_WARP_DIM; d >= 0; d--) {
    for (int x : by_dim[d]) ctx->ph_warp_smem = std::max(ctx->ph_warp_smem, (add(x) + 15) / 16 * 16);
    if (d <= PH_TINY_FP64) ctx->n_ph_tiny64 += (int)by_dim[d].size();
    if (d <= PH_TINY_DIM) ctx->n_ph_tiny_f2 += (int)by_dim[d].size();
  }
  if (std::max(std::max(wf, v1), std::max(src, fixed)) >= (1L << 32))
    throw PnmError{PNM_EINVAL, "problem too large for 32-bit element maps"};
  ctx->ph_dig_smem = std::max(ctx->ph_dig_smem, PH_WARPS * ctx->ph_warp_smem);
  PhItem* d = ctx_alloc<PhItem>(ctx, items.size());
  ctx->ph_exps = ctx_alloc<int2>(ctx, items.size());
  ctx->ph_src = ctx_alloc<int>(ctx, src);
  ctx->ph_wf = ctx_alloc<uint4>(ctx, wf);
  ctx->ph_v1 = ctx_alloc<long long>(ctx, v1);
  ctx->ph_fixed64 = ctx_alloc<double>(ctx, fixed);
  ctx->ph_fixed_f2 = ctx_alloc<f2>(ctx, fixed);
  if (!items.empty()) {
    CUDA_TRY(cudaMemcpyAsync(d, items.data(), sizeof(PhItem) * items.size(), cudaMemcpyHostToDevice, s));
    k_ph_pack<<<(unsigned)items.size(), 128, 0, s>>>(ctx->d, d, ctx->ph_exps, ctx->ph_src, ctx->ph_wf, ctx->ph_v1,
                                                        ctx->ph_fixed64, ctx->ph_fixed_f2);
    CUDA_TRY(cudaGetLastError());
  }
  const int nsys = (int)ctx->sys.size();
  std::vector<long> lo(nsys + 1, ctx->nt);
  long longest = 0;
  for (int k = 0; k < nsys; k++) {
    lo[k] = ctx->sys[k].t_begin;
    longest = std::max(longest, ctx->sys[k].t_end - ctx->sys[k].t_begin);
  }
  // parts of about a thousand amplitudes
  ctx->n_tw_parts = (int)std::max<long>(1, std::min<long>(TW_PARTS, longest / (4 * TW_THREADS)));
  ctx->tw_lo = ctx_alloc<long>(ctx, nsys + 1);
  ctx->tw_parts = ctx_alloc<int>(ctx, (size_t)nsys * TW_PARTS);
  ctx->d.sys_texp = ctx_alloc<int>(ctx, nsys);
  ctx->d.twords = ctx_alloc<unsigned long long>(ctx, ctx->nt);
  CUDA_TRY(cudaMemcpyAsync(ctx->tw_lo, lo.data(), sizeof(long) * (nsys + 1), cudaMemcpyHostToDevice, s));
  const size_t most = std::max(ctx->ph_large_smem, ctx->ph_dig_smem);
  smem_at_least(k_ph_dig<double>, most);
  smem_at_least(k_ph_dig<f2>, most);
  ctx->ph_items = d;
}

template <typename Out>
static void launch_ph_dig(pnm_ctx* ctx, bool linear, cudaStream_t s, cudaStream_t s_tiny) {
  // made before any capture by the host-side callers
  if (!ctx->ph_items) throw PnmError{PNM_EINVAL, "the ph term's operands have not been built"};
  constexpr bool pair = std::is_same<Out, f2>::value;
  const int nl = ctx->n_ph_large, n = ctx->n_ph_big + ctx->n_ph_mid + ctx->n_ph - nl;
  const int ntiny = pair ? ctx->n_ph_tiny_f2 : ctx->n_ph_tiny64, nw = ctx->n_ph_warp - ntiny;
  const int nwb = (nw + PH_WARPS - 1) / PH_WARPS, quad = linear ? 0 : 1;
  Out* xq = reinterpret_cast<Out*>(ctx->d.xq);
  const PhItem* items = ctx->ph_items;
  if (nl + n + nw == 0) s_tiny = s;
  if (nl + n + nw > 0) {
    const dim3 grid(ctx->n_tw_parts, (unsigned)ctx->sys.size());
    k_tmax<<<grid, TW_THREADS, 0, s>>>(ctx->d, ctx->ctl, ctx->tw_lo, ctx->tw_parts);
    k_twords<<<grid, TW_THREADS, 0, s>>>(ctx->d, ctx->ctl, ctx->tw_lo, ctx->tw_parts, ctx->n_tw_parts);
  }
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
// s_tiny: the stream of the smallest channels, which wait for no digits (a captured update runs them
// beside the two passes over the amplitudes; in a context without larger channels they keep s).
void launch_ph64(pnm_ctx* ctx, cudaStream_t s, cudaStream_t s_tiny, bool linear) {
  launch_ph_dig<double>(ctx, linear, s, s_tiny);
}
void launch_ph_f2(pnm_ctx* ctx, cudaStream_t s, cudaStream_t s_tiny) { launch_ph_dig<f2>(ctx, false, s, s_tiny); }

// ------------------------------------------------------------------------ ladder basis
// s(ij, q) = sum over the (one or two) pairs of vector q of sign * t(ij, pair) from the current
// FP64 amplitudes, as digit words of the row's common exponent (dig.cuh), zero words in the
// padding.  One CTA per (channel, ij) row of a channel with V_pppp.  A row that holds an infinity
// or a NaN keeps its FP64 values instead of digits (exponent DIG_NONFINITE; the ladder kernel
// then sums it in FP64).
constexpr int TDIG_THREADS = 128;
__global__ void __launch_bounds__(TDIG_THREADS) k_tdig(DevState D, const LoopCtl* __restrict__ ctl,
                                                       const int2* __restrict__ rows) {
  extern __shared__ double ssum[];
  __shared__ int warp_max[TDIG_THREADS / 32];
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
    e = max(e, dig_exp(v));
  }
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = e;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < TDIG_THREADS / 32; w++) e = max(e, warp_max[w]);
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
    if (e < DIG_NONFINITE) {
      uint32_t b0[8], b1[8];
      dig_expand<8>(dig_interleave(dig_word(dig_fixed(v[0], e)), dig_word(dig_fixed(v[1], e))), b0);
      dig_expand<8>(dig_interleave(dig_word(dig_fixed(v[2], e)), dig_word(dig_fixed(v[3], e))), b1);
#pragma unroll
      for (int u = 0; u < 4; u++) o[f * 4 + u] = make_uint4(b0[2 * u], b1[2 * u], b0[2 * u + 1], b1[2 * u + 1]);
    } else {
      double* raw = reinterpret_cast<double*>(o + f * 4);
#pragma unroll
      for (int u = 0; u < 4; u++) raw[u] = v[u];
    }
  }
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
// through mma.sync) for many.  Per launch with k_tdig (N = 66, n^2 <= 42, FP64): 80 us (V 250 MB in
// 60 us, 4.2 TB/s) against 291 us on the FP64 pipe; symmetric matter, 28 nucleons, n^2 <= 20: 43
// against 119 us; three densities of N = 66, n^2 <= 36, pairs: 126 against 190 us on the FP32 pipe.
constexpr int PP_WARPS = 4, PP_CTAS = 3, PP_DEPTH = 4;  // warps per CTA, CTAs per SM, ring steps
constexpr size_t PP_SMEM = sizeof(uint4) * 256 * PP_DEPTH * PP_WARPS;  // 64 KB: three CTAs per SM
constexpr int PP_MAX_NLAD = 3376;  // ladder basis of a channel (the amplitudes of a row in shared memory)

// sum_cd t(ij, cd) V(cd, ab) in FP64 for a row ij kept as FP64 values (infinities, NaN).
__device__ __noinline__ double pp_nonfinite(const uint4* __restrict__ vstrip, const double* __restrict__ trow, int row,
                                            int nl, int vexp) {
  double s = 0.0;
  for (int k = 0; k < nl; k++) {
    const int q = (k & 7) >> 1, half = (k >> 3) & 1;
    const dig_t w = dig_pick(vstrip[((long)(k >> 4) * 4 + (row >> 3) + 2 * half) * 32 + (row & 7) * 4 + q], k & 1);
    s += trow[((k >> 4) * 4 + q) * 8 + half * 2 + (k & 1)] * dig_to_double((long long)(w - DIG_BIAS), vexp - 1022 - 61);
  }
  return s;
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
// of the item's warps (4 per lane and warp).
template <int SLOTS, typename Out>
__device__ __forceinline__ void pp_pass(const DevState& D, const PPItem& it, const int* __restrict__ rows, int part,
                                        int wk, uint4* __restrict__ ring, DigSum* __restrict__ red) {
  constexpr int Q = 8 / SLOTS;  // rows ij of this pass, and digits per slot
  const int c = it.c, strip = it.strip, nl = it.nl, n0 = it.n0, nr = it.nr;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int steps = (nl + 15) >> 4;
  const uint4* __restrict__ vstrip = reinterpret_cast<const uint4*>(D.vdig + it.voff);
  const uint4* __restrict__ vp = vstrip + lane;
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
  if (part != 0) return;
  for (int p = 1; p < wk; p++)
#pragma unroll
    for (int e = 0; e < 4; e++) {
      sum[e].hi += red[(p * 4 + e) * 32 + lane].hi;
      sum[e].lo += red[(p * 4 + e) * 32 + lane].lo;
    }
  // accumulator columns 2t, 2t + 1: slot s counts 256^(-Q s); the slots of a row added up
  const int vexp = D.ch_vexp[c];
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
    if (col < Q && n0 + col < nr && ab < nl) {
      const int ij = rows ? rows[n0 + col] : n0 + col;
      const int te = D.texp[D.ch_hh_off[c] + ij];
      Out v;
      if (te < DIG_NONFINITE && vexp < DIG_NONFINITE) v = dig_result<Out>(x, dig_power(vexp, te));
      else
        v = Arith<Out>::from_double(
            vexp < DIG_NONFINITE
                ? pp_nonfinite(vstrip, reinterpret_cast<const double*>(tch + (long)ij * steps * 16), row, nl, vexp)
                : __longlong_as_double(0x7ff8000000000000ll));
      reinterpret_cast<Out*>(D.rpp)[D.ch_s_off[c] + (long)ij * nl + ab] = v;
    }
  }
}

// rep_only: the rows ij of the items count the list upd_row of the channel, else every hole pair.
// wk (2 or 4) divides PP_WARPS: PP_WARPS / wk items per CTA.  slots: ring steps per warp, PP_DEPTH or
// as many as a warp has.
template <typename Out>
__global__ void __launch_bounds__(PP_WARPS * 32, PP_CTAS) k_pp(DevState D, const LoopCtl* __restrict__ ctl,
                                                               const PPItem* __restrict__ items, int nitems, int rep_only,
                                                               int wk, int slots) {
  extern __shared__ __align__(16) uint4 pp_ring[];
  __shared__ DigSum red[PP_WARPS * 128];
  const int warp = threadIdx.x >> 5, part = warp % wk;
  const int item = blockIdx.x * (PP_WARPS / wk) + warp / wk;
  PPItem it;
  if (item < nitems) it = items[item];
  // the barrier of pp_pass is the block's only one: warps without work join it here
  if (item >= nitems || sys_done(D, ctl, it.sys)) {
    __syncthreads();
    return;
  }
  const int* __restrict__ rows = rep_only ? D.upd_row + D.ch_uoff[it.c] : nullptr;
  DigSum* mine = red + (warp / wk) * wk * 128;
  uint4* ring = pp_ring + warp * slots * 256;
  const int n = it.nr - it.n0;
  if (n > 4) pp_pass<1, Out>(D, it, rows, part, wk, ring, mine);
  else if (n > 2) pp_pass<2, Out>(D, it, rows, part, wk, ring, mine);
  else pp_pass<4, Out>(D, it, rows, part, wk, ring, mine);
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
// It runs alone on one SM after the last block of the update, so its time adds to every update:
// a chain of dependent round trips, not bandwidth.  Batches of at least FIN_WARP_SYSTEMS systems
// take one warp per system (no block barrier between systems); fewer take the whole block per
// system, which reads the several thousand partials of a large system with four times the loads
// in flight.  FIN_UNROLL partial pairs are requested before the first is added.  120 systems of
// 27 partials each, mixed solve of 20 updates read back whole: 21.0 -> 16.4 ms against the block
// taking the systems one after the other (two reductions and three barriers each); a single
// system of 66 states, 39 updates: 1.143 -> 1.122 ms from the earlier loads.
constexpr int FIN_WARP_SYSTEMS = 4, FIN_UNROLL = 8;

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
// control c are copies read before the sums, so that their loads overlap the partials'.
__device__ __forceinline__ void finalize_one(const FinArgs& f, SysCtl S, const LoopCtl& c, int s, double e, double r,
                                             bool& all_done, bool& bad) {
  if (!S.done) {
    S.iters += 1;
    S.e_new = e;
    S.resid = sqrt(r);
    if (S.iters < f.hist_cap) f.hist[(long)s * f.hist_cap + S.iters] = e;
    const double diff = fabs(e - S.e_old);
    S.e_old = e;
    S.grow = (diff > 2.0 * S.d_old && diff > S.tol) ? S.grow + 1 : 0;
    S.d_old = diff;
    bad = bad || !isfinite(e) || !isfinite(r) || S.grow >= PNM_DIVERGE_STEPS;
    if (diff < S.tol && c.iter + 1 >= c.min_iter) {
      S.done = 1;
      S.frozen_at = c.iter;
    }
    f.sc[s] = S;
  }
  all_done = all_done && S.done;
}

__device__ void finalize_systems(const FinArgs& f, LoopCtl* ctl) {
  __shared__ double sh32f[32];
  const LoopCtl c = *ctl;
  bool all_done = true, bad = false;  // of the systems this thread closes
  double e, r;
  if (f.nsys >= FIN_WARP_SYSTEMS) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    for (int s = warp; s < f.nsys; s += nw) {
      SysCtl S;
      if (lane == 0) S = f.sc[s];
      sum_partials(f, s, lane, 32, e, r);
      e = warp_sum(e);
      r = warp_sum(r);
      if (lane == 0) finalize_one(f, S, c, s, e, r, all_done, bad);
    }
    all_done = __syncthreads_and(all_done);
    bad = __syncthreads_or(bad);
  } else {
    for (int s = 0; s < f.nsys; s++) {
      SysCtl S;
      if (threadIdx.x == 0) S = f.sc[s];
      sum_partials(f, s, threadIdx.x, blockDim.x, e, r);
      block_sum2(e, r, sh32f);
      if (threadIdx.x == 0) finalize_one(f, S, c, s, e, r, all_done, bad);
    }
  }
  if (threadIdx.x == 0) {
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
}

// The last block of a grid to finish runs the finalize step (no waiting: the blocks count
// themselves out with an atomic after a fence, as in the CUDA threadfence reduction).
__device__ void last_block_finalize(const FinArgs& f, LoopCtl* ctl) {
  // only thread 0 wrote the block's partials: its fence orders them before the count
  __shared__ int is_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    is_last = (atomicAdd(&ctl->blocks_done, 1) == (int)gridDim.x - 1);
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  finalize_systems(f, ctl);
  if (threadIdx.x == 0) ctl->blocks_done = 0;
}

// ---------------------------------------------------------------------------- update
// One CTA per item (channel, up to UPD_ROWS hole pairs ij, 128 pp columns).  Jacobi step of
// Eq. (ccd3): the bracket collects v, the non-eps parts of the one-body terms, the pp and hh
// ladders and P(ij)P(ab) Q; then t_new = bracket / eps_ij^ab and t = alpha t_new + (1 - alpha) t_old.
// The residual of the amplitude equation is R = bracket - eps_ij^ab t.  The hh ladder is
// summed in the element arithmetic of T_: FP64, or FP32 pairs from the pair copy of the
// amplitudes (the sweeps with FP32-pair contractions); everything else is FP64.
// With FP32 pairs the pp ladder, the hh ladder and the ph term arrive as pairs (the 8-byte
// slots of rpp and xq) and their sum is formed on the FP32 pipe and converted to FP64 once; the
// denominator, residual, step (alpha / eps_ij^ab prepared per solve, aw) and energy stay FP64.
template <typename T_>
__global__ void __launch_bounds__(128) k_update(DevState D, LoopCtl* __restrict__ ctl,
                                                const int4* __restrict__ items, FinArgs fa,
                                                const T_* __restrict__ tpair, const double* __restrict__ aw) {
  constexpr bool PAIR = std::is_same<T_, f2>::value;
  using A = Arith<T_>;
  // the hh-ladder factor chi_kl^ij of the item's rows: chs[kl][g], zero for rows past ng;
  // per row: its hole pair ij and d_i + d_j of the one-body term
  __shared__ T_ chs[UPD_MAX_NHH][UPD_ROWS];
  __shared__ double row_dij[UPD_ROWS];
  __shared__ int row_ij[UPD_ROWS];
  __shared__ double sh32[32];
  if (ctl->status != 0) return;  // the loop has ended within its body (see pnm_enqueue_loop_body)
  int4 it = items[blockIdx.x];
  int c = it.x, ng = it.w;
  int npp = D.ch_npp[c], nh = D.ch_nhh[c];
  int ab = it.z + threadIdx.x;
  bool frozen = fa.sc[D.ch_sys[c]].done != 0;
  if (sys_settled(fa.sc[D.ch_sys[c]], ctl)) {
    // converged at least two steps ago: both amplitude buffers already hold its values
    if (threadIdx.x == 0) {
      D.eparts[blockIdx.x] = 0.0;
      D.rparts[blockIdx.x] = 0.0;
    }
    last_block_finalize(fa, ctl);
    return;
  }
  bool has_vpp = D.ch_vpp[c] != 0;
  double alpha = ctl->alpha;
  const double* __restrict__ t = cur_t(D, ctl);
  double* __restrict__ tn = next_t(D, ctl);
  long base = D.ch_t_off[c];
  long vho = D.ch_vhh_off[c];
  const UpdRow* __restrict__ rt = D.upd_rowinfo + (long)blockIdx.x * UPD_ROWS;
  if ((int)threadIdx.x < UPD_ROWS) {
    const UpdRow ri = rt[threadIdx.x];
    row_ij[threadIdx.x] = ri.ij;
    row_dij[threadIdx.x] = D.dchi[ri.hx] + D.dchi[ri.hy];
  }
  // chi's columns of the item's rows from the row table (one barrier covers both)
  for (int e = threadIdx.x; e < nh * UPD_ROWS; e += blockDim.x) {
    int kl = e / UPD_ROWS, g = e % UPD_ROWS;
    chs[kl][g] = g < ng ? A::from_double(D.chi_hh[vho + (long)kl * nh + rt[g].ij]) : A::zero();
  }
  __syncthreads();
  double esum = 0.0, rsum = 0.0;
  if (ab < npp) {
    // hh ladder sum_kl t_ab^kl chi_kl^ij for all rows of the item: one pass over the t column
    T_ hs[UPD_ROWS];
#pragma unroll
    for (int g = 0; g < UPD_ROWS; g++) hs[g] = A::zero();
    if (!frozen) {
      const long col = base + ab;
      const T_* __restrict__ tc;
      if constexpr (PAIR) tc = tpair;
      else tc = t;
#pragma unroll 4
      for (int kl = 0; kl < nh; kl++) {
        const T_ tk = tc[col + (long)kl * npp];
#pragma unroll
        for (int g = 0; g < UPD_ROWS; g++) A::mac(hs[g], tk, chs[kl][g]);
      }
    }
    int2 p = D.pp_pair[D.ch_pp_off[c] + ab];
    // one-body part of the bracket: (d_a + d_b - d_i - d_j) t with d_p = chi_p - eps_p
    double da = D.dchi[p.x] + D.dchi[p.y];
#pragma unroll
    for (int g = 0; g < UPD_ROWS; g++) {
      if (g >= ng) break;
      long z = base + (long)row_ij[g] * npp + ab;
      // one amplitude of each spin-flip pair is computed (the one with the smaller index) and
      // written to both; the pair counts twice in the energy and the residual norm
      const int fc = D.fmap[z];
      const long f = (long)(fc > 0 ? fc : -fc) - 1;
      if (f < z) continue;
      const double wgt = f == z ? 1.0 : 2.0;
      double tz = t[z];
      double out = tz;
      double v = D.v_pphh[z];
      if (!frozen) {
        int4 q = D.qmap[z];
        if constexpr (PAIR) {
          // pp ladder + hh ladder + P(ij)P(ab) Q in FP32 pairs, converted once
          const f2* __restrict__ rp = reinterpret_cast<const f2*>(D.rpp);
          const f2* __restrict__ xqp = reinterpret_cast<const f2*>(D.xq);
          f2 corr = hs[g];
          if (has_vpp) {
            int sg;
            const f2 rl = rp[lad_index(D, c, row_ij[g], ab, sg)];
            corr = A::add(corr, sg > 0 ? rl : A::neg(rl));
          }
          if (q.x >= 0) corr = A::add(corr, xqp[q.x]);
          if (q.y >= 0) corr = A::sub(corr, xqp[q.y]);
          if (q.z >= 0) corr = A::sub(corr, xqp[q.z]);
          if (q.w >= 0) corr = A::add(corr, xqp[q.w]);
          const double num = fma(da - row_dij[g], tz, v) + A::to_double(corr);
          const double R = fma(-D.den[z], tz, num);  // bracket - eps_ij^ab t
          rsum = fma(wgt * R, R, rsum);
          out = fma(R, aw[z], tz);                   // t + alpha R / eps_ij^ab
        } else {
          double num = v + (da - row_dij[g]) * tz;
          if (has_vpp) {
            int sg;
            double rl = D.rpp[lad_index(D, c, row_ij[g], ab, sg)];
            num += sg > 0 ? rl : -rl;
          }
          num += A::to_double(hs[g]);
          double ph = 0.0;
          if (q.x >= 0) ph += D.xq[q.x];
          if (q.y >= 0) ph -= D.xq[q.y];
          if (q.z >= 0) ph -= D.xq[q.z];
          if (q.w >= 0) ph += D.xq[q.w];
          num += ph;
          double tnew = num * D.inv_den[z];
          double R = num - D.den[z] * tz;
          rsum += wgt * (R * R);
          out = alpha * tnew + (1.0 - alpha) * tz;
        }
      }
      tn[z] = out;
      if (f != z) tn[f] = fc > 0 ? out : -out;
      esum = fma(wgt * v, out, esum);
    }
  }
  block_sum2(esum, rsum, sh32);
  if (threadIdx.x == 0) {
    D.eparts[blockIdx.x] = esum;
    D.rparts[blockIdx.x] = rsum;
  }
  last_block_finalize(fa, ctl);
}

void launch_update64(pnm_ctx* ctx, int use_cond, cudaGraphConditionalHandle h, bool pair) {
  if (pair)
    k_update<f2><<<ctx->n_grp_items, 128, 0, ctx->stream>>>(ctx->d, ctx->ctl, ctx->grp_items,
                                                            fin_args(ctx, use_cond, h, false), ctx->t_pair,
                                                            pnm_mixed_aw(ctx));
  else
    k_update<double><<<ctx->n_grp_items, 128, 0, ctx->stream>>>(ctx->d, ctx->ctl, ctx->grp_items,
                                                                fin_args(ctx, use_cond, h, false), nullptr,
                                                                nullptr);
}

// Mixed-precision update.  One CTA per item (channel, up to UPD_ROWS hole pairs ij of the rows
// the updates compute, 128 pp columns); each thread owns one column ab and the item's rows.
//   hh ladder   sum_kl t_ab^kl chi_kl^ij in FP32 for all rows of the item from one pass over
//               the FP32 t column (chi's columns of the item's rows staged in shared memory)
//   bracket     corrections in FP32: one-body (d_a + d_b - d_i - d_j) t, pp ladder (ladder
//               layout, k-split planes summed), hh ladder, and the ph term
//               Q_ij^ab - Q_ji^ab - Q_ij^ba + Q_ji^ba gathered from the cross-channel Q (qmap)
//   T scatter   the new FP32 amplitude to its four places in the ph term's T (the positions of
//               the four Q terms, qmap; formed positions only, so the same for the amplitude
//               and its spin flip), which the next ph kernel reads row by row
//   FP64        denominator eps_a + eps_b - eps_i - eps_j, residual R = v + bracket - eps_ij^ab t,
//               step t + alpha R / eps_ij^ab (alpha / eps_ij^ab prepared per solve), energy and
//               residual partial sums; v = <ab|v|ij> regenerated from the system's interaction
//               table (bit for bit the stored element, one FP64 addition) instead of streamed
// Arrays read once per update (t, alpha / eps, flip and Q maps) and the FP64 amplitudes written
// for the next update are streamed with the evict-first policy, so that the ph term's T and Q
// (50 MB each for the held-out batch, read and written at random) and the FP32 amplitudes the
// next update's contractions read stay in L2.
// The FP64 unit of a GB300 runs at about 1/64 of its FP32 rate, so the FP64 work is held to
// eight instructions per amplitude; the new amplitude goes to t (FP64) for itself and to t32 for
// itself and, sign applied, for its spin flip.  The FP64 flips are not read before the mixed
// iteration ends (the update reads t at the amplitudes it computes only); one flip copy of the
// current buffer fills them then (pnm_flip_copy_current).  Rows go in batches of UPD_BATCH with
// all loads of a batch issued before any store (rows past ng repeat the last row and are
// discarded).
__global__ void __launch_bounds__(128, UPD_MIN_BLOCKS) k_update_mix(DevState D, LoopCtl* __restrict__ ctl,
                                                    const int4* __restrict__ items, FinArgs fa,
                                                    const float* __restrict__ rpp, const float* __restrict__ xq,
                                                    const double* __restrict__ aw, float* __restrict__ xt,
                                                    const int* __restrict__ lut_off, int nplanes, long pstride) {
  __shared__ float chs[UPD_MAX_NHH * UPD_ROWS];  // chi32[kl][ij of row g] at kl * UPD_ROWS + g
  __shared__ float row_dij[UPD_ROWS];
  __shared__ double row_eij[UPD_ROWS];
  __shared__ int row_ij[UPD_ROWS];
  __shared__ char4 row_si[UPD_ROWS], row_sj[UPD_ROWS];
  __shared__ double red[2][128];
  if (ctl->status != 0) return;  // the loop has ended within its body (see pnm_enqueue_loop_body)
  int4 it = items[blockIdx.x];
  int c = it.x, ng = it.w;
  int npp = D.ch_npp[c], nh = D.ch_nhh[c];
  int ab = it.z + threadIdx.x;
  const bool col = ab < npp;
  const bool has_vpp = D.ch_vpp[c] != 0;
  // the column's pair data does not depend on the rows: loaded beside the row setup
  int2 p = make_int2(0, 0);
  int lmap = 0;
  if (col) {
    p = D.pp_pair[D.ch_pp_off[c] + ab];
    if (has_vpp) lmap = D.lad_map[D.ch_pp_off[c] + ab];
  }
  const UpdRow* __restrict__ rt = D.upd_rowinfo + (long)blockIdx.x * UPD_ROWS;
  if ((int)threadIdx.x < UPD_ROWS) {
    const UpdRow ri = rt[threadIdx.x];
    row_ij[threadIdx.x] = ri.ij;
    row_dij[threadIdx.x] = D.dchi32[ri.hx] + D.dchi32[ri.hy];
    row_eij[threadIdx.x] = ri.eij;
    row_si[threadIdx.x] = ri.si;
    row_sj[threadIdx.x] = ri.sj;
  }
  float dab = 0.0f;
  double eab = 0.0;
  char4 sa = make_char4(0, 0, 0, 0), sb = sa;
  if (col) {
    dab = D.dchi32[p.x] + D.dchi32[p.y];
    eab = D.eps[p.x] + D.eps[p.y];
    sa = D.nvec[p.x];
    sb = D.nvec[p.y];
  }
  const bool frozen = fa.sc[D.ch_sys[c]].done != 0;
  if (sys_settled(fa.sc[D.ch_sys[c]], ctl)) {
    // converged at least two steps ago: both amplitude buffers already hold its values
    if (threadIdx.x == 0) {
      D.eparts[blockIdx.x] = 0.0;
      D.rparts[blockIdx.x] = 0.0;
    }
    last_block_finalize(fa, ctl);
    return;
  }
  // chi's columns of the item's rows, their indices read from the row table (no wait for the
  // row setup above: one barrier covers both)
  if (!frozen) {
    const float* __restrict__ chi = D.chi32 + D.ch_vhh_off[c];
    for (int e = threadIdx.x; e < nh * UPD_ROWS; e += blockDim.x) {
      const int kl = e / UPD_ROWS, g = e % UPD_ROWS;
      chs[e] = g < ng ? chi[(long)kl * nh + rt[g].ij] : 0.0f;
    }
  }
  __syncthreads();
  const double* __restrict__ t = cur_t(D, ctl);
  const float* __restrict__ t32 = cur_t32(D, ctl);
  double* __restrict__ tn = next_t(D, ctl);
  float* __restrict__ t32n = next_t32(D, ctl);
  const long base = D.ch_t_off[c];
  // energy and residual sums of the amplitudes whose spin flip is another amplitude (counted
  // twice) and of those that are their own flip (counted once)
  double e2 = 0.0, e1 = 0.0, r2 = 0.0, r1 = 0.0;
  if (col) {
    float hh[UPD_ROWS];
#pragma unroll
    for (int g = 0; g < UPD_ROWS; g++) hh[g] = 0.0f;
    if (!frozen) {
      const float* __restrict__ tc = t32 + base + ab;
#pragma unroll UPD_HH_UNROLL
      for (int kl = 0; kl < nh; kl++) {
        const float tk = tc[(long)kl * npp];
        const float4 c0 = *reinterpret_cast<const float4*>(chs + kl * UPD_ROWS);
        const float4 c1 = *reinterpret_cast<const float4*>(chs + kl * UPD_ROWS + 4);
        hh[0] = fmaf(tk, c0.x, hh[0]); hh[1] = fmaf(tk, c0.y, hh[1]);
        hh[2] = fmaf(tk, c0.z, hh[2]); hh[3] = fmaf(tk, c0.w, hh[3]);
        hh[4] = fmaf(tk, c1.x, hh[4]); hh[5] = fmaf(tk, c1.y, hh[5]);
        hh[6] = fmaf(tk, c1.z, hh[6]); hh[7] = fmaf(tk, c1.w, hh[7]);
      }
    }
    const double* __restrict__ lut = D.lut + lut_off[D.ch_sys[c]];
    // the pp ladder's element in the ladder layout: s_off + ij * n_lad + |m| - 1, sign of m
    long lad0 = 0;
    int nl = 0;
    bool lneg = false;
    if (has_vpp) {
      const int m = lmap;
      lneg = m < 0;
      nl = D.ch_nlad[c];
      lad0 = D.ch_s_off[c] + ((m > 0 ? m : -m) - 1);
    }
#pragma unroll
    for (int gb = 0; gb < UPD_ROWS; gb += UPD_BATCH) {
      if (gb >= ng) break;
      long z[UPD_BATCH];
      double tz[UPD_BATCH], wz[UPD_BATCH];
      int fc[UPD_BATCH];
      float t32z[UPD_BATCH], part[UPD_BATCH], qs[UPD_BATCH];
      int4 qm[UPD_BATCH];
#pragma unroll
      for (int j = 0; j < UPD_BATCH; j++) {
        const int g = min(gb + j, ng - 1);
        z[j] = base + (long)row_ij[g] * npp + ab;
        tz[j] = __ldcs(t + z[j]);
        wz[j] = __ldcs(aw + z[j]);
        fc[j] = __ldcs(D.fmap + z[j]);
        t32z[j] = t32[z[j]];
        qm[j] = __ldcs(D.qmap + z[j]);
        float rl = 0.0f;
        if (has_vpp) {
          const long zl = lad0 + (long)row_ij[g] * nl;
          for (int pl = 0; pl < nplanes; pl++) rl += rpp[pl * pstride + zl];
          if (lneg) rl = -rl;
        }
        part[j] = rl;
      }
#pragma unroll
      for (int j = 0; j < UPD_BATCH; j++) {
        // P(ij)P(ab) Q: Q_ij^ab - Q_ji^ab - Q_ij^ba + Q_ji^ba from the cross-channel layout
        const float a0 = qm[j].x >= 0 ? xq[qm[j].x] : 0.0f, a1 = qm[j].y >= 0 ? xq[qm[j].y] : 0.0f;
        const float a2 = qm[j].z >= 0 ? xq[qm[j].z] : 0.0f, a3 = qm[j].w >= 0 ? xq[qm[j].w] : 0.0f;
        qs[j] = (a0 - a1) - (a2 - a3);
      }
#pragma unroll
      for (int j = 0; j < UPD_BATCH; j++) {
        const int g = gb + j;
        if (g >= ng) break;
        // one amplitude of each spin-flip pair is computed (the smaller index) and written to both
        const long f = (long)(fc[j] > 0 ? fc[j] : -fc[j]) - 1;
        if (f < z[j]) continue;
        const double v = v_minnesota_as(sa, sb, row_si[g], row_sj[g], lut);
        double out = tz[j], R = 0.0;
        if (!frozen) {
          const float corr = (dab - row_dij[g]) * t32z[j] + (part[j] + hh[g]) + qs[j];
          R = fma(eab - row_eij[g], tz[j], v) + (double)corr;  // bracket - eps_ij^ab t
          out = fma(R, wz[j], tz[j]);
        }
        const float o32 = (float)out;
        __stcs(tn + z[j], out);
        t32n[z[j]] = o32;
        if (f != z[j]) {
          t32n[f] = fc[j] < 0 ? -o32 : o32;
          e2 = fma(v, out, e2);
          r2 = fma(R, R, r2);
        } else {
          e1 = fma(v, out, e1);
          r1 = fma(R, R, r1);
        }
        if (!frozen) {
          // the T positions of t_ij^ab, t_ji^ab, t_ij^ba, t_ji^ba (the Q positions of the same
          // amplitude; stores only, nothing waits on them)
          if (qm[j].x >= 0) xt[qm[j].x] = o32;
          if (qm[j].y >= 0) xt[qm[j].y] = -o32;
          if (qm[j].z >= 0) xt[qm[j].z] = -o32;
          if (qm[j].w >= 0) xt[qm[j].w] = o32;
        }
      }
    }
  }
  // block sums: per thread in FP64, then 128 values per sum added by one warp
  red[0][threadIdx.x] = fma(2.0, e2, e1);
  red[1][threadIdx.x] = fma(2.0, r2, r1);
  __syncthreads();
  if (threadIdx.x < 32) {
    double es = (red[0][threadIdx.x] + red[0][threadIdx.x + 32]) + (red[0][threadIdx.x + 64] + red[0][threadIdx.x + 96]);
    double rs = (red[1][threadIdx.x] + red[1][threadIdx.x + 32]) + (red[1][threadIdx.x + 64] + red[1][threadIdx.x + 96]);
    es = warp_sum(es);
    rs = warp_sum(rs);
    if (threadIdx.x == 0) {
      D.eparts[blockIdx.x] = es;
      D.rparts[blockIdx.x] = rs;
    }
  }
  last_block_finalize(fa, ctl);
}

void launch_update_mix(pnm_ctx* ctx, const float* rpp, const float* xq, const double* aw, float* xt, int use_cond,
                       cudaGraphConditionalHandle h, int nplanes, long pstride) {
  k_update_mix<<<ctx->n_grp_items, 128, 0, ctx->stream>>>(ctx->d, ctx->ctl, ctx->grp_items,
                                                         fin_args(ctx, use_cond, h, false), rpp, xq, aw, xt,
                                                         ctx->lut_off_d, nplanes, pstride);
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

// Per row (channel, ij) of the amplitudes: 2 if the spin flip maps it onto a later row (it is
// computed by the updates), 0 onto an earlier one (written by that row's update), 1 onto
// itself (its columns are paired among themselves).
__global__ void k_row_mode(DevState D, int nrows, int* __restrict__ mode) {
  int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= nrows) return;
  int2 it = D.row_item[r];
  int npp = D.ch_npp[it.x];
  long z0 = D.ch_t_off[it.x] + (long)it.y * npp;
  int cd = D.fmap[z0];
  long f0 = (long)(cd > 0 ? cd : -cd) - 1;
  mode[r] = (f0 >= z0 && f0 < z0 + npp) ? 1 : (f0 > z0 ? 2 : 0);
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

// Initial amplitudes (MBPT2 guess or zero) into t0 with energy partials.
__global__ void __launch_bounds__(128) k_init(DevState D, int init) {
  __shared__ double sh32[32];
  int2 it = D.row_item[blockIdx.x];
  int c = it.x, ij = it.y;
  int npp = D.ch_npp[c];
  long row = D.ch_t_off[c] + (long)ij * npp;
  int2 h = D.hh_pair[D.ch_hh_off[c] + ij];
  double ei = D.eps[h.x], ej = D.eps[h.y];
  double esum = 0.0;
  for (int ab = threadIdx.x; ab < npp; ab += blockDim.x) {
    long z = row + ab;
    double v = D.v_pphh[z];
    double t;
    if (init == PNM_INIT_MBPT2) {
      int2 p = D.pp_pair[D.ch_pp_off[c] + ab];
      t = v / (ei + ej - D.eps[p.x] - D.eps[p.y]);
      D.t0[z] = t;
    } else if (init == PNM_INIT_ZERO) {
      t = 0.0;
      D.t0[z] = t;
    } else {
      t = D.t0[z];
    }
    esum += v * t;
  }
  esum = block_sum(esum, sh32);
  if (threadIdx.x == 0) {
    D.eparts[blockIdx.x] = esum;
    D.rparts[blockIdx.x] = 0.0;
  }
}

// MBPT2 with v generated on the fly: sum over restricted pairs of v^2 / eps_ij^ab.
__global__ void __launch_bounds__(128) k_mbpt2(DevState D, const int* __restrict__ row_lut_off) {
  __shared__ double sh32[32];
  int2 it = D.row_item[blockIdx.x];
  int c = it.x, ij = it.y;
  int npp = D.ch_npp[c];
  const double* lut = D.lut + row_lut_off[D.ch_sys[c]];
  int2 h = D.hh_pair[D.ch_hh_off[c] + ij];
  char4 si = D.nvec[h.x], sj = D.nvec[h.y];
  double ei = D.eps[h.x], ej = D.eps[h.y];
  double s = 0.0;
  for (int ab = threadIdx.x; ab < npp; ab += blockDim.x) {
    int2 p = D.pp_pair[D.ch_pp_off[c] + ab];
    double v = v_minnesota_as(D.nvec[p.x], D.nvec[p.y], si, sj, lut);
    s += v * v / (ei + ej - D.eps[p.x] - D.eps[p.y]);
  }
  s = block_sum(s, sh32);
  if (threadIdx.x == 0) D.eparts[blockIdx.x] = s;
}

// Sum of row partials per system (fixed order), into out[sys].
__global__ void k_reduce_rows(const double* __restrict__ parts, const int* __restrict__ row_lo,
                              const int* __restrict__ row_hi, double* __restrict__ out) {
  __shared__ double sh32[32];
  int s = blockIdx.x;
  double acc = 0.0;
  for (int r = row_lo[s] + threadIdx.x; r < row_hi[s]; r += blockDim.x) acc += parts[r];
  acc = block_sum(acc, sh32);
  if (threadIdx.x == 0) out[s] = acc;
}

// Energy of the start amplitudes: history[0] per system, reset of the loop state.
__global__ void k_start(const double* __restrict__ parts, const int* __restrict__ row_lo,
                        const int* __restrict__ row_hi, int nsys, SysCtl* __restrict__ sc,
                        LoopCtl* __restrict__ ctl, double* __restrict__ hist, int hist_cap) {
  // one warp per system in batches (as in finalize_systems), else the whole block
  __shared__ double sh32[32];
  const bool by_warp = nsys >= FIN_WARP_SYSTEMS;
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
    ctl->blocks_done = 0;
    ctl->dev_error = 0;
  }
}

// ------------------------------------------------------------------------- host side

static void* dmalloc(pnm_ctx* ctx, size_t bytes) { return pnm_ctx_alloc(ctx, bytes); }

// Static row data of the update items: row g of item i is the (min(g, ng - 1))-th row of its run.
__global__ void k_rowinfo(DevState D, const int4* __restrict__ items, UpdRow* __restrict__ out) {
  const int g = threadIdx.x;
  if (g >= UPD_ROWS) return;
  const int4 it = items[blockIdx.x];
  const int c = it.x, ij = D.upd_row[it.y + min(g, it.w - 1)];
  const int2 h = D.hh_pair[D.ch_hh_off[c] + ij];
  UpdRow r;
  r.ij = ij;
  r.hx = h.x;
  r.hy = h.y;
  r.pad = 0;
  r.si = D.nvec[h.x];
  r.sj = D.nvec[h.y];
  r.eij = D.eps[h.x] + D.eps[h.y];
  out[(long)blockIdx.x * UPD_ROWS + g] = r;
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
  std::vector<int2> abit;
  std::vector<int4> upd;
  std::vector<int> ulo(nsys), uhi(nsys);
  int max_npp = 0, max_nlad = 0;
  for (int c = 0; c < ctx->nch; c++) {
    int npp = ctx->h_npp[c];
    max_npp = std::max(max_npp, npp);
    for (int ab0 = 0; ab0 < npp; ab0 += 128) abit.push_back(make_int2(c, ab0));
    if (!ctx->h_vpp[c]) continue;
    int nl = ctx->h_nlad[c];
    max_nlad = std::max(max_nlad, nl);
  }
  // per-row items (channel, ij, first column), 128 columns each, grouped by system (the
  // learned-start kernels); update items (channel, first ij, first column, rows) with up to
  // UPD_ROWS hole pairs each, fewer when the grid would not fill the GPU
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
  std::vector<int> rmode(ctx->nrows, 2);
  if (ctx->nrows > 0) {
    int* dm = (int*)dmalloc(ctx, sizeof(int) * ctx->nrows);
    k_row_mode<<<(ctx->nrows + 255) / 256, 256, 0, s>>>(ctx->d, ctx->nrows, dm);
    CUDA_TRY(cudaMemcpyAsync(rmode.data(), dm, sizeof(int) * ctx->nrows, cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
  }
  ctx->h_row_mode = rmode;
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
  auto group_items = [&](int G, std::vector<int4>* out, std::vector<int>* glo, std::vector<int>* ghi) {
    size_t n = 0;
    for (int k = 0; k < nsys; k++) {
      if (glo) (*glo)[k] = (int)(out ? out->size() : n);
      for (int c = ctx->sys[k].ch_begin; c < ctx->sys[k].ch_end; c++) {
        int nr = uoff[c + 1] - uoff[c], np = ctx->h_npp[c];
        for (int r0 = 0; r0 < nr; r0 += G)
          for (int ab0 = 0; ab0 < np; ab0 += 128) {
            if (out) out->push_back(make_int4(c, uoff[c] + r0, ab0, std::min(G, nr - r0)));
            n++;
          }
      }
      if (ghi) (*ghi)[k] = (int)(out ? out->size() : n);
    }
    return n;
  };
  int G = UPD_ROWS;
  while (G > 1 && group_items(G, nullptr, nullptr, nullptr) < (size_t)8 * nsm) G >>= 1;
  std::vector<int4> grp;
  std::vector<int> glo(nsys), ghi(nsys);
  group_items(G, &grp, &glo, &ghi);
  // static row data of every update item, filled on the device (pairs and energies live there)
  ctx->d.upd_rowinfo = (UpdRow*)dmalloc(ctx, sizeof(UpdRow) * UPD_ROWS * std::max<size_t>(1, grp.size()));
  ctx->upd_rows = G;
  ctx->max_npp = max_npp;
  ctx->max_nlad = max_nlad;
  std::vector<int> alo(nsys), ahi(nsys);
  int max_nhh = 1;
  for (size_t k = 0; k < abit.size(); k++) max_nhh = std::max(max_nhh, ctx->h_nhh[abit[k].x]);
  for (int k = 0; k < nsys; k++) {
    alo[k] = (int)abit.size();
    ahi[k] = 0;
  }
  for (size_t k = 0; k < abit.size(); k++) {
    int sy = ctx->h_ch_sys[abit[k].x];
    alo[sy] = std::min(alo[sy], (int)k);
    ahi[sy] = std::max(ahi[sy], (int)k + 1);
  }
  for (int k = 0; k < nsys; k++)
    if (ahi[k] == 0) alo[k] = 0;
  ctx->max_nhh = max_nhh;
  if (max_nhh > UPD_MAX_NHH) throw PnmError{PNM_EINVAL, "more hole pairs in one channel than the update supports"};
  int* ad = (int*)dmalloc(ctx, sizeof(int) * 2 * nsys);
  CUDA_TRY(cudaMemcpyAsync(ad, alo.data(), sizeof(int) * nsys, cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemcpyAsync(ad + nsys, ahi.data(), sizeof(int) * nsys, cudaMemcpyHostToDevice, s));
  ctx->ab_lo_d = ad;
  ctx->ab_hi_d = ad + nsys;
  ctx->n_ab_items = (int)abit.size();
  ctx->ab_items = (int2*)dmalloc(ctx, sizeof(int2) * std::max<size_t>(1, abit.size()));
  if (!abit.empty())
    CUDA_TRY(cudaMemcpyAsync(ctx->ab_items, abit.data(), sizeof(int2) * abit.size(),
                             cudaMemcpyHostToDevice, s));
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
  ctx->n_grp_items = (int)grp.size();
  ctx->grp_items = (int4*)dmalloc(ctx, sizeof(int4) * std::max<size_t>(1, grp.size()));
  if (!grp.empty()) {
    CUDA_TRY(cudaMemcpyAsync(ctx->grp_items, grp.data(), sizeof(int4) * grp.size(),
                             cudaMemcpyHostToDevice, s));
    k_rowinfo<<<(unsigned)grp.size(), 32, 0, s>>>(ctx->d, ctx->grp_items, ctx->d.upd_rowinfo);
    CUDA_TRY(cudaGetLastError());
  }
  int* gd = (int*)dmalloc(ctx, sizeof(int) * 2 * nsys);
  CUDA_TRY(cudaMemcpyAsync(gd, glo.data(), sizeof(int) * nsys, cudaMemcpyHostToDevice, s));
  CUDA_TRY(cudaMemcpyAsync(gd + nsys, ghi.data(), sizeof(int) * nsys, cudaMemcpyHostToDevice, s));
  ctx->grp_lo_d = gd;
  ctx->grp_hi_d = gd + nsys;
  // partial sums: one per update item (at least one per row for init/MBPT2)
  size_t nparts = std::max<size_t>(upd.size(), (size_t)ctx->nrows);
  ctx->d.eparts = (double*)dmalloc(ctx, sizeof(double) * nparts);
  ctx->d.rparts = (double*)dmalloc(ctx, sizeof(double) * nparts);
  int mx = 0;
  for (int x = 0; x < ctx->nx; x++) mx = std::max(mx, std::max(ctx->h_x_nph[x], ctx->h_x_nhp[x]));
  ctx->max_x_dim = mx;
  ctx->ctl = (LoopCtl*)dmalloc(ctx, sizeof(LoopCtl));
  CUDA_TRY(cudaMemsetAsync(ctx->ctl, 0, sizeof(LoopCtl), s));
  ctx->small = (double*)dmalloc(ctx, sizeof(double) * 8);
  ctx->sysctl = (SysCtl*)dmalloc(ctx, sizeof(SysCtl) * nsys);
  CUDA_TRY(cudaMemsetAsync(ctx->sysctl, 0, sizeof(SysCtl) * nsys, s));
  ctx->d.sysctl = ctx->sysctl;
  // cross channels of the ph launch: S_z >= 0 (S_z < 0 ones are read at their flips), costliest first;
  // shared memory for the largest (NM = 1: rows/columns; NM = 2: those of the halves, twice)
  // CTA per channel in three size classes (larger than PH_SMALL_DIM: k_ph_big; larger than
  // PH_MID_DIM; the rest), warp per channel (at most PH_WARP_DIM)
  std::vector<int> xb, xm, xl, xw;
  size_t ph_staged = 0;  // three 8-byte matrices of the largest channel: the size limit of a context
  std::vector<long> xcost(ctx->nx, 0);
  for (int x = 0; x < ctx->nx; x++) {
    int c = ctx->h_x_cls[x];
    if (c < 0) continue;
    long ph = ctx->h_x_nph[x], hp = ctx->h_x_nhp[x];
    int d = (int)std::max(ph, hp);
    if (c == 0) {
      d /= 2;
      xcost[x] = ph * hp * hp / 4;
    } else {
      xcost[x] = ph * hp * hp;
    }
    if (d <= PH_WARP_DIM) {
      xw.push_back(x);
      continue;
    }
    int nm = c == 0 ? 2 : 1;
    ph_staged = std::max(ph_staged, ph_smem_bytes(d, nm, sizeof(double)));
    if (d > PH_SMALL_DIM) {
      ctx->ph_big_smem32 = std::max(ctx->ph_big_smem32, ph_smem_bytes(d, nm, sizeof(float)));
      xb.push_back(x);
    } else if (d > PH_MID_DIM) {
      ctx->ph_mid_smem32 = std::max(ctx->ph_mid_smem32, ph_smem_bytes(d, nm, sizeof(float)));
      xm.push_back(x);
    } else {
      ctx->ph_smem32 = std::max(ctx->ph_smem32, ph_smem_bytes(d, nm, sizeof(float)));
      xl.push_back(x);
    }
  }
  auto costlier = [&](int a, int b) { return xcost[a] != xcost[b] ? xcost[a] > xcost[b] : a < b; };
  std::sort(xb.begin(), xb.end(), costlier);
  std::sort(xm.begin(), xm.end(), costlier);
  std::sort(xl.begin(), xl.end(), costlier);
  std::sort(xw.begin(), xw.end(), costlier);
  ctx->n_ph_big = (int)xb.size();
  ctx->n_ph_mid = (int)xm.size();
  ctx->n_ph = (int)xl.size();
  ctx->n_ph_warp = (int)xw.size();
  // list order: big, middle, small, warp
  xl.insert(xl.end(), xw.begin(), xw.end());
  xl.insert(xl.begin(), xm.begin(), xm.end());
  xl.insert(xl.begin(), xb.begin(), xb.end());
  ctx->h_ph_list = xl;
  ctx->ph_list = (int*)dmalloc(ctx, sizeof(int) * std::max<size_t>(1, xl.size()));
  if (!xl.empty())
    CUDA_TRY(cudaMemcpyAsync(ctx->ph_list, xl.data(), sizeof(int) * xl.size(), cudaMemcpyHostToDevice, s));
  if (ph_staged > 227 * 1024 || max_nlad > PP_MAX_NLAD)
    throw PnmError{PNM_EINVAL, "channel too large for the shared-memory tiles"};
  smem_at_least(k_ph<float, PH_THREADS, PNM_PH32_TILE>, ph32_smem(ctx));
  for (int k = 0; k < 2; k++) {
    CUDA_TRY(cudaStreamCreateWithFlags(&ctx->side[k], cudaStreamNonBlocking));
    CUDA_TRY(cudaEventCreateWithFlags(&ctx->ev_join[k], cudaEventDisableTiming));
  }
  CUDA_TRY(cudaEventCreateWithFlags(&ctx->ev_fork, cudaEventDisableTiming));
  smem_at_least(k_tdig, sizeof(double) * max_nlad);
  smem_at_least(k_pp<double>, PP_SMEM);
  smem_at_least(k_pp<f2>, PP_SMEM);
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
  k_mbpt2<<<ctx->nrows, 128, 0, s>>>(ctx->d, ctx->lut_off_d);
  k_reduce_rows<<<nsys, 256, 0, s>>>(ctx->d.eparts, ctx->row_lo_d, ctx->row_hi_d,
                                     ctx->d.rparts);
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
// per row (channel, ij) the partial sums over ab of
//   (4)  t0_ab^ij sum_{c<d} <ab|v|cd> t0_cd^ij,
//   (5)  t0_ab^ij sum_{k<l} t0_ab^kl <kl|v|ij>,
//   (3)  t0_ab^ij [P(ij)P(ab) sum_kc <kb|v|cj> t0_ik^ac],
// into parts[0..3) x nrows.
__global__ void __launch_bounds__(128) k_mbpt3_rows(DevState D, double* __restrict__ parts, int nrows) {
  __shared__ double sh32[32];
  int2 it = D.row_item[blockIdx.x];
  int c = it.x, ij = it.y;
  int npp = D.ch_npp[c], nh = D.ch_nhh[c];
  long base = D.ch_t_off[c], row = base + (long)ij * npp;
  const double* __restrict__ vh = D.v_hhhh + D.ch_vhh_off[c];
  const double* __restrict__ t = D.t0;
  bool has_vpp = D.ch_vpp[c] != 0;
  double e4 = 0.0, e5 = 0.0, e3 = 0.0;
  for (int ab = threadIdx.x; ab < npp; ab += blockDim.x) {
    long z = row + ab;
    // one amplitude of each spin-flip pair, counted twice (the ladder is formed on those rows)
    const int fc = D.fmap[z];
    const long f = (long)(fc > 0 ? fc : -fc) - 1;
    if (f < z) continue;
    double tz = (f == z ? 1.0 : 2.0) * t[z];
    if (has_vpp) {
      int sg;
      double rl = D.rpp[lad_index(D, c, ij, ab, sg)];
      e4 += tz * (sg > 0 ? rl : -rl);
    }
    double hh = 0.0;
    for (int kl = 0; kl < nh; kl++) hh += t[base + (long)kl * npp + ab] * vh[(long)kl * nh + ij];
    e5 += tz * hh;
    int4 q = D.qmap[z];
    double ph = 0.0;
    if (q.x >= 0) ph += D.xq[q.x];
    if (q.y >= 0) ph -= D.xq[q.y];
    if (q.z >= 0) ph -= D.xq[q.z];
    if (q.w >= 0) ph += D.xq[q.w];
    e3 += tz * ph;
  }
  e4 = block_sum(e4, sh32);
  e5 = block_sum(e5, sh32);
  e3 = block_sum(e3, sh32);
  if (threadIdx.x == 0) {
    parts[blockIdx.x] = e4;
    parts[nrows + blockIdx.x] = e5;
    parts[2 * nrows + blockIdx.x] = e3;
  }
}

// out[3 s + {0, 1, 2}] = diagrams (4), (5), (3) of system s.  Replaces the context's
// amplitudes by the MBPT2 guess.
void pnm_mbpt3_all(pnm_ctx* ctx, double* out) {
  cudaStream_t s = ctx->stream;
  pnm_need_digits(ctx);
  int nsys = (int)ctx->sys.size();
  if (!ctx->mbpt3_buf) ctx->mbpt3_buf = (double*)dmalloc(ctx, sizeof(double) * (3 * (size_t)ctx->nrows + 3 * nsys));
  double* parts = ctx->mbpt3_buf;
  double* res = parts + 3 * (size_t)ctx->nrows;
  CUDA_TRY(cudaEventRecord(ctx->ev[0], s));
  // amplitudes of the start in t0, read by the contraction kernels (iteration parity 0, no
  // system frozen)
  CUDA_TRY(cudaMemsetAsync(&ctx->ctl->iter, 0, sizeof(int), s));
  CUDA_TRY(cudaMemsetAsync(&ctx->ctl->skip_done, 0, sizeof(int), s));
  k_init<<<ctx->nrows, 128, 0, s>>>(ctx->d, PNM_INIT_MBPT2);
  pnm_launch_pp(ctx, s, true, false);
  if (ctx->nx > 0) launch_ph64(ctx, s, s, true);  // without cross channels no Q is read
  k_mbpt3_rows<<<ctx->nrows, 128, 0, s>>>(ctx->d, parts, ctx->nrows);
  for (int k = 0; k < 3; k++)
    k_reduce_rows<<<nsys, 256, 0, s>>>(parts + (size_t)k * ctx->nrows, ctx->row_lo_d, ctx->row_hi_d,
                                       res + (size_t)k * nsys);
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
  k_mbpt2<<<ctx->nrows, 128, 0, ctx->stream>>>(d, ctx->lut_off_d);
  k_reduce_rows<<<(int)ctx->sys.size(), 256, 0, ctx->stream>>>(partials, ctx->row_lo_d,
                                                                ctx->row_hi_d, results);
}

// The body of one update, enqueued on the context stream (FP64 path).
// per_row: partials of the per-row mixed update (items upd_items), else of the grouped update.
FinArgs fin_args(pnm_ctx* ctx, int use_cond, cudaGraphConditionalHandle h, bool per_row) {
  FinArgs f;
  f.eparts = ctx->d.eparts;
  f.rparts = ctx->d.rparts;
  f.lo = per_row ? ctx->upd_lo_d : ctx->grp_lo_d;
  f.hi = per_row ? ctx->upd_hi_d : ctx->grp_hi_d;
  f.nsys = (int)ctx->sys.size();
  f.sc = ctx->sysctl;
  f.hist = ctx->hist;
  f.hist_cap = ctx->hist_cap;
  f.use_cond = use_cond;
  f.handle = h;
  return f;
}

template <typename T_>
static void lad_expand(pnm_ctx* ctx, const T_* rs, int planes, long pstride, double* host_out) {
  cudaStream_t s = ctx->stream;
  if (!ctx->expand_buf) ctx->expand_buf = (double*)dmalloc(ctx, sizeof(double) * std::max<long>(ctx->nt, 1));
  if (ctx->nrows > 0)
    k_lad_expand<T_><<<ctx->nrows, 128, 0, s>>>(ctx->d, rs, planes, pstride, ctx->expand_buf);
  CUDA_TRY(cudaGetLastError());
  CUDA_TRY(cudaMemcpyAsync(host_out, ctx->expand_buf, sizeof(double) * ctx->nt, cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));
}

void pnm_lad_expand(pnm_ctx* ctx, const float* rs, int planes, long pstride, double* host_out) {
  lad_expand(ctx, rs, planes, pstride, host_out);
}

void pnm_lad_expand(pnm_ctx* ctx, const double* rs, int planes, long pstride, double* host_out) {
  lad_expand(ctx, rs, planes, pstride, host_out);
}

void pnm_lad_expand(pnm_ctx* ctx, const f2* rs, int planes, long pstride, double* host_out) {
  lad_expand(ctx, rs, planes, pstride, host_out);
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
  k_tdig<<<nrow, TDIG_THREADS, sizeof(double) * ctx->max_nlad, s>>>(ctx->d, ctx->ctl, ctx->lad_rows);
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
  if (pair) k_pp<f2><<<nb, PP_WARPS * 32, smem, s>>>(ctx->d, ctx->ctl, items, n, rep_only ? 1 : 0, wk, slots);
  else k_pp<double><<<nb, PP_WARPS * 32, smem, s>>>(ctx->d, ctx->ctl, items, n, rep_only ? 1 : 0, wk, slots);
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
  unsigned nb = (unsigned)(ctx->nrows + ctx->n_ab_items);
  unsigned nd = (unsigned)((ctx->nsp_total * 32 + 255) / 256);
  prof_begin(ctx, mixed ? KID_TSTATS32 : KID_TSTATS);
  if (mixed) k_tstats<float><<<nb, 128, 0, s>>>(D, ctx->ctl, ctx->nrows, ctx->ab_items);
  else if (pair)
    k_tstats<double, true><<<nb, 128, 0, s>>>(D, ctx->ctl, ctx->nrows, ctx->ab_items, ctx->t_pair,
                                             ctx->vpphh_f2);
  else k_tstats<double><<<nb, 128, 0, s>>>(D, ctx->ctl, ctx->nrows, ctx->ab_items);
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
  if (terms == PNM_TERMS_FULL) pnm_enqueue_stats(ctx, false, pair);
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
static bool is_ph_kernel(const void* f) {
  return f == (const void*)k_ph<float, PH_THREADS, PNM_PH32_TILE> || f == (const void*)k_ph_dig<double> ||
         f == (const void*)k_ph_dig<f2> || f == (const void*)k_ph_tiny<double> || f == (const void*)k_ph_tiny<f2>;
}

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
    v.priority = is_ph_kernel(kp.func) ? least : greatest;
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
  k_init<<<ctx->nrows, 128, 0, s>>>(ctx->d, init);
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
  k_init<<<ctx->nrows, 128, 0, s>>>(ctx->d, init);
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
// faster for this precision mode.  The held amplitudes are saved and restored.
static std::mutex g_sched_mu;
static std::map<std::string, bool> g_sched_cache;  // (shape key, mode) -> one stream

void pnm_tune_schedule(pnm_ctx* ctx, int mode, double alpha) {
  const bool pair = ((mode >> 8) & 1) != 0;
  int m = (mode & 15) == PNM_PREC_FP64 ? (pair ? 2 : 0) : 1;
  if (ctx->sched_tuned[m]) return;
  if (m == 0) pnm_need_digits(ctx);
  const std::string key = pnm_shape_key(ctx) + (m == 1 ? "|mixed" : m == 2 ? "|pair" : "|fp64");
  {
    std::lock_guard<std::mutex> lock(g_sched_mu);
    auto f = g_sched_cache.find(key);
    if (f != g_sched_cache.end()) {
      ctx->serial_sched[m] = f->second;
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
  for (int serial = 0; serial < 2; serial++) {
    ctx->serial_sched[m] = serial != 0;
    CUDA_TRY(cudaMemcpyAsync(ctx->d.t0, save, sizeof(double) * ctx->nt, cudaMemcpyDeviceToDevice, s));
    pnm_start(ctx, PNM_INIT_KEEP, never);
    if (m == 1) pnm_mixed_pack_initial(ctx, alpha);
    pnm_enqueue_body(ctx, mode, 0, 0);
    CUDA_TRY(cudaEventRecord(e0, s));
    for (int k = 0; k < 4; k++) pnm_enqueue_body(ctx, mode, 0, 0);
    CUDA_TRY(cudaEventRecord(e1, s));
    CUDA_TRY(cudaEventSynchronize(e1));
    float ms = 0;
    CUDA_TRY(cudaEventElapsedTime(&ms, e0, e1));
    if (ms < best) {
      best = ms;
      best_serial = serial;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  ctx->serial_sched[m] = best_serial != 0;
  ctx->sched_tuned[m] = true;
  {
    std::lock_guard<std::mutex> lock(g_sched_mu);
    g_sched_cache[key] = ctx->serial_sched[m];
  }
  CUDA_TRY(cudaMemcpyAsync(ctx->d.t0, save, sizeof(double) * ctx->nt, cudaMemcpyDeviceToDevice, s));
  CUDA_TRY(cudaGetLastError());
  CUDA_TRY(cudaStreamSynchronize(s));
}
