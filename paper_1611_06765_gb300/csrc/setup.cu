// setup.cu -- GPU construction of the basis, the channel tables, the index maps and the
// antisymmetrized Minnesota blocks of a pnmcc context.
//
//   basis     Sec. "Single-particle basis for infinite matter": k = 2 pi n / L, L^3 = N/rho,
//             closed shells; state order of the shell loop in Sec. "Developing a CCD code"
//             (shell, then n_x, n_y, n_z ascending, then s = -1 before +1).
//   channels  Sec. "Developing a CCD code": direct channels T (quantum numbers added) and
//             cross channels X (subtracted).  One warp per channel key walks the rows in
//             ascending state order; in a row every partner is unique for a given key, so a
//             ballot/popc prefix gives each pair its lexicographic position with no sort.
//   blocks    Sec. "Two-body interaction" (Minnesota in momentum space) and the particle-hole
//             character blocks t_pphh, v_pphh, v_pppp, v_hhhh, v_hpph of the channel mapping.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>

#include <type_traits>

#include "dig.cuh"
#include "pnm_context.cuh"

namespace {

__device__ __forceinline__ int cube_index(int x, int y, int z, int r) {
  if (x < -r || x > r || y < -r || y > r || z < -r || z > r) return -1;
  int w = 2 * r + 1;
  return ((x + r) * w + (y + r)) * w + (z + r);
}

// Charge label of a state (the .w of its char4): the spin s = +-1 in systems of neutrons only
// (species 1); s + 4t (t = +1 neutron, -1 proton) in systems with protons (species 2: protons
// only, 3: both), so that sums and differences of two labels decode uniquely into (S_z, T_z).
// A channel key's charge slot is (S_z + 2)/2 of 3 (neutrons only) or 3 (S_z + 2)/2 +
// (T_z + 2)/2 of 9.
__device__ __forceinline__ int charge_slot(int wsum, int species) {
  if (species == 1) return (wsum + 2) >> 1;
  int tsum = wsum >= 6 ? 2 : (wsum <= -6 ? -2 : 0);
  int ssum = wsum - 4 * tsum;
  return 3 * ((ssum + 2) >> 1) + ((tsum + 2) >> 1);
}

__device__ __forceinline__ int charge_sum(int slot, int species) {
  if (species == 1) return 2 * slot - 2;
  return (2 * (slot / 3) - 2) + 4 * (2 * (slot % 3) - 2);
}

__device__ __forceinline__ int charge_slots(int species) { return species == 1 ? 3 : 9; }

// State index of (n, w) in a system, or -1.  A lattice point holds 2 states (one species) or
// 4 (s = -1 then +1; within a spin the proton before the neutron).
__device__ __forceinline__ int lookup_state(const int* __restrict__ idx3, int r, int x, int y,
                                            int z, int w, int species) {
  int c = cube_index(x, y, z, r);
  if (c < 0) return -1;
  int sp, slot;
  if (species == 1) {
    if (w != -1 && w != 1) return -1;
    return idx3[2 * c + ((w + 1) >> 1)];
  }
  int t = (w == 3 || w == 5) ? 1 : ((w == -3 || w == -5) ? -1 : 0);
  if (t == 0 || !(species & (t > 0 ? 1 : 2))) return -1;
  sp = w - 4 * t;
  slot = species == 3 ? 2 * ((sp + 1) >> 1) + ((t + 1) >> 1) : (sp + 1) >> 1;
  return idx3[(species == 3 ? 4 : 2) * c + slot];
}

__device__ __forceinline__ void decode_key(int K, int m, int M, int species, int& Px, int& Py,
                                           int& Pz, int& W) {
  int nq = charge_slots(species);
  W = charge_sum(K % nq, species);
  int rest = K / nq;
  Pz = rest % M - m;
  rest /= M;
  Py = rest % M - m;
  Px = rest / M - m;
}

__device__ __forceinline__ int encode_key(int Px, int Py, int Pz, int W, int m, int M, int species) {
  return (((Px + m) * M + (Py + m)) * M + (Pz + m)) * charge_slots(species) + charge_slot(W, species);
}

// Spin s = +-1 of a state's charge label.
__device__ __forceinline__ int spin_of(int w, int species) {
  return species == 1 ? w : w - 4 * (w > 0 ? 1 : -1);
}

// ---------------------------------------------------------------------------- basis
// What the setup kernels need of one system; an array of these covers the whole context, so that
// every kernel is launched once for all systems (a grid row, a channel, a state or a hole pair picks
// its system) instead of once per system: 120 twisted systems would otherwise be 1700 launches of a
// few microseconds of latency each.  All pointers are scratch of the setup.
struct SetupSys {
  int r, m, M, species, N, nsp, sp_off, n2max, nkeys, lut_off, lut_len, twisted;
  double L, phi[3];
  char4* shell;   // states in shell order (twisted systems: before the reorder)
  int* idx3;      // lattice point and charge slot -> state
  int* start;     // first lattice point of each shell
  int* perm;      // shell order -> state (twisted)
  int* cnt;       // pairs per key: hh, pp, ph, hp
  int* key2ch;    // direct key -> channel of the context, -1 where not held
  int* pos_hh;    // hole pair (i < j) -> its place among the context's hole pairs
  int* hbase;     // ordered hole pair -> +-(first amplitude of its row + 1), 0 where not held
  int* pos_pp;    // ordered particle pair -> +-(position in the channel + 1): a < b positive
  int *phch, *phpos, *hpch, *hppos;  // (a,i) and (k,c): cross channel (-1: none) and position
  int4* code;     // [hole][particle]: formed row (a,i) as its first element in the problem of column
                  // code 0 and the step to the other problem, formed column (k,c) as 2 * column + problem
};

// Cube points c = ((x+r)w + (y+r))w + (z+r) are in (n_x, n_y, n_z) lexicographic order, so a
// point's slot in the shell-ordered list is (points in lower shells) + (points of the same
// shell with a smaller cube index).  k_basis_count: one CTA per system counts the shells
// (shared-memory atomics) and writes the shell starts; k_basis_place: one warp per cube point counts
// the same-shell points before it, a lattice line (x, y) per lane and step (two points at most: a
// thread per point that looked at every point before it took 29 us at n2max = 36, this 5), and
// writes the states.
__global__ void k_basis_count(const SetupSys* __restrict__ SS) {
  extern __shared__ int cnt[];  // [n2max + 1]
  const SetupSys& S = SS[blockIdx.x];
  const int n2max = S.n2max, r = S.r, w = 2 * r + 1, ncube = w * w * w;
  for (int k = threadIdx.x; k <= n2max; k += blockDim.x) cnt[k] = 0;
  __syncthreads();
  for (int c = threadIdx.x; c < ncube; c += blockDim.x) {
    int x = c / (w * w) - r, y = (c / w) % w - r, z = c % w - r;
    int n2 = dot3(x, y, z);
    if (n2 <= n2max) atomicAdd(&cnt[n2], 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int k = 0; k <= n2max; k++) {
      S.start[k] = acc;
      acc += cnt[k];
    }
  }
}

// Points z2 in [-r, r] with z2^2 = rest, for rest <= r^2 + 2r.
__device__ __forceinline__ int line_points(int rest) {
  if (rest < 0) return 0;
  const int q = (int)sqrtf((float)rest);  // exact for squares of this size
  return q * q != rest ? 0 : (q == 0 ? 1 : 2);
}

__global__ void __launch_bounds__(256) k_basis_place(const SetupSys* __restrict__ SS, char4* __restrict__ nvec) {
  const SetupSys& S = SS[blockIdx.x];
  const int n2max = S.n2max, r = S.r, species = S.species, w = 2 * r + 1, ncube = w * w * w;
  const int g = species == 3 ? 4 : 2, lane = threadIdx.x & 31;
  const int c = (blockIdx.y * blockDim.x + threadIdx.x) >> 5;
  if (c >= ncube) return;  // whole warps
  const int line = c / w, x = line / w - r, y = line % w - r, z = c % w - r;
  const int n2 = dot3(x, y, z);
  int* __restrict__ idx3 = S.idx3;
  if (n2 > n2max) {
    if (lane < g) idx3[g * c + lane] = -1;
    return;
  }
  // same-shell points on the lattice lines before this one, and before z on its own line
  int rank = 0;
  for (int l = lane; l < line; l += 32) {
    const int x2 = l / w - r, y2 = l % w - r;
    rank += line_points(n2 - x2 * x2 - y2 * y2);
  }
  rank = __reduce_add_sync(0xffffffffu, rank) + (z > 0);
  if (lane != 0) return;
  const int slot = S.start[n2] + rank;
  char4* __restrict__ out = S.twisted ? S.shell : nvec + S.sp_off;
  int j = 0;
  for (int sp = -1; sp <= 1; sp += 2)
    for (int t = -1; t <= 1; t += 2) {
      if (!(species & (t > 0 ? 1 : 2))) continue;
      int lab = species == 1 ? sp : sp + 4 * t;
      out[g * slot + j] = make_char4((char)x, (char)y, (char)z, (char)lab);
      idx3[g * c + j] = g * slot + j;
      j++;
    }
}

// hlut[m] = 1/2 sum_{a=R,S} (V_a / L^3)(pi/kappa_a)^{3/2} exp(-(2 pi/L)^2 m / (4 kappa_a)),
// the half of Vt that the antisymmetrized element adds twice (exact scaling by 1/2).
// With protons the three Gaussians carry different spin-isospin weights: hlut[3m + a] =
// 1/2 (V_a / L^3)(pi/kappa_a)^{3/2} exp(-(2 pi/L)^2 m / (4 kappa_a)) for a = R, T, S.
__global__ void k_lut(const SetupSys* __restrict__ SS, pnm_minnesota P, double* __restrict__ lut) {
  const SetupSys& S = SS[blockIdx.x];
  int m = blockIdx.y * blockDim.x + threadIdx.x;
  if (m >= S.lut_len) return;
  const double L = S.L, L3 = L * L * L;
  double q2 = (2.0 * PNM_PI / L) * (2.0 * PNM_PI / L) * (double)m;
  double* __restrict__ hlut = lut + S.lut_off;
  if (S.species == 1) {
    double vt = P.VR / L3 * pow(PNM_PI / P.kR, 1.5) * exp(-q2 / (4.0 * P.kR)) +
                P.VS / L3 * pow(PNM_PI / P.kS, 1.5) * exp(-q2 / (4.0 * P.kS));
    hlut[m] = 0.5 * vt;
  } else {
    hlut[3 * m] = 0.5 * (P.VR / L3 * pow(PNM_PI / P.kR, 1.5) * exp(-q2 / (4.0 * P.kR)));
    hlut[3 * m + 1] = 0.5 * (P.VT / L3 * pow(PNM_PI / P.kT, 1.5) * exp(-q2 / (4.0 * P.kT)));
    hlut[3 * m + 2] = 0.5 * (P.VS / L3 * pow(PNM_PI / P.kS, 1.5) * exp(-q2 / (4.0 * P.kS)));
  }
}

// ------------------------------------------------------------------ twisted boundaries
// Sec. "Twist-averaged boundary conditions": k = (2 pi n + theta)/L, so the kinetic energy is
// hbar^2/2m (2 pi/L)^2 |n + phi|^2 with phi = theta/(2 pi).  The three axis terms are added
// smallest first and every step is rounded on its own (no fused multiply-add), so that states
// related by a permutation of axes with equal twist components get bit-identical values; with
// phi = 0 the result is the integer n^2.
__device__ __forceinline__ double twisted_n2(char4 sp, double px, double py, double pz) {
  double a = __dadd_rn((double)sp.x, px), b = __dadd_rn((double)sp.y, py);
  double c = __dadd_rn((double)sp.z, pz);
  a = __dmul_rn(a, a);
  b = __dmul_rn(b, b);
  c = __dmul_rn(c, c);
  double lo = fmin(a, b), hi = fmax(a, b);
  double x0 = fmin(lo, c), mid = fmax(lo, c);
  double x1 = fmin(mid, hi), x2 = fmax(mid, hi);
  return __dadd_rn(__dadd_rn(x0, x1), x2);
}
__device__ __forceinline__ double twisted_n2(char4 sp, const SetupSys& S) {
  return twisted_n2(sp, S.phi[0], S.phi[1], S.phi[2]);
}

// Stable reorder by key ("order states by energy and fill holes"): a state's new slot is the
// number of states with a smaller key, or an equal key and a smaller shell-order index.
// Keys are formed into shared memory in tiles of the block size.
constexpr int TWIST_THREADS = 256;
__global__ void __launch_bounds__(TWIST_THREADS) k_twist_rank(const SetupSys* __restrict__ SS, char4* __restrict__ nvec) {
  __shared__ double sk[TWIST_THREADS];
  const SetupSys& S = SS[blockIdx.x];
  const int nsp = S.nsp;
  if (!S.twisted || blockIdx.y * TWIST_THREADS >= nsp) return;
  const char4* __restrict__ in = S.shell;
  int p = blockIdx.y * TWIST_THREADS + threadIdx.x;
  const double kp = p < nsp ? twisted_n2(in[p], S) : 0.0;
  int rank = 0;
  for (int q0 = 0; q0 < nsp; q0 += TWIST_THREADS) {
    int q = q0 + threadIdx.x;
    sk[threadIdx.x] = q < nsp ? twisted_n2(in[q], S) : 0.0;
    __syncthreads();
    int lim = min(TWIST_THREADS, nsp - q0);
    if (p < nsp)
      for (int u = 0; u < lim; u++) {
        double kq = sk[u];
        rank += (kq < kp) || (kq == kp && q0 + u < p);
      }
    __syncthreads();
  }
  if (p < nsp) {
    nvec[S.sp_off + rank] = in[p];
    S.perm[p] = rank;
  }
}

// Cube point -> state index map follows the reorder.
__global__ void k_twist_idx3(const SetupSys* __restrict__ SS) {
  const SetupSys& S = SS[blockIdx.x];
  const int w = 2 * S.r + 1, n = (S.species == 3 ? 4 : 2) * w * w * w;
  int c = blockIdx.y * blockDim.x + threadIdx.x;
  if (S.twisted && c < n && S.idx3[c] >= 0) S.idx3[c] = S.perm[S.idx3[c]];
}

// eps_p = h0_pp + sum_i <pi|v|pi>  (holes are the first N states of the system), 32 states per CTA:
// the elements of 32 holes at a time by all threads into shared memory, then added in the order of
// the holes by one warp, a lane per state (an FP64 addition costs a warp the same with one lane or
// 32 of them at work).  Also the state of opposite spin, and per system whether its N lowest states
// leave no gap (an open shell, a degenerate Fermi level).
__global__ void __launch_bounds__(256) k_eps(const SetupSys* __restrict__ SS, const char4* __restrict__ nvec_all,
                                             const double* __restrict__ lut_all, double hbar2_2m,
                                             double* __restrict__ ekin, double* __restrict__ eps,
                                             int* __restrict__ sp_sys, int* __restrict__ sp_hole,
                                             int* __restrict__ flip, int* __restrict__ open) {
  __shared__ double v[32][33];
  const int sys = blockIdx.x, p0 = blockIdx.y * 32, lane = threadIdx.x & 31;
  const SetupSys& S = SS[sys];
  const int nsp = S.nsp, N = S.N, p = p0 + lane;
  if (p0 >= nsp) return;  // whole CTAs
  const char4* __restrict__ nvec = nvec_all + S.sp_off;
  const double* __restrict__ lut = lut_all + S.lut_off;
  const char4 sp = nvec[min(p, nsp - 1)];
  double acc = 0.0;
  for (int i0 = 0; i0 < N; i0 += 32) {
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; u++) {
      const int k = (threadIdx.x >> 5) + u * 8;
      if (i0 + k < N) {
        const char4 si = nvec[i0 + k];
        v[k][lane] = v_minnesota_as(sp, si, sp, si, lut);
      }
    }
    __syncthreads();
    if (threadIdx.x < 32) {
      const int n = min(32, N - i0);
      for (int k = 0; k < n; k++) acc += v[k][lane];
    }
  }
  if (threadIdx.x >= 32 || p >= nsp) return;
  const int o = S.sp_off + p;
  const double k0 = 2.0 * PNM_PI / S.L, ek = hbar2_2m * k0 * k0 * twisted_n2(sp, S);
  ekin[o] = ek;
  eps[o] = ek + acc;
  sp_sys[o] = sys;
  sp_hole[o] = p < N;
  flip[o] = lookup_state(S.idx3, S.r, sp.x, sp.y, sp.z, sp.w - 2 * spin_of(sp.w, S.species), S.species);
  if (p == N) open[sys] = twisted_n2(nvec[N - 1], S) < twisted_n2(sp, S) ? 0 : 1;
}

// ---------------------------------------------------------------------- channel counts
// Direct keys (total momentum and charge label sum): pairs p < q of one class, counted in hh (both
// holes, index < N) or pp (both particles).  Cross keys (n_p - n_q and the label difference): ph for
// p a particle and q a hole, hp for p a hole and q a particle (a mixed pair counts once in each, with
// opposite keys).  Sums and differences of two states' momenta lie in [-m, m] (m = 2r), and of two
// labels decode uniquely (charge_slot), so every pair has a key.
// k_count_holes: the pairs of the holes p with the later states, one CTA per hole.  k_count_pp: two
// particles per CTA (one of each end of the list, so that all CTAs have the same number of pairs);
// a channel needs hole pairs too, so only pairs of keys that have some are counted: a load per pair
// instead of an atomic (44 us for three N_max = 36 systems with atomics for all, 25 us so).
__global__ void __launch_bounds__(256) k_count_holes(const SetupSys* __restrict__ SS, const char4* __restrict__ nvec_all) {
  const SetupSys& S = SS[blockIdx.x];
  const int nsp = S.nsp, N = S.N, m = S.m, M = S.M, species = S.species, nk = S.nkeys, p = blockIdx.y;
  if (p >= N) return;
  const char4* __restrict__ nvec = nvec_all + S.sp_off;
  int* __restrict__ cnt = S.cnt;
  const char4 a = nvec[p];
  for (int q = p + 1 + threadIdx.x; q < nsp; q += blockDim.x) {
    const char4 b = nvec[q];
    if (q < N) {
      atomicAdd(cnt + encode_key(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w, m, M, species), 1);
    } else {
      atomicAdd(cnt + 2 * nk + encode_key(b.x - a.x, b.y - a.y, b.z - a.z, b.w - a.w, m, M, species), 1);
      atomicAdd(cnt + 3 * nk + encode_key(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w, m, M, species), 1);
    }
  }
}

__global__ void __launch_bounds__(256) k_count_pp(const SetupSys* __restrict__ SS, const char4* __restrict__ nvec_all) {
  const SetupSys& S = SS[blockIdx.x];
  const int np = S.nsp - S.N, m = S.m, M = S.M, species = S.species;
  const char4* __restrict__ nvec = nvec_all + S.sp_off + S.N;
  const int* __restrict__ hh = S.cnt;
  int* __restrict__ pp = S.cnt + S.nkeys;
  for (int half = 0; half < 2; half++) {
    const int p = half ? np - 1 - (int)blockIdx.y : (int)blockIdx.y;
    if (half ? p <= (int)blockIdx.y : 2 * p >= np) return;  // the middle state once
    const char4 a = nvec[p];
#pragma unroll 4
    for (int q = p + 1 + threadIdx.x; q < np; q += blockDim.x) {
      const char4 b = nvec[q];
      const int K = encode_key(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w, m, M, species);
      if (hh[K] > 0) atomicAdd(pp + K, 1);
    }
  }
}

// Channels: the keys with pairs of both classes, ascending per system.  k_keys_count: their numbers
// (direct, cross) in each of KEY_RUNS runs of a system's keys; k_keys_emit: their lists (key, sizes,
// system) over all systems in order, and the map of the direct keys.
constexpr int KEY_THREADS = 256, KEY_RUNS = 48;
__device__ __forceinline__ int key_run(int nkeys) {  // keys of a run, whole warps of them per warp
  return (nkeys + KEY_RUNS * KEY_THREADS - 1) / (KEY_RUNS * KEY_THREADS) * KEY_THREADS;
}
__global__ void __launch_bounds__(KEY_THREADS) k_keys_count(const SetupSys* __restrict__ SS, int* __restrict__ nsel) {
  __shared__ int tot[2];
  const SetupSys& S = SS[blockIdx.x];
  const int nk = S.nkeys, len = key_run(nk), k0 = blockIdx.y * len, k1 = min(nk, k0 + len);
  const int* __restrict__ cnt = S.cnt;
  if (threadIdx.x < 2) tot[threadIdx.x] = 0;
  __syncthreads();
  int d = 0, x = 0;
  for (int K = k0 + threadIdx.x; K < k1; K += KEY_THREADS) {
    d += cnt[K] > 0 && cnt[nk + K] > 0;
    x += cnt[2 * nk + K] > 0 && cnt[3 * nk + K] > 0;
  }
  d = __reduce_add_sync(0xffffffffu, d);
  x = __reduce_add_sync(0xffffffffu, x);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&tot[0], d);
    atomicAdd(&tot[1], x);
  }
  __syncthreads();
  if (threadIdx.x < 2) nsel[2 * (blockIdx.x * KEY_RUNS + blockIdx.y) + threadIdx.x] = tot[threadIdx.x];
}

__global__ void __launch_bounds__(KEY_THREADS) k_keys_emit(const SetupSys* __restrict__ SS, const int* __restrict__ nsel,
                                                           int4* __restrict__ dlist, int4* __restrict__ xlist) {
  __shared__ int before[2], run[KEY_THREADS / 32][2];
  const int sys = blockIdx.x;
  const SetupSys& S = SS[sys];
  const int nk = S.nkeys, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int* __restrict__ cnt = S.cnt;
  if (threadIdx.x < 2) before[threadIdx.x] = 0;
  __syncthreads();
  for (int k = threadIdx.x; k < 2 * (sys * KEY_RUNS + (int)blockIdx.y); k += KEY_THREADS)
    if (nsel[k]) atomicAdd(&before[k & 1], nsel[k]);
  const int len = key_run(nk), part = len / (KEY_THREADS / 32);
  const int k0 = blockIdx.y * len + w * part, k1 = min(nk, k0 + part);
  int d = 0, x = 0;
  for (int K = k0 + lane; K < k1; K += 32) {
    d += cnt[K] > 0 && cnt[nk + K] > 0;
    x += cnt[2 * nk + K] > 0 && cnt[3 * nk + K] > 0;
  }
  d = __reduce_add_sync(0xffffffffu, d);
  x = __reduce_add_sync(0xffffffffu, x);
  if (lane == 0) {
    run[w][0] = d;
    run[w][1] = x;
  }
  __syncthreads();
  int od = before[0], ox = before[1];
  for (int u = 0; u < w; u++) {
    od += run[u][0];
    ox += run[u][1];
  }
  const unsigned lt = (1u << lane) - 1u;
  for (int b = k0; b < k1; b += 32) {
    const int K = b + lane;
    int4 n = make_int4(0, 0, 0, 0);
    if (K < k1) n = make_int4(cnt[K], cnt[nk + K], cnt[2 * nk + K], cnt[3 * nk + K]);
    const bool isd = n.x > 0 && n.y > 0, isx = n.z > 0 && n.w > 0;
    const unsigned bd = __ballot_sync(0xffffffffu, isd), bx = __ballot_sync(0xffffffffu, isx);
    const int pd = od + __popc(bd & lt);
    if (K < k1) S.key2ch[K] = isd ? pd : -1;
    if (isd) dlist[pd] = make_int4(K, n.x, n.y, sys);
    if (isx) xlist[ox + __popc(bx & lt)] = make_int4(K, n.z, n.w, sys);
    od += __popc(bd);
    ox += __popc(bx);
  }
}

// ------------------------------------------------------------------------ channel fill
// Pairs (global state indices) of the channels in lexicographic order and the pair -> position tables
// used by the index maps.
// One CTA per direct channel walks the states p in order, FILL_STEPS steps of 32 per warp at a time;
// in a row every partner q > p is unique for the key, so that ballots and the warps' totals give each
// pair its place (one warp per channel and one step at a time, a chain of 58 lookups of L2 latency,
// took 37 us per N_max = 36 system; 22 us for three so).
constexpr int FILL_STEPS = 4;
__global__ void __launch_bounds__(128) k_fill_direct(const SetupSys* __restrict__ SS, const char4* __restrict__ nvec_all,
                                                     const int* __restrict__ ch_sys, const int* __restrict__ key,
                                                     const int* __restrict__ hh_off, const int* __restrict__ pp_off,
                                                     const int* __restrict__ ch_npp, const long* __restrict__ ch_t_off,
                                                     int2* __restrict__ hh_pair, int2* __restrict__ pp_pair) {
  __shared__ int tot[4][2];
  const int c = blockIdx.x, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const SetupSys& S = SS[ch_sys[c]];
  const int nsp = S.nsp, N = S.N, np = nsp - N, r = S.r, species = S.species, sp_off = S.sp_off;
  const int* __restrict__ idx3 = S.idx3;
  const char4* __restrict__ nvec = nvec_all + sp_off;
  int Px, Py, Pz, Sz;
  decode_key(key[c], S.m, S.M, species, Px, Py, Pz, Sz);
  int* __restrict__ pos_hh = S.pos_hh;
  int* __restrict__ pos_pp = S.pos_pp;
  int* __restrict__ hbase = S.hbase;
  const int npp = ch_npp[c], t1 = (int)ch_t_off[c] + 1, hh0 = hh_off[c], pp0 = pp_off[c];
  int n_hh = 0, n_pp = 0;
  const unsigned lt = (1u << lane) - 1u;
  for (int p0 = 0; p0 < nsp; p0 += 128 * FILL_STEPS) {
    const int p1 = p0 + w * 32 * FILL_STEPS + lane;
    int q[FILL_STEPS], mh = 0, mp = 0;
#pragma unroll
    for (int u = 0; u < FILL_STEPS; u++) {
      const int p = p1 + u * 32;
      q[u] = -1;
      if (p < nsp) {
        const char4 s = nvec[p];
        q[u] = lookup_state(idx3, r, Px - s.x, Py - s.y, Pz - s.z, Sz - s.w, species);
        if (q[u] <= p || (p < N) != (q[u] < N)) q[u] = -1;
      }
    }
#pragma unroll
    for (int u = 0; u < FILL_STEPS; u++) {
      const int p = p1 + u * 32;
      mh += __popc(__ballot_sync(0xffffffffu, q[u] >= 0 && p < N));
      mp += __popc(__ballot_sync(0xffffffffu, q[u] >= 0 && p >= N));
    }
    __syncthreads();
    if (lane == 0) {
      tot[w][0] = mh;
      tot[w][1] = mp;
    }
    __syncthreads();
    int at_hh = n_hh, at_pp = n_pp;
#pragma unroll
    for (int u = 0; u < 4; u++) {
      if (u < w) {
        at_hh += tot[u][0];
        at_pp += tot[u][1];
      }
      n_hh += tot[u][0];
      n_pp += tot[u][1];
    }
#pragma unroll
    for (int u = 0; u < FILL_STEPS; u++) {
      const int p = p1 + u * 32;
      const bool vh = q[u] >= 0 && p < N, vp = q[u] >= 0 && p >= N;
      const unsigned bh = __ballot_sync(0xffffffffu, vh), bp = __ballot_sync(0xffffffffu, vp);
      if (vh) {
        const int k = at_hh + __popc(bh & lt), h = t1 + k * npp;
        hh_pair[hh0 + k] = make_int2(p + sp_off, q[u] + sp_off);
        pos_hh[p * N + q[u]] = hh0 + k;
        hbase[p * N + q[u]] = h;
        hbase[q[u] * N + p] = -h;
      }
      if (vp) {
        const int pos = at_pp + __popc(bp & lt);
        pp_pair[pp0 + pos] = make_int2(p + sp_off, q[u] + sp_off);
        pos_pp[(size_t)(p - N) * np + (q[u] - N)] = pos + 1;
        pos_pp[(size_t)(q[u] - N) * np + (p - N)] = -pos - 1;
      }
      at_hh += __popc(bh);
      at_pp += __popc(bp);
    }
  }
}

// One warp per cross channel, a lane per hole: columns (k,c) in the order of the holes k; rows (a,i)
// in the order of the particles a, each row's place being the number of smaller a (compared from
// shared memory, N ints per warp; the walk over all states instead of the holes took 127 us for three
// N_max = 36 systems, 26 us so).
constexpr int CROSS_WARPS = 4;
__global__ void __launch_bounds__(CROSS_WARPS * 32) k_fill_cross(const SetupSys* __restrict__ SS,
                                                    const char4* __restrict__ nvec_all, int nx, int max_n,
                                                    const int* __restrict__ x_sys, const int* __restrict__ key,
                                                    const int* __restrict__ ph_off, const int* __restrict__ hp_off,
                                                    int2* __restrict__ ph_pair, int2* __restrict__ hp_pair) {
  extern __shared__ int partner[];
  const int x = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (x >= nx) return;  // whole warps; no block barrier
  int* mine = partner + (threadIdx.x >> 5) * max_n;
  const SetupSys& S = SS[x_sys[x]];
  const int nsp = S.nsp, N = S.N, np = nsp - N, r = S.r, species = S.species, sp_off = S.sp_off;
  const int* __restrict__ idx3 = S.idx3;
  const char4* __restrict__ nvec = nvec_all + sp_off;
  int Dx, Dy, Dz, Ds;
  decode_key(key[x], S.m, S.M, species, Dx, Dy, Dz, Ds);
  const int po = ph_off[x], ho = hp_off[x];
  int f_hp = 0;
  const unsigned lt = (1u << lane) - 1u;
  for (int h0 = 0; h0 < N; h0 += 32) {
    const int h = h0 + lane;
    int a = INT_MAX, c = -1;
    if (h < N) {
      const char4 s = nvec[h];
      const int pa = lookup_state(idx3, r, s.x + Dx, s.y + Dy, s.z + Dz, s.w + Ds, species);
      c = lookup_state(idx3, r, s.x - Dx, s.y - Dy, s.z - Dz, s.w - Ds, species);
      if (pa >= N) a = pa;
      mine[h] = a;
    }
    const bool vhp = c >= N;
    const unsigned b = __ballot_sync(0xffffffffu, vhp);
    if (vhp) {
      const int pos = f_hp + __popc(b & lt);
      const size_t e = (size_t)h * np + (c - N);
      hp_pair[ho + pos] = make_int2(h + sp_off, c + sp_off);
      S.hppos[e] = pos;
      S.hpch[e] = x;
    }
    f_hp += __popc(b);
  }
  __syncwarp();
  for (int h = lane; h < N; h += 32) {
    const int a = mine[h];
    if (a == INT_MAX) continue;
    int pos = 0;
    for (int k = 0; k < N; k++) pos += mine[k] < a;
    const size_t e = (size_t)(a - N) * N + h;
    ph_pair[po + pos] = make_int2(a + sp_off, h + sp_off);
    S.phpos[e] = pos;
    S.phch[e] = x;
  }
}

// ------------------------------------------------------------------------ spin flip
// The global spin flip F (every state to the one of opposite spin) leaves H and the
// spin-saturated reference unchanged, so the amplitudes of the solution obey
// t(F i, F j; F a, F b) = t(i, j; a, b) and every cross-channel matrix M of the ph term
// (T, W, <kb|v|cj>, Q) obeys M_F(x)[F r][F c] = M_x[r][c].  For every cross channel it records:
//   x_cls   +1 for S_z = s_a - s_i > 0 (formed in full), 0 for S_z = 0 (F maps the channel
//           onto itself; formed on its spin-up rows), -1 for S_z < 0 (not formed: the update
//           reads the flipped channel F(x) instead, see k_cross_codes);
//   x_fcol  per column (k,c) the column of (F k, F c) in F(x);
//   x_rrow / x_rcol (S_z = 0)  the rows (a,i) and columns (k,c) with spin-up a and k, in order
//           (half of each: the other half are their flips);
//   x_rinv / x_cinv  their inverses: the place of a spin-up row, and of a column v (spin-up) or
//           -v - 1 (the flip of the v-th spin-up column).
// Sets *err when the rows or columns of a channel do not map onto one channel F(x) (a
// reference that is not spin saturated).
// One warp per channel; the spin-up rows and columns are compacted in order with ballots.
__global__ void __launch_bounds__(128) k_xflip(const SetupSys* __restrict__ SS, int nx, const int* __restrict__ x_sys,
                                               const int* __restrict__ x_nph, const int* __restrict__ x_nhp,
                                               const int* __restrict__ x_ph_off, const int* __restrict__ x_hp_off,
                                               const int2* __restrict__ ph_pair, const int2* __restrict__ hp_pair,
                                               const char4* __restrict__ nvec, const int* __restrict__ flip,
                                               int* __restrict__ x_cls, int* __restrict__ x_fcol,
                                               int* __restrict__ x_rrow, int* __restrict__ x_rcol,
                                               int* __restrict__ x_rinv, int* __restrict__ x_cinv, int* __restrict__ err) {
  const int x = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (x >= nx) return;  // warp-uniform
  const SetupSys& S = SS[x_sys[x]];
  const unsigned lt = (1u << lane) - 1u;
  const int nph = x_nph[x], nhp = x_nhp[x], po = x_ph_off[x], ho = x_hp_off[x];
  const int N = S.N, np = S.nsp - N, species = S.species;
  bool bad = nph <= 0 || nhp <= 0;
  int sz = 0, mir = -1, nr = 0, nc = 0;
  if (!bad) {
    int2 p0 = ph_pair[po];
    sz = spin_of(nvec[p0.x].w, species) - spin_of(nvec[p0.y].w, species);
  }
  for (int k0 = 0; k0 < nph && !bad; k0 += 32) {
    const int k = k0 + lane;
    bool lbad = false, up = false;
    int ch = -1;
    if (k < nph) {
      int2 ai = ph_pair[po + k];
      const int fa = flip[ai.x], fi = flip[ai.y];
      if (fa < N || fi < 0 || fi >= N) {
        lbad = true;
      } else {
        ch = S.phch[(size_t)(fa - N) * N + fi];
        if (ch < 0) lbad = true;
        up = sz == 0 && spin_of(nvec[ai.x].w, species) > 0;
      }
    }
    if (mir < 0) mir = __shfl_sync(0xffffffffu, ch, 0);
    bad = __any_sync(0xffffffffu, lbad || (k < nph && ch != mir));
    unsigned bu = __ballot_sync(0xffffffffu, up);
    if (up) {
      const int v = nr + __popc(bu & lt);
      x_rrow[po + v] = k;
      x_rinv[po + k] = v;
    }
    nr += __popc(bu);
  }
  for (int k0 = 0; k0 < nhp && !bad; k0 += 32) {
    const int k = k0 + lane;
    bool lbad = false, up = false;
    if (k < nhp) {
      int2 hc = hp_pair[ho + k];
      const int fh = flip[hc.x], fp = flip[hc.y];
      if (fh < 0 || fh >= N || fp < N) {
        lbad = true;
      } else {
        x_fcol[ho + k] = S.hppos[(size_t)fh * np + (fp - N)];
        up = sz == 0 && spin_of(nvec[hc.x].w, species) > 0;
      }
    }
    bad = __any_sync(0xffffffffu, lbad);
    unsigned bu = __ballot_sync(0xffffffffu, up);
    if (up) {
      const int v = nc + __popc(bu & lt);
      x_rcol[ho + v] = k;
      x_cinv[ho + k] = v;
      x_cinv[ho + x_fcol[ho + k]] = -v - 1;
    }
    nc += __popc(bu);
  }
  if (lane != 0) return;
  if (!bad && sz == 0 && (2 * nr != nph || 2 * nc != nhp || mir != x)) bad = true;
  if (!bad && sz != 0 && mir == x) bad = true;
  x_cls[x] = sz > 0 ? 1 : (sz == 0 ? 0 : -1);
  if (bad) atomicExch(err, 1);
}

// ------------------------------------------------------------------------- index maps
// Cross-channel description of the index maps.
struct CrossTables {
  const int *x_sys, *x_nph, *x_nhp, *x_cls, *x_ph_off, *x_hp_off, *x_rrow, *x_rcol, *x_fcol, *x_rinv, *x_cinv;
  const long *x_t_off, *x_c_off;
};

// Row and column of a cross channel behind element (m, u, v) of its formed matrices: S_z > 0 rows
// and columns as they are (m = 0); S_z = 0 the u-th spin-up row, and of the v-th spin-up column
// (m = 0) or of its flip (m = 1).
struct FormedChannel {
  int nm, R, H, W;  // problems, rows, columns, row stride
  const int *rrow, *rcol, *fcol;
  __device__ FormedChannel(const CrossTables& X, int x)
      : nm(X.x_cls[x] < 0 ? 0 : (X.x_cls[x] == 0 ? 2 : 1)), R(nm == 2 ? X.x_nph[x] >> 1 : X.x_nph[x]),
        H(nm == 2 ? X.x_nhp[x] >> 1 : X.x_nhp[x]), W(formed_width(H)), rrow(X.x_rrow + X.x_ph_off[x]),
        rcol(X.x_rcol + X.x_hp_off[x]), fcol(X.x_fcol + X.x_hp_off[x]) {}
  __device__ int row(int u) const { return nm == 2 ? rrow[u] : u; }
  __device__ int col(int m, int v) const { return nm == 2 ? (m ? fcol[rcol[v]] : rcol[v]) : v; }
};

// Position of Q_x[(p,h)][(h2,p2)].  The ph kernels form Q (and read T) only in the cross channels
// with S_z >= 0 and, in those with S_z = 0, only in the rows of a spin-up particle; every other
// position is replaced by that of its spin flip Q_F(x)[(Fp,Fh)][(Fh2,Fp2)], which holds the same
// value for flip-symmetric amplitudes.  Whether the element is replaced depends on its row alone, and
// a flip changes a column of a channel with S_z = 0 into the same column of the other problem, so the
// position is the sum of a code of the row and one of the column.  One thread per (hole, particle)
// here writes both, and an amplitude's four positions are four loads (k_amplitudes) instead of the
// whole chain of tables four times (110 us per N=66, N_max=36 system).
__global__ void __launch_bounds__(128) k_cross_codes(const SetupSys* __restrict__ SS, CrossTables X,
                                                     const char4* __restrict__ nvec, const int* __restrict__ flip_all) {
  const SetupSys& S = SS[blockIdx.x];
  const int N = S.N, np = S.nsp - N, e = blockIdx.y * blockDim.x + threadIdx.x;
  if (e >= np * N) return;
  const int* __restrict__ flip = flip_all + S.sp_off;
  const int h = e / np, p = e % np + N, fh = flip[h], fp = flip[p];
  const bool mapped = fh >= 0 && fh < N && fp >= N;
  int4 code = make_int4(-1, 0, 0, 0);
  size_t u = (size_t)(p - N) * N + h;
  int g = S.phch[u];
  if (g >= 0 && mapped) {  // as a row (p, h)
    bool flipped = false;
    if (X.x_cls[g] < 0 || (X.x_cls[g] == 0 && spin_of(nvec[S.sp_off + p].w, S.species) < 0)) {
      flipped = true;
      u = (size_t)(fp - N) * N + fh;
      g = S.phch[u];
    }
    if (g >= 0) {
      const bool zero = X.x_cls[g] == 0;
      const int W = formed_width(zero ? X.x_nhp[g] >> 1 : X.x_nhp[g]);
      const int row = zero ? X.x_rinv[X.x_ph_off[g] + S.phpos[u]] : S.phpos[u];
      const int other = zero ? (X.x_nph[g] >> 1) * W : 0;  // from one problem to the other
      const int first = (int)X.x_t_off[g] + row * W;
      code.x = zero && flipped ? first + other : first;
      code.y = zero && flipped ? -other : other;
    }
  }
  u = e;
  g = S.hpch[u];
  if (g >= 0 && mapped) {  // as a column (h, p)
    if (X.x_cls[g] < 0) {
      u = (size_t)fh * np + (fp - N);
      g = S.hpch[u];
    }
    if (g >= 0) {
      const int col = S.hppos[u];
      code.z = 2 * col;
      if (X.x_cls[g] == 0) {
        const int v = X.x_cinv[X.x_hp_off[g] + col];
        code.z = v < 0 ? 2 * (-v - 1) + 1 : 2 * v;
      }
    }
  }
  S.code[e] = code;
}

__device__ __forceinline__ int q_position(int4 row, int4 col) {
  return row.x < 0 ? -1 : row.x + (col.z >> 1) + (col.z & 1) * row.y;
}

// Sign * (index + 1) of t_{h1 h2}^{p1 p2} (system-local states) in the restricted direct blocks from
// the code hb of its hole pair; 0 where it vanishes (p1 = p2 or h1 = h2) or its channel is not held.
__device__ __forceinline__ int t_code(int p1, int p2, int hb, int N, int np, const int* __restrict__ pos_pp) {
  if (p1 == p2 || hb == 0) return 0;
  const int pos = pos_pp[(size_t)(p1 - N) * np + (p2 - N)], code = abs(hb) + abs(pos) - 1;
  return (hb > 0) == (pos > 0) ? code : -code;
}

// Static data of the amplitudes of one row (channel, ij) per CTA:
//   v_pphh   <ab|v|ij>
//   den, inv_den   eps_ij^ab = e_i + e_j - e_a - e_b (HF energies) and its reciprocal
//            (these three once per pair of an amplitude and its spin flip, for both)
//   fmap     the position code of the spin-flipped amplitude (sign * (index + 1)); the flipped row is
//            one row, so only the position of its particle pair is looked up
//   qmap     the positions of Q_ij^ab, Q_ji^ab, Q_ij^ba, Q_ji^ba with Q_ij^ab = Q_x[(a,i)][(j,b)]
// and mode of the row: 2 if the spin flip maps it onto a later row (it is computed by the updates),
// 0 onto an earlier one (written by that row's update), 1 onto itself (its columns are paired among
// themselves).
// Bound by the FP64 divisions and the gathers, which overlap here; as four kernels, one after the
// other for every system, 158 us per N=66, N_max=36 system, 70 us for three systems here.
__global__ void __launch_bounds__(128) k_amplitudes(const SetupSys* __restrict__ SS, DevState D,
                                                    const int* __restrict__ flip_all, int* __restrict__ mode,
                                                    int* __restrict__ err) {
  const int2 it = D.row_item[blockIdx.x];
  const int c = it.x, ij = it.y;
  const SetupSys& S = SS[D.ch_sys[c]];
  const int N = S.N, np = S.nsp - N, sp_off = S.sp_off, npp = D.ch_npp[c];
  const int2 h = D.hh_pair[D.ch_hh_off[c] + ij];
  const int i = h.x - sp_off, j = h.y - sp_off;
  const int* __restrict__ flip = flip_all + sp_off;
  const int* __restrict__ pos_pp = S.pos_pp;
  const int4* __restrict__ code_i = S.code + (long)i * np - N;
  const int4* __restrict__ code_j = S.code + (long)j * np - N;
  const double* __restrict__ lut = D.lut + S.lut_off;
  const int2* __restrict__ pairs = D.pp_pair + D.ch_pp_off[c];
  const int fi = flip[i], fj = flip[j];
  const bool held = fi >= 0 && fi < N && fj >= 0 && fj < N;
  const int hb = held ? S.hbase[fi * N + fj] : 0;
  const char4 si = D.nvec[h.x], sj = D.nvec[h.y];
  const double eij = D.eps[h.x] + D.eps[h.y];
  const long base = D.ch_t_off[c] + (long)ij * npp;
  for (int ab = threadIdx.x; ab < npp; ab += blockDim.x) {
    const int2 pb = pairs[ab];
    const int a = pb.x - sp_off, b = pb.y - sp_off, fa = flip[a], fb = flip[b];
    const int4 ai = code_i[a], aj = code_j[a], bi = code_i[b], bj = code_j[b];
    const int code = fa >= N && fb >= N ? t_code(fa, fb, hb, N, np, pos_pp) : 0;
    const long z = base + ab, f = (long)(code > 0 ? code : -code) - 1;
    if (f >= z || f < 0) {
      const double v = v_minnesota_as(D.nvec[pb.x], D.nvec[pb.y], si, sj, lut);
      const double d = eij - D.eps[pb.x] - D.eps[pb.y], y = 1.0 / d;
      D.v_pphh[z] = v;
      D.den[z] = d;
      D.inv_den[z] = y;
      if (f > z) {
        D.v_pphh[f] = code > 0 ? v : -v;
        D.den[f] = d;
        D.inv_den[f] = y;
      }
    }
    D.qmap[base + ab] = make_int4(q_position(ai, bj), q_position(aj, bi), q_position(bi, aj), q_position(bj, ai));
    if (code == 0) atomicExch(err, 1);
    D.fmap[base + ab] = code;
    if (ab == 0) mode[blockIdx.x] = f >= base && f < base + npp ? 1 : (f > base ? 2 : 0);
  }
}

// The formed matrices of one cross channel per CTA:
//   xmap   T_x[(a,i)][(k,c)] = t_ik^ac, read from the restricted direct block with its sign: sign *
//          (t index + 1), 0 where the element vanishes (a = c or i = k) and in the padding
//   x_w    W_x[(k,c)][(e,l)] = <kl|v|ce>, stored as W_x^T, so the ph kernel stages it with coalesced loads
//   x_v1   V1_x[(k,c)][(j,b)] = <kb|v|cj>
// zero in the padding.  The states of the rows and columns are staged in shared memory.
__global__ void __launch_bounds__(128) k_cross(const SetupSys* __restrict__ SS, CrossTables X, DevState D) {
  extern __shared__ __align__(16) unsigned char xsm[];
  const int x = blockIdx.x;
  const FormedChannel f(X, x);
  if (f.nm == 0) return;
  const SetupSys& S = SS[X.x_sys[x]];
  const int N = S.N, np = S.nsp - N, po = X.x_ph_off[x], ho = X.x_hp_off[x], C = f.nm * f.H;
  const int* __restrict__ pos_pp = S.pos_pp;
  const int* __restrict__ hbase = S.hbase;
  const double* __restrict__ lut = D.lut + S.lut_off;
  int2* rs = reinterpret_cast<int2*>(xsm);  // rows (a,i), then columns (k,c): system-local states
  int2* cs = rs + f.R;
  char4* ra = reinterpret_cast<char4*>(cs + C);  // a and i of the rows, k and c of the columns
  char4 *ri = ra + f.R, *ck = ri + f.R, *cc = ck + C;
  for (int u = threadIdx.x; u < f.R; u += blockDim.x) {
    const int2 ai = D.ph_pair[po + f.row(u)];
    rs[u] = make_int2(ai.x - S.sp_off, ai.y - S.sp_off);
    ra[u] = D.nvec[ai.x];
    ri[u] = D.nvec[ai.y];
  }
  for (int v = threadIdx.x; v < C; v += blockDim.x) {
    const int2 kc = D.hp_pair[ho + f.col(v >= f.H, v >= f.H ? v - f.H : v)];
    cs[v] = make_int2(kc.x - S.sp_off, kc.y - S.sp_off);
    ck[v] = D.nvec[kc.x];
    cc[v] = D.nvec[kc.y];
  }
  __syncthreads();
  const long to = X.x_t_off[x], co = X.x_c_off[x];
  for (int e = threadIdx.x; e < f.nm * f.R * f.W; e += blockDim.x) {
    const int mu = e / f.W, v = e - mu * f.W, m = mu >= f.R, u = mu - m * f.R;
    int code = 0;
    double y = 0.0;
    if (v < f.H) {
      const int2 ai = rs[u], kc = cs[m * f.H + v];
      code = t_code(ai.x, kc.y, hbase[ai.y * N + kc.x], N, np, pos_pp);
      y = v_minnesota_as(ck[m * f.H + v], ri[u], cc[m * f.H + v], ra[u], lut);
    }
    D.xmap[to + e] = code;
    D.x_w[to + e] = y;
  }
  for (int e = threadIdx.x; e < f.nm * f.H * f.W; e += blockDim.x) {
    const int mr = e / f.W, v = e - mr * f.W, m = mr >= f.H, r = mr - m * f.H;
    double y = 0.0;
    if (v < f.H) y = v_minnesota_as(ck[r], cc[m * f.H + v], cc[r], ck[m * f.H + v], lut);
    D.x_v1[co + e] = y;
  }
}

// Pairs containing each state (for the one-body intermediates): count then fill, in the order of the
// partners d of the same class.  One CTA per state, four steps of 32 partners per warp at a time (a
// warp per state walked the partners in a chain of 58 steps: 41 us per N_max = 36 system and pass).
constexpr int OCC_THREADS = 128, OCC_STEPS = 4;
__global__ void __launch_bounds__(OCC_THREADS) k_occ(int fill, const SetupSys* __restrict__ SS, const int* __restrict__ sp_sys,
                                                     const char4* __restrict__ nvec_all, const int* __restrict__ ch_pp_off,
                                                     int* __restrict__ occ_cnt, const int* __restrict__ occ_off,
                                                     int* __restrict__ occ_idx) {
  __shared__ int tot[OCC_THREADS / 32];
  const SetupSys& S = SS[sp_sys[blockIdx.x]];
  const int N = S.N, np = S.nsp - N, p = (int)blockIdx.x - S.sp_off, w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool hole = p < N;
  const int lo = hole ? 0 : N, hi = hole ? N : S.nsp;
  const char4* __restrict__ nvec = nvec_all + S.sp_off;
  const int* __restrict__ key2ch = S.key2ch;
  const char4 sp = nvec[p];
  const unsigned lt = (1u << lane) - 1u;
  int n = 0;
  for (int d0 = lo; d0 < hi; d0 += OCC_THREADS * OCC_STEPS) {
    int ch[OCC_STEPS], d1 = d0 + w * 32 * OCC_STEPS + lane, mine = 0;
    unsigned b[OCC_STEPS];
#pragma unroll
    for (int u = 0; u < OCC_STEPS; u++) {
      const int d = d1 + u * 32;
      ch[u] = -1;
      if (d < hi && d != p) {
        const char4 sd = nvec[d];
        ch[u] = key2ch[encode_key(sp.x + sd.x, sp.y + sd.y, sp.z + sd.z, sp.w + sd.w, S.m, S.M, S.species)];
      }
    }
#pragma unroll
    for (int u = 0; u < OCC_STEPS; u++) {
      b[u] = __ballot_sync(0xffffffffu, ch[u] >= 0);
      mine += __popc(b[u]);
    }
    __syncthreads();
    if (lane == 0) tot[w] = mine;
    __syncthreads();
    int at = n;
    for (int u = 0; u < OCC_THREADS / 32; u++) {
      if (u < w) at += tot[u];
      n += tot[u];
    }
    if (!fill) continue;
    at += occ_off[blockIdx.x];
#pragma unroll
    for (int u = 0; u < OCC_STEPS; u++) {
      const int d = d1 + u * 32;
      if (ch[u] >= 0)
        occ_idx[at + __popc(b[u] & lt)] = hole ? S.pos_hh[min(p, d) * N + max(p, d)]
                                               : ch_pp_off[ch[u]] + abs(S.pos_pp[(size_t)(p - N) * np + (d - N)]) - 1;
      at += __popc(b[u]);
    }
  }
  if (!fill && threadIdx.x == 0) occ_cnt[blockIdx.x] = n;
}

// ---------------------------------------------------------------------- ladder basis
// For two neutrons <ab|v|cd> acts only on the spin singlet: with each pp pair of an S_z = 0
// channel written with its spin-up particle first (sign e = -1 when the stored order is the
// other one), the element e_x e_z <x|v|z> depends on the spatial pair of z only through the
// two Gaussians of n_u - n_u' and n_u - n_d', so it is the same for z and its partner z'
// (spatial labels of the two spins exchanged).  The pp ladder R_x = sum_z <x|v|z> t_z is then
// R_x = e_x sum_c W(c(x), c) s_c with one vector per partner couple, s_c = e_z t_z + e_z' t_z'
// and W(c, c') = e e' <rep c|v|rep c'>: a quarter of the elements and of the products.  Other
// channels (systems with protons) keep one vector per pair.
// One CTA (256 threads) per channel with a V_pppp block; dynamic shared memory holds three
// ints per pair: partner position, sign e, rank of a representative.
constexpr int LAD_THREADS = 256;
__global__ void __launch_bounds__(LAD_THREADS) k_ladder_basis(
    const SetupSys* __restrict__ SS, const int* __restrict__ chans, const int* __restrict__ ch_sys,
    const int* __restrict__ ch_pp_off, const int* __restrict__ ch_npp, const int2* __restrict__ pp_pair,
    const char4* __restrict__ nvec, int* __restrict__ lad_map, int2* __restrict__ lad_mem, int* __restrict__ ch_nlad) {
  extern __shared__ int lsm[];
  __shared__ int warp_tot[LAD_THREADS / 32];
  __shared__ int base_sh;
  int c = chans[blockIdx.x];
  int off = ch_pp_off[c], npp = ch_npp[c];
  const SetupSys& S = SS[ch_sys[c]];
  const int species = S.species, N = S.N, nsp = S.nsp, r = S.r;
  const int* __restrict__ idx3 = S.idx3;
  const int* __restrict__ pos_pp = S.pos_pp;
  if (species != 1) {  // no reduction: one vector per pair
    for (int x = threadIdx.x; x < npp; x += blockDim.x) {
      lad_map[off + x] = x + 1;
      lad_mem[off + x] = make_int2(x + 1, 0);
    }
    if (threadIdx.x == 0) ch_nlad[c] = npp;
    return;
  }
  int* part = lsm;
  int* sgn = lsm + npp;
  int* rnk = lsm + 2 * npp;
  int np = nsp - N;
  for (int x = threadIdx.x; x < npp; x += blockDim.x) {
    int2 pr = pp_pair[off + x];
    char4 sa = nvec[pr.x], sb = nvec[pr.y];
    bool a_up = sa.w > 0;
    char4 su = a_up ? sa : sb, sd = a_up ? sb : sa;
    sgn[x] = a_up ? 1 : -1;
    int u2 = lookup_state(idx3, r, sd.x, sd.y, sd.z, 1, 1);   // spin up at the down momentum
    int d2 = lookup_state(idx3, r, su.x, su.y, su.z, -1, 1);  // spin down at the up momentum
    int p1 = min(u2, d2), p2 = max(u2, d2);
    part[x] = (p1 < N) ? x : pos_pp[(size_t)(p1 - N) * np + (p2 - N)] - 1;
  }
  if (threadIdx.x == 0) base_sh = 0;
  __syncthreads();
  // rank of each representative (partner position >= own position) in pair order
  int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int x0 = 0; x0 < npp; x0 += blockDim.x) {
    int x = x0 + threadIdx.x;
    bool rep = x < npp && part[x] >= x;
    unsigned bal = __ballot_sync(0xffffffffu, rep);
    if (lane == 0) warp_tot[warp] = __popc(bal);
    __syncthreads();
    int before = base_sh;
    for (int w = 0; w < warp; w++) before += warp_tot[w];
    if (rep) rnk[x] = before + __popc(bal & ((1u << lane) - 1u));
    __syncthreads();
    if (threadIdx.x == 0) {
      int tot = 0;
      for (int w = 0; w < LAD_THREADS / 32; w++) tot += warp_tot[w];
      base_sh += tot;
    }
    __syncthreads();
  }
  for (int x = threadIdx.x; x < npp; x += blockDim.x) {
    int px = part[x];
    int rk = px >= x ? rnk[x] : rnk[px];
    lad_map[off + x] = (rk + 1) * sgn[x];
    if (px >= x) lad_mem[off + rk] = make_int2((x + 1) * sgn[x], px != x ? (px + 1) * sgn[px] : 0);
  }
  if (threadIdx.x == 0) ch_nlad[c] = base_sh;
}

// W(c, c') = e e' <rep c|v|rep c'> for the 16 rows of one strip of a channel per CTA, as digit
// words (dig.cuh) in the order the ladder kernel's tensor-core fragments read them: per 16-column
// step four groups (row half + 2 column half) of 32 lanes with two neighbouring columns each
// (interleaved), zero past the matrix.  The channel's representative pair states, their signs and the
// interaction table (as integers) are staged in shared memory; no FP64 arithmetic.
// The BF16 tiles of the mixed ladder (k_pack_v) come from the same integers.
constexpr int VLAD_ROWS = 16;
__global__ void __launch_bounds__(256) k_v_dig(const int4* __restrict__ items, const int* __restrict__ ch_pp_off,
                                               const int* __restrict__ ch_nlad, const long* __restrict__ ch_vd_off,
                                               const int2* __restrict__ lad_mem, const int2* __restrict__ pp_pair,
                                               const char4* __restrict__ nvec, const double* __restrict__ lut,
                                               int* __restrict__ ch_vexp, unsigned* __restrict__ vtop, double* __restrict__ v64_all,
                                               const int* __restrict__ ch_sys, const int* __restrict__ sys_steep,
                                               dig_t* __restrict__ vdig) {
  extern __shared__ __align__(16) unsigned char vsm[];
  __shared__ int sh_max;
  __shared__ unsigned sh_top;
  long long* xlut = reinterpret_cast<long long*>(vsm);
  const int4 it = items[blockIdx.x];  // channel, first row, interaction table and its size (< 0: with protons)
  const int c = it.x, r0 = it.y, lut_elems = abs(it.w);
  double* __restrict__ v64 = v64_all && sys_steep[ch_sys[c]] ? v64_all : nullptr;
  int nl = ch_nlad[c], off = ch_pp_off[c];
  char4* sa = reinterpret_cast<char4*>(xlut + lut_elems);
  char4* sb = sa + nl;
  int* sg = reinterpret_cast<int*>(sb + nl);
  const int e = stage_fixed_lut(lut + it.z, lut_elems, it.w < 0, xlut, &sh_max);
  for (int q = threadIdx.x; q < nl; q += blockDim.x) {
    int m = lad_mem[off + q].x;
    int pos = (m > 0 ? m : -m) - 1;
    int2 pr = pp_pair[off + pos];
    sa[q] = nvec[pr.x];
    sb[q] = nvec[pr.y];
    sg[q] = m > 0 ? 1 : -1;
  }
  if (threadIdx.x == 0) {
    ch_vexp[c] = e;
    sh_top = 0;
  }
  __syncthreads();
  const int steps = (nl + 15) >> 4;
  uint4* out = reinterpret_cast<uint4*>(vdig + ch_vd_off[c]) + (long)(r0 >> 4) * steps * 128;
  unsigned top = 0;
  for (int f = threadIdx.x; f < steps * 128; f += blockDim.x) {
    const int lane = f & 31, g = (f >> 5) & 3, ks = f >> 7;
    const int row = r0 + (lane >> 2) + (g & 1) * 8, col = ks * 16 + (lane & 3) * 2 + (g >> 1) * 8;
    dig_t w[2];
#pragma unroll
    for (int k = 0; k < 2; k++) {
      const int q = col + k;
      long long v = 0;
      if (row < nl && q < nl) {
        v = v_minnesota_fixed(sa[q], sb[q], sa[row], sb[row], xlut);
        v = sg[row] * sg[q] > 0 ? v : -v;
        if (v64) {
          const double y = v_minnesota_as(sa[q], sb[q], sa[row], sb[row], lut + it.z);
          v64[ch_vd_off[c] + (long)row * steps * 16 + q] = sg[row] * sg[q] > 0 ? y : -y;
        }
      }
      top = max(top, dig_top(v));
      w[k] = dig_word(v);
    }
    out[f] = dig_interleave(w[0], w[1]);
  }
  top = __reduce_max_sync(0xffffffffu, top);
  if ((threadIdx.x & 31) == 0) atomicMax(&sh_top, top);
  __syncthreads();
  if (threadIdx.x == 0) vtop[ch_vd_off[c] / 256 + (r0 >> 4) * steps] = sh_top;
}

__global__ void k_v_hhhh(const SetupSys* __restrict__ SS, const int* __restrict__ ch_sys,
                         const int* __restrict__ ch_hh_off, const int* __restrict__ ch_nhh,
                         const long* __restrict__ ch_vhh_off, const int2* __restrict__ hh_pair,
                         const char4* __restrict__ nvec, const double* __restrict__ lut_all,
                         double* __restrict__ v_hhhh) {
  const int c = blockIdx.x, nh = ch_nhh[c];
  const double* __restrict__ lut = lut_all + SS[ch_sys[c]].lut_off;
  for (int e = threadIdx.x; e < nh * nh; e += blockDim.x) {
    int kl = e / nh, ij = e % nh;
    int2 a = hh_pair[ch_hh_off[c] + kl], b = hh_pair[ch_hh_off[c] + ij];
    v_hhhh[ch_vhh_off[c] + e] = v_minnesota_as(nvec[a.x], nvec[a.y], nvec[b.x], nvec[b.y], lut);
  }
}

template <typename T>
T* dalloc(size_t n, std::vector<void*>& owned, cudaStream_t s) {
  void* p = pnm_pool_alloc(s, std::max<size_t>(n, 1) * sizeof(T));
  owned.push_back(p);
  return (T*)p;
}

template <typename T>
void h2d(T* d, const std::vector<T>& h, cudaStream_t s) {
  if (!h.empty()) CUDA_TRY(cudaMemcpyAsync(d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice, s));
}

template <typename T>
std::vector<T> d2h(const T* d, size_t n, cudaStream_t s) {
  std::vector<T> h(n);
  if (n) {
    CUDA_TRY(cudaMemcpyAsync(h.data(), d, n * sizeof(T), cudaMemcpyDeviceToHost, s));
    CUDA_TRY(cudaStreamSynchronize(s));
  }
  return h;
}

int isqrt_floor(int x) {
  int r = (int)std::floor(std::sqrt((double)x));
  while (r * r > x) r--;
  while ((r + 1) * (r + 1) <= x) r++;
  return r;
}

}  // namespace

// Device memory that lives only during setup; its release is ordered on the context's stream.
struct SetupScratch {
  cudaStream_t stream;
  std::vector<void*> owned;
  explicit SetupScratch(cudaStream_t s) : stream(s) {}
  SetupScratch(const SetupScratch&) = delete;
  ~SetupScratch() {
    for (void* p : owned) pnm_pool_free(stream, p);
  }
  template <typename T>
  T* get(size_t n) {
    return dalloc<T>(n, owned, stream);
  }
};

// Arrays of one allocation: pointers to set once its address is known.
struct ScratchLayout {
  std::vector<std::pair<void*, size_t>> at;
  size_t bytes = 0;
  template <typename T>
  void add(T*& p, size_t n) {
    at.push_back({&p, bytes});
    bytes += (n * sizeof(T) + 15) / 16 * 16;
  }
  void place(char* base) {
    for (auto& a : at) {
      char* p = base + a.second;
      std::memcpy(a.first, &p, sizeof(p));
    }
  }
};

// Host arrays that go to the device in one copy.
struct Upload {
  ScratchLayout lay;
  std::vector<char> buf;
  template <typename T>
  void add(T*& p, const std::vector<T>& h) {
    lay.add(p, h.size());
    const size_t o = lay.at.back().second;
    buf.resize(std::max<size_t>(lay.bytes, 1));
    if (!h.empty()) std::memcpy(buf.data() + o, h.data(), h.size() * sizeof(T));
  }
  void send(char* d, cudaStream_t s) {
    h2d(d, buf, s);
    lay.place(d);
  }
};

// The digit words of the ladder-basis V_pppp (the FP64 and FP32-pair pp ladder): built once, on
// first use.
void pnm_need_vdig(pnm_ctx* ctx) {
  if (ctx->d.vdig) return;
  cudaStream_t s = ctx->stream;
  DevState& D = ctx->d;
  pnm_need_pp_lists(ctx);
  D.tdig = ctx_alloc<dig_t>(ctx, ctx->ntdig);
  D.texp = ctx_alloc<int>(ctx, ctx->n_hh_pairs);
  D.ttop = ctx_alloc<unsigned>(ctx, ctx->n_hh_pairs);
  D.vtop = ctx_alloc<unsigned>(ctx, ctx->nvdig / 256);
  if (std::find(ctx->h_steep.begin(), ctx->h_steep.end(), 1) != ctx->h_steep.end()) {  // before any capture
    D.sys_steep = ctx_alloc<int>(ctx, ctx->h_steep.size());
    h2d(D.sys_steep, ctx->h_steep, s);
    D.v64 = ctx_alloc<double>(ctx, ctx->nvdig);
    ctx->s64 = ctx_alloc<double>(ctx, std::max<long>(ctx->ns, 1));
  }
  D.vdig = ctx_alloc<dig_t>(ctx, std::max<long>(ctx->nvdig, 1));
  smem_at_least(k_v_dig, ctx->vl_smem);
  if (ctx->n_vl_items > 0)
    k_v_dig<<<ctx->n_vl_items, 256, ctx->vl_smem, s>>>(ctx->vl_items, D.ch_pp_off, D.ch_nlad, D.ch_vd_off, D.lad_mem,
                                                       D.pp_pair, D.nvec, D.lut, D.ch_vexp, D.vtop, D.v64, D.ch_sys, D.sys_steep, D.vdig);
  CUDA_TRY(cudaGetLastError());
}

void pnm_build(pnm_ctx* ctx, int nsys, const int* Ns, const int* Zs, const double* rhos,
               const int* n2maxs, const double* thetas, const pnm_minnesota& P) {
  cudaStream_t s = ctx->stream;
  DevState& D = ctx->d;
  std::vector<SysInfo>& sys = ctx->sys;
  sys.resize(nsys);
  SetupScratch scr(s);
  ctx->hbar2_2m = P.hbar2_2m;

  // ---- sizes per system
  int nsp_total = 0, lut_total = 0;
  for (int k = 0; k < nsys; k++) {
    SysInfo& S = sys[k];
    int Nn = Ns[k], Z = Zs ? Zs[k] : 0;
    if (Nn < 0 || Z < 0 || (Nn > 0 && Z > 0 && Nn != Z))
      throw PnmError{PNM_EINVAL, "system " + std::to_string(k) +
                                     ": neutrons only, protons only, or equal numbers of both"};
    S.N = Nn + Z;
    S.Z = Z;
    S.species = (Nn > 0 ? 1 : 0) | (Z > 0 ? 2 : 0);
    S.rho = rhos[k];
    S.n2max = n2maxs[k];
    if (S.N <= 0 || !(S.rho > 0.0) || S.n2max < 0 || S.n2max > 400)
      throw PnmError{PNM_EINVAL, "invalid N, rho or n2max"};
    S.r = isqrt_floor(S.n2max);
    S.m = 2 * S.r;
    S.M = 2 * S.m + 1;
    S.nkeys = S.M * S.M * S.M * (S.species == 1 ? 3 : 9);
    S.L = std::cbrt((double)S.N / S.rho);
    for (int a = 0; a < 3; a++) {
      double th = thetas ? thetas[3 * k + a] : 0.0;
      if (!std::isfinite(th)) throw PnmError{PNM_EINVAL, "twist angle is not finite"};
      S.phi[a] = th / (2.0 * PNM_PI);
    }
    // lattice points with n^2 <= n2max, counted line by line
    int points = 0;
    for (int x = -S.r; x <= S.r; x++)
      for (int y = -S.r; y <= S.r; y++)
        if (x * x + y * y <= S.n2max) points += 2 * isqrt_floor(S.n2max - x * x - y * y) + 1;
    S.nsp = (S.species == 3 ? 4 : 2) * points;
    if (S.N >= S.nsp) throw PnmError{PNM_EINVAL, "no particle states: n2max too small for N"};
    S.sp_off = nsp_total;
    nsp_total += S.nsp;
    // exp(-q^2 / 4 kappa) of the widest Gaussian at q = (2 pi / L) 2 sqrt(n2max)
    const double q1 = 2.0 * PNM_PI / S.L;
    double kappa = std::max(P.VR != 0.0 ? P.kR : 0.0, P.VS != 0.0 ? P.kS : 0.0);
    if (S.species != 1 && P.VT != 0.0) kappa = std::max(kappa, P.kT);
    const double octaves = kappa > 0.0 ? q1 * q1 * S.n2max / kappa / std::log(2.0) : 0.0;
    ctx->fall = std::max(ctx->fall, octaves);
    ctx->h_steep.push_back(octaves > (S.species == 1 ? PP_STEEP : PP_STEEP_PROTONS));
    S.lut_off = lut_total;
    S.lut_len = 4 * S.n2max + 1;
    lut_total += S.lut_len * (S.species == 1 ? 1 : 3);  // interleaved R, T, S halves with protons
  }
  ctx->nsp_total = nsp_total;

  // ---- scratch tables of every system in one allocation: first those that start as zero, then those
  // that start as -1, then the rest
  std::vector<SetupSys> hs(nsys);
  int max_n = 0, max_ncube = 0, max_nsp = 0, max_lut = 0, max_n2 = 0, max_g = 2;
  long max_np_n = 0;
  bool any_twist = false;
  size_t zero_end = 0, ones_end = 0;
  {
    ScratchLayout lay;
    for (int pass = 0; pass < 3; pass++) {
      for (int k = 0; k < nsys; k++) {
        const SysInfo& S = sys[k];
        SetupSys& H = hs[k];
        const size_t np = S.nsp - S.N, w = 2 * S.r + 1, ncube = w * w * w, g = S.species == 3 ? 4 : 2;
        if (pass == 0) {
          H.r = S.r; H.m = S.m; H.M = S.M; H.species = S.species; H.N = S.N; H.nsp = S.nsp;
          H.sp_off = S.sp_off; H.n2max = S.n2max; H.nkeys = S.nkeys; H.lut_off = S.lut_off; H.lut_len = S.lut_len;
          H.L = S.L;
          H.twisted = 0;
          for (int a = 0; a < 3; a++) {
            H.phi[a] = S.phi[a];
            if (S.phi[a] != 0.0) H.twisted = 1;
          }
          any_twist = any_twist || H.twisted;
          max_ncube = std::max(max_ncube, (int)ncube);
          max_g = std::max(max_g, (int)g);
          max_n = std::max(max_n, S.N);
          max_nsp = std::max(max_nsp, S.nsp);
          max_lut = std::max(max_lut, S.lut_len);
          max_n2 = std::max(max_n2, S.n2max);
          max_np_n = std::max(max_np_n, (long)(np * S.N));
          lay.add(H.cnt, 4 * (size_t)S.nkeys);
          lay.add(H.hbase, (size_t)S.N * S.N);
        } else if (pass == 1) {
          lay.add(H.phch, np * S.N);
          lay.add(H.hpch, np * S.N);
        } else {
          lay.add(H.shell, H.twisted ? (size_t)S.nsp : 0);
          lay.add(H.perm, H.twisted ? (size_t)S.nsp : 0);
          lay.add(H.idx3, g * ncube);
          lay.add(H.start, (size_t)S.n2max + 1);
          lay.add(H.key2ch, (size_t)S.nkeys);
          lay.add(H.pos_hh, (size_t)S.N * S.N);
          lay.add(H.pos_pp, np * np);
          lay.add(H.phpos, np * S.N);
          lay.add(H.hppos, np * S.N);
          lay.add(H.code, np * S.N);
        }
      }
      if (pass == 0) zero_end = lay.bytes;
      if (pass == 1) ones_end = lay.bytes;
    }
    char* base = scr.get<char>(lay.bytes);
    lay.place(base);
    CUDA_TRY(cudaMemsetAsync(base, 0, zero_end, s));
    if (ones_end > zero_end) CUDA_TRY(cudaMemsetAsync(base + zero_end, 0xff, ones_end - zero_end, s));
  }
  SetupSys* SS = scr.get<SetupSys>(nsys);
  h2d(SS, hs, s);

  // ---- basis, interaction tables, HF energies, pair counts, channels (every system in one launch)
  D.nvec = dalloc<char4>(nsp_total, ctx->owned, s);
  D.eps = dalloc<double>(nsp_total, ctx->owned, s);
  D.ekin = dalloc<double>(nsp_total, ctx->owned, s);
  D.sp_sys = dalloc<int>(nsp_total, ctx->owned, s);
  D.sp_hole = dalloc<int>(nsp_total, ctx->owned, s);
  D.lut = dalloc<double>(lut_total, ctx->owned, s);
  D.dchi = dalloc<double>(nsp_total, ctx->owned, s);
  long nkeys_total = 0;
  for (const SysInfo& S : sys) nkeys_total += S.nkeys;
  int* flip = scr.get<int>(nsp_total);
  // whether a system is open; then per system and run of its keys the channels of both kinds
  const size_t n_found = (1 + 2 * KEY_RUNS) * (size_t)nsys;
  int* found = scr.get<int>(n_found);
  int4* dlist = scr.get<int4>(nkeys_total);
  int4* xlist = scr.get<int4>(nkeys_total);
  const unsigned ny = (unsigned)nsys;
  auto blocks = [](long n, int per) { return (unsigned)((n + per - 1) / per); };
  k_basis_count<<<ny, 512, (max_n2 + 1) * sizeof(int), s>>>(SS);
  k_basis_place<<<dim3(ny, blocks(max_ncube, 8)), 256, 0, s>>>(SS, D.nvec);
  if (any_twist) {
    k_twist_rank<<<dim3(ny, blocks(max_nsp, TWIST_THREADS)), TWIST_THREADS, 0, s>>>(SS, D.nvec);
    k_twist_idx3<<<dim3(ny, blocks((long)max_g * max_ncube, 256)), 256, 0, s>>>(SS);
  }
  k_lut<<<dim3(ny, blocks(max_lut, 128)), 128, 0, s>>>(SS, P, D.lut);
  k_eps<<<dim3(ny, blocks(max_nsp, 32)), 256, 0, s>>>(SS, D.nvec, D.lut, P.hbar2_2m, D.ekin, D.eps, D.sp_sys, D.sp_hole,
                                                     flip, found);
  k_count_holes<<<dim3(ny, max_n), 256, 0, s>>>(SS, D.nvec);
  k_count_pp<<<dim3(ny, blocks(max_nsp, 2)), 256, 0, s>>>(SS, D.nvec);
  k_keys_count<<<dim3(ny, KEY_RUNS), KEY_THREADS, 0, s>>>(SS, found + nsys);
  k_keys_emit<<<dim3(ny, KEY_RUNS), KEY_THREADS, 0, s>>>(SS, found + nsys, dlist, xlist);
  CUDA_TRY(cudaGetLastError());
  const std::vector<int> hfound = d2h(found, n_found, s);
  std::vector<int> nch_sys(nsys, 0), nx_sys(nsys, 0);
  long n_direct = 0, n_cross = 0;
  for (int k = 0; k < nsys; k++) {
    if (hfound[k] && !hs[k].twisted)
      throw PnmError{PNM_EINVAL, "N = " + std::to_string(sys[k].N) + " does not close a shell"};
    if (hfound[k])
      throw PnmError{PNM_EINVAL, "system " + std::to_string(k) + ": N = " + std::to_string(sys[k].N) +
                                     " leaves no gap at this twist (degenerate Fermi level)"};
    for (int u = 0; u < KEY_RUNS; u++) {
      nch_sys[k] += hfound[nsys + 2 * (k * KEY_RUNS + u)];
      nx_sys[k] += hfound[nsys + 2 * (k * KEY_RUNS + u) + 1];
    }
    n_direct += nch_sys[k];
    n_cross += nx_sys[k];
  }
  std::vector<int4> hd(n_direct), hx(n_cross);
  if (n_direct) CUDA_TRY(cudaMemcpyAsync(hd.data(), dlist, sizeof(int4) * n_direct, cudaMemcpyDeviceToHost, s));
  if (n_cross) CUDA_TRY(cudaMemcpyAsync(hx.data(), xlist, sizeof(int4) * n_cross, cudaMemcpyDeviceToHost, s));
  CUDA_TRY(cudaStreamSynchronize(s));

  // ---- channel metadata and offsets (host prefix sums over channels)
  const int C = (int)n_direct, NX = (int)n_cross;
  std::vector<int> h_ch_sys(C), h_key(C), h_nhh(C), h_npp(C), h_hh_off(C), h_pp_off(C), h_vpp(C);
  std::vector<long> h_t_off(C), h_vhh_off(C);
  std::vector<int2> h_rows;
  std::vector<int> h_lad_chans;  // channels with a V_pppp block
  std::vector<int> h_x_sys(NX), h_x_key(NX), h_x_nph(NX), h_x_nhp(NX), h_x_ph_off(NX), h_x_hp_off(NX), h_x_cls(NX);
  std::vector<long> h_x_t_off(NX), h_x_c_off(NX);
  long t_acc = 0, vhh_acc = 0, xt_acc = 0, xc_acc = 0, xt_full = 0;
  int hh_acc = 0, pp_acc = 0, ph_acc = 0, hp_acc = 0, max_npp = 0, max_cross = 0;
  for (int k = 0, g = 0, x = 0; k < nsys; k++) {
    SysInfo& S = sys[k];
    S.ch_begin = g;
    S.t_begin = t_acc;
    S.row_begin = (int)h_rows.size();
    for (int e = g + nch_sys[k]; g < e; g++) {
      const int K = hd[g].x, nhh = hd[g].y, npp = hd[g].z;
      h_ch_sys[g] = k;
      h_key[g] = K;
      h_nhh[g] = nhh;
      h_npp[g] = npp;
      h_hh_off[g] = hh_acc;
      h_pp_off[g] = pp_acc;
      h_t_off[g] = t_acc;
      h_vhh_off[g] = vhh_acc;
      // <ab|v|cd> vanishes for identical-nucleon pairs of equal spin (|S_z| = |T_z| = 2); in
      // neutron-only systems that leaves S_z = 0
      int slot = S.species == 1 ? K % 3 : K % 9;
      bool has_vpp = S.species == 1 ? slot == 1 : !(slot / 3 != 1 && slot % 3 != 1);
      h_vpp[g] = has_vpp ? 1 : 0;
      if (has_vpp) {
        h_lad_chans.push_back(g);
        max_npp = std::max(max_npp, npp);
      }
      for (int ij = 0; ij < nhh; ij++) h_rows.push_back(make_int2(g, ij));
      hh_acc += nhh;
      pp_acc += npp;
      t_acc += (long)nhh * npp;
      vhh_acc += (long)nhh * nhh;
    }
    S.ch_end = g;
    S.t_end = t_acc;
    S.row_end = (int)h_rows.size();
    S.x_begin = x;
    for (int e = x + nx_sys[k]; x < e; x++) {
      const int K = hx[x].x, nph = hx[x].y, nhp = hx[x].z;
      h_x_sys[x] = k;
      h_x_key[x] = K;
      h_x_nph[x] = nph;
      h_x_nhp[x] = nhp;
      h_x_ph_off[x] = ph_acc;
      h_x_hp_off[x] = hp_acc;
      h_x_t_off[x] = xt_acc;
      h_x_c_off[x] = xc_acc;
      // the formed matrices of the ph term: S_z > 0 whole, S_z = 0 the spin-up rows (the spin of a
      // key's charge slot is that of its first index)
      const int cls = (S.species == 1 ? K % 3 : (K % 9) / 3) - 1;
      h_x_cls[x] = cls;
      ph_acc += nph;
      hp_acc += nhp;
      xt_full += (long)nph * nhp;
      if (cls >= 0) {
        const int nm = cls == 0 ? 2 : 1, R = nph / nm, H = nhp / nm;
        xt_acc += (long)nm * R * formed_width(H);
        xc_acc += (long)nm * H * formed_width(H);
        max_cross = std::max(max_cross, nph + nhp);
      }
    }
    S.x_end = x;
  }
  if (!fits_maps(t_acc, xt_full, xt_acc, xc_acc))
    throw PnmError{PNM_EINVAL, "problem too large for 32-bit element maps"};
  const int nrows = (int)h_rows.size();
  ctx->nch = C;
  ctx->nx = NX;
  ctx->nt = t_acc;
  ctx->nvhh = vhh_acc;
  ctx->nxt = xt_acc;
  ctx->nxc = xc_acc;
  ctx->nrows = nrows;
  ctx->n_hh_pairs = hh_acc;
  ctx->n_pp_pairs = pp_acc;

  int *x_nph, *x_nhp, *x_ph_off, *x_hp_off, *x_sys, *x_key, *lad_chans;
  long *x_t_off, *x_c_off;
  {
    Upload up;
    up.add(D.ch_sys, h_ch_sys);
    up.add(D.ch_key, h_key);
    up.add(D.ch_nhh, h_nhh);
    up.add(D.ch_npp, h_npp);
    up.add(D.ch_hh_off, h_hh_off);
    up.add(D.ch_pp_off, h_pp_off);
    up.add(D.ch_vpp, h_vpp);
    up.add(D.ch_t_off, h_t_off);
    up.add(D.ch_vhh_off, h_vhh_off);
    up.add(D.row_item, h_rows);
    up.send(dalloc<char>(up.buf.size(), ctx->owned, s), s);
    Upload xu;  // only the setup reads these
    xu.add(x_sys, h_x_sys);
    xu.add(x_key, h_x_key);
    xu.add(x_nph, h_x_nph);
    xu.add(x_nhp, h_x_nhp);
    xu.add(x_ph_off, h_x_ph_off);
    xu.add(x_hp_off, h_x_hp_off);
    xu.add(x_t_off, h_x_t_off);
    xu.add(x_c_off, h_x_c_off);
    xu.add(lad_chans, h_lad_chans);
    xu.send(scr.get<char>(xu.buf.size()), s);
  }

  D.hh_pair = dalloc<int2>(hh_acc, ctx->owned, s);
  D.pp_pair = dalloc<int2>(pp_acc, ctx->owned, s);
  D.ph_pair = dalloc<int2>(ph_acc, ctx->owned, s);
  D.hp_pair = dalloc<int2>(hp_acc, ctx->owned, s);
  D.fmap = dalloc<int>(t_acc, ctx->owned, s);
  D.xmap = dalloc<int>(xt_acc, ctx->owned, s);
  D.qmap = dalloc<int4>(t_acc, ctx->owned, s);
  D.v_pphh = dalloc<double>(t_acc, ctx->owned, s);
  D.den = dalloc<double>(t_acc, ctx->owned, s);
  D.inv_den = dalloc<double>(t_acc, ctx->owned, s);
  D.lad_map = dalloc<int>(pp_acc, ctx->owned, s);
  D.lad_mem = dalloc<int2>(pp_acc, ctx->owned, s);
  D.v_hhhh = dalloc<double>(vhh_acc, ctx->owned, s);
  D.x_v1 = dalloc<double>(xc_acc, ctx->owned, s);
  D.x_w = dalloc<double>(xt_acc, ctx->owned, s);
  D.t0 = dalloc<double>(t_acc, ctx->owned, s);
  CUDA_TRY(cudaMemsetAsync(D.t0, 0, sizeof(double) * std::max<long>(t_acc, 1), s));  // held amplitudes of a new context
  D.t1 = dalloc<double>(t_acc, ctx->owned, s);
  D.chi_hh = dalloc<double>(vhh_acc, ctx->owned, s);
  D.sab = dalloc<double>(pp_acc, ctx->owned, s);
  D.sij = dalloc<double>(hh_acc, ctx->owned, s);
  D.xq = dalloc<double>(xt_acc, ctx->owned, s);
  D.ch_vexp = dalloc<int>(C, ctx->owned, s);
  D.ch_nlad = dalloc<int>(C, ctx->owned, s);

  // ---- pair lists, maps, V blocks.  Flip tables and the results the host reads (pairs per state,
  // ladder sizes, row modes, whether the flip tables close) in one block that starts as zero: valid
  // indices also where a channel that does not map onto one leaves gaps.
  const size_t n_flip = 2 * ((size_t)ph_acc + hp_acc) + hp_acc + NX, n_read = (size_t)nsp_total + C + nrows + 1;
  int* block = scr.get<int>(n_flip + n_read);
  CUDA_TRY(cudaMemsetAsync(block, 0, sizeof(int) * (n_flip + n_read), s));
  int *x_rrow = block, *x_rinv = x_rrow + ph_acc, *x_rcol = x_rinv + ph_acc, *x_cinv = x_rcol + hp_acc;
  int *x_fcol = x_cinv + hp_acc, *x_cls = x_fcol + hp_acc;
  int *read = block + n_flip, *occ_cnt = read, *nlad = occ_cnt + nsp_total, *mode = nlad + C, *flip_err = mode + nrows;
  const CrossTables X{x_sys, x_nph, x_nhp, x_cls, x_ph_off, x_hp_off, x_rrow, x_rcol, x_fcol, x_rinv, x_cinv, x_t_off, x_c_off};
  const size_t fsm = CROSS_WARPS * sizeof(int) * (size_t)max_n;
  const size_t csm = 2 * sizeof(int2) * (size_t)max_cross, lsm = 3 * sizeof(int) * (size_t)max_npp;
  if (csm > 200 * 1024) throw PnmError{PNM_EINVAL, "channel too large for the shared-memory tiles"};
  if (lsm > 200 * 1024) throw PnmError{PNM_EINVAL, "channel too large for the ladder basis"};
  smem_at_least(k_fill_cross, fsm);
  smem_at_least(k_cross, csm);
  smem_at_least(k_ladder_basis, lsm);
  if (C > 0)
    k_fill_direct<<<C, 128, 0, s>>>(SS, D.nvec, D.ch_sys, D.ch_key, D.ch_hh_off, D.ch_pp_off, D.ch_npp,
                                               D.ch_t_off, D.hh_pair, D.pp_pair);
  if (NX > 0) {
    k_fill_cross<<<blocks(NX, CROSS_WARPS), CROSS_WARPS * 32, fsm, s>>>(SS, D.nvec, NX, max_n, x_sys, x_key, x_ph_off, x_hp_off, D.ph_pair, D.hp_pair);
    k_xflip<<<blocks(NX, 4), 128, 0, s>>>(SS, NX, x_sys, x_nph, x_nhp, x_ph_off, x_hp_off, D.ph_pair, D.hp_pair, D.nvec,
                                          flip, x_cls, x_fcol, x_rrow, x_rcol, x_rinv, x_cinv, flip_err);
    k_cross<<<NX, 128, csm, s>>>(SS, X, D);
  }
  k_cross_codes<<<dim3(ny, blocks(max_np_n, 128)), 128, 0, s>>>(SS, X, D.nvec, flip);
  if (nrows > 0) k_amplitudes<<<nrows, 128, 0, s>>>(SS, D, flip, mode, flip_err);
  if (C > 0)
    k_v_hhhh<<<C, 128, 0, s>>>(SS, D.ch_sys, D.ch_hh_off, D.ch_nhh, D.ch_vhh_off, D.hh_pair, D.nvec, D.lut, D.v_hhhh);
  k_occ<<<nsp_total, OCC_THREADS, 0, s>>>(0, SS, D.sp_sys, D.nvec, D.ch_pp_off, occ_cnt, nullptr, nullptr);
  // ladder basis of the pp ladder (pairs and the partner tables are ready)
  if (!h_lad_chans.empty())
    k_ladder_basis<<<(unsigned)h_lad_chans.size(), LAD_THREADS, lsm, s>>>(SS, lad_chans, D.ch_sys, D.ch_pp_off, D.ch_npp,
                                                                        D.pp_pair, D.nvec, D.lad_map, D.lad_mem, nlad);
  CUDA_TRY(cudaGetLastError());
  if (C > 0) CUDA_TRY(cudaMemcpyAsync(D.ch_nlad, nlad, sizeof(int) * C, cudaMemcpyDeviceToDevice, s));
  const std::vector<int> hr = d2h(read, n_read, s);
  if (hr[n_read - 1]) throw PnmError{PNM_EINVAL, "spin-flip tables not closed (reference not spin saturated)"};
  std::vector<int> h_occ_off(nsp_total + 1, 0);
  for (int p = 0; p < nsp_total; p++) h_occ_off[p + 1] = h_occ_off[p] + hr[p];
  std::vector<int> h_nlad(hr.begin() + nsp_total, hr.begin() + nsp_total + C);
  ctx->h_row_mode.assign(hr.begin() + nsp_total + C, hr.begin() + nsp_total + C + nrows);
  std::vector<long> h_s_off(C, 0), h_vd_off(C, -1), h_td_off(C, 0);
  long s_acc = 0, vd_acc = 0, td_acc = 0;
  int max_nlad = 0;
  std::vector<int4> vl_items;  // work list of the ladder V
  for (int c = 0; c < C; c++) {
    h_s_off[c] = s_acc;
    if (!h_vpp[c]) continue;
    h_vd_off[c] = vd_acc;
    h_td_off[c] = td_acc;
    const long wide = (h_nlad[c] + 15) / 16 * 16;  // rows and columns padded to the tiles of the products
    s_acc += (long)h_nhh[c] * h_nlad[c];
    vd_acc += wide * wide;
    td_acc += 2 * h_nhh[c] * wide;  // FP16 digits: 16 bytes per element
    max_nlad = std::max(max_nlad, h_nlad[c]);
    const SysInfo& S = sys[h_ch_sys[c]];
    const int table = S.species == 1 ? S.lut_len : -3 * S.lut_len;
    for (int r0 = 0; r0 < h_nlad[c]; r0 += VLAD_ROWS) vl_items.push_back(make_int4(c, r0, S.lut_off, table));
  }
  ctx->ns = s_acc;
  ctx->nvdig = vd_acc;
  {
    Upload up;
    up.add(D.occ_off, h_occ_off);
    up.add(D.ch_s_off, h_s_off);
    up.add(D.ch_vd_off, h_vd_off);
    up.add(D.ch_td_off, h_td_off);
    up.add(ctx->vl_items, vl_items);
    up.send(dalloc<char>(up.buf.size(), ctx->owned, s), s);
  }
  D.occ_idx = dalloc<int>(h_occ_off[nsp_total], ctx->owned, s);
  k_occ<<<nsp_total, OCC_THREADS, 0, s>>>(1, SS, D.sp_sys, D.nvec, D.ch_pp_off, nullptr, D.occ_off, D.occ_idx);
  D.vdig = nullptr;  // the ladder V is built on first use
  D.v64 = nullptr;
  D.sys_steep = nullptr;
  D.rpp = dalloc<double>(s_acc, ctx->owned, s);
  ctx->ntdig = td_acc;
  ctx->n_vl_items = (int)vl_items.size();
  if (!vl_items.empty()) {
    int most = 0;
    for (const SysInfo& S : sys) most = std::max(most, S.lut_len * (S.species == 1 ? 1 : 3));
    size_t smem = sizeof(double) * most + (2 * sizeof(char4) + sizeof(int)) * (size_t)max_nlad;
    if (smem > 200 * 1024) throw PnmError{PNM_EINVAL, "channel too large for the staged ladder V"};
    ctx->vl_smem = smem;
  }
  ctx->h_ch_sys = std::move(h_ch_sys);
  ctx->h_key = std::move(h_key);
  ctx->h_nhh = std::move(h_nhh);
  ctx->h_npp = std::move(h_npp);
  ctx->h_hh_off = std::move(h_hh_off);
  ctx->h_pp_off = std::move(h_pp_off);
  ctx->h_vpp = std::move(h_vpp);
  ctx->h_t_off = std::move(h_t_off);
  ctx->h_vhh_off = std::move(h_vhh_off);
  ctx->h_rows = std::move(h_rows);
  ctx->h_x_sys = std::move(h_x_sys);
  ctx->h_x_nph = std::move(h_x_nph);
  ctx->h_x_nhp = std::move(h_x_nhp);
  ctx->h_x_t_off = std::move(h_x_t_off);
  ctx->h_x_c_off = std::move(h_x_c_off);
  ctx->h_x_cls = std::move(h_x_cls);
  ctx->h_x_ph_off = std::move(h_x_ph_off);
  ctx->h_x_hp_off = std::move(h_x_hp_off);
  ctx->h_nlad = std::move(h_nlad);
  ctx->h_s_off = std::move(h_s_off);
  ctx->h_vd_off = std::move(h_vd_off);
  CUDA_TRY(cudaGetLastError());
}
