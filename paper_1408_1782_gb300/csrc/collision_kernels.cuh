// Fast Fourier spectral collision operator C[W] = C_c[W] + C_d[W] of
// Lu & Mendl, Sec. 3.2, for 2x2 Hermitian Wigner matrices in Pauli form.
//
// Fine ("doubly padded") grid: n = 2N points per dimension, v' = -L + (L/N) i',
// fine frequencies sigma in [-N, N-1] (standard wrap).  A field on Xi is
// zero-padded to the fine grid; products of at most three Xi-limited fields
// are then free of aliasing on Xi (Sec. 1 and Sec. 3.2, "double zero padding").
// Real fields travel two at a time as the real and imaginary parts of one
// complex field; every kernel multiplier (phi, psi, psi', K) is real and has
// definite parity, so the pairing is exact.
//
// Terms (w = Pauli components, eta = diag(1,-1,-1,-1)):
//   C_c  = -2 (D x w).sigma,  D(v) = int int P(1/(u.u')) (2w0(v+u)-1) w_vec(v+u+u')   (I1, eq. CcPauliCarleman)
//   C_d  = 2 pi K2 (1 - W) - 2 pi K3.sigma + pi {W, K4.sigma}                         (I2, I3, I4, eq. CdPauli)
//   K2   = sum_a eta_a int int delta(u.u') w_a(v+u) w_a(v+u')
//   K3_b = sum_a eta_a int int delta(u.u') w_a(v+u) w_a(v+u') (eta w)_b(v+u+u')
//   K4_b = int int delta(u.u') (2 w0(v+u) - 1) (eta w)_b(v+u+u')
// with G_J (eq. approxG), H_J (eq. approxH-J) and the Hu-Ying form H_JM
// (eq. approxH-JM) for K3.  Algebraic regroupings relative to the printed
// algorithm (exact up to rounding):
//   * I1: K_j'(sigma) = sum_j omega_G[j][j'] phi_j(sigma) is tabulated, so the
//     J^2 outer convolutions become J (the j-sum is linear and acts after the
//     first convolution);
//   * psi'_j = psi_{j + J/2} (theta_j^perp = theta_{j+J/2} up to sign, psi even),
//     so the I2 and I4 inverse transforms are shared;
//   * I3: the weight (pi/J) w_m is split as sqrt((pi/J) w_m) into both shifted
//     factors; each accumulated K3 term carries it exactly once.
//
// Precision: every kernel is a template on the real type T of its transforms,
// products and per-unit accumulations (double: the plain FP64 form; float: the
// FP32-split form).  The state W comes in and C[W] goes out in FP64.  The per-unit
// K3 partial sums are reduced to FP64 sums in both forms (the FP32 values no less
// accurately than by FP64 additions, float_sum.cuh); they are rounded to T once, the
// real-space ones with the rest of C on the grid, the Fourier-space ones with the
// spectrum of C that they are added to.
#pragma once

#include <cmath>
#include <cstdio>
#include <type_traits>

#include "fft.cuh"
#include "float_sum.cuh"
#include "internal.h"
#include "tmem.cuh"

namespace qbe {

namespace {

constexpr double kPi = 3.14159265358979323846;

// Fine frequency index k (0..n-1) lies in Xi without its -N/2 line.
template <int n>
__device__ __forceinline__ bool in_xi(int k) {
  constexpr int N = n / 2;
  return (k < N / 2) || (k > n - N / 2);
}

// Fourier-space partials are kept only on the frequencies the final projection keeps (in_xi in both
// coordinates, n/2 - 1 per coordinate): xi_slot is the compact index, ascending in the permuted
// position, or -1.  Position B k1 + t holds a frequency of Xi where xi_t<B>(t); its -N/2 line sits at
// k1 = 0, t = 3 B / 4.
template <int n>
__host__ __device__ constexpr int xi_kept() {
  return n / 2 - 1;
}
template <int n>
__host__ __device__ constexpr int xi_slot(int pos) {
  constexpr int B = Split<n>::B;
  const int k1 = pos / B, t = pos % B;
  if (!xi_t<B>(t) || pos == 3 * B / 4) return -1;
  return k1 * (B / 2) + (t < B / 4 ? t : t - B / 2) - (pos > 3 * B / 4 ? 1 : 0);
}
template <int n>
__device__ __forceinline__ void build_xi_slots(int* slot) {
  for (int pos = threadIdx.x; pos < n; pos += blockDim.x) slot[pos] = xi_slot<n>(pos);
  __syncthreads();
}
template <int n>
__device__ __forceinline__ void build_xi_slots(int* slot, int* kept_pos) {
  for (int pos = threadIdx.x; pos < n; pos += blockDim.x) {
    const int k = xi_slot<n>(pos);
    slot[pos] = k;
    if (k >= 0) kept_pos[k] = pos;
  }
  __syncthreads();
}

template <class C2>
__device__ __forceinline__ void zero_fields(C2* p, int count) {
  for (int i = threadIdx.x; i < count; i += blockDim.x) p[i] = mk2((typename RealOf<C2>::type)0, (typename RealOf<C2>::type)0);
  __syncthreads();
}

template <class C2>
__device__ __forceinline__ void zero_fields_team(C2* p, int count) {
  for (int i = element_first(); i < count; i += element_stride()) p[i] = mk2((typename RealOf<C2>::type)0, (typename RealOf<C2>::type)0);
  team_sync();
}

template <class T>
__device__ __forceinline__ typename Vec2Of<T>::type zero2() {
  return mk2((T)0, (T)0);
}

// Job of a global I3 unit: the last job whose first unit is <= gunit (uniform across the block).
template <class T>
__device__ __forceinline__ int i3_job_of(const I3Jobs<T>& jobs, int gunit) {
  int k = 0;
  while (k + 1 < jobs.njobs && gunit >= jobs.job[k + 1].unit_begin) ++k;
  return k;
}

// Node group at item `it` of a chunk that ends at it1 (items as in i3_chunk_begin): node m, with its
// partner M-1-m where `pair` is set, and the pairs q in [q0, q1) of the first index of U_ab (w_0 + i w_1,
// w_2 + i w_3) that the chunk covers; `next` is the item after it.
struct I3Group {
  int m, q0, q1, next;
  bool pair;
};
__device__ __forceinline__ I3Group i3_group_at(int it, int it1, int M) {
  I3Group g;
  g.m = it >> 1;
  g.pair = !((M & 1) && it == M - 1);
  if (!g.pair) {
    g.q0 = 0;
    g.q1 = 2;
    g.next = it + 1;
  } else {
    g.q0 = it & 1;
    g.q1 = (g.q0 == 0 && it + 1 < it1) ? 2 : g.q0 + 1;
    g.next = it + g.q1 - g.q0;
  }
  return g;
}

// --------------------------------------------------------------------------
// Prep: Xi coefficients of the four Pauli components (paired) and the
// fine-grid interpolants.  One team per cell and coefficient pair.  (Outside Xi the
// coefficients are zero and not stored: no kernel reads there.)
//   what[c][0] = w0^ + i w1^, [1] = w2^ + i w3^, [2] = w1^ + i w2^, [3] = w3^
//   wfine[c][0] = w0 + i w1, [1] = w2 + i w3  on the fine grid;
//   wplane (may be null): the same four components as planes [c][4][n*n] in thread_order.
// The coarse DFT is the fine forward FFT of the zero-interleaved samples
// (its spectrum repeats with period N), scaled by 1/N^2 and cut to Xi.
// --------------------------------------------------------------------------
template <int n, class T, int CB>
__global__ void __launch_bounds__(kThreads, (cell_min_blocks<n, T, CB>()))
    k_prep(const double* __restrict__ w, typename Vec2Of<T>::type* what, typename Vec2Of<T>::type* wfine, T* wplane,
           typename Vec2Of<T>::type* ws, const typename Vec2Of<T>::type* __restrict__ gtw) {
  using C2 = typename Vec2Of<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* tw = reinterpret_cast<C2*>(smem_raw);
  C2* sm = tw + n;
  load_twiddles<n>(tw, gtw);
  constexpr int N = n / 2, P = n * n;
  const int cq = cluster_index(), c = cq >> 2, q = cq & 3;   // one team per cell and coefficient pair
  const double* wc = w + (size_t)c * 4 * N * N;
  C2* G = ws + (size_t)cq * P;
  const T invN2 = (T)(1.0 / ((double)N * N));
  constexpr int B = Split<n>::B;
  C2* out = what + ((size_t)c * 4 + q) * P;
  const int a = (q == 0) ? 0 : (q == 1) ? 2 : (q == 2) ? 1 : 3;
  const int b = (q == 0) ? 1 : (q == 1) ? 3 : (q == 2) ? 2 : -1;
  even_row_pass<n, -1, CB>(
      sm, tw,
      [&](int ix, int iy) {
        if (iy & 1) return zero2<T>();
        const int i = ix >> 1, j = iy >> 1;
        return mk2((T)wc[(a * N + i) * N + j], b >= 0 ? (T)wc[(b * N + i) * N + j] : (T)0);
      },
      [&](int ix, int iy, C2 v) {
        if (xi_t<B>(iy % B)) G[ix * n + iy] = v;
      });
  auto load = [&](int ix, int iy) { return (ix & 1) ? zero2<T>() : ldc<n, CB>(&G[ix * n + iy]); };
  auto coef = [&](int ix, int iy, C2 v) {
    const bool keep = xi_slot<n>(ix) >= 0 && xi_slot<n>(iy) >= 0;
    const C2 z = keep ? cscale(v, invN2) : zero2<T>();
    out[ix * n + iy] = z;
    return z;
  };
  if (q >= 2) {
    xi_col_filter<n, true, false, CB>(sm, tw, load, coef, [](int, int, C2) {});
    return;
  }
  xi_col_filter<n, true, true, CB>(sm, tw, load, coef, [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
  C2* fine = wfine + ((size_t)c * 2 + q) * P;
  row_pass<n, 1, false, 0, CB, true>(
      sm, tw, [&](int ix, int iy) { return xi_t<B>(iy % B) ? ldc<n, CB>(&G[ix * n + iy]) : zero2<T>(); }, NoMid(),
      [&](int ix, int iy, C2 v) {
        fine[ix * n + iy] = v;
        if (wplane) {
          T* pl = wplane + ((size_t)c * 4 + 2 * q) * P + thread_order<n>(ix, iy);
          pl[0] = v.x;
          pl[P] = v.y;
        }
      });
}

// --------------------------------------------------------------------------
// The per-cell terms before I3, one team per (cell c, angle chunk ch, pair p) and kind:
//   I1 (conservative part): D^_b(sigma) = sum_j' K_j'(sigma) FFT[(2w0-1) IFFT(phi'_j' w_b^)], pairs
//     (w1 + i w2) and (w3); angles j' in [J ch / nch, J (ch + 1) / nch); D partial [c][ch][p]
//   I2 and I4, over angle pairs (j, j + J/2), j in chunk ch of J/2, F_{a,j} = IFFT(psi_j w_a^) (real),
//     pairs (0,1), (2,3):
//     K2  += 2 (pi/J) sum_a eta_a F_{a,j} F_{a,j+J/2}                                 partial [c][ch][p]
//     K4^ += (pi/J) [psi_j FFT((2w0-1) F_{.,j+J/2}) + psi_{j+J/2} FFT((2w0-1) F_{.,j})] / n^2
// Teams [0, 2 nch ncells) take I1, the next as many I2/I4 (both kinds in one launch: with few cells
// neither fills the GPU); `first` is the team of the launch's first block.  The inverse transforms skip
// what lies outside Xi.
// --------------------------------------------------------------------------
template <int n, class T>
struct CellTerms {
  using C2 = typename Vec2Of<T>::type;
  const C2* what;
  const C2* wfine;
  C2* D;          // [c][ch][2][P]
  T* K2;          // [c][ch][2][P], cells k2_cell reals apart
  C2* K4;         // [c][ch][2][P]
  size_t k2_cell;
  C2* ws1;        // one field per I1 team
  C2* ws24;       // three fields per I2/I4 team
  const C2* tw;
  const T* phip;
  const T* Ktab;
  const T* psi;
  int J, nch, teams1, first;
};

template <int n, class T, int CB>
__global__ void __launch_bounds__(kThreads, (cell_min_blocks<n, T, CB>()))
    k_i124(const CellTerms<n, T> a) {
  using C2 = typename Vec2Of<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* tw = reinterpret_cast<C2*>(smem_raw);
  C2* sm = tw + n;
  load_twiddles<n>(tw, a.tw);
  constexpr int P = n * n, B = Split<n>::B;
  const int team = cluster_index() + a.first, J = a.J, nch = a.nch;
  const bool i1 = team < a.teams1;
  const int id = i1 ? team : team - a.teams1;
  const int p = id & 1, cch = id >> 1, c = cch / nch, ch = cch % nch;
  const C2* wf0 = a.wfine + (size_t)c * 2 * P;
  auto load_xi = [&](const C2* G) {
    return [G](int ix, int iy) { return xi_t<B>(iy % B) ? ldc<n, CB>(&G[ix * n + iy]) : zero2<T>(); };
  };
  if (i1) {
    C2* G = a.ws1 + (size_t)id * P;
    C2* Dp = a.D + (size_t)id * P;
    const C2* in = a.what + ((size_t)c * 4 + 2 + p) * P;
    zero_fields_team(Dp, P);
    for (int jp = J * ch / nch; jp < J * (ch + 1) / nch; ++jp) {
      const T* ph = a.phip + (size_t)jp * P;
      const T* K = a.Ktab + (size_t)jp * P;
      xi_col_pass<n, CB>(
          sm, tw, [&](int ix, int iy) { return cscale(in[ix * n + iy], ph[ix * n + iy]); },
          [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
      row_pass<n, 1, true, -1, CB, true>(
          sm, tw, load_xi(G), [&](int ix, int iy, C2 v) { return cscale(v, (T)2 * wf0[ix * n + iy].x - (T)1); },
          [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
      col_pass<n, -1, false, 0, CB>(
          sm, tw, [&](int ix, int iy) { return ldc<n, CB>(&G[ix * n + iy]); }, NoMid(),
          [&](int ix, int iy, C2 v) {
            const T k = K[ix * n + iy];
            const C2 d = Dp[ix * n + iy];
            Dp[ix * n + iy] = mk2(fmaT(k, v.x, d.x), fmaT(k, v.y, d.y));
          });
    }
    return;
  }
  C2* FA = a.ws24 + (size_t)id * 3 * P;
  C2* FB = FA + P;
  C2* G = FA + 2 * P;
  T* K2 = a.K2 + c * a.k2_cell + ((size_t)ch * 2 + p) * P;
  C2* K4 = a.K4 + (size_t)id * P;
  for (int i = element_first(); i < P; i += element_stride()) K2[i] = (T)0;
  zero_fields_team(K4, P);
  const C2* in = a.what + ((size_t)c * 4 + p) * P;
  const T wj = (T)(kPi / J);
  const T scale = (T)(kPi / J / (double)P);
  const T e0 = p == 0 ? (T)1 : (T)-1;   // eta of component 2 p
  const int H = J / 2;
  for (int j = H * ch / nch; j < H * (ch + 1) / nch; ++j) {
    const int jp = j + J / 2;
    for (int h = 0; h < 2; ++h) {
      const T* ps = a.psi + (size_t)(h == 0 ? j : jp) * P;
      C2* F = h == 0 ? FA : FB;
      xi_col_pass<n, CB>(
          sm, tw, [&](int ix, int iy) { return cscale(in[ix * n + iy], ps[ix * n + iy]); },
          [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
      row_pass<n, 1, false, 0, CB, true>(
          sm, tw, load_xi(G), NoMid(), [&](int ix, int iy, C2 v) { F[ix * n + iy] = v; });
    }
    for (int i = element_first(); i < P; i += element_stride()) {
      const C2 fa = ldc<n, CB>(&FA[i]), fb = ldc<n, CB>(&FB[i]);
      K2[i] = fmaT((T)2 * wj, e0 * fa.x * fb.x - fa.y * fb.y, K2[i]);
    }
    team_sync();
    for (int h = 0; h < 2; ++h) {
      const C2* F = h == 0 ? FB : FA;   // psi_j pairs with F_{j+J/2}
      const T* ps = a.psi + (size_t)(h == 0 ? j : jp) * P;
      row_pass<n, -1, false, 0, CB>(
          sm, tw, [&](int ix, int iy) { return cscale(ldc<n, CB>(&F[ix * n + iy]), (T)2 * wf0[ix * n + iy].x - (T)1); },
          NoMid(), [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
      col_pass<n, -1, false, 0, CB>(
          sm, tw, [&](int ix, int iy) { return ldc<n, CB>(&G[ix * n + iy]); }, NoMid(),
          [&](int ix, int iy, C2 v) {
            const T k = scale * ps[ix * n + iy];
            const C2 d = K4[ix * n + iy];
            K4[ix * n + iy] = mk2(fmaT(k, v.x, d.x), fmaT(k, v.y, d.y));
          });
    }
  }
}

// Blocks of a grid-stride kernel over `count` elements (counted in 64 bits: a call may hold millions of cells).
inline unsigned element_blocks(size_t count) {
  const size_t b = (count + kThreads - 1) / kThreads, most = 152 * 32;
  return (unsigned)(b < most ? b : most);
}

// Sums of the partials of k_i124 of each cell, in order: D and K4 (2 complex fields each) over the nch
// chunks (skipped with one: the kernel writes the sums), K2 (real) over its 2 nch planes.
template <class T>
__global__ void __launch_bounds__(kThreads) k_reduce_chunks(const T* __restrict__ Dpart, const T* __restrict__ K2part,
                                                            const T* __restrict__ K4part, T* Dacc, T* K2acc, T* K4acc,
                                                            int nch, int ncells, size_t P, size_t k2_cell) {
  const size_t per_c = nch > 1 ? 4 * P : 0;   // reals of D and of K4 per cell
  const size_t total = (size_t)ncells * (2 * per_c + P);
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const T* p;
    T* dst;
    size_t stride;
    int planes = nch;
    if (i < (size_t)ncells * 2 * per_c) {
      const bool second = i >= (size_t)ncells * per_c;
      const size_t k = second ? i - (size_t)ncells * per_c : i;
      stride = per_c;
      p = (second ? K4part : Dpart) + (k / per_c * nch) * per_c + k % per_c;
      dst = (second ? K4acc : Dacc) + k;
    } else {
      const size_t k = i - (size_t)ncells * 2 * per_c;
      stride = P;
      planes = 2 * nch;
      p = K2part + k / P * k2_cell + k % P;
      dst = K2acc + k;
    }
    T sum = p[0];
    for (int ch = 1; ch < planes; ++ch) sum += p[(size_t)ch * stride];
    *dst = sum;
  }
}

// --------------------------------------------------------------------------
// I3 (dominant, Hu-Ying form eq. approxH-JM).  Persistent blocks over units
// (cell, j, m-chunk).  For each m:
//   Sigma_p = IFFT(e^{i alpha_jm.sigma} sqrt(c_jm) w^_pair p)   (shifted fields S_a = w_a(v + rho_m theta_j))
//   for a, p:  T = IFFT(psi'_j FFT(w_a Sigma_p)) / n^2;  acc_p += eta_a S_a T
// The unit's partial sum acc[2][n*n] (pairs (0,1), (2,3), real space) is
// written to its own slot of K3part and reduced in fixed order later.
// --------------------------------------------------------------------------
// The staged kernel's launch shape (threads per block, shared-memory chunk bytes of its row and
// column passes, blocks per SM) is a template parameter: the autotuner chooses among the
// instantiated shapes (i3_variant below).
template <int n, class T, int NTH = 256, int CB = 65536, int MINB = 3>
__global__ void __launch_bounds__(NTH, MINB)
    k_i3(const I3Jobs<T> jobs, typename Vec2Of<T>::type* ws, const typename Vec2Of<T>::type* __restrict__ gtw) {
  using C2 = typename Vec2Of<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* tw = reinterpret_cast<C2*>(smem_raw);
  C2* sm = tw + n;
  __shared__ int xcols[n];          // permuted positions whose frequency lies in Xi (incl. its -N/2 line)
  __shared__ unsigned char xmask[n];
  if (threadIdx.x == 0) {
    int cnt = 0;
    for (int pos = 0; pos < n; ++pos) {
      const int k = freq_of_pos<n>(pos);
      const bool in = (k < n / 4) || (k >= n - n / 4);
      xmask[pos] = in ? 1 : 0;
      if (in) xcols[cnt++] = pos;
    }
  }
  load_twiddles<n>(tw, gtw);
  constexpr int P = n * n;
  C2* slot = ws + (size_t)blockIdx.x * 3 * P;
  C2* Sig = slot;           // [2][P]
  C2* G = slot + 2 * P;
  for (int gunit = blockIdx.x; gunit < jobs.total; gunit += gridDim.x) {
    const I3Job<T>& jb = jobs.job[i3_job_of(jobs, gunit)];
    const int unit = gunit - jb.unit_begin;
    const int J = jb.J, M = jb.M, nmc = jb.nmc;
    const C2* what = jb.what;
    const T* __restrict__ psip_s = jb.psip_s;
    const C2* __restrict__ phase = jb.phase;
    const int c = unit / (J * nmc);
    const int j = (unit / nmc) % J;
    const int mc = unit % nmc;
    C2* acc = jb.K3part + (size_t)unit * 2 * P;
    zero_fields(acc, 2 * P);
    const T* psp = psip_s + (size_t)j * P;
    const C2* wf = jb.wfine + (size_t)c * 2 * P;
    const int m0 = i3_chunk_begin(mc, nmc, M), m1 = i3_chunk_begin(mc + 1, nmc, M);
    for (int m = m0; m < m1; ++m) {
      const C2* px = phase + ((size_t)j * M + m) * 2 * n;
      const C2* py = px + n;
      for (int p = 0; p < 2; ++p) {
        const C2* in = what + ((size_t)c * 4 + p) * P;
        C2* S = Sig + (size_t)p * P;
        // only the n/2 columns (y frequencies) of Xi are non-zero: transform those
        col_pass_list<n, 1, false, 0, CB, true>(
            sm, tw, xcols, n / 2,
            [&](int ix, int iy) { return xmask[ix] ? cmul(in[ix * n + iy], cmul(px[ix], py[iy])) : zero2<T>(); },
            NoMid(), [&](int ix, int iy, C2 v) { S[ix * n + iy] = v; });
        row_pass<n, 1, false, 0, CB, true>(
            sm, tw, [&](int ix, int iy) { return xmask[iy] ? S[ix * n + iy] : zero2<T>(); }, NoMid(),
            [&](int ix, int iy, C2 v) { S[ix * n + iy] = v; });
      }
      for (int a = 0; a < 4; ++a) {
        const C2* wa = wf + (size_t)(a >> 1) * P;
        const C2* Sa = Sig + (size_t)(a >> 1) * P;
        const bool im = (a & 1) != 0;
        const bool pos_eta = (a == 0);
        for (int p = 0; p < 2; ++p) {
          const C2* Sp = Sig + (size_t)p * P;
          C2* accp = acc + (size_t)p * P;
          row_pass<n, -1, false, 0, CB>(
              sm, tw,
              [&](int ix, int iy) {
                const C2 z = wa[ix * n + iy];
                return cscale(Sp[ix * n + iy], im ? z.y : z.x);
              },
              NoMid(), [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
          col_conv_pass<n, CB>(
              sm, tw, [&](int ix, int iy) { return G[ix * n + iy]; },
              [&](int ix, int iy) { return psp[ix * n + iy]; },
              [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
          row_pass<n, 1, false, 0, CB>(
              sm, tw, [&](int ix, int iy) { return G[ix * n + iy]; }, NoMid(),
              [&](int ix, int iy, C2 v) {
                // eta_a = +1 for a = 0, -1 otherwise: the sign goes into the FMAs
                const C2 s = Sa[ix * n + iy];
                const T f = im ? s.y : s.x;
                const C2 d = accp[ix * n + iy];
                accp[ix * n + iy] = pos_eta ? mk2(fmaT(f, v.x, d.x), fmaT(f, v.y, d.y))
                                            : mk2(fmaT(-f, v.x, d.x), fmaT(-f, v.y, d.y));
              });
        }
      }
    }
  }
}

// --------------------------------------------------------------------------
// I3 with the transform field resident in shared memory (FP32, n <= 128: an
// n x (n+1) complex float field is at most 129 KB), nodes in pairs as in k_i3_sf
// (i3_staged_fused.cuh).  Each convolution (row FFT, column psi' convolution, row
// IFFT) runs entirely on chip; global memory holds the two shifted fields and V_q
// per block and the partial sums.
// --------------------------------------------------------------------------
constexpr int kThreadsI3Smem = 1024;

template <int n>
__global__ void __launch_bounds__(kThreadsI3Smem, 1) k_i3_smem(const I3Jobs<float> jobs, float2* ws,
                                                             const float2* __restrict__ gtw) {
  using C2 = float2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* tw = reinterpret_cast<C2*>(smem_raw);
  C2* G = tw + n;                       // [n][LS]
  float* psm = reinterpret_cast<float*>(G + n * (n + 1));   // psi'_j of the current unit, [n][n]
  constexpr int LS = n + 1, P = n * n;
  constexpr int NQ = xi_kept<n>(), Q = NQ * NQ;
  constexpr int kIter = (P + kThreadsI3Smem - 1) / kThreadsI3Smem;
  __shared__ unsigned char xmask[n];
  __shared__ int kslot[n];
  __shared__ int kcols[n];
  for (int pos = threadIdx.x; pos < n; pos += blockDim.x) xmask[pos] = xi_t<Split<n>::B>(pos % Split<n>::B) ? 1 : 0;
  build_xi_slots<n>(kslot, kcols);
  load_twiddles<n>(tw, gtw);
  C2* Sig = ws + (size_t)blockIdx.x * 3 * P;   // [2][P]
  C2* V = Sig + 2 * P;
  for (int gunit = blockIdx.x; gunit < jobs.total; gunit += gridDim.x) {
    const I3Job<float>& jb = jobs.job[i3_job_of(jobs, gunit)];
    const int unit = gunit - jb.unit_begin;
    const int J = jb.J, M = jb.M, nmc = jb.nmc;
    const C2* what = jb.what;
    const float* __restrict__ psip_s = jb.psip_s;
    const C2* __restrict__ phase = jb.phase;
    const int c = unit / (J * nmc);
    const int j = (unit / nmc) % J;
    const int mc = unit % nmc;
    float* K = reinterpret_cast<float*>(jb.K3part + (size_t)unit * 2 * P);   // [4][P]
    C2* spec = jb.K3spec + (size_t)unit * 2 * Q;
    {
      const float4* src = reinterpret_cast<const float4*>(psip_s + (size_t)j * P);
      float4* dst = reinterpret_cast<float4*>(psm);
      for (int i4 = threadIdx.x; i4 < P / 4; i4 += blockDim.x) dst[i4] = src[i4];
      __syncthreads();
    }
    const C2* __restrict__ wf = jb.wfine + (size_t)c * 2 * P;
    const int it1 = i3_chunk_begin(mc + 1, nmc, M);
    bool k_first = true, s_first[2] = {true, true};
    for (int it = i3_chunk_begin(mc, nmc, M); it < it1;) {
      const I3Group gr = i3_group_at(it, it1, M);
      it = gr.next;
      const C2* px = phase + ((size_t)j * M + gr.m) * 2 * n;
      const C2* py = px + n;
      for (int p = 0; p < 2; ++p) {
        const C2* in = what + ((size_t)c * 4 + p) * P;
        for (int idx = threadIdx.x; idx < P; idx += blockDim.x) {
          const int ix = idx / n, iy = idx % n;
          G[ix * LS + iy] = (xmask[ix] && xmask[iy]) ? cmul(in[idx], cmul(px[ix], py[iy])) : zero2<float>();
        }
        __syncthreads();
        fft_lines<n, 1, true>(G, n, 1, LS, tw);     // columns (along ix), input zero outside Xi
        fft_lines<n, 1, true>(G, n, LS, 1, tw);     // rows (along iy), zero outside the Xi columns
        C2* S = Sig + (size_t)p * P;
        for (int idx = threadIdx.x; idx < P; idx += blockDim.x) S[idx] = G[(idx / n) * LS + idx % n];
        __syncthreads();
      }
      for (int q = gr.q0; q < gr.q1; ++q) {
        const C2* __restrict__ wq = wf + (size_t)q * P;
        const C2* Sq = Sig + (size_t)q * P;
        const float e0 = q == 0 ? 1.f : -1.f;
        for (int b = 0; b < 4; ++b) {
          const float* Sb = reinterpret_cast<const float*>(Sig + (size_t)(b >> 1) * P) + (b & 1);
          const float* __restrict__ wb = reinterpret_cast<const float*>(wf + (size_t)(b >> 1) * P) + (b & 1);
          float* Kb = K + (size_t)b * P;
          const float eb = b == 0 ? 1.f : -1.f;
          // element loops with a compile-time trip count, unrolled so each thread keeps several
          // L2 loads in flight (one block per SM leaves few warps to hide their latency)
#pragma unroll 8
          for (int k = 0; k < kIter; ++k) {
            const int idx = threadIdx.x + k * kThreadsI3Smem;
            if (kIter * kThreadsI3Smem == P || idx < P) G[(idx / n) * LS + idx % n] = cscale(wq[idx], Sb[2 * idx]);
          }
          __syncthreads();
          fft_lines<n, -1>(G, n, LS, 1, tw);                                           // rows forward
          fft_conv_lines<n>(G, n, 1, LS, tw, [&](int l, int pos) { return psm[pos * n + l]; });   // columns
          fft_lines<n, 1>(G, n, LS, 1, tw);                                            // rows inverse
#pragma unroll 8
          for (int k = 0; k < kIter; ++k) {
            const int idx = threadIdx.x + k * kThreadsI3Smem;
            if (kIter * kThreadsI3Smem == P || idx < P) {
              const C2 u = G[(idx / n) * LS + idx % n];
              const C2 s2 = Sq[idx];
              const float t = fmaT(e0 * s2.x, u.x, -s2.y * u.y);
              if (k_first) Kb[idx] = t;
              else atomicAdd(Kb + idx, t);     // no other thread adds to this point
              const float f = eb * wb[2 * idx], fx = -e0 * f;
              if (b == 0) {
                V[idx] = mk2(fx * u.x, f * u.y);
              } else {
                const C2 d = V[idx];
                V[idx] = mk2(fmaT(fx, u.x, d.x), fmaT(f, u.y, d.y));
              }
            }
          }
          __syncthreads();
        }
        k_first = false;
        if (!gr.pair) continue;
        for (int idx = threadIdx.x; idx < P; idx += blockDim.x) G[(idx / n) * LS + idx % n] = V[idx];
        __syncthreads();
        fft_lines<n, -1>(G, n, LS, 1, tw);    // rows
        fft_lines<n, -1>(G, n, 1, LS, tw);    // columns
        C2* dst = spec + (size_t)q * Q;
        const bool first = s_first[q];
        s_first[q] = false;
        for (int e = threadIdx.x; e < Q; e += blockDim.x) {
          const int ix = kcols[e / NQ], iy = kcols[e % NQ];
          const C2 z = cmulc(G[ix * LS + iy], cmul(px[ix], py[iy]));
          dst[e] = first ? z : cadd(dst[e], z);
        }
        __syncthreads();
      }
    }
    for (int q = 0; q < 2; ++q)
      if (s_first[q]) zero_fields(spec + (size_t)q * Q, Q);
  }
}

template <int n>
constexpr bool use_i3_smem() {
  return n <= 128;
}

template <int n>
constexpr size_t i3_smem_bytes() {   // twiddles, the field (padded rows), psi'_j
  return (size_t)(n + n * (n + 1)) * sizeof(float2) + (size_t)n * n * sizeof(float);
}

#include "i3_fused.cuh"
#include "i3_staged_fused.cuh"
#include "i3_tmem.cuh"
#include "i3_lines.cuh"

// Padded sizes with the fused shared-memory FP32 kernel (whole row tasks per thread for its shapes).
template <int n>
__host__ __device__ constexpr bool use_i3_fused() {
  return n == 64 || n == 96 || n == 128;
}
// Its launch shapes per size: (threads, blocks per SM, accumulation mode of k_i3_fused), and the
// default variant (I3 launch, J = M = 32, on a GB300).  N = 16, 256 cells: 5.0 ms for k_i3_tmem.  N = 32,
// 128 cells: 12.5 ms for k_i3_tmem (variant 0; 28.6 ms for the fused kernel with register accumulation that
// it replaces), 38.8 and 52.3 for shapes 1 and 2, 19.6 for k_i3_smem.  N = 48, 64 cells: 14.3 for k_i3_lines
// (variant 3; 25.2 for k_i3_smem, which it replaces, 38.5 node by node), 38.8, 40.4, 53.2 for the fused shapes.  N = 64,
// 128 cells: 47.6 for k_i3_tmem (variant 4; 88.6 for the warp-local kernel, node by node, that it
// replaces), 101.1, 116.4, 114.5 for shapes 0 to 2, 83.1 for k_i3_smem.
template <int n> struct FusedShapes;
template <> struct FusedShapes<64> {   // variant 0: k_i3_tmem
  static constexpr int T0 = 0, B0 = 0, M0 = 1, T1 = 512, B1 = 2, M1 = 2, T2 = 256, B2 = 4, M2 = 2, DEFAULT = 0;
};
template <> struct FusedShapes<96> {   // variant 3: k_i3_lines
  static constexpr int T0 = 768, B0 = 1, M0 = 0, T1 = 768, B1 = 1, M1 = 2, T2 = 384, B2 = 2, M2 = 2, DEFAULT = 3;
};
template <> struct FusedShapes<128> {   // variant 4: k_i3_tmem
  static constexpr int T0 = 512, B0 = 1, M0 = 1, T1 = 1024, B1 = 1, M1 = 2, T2 = 1024, B2 = 1, M2 = 0, DEFAULT = 4;
};

// --------------------------------------------------------------------------
// I3 on padded grids above 128 points in FP32 (n = 192, 256: one field is 288 or 512 KB, more
// than one block's shared memory).  A cluster of kI3Cluster CTAs works on one unit at a time:
// CTA r holds rows [r R, r R + R) of the transform field (R = n / kI3Cluster) for the row
// transforms and columns [r R, r R + R) for the column psi' convolution, with the angle's psi'
// columns in shared memory.  The transposes between the two go through the cluster's field in
// global memory, stored transposed (G'[ky][x]) so that the line stages load and store it directly,
// coalesced, ordered by cluster barriers; per cluster that field and the two shifted fields
// (3 n^2 complex values) stay L2-resident, where 152 independent units of the staged kernel
// (about 2.5 MB each) would not.  Same units and line transforms as k_i3.  Every CTA of a cluster
// runs the same loop trip counts, so every barrier is reached by all of them (hardware barriers,
// no spin waits).
// --------------------------------------------------------------------------
// Measured at N = 128 (32 cells, C[W] I3 launch), element passes through shared memory around
// every global access: 4 CTAs x 1024 threads 239.9 ms; 8 CTAs x 512 threads (two CTAs of
// different clusters per SM) 255.4 ms; the staged k_i3 294.5 ms.  With the line stages reading
// and writing the transposed field directly: 219.1 ms (1024 threads, mode 0 below), 192.4 ms
// (512 threads, mode 1 node by node), 132.4 ms (mode 1, nodes in pairs, the sums over a in registers).
// Those took 64 of a thread's 128 registers; in tensor memory they leave room for both of its tasks' loads at
// a time: 14 cells 58.0 -> 42.7 ms, N = 96, 32 cells 70.8 -> 62.6 ms; with the operands in thread_order 40.8
// and 59.8 ms.  What is left is L2 traffic (60 bytes per point and convolution, 32 of them the two
// transposes) between phases that four blocks share; the transposes as stores into the other blocks' shared
// memory took 44.8 ms, the field in 16-byte words of two lines 41.7.
constexpr int kI3Cluster = 4;             // CTAs per cluster
constexpr int kThreadsI3Cluster = 1024;   // threads per CTA of mode 0

template <int n>
__host__ __device__ constexpr bool use_i3_cluster() {
  return n > 128;
}

template <int n>
__host__ __device__ constexpr int i3_cluster_slab() {   // complex elements of the row / column slab
  constexpr int R = n / kI3Cluster;
  return R * (n + 1) > n * R ? R * (n + 1) : n * R;
}

template <int n>
constexpr size_t i3_cluster_smem_bytes() {   // twiddles (two orders), the slab, psi' columns
  return (size_t)(2 * n + i3_cluster_slab<n>()) * sizeof(float2) + (size_t)n * (n / kI3Cluster) * sizeof(float);
}

// The cluster kernel's launch shapes: NT threads per CTA and the accumulation mode.  MODE 0: loop a
// (outer), p (inner), each convolution's last stage adds eta_a S_a T into the unit's partial sum in
// global memory (read-modify-write per convolution).  MODE 1: loop p (outer), a (inner), the last
// stage accumulates over a in tensor memory (each thread owns the same points in every convolution);
// NT = R B / 2, so that every thread owns two row tasks.
template <int n>
constexpr int i3_cluster_threads(int mode) {
  return mode == 0 ? kThreadsI3Cluster : (n / kI3Cluster) * Split<n>::B / 2;
}

template <int n, int NT, int MODE>
__global__ void __cluster_dims__(kI3Cluster, 1, 1) __launch_bounds__(NT, 1)
    k_i3_cluster(const I3Jobs<float> jobs, float2* ws, const float2* __restrict__ gtw) {
  static_assert(n / kI3Cluster * n >= NT, "at least one element per thread in every phase");
  using C2 = float2;
  constexpr int R = n / kI3Cluster, LS = n + 1, P = n * n;
  constexpr int XC = (n / 2) / kI3Cluster;           // Xi columns per CTA in the shift transforms
  constexpr int A = Split<n>::A, B = Split<n>::B;
  constexpr int TA = (R * B + NT - 1) / NT;          // row tasks (r, t2) per thread in an A stage
  constexpr int TB = (R * A + NT - 1) / NT;          // tasks (r, k1) per thread in a B stage
  constexpr int W4 = TA * A / 4;                     // MODE 1: words of a thread in a plane of R rows
  constexpr int NQ = xi_kept<n>(), Q = NQ * NQ;
  static_assert(MODE == 0 || R * B == 2 * NT, "accumulation at the thread's own points: two row tasks per thread");
  static_assert(n % kI3Cluster == 0 && (n / 2) % kI3Cluster == 0, "cluster split");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* tw = reinterpret_cast<C2*>(smem_raw);
  C2* twT = tw + n;                                  // twT[k1 B + t2] = tw[t2 A + k1] (t2-fastest lanes)
  C2* F = twT + n;                                   // [R][LS] row or line slab, [n][XC] shift column slab
  float* psl = reinterpret_cast<float*>(F + i3_cluster_slab<n>());   // psi'_j of this CTA's lines, [n][R]
  __shared__ int xcols[n];
  __shared__ unsigned char xmask[n];
  if (threadIdx.x == 0) {
    int cnt = 0;
    for (int pos = 0; pos < n; ++pos) {
      const int k = freq_of_pos<n>(pos);
      const bool in = (k < n / 4) || (k >= n - n / 4);
      xmask[pos] = in ? 1 : 0;
      if (in) xcols[cnt++] = pos;
    }
  }
  for (int pos = threadIdx.x; pos < n; pos += NT) twT[(pos % A) * B + pos / A] = gtw[pos];
  load_twiddles<n>(tw, gtw);
  __shared__ uint32_t tm_slot;
  uint32_t tm_base = 0, tv = 0;                      // MODE 1: V_q, per row task A real, A imaginary parts
  if constexpr (MODE == 1) {
    tm_base = tmem_alloc<tmem_columns(NT, 2 * TA * A)>(&tm_slot);
    tv = tmem_mine<2 * TA * A>(tm_base);
  }
  const int tid = threadIdx.x;
  const int rank = cluster_rank();
  const int r0 = rank * R;                           // this CTA's first row / column
  C2* Gs = ws + (size_t)cluster_index() * 3 * P;     // the cluster's transform field
  C2* Sig = Gs + P;                                  // the two shifted pairs
  // One Psi'_j convolution of the field load(idx) (idx = r n + y, r a row of this CTA), with the
  // last stage's results handed to epi(i, t1, idx, v) (i: the thread's row task, t1: its element).
  // Between the passes the cluster's field is stored transposed, Gs'[ky][x] (ky in the row
  // transform's permuted order): the row passes reach it from stage B (lanes = consecutive rows of
  // this CTA) and the line pass from stage A (contiguous in x), so every global access is inside a
  // line stage and coalesced.
  // Each stage loads both of a thread's tasks before it transforms the first: the loads' latency is what
  // bounds the kernel.
  auto a_task = [&](int i, int& r, int& t2) {        // row task i of the thread
    const int task = tid + i * NT;
    r = task / B;
    t2 = task % B;
    return TA * NT == R * B || task < R * B;
  };
  auto b_task = [&](int i, int& r, int& k1) {
    const int task = tid + i * NT;
    r = task % R;
    k1 = task / R;
    return TB * NT == R * A || task < R * A;
  };
  // lines of v through stage A into F
  auto stage_a_forward = [&](C2 (&v)[A], int r, int t2) {
    dft<A, -1>(v);
#pragma unroll
    for (int k1 = 1; k1 < A; ++k1) v[k1] = cmul(v[k1], twT[k1 * B + t2]);
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) F[r * LS + B * k1 + t2] = v[k1];
  };
  auto stage_a_inverse = [&](C2 (&v)[A], int r, int t2) {
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) v[k1] = F[r * LS + B * k1 + t2];
#pragma unroll
    for (int k1 = 1; k1 < A; ++k1) v[k1] = cmulc(v[k1], twT[k1 * B + t2]);
    dft<A, 1>(v);
  };
  auto convolve = [&](auto load, auto epi) {
    int r, t2, k1;
    {
      C2 v[TA][A];
#pragma unroll
      for (int i = 0; i < TA; ++i)                   // forward rows: stage A loads the product
        if (a_task(i, r, t2)) load(i, r, t2, v[i]);
#pragma unroll
      for (int i = 0; i < TA; ++i)
        if (a_task(i, r, t2)) stage_a_forward(v[i], r, t2);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TB; ++i)
      if (b_task(i, r, k1)) {
        C2 b[B];
#pragma unroll
        for (int t = 0; t < B; ++t) b[t] = F[r * LS + B * k1 + t];
        dft<B, -1>(b);
#pragma unroll
        for (int t = 0; t < B; ++t) Gs[(size_t)(B * k1 + t) * n + r0 + r] = b[t];
      }
    cluster_sync_global();                           // all rows transformed
    // psi' convolution along x on this CTA's lines ky in [r0, r0 + R)
    {
      C2 v[TA][A];
#pragma unroll
      for (int i = 0; i < TA; ++i)
        if (a_task(i, r, t2)) {
#pragma unroll
          for (int t1 = 0; t1 < A; ++t1) v[i][t1] = __ldcg(&Gs[(size_t)(r0 + r) * n + B * t1 + t2]);
        }
#pragma unroll
      for (int i = 0; i < TA; ++i)
        if (a_task(i, r, t2)) stage_a_forward(v[i], r, t2);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TB; ++i)
      if (b_task(i, r, k1)) {
        C2 b[B];
#pragma unroll
        for (int t = 0; t < B; ++t) b[t] = F[r * LS + B * k1 + t];
        dft<B, -1>(b);
        float sc[B];
#pragma unroll
        for (int t = 0; t < B; ++t) sc[t] = psl[(B * k1 + t) * R + r];
        dft_scaled<B, 1>(b, sc);
#pragma unroll
        for (int t = 0; t < B; ++t) F[r * LS + B * k1 + t] = b[t];
      }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TA; ++i)
      if (a_task(i, r, t2)) {
        C2 v[A];
        stage_a_inverse(v, r, t2);
#pragma unroll
        for (int t1 = 0; t1 < A; ++t1) Gs[(size_t)(r0 + r) * n + B * t1 + t2] = v[t1];
      }
    cluster_sync_global();                           // all lines convolved
    // inverse rows on this CTA's rows: stage B loads, the epilogue takes stage A
    {
      C2 b[TB][B];
#pragma unroll
      for (int i = 0; i < TB; ++i)
        if (b_task(i, r, k1)) {
#pragma unroll
          for (int t = 0; t < B; ++t) b[i][t] = __ldcg(&Gs[(size_t)(B * k1 + t) * n + r0 + r]);
        }
#pragma unroll
      for (int i = 0; i < TB; ++i)
        if (b_task(i, r, k1)) {
          dft<B, 1>(b[i]);
#pragma unroll
          for (int t = 0; t < B; ++t) F[r * LS + B * k1 + t] = b[i][t];
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TA; ++i)
      if (a_task(i, r, t2)) epi(i, r, t2);
    __syncthreads();
  };
  for (int gunit = cluster_index(); gunit < jobs.total; gunit += cluster_count()) {
    const I3Job<float>& jb = jobs.job[i3_job_of(jobs, gunit)];
    const int unit = gunit - jb.unit_begin;
    const int J = jb.J, M = jb.M, nmc = jb.nmc;
    const C2* what = jb.what;
    const C2* __restrict__ phase = jb.phase;
    const int c = unit / (J * nmc);
    const int j = (unit / nmc) % J;
    const int mc = unit % nmc;
    C2* acc = jb.K3part + (size_t)unit * 2 * P;
    if (MODE == 0) {
      #pragma unroll 1
      for (int idx = tid; idx < R * n; idx += NT) {
        acc[(size_t)r0 * n + idx] = zero2<float>();
        acc[P + (size_t)r0 * n + idx] = zero2<float>();
      }
    }
    const float* __restrict__ psp = jb.psip_s + (size_t)j * P;
    #pragma unroll 1
    for (int idx = tid; idx < n * R; idx += NT) psl[idx] = psp[(idx / R) * n + r0 + idx % R];
    __syncthreads();
    const C2* wf = jb.wfine + (size_t)c * 2 * P;     // MODE 0
    const float* __restrict__ wp = jb.wplane + (size_t)c * 4 * P + (size_t)r0 * n;   // MODE 1: this block's rows
    const int it1 = i3_chunk_begin(mc + 1, nmc, M);
    C2* spec = jb.K3spec + (size_t)unit * 2 * Q;     // MODE 1
    bool k_first = true, s_first0 = true, s_first1 = true;
    for (int it = i3_chunk_begin(mc, nmc, M); it < it1;) {
      I3Group gr = {it, 0, 2, it + 1, false};        // MODE 0: an item is a node
      if constexpr (MODE == 1) gr = i3_group_at(it, it1, M);
      it = gr.next;
      const C2* px = phase + ((size_t)j * M + gr.m) * 2 * n;
      const C2* py = px + n;
      cluster_sync_global();                         // the previous m's (or unit's) Sig and Gs are read
      // shifted fields, column transforms over this CTA's share of the Xi columns
      for (int p = 0; p < 2; ++p) {
        const C2* in = what + ((size_t)c * 4 + p) * P;
        C2* S = Sig + (size_t)p * P;
        #pragma unroll 1
        for (int idx = tid; idx < n * XC; idx += NT) {
          const int ix = idx / XC, cc = idx % XC, iy = xcols[rank * XC + cc];
          F[idx] = xmask[ix] ? cmul(in[ix * n + iy], cmul(px[ix], py[iy])) : zero2<float>();
        }
        __syncthreads();
        fft_lines<n, 1, true>(F, XC, 1, XC, tw);
        #pragma unroll 1
        for (int idx = tid; idx < n * XC; idx += NT) {
          const int ix = idx / XC, cc = idx % XC;
          S[ix * n + xcols[rank * XC + cc]] = F[idx];
        }
        __syncthreads();
      }
      cluster_sync_global();                         // the Xi columns of both shifted fields are complete
      // row transforms over this CTA's rows (columns outside Xi are zero)
      for (int p = 0; p < 2; ++p) {
        C2* S = Sig + (size_t)p * P + (size_t)r0 * n;
        #pragma unroll 1
        for (int idx = tid; idx < R * n; idx += NT) {
          const int r = idx / n, iy = idx % n;
          F[r * LS + iy] = xmask[iy] ? __ldcg(&S[idx]) : zero2<float>();
        }
        __syncthreads();
        fft_lines<n, 1, true>(F, R, LS, 1, tw);
        if constexpr (MODE == 0) {
          #pragma unroll 1
          for (int idx = tid; idx < R * n; idx += NT) S[idx] = F[(idx / n) * LS + idx % n];
        } else {                                     // the rows' two planes, in thread_order
          float4* S4 = reinterpret_cast<float4*>(S) + tid;
#pragma unroll 2
          for (int w = 0; w < W4; ++w) {
            const int task = tid + w / (A / 4) * NT;
            const C2* f = F + task / B * LS + task % B + B * (w % (A / 4) * 4);
            const C2 z0 = f[0], z1 = f[B], z2 = f[2 * B], z3 = f[3 * B];
            S4[w * NT] = make_float4(z0.x, z1.x, z2.x, z3.x);
            S4[(W4 + w) * NT] = make_float4(z0.y, z1.y, z2.y, z3.y);
          }
        }
        __syncthreads();
      }
      // from here on this CTA reads only its own rows of the shifted fields
      if constexpr (MODE == 0) {
        for (int a = 0; a < 4; ++a) {
          // component im of the fine pair and of the shifted pair, loaded as single floats
          const int im = a & 1;
          const float* wa = reinterpret_cast<const float*>(wf + (size_t)(a >> 1) * P + (size_t)r0 * n) + im;
          const float* Sa = reinterpret_cast<const float*>(Sig + (size_t)(a >> 1) * P + (size_t)r0 * n) + im;
          const float eta = (a == 0) ? 1.f : -1.f;
          for (int p = 0; p < 2; ++p) {
            const C2* Sp = Sig + (size_t)p * P + (size_t)r0 * n;
            C2* accp = acc + (size_t)p * P + (size_t)r0 * n;
            convolve([&](int, int r, int t2, C2 (&v)[A]) {
#pragma unroll
                       for (int t1 = 0; t1 < A; ++t1) {
                         const int idx = r * n + B * t1 + t2;
                         v[t1] = cscale(Sp[idx], wa[2 * idx]);
                       }
                     },
                     [&](int, int r, int t2) {
                       C2 v[A];
                       stage_a_inverse(v, r, t2);
#pragma unroll
                       for (int t1 = 0; t1 < A; ++t1) {
                         const int idx = r * n + B * t1 + t2;
                         const float f = eta * Sa[2 * idx];
                         const C2 d = accp[idx];
                         accp[idx] = mk2(fmaT(f, v[t1].x, d.x), fmaT(f, v[t1].y, d.y));
                       }
                     });
          }
        }
      } else {
        const int xl0 = rank * XC;                   // this CTA's share of the n / 2 lines ky of Xi
        auto xi_line = [&](int cc) { return xcols[xl0 + cc]; };
        for (int q = gr.q0; q < gr.q1; ++q) {
          // this thread's words of the rows' planes
          const float4* wq = reinterpret_cast<const float4*>(wp + (size_t)(2 * q) * P) + tid;
          const float4* Sq = reinterpret_cast<const float4*>(Sig + (size_t)q * P + (size_t)r0 * n) + tid;
          const float e0 = q == 0 ? 1.f : -1.f;
          for (int b = 0; b < 4; ++b) {
            const float4* Sb =
                reinterpret_cast<const float4*>(Sig + (size_t)(b >> 1) * P + (size_t)r0 * n) + (b & 1) * W4 * NT + tid;
            const float4* wb = reinterpret_cast<const float4*>(wp + (size_t)b * P) + tid;
            float4* Kb = reinterpret_cast<float4*>(reinterpret_cast<float*>(acc) + (size_t)b * P + (size_t)r0 * n) + tid;
            const float eb = b == 0 ? 1.f : -1.f;
            convolve([&](int i, int, int, C2 (&v)[A]) {
#pragma unroll
                       for (int g = 0; g < A / 4; ++g) {
                         const int w = (i * (A / 4) + g) * NT;
                         const float4 sb = Sb[w], wx = wq[w], wy = wq[P / 4 + w];
#pragma unroll
                         for (int t = 0; t < 4; ++t)
                           v[4 * g + t] = mk2(quad_at(wx, t) * quad_at(sb, t), quad_at(wy, t) * quad_at(sb, t));
                       }
                     },
                     [&](int i, int r, int t2) {
                       float4 sx[A / 4], sy[A / 4], wv[A / 4];
#pragma unroll
                       for (int g = 0; g < A / 4; ++g) {
                         const int w = (i * (A / 4) + g) * NT;
                         sx[g] = Sq[w];
                         sy[g] = Sq[W4 * NT + w];
                         wv[g] = wb[w];
                       }
                       C2 v[A];
                       stage_a_inverse(v, r, t2);
                       const uint32_t tvi = tv + 2 * A * i;
#pragma unroll
                       for (int g = 0; g < A / 4; ++g) {
                         float Vx[4] = {}, Vy[4] = {}, k[4];
                         if (b > 0) {
                           tmem_ld(tvi + 4 * g, Vx);
                           tmem_ld(tvi + A + 4 * g, Vy);
                           tmem_wait_ld(Vx);
                           tmem_wait_ld(Vy);
                         }
#pragma unroll
                         for (int t = 0; t < 4; ++t) {
                           const C2 u = v[4 * g + t];
                           k[t] = fmaT(e0 * quad_at(sx[g], t), u.x, -quad_at(sy[g], t) * u.y);
                           const float f = eb * quad_at(wv[g], t);
                           Vx[t] = fmaT(-e0 * f, u.x, Vx[t]);
                           Vy[t] = fmaT(f, u.y, Vy[t]);
                         }
                         float4* kp = Kb + (i * (A / 4) + g) * NT;   // no other thread adds to these points
                         if (k_first) *kp = make_float4(k[0], k[1], k[2], k[3]);
                         else red_add4(kp, k[0], k[1], k[2], k[3]);
                         tmem_st(tvi + 4 * g, Vx);
                         tmem_st(tvi + A + 4 * g, Vy);
                       }
                       tmem_wait_st();               // loaded again after the next convolution
                     });
          }
          k_first = false;
          if (!gr.pair) continue;
          // V_q shifted back: forward rows from the registers into the Xi lines of Gs'
#pragma unroll
          for (int i = 0; i < TA; ++i) {
            const int task = tid + i * NT, r = task / B, t2 = task % B;
            float Vx[A], Vy[A];
            tmem_ld(tv + 2 * A * i, Vx);
            tmem_ld(tv + 2 * A * i + A, Vy);
            tmem_wait_ld(Vx);
            tmem_wait_ld(Vy);
            C2 v[A];
#pragma unroll
            for (int t1 = 0; t1 < A; ++t1) v[t1] = mk2(Vx[t1], Vy[t1]);
            stage_a_forward(v, r, t2);
          }
          __syncthreads();
#pragma unroll
          for (int i = 0; i < TB; ++i) {
            const int task = tid + i * NT;
            if (TB * NT == R * A || task < R * A) {
              const int r = task % R, k1 = task / R;
              C2 b[B];
#pragma unroll
              for (int t = 0; t < B; ++t) b[t] = F[r * LS + B * k1 + t];
              dft<B, -1>(b);
#pragma unroll
              for (int t = 0; t < B; ++t)
                if (xi_t<B>(t)) Gs[(size_t)(B * k1 + t) * n + r0 + r] = b[t];
            }
          }
          cluster_sync_global();                     // the Xi lines are complete
          // forward along x on this CTA's Xi lines, times the conjugate phase
          for (int task = tid; task < XC * B; task += NT) {
            const int cc = task / B, t2 = task % B, ky = xi_line(cc);
            C2 v[A];
#pragma unroll
            for (int t1 = 0; t1 < A; ++t1) v[t1] = __ldcg(&Gs[(size_t)ky * n + B * t1 + t2]);
            dft<A, -1>(v);
#pragma unroll
            for (int k1 = 1; k1 < A; ++k1) v[k1] = cmul(v[k1], twT[k1 * B + t2]);
#pragma unroll
            for (int k1 = 0; k1 < A; ++k1) F[cc * LS + B * k1 + t2] = v[k1];
          }
          __syncthreads();
          const bool first = q == 0 ? s_first0 : s_first1;
          if (q == 0) s_first0 = false;
          else s_first1 = false;
          for (int task = tid; task < XC * A; task += NT) {
            const int cc = task % XC, k1 = task / XC, ky = xi_line(cc), sy = xi_slot<n>(ky);
            C2 b[B];
#pragma unroll
            for (int t = 0; t < B; ++t) b[t] = F[cc * LS + B * k1 + t];
            dft<B, -1>(b);
            if (sy < 0) continue;
            const C2 pyy = py[ky];
#pragma unroll
            for (int t = 0; t < B; ++t)
              if (xi_t<B>(t)) {
                const int sx = xi_slot<n>(B * k1 + t);
                if (sx >= 0) {
                  const C2 z = cmulc(b[t], cmul(px[B * k1 + t], pyy));
                  C2* o = spec + (size_t)q * Q + sx * NQ + sy;
                  *o = first ? z : cadd(*o, z);
                }
              }
          }
          cluster_sync_global();                     // Gs is rewritten by the next convolution
        }
      }
    }
    if constexpr (MODE == 1) {
      for (int e = rank * NT + tid; e < Q; e += kI3Cluster * NT) {
        if (s_first0) spec[e] = zero2<float>();
        if (s_first1) spec[Q + e] = zero2<float>();
      }
    }
  }
  if constexpr (MODE == 1) tmem_free<tmem_columns(NT, 2 * TA * A)>(tm_base);
}

// --------------------------------------------------------------------------
// Sums of the per-unit I3 partials of each cell, in FP64: the np fine-grid values (2 n^2 complex) and
// the nq Fourier-space values (kept frequencies; nq = 0 where the launch wrote none), 16 bytes per
// load.  A block takes 256 / G such words with G threads each, thread g the units u = g mod G, added in
// the order of g.  Bound by HBM (or L2, where the partials still sit there).  It was part of k_assemble,
// whose one block per cell read a single cell's partials alone: at one cell of N = 32, J = M = 32, 1024
// units, 5.2 of the 5.5 ms of that kernel.
// FP32 partials are added as unevaluated sums of three floats, runs of 64 of them in FP64 (FloatSum):
// converting and adding each value in FP64 bound the kernel at a fifth of the memory rate (two FP64 lanes
// per clock), 128 cells of N = 64 1234 us against 248 us.
// sum: [ncells][np] and spec_sum: [ncells][nq] (FP32), or null (FP64): in place into the cell's first unit.
// order_n: padded grid size where the partials' four planes are in thread_order, else 0.
// --------------------------------------------------------------------------
template <class T, int G>
__global__ void __launch_bounds__(256) k_reduce_k3(typename Vec2Of<T>::type* part, double2* sum,
                                                   typename Vec2Of<T>::type* spec, double2* spec_sum, int nparts,
                                                   int np, int nq, int chunks, int order_n) {
  using Word = typename std::conditional<sizeof(T) == 8, double2, float4>::type;
  constexpr int PT = 256 / G, VEC = sizeof(T) == 8 ? 1 : 2;   // complex values per word
  const size_t c = blockIdx.x / chunks;
  const int i = ((blockIdx.x % chunks) * PT + threadIdx.x % PT) * VEC, g = threadIdx.x / PT;
  const bool real_space = i < np;
  Word* src = reinterpret_cast<Word*>(real_space ? part + c * nparts * np + i : spec + c * nparts * nq + (i - np));
  const size_t stride = (size_t)(real_space ? np : nq) / VEC;
  double s[2 * VEC] = {};
  FloatSum a[VEC == 2 ? 4 : 1];   // FP32: the thread's last run
  if (i < np + nq) {
    if constexpr (VEC == 1) {
#pragma unroll 8
      for (int u = g; u < nparts; u += G) {
        const Word v = src[(size_t)u * stride];
        s[0] += v.x;
        s[1] += v.y;
      }
    } else {
      for (int u0 = g; u0 < nparts; u0 += G * FloatSum::kRun) {
        const int u1 = min(nparts, u0 + G * FloatSum::kRun);
        if (u0 > g) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            s[k] += a[k].value();
            a[k] = FloatSum();
          }
        }
#pragma unroll 8
        for (int u = u0; u < u1; u += G) {
          const Word v = src[(size_t)u * stride];
          a[0].add(v.x);
          a[1].add(v.y);
          a[2].add(v.z);
          a[3].add(v.w);
        }
      }
    }
  }
  if constexpr (VEC == 2) {
    // Few values a thread (G > 1): their sums are merged as floats, FP64 additions (24 a thread) would be most of
    // the work.
    const bool merged = G > 1 && nparts <= FloatSum::kMerged;
    if constexpr (G > 1) {
      __shared__ double red[G][2 * VEC][PT + PT / 2];   // doubles, or three floats a value
      float* fl = &reinterpret_cast<float*>(red)[threadIdx.x % PT];
      auto at = [&](int part, int j, int k) -> float& { return fl[((part * G + j) * 4 + k) * PT]; };
      if (merged) {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          at(0, g, k) = a[k].hi;
          at(1, g, k) = a[k].mid;
          at(2, g, k) = a[k].lo;
        }
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) red[g][k][threadIdx.x % PT] = s[k] + a[k].value();
      }
      __syncthreads();
      if (g > 0) return;
      if (merged) {
        for (int j = 1; j < G; ++j)
#pragma unroll
          for (int k = 0; k < 4; ++k) a[k].merge(at(0, j, k), at(1, j, k), at(2, j, k));
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) s[k] = red[0][k][threadIdx.x];
        for (int j = 1; j < G; ++j)
#pragma unroll
          for (int k = 0; k < 4; ++k) s[k] += red[j][k][threadIdx.x];
      }
    }
    if (G == 1 || merged) {
#pragma unroll
      for (int k = 0; k < 4; ++k) s[k] = nparts > G * FloatSum::kRun ? s[k] + a[k].value() : a[k].value();
    }
  } else if constexpr (G > 1) {
    __shared__ double red[G][2 * VEC][PT];
#pragma unroll
    for (int k = 0; k < 2 * VEC; ++k) red[g][k][threadIdx.x % PT] = s[k];
    __syncthreads();
    if (g > 0) return;
    for (int j = 1; j < G; ++j)
#pragma unroll
      for (int k = 0; k < 2 * VEC; ++k) s[k] += red[j][k][threadIdx.x];
  }
  if (i >= np + nq) return;
  if (VEC == 2 && real_space && order_n) {   // thread_order planes (FP32, sum given) into rows
    const int P = order_n * order_n;
    const ThreadWord w = thread_word(order_n, 2 * i % P / 4);
    double* dst = reinterpret_cast<double*>(sum + c * np) + 2 * i / P * P + w.first;
#pragma unroll
    for (int k = 0; k < 2 * VEC; ++k) dst[w.step * k] = s[k];
  } else if (VEC == 2) {
    double2* o = real_space ? sum + c * np + i : spec_sum + c * nq + (i - np);
#pragma unroll
    for (int k = 0; k < VEC; ++k) o[k] = mk2(s[2 * k], s[2 * k + 1]);
  } else {
    T* o = reinterpret_cast<T*>(src);
#pragma unroll
    for (int k = 0; k < 2 * VEC; ++k) o[k] = (T)s[k];
  }
}

// One thread per word where that gives a thousand threads per SM, eight otherwise: short columns of loads,
// more of them in flight.  The order of a sum depends on it, so the line goes by the cells nb that the
// workspace holds (the allocation-free entry, which has none of its own: one), as the chunks do: one handle
// gives a cell the same bits in a call of one cell and of all.
template <class T>
void reduce_partials(typename Vec2Of<T>::type* part, double2* sum, typename Vec2Of<T>::type* spec,
                     double2* spec_sum, int nparts, int np, int nq, int nb, int ncells, int order_n, cudaStream_t s) {
  constexpr int VEC = sizeof(T) == 8 ? 1 : 2;
  const int words = (np + nq) / VEC;
  if (nparts >= 16 && (long long)words * nb < 152 * 1024) {
    const int chunks = (words + 31) / 32;
    k_reduce_k3<T, 8><<<(unsigned)chunks * ncells, 256, 0, s>>>(part, sum, spec, spec_sum, nparts, np, nq,
                                                                chunks, order_n);
  } else {
    const int chunks = (words + 255) / 256;
    k_reduce_k3<T, 1><<<(unsigned)chunks * ncells, 256, 0, s>>>(part, sum, spec, spec_sum, nparts, np, nq,
                                                                chunks, order_n);
  }
}

// Real-space D pairs and K4 pairs of each cell (inverse 2-D transforms), DK[c][4][P]: one team per cell
// and pair.
template <int n, class T, int CB>
__global__ void __launch_bounds__(kThreads, (cell_min_blocks<n, T, CB>()))
    k_dk_fields(const typename Vec2Of<T>::type* Dacc, const typename Vec2Of<T>::type* K4acc,
                typename Vec2Of<T>::type* DK, const typename Vec2Of<T>::type* __restrict__ gtw) {
  using C2 = typename Vec2Of<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* tw = reinterpret_cast<C2*>(smem_raw);
  C2* sm = tw + n;
  load_twiddles<n>(tw, gtw);
  constexpr int P = n * n;
  const int c = cluster_index() >> 2, f = cluster_index() & 3;
  const C2* in = (f < 2) ? (Dacc + ((size_t)c * 2 + f) * P) : (K4acc + ((size_t)c * 2 + (f - 2)) * P);
  C2* out = DK + (size_t)cluster_index() * P;
  col_pass<n, 1, false, 0, CB>(
      sm, tw, [&](int ix, int iy) { return in[ix * n + iy]; }, NoMid(),
      [&](int ix, int iy, C2 v) { out[ix * n + iy] = v; });
  row_pass<n, 1, false, 0, CB>(
      sm, tw, [&](int ix, int iy) { return ldc<n, CB>(&out[ix * n + iy]); }, NoMid(),
      [&](int ix, int iy, C2 v) { out[ix * n + iy] = v; });
}

// --------------------------------------------------------------------------
// Assemble C on the fine grid from D, K2, K3, K4 (Pauli formulas of Sec. 3.1),
// then FFT, cut to Xi (without the -N/2 line), inverse FFT and sample the
// coarse nodes.  One team per cell and pair (C_0, C_1) or (C_2, C_3); the pointwise
// formulas are evaluated on the load of the first pass, and after it only the Xi
// columns and the even rows are transformed.  k3: the reduced K3 of a cell (FP64),
// k3_stride apart; spec (null after a node-by-node kernel): their Fourier-space parts (FP64),
// added to the spectrum of C inside the projection (C_0 holds -2 pi K3_0 and C_c holds
// +2 pi K3raw_c; the sign of component 0 is already in spec).
// --------------------------------------------------------------------------
template <int n, class T, int CB>
__global__ void __launch_bounds__(kThreads, (cell_min_blocks<n, T, CB>()))
    k_assemble(const typename Vec2Of<T>::type* wfine, const typename Vec2Of<T>::type* DK, const T* K2acc,
               const double2* k3, size_t k3_stride, const double2* spec, size_t spec_stride,
               typename Vec2Of<T>::type* ws, const typename Vec2Of<T>::type* __restrict__ gtw, double* cout) {
  using C2 = typename Vec2Of<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* tw = reinterpret_cast<C2*>(smem_raw);
  C2* sm = tw + n;
  load_twiddles<n>(tw, gtw);
  constexpr int N = n / 2, P = n * n, NQ = xi_kept<n>(), Q = NQ * NQ, B = Split<n>::B;
  const int c = cluster_index() >> 1, p = cluster_index() & 1;
  C2* H = ws + (size_t)cluster_index() * P;
  const C2* dk = DK + (size_t)c * 4 * P;
  const double2* k3c = k3 + c * k3_stride;
  const double* k3r = reinterpret_cast<const double*>(k3c);
  const C2* wf0 = wfine + (size_t)c * 2 * P;
  const C2* wf1 = wf0 + P;
  const T* K2 = K2acc + (size_t)c * P;
  const double tp = 2.0 * kPi;
  const T invP = (T)(1.0 / (double)P);
  double* co = cout + (size_t)c * 4 * N * N;
  const double2* Hs = spec ? spec + c * spec_stride + (size_t)p * Q : nullptr;
  row_pass<n, -1, false, 0, CB>(
      sm, tw,
      [&](int ix, int iy) {
        const int i = ix * n + iy;
        // node-by-node kernels: pairs (K3_0, K3_1), (K3_2, K3_3); kernels in pairs: four planes
        const double2 k3p = spec ? mk2(k3r[2 * p * P + i], k3r[(2 * p + 1) * P + i]) : k3c[p * P + i];
        const double w0 = wf0[i].x, w1 = wf0[i].y, w2 = wf1[i].x, w3 = wf1[i].y;
        const C2 s0 = dk[i], s1 = dk[P + i], s2 = dk[2 * P + i], s3 = dk[3 * P + i];
        const double D1 = s0.x, D2 = s0.y, D3 = s1.x;
        const double K40 = s2.x, K41 = -(double)s2.y;   // eta_b applied
        const double K42 = -(double)s3.x, K43 = -(double)s3.y;
        const double k2 = K2[i];
        if (p == 0) {
          const double K30 = k3p.x, K31 = -k3p.y;
          const double C0 = tp * (k2 * (1.0 - w0) - K30 + w0 * K40 + w1 * K41 + w2 * K42 + w3 * K43);
          const double C1 = -2.0 * (D2 * w3 - D3 * w2) + tp * (-k2 * w1 - K31 + w0 * K41 + K40 * w1);
          return mk2((T)C0, (T)C1);
        }
        const double K32 = -k3p.x, K33 = -k3p.y;
        const double C2v = -2.0 * (D3 * w1 - D1 * w3) + tp * (-k2 * w2 - K32 + w0 * K42 + K40 * w2);
        const double C3 = -2.0 * (D1 * w2 - D2 * w1) + tp * (-k2 * w3 - K33 + w0 * K43 + K40 * w3);
        return mk2((T)C2v, (T)C3);
      },
      NoMid(),
      [&](int ix, int iy, C2 v) {
        if (xi_t<B>(iy % B)) H[ix * n + iy] = v;
      });
  xi_col_filter<n, true, true, CB>(
      sm, tw, [&](int ix, int iy) { return ldc<n, CB>(&H[ix * n + iy]); },
      [&](int ix, int iy, C2 v) {
        const int sx = xi_slot<n>(ix), sy = xi_slot<n>(iy);
        if (sx < 0 || sy < 0) return zero2<T>();
        if (Hs) {
          const double2 h = Hs[sx * NQ + sy];
          v = mk2((T)fma(tp, h.x, (double)v.x), (T)fma(tp, h.y, (double)v.y));
        }
        return cscale(v, invP);
      },
      [&](int ix, int iy, C2 v) {
        if (!(ix & 1)) H[ix * n + iy] = v;
      });
  even_row_pass<n, 1, CB, true>(
      sm, tw, [&](int ix, int iy) { return xi_t<B>(iy % B) ? ldc<n, CB>(&H[ix * n + iy]) : zero2<T>(); },
      [&](int ix, int iy, C2 v) {
        if (!(iy & 1)) {
          const int i = ix >> 1, j = iy >> 1;
          co[((2 * p) * N + i) * N + j] = (double)v.x;
          co[((2 * p + 1) * N + i) * N + j] = (double)v.y;
        }
      });
}

}  // namespace

template <int n, class T, int CB>
size_t cell_smem_bytes() {
  using C2 = typename Vec2Of<T>::type;
  return (size_t)(n + Chunk<n, sizeof(C2), CB>::SMEM_ELEMS) * sizeof(C2);
}
// Blocks per team of a per-cell kernel over `teams` teams: 1, 2, 4 or 8, the most that stay within three
// blocks per SM, or one where that is fewer than `least`.  The FP64 passes of one cell keep one SM's FP64 unit
// (two lanes per clock) busy while the others idle, the FP32 ones wait for its latency.  One cell, N = 32 FP64,
// per C[W]: k_prep 279 -> 31 us, I1 and I2/I4 817 -> 283 us; two steps of it 18.8 -> 14.7 ms.
inline int cell_team(int teams, int least) {
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  int size = 1;
  while (size < 8 && 2LL * size * teams <= 3LL * nsm) size *= 2;
  return size < least ? 1 : size;
}
// The smallest team worth its cluster barriers.  A team's chunk is n / 8 lines, so a block of a team of s runs
// 8 / s chunks per pass, one after the other, where a block alone runs one or two larger ones.  Measured (ncu,
// one / two / four / eight blocks, us; 50, 100 and 200 teams take 8, 4 and 2): n = 16 k_i24_vjp, FP32, 50:
// 28/165/99/67; n = 32, FP32, 50: 46/161/100/72, FP64, 50: 293/757/400/225, 100: 292/766/409/445; n = 64, FP32,
// 100: 159/266/162/219, 200: 199/289/348/326, FP64, 200: 2353/1875/1883/1942; n = 96, FP32, 200:
// 632/543/536/503.  k_assemble (ASSEMBLE) gains earlier in FP32, by its formulas in FP64: n = 32, 50: 16/22/16/12;
// n = 64, 200: 96/71/62/58.
template <int n, class T, bool ASSEMBLE>
constexpr int least_team() {
  constexpr bool fp32 = std::is_same<T, float>::value && !ASSEMBLE;
  return n == 16 ? 16 : n == 32 ? (fp32 ? 16 : 8) : n == 64 ? (fp32 ? 4 : 2) : 2;
}
// Launches a per-cell kernel over `teams` teams: `one` with a block each, `several` with a cluster each.
template <class... K, class... Args>
cudaError_t launch_cells(void (*one)(K...), void (*several)(K...), int least, int teams, size_t smem_one,
                         size_t smem_several, cudaStream_t s, Args... args) {
  const int size = cell_team(teams, least);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)teams * size);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = size == 1 ? smem_one : smem_several;
  cfg.stream = s;
  cudaLaunchAttribute attr = {};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = size;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = size == 1 ? 0 : 1;
  return cudaLaunchKernelEx(&cfg, size == 1 ? one : several, static_cast<K>(args)...);
}
#define QBE_TEAM_CB team_cb<n, typename Vec2Of<T>::type>()
#define QBE_CELLS_OF(assemble, kernel, teams, s, ...)                                                       \
  launch_cells(kernel<n, T, kCellCB>, kernel<n, T, QBE_TEAM_CB>, least_team<n, T, assemble>(), teams,       \
               cell_smem_bytes<n, T, kCellCB>(), cell_smem_bytes<n, T, QBE_TEAM_CB>(), s, __VA_ARGS__)
#define QBE_CELLS(kernel, teams, s, ...) QBE_CELLS_OF(false, kernel, teams, s, __VA_ARGS__)
#define QBE_CELLS_SMEM(kernel)                                                                              \
  cudaFuncSetAttribute(kernel<n, T, kCellCB>, cudaFuncAttributeMaxDynamicSharedMemorySize,                  \
                       (int)cell_smem_bytes<n, T, kCellCB>());                                              \
  cudaFuncSetAttribute(kernel<n, T, QBE_TEAM_CB>, cudaFuncAttributeMaxDynamicSharedMemorySize,              \
                       (int)cell_smem_bytes<n, T, QBE_TEAM_CB>())

template <int n, class T, int CB>
size_t i3_staged_smem_bytes() {
  using C2 = typename Vec2Of<T>::type;
  return (size_t)(n + Chunk<n, sizeof(C2), CB>::SMEM_ELEMS) * sizeof(C2);
}

// Launch variants of the I3 kernel for padded size n and transform type T: the shapes the
// autotuner chooses among (i3_default_variant gives the one a new handle starts with).
//   FP64 (every size): the staged kernel, node by node, as (threads, chunk bytes, blocks per SM)
//     0: (256, 64 KB, 3)   1: (128, 32 KB, 6);  k_i3_sf, nodes in pairs, 2: (256, 64 KB, 3)
//     3: (128, 32 KB, 6).  Variant 0 also serves the allocation-free entry point, whose static array
//     has no room for the pairs' Fourier-space partials at the sizes it accepts.
//   FP32, n = 64, 96, 128: 0, 1, 2: the fused shared-memory kernel in the FusedShapes<n> shapes
//     (0 at n = 64: k_i3_tmem), 3: k_i3_smem (1024 threads, element passes through shared memory; at
//     n = 96 k_i3_lines), 4 (n = 128): k_i3_tmem
//   FP32, n = 32: k_i3_tmem;  n = 16: k_i3_smem;  FP32, n > 128: the cluster kernel, 0: 1024 threads per CTA with a
//     partial-sum update per convolution, 1: two row tasks per thread, node pairs, sums in tensor memory.
struct I3Launch {
  const void* fn = nullptr;
  int threads = 0;
  size_t smem = 0;
  bool cluster = false;
  const char* name = "";
  int teams = 1;   // units a block works on at a time
};

template <int n>
I3Launch i3_tmem_launch() {
  using S = TmShape<n>;
  return {(const void*)k_i3_tmem<n>, S::NT, S::smem, false,
          n == 128 ? "node pairs, tensor-memory exchanges, one team of 512 threads per block"
          : n == 64 ? "node pairs, tensor-memory exchanges, four teams of 128 threads per block"
                    : "node pairs, a warp per unit, sixteen per block", S::TEAMS};
}

template <int n, class T>
constexpr int i3_nvariants() {
  if constexpr (std::is_same<T, float>::value) {
    if constexpr (use_i3_cluster<n>()) return 2;
    else if constexpr (use_i3_fused<n>()) return n == 128 ? 5 : 4;   // 128 points: + k_i3_tmem
    else return 1;
  } else {
    return 4;
  }
}

// Whether a variant's partials are planes in thread_order (k_i3_tmem, k_i3_lines, k_i3_cluster in pairs).
template <int n, class T>
constexpr bool i3_variant_thread_order(int v) {
  return std::is_same<T, float>::value &&
         (n == 32 || (n == 64 && v == 0) || (n == 96 && v == 3) || (n == 128 && v == 4) || (use_i3_cluster<n>() && v == 1));
}

template <int n, class T>
I3Launch i3_variant(int v) {
  I3Launch l;
  if constexpr (std::is_same<T, float>::value && use_i3_cluster<n>()) {
    constexpr int NT1 = i3_cluster_threads<n>(1);
    if (v == 1)
      l = {(const void*)k_i3_cluster<n, NT1, 1>, NT1, i3_cluster_smem_bytes<n>(), true,
           n == 256 ? "node pairs, cluster of 4 CTAs x 512 threads, sums in tensor memory"
                    : "node pairs, cluster of 4 CTAs x 384 threads, sums in tensor memory"};
    else
      l = {(const void*)k_i3_cluster<n, kThreadsI3Cluster, 0>, kThreadsI3Cluster, i3_cluster_smem_bytes<n>(), true,
           "cluster of 4 CTAs x 1024 threads"};
  } else if constexpr (std::is_same<T, float>::value && use_i3_fused<n>()) {
    using S = FusedShapes<n>;
    constexpr const char* names[3] = {"fused, per-convolution partial sums", "fused, register accumulation",
                                      "fused, paired w with register accumulation"};
    if (v == 0) {
      if constexpr (n == 64) l = i3_tmem_launch<n>();
      else l = {(const void*)k_i3_fused<n, S::T0, S::B0, S::M0>, S::T0, i3_fused_smem_bytes<n>(), false, names[S::M0]};
    } else if (v == 1)
      l = {(const void*)k_i3_fused<n, S::T1, S::B1, S::M1>, S::T1, i3_fused_smem_bytes<n>(), false, names[S::M1]};
    else if (v == 2)
      l = {(const void*)k_i3_fused<n, S::T2, S::B2, S::M2>, S::T2, i3_fused_smem_bytes<n>(), false, names[S::M2]};
    else if constexpr (n == 96) {
      using L = LineShape<n>;
      l = {(const void*)k_i3_lines<n>, L::NT, L::smem, false, "node pairs, shared-memory, two teams of 384 threads per block",
           L::TEAMS};
    } else
      l = {(const void*)k_i3_smem<n>, kThreadsI3Smem, i3_smem_bytes<n>(), false, "node pairs, shared-memory, 1024 threads"};
    if constexpr (n == 128) {
      if (v == 4) l = i3_tmem_launch<n>();
    }
  } else if constexpr (std::is_same<T, float>::value && n == 32) {
    l = i3_tmem_launch<n>();
  } else if constexpr (std::is_same<T, float>::value) {
    l = {(const void*)k_i3_smem<n>, kThreadsI3Smem, i3_smem_bytes<n>(), false, "node pairs, shared-memory, 1024 threads"};
  } else {
    if (v == 1)
      l = {(const void*)k_i3<n, T, 128, 32768, 6>, 128, i3_staged_smem_bytes<n, T, 32768>(), false,
           "staged, 128 threads, 32 KB chunks"};
    else if (v == 2)
      l = {(const void*)k_i3_sf<n, T, 256, 65536, 3>, 256, i3_sf_smem_bytes<n, T, 65536>(), false,
           "staged with fused loads and stores, 256 threads, 64 KB chunks"};
    else if (v == 3)
      l = {(const void*)k_i3_sf<n, T, 128, 32768, 6>, 128, i3_sf_smem_bytes<n, T, 32768>(), false,
           "staged with fused loads and stores, 128 threads, 32 KB chunks"};
    else
      l = {(const void*)k_i3<n, T, 256, 65536, 3>, 256, i3_staged_smem_bytes<n, T, 65536>(), false,
           "staged, 256 threads, 64 KB chunks"};
  }
  return l;
}

template <int n, class T>
void set_smem_attributes() {
  static unsigned long long done = 0;
  if (!first_on_device(done)) return;
  QBE_CELLS_SMEM(k_prep);
  QBE_CELLS_SMEM(k_i124);
  QBE_CELLS_SMEM(k_dk_fields);
  QBE_CELLS_SMEM(k_assemble);
  for (int v = 0; v < i3_nvariants<n, T>(); ++v) {
    const I3Launch l = i3_variant<n, T>(v);
    cudaFuncSetAttribute(l.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)l.smem);
  }
}

// Clusters of the cluster variant v of k_i3_cluster<n> that can be resident at once on the current
// device (cached per device and variant).
template <int n>
int i3_max_clusters(int v) {
  static int cached[64][2] = {};
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  v = (v == 1) ? 1 : 0;
  if (cached[dev & 63][v] > 0) return cached[dev & 63][v];
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const I3Launch l = i3_variant<n, float>(v);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kI3Cluster * (nsm > 0 ? nsm : 1));
  cfg.blockDim = dim3(l.threads);
  cfg.dynamicSmemBytes = l.smem;
  int ncl = 0;
  if (cudaOccupancyMaxActiveClusters(&ncl, l.fn, &cfg) != cudaSuccess || ncl < 1) {
    cudaGetLastError();
    ncl = (nsm > 0 ? nsm : 1) / kI3Cluster;
  }
  cached[dev & 63][v] = ncl < 1 ? 1 : ncl;
  return cached[dev & 63][v];
}

// Resident blocks per SM of an I3 variant (at least 1).
template <int n, class T>
int i3_blocks_per_sm(int v) {
  set_smem_attributes<n, T>();
  if (v < 0 || v >= i3_nvariants<n, T>()) v = 0;
  const I3Launch l = i3_variant<n, T>(v);
  int b = 0;
  if constexpr (std::is_same<T, float>::value && use_i3_cluster<n>()) {
    int dev = 0, nsm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    b = (i3_max_clusters<n>(v) * kI3Cluster + nsm - 1) / (nsm > 0 ? nsm : 1);
  } else if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, l.fn, l.threads, l.smem) != cudaSuccess) {
    cudaGetLastError();
    b = 1;
  }
  return b < 1 ? 1 : b;
}

template <int n, class T>
int i3_variant_count() {
  return i3_nvariants<n, T>();
}

// The variant a new handle starts with (the fastest measured on a GB300 for this size).  FP64, I3
// launch in ms for variants 0..3 (J = M = 32; 0 and 1 node by node, 2 and 3 in pairs): N = 16, 128
// cells 135.5 135.1 76.9 77.1; N = 32, 128 cells 646.9 635.0 365.3 371.5; N = 48, 64 cells 861.7 879.5
// 486.7 499.6; N = 64, 32 cells 746.4 755.8 423.6 433.1; N = 128, 8 cells 926.8 935.8 521.0 533.0 (the
// fused line stages node by node: 132.9, 625.3, 860.3, 732.5, 885.5 for variant 2).
// FP32 cluster kernel (I3 launch, J = M = 32): N = 128, 32 cells 216.2 ms (variant 0, node by node),
// 132.4 ms (variant 1, in pairs; 192.4 node by node); N = 96, 64 cells 217.1 and 141.7 (208.9) ms.
template <int n, class T>
int i3_default_variant() {
  if constexpr (std::is_same<T, float>::value && use_i3_fused<n>()) return FusedShapes<n>::DEFAULT;
  else if constexpr (std::is_same<T, float>::value && use_i3_cluster<n>()) return 1;
  else if constexpr (std::is_same<T, double>::value) return 2;
  else return 0;
}

// Work units (or, for the cluster form, clusters) a launch of variant v with `grid` blocks and
// `total` units processes at once: the persistent grid the launcher uses (see i3_group_n).  Unit u
// goes to block (cluster) u mod this number.
template <int n, class T>
int i3_variant_concurrency(int v, int grid, int total) {
  if (v < 0 || v >= i3_nvariants<n, T>()) v = 0;
  int g = total < grid ? total : grid;
  if constexpr (std::is_same<T, float>::value && use_i3_cluster<n>()) {
    int ncl = grid / kI3Cluster;
    const int cmax = i3_max_clusters<n>(v);
    if (ncl > cmax) ncl = cmax;
    if (ncl > total) ncl = total;
    g = ncl < 1 ? 1 : ncl;
  } else {
    int dev = 0, nsm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int gmax = nsm * i3_blocks_per_sm<n, T>(v);
    if (g > gmax) g = gmax;
    g *= i3_variant<n, T>(v).teams;
  }
  return g < 1 ? 1 : g;
}

// Variants that take the radial nodes in pairs (Fourier-space partials beside the real-space ones).
template <int n, class T>
bool i3_variant_paired(int v) {
  if constexpr (std::is_same<T, double>::value) return v >= 2;
  else if constexpr (n > 128) return v == 1;
  else return n <= 32 || v == 3 || v == (n == 128 ? 4 : n == 64 ? 0 : 3);
}

template <int n, class T>
const char* i3_variant_name(int v) {
  if (v < 0 || v >= i3_nvariants<n, T>()) return nullptr;
  return i3_variant<n, T>(v).name;
}

// I1 and I2/I4 of ncells cells (k_i124), then its partials summed into Dacc, K2acc, K4acc.  One launch
// for both kinds; two where they are timed apart, or share their scratch (the workspace without K2part
// has six fields per cell, and keeps the K2 planes in the coefficients that only I1 reads).
template <int n, class T>
cudaError_t per_cell_terms(const Tables& t, CollisionWork& cw, typename Vec2Of<T>::type* ws, int ncells,
                           cudaStream_t s, long long& launches, KernelTimer* tm) {
  using C2 = typename Vec2Of<T>::type;
  constexpr size_t P = (size_t)n * n;
  const TabPtrs<T> tb = tab_ptrs<T>(t);
  const int nch = cw.nch < 1 ? 1 : cw.nch;
  const bool own_k2 = cw.K2part != nullptr;
  CellTerms<n, T> a;
  a.what = (const C2*)cw.what;
  a.wfine = (const C2*)cw.wfine;
  a.D = (C2*)(nch > 1 ? cw.Dpart : cw.Dacc);
  a.K4 = (C2*)(nch > 1 ? cw.K4part : cw.K4acc);
  a.K2 = own_k2 ? (T*)cw.K2part : (T*)((C2*)cw.what + 2 * P);
  a.k2_cell = own_k2 ? 2 * (size_t)nch * P : 8 * P;
  a.tw = tb.tw;
  a.phip = tb.phip;
  a.Ktab = tb.Ktab;
  a.psi = tb.psi;
  a.J = t.J;
  a.nch = nch;
  a.teams1 = 2 * ncells * nch;
  a.first = 0;
  a.ws1 = ws;
  a.ws24 = own_k2 ? ws + a.teams1 * P : ws;
  const bool apart = !own_k2 || (tm && tm->on);
  if (tm && apart) tm->begin(KG_I1, s);
  cudaError_t e = QBE_CELLS(k_i124, apart ? a.teams1 : 2 * a.teams1, s, a);
  if (e != cudaSuccess) return e;
  if (tm && apart) tm->end(s);
  if (apart) {
    a.first = a.teams1;
    if (tm) tm->begin(KG_I24, s);
    e = QBE_CELLS(k_i124, a.teams1, s, a);
    if (e != cudaSuccess) return e;
    ++launches;
  }
  k_reduce_chunks<T><<<element_blocks((size_t)ncells * (nch > 1 ? 9 : 1) * P), kThreads, 0, s>>>(
      (const T*)a.D, a.K2, (const T*)a.K4, (T*)cw.Dacc, (T*)cw.K2acc, (T*)cw.K4acc, nch, ncells, P, a.k2_cell);
  if (tm && apart) tm->end(s);
  launches += 2;
  return cudaGetLastError();
}

// The collision operator in three parts: the per-cell terms before I3 (prep, I1, I2/I4), the I3
// launch (a work queue over the units of one or several simulations of the same padded size), and
// the per-cell assembly.  collide_batch_n runs all three for one simulation.
template <int n, class T>
cudaError_t collide_pre_n(const Tables& t, CollisionWork& cw, const double* w, int ncells, cudaStream_t s,
                          long long& launches, KernelTimer* tm) {
  using C2 = typename Vec2Of<T>::type;
  set_smem_attributes<n, T>();
  const TabPtrs<T> tb = tab_ptrs<T>(t);
  C2* what = (C2*)cw.what;
  C2* wfine = (C2*)cw.wfine;
  C2* ws = (C2*)cw.ws;
  auto begin = [&](int g) { if (tm) tm->begin(g, s); };
  auto end = [&]() { if (tm) tm->end(s); };
  begin(KG_PREP);
  cudaError_t e = QBE_CELLS(k_prep, 4 * ncells, s, w, what, wfine, (T*)cw.wplane, ws, tb.tw);
  end();
  if (e != cudaSuccess) return e;
  e = per_cell_terms<n, T>(t, cw, ws, ncells, s, launches, tm);
  if (e != cudaSuccess) return e;
  ++launches;
  return cudaGetLastError();
}

template <int n, class T>
I3Job<T> i3_job(const Tables& t, const CollisionWork& cw, int ncells, int unit_begin) {
  using C2 = typename Vec2Of<T>::type;
  const TabPtrs<T> tb = tab_ptrs<T>(t);
  I3Job<T> jb;
  jb.what = (const C2*)cw.what;
  jb.wfine = (const C2*)cw.wfine;
  jb.wplane = (const T*)cw.wplane;
  jb.K3part = (C2*)cw.K3part;
  jb.K3spec = (C2*)cw.K3spec;
  jb.psip_s = tb.psip_s;
  jb.phase = tb.phase;
  jb.J = t.J;
  jb.M = t.M;
  jb.nmc = cw.nmc;
  jb.unit_begin = unit_begin;
  jb.nunits = ncells * t.J * cw.nmc;
  return jb;
}

// I3 over the units of njobs simulations (same n and precision, njobs <= kMaxI3Jobs); ws must hold
// i3_fields (2N)^2 complex values for each of `grid` blocks (the cluster form uses one such slot per
// cluster of kI3Cluster blocks).
template <int n, class T>
cudaError_t i3_group_n(const Tables* const* tabs, const CollisionWork* const* cws, const int* ncells, int njobs,
                       void* ws, int grid, cudaStream_t s, long long& launches, int max_units) {
  using C2 = typename Vec2Of<T>::type;
  if (njobs < 1 || njobs > kMaxI3Jobs) return cudaErrorInvalidValue;
  set_smem_attributes<n, T>();
  I3Jobs<T> jobs;
  jobs.njobs = njobs;
  int total = 0;
  for (int k = 0; k < njobs; ++k) {
    jobs.job[k] = i3_job<n, T>(*tabs[k], *cws[k], ncells[k], total);
    total += jobs.job[k].nunits;
  }
  jobs.total = (max_units > 0 && max_units < total) ? max_units : total;   // a prefix (autotuner samples)
  total = jobs.total;
  if (total == 0) return cudaSuccess;
  const TabPtrs<T> tb = tab_ptrs<T>(*tabs[0]);
  int v = cws[0]->i3_variant;
  if (v < 0 || v >= i3_nvariants<n, T>()) v = 0;
  const bool paired = i3_variant_paired<n, T>(v);
  for (int k = 0; k < njobs; ++k) {
    if (paired && !cws[k]->K3spec) return cudaErrorInvalidValue;
    cws[k]->i3_paired = paired;
    cws[k]->i3_thread_order = i3_variant_thread_order<n, T>(v);
  }
  const I3Launch l = i3_variant<n, T>(v);
  int g = total < grid ? total : grid;
  if constexpr (std::is_same<T, float>::value && use_i3_cluster<n>()) {
    int ncl = grid / kI3Cluster;
    const int cmax = i3_max_clusters<n>(v);
    if (ncl > cmax) ncl = cmax;
    if (ncl > total) ncl = total;
    if (ncl < 1) ncl = 1;
    g = ncl * kI3Cluster;
  } else {
    int dev = 0, nsm = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const int gmax = nsm * i3_blocks_per_sm<n, T>(v);      // persistent: never more than fit at once
    if (g > gmax) g = gmax;
  }
  C2* wsp = (C2*)ws;
  const C2* twp = tb.tw;
  void* args[] = {(void*)&jobs, (void*)&wsp, (void*)&twp};
  cudaError_t e = cudaLaunchKernel(l.fn, dim3(g), dim3(l.threads), args, l.smem, s);
  ++launches;
  return e != cudaSuccess ? e : cudaGetLastError();
}

template <int n, class T>
cudaError_t collide_post_n(const Tables& t, CollisionWork& cw, double* c, int ncells, cudaStream_t s,
                           long long& launches, KernelTimer* tm) {
  using C2 = typename Vec2Of<T>::type;
  set_smem_attributes<n, T>();
  const TabPtrs<T> tb = tab_ptrs<T>(t);
  if (tm) tm->begin(KG_ASSEMBLE, s);
  constexpr int np = 2 * n * n;
  constexpr int nq = 2 * xi_kept<n>() * xi_kept<n>();
  const int nparts = t.J * cw.nmc, nqp = cw.i3_paired ? nq : 0;
  C2* part_s = cw.i3_paired ? (C2*)cw.K3spec : nullptr;
  reduce_partials<T>((C2*)cw.K3part, cw.K3sum, part_s, cw.K3ssum, nparts, np, nqp, cw.order_nb, ncells,
                     cw.i3_thread_order ? n : 0, s);
  const double2* spec = !cw.i3_paired ? nullptr : cw.K3ssum ? cw.K3ssum : (const double2*)cw.K3spec;
  const double2* k3 = cw.K3sum ? cw.K3sum : (const double2*)cw.K3part;
  C2* DK = (C2*)cw.ws;   // [ncells][4][P], then a field per (cell, pair)
  cudaError_t e = QBE_CELLS(k_dk_fields, 4 * ncells, s, (C2*)cw.Dacc, (C2*)cw.K4acc, DK, tb.tw);
  if (e != cudaSuccess) return e;
  e = QBE_CELLS_OF(true, k_assemble, 2 * ncells, s, (C2*)cw.wfine, DK, (T*)cw.K2acc, k3,
                cw.K3sum ? (size_t)np : (size_t)nparts * np, spec, cw.K3ssum ? (size_t)nq : (size_t)nparts * nq,
                DK + (size_t)ncells * 4 * n * n, tb.tw, c);
  if (tm) tm->end(s);
  if (e != cudaSuccess) return e;
  launches += 3;
  return cudaGetLastError();
}

template <int n, class T>
cudaError_t collide_batch_n(const Tables& t, CollisionWork& cw, const double* w, double* c, int ncells,
                            cudaStream_t s, long long& launches, KernelTimer* tm) {
  cudaError_t e = collide_pre_n<n, T>(t, cw, w, ncells, s, launches, tm);
  if (e != cudaSuccess) return e;
  const Tables* tp = &t;
  const CollisionWork* cp = &cw;
  if (tm) tm->begin(KG_I3, s);
  e = i3_group_n<n, T>(&tp, &cp, &ncells, 1, cw.ws, cw.grid_i3, s, launches, 0);
  if (tm) tm->end(s);
  if (e != cudaSuccess) return e;
  return collide_post_n<n, T>(t, cw, c, ncells, s, launches, tm);
}

}  // namespace qbe
