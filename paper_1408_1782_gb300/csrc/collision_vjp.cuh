// Vector-Jacobian product of the discrete collision operator: given a
// cotangent lambda of C[W] on the velocity grid, the gradient of <lambda, C[W]>
// with respect to W.  Used by the adjoint of the split time step.
//
// Every dependence of C on W goes through the fine-grid interpolant w^fine
// = I(W) (band-limited to Xi), so the kernels accumulate a fine-grid cotangent
// nu_a of each Pauli component and finish with I^T nu = 4 E P nu (band-limit
// to Xi, sample the coarse nodes; E samples the even fine nodes).  The
// transposes used, all exact for the discrete operators:
//   * a Fourier multiplier m(sigma) transposes to m(-sigma): even real
//     multipliers (psi, psi') are self-adjoint; odd ones are handled as the
//     real operators "multiply by i phi'" and "multiply by i K", which are
//     antisymmetric;
//   * the Hu-Ying shift S (multiplier e^{i alpha.sigma}) transposes to the
//     shift back (conjugate phase);
//   * the projection of C_fine to Xi is self-adjoint; sampling transposes to
//     zero interleaving.
// With lambda band-limited by that projection, the only frequency at which
// these statements need care (the unpaired -N line of the padded grid) never
// reaches Xi.  Terms (as in the forward kernels, raw accumulators):
//   D_b = -K'(f A_{j'} w_b),   K2 = 2 (pi/J) sum eta_a F_{a,j} F_{a,j+J/2},
//   K4raw_b = (pi/J) sum_j Psi_j(f F_{b,j+J/2}),
//   K3raw_b = sum_{j,m,a} eta_a S(w_a) Psi'_j(w_a S(w_b)),   f = 2 w0 - 1.
#pragma once

#include "collision_kernels.cuh"

namespace qbe {

namespace {

template <class C2>
__device__ __forceinline__ C2 mul_i(C2 v, typename RealOf<C2>::type s) {   // v * (i s)
  return mk2(-s * v.y, s * v.x);
}

// --------------------------------------------------------------------------
// mu = P(E^T lambda) on the fine grid: MU[c][2] (pairs (0,1), (2,3)) and muh[c][2], 2 pi times the Xi
// coefficients of the pairs mu_0 + i mu_1, mu_2 + i mu_3 (outside Xi not stored).  One team per cell and
// pair.
// --------------------------------------------------------------------------
template <int n, class T, int CB>
__global__ void __launch_bounds__(kThreads, (cell_min_blocks<n, T, CB>()))
    k_vjp_mu(const double* __restrict__ lam, typename Vec2Of<T>::type* MU, typename Vec2Of<T>::type* muh,
             const typename Vec2Of<T>::type* __restrict__ gtw) {
  using C2 = typename Vec2Of<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* tw = reinterpret_cast<C2*>(smem_raw);
  C2* sm = tw + n;
  load_twiddles<n>(tw, gtw);
  constexpr int N = n / 2, P = n * n, B = Split<n>::B;
  const int c = cluster_index() >> 1, p = cluster_index() & 1;
  C2* M = MU + (size_t)cluster_index() * P;
  C2* muhp = muh + (size_t)cluster_index() * P;
  const double* lc = lam + (size_t)c * 4 * N * N;
  const T invP = (T)(1.0 / (double)P);
  even_row_pass<n, -1, CB>(
      sm, tw,
      [&](int ix, int iy) {
        if (iy & 1) return zero2<T>();
        const int i = ix >> 1, j = iy >> 1;
        return mk2((T)lc[((2 * p) * N + i) * N + j], (T)lc[((2 * p + 1) * N + i) * N + j]);
      },
      [&](int ix, int iy, C2 v) {
        if (xi_t<B>(iy % B)) M[ix * n + iy] = v;
      });
  xi_col_filter<n, true, true, CB>(
      sm, tw, [&](int ix, int iy) { return (ix & 1) ? zero2<T>() : ldc<n, CB>(&M[ix * n + iy]); },
      [&](int ix, int iy, C2 v) {
        const bool keep = xi_slot<n>(ix) >= 0 && xi_slot<n>(iy) >= 0;
        const C2 z = keep ? cscale(v, invP) : zero2<T>();
        muhp[ix * n + iy] = cscale(z, (T)(2.0 * kPi));
        return z;
      },
      [&](int ix, int iy, C2 v) { M[ix * n + iy] = v; });
  row_pass<n, 1, false, 0, CB, true>(
      sm, tw, [&](int ix, int iy) { return xi_t<B>(iy % B) ? ldc<n, CB>(&M[ix * n + iy]) : zero2<T>(); }, NoMid(),
      [&](int ix, int iy, C2 v) { M[ix * n + iy] = v; });
}

// --------------------------------------------------------------------------
// Seed: the transpose of the pointwise Pauli assembly, from mu (k_vjp_mu) and the forward D and K4
// fields (k_dk_fields).  Outputs: nu[c][2] (direct cotangent of the w pairs), nuf[c] (cotangent of
// f = 2 w0 - 1), muD[c][2] (pairs (D1,D2),(D3,-)), muK2[c], mu4[c][2] (raw K4
// pairs), mu3[c][2] (raw K3 pairs), mupl[c][4] (may be null: mu3 as planes in thread_order).
// --------------------------------------------------------------------------
template <int n, class T>
__global__ void __launch_bounds__(kThreads) k_vjp_seed(
    const typename Vec2Of<T>::type* MUall, const typename Vec2Of<T>::type* DKall,
    const typename Vec2Of<T>::type* wfine, const T* K2acc, typename Vec2Of<T>::type* nu, T* nuf,
    typename Vec2Of<T>::type* muD, T* muK2, typename Vec2Of<T>::type* mu4, typename Vec2Of<T>::type* mu3, T* mupl,
    int ncells) {
  using C2 = typename Vec2Of<T>::type;
  constexpr int P = n * n;
  for (size_t g = (size_t)blockIdx.x * kThreads + threadIdx.x; g < (size_t)ncells * P;
       g += (size_t)gridDim.x * kThreads) {
    const int c = (int)(g / P), i = (int)(g % P);
    const C2* MU = MUall + (size_t)c * 2 * P;
    const C2* DK = DKall + (size_t)c * 4 * P;
    const C2* wf0 = wfine + (size_t)c * 2 * P;
    const C2* wf1 = wf0 + P;
    const T* K2 = K2acc + (size_t)c * P;
    C2* nuc = nu + (size_t)c * 2 * P;
    T* nufc = nuf + (size_t)c * P;
    C2* muDc = muD + (size_t)c * 2 * P;
    T* muK2c = muK2 + (size_t)c * P;
    C2* mu4c = mu4 + (size_t)c * 2 * P;
    C2* mu3c = mu3 + (size_t)c * 2 * P;
    const double tp = 2.0 * kPi;
    const C2 mu01 = MU[i], mu23 = MU[P + i];
    const C2 dk0 = DK[i], dk1 = DK[P + i], dk2 = DK[2 * P + i], dk3 = DK[3 * P + i];
    const double m0 = mu01.x, m1 = mu01.y, m2 = mu23.x, m3 = mu23.y;
    const double w0 = wf0[i].x, w1 = wf0[i].y, w2 = wf1[i].x, w3 = wf1[i].y;
    const double D1 = dk0.x, D2 = dk0.y, D3 = dk1.x;
    const double K40 = dk2.x, K41 = -(double)dk2.y;
    const double K42 = -(double)dk3.x, K43 = -(double)dk3.y;
    const double k2 = K2[i];
    // C0 = 2pi[K2(1-w0) - K3_0 + w0 K4_0 + w.K4];  C_c = -2 (D x w)_c + 2pi[-K2 w_c - K3_c + w0 K4_c + K4_0 w_c]
    const double g0 = tp * (m0 * (K40 - k2) + m1 * K41 + m2 * K42 + m3 * K43);
    // -2 (mu x D)_c + 2 pi (m0 K4_c + m_c (K4_0 - K2))
    const double g1 = -2.0 * (m2 * D3 - m3 * D2) + tp * (m0 * K41 + m1 * (K40 - k2));
    const double g2 = -2.0 * (m3 * D1 - m1 * D3) + tp * (m0 * K42 + m2 * (K40 - k2));
    const double g3 = -2.0 * (m1 * D2 - m2 * D1) + tp * (m0 * K43 + m3 * (K40 - k2));
    nuc[i] = mk2((T)g0, (T)g1);
    nuc[P + i] = mk2((T)g2, (T)g3);
    nufc[i] = (T)0;
    // muD = -2 (w x mu)
    const double dd1 = -2.0 * (w2 * m3 - w3 * m2), dd2 = -2.0 * (w3 * m1 - w1 * m3), dd3 = -2.0 * (w1 * m2 - w2 * m1);
    muDc[i] = mk2((T)dd1, (T)dd2);
    muDc[P + i] = mk2((T)dd3, (T)0);
    muK2c[i] = (T)(tp * (m0 * (1.0 - w0) - m1 * w1 - m2 * w2 - m3 * w3));
    // K4_b = eta_b raw_b
    const double q0 = tp * (m0 * w0 + m1 * w1 + m2 * w2 + m3 * w3);
    const double q1 = -tp * (m0 * w1 + m1 * w0), q2 = -tp * (m0 * w2 + m2 * w0), q3 = -tp * (m0 * w3 + m3 * w0);
    mu4c[i] = mk2((T)q0, (T)q1);
    mu4c[P + i] = mk2((T)q2, (T)q3);
    // K3_b = eta_b raw_b, C_b has -2 pi K3_b
    mu3c[i] = mk2((T)(-tp * m0), (T)(tp * m1));
    mu3c[P + i] = mk2((T)(tp * m2), (T)(tp * m3));
    if (mupl) {
      T* pl = mupl + (size_t)c * 4 * P + thread_order<n>(i / n, i % n);
      pl[0] = mu3c[i].x;
      pl[P] = mu3c[i].y;
      pl[2 * P] = mu3c[P + i].x;
      pl[3 * P] = mu3c[P + i].y;
    }
  }
}

// --------------------------------------------------------------------------
// I1 transpose.  D_b = -K'(f A w_b) with A = "multiply by i phi'_j'", K' = "by i K_j'":
//   nu_f += sum_j' (K' mu_b)(A w_b),   nu_b += -A(f K' mu_b).  One block per cell.
// --------------------------------------------------------------------------
template <int n, class T, int CB>
__global__ void __launch_bounds__(kThreads, (cell_min_blocks<n, T, CB>()))
    k_i1_vjp(const typename Vec2Of<T>::type* what, const typename Vec2Of<T>::type* wfine,
             const typename Vec2Of<T>::type* muD, typename Vec2Of<T>::type* nu, T* nuf, typename Vec2Of<T>::type* ws,
             const typename Vec2Of<T>::type* __restrict__ gtw, const T* __restrict__ phip,
             const T* __restrict__ Ktab, int J, int nch) {
  using C2 = typename Vec2Of<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* tw = reinterpret_cast<C2*>(smem_raw);
  C2* sm = tw + n;
  load_twiddles<n>(tw, gtw);
  constexpr int P = n * n, B = Split<n>::B;
  // block (cell c, angle chunk ch); with nch > 1, nu and nuf are per-(cell, chunk) partials (zeroed
  // here, completed by k_i24_vjp, summed by k_add_chunks), with nch = 1 the cell's own accumulators
  const int c = cluster_index() / nch, ch = cluster_index() % nch;
  C2* slot = ws + (size_t)cluster_index() * 3 * P;
  C2* Aw = slot;          // A w_pair
  C2* Bm = slot + P;      // K' mu_pair
  C2* G = slot + 2 * P;
  const C2* wf0 = wfine + (size_t)c * 2 * P;
  C2* nuc = nu + (size_t)cluster_index() * 2 * P;
  T* nufc = nuf + (size_t)cluster_index() * P;
  if (nch > 1) {
    zero_fields_team(nuc, 2 * P);
    for (int i = element_first(); i < P; i += element_stride()) nufc[i] = (T)0;
    team_sync();
  }
  const T invP = (T)(1.0 / (double)P);
  for (int jp = J * ch / nch; jp < J * (ch + 1) / nch; ++jp) {
    const T* ph = phip + (size_t)jp * P;
    const T* K = Ktab + (size_t)jp * P;
    for (int p = 0; p < 2; ++p) {
      const C2* in = what + ((size_t)c * 4 + 2 + p) * P;
      const C2* mu = muD + ((size_t)c * 2 + p) * P;
      // Aw = IFFT(i phi' w^)
      xi_col_pass<n, CB>(
          sm, tw, [&](int ix, int iy) { return mul_i(in[ix * n + iy], ph[ix * n + iy]); },
          [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
      row_pass<n, 1, false, 0, CB, true>(
          sm, tw, [&](int ix, int iy) { return xi_t<B>(iy % B) ? ldc<n, CB>(&G[ix * n + iy]) : zero2<T>(); }, NoMid(),
          [&](int ix, int iy, C2 v) { Aw[ix * n + iy] = v; });
      // Bm = IFFT(i K FFT(mu))   (K already carries 1/n^2)
      row_pass<n, -1, false, 0, CB>(
          sm, tw, [&](int ix, int iy) { return mu[ix * n + iy]; }, NoMid(),
          [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
      col_pass<n, -1, true, 1, CB>(
          sm, tw, [&](int ix, int iy) { return ldc<n, CB>(&G[ix * n + iy]); },
          [&](int ix, int iy, C2 v) { return mul_i(v, K[ix * n + iy]); },
          [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
      row_pass<n, 1, false, 0, CB>(
          sm, tw, [&](int ix, int iy) { return ldc<n, CB>(&G[ix * n + iy]); }, NoMid(),
          [&](int ix, int iy, C2 v) { Bm[ix * n + iy] = v; });
      // nu_f += Re.Re + Im.Im ;  then -A(f Bm) into nu (pair layout of this p)
      row_pass<n, -1, false, 0, CB>(
          sm, tw,
          [&](int ix, int iy) {
            const int i = ix * n + iy;
            const C2 a = ldc<n, CB>(&Aw[i]), b = ldc<n, CB>(&Bm[i]);
            nufc[i] += a.x * b.x + a.y * b.y;
            return cscale(b, (T)2 * wf0[i].x - (T)1);
          },
          NoMid(), [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
      col_pass<n, -1, true, 1, CB>(
          sm, tw, [&](int ix, int iy) { return ldc<n, CB>(&G[ix * n + iy]); },
          [&](int ix, int iy, C2 v) { return mul_i(v, -ph[ix * n + iy] * invP); },
          [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
      row_pass<n, 1, false, 0, CB>(
          sm, tw, [&](int ix, int iy) { return ldc<n, CB>(&G[ix * n + iy]); }, NoMid(),
          [&](int ix, int iy, C2 v) {
            const int i = ix * n + iy;
            // pair p = 0 carries components (1, 2) -> nu pair 0 .y and nu pair 1 .x; p = 1 carries (3, -)
            if (p == 0) {
              nuc[i].y += v.x;
              nuc[P + i].x += v.y;
            } else {
              nuc[P + i].y += v.x;
            }
          });
    }
  }
}

// --------------------------------------------------------------------------
// I2/I4 transpose.  F_{a,j} = Psi_j w_a (even multipliers: self-adjoint).
//   K2 = 2 (pi/J) sum_{j<J/2} sum_a eta_a F_{a,j} F_{a,j'} ,  j' = j + J/2
//   K4raw_b = (pi/J) sum_{j<J/2} [Psi_j(f F_{b,j'}) + Psi_j'(f F_{b,j})]
// One block per cell.
// --------------------------------------------------------------------------
template <int n, class T, int CB>
__global__ void __launch_bounds__(kThreads, (cell_min_blocks<n, T, CB>()))
    k_i24_vjp(const typename Vec2Of<T>::type* what, const typename Vec2Of<T>::type* wfine, const T* muK2,
              const typename Vec2Of<T>::type* mu4, typename Vec2Of<T>::type* nu, T* nuf,
              typename Vec2Of<T>::type* ws, const typename Vec2Of<T>::type* __restrict__ gtw,
              const T* __restrict__ psi, int J, int nch) {
  using C2 = typename Vec2Of<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* tw = reinterpret_cast<C2*>(smem_raw);
  C2* sm = tw + n;
  load_twiddles<n>(tw, gtw);
  constexpr int P = n * n, B = Split<n>::B;
  // block (cell c, chunk ch of the J/2 angle pairs); nu, nuf as in k_i1_vjp
  const int c = cluster_index() / nch, ch = cluster_index() % nch;
  C2* slot = ws + (size_t)cluster_index() * 7 * P;
  C2* FA = slot;             // [2] F_{.,j}
  C2* FB = slot + 2 * P;     // [2] F_{.,j'}
  C2* PM = slot + 4 * P;     // [2] Psi(mu4) for the current direction
  C2* G = slot + 6 * P;
  const C2* wf0 = wfine + (size_t)c * 2 * P;
  const T* mk2c = muK2 + (size_t)c * P;
  const C2* m4 = mu4 + (size_t)c * 2 * P;
  C2* nuc = nu + (size_t)cluster_index() * 2 * P;
  T* nufc = nuf + (size_t)cluster_index() * P;
  const T wj = (T)(kPi / J);
  const T invP = (T)(1.0 / (double)P);
  const int H = J / 2;
  for (int j = H * ch / nch; j < H * (ch + 1) / nch; ++j) {
    const int jq = j + J / 2;
    for (int p = 0; p < 2; ++p) {
      const C2* in = what + ((size_t)c * 4 + p) * P;
      for (int h = 0; h < 2; ++h) {
        const T* ps = psi + (size_t)(h == 0 ? j : jq) * P;
        C2* F = (h == 0 ? FA : FB) + (size_t)p * P;
        xi_col_pass<n, CB>(
            sm, tw, [&](int ix, int iy) { return cscale(in[ix * n + iy], ps[ix * n + iy]); },
            [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
        row_pass<n, 1, false, 0, CB, true>(
            sm, tw, [&](int ix, int iy) { return xi_t<B>(iy % B) ? ldc<n, CB>(&G[ix * n + iy]) : zero2<T>(); }, NoMid(),
            [&](int ix, int iy, C2 v) { F[ix * n + iy] = v; });
      }
    }
    for (int h = 0; h < 2; ++h) {
      const T* ps = psi + (size_t)(h == 0 ? j : jq) * P;       // Psi_j pairs with F_{j'}, Psi_j' with F_j
      const T* pq = psi + (size_t)(h == 0 ? jq : j) * P;
      const C2* Fo = (h == 0 ? FB : FA);                          // the other direction's F
      for (int p = 0; p < 2; ++p) {
        const C2* F = Fo + (size_t)p * P;
        const C2* mup = m4 + (size_t)p * P;
        C2* PMp = PM + (size_t)p * P;
        const T eta0 = (p == 0) ? (T)1 : (T)-1;
        // K2 part: nu_a += 2 (pi/J) eta_a Psi_{dir}(muK2 * F_other)
        // K4 part: PMp = Psi_{dir}(mu4_pair)
        for (int part = 0; part < 2; ++part) {
          row_pass<n, -1, false, 0, CB>(
              sm, tw,
              [&](int ix, int iy) {
                const int i = ix * n + iy;
                return part == 0 ? cscale(ldc<n, CB>(&F[i]), mk2c[i]) : mup[i];
              },
              NoMid(), [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
          col_pass<n, -1, true, 1, CB>(
              sm, tw, [&](int ix, int iy) { return ldc<n, CB>(&G[ix * n + iy]); },
              [&](int ix, int iy, C2 v) { return cscale(v, ps[ix * n + iy] * invP); },
              [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
          row_pass<n, 1, false, 0, CB>(
              sm, tw, [&](int ix, int iy) { return ldc<n, CB>(&G[ix * n + iy]); }, NoMid(),
              [&](int ix, int iy, C2 v) {
                const int i = ix * n + iy;
                if (part == 0) {
                  C2 o = nuc[(size_t)p * P + i];
                  o.x += (T)2 * wj * eta0 * v.x;     // eta of component 2p
                  o.y += (T)2 * wj * (T)(-1) * v.y;  // eta of component 2p+1 (always -1)
                  nuc[(size_t)p * P + i] = o;
                } else {
                  PMp[i] = v;
                }
              });
        }
        // nu_f += (pi/J) PM . F_other ; nu_b += (pi/J) Psi_other(f PM)
        row_pass<n, -1, false, 0, CB>(
            sm, tw,
            [&](int ix, int iy) {
              const int i = ix * n + iy;
              const C2 pmv = ldc<n, CB>(&PMp[i]), fv = ldc<n, CB>(&F[i]);
              nufc[i] += wj * (pmv.x * fv.x + pmv.y * fv.y);
              return cscale(pmv, (T)2 * wf0[i].x - (T)1);
            },
            NoMid(), [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
        col_pass<n, -1, true, 1, CB>(
            sm, tw, [&](int ix, int iy) { return ldc<n, CB>(&G[ix * n + iy]); },
            [&](int ix, int iy, C2 v) { return cscale(v, pq[ix * n + iy] * invP); },
            [&](int ix, int iy, C2 v) { G[ix * n + iy] = v; });
        row_pass<n, 1, false, 0, CB>(
            sm, tw, [&](int ix, int iy) { return ldc<n, CB>(&G[ix * n + iy]); }, NoMid(),
            [&](int ix, int iy, C2 v) {
              const int i = ix * n + iy;
              C2 o = nuc[(size_t)p * P + i];
              o.x += wj * v.x;
              o.y += wj * v.y;
              nuc[(size_t)p * P + i] = o;
            });
      }
    }
  }
}

// nu[c] += sum_ch nupart[c][ch] (2 complex fields) and nuf[c] += sum_ch nufpart[c][ch] (1 real
// field), in chunk order: the per-(cell, chunk) partials of k_i1_vjp + k_i24_vjp.
template <class T>
__global__ void __launch_bounds__(kThreads) k_add_chunks(const T* __restrict__ nupart, const T* __restrict__ nufpart,
                                                         T* nu, T* nuf, int nch, int ncells, size_t P) {
  const size_t per_c = 4 * P;
  const size_t total = (size_t)ncells * (per_c + P);
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const T* src;
    T* dst;
    size_t c, e, stride;
    if (i < (size_t)ncells * per_c) {
      c = i / per_c; e = i % per_c; src = nupart; dst = nu; stride = per_c;
    } else {
      const size_t k = i - (size_t)ncells * per_c;
      c = k / P; e = k % P; src = nufpart; dst = nuf; stride = P;
    }
    const T* p = src + (c * nch) * stride + e;
    T sum = p[0];
    for (int ch = 1; ch < nch; ++ch) sum += p[(size_t)ch * stride];
    dst[c * stride + e] += sum;
  }
}

// --------------------------------------------------------------------------
// I3 transpose (Hu-Ying term), nodes in pairs as in k_i3_sf (i3_staged_fused.cuh).  With s = S w,
// U_ab = Psi'(w_a s_b), K3raw_b = sum_a eta_a s_a U_ab (node m) and K3raw_a = S*[sum_b eta_b w_b U_ab]
// (its partner), cotangents mu_b of K3raw_b and nu = S mu:
//   Z_ab = Psi'(eta_a mu_b s_a + eta_b nu_a w_b)                 (cotangent of w_a s_b)
//   R_a += sum_b Z_ab s_b,  R_b += eta_b sum_a nu_a U_ab          (of w, real space)
//   X_b  = sum_a Z_ab w_a,  X_a += eta_a sum_b mu_b U_ab          (of s, then S* X of w, Fourier space)
// The middle node of an odd M has no partner and no nu.  With the first index in pairs q (2q, 2q + 1)
// a pair of nodes takes 8 complex convolutions for U and 8 for Z, 4 shifts and 2 transforms back, half
// of what its two nodes take one by one.
// Persistent blocks over units (cell, j, m-chunk); per unit outputs a real-space partial R[4][P] (planes)
// and a spectral partial [2][Q] on the kept frequencies (Q = (n/2 - 1)^2).
// Several cotangents (K of them, mu3 / muh / part_r / part_s of cotangent k at offsets k * mu_stride,
// k * part_stride and k * spart_stride) share the shifted fields and the U convolutions, which depend on
// the state only: per pair 8 + 8 K convolutions instead of 16 K.
// Bound by FP64 issue like k_i3_sf.
// --------------------------------------------------------------------------
constexpr int kVjpCB = 65536;
template <int n, class T>
__global__ void __launch_bounds__(kThreads, 3) k_i3_vjp(
    const typename Vec2Of<T>::type* what, const typename Vec2Of<T>::type* wfine,
    const typename Vec2Of<T>::type* mu3, const typename Vec2Of<T>::type* muh, typename Vec2Of<T>::type* part_r,
    typename Vec2Of<T>::type* part_s, typename Vec2Of<T>::type* ws, const T* __restrict__ psip_s,
    const typename Vec2Of<T>::type* __restrict__ phase, int J, int M, int nmc, int nunits, int K, size_t mu_stride, size_t part_stride, size_t spart_stride) {
  using C2 = typename Vec2Of<T>::type;
  using Lines = StagedLines<n, T, kThreads, kVjpCB>;
  constexpr int P = n * n, Q = Lines::Q;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int kslot[n];
  C2* slot = ws + (size_t)blockIdx.x * (3 + 4 * K) * P;
  C2* Sig = slot;                                  // [2][P] shifted pairs of the state
  C2* Nu = slot + 3 * P;                           // [K][2][P] shifted pairs of the cotangents
  T* X = reinterpret_cast<T*>(slot + (3 + 2 * K) * (size_t)P);   // [K][4][P]
  Lines ln;
  ln.init(reinterpret_cast<C2*>(smem_raw));
  ln.kslot = kslot;
  ln.G = slot + 2 * P;
  build_xi_slots<n>(kslot);
  for (int unit = blockIdx.x; unit < nunits; unit += gridDim.x) {
    const int c = unit / (J * nmc);
    const int j = (unit / nmc) % J;
    const int mc = unit % nmc;
    for (int k = 0; k < K; ++k) {
      zero_fields(part_r + k * part_stride + (size_t)unit * 2 * P, 2 * P);
      zero_fields(part_s + k * spart_stride + (size_t)unit * 2 * Q, 2 * Q);
    }
    const T* __restrict__ psp = psip_s + (size_t)j * P;
    const C2* wf = wfine + (size_t)c * 2 * P;
    const int it1 = i3_chunk_begin(mc + 1, nmc, M);
    for (int it = i3_chunk_begin(mc, nmc, M); it < it1;) {
      const I3Group gr = i3_group_at(it, it1, M);
      it = gr.next;
      const C2* px = phase + ((size_t)j * M + gr.m) * 2 * n;
      const C2* py = px + n;
      // shifted pairs of the state, then of each cotangent (component 0 of mu3 is -2 pi mu_0)
      for (int f = 0; f < (gr.pair ? 2 + 2 * K : 2); ++f) {
        const int k = (f - 2) >> 1, p = f & 1;
        const C2* in = f < 2 ? what + ((size_t)c * 4 + p) * P : muh + k * mu_stride + ((size_t)c * 2 + p) * P;
        C2* S = f < 2 ? Sig + (size_t)p * P : Nu + ((size_t)2 * k + p) * P;
        const T sx = (f >= 2 && p == 0) ? (T)-1 : (T)1;
        ln.shift(in, px, py, [&](int idx, C2 v) { S[idx] = mk2(sx * v.x, v.y); });
      }
      zero_fields(reinterpret_cast<C2*>(X), 2 * K * P);
      for (int q = gr.q0; q < gr.q1; ++q) {
        const C2* wq = wf + (size_t)q * P;
        const C2* Sq = Sig + (size_t)q * P;
        const T e0 = q == 0 ? (T)1 : (T)-1;
        for (int b = 0; b < 4; ++b) {
          const T* Sb = reinterpret_cast<const T*>(Sig + (size_t)(b >> 1) * P) + (b & 1);
          const T* wb = reinterpret_cast<const T*>(wf + (size_t)(b >> 1) * P) + (b & 1);
          const T eb = b == 0 ? (T)1 : (T)-1;
          const size_t mu_b = ((size_t)c * 2 + (b >> 1)) * P * 2 + (b & 1);   // of component b in the pairs of mu3
          // U: X_q += eta_q mu_b U, R_b += eta_b nu_q . U
          ln.convolve(
              psp, [&](int idx) { return cscale(wq[idx], Sb[2 * idx]); },
              [&](int idx, C2 v) {
                for (int k = 0; k < K; ++k) {
                  const T m = reinterpret_cast<const T*>(mu3 + k * mu_stride)[mu_b + 2 * idx];
                  T* Xq = X + ((size_t)4 * k + 2 * q) * P + idx;
                  Xq[0] = fmaT(e0 * m, v.x, Xq[0]);
                  Xq[P] = fmaT(-m, v.y, Xq[P]);
                  if (gr.pair) {
                    const C2 nu = Nu[((size_t)2 * k + q) * P + idx];
                    T* Rb = reinterpret_cast<T*>(part_r + k * part_stride + (size_t)unit * 2 * P) + (size_t)b * P + idx;
                    *Rb = fmaT(eb * nu.x, v.x, fmaT(eb * nu.y, v.y, *Rb));
                  }
                }
              });
          // Z per cotangent: R_q += s_b Z, X_b += w_q . Z
          for (int k = 0; k < K; ++k) {
            const T* mub = reinterpret_cast<const T*>(mu3 + k * mu_stride) + mu_b;
            const C2* nuq = Nu + ((size_t)2 * k + q) * P;
            T* Rq = reinterpret_cast<T*>(part_r + k * part_stride + (size_t)unit * 2 * P) + (size_t)2 * q * P;
            T* Xb = X + ((size_t)4 * k + b) * P;
            ln.convolve(
                psp,
                [&](int idx) {
                  const T m = mub[2 * idx];
                  const C2 s = Sq[idx];
                  C2 g = mk2(e0 * m * s.x, -m * s.y);
                  if (gr.pair) {
                    const C2 nu = nuq[idx];
                    const T f = eb * wb[2 * idx];
                    g = mk2(fmaT(f, nu.x, g.x), fmaT(f, nu.y, g.y));
                  }
                  return g;
                },
                [&](int idx, C2 v) {
                  const T s = Sb[2 * idx];
                  const C2 wv = wq[idx];
                  Rq[idx] = fmaT(s, v.x, Rq[idx]);
                  Rq[P + idx] = fmaT(s, v.y, Rq[P + idx]);
                  Xb[idx] = fmaT(wv.x, v.x, fmaT(wv.y, v.y, Xb[idx]));
                });
          }
        }
      }
      for (int k = 0; k < K; ++k)
        for (int p = 0; p < 2; ++p) {
          const T* Xp = X + ((size_t)4 * k + 2 * p) * P;
          ln.shift_back(px, py, part_s + k * spart_stride + (size_t)unit * 2 * Q + (size_t)p * Q, false,
                        [&](int idx) { return mk2(Xp[idx], Xp[P + idx]); });
        }
    }
  }
}

// --------------------------------------------------------------------------
// The same with the transform field resident in shared memory (FP32, n <= 128),
// the counterpart of k_i3_smem: each convolution's epilogue adds its terms straight
// into the accumulators (R in the unit's partial, X in scratch).
// --------------------------------------------------------------------------
template <int n>
__global__ void __launch_bounds__(kThreadsI3Smem, 1) k_i3_vjp_smem(
    const float2* what, const float2* wfine, const float2* mu3, const float2* muh, float2* part_r, float2* part_s,
    float2* ws, const float2* __restrict__ gtw, const float* __restrict__ psip_s, const float2* __restrict__ phase,
    int J, int M, int nmc, int nunits, int K, size_t mu_stride, size_t part_stride, size_t spart_stride) {
  using C2 = float2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* tw = reinterpret_cast<C2*>(smem_raw);
  C2* G = tw + n;
  float* psm = reinterpret_cast<float*>(G + n * (n + 1));
  constexpr int LS = n + 1, P = n * n;
  constexpr int NQ = xi_kept<n>(), Q = NQ * NQ;
  constexpr int kIter = (P + kThreadsI3Smem - 1) / kThreadsI3Smem;
  __shared__ unsigned char xmask[n];
  __shared__ int kslot[n];
  __shared__ int kcols[n];
  for (int pos = threadIdx.x; pos < n; pos += blockDim.x) xmask[pos] = xi_t<Split<n>::B>(pos % Split<n>::B) ? 1 : 0;
  build_xi_slots<n>(kslot, kcols);
  load_twiddles<n>(tw, gtw);
  C2* slot = ws + (size_t)blockIdx.x * (2 + 4 * K) * P;
  C2* Sig = slot;                                                 // [2][P]
  C2* Nu = slot + 2 * P;                                          // [K][2][P]
  float* X = reinterpret_cast<float*>(slot + (2 + 2 * K) * (size_t)P);   // [K][4][P]
  // element loop over the field with a compile-time trip count
  auto elements = [&](auto body) {
#pragma unroll 4
    for (int k = 0; k < kIter; ++k) {
      const int idx = threadIdx.x + k * kThreadsI3Smem;
      if (kIter * kThreadsI3Smem == P || idx < P) body(idx, G[(idx / n) * LS + idx % n]);
    }
    __syncthreads();
  };
  for (int unit = blockIdx.x; unit < nunits; unit += gridDim.x) {
    const int c = unit / (J * nmc);
    const int j = (unit / nmc) % J;
    const int mc = unit % nmc;
    for (int k = 0; k < K; ++k) {
      zero_fields(part_r + k * part_stride + (size_t)unit * 2 * P, 2 * P);
      zero_fields(part_s + k * spart_stride + (size_t)unit * 2 * Q, 2 * Q);
    }
    {
      const float4* src = reinterpret_cast<const float4*>(psip_s + (size_t)j * P);
      float4* dst = reinterpret_cast<float4*>(psm);
      for (int i4 = threadIdx.x; i4 < P / 4; i4 += blockDim.x) dst[i4] = src[i4];
      __syncthreads();
    }
    const C2* __restrict__ wf = wfine + (size_t)c * 2 * P;
    auto convolve = [&]() {
      fft_lines<n, -1>(G, n, LS, 1, tw);
      fft_conv_lines<n>(G, n, 1, LS, tw, [&](int l, int pos) { return psm[pos * n + l]; });
      fft_lines<n, 1>(G, n, LS, 1, tw);
    };
    const int it1 = i3_chunk_begin(mc + 1, nmc, M);
    for (int it = i3_chunk_begin(mc, nmc, M); it < it1;) {
      const I3Group gr = i3_group_at(it, it1, M);
      it = gr.next;
      const C2* px = phase + ((size_t)j * M + gr.m) * 2 * n;
      const C2* py = px + n;
      for (int f = 0; f < (gr.pair ? 2 + 2 * K : 2); ++f) {
        const int k = (f - 2) >> 1, p = f & 1;
        const C2* in = f < 2 ? what + ((size_t)c * 4 + p) * P : muh + k * mu_stride + ((size_t)c * 2 + p) * P;
        C2* S = f < 2 ? Sig + (size_t)p * P : Nu + ((size_t)2 * k + p) * P;
        const float sx = (f >= 2 && p == 0) ? -1.f : 1.f;   // component 0 of mu3 is -2 pi mu_0
        elements([&](int idx, C2& g) {
          const int ix = idx / n, iy = idx % n;
          g = (xmask[ix] && xmask[iy]) ? cmul(in[idx], cmul(px[ix], py[iy])) : zero2<float>();
        });
        fft_lines<n, 1, true>(G, n, 1, LS, tw);   // shifts: input zero outside Xi x Xi
        fft_lines<n, 1, true>(G, n, LS, 1, tw);
        elements([&](int idx, C2& g) { S[idx] = mk2(sx * g.x, g.y); });
      }
      zero_fields(reinterpret_cast<C2*>(X), 2 * K * P);
      for (int q = gr.q0; q < gr.q1; ++q) {
        const C2* __restrict__ wq = wf + (size_t)q * P;
        const C2* Sq = Sig + (size_t)q * P;
        const float e0 = q == 0 ? 1.f : -1.f;
        for (int b = 0; b < 4; ++b) {
          const float* Sb = reinterpret_cast<const float*>(Sig + (size_t)(b >> 1) * P) + (b & 1);
          const float* __restrict__ wb = reinterpret_cast<const float*>(wf + (size_t)(b >> 1) * P) + (b & 1);
          const float eb = b == 0 ? 1.f : -1.f;
          const size_t mu_b = ((size_t)c * 2 + (b >> 1)) * P * 2 + (b & 1);
          // U: X_q += eta_q mu_b U, R_b += eta_b nu_q . U
          elements([&](int idx, C2& g) { g = cscale(wq[idx], Sb[2 * idx]); });
          convolve();
          for (int k = 0; k < K; ++k) {
            const float* __restrict__ mb = reinterpret_cast<const float*>(mu3 + k * mu_stride) + mu_b;
            const C2* nuq = Nu + ((size_t)2 * k + q) * P;
            float* Xq = X + ((size_t)4 * k + 2 * q) * P;
            float* Rb = reinterpret_cast<float*>(part_r + k * part_stride + (size_t)unit * 2 * P) + (size_t)b * P;
            elements([&](int idx, C2& g) {
              const float m = mb[2 * idx];
              Xq[idx] = fmaf(e0 * m, g.x, Xq[idx]);
              Xq[P + idx] = fmaf(-m, g.y, Xq[P + idx]);
              if (gr.pair) {
                const C2 nu = nuq[idx];
                Rb[idx] = fmaf(eb * nu.x, g.x, fmaf(eb * nu.y, g.y, Rb[idx]));
              }
            });
          }
          // Z per cotangent: R_q += s_b Z, X_b += w_q . Z
          for (int k = 0; k < K; ++k) {
            const float* __restrict__ mb = reinterpret_cast<const float*>(mu3 + k * mu_stride) + mu_b;
            const C2* nuq = Nu + ((size_t)2 * k + q) * P;
            float* Rq = reinterpret_cast<float*>(part_r + k * part_stride + (size_t)unit * 2 * P) + (size_t)2 * q * P;
            float* Xb = X + ((size_t)4 * k + b) * P;
            elements([&](int idx, C2& g) {
              const float m = mb[2 * idx];
              const C2 s = Sq[idx];
              g = mk2(e0 * m * s.x, -m * s.y);
              if (gr.pair) {
                const C2 nu = nuq[idx];
                const float f = eb * wb[2 * idx];
                g = mk2(fmaf(f, nu.x, g.x), fmaf(f, nu.y, g.y));
              }
            });
            convolve();
            elements([&](int idx, C2& g) {
              const float s = Sb[2 * idx];
              const C2 wv = wq[idx];
              Rq[idx] = fmaf(s, g.x, Rq[idx]);
              Rq[P + idx] = fmaf(s, g.y, Rq[P + idx]);
              Xb[idx] = fmaf(wv.x, g.x, fmaf(wv.y, g.y, Xb[idx]));
            });
          }
        }
      }
      for (int kc = 0; kc < K; ++kc) {
        for (int p = 0; p < 2; ++p) {
          const float* Xp = X + ((size_t)4 * kc + 2 * p) * P;
          C2* dst = part_s + kc * spart_stride + (size_t)unit * 2 * Q + (size_t)p * Q;
          elements([&](int idx, C2& g) { g = mk2(Xp[idx], Xp[P + idx]); });
          fft_lines<n, -1>(G, n, LS, 1, tw);    // rows
          fft_lines<n, -1>(G, n, 1, LS, tw);    // columns
          // accumulated on the kept frequencies only
          for (int e = threadIdx.x; e < Q; e += blockDim.x) {
            const int ix = kcols[e / NQ], iy = kcols[e % NQ];
            dst[e] = cadd(dst[e], cmulc(G[ix * LS + iy], cmul(px[ix], py[iy])));
          }
          __syncthreads();
        }
      }
    }
  }
}

#include "i3_vjp_tmem.cuh"

// --------------------------------------------------------------------------
// Final: nu = direct + I1 + I2/I4 + 2 nu_f (into w0) + R, the reduced I3 real-space
// partials (planes [4][P], FP64); gradient = 4 E P (nu + IFFT(H) / n^2) with H the
// reduced I3 spectral partials (k_reduce_k3).  P keeps the kept frequencies only and FFT(IFFT(H)) =
// n^2 H, so H (stored on those frequencies) is added to FFT(nu) there.
// One team per cell and pair; writes grad[c][4][N][N] (FP64).
// --------------------------------------------------------------------------
template <int n, class T, int CB>
__global__ void __launch_bounds__(kThreads, (cell_min_blocks<n, T, CB>()))
    k_vjp_final(const typename Vec2Of<T>::type* nu, const T* nuf, const double* R, size_t r_stride,
                const double2* spec, size_t spec_stride, typename Vec2Of<T>::type* ws,
                const typename Vec2Of<T>::type* __restrict__ gtw, double* grad, int accumulate) {
  using C2 = typename Vec2Of<T>::type;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2* tw = reinterpret_cast<C2*>(smem_raw);
  C2* sm = tw + n;
  load_twiddles<n>(tw, gtw);
  constexpr int N = n / 2, P = n * n, B = Split<n>::B;
  constexpr int NQ = xi_kept<n>(), Q = NQ * NQ;
  const int c = cluster_index() >> 1, p = cluster_index() & 1;
  C2* F = ws + (size_t)cluster_index() * P;
  const double* Rc = R + c * r_stride + (size_t)2 * p * P;
  const double2* Hp = spec + c * spec_stride + (size_t)p * Q;
  const C2* nup = nu + ((size_t)c * 2 + p) * P;
  const T* nufc = nuf + (size_t)c * P;
  const T invP = (T)(1.0 / (double)P);
  // 4 E P (V + IFFT(H) / n^2), V the total real-space cotangent of the pair
  row_pass<n, -1, false, 0, CB>(
      sm, tw,
      [&](int ix, int iy) {
        const int i = ix * n + iy;
        const C2 d = nup[i];
        double vx = (double)d.x + Rc[i];
        const double vy = (double)d.y + Rc[P + i];
        if (p == 0) vx += 2.0 * (double)nufc[i];
        return mk2((T)vx, (T)vy);
      },
      NoMid(),
      [&](int ix, int iy, C2 v) {
        if (xi_t<B>(iy % B)) F[ix * n + iy] = v;
      });
  xi_col_filter<n, true, true, CB>(
      sm, tw, [&](int ix, int iy) { return ldc<n, CB>(&F[ix * n + iy]); },
      [&](int ix, int iy, C2 v) {
        const int sx = xi_slot<n>(ix), sy = xi_slot<n>(iy);
        if (sx < 0 || sy < 0) return zero2<T>();
        const double2 h = Hp[sx * NQ + sy];
        return cscale(mk2((T)((double)v.x + h.x), (T)((double)v.y + h.y)), invP);
      },
      [&](int ix, int iy, C2 v) {
        if (!(ix & 1)) F[ix * n + iy] = v;
      });
  double* g = grad + (size_t)c * 4 * N * N;
  even_row_pass<n, 1, CB, true>(
      sm, tw, [&](int ix, int iy) { return xi_t<B>(iy % B) ? ldc<n, CB>(&F[ix * n + iy]) : zero2<T>(); },
      [&](int ix, int iy, C2 v) {
        if (!(iy & 1)) {
          const int i = ix >> 1, j = iy >> 1;
          double* g0 = g + ((2 * p) * N + i) * N + j;
          double* g1 = g + ((2 * p + 1) * N + i) * N + j;
          *g0 = (accumulate ? *g0 : 0.0) + 4.0 * (double)v.x;
          *g1 = (accumulate ? *g1 : 0.0) + 4.0 * (double)v.y;
        }
      });
}

}  // namespace

// I3 transpose kernels per (n, T): staged in FP64 and above 128 points; in FP32 the teams with
// tensor-memory exchanges at 32, 64 and 128 points, the element-pass shared-memory kernel at 16 and 96
// and as variant 1 at 128.
template <int n, class T>
constexpr bool vjp_tmem() {
  return std::is_same<T, float>::value && (n == 32 || n == 64 || n == 128);
}
template <int n, class T>
constexpr bool vjp_smem() {
  return std::is_same<T, float>::value && (n == 16 || n == 96 || n == 128);
}
template <int n, class T>
constexpr bool vjp_staged() {
  return !vjp_tmem<n, T>() && !vjp_smem<n, T>();
}

template <int n, class T>
void set_vjp_smem_attributes() {
  static unsigned long long done = 0;
  if (!first_on_device(done)) return;
  QBE_CELLS_SMEM(k_vjp_mu);
  QBE_CELLS_SMEM(k_i1_vjp);
  QBE_CELLS_SMEM(k_i24_vjp);
  QBE_CELLS_SMEM(k_vjp_final);
  if constexpr (vjp_staged<n, T>())
    cudaFuncSetAttribute(k_i3_vjp<n, T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)i3_sf_smem_bytes<n, T, kVjpCB>());
  if constexpr (vjp_smem<n, T>())
    cudaFuncSetAttribute(k_i3_vjp_smem<n>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)i3_smem_bytes<n>());
  if constexpr (vjp_tmem<n, T>())
    cudaFuncSetAttribute(k_i3_vjp_tmem<n>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TmShape<n>::smem);
}

// Forward prep/I1/I2+I4 once (the VJP needs wfine, D^, K2, K4^), then per cotangent the seed and the
// I1 and I2/I4 transposes, one I3 transpose launch for all K cotangents, and per cotangent the final
// assembly.  Cotangent k uses copy k of every cotangent buffer of vw.
template <int n, class T>
cudaError_t collide_vjp_n(const Tables& t, CollisionWork& cw, VjpWork& vw, const double* w, const double* const* lam,
                          double* const* grad, int K, int ncells, int accumulate, cudaStream_t s, long long& launches,
                          KernelTimer* tm) {
  using C2 = typename Vec2Of<T>::type;
  set_smem_attributes<n, T>();
  set_vjp_smem_attributes<n, T>();
  const TabPtrs<T> tb = tab_ptrs<T>(t);
  C2* what = (C2*)cw.what;
  C2* wfine = (C2*)cw.wfine;
  C2* Dacc = (C2*)cw.Dacc;
  T* K2acc = (T*)cw.K2acc;
  C2* K4acc = (C2*)cw.K4acc;
  C2* ws = (C2*)vw.ws;
  constexpr size_t P = (size_t)n * n;
  const size_t c_stride = (size_t)vw.nb * 2 * P;           // complex cotangent buffers, per cotangent
  const size_t r_stride = (size_t)vw.nb * P;               // real cotangent buffers, per cotangent
  const size_t nparts = (size_t)vw.nb * t.J * vw.nmc;
  const size_t part_stride = nparts * 2 * P;
  const size_t spart_stride = nparts * 2 * (size_t)xi_kept<n>() * xi_kept<n>();
  auto begin = [&](int g) { if (tm) tm->begin(g, s); };
  auto end = [&]() { if (tm) tm->end(s); };
  begin(KG_VJP);
  cudaError_t e = QBE_CELLS(k_prep, 4 * ncells, s, w, what, wfine, (T*)cw.wplane, ws, tb.tw);
  if (e != cudaSuccess) return e;
  ++launches;
  {
    e = per_cell_terms<n, T>(t, cw, ws, ncells, s, launches, nullptr);
    if (e != cudaSuccess) return e;
  }
  C2* DK = ws;   // [ncells][4][P] real-space D and K4 pairs of the state
  e = QBE_CELLS(k_dk_fields, 4 * ncells, s, Dacc, K4acc, DK, tb.tw);
  if (e != cudaSuccess) return e;
  ++launches;
  for (int k = 0; k < K; ++k) {
    C2* nu = (C2*)vw.nu + k * c_stride;
    T* nuf = (T*)vw.nuf + k * r_stride;
    C2* muD = (C2*)vw.muD + k * c_stride;
    T* muK2 = (T*)vw.muK2 + k * r_stride;
    C2* mu4 = (C2*)vw.mu4 + k * c_stride;
    C2* mu3 = (C2*)vw.mu3 + k * c_stride;
    C2* muh = (C2*)vw.muh + k * c_stride;
    T* mupl = vw.mupl ? (T*)vw.mupl + k * 2 * c_stride : nullptr;
    C2* MU = DK + (size_t)ncells * 4 * P;   // [ncells][2][P]
    e = QBE_CELLS(k_vjp_mu, 2 * ncells, s, lam[k], MU, muh, tb.tw);
    if (e != cudaSuccess) return e;
    if (k > 0) {   // the I1 and I2/I4 transposes of the cotangent before used the scratch
      e = QBE_CELLS(k_dk_fields, 4 * ncells, s, Dacc, K4acc, DK, tb.tw);
      if (e != cudaSuccess) return e;
      ++launches;
    }
    const size_t seed_blocks = ((size_t)ncells * P + kThreads - 1) / kThreads;
    k_vjp_seed<n, T><<<(unsigned)(seed_blocks < 65535 ? seed_blocks : 65535), kThreads, 0, s>>>(
        MU, DK, wfine, K2acc, nu, nuf, muD, muK2, mu4, mu3, mupl, ncells);
    ++launches;
    // I1 and I2/I4 transposes over (cell, angle chunk) blocks; their per-chunk cotangents go to the
    // forward's chunk-partial buffers (free once per_cell_terms has reduced them) and are summed in
    // chunk order into nu and nuf
    const int nch = cw.nch < 1 ? 1 : cw.nch;
    C2* nup = nch > 1 ? (C2*)cw.Dpart : nu;
    T* nufp = nch > 1 ? (T*)cw.K2part : nuf;
    e = QBE_CELLS(k_i1_vjp, ncells * nch, s, what, wfine, muD, nup, nufp, ws, tb.tw, tb.phip, tb.Ktab, t.J, nch);
    if (e != cudaSuccess) return e;
    e = QBE_CELLS(k_i24_vjp, ncells * nch, s, what, wfine, muK2, mu4, nup, nufp, ws, tb.tw, tb.psi, t.J, nch);
    if (e != cudaSuccess) return e;
    launches += 3;
    if (nch > 1) {
      k_add_chunks<T><<<element_blocks((size_t)ncells * 5 * P), kThreads, 0, s>>>(
          (const T*)nup, (const T*)nufp, (T*)nu, nuf, nch, ncells, P);
      ++launches;
    }
  }
  end();
  const int nunits = ncells * t.J * vw.nmc;
  const int grid = nunits < vw.grid ? nunits : vw.grid;
  begin(KG_VJP_I3);
  bool done = false, tmem = false;
  if constexpr (vjp_tmem<n, T>()) {
    tmem = K == 1 && vw.i3v == 0;
    if (tmem) {
      k_i3_vjp_tmem<n><<<grid, TmShape<n>::NT, TmShape<n>::smem, s>>>(
          what, (const T*)cw.wplane, (const T*)vw.mupl, (C2*)vw.muh, (C2*)vw.part_r, (C2*)vw.part_s, ws, tb.psip_s,
          tb.phase, t.J, t.M, vw.nmc, nunits);
      done = true;
    }
  }
  if constexpr (vjp_smem<n, T>()) {
    if (!done)
      k_i3_vjp_smem<n><<<grid, kThreadsI3Smem, i3_smem_bytes<n>(), s>>>(
          what, wfine, (C2*)vw.mu3, (C2*)vw.muh, (C2*)vw.part_r, (C2*)vw.part_s, ws, tb.tw, tb.psip_s, tb.phase, t.J,
          t.M, vw.nmc, nunits, K, c_stride, part_stride, spart_stride);
    done = true;
  }
  if constexpr (vjp_staged<n, T>()) {
    k_i3_vjp<n, T><<<grid, kThreads, i3_sf_smem_bytes<n, T, kVjpCB>(), s>>>(
        what, wfine, (C2*)vw.mu3, (C2*)vw.muh, (C2*)vw.part_r, (C2*)vw.part_s, ws, tb.psip_s, tb.phase, t.J, t.M,
        vw.nmc, nunits, K, c_stride, part_stride, spart_stride);
    done = true;
  }
  if (!done) return cudaErrorInvalidValue;
  end();
  ++launches;
  begin(KG_VJP);
  const int units = t.J * vw.nmc;
  constexpr int np = 2 * n * n, nq = 2 * xi_kept<n>() * xi_kept<n>();
  for (int k = 0; k < K; ++k) {
    C2* pr = (C2*)vw.part_r + k * part_stride;
    C2* ps = (C2*)vw.part_s + k * spart_stride;
    reduce_partials<T>(pr, cw.K3sum, ps, cw.K3ssum, units, np, nq, vw.nb, ncells, tmem ? n : 0, s);
    const double* R = cw.K3sum ? (const double*)cw.K3sum : (const double*)pr;
    const double2* H = cw.K3ssum ? cw.K3ssum : (const double2*)ps;
    e = QBE_CELLS(k_vjp_final, 2 * ncells, s, (C2*)vw.nu + k * c_stride, (T*)vw.nuf + k * r_stride, R,
                  (cw.K3sum ? (size_t)1 : (size_t)units) * 2 * np, H, (cw.K3ssum ? (size_t)1 : (size_t)units) * nq, ws,
                  tb.tw, grad[k], accumulate);
    if (e != cudaSuccess) return e;
    launches += 2;
  }
  end();
  return cudaGetLastError();
}

template <int n, class T>
int i3_vjp_blocks_per_sm() {
  set_vjp_smem_attributes<n, T>();
  int b = 0;
  if constexpr (vjp_tmem<n, T>()) b = 1;   // a block of 512 threads with the SM's tensor memory (and variant 1: 1)
  else if constexpr (vjp_smem<n, T>())
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_i3_vjp_smem<n>, kThreadsI3Smem, i3_smem_bytes<n>());
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_i3_vjp<n, T>, kThreads, i3_sf_smem_bytes<n, T, kVjpCB>());
  return b < 1 ? 1 : b;
}

}  // namespace qbe
