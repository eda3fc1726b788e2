// Transpose of the I3 (Hu-Ying, eq. approxH-JM) term's derivative in FP32 on padded grids of 32, 64
// and 128 points, one cotangent per product: the node pairs of k_i3_vjp on the teams and
// tensor-memory exchanges of k_i3_tmem.  Included by collision_vjp.cuh inside its anonymous namespace.
//
// Per pair of nodes, q and b the two convolutions U and Z run on one copy of the code.  X_q's sums
// over b live in tensor memory; every other sum is added in memory at the thread's own points by
// reductions (no other thread adds there, so the order is fixed): R[4][P] is the unit's real-space
// partial, X[4][P] the team's scratch, written first by the Z convolutions of the pair's first q.
// I3 transpose, 24 cells of N = 64, J = M = 32: 48 (node by node, transforms exchanged in shared memory)
// -> 24.0 ms.
#pragma once

template <int n>
__global__ void __launch_bounds__(TmShape<n>::NT, 1) k_i3_vjp_tmem(
    const float2* what, const float* wplane, const float* mupl, const float2* muh, float2* part_r, float2* part_s,
    float2* ws, const float* __restrict__ psip_s, const float2* __restrict__ phase, int J, int M, int nmc,
    int nunits) {
  using C2 = float2;
  using Sh = TmShape<n>;
  constexpr int P = n * n, H = Sh::H, TT = Sh::TEAM_THREADS;
  constexpr int NQ = xi_kept<n>(), Q = NQ * NQ;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint32_t tm_slot;
  const uint32_t tm_base = tmem_alloc<Sh::COLS>(&tm_slot);
  const TmLine<n> ln = tm_setup<n>(smem_raw, tm_base);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, h = ln.h;
  const int team = (w >> 2) / H * (4 / Sh::SPT) + (w & 3) / Sh::SPT;
  const int L = 32 * ((w & 3) % Sh::SPT) + lane;
  const int tt = L + n * h;
  C2* F = reinterpret_cast<C2*>(smem_raw + Sh::tw_bytes + team * Sh::team_bytes);
  float* psm = reinterpret_cast<float*>(F + n * Sh::LS);
  const uint32_t tv = ln.ex + Sh::EX + 64 * h;                     // X_q: real parts, then imaginary parts
  const int slot = team * gridDim.x + blockIdx.x, nslots = gridDim.x * Sh::TEAMS;
  float* S = reinterpret_cast<float*>(ws) + (size_t)slot * 12 * P;  // [4][P] shifted components of the state
  float* Nu = S + 4 * P;                                            // [4][P] of the cotangent
  float* X = Nu + 4 * P;                                            // [4][P]
  auto keep_step = [&]() {   // as in k_i3_tmem
    if constexpr (Sh::TEAMS > 1) __syncthreads();
  };
  for (int g0 = 0; g0 < nunits; g0 += nslots) {
    const bool have = g0 + slot < nunits;
    const int unit = have ? g0 + slot : 0;
    const int c = unit / (J * nmc);
    const int j = (unit / nmc) % J;
    const int mc = unit % nmc;
    float* R = reinterpret_cast<float*>(part_r + (size_t)unit * 2 * P);   // [4][P]
    C2* ps = part_s + (size_t)unit * 2 * Q;
    if (have) {
      const float* __restrict__ src = psip_s + (size_t)j * P;
      for (int i = tt; i < P; i += Sh::TEAM_THREADS) psm[freq_of_pos<n>(i % n) * n + freq_of_pos<n>(i / n)] = src[i];
#pragma unroll 4
      for (int i = 0; i < 32; ++i) tm_quad(R, tt)[i * TT] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const float* __restrict__ W = wplane + (size_t)c * 4 * P;
    const float* __restrict__ Mu = mupl + (size_t)c * 4 * P;
    int it = i3_chunk_begin(mc, nmc, M);
    const int it1 = have ? i3_chunk_begin(mc + 1, nmc, M) : it;
    bool s_first = true;
    for (;;) {
      const bool more = it < it1;
      if constexpr (Sh::TEAMS > 1) {
        if (!__syncthreads_or(more)) break;
      } else {
        if (!more) break;
      }
      I3Group gr = {0, 0, 0, it, false};
      if (more) gr = i3_group_at(it, it1, M);
      it = gr.next;
      const C2* px = phase + ((size_t)j * M + gr.m) * 2 * n;
      const C2* py = px + n;
      // shifted components of the state, then of the cotangent (component 0 of mu3 is -2 pi mu_0)
#pragma unroll 1
      for (int f = 0; f < 4; ++f) {
        keep_step();
        const int p = f & 1;
        if (more && (f < 2 || gr.pair))
          tm_shift<n>(ln, F, L, team, tt, (f < 2 ? what + ((size_t)c * 4 + p) * P : muh + ((size_t)c * 2 + p) * P), px,
                      py, (f < 2 ? S : Nu) + (size_t)(2 * p) * P, f == 2 ? -1.f : 1.f);
      }
#pragma unroll 1
      for (int q = 0; q < 2; ++q) {
        const bool on = q >= gr.q0 && q < gr.q1;
        const bool first_q = q == gr.q0;
        const float4* __restrict__ Wq = tm_quad(W + (size_t)(2 * q) * P, tt);
        const float4* Sq = tm_quad(S + (size_t)(2 * q) * P, tt);      // rewritten every pair: plain (coherent) loads
        const float4* Nq = tm_quad(Nu + (size_t)(2 * q) * P, tt);
        const float e0 = q == 0 ? 1.f : -1.f;
        C2 v[32];
#pragma unroll 1
        for (int bz = 0; bz < 8; ++bz) {
          keep_step();
          if (!on) continue;
          const int b = bz >> 1;
          const bool z = (bz & 1) != 0;
          const float4* __restrict__ wb = tm_quad(W + (size_t)b * P, tt);
          const float4* __restrict__ mb = tm_quad(Mu + (size_t)b * P, tt);
          const float4* Sb = tm_quad(S + (size_t)b * P, tt);
          const float eb = b == 0 ? 1.f : -1.f;
          if (!z) {   // U = Psi'((w_2q + i w_2q+1) s_b)
#pragma unroll
            for (int g = 0; g < 8; ++g) {
              const float4 sb = Sb[g * TT], wx = Wq[g * TT], wy = Wq[P / 4 + g * TT];
#pragma unroll
              for (int i = 0; i < 4; ++i)
                v[4 * g + i] = mk2(quad_at(wx, i) * quad_at(sb, i), quad_at(wy, i) * quad_at(sb, i));
            }
          } else {    // Z = Psi'(mu_b (eta s)_q + eta_b w_b nu_q)
#pragma unroll
            for (int g = 0; g < 8; ++g) {
              const float4 m4 = mb[g * TT], sx = Sq[g * TT], sy = Sq[P / 4 + g * TT];
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const float m = quad_at(m4, i);
                v[4 * g + i] = mk2(e0 * m * quad_at(sx, i), -m * quad_at(sy, i));
              }
              if (gr.pair) {
                const float4 w4 = wb[g * TT], nx = Nq[g * TT], ny = Nq[P / 4 + g * TT];
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  const float f = eb * quad_at(w4, i);
                  C2& z = v[4 * g + i];
                  z = mk2(fmaf(f, quad_at(nx, i), z.x), fmaf(f, quad_at(ny, i), z.y));
                }
              }
            }
          }
          // the epilogue's operands: mu_b, nu_q or s_b, w_q; the first words before the last stage
          const float4 *o0 = z ? Sb : mb, *o1 = z ? Wq : Nq;
          const bool two = z || gr.pair;
          float4 op[3] = {};
          auto fetch = [&](int g) {
            op[0] = o0[g * TT];
            if (two) {
              op[1] = o1[g * TT];
              op[2] = o1[P / 4 + g * TT];
            }
          };
          tm_convolve<n>(ln, F, psm, L, team, v, [&]() { fetch(0); });
          if constexpr (Sh::TEAMS > 1) fetch(0);
          if (!z) {
            // X_q += mu_b (eta_2q Re U, eta_2q+1 Im U);  R_b += eta_b nu_q . U
            float4* Rb = tm_quad(R + (size_t)b * P, tt);
#pragma unroll
            for (int g = 0; g < 8; ++g) {
              float Vx[4] = {}, Vy[4] = {}, r[4];
              if (b > 0) {
                tmem_ld(tv + 4 * g, Vx);
                tmem_ld(tv + 32 + 4 * g, Vy);
                tmem_wait_ld(Vx);
                tmem_wait_ld(Vy);
              }
              const float4 m4 = op[0], nx = op[1], ny = op[2];
              if (g < 7) fetch(g + 1);
#pragma unroll
              for (int t = 0; t < 4; ++t) {
                const C2 u = v[4 * g + t];
                const float m = quad_at(m4, t);
                Vx[t] = fmaf(e0 * m, u.x, Vx[t]);
                Vy[t] = fmaf(-m, u.y, Vy[t]);
                r[t] = eb * fmaf(quad_at(nx, t), u.x, quad_at(ny, t) * u.y);
              }
              if (gr.pair) red_add4(Rb + g * TT, r[0], r[1], r[2], r[3]);
              tmem_st(tv + 4 * g, Vx);
              tmem_st(tv + 32 + 4 * g, Vy);
            }
            tmem_wait_st();
          } else {
            // R_q += s_b Z;  X_b += w_q . Z
            float4* Rq = tm_quad(R + (size_t)(2 * q) * P, tt);
            float4* Xb = tm_quad(X + (size_t)b * P, tt);
#pragma unroll
            for (int g = 0; g < 8; ++g) {
              const float4 sb = op[0], wx = op[1], wy = op[2];
              if (g < 7) fetch(g + 1);
              float d[4];
#pragma unroll
              for (int i = 0; i < 4; ++i)
                d[i] = fmaf(quad_at(wx, i), v[4 * g + i].x, quad_at(wy, i) * v[4 * g + i].y);
              const C2* u = v + 4 * g;
              red_add4(Rq + g * TT, sb.x * u[0].x, sb.y * u[1].x, sb.z * u[2].x, sb.w * u[3].x);
              red_add4(Rq + P / 4 + g * TT, sb.x * u[0].y, sb.y * u[1].y, sb.z * u[2].y, sb.w * u[3].y);
              if (first_q) Xb[g * TT] = make_float4(d[0], d[1], d[2], d[3]);
              else red_add4(Xb + g * TT, d[0], d[1], d[2], d[3]);
            }
          }
        }
        if (!on) continue;
        tmem_ld_c<32>(tv, tv + 32, v);
        tmem_wait_ld_c<32>(v);
        float4* Xq = tm_quad(X + (size_t)(2 * q) * P, tt);
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          const C2* z = v + 4 * g;
          red_add4(Xq + g * TT, z[0].x, z[1].x, z[2].x, z[3].x);
          red_add4(Xq + P / 4 + g * TT, z[0].y, z[1].y, z[2].y, z[3].y);
        }
      }
      // X shifted back (its sums are in L2: loads that bypass L1)
#pragma unroll 1
      for (int p = 0; p < 2; ++p) {
        keep_step();
        if (!more) continue;
        C2 v[32];
        const float4* Xp = tm_quad(X + (size_t)(2 * p) * P, tt);
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          const float4 x = __ldcg(Xp + g * TT), y = __ldcg(Xp + P / 4 + g * TT);
#pragma unroll
          for (int i = 0; i < 4; ++i) v[4 * g + i] = mk2(quad_at(x, i), quad_at(y, i));
        }
        tm_shift_back<n>(ln, F, L, team, tt, v, px, py, ps + (size_t)p * Q, s_first);
      }
      s_first = false;
    }
    tm_team_sync<n>(team);   // psm is reloaded by the next unit
  }
  tmem_free<Sh::COLS>(tm_base);
}
