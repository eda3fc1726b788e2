// I3 (Hu-Ying term, eq. approxH-JM) in FP32 on the padded grid of 96 points, nodes in pairs
// (i3_staged_fused.cuh), two teams of 384 threads per block, each on a unit of its own.  Included by
// collision_kernels.cuh inside its anonymous namespace.
//
// A team's field F[x][y] stays in shared memory (pitch n + 1).  A line of n = A B points takes an A stage
// (t2 fixed, radix A over t1) and a B stage (k1 fixed, radix B over t); a warp's lanes are 32 consecutive
// lines at one t2 or k1, so that every access to F, along x or y, is free of bank conflicts and the
// twiddles are uniform in a warp.  The first A stage multiplies the operands and the last one hands its
// results to the sums, so the field goes through shared memory six times per convolution (k_i3_smem, with
// passes of their own for those: eight times, and a block-wide barrier for each).  Each thread owns the
// same points in both, hence the operands lie in thread_order and V_q in tensor memory.
//
// The two teams keep no common time: the loads of one overlap the transforms of the other.  64 cells of
// N = 48, J = M = 32: 25.2 (k_i3_smem) -> 14.3 ms.
#pragma once

template <int n>
struct LineShape {
  static constexpr int A = Split<n>::A, B = Split<n>::B, LS = n + 1, P = n * n;
  static constexpr int TT = n * B / 2, TEAMS = 2, NT = TT * TEAMS;   // two A tasks per thread
  static constexpr int TA = 2, TB = n * A / TT, X = n / 2;           // tasks per thread, Xi lines
  static constexpr int W = A / 4;                                    // words per task in a plane
  static constexpr int COLS = tmem_columns(NT, 2 * TA * A);
  static constexpr size_t team_bytes = (size_t)n * LS * sizeof(float2) + (size_t)P * sizeof(float);
  static constexpr size_t smem = n * sizeof(float2) + TEAMS * team_bytes;
  static_assert(n * A % TT == 0 && A % 4 == 0 && n % 32 == 0 && X * B == TT && TT % 128 == 0, "whole warps of lines");
};

template <int n>
struct LineTeam {
  using Sh = LineShape<n>;
  static constexpr int A = Sh::A, B = Sh::B, LS = Sh::LS, TT = Sh::TT, TA = Sh::TA, TB = Sh::TB, X = Sh::X;
  float2* F;
  const float2* tw;    // [B k1 + t2] exp(-2 pi i k1 t2 / n)
  const float* psm;    // psi'_j, [pos][line]
  int team, t;
  __device__ __forceinline__ void sync() const {
    asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(TT) : "memory");
  }
  // element e of line L: a row (along y) or a column (along x)
  template <bool ROW>
  __device__ __forceinline__ float2& at(int L, int e) const {
    return ROW ? F[L * LS + e] : F[e * LS + L];
  }
  template <bool ROW>
  __device__ __forceinline__ void put_a(float2 (&v)[A], int L, int t2) const {
    dft<A, -1>(v);
    at<ROW>(L, t2) = v[0];
#pragma unroll
    for (int k1 = 1; k1 < A; ++k1) at<ROW>(L, B * k1 + t2) = cmul(v[k1], tw[B * k1 + t2]);
  }
  template <bool ROW>
  __device__ __forceinline__ void get_a(float2 (&v)[A], int L, int t2) const {
    v[0] = at<ROW>(L, t2);
#pragma unroll
    for (int k1 = 1; k1 < A; ++k1) v[k1] = cmulc(at<ROW>(L, B * k1 + t2), tw[B * k1 + t2]);
    dft<A, 1>(v);
  }
  // the rows' B stage in place; XI: only the frequencies (forward: results, inverse: inputs) of Xi
  template <int DIR, bool XI>
  __device__ __forceinline__ void rows_b() const {
#pragma unroll 1
    for (int i = 0; i < TB; ++i) {
      const int task = t + i * TT, L = task % n, k1 = task / n;
      float2 b[B];
#pragma unroll
      for (int s = 0; s < B; ++s) b[s] = DIR > 0 && XI && !xi_t<B>(s) ? zero2<float>() : at<true>(L, B * k1 + s);
      dft<B, DIR>(b);
#pragma unroll
      for (int s = 0; s < B; ++s)
        if (DIR > 0 || !XI || xi_t<B>(s)) at<true>(L, B * k1 + s) = b[s];
    }
  }
  // One Psi'_j convolution: load(i, v) gives task i's elements, epi(i, v) takes the results at the same points.
  template <class LOAD, class EPI>
  __device__ __forceinline__ void convolve(LOAD load, EPI epi) const {
#pragma unroll 1
    for (int i = 0; i < TA; ++i) {
      float2 v[A];
      load(i, v);
      put_a<true>(v, (t + i * TT) % n, (t + i * TT) / n);
    }
    sync();
    rows_b<-1, false>();
    sync();
#pragma unroll 1
    for (int i = 0; i < TA; ++i) {
      const int L = (t + i * TT) % n, t2 = (t + i * TT) / n;
      float2 v[A];
#pragma unroll
      for (int t1 = 0; t1 < A; ++t1) v[t1] = at<false>(L, B * t1 + t2);
      put_a<false>(v, L, t2);
    }
    sync();
#pragma unroll 1
    for (int i = 0; i < TB; ++i) {
      const int task = t + i * TT, L = task % n, k1 = task / n;
      float2 b[B];
      float sc[B];
#pragma unroll
      for (int s = 0; s < B; ++s) {
        b[s] = at<false>(L, B * k1 + s);
        sc[s] = psm[(B * k1 + s) * n + L];
      }
      dft<B, -1>(b);
      dft_scaled<B, 1>(b, sc);
#pragma unroll
      for (int s = 0; s < B; ++s) at<false>(L, B * k1 + s) = b[s];
    }
    sync();
#pragma unroll 1
    for (int i = 0; i < TA; ++i) {
      const int L = (t + i * TT) % n, t2 = (t + i * TT) / n;
      float2 v[A];
      get_a<false>(v, L, t2);
#pragma unroll
      for (int t1 = 0; t1 < A; ++t1) at<false>(L, B * t1 + t2) = v[t1];
    }
    sync();
    rows_b<1, false>();
    sync();
#pragma unroll 1
    for (int i = 0; i < TA; ++i) {
      float2 v[A];
      get_a<true>(v, (t + i * TT) % n, (t + i * TT) / n);
      epi(i, v);
    }
  }
  // The shifted pair (Xi coefficients `in` times the phase, inverse transform) into the planes Sx, Sx + P.
  __device__ __forceinline__ void shift(const float2* __restrict__ in, const float2* px, const float2* py,
                                        float* Sx) const {
    sync();
#pragma unroll 1
    for (int task = t; task < X * A; task += TT) {
      const int iy = xi_position<n>(task % X), k1 = task / X;
      float2 b[B];
#pragma unroll
      for (int s = 0; s < B; ++s) {
        const int ix = B * k1 + s;
        b[s] = xi_t<B>(s) ? cmul(in[ix * n + iy], cmul(px[ix], py[iy])) : zero2<float>();
      }
      dft<B, 1>(b);
#pragma unroll
      for (int s = 0; s < B; ++s) at<false>(iy, B * k1 + s) = b[s];
    }
    sync();
    {
      const int iy = xi_position<n>(t % X), t2 = t / X;
      float2 v[A];
      get_a<false>(v, iy, t2);
#pragma unroll
      for (int t1 = 0; t1 < A; ++t1) at<false>(iy, B * t1 + t2) = v[t1];
    }
    sync();
    rows_b<1, true>();
    sync();
#pragma unroll 1
    for (int i = 0; i < TA; ++i) {
      float2 v[A];
      get_a<true>(v, (t + i * TT) % n, (t + i * TT) / n);
      float4* S4 = reinterpret_cast<float4*>(Sx) + i * Sh::W * TT + t;
#pragma unroll
      for (int g = 0; g < Sh::W; ++g) {
        const float2* z = v + 4 * g;
        S4[g * TT] = make_float4(z[0].x, z[1].x, z[2].x, z[3].x);
        S4[Sh::P / 4 + g * TT] = make_float4(z[0].y, z[1].y, z[2].y, z[3].y);
      }
    }
  }
  // The transform back of get(i, v): its Xi coefficients times the conjugate phase, added to dst [sx][sy].
  template <class GET>
  __device__ __forceinline__ void shift_back(GET get, const float2* px, const float2* py, float2* dst,
                                             bool first) const {
    constexpr int NQ = xi_kept<n>();
#pragma unroll 1
    for (int i = 0; i < TA; ++i) {
      float2 v[A];
      get(i, v);
      put_a<true>(v, (t + i * TT) % n, (t + i * TT) / n);
    }
    sync();
    rows_b<-1, true>();
    sync();
    {
      const int iy = xi_position<n>(t % X), t2 = t / X;
      float2 v[A];
#pragma unroll
      for (int t1 = 0; t1 < A; ++t1) v[t1] = at<false>(iy, B * t1 + t2);
      put_a<false>(v, iy, t2);
    }
    sync();
#pragma unroll 1
    for (int task = t; task < X * A; task += TT) {
      const int iy = xi_position<n>(task % X), k1 = task / X, sy = xi_slot<n>(iy);
      float2 b[B];
#pragma unroll
      for (int s = 0; s < B; ++s) b[s] = at<false>(iy, B * k1 + s);
      dft<B, -1>(b);
#pragma unroll
      for (int s = 0; s < B; ++s) {
        const int ix = B * k1 + s, sx = xi_t<B>(s) ? xi_slot<n>(ix) : -1;
        if (sx >= 0 && sy >= 0) {
          const float2 z = cmulc(b[s], cmul(px[ix], py[iy]));
          float2* o = dst + sx * NQ + sy;
          *o = first ? z : cadd(*o, z);
        }
      }
    }
    sync();
  }
};

template <int n>
__global__ void __launch_bounds__(LineShape<n>::NT, 1) k_i3_lines(const I3Jobs<float> jobs, float2* ws,
                                                                 const float2* __restrict__ gtw) {
  using C2 = float2;
  using Sh = LineShape<n>;
  constexpr int A = Sh::A, B = Sh::B, P = Sh::P, TT = Sh::TT, TA = Sh::TA, W4 = Sh::W;
  constexpr int NQ = xi_kept<n>(), Q = NQ * NQ;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint32_t tm_slot;
  const uint32_t tm_base = tmem_alloc<Sh::COLS>(&tm_slot);
  const uint32_t tv = tmem_mine<2 * TA * A>(tm_base);   // V_q: per task A real, A imaginary parts
  C2* tw = reinterpret_cast<C2*>(smem_raw);
  for (int pos = threadIdx.x; pos < n; pos += Sh::NT) tw[(pos % A) * B + pos / A] = gtw[pos];
  __syncthreads();
  LineTeam<n> tm;
  tm.team = threadIdx.x / TT;
  tm.t = threadIdx.x % TT;
  tm.tw = tw;
  tm.F = reinterpret_cast<C2*>(smem_raw + n * sizeof(C2) + tm.team * Sh::team_bytes);
  float* psm = reinterpret_cast<float*>(tm.F + n * Sh::LS);
  tm.psm = psm;
  const int slot = tm.team * gridDim.x + blockIdx.x, nslots = gridDim.x * Sh::TEAMS;   // few units: over the blocks first
  float* S = reinterpret_cast<float*>(ws) + (size_t)slot * 4 * P;   // [4][P] shifted components
  auto words = [&](const float* plane) { return reinterpret_cast<const float4*>(plane) + tm.t; };
  for (int gunit = slot; gunit < jobs.total; gunit += nslots) {
    const I3Job<float>& jb = jobs.job[i3_job_of(jobs, gunit)];
    const int unit = gunit - jb.unit_begin;
    const int J = jb.J, M = jb.M, nmc = jb.nmc;
    const C2* what = jb.what;
    const C2* __restrict__ phase = jb.phase;
    const int c = unit / (J * nmc);
    const int j = (unit / nmc) % J;
    const int mc = unit % nmc;
    float* K = reinterpret_cast<float*>(jb.K3part + (size_t)unit * 2 * P);   // [4][P], thread_order
    C2* spec = jb.K3spec + (size_t)unit * 2 * Q;
    const float4* src = reinterpret_cast<const float4*>(jb.psip_s + (size_t)j * P);
    for (int i = tm.t; i < P / 4; i += TT) reinterpret_cast<float4*>(psm)[i] = src[i];
    const float* __restrict__ Wp = jb.wplane + (size_t)c * 4 * P;
    const int it1 = i3_chunk_begin(mc + 1, nmc, M);
    bool k_first = true, s_first0 = true, s_first1 = true;
    for (int it = i3_chunk_begin(mc, nmc, M); it < it1;) {
      const I3Group gr = i3_group_at(it, it1, M);
      it = gr.next;
      const C2* px = phase + ((size_t)j * M + gr.m) * 2 * n;
      const C2* py = px + n;
#pragma unroll 1
      for (int p = 0; p < 2; ++p) tm.shift(what + ((size_t)c * 4 + p) * P, px, py, S + (size_t)(2 * p) * P);
#pragma unroll 1
      for (int q = gr.q0; q < gr.q1; ++q) {
        const float4* __restrict__ Wq = words(Wp + (size_t)(2 * q) * P);
        const float4* Sq = words(S + (size_t)(2 * q) * P);      // rewritten every pair: plain (coherent) loads
        const float e0 = q == 0 ? 1.f : -1.f;
#pragma unroll 1
        for (int b = 0; b < 4; ++b) {
          const float4* __restrict__ wb = words(Wp + (size_t)b * P);
          const float4* Sb = words(S + (size_t)b * P);
          float4* Kb = reinterpret_cast<float4*>(K + (size_t)b * P) + tm.t;
          const float eb = b == 0 ? 1.f : -1.f;
          tm.convolve(
              [&](int i, C2 (&v)[A]) {   // U = Psi'((w_2q + i w_2q+1) s_b)
#pragma unroll
                for (int g = 0; g < W4; ++g) {
                  const int e = (i * W4 + g) * TT;
                  const float4 sb = Sb[e], wx = Wq[e], wy = Wq[P / 4 + e];
#pragma unroll
                  for (int s = 0; s < 4; ++s)
                    v[4 * g + s] = mk2(quad_at(wx, s) * quad_at(sb, s), quad_at(wy, s) * quad_at(sb, s));
                }
              },
              // K3_b += eta_2q s_2q Re U + eta_2q+1 s_2q+1 Im U (no other thread adds to these points);
              // V_q += eta_b w_b U (x part of q = 0 with the sign that C_0 has against C_1..C_3, see k_assemble)
              [&](int i, C2 (&v)[A]) {
                const uint32_t tvi = tv + 2 * A * i;
#pragma unroll
                for (int g = 0; g < W4; ++g) {
                  const int e = (i * W4 + g) * TT;
                  const float4 sx = Sq[e], sy = Sq[P / 4 + e], wv = wb[e];
                  float Vx[4] = {}, Vy[4] = {}, k[4];
                  if (b > 0) {
                    tmem_ld(tvi + 4 * g, Vx);
                    tmem_ld(tvi + A + 4 * g, Vy);
                    tmem_wait_ld(Vx);
                    tmem_wait_ld(Vy);
                  }
#pragma unroll
                  for (int s = 0; s < 4; ++s) {
                    const C2 u = v[4 * g + s];
                    k[s] = fmaf(e0 * quad_at(sx, s), u.x, -quad_at(sy, s) * u.y);
                    const float f = eb * quad_at(wv, s);
                    Vx[s] = fmaf(-e0 * f, u.x, Vx[s]);
                    Vy[s] = fmaf(f, u.y, Vy[s]);
                  }
                  if (k_first) Kb[e] = make_float4(k[0], k[1], k[2], k[3]);
                  else red_add4(Kb + e, k[0], k[1], k[2], k[3]);
                  tmem_st(tvi + 4 * g, Vx);
                  tmem_st(tvi + A + 4 * g, Vy);
                }
                tmem_wait_st();   // V_q is loaded again after the next convolution
              });
        }
        k_first = false;
        if (!gr.pair) continue;
        tm.shift_back(
            [&](int i, C2 (&v)[A]) {
              float Vx[A], Vy[A];
              tmem_ld(tv + 2 * A * i, Vx);
              tmem_ld(tv + 2 * A * i + A, Vy);
              tmem_wait_ld(Vx);
              tmem_wait_ld(Vy);
#pragma unroll
              for (int t1 = 0; t1 < A; ++t1) v[t1] = mk2(Vx[t1], Vy[t1]);
            },
            px, py, spec + (size_t)q * Q, q == 0 ? s_first0 : s_first1);
        if (q == 0) s_first0 = false;
        else s_first1 = false;
      }
    }
    for (int e = tm.t; e < Q; e += TT) {
      if (s_first0) spec[e] = zero2<float>();
      if (s_first1) spec[Q + e] = zero2<float>();
    }
    tm.sync();   // psm is reloaded by the next unit
  }
  tmem_free<Sh::COLS>(tm_base);
}
