// I3 (Hu-Ying term, eq. approxH-JM) in FP32 on padded grids of 32, 64 and 128 points, nodes in pairs
// (i3_staged_fused.cuh), with the line transforms' exchanges in tensor memory.  Included by
// collision_kernels.cuh inside its anonymous namespace.
//
// A team of n / 32 x n threads works on one n x n field: thread (line L of n, h of H = n / 32), each
// with 32 elements of its line in registers.  A line of n = 32 H points is
//   forward:  elements H t1 + h, radix 32 over t1 in registers; exchange; thread h takes
//             k1 in [32 h / H, 32 (h + 1) / H) and the H values t2 of each: twiddles and radix H;
//             frequencies k1 + 32 k2
//   inverse:  the same backwards.
// The H threads of a line sit on the same lane of warps of equal index mod 4, which share a quarter
// of the tensor memory's lanes, so the exchange goes through 2 n of the lane's 512 columns with a
// named barrier of those H warps (none at n = 32).  Columns are written by the thread that read them
// last, or after a team barrier.  H x 64 further columns hold V_q, 64 words per thread.
// A block of 512 threads, one per SM, is one team at n = 128, holds four at 64 and sixteen (a warp
// each) at 32; teams run independent units, so that the loads of one overlap the transforms of
// another.
//
// What bounds it: the kernel it replaces at n = 128 (two register stages of radix 8 and 16, exchanges
// in shared memory) passed the field through the L1 / shared-memory pipe twelve times per convolution
// and kept that pipe 73 % busy with the FMA pipe at 38 %; here only the two transpositions between
// the x and the y lines go through shared memory, four passes (25 %), and the time is the sum of the
// issue slots (55 %) and of the operand loads between them (28 bytes per point and convolution from
// L2), which one team per SM cannot overlap.  Figures: FusedShapes.
//
// The field F[kx][.] between the passes has a row pitch of n + 1: threads of consecutive iy (x pass)
// write F[kx][iy], threads of consecutive kx (y pass) read F[kx][y], both free of bank conflicts.
// Per convolution: x lines forward (lanes = iy, so the loads of the product are coalesced), y lines
// forward, psi'_j, inverse (lanes = kx), x lines inverse; the team synchronises twice.
#pragma once

template <int n>
struct TmShape {
  static constexpr int H = n / 32, JPT = 32 / H;        // threads per line, k1 per thread
  static constexpr int NT = 512, TEAM_THREADS = n * H;
  static constexpr int TEAMS = NT / TEAM_THREADS;       // teams (units at a time) per block: 1, 4, 16
  static constexpr int SPT = n / 32;                    // lane quarters of a team (its lines / 32)
  static constexpr int LS = n + 1;
  static constexpr int EX = H > 1 ? 2 * n : 0;          // exchange columns of a team
  static constexpr int REP = 4 / H;                     // teams stacked on the same lanes
  static constexpr int COLS = REP * (EX + 64 * H);      // 512, 512, 256
  static constexpr size_t tw_bytes = 32 * (sizeof(float4) + sizeof(float2));
  static constexpr size_t team_bytes = (size_t)n * LS * sizeof(float2) + (size_t)n * n * sizeof(float);
  static constexpr size_t smem = tw_bytes + TEAMS * team_bytes;
  static_assert(n == 32 || n == 64 || n == 128, "32 elements per thread, whole teams per block");
  static_assert((COLS & (COLS - 1)) == 0 && COLS <= 512, "tensor memory of one block per SM");
};

template <int n>
struct TmLine {          // one thread's place in the line transforms
  uint32_t ex;           // the team's columns of the thread's lane: the exchange's, then V_q's
  int h, bar;
  const float4* w12;     // [32] exp(-2 pi i k1 / n), exp(-4 pi i k1 / n)
  const float2* w3;      // [32] exp(-6 pi i k1 / n)
};

// The threads of every lane of this warp's 32 have their tcgen05.st done before any loads.
template <int n>
__device__ __forceinline__ void tm_exchange_sync(const TmLine<n>& t) {
  tmem_wait_st();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  asm volatile("bar.sync %0, %1;" ::"r"(t.bar), "n"(32 * TmShape<n>::H) : "memory");
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Team barrier that also orders tensor-memory accesses of the team's threads.
template <int n>
__device__ __forceinline__ void tm_team_sync(int team) {
  if constexpr (n == 32) {
    __syncwarp();
  } else {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(TmShape<n>::TEAM_THREADS) : "memory");
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  }
}

// Forward, first part: v[t1] = element H t1 + h in; b[H j + t2] out, the radix-H inputs of
// k1 = JPT h + j.  (In place: v is b.)
template <int n>
__device__ __forceinline__ void tm_fwd_a(const TmLine<n>& t, float2 (&v)[32]) {
  constexpr int H = TmShape<n>::H, JPT = TmShape<n>::JPT;
  dft<32, -1>(v);
  if constexpr (H > 1) {
    tmem_st_c<32>(t.ex + 64 * t.h, t.ex + 64 * t.h + 32, v);
    tm_exchange_sync(t);
#pragma unroll
    for (int t2 = 0; t2 < H; ++t2)
      tmem_ld_c<JPT, H>(t.ex + 64 * t2 + JPT * t.h, t.ex + 64 * t2 + 32 + JPT * t.h, v + t2);
    tmem_wait_ld_c<32>(v);
  }
}
// Inverse, second part: b[H j + t2] in, v[t1] = element H t1 + h out.  (In place.)
template <int n>
__device__ __forceinline__ void tm_inv_a(const TmLine<n>& t, float2 (&v)[32]) {
  constexpr int H = TmShape<n>::H, JPT = TmShape<n>::JPT;
  if constexpr (H > 1) {
#pragma unroll
    for (int t2 = 0; t2 < H; ++t2)
      tmem_st_c<JPT, H>(t.ex + 64 * t2 + JPT * t.h, t.ex + 64 * t2 + 32 + JPT * t.h, v + t2);
    tm_exchange_sync(t);
    tmem_ld_c<32>(t.ex + 64 * t.h, t.ex + 64 * t.h + 32, v);
    tmem_wait_ld_c<32>(v);
  }
  dft<32, 1>(v);
}
// a + w b and a - w b.
__device__ __forceinline__ void tm_butterfly(float2 a, float2 b, float wx, float wy, float2& p, float2& m) {
  p = mk2(fmaf(wx, b.x, fmaf(-wy, b.y, a.x)), fmaf(wx, b.y, fmaf(wy, b.x, a.y)));
  m = mk2(fmaf(-wx, b.x, fmaf(wy, b.y, a.x)), fmaf(-wx, b.y, fmaf(-wy, b.x, a.y)));
}
// Forward, second part for one k1: twiddles and radix H, b[t2] -> b[k2].
template <int n>
__device__ __forceinline__ void tm_fwd_b(const TmLine<n>& t, int j, float2* b) {
  constexpr int H = TmShape<n>::H, JPT = TmShape<n>::JPT;
  if constexpr (H == 1) return;
  const float4 w = t.w12[JPT * t.h + j];   // w1, w2
  if constexpr (H == 2) {
    float2 p, m;
    tm_butterfly(b[0], b[1], w.x, w.y, p, m);
    b[0] = p;
    b[1] = m;
  } else if constexpr (H == 4) {
    float2 s, d, e, f;
    tm_butterfly(b[0], b[2], w.z, w.w, s, d);
    tm_butterfly(b[1], b[3], w.z, w.w, e, f);
    tm_butterfly(s, e, w.x, w.y, b[0], b[2]);
    tm_butterfly(d, f, w.y, -w.x, b[1], b[3]);   // -i w1
  }
}
// Inverse, first part for one k1: b[k2] -> radix H and conjugate twiddles, b[t2].
template <int n>
__device__ __forceinline__ void tm_inv_twiddle(const TmLine<n>& t, int j, float2* b) {
  constexpr int H = TmShape<n>::H, JPT = TmShape<n>::JPT;
  const float4 w = t.w12[JPT * t.h + j];
  b[1] = cmulc(b[1], mk2(w.x, w.y));
  if constexpr (H == 4) {
    b[2] = cmulc(b[2], mk2(w.z, w.w));
    b[3] = cmulc(b[3], t.w3[JPT * t.h + j]);
  }
}
// sc(k2): real scales of the inputs (SCALED), folded into the first sums: one product and two FMAs per
// component of a pair.
struct TmNoScale {
  __device__ float operator()(int) const { return 1.f; }
};
template <int n, bool SCALED = false, class SC = TmNoScale>
__device__ __forceinline__ void tm_inv_b(const TmLine<n>& t, int j, float2* b, SC sc = SC()) {
  constexpr int H = TmShape<n>::H;
  auto sums = [&](int iu, int ix, float2& p, float2& m) {
    const float2 u = b[iu];
    if constexpr (SCALED) {
      const float cu = sc(iu);
      const float2 x = cscale(b[ix], sc(ix));
      p = mk2(fmaf(u.x, cu, x.x), fmaf(u.y, cu, x.y));
      m = mk2(fmaf(u.x, cu, -x.x), fmaf(u.y, cu, -x.y));
    } else {
      const float2 x = b[ix];
      p = cadd(u, x);
      m = csub(u, x);
    }
  };
  if constexpr (H == 1) {
    if constexpr (SCALED) b[0] = cscale(b[0], sc(0));
  } else if constexpr (H == 2) {
    float2 p, m;
    sums(0, 1, p, m);
    b[0] = p;
    b[1] = m;
    tm_inv_twiddle(t, j, b);
  } else {
    float2 s, d, e, f;
    sums(0, 2, s, d);
    sums(1, 3, e, f);
    b[0] = cadd(s, e);
    b[2] = csub(s, e);
    b[1] = mk2(d.x - f.y, d.y + f.x);
    b[3] = mk2(d.x + f.y, d.y - f.x);
    tm_inv_twiddle(t, j, b);
  }
}
// The Xi frequencies (k < n/4 or k >= 3 n/4) of one k1: XI_PER of them per k1, tm_xi_k(i) the i-th.
template <int n>
struct TmXi {
  static constexpr int PER = TmShape<n>::H == 4 ? 2 : 1;
};
// Whether k1 (at n = 32: any other n has some Xi frequency for every k1) holds one.
template <int n>
__device__ __forceinline__ bool tm_xi_has(int k1) {
  return n > 32 || k1 < 8 || k1 >= 24;
}
template <int n>
__device__ __forceinline__ int tm_xi_k(const TmLine<n>& t, int k1, int i) {
  if constexpr (TmShape<n>::H == 4) return k1 + 96 * i;          // k2 = 0, 3
  else if constexpr (TmShape<n>::H == 2) return k1 + 32 * t.h;   // k1 < 16: k2 = 0, else 1
  else return k1;
}
// tm_inv_b with the Xi frequencies only: x[i] at tm_xi_k(i), the others zero.
template <int n>
__device__ __forceinline__ void tm_inv_b_xi(const TmLine<n>& t, int j, const float2* x, float2* b) {
  constexpr int H = TmShape<n>::H;
  if constexpr (H == 1) {
    b[0] = x[0];
  } else if constexpr (H == 2) {
    b[0] = x[0];
    b[1] = t.h ? mk2(-x[0].x, -x[0].y) : x[0];
    tm_inv_twiddle(t, j, b);
  } else {
    b[0] = cadd(x[0], x[1]);
    b[2] = csub(x[0], x[1]);
    b[1] = mk2(x[0].x + x[1].y, x[0].y - x[1].x);   // x0 - i x3
    b[3] = mk2(x[0].x - x[1].y, x[0].y + x[1].x);
    tm_inv_twiddle(t, j, b);
  }
}
// Output of tm_fwd_b at the i-th Xi frequency.
template <int n>
__device__ __forceinline__ float2 tm_xi_of(const TmLine<n>& t, const float2* b, int i) {
  if constexpr (TmShape<n>::H == 4) return b[3 * i];
  else if constexpr (TmShape<n>::H == 2) return t.h ? b[1] : b[0];
  else return b[0];
}
// The s-th permuted position (of n / 2, ascending) whose frequency lies in Xi.
template <int n>
__device__ __forceinline__ int tm_xi_pos(int s) {
  constexpr int B = Split<n>::B;
  const int k1 = s / (B / 2), t = s % (B / 2);
  return B * k1 + (t < B / 4 ? t : t + B / 2);
}

// Xi line of the thread in the passes over the n / 2 lines of Xi, whose threads L >= n / 2 idle: at
// n = 32 they run along (a line's warp is not split) on line 0 and store nothing.
template <int n>
__device__ __forceinline__ int tm_xi_line(int L) {
  return L < n / 4 ? L : L < n / 2 ? L + n / 2 : 0;
}

// The calling thread's words of a plane in thread_order: elements 4 g .. 4 g + 3 are word g * TEAM_THREADS.
__device__ __forceinline__ float4* tm_quad(float* plane, int tt) { return reinterpret_cast<float4*>(plane) + tt; }
__device__ __forceinline__ const float4* tm_quad(const float* plane, int tt) {
  return reinterpret_cast<const float4*>(plane) + tt;
}

// The shifted pair S (phase-multiplied Xi coefficients `in`, inverse 2-D transform) into planes Sx (times
// sign_x), Sx + P, in thread_order: y lines of the n / 2 lines kx of Xi, then the x lines.  Starts and ends with F free.
template <int n>
__device__ __forceinline__ void tm_shift(const TmLine<n>& ln, float2* F, int L, int team, int tt,
                                         const float2* __restrict__ in, const float2* px, const float2* py,
                                         float* Sx, float sign_x = 1.f) {
  constexpr int LS = TmShape<n>::LS, H = TmShape<n>::H, JPT = TmShape<n>::JPT, P = n * n, PER = TmXi<n>::PER;
  constexpr int TT = TmShape<n>::TEAM_THREADS, X = n / 2;
  const int kxi = tm_xi_line<n>(L);
  for (int e = tt; e < X * X; e += TT) {
    const int xp = tm_xi_pos<n>(e / X), yp = tm_xi_pos<n>(e % X);
    F[freq_of_pos<n>(yp) * LS + freq_of_pos<n>(xp)] = cmul(in[xp * n + yp], cmul(px[xp], py[yp]));
  }
  tm_team_sync<n>(team);
  // Several teams: two passes over one copy of the code (the instruction cache).
#pragma unroll(TmShape<n>::TEAMS == 1 ? 2 : 1)
  for (int pass = 0; pass < 2; ++pass) {
    float2 v[32];
    const bool active = pass == 1 || L < n / 2;     // uniform in a warp where the line has an exchange
    if (H == 1 || active) {
      const float2* src = F + (pass == 0 ? kxi : L * LS);
      const int sk = pass == 0 ? LS : 1;
#pragma unroll
      for (int j = 0; j < JPT; ++j) {
        const int k1 = JPT * ln.h + j;
        float2 x[PER];
#pragma unroll
        for (int i = 0; i < PER; ++i) x[i] = tm_xi_has<n>(k1) ? src[tm_xi_k(ln, k1, i) * sk] : zero2<float>();
        tm_inv_b_xi(ln, j, x, v + H * j);
      }
      tm_inv_a(ln, v);
      if (pass == 0) {
        if (active) {
#pragma unroll
          for (int t1 = 0; t1 < 32; ++t1) F[(H * t1 + ln.h) * LS + kxi] = v[t1];
        }
      } else {
#pragma unroll
        for (int g = 0; g < 8; ++g) {
          const float2* z = v + 4 * g;
          tm_quad(Sx, tt)[g * TT] = make_float4(sign_x * z[0].x, sign_x * z[1].x, sign_x * z[2].x, sign_x * z[3].x);
          tm_quad(Sx + P, tt)[g * TT] = make_float4(z[0].y, z[1].y, z[2].y, z[3].y);
        }
      }
    }
    tm_team_sync<n>(team);
  }
}

// The transform back: the field v (natural order, element H t1 + h of x line L = iy) to its Xi
// coefficients times the conjugate phase, added to (or, with `first`, put into) dst on the kept
// frequencies [sx][sy].  Starts and ends with F free.
template <int n>
__device__ __forceinline__ void tm_shift_back(const TmLine<n>& ln, float2* F, int L, int team, int tt, float2 (&v)[32],
                                              const float2* px, const float2* py, float2* dst, bool first) {
  constexpr int LS = TmShape<n>::LS, H = TmShape<n>::H, JPT = TmShape<n>::JPT, PER = TmXi<n>::PER;
  constexpr int TT = TmShape<n>::TEAM_THREADS, X = n / 2, NQ = xi_kept<n>();
  const int kxi = tm_xi_line<n>(L);
#pragma unroll(TmShape<n>::TEAMS == 1 ? 2 : 1)
  for (int pass = 0; pass < 2; ++pass) {
    const bool active = pass == 0 || L < n / 2;
    if (H == 1 || active) {
      if (pass == 1) {
#pragma unroll
        for (int t1 = 0; t1 < 32; ++t1) v[t1] = F[kxi * LS + H * t1 + ln.h];
      }
      tm_fwd_a(ln, v);
      float2* dst_f = F + (pass == 0 ? L : kxi * LS);
      const int sk = pass == 0 ? LS : 1;
#pragma unroll
      for (int j = 0; j < JPT; ++j) {
        const int k1 = JPT * ln.h + j;
        tm_fwd_b(ln, j, v + H * j);
#pragma unroll
        for (int i = 0; i < PER; ++i)
          if (active && tm_xi_has<n>(k1)) dst_f[tm_xi_k(ln, k1, i) * sk] = tm_xi_of(ln, v + H * j, i);
      }
    }
    tm_team_sync<n>(team);
  }
  for (int e = tt; e < X * X; e += TT) {
    const int xp = tm_xi_pos<n>(e / X), yp = tm_xi_pos<n>(e % X);
    const int sx = xi_slot<n>(xp), sy = xi_slot<n>(yp);
    if (sx >= 0 && sy >= 0) {
      const float2 z = cmulc(F[freq_of_pos<n>(xp) * LS + freq_of_pos<n>(yp)], cmul(px[xp], py[yp]));
      float2* o = dst + sx * NQ + sy;
      *o = first ? z : cadd(*o, z);
    }
  }
  tm_team_sync<n>(team);
}

struct TmNothing {
  __device__ void operator()() const {}
};
// One Psi'_j convolution of the field v (natural order, element H t1 + h of x line L = iy), in place.
// Starts with F free of unread values of other threads; so it ends.
// pre() runs before the last line stage (one team per block: loads whose latency that stage covers).
template <int n, class PRE = TmNothing>
__device__ __forceinline__ void tm_convolve(const TmLine<n>& ln, float2* F, const float* psm, int L, int team,
                                            float2 (&v)[32], PRE pre = PRE()) {
  constexpr int LS = TmShape<n>::LS, H = TmShape<n>::H, JPT = TmShape<n>::JPT;
  auto to_lines_of_y = [&]() {
#pragma unroll
    for (int j = 0; j < JPT; ++j)
#pragma unroll
      for (int k2 = 0; k2 < H; ++k2) F[(JPT * ln.h + j + 32 * k2) * LS + L] = v[H * j + k2];
    tm_team_sync<n>(team);
#pragma unroll
    for (int t1 = 0; t1 < 32; ++t1) v[t1] = F[L * LS + H * t1 + ln.h];
  };
  auto to_lines_of_x = [&]() {
#pragma unroll
    for (int t1 = 0; t1 < 32; ++t1) F[L * LS + H * t1 + ln.h] = v[t1];
    tm_team_sync<n>(team);
#pragma unroll
    for (int j = 0; j < JPT; ++j)
#pragma unroll
      for (int k2 = 0; k2 < H; ++k2) v[H * j + k2] = F[(JPT * ln.h + j + 32 * k2) * LS + L];
  };
  const float* ps = psm + JPT * ln.h * n + L;
  if constexpr (TmShape<n>::TEAMS == 1) {
    tm_fwd_a(ln, v);
#pragma unroll
    for (int j = 0; j < JPT; ++j) tm_fwd_b(ln, j, v + H * j);
    to_lines_of_y();
    tm_fwd_a(ln, v);
#pragma unroll
    for (int j = 0; j < JPT; ++j) {
      tm_fwd_b(ln, j, v + H * j);
      tm_inv_b<n, true>(ln, j, v + H * j, [&](int k2) { return ps[(j + 32 * k2) * n]; });
    }
    tm_inv_a(ln, v);
    to_lines_of_x();
#pragma unroll
    for (int j = 0; j < JPT; ++j) tm_inv_b(ln, j, v + H * j);
    pre();
    tm_inv_a(ln, v);
  } else {
    // one copy of the code each way: several teams share the instruction cache
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
      tm_fwd_a(ln, v);
#pragma unroll
      for (int j = 0; j < JPT; ++j) tm_fwd_b(ln, j, v + H * j);
      if (pass == 0) to_lines_of_y();
    }
#pragma unroll
    for (int j = 0; j < JPT; ++j)
#pragma unroll
      for (int k2 = 0; k2 < H; ++k2) v[H * j + k2] = cscale(v[H * j + k2], ps[(j + 32 * k2) * n]);
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
      for (int j = 0; j < JPT; ++j) tm_inv_b(ln, j, v + H * j);
      tm_inv_a(ln, v);
      if (pass == 0) to_lines_of_x();
    }
  }
}

// Places of the calling thread, its team's shared memory and the twiddles (rounded once, from double).
template <int n>
__device__ __forceinline__ TmLine<n> tm_setup(unsigned char* smem_raw, uint32_t tm_base) {
  float4* w12 = reinterpret_cast<float4*>(smem_raw);
  float2* w3 = reinterpret_cast<float2*>(w12 + 32);
  if (threadIdx.x < 32) {
    double sn, cs;
    float r[6];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      sincospi(-2.0 * (double)((i + 1) * threadIdx.x) / n, &sn, &cs);
      r[2 * i] = (float)cs;
      r[2 * i + 1] = (float)sn;
    }
    w12[threadIdx.x] = make_float4(r[0], r[1], r[2], r[3]);
    w3[threadIdx.x] = mk2(r[4], r[5]);
  }
  __syncthreads();
  const int w = threadIdx.x >> 5;
  TmLine<n> ln;
  const int rep = (w >> 2) / TmShape<n>::H;
  ln.ex = tm_base + ((32u * (w & 3)) << 16) + rep * (TmShape<n>::EX + 64 * TmShape<n>::H);
  ln.h = (w >> 2) % TmShape<n>::H;
  ln.bar = 5 + 4 * rep + (w & 3);   // team barriers: 1 .. 4
  ln.w12 = w12;
  ln.w3 = w3;
  return ln;
}

template <int n>
__global__ void __launch_bounds__(TmShape<n>::NT, 1) k_i3_tmem(const I3Jobs<float> jobs, float2* ws,
                                                              const float2* __restrict__) {
  using C2 = float2;
  using Sh = TmShape<n>;
  constexpr int P = n * n, H = Sh::H, TT = Sh::TEAM_THREADS;
  constexpr int NQ = xi_kept<n>(), Q = NQ * NQ;
  constexpr int D = 1;    // words fetched ahead (n = 128: 1 47.6, 2 48.1, 3 49.0 ms; groups of two fetched at once 49.0)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ uint32_t tm_slot;
  const uint32_t tm_base = tmem_alloc<Sh::COLS>(&tm_slot);
  const TmLine<n> ln = tm_setup<n>(smem_raw, tm_base);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, h = ln.h;
  const int team = (w >> 2) / H * (4 / Sh::SPT) + (w & 3) / Sh::SPT;   // of the block
  const int L = 32 * ((w & 3) % Sh::SPT) + lane;                   // line of the thread
  const int tt = L + n * h;                                        // thread of the team
  C2* F = reinterpret_cast<C2*>(smem_raw + Sh::tw_bytes + team * Sh::team_bytes);   // [n][LS]
  float* psm = reinterpret_cast<float*>(F + n * Sh::LS);           // psi'_j of the current unit, [ky][kx]
  const uint32_t tv = ln.ex + Sh::EX + 64 * h;                     // V_q: real parts, then imaginary parts
  const int slot = team * gridDim.x + blockIdx.x, nslots = gridDim.x * Sh::TEAMS;   // few units: over the blocks first
  float* S = reinterpret_cast<float*>(ws) + (size_t)slot * 4 * P;  // [4][P] shifted components
  // The teams of a block keep step (a block barrier per node group and convolution): one that is a
  // convolution ahead of another evicts its instructions (no_instruction was the largest stall).  n = 64, 128 cells: 15.1 ms out of step,
  // 13.6 ms in step.
  auto keep_step = [&]() {
    if constexpr (Sh::TEAMS > 1) __syncthreads();
  };
  for (int g0 = 0; g0 < jobs.total; g0 += nslots) {
    const bool have = g0 + slot < jobs.total;
    const int gunit = have ? g0 + slot : 0;
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
    if (have) {
      const float* __restrict__ src = jb.psip_s + (size_t)j * P;
      for (int i = tt; i < P; i += Sh::TEAM_THREADS) psm[freq_of_pos<n>(i % n) * n + freq_of_pos<n>(i / n)] = src[i];
    }
    const float* __restrict__ W = jb.wplane + (size_t)c * 4 * P;   // [4][P]
    int it = i3_chunk_begin(mc, nmc, M);
    const int it1 = have ? i3_chunk_begin(mc + 1, nmc, M) : it;
    bool k_first = true, s_first0 = true, s_first1 = true;
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
      if (more) {
#pragma unroll 1
        for (int p = 0; p < 2; ++p)
          tm_shift<n>(ln, F, L, team, tt, what + ((size_t)c * 4 + p) * P, px, py, S + (size_t)(2 * p) * P);
      }
#pragma unroll 1
      for (int q = Sh::TEAMS > 1 ? 0 : gr.q0; q < (Sh::TEAMS > 1 ? 2 : gr.q1); ++q) {
        const bool on = Sh::TEAMS == 1 || (q >= gr.q0 && q < gr.q1);
        const float4* __restrict__ Wq = tm_quad(W + (size_t)(2 * q) * P, tt);
        const float4* Sq = tm_quad(S + (size_t)(2 * q) * P, tt);      // rewritten every pair: plain (coherent) loads
        const float e0 = q == 0 ? 1.f : -1.f;
        C2 v[32];
#pragma unroll 1
        for (int b = 0; b < 4; ++b) {
          keep_step();
          if (!on) continue;
          const float4* __restrict__ wb = tm_quad(W + (size_t)b * P, tt);
          const float4* Sb = tm_quad(S + (size_t)b * P, tt);
          float4* Kb = tm_quad(K + (size_t)b * P, tt);
          // U = Psi'((w_2q + i w_2q+1) s_b)
#pragma unroll
          for (int g = 0; g < 8; ++g) {
            const float4 sb = Sb[g * TT], wx = Wq[g * TT], wy = Wq[P / 4 + g * TT];
#pragma unroll
            for (int i = 0; i < 4; ++i)
              v[4 * g + i] = mk2(quad_at(wx, i) * quad_at(sb, i), quad_at(wy, i) * quad_at(sb, i));
          }
          // the epilogue's operands, D words of each plane ahead
          float4 op[D][3];
          auto fetch = [&](int g) {
            op[g % D][0] = Sq[g * TT];
            op[g % D][1] = Sq[P / 4 + g * TT];
            op[g % D][2] = wb[g * TT];
          };
          tm_convolve<n>(ln, F, psm, L, team, v, [&]() {
#pragma unroll
            for (int g = 0; g < D; ++g) fetch(g);
          });
          if constexpr (Sh::TEAMS > 1) {
#pragma unroll
            for (int g = 0; g < D; ++g) fetch(g);
          }
          // K3_b += eta_2q s_2q Re U + eta_2q+1 s_2q+1 Im U (no other thread adds to this point of the
          // unit's partial: a reduction in memory instead of a load and a store);  V_q += eta_b w_b U
          // (x part of q = 0 with the sign that C_0 has against C_1..C_3, see k_assemble)
          const float eb = b == 0 ? 1.f : -1.f;
#pragma unroll
          for (int g = 0; g < 8; ++g) {
            float Vx[4] = {}, Vy[4] = {}, k[4];
            if (b > 0) {
              tmem_ld(tv + 4 * g, Vx);
              tmem_ld(tv + 32 + 4 * g, Vy);
              tmem_wait_ld(Vx);
              tmem_wait_ld(Vy);
            }
            const float4 sx = op[g % D][0], sy = op[g % D][1], wv = op[g % D][2];
            if (g + D < 8) fetch(g + D);
#pragma unroll
            for (int t = 0; t < 4; ++t) {
              const C2 u = v[4 * g + t];
              k[t] = fmaf(e0 * quad_at(sx, t), u.x, -quad_at(sy, t) * u.y);
              const float f = eb * quad_at(wv, t);
              Vx[t] = fmaf(-e0 * f, u.x, Vx[t]);
              Vy[t] = fmaf(f, u.y, Vy[t]);
            }
            if (k_first) Kb[g * TT] = make_float4(k[0], k[1], k[2], k[3]);
            else red_add4(Kb + g * TT, k[0], k[1], k[2], k[3]);
            tmem_st(tv + 4 * g, Vx);
            tmem_st(tv + 32 + 4 * g, Vy);
          }
          tmem_wait_st();   // V_q is loaded again after the next convolution
        }
        if (!on) continue;
        k_first = false;
        if (!gr.pair) continue;
        tmem_ld_c<32>(tv, tv + 32, v);
        tmem_wait_ld_c<32>(v);
        tm_shift_back<n>(ln, F, L, team, tt, v, px, py, spec + (size_t)q * Q, q == 0 ? s_first0 : s_first1);
        if (q == 0) s_first0 = false;
        else s_first1 = false;
      }
    }
    if (have)
      for (int e = tt; e < Q; e += Sh::TEAM_THREADS) {
        if (s_first0) spec[e] = zero2<float>();
        if (s_first1) spec[Q + e] = zero2<float>();
      }
    tm_team_sync<n>(team);   // psm is reloaded by the next unit
  }
  tmem_free<Sh::COLS>(tm_base);
}
