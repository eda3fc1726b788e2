// I3 (Hu-Ying term, eq. approxH-JM) for fields larger than one block's shared memory (the FP64 form):
// the radial nodes taken in pairs +-rho_m, staged row and line passes with every global load and
// store fused into a line stage.  Included by collision_kernels.cuh inside its anonymous namespace.
//
// Node pairs.  With S the shift by node m (rho_m < 0) and S* = S^-1 that of its partner M-1-m (the
// Gauss-Legendre nodes are symmetric, with equal weights), write s_a = S w_a.  Translations commute
// with Psi'_j and with products, so
//   sum_a eta_a S*w_a Psi'(w_a S*w_b) = S*[ sum_a eta_a w_a Psi'(s_a w_b) ]
// and both nodes of the pair use the same sixteen real convolutions U_ab = Psi'(w_a s_b):
//   node m:      K3_b += sum_a eta_a s_a U_ab          (real space)
//   node M-1-m:  K3_a += S*[ sum_b eta_b w_b U_ab ]    (Fourier space, on the kept frequencies)
// The product of three Xi-limited fields aliases only outside Xi on the padded grid and Xi is all that
// the final projection keeps, so the regrouping is exact up to rounding.  Per pair: 2 shifts, 8 complex
// convolutions, 2 transforms back, against 4 shifts and 16 convolutions node by node.  The middle node
// of an odd M (rho = 0) has no partner.
//
// What bounds it: FP64 issue (two lanes per clock and SM); the scratch traffic through L2 is nearly
// free beside it.  I3 launch, J = M = 32, on a GB300, node by node -> in pairs: see i3_default_variant.
//
// The block's scratch field between the passes is stored transposed, G'[ky][x] (ky in the row
// transform's permuted order), so that each pass reads and writes it with coalesced accesses
// straight from its line stages:
//   row pass, forward:  stage A loads the product (tasks (row, t2), t2-fastest), stage B stores its
//                       B spectral values of a row into B lines of G' (lanes = consecutive rows);
//   line pass (x):      stage A loads a line of G' (contiguous in x), stage B with the psi'_j
//                       multiplier between forward and inverse, stage A stores the line back;
//   row pass, inverse:  stage B loads B lines of G' at its row (lanes = consecutive rows), stage A
//                       hands its results to the accumulations.
// The shifts run the lines and then the rows, the transforms back the rows and then the lines, both
// with the n / 2 lines of Xi only and with the Xi values only of each spectral stage (xi_t).
// Shared memory holds one chunk at a time; no pass copies a chunk through it without transforming.
#pragma once

// The passes of one block on its scratch field G', with one chunk sm of shared memory.
template <int n, class T, int NTH, int CB>
struct StagedLines {
  using C2 = typename Vec2Of<T>::type;
  static constexpr int A = Split<n>::A, B = Split<n>::B, P = n * n;
  static constexpr int RC = Chunk<n, sizeof(C2), CB>::RC, CC = Chunk<n, sizeof(C2), CB>::CC,
                       LS = Chunk<n, sizeof(C2), CB>::LS;
  static constexpr int NQ = xi_kept<n>(), Q = NQ * NQ;
  static_assert(RC == CC, "row and line chunks share the buffer");
  // FP64: twiddles merged into the second stage of a line (dft_merged), forward [k1][B - 1] (a warp shares k1,
  // and k1 = 0 has none), inverse [A - 1][t2] (t2-fastest lanes).  A 128-point line takes 2324 (forward) and
  // 2336 instead of 2464 FP64 instructions, and the FP64 pipe is what bounds these kernels: k_i3_sf took
  // 423.6 -> 389.4 ms (32 cells at N = 64, J = M = 32), 365.3 -> 330.5 (128 cells, N = 32), 486.7 -> 466.6
  // (64 cells, N = 48, whose radix-12 inverse keeps its products), the transpose 415 -> 381 (16 cells, N = 64).
  // FP32 keeps the products, [k1][t2]: a merged line alone rounds 8-13% worse (FP32, n = 16..128).
  static constexpr bool kMergeB = sizeof(T) == 8, kMergeA = kMergeB && (A & (A - 1)) == 0;
  static constexpr int kTwF = kMergeB ? A * (B - 1) : 0, kTwI = kMergeA ? (A - 1) * B : n;
  C2* twF;
  C2* twI;
  C2* sm;            // one chunk: [RC][LS] rows, or [CC][LS] lines of G'
  const int* kslot;  // [n] xi_slot
  C2* G;             // G'[ky][x] between the passes

  // the li-th of the n / 2 lines ky of Xi: its permuted position
  __device__ __forceinline__ static int xi_line(int li) {
    const int k1 = li / (B / 2), t = li % (B / 2);
    return B * k1 + (t < B / 4 ? t : t + B / 2);
  }
  __device__ __forceinline__ void init(C2* smem) {
    twF = smem;
    twI = twF + kTwF;
    sm = twI + kTwI;
    for (int i = threadIdx.x; i < kTwF; i += NTH) twF[i] = root(-merged_exponent<B>(i % (B - 1), i / (B - 1), A));
    for (int i = threadIdx.x; i < kTwI; i += NTH)
      twI[i] = kMergeA ? root(merged_exponent<A>(i / B, i % B, B)) : root(-(i / B) * (i % B));
  }
  // between the stages of a forward line
  __device__ __forceinline__ void twiddle_forward(C2 (&v)[A], int t2) const {
    if constexpr (!kMergeB) {
#pragma unroll
      for (int k1 = 1; k1 < A; ++k1) v[k1] = cmul(v[k1], twI[k1 * B + t2]);
    }
  }
  __device__ static C2 root(int m) {   // exp(2 pi i m / n)
    double sn, cs;
    sincospi(2.0 * (double)m / n, &sn, &cs);
    return mk2((T)cs, (T)sn);
  }
  // second stage of a forward line: b[t2] -> spectrum values of k1 + A (0..B-1)
  __device__ __forceinline__ void stage_b_forward(C2 (&b)[B], int k1) const {
    if (!kMergeB || k1 == 0) {
      dft<B, -1>(b);
    } else {
      const C2* w = twF + k1 * (B - 1);
      dft_merged<B>(b, [&](int e) { return w[e]; });
    }
  }
  // second stage of an inverse line: v[k1] -> elements B (0..A-1) + t2
  __device__ __forceinline__ void stage_a_inverse(C2 (&v)[A], int t2) const {
    if constexpr (kMergeA) {
      const C2* w = twI + t2;
      dft_merged<A>(v, [&](int e) { return w[e * B]; });
    } else {
#pragma unroll
      for (int k1 = 1; k1 < A; ++k1) v[k1] = cmulc(v[k1], twI[k1 * B + t2]);
      dft<A, 1>(v);
    }
  }
  // rows of load(idx), idx = row * n + y, into lines of G' (XI: into the Xi lines only)
  template <bool XI, class LOAD>
  __device__ __forceinline__ void rows_forward(LOAD load) const {
    const int tid = threadIdx.x;
    for (int r0 = 0; r0 < n; r0 += RC) {
      for (int task = tid; task < RC * B; task += NTH) {
        const int r = task / B, t2 = task % B;
        C2 v[A];
#pragma unroll
        for (int t1 = 0; t1 < A; ++t1) v[t1] = load((r0 + r) * n + B * t1 + t2);
        dft<A, -1>(v);
        twiddle_forward(v, t2);
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) sm[r * LS + B * k1 + t2] = v[k1];
      }
      __syncthreads();
      for (int task = tid; task < RC * A; task += NTH) {
        const int r = task % RC, k1 = task / RC;
        const C2* base = sm + r * LS + B * k1;
        C2 b[B];
#pragma unroll
        for (int t = 0; t < B; ++t) b[t] = base[t];
        stage_b_forward(b, k1);
#pragma unroll
        for (int t = 0; t < B; ++t)
          if (!XI || xi_t<B>(t)) G[(B * k1 + t) * n + r0 + r] = b[t];
      }
      __syncthreads();
    }
  }
  // rows of G' back to real space, handed to epi(idx, v) (XI: only the Xi lines are non-zero)
  template <bool XI, class EPI>
  __device__ __forceinline__ void rows_inverse(EPI epi) const {
    const int tid = threadIdx.x;
    for (int r0 = 0; r0 < n; r0 += RC) {
      for (int task = tid; task < RC * A; task += NTH) {
        const int r = task % RC, k1 = task / RC;
        C2* base = sm + r * LS + B * k1;
        C2 b[B];
#pragma unroll
        for (int t = 0; t < B; ++t) b[t] = (!XI || xi_t<B>(t)) ? G[(B * k1 + t) * n + r0 + r] : zero2<T>();
        if constexpr (XI) dft_xi<B, 1>(b);
        else dft<B, 1>(b);
#pragma unroll
        for (int t = 0; t < B; ++t) base[t] = b[t];
      }
      __syncthreads();
      for (int task = tid; task < RC * B; task += NTH) {
        const int r = task / B, t2 = task % B;
        C2 v[A];
#pragma unroll
        for (int k1 = 0; k1 < A; ++k1) v[k1] = sm[r * LS + B * k1 + t2];
        stage_a_inverse(v, t2);
#pragma unroll
        for (int t1 = 0; t1 < A; ++t1) epi((r0 + r) * n + B * t1 + t2, v[t1]);
      }
      __syncthreads();
    }
  }
  // stage A of lines in shared memory, back into G' (inverse)
  __device__ __forceinline__ void lines_out(int nl, int c0, bool xi) const {
    for (int task = threadIdx.x; task < nl * B; task += NTH) {
      const int cc = task / B, t2 = task % B, ky = xi ? xi_line(c0 + cc) : c0 + cc;
      C2 v[A];
#pragma unroll
      for (int k1 = 0; k1 < A; ++k1) v[k1] = sm[cc * LS + B * k1 + t2];
      stage_a_inverse(v, t2);
#pragma unroll
      for (int t1 = 0; t1 < A; ++t1) G[ky * n + B * t1 + t2] = v[t1];
    }
    __syncthreads();
  }
  // stage A of lines of G' into shared memory (forward)
  __device__ __forceinline__ void lines_in(int nl, int c0, bool xi) const {
    for (int task = threadIdx.x; task < nl * B; task += NTH) {
      const int cc = task / B, t2 = task % B, ky = xi ? xi_line(c0 + cc) : c0 + cc;
      C2 v[A];
#pragma unroll
      for (int t1 = 0; t1 < A; ++t1) v[t1] = G[ky * n + B * t1 + t2];
      dft<A, -1>(v);
      twiddle_forward(v, t2);
#pragma unroll
      for (int k1 = 0; k1 < A; ++k1) sm[cc * LS + B * k1 + t2] = v[k1];
    }
    __syncthreads();
  }
  // Psi'_j of the field load(idx), handed to epi(idx, v)
  template <class LOAD, class EPI>
  __device__ __forceinline__ void convolve(const T* __restrict__ psp, LOAD load, EPI epi) const {
    rows_forward<false>(load);
    for (int c0 = 0; c0 < n; c0 += CC) {
      lines_in(CC, c0, false);
      for (int task = threadIdx.x; task < CC * A; task += NTH) {
        const int cc = task % CC, k1 = task / CC;
        C2* base = sm + cc * LS + B * k1;
        C2 z[B];
#pragma unroll
        for (int t = 0; t < B; ++t) z[t] = base[t];
        stage_b_forward(z, k1);
        T sc[B];
#pragma unroll
        for (int t = 0; t < B; ++t) sc[t] = psp[(B * k1 + t) * n + c0 + cc];
        dft_scaled<B, 1>(z, sc);
#pragma unroll
        for (int t = 0; t < B; ++t) base[t] = z[t];
      }
      __syncthreads();
      lines_out(CC, c0, false);
    }
    rows_inverse<false>(epi);
  }
  // The shift S of the Xi coefficients `in`, handed to epi(idx, v): the Xi lines along x, then the rows
  template <class EPI>
  __device__ __forceinline__ void shift(const C2* in, const C2* px, const C2* py, EPI epi) const {
    for (int c0 = 0; c0 < n / 2; c0 += CC) {
      const int nl = (n / 2 - c0) < CC ? (n / 2 - c0) : CC;
      for (int task = threadIdx.x; task < nl * A; task += NTH) {
        const int cc = task % nl, k1 = task / nl, ky = xi_line(c0 + cc);
        const C2 pyy = py[ky];
        C2* base = sm + cc * LS + B * k1;
        C2 b[B];
#pragma unroll
        for (int t = 0; t < B; ++t)
          b[t] = xi_t<B>(t) ? cmul(in[(B * k1 + t) * n + ky], cmul(px[B * k1 + t], pyy)) : zero2<T>();
        dft_xi<B, 1>(b);
#pragma unroll
        for (int t = 0; t < B; ++t) base[t] = b[t];
      }
      __syncthreads();
      lines_out(nl, c0, true);
    }
    rows_inverse<true>(epi);
  }
  // The shift back S* of the field load(idx): rows, then the Xi lines along x, times the conjugate phase,
  // added to (or, with `first`, put into) dst on the kept frequencies
  template <class LOAD>
  __device__ __forceinline__ void shift_back(const C2* px, const C2* py, C2* dst, bool first, LOAD load) const {
    rows_forward<true>(load);
    for (int c0 = 0; c0 < n / 2; c0 += CC) {
      const int nl = (n / 2 - c0) < CC ? (n / 2 - c0) : CC;
      lines_in(nl, c0, true);
      for (int task = threadIdx.x; task < nl * A; task += NTH) {
        const int cc = task % nl, k1 = task / nl, ky = xi_line(c0 + cc), sy = kslot[ky];
        const C2* base = sm + cc * LS + B * k1;
        C2 b[B];
#pragma unroll
        for (int t = 0; t < B; ++t) b[t] = base[t];
        stage_b_forward(b, k1);
        if (sy < 0) continue;
        const C2 pyy = py[ky];
#pragma unroll
        for (int t = 0; t < B; ++t)
          if (xi_t<B>(t)) {
            const int sx = kslot[B * k1 + t];
            if (sx >= 0) {
              const C2 z = cmulc(b[t], cmul(px[B * k1 + t], pyy));
              C2* o = dst + sx * NQ + sy;
              *o = first ? z : cadd(*o, z);
            }
          }
      }
      __syncthreads();
    }
  }
};

template <int n, class T, int NTH, int CB, int MINB>
__global__ void __launch_bounds__(NTH, MINB)
    k_i3_sf(const I3Jobs<T> jobs, typename Vec2Of<T>::type* ws, const typename Vec2Of<T>::type* __restrict__) {
  using C2 = typename Vec2Of<T>::type;
  using Lines = StagedLines<n, T, NTH, CB>;
  constexpr int P = n * n, Q = Lines::Q;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int kslot[n];
  C2* slot = ws + (size_t)blockIdx.x * 4 * P;
  C2* Sig = slot;           // [2][P] shifted pairs s_0 + i s_1, s_2 + i s_3
  C2* V = slot + 3 * P;     // sum_b eta_b w_b U_ab of the current pair of a
  Lines ln;
  ln.init(reinterpret_cast<C2*>(smem_raw));
  ln.kslot = kslot;
  ln.G = slot + 2 * P;
  build_xi_slots<n>(kslot);
  for (int gunit = blockIdx.x; gunit < jobs.total; gunit += gridDim.x) {
    const I3Job<T>& jb = jobs.job[i3_job_of(jobs, gunit)];
    const int unit = gunit - jb.unit_begin;
    const int J = jb.J, M = jb.M, nmc = jb.nmc;
    const C2* what = jb.what;
    const C2* __restrict__ phase = jb.phase;
    const int c = unit / (J * nmc);
    const int j = (unit / nmc) % J;
    const int mc = unit % nmc;
    T* K = reinterpret_cast<T*>(jb.K3part + (size_t)unit * 2 * P);   // [4][P]
    C2* spec = jb.K3spec + (size_t)unit * 2 * Q;
    const T* __restrict__ psp = jb.psip_s + (size_t)j * P;
    const C2* wf = jb.wfine + (size_t)c * 2 * P;
    const int it1 = i3_chunk_begin(mc + 1, nmc, M);
    bool k_first = true, s_first[2] = {true, true};
    for (int it = i3_chunk_begin(mc, nmc, M); it < it1;) {
      const I3Group gr = i3_group_at(it, it1, M);
      it = gr.next;
      const C2* px = phase + ((size_t)j * M + gr.m) * 2 * n;
      const C2* py = px + n;
      for (int p = 0; p < 2; ++p) {
        C2* S = Sig + (size_t)p * P;
        ln.shift(what + ((size_t)c * 4 + p) * P, px, py, [&](int idx, C2 v) { S[idx] = v; });
      }
      for (int q = gr.q0; q < gr.q1; ++q) {
        const C2* wq = wf + (size_t)q * P;
        const C2* Sq = Sig + (size_t)q * P;
        for (int b = 0; b < 4; ++b) {
          // U_{2q,b} + i U_{2q+1,b} = Psi'((w_2q + i w_2q+1) s_b);
          // K3_b += eta_2q s_2q Re U + eta_2q+1 s_2q+1 Im U;  V_q += eta_b w_b U (x part of q = 0 with the
          // sign that C_0 has against C_1..C_3, see k_assemble)
          const T* Sb = reinterpret_cast<const T*>(Sig + (size_t)(b >> 1) * P) + (b & 1);
          const T* wb = reinterpret_cast<const T*>(wf + (size_t)(b >> 1) * P) + (b & 1);
          T* Kb = K + (size_t)b * P;
          const T e0 = q == 0 ? (T)1 : (T)-1, eb = b == 0 ? (T)1 : (T)-1;
          ln.convolve(
              psp, [&](int idx) { return cscale(wq[idx], Sb[2 * idx]); },
              [&](int idx, C2 v) {
                const C2 s = Sq[idx];
                const T k = fmaT(e0 * s.x, v.x, -s.y * v.y);
                Kb[idx] = k_first ? k : Kb[idx] + k;
                if (gr.pair) {
                  const T f = eb * wb[2 * idx], fx = -e0 * f;
                  if (b == 0) {
                    V[idx] = mk2(fx * v.x, f * v.y);
                  } else {
                    const C2 d = V[idx];
                    V[idx] = mk2(fmaT(fx, v.x, d.x), fmaT(f, v.y, d.y));
                  }
                }
              });
        }
        k_first = false;
        if (!gr.pair) continue;
        ln.shift_back(px, py, spec + (size_t)q * Q, s_first[q], [&](int idx) { return V[idx]; });
        s_first[q] = false;
      }
    }
    for (int q = 0; q < 2; ++q)
      if (s_first[q]) zero_fields(spec + (size_t)q * Q, Q);
  }
}

template <int n, class T, int CB>
constexpr size_t i3_sf_smem_bytes() {   // twiddles and one chunk of RC padded lines
  using L = StagedLines<n, T, 256, CB>;
  return (size_t)(L::kTwF + L::kTwI + L::RC * L::LS) * sizeof(typename L::C2);
}
