// Block-level FFT building blocks for the spectral collision operator.
//
// A length-n DFT (n = A*B) is done in two in-place stages on a line of
// double2 values (Cooley-Tukey "four-step" split, no reordering pass):
//   t = B*t1 + t2,  k = k1 + A*k2
//   forward: X[k1 + A k2] = sum_t2 e^{-2pi i t2 k2/B} [ e^{-2pi i t2 k1/n} sum_t1 e^{-2pi i t1 k1/A} x[B t1 + t2] ]
// Stage 1 reads positions B*t1 + t2 and writes back to the same positions
// (holding index k1 at B*k1 + t2); stage 2 reads the B contiguous values at
// B*k1 + (0..B-1) and writes them back in place.  The spectrum therefore sits
// in the "permuted" order pos(k) = B*(k mod A) + (k div A).  The inverse runs
// the two stages backwards and takes permuted input to natural output.  All
// spectral-space tables of the library are stored in this permuted order.
//
// Sign convention: forward = sum x e^{-2 pi i ...}, inverse = sum X e^{+2 pi i ...},
// both unnormalised.
#pragma once

#include <cuda_runtime.h>

namespace qbe {

template <int n> struct Split;
template <> struct Split<16>  { static constexpr int A = 4,  B = 4;  };
template <> struct Split<32>  { static constexpr int A = 4,  B = 8;  };
template <> struct Split<64>  { static constexpr int A = 8,  B = 8;  };
template <> struct Split<128> { static constexpr int A = 8,  B = 16; };
template <> struct Split<256> { static constexpr int A = 16, B = 16; };
template <> struct Split<96>  { static constexpr int A = 12, B = 8;  };
template <> struct Split<192> { static constexpr int A = 12, B = 16; };

// Planes whose points only their own thread reads are stored in the thread order of the FP32 I3 kernel of
// their size: 16-byte words of four elements of a thread, consecutive threads side by side.
//   n = 96 (k_i3_lines): thread t of 384 holds, in task i = 0, 1, the elements y = 8 t1 + t2 of line x, where
//   96 t2 + x = t + 384 i;
//   n = 32, 64, 128 = 32 H (k_i3_tmem): thread y + n h holds the elements x = H t1 + h of line y;
//   n > 128 (k_i3_cluster): block x / R of four holds R rows; thread t of its NT = R B / 2 holds, in each of
//   its two tasks r B + t2 = t + i NT, the elements y = B t1 + t2 of row r.
// Words of a plane: the point x n + y of the first element and the step to the next three.
struct ThreadWord {
  int first, step;
};
__host__ __device__ __forceinline__ ThreadWord thread_word(int n, int word) {
  if (n == 96) {
    const int ig = word / 384, task = word % 384 + ig / 3 * 384;
    return {task % n * n + 8 * (ig % 3 * 4) + task / n, 8};
  }
  if (n <= 128) {
    const int H = n / 32, t = word % (n * H);
    return {(H * (word / (n * H) * 4) + t / n) * n + t % n, H * n};
  }
  const int B = 16, A4 = n / B / 4, R = n / 4, NT = R * B / 2;
  const int block = word / (R * n / 4), w = word % (R * n / 4), ig = w / NT, task = w % NT + ig / A4 * NT;
  return {(block * R + task / B) * n + B * (ig % A4 * 4) + task % B, B};
}
// Place of point (x, y).
template <int n>
__host__ __device__ __forceinline__ int thread_order(int x, int y) {
  if constexpr (n == 96) {
    const int task = y % 8 * n + x, t1 = y / 8;
    return ((task / 384 * 3 + t1 / 4) * 384 + task % 384) * 4 + t1 % 4;
  } else if constexpr (n <= 128) {
    constexpr int H = n < 32 ? 1 : n / 32;
    const int t1 = x / H;
    return ((t1 / 4) * n * H + y + n * (x % H)) * 4 + t1 % 4;
  } else {
    constexpr int A = Split<n>::A, B = Split<n>::B, R = n / 4, NT = R * B / 2;
    const int task = x % R * B + y % B, t1 = y / B;
    return x / R * R * n + ((task / NT * (A / 4) + t1 / 4) * NT + task % NT) * 4 + t1 % 4;
  }
}

// Frequency index (0..n-1, standard wrap) stored at permuted position pos.
template <int n>
__host__ __device__ __forceinline__ int freq_of_pos(int pos) {
  constexpr int A = Split<n>::A, B = Split<n>::B;
  return pos / B + A * (pos % B);
}
// Permuted position of frequency index k.
template <int n>
__host__ __device__ __forceinline__ int pos_of_freq(int k) {
  constexpr int A = Split<n>::A, B = Split<n>::B;
  return B * (k % A) + k / A;
}

// The team of a pass: the blocks of a cluster (a plain launch is a cluster of one).  Its blocks share
// the chunks of every pass, and data that one block writes and another reads goes through L2 between
// cluster barriers (release / acquire at cluster scope; the reads of teams of several blocks bypass L1: ldc).
__device__ __forceinline__ int cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return (int)r;
}
__device__ __forceinline__ int cluster_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return (int)r;
}
__device__ __forceinline__ int cluster_index() {
  unsigned r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return (int)r;
}
__device__ __forceinline__ int cluster_count() {
  unsigned r;
  asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
  return (int)r;
}
// All threads of all blocks of the cluster.
__device__ __forceinline__ void cluster_sync_global() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void team_sync() {
  if (cluster_size() > 1) cluster_sync_global();
  else __syncthreads();
}
// Chunk bytes of the per-cell kernels: one block per team takes 64 KB chunks; in a team of several
// blocks a chunk is n / 8 rows or columns, so that up to 8 blocks share a pass.
constexpr int kCellCB = 65536;
template <int n, class C>
__host__ __device__ constexpr int team_cb() {
  return n * (n / 8) * (int)sizeof(C);
}
// Whether a kernel of these chunks is launched with one block per team only: it needs no rank, no cluster
// barrier, and reads its own writes through L1 (up to n = 64; larger fields only evict what L1 holds).  At
// small n a pass is little more than its latency, and the ranks read and L1 bypassed in every pass took up to
// a third of a kernel: FP32, 100 blocks, n = 16 k_i1_vjp 29.1 -> 21.2 us, k_i24_vjp 38.6 -> 26.9; n = 32
// k_i24_vjp 58.4 -> 46.4; FP64, n = 16 128.4 -> 116.6.
template <int n, class C, int CB>
__host__ __device__ constexpr bool lone_block() {
  return CB == kCellCB && team_cb<n, C>() != kCellCB;
}
// Load of what the team has written.
template <int n, int CB, class C>
__device__ __forceinline__ C ldc(const C* p) {
  if constexpr (lone_block<n, C, CB>() && n <= 64) return *p;
  else return __ldcg(p);
}
// Rank and size of the team that shares the chunks of a pass.
template <int n, class C, int CB>
__device__ __forceinline__ int pass_rank() {
  if constexpr (lone_block<n, C, CB>()) return 0;
  else return cluster_rank();
}
template <int n, class C, int CB>
__device__ __forceinline__ int pass_ranks() {
  if constexpr (lone_block<n, C, CB>()) return 1;
  else return cluster_size();
}
// Element loops shared by the team: for (i = element_first(); i < count; i += element_stride()).
__device__ __forceinline__ int element_first() { return cluster_rank() * blockDim.x + threadIdx.x; }
__device__ __forceinline__ int element_stride() { return cluster_size() * blockDim.x; }

// Real type of a complex vector type, and fused multiply-add per precision.
template <class C2> struct RealOf;
template <> struct RealOf<double2> { using type = double; };
template <> struct RealOf<float2> { using type = float; };
template <class T> struct Vec2Of;
template <> struct Vec2Of<double> { using type = double2; };
template <> struct Vec2Of<float> { using type = float2; };
__device__ __forceinline__ double fmaT(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fmaT(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double2 mk2(double x, double y) { return make_double2(x, y); }
__device__ __forceinline__ float2 mk2(float x, float y) { return make_float2(x, y); }

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaT(a.x, b.x, -a.y * b.y), fmaT(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
  return make_float2(fmaT(a.x, b.x, a.y * b.y), fmaT(a.y, b.x, -a.x * b.y));
}
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }

__device__ __forceinline__ double2 cadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 csub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fmaT(a.x, b.x, -a.y * b.y), fmaT(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 cmulc(double2 a, double2 b) {  // a * conj(b)
  return make_double2(fmaT(a.x, b.x, a.y * b.y), fmaT(a.y, b.x, -a.x * b.y));
}
__device__ __forceinline__ double2 cscale(double2 a, double s) { return make_double2(a.x * s, a.y * s); }

// cos(2 pi k / 32) for integer k (mathematical constants cos(pi j / 16)).
__host__ __device__ constexpr double cos32(int k) {
  constexpr double c1 = 0.98078528040323044913;   // cos(pi/16)
  constexpr double c2 = 0.92387953251128675613;   // cos(pi/8)
  constexpr double c3 = 0.83146961230254523708;   // cos(3 pi/16)
  constexpr double c4 = 0.70710678118654752440;   // cos(pi/4)
  constexpr double c5 = 0.55557023301960222474;   // cos(5 pi/16)
  constexpr double c6 = 0.38268343236508977173;   // cos(3 pi/8)
  constexpr double c7 = 0.19509032201612826785;   // cos(7 pi/16)
  k &= 31;
  k = k > 16 ? 32 - k : k;
  const double s = k > 8 ? -1.0 : 1.0;
  k = k > 8 ? 16 - k : k;
  return k == 8 ? 0.0 : s * (k == 0 ? 1.0 : k == 1 ? c1 : k == 2 ? c2 : k == 3 ? c3 : k == 4 ? c4 : k == 5 ? c5
                             : k == 6 ? c6 : c7);
}
__host__ __device__ constexpr double sin32(int k) { return cos32(k - 8); }
// FP32 constants c = cos(2 pi k / 32) and r = tan(2 pi k / 32) of the cosine-factored butterflies of radix 32
// (the I3 kernels with tensor-memory exchanges), for 0 < k < 16, k != 8: of the floats within two units in the
// last place the pair whose turn c + i c r is nearest to length 1 (plus a twentieth of its error in angle).
// Rounded each by itself they shorten a line's low frequencies by up to 3e-8 a stage, the same in every
// convolution, so that the errors add up over the nodes; two stages of radix 8 and 16 average over more
// constants.  Error of C[W] at N = 16, 32, 64 (J = M = 16, six states): 5.2, 5.8, 6.4e-7 -> 5.0, 5.8, 6.0e-7
// (node by node 4.8, 5.5, 5.7e-7).  Not taken: such pairs in every radix (N = 64 6.8e-7: what I3 and the other
// terms have in common cancels in C), radix 32 as 4 x 8 (5.6e-7 at N = 32, the same at 64, 2.7 and 6 % slower at
// N = 64 and 16).
struct Turn {
  float c, r;
};
__host__ __device__ constexpr Turn turn32(int k) {
  const int m = k > 8 ? 16 - k : k;
  const Turn t = m == 1 ? Turn{0x1.f6297cp-1f, 0x1.975f62p-3f}
               : m == 2 ? Turn{0x1.d906bcp-1f, 0x1.a8279ep-2f}
               : m == 3 ? Turn{0x1.a9b662p-1f, 0x1.561b84p-1f}
               : m == 4 ? Turn{0x1.6a09e8p-1f, 0x1.fffffcp-1f}
               : m == 5 ? Turn{0x1.1c73b4p-1f, 0x1.7f218ep+0f}
               : m == 6 ? Turn{0x1.87de2ep-2f, 0x1.3504f0p+1f}
                        : Turn{0x1.8f8b84p-3f, 0x1.41bfeep+2f};
  return k > 8 ? Turn{-t.c, -t.r} : t;
}

// x * exp(SIGN * 2 pi i k / R) for R <= 32, k a compile-time constant after unrolling.
template <int R, int SIGN, class C2>
__device__ __forceinline__ C2 twid(int k, C2 x) {
  using T = typename RealOf<C2>::type;
  const int k32 = (k * (32 / R)) & 31;
  if (k32 == 0) return x;
  if (k32 == 16) return mk2(-x.x, -x.y);
  if (k32 == 8) return SIGN > 0 ? mk2(-x.y, x.x) : mk2(x.y, -x.x);
  if (k32 == 24) return SIGN > 0 ? mk2(x.y, -x.x) : mk2(-x.y, x.x);
  const T c = (T)cos32(k32), s = (T)(SIGN * sin32(k32));
  return mk2(fmaT(x.x, c, -x.y * s), fmaT(x.x, s, x.y * c));
}

__host__ __device__ constexpr int ilog2c(int r) { return r <= 1 ? 0 : 1 + ilog2c(r / 2); }
// Bit reversal of i within `bits` <= 5 bits (closed form so that it folds after unrolling).
__host__ __device__ constexpr int bitrev(int i, int bits) {
  return (((i & 1) << 4) | ((i & 2) << 2) | (i & 4) | ((i & 8) >> 2) | ((i & 16) >> 4)) >> (5 - bits);
}

// One radix-2 decimation-in-time stage of butterfly span S on R registers.
// Butterflies with a non-trivial twiddle w = c + i s use the cosine-factored
// form (u +- w x) = u +- c (x + (s/c) i x): six FMAs instead of two products,
// two FMAs and four additions (|s/c| <= tan(3 pi/8) for R <= 16, tan(7 pi/16) for R = 32; the factor c
// takes the ratio's size out again).
template <int R, int SIGN, int S, class C2>
struct DftStage {
  __device__ __forceinline__ static void run(C2 (&b)[R]) {
    using T = typename RealOf<C2>::type;
#pragma unroll
    for (int g = 0; g < R; g += S) {
#pragma unroll
      for (int k = 0; k < S / 2; ++k) {
        const int k32 = (k * (32 / S)) & 31;
        const C2 u = b[g + k];
        const C2 x = b[g + k + S / 2];
        if ((k32 & 7) == 0) {
          const C2 t = twid<32, SIGN>(k32, x);
          b[g + k] = cadd(u, t);
          b[g + k + S / 2] = csub(u, t);
        } else {
          const T c = sizeof(T) == 4 && R == 32 ? (T)turn32(k32).c : (T)cos32(k32);
          const T r = sizeof(T) == 4 && R == 32 ? (T)(SIGN * turn32(k32).r) : (T)((SIGN * sin32(k32)) / cos32(k32));
          const T qx = fmaT(-r, x.y, x.x);
          const T qy = fmaT(r, x.x, x.y);
          b[g + k] = mk2(fmaT(c, qx, u.x), fmaT(c, qy, u.y));
          b[g + k + S / 2] = mk2(fmaT(-c, qx, u.x), fmaT(-c, qy, u.y));
        }
      }
    }
    DftStage<R, SIGN, 2 * S, C2>::run(b);
  }
};
template <int R, int SIGN, class C2>
struct DftStage<R, SIGN, 2 * R, C2> {
  __device__ __forceinline__ static void run(C2 (&)[R]) {}
};

// cos(2 pi k / 12) for integer k.
__host__ __device__ constexpr double cos12(int k) {
  constexpr double h3 = 0.86602540378443864676;   // sqrt(3)/2
  k = ((k % 12) + 12) % 12;
  return k == 0 ? 1.0 : k == 1 ? h3 : k == 2 ? 0.5 : k == 3 ? 0.0 : k == 4 ? -0.5 : k == 5 ? -h3
       : k == 6 ? -1.0 : k == 7 ? -h3 : k == 8 ? -0.5 : k == 9 ? 0.0 : k == 10 ? 0.5 : h3;
}
__host__ __device__ constexpr double sin12(int k) { return cos12(k - 3); }

// In-register DFT of length R (natural order in and out): R a power of two <= 32
// (radix-2 decimation in time), or R = 3 * 2^q <= 12 (one radix-3 decimation-in-time
// step on top of power-of-two sub-DFTs).
template <int R, int SIGN, class C2, bool POW2 = ((R & (R - 1)) == 0)>
struct Dft;

template <int R, int SIGN, class C2>
struct Dft<R, SIGN, C2, true> {
  __device__ __forceinline__ static void run(C2 (&a)[R]) {
    constexpr int L2 = ilog2c(R);
    C2 b[R];
#pragma unroll
    for (int i = 0; i < R; ++i) b[i] = a[bitrev(i, L2)];
    DftStage<R, SIGN, 2, C2>::run(b);
#pragma unroll
    for (int i = 0; i < R; ++i) a[i] = b[i];
  }
};

template <int R, int SIGN, class C2>
struct Dft<R, SIGN, C2, false> {
  static_assert(R % 3 == 0 && R <= 12, "mixed-radix DFT supports 3, 6, 12");
  __device__ __forceinline__ static void run(C2 (&a)[R]) {
    using T = typename RealOf<C2>::type;
    constexpr int Q = R / 3;
    C2 s0[Q], s1[Q], s2[Q];
#pragma unroll
    for (int t = 0; t < Q; ++t) { s0[t] = a[3 * t]; s1[t] = a[3 * t + 1]; s2[t] = a[3 * t + 2]; }
    Dft<Q, SIGN, C2>::run(s0);
    Dft<Q, SIGN, C2>::run(s1);
    Dft<Q, SIGN, C2>::run(s2);
    const T h3 = (T)(SIGN * 0.86602540378443864676);   // SIGN * sqrt(3)/2
#pragma unroll
    for (int k = 0; k < Q; ++k) {
      // twiddles exp(SIGN 2 pi i r k / R), r = 1, 2 (angles in twelfths: (12/R) r k)
      const int e1 = (12 / R) * k, e2 = 2 * (12 / R) * k;
      const C2 x0 = s0[k];
      C2 x1 = s1[k], x2 = s2[k];
      if (e1 % 12 != 0) {
        const T c = (T)cos12(e1), sn = (T)(SIGN * sin12(e1));
        x1 = mk2(fmaT(x1.x, c, -x1.y * sn), fmaT(x1.x, sn, x1.y * c));
      }
      if (e2 % 12 != 0) {
        const T c = (T)cos12(e2), sn = (T)(SIGN * sin12(e2));
        x2 = mk2(fmaT(x2.x, c, -x2.y * sn), fmaT(x2.x, sn, x2.y * c));
      }
      // radix-3 butterfly with w = exp(SIGN 2 pi i / 3)
      const C2 t1 = cadd(x1, x2);
      const C2 t2 = mk2(fmaT((T)-0.5, t1.x, x0.x), fmaT((T)-0.5, t1.y, x0.y));
      const C2 d = csub(x1, x2);
      a[k] = cadd(x0, t1);   // and t2 +- i SIGN sqrt(3)/2 (x1 - x2), as FMAs
      a[k + Q] = mk2(fmaT(-h3, d.y, t2.x), fmaT(h3, d.x, t2.y));
      a[k + 2 * Q] = mk2(fmaT(h3, d.y, t2.x), fmaT(-h3, d.x, t2.y));
    }
  }
};

template <int R, int SIGN, class C2>
__device__ __forceinline__ void dft(C2 (&a)[R]) {
  Dft<R, SIGN, C2>::run(a);
}

// DFT of length R (a power of two) of the inputs a[i] multiplied by real scales sc[i], the scaling
// fused into the first radix-2 stage: u su +- x sx as t = x sx (one multiplication per component)
// and two FMAs, instead of two multiplications and two additions per component.
template <int R, int SIGN, class C2>
__device__ __forceinline__ void dft_scaled(C2 (&a)[R], const typename RealOf<C2>::type (&sc)[R]) {
  static_assert((R & (R - 1)) == 0 && R >= 2, "power-of-two length");
  constexpr int L2 = ilog2c(R);
  C2 b[R];
#pragma unroll
  for (int g = 0; g < R; g += 2) {
    const int iu = bitrev(g, L2), ix = bitrev(g + 1, L2);
    const C2 u = a[iu], x = a[ix];
    const C2 t = mk2(x.x * sc[ix], x.y * sc[ix]);
    b[g] = mk2(fmaT(u.x, sc[iu], t.x), fmaT(u.y, sc[iu], t.y));
    b[g + 1] = mk2(fmaT(u.x, sc[iu], -t.x), fmaT(u.y, sc[iu], -t.y));
  }
  DftStage<R, SIGN, 4, C2>::run(b);
#pragma unroll
  for (int i = 0; i < R; ++i) a[i] = b[i];
}

// DFT of length R (a power of two) at shifted frequencies: the twiddle factors between the two stages of a
// line, w^(k1 t) on input t, merged into the butterflies.  tw(S / 2 - 1 + k) is the factor of butterfly k of
// the stage of span S (merged_twiddle).  With p = u + w x as four FMAs and u - w x = 2 u - p as two more, a
// butterfly takes six instructions; the twiddle products of their own took R - 1 times four.
template <int R, int S, class C2>
struct MergedStage {
  template <class TW>
  __device__ __forceinline__ static void run(C2 (&b)[R], TW tw) {
    using T = typename RealOf<C2>::type;
#pragma unroll
    for (int k = 0; k < S / 2; ++k) {
      const C2 w = tw(S / 2 - 1 + k);
#pragma unroll
      for (int g = 0; g < R; g += S) {
        const C2 u = b[g + k], x = b[g + k + S / 2];
        const C2 p = mk2(fmaT(w.x, x.x, fmaT(-w.y, x.y, u.x)), fmaT(w.x, x.y, fmaT(w.y, x.x, u.y)));
        b[g + k] = p;
        b[g + k + S / 2] = mk2(fmaT((T)2, u.x, -p.x), fmaT((T)2, u.y, -p.y));
      }
    }
    MergedStage<R, 2 * S, C2>::run(b, tw);
  }
};
template <int R, class C2>
struct MergedStage<R, 2 * R, C2> {
  template <class TW>
  __device__ __forceinline__ static void run(C2 (&)[R], TW) {}
};
template <int R, class C2, class TW>
__device__ __forceinline__ void dft_merged(C2 (&a)[R], TW tw) {
  constexpr int L2 = ilog2c(R);
  C2 b[R];
#pragma unroll
  for (int i = 0; i < R; ++i) b[i] = a[bitrev(i, L2)];
  MergedStage<R, 2, C2>::run(b, tw);
#pragma unroll
  for (int i = 0; i < R; ++i) a[i] = b[i];
}
// Exponent m of the factor exp(-+2 pi i m / n) that entry e = S / 2 - 1 + k of a length-R stage takes at
// shift s, with step Q = n / R between its frequencies: (s + Q k) R / S.
template <int R>
__host__ __device__ constexpr int merged_exponent(int e, int s, int Q) {
  int S = 2;
  while (S / 2 - 1 + S / 2 <= e) S *= 2;
  return (s + Q * (e - (S / 2 - 1))) * (R / S);
}

// Band-limited (Xi) frequencies |k| < n/4 of a line of n = A B points: in the permuted order
// pos = B k1 + t of frequency k1 + A t they are the t below B / 4 and from 3 B / 4 on, for every k1.
template <int B>
__host__ __device__ constexpr bool xi_t(int t) {
  return t < B / 4 || t >= 3 * B / 4;
}

// DFT of a stage-B line (length R = B >= 4) whose inputs vanish outside Xi, with the first radix-2
// stage reduced to copies: its butterflies pair a[r] with a[r + R / 2], and one of the two is zero.
template <int R, int SIGN, class C2>
__device__ __forceinline__ void dft_xi(C2 (&a)[R]) {
  static_assert((R & (R - 1)) == 0 && R >= 4, "power-of-two length");
  constexpr int L2 = ilog2c(R);
  C2 b[R];
#pragma unroll
  for (int g = 0; g < R; g += 2) {
    const int r = bitrev(g, L2);   // 0 .. R/2 - 1; bitrev(g + 1) = r + R / 2
    if (r < R / 4) {
      b[g] = a[r];
      b[g + 1] = a[r];
    } else {
      b[g] = a[r + R / 2];
      b[g + 1] = mk2(-a[r + R / 2].x, -a[r + R / 2].y);
    }
  }
  DftStage<R, SIGN, 4, C2>::run(b);
#pragma unroll
  for (int i = 0; i < R; ++i) a[i] = b[i];
}

// FFT of nl lines of length n held in shared (or global) memory:
// element e of line l at buf[l*ls + e*es].  tw[t2*A + k1] = exp(-2 pi i t2 k1 / n).
// SIGN < 0: forward, natural -> permuted.  SIGN > 0: inverse, permuted -> natural.
// XI (inverse only): the input is zero outside Xi, so the first stage reads the Xi values of each
// line only and runs dft_xi.
// Must be called by every thread of the block; ends with __syncthreads().
template <int n, int SIGN, bool XI = false, class C2>
__device__ __forceinline__ void fft_lines(C2* buf, int nl, int ls, int es, const C2* __restrict__ tw) {
  constexpr int A = Split<n>::A, B = Split<n>::B;
  const int tid = threadIdx.x, nt = blockDim.x;
  if (SIGN < 0) {
    for (int task = tid; task < nl * B; task += nt) {
      const int l = task % nl, t2 = task / nl;
      C2* base = buf + l * ls + t2 * es;
      C2 a[A];
#pragma unroll
      for (int t1 = 0; t1 < A; ++t1) a[t1] = base[B * t1 * es];
      dft<A, -1>(a);
#pragma unroll
      for (int k1 = 1; k1 < A; ++k1) a[k1] = cmul(a[k1], tw[t2 * A + k1]);
#pragma unroll
      for (int k1 = 0; k1 < A; ++k1) base[B * k1 * es] = a[k1];
    }
    __syncthreads();
    for (int task = tid; task < nl * A; task += nt) {
      const int l = task % nl, k1 = task / nl;
      C2* base = buf + l * ls + B * k1 * es;
      C2 b[B];
#pragma unroll
      for (int t2 = 0; t2 < B; ++t2) b[t2] = base[t2 * es];
      dft<B, -1>(b);
#pragma unroll
      for (int k2 = 0; k2 < B; ++k2) base[k2 * es] = b[k2];
    }
    __syncthreads();
  } else {
    for (int task = tid; task < nl * A; task += nt) {
      const int l = task % nl, k1 = task / nl;
      C2* base = buf + l * ls + B * k1 * es;
      C2 b[B];
      if constexpr (XI) {
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2)
          b[k2] = xi_t<B>(k2) ? base[k2 * es] : mk2((typename RealOf<C2>::type)0, (typename RealOf<C2>::type)0);
        dft_xi<B, 1>(b);
      } else {
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) b[k2] = base[k2 * es];
        dft<B, 1>(b);
      }
#pragma unroll
      for (int t2 = 0; t2 < B; ++t2) base[t2 * es] = b[t2];
    }
    __syncthreads();
    for (int task = tid; task < nl * B; task += nt) {
      const int l = task % nl, t2 = task / nl;
      C2* base = buf + l * ls + t2 * es;
      C2 a[A];
#pragma unroll
      for (int k1 = 0; k1 < A; ++k1) a[k1] = base[B * k1 * es];
#pragma unroll
      for (int k1 = 1; k1 < A; ++k1) a[k1] = cmulc(a[k1], tw[t2 * A + k1]);
      dft<A, 1>(a);
#pragma unroll
      for (int t1 = 0; t1 < A; ++t1) base[B * t1 * es] = a[t1];
    }
    __syncthreads();
  }
}

// Circular convolution along lines: forward FFT, multiplication of each
// spectral value by mul(line, pos) (pos = permuted position), inverse FFT.  The
// second forward stage, the multiplication and the first inverse stage act on
// the same B contiguous values, so they are fused in registers.
template <int n, class C2, class MUL>
__device__ __forceinline__ void fft_conv_lines(C2* buf, int nl, int ls, int es, const C2* __restrict__ tw, MUL mul) {
  constexpr int A = Split<n>::A, B = Split<n>::B;
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int task = tid; task < nl * B; task += nt) {
    const int l = task % nl, t2 = task / nl;
    C2* base = buf + l * ls + t2 * es;
    C2 a[A];
#pragma unroll
    for (int t1 = 0; t1 < A; ++t1) a[t1] = base[B * t1 * es];
    dft<A, -1>(a);
#pragma unroll
    for (int k1 = 1; k1 < A; ++k1) a[k1] = cmul(a[k1], tw[t2 * A + k1]);
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) base[B * k1 * es] = a[k1];
  }
  __syncthreads();
  for (int task = tid; task < nl * A; task += nt) {
    const int l = task % nl, k1 = task / nl;
    C2* base = buf + l * ls + B * k1 * es;
    C2 b[B];
#pragma unroll
    for (int t2 = 0; t2 < B; ++t2) b[t2] = base[t2 * es];
    dft<B, -1>(b);
    typename RealOf<C2>::type sc[B];
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) sc[k2] = (typename RealOf<C2>::type)mul(l, B * k1 + k2);
    dft_scaled<B, 1>(b, sc);
#pragma unroll
    for (int t2 = 0; t2 < B; ++t2) base[t2 * es] = b[t2];
  }
  __syncthreads();
  for (int task = tid; task < nl * B; task += nt) {
    const int l = task % nl, t2 = task / nl;
    C2* base = buf + l * ls + t2 * es;
    C2 a[A];
#pragma unroll
    for (int k1 = 0; k1 < A; ++k1) a[k1] = base[B * k1 * es];
#pragma unroll
    for (int k1 = 1; k1 < A; ++k1) a[k1] = cmulc(a[k1], tw[t2 * A + k1]);
    dft<A, 1>(a);
#pragma unroll
    for (int t1 = 0; t1 < A; ++t1) base[B * t1 * es] = a[t1];
  }
  __syncthreads();
}

// Chunk sizes (rows per row-pass chunk, columns per column-pass chunk) so that a
// chunk of complex doubles occupies about 64 KB of shared memory (three blocks
// per SM fit) and the radix-B stage has at least one task per thread.
__host__ __device__ constexpr int largest_divisor_le(int n, int cap) {
  return cap >= n ? n : (n % cap == 0 ? cap : largest_divisor_le(n, cap - 1));
}

template <int n, int ELEM = 16, int CB = 65536> struct Chunk {
  static constexpr int RC0 = CB / (n * ELEM);
  static constexpr int RC = largest_divisor_le(n, RC0);
  static constexpr int CC = RC;
  static constexpr int LS = n + 1;                 // padded row stride (odd => no bank conflicts)
  static constexpr int SMEM_ELEMS = (RC * LS > CC * n ? RC * LS : CC * n);
};

// Resident blocks that a kernel of lone blocks is compiled for at up to 64 points, at most what its chunk
// leaves of shared memory: free to unroll the passes of known chunks, the compiler went to twice the registers
// (k_i1_vjp at n = 16, FP64, 400 blocks: 48 -> 128 registers, 369 -> 526 us).  0: its own choice.
template <int n, class T, int CB>
__host__ __device__ constexpr int cell_min_blocks() {
  using C2 = typename Vec2Of<T>::type;
  if (!lone_block<n, C2, CB>() || n > 64) return 0;
  return 4 * (n + Chunk<n, sizeof(C2), CB>::SMEM_ELEMS) * sizeof(C2) <= 220 * 1024 ? 4 : 3;
}

// Row pass over an n x n field (rows = fixed ix, transform along iy), its chunks shared by the team:
// for each chunk: sm[r][iy] = ld(ix, iy); [FFT DIR1]; [sm = mid(ix, iy, sm)]; [FFT DIR2]; st(ix, iy, sm).
// DIR = 0 skips that transform; HAS_MID selects the pointwise middle step.
template <int n, int DIR1, bool HAS_MID, int DIR2, int CB = 65536, bool XI = false, class C2, class LD, class MID,
          class ST>
__device__ __forceinline__ void row_pass(C2* sm, const C2* tw, LD ld, MID mid, ST st) {
  constexpr int RC = Chunk<n, sizeof(C2), CB>::RC, LS = Chunk<n, sizeof(C2), CB>::LS;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int ranks = pass_ranks<n, C2, CB>();
  for (int r0 = pass_rank<n, C2, CB>() * RC; r0 < n; r0 += ranks * RC) {
#pragma unroll 4
    for (int idx = tid; idx < RC * n; idx += nt) {
      const int r = idx / n, iy = idx % n;
      sm[r * LS + iy] = ld(r0 + r, iy);
    }
    __syncthreads();
    if (DIR1 != 0) fft_lines<n, (DIR1 < 0 ? -1 : 1), XI>(sm, RC, LS, 1, tw);
    if (HAS_MID) {
  #pragma unroll 4
    for (int idx = tid; idx < RC * n; idx += nt) {
        const int r = idx / n, iy = idx % n;
        sm[r * LS + iy] = mid(r0 + r, iy, sm[r * LS + iy]);
      }
      __syncthreads();
    }
    if (DIR2 != 0) fft_lines<n, (DIR2 < 0 ? -1 : 1)>(sm, RC, LS, 1, tw);
#pragma unroll 4
    for (int idx = tid; idx < RC * n; idx += nt) {
      const int r = idx / n, iy = idx % n;
      st(r0 + r, iy, sm[r * LS + iy]);
    }
    __syncthreads();
  }
  if (ranks > 1) cluster_sync_global();
}

// Column pass (transform along ix) over chunks of CC columns held as sm[ix][c].
template <int n, int DIR1, bool HAS_MID, int DIR2, int CB = 65536, class C2, class LD, class MID, class ST>
__device__ __forceinline__ void col_pass(C2* sm, const C2* tw, LD ld, MID mid, ST st) {
  constexpr int CC = Chunk<n, sizeof(C2), CB>::CC;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int ranks = pass_ranks<n, C2, CB>();
  for (int c0 = pass_rank<n, C2, CB>() * CC; c0 < n; c0 += ranks * CC) {
#pragma unroll 4
    for (int idx = tid; idx < CC * n; idx += nt) {
      const int ix = idx / CC, c = idx % CC;
      sm[ix * CC + c] = ld(ix, c0 + c);
    }
    __syncthreads();
    if (DIR1 != 0) fft_lines<n, (DIR1 < 0 ? -1 : 1)>(sm, CC, 1, CC, tw);
    if (HAS_MID) {
  #pragma unroll 4
    for (int idx = tid; idx < CC * n; idx += nt) {
        const int ix = idx / CC, c = idx % CC;
        sm[ix * CC + c] = mid(ix, c0 + c, sm[ix * CC + c]);
      }
      __syncthreads();
    }
    if (DIR2 != 0) fft_lines<n, (DIR2 < 0 ? -1 : 1)>(sm, CC, 1, CC, tw);
#pragma unroll 4
    for (int idx = tid; idx < CC * n; idx += nt) {
      const int ix = idx / CC, c = idx % CC;
      st(ix, c0 + c, sm[ix * CC + c]);
    }
    __syncthreads();
  }
  if (ranks > 1) cluster_sync_global();
}

// Passes over n / 2 of the lines: the chunks are halved where a chunk is n / 8 lines (teams of up to eight
// blocks), so that eight blocks share these passes too.
template <int n, int CHUNK>
__host__ __device__ constexpr int half_chunk() {
  return (CHUNK == n / 8 && CHUNK > 1) ? CHUNK / 2 : CHUNK;
}
// The li-th of the n / 2 permuted positions of Xi.
template <int n>
__host__ __device__ __forceinline__ int xi_position(int li) {
  constexpr int B = Split<n>::B;
  const int k1 = li / (B / 2), t = li % (B / 2);
  return B * k1 + (t < B / 4 ? t : t + B / 2);
}

// Column passes over the n / 2 columns iy of Xi.  FWD: forward transform of ld(ix, iy), then mid(ix, iy, v)
// on the Xi rows (permuted positions); without FWD ld gives the spectrum and is called for Xi rows only.
// INV: inverse transform (zero outside the Xi rows), then st(ix, iy, v) on every row.
template <int n, bool FWD, bool INV, int CB = 65536, class C2, class LD, class MID, class ST>
__device__ __forceinline__ void xi_col_filter(C2* sm, const C2* tw, LD ld, MID mid, ST st) {
  constexpr int CC = half_chunk<n, Chunk<n, sizeof(C2), CB>::CC>(), B = Split<n>::B;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int ranks = pass_ranks<n, C2, CB>();
  for (int c0 = pass_rank<n, C2, CB>() * CC; c0 < n / 2; c0 += ranks * CC) {
    const int nc = (n / 2 - c0) < CC ? (n / 2 - c0) : CC;
#pragma unroll 4
    for (int idx = tid; idx < nc * n; idx += nt) {
      const int ix = idx / nc, c = idx % nc;
      if (FWD || xi_t<B>(ix % B)) sm[ix * CC + c] = ld(ix, xi_position<n>(c0 + c));
    }
    __syncthreads();
    if constexpr (FWD) {
      fft_lines<n, -1>(sm, nc, 1, CC, tw);
#pragma unroll 4
      for (int idx = tid; idx < nc * n; idx += nt) {
        const int ix = idx / nc, c = idx % nc;
        if (xi_t<B>(ix % B)) sm[ix * CC + c] = mid(ix, xi_position<n>(c0 + c), sm[ix * CC + c]);
      }
      __syncthreads();
    }
    if constexpr (INV) {
      fft_lines<n, 1, true>(sm, nc, 1, CC, tw);
#pragma unroll 4
      for (int idx = tid; idx < nc * n; idx += nt) {
        const int ix = idx / nc, c = idx % nc;
        st(ix, xi_position<n>(c0 + c), sm[ix * CC + c]);
      }
      __syncthreads();
    }
  }
  if (ranks > 1) cluster_sync_global();
}
template <int n, int CB = 65536, class C2, class LD, class ST>
__device__ __forceinline__ void xi_col_pass(C2* sm, const C2* tw, LD ld, ST st) {
  xi_col_filter<n, false, true, CB>(sm, tw, ld, [](int, int, C2 v) { return v; }, st);
}
// Row pass over the even rows ix (the coarse nodes, or a zero-interleaved coarse field).
template <int n, int DIR, int CB = 65536, bool XI = false, class C2, class LD, class ST>
__device__ __forceinline__ void even_row_pass(C2* sm, const C2* tw, LD ld, ST st) {
  constexpr int RC = half_chunk<n, Chunk<n, sizeof(C2), CB>::RC>(), LS = Chunk<n, sizeof(C2), CB>::LS;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int ranks = pass_ranks<n, C2, CB>();
  for (int r0 = pass_rank<n, C2, CB>() * RC; r0 < n / 2; r0 += ranks * RC) {
    const int nr = (n / 2 - r0) < RC ? (n / 2 - r0) : RC;
#pragma unroll 4
    for (int idx = tid; idx < nr * n; idx += nt) sm[idx / n * LS + idx % n] = ld(2 * (r0 + idx / n), idx % n);
    __syncthreads();
    fft_lines<n, DIR, XI>(sm, nr, LS, 1, tw);
#pragma unroll 4
    for (int idx = tid; idx < nr * n; idx += nt) st(2 * (r0 + idx / n), idx % n, sm[idx / n * LS + idx % n]);
    __syncthreads();
  }
  if (ranks > 1) cluster_sync_global();
}

// Column pass doing a circular convolution along ix for each column iy:
// sm[ix][c] = ld(ix, iy); forward FFT; times mul(pos_x, iy); inverse FFT; st(ix, iy, value).
template <int n, int CB = 65536, class C2, class LD, class MUL, class ST>
__device__ __forceinline__ void col_conv_pass(C2* sm, const C2* tw, LD ld, MUL mul, ST st) {
  constexpr int CC = Chunk<n, sizeof(C2), CB>::CC;
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int c0 = 0; c0 < n; c0 += CC) {
#pragma unroll 4
    for (int idx = tid; idx < CC * n; idx += nt) {
      const int ix = idx / CC, c = idx % CC;
      sm[ix * CC + c] = ld(ix, c0 + c);
    }
    __syncthreads();
    fft_conv_lines<n>(sm, CC, 1, CC, tw, [&](int l, int pos) { return mul(pos, c0 + l); });
#pragma unroll 4
    for (int idx = tid; idx < CC * n; idx += nt) {
      const int ix = idx / CC, c = idx % CC;
      st(ix, c0 + c, sm[ix * CC + c]);
    }
    __syncthreads();
  }
}

// Column pass over a subset of columns cols[0..ncols) (chunks of CC columns).
template <int n, int DIR1, bool HAS_MID, int DIR2, int CB = 65536, bool XI = false, class C2, class LD, class MID,
          class ST>
__device__ __forceinline__ void col_pass_list(C2* sm, const C2* tw, const int* cols, int ncols, LD ld, MID mid,
                                              ST st) {
  constexpr int CC = Chunk<n, sizeof(C2), CB>::CC;
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int c0 = 0; c0 < ncols; c0 += CC) {
    const int nc = (ncols - c0) < CC ? (ncols - c0) : CC;
#pragma unroll 4
    for (int idx = tid; idx < nc * n; idx += nt) {
      const int ix = idx / nc, c = idx % nc;
      sm[ix * CC + c] = ld(ix, cols[c0 + c]);
    }
    __syncthreads();
    if (DIR1 != 0) fft_lines<n, (DIR1 < 0 ? -1 : 1), XI>(sm, nc, 1, CC, tw);
    if (HAS_MID) {
  #pragma unroll 4
    for (int idx = tid; idx < nc * n; idx += nt) {
        const int ix = idx / nc, c = idx % nc;
        sm[ix * CC + c] = mid(ix, cols[c0 + c], sm[ix * CC + c]);
      }
      __syncthreads();
    }
    if (DIR2 != 0) fft_lines<n, (DIR2 < 0 ? -1 : 1)>(sm, nc, 1, CC, tw);
#pragma unroll 4
    for (int idx = tid; idx < nc * n; idx += nt) {
      const int ix = idx / nc, c = idx % nc;
      st(ix, cols[c0 + c], sm[ix * CC + c]);
    }
    __syncthreads();
  }
}

struct NoMid {
  template <class C2>
  __device__ C2 operator()(int, int, C2 v) const { return v; }
};

// Load the n-point twiddle table into shared memory.
template <int n, class C2>
__device__ __forceinline__ void load_twiddles(C2* sm_tw, const C2* __restrict__ g_tw) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) sm_tw[i] = g_tw[i];
  __syncthreads();
}

}  // namespace qbe
