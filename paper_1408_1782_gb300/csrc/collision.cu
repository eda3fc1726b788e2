// Size dispatch and workspace allocation of the collision operator; the
// kernels are instantiated per fine-grid size in collision_n*.cu.
#include <climits>
#include <utility>
#include <vector>

#include "internal.h"

namespace qbe {

cudaError_t collide_batch(const Tables& t, CollisionWork& cw, const double* w, double* c, int ncells,
                          cudaStream_t s, long long& launches, KernelTimer* tm) {
  if (cw.prec == 1) {
    switch (t.n) {
      case 16: return collide_batch_n<16, float>(t, cw, w, c, ncells, s, launches, tm);
      case 32: return collide_batch_n<32, float>(t, cw, w, c, ncells, s, launches, tm);
      case 64: return collide_batch_n<64, float>(t, cw, w, c, ncells, s, launches, tm);
      case 128: return collide_batch_n<128, float>(t, cw, w, c, ncells, s, launches, tm);
      case 256: return collide_batch_n<256, float>(t, cw, w, c, ncells, s, launches, tm);
    case 96: return collide_batch_n<96, float>(t, cw, w, c, ncells, s, launches, tm);
    case 192: return collide_batch_n<192, float>(t, cw, w, c, ncells, s, launches, tm);
      default: return cudaErrorInvalidValue;
    }
  }
  switch (t.n) {
    case 16: return collide_batch_n<16, double>(t, cw, w, c, ncells, s, launches, tm);
    case 32: return collide_batch_n<32, double>(t, cw, w, c, ncells, s, launches, tm);
    case 64: return collide_batch_n<64, double>(t, cw, w, c, ncells, s, launches, tm);
    case 128: return collide_batch_n<128, double>(t, cw, w, c, ncells, s, launches, tm);
    case 256: return collide_batch_n<256, double>(t, cw, w, c, ncells, s, launches, tm);
    case 96: return collide_batch_n<96, double>(t, cw, w, c, ncells, s, launches, tm);
    case 192: return collide_batch_n<192, double>(t, cw, w, c, ncells, s, launches, tm);
    default: return cudaErrorInvalidValue;
  }
}


#define QBE_SIZE_SWITCH(CALL, FAIL)                                   \
  if (prec == 1) {                                                    \
    switch (n) {                                                      \
      case 16: return CALL(16, float); case 32: return CALL(32, float); \
      case 64: return CALL(64, float); case 128: return CALL(128, float); \
      case 256: return CALL(256, float); case 96: return CALL(96, float); \
      case 192: return CALL(192, float); default: return FAIL;          \
    }                                                                 \
  }                                                                   \
  switch (n) {                                                        \
    case 16: return CALL(16, double); case 32: return CALL(32, double); \
    case 64: return CALL(64, double); case 128: return CALL(128, double); \
    case 256: return CALL(256, double); case 96: return CALL(96, double); \
    case 192: return CALL(192, double); default: return FAIL;           \
  }

int i3_variants(int n, int prec) {
#define QBE_CALL(nn, T) i3_variant_count<nn, T>()
  QBE_SIZE_SWITCH(QBE_CALL, 0)
#undef QBE_CALL
}

int i3_default(int n, int prec) {
#define QBE_CALL(nn, T) i3_default_variant<nn, T>()
  QBE_SIZE_SWITCH(QBE_CALL, 0)
#undef QBE_CALL
}

int i3_variant_bps(int n, int prec, int variant) {
#define QBE_CALL(nn, T) i3_blocks_per_sm<nn, T>(variant)
  QBE_SIZE_SWITCH(QBE_CALL, 1)
#undef QBE_CALL
}

int i3_concurrency(int n, int prec, int variant, int grid, int total) {
#define QBE_CALL(nn, T) i3_variant_concurrency<nn, T>(variant, grid, total)
  QBE_SIZE_SWITCH(QBE_CALL, 1)
#undef QBE_CALL
}

const char* i3_variant_desc(int n, int prec, int variant) {
#define QBE_CALL(nn, T) i3_variant_name<nn, T>(variant)
  QBE_SIZE_SWITCH(QBE_CALL, nullptr)
#undef QBE_CALL
}

bool i3_paired(int n, int prec, int variant) {
#define QBE_CALL(nn, T) i3_variant_paired<nn, T>(variant)
  QBE_SIZE_SWITCH(QBE_CALL, false)
#undef QBE_CALL
}

namespace {
// Two-dimensional transforms of a middle node, a node pair and half a pair.
struct NodeCost {
  double mid, pair, half;
};
constexpr NodeCost kForwardCost = {18, 20, 11};      // 2 shifts, 2 per convolution (8 or 4), back 2 or 1
constexpr NodeCost kTransposeCost = {36, 38, 22};    // 2 or 4 shifts, 16 or 8 convolutions, 2 back

double chunk_cost(int begin, int end, int M, const NodeCost& c) {
  double cost = 0;
  for (int it = begin; it < end;) {
    if ((M & 1) && it == M - 1) {
      cost += c.mid;
      it += 1;
    } else if ((it & 1) == 0 && it + 1 < end) {
      cost += c.pair;
      it += 2;
    } else {
      cost += c.half;
      it += 1;
    }
  }
  return cost;
}

// m-chunks per (cell, angle) for a launch that works on G units at a time, unit u on slot u mod G: `base`,
// or up to three times as many (at least `most_at_least`, at most M) where that evens out the slots'
// loads by more than a hundredth, within 4 GB of partials and 1.5 GB more than `base` takes.  A unit's fixed
// costs (its tables loaded, its partials written and reduced) count per_unit transforms.
int even_chunks(long long cj, int G, int M, int base, int most_at_least, size_t unit_bytes, const NodeCost& c,
                double per_unit) {
  double best = 0;
  int best_nmc = base;
  const int most = 3 * base > most_at_least ? 3 * base : most_at_least;
  for (int want = base; want <= most && want <= M; ++want) {
    const int mch = (M + want - 1) / want, nmc = (M + mch - 1) / mch;
    const long long units = cj * nmc;
    const size_t bytes = (size_t)units * unit_bytes, more = (size_t)(units - cj * base) * unit_bytes;
    if (want > base && (nmc == base || bytes > ((size_t)4 << 30) || more > ((size_t)3 << 29))) continue;
    const int g = G < units ? G : (int)units;
    std::vector<double> load(g, 0.0), cost(nmc);
    for (int mc = 0; mc < nmc; ++mc)
      cost[mc] = per_unit + chunk_cost(i3_chunk_begin(mc, nmc, M), i3_chunk_begin(mc + 1, nmc, M), M, c);
    for (long long u = 0; u < units; ++u) load[u % g] += cost[u % nmc];
    double mx = 0;
    for (double l : load) mx = l > mx ? l : mx;
    if (want == base || mx < 0.99 * best) {
      best = mx;
      best_nmc = nmc;
    }
  }
  return best_nmc;
}

// Buffers in one device allocation, each on a 256-byte boundary: creating a handle is a single cudaMalloc per
// workspace, and one that does not fit leaves nothing behind.
struct Carve {
  std::vector<std::pair<void**, size_t>> parts;
  size_t total = 0;
  template <class T>
  void add(T*& p, size_t bytes) {
    parts.push_back({(void**)&p, total});
    total += (bytes + 255) & ~(size_t)255;
  }
  cudaError_t take(void*& mem) const {
    const cudaError_t e = cudaMalloc(&mem, total);
    if (e != cudaSuccess) {
      mem = nullptr;
      cudaGetLastError();   // the caller may try a smaller one
      return e;
    }
    for (const auto& p : parts) *p.first = (unsigned char*)mem + p.second;
    return cudaSuccess;
  }
};
}  // namespace

double i3_chunk_cost(int begin, int end, int M, bool paired) {
  return paired ? chunk_cost(begin, end, M, kForwardCost) : kForwardCost.mid * (end - begin);
}

// Angle chunks per cell of the I1 and I2/I4 kernels: enough (cell, chunk) blocks to fill about one
// wave of the device (3 resident 256-thread blocks per SM), at most J/2 (the I2/I4 angle pairs).
int per_cell_chunks(int nb, int J) {
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int cap = 3 * (nsm > 0 ? nsm : 1);
  int nch = (cap + nb / 2) / (nb > 0 ? nb : 1);
  if (nch > J / 2) nch = J / 2;
  return nch < 1 ? 1 : nch;
}

cudaError_t alloc_collision_work(const Tables& t, int nb, CollisionWork& cw, int prec, int most_chunks) {
  const size_t P = (size_t)t.n * t.n;
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int nv = i3_variants(t.n, prec);
  if (nv < 1) return cudaErrorInvalidValue;
  const int v0 = i3_default(t.n, prec);
  const int bps = i3_variant_bps(t.n, prec, v0);
  int bps_max = bps;
  for (int v = 0; v < nv; ++v) {
    const int b = i3_variant_bps(t.n, prec, v);
    if (b > bps_max) bps_max = b;
  }
  cw.prec = prec;
  cw.nb = cw.order_nb = nb;
  cw.i3_variant = v0;
  cw.grid_i3 = nsm * bps;
  cw.grid_max = nsm * bps_max;
  // enough (cell, j, m-chunk) units for about 8 waves of the persistent grid (of its teams, where a
  // block works on several units at a time)
  int slots = i3_concurrency(t.n, prec, v0, cw.grid_i3, INT_MAX);
  if (slots < cw.grid_i3) slots = cw.grid_i3;
  const long long cj = (long long)nb * t.J, want_nmc = (8LL * slots + cj - 1) / cj;
  int nmc = (int)(want_nmc < t.M ? want_nmc : t.M);
  if (most_chunks > 0 && nmc > most_chunks) nmc = most_chunks;
  if (nmc < 1) nmc = 1;
  if (nmc > t.M) nmc = t.M;
  const size_t N = t.N, Q = (N - 1) * (N - 1);
  const size_t cz = prec == 1 ? sizeof(float2) : sizeof(double2);   // complex element
  const size_t rz = cz / 2;                                           // real element
  bool any_paired = false;
  for (int v = 0; v < nv; ++v) any_paired = any_paired || i3_paired(t.n, prec, v);
  const size_t part_bytes = (2 * P + (any_paired ? 2 * Q : 0)) * cz;
  auto set_chunks = [&](int want) {
    cw.mch = (t.M + want - 1) / want;
    cw.nmc = (t.M + cw.mch - 1) / cw.mch;
  };
  set_chunks(nmc);
  if (most_chunks == 0 && i3_paired(t.n, prec, v0))
    set_chunks(even_chunks(cj, i3_concurrency(t.n, prec, v0, cw.grid_i3, INT_MAX), t.M, cw.nmc, 1, part_bytes,
                           kForwardCost, 0.4));
  const size_t nparts = (size_t)nb * t.J * cw.nmc;
  cw.nparts_cap = nparts;
  cw.ws_slots = nb > cw.grid_i3 ? nb : cw.grid_i3;
  cw.nch = per_cell_chunks(nb, t.J);
  size_t ws_fields = 6 * (size_t)nb;
  if (5 * (size_t)nb * cw.nch > ws_fields) ws_fields = 5 * (size_t)nb * cw.nch;
  if (3 * (size_t)cw.grid_max > ws_fields) ws_fields = 3 * (size_t)cw.grid_max;
  // A requested grid is cut to this many blocks (and a launch to the resident ones, at most grid_max).
  cw.grid_cap = (int)(ws_fields / 3 < (size_t)INT_MAX ? ws_fields / 3 : INT_MAX);
  // fields per block of the kernels that take the nodes in pairs: four in FP64; in FP32 two per team, of
  // which a block has (128 / n)^2
  cw.i3_fields = prec == 0 ? 4 : t.n == 64 ? 8 : t.n == 32 ? 32 : t.n == 96 ? 4 : 3;
  if ((size_t)cw.i3_fields * cw.grid_max > ws_fields) ws_fields = (size_t)cw.i3_fields * cw.grid_max;
  // k_i124: per (cell, chunk, pair) one field for I1 and three for I2/I4
  if (8 * (size_t)nb * cw.nch > ws_fields) ws_fields = 8 * (size_t)nb * cw.nch;
  cw.ws_fields = ws_fields;
  Carve mem;
  mem.add(cw.what, (size_t)nb * 4 * P * cz);
  mem.add(cw.wfine, (size_t)nb * 2 * P * cz);
  if (prec == 1 && t.n != 16) mem.add(cw.wplane, (size_t)nb * 4 * P * rz);
  mem.add(cw.Dacc, (size_t)nb * 2 * P * cz);
  mem.add(cw.K2acc, (size_t)nb * P * rz);
  mem.add(cw.K4acc, (size_t)nb * 2 * P * cz);
  mem.add(cw.K2part, (size_t)nb * cw.nch * 2 * P * rz);
  if (cw.nch > 1) {
    mem.add(cw.Dpart, (size_t)nb * cw.nch * 2 * P * cz);
    mem.add(cw.K4part, (size_t)nb * cw.nch * 2 * P * cz);
  }
  mem.add(cw.K3part, nparts * 2 * P * cz);
  if (any_paired) mem.add(cw.K3spec, nparts * 2 * Q * cz);
  if (prec == 1) mem.add(cw.K3sum, (size_t)nb * 2 * P * sizeof(double2));
  if (prec == 1) mem.add(cw.K3ssum, (size_t)nb * 2 * Q * sizeof(double2));
  mem.add(cw.ws, ws_fields * P * cz);
  mem.add(cw.cbuf, (size_t)nb * 4 * N * N * sizeof(double));
  mem.add(cw.wbuf, (size_t)nb * 4 * N * N * sizeof(double));
  const cudaError_t e = mem.take(cw.mem);
  if (e != cudaSuccess) cw = CollisionWork();
  return e;
}

void free_collision_work(CollisionWork& cw) {
  cudaFree(cw.mem);
  cw = CollisionWork();
}


#define QBE_VJP_SWITCH(T, CALL)                       \
  switch (t.n) {                                      \
    case 16: return CALL(16, T);                      \
    case 32: return CALL(32, T);                      \
    case 64: return CALL(64, T);                      \
    case 128: return CALL(128, T);                    \
    case 256: return CALL(256, T);                    \
    case 96: return CALL(96, T);                      \
    case 192: return CALL(192, T);                    \
    default: break;                                   \
  }

namespace {
int vjp_bps(const Tables& t, int prec) {
#define QBE_BPS(n, T) i3_vjp_blocks_per_sm<n, T>()
  if (prec == 1) {
    QBE_VJP_SWITCH(float, QBE_BPS)
  } else {
    QBE_VJP_SWITCH(double, QBE_BPS)
  }
#undef QBE_BPS
  return 0;
}
}  // namespace

cudaError_t collide_pre(const Tables& t, CollisionWork& cw, const double* w, int ncells, cudaStream_t s,
                        long long& launches) {
#define QBE_PRE_CALL(n, T) collide_pre_n<n, T>(t, cw, w, ncells, s, launches, nullptr)
  if (cw.prec == 1) {
    QBE_VJP_SWITCH(float, QBE_PRE_CALL)
  } else {
    QBE_VJP_SWITCH(double, QBE_PRE_CALL)
  }
#undef QBE_PRE_CALL
  return cudaErrorInvalidValue;
}

cudaError_t collide_post(const Tables& t, CollisionWork& cw, double* c, int ncells, cudaStream_t s,
                         long long& launches) {
#define QBE_POST_CALL(n, T) collide_post_n<n, T>(t, cw, c, ncells, s, launches, nullptr)
  if (cw.prec == 1) {
    QBE_VJP_SWITCH(float, QBE_POST_CALL)
  } else {
    QBE_VJP_SWITCH(double, QBE_POST_CALL)
  }
#undef QBE_POST_CALL
  return cudaErrorInvalidValue;
}

cudaError_t i3_group(const Tables* const* tabs, const CollisionWork* const* cws, const int* ncells, int njobs,
                     void* ws, int grid, cudaStream_t s, long long& launches, int max_units) {
  if (njobs < 1) return cudaErrorInvalidValue;
  const Tables& t = *tabs[0];
  for (int k = 1; k < njobs; ++k)
    if (tabs[k]->n != t.n || cws[k]->prec != cws[0]->prec) return cudaErrorInvalidValue;
#define QBE_GROUP_CALL(n, T) i3_group_n<n, T>(tabs, cws, ncells, njobs, ws, grid, s, launches, max_units)
  if (cws[0]->prec == 1) {
    QBE_VJP_SWITCH(float, QBE_GROUP_CALL)
  } else {
    QBE_VJP_SWITCH(double, QBE_GROUP_CALL)
  }
#undef QBE_GROUP_CALL
  return cudaErrorInvalidValue;
}

cudaError_t collide_vjp(const Tables& t, CollisionWork& cw, VjpWork& vw, const double* w, const double* const* lam,
                        double* const* grad, int K, int ncells, int accumulate, cudaStream_t s, long long& launches,
                        KernelTimer* tm) {
  if (ncells > cw.nb || ncells > vw.nb || cw.prec != vw.prec || K < 1 || K > vw.kcap) return cudaErrorInvalidValue;
#define QBE_VJP_CALL(n, T) collide_vjp_n<n, T>(t, cw, vw, w, lam, grad, K, ncells, accumulate, s, launches, tm)
  if (vw.prec == 1) {
    QBE_VJP_SWITCH(float, QBE_VJP_CALL)
  } else {
    QBE_VJP_SWITCH(double, QBE_VJP_CALL)
  }
#undef QBE_VJP_CALL
  return cudaErrorInvalidValue;
}

// Cotangents one collision product should carry.  The staged transpose kernels (FP64, and FP32 on grids above
// 128 points) are bound by their transforms, so sharing the state's U convolutions saves work: I3 transpose,
// FP64, N = 64, 16 cells, J = M = 32, 381 ms for one, 598 for two, 1032 for four; FP32, N = 128, 196 and 347 ms.
// The FP32 shared-memory kernel is bound by its sums in global memory, whose working set leaves L2 further with
// every cotangent (16 cells of N = 48: 12.7 ms for one, 28.2 for two; N = 64, variant 1: 27.4 and 57.3); the
// tensor-memory kernel (15.9 ms there) holds one cotangent's sums, with no room for a second.  Both take one at a
// time.
int vjp_cotangent_group(const Tables& t, int prec) { return (prec == 1 && t.n <= 128) ? 1 : kMaxCotangents; }

int vjp_i3_variants(int n, int prec) { return (prec == 1 && n == 128) ? 2 : 1; }

cudaError_t alloc_vjp_work(const Tables& t, int nb, VjpWork& vw, int prec, int kcap, int most_chunks) {
  const size_t P = (size_t)t.n * t.n;
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int bps = vjp_bps(t, prec);
  if (bps < 1) return cudaErrorInvalidValue;
  if (kcap < 1 || kcap > kMaxCotangents) return cudaErrorInvalidValue;
  vw.prec = prec;
  vw.nb = nb;
  vw.kcap = kcap;
  vw.grid = nsm * bps;
  // teams (units at a time) of a block of the FP32 kernels with tensor-memory exchanges
  const bool tm = prec == 1 && (t.n == 32 || t.n == 64 || t.n == 128);
  const int teams = tm ? (128 / t.n) * (128 / t.n) : 1;
  // about 4 waves of (cell, j, m-chunk) units
  const long long cj = (long long)nb * t.J, want_nmc = (4LL * vw.grid * teams + cj - 1) / cj;
  int nmc = (int)(want_nmc < t.M ? want_nmc : t.M);
  if (most_chunks > 0 && nmc > most_chunks) nmc = most_chunks;
  if (nmc < 1) nmc = 1;
  vw.mch = (t.M + nmc - 1) / nmc;
  vw.nmc = (t.M + vw.mch - 1) / vw.mch;
  if (most_chunks == 0) {
    const size_t Q1 = (size_t)(t.n / 2 - 1) * (t.n / 2 - 1);
    // (of as many cotangents as a product can carry: the chunking, and with it the order of the sums, must
    // not depend on how many this workspace holds)
    const size_t unit_bytes =
        (size_t)vjp_cotangent_group(t, prec) * 2 * (P + Q1) * (prec == 1 ? sizeof(float2) : sizeof(double2));
    vw.nmc = even_chunks(cj, vw.grid * teams, t.M, vw.nmc, 8, unit_bytes, kTransposeCost, 1.0);
    vw.mch = (t.M + vw.nmc - 1) / vw.nmc;
  }
  const size_t nparts = (size_t)nb * t.J * vw.nmc;
  // per-cell kernels: 7 fields per cell; I3 transpose per block: 3 + 4 K fields (staged; the
  // shared-memory kernel one less), 6 per team
  const size_t per_block = tm ? (6 * (size_t)teams > 2 + 4 * (size_t)kcap ? 6 * (size_t)teams : 2 + 4 * (size_t)kcap)
                              : 3 + 4 * (size_t)kcap;
  size_t ws_fields = 7 * (size_t)nb;
  if (per_block * vw.grid > ws_fields) ws_fields = per_block * vw.grid;
  // per (cell, angle chunk): the recomputed forward's I1 and I2/I4 teams 8 fields, the I2/I4
  // transpose 7
  const size_t nch = (size_t)per_cell_chunks(nb, t.J);
  if (8 * (size_t)nb * nch > ws_fields) ws_fields = 8 * (size_t)nb * nch;
  const size_t kc = (size_t)kcap;
  const size_t cz = prec == 1 ? sizeof(float2) : sizeof(double2);
  const size_t rz = cz / 2;
  Carve mem;
  mem.add(vw.nu, kc * nb * 2 * P * cz);
  mem.add(vw.nuf, kc * nb * P * rz);
  mem.add(vw.muD, kc * nb * 2 * P * cz);
  mem.add(vw.muK2, kc * nb * P * rz);
  mem.add(vw.mu4, kc * nb * 2 * P * cz);
  mem.add(vw.mu3, kc * nb * 2 * P * cz);
  mem.add(vw.muh, kc * nb * 2 * P * cz);
  if (tm) mem.add(vw.mupl, kc * nb * 4 * P * rz);
  mem.add(vw.part_r, kc * nparts * 2 * P * cz);
  const size_t Q = (size_t)(t.n / 2 - 1) * (t.n / 2 - 1);   // kept frequencies (Fourier-space partials)
  mem.add(vw.part_s, kc * nparts * 2 * Q * cz);
  mem.add(vw.ws, ws_fields * P * cz);
  const cudaError_t e = mem.take(vw.mem);
  if (e != cudaSuccess) vw = VjpWork();
  return e;
}

void free_vjp_work(VjpWork& vw) {
  cudaFree(vw.mem);
  vw = VjpWork();
}

}  // namespace qbe
