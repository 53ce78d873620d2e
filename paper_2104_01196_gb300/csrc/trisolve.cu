// The triangular solve of exact Gauss-Seidel / SOR, (D + omega T) g = r by
// D^{-1}:  g_i = rhat_i - omega sum_k T_ik g_k, then x_i += omega g_i, in one
// launch for the whole triangle (or one per level where there are few: by_level).
//
// What bounds it is the chain of levels: a 100^3 stencil has 298 of them,
// each a dependent step, against 24 us of memory traffic for the sweep.  One
// launch per level cost 4.9 us a step (1450 us per half sweep); a grid
// barrier per level would cost 1.3 us on top of a level's own round trips.
// Here no level waits for another as a whole: rows are solved as soon as
// their own dependencies are.  g is its own flag -- every entry starts as
// kPending, a NaN pattern no result takes, and a reader polls the eight bytes
// it needs anyway -- so a step costs one store to L2, one load from it and
// the row's products.
//
// Rows are stored in level order, entries with the place of their column in
// that order, so the rows of a warp (one chunk: rows of one level) write one
// run of g and read a few runs of it; in natural order a level's rows are
// strided and every lane would poll a sector of its own.  A warp takes the
// next chunk from a counter.  Chunks are handed out in level order and a warp
// finishes its chunk before its next one, so the first unfinished chunk
// always has its dependencies solved and a running warp: the kernel needs no
// co-resident grid.  Waits are bounded all the same; a warp that gives up
// records GS2_ERR_TIMEOUT and leaves.
//
// Measured, a symmetric sweep (two half sweeps, residuals included), against a
// launch per level: 100^3 Laplacian (298 levels) 2894 -> 535 us, 0.85 us a
// level; 200^2 Laplacian (399 levels) 2359 -> 452; a chain of 3,000 rows 11,700
// -> 2980; Q1 elasticity on 28^3 nodes 10,080 -> 1395.  One, two and four blocks
// per SM differ by 3%.
#include <algorithm>
#include <cstring>
#include <vector>

#include "tiles.cuh"

namespace gs2 {

constexpr unsigned long long kPending = ~0ull;
constexpr int kTriThreads = 256;
constexpr int kTriBlocksPerSm = 2;

// every entry of g pending, the chunk counter at 0
__global__ void k_tri_begin(int n, unsigned long long* g, int* ticket, const int* skip) {
  pdl_wait();
  if (skip && *skip) return;
  const int i0 = blockIdx.x * blockDim.x + threadIdx.x;
  for (int i = i0; i < n; i += gridDim.x * blockDim.x) g[i] = kPending;
  if (i0 == 0) *ticket = 0;
}

__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// K lanes per row (32 / K rows a chunk): lane l of a row takes entries l,
// l + K, ..., G of them in flight at once.  The products are summed from zero
// and subtracted from rhat at the end: a sum that starts at rhat is one
// dependent FP64 operation shorter (33 ns, 4% of the solve), but rounds every
// product at rhat's size (distance from the exact sweep 13% to 17% larger).
// Skipping the empty slots' products by a branch cost more than they do
// (+10%), and so did waiting by warp instead of by lane (+5%, +50% on rows
// of a few dozen entries); a sleep between polls changed nothing.
template <int K, int G>
__global__ void __launch_bounds__(kTriThreads, kTriBlocksPerSm)
k_trisolve(TriView T, const double* __restrict__ rhat, double* x, double omega, int x_zero,
           const int* skip, int* err) {
  pdl_wait();
  if (skip && *skip) return;
  const int lane = threadIdx.x & 31, q = lane / K, l = lane % K;
  int c = 0;
  if (lane == 0) c = atomicAdd(T.ticket, 1);
  c = __shfl_sync(0xffffffffu, c, 0);
  while (c < T.nchunks) {
    int next = 0;
    if (lane == 0) next = atomicAdd(T.ticket, 1);  // arrives while this chunk waits
    const int2 ch = __ldg(T.chunk + c);
    const int p = ch.x + q;
    const bool own = q < ch.y;
    int a = 0, e = 0, row = 0;
    double s = 0.0, rh = 0.0, xi = 0.0;
    if (own) {
      a = __ldg(T.rp + p);
      e = __ldg(T.rp + p + 1);
      if (l == 0) {
        row = __ldg(T.rows + p);
        rh = rhat[row];
        if (!x_zero) xi = x[row];
      }
    }
    bool ok = true;
    for (int k = a + l; k < e; k += G * K) {
      int d[G];
      double v[G];
      unsigned long long y[G];
#pragma unroll
      for (int j = 0; j < G; ++j) {
        const bool in = k + j * K < e;
        d[j] = in ? __ldg(T.ci + k + j * K) : -1;
        v[j] = in ? __ldg(T.va + k + j * K) : 0.0;
      }
#pragma unroll
      for (int j = 0; j < G; ++j) y[j] = d[j] >= 0 ? ld_relaxed(T.g + d[j]) : 0ull;
      long long t0 = 0;
      for (;;) {
        bool wait = false;
#pragma unroll
        for (int j = 0; j < G; ++j) wait = wait || y[j] == kPending;
        if (!wait) break;
#pragma unroll
        for (int j = 0; j < G; ++j)
          if (y[j] == kPending) y[j] = ld_relaxed(T.g + d[j]);
        const long long t = clock64();
        if (t0 == 0) t0 = t;
        if (t - t0 > kWaitBudgetCycles) {
          ok = false;
          break;
        }
      }
      if (!ok) break;
#pragma unroll
      for (int j = 0; j < G; ++j)
        s = fma(v[j], __longlong_as_double((long long)y[j]), s);
    }
    if (__any_sync(0xffffffffu, !ok)) {
      if (lane == 0 && err) atomicExch(err, (int)GS2_ERR_TIMEOUT);
      return;
    }
    if (K > 1) s = group_sum<K, double>(s);
    if (own && l == 0) {
      const double gi = rh - omega * s;
      unsigned long long bits = (unsigned long long)__double_as_longlong(gi);
      if (bits == kPending) bits = 0x7ff8000000000000ull;  // a NaN, but not that one
      st_relaxed(T.g + p, bits);
      x[row] = xi + omega * gi;
    }
    c = __shfl_sync(0xffffffffu, next, 0);
  }
}

// One level: rows p0 .. p1 of the level order, g of the earlier levels final.
// The arithmetic of a row is that of k_trisolve.
template <int K>
__global__ void __launch_bounds__(kTriThreads)
k_level(int p0, int p1, TriView T, const double* __restrict__ rhat, double* x, double omega,
        int x_zero, const int* skip) {
  pdl_wait();
  if (skip && *skip) return;
  double* g = (double*)T.g;
  const int q = threadIdx.x / K, l = threadIdx.x % K;
  constexpr int R = kTriThreads / K;
  for (int base = p0 + blockIdx.x * R; base < p1; base += gridDim.x * R) {
    const int p = base + q;
    const bool own = p < p1;
    double s = 0.0, rh = 0.0, xi = 0.0;
    int row = 0;
    if (own) {
      if (l == 0) {
        row = __ldg(T.rows + p);
        rh = rhat[row];
        if (!x_zero) xi = x[row];
      }
      const int e = __ldg(T.rp + p + 1);
      for (int k = __ldg(T.rp + p) + l; k < e; k += K)
        s = fma(__ldg(T.va + k), g[__ldg(T.ci + k)], s);
    }
    if (K > 1) s = group_sum<K, double>(s);
    if (own && l == 0) {
      const double gi = rh - omega * s;
      g[p] = gi;
      x[row] = xi + omega * gi;
    }
  }
}

// entries of the rows in level order (rp: their places): the place of each
// entry's column, and its value
__global__ void k_tri_place(int n, const int* __restrict__ rows, int* place) {
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x)
    place[rows[p]] = p;
}
__global__ void k_tri_entries(int n, const int* __restrict__ rows, const int* __restrict__ place,
                              const int* __restrict__ rp0, const int* __restrict__ ci0,
                              const double* __restrict__ va0, const int* __restrict__ rp, int* ci,
                              double* va) {
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
    const int a0 = rp0[rows[p]], a = rp[p], len = rp[p + 1] - a;
    for (int k = 0; k < len; ++k) {
      ci[a + k] = place[ci0[a0 + k]];
      va[a + k] = va0[a0 + k];
    }
  }
}

void tri_upload(gs2_handle* h, const DevCsr& M, const std::vector<int>& rows,
                const std::vector<int>& rp, TriSolve& T) {
  const int n = M.n;
  if (n == 0) return;
  // lanes per row: short rows one, so that a chunk is 32 rows; longer rows
  // more, as a lane's groups of four entries wait one after another (Q1
  // elasticity, 37 entries: 8 lanes 965 us a sweep, 16 lanes 921)
  T.lanes = M.mean_row <= 6.0 ? 1 : M.mean_row <= 24.0 ? 4 : 16;
  if (h->for_pack) T.lanes = M.tpr >= 8 ? 16 : 1;  // (as far as can be, whatever the others)
  T.width = 0;
  for (int p = 0; p < n; ++p) T.width = std::max(T.width, rp[p + 1] - rp[p]);
  const int per = 32 / T.lanes;
  std::vector<int2> chunk;
  chunk.reserve(n / per + T.levels.size());
  for (size_t v = 0; v + 1 < T.levels.size(); ++v)
    for (int p = T.levels[v]; p < T.levels[v + 1]; p += per)
      chunk.push_back(make_int2(p, std::min(per, T.levels[v + 1] - p)));
  T.nchunks = (int)chunk.size();
  // one allocation, and one upload of rows, entry places and chunks
  const size_t head = sizeof(int) * (2 * (size_t)n + 2) + sizeof(int2) * chunk.size();
  auto up = [](size_t x) { return (x + 255) / 256 * 256; };
  char* base = (char*)h->dalloc(up(head) + up(sizeof(int) * M.nnz) + up(sizeof(double) * M.nnz) +
                                up(sizeof(double) * n) + sizeof(int));
  std::vector<int> host(head / sizeof(int));
  std::copy(rows.begin(), rows.end(), host.begin());
  std::copy(rp.begin(), rp.end(), host.begin() + n);
  std::memcpy(host.data() + 2 * (size_t)n + 2, chunk.data(), sizeof(int2) * chunk.size());
  h->h2d(base, host.data(), head);
  T.rows = (int*)base;
  T.rp = T.rows + n;
  T.chunk = (int2*)(T.rows + 2 * (size_t)n + 2);
  base += up(head);
  T.ci = (int*)base;
  base += up(sizeof(int) * M.nnz);
  T.va = (double*)base;
  base += up(sizeof(double) * M.nnz);
  T.g = (unsigned long long*)base;
  base += up(sizeof(double) * n);
  T.ticket = (int*)base;
  // the column -> place map is needed only here: it lies in g until the
  // first solve
  int* place = (int*)T.g;
  k_tri_place<<<vec_blocks(h, n), kVecThreads, 0, h->stream>>>(n, T.rows, place);
  GS2_LAUNCH_CHECK();
  k_tri_entries<<<vec_blocks(h, n), kVecThreads, 0, h->stream>>>(n, T.rows, place, M.rp, M.ci,
                                                                M.va, T.rp, T.ci, T.va);
  GS2_LAUNCH_CHECK();
}

// Few levels of many rows are cheaper as a launch per level: a level then costs
// 3 to 4 us, but its rows stream without the fill of g, the counter and the
// polls, which cost about 20 us per million rows.  The line is where the two
// cross on 7-point rows in 1 to 33 levels, half sweeps in us, residual included
// (launch per level / one launch):
//                 1 level       3            5            9            17           33
//     4,096 rows  5.7 / 7.2     9.1 / 8.3    12.5 / 9.4   19 / 12      35 / 18      63 / 28
//    32,768       5.8 / 7.3     9.3 / 9.2    13.6 / 10.7  22 / 15      34 / 20      67 / 32
//   262,144       6.3 / 14.2    14.9 / 19.4  20.2 / 20.7  27 / 22      44 / 30      75 / 44
// 2,097,152       32 / 73       81 / 126     86 / 128     95 / 128     118 / 131    155 / 131
// (Longer rows in so few levels favour the launches more.)  Both forms give the
// same bits.
static bool by_level(const TriSolve& T, int n) {
  return (int64_t)T.levels.size() - 1 <= 2 + n / 100000;
}

void launch_trisolve(gs2_handle* h, const TriSolve& T, const double* rhat, double* x,
                     double omega, bool x_zero, const int* skip) {
  if (h->n == 0) return;
  const int n = (int)h->n;
  const TriView v{T.nchunks, T.chunk, T.rows, T.rp, T.ci, T.va, T.g, T.ticket};
  if (by_level(T, n)) {
    auto fn = T.lanes == 16 ? k_level<16> : T.lanes == 4 ? k_level<4> : k_level<1>;
    const int R = kTriThreads / T.lanes;
    for (size_t q = 0; q + 1 < T.levels.size(); ++q) {
      const int p0 = T.levels[q], p1 = T.levels[q + 1];
      const int grid = std::max(1, std::min((p1 - p0 + R - 1) / R, 8 * h->nsm));
      launch_pdl(fn, grid, kTriThreads, 0, h->stream, p0, p1, v, rhat, x, omega, x_zero ? 1 : 0,
                 skip);
      GS2_LAUNCH_CHECK();
    }
    return;
  }
  launch_pdl(k_tri_begin, vec_blocks(h, n), kVecThreads, 0, h->stream, n, T.g, T.ticket, skip);
  GS2_LAUNCH_CHECK();
  const int warps = kTriThreads / 32;
  const int grid = std::max(1, std::min((T.nchunks + warps - 1) / warps,
                                        kTriBlocksPerSm * h->nsm));
  // one lane a row: no more slots in flight than the longest row has
  auto fn = T.lanes == 16  ? k_trisolve<16, 4>
            : T.lanes == 4 ? k_trisolve<4, 4>
            : T.width > 3  ? k_trisolve<1, 4>
            : T.width == 3 ? k_trisolve<1, 3>
                           : k_trisolve<1, 2>;
  launch_pdl(fn, grid, kTriThreads, 0, h->stream, v, rhat, x, omega, x_zero ? 1 : 0, skip,
             h->dev_err);
  GS2_LAUNCH_CHECK();
}

}  // namespace gs2
