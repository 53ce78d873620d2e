// GS2 sweeps of a small stencil system in one launch: one thread-block
// cluster, one row a thread.
//
// A symmetric sweep of a 4,096-row system is four row kernels of about 2 us
// each, nearly all of it launch and the round trips place -> columns ->
// gathers that every kernel repeats.  Here a row's entries (at most four to
// either side of the diagonal) are loaded into registers once, its entry of
// every vector lies in the shared memory of the CTA that owns it, and other
// rows' entries are read there as distributed shared memory, at addresses
// formed once.  The CTAs meet at the hardware cluster barrier between phases;
// all CTAs of a cluster run at once and each passes every barrier, so no wait
// depends on anything outside the cluster.  The arithmetic of a row is that
// of the row kernels, entry for entry in stored order.
//
#include <algorithm>
#include <map>
#include <mutex>

#include "internal.cuh"

namespace gs2 {

constexpr int kSmCtas = 16;
constexpr int kSmThreads = 512;
constexpr int kSmSide = 4;  // entries of a row to either side of the diagonal

// The sizes it takes, by the row kernels that it replaces: the launches saved
// grow with them, and beyond 256 rows an SM its FP64 pipe sets the time of a
// phase.  The lines are where the two cross on 7-point rows (5-point rows cross
// later, at 5,500 and 6,500 rows); back-to-back calls, us, row kernels / one
// launch:
//                          400 rows    4,096       5,832       6,859       8,000
//   forward (2 kernels)    5.3  4.2    5.3  5.3    5.5  6.0    5.3  6.3    5.3  6.8
//   symmetric (4)          8.7  5.8    9.3  7.3    8.9  8.7    8.9  9.5    8.8 10.1
//   symmetric, 2 inner (6) 12.1 7.0    13.4 9.0    13.6 10.8   13.8 11.8   13.3 12.7
//   symmetric, 3 inner (8) 15.7 8.4    17.5 10.8   17.8 13.1   17.9 14.4   17.6 15.5
// (400 rows of a 5-point stencil.)
static int64_t small_rows(int64_t kernels) {
  return kernels >= 6 ? 8192 : kernels >= 4 ? 6000 : 4096;
}

struct SmallArgs {
  int n, R;  // rows, rows per CTA
  const int *Arp, *Aci, *Lrp, *Urp;
  const double *Ava, *Lva, *Uva, *dinv, *b;
  double* x;
  int sweeps, inner, dir;
  double omega, gamma;
};

__device__ __forceinline__ unsigned sm_map(unsigned addr, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ double sm_load(unsigned addr) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr));
  return v;
}
__device__ __forceinline__ void sm_barrier() {
  asm volatile(
      "barrier.cluster.arrive.release.aligned;\n\t"
      "barrier.cluster.wait.acquire.aligned;" ::
          : "memory");
}

__global__ void __launch_bounds__(kSmThreads, 1) k_small_sweeps(SmallArgs a) {
  // vector v of this CTA's row t at vec[v][t]: x and two inner iterates
  __shared__ double vec[3][kSmThreads];
  pdl_wait();
  unsigned rank;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  const int t = threadIdx.x, row = (int)rank * a.R + t;
  const bool own = t < a.R && row < a.n;
  const unsigned vec0 = (unsigned)__cvta_generic_to_shared(&vec[0][0]);
  constexpr unsigned kStep = 8u * kSmThreads;  // from one vector to the next

  int nl = 0, nu = 0;
  double al[kSmSide], au[kSmSide], tl[kSmSide], tu[kSmSide];
  unsigned pl[kSmSide], pu[kSmSide];  // addresses of the entries' x
  double ad = 0.0, d = 0.0, b = 0.0, x = 0.0;
#pragma unroll
  for (int k = 0; k < kSmSide; ++k) {
    al[k] = au[k] = tl[k] = tu[k] = 0.0;
    pl[k] = pu[k] = vec0;
  }
  if (own) {
    const int r0 = a.Arp[row], l0 = a.Lrp[row], u0 = a.Urp[row];
    nl = a.Lrp[row + 1] - l0;
    nu = a.Urp[row + 1] - u0;
    d = a.dinv[row];
    b = a.b[row];
    x = a.x[row];
    ad = a.Ava[r0 + nl];
    auto place = [&](int col) {
      const int o = col / a.R;
      return sm_map(vec0 + 8u * (unsigned)(col - o * a.R), (unsigned)o);
    };
#pragma unroll
    for (int k = 0; k < kSmSide; ++k) {
      if (k < nl) {
        al[k] = a.Ava[r0 + k];
        tl[k] = a.Lva[l0 + k];
        pl[k] = place(a.Aci[r0 + k]);
      }
      if (k < nu) {
        au[k] = a.Ava[r0 + nl + 1 + k];
        tu[k] = a.Uva[u0 + k];
        pu[k] = place(a.Aci[r0 + nl + 1 + k]);
      }
    }
    vec[0][t] = x;
  }
  // the warp's longest rows: slots beyond them issue nothing on the FP64 pipe
  const int wl = __reduce_max_sync(0xffffffffu, nl), wu = __reduce_max_sync(0xffffffffu, nu);
  // s + sum of one side's values times vector v
  auto side = [&](double s, const double (&val)[kSmSide], const unsigned (&adr)[kSmSide], int cnt,
                  int most, int v) {
    double g[kSmSide];
#pragma unroll
    for (int k = 0; k < kSmSide; ++k) g[k] = k < cnt ? sm_load(adr[k] + (unsigned)v * kStep) : 0.0;
#pragma unroll
    for (int k = 0; k < kSmSide; ++k)
      if (k < most) {
        if (k < cnt) s = fma(val[k], g[k], s);
      }
    return s;
  };
  const bool damped = a.gamma != 1.0;
  for (int s = 0; s < a.sweeps; ++s) {
    for (int half = 0; half < 2; ++half) {
      const bool fwd = half == 0;
      if (a.dir == (fwd ? GS2_BACKWARD : GS2_FORWARD)) continue;
      sm_barrier();  // x complete
      // rhat = D^{-1} (b - A x), the inner iterate g_0
      double r = side(0.0, al, pl, nl, wl, 0);
      r = fma(ad, x, r);
      r = side(r, au, pu, nu, wu, 0);
      const double rh = d * (b - r);
      double g = rh;
      int cur = 1;
      for (int j = 0; j < a.inner; ++j) {
        if (own) vec[cur][t] = g;
        sm_barrier();  // g complete
        const double sum = fwd ? side(0.0, tl, pl, nl, wl, cur) : side(0.0, tu, pu, nu, wu, cur);
        const double go = rh - a.omega * sum;
        g = damped ? (1.0 - a.gamma) * g + a.gamma * go : go;
        cur ^= 3;
      }
      // every read of the old x ends before the first write of the new one: the
      // barriers of the inner sweeps lie between them, else one of its own
      if (a.inner == 0) sm_barrier();
      x = fma(a.omega, g, x);
      if (own) vec[0][t] = x;
    }
  }
  if (own) a.x[row] = x;
  sm_barrier();  // no CTA leaves while another may still read its memory
}

// Whether the sweeps of p on h take the one-launch form: FP64 non-compact GS2
// on a small system whose rows hold at most four entries to either side, the
// columns before the diagonal stored first.
bool small_sweeps_eligible(gs2_handle* h, const gs2_params* p) {
  const int64_t kernels = (p->direction == GS2_SYMMETRIC ? 2 : 1) * (int64_t)(1 + p->inner) *
                          p->outer * std::max(1, p->local_sweeps);
  if (h->n < 1 || h->n > small_rows(kernels) || h->pack || !h->parted || profiling_active(h))
    return false;
  if (p->kind != GS2_PC_GS2 || p->precision != GS2_FP64 || p->form != GS2_NONCOMPACT ||
      p->parts > 1)
    return false;
  longest_rows(h);
  if (h->cl_wl > kSmSide || h->cl_wu > kSmSide) return false;
  // the kernel's cluster must fit the GPU (asked once per process and shape)
  static std::mutex mu;
  static std::map<std::pair<int, int>, bool> fits;  // (device, CTAs)
  const int R = small_rows_per_cta(h->n), C = (int)((h->n + R - 1) / R);
  std::lock_guard<std::mutex> g(mu);
  auto it = fits.find({h->device, C});
  if (it != fits.end()) return it->second;
  bool ok = cudaFuncSetAttribute((const void*)k_small_sweeps,
                                 cudaFuncAttributeNonPortableClusterSizeAllowed,
                                 1) == cudaSuccess;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)C);
  cfg.blockDim = dim3((unsigned)kSmThreads);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim = {(unsigned)C, 1, 1};
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int clusters = 0;
  ok = ok && cudaOccupancyMaxActiveClusters(&clusters, (const void*)k_small_sweeps, &cfg) ==
                 cudaSuccess;
  if (!ok) cudaGetLastError();  // not an error of the caller's: the row kernels take it
  return fits[{h->device, C}] = ok && clusters >= 1;
}

// rows per CTA: whole warps, at least two, over at most 16 CTAs
int small_rows_per_cta(int64_t n) {
  const int R = (int)((n + kSmCtas - 1) / kSmCtas);
  return std::max(64, (R + 31) / 32 * 32);
}

void launch_small_sweeps(gs2_handle* h, const double* b, double* x, const gs2_params* p) {
  SmallArgs a{};
  a.n = (int)h->n;
  a.R = small_rows_per_cta(h->n);
  a.Arp = h->A.rp;
  a.Aci = h->A.ci;
  a.Ava = h->A.va;
  a.Lrp = h->L.rp;
  a.Lva = h->L.va;
  a.Urp = h->U.rp;
  a.Uva = h->U.va;
  a.dinv = h->dinv;
  a.b = b;
  a.x = x;
  a.sweeps = p->outer * std::max(1, p->local_sweeps);
  a.inner = p->inner;
  a.dir = p->direction;
  a.omega = p->omega;
  a.gamma = p->gamma;
  const int C = (a.n + a.R - 1) / a.R;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)C);
  cfg.blockDim = dim3((unsigned)a.R);
  cfg.stream = h->stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim = {(unsigned)C, 1, 1};
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  GS2_CUDA(cudaLaunchKernelEx(&cfg, k_small_sweeps, a));
  GS2_LAUNCH_CHECK();
}

}  // namespace gs2
