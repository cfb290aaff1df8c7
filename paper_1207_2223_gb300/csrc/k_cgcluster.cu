// CG iterations of a mixed-precision solve on a small lattice inside one thread
// block cluster (the CG routine of Sec. 3): the three passes of k_cglo.cu on up
// to 16 SMs, with the cluster's hardware barrier after each pass instead of a
// kernel boundary.
//
// On these lattices a pass is a chain of trips to L2, not bytes or arithmetic: a
// kernel launch, the halt flag, the loads, an atomic ticket, the partial sums, the
// scalars.  Inside a cluster a pass ends with one exchange: every block writes its
// partial sum into the shared memory of all blocks and arrives at the barrier,
// which also orders the fields written to global memory; every block then derives
// alpha, beta and the halt decision itself from the same sums in the same order.
// 8^4 with FP16 storage: 18.6 us per iteration as three kernels of a graph, 17.1 with
// their launches overlapped (launch_pdl), 13.9 here.  A device-wide barrier in
// software (a cooperative launch on all SMs) was slower than kernel boundaries: 22.5.
#include <atomic>

#include "lq_internal.h"

namespace lq {

namespace {

constexpr int kMaxCluster = 16;

struct ClusterArgs {
  SpinorRef r, p, t, x;
  const void* gauge;
  SolverState* st;
  int max_iters;
};

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cluster_size() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// All threads of the cluster; global and shared writes before it are visible after it (release and acquire, so
// that plain loads of what other blocks wrote before it do not see older lines).  Not the .aligned forms: it is
// entered after loops whose trip count differs within the last warp of a ragged lattice, and nothing
// promises that the lanes of a warp have met again by then.
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}

// Barrier of the cluster; f(sum of all threads' v, in a fixed order) in the first thread of every
// block, the block waiting for it.  FP64 operations issue at 2 per clock and SM, so nothing of the
// scalar work is done by all threads (every thread adding the blocks' sums and dividing took 5000 of
// the 29,000 clocks of an iteration at 8^4).  slots: [2][kMaxCluster] shared, by the parity of the
// calls, so that a block one call ahead does not overwrite what another still reads.
template <class F>
__device__ __forceinline__ void cluster_sum(double v, double (*slots)[kMaxCluster], int parity, const F& f) {
  __shared__ double sh[32];
  double w[1] = {v};
  block_sum<1>(w, sh);                               // w valid in warp 0
  const unsigned n = cluster_size();
  if (threadIdx.x < n) {
    unsigned local = static_cast<unsigned>(__cvta_generic_to_shared(&slots[parity][cluster_rank()])), remote;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(threadIdx.x));
    asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(w[0]) : "memory");
  }
  cluster_barrier();
  if (threadIdx.x < 32) {
    double x = threadIdx.x < n ? slots[parity][threadIdx.x] : 0.0;
#pragma unroll
    for (int o = kMaxCluster / 2; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (threadIdx.x == 0) f(x);
  }
  __syncthreads();
}

// Load mode 0: the neighbours' elements come from other blocks of this launch, ordered by cluster_barrier.
template <bool DAG, GStore G, SStore S>
__device__ __forceinline__ void stencil(const Geom& geo, const GaugeRef& U, const SpinorRef& in, int s, float kappa,
                                        cplx<float> acc[12]) {
  int c[4];
  site_coords(geo, s, c);
  hop_dir<0, DAG, G, S, float, SingleIndex, true, 0>(geo, U, in, s, c, acc);
  hop_dir<1, DAG, G, S, float, SingleIndex, false, 0>(geo, U, in, s, c, acc);
  hop_dir<2, DAG, G, S, float, SingleIndex, false, 0>(geo, U, in, s, c, acc);
  hop_dir<3, DAG, G, S, float, SingleIndex, false, 0>(geo, U, in, s, c, acc);
  cplx<float> ctr[12];
  load_spinor<S, float, 0>(in, geo.V, s, ctr);
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    acc[k].re = fmaf(-kappa, acc[k].re, ctr[k].re);
    acc[k].im = fmaf(-kappa, acc[k].im, ctr[k].im);
  }
}

template <GStore G, SStore S>
__global__ void __launch_bounds__(512, 1) cg_cluster_kernel(Geom geo, ClusterArgs a, float kappa) {
  __shared__ double slots[2][kMaxCluster];
  SolverState* st = a.st;
  // the state is read here and written only after a barrier, which every block reaches after reading
  if (*(volatile int*)&st->halt) return;
  const GaugeRef U{a.gauge};
  const int first = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
  const bool boss = blockIdx.x == 0;
  // scalars of the iteration: thread 0 of every block carries them along, block 0 writes them back
  double rr = 0.0, alpha = 0.0, tt = 0.0;
  int iter = 0, since = 0;
  if (threadIdx.x == 0) {
    rr = st->rr;
    iter = st->iter;
    since = st->iter_since_ru;
  }
  __shared__ float s_coef;                            // alpha, beta
  __shared__ int s_stop;
  cluster_barrier();                                  // every block of the cluster is resident before any writes to it
  for (int it = 0; it < a.max_iters; ++it) {
    // t = M p, alpha = rr / |t|^2
    double red = 0.0;
    for (int s = first; s < geo.V; s += stride) {
      cplx<float> v[12];
      stencil<false, G, S>(geo, U, a.p, s, kappa, v);
      store_spinor<S, float>(a.t, geo.V, s, v);
      red += site_norm2(v);
    }
    cluster_sum(red, slots, 0, [&](double sum) {
      tt = sum;
      const bool bad = !(tt > 0.0) || !isfinite(tt) || !isfinite(rr);
      alpha = bad ? 0.0 : rr / tt;
      s_coef = (float)alpha;
      s_stop = bad;
      if (bad && boss) {
        st->tt = tt;
        st->breakdown = 1;
        st->halt = 1;
        st->alpha = 0.0;
        st->rr = rr;
        st->iter = iter;
        st->iter_since_ru = since;
      }
    });
    if (s_stop) break;
    const float al = s_coef;
    // r -= alpha M^dag t, x += alpha p, beta, halt decision
    red = 0.0;
    for (int s = first; s < geo.V; s += stride) {
      cplx<float> v[12], rv[12], xv[12], pv[12];
      stencil<true, G, S>(geo, U, a.t, s, kappa, v);
      load_spinor<S, float, 0>(a.r, geo.V, s, rv);
      load_spinor<xlo_store(S), float, 0>(a.x, geo.V, s, xv);
      load_spinor<S, float, 0>(a.p, geo.V, s, pv);
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        rv[k] = {fmaf(-al, v[k].re, rv[k].re), fmaf(-al, v[k].im, rv[k].im)};
        xv[k] = {fmaf(al, pv[k].re, xv[k].re), fmaf(al, pv[k].im, xv[k].im)};
      }
      store_spinor<S, float>(a.r, geo.V, s, rv);
      store_spinor<xlo_store(S), float>(a.x, geo.V, s, xv);
      red += site_norm2(rv);
    }
    cluster_sum(red, slots, 1, [&](double rr_new) {
      const bool finite = isfinite(rr_new);
      ++since;
      const bool halt = !finite || rr_new <= st->stop2 || (st->ru_every > 0 && since >= st->ru_every) ||
                        (st->delta2 > 0.0 && rr_new < st->delta2 * st->rr_ref) || iter + 1 >= st->maxiter;
      const double beta = rr_new / rr;
      s_coef = (float)beta;
      s_stop = halt;
      if (boss) {
        if (st->hist != nullptr && iter < st->hist_len) st->hist[iter] = sqrt(rr_new / st->phi2);
        if (halt || it == a.max_iters - 1) {
          st->tt = tt;
          st->alpha = alpha;
          st->beta = beta;
          st->rr_prev = rr;
          st->rr = rr_new;
          st->iter = iter + 1;
          st->iter_since_ru = since;
          if (!finite) st->breakdown = 1;
          if (halt) st->halt = 1;
        }
      }
      ++iter;
      rr = rr_new;
    });
    if (s_stop) break;
    // p = r + beta p
    const float be = s_coef;
    for (int s = first; s < geo.V; s += stride) {
      cplx<float> rv[12], pv[12];
      load_spinor<S, float, 0>(a.r, geo.V, s, rv);
      load_spinor<S, float, 0>(a.p, geo.V, s, pv);
#pragma unroll
      for (int k = 0; k < 12; ++k) pv[k] = {fmaf(be, pv[k].re, rv[k].re), fmaf(be, pv[k].im, rv[k].im)};
      store_spinor<S, float>(a.p, geo.V, s, pv);
    }
    cluster_barrier();
  }
  cluster_barrier();                                  // no block leaves while another may still write to its slots
}

template <GStore G, SStore S>
cudaError_t run(lq_ctx* c, const void* gauge, int n, double kappa, cudaStream_t stream) {
  auto kern = &cg_cluster_kernel<G, S>;
  const int k = (int)S, V = c->geo.V;
  // a warp per SM first, then more warps: one site per thread up to 16 blocks of 512
  int blocks = 1;
  while (blocks < kMaxCluster && blocks * 32 < V) blocks <<= 1;
  const int bs = std::min(512, ((V + blocks - 1) / blocks + 31) & ~31);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(bs);
  cfg.stream = stream;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = blocks;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  // more than 8 blocks in a cluster have to be allowed, once per kernel and device
  static std::atomic<unsigned long long> allowed{0};
  if (!(allowed.load() >> (c->device & 63) & 1)) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    allowed.fetch_or(1ull << (c->device & 63));
  }
  ClusterArgs a{c->r_lo[k].ref(), c->p_lo[k].ref(), c->t_lo[k].ref(), c->x_lo[k].ref(), gauge, c->state, n};
  return cudaLaunchKernelEx(&cfg, kern, c->geo, a, (float)kappa);
}

}  // namespace

// Up to kClusterMaxSites sites, where the device has room for a cluster of 16 (a partition of a GPU
// may not).  Not with the optional stencils.
bool cluster_takes(const lq_ctx* c, int prec) {
  if (prec == LQ_F64 || c->geo.V > kClusterMaxSites || c->staged || (c->pair_sites && prec == LQ_I16_12)) return false;
  static std::atomic<unsigned long long> known{0}, room{0};
  const unsigned long long bit = 1ull << (c->device & 63);
  if (!(known.load() & bit)) {
    auto kern = &cg_cluster_kernel<GStore::F32_18, SStore::F32>;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(kMaxCluster);
    cfg.blockDim = dim3(512);
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kMaxCluster;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int n = 0;
    const bool ok = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0;
    if (!ok) cudaGetLastError();
    if (ok) room.fetch_or(bit);
    known.fetch_or(bit);
  }
  return (room.load() & bit) != 0;
}

cudaError_t cg_cluster_iterations(lq_ctx* c, int prec, int n, double kappa, cudaStream_t stream) {
  const void* gauge = c->gauge_lo[prec];
  switch (prec) {
    case LQ_F32: return run<GStore::F32_18, SStore::F32>(c, gauge, n, kappa, stream);
    case LQ_F32_12: return run<GStore::F32_12, SStore::F32>(c, gauge, n, kappa, stream);
    case LQ_F16_12: return run<GStore::F16_12, SStore::F16>(c, gauge, n, kappa, stream);
    case LQ_BF16_12: return run<GStore::BF16_12, SStore::BF16>(c, gauge, n, kappa, stream);
    case LQ_I16_12: return run<GStore::I16_12, SStore::I16>(c, gauge, n, kappa, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lq
