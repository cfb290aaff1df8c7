// M^dag M on caller buffers without any device allocation.
//
// Some callers cannot let a library allocate device memory: an application
// that hands all of its GPU memory to its own pool allocator and forbids
// cudaMalloc after start-up, or a plugin that runs under a fixed memory
// budget set by its host program.  lq_apply_MdagM_static serves them: it
// takes the gauge field and the spinors in the canonical layout directly
// from device buffers the caller owns, and keeps its one intermediate
// field (M in) and the sites' exponent words in fixed-size arrays compiled into
// this library.
//
// The arrays are file-scope __device__ variables.  Their names, used in host
// code, are only host-side stand-ins and not device addresses, so host code
// asks the runtime for the device addresses (cudaGetSymbolAddress) once per
// device, with that device current, and passes the result to the kernels.
#include <mutex>
#include <string>

#include "lq_fix64.cuh"

namespace lq {

// Largest lattice the array holds: 65,536 sites (for example 16^4), one FP64
// spinor of 12 complex numbers per site = 12 MiB, and two words per site = 0.5 MiB.
// Every GPU that loads the library holds these arrays until the process exits.
constexpr int kStaticMaxSites = 65536;

static __device__ __align__(256) double2 g_static_scratch[(size_t)kStaticMaxSites * 12];

// Site words of the input (ExpRange, with kBadLinks) and of M in.
static __device__ int g_static_word[2][kStaticMaxSites];

// Some link of the site is not unitary (unit_length): its hops take FP64 arithmetic.
constexpr int kBadLinks = 1 << 17;

// The word of every site of the input and of its four links; one thread per site and link
// direction, direction 0 also reads the spinor.  The fixed-point operator below needs both before
// it reads a site, and canonical buffers come without them.
__global__ void __launch_bounds__(256) static_scan_kernel(int V, const double2* __restrict__ U,
                                                          const double2* __restrict__ in, int* __restrict__ word) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;      // four consecutive threads per site
  const int s = idx >> 2, mu = idx & 3;
  const bool active = s < V;
  bool bad = false;
  ExpRange r;
  if (active) {
    const double2* u = U + (size_t)idx * 9;
    float row[3] = {0.f, 0.f, 0.f}, col[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const double2 w = u[k];
      const float a = (float)w.x, b = (float)w.y, n = a * a + b * b;
      row[k / 3] += n;
      col[k % 3] += n;
    }
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) ok = ok && unit_length(row[k]) && unit_length(col[k]);
    bad = !ok;
    cplx<double> v[3];                                          // thread mu reads spin mu
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double2 w = in[(size_t)s * 12 + 3 * mu + k];
      v[k] = {w.x, w.y};
    }
    r.spin(v);
  }
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    r.mx = max(r.mx, __shfl_xor_sync(0xffffffffu, r.mx, o));
    r.mn = min(r.mn, __shfl_xor_sync(0xffffffffu, r.mn, o));
    r.lo |= __shfl_xor_sync(0xffffffffu, r.lo, o);
    bad |= __shfl_xor_sync(0xffffffffu, (int)bad, o) != 0;
  }
  if (active && mu == 0) word[s] = r.word() | (bad ? kBadLinks : 0);
}

// Canonical buffers: 12 complex numbers per site, links [site][mu][3][3], converted as they are read.
struct CanonAccess {
  const double2* psi;
  const double2* U;
  __device__ __forceinline__ const double2* site(int comp, int n) const { return psi + (size_t)n * 12 + comp; }
  __device__ __forceinline__ double2 spin(const double2* p, int k) const { return p[k]; }
  __device__ __forceinline__ const double2* link(int mu, int s) const { return U + ((size_t)s * 4 + mu) * 9; }
  __device__ __forceinline__ int4 element(const double2* p, int e) const { return fix_link(__ldg(p + e)); }
  __device__ __forceinline__ double2 element64(int mu, int e, int s) const { return __ldg(link(mu, s) + e); }
};

// out = in - kappa * H in (DAG: in - kappa * H^dag in) in fixed point (lq_fix64.cuh) on canonical
// buffers, two threads per site.  win: words of the input; wlink: the words that hold kBadLinks;
// wout (may be null): the words of out.  8^4: one thread per site in FP64 arithmetic 65 us,
// bound by the FP64 pipe of the 16 SMs its blocks reached; here 35 us for the whole call (131).
// DIR: split by direction (fix_dir_site), four warps per 16 sites.
template <bool DAG, bool DIR>
__global__ void __launch_bounds__(DIR ? 128 : kFixBlock, DIR ? 4 : 2)
    hop_canonical_kernel(Geom geo, const double2* __restrict__ U, const double2* in, const int* win, const int* wlink,
                         double2* out, int* wout, double kappa) {
  pdl_wait();
  const CanonAccess acc{in, U};
  const int lane = threadIdx.x & 31, dir = DIR ? (int)threadIdx.x >> 5 : 0, half = threadIdx.x & 1;
  const int s0 = DIR ? (int)blockIdx.x * 16 + (lane >> 1) : (int)(blockIdx.x * blockDim.x + threadIdx.x) >> 1;
  const bool active = s0 < geo.V;
  const int s = active ? s0 : 0;
  int c[4];
  site_coords(geo, s, c);
  int f[4], b[4], E = kFixMinExp, any = wlink[s] & kBadLinks;
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    f[m] = nbr_fwd(geo, s, c, m);
    b[m] = nbr_bwd(geo, s, c, m);
    const int wf = win[f[m]], wb = win[b[m]];
    any |= (wf | wb) & kFixSlow;
    any |= wlink[b[m]] & kBadLinks;
    E = max(E, max(wf & 0x7ff, wb & 0x7ff));
  }
  const bool slow = any != 0;
  cplx<double> v[6];
  if constexpr (DIR) {
    __shared__ long long part[3][12][32];
    fix_dir_site<DAG>(geo, acc, s, c, f, b, E, slow, lane, dir, kappa, part, v);
    if (dir > 0) return;
  } else {
    FixAcc a;
    if (!slow) {
      fix_clear(a);
      fix_hops<DAG>(geo, acc, s, c, f, b, half, E, a);
    } else {
      FixAcc t64;
      split_site64<DAG>(geo, acc, s, half, &t64);
      a = t64;
    }
    fix_finish(acc, a, s, half, slow, slow ? -kappa : -kappa * __hiloint2double((E - 56) << 20, 0), v);
  }
  if (active) {
#pragma unroll
    for (int k = 0; k < 6; ++k) out[(size_t)s * 12 + fix_comp(half, k)] = make_double2(v[k].re, v[k].im);
  }
  if (wout) {
    ExpRange r;
    r.spin(v);
    r.spin(v + 3);
    r.mx = max(r.mx, __shfl_xor_sync(0xffffffffu, r.mx, 1));
    r.mn = min(r.mn, __shfl_xor_sync(0xffffffffu, r.mn, 1));
    r.lo |= __shfl_xor_sync(0xffffffffu, r.lo, 1);
    if (active && half == 0) wout[s] = r.word();
  }
}

namespace {

// True when p is device (or managed) memory.  cudaPointerGetAttributes
// allocates nothing; host memory, including pinned or unregistered host
// buffers, is refused before any kernel sees it.
bool static_device_ptr(const void* p) {
  cudaPointerAttributes a;
  if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

constexpr int kMaxDevices = 64;
std::mutex g_static_mutex;
double2* g_static_addr[kMaxDevices] = {};
int* g_static_word_addr[kMaxDevices] = {};

// Device address of the scratch array on the current device, looked up once
// per device (the first call on each device) and kept for the life of the
// process.  A device reset (cudaDeviceReset, or a reset of the primary
// context) unloads the module that holds the array, so calls after one are
// not supported.
cudaError_t static_scratch_address(double2** out, int** word) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_static_mutex);
  if (!g_static_addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess) return e;
    void* q = nullptr;
    e = cudaGetSymbolAddress(&q, g_static_word);
    if (e != cudaSuccess) return e;
    g_static_addr[dev] = static_cast<double2*>(p);
    g_static_word_addr[dev] = static_cast<int*>(q);
  }
  *out = g_static_addr[dev];
  *word = g_static_word_addr[dev];
  return cudaSuccess;
}

}  // namespace
}  // namespace lq

// Error text for the static entry point (read with lq_last_error(NULL)).
void lq_set_global_error(const std::string& msg);

extern "C" lq_status lq_apply_MdagM_static(double* out, const double* U, const double* in, const int dims[4],
                                           int t_antiperiodic, double kappa, void* cuda_stream) {
  using namespace lq;
  if (!out || !U || !in || !dims) {
    lq_set_global_error("lq_apply_MdagM_static: null argument");
    return LQ_ERR_ARG;
  }
  // Each extent is checked before it enters the product, and the product stops
  // growing as soon as it passes the limit, so it cannot overflow.
  long long V = 1;
  for (int m = 0; m < 4; ++m) {
    if (dims[m] < 2) {
      lq_set_global_error("lq_apply_MdagM_static: every lattice extent must be >= 2");
      return LQ_ERR_SHAPE;
    }
    if (dims[m] > kStaticMaxSites || V * dims[m] > kStaticMaxSites) {
      lq_set_global_error("lq_apply_MdagM_static: lattice " + std::to_string(dims[0]) + "x" +
                          std::to_string(dims[1]) + "x" + std::to_string(dims[2]) + "x" + std::to_string(dims[3]) +
                          " has more sites than the built-in scratch array holds (at most " +
                          std::to_string(kStaticMaxSites) + ")");
      return LQ_ERR_SHAPE;
    }
    V *= dims[m];
  }
  const uintptr_t mis = (reinterpret_cast<uintptr_t>(out) | reinterpret_cast<uintptr_t>(U) |
                         reinterpret_cast<uintptr_t>(in)) & 15u;
  if (mis) {
    lq_set_global_error("lq_apply_MdagM_static: buffers must be 16-byte aligned");
    return LQ_ERR_ARG;
  }
  if (!static_device_ptr(out) || !static_device_ptr(U) || !static_device_ptr(in)) {
    lq_set_global_error("lq_apply_MdagM_static: U, in and out must be device buffers");
    return LQ_ERR_ARG;
  }
  double2* scratch = nullptr;
  int* word = nullptr;
  cudaError_t e = static_scratch_address(&scratch, &word);
  if (e != cudaSuccess) {
    cudaGetLastError();
    lq_set_global_error(std::string("lq_apply_MdagM_static: cudaGetSymbolAddress: ") + cudaGetErrorString(e));
    return LQ_ERR_CUDA;
  }
  Geom geo{};
  geo.V = (int)V;
  for (int m = 0; m < 4; ++m) geo.L[m] = dims[m];
  geo.stride[0] = 1;
  for (int m = 1; m < 4; ++m) geo.stride[m] = geo.stride[m - 1] * dims[m - 1];
  geo.antiperiodic = t_antiperiodic ? 1 : 0;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const double2 *Uc = reinterpret_cast<const double2*>(U), *ic = reinterpret_cast<const double2*>(in);
  int *w0 = word, *w1 = word + kStaticMaxSites;
  static_scan_kernel<<<grid_for(4 * geo.V, 128), 128, 0, st>>>(geo.V, Uc, ic, w0);
  // scratch = M in (every site written before it is read: nothing to clear)
  double2* oc = reinterpret_cast<double2*>(out);
  const bool few = geo.V <= kFixDirSites;                          // as launch_dslash_fix
  const int grid = few ? grid_for(geo.V, 16) : grid_for(2 * geo.V, kFixBlock), bs = few ? 128 : kFixBlock;
  auto m = few ? &hop_canonical_kernel<false, true> : &hop_canonical_kernel<false, false>;
  auto mdag = few ? &hop_canonical_kernel<true, true> : &hop_canonical_kernel<true, false>;
  launch_pdl(m, grid, bs, 0, st, geo, Uc, ic, w0, w0, scratch, w1, kappa);
  // out = M^dag scratch
  launch_pdl(mdag, grid, bs, 0, st, geo, Uc, scratch, w1, w0, oc, nullptr, kappa);
  e = cudaGetLastError();
  if (e != cudaSuccess) {
    lq_set_global_error(std::string("lq_apply_MdagM_static: launch: ") + cudaGetErrorString(e));
    return LQ_ERR_CUDA;
  }
  return LQ_OK;
}
