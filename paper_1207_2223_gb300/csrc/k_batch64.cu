// FP64 reliable updates of the batched solver (the CG routine of Sec. 3 over a
// batch of systems): per column r = phi - M^dag M x with the fixed-point FP64
// operator (lq_fix64.cuh), two launches for the whole batch.  The blocks of the
// one wave are shared out over the columns by volume, a block works on one
// column, and the last block of a column adds its partial sums and applies the
// per-column rule (freeze at the tolerance, restart on drift).  Columns that
// are frozen already are left alone: their x does not change any more.
#include "lq_batch.cuh"

namespace lq {

namespace {

struct FixCols {
  Geom geo[kMaxSys];
  FixGauge U[kMaxSys];
  double kappa[kMaxSys];
  int sys[kMaxCols], off[kMaxCols];
  int block0[kMaxCols + 1];        // first block of each column
  int ncols, total;
};

// a column's |r|^2 after its update
struct FinBatch {
  BatchState* st;
  int col;
  __device__ void operator()(double rr) const {
    reliable_update_column(st, col, rr);
    st->iter_since_ru = 0;
    st->halt = 0;
  }
};

template <bool RESIDUAL, SStore S, int MINB>
__global__ void __launch_bounds__(kFixBlock, MINB)
    batch_fix_kernel(const __grid_constant__ FixCols fc, SpinorRef in, SpinorRef out, SpinorRef phi, BatchState* st,
                     BatchReduce br) {
  int col = 0;
  while (col + 1 < fc.ncols && (int)blockIdx.x >= fc.block0[col + 1]) ++col;
  if (*(volatile const int*)&st->done[col]) return;     // set only after all blocks of the column passed here
  const int k = fc.sys[col], block = (int)blockIdx.x - fc.block0[col], nblocks = fc.block0[col + 1] - fc.block0[col];
  const int first = (block * (int)blockDim.x + (int)threadIdx.x) >> 1, stride = (nblocks * (int)blockDim.x) >> 1;
  double red[1] = {0.0};
  if constexpr (!RESIDUAL) {
    const FixEpiStore epi{out};
    fix_sites<false, MINB == 2 ? kFixBlock : 0>(fc.geo[k], fc.U[k], in, fc.total, fc.off[col], fc.kappa[k], epi, first, stride, red);
  } else {
    const FixEpiResidual<S, true, FinBatch, false> epi{phi, SpinorRef{nullptr, nullptr}, out, FinBatch{st, col}};
    fix_sites<true, MINB == 2 ? kFixBlock : 0>(fc.geo[k], fc.U[k], in, fc.total, fc.off[col], fc.kappa[k], epi, first, stride, red);
    const ReduceScratch rs{br.partials + (size_t)col * br.max_blocks, br.ticket + col, br.max_blocks};
    double tot[1];
    if (grid_sum<1>(red, rs, tot, block, nblocks)) epi.finalize(tot);
  }
}

template <bool RESIDUAL, SStore S>
void launch(const Batch64Args& a, FixCols fc, SpinorRef in, SpinorRef out, cudaStream_t st) {
  static std::atomic<int> waves[kFixDevices];
  const int wave = fix_wave(reinterpret_cast<const void*>(&batch_fix_kernel<RESIDUAL, S, 2>), kFixBlock, waves);
  long long pairs = 0;
  for (int c = 0; c < fc.ncols; ++c) pairs += fc.geo[fc.sys[c]].V;
  int bs = kFixBlock;                                   // smaller blocks when the batch leaves SMs idle
  while (bs > 32 && 2 * pairs < (long long)a.sms * bs) bs >>= 1;
  int n = 0;
  for (int c = 0; c < fc.ncols; ++c) {
    const int V = fc.geo[fc.sys[c]].V, need = grid_for(2 * V, bs);
    const int share = (int)((double)wave * V / (double)pairs);
    fc.block0[c] = n;
    n += std::max(1, std::min(std::min(need, share), a.br.max_blocks));
  }
  fc.block0[fc.ncols] = n;
  if (n <= a.sms) batch_fix_kernel<RESIDUAL, S, 1><<<n, bs, 0, st>>>(fc, in, out, a.phi, a.st, a.br);
  else batch_fix_kernel<RESIDUAL, S, 2><<<n, bs, fix_smem(kFixBlock), st>>>(fc, in, out, a.phi, a.st, a.br);
}

}  // namespace

void batch_true_residual(const Batch64Args& a, const BatchDesc& bd, SStore s, cudaStream_t st) {
  FixCols fc{};
  fc.total = bd.total;
  fc.ncols = bd.ncols;
  for (int k = 0; k < bd.nsys; ++k) {
    fc.geo[k] = bd.sys[k].geo;
    fc.U[k] = bd.sys[k].fix;
    fc.kappa[k] = bd.sys[k].kappa;
    for (int r = 0; r < bd.sys[k].R; ++r) {
      fc.sys[bd.sys[k].col + r] = k;
      fc.off[bd.sys[k].col + r] = bd.sys[k].off + r * bd.sys[k].geo.V;
    }
  }
  launch<false, SStore::F32>(a, fc, a.x, a.tmp, st);
  switch (s) {
    case SStore::F16: launch<true, SStore::F16>(a, fc, a.tmp, a.rlo, st); break;
    case SStore::BF16: launch<true, SStore::BF16>(a, fc, a.tmp, a.rlo, st); break;
    case SStore::I16: launch<true, SStore::I16>(a, fc, a.tmp, a.rlo, st); break;
    default: launch<true, SStore::F32>(a, fc, a.tmp, a.rlo, st); break;
  }
}

}  // namespace lq
