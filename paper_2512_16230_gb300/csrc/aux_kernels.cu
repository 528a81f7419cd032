// Dispatch of the kernels around the time step to the lattice's instantiation (io_kernels.cuh):
// population gather/scatter for I/O, the macroscopic-field readout (Eq. (2-4-2) / (2-4-1)) and the
// FP64 conservation sums; and the conversion of a cell field to the compute dtype.
#include "lbm_internal.cuh"

namespace lbm {

namespace {

lbm_status run_io(lbm_model* m, const IoCall& io) {
  switch (m->lat->kind) {
    case LBM_RD2Q13: return Launch<LBM_RD2Q13>::io(m, io);
    case LBM_RD2Q17: return Launch<LBM_RD2Q17>::io(m, io);
    case LBM_RD2Q21: return Launch<LBM_RD2Q21>::io(m, io);
    case LBM_RD2Q25: return Launch<LBM_RD2Q25>::io(m, io);
    case LBM_RD3Q33: return Launch<LBM_RD3Q33>::io(m, io);
    case LBM_RD3Q45: return Launch<LBM_RD3Q45>::io(m, io);
    case LBM_RD3Q53: return Launch<LBM_RD3Q53>::io(m, io);
    case LBM_RD2Q9: return Launch<LBM_RD2Q9>::io(m, io);
    case LBM_RD3Q27: return Launch<LBM_RD3Q27>::io(m, io);
  }
  return set_error(LBM_ERR_ARG, "unknown lattice kind");
}

template <class CT>
__global__ void k_to_compute(const double* __restrict__ src, CT* __restrict__ dst, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = CT(src[i]);
}

}  // namespace

lbm_status launch_gather(lbm_model* m, double* out) {
  return run_io(m, IoCall{IoCall::kGather, "gather launch", nullptr, out, nullptr, nullptr});
}

lbm_status launch_scatter(lbm_model* m, const double* in) {
  return run_io(m, IoCall{IoCall::kScatter, "scatter launch", in, nullptr, nullptr, nullptr});
}

lbm_status launch_fields(lbm_model* m, double* rho, double* u) {
  return run_io(m, IoCall{IoCall::kFields, "fields launch", nullptr, rho, u, nullptr});
}

lbm_status launch_phi_from_populations(lbm_model* m) {
  return run_io(m, IoCall{IoCall::kPhi, "phi launch", nullptr, nullptr, nullptr, m->phi_prev});
}

lbm_status launch_density_history(lbm_model* m) {
  return run_io(m, IoCall{IoCall::kPhi, "density history launch", nullptr, nullptr, nullptr, m->rho_hist[m->hist_cur]});
}

lbm_status launch_to_compute(lbm_model* m, const double* src, void* dst) {
  const int grid = (m->ncells + 127) / 128;
  if (m->store == LBM_F64)
    k_to_compute<double><<<grid, 128, 0, m->stream>>>(src, static_cast<double*>(dst), m->ncells);
  else
    k_to_compute<float><<<grid, 128, 0, m->stream>>>(src, static_cast<float*>(dst), m->ncells);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return cuda_error(err, "field conversion launch");
  m->launches += 1;
  return LBM_OK;
}

lbm_status launch_sums(lbm_model* m) {
  return run_io(m, IoCall{IoCall::kSums, "sums launch", nullptr, m->sums, m->partials, nullptr});
}

lbm_status launch_sums_into(lbm_model* m, double* partials, int partial_slots, double* out) {
  if (partial_slots < kRedBlocks) return set_error(LBM_ERR_ARG, "reduction scratch too small");
  return run_io(m, IoCall{IoCall::kSums, "sums launch", nullptr, out, partials, nullptr});
}

}  // namespace lbm
