// gemm_tc_n64.cu -- the 64-wide launch shapes of the tensor-core integer GEMM (calls of few tiles); a
// translation unit of its own so that the parts of the GEMM compile in parallel.
#include "gemm_tc.cuh"

namespace ilw {

template <bool AF16, bool GELU>
cudaError_t run_n64(const GemmProblem &gp, const EpiParams &ep, cudaStream_t s) {
    return run<64, GELU ? (AF16 ? 5 : 4) : (AF16 ? 6 : 5), 1, AF16, false, GELU>(gp, ep, s);
}

cudaError_t run_n64_split(const GemmProblem &gp, const EpiParams &ep, cudaStream_t s) {
    return run<64, 5, kMaxBranches, false, false, false>(gp, ep, s);
}

template cudaError_t run_n64<true, true>(const GemmProblem &, const EpiParams &, cudaStream_t);
template cudaError_t run_n64<true, false>(const GemmProblem &, const EpiParams &, cudaStream_t);
template cudaError_t run_n64<false, true>(const GemmProblem &, const EpiParams &, cudaStream_t);
template cudaError_t run_n64<false, false>(const GemmProblem &, const EpiParams &, cudaStream_t);

}  // namespace ilw
