// Overflow masks of the straight-through estimator STE^OF (App. D of the paper) from the packed kernel:
// 64x64 tile with 4x8 or 32x32 tile with 4x4 outputs per thread, floor quantisers, sequential or chunk-16 order.
#include "lba_kernel.cuh"

namespace lba {
namespace {

template <int BM, int BN, int TM, int TN, int PQ, int ORD, int LD>
cudaError_t launch_tile(const Problem& p, cudaStream_t stream) {
  const dim3 grid((unsigned)((p.M + BM - 1) / BM), (unsigned)((p.N + BN - 1) / BN), 1);
  auto kernel = lba_contract_packed_kernel<BM, BN, TM, TN, PQ, 0, ORD, LD, 1>;
  constexpr size_t smem = packed_ste_smem_bytes<BM, BN, TM, TN>();
  static_assert(smem <= 48 * 1024, "no opt-in needed");
  return launch_after(kernel, grid, (BM / TM) * (BN / TN), smem, stream, p);
}

template <int PQ, int ORD, int LD>
cudaError_t launch(bool small, const Problem& p, cudaStream_t stream) {
  return small ? launch_tile<32, 32, 4, 4, PQ, ORD, LD>(p, stream) : launch_tile<64, 64, 4, 8, PQ, ORD, LD>(p, stream);
}

template <int PQ, int ORD>
cudaError_t by_loader(bool small, int load, const Problem& p, cudaStream_t stream) {
  return load == LD_GEMM_VEC ? launch<PQ, ORD, LD_GEMM_VEC>(small, p, stream) : launch<PQ, ORD, LD_GEMM_ROWS>(small, p, stream);
}

template <int ORD>
cudaError_t by_product(bool small, int pq, int load, const Problem& p, cudaStream_t stream) {
  switch (pq) {
    case PQ_NONE: return by_loader<PQ_NONE, ORD>(small, load, p, stream);
    case PQ_MASK: return by_loader<PQ_MASK, ORD>(small, load, p, stream);
    case PQ_CUT_ANY: return by_loader<PQ_CUT_ANY, ORD>(small, load, p, stream);
    default: return by_loader<PQ_MASK_SAT, ORD>(small, load, p, stream);
  }
}

}  // namespace

// small: the 32x32 tile; pq: PackedProd; chunk16: 0 = sequential order, 1 = chunks of 16
cudaError_t launch_ste_packed(bool small, int pq, int chunk16, int load, const Problem& p, cudaStream_t stream) {
  return chunk16 ? by_product<ORD_CHUNK16>(small, pq, load, p, stream) : by_product<ORD_SEQ>(small, pq, load, p, stream);
}

}  // namespace lba
