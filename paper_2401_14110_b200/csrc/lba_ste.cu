// Re-computation passes for the fine-grained straight-through estimators (Sec. 4, App. D of the paper): the
// forward chain of every output is replayed with the tracking variants of the scalar kernel, which report
// the last overflow (recursive estimator) or one bit per FMAq step (overflow and difference estimators).
#include "lba_kernel.cuh"

namespace lba {

namespace {

template <int BM, int BN, int QM, int ORD, int LD, int TRACK>
cudaError_t launch_tile(const Problem& p, cudaStream_t stream) {
  constexpr int TM = 4, TN = 4;
  const dim3 grid((unsigned)((p.M + BM - 1) / BM), (unsigned)((p.N + BN - 1) / BN), 1);
  lba_contract_kernel<BM, BN, TM, TN, QM, ORD, LD, TRACK><<<grid, (BM / TM) * (BN / TN), 0, stream>>>(p);
  return cudaGetLastError();
}

template <int QM, int ORD, int LD, int TRACK>
cudaError_t launch(bool small, const Problem& p, cudaStream_t stream) {
  if constexpr (TRACK == TRACK_MASK_DIFF && ORD == ORD_CHUNK_SLAB) return launch_tile<64, 64, QM, ORD, LD, TRACK>(p, stream);  // the host's only choice
  else return small ? launch_tile<32, 32, QM, ORD, LD, TRACK>(p, stream) : launch_tile<64, 64, QM, ORD, LD, TRACK>(p, stream);
}

template <int QM, int ORD, int TRACK>
cudaError_t by_loader(bool small, int load, const Problem& p, cudaStream_t stream) {
  return load == LD_GEMM_VEC ? launch<QM, ORD, LD_GEMM_VEC, TRACK>(small, p, stream)
                             : launch<QM, ORD, LD_GEMM_ROWS, TRACK>(small, p, stream);
}

template <int QM, int TRACK>
cudaError_t by_order(bool small, int ord, int load, const Problem& p, cudaStream_t stream) {
  switch (ord) {
    case ORD_SEQ: return by_loader<QM, ORD_SEQ, TRACK>(small, load, p, stream);
    case ORD_CHUNK_SLAB: return by_loader<QM, ORD_CHUNK_SLAB, TRACK>(small, load, p, stream);
    case ORD_CHUNK_ANY: return by_loader<QM, ORD_CHUNK_ANY, TRACK>(small, load, p, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

// small: the 32x32 tile; qm: QM_FLOOR_FAST (Q_prod is the flush alone) or QM_FLOOR_FULL
cudaError_t launch_last_overflow(bool small, int qm, int load, const Problem& p, cudaStream_t stream) {
  return qm == QM_FLOOR_FAST ? by_loader<QM_FLOOR_FAST, ORD_SEQ, TRACK_LAST_OF>(small, load, p, stream)
                             : by_loader<QM_FLOOR_FULL, ORD_SEQ, TRACK_LAST_OF>(small, load, p, stream);
}

// ord: ORD_SEQ, ORD_CHUNK_SLAB (chunk a multiple of the slab length) or ORD_CHUNK_ANY; diff: 0 = STE^OF, 1 = STE^DIFF
cudaError_t launch_ste_mask(bool small, int qm, int ord, int diff, int load, const Problem& p, cudaStream_t stream) {
  if (qm == QM_FLOOR_FAST)
    return diff ? by_order<QM_FLOOR_FAST, TRACK_MASK_DIFF>(small, ord, load, p, stream)
                : by_order<QM_FLOOR_FAST, TRACK_MASK_OF>(small, ord, load, p, stream);
  return diff ? by_order<QM_FLOOR_FULL, TRACK_MASK_DIFF>(small, ord, load, p, stream)
              : by_order<QM_FLOOR_FULL, TRACK_MASK_OF>(small, ord, load, p, stream);
}

}  // namespace lba
