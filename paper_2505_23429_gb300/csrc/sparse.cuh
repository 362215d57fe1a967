// Sparse MPO action with staged input rows (sparse.cu).
#pragma once
#include "kernels.cuh"

namespace a2 {

// element kinds of the stages: BF16, a value as three BF16 planes, as an FP32 pair, FP64
enum StKind { ST_BF16 = 0, ST_PLANES = 1, ST_DF = 2, ST_F64 = 3 };

// Runs the stage (geometry and meaning as for sparse_rows_apply and its variants) on the
// kernel with staged rows and returns true, or returns false, having done nothing, where the
// general kernels are the better or the only ones.  in must not overlap out.
bool sparse_staged(const SparseRows<float>& sp, const SparseGeom& g, int in_kind, const void* in,
                   long long in_plane, int out_kind, void* out, long long out_plane,
                   cudaStream_t s);

}  // namespace a2
