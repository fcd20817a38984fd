// Workspace of the energy steps' stencil form (energy_rows.cuh): host code only.
#pragma once
#include <cuda_runtime_api.h>

#include <cstddef>

namespace tn {

struct alignas(32) WedgeFlow {  // per-wedge velocity terms of the energy rows
  double vt, l0, l1, mu;
};
struct RowsWorkspace {
  double* rows = nullptr;
  WedgeFlow* wq = nullptr;
};

// Whether the workspace is there: allocated with the first call that finds room for it and kept with the mesh; not
// taken (element residuals then) when it exceeds a quarter of the memory that is free at this call, or while the
// stream is being captured.  Nothing is remembered of a refusal: the next call asks again.
inline bool rows_ready(RowsWorkspace& W, size_t rows_bytes, size_t wedge_bytes, cudaStream_t st) {
  if (W.rows) return true;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
    cudaGetLastError();
    return false;
  }
  size_t fr = 0, tot = 0;
  bool ok = cudaMemGetInfo(&fr, &tot) == cudaSuccess && rows_bytes + wedge_bytes <= fr / 4;
  ok = ok && cudaMalloc((void**)&W.rows, rows_bytes) == cudaSuccess;
  if (ok && cudaMalloc((void**)&W.wq, wedge_bytes) != cudaSuccess) {
    cudaFree(W.rows);
    ok = false;
  }
  if (!ok) W = RowsWorkspace{};
  cudaGetLastError();
  return ok;
}

}  // namespace tn
