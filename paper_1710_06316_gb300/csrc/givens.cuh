// givens.cuh -- Givens update of the GMRES Hessenberg matrix on the device: by one thread on
// global memory, and by a block through shared memory.  H is stored by columns of m + 1.
#pragma once

namespace afmpb {

// Givens update of Hessenberg column j: the new column from hcol, the earlier rotations
// applied, a new rotation zeroing its subdiagonal, the residual estimate |g[j + 1]|.
__device__ __forceinline__ void givens_update(int j, int m, const double *__restrict__ hcol, double *__restrict__ H,
                                              double *__restrict__ cs, double *__restrict__ sn, double *__restrict__ g,
                                              double *__restrict__ res) {
  double *col = H + (int64_t)j * (m + 1);
  for (int i = 0; i <= j + 1; ++i) col[i] = hcol[i];
  for (int i = 0; i < j; ++i) {
    const double a = col[i], b = col[i + 1];
    col[i] = cs[i] * a + sn[i] * b;
    col[i + 1] = -sn[i] * a + cs[i] * b;
  }
  const double a = col[j], b = col[j + 1];
  const double den = hypot(a, b);
  cs[j] = den > 0 ? a / den : 1.0;
  sn[j] = den > 0 ? b / den : 0.0;
  col[j] = den;
  col[j + 1] = 0.0;
  g[j + 1] = -sn[j] * g[j];
  g[j] = cs[j] * g[j];
  res[0] = fabs(g[j + 1]);
}

// givens_update by a block: column, rotations and the new entry pass through shared memory
// (a thread on global memory waits for each of the column's j dependent updates).
constexpr int kGivensShared = 256;
__device__ __forceinline__ void givens_update_block(int j, int m, double nrm, double *__restrict__ hcol,
                                                    double *__restrict__ H, double *__restrict__ cs,
                                                    double *__restrict__ sn, double *__restrict__ g,
                                                    double *__restrict__ res) {
  __shared__ double col[kGivensShared + 1], c[kGivensShared], z[kGivensShared];
  if (threadIdx.x == 0) hcol[j + 1] = nrm;
  if (j >= kGivensShared) {
    __syncthreads();
    if (threadIdx.x == 0) givens_update(j, m, hcol, H, cs, sn, g, res);
    __syncthreads();
    return;
  }
  for (int i = threadIdx.x; i < j; i += blockDim.x) {
    c[i] = cs[i];
    z[i] = sn[i];
  }
  for (int i = threadIdx.x; i <= j; i += blockDim.x) col[i] = hcol[i];
  __syncthreads();
  if (threadIdx.x == 0) {
    double a = col[0];
    for (int i = 0; i < j; ++i) {                       // a: the rotated entry i so far
      const double b = col[i + 1];
      col[i] = c[i] * a + z[i] * b;
      a = -z[i] * a + c[i] * b;
    }
    const double den = hypot(a, nrm), gj = g[j];
    const double cj = den > 0 ? a / den : 1.0, sj = den > 0 ? nrm / den : 0.0;
    col[j] = den;
    cs[j] = cj;
    sn[j] = sj;
    g[j + 1] = -sj * gj;
    g[j] = cj * gj;
    res[0] = fabs(sj * gj);
  }
  __syncthreads();
  double *out = H + (int64_t)j * (m + 1);
  for (int i = threadIdx.x; i <= j + 1; i += blockDim.x) out[i] = i <= j ? col[i] : 0.0;
}

}  // namespace afmpb
