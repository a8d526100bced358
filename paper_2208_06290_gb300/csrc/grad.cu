// Small kernels of the gradient of  loss = sum_j b_j^T A^{-1} b_j + log|det A|
// with respect to b, the leaf blocks D_b and the bases U_big, V_big
// (the sequencing is in api.cu, hodlr_grad).
#include "hodlr_internal.cuh"

namespace hodlr {

// Identity blocks: E(b*m + i, j) = delta_ij for every leaf b (N x m, ld N).
__global__ void leaf_identity_kernel(int64_t N, int m, double* E) {
  const int j = blockIdx.y;
  for (int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; row < N; row += (int64_t)gridDim.x * blockDim.x)
    E[(int64_t)j * N + row] = (row % m) == j ? 1.0 : 0.0;
}

cudaError_t launch_leaf_identity(int64_t N, int m, double* E, cudaStream_t s) {
  ProfScope prof_(KC_VECTOR, s);
  note_work(8.0 * N * m, 0.0);
  int64_t b = (N + 255) / 256;
  dim3 grid((unsigned)(b < 4096 ? b : 4096), m);
  { leaf_identity_kernel<<<grid, 256, 0, s>>>(N, m, E); note_launches(1); }
  return cudaGetLastError();
}

// out_b(i, j) = beta * out_b(i, j) + alpha * sum_t A(b m + i, t) B(b m + j, t)
//               + (Tadd ? Tadd(b m + j, i) : 0)          for every leaf b,
// out in the leaf-block layout of D (column-major m x m blocks), A and B
// N x K column-major, Tadd N x m column-major (ld N).
template <typename TB>
cudaError_t launch_leaf_outer(int64_t N, int m, int K, const double* A, int64_t lda, const TB* B, int64_t ldb,
                              double alpha, double beta, const double* Tadd, double* out, cudaStream_t s) {
  ProfScope prof_(KC_LEAF_MATVEC, s);
  note_work((8.0 + sizeof(TB)) * (double)N * K +
                8.0 * ((double)N * m * (beta != 0.0 ? 2 : 1) + (Tadd ? (double)N * m : 0.0)),
            2.0 * (double)N * m * K);
  return launch_leaf_outer_split(N, m, K, A, lda, B, ldb, alpha, beta, Tadd, out, s);
}
template cudaError_t launch_leaf_outer<double>(int64_t, int, int, const double*, int64_t, const double*, int64_t,
                                               double, double, const double*, double*, cudaStream_t);
template cudaError_t launch_leaf_outer<float>(int64_t, int, int, const double*, int64_t, const float*, int64_t,
                                              double, double, const double*, double*, cudaStream_t);

// H_alpha for the children of every parent at child level c, from
// G = K~^{-T}: the first child gets G21 = G(r:2r, 0:r), the second G12 =
// G(0:r, r:2r). Written as r x r column-major slots per child (node index),
// H and, if HT != null, H^T.
__global__ void coupling_h_kernel(int r, const double* __restrict__ Kinv, double* __restrict__ H,
                                  double* __restrict__ HT) {
  const int n = 2 * r;
  const int64_t j = blockIdx.x;
  const double* Kj = Kinv + (size_t)j * n * n;
  for (int e = threadIdx.x; e < 2 * r * r; e += blockDim.x) {
    const int child = e / (r * r);
    const int a = (e % (r * r)) % r, b = (e % (r * r)) / r;
    // G(p, q) = Kinv(q, p) = Kj[p * n + q]
    const double v = child == 0 ? Kj[(size_t)(r + a) * n + b] : Kj[(size_t)a * n + r + b];
    const int64_t node = 2 * j + child;
    H[(size_t)node * r * r + (size_t)b * r + a] = v;
    if (HT) HT[(size_t)node * r * r + (size_t)a * r + b] = v;
  }
}

cudaError_t launch_coupling_h(const Factor& F, int c, double* H, double* HT, cudaStream_t s) {
  ProfScope prof_(KC_VECTOR, s);
  const int r = F.d.r;
  const int64_t parents = (int64_t)1 << (c - 1);
  note_work(8.0 * parents * (4.0 * r * r + 4.0 * r * r), 0.0);
  { coupling_h_kernel<<<(unsigned)parents, 128, 0, s>>>(r, F.K + F.Koff[c] * 4 * r * r, H, HT); note_launches(1); }
  return cudaGetLastError();
}

}  // namespace hodlr
