// Boundary-element set-up (Sec. 4.3): constant elements, no nodes at the corners, 4n
// equal elements on the square, collocation at their midpoints.  The single-layer
// matrix S_mk = int_{Gamma_k} G(y_m, y) dGamma (left side of Eq. e:ubound) is assembled in
// FP64 from the closed-form element integral (Sec. 4.2).  The square's symmetries split it:
//
//  Rotation.  S is block circulant over the four sides, so a 4-point DFT over the side index gives
//  C^0 = S0+S1+S2+S3, C^2 = S0-S1+S2-S3 and A + iB, A = S0 - S2, B = S1 - S3 (n x n).
//  Reflection.  Reversing the elements of every side (J) maps side 1 to side 3: J C^0 J = C^0,
//  J C^2 J = C^2, J A J = A, J B J = -B.  On the sums and differences of mirrored elements,
//  v_e[k] = v[k] + v[n-1-k] and v_o[k] = v[k] - v[n-1-k], k < h = n / 2, each matrix X acts through
//  h x h blocks X_e = X[m][k] + X[m][n-1-k], X_o = X[m][k] - X[m][n-1-k]: (X v)_e = X_e v_e and
//  (X v)_o = X_o v_o for C^0, C^2 and A; (B v)_e = B_o v_o and (B v)_o = B_e v_e.
//
// So a matrix of this kind is stored as h rows of [C0e | C0o | C2e | C2o | Ae | Ao | Bo | Be], 4n values
// each (the folded form): half the entries and multiply-adds of the side-DFT form alone.  The
// inverse of S has the form again; its blocks are inverted once (LU with partial pivoting by
// cuSOLVER, then the triangular solves against the identity): four h x h, and A + iB, which in
// the basis diag(1, i) is the real [[Ae, -Bo], [Be, Ao]].  The inversion is set-up, not the apply's path.
#include <cusolverDn.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>
#include <vector>

#include "handle.cuh"

namespace fmmpc {

namespace {

inline unsigned nblk(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

// along-side coordinate and signed normal offset (node units) of a point, per side
__device__ __forceinline__ void side_coords_d(int side, double np1, double x, double y, double &u, double &d) {
  switch (side) {
    case 0: u = x; d = -y; break;
    case 1: u = y; d = x - np1; break;
    case 2: u = np1 - x; d = y - np1; break;
    default: u = np1 - y; d = -x; break;
  }
}

__device__ __forceinline__ double seg_log_int_d(double s1, double ell, double d) {
  const double s2 = s1 + ell;
  const double A1 = s1 * s1 + d * d, A2 = s2 * s2 + d * d;
  double v = 0.5 * (ell * log(A2) + s1 * log1p(ell * (s1 + s2) / A1)) - ell;
  if (d != 0.0) v += d * atan2(ell * d, d * d + s1 * s2);
  return v;
}

// Matrices in the folded form (rows m < h of the first block row [S0 | S1 | S2 | S3]):
//  SINGLE  S_mk = -(h/2pi) (int_k ln|y_m - y|_node ds_node + l ln h)  (physical units)
//  DOUBLE  diag I + K, K_mk = int_k dG/dn_y(y_m, y) dGamma = (1/2pi) atan2(l d, d^2 + s1 s2) with d
//          the signed normal offset of y_m from element k's line (zero on the same side): diag =
//          -1/2 the system (-1/2 I + K) mu = -(V r)|_Gamma of the double-layer correction, diag
//          = 1/2 the boundary data term of Eq. e:ubound.
enum class BemMatrix { SINGLE, DOUBLE };

// entry (m, element k of side sk), the collocation point m on side 0; a, b: h and ln h, or diag and unused
template <BemMatrix KIND>
__device__ __forceinline__ double bem_entry(int n, int m, int sk, int k, double a, double b) {
  const double ell = (n + 1.0) / n, np1 = n + 1.0;
  if (KIND == BemMatrix::DOUBLE && sk == 0) return k == m ? a : 0.0;
  double u, d;
  side_coords_d(sk, np1, (m + 0.5) * ell, 0.0, u, d);
  if (KIND == BemMatrix::SINGLE) {
    const double I = sk == 0 ? seg_log_int_d((k - m - 0.5) * ell, ell, 0.0)  // same side: exact offsets
                             : seg_log_int_d(k * ell - u, ell, d);
    return -(a / (2.0 * PI)) * (I + ell * b);
  }
  const double s1 = k * ell - u, s2 = s1 + ell;
  return atan2(ell * d, d * d + s1 * s2) / (2.0 * PI);
}

// Row m < h of the folded form, T[m] (4n values): thread per (m, k < h), the eight entries of columns k and
// n - 1 - k of every side.
template <BemMatrix KIND>
__global__ void k_bem_fold(int n, double a, double b, double *__restrict__ T) {
  const int h = n >> 1;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)h * h) return;
  const int m = (int)(t / h), k = (int)(t % h);
  double x[2][4];  // C^0, C^2, A, B at columns k and n - 1 - k
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    double s[4];
#pragma unroll 1
    for (int sk = 0; sk < 4; ++sk) s[sk] = bem_entry<KIND>(n, m, sk, j ? n - 1 - k : k, a, b);
    x[j][0] = (s[0] + s[2]) + (s[1] + s[3]);
    x[j][1] = (s[0] + s[2]) - (s[1] + s[3]);
    x[j][2] = s[0] - s[2];
    x[j][3] = s[1] - s[3];
  }
  double *o = T + (int64_t)m * 4 * n + k;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    o[(2 * q) * h] = x[0][q] + x[1][q];
    o[(2 * q + 1) * h] = x[0][q] - x[1][q];
  }
  o[6 * h] = x[0][3] - x[1][3];  // Bo
  o[7 * h] = x[0][3] + x[1][3];  // Be
}

// The blocks to invert, from the folded form: X[4] (h x h each) and M = [[Ae, -Bo], [Be, Ao]] (n x n);
// and back (the inverse's Bo is minus the upper right block).
template <bool PACK>
__global__ void k_bem_blocks(int n, double *__restrict__ T, double *__restrict__ X, double *__restrict__ M) {
  const int h = n >> 1;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)h * h) return;
  const int64_t m = t / h;
  const int k = (int)(t % h);
  double *o = T + m * 4 * n + k, *ae = M + m * n + k, *bo = ae + h, *be = M + (m + h) * n + k, *ao = be + h;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (PACK) o[q * h] = X[q * (int64_t)h * h + t];
    else X[q * (int64_t)h * h + t] = o[q * h];
  }
  if (PACK) {
    o[4 * h] = *ae;
    o[5 * h] = *ao;
    o[6 * h] = -*bo;
    o[7 * h] = *be;
  } else {
    *ae = o[4 * h];
    *ao = o[5 * h];
    *bo = -o[6 * h];
    *be = o[7 * h];
  }
}

__global__ void k_identity(int N, double *__restrict__ B) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < (int64_t)N * N) B[t] = (t / N == t % N) ? 1.0 : 0.0;
}

// |A_kk| of the N x N matrix A
__global__ void k_diag_abs(int N, const double *__restrict__ A, double *__restrict__ d) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < N) d[k] = fabs(A[(int64_t)k * N + k]);
}

#define FMMPC_CUSOLVER(call)                                                                   \
  do {                                                                                          \
    const cusolverStatus_t st_ = (call);                                                        \
    if (st_ != CUSOLVER_STATUS_SUCCESS)                                                         \
      throw ::fmmpc::Error(FMMPC_ERR_CUDA, std::string(#call) + ": cuSOLVER status " + std::to_string((int)st_)); \
  } while (0)

// One cuSOLVER handle per device for the process (creating one costs milliseconds).
cusolverDnHandle_t solver_handle() {
  static std::mutex mu;
  static std::map<int, cusolverDnHandle_t> handles;
  int dev = 0;
  FMMPC_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(mu);
  auto it = handles.find(dev);
  if (it != handles.end()) return it->second;
  cusolverDnHandle_t h = nullptr;
  FMMPC_CUSOLVER(cusolverDnCreate(&h));
  handles[dev] = h;
  return h;
}

// In-place inverse of the N x N matrix A (row-major, device), by LU with partial pivoting and the
// two triangular solves against the identity.  Row-major A is the column-major A^T, and
// inv(A^T) read row-major is inv(A), so the factorisation runs on the buffer as it is.  Returns
// the smallest |U_kk| (0 for a singular matrix).  Calls are serialised on the handle's stream.
double lu_invert(double *A, int N, cudaStream_t s, DevPool &tmp) {
  static std::mutex mu;
  std::lock_guard<std::mutex> lock(mu);  // the per-device solver handle is shared
  cusolverDnHandle_t h = solver_handle();
  FMMPC_CUSOLVER(cusolverDnSetStream(h, s));
  int lwork = 0;
  FMMPC_CUSOLVER(cusolverDnDgetrf_bufferSize(h, N, N, A, N, &lwork));
  double *work = tmp.get<double>((size_t)std::max(lwork, 1));
  int *ipiv = tmp.get<int>(N), *info = tmp.get<int>(2);
  double *dabs = tmp.get<double>(N), *B = tmp.get<double>((size_t)N * N);
  FMMPC_CUSOLVER(cusolverDnDgetrf(h, N, N, A, N, work, ipiv, info));
  k_diag_abs<<<nblk(N), 256, 0, s>>>(N, A, dabs);
  k_identity<<<nblk((int64_t)N * N), 256, 0, s>>>(N, B);
  FMMPC_LAUNCH_CHECK();
  FMMPC_CUSOLVER(cusolverDnDgetrs(h, CUBLAS_OP_N, N, N, A, N, ipiv, B, N, info + 1));
  FMMPC_CUDA(cudaMemcpyAsync(A, B, sizeof(double) * N * N, cudaMemcpyDeviceToDevice, s));
  std::vector<double> ha(N);
  int hinfo[2] = {0, 0};
  FMMPC_CUDA(cudaMemcpyAsync(ha.data(), dabs, sizeof(double) * N, cudaMemcpyDeviceToHost, s));
  FMMPC_CUDA(cudaMemcpyAsync(hinfo, info, sizeof(int) * 2, cudaMemcpyDeviceToHost, s));
  FMMPC_CUDA(cudaStreamSynchronize(s));
  if (hinfo[0] > 0) return 0.0;  // U_kk == 0 at k = info - 1
  if (hinfo[0] < 0 || hinfo[1] != 0)
    throw Error(FMMPC_ERR_CUDA, "cuSOLVER getrf/getrs: invalid argument " + std::to_string(hinfo[0] ? hinfo[0] : hinfo[1]));
  double amin = ha[0];
  for (int k = 0; k < N; ++k) amin = std::min(amin, ha[k]);
  return amin;
}

// T: the folded form of a matrix of the square's symmetry, replaced by its inverse's.  False if a
// block is singular.
bool invert_folded(int n, double *T, cudaStream_t s, DevPool &tmp) {
  const int h = n >> 1;
  double *X = tmp.get<double>((size_t)4 * h * h), *M = tmp.get<double>((size_t)n * n);
  k_bem_blocks<false><<<nblk((int64_t)h * h), 256, 0, s>>>(n, T, X, M);
  FMMPC_LAUNCH_CHECK();
  for (int q = 0; q < 4; ++q)
    if (!(lu_invert(X + (size_t)q * h * h, h, s, tmp) > 0.0)) return false;
  if (!(lu_invert(M, n, s, tmp) > 0.0)) return false;
  k_bem_blocks<true><<<nblk((int64_t)h * h), 256, 0, s>>>(n, T, X, M);
  FMMPC_LAUNCH_CHECK();
  return true;
}

}  // namespace

namespace {
// x = hi + lo, hi = fl32(x), lo = fl32(x - hi)
__global__ void k_split_f2(int64_t total, const double *__restrict__ x, float *__restrict__ hi, float *__restrict__ lo) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= total) return;
  const double v = x[t];
  const float h = (float)v;
  hi[t] = h;
  lo[t] = (float)(v - (double)h);
}
}  // namespace

void init_bem(fmmpc_handle &H, DevPool &tmp) {
  const Geo &g = H.g;
  const int n = g.n, N = g.NG;
  const size_t nt = (size_t)(n / 2) * N;  // the folded form
  cudaStream_t s = H.stream;
  H.Sinv = H.pool.get<double>(nt);
  k_bem_fold<BemMatrix::SINGLE><<<nblk((int64_t)(n / 2) * (n / 2)), 256, 0, s>>>(n, g.h, g.lnh, H.Sinv);
  FMMPC_LAUNCH_CHECK();
  if (!invert_folded(n, H.Sinv, s, tmp))
    throw Error(FMMPC_ERR_INVALID, "single-layer BEM matrix is singular for this domain");
  if (H.prec != FMMPC_PREC_FP64) {  // the single-precision forms apply it in two-word FP32
    H.Sinv_hi = H.pool.get<float>(nt);
    H.Sinv_lo = H.pool.get<float>(nt);
    k_split_f2<<<nblk((int64_t)nt), 256, 0, s>>>((int64_t)nt, H.Sinv, H.Sinv_hi, H.Sinv_lo);
    FMMPC_LAUNCH_CHECK();
  }
  FMMPC_CUDA(cudaStreamSynchronize(s));
}

// The folded form T' of S^T from T of S: the side index is reversed, so C^0, C^2 and A transpose and
// B becomes -B^T, whose folded blocks are Bo' = -Be^T, Be' = -Bo^T.
__global__ void k_bem_transpose(int n, const double *__restrict__ T, double *__restrict__ Tt) {
  const int h = n >> 1;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)h * 4 * n) return;
  const int64_t mrow = t / (4 * n);
  const int c = (int)(t % (4 * n)), blk = c / h, k = c % h;
  const int from = blk == 6 ? 7 : (blk == 7 ? 6 : blk);
  const double v = T[(int64_t)k * 4 * n + (int64_t)from * h + mrow];
  Tt[t] = blk >= 6 ? -v : v;
}

// S^{-T} for the transpose pass, formed on first use.
void init_bem_transpose(fmmpc_handle &H) {
  if (H.SinvT) return;
  const int n = H.g.n;
  const size_t nt = (size_t)(n / 2) * 4 * n;
  double *Tt = H.pool.get<double>(nt);
  k_bem_transpose<<<nblk((int64_t)nt), 256, 0, H.stream>>>(n, H.Sinv, Tt);
  FMMPC_LAUNCH_CHECK();
  FMMPC_CUDA(cudaStreamSynchronize(H.stream));
  H.SinvT = Tt;
}

// The inverse of -1/2 I + K in the folded form (the same symmetries), for the double-layer
// correction; formed on first use.
void init_bem_dl(fmmpc_handle &H) {
  if (H.Kdl_inv) return;
  const Geo &g = H.g;
  const int n = g.n, N = g.NG;
  const size_t nt = (size_t)(n / 2) * N;
  cudaStream_t s = H.stream;
  DevPool tmp;
  double *T = nullptr;
  float *th = nullptr, *tl = nullptr;
  try {
    T = H.pool.get<double>(nt);
    k_bem_fold<BemMatrix::DOUBLE><<<nblk((int64_t)(n / 2) * (n / 2)), 256, 0, s>>>(n, -0.5, 0.0, T);
    FMMPC_LAUNCH_CHECK();
    if (!invert_folded(n, T, s, tmp))
      throw Error(FMMPC_ERR_INVALID, "double-layer BEM matrix is singular for this domain");
    if (H.prec != FMMPC_PREC_FP64) {
      th = H.pool.get<float>(nt);
      tl = H.pool.get<float>(nt);
      k_split_f2<<<nblk((int64_t)nt), 256, 0, s>>>((int64_t)nt, T, th, tl);
      FMMPC_LAUNCH_CHECK();
    }
    FMMPC_CUDA(cudaStreamSynchronize(s));
    H.Kdl_inv = T;
    H.Kdl_hi = th;
    H.Kdl_lo = tl;
  } catch (...) {  // the handle keeps nothing of it
    cudaStreamSynchronize(s);
    H.pool.give_back(T, sizeof(double) * nt);
    H.pool.give_back(th, sizeof(float) * nt);
    H.pool.give_back(tl, sizeof(float) * nt);
    throw;
  }
}

// 1/2 I + K in the folded form, the boundary data term of Eq. e:ubound, for apply_bc; formed
// on its first call, in the stream's order and without a wait.  Summing the 16 n^2 atan2 of K g
// directly took 1160 us at n = 1024; the 3 n^2 multiply-adds of the folded form take 9 us.  The
// handle's stream is not being captured.  Not formed where there is no memory for it (then for good):
// the caller sums directly.
void init_bem_bc(fmmpc_handle &H) {
  if (H.Kbc || H.no_bc_tables) return;
  const int n = H.g.n;
  const size_t nt = (size_t)(n / 2) * H.g.NG, nv = (size_t)H.g.NG * H.nrhs_max;
  double *T = static_cast<double *>(H.pool.try_alloc_beside_captures(sizeof(double) * (nt + 2 * nv)));
  if (!T) {
    H.no_bc_tables = true;
    return;
  }
  k_bem_fold<BemMatrix::DOUBLE><<<nblk((int64_t)(n / 2) * (n / 2)), 256, 0, H.stream>>>(n, 0.5, 0.0, T);
  FMMPC_LAUNCH_CHECK();
  H.bc_vt = T + nt;
  H.bc_kg = H.bc_vt + nv;
  H.Kbc = T;
}

}  // namespace fmmpc
