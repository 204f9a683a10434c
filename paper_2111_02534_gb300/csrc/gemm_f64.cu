// FP64 launchers of the mode-product GEMM (gemm_kernel.cuh): the H-apply of Eq.
// tensor_op1D / Eq. tensor_op2D with V and the shift fused into the epilogue, and the
// fast-diagonalisation preconditioner of Sec. 4.2 with the division fused.
//
// GB300 has no FP64 tensor-core path (tcgen05 has no f64 kind), so these run on the
// FP64 FMA pipe, which they keep busy on every active cycle.
#include "gemm_kernel.cuh"

namespace tps {

gemm::TileCache &gemm::tile_cache() {
  static TileCache cache;
  return cache;
}

using gemm::GemmArgs;
using gemm::base_args;
using gemm::left;

namespace {
// How the products of an operator share their K (GemmArgs::split).  The order in which a
// product's terms are added follows from it, so it is chosen by the operator alone: a vector's
// result has the same bits whatever the number of vectors in the call.
//  * 8 for 1D operators (K is the grid size) and small 2D ones, whose few outputs leave schedulers
//    idle otherwise: 64 x 64, 1 vector 9 us, 17 with 2; 6^2 x 20^2 19 and 23.
//  * 2 for 2D operators: K is short, and eight pieces cost seven additions for each output of 12
//    to 64 products.  H-apply with 2, 8 and tiled, 8 vectors: 16^4 80, 132 and 124 us; 24^4 533,
//    638 and 844; 36^4 4.37, 4.64 and 5.88 ms; 48^4 13.6, 18.1 and 14.2.
//  * 0, the tiled kernel, for modes that fill its tiles: 32^4, 8 vectors 1.82 ms, 1.85 with 2
//    (1 vector 0.27 and 0.25); 64^4, 1 vector 7.04 and 7.12.
int f64_split(const DevOperator &op) {
  if (op.nmodes == 2 || op.N < (1LL << 15)) return 8;
  for (int k = 0; k < 4; ++k)
    if (op.n[k] % 32) return 2;
  return 0;
}
inline void gemm64(GemmArgs g, int split, cudaStream_t s) {
  g.split = split;
  gemm::gemm<double, double, double, double>(g, s);
}
inline void right64(const double *A, long long rows, int n, const double *B, double *C, int split,
                    cudaStream_t s) {
  gemm::right_chunked<double, double, double, double>(A, rows, n, B, C, s, split);
}
}  // namespace

void launch_apply_h(const DevOperator &op, const double *psi, double *out, int nvec,
                    const double *theta_dev, double theta, cudaStream_t s) {
  if (nvec <= 0) return;
  const int split = f64_split(op);
  if (op.nmodes == 2) {
    const int nx = op.n[0], ny = op.n[1];
    GemmArgs g = base_args();
    g.M = nx;
    g.Nc = ny;
    g.batch = nvec;
    g.nphase = 2;
    g.K[0] = nx;
    g.A[0] = {op.K[0], nx, 0};
    g.B[0] = {psi, ny, op.N};
    g.K[1] = ny;
    g.A[1] = {psi, ny, op.N};
    g.B[1] = {op.KT[1], ny, 0};
    g.C = out;
    g.ldc = ny;
    g.bsc = op.N;
    g.epi = gemm::EPI_HAPPLY;
    g.E = {psi, ny, op.N};
    g.V = op.V;
    g.ldv = ny;
    g.vbs = 0;
    g.vmod = 1;
    g.theta = theta_dev;
    g.theta_div = 1;
    g.theta0 = theta;
    gemm64(g, split, s);
    return;
  }
  // 2D: [v][x1][x2][y1][y2]
  const int n0 = op.n[0], n1 = op.n[1], n2 = op.n[2], n3 = op.n[3];
  const long long s23 = (long long)n2 * n3, s123 = (long long)n1 * s23;
  {  // fused y1 + y2 products over every (v, x1, x2) slab, V and theta in the epilogue
    GemmArgs g = base_args();
    g.M = n2;
    g.Nc = n3;
    g.batch = nvec * n0 * n1;
    g.nphase = 2;
    g.K[0] = n2;
    g.A[0] = {op.K[2], n2, 0};
    g.B[0] = {psi, n3, s23};
    g.K[1] = n3;
    g.A[1] = {psi, n3, s23};
    g.B[1] = {op.KT[3], n3, 0};
    g.C = out;
    g.ldc = n3;
    g.bsc = s23;
    g.epi = gemm::EPI_HAPPLY;
    g.E = {psi, n3, s23};
    g.V = op.V;
    g.ldv = n3;
    g.vbs = s23;
    g.vmod = (long long)n0 * n1;
    g.theta = theta_dev;
    g.theta_div = (long long)n0 * n1;
    g.theta0 = theta;
    gemm64(g, split, s);
  }
  {  // x2 product, accumulated
    GemmArgs g = left(op.K[1], n1, psi, s23, s23, s123, out, nvec * n0);
    g.epi = gemm::EPI_ACCUM;
    gemm64(g, split, s);
  }
  {  // x1 product, accumulated
    GemmArgs g = left(op.K[0], n0, psi, s123, s123, op.N, out, nvec);
    g.epi = gemm::EPI_ACCUM;
    gemm64(g, split, s);
  }
}

void launch_apply_prec(const DevOperator &op, const double *r, double *out, int nvec,
                       double sigma, ApplyWorkspace &ws, cudaStream_t s) {
  if (nvec <= 0) return;
  const int split = f64_split(op);
  double *t0 = ws.t0, *t1 = ws.t1;
  if (op.nmodes == 2) {
    const int nx = op.n[0], ny = op.n[1];
    right64(r, (long long)nvec * nx, ny, op.S[1], t0, split, s);                   // R S_y
    GemmArgs g = left(op.ST[0], nx, t0, ny, ny, op.N, t1, nvec);           // S_x^T (R S_y)
    g.epi = gemm::EPI_DIVIDE2;
    g.lamM = op.lam[0];
    g.lamN = op.lam[1];
    g.sigma = sigma;
    gemm64(g, split, s);
    gemm64(left(op.S[0], nx, t1, ny, ny, op.N, t0, nvec), split, s);               // S_x (..)
    right64(t0, (long long)nvec * nx, ny, op.ST[1], out, split, s);                // (..) S_y^T
    return;
  }
  const int n0 = op.n[0], n1 = op.n[1], n2 = op.n[2], n3 = op.n[3];
  const long long s23 = (long long)n2 * n3, s123 = (long long)n1 * s23;
  right64(r, (long long)nvec * n0 * n1 * n2, n3, op.S[3], t0, split, s);
  gemm64(left(op.ST[2], n2, t0, n3, n3, s23, t1, nvec * n0 * n1), split, s);
  gemm64(left(op.ST[1], n1, t1, s23, s23, s123, t0, nvec * n0), split, s);
  {
    GemmArgs g = left(op.ST[0], n0, t0, s123, s123, op.N, t1, nvec);
    g.epi = gemm::EPI_DIVIDE4;
    g.lamM = op.lam[0];
    g.lamN = op.lam[1];
    g.lam2 = op.lam[2];
    g.lam3 = op.lam[3];
    g.n2 = n2;
    g.n3 = n3;
    g.sigma = sigma;
    gemm64(g, split, s);
  }
  gemm64(left(op.S[0], n0, t1, s123, s123, op.N, t0, nvec), split, s);
  gemm64(left(op.S[1], n1, t0, s23, s23, s123, t1, nvec * n0), split, s);
  gemm64(left(op.S[2], n2, t1, n3, n3, s23, t0, nvec * n0 * n1), split, s);
  right64(t0, (long long)nvec * n0 * n1 * n2, n3, op.ST[3], out, split, s);
}

}  // namespace tps
