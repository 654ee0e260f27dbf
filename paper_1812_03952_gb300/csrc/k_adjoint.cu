// Adjoint kernels: transposed block SpMV (a gather, no explicit transpose),
// block transposition of values, the pattern-restricted outer product
// -lambda_i x_j^T and its chain through the harmonic transmissibility to
// theta = ln k.
#include "trs_kernels.cuh"

namespace trs {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

inline unsigned grid_of(int64_t n) { return (unsigned)((n + kThreads - 1) / kThreads); }

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// y_i = alpha * sum_j (A_ji)^T x_j + beta * y_i.  For a cell row the blocks
// A_ji of its 7-point neighbours sit in the neighbour's opposite slot; blocks
// of the tail are found through the column lists tc_*.
template <int B>
__global__ void __launch_bounds__(kThreads) k_spmv_t(MatView<double> A, const int64_t *tc_ptr, const int64_t *tc_src,
                                                     const int32_t *tc_row, const double *x, double *y, double alpha,
                                                     double beta, int64_t cell_blocks) {
  pdl_enter();
  constexpr int BB = B * B;
  const int64_t nc = A.g.nc;
  if (blockIdx.x < cell_blocks) {
    const int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x;
    if (i >= nc) return;
    double acc[B] = {};
    const unsigned m = A.emask[i];
#pragma unroll
    for (int s = 0; s < kSlots; s++) {
      if (!((m >> s) & 1u)) continue;
      const int64_t j = i + A.g.off[s];
      const int so = kSlots - 1 - s;
      const double *blk = A.ell + (int64_t)so * BB * nc + j;
#pragma unroll
      for (int r = 0; r < B; r++) {
        const double xr = x[j * B + r];
#pragma unroll
        for (int c = 0; c < B; c++) acc[c] = fma(blk[(int64_t)(r * B + c) * nc], xr, acc[c]);
      }
    }
    for (int64_t t = tc_ptr[i]; t < tc_ptr[i + 1]; t++) {
      const int64_t j = tc_row[t];
      const double *blk = A.tval + tc_src[t] * BB;
#pragma unroll
      for (int r = 0; r < B; r++)
#pragma unroll
        for (int c = 0; c < B; c++) acc[c] = fma(blk[r * B + c], x[j * B + r], acc[c]);
    }
#pragma unroll
    for (int c = 0; c < B; c++)
      y[i * B + c] = (beta == 0.0) ? alpha * acc[c] : fma(alpha, acc[c], beta * y[i * B + c]);
  } else {
    const int lane = threadIdx.x & 31;
    const int64_t i = nc + (blockIdx.x - cell_blocks) * (int64_t)kWarps + (threadIdx.x >> 5);
    if (i >= A.g.n_rows) return;
    double acc[B] = {};
    for (int64_t t = tc_ptr[i] + lane; t < tc_ptr[i + 1]; t += 32) {
      const int64_t j = tc_row[t];
      const double *blk = A.tval + tc_src[t] * BB;
#pragma unroll
      for (int r = 0; r < B; r++)
#pragma unroll
        for (int c = 0; c < B; c++) acc[c] = fma(blk[r * B + c], x[j * B + r], acc[c]);
    }
#pragma unroll
    for (int c = 0; c < B; c++) acc[c] = warp_sum(acc[c]);
    if (lane == 0)
#pragma unroll
      for (int c = 0; c < B; c++)
        y[i * B + c] = (beta == 0.0) ? alpha * acc[c] : fma(alpha, acc[c], beta * y[i * B + c]);
  }
}

// Cell part of A^T: the block in slot s of cell i is the transpose of the
// block in the opposite slot of cell j = i + off[s] (the slots are geometric,
// so that block is always in A's ELL part).  One thread per (slot, cell):
// for a fixed element the reads and the writes are both unit-stride in i.
template <int B>
__global__ void __launch_bounds__(kThreads) k_transpose_ell(Geom g, const uint8_t *__restrict__ emask_dst,
                                                            const double *__restrict__ ell_src,
                                                            double *__restrict__ ell_dst) {
  pdl_enter();
  constexpr int BB = B * B;
  const int64_t nc = g.nc;
  const int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x;
  if (i >= nc) return;
  const int s = blockIdx.y;
  double *dst = ell_dst + (int64_t)s * BB * nc + i;
  if ((emask_dst[i] >> s) & 1u) {
    const double *src = ell_src + (int64_t)(kSlots - 1 - s) * BB * nc + (i + g.off[s]);
#pragma unroll
    for (int r = 0; r < B; r++)
#pragma unroll
      for (int c = 0; c < B; c++) dst[(int64_t)(r * B + c) * nc] = src[(int64_t)(c * B + r) * nc];
  } else {
#pragma unroll
    for (int e = 0; e < BB; e++) dst[(int64_t)e * nc] = 0.0;
  }
}

// Tail part of A^T: entry t of the tail is canonical block tq[t]; its source
// is canonical block src_canon[tq[t]] of A, wherever A keeps it.
__global__ void __launch_bounds__(kThreads) k_transpose_tail(int b, int64_t ntail, const int64_t *__restrict__ tq,
                                                             const int64_t *__restrict__ src_canon,
                                                             const int64_t *__restrict__ map_src,
                                                             const double *__restrict__ ell_src,
                                                             const double *__restrict__ tval_src, int64_t nc,
                                                             double *__restrict__ tval_dst) {
  pdl_enter();
  const int bb = b * b;
  const int64_t idx = blockIdx.x * (int64_t)kThreads + threadIdx.x;
  if (idx >= ntail * bb) return;
  const int64_t t = idx / bb;
  const int e = (int)(idx % bb), r = e / b, c = e % b;
  const int64_t ls = map_src[src_canon[tq[t]]];
  const int es = c * b + r;  // transposed element
  tval_dst[idx] = ls < kSlots * nc ? ell_src[((ls / nc) * bb + es) * nc + ls % nc]
                                   : tval_src[(ls - kSlots * nc) * bb + es];
}

// dA_p = -lambda_i x_j^T of pattern entry p = (i, j), a block of threads per
// kOuterRun entries: their rows and columns are read once, and the index
// arithmetic is 32-bit.  Bound by the FP64 unit (one product per value at 2 per
// clock and SM: 43 us for the 25 million values of a 100x80x50 grid with b = 3;
// 118 us with a thread per
// value and 64-bit index arithmetic, now 62).
constexpr int kOuterRun = 256;

template <int B>
__global__ void __launch_bounds__(kThreads) k_outer_product(int64_t nnzb, const int32_t *urow, const int32_t *ucol,
                                                            const double *lambda, const double *x, double *dA) {
  pdl_enter();
  constexpr int BB = B * B;
  __shared__ int32_t row[kOuterRun], col[kOuterRun];
  const int64_t p0 = blockIdx.x * (int64_t)kOuterRun;
  const int np = (int)(nnzb - p0 < kOuterRun ? nnzb - p0 : kOuterRun);
  if ((int)threadIdx.x < np) {
    row[threadIdx.x] = urow[p0 + threadIdx.x];
    col[threadIdx.x] = ucol[p0 + threadIdx.x];
  }
  __syncthreads();
  double *out = dA + p0 * BB;
#pragma unroll 4
  for (int e = threadIdx.x; e < np * BB; e += kThreads) {
    const int p = e / BB, rc = e % BB;
    out[e] = -(lambda[(int64_t)row[p] * B + rc / B] * x[(int64_t)col[p] * B + rc % B]);
  }
}

// dL/dtheta_i = sum over the faces f of i of dL/dT_f * T_f * k_j / (k_i + k_j),
// dL/dT_f = lambda_i^T M_if (x_j - x_i) + lambda_j^T M_jf' (x_i - x_j): the
// contraction of -lambda x^T with dA/dT_f (A_ij = -T M_if, A_ii += T M_if, and
// the same from cell j); T_f the harmonic mean, so T_f k_j / (k_i + k_j) =
// 2 c k_i r_j^2 with r_j = k_j / (k_i + k_j).
//
// Bound by the FP64 unit (2 operations per clock and SM).  A block of threads
// takes a tile of 8 x 8 x 4 cells and goes over its faces, its boundary's
// included (3.5 per cell; a thread per cell does 6): a face's contraction, its
// one division and both its cells' terms are formed once and left in shared
// memory, one place per cell and face, and every cell sums its own in slot
// order, so no sum depends on timing and no memory outside the tile is written.
// exp is taken once per cell of the tile and its halo.  The dots run over the
// columns first (B^2 + B operations a side instead of 2 B^2).  100x80x50,
// b = 3: 297 us with a thread per cell, now 149.  A face that A does not store
// (a sealed fault, an inactive cell) adds nothing; its mask byte is looked at
// last, so that no load waits for it.
constexpr int kTileX = 8, kTileY = 8, kTileZ = 4, kTileCells = kTileX * kTileY * kTileZ;
constexpr int kTileThreads = 128;
constexpr int kFacesX = (kTileX + 1) * kTileY * kTileZ, kFacesY = kTileX * (kTileY + 1) * kTileZ,
              kFacesZ = kTileX * kTileY * (kTileZ + 1);
constexpr int kHaloX = kTileX + 2, kHaloY = kTileY + 2, kHaloZ = kTileZ + 2;

template <int B>
__global__ void __launch_bounds__(kTileThreads) k_chain_theta(Geom g, int tiles_x, int tiles_y, const uint8_t *emask,
                                                              const double *perm, int is_log, double kvkh, double c_t,
                                                              const double *M, const double *lambda, const double *x,
                                                              double *dtheta) {
  pdl_enter();
  constexpr int BB = B * B;
  __shared__ double kk[kHaloZ][kHaloY][kHaloX];
  __shared__ double part[6][kTileCells];
  const int tile = (int)blockIdx.x;
  const int x0 = tile % tiles_x * kTileX, y0 = tile / tiles_x % tiles_y * kTileY,
            z0 = tile / (tiles_x * tiles_y) * kTileZ;
  auto inside = [&](int cx, int cy, int cz) {
    return cx >= 0 && cx < g.nx && cy >= 0 && cy < g.ny && cz >= 0 && cz < g.nz;
  };
  auto cell = [&](int cx, int cy, int cz) { return ((int64_t)cz * g.ny + cy) * g.nx + cx; };
  for (int e = threadIdx.x; e < kHaloX * kHaloY * kHaloZ; e += kTileThreads) {
    const int hx = e % kHaloX, hy = e / kHaloX % kHaloY, hz = e / (kHaloX * kHaloY);
    const int cx = x0 + hx - 1, cy = y0 + hy - 1, cz = z0 + hz - 1;
    double v = 0.0;
    if (inside(cx, cy, cz)) {
      v = perm[cell(cx, cy, cz)];
      if (is_log) v = exp(v);
    }
    kk[hz][hy][hx] = v;
  }
  __syncthreads();
  for (int f = threadIdx.x; f < kFacesX + kFacesY + kFacesZ; f += kTileThreads) {
    // the lower cell of the face, from -1 along its direction a
    int lx, ly, lz, a;
    if (f < kFacesX) {
      a = 0; lx = f % (kTileX + 1) - 1; ly = f / (kTileX + 1) % kTileY; lz = f / ((kTileX + 1) * kTileY);
    } else if (f < kFacesX + kFacesY) {
      const int h = f - kFacesX;
      a = 1; lx = h % kTileX; ly = h / kTileX % (kTileY + 1) - 1; lz = h / (kTileX * (kTileY + 1));
    } else {
      const int h = f - kFacesX - kFacesY;
      a = 2; lx = h % kTileX; ly = h / kTileX % kTileY; lz = h / (kTileX * kTileY) - 1;
    }
    const int ux = lx + (a == 0), uy = ly + (a == 1), uz = lz + (a == 2);
    if (!inside(x0 + lx, y0 + ly, z0 + lz) || !inside(x0 + ux, y0 + uy, z0 + uz)) continue;
    const int64_t i = cell(x0 + lx, y0 + ly, z0 + lz), j = cell(x0 + ux, y0 + uy, z0 + uz);
    const double ki = kk[lz + 1][ly + 1][lx + 1], kj = kk[uz + 1][uy + 1][ux + 1];
    const double den = ki + kj;
    const bool stored = (emask[i] >> (kSelf + 1 + a)) & 1u;
    double gi = 0.0, gj = 0.0;
    if (den != 0.0) {
      const double *Mi = M + (i * 6 + 3 + a) * BB, *Mj = M + (j * 6 + 2 - a) * BB;
      double dx[B], dLdT = 0.0;
#pragma unroll
      for (int c = 0; c < B; c++) dx[c] = x[j * B + c] - x[i * B + c];
#pragma unroll
      for (int r = 0; r < B; r++) {
        double si = Mi[r * B] * dx[0], sj = Mj[r * B] * dx[0];
#pragma unroll
        for (int c = 1; c < B; c++) {
          si = fma(Mi[r * B + c], dx[c], si);
          sj = fma(Mj[r * B + c], dx[c], sj);
        }
        dLdT = fma(lambda[i * B + r], si, dLdT);
        dLdT = fma(-lambda[j * B + r], sj, dLdT);
      }
      double ri, rj;
      if (fabs(den) > 1e-290) {
        const double inv = 1.0 / den;
        ri = ki * inv;
        rj = kj * inv;
      } else {   // 1 / den would overflow
        ri = ki / den;
        rj = kj / den;
      }
      // T = c 2 k_i k_j / (k_i + k_j)
      const double w = dLdT * ((a == 2 ? c_t * kvkh : c_t) * (2.0 * ki * rj));
      gi = stored ? w * rj : 0.0;
      gj = stored ? w * ri : 0.0;
    }
    auto inner = [&](int cx, int cy, int cz) {
      return cx >= 0 && cx < kTileX && cy >= 0 && cy < kTileY && cz >= 0 && cz < kTileZ;
    };
    if (inner(lx, ly, lz)) part[3 + a][(lz * kTileY + ly) * kTileX + lx] = gi;
    if (inner(ux, uy, uz)) part[2 - a][(uz * kTileY + uy) * kTileX + ux] = gj;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < kTileCells; e += kTileThreads) {
    const int cx = x0 + e % kTileX, cy = y0 + e / kTileX % kTileY, cz = z0 + e / (kTileX * kTileY);
    if (!inside(cx, cy, cz)) continue;
    const bool on[6] = {cz > 0, cy > 0, cx > 0, cx + 1 < g.nx, cy + 1 < g.ny, cz + 1 < g.nz};
    double acc = 0.0;
#pragma unroll
    for (int d = 0; d < 6; d++)
      if (on[d]) acc = acc + part[d][e];
    dtheta[cell(cx, cy, cz)] = acc;
  }
}

}  // namespace

void launch_spmv_t(int b, const trs_bsr &A, const double *x, double *y, double alpha, double beta,
                   cudaStream_t s) {
  const int64_t cb = (A.g.nc + kThreads - 1) / kThreads;
  const int64_t lb = (A.g.n_rows - A.g.nc + kWarps - 1) / kWarps;
  if (cb + lb == 0) return;
  TRS_DISPATCH_B(b, launch_pdl(k_spmv_t<B>, (unsigned)(cb + lb), kThreads, 0, s, A.view(), A.tc_ptr.p, A.tc_src.p,
                                                                         A.tc_row.p, x, y, alpha, beta, cb));
  TRS_LAUNCHED();
}

void launch_transpose_values(const trs_bsr &A, trs_bsr &AT, cudaStream_t s) {
  const int64_t nc = AT.g.nc;
  if (nc) {
    TRS_DISPATCH_B(A.b, launch_pdl(k_transpose_ell<B>, dim3(grid_of(nc), kSlots), dim3(kThreads), 0, s, AT.g,
                                   (const uint8_t *)AT.emask.p, (const double *)A.ell.p, AT.ell.p));
  }
  if (AT.ntail) {
    const int bb = A.b * A.b;
    launch_pdl(k_transpose_tail, grid_of(AT.ntail * bb), kThreads, 0, s, A.b, AT.ntail, (const int64_t *)AT.ttail.p,
               (const int64_t *)AT.tsrc.p, (const int64_t *)A.map.p, (const double *)A.ell.p,
               (const double *)A.tval.p, A.g.nc, AT.tval.p);
  }
  TRS_LAUNCHED();
}

void launch_outer_product(int b, const trs_bsr &A, const double *lambda, const double *x, double *dA,
                          cudaStream_t s) {
  if (!A.nnzb) return;
  TRS_DISPATCH_B(b, launch_pdl(k_outer_product<B>, (unsigned)((A.nnzb + kOuterRun - 1) / kOuterRun), kThreads, 0, s,
                               A.nnzb, A.urow.p, A.ucol.p, lambda, x, dA));
  TRS_LAUNCHED();
}

void launch_chain_theta(int b, const trs_bsr &A, const double *perm, int perm_is_log, double kvkh, double c_t,
                        const double *M, const double *lambda, const double *x, double *dtheta, cudaStream_t s) {
  if (!A.g.nc) return;
  const int tx = (A.g.nx + kTileX - 1) / kTileX, ty = (A.g.ny + kTileY - 1) / kTileY,
            tz = (A.g.nz + kTileZ - 1) / kTileZ;
  TRS_DISPATCH_B(b, launch_pdl(k_chain_theta<B>, (unsigned)((int64_t)tx * ty * tz), kTileThreads, 0, s, A.g, tx, ty,
                               A.emask.p, perm, perm_is_log, kvkh, c_t, M, lambda, x, dtheta));
  TRS_LAUNCHED();
}

}  // namespace trs
