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

// dA_p = -lambda_i x_j^T of pattern entry p = (i, j), a block of threads per run
// of up to kOuterRun entries: their rows and columns are read once, and the index
// arithmetic is 32-bit.  Bound by the FP64 unit (one product per value at 2 per
// clock and SM: 43 us for the 25 million values of a 100x80x50 grid with b = 3;
// 118 us with a thread per value and 64-bit index arithmetic, now 62).
constexpr int kOuterRun = 256;

template <int B>
__global__ void __launch_bounds__(kThreads) k_outer_product(int64_t nnzb, int run, const int32_t *urow,
                                                            const int32_t *ucol, const double *lambda,
                                                            const double *x, double *dA) {
  pdl_enter();
  constexpr int BB = B * B;
  __shared__ int32_t row[kOuterRun], col[kOuterRun];
  const int64_t p0 = blockIdx.x * (int64_t)run;
  const int np = (int)(nnzb - p0 < run ? nnzb - p0 : run);
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

// Matrices of up to 2^20 values (8 MB) take shorter runs, for eight blocks per SM,
// down to 4 values a thread (16x16x8, b = 5: 25.3 us a call by whole runs, now 21.6),
// in multiples of 16 entries, so that every block writes whole 128-byte lines.
// Above, a call gains 2 to 4 us of 25 to 35, but between 20 and 45 MB, where dA and
// the chain's blocks just fit one die's L2, whole runs leave more of the latter
// there: 40x40x20, b = 4, with the chain 38 us, 120 with runs of 192.
int outer_run(int64_t nnzb, int b) {
  if (nnzb * b * b > (int64_t(1) << 20)) return kOuterRun;
  const int64_t even = nnzb / (8 * 152), least = 4 * kThreads / (b * b);
  return (int)std::min<int64_t>(kOuterRun, (std::max(even, least) + 15) / 16 * 16);
}

// dL/dtheta_i = sum over the faces f of i of dL/dT_f * T_f * k_j / (k_i + k_j),
// dL/dT_f = lambda_i^T M_if (x_j - x_i) + lambda_j^T M_jf' (x_i - x_j): the
// contraction of -lambda x^T with dA/dT_f (A_ij = -T M_if, A_ii += T M_if, and
// the same from cell j); T_f the harmonic mean, so T_f k_j / (k_i + k_j) =
// 2 c k_i r_j^2 with r_j = k_j / (k_i + k_j).
//
// Bound by the FP64 unit (2 operations per clock and SM).  A block of threads
// takes a tile of up to 256 cells and goes over its faces, its boundary's
// included (3.5 per cell of an 8 x 8 x 4 tile; a thread per cell does 6): a
// face's contraction, its one division and both its cells' terms are formed once
// and left in shared memory, one place per cell and face, and every cell sums its
// own in slot order, so no sum depends on timing or on the tile, and no memory
// outside the tile is written.  exp is taken once per cell of the tile and of the
// layers around it.  The dots run over the columns first (B^2 + B operations a
// side instead of 2 B^2).  A thread's blocks of M come value by value, 4 sectors
// per 72 or 200 bytes, and have to stay in L1 meanwhile: shared memory takes 100
// KB of an SM (5 blocks), not all that would fit.  100x80x50, b = 3: 297 us with
// a thread per cell, now 132, 172 with 164 KB of shared memory (b = 5: a call of
// 701 us, now 272, 459 with 164 KB).  A face that A does not store (a sealed fault,
// an inactive cell) adds nothing; its mask byte is looked at last, so that no load
// waits for it.
constexpr int kTileCells = 256;
constexpr int kBoxX = 3, kBoxY = 3, kBoxZ = 2;   // log2 of a box's tile, 8 x 8 x 4: constants in its kernel
constexpr int kTileThreads = 128;
constexpr int kTileCarveout = 44;   // per cent of 228 KB

// Extents of a tile, powers of two (cell e of the tile: x lowest), and the
// number of tiles along x and y.
struct ChainTile {
  int sx, sy, sz;   // log2 of the extents
  int tiles_x, tiles_y;
};

// 8 x 8 x 4, but no direction longer than the grid needs; what that leaves goes
// to the others in turn, as far as they have cells, so that a section or a
// column fills its tiles like a box.  A call at b = 3 with a thread per cell, with
// 8 x 8 x 4 for every grid, and now: 1 x 1 x 400,000 155, 1967 and 81 us;
// 1 x 600 x 700 280, 903 and 128; 700 x 600 x 1 280, 151 and 119.
ChainTile chain_tile(const Geom &g) {
  const int n[3] = {g.nx, g.ny, g.nz};
  int s[3] = {kBoxX, kBoxY, kBoxZ}, spare = 0;
  for (int a = 0; a < 3; a++)
    while (s[a] > 0 && (1 << (s[a] - 1)) >= n[a]) { s[a]--; spare++; }
  for (bool more = true; spare && more;) {
    more = false;
    for (int a = 0; a < 3; a++)
      if (spare && (1 << s[a]) < n[a]) { s[a]++; spare--; more = true; }
  }
  return {s[0], s[1], s[2], ((n[0] - 1) >> s[0]) + 1, ((n[1] - 1) >> s[1]) + 1};
}

template <int B, bool BOX>
__global__ void __launch_bounds__(kTileThreads) k_chain_theta(Geom g, ChainTile t, const uint8_t *emask,
                                                              const double *perm, int is_log, double kvkh, double c_t,
                                                              const double *M, const double *lambda, const double *x,
                                                              double *dtheta) {
  pdl_enter();
  constexpr int BB = B * B;
  // permeabilities: the tile's cells, then for each direction that the tile does
  // not cover the layer before the tile and the layer after it (a tile that does
  // not cover a direction has 8, 8 and 4 cells and more along x, y and z)
  __shared__ double kk[kTileCells + 2 * (kTileCells / 8 + kTileCells / 8 + kTileCells / 4)];
  __shared__ double part[6][kTileCells];
  const int sx = BOX ? kBoxX : t.sx, sy = BOX ? kBoxY : t.sy, sz = BOX ? kBoxZ : t.sz;
  const int sxy = sx + sy, sc = sxy + sz, cells = 1 << sc;
  const int mx = (1 << sx) - 1, my = (1 << sy) - 1, mxy = (1 << sxy) - 1;
  // cells of a layer across x, y, z
  const int n0 = g.nx > 1 << sx ? cells >> sx : 0, n1 = g.ny > 1 << sy ? cells >> sy : 0,
            n2 = g.nz > 1 << sz ? cells >> sz : 0;
  const int tile = (int)blockIdx.x;
  const int x0 = tile % t.tiles_x << sx, y0 = tile / t.tiles_x % t.tiles_y << sy,
            z0 = tile / (t.tiles_x * t.tiles_y) << sz;
  struct At { int x, y, z; };   // relative to the tile
  auto at_cell = [&](int e) { return At{e & mx, e >> sx & my, e >> sxy}; };
  auto at_layer = [&](int a, int q, int v) {
    return a == 0 ? At{v, q & my, q >> sy} : a == 1 ? At{q & mx, v, q >> sx} : At{q & mx, q >> sx, v};
  };
  auto direction = [&](int &q, int per) {   // of place q of the layers, per places each; q: place in the direction
    if (q < per * n0) return 0;
    q -= per * n0;
    if (q < per * n1) return 1;
    q -= per * n1;
    return 2;
  };
  auto layer_size = [&](int a) { return a == 0 ? n0 : a == 1 ? n1 : n2; };
  auto layer_base = [&](int a) { return cells + 2 * (a == 0 ? 0 : a == 1 ? n0 : n0 + n1); };
  auto inside = [&](At p) {
    return x0 + p.x >= 0 && x0 + p.x < g.nx && y0 + p.y >= 0 && y0 + p.y < g.ny && z0 + p.z >= 0 && z0 + p.z < g.nz;
  };
  auto cell = [&](At p) { return ((int64_t)(z0 + p.z) * g.ny + (y0 + p.y)) * g.nx + (x0 + p.x); };
  for (int e = threadIdx.x; e < cells + 2 * (n0 + n1 + n2); e += kTileThreads) {
    At p;
    if (e < cells) {
      p = at_cell(e);
    } else {
      int q = e - cells;
      const int a = direction(q, 2), n = layer_size(a);
      p = q < n ? at_layer(a, q, -1) : at_layer(a, q - n, a == 0 ? 1 << sx : a == 1 ? 1 << sy : 1 << sz);
    }
    double v = 0.0;
    if (inside(p)) {
      v = perm[cell(p)];
      if (is_log) v = exp(v);
    }
    kk[e] = v;
  }
  __syncthreads();
  // the upper faces of the tile's cells, direction by direction, then the lower faces of the tile
  for (int f = threadIdx.x; f < 3 * cells + n0 + n1 + n2; f += kTileThreads) {
    int a, el, eu, kl, ku;   // direction; cells below and above (-1: outside the tile), and their places in kk
    At lo;
    if (f < 3 * cells) {
      a = f >> sc;
      el = kl = f & (cells - 1);
      lo = at_cell(el);
      const bool last = a == 0 ? lo.x == mx : a == 1 ? lo.y == my : lo.z == (1 << sz) - 1;
      eu = last ? -1 : el + (a == 0 ? 1 : a == 1 ? 1 << sx : 1 << sxy);
      ku = !last ? eu
                 : layer_base(a) + layer_size(a) +
                       (a == 0 ? el >> sx : a == 1 ? (el & mx) | el >> sxy << sx : el & mxy);
    } else {
      int q = f - 3 * cells;
      a = direction(q, 1);
      el = -1;
      kl = layer_base(a) + q;
      lo = at_layer(a, q, -1);
      eu = ku = a == 0 ? q << sx : a == 1 ? (q & mx) | q >> sx << sxy : q;
    }
    const At up{lo.x + (a == 0), lo.y + (a == 1), lo.z + (a == 2)};
    if (!inside(lo) || !inside(up)) continue;
    const int64_t i = cell(lo), j = cell(up);
    const double ki = kk[kl], kj = kk[ku];
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
    if (el >= 0) part[3 + a][el] = gi;
    if (eu >= 0) part[2 - a][eu] = gj;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < cells; e += kTileThreads) {
    const At p = at_cell(e);
    if (!inside(p)) continue;
    const int cx = x0 + p.x, cy = y0 + p.y, cz = z0 + p.z;
    const bool on[6] = {cz > 0, cy > 0, cx > 0, cx + 1 < g.nx, cy + 1 < g.ny, cz + 1 < g.nz};
    double acc = 0.0;
#pragma unroll
    for (int d = 0; d < 6; d++)
      if (on[d]) acc = acc + part[d][e];
    dtheta[cell(p)] = acc;
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
  const int run = outer_run(A.nnzb, b);
  TRS_DISPATCH_B(b, launch_pdl(k_outer_product<B>, (unsigned)((A.nnzb + run - 1) / run), kThreads, 0, s, A.nnzb, run,
                               A.urow.p, A.ucol.p, lambda, x, dA));
  TRS_LAUNCHED();
}

void launch_chain_theta(int b, const trs_bsr &A, const double *perm, int perm_is_log, double kvkh, double c_t,
                        const double *M, const double *lambda, const double *x, double *dtheta, cudaStream_t s) {
  if (!A.g.nc) return;
  const ChainTile t = chain_tile(A.g);
  const int64_t tiles = (int64_t)t.tiles_x * t.tiles_y * (((A.g.nz - 1) >> t.sz) + 1);
  const bool box = t.sx == kBoxX && t.sy == kBoxY && t.sz == kBoxZ;
  TRS_DISPATCH_B(b, {
    // the constants take registers from the contraction at b = 4 and 5 (100x80x50, b = 5: 253 us, 272 with them;
    // b = 3: 135, with them 132; 16x16x8, b = 3: 20.3, with them 19.5)
    const auto kernel = B <= 3 && box ? k_chain_theta<B, B <= 3> : k_chain_theta<B, false>;
    set_attribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, kTileCarveout);
    launch_pdl(kernel, (unsigned)tiles, kTileThreads, 0, s, A.g, t, A.emask.p, perm, perm_is_log, kvkh, c_t, M, lambda,
               x, dtheta);
  });
  TRS_LAUNCHED();
}

}  // namespace trs
