// Block Krylov (block Lanczos with full re-orthogonalisation) for the
// A-harmonic local eigenproblem S x = lambda T x, run on the shift-invert
// operator M = S^{-1} T, which is self-adjoint in the T inner product.
//
// Vectors are kept in their A-harmonic extension phi = E x (full Omega*
// layout); M phi = E [K^{-1} B phi]_2 with B = D_mu K D_mu (one K solve and one
// A11 solve per block).  M is self-adjoint in the inner product
// N = S + sigma T, <phi_a, phi_b>_N = phi_a^T (K + sigma B) phi_b, which is
// definite on the rigid modes (where S vanishes) and on the near-null space of
// T (vectors living where mu ~ 0, which T alone cannot see), so rounding noise
// is never normalised into the basis.  With Q_m N-orthonormal,
// M Q_m = Q_m H_m + Q_{m+1} R_{m+1} E_m^T; a Ritz pair (mu, y) of H_m gives
// lambda = 1/mu and the relative residual ||M x - mu x||_N / (mu ||x||_N) =
// ||R_{m+1} y_last|| / mu without extra solves; x^T T x = 1 / (lambda + sigma)
// gives the B-normalised eigenvector.
#include "internal.h"

namespace {

constexpr double KSIGMA = 1e-2;   // N = S + KSIGMA T

// Rayleigh-Ritz work arrays: wanted mu (descending) and their indices [N][PST], the
// rotations' tangents [RR_BATCH or N][rounds][MQ / 2], rounds run [N]
struct RrWork {
  double* mu;
  float* log;
  int* perm;
  int* rounds;
};

// y = alpha [D_mu] K [D_mu] x on KB-wide blocks: 4 nodes per warp, lane % 8 = column.
__global__ void __launch_bounds__(256)
k_stencil_kb(const SubDev* __restrict__ subs, const int* __restrict__ active, int src, int dst, int mode,
             double alpha) {
  const int sidx = blockIdx.y;
  if (active != nullptr && !active[sidx]) return;
  const SubDev& s = subs[sidx];
  const int lane = threadIdx.x & 31, col = lane & (KB - 1);
  const int node = (blockIdx.x * 8 + (threadIdx.x >> 5)) * (32 / KB) + (lane / KB);
  if (node >= s.nnode) return;
  const double* x = mv_ptr(s, src);
  double* y = mv_ptr(s, dst);
  const int k = node / s.npl, q = node % s.npl;
  const int qi = q / s.nyn, qj = q % s.nyn;
  const double* st = s.stencil + (size_t)node * 243;
  double y0 = 0.0, y1 = 0.0, y2 = 0.0, z0 = 0.0, z1 = 0.0, z2 = 0.0;
  for (int slot = 0; slot < 27; ++slot) {
    const int di = slot / 9 - 1, dj = (slot / 3) % 3 - 1, dk = slot % 3 - 1;
    const int ni = qi + di, nj = qj + dj, nk = k + dk;
    if (ni < 0 || ni >= s.nxn || nj < 0 || nj >= s.nyn || nk < 0 || nk >= s.nzn) continue;
    const int nb = nk * s.npl + ni * s.nyn + nj;
    const double* xr = x + (size_t)nb * 3 * KB + col;
    const double* c = st + slot * 9;
    if (mode == 4) {
      // N x = K x + sigma D_mu K D_mu x in one pass (sigma = alpha)
      const double x0 = xr[0], x1 = xr[KB], x2 = xr[2 * KB], m = s.mu[nb];
      const double k0 = fma(c[0], x0, fma(c[1], x1, c[2] * x2));
      const double k1 = fma(c[3], x0, fma(c[4], x1, c[5] * x2));
      const double k2 = fma(c[6], x0, fma(c[7], x1, c[8] * x2));
      y0 += k0; y1 += k1; y2 += k2;
      z0 = fma(m, k0, z0); z1 = fma(m, k1, z1); z2 = fma(m, k2, z2);
      continue;
    }
    const double sc = (mode & 1) ? s.mu[nb] : 1.0;
    const double x0 = sc * xr[0], x1 = sc * xr[KB], x2 = sc * xr[2 * KB];
    y0 = fma(c[0], x0, fma(c[1], x1, fma(c[2], x2, y0)));
    y1 = fma(c[3], x0, fma(c[4], x1, fma(c[5], x2, y1)));
    y2 = fma(c[6], x0, fma(c[7], x1, fma(c[8], x2, y2)));
  }
  double* yr = y + (size_t)node * 3 * KB + col;
  if (mode == 4) {
    const double sm = alpha * s.mu[node];
    yr[0] = fma(sm, z0, y0);
    yr[KB] = fma(sm, z1, y1);
    yr[2 * KB] = fma(sm, z2, y2);
    return;
  }
  const double post = alpha * ((mode & 2) ? s.mu[node] : 1.0);
  yr[0] = post * y0;
  yr[KB] = post * y1;
  yr[2 * KB] = post * y2;
}

// Rows per partial sum of a Gram product: the fewest of 64 .. 512 with at most
// GRAM_KB_PARTS partial sums over all subdomains (whose slots d_gram_part holds in any
// case).  FP64 bound once every SM has work; 512 rows leave few subdomains on few SMs:
// 40 x 6 x 12 beam, 8 subdomains, 8 to 96 columns: 407 products 24 -> 5 ms.
int gram_kb_rows(const msgfem* h, int nfull) {
  int rows = 64;
  while (rows < 512 && (size_t)h->N * ((nfull + rows - 1) / rows) > GRAM_KB_PARTS) rows *= 2;
  return rows;
}

// Partial sums of G[a][b] = sum_r X[r][a] Y[r][b], a < nx (X of stride xs),
// b < KB (Y of stride KB), over krows rows (a multiple of 32).  Up to 16 columns of X the
// threads form 2 or 4 groups that share the rows.
__global__ void __launch_bounds__(256)
k_gram_kb_partial(const SubDev* __restrict__ subs, const int* __restrict__ active, int wx, int xs, int nx, int wy,
                  int only_floating, double* __restrict__ part, int nchunk, int krows) {
  const int sidx = blockIdx.y;
  if (active != nullptr && !active[sidx]) return;
  const SubDev& s = subs[sidx];
  if (only_floating && !s.floating) return;
  __shared__ double Xs[32][MQ + 1];
  __shared__ double Ys[32][KB];
  const double* X = mv_ptr(s, wx);
  const double* Yv = mv_ptr(s, wy);
  const int tid = threadIdx.x;
  const int nout = nx * KB, groups = nx <= 8 ? 4 : (nx <= 16 ? 2 : 1), per = 256 / groups;
  const int g = tid / per, nr = 32 / groups, f0 = g * nr;
  double acc[3] = {0.0, 0.0, 0.0};
  const int r0 = blockIdx.x * krows;
  const int r1 = min(r0 + krows, s.nfull);
  for (int rb = r0; rb < r1; rb += 32) {
    for (int e = tid; e < 32 * nx; e += 256) {
      const int rr = rb + e / nx;
      Xs[e / nx][e % nx] = rr < r1 ? X[(size_t)rr * xs + e % nx] : 0.0;
    }
    for (int e = tid; e < 32 * KB; e += 256) {
      const int rr = rb + e / KB;
      Ys[e / KB][e % KB] = rr < r1 ? Yv[(size_t)rr * KB + e % KB] : 0.0;
    }
    __syncthreads();
    for (int i = 0; i < 3; ++i) {
      const int o = tid % per + 256 * i;
      if (o >= nout) break;
      const int a = o / KB, b = o % KB;
      double v = acc[i];
#pragma unroll 8
      for (int r = 0; r < nr; ++r) v = fma(Xs[f0 + r][a], Ys[f0 + r][b], v);
      acc[i] = v;
    }
    __syncthreads();
  }
  double* out = part + ((size_t)sidx * nchunk + blockIdx.x) * MQ * KB;
  if (groups > 1) {   // nout <= per: one output per thread
    double* sum = &Xs[0][0];
    sum[tid] = acc[0];
    __syncthreads();
    if (tid < nout) {
      double v = sum[tid];
      for (int q = 1; q < groups; ++q) v += sum[tid + q * per];
      out[tid] = v;
    }
    return;
  }
  for (int i = 0; i < 3; ++i) {
    const int o = tid + 256 * i;
    if (o < nout) out[o] = acc[i];
  }
}

__global__ void k_gram_kb_reduce(const SubDev* __restrict__ subs, const int* __restrict__ active, int nx,
                                 int only_floating, const double* __restrict__ part, int nchunk, int krows) {
  const int sidx = blockIdx.x;
  if (active != nullptr && !active[sidx]) return;
  const SubDev& s = subs[sidx];
  if (only_floating && !s.floating) return;
  const int nc = (s.nfull + krows - 1) / krows;
  for (int o = threadIdx.x; o < nx * KB; o += blockDim.x) {
    double acc = 0.0;
    for (int c = 0; c < nc; ++c) acc += part[((size_t)sidx * nchunk + c) * MQ * KB + o];
    s.Hc[o] = acc;
  }
}

// Y -= X Hc with X of stride xs and nx columns, Y a KB-wide block.
__global__ void __launch_bounds__(256)
k_update_kb(const SubDev* __restrict__ subs, const int* __restrict__ active, int wx, int xs, int nx, int wy,
            int only_floating) {
  const int sidx = blockIdx.y;
  if (active != nullptr && !active[sidx]) return;
  const SubDev& s = subs[sidx];
  if (only_floating && !s.floating) return;
  __shared__ double C[MQ][KB];
  for (int e = threadIdx.x; e < nx * KB; e += 256) C[e / KB][e % KB] = s.Hc[e];
  __syncthreads();
  const double* X = mv_ptr(s, wx);
  double* Y = mv_ptr(s, wy);
  const int col = threadIdx.x % KB;
  for (int r = blockIdx.x * (256 / KB) + threadIdx.x / KB; r < s.nfull; r += gridDim.x * (256 / KB)) {
    const double* xr = X + (size_t)r * xs;
    double acc = Y[(size_t)r * KB + col];
    for (int a = 0; a < nx; ++a) acc = fma(-xr[a], C[a][col], acc);
    Y[(size_t)r * KB + col] = acc;
  }
}

// H[a][j KB + c] (+)= Hc[a][c], a < m.
__global__ void k_h_accum(const SubDev* __restrict__ subs, const int* __restrict__ active, int m, int j, int add) {
  const int sidx = blockIdx.x;
  if (active != nullptr && !active[sidx]) return;
  const SubDev& s = subs[sidx];
  for (int e = threadIdx.x; e < m * KB; e += blockDim.x) {
    const int a = e / KB, c = e % KB;
    double* h = s.H + (size_t)a * MQ + j * KB + c;
    *h = add ? *h + s.Hc[e] : s.Hc[e];
  }
}

// One pass of CholeskyQR2 of a KB-wide block in the N inner product:
// Hc = W^T N W = L L^T and Y[0:KB][0:KB] = L^{-T}.  Pass 1 drops columns that
// are rounding noise -- a pivot below 1e-12 of the column's own squared norm
// (dependent inside the block) or below 1e-20 of its squared norm before
// Gram-Schmidt (the Krylov space is exhausted) -- and keeps R1 = L^T in
// Y[KB:2KB][0:KB].  Pass 2 re-orthonormalises the surviving columns and, for
// j >= 0, stores R_{j+1} = L2^T R1 in H[(j+1) KB + r][j KB + c].
// One warp per subdomain, a lane per row of the column's elimination and per column of
// the inverse (50 us in one thread,
// 16 here).
__global__ void k_cholqr_kb(const SubDev* __restrict__ subs, const int* __restrict__ active, int j, int pass) {
  const int sidx = blockIdx.x;
  if (active != nullptr && !active[sidx]) return;
  const SubDev& s = subs[sidx];
  __shared__ double G[KB][KB], L[KB][KB], U[KB][KB], R1[KB][KB];
  const int lane = threadIdx.x;
  for (int e = lane; e < KB * KB; e += 32) {
    const int a = e / KB, b = e % KB;
    G[a][b] = 0.5 * (s.Hc[a * KB + b] + s.Hc[b * KB + a]);
    L[a][b] = U[a][b] = 0.0;
    R1[a][b] = pass == 2 ? s.Y[(KB + a) * PST + b] : 0.0;
  }
  __syncwarp();
  // lanes c, c + 8, c + 16, c + 24: squared norm of column c before Gram-Schmidt
  double n0 = 0.0;
  if (pass == 1 && j >= 0)
    for (int a = lane / KB; a < (j + 1) * KB; a += 32 / KB) {
      const double hc = s.H[(size_t)a * MQ + j * KB + lane % KB];
      n0 += hc * hc;
    }
  n0 += __shfl_xor_sync(0xffffffffu, n0, 8);
  n0 += __shfl_xor_sync(0xffffffffu, n0, 16);
  n0 += G[lane % KB][lane % KB];
  unsigned dead = 0;   // the same in every lane
  for (int c = 0; c < KB; ++c) {
    double v = G[c][c];
    for (int k = 0; k < c; ++k) v -= L[c][k] * L[c][k];
    const double nc = __shfl_sync(0xffffffffu, n0, c);
    if (!(G[c][c] > 0.0) || !(v > 1e-12 * G[c][c]) || !(v > 1e-20 * nc)) {
      dead |= 1u << c;
      if (lane == 0) s.status[3] = 1;
      continue;
    }
    const double d = sqrt(v);
    double w = d;
    if (lane > c && lane < KB) {
      w = G[lane][c];
      for (int k = 0; k < c; ++k) w -= L[lane][k] * L[c][k];
      w /= d;
    }
    if (lane >= c && lane < KB) L[lane][c] = w;
    __syncwarp();
  }
  if (lane < KB && !((dead >> lane) & 1)) {
    const int c = lane;
    for (int i = c; i >= 0; --i) {
      if ((dead >> i) & 1) continue;
      double v = (i == c) ? 1.0 : 0.0;
      for (int k = i + 1; k <= c; ++k) v -= L[k][i] * U[k][c];
      U[i][c] = v / L[i][i];
    }
  }
  __syncwarp();
  for (int e = lane; e < KB * KB; e += 32) {
    const int r = e / KB, c = e % KB;
    s.Y[r * PST + c] = U[r][c];
    if (pass == 1) {
      s.Y[(KB + r) * PST + c] = L[c][r];
    } else if (j >= 0) {
      double v = 0.0;
      for (int k = 0; k < KB; ++k) v += L[k][r] * R1[k][c];   // (L2^T R1)[r][c]
      s.H[(size_t)((j + 1) * KB + r) * MQ + j * KB + c] = v;
    }
  }
}

// X <- X Y[0:KB][0:KB] on a KB-wide block.
__global__ void __launch_bounds__(256)
k_rotate_kb(const SubDev* __restrict__ subs, const int* __restrict__ active, int which) {
  const int sidx = blockIdx.y;
  if (active != nullptr && !active[sidx]) return;
  const SubDev& s = subs[sidx];
  __shared__ double Ys[KB][KB];
  if (threadIdx.x < KB * KB) Ys[threadIdx.x / KB][threadIdx.x % KB] = s.Y[(threadIdx.x / KB) * PST + threadIdx.x % KB];
  __syncthreads();
  double* X = mv_ptr(s, which);
  const int col = threadIdx.x % KB;
  for (int r = blockIdx.x * (256 / KB) + threadIdx.x / KB; r < s.nfull; r += gridDim.x * (256 / KB)) {
    double xr[KB];
#pragma unroll
    for (int a = 0; a < KB; ++a) xr[a] = X[(size_t)r * KB + a];
    __syncwarp();
    double acc = 0.0;
#pragma unroll
    for (int a = 0; a < KB; ++a) acc = fma(xr[a], Ys[a][col], acc);
    X[(size_t)r * KB + col] = acc;
  }
}

// dst[:, j KB + c] = src[:, c] (dst = QB or NQ)
__global__ void k_store_block(const SubDev* __restrict__ subs, const int* __restrict__ active, int src, int j,
                              int dst) {
  const int sidx = blockIdx.y;
  if (active != nullptr && !active[sidx]) return;
  const SubDev& s = subs[sidx];
  const double* X = mv_ptr(s, src);
  double* D = mv_ptr(s, dst);
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < (size_t)s.nfull * KB;
       e += (size_t)gridDim.x * blockDim.x)
    D[(e / KB) * MQ + j * KB + e % KB] = X[e];
}

__global__ void k_zero_kb(const SubDev* __restrict__ subs, const int* __restrict__ active, int which, int col0_only) {
  if (active != nullptr && !active[blockIdx.y]) return;
  const SubDev& s = subs[blockIdx.y];
  double* X = mv_ptr(s, which);
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < (size_t)s.nfull * KB;
       e += (size_t)gridDim.x * blockDim.x)
    X[e] = 0.0;
  (void)col0_only;
}

// Start block on the rows of DoF class fill_cls (counter-based uniform(-1, 1)),
// zero elsewhere: B2 for the A-harmonic problem, B1 for GenEO.
__device__ __forceinline__ uint64_t mix64(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

__global__ void k_random_kb(const SubDev* __restrict__ subs, const int* __restrict__ active, int which,
                            unsigned long long seed, int fill_cls) {
  const int sidx = blockIdx.y;
  if (active != nullptr && !active[sidx]) return;
  const SubDev& s = subs[sidx];
  double* X = mv_ptr(s, which);
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < (size_t)s.nfull * KB;
       e += (size_t)gridDim.x * blockDim.x) {
    const int row = (int)(e / KB), col = (int)(e % KB);
    const int q = (row / 3) % s.npl;
    double v = 0.0;
    if (s.cls[q] == fill_cls) {
      const uint64_t key = mix64(seed ^ mix64(((uint64_t)sidx << 40) ^ ((uint64_t)row << 8) ^ col));
      v = (double)(key >> 11) * (2.0 / 9007199254740992.0) - 1.0;
    }
    X[e] = v;
  }
}

__global__ void k_mask_kb(const SubDev* __restrict__ subs, const int* __restrict__ active, int which, int keep) {
  const int sidx = blockIdx.y;
  if (active != nullptr && !active[sidx]) return;
  const SubDev& s = subs[sidx];
  double* X = mv_ptr(s, which);
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < (size_t)s.nfull * KB;
       e += (size_t)gridDim.x * blockDim.x) {
    const int q = (int)(e / KB / 3) % s.npl;
    if (!((keep >> s.cls[q]) & 1)) X[e] = 0.0;
  }
}

__global__ void k_zero_pins_kb(const SubDev* __restrict__ subs, const int* __restrict__ active, int which) {
  if (active != nullptr && !active[blockIdx.x]) return;
  const SubDev& s = subs[blockIdx.x];
  if (!s.floating) return;
  double* X = mv_ptr(s, which);
  const int i = threadIdx.x / KB, c = threadIdx.x % KB;
  if (i < 6 && s.pin[i] >= 0) X[(size_t)s.pin[i] * KB + c] = 0.0;
}

// dst[:, 0] = sign * bload, other columns zero (KB-wide block)
__global__ void k_load_col_kb(const SubDev* __restrict__ subs, const int* __restrict__ active, int which, double sign) {
  if (active != nullptr && !active[blockIdx.y]) return;
  const SubDev& s = subs[blockIdx.y];
  double* X = mv_ptr(s, which);
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < (size_t)s.nfull * KB;
       e += (size_t)gridDim.x * blockDim.x)
    X[e] = (e % KB == 0) ? sign * s.bload[e / KB] : 0.0;
}

__global__ void k_take_col_kb(const SubDev* __restrict__ subs, const int* __restrict__ active, int which) {
  if (active != nullptr && !active[blockIdx.y]) return;
  const SubDev& s = subs[blockIdx.y];
  const double* X = mv_ptr(s, which);
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < s.nfull; r += gridDim.x * blockDim.x)
    s.psi[r] = X[(size_t)r * KB];
}

// Rayleigh-Ritz on the leading m x m block of H (symmetrised): parallel cyclic
// Jacobi; the nw largest mu give theta = 1/mu ascending, Yk[:, i] their coefficient
// vectors, resid[i] = theta_i ||R_{m+1} y_last||.
//
// One SM's FP64 pipe (1.6 FMA per clock) bounds it, so the arithmetic is kept small
// and the vectors leave the iteration:
//  * a round's m / 2 disjoint rotations update the symmetric matrix as 2 x 2 blocks
//    of pairs (k <= l), read and written once;
//  * rotations are scaled, A = D S D with J = c [1 t; -t 1]: the c go into D and an
//    entry costs one FMA per side (8 per 2 x 2 block instead of 16);
//  * the angle needs no FP64 accuracy (a rotation by a slightly wrong angle is still
//    a similarity): t is formed in FP32, c = (1 + t^2)^{-1/2} to FP64 by Newton steps;
//  * only t is logged (4 bytes per rotation); the wanted vectors are formed after
//    the iteration by applying the rotations backwards to unit vectors, four columns
//    per CTA (k_rr_vectors).
// 65 calls (m = 24 to 96) of the GenEO comparison on eight subdomains 452 -> 142 ms,
// 9 calls on the C-section's 16 subdomains 50.6 -> 16.8 ms (every rotation applied to
// rows, columns and vectors before).
constexpr int RR_SWEEPS = 30;
constexpr int RR_ROUNDS = RR_SWEEPS * (MQ - 1);
// The log of a subdomain takes 547 KB (the most sweeps at the largest basis), so that of
// the subdomains of one launch only is kept: two rounds of the two CTAs that an SM holds.
constexpr int RR_BATCH = 608;

// pair k of round r of the round-robin order of mm (even) indices
__device__ __forceinline__ void rr_pair(int k, int r, int mm, int& a, int& b) {
  a = (k == 0) ? 0 : ((r + k - 1) % (mm - 1)) + 1;
  b = ((r + mm - 2 - k) % (mm - 1)) + 1;
  if (a > b) { const int t = a; a = b; b = t; }
}

// w^{-1/2} for w in [1, 2]: FP32 seed, two Newton steps
__device__ __forceinline__ double rr_rsqrt(double w) {
  double y = (double)rsqrtf((float)w);
  y = y * fma(-0.5 * w * y, y, 1.5);
  return y * fma(-0.5 * w * y, y, 1.5);
}

__global__ void __launch_bounds__(512)
k_rr_jacobi(const SubDev* __restrict__ subs, const int* __restrict__ active, const int* __restrict__ mvec,
            const int* __restrict__ nwvec, RrWork wk) {
  const int sidx = blockIdx.x;
  if (active != nullptr && !active[sidx]) return;
  const SubDev& s = subs[sidx];
  const int m = mvec[sidx], nw = nwvec[sidx];
  if (m <= 0 || nw <= 0) return;
  extern __shared__ double sh[];
  double (*A)[MQ + 1] = reinterpret_cast<double (*)[MQ + 1]>(sh);   // entries (i, j), j <= i
  __shared__ double d[MQ], id[MQ], al[MQ / 2], be[MQ / 2];
  __shared__ int pa[MQ / 2], pb[MQ / 2];
  __shared__ double red_off[16], red_tot[16];
  __shared__ int again;
  const int tid = threadIdx.x, np = m / 2;      // m is a multiple of KB
  float* log = wk.log + (size_t)sidx * RR_ROUNDS * (MQ / 2);
  for (int e = tid; e < m * m; e += 512) {
    const int r = e / m, c = e % m;
    if (c <= r) A[r][c] = 0.5 * (s.H[(size_t)r * MQ + c] + s.H[(size_t)c * MQ + r]);
  }
  if (tid < m) { d[tid] = 1.0; id[tid] = 1.0; }
  __syncthreads();
  int rounds = 0;
  for (int sweep = 0; sweep < RR_SWEEPS; ++sweep) {
    // apply the scaling, off-diagonal and total Frobenius mass
    double off = 0.0, tot = 0.0;
    for (int e = tid; e < m * m; e += 512) {
      const int i = e / m, j = e % m;
      if (j > i) continue;
      const double v = A[i][j] * d[i] * d[j];
      A[i][j] = v;
      if (i != j) off += 2.0 * v * v;
      else tot += v * v;
    }
    tot += off;
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      tot += __shfl_xor_sync(0xffffffffu, tot, o);
    }
    if ((tid & 31) == 0) { red_off[tid >> 5] = off; red_tot[tid >> 5] = tot; }
    __syncthreads();
    if (tid < m) { d[tid] = 1.0; id[tid] = 1.0; }
    if (tid == 0) {
      double so = 0.0, st = 0.0;
      for (int w = 0; w < 16; ++w) { so += red_off[w]; st += red_tot[w]; }
      again = so > 1e-30 * st;
    }
    __syncthreads();
    if (!again) break;
    for (int round = 0; round < m - 1; ++round, ++rounds) {
      if (tid < np) {
        int p, q;
        rr_pair(tid, round, m, p, q);
        pa[tid] = p;
        pb[tid] = q;
        // t = sign / (|tau| + sqrt(1 + tau^2)), tau = (a_qq - a_pp) / (2 a_pq)
        const double dp = d[p], dq = d[q];
        const double diff = A[q][q] * dq * dq - A[p][p] * dp * dp, twice = 2.0 * A[q][p] * dp * dq;
        float t = 0.f;
        if (fabs(twice) > 1e-36) {
          const float tau = (float)(diff) / (float)twice;
          t = copysignf(1.f, tau) / (fabsf(tau) + sqrtf(fmaf(tau, tau, 1.f)));
          if (!(fabsf(t) <= 1.f)) t = 0.f;
        }
        const double td = (double)t, w = fma(td, td, 1.0), c = rr_rsqrt(w);
        al[tid] = td * dq * id[p];
        be[tid] = td * dp * id[q];
        d[p] = c * dp;
        d[q] = c * dq;
        id[p] *= w * c;
        id[q] *= w * c;
        log[(size_t)rounds * (MQ / 2) + tid] = t;
      }
      __syncthreads();
      // blocks (k, l), k <= l: rows k and np - 1 - k hold np + 1 of them together
      for (int e = tid; e < np / 2 * (np + 1); e += 512) {
        const int r = e / (np + 1), c = e % (np + 1);
        const int k = c < np - r ? r : np - 1 - r, l = c < np - r ? r + c : k + c - (np - r);
        const int p0 = pa[k], q0 = pb[k], p1 = pa[l], q1 = pb[l];
        double* xa = p0 > p1 ? &A[p0][p1] : &A[p1][p0];
        double* xb = p0 > q1 ? &A[p0][q1] : &A[q1][p0];
        double* xc = q0 > p1 ? &A[q0][p1] : &A[p1][q0];
        double* xd = q0 > q1 ? &A[q0][q1] : &A[q1][q0];
        const double a = *xa, b = *xb, cc = *xc, dd = *xd;
        const double ak = al[k], bk = be[k], aL = al[l], bL = be[l];
        const double a1 = fma(-ak, cc, a), c1 = fma(bk, a, cc), b1 = fma(-ak, dd, b), d1 = fma(bk, b, dd);
        *xa = fma(-aL, b1, a1);
        *xd = fma(bL, c1, d1);
        if (k != l) *xc = fma(-aL, d1, c1);   // (k, k): the same entry as b
        *xb = fma(bL, a1, b1);
      }
      __syncthreads();
    }
  }
  // descending mu by counting; ties by index
  __shared__ double mu[MQ];
  if (tid < m) mu[tid] = A[tid][tid] * d[tid] * d[tid];
  __syncthreads();
  if (tid < m) {
    int rank = 0;
    for (int j = 0; j < m; ++j) rank += (mu[j] > mu[tid] || (mu[j] == mu[tid] && j < tid)) ? 1 : 0;
    // an operator with a NaN or an infinity has no Ritz pairs: every rank is written (none
    // keeps an earlier call's value) as invalid
    double mass = 0.0;
    for (int w = 0; w < 16; ++w) mass += red_tot[w];
    const bool bad = !(mass <= 1.7e308);
    if (bad) rank = tid;
    if (rank < nw && rank < PST) {
      wk.perm[sidx * PST + rank] = tid;
      wk.mu[sidx * PST + rank] = bad ? NAN : mu[tid];
    }
  }
  if (tid == 0) wk.rounds[sidx] = rounds;
}

constexpr int RR_CHUNK = 32;   // rounds whose rotations are staged at once

__global__ void __launch_bounds__(4 * (MQ / 2))
k_rr_vectors(const SubDev* __restrict__ subs, const int* __restrict__ active, const int* __restrict__ mvec,
             const int* __restrict__ nwvec, RrWork wk) {
  const int sidx = blockIdx.y;
  if (active != nullptr && !active[sidx]) return;
  const SubDev& s = subs[sidx];
  const int m = mvec[sidx], nw = nwvec[sidx];
  if (m <= 0 || nw <= 0) return;
  __shared__ double x[MQ][4];
  __shared__ double2 cs[RR_CHUNK][MQ / 2];
  const int tid = threadIdx.x, k = tid >> 2, c = tid & 3, col = blockIdx.x * 4 + c, np = m / 2;
  const bool live = col < nw;
  const int src = live ? wk.perm[sidx * PST + col] : -1;
  for (int a = k; a < MQ; a += MQ / 2) x[a][c] = (a == src) ? 1.0 : 0.0;
  if (blockIdx.x * 4 < nw) {
    const float* log = wk.log + (size_t)sidx * RR_ROUNDS * (MQ / 2);
    // V e = J_1 (J_2 ( ... J_n e)), each round's disjoint rotations at once
    for (int r1 = wk.rounds[sidx]; r1 > 0; r1 -= RR_CHUNK) {
      const int r0 = max(0, r1 - RR_CHUNK);
      __syncthreads();
      for (int e = tid; e < (r1 - r0) * np; e += blockDim.x) {
        const int r = e / np, i = e % np;
        const double t = (double)log[(size_t)(r0 + r) * (MQ / 2) + i], cv = rr_rsqrt(fma(t, t, 1.0));
        cs[r][i] = make_double2(cv, cv * t);
      }
      __syncthreads();
      for (int r = r1 - 1; r >= r0; --r) {
        if (k < np) {
          int p, q;
          rr_pair(k, r % (m - 1), m, p, q);
          const double2 g = cs[r - r0][k];
          const double xp = x[p][c], xq = x[q][c];
          x[p][c] = fma(g.x, xp, g.y * xq);
          x[q][c] = fma(g.x, xq, -g.y * xp);
        }
        __syncthreads();
      }
    }
  }
  __syncthreads();
  for (int a = k; a < MQ; a += MQ / 2)
    if (col < PST) s.Yk[(size_t)a * PST + col] = (live && a < m) ? x[a][c] : 0.0;
  if (k == 0 && live) {
    // Ritz values of M in the N = S + sigma T inner product lie in [0, 1 / sigma];
    // a wanted one below 1e-14 (lambda above 1e14) comes from a basis that broke down
    const double mu = wk.mu[sidx * PST + col];
    const bool valid = mu > 1e-14;
    const double th = valid ? 1.0 / mu : 1e300;
    double r2 = 0.0;
    for (int r = 0; r < KB; ++r) {
      double v = 0.0;
      for (int j = 0; j < KB; ++j) v += s.H[(size_t)(m + r) * MQ + (m - KB + j)] * x[m - KB + j][c];
      r2 += v * v;
    }
    s.theta[col] = th;
    // no positive Ritz value (a basis that broke down, e.g. from a non-finite
    // start block whose columns were all dropped): never converged
    s.resid[col] = valid ? th * sqrt(r2) : INFINITY;
  }
}

// dst[:, i] = src[:, 0:m] Yk[:, i] for i < nw, zero for i >= nw (src = QB:
// Ritz vectors; src = NQ: their N products); with scale = 1 the columns are
// B-normalised (factor sqrt(theta_i + sigma)).
__global__ void __launch_bounds__(256)
k_ritz(const SubDev* __restrict__ subs, const int* __restrict__ active, const int* __restrict__ mvec,
       const int* __restrict__ nwvec, int scale, int src, int dst) {
  const int sidx = blockIdx.y;
  if (active != nullptr && !active[sidx]) return;
  const SubDev& s = subs[sidx];
  const int m = mvec[sidx], nw = nwvec[sidx];
  __shared__ double Ys[MQ][PST];
  for (int e = threadIdx.x; e < MQ * PST; e += 256) Ys[e / PST][e % PST] = s.Yk[e];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int r = blockIdx.x * 8 + (threadIdx.x >> 5); r < s.nfull; r += gridDim.x * 8) {
    const double* q = mv_ptr(s, src) + (size_t)r * MQ;
    double acc = 0.0;
    for (int a0 = 0; a0 < m; a0 += 32) {
      const double qv = (a0 + lane < m) ? q[a0 + lane] : 0.0;
      const int na = min(32, m - a0);
      for (int a = 0; a < na; ++a) acc = fma(__shfl_sync(0xffffffffu, qv, a), Ys[a0 + a][lane], acc);
    }
    mv_ptr(s, dst)[(size_t)r * PST + lane] = (lane < nw) ? (scale ? acc * sqrt(s.theta[lane] + KSIGMA) : acc) : 0.0;
  }
}

// Thick restart, basis part: dst[:, 0:k] = ritz[:, 0:k] (Ritz vectors),
// dst[:, k:k+KB] = block (the residual block Q_{m+1}); run for QB and for NQ.
__global__ void k_restart_basis(const SubDev* __restrict__ subs, const int* __restrict__ active, int k, int ritz,
                                int block, int dst) {
  const int sidx = blockIdx.y;
  if (active != nullptr && !active[sidx]) return;
  const SubDev& s = subs[sidx];
  const double* R = mv_ptr(s, ritz);
  const double* B = mv_ptr(s, block);
  double* D = mv_ptr(s, dst);
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < (size_t)s.nfull * (k + KB);
       e += (size_t)gridDim.x * blockDim.x) {
    const size_t r = e / (k + KB);
    const int c = (int)(e % (k + KB));
    D[r * MQ + c] = c < k ? R[r * PST + c] : B[r * KB + (c - k)];
  }
}

// H = 0 for the active subdomains before a Krylov run: the Lanczos steps write
// only the block upper Hessenberg part, and a thick restart of an earlier run
// leaves its arrow rows below it.
__global__ void k_zero_h(const SubDev* __restrict__ subs, const int* __restrict__ active) {
  const int sidx = blockIdx.x;
  if (active != nullptr && !active[sidx]) return;
  double* H = subs[sidx].H;
  for (int e = threadIdx.x; e < (MQ + KB) * MQ; e += blockDim.x) H[e] = 0.0;
}

// Thick restart, projected operator: H = [diag(mu) ; R_{m+1} Y_last] in the
// first k columns, zero elsewhere (the next block's coefficients are filled by
// Gram-Schmidt).  One block per subdomain.
__global__ void k_restart_h(const SubDev* __restrict__ subs, const int* __restrict__ active, int m, int k) {
  const int sidx = blockIdx.x;
  if (active != nullptr && !active[sidx]) return;
  const SubDev& s = subs[sidx];
  __shared__ double RY[KB][PST];
  __shared__ double mu[PST];
  for (int e = threadIdx.x; e < KB * k; e += blockDim.x) {
    const int r = e / k, i = e % k;
    double v = 0.0;
    for (int c = 0; c < KB; ++c) v += s.H[(size_t)(m + r) * MQ + (m - KB + c)] * s.Yk[(size_t)(m - KB + c) * PST + i];
    RY[r][i] = v;
  }
  if (threadIdx.x < k) mu[threadIdx.x] = 1.0 / s.theta[threadIdx.x];
  __syncthreads();
  for (size_t e = threadIdx.x; e < (size_t)(MQ + KB) * MQ; e += blockDim.x) {
    const int r = (int)(e / MQ), c = (int)(e % MQ);
    double v = 0.0;
    if (c < k) {
      if (r == c) v = mu[c];
      else if (r >= k && r < k + KB) v = RY[r - k][c];
    }
    s.H[e] = v;
  }
}

}  // namespace

static int max_nnode_k(msgfem* h) {
  int m = 0;
  for (const auto& s : h->sub) m = std::max(m, s.nnode);
  return m;
}

void launch_stencil_kb(msgfem* h, int src, int dst, int mode, double alpha) {
  dim3 grid((max_nnode_k(h) + 31) / 32, h->N);
  k_stencil_kb<<<grid, 256, 0, h->stream>>>(h->d_sub, h->d_flags, src, dst, mode, alpha); ++g_launch_count;
}

// Hc[0:nx][0:KB] = X[:, 0:nx]^T Y
void launch_gram_kb(msgfem* h, int wx, int xs, int nx, int wy, int only_floating) {
  const int nfull = 3 * max_nnode_k(h), krows = gram_kb_rows(h, nfull), nchunk = (nfull + krows - 1) / krows;
  dim3 grid(nchunk, h->N);
  k_gram_kb_partial<<<grid, 256, 0, h->stream>>>(h->d_sub, h->d_flags, wx, xs, nx, wy, only_floating,
                                                 h->d_gram_part, nchunk, krows); ++g_launch_count;
  k_gram_kb_reduce<<<h->N, 256, 0, h->stream>>>(h->d_sub, h->d_flags, nx, only_floating, h->d_gram_part, nchunk, krows);
  ++g_launch_count;
}

// CTAs per subdomain of the row-wise block kernels (32 rows per pass): 256 rows each, or
// down to 32 while that leaves less than about eight CTAs per SM.
static int row_ctas(msgfem* h) {
  const int rows = 3 * max_nnode_k(h);
  return std::max(1, std::min((rows + 31) / 32, std::max((rows + 255) / 256, 1216 / h->N)));
}

void launch_update_kb(msgfem* h, int wx, int xs, int nx, int wy, int only_floating) {
  dim3 grid(row_ctas(h), h->N);
  k_update_kb<<<grid, 256, 0, h->stream>>>(h->d_sub, h->d_flags, wx, xs, nx, wy, only_floating); ++g_launch_count;
}

void launch_h_accum(msgfem* h, int m, int j, int add) {
  k_h_accum<<<h->N, 256, 0, h->stream>>>(h->d_sub, h->d_flags, m, j, add); ++g_launch_count;
}

void launch_cholqr_kb(msgfem* h, int j, int pass) { k_cholqr_kb<<<h->N, 32, 0, h->stream>>>(h->d_sub, h->d_flags, j, pass); ++g_launch_count; }

void launch_rotate_kb(msgfem* h, int which) {
  dim3 grid(row_ctas(h), h->N);
  k_rotate_kb<<<grid, 256, 0, h->stream>>>(h->d_sub, h->d_flags, which); ++g_launch_count;
}

void launch_store_block(msgfem* h, int src, int j, int dst) {
  dim3 grid(256, h->N);
  k_store_block<<<grid, 256, 0, h->stream>>>(h->d_sub, h->d_flags, src, j, dst); ++g_launch_count;
}

void launch_random_kb(msgfem* h, int which, unsigned long long seed) {
  dim3 grid(256, h->N);
  k_random_kb<<<grid, 256, 0, h->stream>>>(h->d_sub, h->d_flags, which, seed, h->geneo ? 1 : 2); ++g_launch_count;
}

void launch_mask_kb(msgfem* h, int which, int keep) {
  dim3 grid(256, h->N);
  k_mask_kb<<<grid, 256, 0, h->stream>>>(h->d_sub, h->d_flags, which, keep); ++g_launch_count;
}

void launch_zero_pins_kb(msgfem* h, int which) { k_zero_pins_kb<<<h->N, 6 * KB, 0, h->stream>>>(h->d_sub, h->d_flags, which); ++g_launch_count; }

void launch_load_col_kb(msgfem* h, int which, double sign) {
  dim3 grid(256, h->N);
  k_load_col_kb<<<grid, 256, 0, h->stream>>>(h->d_sub, h->d_flags, which, sign); ++g_launch_count;
}

void launch_take_col_kb(msgfem* h, int which) {
  dim3 grid(64, h->N);
  k_take_col_kb<<<grid, 256, 0, h->stream>>>(h->d_sub, h->d_flags, which); ++g_launch_count;
}

void launch_zero_kb(msgfem* h, int which) {
  dim3 grid(256, h->N);
  k_zero_kb<<<grid, 256, 0, h->stream>>>(h->d_sub, h->d_flags, which, 0); ++g_launch_count;
}

// bytes of the Rayleigh-Ritz work arrays of N subdomains
size_t rr_bytes(int N) {
  return (size_t)N * (PST * (sizeof(double) + sizeof(int)) + 8) +
         (size_t)std::min(N, RR_BATCH) * RR_ROUNDS * (MQ / 2) * sizeof(float);
}

void launch_rr_krylov(msgfem* h, const int* d_m, const int* d_nw) {
  static bool attr = false;
  const int smem = MQ * (MQ + 1) * (int)sizeof(double);
  if (!attr) {
    cudaFuncSetAttribute(k_rr_jacobi, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    attr = true;
  }
  RrWork wk;
  char* base = static_cast<char*>(h->d_rr);
  wk.mu = reinterpret_cast<double*>(base);
  wk.log = reinterpret_cast<float*>(wk.mu + (size_t)h->N * PST);
  wk.perm = reinterpret_cast<int*>(wk.log + (size_t)std::min(h->N, RR_BATCH) * RR_ROUNDS * (MQ / 2));
  wk.rounds = wk.perm + (size_t)h->N * PST;
  for (int first = 0; first < h->N; first += RR_BATCH) {   // the arrays from the batch's first subdomain on
    const int n = std::min(RR_BATCH, h->N - first);
    k_rr_jacobi<<<n, 512, smem, h->stream>>>(h->d_sub + first, h->d_flags + first, d_m + first, d_nw + first, wk);
    k_rr_vectors<<<dim3(PST / 4, n), 4 * (MQ / 2), 0, h->stream>>>(h->d_sub + first, h->d_flags + first, d_m + first,
                                                                  d_nw + first, wk);
    g_launch_count += 2;
    wk.mu += (size_t)RR_BATCH * PST;
    wk.perm += (size_t)RR_BATCH * PST;
    wk.rounds += RR_BATCH;
  }
}

void launch_ritz(msgfem* h, const int* d_m, const int* d_nw, int scale, bool masked, int src, int dst) {
  dim3 grid(std::max(1, (3 * max_nnode_k(h) + 8 * 16 - 1) / (8 * 16)), h->N);
  k_ritz<<<grid, 256, 0, h->stream>>>(h->d_sub, masked ? h->d_flags : nullptr, d_m, d_nw, scale, src, dst);
  ++g_launch_count;
}

void launch_zero_h(msgfem* h) {
  k_zero_h<<<h->N, 256, 0, h->stream>>>(h->d_sub, h->d_flags);
  ++g_launch_count;
}

// Thick restart: QB = [Ritz vectors (PHI) | W], NQ = [their N products (CW) | N W (ZB)]
void launch_restart(msgfem* h, int m, int k) {
  dim3 grid(256, h->N);
  k_restart_basis<<<grid, 256, 0, h->stream>>>(h->d_sub, h->d_flags, k, MV_PHI, MV_WB, MV_QB); ++g_launch_count;
  k_restart_basis<<<grid, 256, 0, h->stream>>>(h->d_sub, h->d_flags, k, MV_CW, MV_ZB, MV_NQ); ++g_launch_count;
  k_restart_h<<<h->N, 256, 0, h->stream>>>(h->d_sub, h->d_flags, m, k); ++g_launch_count;
}
