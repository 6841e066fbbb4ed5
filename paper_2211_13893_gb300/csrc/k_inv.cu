// Inverse form of the layer-block solver (the default of the block Krylov path).
//
// K and A11 are block tridiagonal over the node layers, with dense diagonal
// blocks D_l and couplings C_l = A[layer l, layer l - 1] that hold 27 non-zeros
// per row (the node stencil).  Instead of the block Cholesky factors L_l and
// E_l = C_l L_{l-1}^{-T} (dense) this form keeps only the inverses of the Schur
// complements,
//   S_l = D_l - C_l S_{l-1}^{-1} C_l^T,
// and applies the couplings from the stencil:
//   forward   z_l = b_l - C_l u_{l-1},  u_l = S_l^{-1} z_l
//   backward  x_l = u_l - S_l^{-1} C_{l+1}^T x_{l+1}.
// Per layer of n DoFs the factorisation takes n^3 flops (one SPD inverse) plus
// 54 n^2 fused multiply-adds for the sparse triple product, against 8/3 n^3
// for the block Cholesky with its block inverses, and a solve reads 2 n^2
// numbers against 3 n^2.
//
// The layers are eliminated from both ends towards the middle layer
// (two half chains per matrix, the middle Schur complement takes both): the
// same work in half as many dependent steps.
//
// The inverse of a Schur complement is the symmetric sweep operator (block
// Gauss-Jordan) over its T x T tiles of 64: for k = 0 .. T - 1
//   P = S_kk^{-1};  W_i = S_ik P;  S_ij -= W_i S_jk^T (i, j != k);
//   S_ik = W_i, S_ki = W_i^T, S_kk = -P,
// which leaves -S^{-1} (kept with that sign).  Every sweep touches the whole
// matrix, so the tasks of a step stay numerous to the end.  Measured on the CPU
// in the same arithmetic it is as accurate as the block Cholesky with explicit
// block inverses in FP64, and a better FP32 preconditioner (c2's interior K:
// 4 CG steps to 1e-11 where the Cholesky form takes 5 to 6).
//
// Measured on one GB300 against the block Cholesky (factorisation / all solves of a
// local stage, ms): 36 x 12 x 39 beam FP64 345 -> 41 / 424 -> 41; 192 x 12 x 39 beam
// mixed 102 -> 72 / 374 -> 154; C-section of 16 subdomains mixed 85 -> 42 / 409 -> 124;
// 47 x 7 x 13 beam FP64 whole pass 156 -> 31.
#include "internal.h"

#include <cooperative_groups.h>
#include <cstring>
#include <type_traits>

#include "tc_gemm.cuh"

namespace cg = cooperative_groups;

// One matrix (K or A11) of one subdomain.  The kept DoFs of a layer are all
// three components of a nic x njc box of in-plane nodes.
struct InvMat {
  int sub, mat;
  int ia, ja, nic, njc;        // kept node box
  int n, b, nL, mid;           // kept / padded layer size, layers, middle layer
  int npl, nyn;
  int pinned;                  // K of a floating subdomain: rows pin[] of layer 0 are out
  int pin[6];                  // compact rows in layer 0
  int sg;                      // FP32: ranks of the solve's clusters (0: no k_inv_solve_f32)
  const double* stencil;
  void* D;                     // [nL][b][b] S_l, then -S_l^{-1}
  void* E;                     // [nL - 1][b][b] scratch of the triple products
  void* L;                     // [nL][b][b]: sweep scratch, then the packed couplings
  void* yc;                    // [nL][b][KB] u of the forward sweep
};

namespace {

enum { IV_SCHUR_A = 0, IV_SCHUR_B, IV_PIVOT, IV_PANEL, IV_UPDATE };
struct InvTask {
  int type, m, layer, k, i, j;
};

constexpr int NBLK = 8;   // nodes per coupling task

// scratch of the sweep of layer l: the old tile column k and the pivot inverse
template <typename T>
__device__ __forceinline__ T* old_col(const InvMat& m, int l) { return static_cast<T*>(m.L) + (size_t)l * m.b * m.b; }
template <typename T>
__device__ __forceinline__ T* pivot_inv(const InvMat& m, int l) {
  return static_cast<T*>(m.L) + (size_t)l * m.b * m.b + (m.b > TILE ? (size_t)m.b * TILE : 0);
}
template <typename T>
__device__ __forceinline__ T* layer_block(const InvMat& m, int l) { return static_cast<T*>(m.D) + (size_t)l * m.b * m.b; }
// scratch of the triple product that couples layer l to layer l + dk
template <typename T>
__device__ __forceinline__ T* triple_scratch(const InvMat& m, int l, int dk) {
  return static_cast<T*>(m.E) + (size_t)(dk < 0 ? l - 1 : l) * m.b * m.b;
}

__device__ __forceinline__ bool pinned_row(const InvMat& m, int layer, int row) {
  if (!m.pinned || layer != 0) return false;
#pragma unroll
  for (int i = 0; i < 6; ++i)
    if (m.pin[i] == row) return true;
  return false;
}

// Entry (r, c) of the coupling block of kept node p in layer l with neighbour
// slot s9 (0 .. 8, in-plane) in layer l + dk; zero outside the kept box and at pins.
__device__ __forceinline__ double coupling(const InvMat& m, int l, int p, int dk, int s9, int r, int c) {
  const int i = p / m.njc, j = p % m.njc, di = s9 / 3 - 1, dj = s9 % 3 - 1;
  if (i + di < 0 || i + di >= m.nic || j + dj < 0 || j + dj >= m.njc) return 0.0;
  if (m.pinned && (pinned_row(m, l, 3 * p + r) || pinned_row(m, l + dk, 3 * (p + di * m.njc + dj) + c))) return 0.0;
  const size_t node = (size_t)l * m.npl + (size_t)(m.ia + i) * m.nyn + m.ja + j;
  return m.stencil[node * 243 + (size_t)((di + 1) * 9 + (dj + 1) * 3 + dk + 1) * 9 + r * 3 + c];
}

// Rows of 8 kept nodes times a row-major matrix X: three outputs per node and
// column, 27 products each; columns along the lanes (coalesced), the
// coefficients broadcast from shared memory.  The FP64 form is bound by the
// FP64 pipe, the FP32 form by the shared-memory broadcasts.
template <typename T>
__device__ __forceinline__ void couple_rows(const InvMat& m, int nb, int dk, int layer, int q, const T* X, T* coef,
                                            T (&acc)[2][3]) {
  const int tid = threadIdx.x, nn = m.n / 3;
  for (int e = tid; e < NBLK * 81; e += 256) {
    const int p = nb * NBLK + e / 81, s9 = (e % 81) / 9, rc = e % 9;
    coef[e] = p < nn ? (T)coupling(m, layer, p, dk, s9, rc / 3, rc % 3) : (T)0;
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int pl = (tid >> 6) * 2 + u, p = nb * NBLK + pl;
#pragma unroll
    for (int r = 0; r < 3; ++r) acc[u][r] = (T)0;
    if (p >= nn || q >= m.n) continue;
    const int i = p / m.njc, j = p % m.njc;
#pragma unroll
    for (int s9 = 0; s9 < 9; ++s9) {
      const int di = s9 / 3 - 1, dj = s9 % 3 - 1;
      if (i + di < 0 || i + di >= m.nic || j + dj < 0 || j + dj >= m.njc) continue;
      const T* x = X + (size_t)(3 * (p + di * m.njc + dj)) * m.b + q;
      const T x0 = x[0], x1 = x[m.b], x2 = x[2 * (size_t)m.b];
      const T* c = coef + pl * 81 + s9 * 9;
#pragma unroll
      for (int r = 0; r < 3; ++r) acc[u][r] = fma(c[3 * r], x0, fma(c[3 * r + 1], x1, fma(c[3 * r + 2], x2, acc[u][r])));
    }
  }
}

// ---------------------------------------------------------------------------
// FP64 products in exact digit products on the tensor cores.
//
// One SM does 1.6 FP64 FMAs per clock but 956 FP16 ones (mma.sync m16n8k16, both
// measured), and its FP32 accumulation of integers is exact below 2^24.  A number is
// written as a 61-bit integer below the largest of its row (matrix) or column
// (vector) in seven balanced base-512 digits, n_i in [-256, 255], exact in FP16; of
// the 49 digit products the 28 of weight 512^6 and up are formed, those of one weight
// in one accumulator: 32 columns of k add at most 7 x 32 x 2^16 < 2^24.  After every 32
// columns the seven sums go into two 64-bit integers, so what is formed is exact.  The
// error of a product is the rounding of its operands (2^-61 of their row or column
// maximum) and the 21 digit products left out: 2^-61 of the operands' product in the
// median of random ones, at most 2^-56.4 of row maximum times column maximum (all digits
// -256).  The DFMA chain rounds every partial sum to 2^-53 of itself.  The digits' bound is
// one of the whole row, not of its small entries; emulated on the CPU, solutions at
// fibre-to-matrix ratios from 4 to 10^8 and on bricks graded 1 : 1,000 are as accurate with
// them as with FP64 products (the explicit inverse decides: INV_COND_A11).
//
// Digits are cut from biased integers, X + sum 256 512^i: a 9-bit field d is the
// digit d + 256, and 0x6400 | d is 1024 + d in FP16.  The factorisation leaves every
// layer's -S^{-1} in that form in place (8 bytes per entry, 16 x 16 blocks in fragment
// order: a lane's operands are four 16-byte vectors), so that a solve streams it with
// bulk copies as before and spends five instructions per pair of digits; the
// right-hand side's digits are cut once per layer by the rank that owns the node
// and written to every rank of the cluster.  Taken whenever a layer's digits and
// coefficients fit in shared memory (layers up to about 1,000 DoFs); above, FP64 FMAs.
// Whole passes with FP64 FMAs -> digits: 36 x 12 x 39 beam 306 -> 204 ms (solves 158 ->
// 54, 41 since), 47 x 7 x 13 beam 77 -> 50, 24 x 4 x 12 beam 29 -> 20, Schwarz PCG 45 -> 29; the
// passes' errors against a dense 64-bit reference are unchanged.
constexpr int DIG = 7;
constexpr long long DIG_BIAS = 256ll * (0x7fffffffffffffffll / 511);   // sum of 256 512^i, i < 7

// x 2^(60 - emax) rounded to nearest (|x| < 2^(emax + 1), biased exponents), plus the bias
__device__ __forceinline__ long long biased_fixed(double x, int emax) {
  const long long xb = __double_as_longlong(x);
  const int ex = (int)(xb >> 52) & 0x7ff, sh = emax - ex - 8;
  const long long m = (xb & 0xfffffffffffffll) | (1ll << 52);
  long long v;
  if (ex == 0 || sh > 60) v = 0;               // zero, subnormal or below half a unit
  else if (sh <= 0) v = m << -sh;
  else v = (m + (1ll << (sh - 1))) >> sh;
  return (xb < 0 ? -v : v) + DIG_BIAS;
}

// digit i of two biased integers as a pair of FP16 numbers
__device__ __forceinline__ uint32_t digit_pair(long long x0, long long x1, int i) {
  const uint32_t d = (__byte_perm((uint32_t)(x0 >> (9 * i)), (uint32_t)(x1 >> (9 * i)), 0x5410) & 0x01ff01ffu) | 0x64006400u;
  uint32_t r;
  asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(d), "r"(0xe500e500u));   // - 1280
  return r;
}

__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// sums of the seven weights (512^6 .. 512^12) into hi 2^27 + lo
__device__ __forceinline__ void digit_flush(const float (&acc)[DIG][4], int e, long long& hi, long long& lo) {
  lo += (long long)__float2int_rn(acc[0][e]) + ((long long)__float2int_rn(acc[1][e]) << 9) +
        ((long long)__float2int_rn(acc[2][e]) << 18);
  hi += (long long)__float2int_rn(acc[3][e]) + ((long long)__float2int_rn(acc[4][e]) << 9) +
        ((long long)__float2int_rn(acc[5][e]) << 18) + ((long long)__float2int_rn(acc[6][e]) << 27);
}

// (hi 2^27 + lo) 2^e for any int e
__device__ __forceinline__ double digit_value(long long hi, long long lo, int e) {
  const double v = fma((double)hi, 0x1p27, (double)lo);
  if (e >= -1022 && e <= 1023) return v * __hiloint2double((e + 1023) << 20, 0);
  return scalbn(v, e);
}

// v 2^e for a 64 x 64 x 64 digit product (|hi| < 2^50, |lo| < 2^45): conversions by
// the 1.5 2^52 constant, the scale by the exponent field (four FP64 instructions
// per result with the caller's subtraction: they are a third of a tile's time)
__device__ __forceinline__ double tile_digit_value(long long hi, long long lo, int e) {
  const double dh = __longlong_as_double(0x4338000000000000ll + hi) - 0x1.8p52;
  const double dl = __longlong_as_double(0x4338000000000000ll + lo) - 0x1.8p52;
  const double v = fma(dh, 0x1p27, dl);
  const long long vb = __double_as_longlong(v);
  const int ev = (int)(vb >> 52) & 0x7ff;
  if (ev != 0 && ev + e > 0 && ev + e < 0x7ff) return __longlong_as_double(vb + ((long long)e << 52));
  return scalbn(v, e);
}

// Product of two 64 x 64 FP64 tiles, A B^T, in digits: f(r, c, v0, v1) receives the
// entries (r, c) and (r, c + 1), every entry once.  Shared memory: A as FP16 digits in
// fragment order (7 x 8 KiB), B as biased integers in fragment order (32 KiB), two
// CTAs per SM; warp w forms 16 rows x 32 columns, 8 at a time.  Digit scales are the
// rows' maxima within the tile.  copy (may be null) receives A.
constexpr int DIGIT_TILE_SMEM = DIG * 8192 + 32768;

template <typename F>
__device__ __forceinline__ void digit_tile(const double* A, int lda, const double* B, int ldb, unsigned char* sm,
                                           int (*em)[TILE], double* copy, F f) {
  uint32_t* ad = reinterpret_cast<uint32_t*>(sm);                               // [DIG][4 kb][4 rt][32 lanes][4]
  longlong2* bf = reinterpret_cast<longlong2*>(sm + DIG * 8192);                // [4 kb][8 nt][2][32 lanes]
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  {
    const int r = tid & 63, kb = tid >> 6, g = r & 7;
    double2 xa[8], xb[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      xa[c] = *reinterpret_cast<const double2*>(A + (size_t)r * lda + kb * 16 + 2 * c);
      xb[c] = *reinterpret_cast<const double2*>(B + (size_t)r * ldb + kb * 16 + 2 * c);
    }
    if (tid < TILE) em[0][tid] = em[1][tid] = 0;
    __syncthreads();
    int ma = 0, mb = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      ma = max(ma, max((__double2hiint(xa[c].x) >> 20) & 0x7ff, (__double2hiint(xa[c].y) >> 20) & 0x7ff));
      mb = max(mb, max((__double2hiint(xb[c].x) >> 20) & 0x7ff, (__double2hiint(xb[c].y) >> 20) & 0x7ff));
    }
    atomicMax(&em[0][r], ma);
    atomicMax(&em[1][r], mb);
    if (copy != nullptr)
#pragma unroll
      for (int c = 0; c < 8; ++c) *reinterpret_cast<double2*>(copy + r * TILE + kb * 16 + 2 * c) = xa[c];
    __syncthreads();
    const int ea = em[0][r], eb = em[1][r];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int fl = g * 4 + (c & 3), kj = c >> 2;
      const long long u0 = biased_fixed(xa[c].x, ea), u1 = biased_fixed(xa[c].y, ea);
#pragma unroll
      for (int i = 0; i < DIG; ++i)
        ad[(((i * 4 + kb) * 4 + (r >> 4)) * 32 + fl) * 4 + ((r >> 3) & 1) + 2 * kj] = digit_pair(u0, u1, i);
      bf[((kb * 8 + (r >> 3)) * 2 + kj) * 32 + fl] = make_longlong2(biased_fixed(xb[c].x, eb), biased_fixed(xb[c].y, eb));
    }
  }
  __syncthreads();
  const int rt = w & 3;
#pragma unroll 1
  for (int nt = (w >> 2) * 4; nt < (w >> 2) * 4 + 4; ++nt) {
    long long hi[4] = {}, lo[4] = {};
#pragma unroll 1
    for (int kp = 0; kp < 2; ++kp) {
      float acc[DIG][4];
#pragma unroll
      for (int i = 0; i < DIG; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[i][e] = 0.f;
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) {
        const int kb = 2 * kp + kk;
        const longlong2 y0 = bf[((kb * 8 + nt) * 2) * 32 + lane], y1 = bf[((kb * 8 + nt) * 2 + 1) * 32 + lane];
        uint32_t bz[DIG][2];
#pragma unroll
        for (int i = 0; i < DIG; ++i) {
          bz[i][0] = digit_pair(y0.x, y0.y, i);
          bz[i][1] = digit_pair(y1.x, y1.y, i);
        }
#pragma unroll
        for (int i = 0; i < DIG; ++i) {
          const uint4 v = *reinterpret_cast<const uint4*>(ad + (((i * 4 + kb) * 4 + rt) * 32 + lane) * 4);
          const uint32_t av[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int j = DIG - 1 - i; j < DIG; ++j) mma_f16(acc[i + j - (DIG - 1)], av, bz[j]);
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) digit_flush(acc, e, hi[e], lo[e]);
    }
    const int c = nt * 8 + 2 * (lane & 3), e0 = em[1][c], e1 = em[1][c + 1];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = rt * 16 + (lane >> 2) + 8 * h, er = em[0][r];
      double v0 = tile_digit_value(hi[2 * h], lo[2 * h], er + e0 - 2 * 1023 - 66);
      double v1 = tile_digit_value(hi[2 * h + 1], lo[2 * h + 1], er + e1 - 2 * 1023 - 66);
      const double nan = __longlong_as_double(0x7ff8000000000000ll);
      if (er == 0x7ff || e0 == 0x7ff) v0 = nan;   // Inf or NaN operands
      if (er == 0x7ff || e1 == 0x7ff) v1 = nan;
      f(r, c, v0, v1);
    }
  }
}

// Product of two 32 x 32 matrices in shared memory, A B^T, in digits: A(r, k) = A[r ar +
// k ac], B likewise; f(r, c, v) receives every entry once.  A warp forms 16 rows x 8
// columns and cuts its operands' digits itself (row maxima over its quads of lanes).
template <typename F>
__device__ __forceinline__ void digit_32(const double* A, int ar, int ac, const double* B, int br, int bc, F f) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const double* a0 = A + ((w & 1) * 16 + g) * ar;
  const double* a1 = a0 + 8 * ar;
  const double* b0 = B + ((w >> 1) * 8 + g) * br;
  auto col = [&](int q) { return (q >> 2) * 16 + 2 * t + (q & 1) + 8 * ((q >> 1) & 1); };
  int e0 = 0, e1 = 0, eb = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    e0 = max(e0, (__double2hiint(a0[col(q) * ac]) >> 20) & 0x7ff);
    e1 = max(e1, (__double2hiint(a1[col(q) * ac]) >> 20) & 0x7ff);
    eb = max(eb, (__double2hiint(b0[col(q) * bc]) >> 20) & 0x7ff);
  }
#pragma unroll
  for (int o = 1; o < 4; o <<= 1) {
    e0 = max(e0, __shfl_xor_sync(0xffffffffu, e0, o));
    e1 = max(e1, __shfl_xor_sync(0xffffffffu, e1, o));
    eb = max(eb, __shfl_xor_sync(0xffffffffu, eb, o));
  }
  float acc[DIG][4];
#pragma unroll
  for (int i = 0; i < DIG; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[i][e] = 0.f;
#pragma unroll 1
  for (int kk = 0; kk < 2; ++kk) {
    long long xa[2][4], xb[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int c = col(4 * kk + q);
      xa[0][q] = biased_fixed(a0[c * ac], e0);
      xa[1][q] = biased_fixed(a1[c * ac], e1);
      xb[q] = biased_fixed(b0[c * bc], eb);
    }
    uint32_t bz[DIG][2];
#pragma unroll
    for (int i = 0; i < DIG; ++i) {
      bz[i][0] = digit_pair(xb[0], xb[1], i);
      bz[i][1] = digit_pair(xb[2], xb[3], i);
    }
#pragma unroll
    for (int i = 0; i < DIG; ++i) {
      const uint32_t av[4] = {digit_pair(xa[0][0], xa[0][1], i), digit_pair(xa[1][0], xa[1][1], i),
                              digit_pair(xa[0][2], xa[0][3], i), digit_pair(xa[1][2], xa[1][3], i)};
#pragma unroll
      for (int j = DIG - 1 - i; j < DIG; ++j) mma_f16(acc[i + j - (DIG - 1)], av, bz[j]);
    }
  }
  const int ec[2] = {__shfl_sync(0xffffffffu, eb, 8 * t), __shfl_sync(0xffffffffu, eb, 8 * t + 4)};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    long long hi = 0, lo = 0;
    digit_flush(acc, e, hi, lo);
    const int er = e < 2 ? e0 : e1;
    double v = tile_digit_value(hi, lo, er + ec[e & 1] - 2 * 1023 - 66);
    if (er == 0x7ff || ec[e & 1] == 0x7ff) v = __longlong_as_double(0x7ff8000000000000ll);   // Inf or NaN operands
    f((w & 1) * 16 + g + 8 * (e >> 1), (w >> 1) * 8 + 2 * t + (e & 1), v);
  }
}

constexpr int LDH = 33;   // row stride of the 32 x 32 matrices of tile_sweep

// Inverse of a 32 x 32 SPD matrix in shared memory, in place, by the scalar sweep operator
// in FP64 registers: a 16 x 16 thread grid, each thread the entries (ty + 16 p, tx + 16 q)
// with p >= q.  Per pivot the column and the pivot's reciprocal are published, one warp
// scales the column (every thread scaling its own two values took as long as the update:
// a warp's FP64 instruction occupies the SM's pipe for 20 clocks), and all update.  True
// in the threads that met a non-positive pivot.
__device__ __forceinline__ bool sweep_32(double* M, double (*v)[32], double* rinv, double* ws) {
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  double a[2][2];
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int q = 0; q <= p; ++q) a[p][q] = M[(ty + 16 * p) * LDH + tx + 16 * q];
  bool bad = false;
#pragma unroll
  for (int kb = 0; kb < 2; ++kb) {
#pragma unroll 1
    for (int kr = 0; kr < 16; ++kr) {
      double* vs = v[kr & 1];
      if (tx == kr) {
#pragma unroll
        for (int p = kb; p < 2; ++p) vs[ty + 16 * p] = a[p][kb];
        if (ty == kr) {
          double d = a[kb][kb];
          if (!(d > 0.0)) { bad = true; d = 1e-300; }
          rinv[kr & 1] = 1.0 / d;
        }
      }
      if (ty == kr) {
#pragma unroll
        for (int q = 0; q < kb; ++q) vs[tx + 16 * q] = a[kb][q];
      }
      __syncthreads();
      const double r = rinv[kr & 1];
      if (tid < 32) ws[tid] = vs[tid] * r;
      __syncthreads();
      double vj[2], wi[2];
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        vj[p] = vs[tx + 16 * p];
        wi[p] = ws[ty + 16 * p];
      }
#pragma unroll
      for (int p = 0; p < 2; ++p)
#pragma unroll
        for (int q = 0; q <= p; ++q) a[p][q] = fma(-wi[p], vj[q], a[p][q]);
      if (tx == kr) {
#pragma unroll
        for (int p = kb; p < 2; ++p) a[p][kb] = wi[p];
      }
      if (ty == kr) {
#pragma unroll
        for (int q = 0; q <= kb; ++q) a[kb][q] = ws[tx + 16 * q];
        if (tx == kr) a[kb][kb] = -r;
      }
    }
  }
#pragma unroll
  for (int p = 0; p < 2; ++p)
#pragma unroll
    for (int q = 0; q <= p; ++q) {
      M[(ty + 16 * p) * LDH + tx + 16 * q] = -a[p][q];
      if (q < p) M[(tx + 16 * q) * LDH + ty + 16 * p] = -a[p][q];
    }
  __syncthreads();
  return bad;
}

// Inverse of a 64 x 64 SPD tile X (its lower half), FP64 for either type, by blocks of 32:
//   W = A21 A11^{-1}, S = A22 - W A21^T, V = S^{-1} W,
//   X^{-1} = [A11^{-1} + W^T V, -V^T; -V, S^{-1}],
// the two inverses by scalar sweeps, the products in digits.  A chain of these inverses is
// the critical path of a factorisation (the CTA that updates the next pivot tile inverts
// it).  One SM's FP64 pipe (1.6 FMAs per clock) bounded 64 scalar pivots at 53 us; here
// about 31.  Whole passes: 24 x 4 x 12 beam 14.5 -> 13.7 ms, 47 x 7 x 13 beam 34.2 -> 32.7
// (mixed 46.3 -> 44.9), 36 x 12 x 39 beam 127.6 -> 121.7, C-section 328 -> 322.
// sm: 4 x 32 x 33 doubles; X may lie in it.
template <typename T>
__device__ void tile_sweep(const T* X, int ldx, T* P, unsigned char* sm, int* notspd, int sub) {
  __shared__ double v[2][32], ws[32];
  __shared__ double rinv[2];
  double* M11 = reinterpret_cast<double*>(sm);
  double* M21 = M11 + 32 * LDH;
  double* M22 = M21 + 32 * LDH;
  double* W = M22 + 32 * LDH;
  const int tid = threadIdx.x;
  {
    T x[12];   // rows of the lower half, 32 x 32 blocks 11, 21, 22
#pragma unroll
    for (int i = 0; i < 12; ++i) {
      const int e = (i & 3) * 256 + tid, r = e >> 5, c = e & 31, blk = i >> 2;
      const int rr = max(r, c), cc = min(r, c);   // diagonal blocks: from the lower half
      x[i] = blk == 1 ? X[(size_t)(32 + r) * ldx + c] : X[(size_t)(blk * 16 + rr) * ldx + blk * 16 + cc];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 12; ++i) {
      const int e = (i & 3) * 256 + tid;
      M11[(i >> 2) * 32 * LDH + (e >> 5) * LDH + (e & 31)] = (double)x[i];
    }
    __syncthreads();
  }
  bool bad = sweep_32(M11, v, rinv, ws);
  digit_32(M21, LDH, 1, M11, LDH, 1, [&](int r, int c, double y) { W[r * LDH + c] = y; });
  __syncthreads();
  digit_32(W, LDH, 1, M21, LDH, 1, [&](int r, int c, double y) {
    if (c > r) return;
    M22[r * LDH + c] -= y;
    if (c < r) M22[c * LDH + r] = M22[r * LDH + c];
  });
  __syncthreads();
  bad |= sweep_32(M22, v, rinv, ws);
  double* V = M21;
  digit_32(M22, LDH, 1, W, 1, LDH, [&](int r, int c, double y) {
    V[r * LDH + c] = y;
    P[(32 + r) * TILE + c] = (T)-y;
  });
  __syncthreads();
  digit_32(W, 1, LDH, V, 1, LDH, [&](int r, int c, double y) {
    if (c > r) return;
    const T p = (T)(M11[r * LDH + c] + y);
    P[r * TILE + c] = p;
    if (c < r) P[c * TILE + r] = p;
  });
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int e = i * 256 + tid, r = e >> 5, c = e & 31;
    P[(32 + r) * TILE + 32 + c] = (T)M22[r * LDH + c];
    P[r * TILE + 32 + c] = (T)-V[c * LDH + r];
  }
  if (bad) atomicExch(&notspd[sub], 1);
}

// FP32 tiles: operands staged in shared memory as [k][row] (row stride in floats)
constexpr int LDF = 68;
template <typename T>
constexpr int inv_step_smem() {
  return sizeof(T) == 8 ? DIGIT_TILE_SMEM : 2 * TILE * LDF * (int)sizeof(float);
}

// rows of a 64 x 64 tile (leading dimension ld) into shared memory
__device__ __forceinline__ void stage_tile(const float* G, int ld, float* S) {
  const int r = threadIdx.x & 63, k0 = (threadIdx.x >> 6) * 16;
  float4 x[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) x[c] = *reinterpret_cast<const float4*>(G + (size_t)r * ld + k0 + 4 * c);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    S[(k0 + 4 * c) * LDF + r] = x[c].x;
    S[(k0 + 4 * c + 1) * LDF + r] = x[c].y;
    S[(k0 + 4 * c + 2) * LDF + r] = x[c].z;
    S[(k0 + 4 * c + 3) * LDF + r] = x[c].w;
  }
}

// acc = A B^T of two staged 64 x 64 tiles: rows 4 ty .., columns 4 tx ..
__device__ __forceinline__ void tile_product(const float* As, const float* Bs, float (&acc)[4][4]) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[p][q] = 0.f;
#pragma unroll 16
  for (int k = 0; k < TILE; ++k) {
    const float4 av = *reinterpret_cast<const float4*>(As + k * LDF + 4 * ty);
    const float4 bv = *reinterpret_cast<const float4*>(Bs + k * LDF + 4 * tx);
    const float a[4] = {av.x, av.y, av.z, av.w}, b[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[p][q] = fmaf(a[p], b[q], acc[p][q]);
  }
}

// One step of the factorisation: independent tasks, one CTA each.
template <typename T>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 3 : 2)
k_inv_step(const InvTask* __restrict__ tasks, const InvMat* __restrict__ mats, const int* __restrict__ active,
           int* __restrict__ notspd) {
  const InvTask t = tasks[blockIdx.x];
  const InvMat& m = mats[t.m];
  if (active != nullptr && !active[m.sub]) return;
  extern __shared__ __align__(16) unsigned char smem_iv[];
  __shared__ int em[2][TILE];
  const int tid = threadIdx.x, b = m.b;
  T* S = layer_block<T>(m, t.layer);
  if (t.type == IV_SCHUR_A) {
    // (C X)^T with X = -S^{-1} of layer layer + k: rows q, columns of layer `layer`
    T acc[2][3];
    const int q = t.j * TILE + (tid & 63);
    couple_rows<T>(m, t.i, t.k, t.layer, q, layer_block<T>(m, t.layer + t.k), reinterpret_cast<T*>(smem_iv), acc);
    T* W = triple_scratch<T>(m, t.layer, t.k);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int p = t.i * NBLK + (tid >> 6) * 2 + u;
      if (p < m.n / 3 && q < m.n)
#pragma unroll
        for (int r = 0; r < 3; ++r) W[(size_t)q * b + 3 * p + r] = acc[u][r];
    }
    return;
  }
  if (t.type == IV_SCHUR_B) {
    // D += C (C X)^T on and below the diagonal, mirrored
    T acc[2][3];
    const int q = t.j * TILE + (tid & 63);
    couple_rows<T>(m, t.i, t.k, t.layer, q, triple_scratch<T>(m, t.layer, t.k), reinterpret_cast<T*>(smem_iv), acc);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int p = t.i * NBLK + (tid >> 6) * 2 + u;
      if (p < m.n / 3 && q < m.n)
#pragma unroll
        for (int r = 0; r < 3; ++r) {
          const int row = 3 * p + r;
          if (q > row) continue;
          const T v = S[(size_t)row * b + q] + acc[u][r];
          S[(size_t)row * b + q] = v;
          if (q < row) S[(size_t)q * b + row] = v;
        }
    }
    return;
  }
  if (t.type == IV_PIVOT) {
    tile_sweep<T>(S, b, pivot_inv<T>(m, t.layer), smem_iv, notspd, m.sub);
    return;
  }
  const int k = t.k;
  T* P = pivot_inv<T>(m, t.layer);
  T* C = old_col<T>(m, t.layer);
  if (t.type == IV_PANEL && k == 0 && m.yc != nullptr) {   // the diagonal before any update (k_inv_condition)
    if (tid < TILE) {
      const size_t r = (size_t)t.i * TILE + tid;
      static_cast<T*>(m.yc)[(size_t)t.layer * b + r] = S[r * b + r];
    }
    __syncthreads();
  }
  if (t.type == IV_PANEL && t.i == k) {
    T* Skk = S + (size_t)k * TILE * b + (size_t)k * TILE;
    for (int e = tid; e < TILE * TILE; e += 256) Skk[(size_t)(e >> 6) * b + (e & 63)] = -P[e];
    return;
  }
  T* Sik = S + (size_t)t.i * TILE * b + (size_t)k * TILE;
  // IV_PANEL: W_i = S_ik P in place and mirrored, the old tile kept in C;
  // IV_UPDATE: S_ij -= W_i old_j^T, mirrored; the next pivot tile is swept at once
  T* Ski = S + (size_t)k * TILE * b + (size_t)t.i * TILE;
  T* Sij = S + (size_t)t.i * TILE * b + (size_t)t.j * TILE;
  T* Sji = S + (size_t)t.j * TILE * b + (size_t)t.i * TILE;
  const bool diag = t.i == t.j;
  if constexpr (sizeof(T) == 8) {
    if (t.type == IV_PANEL) {
      digit_tile(Sik, b, P, TILE, smem_iv, em, C + (size_t)t.i * TILE * TILE, [&](int r, int c, double v0, double v1) {
        *reinterpret_cast<double2*>(Sik + (size_t)r * b + c) = make_double2(v0, v1);
        Ski[(size_t)c * b + r] = v0;
        Ski[(size_t)(c + 1) * b + r] = v1;
      });
      return;
    }
    digit_tile(Sik, b, C + (size_t)t.j * TILE * TILE, TILE, smem_iv, em, nullptr, [&](int r, int c, double v0, double v1) {
      if (!diag) {
        double2* o = reinterpret_cast<double2*>(Sij + (size_t)r * b + c);
        double2 x = *o;
        x.x -= v0;
        x.y -= v1;
        *o = x;
        Sji[(size_t)c * b + r] = x.x;
        Sji[(size_t)(c + 1) * b + r] = x.y;
        return;
      }
      // diagonal tile: lower half and its mirror image
      if (c <= r) Sij[(size_t)c * b + r] = Sij[(size_t)r * b + c] -= v0;
      if (c + 1 <= r) Sij[(size_t)(c + 1) * b + r] = Sij[(size_t)r * b + c + 1] -= v1;
    });
    if (diag && t.i == k + 1) {
      __syncthreads();   // the tile's stores are visible to the CTA
      tile_sweep<T>(Sij, b, P, smem_iv, notspd, m.sub);
    }
  } else {
    float* As = reinterpret_cast<float*>(smem_iv);
    float* Bs = As + TILE * LDF;
    const int tx = tid & 15, ty = tid >> 4;
    const bool panel = t.type == IV_PANEL;
    T* Ci = C + (size_t)t.i * TILE * TILE;
    stage_tile(Sik, b, As);
    stage_tile(panel ? P : C + (size_t)t.j * TILE * TILE, TILE, Bs);
    __syncthreads();
    float acc[4][4];
    tile_product(As, Bs, acc);
    if (panel)
      for (int e = tid; e < TILE * TILE; e += 256) Ci[e] = As[(e & 63) * LDF + (e >> 6)];
    __syncthreads();
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = 4 * ty + p, c = 4 * tx + q;
        if (panel) {
          As[r * LDF + c] = acc[p][q];
          continue;
        }
        if (diag && c > r) continue;
        const float v = Sij[(size_t)r * b + c] - acc[p][q];
        As[r * LDF + c] = v;
        if (diag) As[c * LDF + r] = v;
      }
    __syncthreads();
    T* out = panel ? Sik : Sij;
    T* mir = panel ? Ski : Sji;
    for (int e = tid; e < TILE * TILE; e += 256) {
      const int r = e >> 6, c = e & 63;
      out[(size_t)r * b + c] = As[r * LDF + c];
      if (panel || !diag) mir[(size_t)r * b + c] = As[c * LDF + r];
    }
    if (!panel && diag && t.i == k + 1) tile_sweep<T>(As, LDF, P, smem_iv, notspd, m.sub);
  }
}

// Conditioning of the Schur complements: the largest S_ii (S^{-1})_ii of the matrix's
// layers into cond[2 sub + mat] (zeroed before; as the bits of a positive float), infinity
// when a pivot was not positive or the value is no number.  D holds -S^{-1}, yc the
// diagonals of S.
template <typename T>
__global__ void __launch_bounds__(128)
k_inv_condition(const InvMat* __restrict__ mats, const int* __restrict__ active, const int* __restrict__ notspd,
                int* __restrict__ cond) {
  const InvMat& m = mats[blockIdx.x];
  const int l = blockIdx.y;
  if (l >= m.nL || (active != nullptr && !active[m.sub])) return;
  const T* D = layer_block<T>(m, l);
  const T* d = static_cast<const T*>(m.yc) + (size_t)l * m.b;
  float g = notspd[m.sub] ? INFINITY : 0.f;
  for (int r = threadIdx.x; r < m.n; r += 128) {
    const float v = (float)(-D[(size_t)r * m.b + r] * d[r]);
    g = v >= 0.f ? fmaxf(g, v) : INFINITY;
  }
  for (int o = 16; o > 0; o >>= 1) g = fmaxf(g, __shfl_xor_sync(0xffffffffu, g, o));
  if ((threadIdx.x & 31) == 0) atomicMax(&cond[2 * m.sub + m.mat], __float_as_int(g));
}

// Couplings of every layer in the solver's precision, packed per node for the
// solves: [layer][2: towards layer - 1, layer + 1][node][9 neighbours][3][3],
// node counts padded to a multiple of 4 (every rank's share is then a copy on a
// 16-byte boundary; 2 x 81 padded nodes fit in the b x b slot of a layer).
__host__ __device__ __forceinline__ int up4(int v) { return (v + 3) & ~3; }
template <typename T>
__global__ void k_inv_pack(const InvMat* __restrict__ mats, const int* __restrict__ active) {
  const InvMat& m = mats[blockIdx.x];
  if (active != nullptr && !active[m.sub]) return;
  const int nn = m.n / 3, np = up4(nn);
  for (int l = blockIdx.y; l < m.nL; l += gridDim.y) {
    T* out = static_cast<T*>(m.L) + (size_t)l * m.b * m.b;
    for (int e = threadIdx.x; e < 2 * np * 81; e += blockDim.x) {
      const int dir = e / (np * 81), p = (e / 81) % np, s = e % 81, dk = dir ? 1 : -1;
      double v = 0.0;
      if (p < nn && l + dk >= 0 && l + dk < m.nL) v = coupling(m, l, p, dk, s / 9, (s % 9) / 3, s % 3);
      out[e] = (T)v;
    }
  }
}

// ---------------------------------------------------------------------------
// Solve of KB right-hand sides.  One thread-block cluster of G CTAs per half
// chain: rank g holds a contiguous share of the layer's rows (in stages of RS
// rows) and of its nodes.  Per layer: (1) the sparse step on the own nodes, z to
// every rank's shared memory; cluster barrier; (2) the own rows of S^{-1} z,
// results to the ranks whose nodes neighbour them; cluster barrier.  The rows of
// S^{-1} are contiguous in memory and depend on nothing, so they stream through
// a ring of bulk copies (cp.async.bulk, one per stage) that runs ahead across
// the layers: the ring is full again when the barriers are passed.  Serves the layers
// that neither k_inv_solve_f32 nor k_inv_solve_fx takes (more than about 1,000 DoFs).
struct InvSolveArgs {
  const InvMat* mats;
  const int* list;          // matrices (largest first)
  const SubDev* subs;
  const int* active;
  int src, dst, stride, coloff, neg, add;
  int ring, smem_z, smem_u, smem_c, smem_r;   // stages, byte offsets of the shared arrays
  int* err;
};

template <typename T>
__device__ __forceinline__ int zpos(int row, int col) {
  // rows in chunks of one 16-byte vector, each chunk padded by 16 bytes (bank
  // groups of the eight lanes of a 128-bit phase differ)
  constexpr int VN = 16 / sizeof(T);
  return (row / VN) * (VN * (KB + 1)) + (row % VN) * KB + col;
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src),
      "r"(bytes), "r"(bar)
      : "memory");
}

template <typename T, int RS, bool BACK>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 2 : 1)
k_inv_solve(const InvSolveArgs a) {
  constexpr int VN = 16 / sizeof(T);
  constexpr int KS = 8 / (RS / 4);            // warps that share a row group (4 rows), splitting k
  using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
  cg::cluster_group cl = cg::this_cluster();
  const int G = (int)cl.num_blocks(), g = (int)cl.block_rank();
  const int task = blockIdx.x / G, half = task & 1;
  const InvMat m = a.mats[a.list[task >> 1]];
  if (a.active != nullptr && !a.active[m.sub]) return;   // uniform over the cluster
  // layers of this half chain, in order: forward from the end, backward from the middle
  const int nch = half ? m.nL - 1 - m.mid : m.mid;        // layers without the middle one
  const int steps = BACK ? nch + 1 : nch;
  if (!BACK && nch == 0) return;
  if (BACK && half && nch == 0) return;
  auto layer_of = [&](int t) {
    if (BACK) return half ? m.mid + t : m.mid - t;
    return half ? m.nL - 1 - t : t;
  };
  extern __shared__ __align__(128) unsigned char smem_sv[];
  T* ring = reinterpret_cast<T*>(smem_sv);
  T* zb = reinterpret_cast<T*>(smem_sv + a.smem_z);
  T* uw = reinterpret_cast<T*>(smem_sv + a.smem_u);
  T* cf = reinterpret_cast<T*>(smem_sv + a.smem_c);
  T* red = reinterpret_cast<T*>(smem_sv + a.smem_r);      // [2][KS][RS][KB]
  __shared__ __align__(8) unsigned long long bars[9];     // ring slots, couplings
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int b = m.b, nn = m.n / 3;
  const int NS = (m.n + RS - 1) / RS, s0 = NS * g / G, s1 = NS * (g + 1) / G, ns = s1 - s0;
  const int npc = up4((nn + G - 1) / G), p0 = min(nn, npc * g), p1 = min(nn, p0 + npc);
  const int wlo = max(0, p0 - m.njc - 1);                 // first node of the window of neighbour values
  const uint32_t ring_s = tc::saddr(ring), bar0 = tc::saddr(bars), cf_s = tc::saddr(cf);
  const uint32_t stage_bytes = (uint32_t)(RS * b * sizeof(T));
  const int total = ns * steps;
  bool ok = true;
  int issued = 0;   // stages requested (thread 0)
  auto issue = [&](int i) {
    issued = i + 1;
    const int l = layer_of(i / ns), s = s0 + i % ns;
    const uint32_t bar = bar0 + 8 * (i % a.ring);
    tc::mbar_expect_tx(bar, stage_bytes);
    bulk_load(ring_s + (uint32_t)(i % a.ring) * stage_bytes, static_cast<const T*>(m.D) + ((size_t)l * b + (size_t)s * RS) * b,
              stage_bytes, bar);
  };
  // couplings of the own nodes in the layer of step t: towards the previous
  // layer of the chain (forward) or towards the middle (backward)
  const int cdir = BACK ? (half ? 0 : 1) : (half ? 1 : 0);
  const uint32_t cbytes = p1 > p0 ? (uint32_t)(up4(p1 - p0) * 81 * sizeof(T)) : 0;
  auto coupling_ptr = [&](int l, int dir) {
    return static_cast<const T*>(m.L) + (size_t)l * b * b + ((size_t)dir * up4(nn) + p0) * 81;
  };
  if (tid == 0) {
    for (int i = 0; i < 9; ++i) tc::mbar_init(bar0 + 8 * i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int i = 0; i < a.ring && i < total; ++i) issue(i);
  }
  for (int e = tid; e < ((b + VN - 1) / VN) * VN * (KB + 1); e += 256) zb[e] = (T)0;
  __syncthreads();
  const SubDev& sd = a.subs[m.sub];
  const double* src = mv_ptr(sd, a.src) + a.coloff;
  double* dst = mv_ptr(sd, a.dst) + a.coloff;
  T* yc = static_cast<T*>(m.yc);
  const T sgn = a.neg ? (T)-1 : (T)1;
  int cphase = 0, ci = 0;   // coupling copies waited for; stages consumed
  int waited = 0;           // stages whose copies have arrived
  bool cpend = false;
  cl.sync();   // no remote store before every CTA of the cluster has cleared its arrays
  for (int t = 0; t < steps; ++t) {
    const int l = layer_of(t);
    // ---- sparse step on the own nodes
    const bool first = t == 0;
    if (cpend) {
      if (ok) ok = tc::mbar_wait(bar0 + 64, cphase & 1);
      ++cphase;
    }
    for (int e = tid; e < (p1 - p0) * KB; e += 256) {
      const int pl = e / KB, col = e % KB, p = p0 + pl;
      const int i = p / m.njc, j = p % m.njc;
      T z[3] = {(T)0, (T)0, (T)0};
      if (!BACK || first) {
        const size_t node = (size_t)l * m.npl + (size_t)(m.ia + i) * m.nyn + m.ja + j;
#pragma unroll
        for (int r = 0; r < 3; ++r) z[r] = sgn * (T)src[(node * 3 + r) * a.stride + col];
        if (m.pinned && l == 0)
#pragma unroll
          for (int r = 0; r < 3; ++r)
            if (pinned_row(m, 0, 3 * p + r)) z[r] = (T)0;
      }
      auto sub_coupling = [&](const T* c, const T* u) {   // z -= C u, u indexed by row * KB
        T acc[3] = {(T)0, (T)0, (T)0};
#pragma unroll
        for (int s9 = 0; s9 < 9; ++s9) {
          const int di = s9 / 3 - 1, dj = s9 % 3 - 1;
          if (i + di < 0 || i + di >= m.nic || j + dj < 0 || j + dj >= m.njc) continue;
          const T* x = u + (ptrdiff_t)(3 * (p + di * m.njc + dj)) * KB + col;
          const T x0 = x[0], x1 = x[KB], x2 = x[2 * KB];
#pragma unroll
          for (int r = 0; r < 3; ++r)
            acc[r] = fma(c[s9 * 9 + 3 * r], x0, fma(c[s9 * 9 + 3 * r + 1], x1, fma(c[s9 * 9 + 3 * r + 2], x2, acc[r])));
        }
#pragma unroll
        for (int r = 0; r < 3; ++r) z[r] -= acc[r];
      };
      if (BACK && first) {
        // middle layer: both half chains' u from memory
        if (m.mid > 0) sub_coupling(coupling_ptr(l, 0) + (size_t)pl * 81, yc + (size_t)(l - 1) * b * KB);
        if (m.mid + 1 < m.nL) sub_coupling(coupling_ptr(l, 1) + (size_t)pl * 81, yc + (size_t)(l + 1) * b * KB);
      } else if (!first) {
        sub_coupling(cf + (size_t)pl * 81, uw - (ptrdiff_t)wlo * 3 * KB);
      }
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        const int pos = zpos<T>(3 * p + r, col);
        for (int q = 0; q < G; ++q) cl.map_shared_rank(zb, q)[pos] = z[r];
      }
    }
    cl.sync();
    // the coupling buffer is free: request the next layer's
    cpend = t + 1 < steps && cbytes > 0;
    if (cpend && ok && tid == 0) {
      tc::fence_async_smem();
      tc::mbar_expect_tx(bar0 + 64, cbytes);
      bulk_load(cf_s, coupling_ptr(layer_of(t + 1), cdir), cbytes, bar0 + 64);
    }
    // ---- dense step on the own rows
    const int nchunk = (m.n + VN - 1) / VN;
    for (int s = s0; s < s1; ++s, ++ci) {
      const int slot = ci % a.ring;
      if (ok) {
        ok = tc::mbar_wait(bar0 + 8 * slot, (ci / a.ring) & 1);
        if (ok) waited = ci + 1;
      }
      const T* st = ring + (size_t)slot * RS * b;
      const int rg = w / KS, ks = w % KS;
      T acc[32];
#pragma unroll
      for (int e = 0; e < 32; ++e) acc[e] = (T)0;
      const T* a0 = st + (size_t)rg * 4 * b;
#pragma unroll 1
      for (int c = ks * 32 + lane; c < nchunk; c += 32 * KS) {
        T av[4][VN];
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const V x = *reinterpret_cast<const V*>(a0 + (size_t)r * b + c * VN);
          const T* e = reinterpret_cast<const T*>(&x);
#pragma unroll
          for (int q = 0; q < VN; ++q) av[r][q] = e[q];
        }
        const T* zp = zb + (size_t)c * VN * (KB + 1);
#pragma unroll
        for (int q = 0; q < VN; ++q) {
          T zv[KB];
#pragma unroll
          for (int h = 0; h < KB / VN; ++h) {
            const V x = *reinterpret_cast<const V*>(zp + q * KB + h * VN);
            const T* e = reinterpret_cast<const T*>(&x);
#pragma unroll
            for (int o = 0; o < VN; ++o) zv[h * VN + o] = e[o];
          }
#pragma unroll
          for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int o = 0; o < KB; ++o) acc[r * KB + o] = fma(av[r][q], zv[o], acc[r * KB + o]);
        }
      }
      // lane L ends with the sum of entry L (row L / KB, column L % KB)
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const bool up = lane & off;
#pragma unroll
        for (int e = 0; e < off; ++e) {
          const T send = up ? acc[e] : acc[e + off];
          const T keep = up ? acc[e + off] : acc[e];
          acc[e] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
      }
      T* rd = red + (size_t)(ci & 1) * KS * RS * KB;
      rd[((size_t)ks * RS + rg * 4) * KB + lane] = acc[0];
      __syncthreads();
      if (tid == 0 && ok && ci + a.ring < total) {
        tc::fence_async_smem();
        issue(ci + a.ring);
      }
      for (int e = tid; e < RS * KB; e += 256) {
        const int row = s * RS + e / KB, col = e % KB;
        if (row >= m.n) continue;
        T y = rd[e];
#pragma unroll
        for (int q = 1; q < KS; ++q) y += rd[q * RS * KB + e];
        T* yp = yc + ((size_t)l * b + row) * KB + col;
        T x;   // the block holds -S^{-1}
        if (BACK && !first) x = *yp + (-y);
        else x = -y;
        if (!BACK) *yp = x;
        else if (!first || half == 0) {
          const int p = row / 3;
          const size_t node = (size_t)l * m.npl + (size_t)(m.ia + p / m.njc) * m.nyn + m.ja + p % m.njc;
          double* o = dst + (node * 3 + row % 3) * a.stride + col;
          *o = a.add ? *o + (double)x : (double)x;
        }
        if (t + 1 < steps) {
          const int p = row / 3;
          for (int q = 0; q < G; ++q) {
            const int q0 = min(nn, npc * q), lo = max(0, q0 - m.njc - 1), hi = min(nn, min(nn, q0 + npc) + m.njc + 1);
            if (p >= lo && p < hi) cl.map_shared_rank(uw, q)[(size_t)(row - 3 * lo) * KB + col] = x;
          }
        }
      }
    }
    cl.sync();
  }
  if (!__syncthreads_and(ok) && tid == 0) {
    // a copy did not arrive within its limit: wait once more for those in flight, then report
    for (int i = waited; i < issued; ++i) tc::mbar_wait(bar0 + 8 * (i % a.ring), (i / a.ring) & 1);
    if (cphase > 0) tc::mbar_wait(bar0 + 64, (cphase - 1) & 1);
    if (a.err != nullptr) atomicExch(a.err, KERR_SOLVE_COPY);
  }
}

// ---------------------------------------------------------------------------
// FP32 solve of layers up to 1,024 DoFs.  The cluster, the chain and the sparse step are
// those of k_inv_solve; the dense step is laid out so that neither shuffles nor CTA
// barriers stand in its loop:
//   - lane = row: a rank owns up to 8 blocks of 32 rows, a warp a fixed eighth of the
//     columns; a lane adds 4 columns x 8 right-hand sides for its row of every block in
//     packed FMAs, z comes as shared-memory broadcasts, 24 reads of 128 bytes per 512
//     entries of 4 blocks (rows across 32 lanes of k: 48, and 31 shuffles per 4 rows);
//   - the factorisation's last kernel puts -S^{-1} into that order (k_inv_pack_f32), so a
//     warp streams its own 512-byte rows of lanes with its own ring of bulk copies and
//     mbarriers and waits for nobody until the layer's end;
//   - there the eight warps' sums are added through shared memory, and all threads write
//     the results (two warps after every stage before).
// All solves of a local stage, k_inv_solve -> here: C-section of 16 subdomains (layers up
// to 714 and 912 DoFs) 188 -> 124 ms, 192 x 12 x 39 beam (570 and 693) 204 -> 154 ms
// (3.1 TB/s, 46 % of the HBM copy rate), 48 beams (210 and 225) 42 -> 23 ms, 47 x 7 x 13
// beam (360 and 408, 20 half chains) 20 -> 17 ms.  Bound by the steps' latency: of a step of
// 21 us on 912 DoFs the products take about 8 in issue slots (two CTAs per SM), the sparse
// step, two cluster barriers and the wait for the slowest rank the rest (issue slots 36 %
// busy, DRAM 32 %, barriers the largest stall).
constexpr int F32_BLOCKS = 8;    // blocks of 32 rows per rank
constexpr int F32_WIDE = 1024;   // widest layer

// -S^{-1} of layer l in the order of the solve: the triple products' scratch, the last
// layer in layer 0's place (packed before)
__device__ __forceinline__ float* packed_layer(const InvMat& m, int l) {
  return l + 1 < m.nL ? static_cast<float*>(m.E) + (size_t)l * m.b * m.b : static_cast<float*>(m.D);
}
// blocks of 32 rows per rank of a cluster of G
__host__ __device__ __forceinline__ int f32_blocks(int n, int G) { return ((n + 31) / 32 + G - 1) / G; }

// Layer l < nL - 1 (last = 0) or nL - 1 (last = 1), block of 32 rows: rank's strip of Rg
// rows, then [column / 4][row of the strip][4]; zero outside the n x n matrix.
__global__ void __launch_bounds__(256)
k_inv_pack_f32(const InvMat* __restrict__ mats, const int* __restrict__ active, int last) {
  const InvMat& m = mats[blockIdx.x];
  if (m.sg == 0 || (active != nullptr && !active[m.sub])) return;
  const int l = last ? m.nL - 1 : blockIdx.y, rb = blockIdx.z, nb = (m.n + 31) / 32, kp = nb * 32;
  if (rb >= nb || (!last && l >= m.nL - 1)) return;
  __shared__ float4 tile[32][33];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int nbr = f32_blocks(m.n, m.sg), g = rb / nbr, Rg = 32 * min(nbr, nb - g * nbr);
  const float* D = static_cast<const float*>(m.D) + ((size_t)l * m.b + (size_t)rb * 32) * m.b;
  float4* out = reinterpret_cast<float4*>(packed_layer(m, l)) + (size_t)g * nbr * 32 * (kp / 4) + (rb - g * nbr) * 32;
  for (int c0 = 0; c0 < kp / 4; c0 += 32) {
    for (int r = w; r < 32; r += 8) {
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
      const int c = 4 * (c0 + lane);
      if (rb * 32 + r < m.n && c < m.n) {
        x = *reinterpret_cast<const float4*>(D + (size_t)r * m.b + c);
        if (c + 1 >= m.n) x.y = 0.f;
        if (c + 2 >= m.n) x.z = 0.f;
        if (c + 3 >= m.n) x.w = 0.f;
      }
      tile[r][lane] = x;
    }
    __syncthreads();
    for (int c = w; c < 32 && c0 + c < kp / 4; c += 8) out[(size_t)(c0 + c) * Rg + lane] = tile[lane][c];
    __syncthreads();
  }
}

__device__ __forceinline__ unsigned long long dup2(float x) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float2 split2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}

// A warp's ring: groups of 4 columns x Rg rows, in the order they are used
struct F32Ring {
  uint32_t smem, bar, bytes;   // first slot, first mbarrier, bytes per group
  int depth, used;             // slots; groups consumed
  bool ok;
};

// Dense step of one layer for NR blocks of rows: the warp's ngrp groups against z, the
// eight warps' sums added into red[4][2][Rg][4] (to be summed over its four slots).
template <int NR, typename Issue>
__device__ __forceinline__ void dense_f32(F32Ring& rg, const float4* slots, const float* z, int ngrp, float* red,
                                          Issue issue) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  unsigned long long acc[NR][4];
#pragma unroll
  for (int r = 0; r < NR; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[r][c] = 0ull;
#pragma unroll 1
  for (int i = 0; i < ngrp; ++i, ++rg.used) {
    const int slot = rg.used % rg.depth;
    if (rg.ok) rg.ok = tc::mbar_wait(rg.bar + 8 * slot, (rg.used / rg.depth) & 1);
    const float4* sp = slots + slot * NR * 32 + lane;
    const float* zp = z + i * 4 * KB;
    float4 sv[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) sv[r] = sp[r * 32];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const ulonglong2 z0 = *reinterpret_cast<const ulonglong2*>(zp + q * KB);
      const ulonglong2 z1 = *reinterpret_cast<const ulonglong2*>(zp + q * KB + 4);
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const unsigned long long x = dup2(q == 0 ? sv[r].x : q == 1 ? sv[r].y : q == 2 ? sv[r].z : sv[r].w);
        fma2(acc[r][0], x, z0.x);
        fma2(acc[r][1], x, z0.y);
        fma2(acc[r][2], x, z1.x);
        fma2(acc[r][3], x, z1.y);
      }
    }
    __syncwarp();
    issue();   // the slot is free
  }
  float4* rd = reinterpret_cast<float4*>(red) + (size_t)(w & 3) * 2 * NR * 32 + lane;
  auto put = [&](bool add) {
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const float2 u = split2(acc[r][2 * hf]), v = split2(acc[r][2 * hf + 1]);
        float4* o = rd + (hf * NR + r) * 32;
        float4 x = make_float4(u.x, u.y, v.x, v.y);
        if (add) x = make_float4(x.x + o->x, x.y + o->y, x.z + o->z, x.w + o->w);
        *o = x;
      }
  };
  if (w >= 4) put(false);
  __syncthreads();
  if (w < 4) put(true);
  __syncthreads();
}

template <bool BACK>
__global__ void __launch_bounds__(256, 2)
k_inv_solve_f32(const InvSolveArgs a) {
  cg::cluster_group cl = cg::this_cluster();
  const int G = (int)cl.num_blocks(), g = (int)cl.block_rank();
  const int task = blockIdx.x / G, half = task & 1;
  const InvMat& m = a.mats[a.list[task >> 1]];
  if (a.active != nullptr && !a.active[m.sub]) return;   // uniform over the cluster
  const int nch = half ? m.nL - 1 - m.mid : m.mid;        // layers without the middle one
  const int steps = BACK ? nch + 1 : nch;
  if (!BACK && nch == 0) return;
  if (BACK && half && nch == 0) return;
  const int mid = m.mid, nL = m.nL;
  auto layer_of = [&](int t) {
    if (BACK) return half ? mid + t : mid - t;
    return half ? nL - 1 - t : t;
  };
  extern __shared__ __align__(128) unsigned char smem_sv[];
  float* ring = reinterpret_cast<float*>(smem_sv);
  float* zb = reinterpret_cast<float*>(smem_sv + a.smem_z);   // [b][KB]
  float* uw = reinterpret_cast<float*>(smem_sv + a.smem_u);
  float* cf = reinterpret_cast<float*>(smem_sv + a.smem_c);
  float* red = reinterpret_cast<float*>(smem_sv + a.smem_r);  // [4][2][Rg][4]
  __shared__ __align__(8) unsigned long long bars[65];        // the warps' ring slots, couplings
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int b = m.b, n = m.n, nn = n / 3, njc = m.njc, nic = m.nic;
  const int nbr = f32_blocks(n, G), nb = max(0, min(nbr, (n + 31) / 32 - g * nbr));   // own blocks of 32 rows
  const int r0 = g * nbr * 32, nrow = max(0, min(n - r0, nb * 32));
  const int npc = up4((nn + G - 1) / G), p0 = min(nn, npc * g), p1 = min(nn, p0 + npc);
  const int wlo = max(0, p0 - njc - 1);                       // first node of the window of neighbour values
  const uint32_t bar0 = tc::saddr(bars), cbar = bar0 + 8 * 64, cf_s = tc::saddr(cf);
  // the warp's ring: its eighth of the columns, group by group, layer by layer
  const int ngrp = (n + 31) / 32, total = nb > 0 ? ngrp * steps : 0;
  F32Ring rg;
  rg.depth = a.ring;
  rg.bytes = (uint32_t)nb * 512;
  rg.smem = tc::saddr(ring) + (uint32_t)w * a.ring * rg.bytes;
  rg.bar = bar0 + 8 * 8 * w;
  rg.used = 0;
  rg.ok = true;
  const float4* slots = reinterpret_cast<const float4*>(ring) + (size_t)w * a.ring * nb * 32;
  int issued = 0, ist = 0, isg = 0;   // groups requested; step and group of the next (lane 0)
  auto issue = [&]() {
    if (lane != 0 || issued >= total || !rg.ok) return;
    const int slot = issued % rg.depth;
    tc::fence_async_smem();
    tc::mbar_expect_tx(rg.bar + 8 * slot, rg.bytes);
    bulk_load(rg.smem + slot * rg.bytes,
              packed_layer(m, layer_of(ist)) + ((size_t)r0 * ngrp * 8 + (size_t)(w * ngrp + isg) * nb * 32) * 4, rg.bytes,
              rg.bar + 8 * slot);
    ++issued;
    if (++isg == ngrp) { isg = 0; ++ist; }
  };
  const int cdir = BACK ? (half ? 0 : 1) : (half ? 1 : 0);
  const uint32_t cbytes = p1 > p0 ? (uint32_t)(up4(p1 - p0) * 81 * sizeof(float)) : 0;
  auto coupling_ptr = [&](int l, int dir) {
    return static_cast<const float*>(m.L) + (size_t)l * b * b + ((size_t)dir * up4(nn) + p0) * 81;
  };
  if (tid == 0) {
    for (int i = 0; i < 65; ++i) tc::mbar_init(bar0 + 8 * i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int e = tid; e < b * KB; e += 256) zb[e] = 0.f;
  __syncthreads();
  for (int i = 0; i < a.ring; ++i) issue();
  const SubDev& sd = a.subs[m.sub];
  const double* src = mv_ptr(sd, a.src) + a.coloff;
  double* dst = mv_ptr(sd, a.dst) + a.coloff;
  float* yc = static_cast<float*>(m.yc);
  const float sgn = a.neg ? -1.f : 1.f;
  int cphase = 0;   // coupling copies waited for
  bool cpend = false, cok = true;
  // sparse step: task e = ((node, component), half of the columns); the source values of
  // a thread's first task of the next layer are requested before the dense step
  const int ntask = (p1 - p0) * 6;
  auto source = [&](int l, int e, double (&v)[4]) {
    const int p = p0 + e / 6, r = (e % 6) >> 1;
    const size_t node = (size_t)l * m.npl + (size_t)(m.ia + p / njc) * m.nyn + m.ja + p % njc;
#pragma unroll
    for (int c = 0; c < 4; ++c) v[c] = src[(node * 3 + r) * a.stride + (e & 1) * 4 + c];
  };
  double pre[4] = {0.0, 0.0, 0.0, 0.0};
  if (tid < ntask) source(layer_of(0), tid, pre);
  cl.sync();   // no remote store before every CTA of the cluster has cleared its arrays
  for (int t = 0; t < steps; ++t) {
    const int l = layer_of(t);
    const bool first = t == 0;
    if (cpend) {
      if (cok) cok = tc::mbar_wait(cbar, cphase & 1);
      ++cphase;
    }
    for (int e = tid; e < ntask; e += 256) {
      const int pl = e / 6, r = (e % 6) >> 1, c0 = (e & 1) * 4, p = p0 + pl;
      const int i = p / njc, j = p % njc;
      float z[4] = {0.f, 0.f, 0.f, 0.f};
      if (!BACK || first) {
        double v[4] = {pre[0], pre[1], pre[2], pre[3]};
        if (e != tid) source(l, e, v);
#pragma unroll
        for (int c = 0; c < 4; ++c) z[c] = pinned_row(m, l, 3 * p + r) ? 0.f : sgn * (float)v[c];
      }
      auto sub_coupling = [&](const float* c, const float* u) {   // z -= C u, u indexed by row * KB
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int s9 = 0; s9 < 9; ++s9) {
          const int di = s9 / 3 - 1, dj = s9 % 3 - 1;
          if (i + di < 0 || i + di >= nic || j + dj < 0 || j + dj >= njc) continue;
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const float4 x = *reinterpret_cast<const float4*>(u + (ptrdiff_t)(3 * (p + di * njc + dj) + q) * KB + c0);
            const float cv = c[s9 * 9 + 3 * r + q];
            acc[0] = fmaf(cv, x.x, acc[0]);
            acc[1] = fmaf(cv, x.y, acc[1]);
            acc[2] = fmaf(cv, x.z, acc[2]);
            acc[3] = fmaf(cv, x.w, acc[3]);
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) z[q] -= acc[q];
      };
      if (BACK && first) {
        // middle layer: both half chains' u from memory
        if (mid > 0) sub_coupling(coupling_ptr(l, 0) + (size_t)pl * 81, yc + (size_t)(l - 1) * b * KB);
        if (mid + 1 < nL) sub_coupling(coupling_ptr(l, 1) + (size_t)pl * 81, yc + (size_t)(l + 1) * b * KB);
      } else if (!first) {
        sub_coupling(cf + (size_t)pl * 81, uw - (ptrdiff_t)wlo * 3 * KB);
      }
      for (int q = 0; q < G; ++q)
        *reinterpret_cast<float4*>(cl.map_shared_rank(zb, q) + (3 * p + r) * KB + c0) = make_float4(z[0], z[1], z[2], z[3]);
    }
    cl.sync();
    // the coupling buffer is free: request the next layer's
    cpend = t + 1 < steps && cbytes > 0;
    if (cpend && cok && tid == 0) {
      tc::fence_async_smem();
      tc::mbar_expect_tx(cbar, cbytes);
      bulk_load(cf_s, coupling_ptr(layer_of(t + 1), cdir), cbytes, cbar);
    }
    // ---- dense step on the own rows
    if (!BACK && t + 1 < steps && tid < ntask) source(layer_of(t + 1), tid, pre);
    float4 prey = make_float4(0.f, 0.f, 0.f, 0.f);   // u of the thread's first result
    if (BACK && !first && tid < 2 * nrow) {
      const int hf = tid >= nrow;
      prey = *reinterpret_cast<const float4*>(yc + ((size_t)l * b + r0 + tid - hf * nrow) * KB + 4 * hf);
    }
    const float* zw = zb + (size_t)w * ngrp * 4 * KB;
    switch (nb) {
      case 1: dense_f32<1>(rg, slots, zw, ngrp, red, issue); break;
      case 2: dense_f32<2>(rg, slots, zw, ngrp, red, issue); break;
      case 3: dense_f32<3>(rg, slots, zw, ngrp, red, issue); break;
      case 4: dense_f32<4>(rg, slots, zw, ngrp, red, issue); break;
      case 5: dense_f32<5>(rg, slots, zw, ngrp, red, issue); break;
      case 6: dense_f32<6>(rg, slots, zw, ngrp, red, issue); break;
      case 7: dense_f32<7>(rg, slots, zw, ngrp, red, issue); break;
      case 8: dense_f32<8>(rg, slots, zw, ngrp, red, issue); break;
    }
    for (int e = tid; e < 2 * nrow; e += 256) {
      const int hf = e >= nrow, rl = e - hf * nrow, row = r0 + rl, c0 = 4 * hf;
      float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const float4 v = reinterpret_cast<const float4*>(red)[(size_t)(q * 2 + hf) * nb * 32 + rl];
        y = make_float4(y.x + v.x, y.y + v.y, y.z + v.z, y.w + v.w);
      }
      float4* yp = reinterpret_cast<float4*>(yc + ((size_t)l * b + row) * KB + c0);
      float4 x = make_float4(-y.x, -y.y, -y.z, -y.w);   // the block holds -S^{-1}
      if (BACK && !first) {
        const float4 u = e == tid ? prey : *yp;
        x = make_float4(u.x + x.x, u.y + x.y, u.z + x.z, u.w + x.w);
      }
      const int p = row / 3;
      if (!BACK) *yp = x;
      else if (!first || half == 0) {
        const size_t node = (size_t)l * m.npl + (size_t)(m.ia + p / njc) * m.nyn + m.ja + p % njc;
        double* o = dst + (node * 3 + row % 3) * a.stride + c0;
        const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) o[c] = a.add ? o[c] + (double)xv[c] : (double)xv[c];
      }
      if (t + 1 < steps)
        for (int q = 0; q < G; ++q) {
          const int q0 = min(nn, npc * q), lo = max(0, q0 - njc - 1), hi = min(nn, min(nn, q0 + npc) + njc + 1);
          if (p >= lo && p < hi) *reinterpret_cast<float4*>(cl.map_shared_rank(uw, q) + (row - 3 * lo) * KB + c0) = x;
        }
    }
    cl.sync();
  }
  if (!__syncthreads_and(rg.ok && cok)) {
    // a copy did not arrive within its limit: wait once more for those in flight, then report
    if (lane == 0)
      for (int i = max(0, issued - rg.depth); i < issued; ++i)
        tc::mbar_wait(rg.bar + 8 * (i % rg.depth), (i / rg.depth) & 1);
    if (tid == 0 && cphase > 0) tc::mbar_wait(cbar, (cphase - 1) & 1);
    if (tid == 0 && a.err != nullptr) atomicExch(a.err, KERR_SOLVE_COPY);
  }
}

// ---------------------------------------------------------------------------
// FP64 solve in digit products
constexpr int FX_WARPS = 16;                    // two groups of eight
constexpr int FX_STAGE = FX_WARPS * 2048;       // bytes of a ring level: a 16 x 16 block for each warp
constexpr int FX_RED = 2 * 4 * 128 * 16;        // bytes of the partial sums of the groups' strips

// biased exponents of the rows of layer l (at the end of the layer's L slot)
__device__ __forceinline__ int* row_exponents(const InvMat& m, int l) {
  return reinterpret_cast<int*>(static_cast<double*>(m.L) + (size_t)(l + 1) * m.b * m.b - m.b / 2);
}

// -S^{-1} of every layer to biased integers in fragment order, in place: one strip of 16 rows per CTA
__global__ void __launch_bounds__(256)
k_inv_digits(const InvMat* __restrict__ mats, const int* __restrict__ active) {
  const InvMat& m = mats[blockIdx.x];
  if (active != nullptr && !active[m.sub]) return;
  const int l = blockIdx.y, s = blockIdx.z, nkb = (m.n + 15) / 16;
  if (l >= m.nL || s >= nkb) return;
  extern __shared__ __align__(16) unsigned char smem_dg[];
  double* v = reinterpret_cast<double*>(smem_dg);
  __shared__ int em[16];
  const int tid = threadIdx.x, b = m.b, ld = b + 2;
  double* D = static_cast<double*>(m.D) + ((size_t)l * b + (size_t)s * 16) * b;
  if (tid < 16) em[tid] = 0;
  __syncthreads();
  for (int e = tid; e < 16 * b; e += 256) {
    const int r = e / b, c = e % b;
    const double x = D[e];
    v[r * ld + c] = x;
    atomicMax(&em[r], (__double2hiint(x) >> 20) & 0x7ff);
  }
  __syncthreads();
  long long* out = reinterpret_cast<long long*>(D);
  for (int e = tid; e < nkb * 256; e += 256) {
    const int kb = e >> 8, j = (e >> 6) & 3, lane = (e >> 1) & 31;
    const int r = (lane >> 2) + 8 * (j & 1), c = kb * 16 + 2 * (lane & 3) + 8 * (j >> 1) + (e & 1);
    out[e] = biased_fixed(v[r * ld + c], em[r]);
  }
  if (tid < 16) row_exponents(m, l)[s * 16 + tid] = em[tid];
}

// Two groups of eight warps take the rank's strips in turn; a warp owns an eighth of the
// columns and streams its blocks through its own ring (nobody else waits for them); the
// eight sums of a strip, 64-bit integers, meet in shared memory once per strip and the
// results are written once per layer.
// Bound by the integer and FP16 pipes (five instructions per pair of digits) and, per
// layer, the FP64 sparse step (6 us of 37 on 693 DoFs and 8 ranks) and three barriers.  A
// stage of 16 blocks per CTA with shared 64-bit atomics and a CTA barrier per stage took
// 1.00 ms per half solve of the 36 x 12 x 39 beam, 0.75 here (0.86 with one group of eight
// warps); whole passes 139.4 -> 127.6 ms, 47 x 7 x 13 beam 37.0 -> 34.2, GenEO comparison
// 211 -> 207, Schwarz PCG 15.9 -> 15.4.
template <bool BACK>
__global__ void __launch_bounds__(32 * FX_WARPS, 1)
k_inv_solve_fx(const InvSolveArgs a) {
  cg::cluster_group cl = cg::this_cluster();
  const int G = (int)cl.num_blocks(), g = (int)cl.block_rank();
  const int task = blockIdx.x / G, half = task & 1;
  const InvMat m = a.mats[a.list[task >> 1]];
  if (a.active != nullptr && !a.active[m.sub]) return;   // uniform over the cluster
  const int nch = half ? m.nL - 1 - m.mid : m.mid;
  const int steps = BACK ? nch + 1 : nch;
  if (nch == 0 && (!BACK || half)) return;
  auto layer_of = [&](int t) {
    if (BACK) return half ? m.mid + t : m.mid - t;
    return half ? m.nL - 1 - t : t;
  };
  extern __shared__ __align__(128) unsigned char smem_fs[];
  unsigned char* ring = smem_fs;
  uint32_t* zd = reinterpret_cast<uint32_t*>(smem_fs + a.smem_z);   // [DIG][8 nkb pairs of rows][KB] FP16 pairs
  double* uw = reinterpret_cast<double*>(smem_fs + a.smem_u);
  double* cf = reinterpret_cast<double*>(smem_fs + a.smem_c);
  longlong2* red = reinterpret_cast<longlong2*>(smem_fs + a.smem_r);          // [2 groups][4][128]
  double* zo = reinterpret_cast<double*>(smem_fs + a.smem_r + FX_RED);        // z of the own nodes, then the results
  __shared__ __align__(8) unsigned long long bars[8 * FX_WARPS + 1];
  __shared__ int zm[KB], zmax[8][KB];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, grp = w >> 3, wg = w & 7, gt = tid & 255;
  const int b = m.b, nn = m.n / 3, nkb = (m.n + 15) / 16;
  const int s0 = nkb * g / G, s1 = nkb * (g + 1) / G, ns = s1 - s0;
  const int npc = up4((nn + G - 1) / G), p0 = min(nn, npc * g), p1 = min(nn, p0 + npc);
  const int wlo = max(0, p0 - m.njc - 1);
  const uint32_t bar0 = tc::saddr(bars), cbar = bar0 + 8 * 8 * FX_WARPS, cf_s = tc::saddr(cf);
  // the warp's ring: its blocks of the group's strips, layer by layer
  const int kw0 = nkb * wg / 8, nw = nkb * (wg + 1) / 8 - kw0, nsg = (ns + 1 - grp) / 2;
  const int total = nsg * nw * steps, depth = a.ring;
  const uint32_t ring_s = tc::saddr(ring) + (uint32_t)w * depth * 2048, wbar = bar0 + 8 * 8 * w;
  const longlong2* slots = reinterpret_cast<const longlong2*>(ring) + (size_t)w * depth * 128;
  bool ok = true, cok = true;
  int used = 0, issued = 0, ist = 0, iss = 0, isb = 0;   // blocks consumed, requested; step, strip, block of the next
  auto issue = [&]() {
    if (lane != 0 || issued >= total || !ok) return;
    const int slot = issued % depth;
    tc::fence_async_smem();
    tc::mbar_expect_tx(wbar + 8 * slot, 2048u);
    bulk_load(ring_s + slot * 2048u,
              static_cast<const double*>(m.D) + ((size_t)layer_of(ist) * b + (size_t)(s0 + grp + 2 * iss) * 16) * b +
                  (size_t)(kw0 + isb) * 256,
              2048u, wbar + 8 * slot);
    ++issued;
    if (++isb == nw) {
      isb = 0;
      if (++iss == nsg) { iss = 0; ++ist; }
    }
  };
  const int cdir = BACK ? (half ? 0 : 1) : (half ? 1 : 0);
  const uint32_t cbytes = p1 > p0 ? (uint32_t)(up4(p1 - p0) * 81 * sizeof(double)) : 0;
  auto coupling_ptr = [&](int l, int dir) {
    return static_cast<const double*>(m.L) + (size_t)l * b * b + ((size_t)dir * up4(nn) + p0) * 81;
  };
  if (tid == 0) {
    for (int i = 0; i < 8 * FX_WARPS + 1; ++i) tc::mbar_init(bar0 + 8 * i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int e = tid; e < DIG * nkb * 8 * KB; e += 32 * FX_WARPS) zd[e] = 0u;
  if (tid < KB) zm[tid] = 0;
  __syncthreads();
  for (int i = 0; i < depth; ++i) issue();
  const SubDev& sd = a.subs[m.sub];
  const double* src = mv_ptr(sd, a.src) + a.coloff;
  double* dst = mv_ptr(sd, a.dst) + a.coloff;
  double* yc = static_cast<double*>(m.yc);
  const double sgn = a.neg ? -1.0 : 1.0;
  int cphase = 0;
  bool cpend = false;
  cl.sync();   // no remote store before every CTA of the cluster has cleared its arrays
  for (int t = 0; t < steps; ++t) {
    const int l = layer_of(t);
    const bool first = t == 0;
    if (cpend) {
      if (cok) cok = tc::mbar_wait(cbar, cphase & 1);
      ++cphase;
    }
    // ---- sparse step on the own nodes (FP64), the largest exponent per column
    int mx = 0;
    for (int e = tid; e < (p1 - p0) * KB; e += 32 * FX_WARPS) {
      const int pl = e / KB, col = e % KB, p = p0 + pl;
      const int i = p / m.njc, j = p % m.njc;
      double z[3] = {0.0, 0.0, 0.0};
      if (!BACK || first) {
        const size_t node = (size_t)l * m.npl + (size_t)(m.ia + i) * m.nyn + m.ja + j;
#pragma unroll
        for (int r = 0; r < 3; ++r) z[r] = sgn * src[(node * 3 + r) * a.stride + col];
        if (m.pinned && l == 0)
#pragma unroll
          for (int r = 0; r < 3; ++r)
            if (pinned_row(m, 0, 3 * p + r)) z[r] = 0.0;
      }
      auto sub_coupling = [&](const double* c, const double* u) {
        double acc[3] = {0.0, 0.0, 0.0};
#pragma unroll
        for (int s9 = 0; s9 < 9; ++s9) {
          const int di = s9 / 3 - 1, dj = s9 % 3 - 1;
          if (i + di < 0 || i + di >= m.nic || j + dj < 0 || j + dj >= m.njc) continue;
          const double* x = u + (ptrdiff_t)(3 * (p + di * m.njc + dj)) * KB + col;
          const double x0 = x[0], x1 = x[KB], x2 = x[2 * KB];
#pragma unroll
          for (int r = 0; r < 3; ++r)
            acc[r] = fma(c[s9 * 9 + 3 * r], x0, fma(c[s9 * 9 + 3 * r + 1], x1, fma(c[s9 * 9 + 3 * r + 2], x2, acc[r])));
        }
#pragma unroll
        for (int r = 0; r < 3; ++r) z[r] -= acc[r];
      };
      if (BACK && first) {
        if (m.mid > 0) sub_coupling(coupling_ptr(l, 0) + (size_t)pl * 81, yc + (size_t)(l - 1) * b * KB);
        if (m.mid + 1 < m.nL) sub_coupling(coupling_ptr(l, 1) + (size_t)pl * 81, yc + (size_t)(l + 1) * b * KB);
      } else if (!first) {
        sub_coupling(cf + (size_t)pl * 81, uw - (ptrdiff_t)wlo * 3 * KB);
      }
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        zo[(3 * pl + r) * KB + col] = z[r];
        mx = max(mx, (__double2hiint(z[r]) >> 20) & 0x7ff);
      }
    }
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
    if (lane < KB) atomicMax(&zm[lane], mx);
    __syncthreads();
    if (tid < G * KB) cl.map_shared_rank(&zmax[g][tid % KB], tid / KB)[0] = zm[tid % KB];
    cl.sync();
    // the coupling buffer is free: request the next layer's
    cpend = t + 1 < steps && cbytes > 0;
    if (cpend && cok && tid == 0) {
      tc::fence_async_smem();
      tc::mbar_expect_tx(cbar, cbytes);
      bulk_load(cf_s, coupling_ptr(layer_of(t + 1), cdir), cbytes, cbar);
    }
    // ---- digits of the own rows (in pairs) to every rank
    if (tid < KB) zm[tid] = 0;
    {
      const int rows = 3 * (p1 - p0), col = tid % KB;
      int ez = 0;
      for (int q = 0; q < G; ++q) ez = max(ez, zmax[q][col]);
      for (int e = tid; e < (rows + 1) / 2 * KB; e += 32 * FX_WARPS) {
        const int rp = e / KB;
        const long long x0 = biased_fixed(zo[2 * rp * KB + col], ez);
        const long long x1 = 2 * rp + 1 < rows ? biased_fixed(zo[(2 * rp + 1) * KB + col], ez) : DIG_BIAS;
        uint32_t dg[DIG];
#pragma unroll
        for (int i = 0; i < DIG; ++i) dg[i] = digit_pair(x0, x1, i);
        const int pos = (3 * p0 / 2 + rp) * KB + col;
        for (int q = 0; q < G; ++q) {
          uint32_t* z = cl.map_shared_rank(zd, q) + pos;
#pragma unroll
          for (int i = 0; i < DIG; ++i) z[i * nkb * 8 * KB] = dg[i];
        }
      }
    }
    cl.sync();
    // ---- dense step on the own strips of 16 rows
    int ezc = 0;   // of the column of the strip's sums that this thread adds up
    for (int q = 0; q < G; ++q) ezc = max(ezc, zmax[q][(gt >> 1) % KB]);
    auto group_sync = [&]() { asm volatile("bar.sync %0, 256;" ::"r"(1 + grp) : "memory"); };
    longlong2* rd = red + grp * 4 * 128;
    for (int s = s0 + grp; s < s1; s += 2) {
      const int er = row_exponents(m, l)[s * 16 + (gt >> 1) / KB];
      long long hi[4] = {}, lo[4] = {};
      for (int k0 = 0; k0 < nw; k0 += 2) {
        float acc[DIG][4];
#pragma unroll
        for (int i = 0; i < DIG; ++i)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[i][e] = 0.f;
        for (int kb = k0; kb < min(nw, k0 + 2); ++kb, ++used) {
          const int slot = used % depth;
          if (ok) ok = tc::mbar_wait(wbar + 8 * slot, (used / depth) & 1);
          const longlong2* ap = slots + slot * 128;
          longlong2 x[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) x[j] = ap[j * 32 + lane];
          uint32_t bz[DIG][2];
          const uint32_t* zp = zd + ((kw0 + kb) * 8 + (lane & 3)) * KB + (lane >> 2);
#pragma unroll
          for (int i = 0; i < DIG; ++i) {
            bz[i][0] = zp[i * nkb * 8 * KB];
            bz[i][1] = zp[i * nkb * 8 * KB + 4 * KB];
          }
          __syncwarp();
          issue();   // the slot is free
#pragma unroll
          for (int i = 0; i < DIG; ++i) {
            uint32_t av[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) av[j] = digit_pair(x[j].x, x[j].y, i);
#pragma unroll
            for (int j = DIG - 1 - i; j < DIG; ++j) mma_f16(acc[i + j - (DIG - 1)], av, bz[j]);
          }
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) digit_flush(acc, e, hi[e], lo[e]);
      }
      auto entry = [&](int e) {
        return (wg & 3) * 128 + ((lane >> 2) + 8 * (e >> 1)) * KB + 2 * (lane & 3) + (e & 1);
      };
      group_sync();   // the previous strip's sums have been read
      if (wg >= 4)
#pragma unroll
        for (int e = 0; e < 4; ++e) rd[entry(e)] = make_longlong2(hi[e], lo[e]);
      group_sync();
      if (wg < 4)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const longlong2 v = rd[entry(e)];
          rd[entry(e)] = make_longlong2(hi[e] + v.x, lo[e] + v.y);
        }
      group_sync();
      // threads 2 i, 2 i + 1 of the group: the high and the low sum of entry i
      const long long* part = reinterpret_cast<const long long*>(rd) + gt;
      long long sum = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) sum += part[q * 256];
      const long long other = __shfl_xor_sync(0xffffffffu, sum, 1);
      if (!(tid & 1)) {
        double y = digit_value(sum, other, er + ezc - 2 * 1023 - 66);
        if (er == 0x7ff || ezc == 0x7ff) y = __longlong_as_double(0x7ff8000000000000ll);   // Inf or NaN operands
        zo[(s - s0) * 128 + (gt >> 1)] = y;
      }
    }
    __syncthreads();
    for (int e = tid; e < ns * 128; e += 32 * FX_WARPS) {
      const int row = s0 * 16 + e / KB, col = e % KB;
      if (row >= m.n) continue;
      const double y = zo[e];
      double* yp = yc + ((size_t)l * b + row) * KB + col;
      const double x = (BACK && !first) ? *yp - y : -y;   // the block holds -S^{-1}
      const int p = row / 3;
      if (!BACK) *yp = x;
      else if (!first || half == 0) {
        const size_t node = (size_t)l * m.npl + (size_t)(m.ia + p / m.njc) * m.nyn + m.ja + p % m.njc;
        double* o = dst + (node * 3 + row % 3) * a.stride + col;
        *o = a.add ? *o + x : x;
      }
      if (t + 1 < steps)
        for (int q = 0; q < G; ++q) {
          const int q0 = min(nn, npc * q), lo_n = max(0, q0 - m.njc - 1), hi_n = min(nn, min(nn, q0 + npc) + m.njc + 1);
          if (p >= lo_n && p < hi_n) cl.map_shared_rank(uw, q)[(size_t)(row - 3 * lo_n) * KB + col] = x;
        }
    }
    cl.sync();
  }
  if (!__syncthreads_and(ok && cok)) {
    if (lane == 0)
      for (int i = max(0, issued - depth); i < issued; ++i) tc::mbar_wait(wbar + 8 * (i % depth), (i / depth) & 1);
    if (tid == 0 && cphase > 0) tc::mbar_wait(cbar, (cphase - 1) & 1);
    if (tid == 0 && a.err != nullptr) atomicExch(a.err, KERR_SOLVE_COPY);
  }
}

}  // namespace

// ---------------------------------------------------------------------------
// host side

struct InvForm {
  std::vector<InvMat> mats;        // K and A11 of every subdomain (A11 may have no DoFs: not listed)
  InvMat* d_mats = nullptr;
  struct Solve {
    std::vector<int> list;         // matrices of one kind in a wave, largest first
    int* d_list = nullptr;
    int G = 1, ring = 2, smem_z = 0, smem_u = 0, smem_c = 0, smem_r = 0, smem = 0;
    bool rows32 = false;           // k_inv_solve_f32 (FP32, layers up to F32_WIDE)
  };
  struct Wave {
    std::vector<std::vector<SchedStep>> steps;   // per stream group
    InvTask* d_tasks = nullptr;
    std::vector<int> all;          // every matrix of the wave (packing)
    Solve solve[2];
  };
  std::vector<Wave> waves;
  // coarse matrix: sweep tasks of its T x T tiles (coarse_inv_build)
  InvMat* d_cmat = nullptr;
  InvTask* d_ctasks = nullptr;
  std::vector<SchedStep> csteps;
  int rs = 8;                      // rows per stage of the solves (by the widest layer and the type)
  bool digits = false;             // FP64: solves in digit products (k_inv_solve_fx)
  int* d_cond = nullptr;           // [2 N] conditioning of the matrices' Schur complements (float bits)
};

namespace {

constexpr int INV_SMEM = 225 * 1024;   // shared memory of one solve CTA

// Conditioning of the layers' Schur complements, gam = max_i S_ii (S^{-1})_ii, up to which
// their explicit inverses serve; beyond it a call goes over to the block Cholesky.  A
// product with S^{-1} is off by about eps gam, the block Cholesky's by less where the
// material or the mesh makes gam large.
// FP64, energy error of the particular functions against a refined 64-bit solution,
// inverse form / block Cholesky by gam of A11: up to 700 0.6 to 1.9 (E1 / E2 from 2 to
// 2,500; bricks of aspect ratio 1 to 60), nu = 0.499 at 150 3.2; E1 / E2 = 25,000 on cubes
// 4,000 13; nu = 0.49999 3,700 120; E1 / E2 = 250,000 42,000 190.  K (whose solves only
// steer the iteration; its eigen-residuals were level up to 170,000, fifty times larger at
// 3e7) has 20 to 4,400 on plies with aspect ratios up to 15 and curved sections.
// Mixed (CG and refinement take the factors as a preconditioner): steps and residuals as
// with the block Cholesky up to 26,000; at 170,000 a run ended at 3e-2 instead of 1e-6,
// and from 65,000 on pivots turn non-positive where the block Cholesky's do not.
constexpr float INV_COND_A11 = 1e3f, INV_COND_K = 1e5f, INV_COND_F32 = 5e4f;

template <typename T, int RS>
const void* solve_kernel_ptr(bool back) {
  return back ? (const void*)k_inv_solve<T, RS, true> : (const void*)k_inv_solve<T, RS, false>;
}
const void* solve_kernel(const msgfem* h, const InvForm& f, const InvForm::Solve& s, bool back) {
  if (s.rows32) return back ? (const void*)k_inv_solve_f32<true> : (const void*)k_inv_solve_f32<false>;
  if (f.digits) return back ? (const void*)k_inv_solve_fx<true> : (const void*)k_inv_solve_fx<false>;
  if (!h->mixed) return solve_kernel_ptr<double, 4>(back);
  return f.rs == 8 ? solve_kernel_ptr<float, 8>(back) : solve_kernel_ptr<float, 4>(back);
}

int solve_threads(const InvForm& f) { return f.digits ? 32 * FX_WARPS : 256; }
// fewest ring levels of a solve
int ring_min(const InvForm& f, const InvForm::Solve& s) { return f.digits || s.rows32 ? 1 : 2; }

// shared-memory layout of a solve over the listed matrices with G CTAs per
// cluster and `ring` stages; the total in bytes
int solve_layout(const msgfem* h, const InvForm& f, InvForm::Solve& s, int G, int ring) {
  const int es = h->mixed ? 4 : 8, vn = 16 / es;
  auto up = [](size_t v) { return (v + 127) / 128 * 128; };
  size_t st = 0, z = 0, u = 0, c = 0, o = 0;
  int wide = 0;
  for (int i : s.list) wide = std::max(wide, f.mats[i].b);
  s.rows32 = h->mixed && wide <= F32_WIDE;
  for (int i : s.list) {
    const InvMat& m = f.mats[i];
    const int nn = m.n / 3, npc = up4((nn + G - 1) / G);
    if (f.digits) {
      o = std::max(o, FX_RED + (size_t)std::max(npc * 3, ((m.n + 15) / 16 + G - 1) / G * 16) * KB * es);
      z = std::max(z, (size_t)((m.n + 15) / 16) * DIG * 8 * KB * 4);
      st = FX_STAGE;
    } else if (s.rows32) {
      const int rows = 32 * f32_blocks(m.n, G);
      if (rows > 32 * F32_BLOCKS) return 1 << 30;
      st = std::max(st, (size_t)rows * 16 * 8);          // a group of every warp
      z = std::max(z, (size_t)m.b * KB * es);
      o = std::max(o, (size_t)rows * KB * es * 4);
    } else {
      st = std::max(st, (size_t)f.rs * m.b * es);
      z = std::max(z, (size_t)((m.b + vn - 1) / vn) * vn * (KB + 1) * es);
    }
    u = std::max(u, (size_t)std::min(nn, npc + 2 * (m.njc + 1)) * 3 * KB * es);
    c = std::max(c, (size_t)npc * 81 * es);
  }
  s.G = G;
  s.ring = ring;
  s.smem_z = (int)up(st * ring);
  s.smem_u = (int)(s.smem_z + up(z));
  s.smem_c = (int)(s.smem_u + up(u));
  s.smem_r = (int)(s.smem_c + up(c));
  s.smem = (int)(s.smem_r + up(f.digits || s.rows32 ? o : (size_t)2 * (8 / (f.rs / 4)) * f.rs * KB * es));
  return s.smem;
}

int resident_clusters(const void* kernel, int G, int smem, int threads) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(G);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = G;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

// Cluster size and ring depth of a solve: the largest cluster with which every
// half chain is resident at once (they run side by side), with the deepest ring
// that one CTA per SM holds, or half an SM's shared memory when that makes more
// half chains resident; with more half chains than SMs one CTA each.
// FP32 layers up to F32_WIDE and digit solves: the fewest rounds of resident half chains, then the widest
// cluster.  All solves of a local stage, ms, by CTAs per half chain: 32 half chains of 912
// DoFs 8: 124, 4: 144; 64 of 570 (4 resident at once, 8 in two rounds) 8: 204, 4: 170;
// 192 of 225 DoFs 8: 66, 4: 38, 2: 31, 1: 34; 20 of 408 8: 20, 4: 20, 2: 27.  The ring's
// depth (2 to 8) changes none of them by more than 3 %, so one level is enough where it
// saves a round: 64 half chains of 693 and 570 DoFs 163 -> 154, 192 of 225 24.6 -> 23.5.
// Sizes that are no powers of two serve what just misses one (FP64, 20 half chains: 6
// instead of 4, 47 x 7 x 13 beam 32.7 -> 30.6 ms; layers of fewer blocks than 8: Schwarz
// PCG 15.5 -> 14.4, GenEO comparison 206 -> 202).
void choose_solve(const msgfem* h, const InvForm& f, InvForm::Solve& s) {
  const int chains = 2 * (int)s.list.size();
  int most = 1;
  solve_layout(h, f, s, 8, 2);   // the kernel
  const int strip = f.digits ? 16 : s.rows32 ? 32 : f.rs;
  for (int i : s.list) most = std::max(most, (f.mats[i].n + strip - 1) / strip / (f.digits || s.rows32 ? 1 : 2));
  auto fit = [&](int G, int limit) {
    int ring = 8;
    while (ring > ring_min(f, s) && solve_layout(h, f, s, G, ring) > limit) --ring;
    return solve_layout(h, f, s, G, ring) <= limit;
  };
  if (s.rows32 || f.digits) {
    int best = 0, rounds = 0, ring = 0;
    for (int G = 8; G >= 1; --G)
      for (int limit : {INV_SMEM, 108 * 1024}) {
        if (G > most || !fit(G, limit)) continue;
        const int res = std::max(1, resident_clusters(solve_kernel(h, f, s, true), G, s.smem, solve_threads(f)));
        const int n = (chains + res - 1) / res;
        if (best == 0 || n < rounds) {
          best = G;
          rounds = n;
          ring = s.ring;
        }
      }
    solve_layout(h, f, s, best, ring);
    return;
  }
  for (int G : {8, 4, 2, 1}) {
    if (G > 1 && G > most) continue;
    for (int limit : {INV_SMEM, 108 * 1024}) {
      if (!fit(G, limit)) continue;
      if (resident_clusters(solve_kernel(h, f, s, true), G, s.smem, solve_threads(f)) >= chains) return;
    }
  }
  if (fit(1, 108 * 1024)) return;
  for (int G : {1, 2, 4, 8})
    if (fit(G, INV_SMEM)) return;
}

}  // namespace

// Eligibility and geometry.  The inverse form serves the block Krylov solver
// with the default kernels; a request for a particular Cholesky schedule, tile
// kernel, tile precision or solve kernel keeps the block Cholesky, and so do
// layers whose solve stages do not fit in shared memory.
bool inv_create(msgfem* h) {
  const msgfem_options& o = h->opt;
  if (o.solver != 0 || o.solve_kernel != 0 || o.factor_schedule != 0 || o.factor_kernel != 0 || o.tile_chol != 0)
    return false;
  InvForm* f = new InvForm();
  const int es = h->mixed ? 4 : 8;
  int bmax = TILE;
  bool good = true;
  for (int j = 0; j < h->N && good; ++j) {
    const SubDev& s = h->sub[j];
    const HostSub& hs = h->hsub[j];
    for (int mat = 0; mat < 2 && good; ++mat) {
      InvMat m;
      memset(&m, 0, sizeof(m));
      m.sub = j;
      m.mat = mat;
      m.n = mat == 0 ? s.nK : s.nA;
      m.b = mat == 0 ? s.bK : s.bA;
      m.nL = s.nzn;
      m.mid = s.nzn / 2;
      m.npl = s.npl;
      m.nyn = s.nyn;
      m.stencil = s.stencil;
      m.D = h->mixed ? (void*)(mat == 0 ? s.DKf : s.DAf) : (void*)(mat == 0 ? s.DK : s.DA);
      m.E = h->mixed ? (void*)(mat == 0 ? s.EKf : s.EAf) : (void*)(mat == 0 ? s.EK : s.EA);
      m.L = h->mixed ? (void*)(mat == 0 ? s.LKf : s.LAf) : (void*)(mat == 0 ? s.LK : s.LA);
      m.yc = h->mixed ? (void*)(mat == 0 ? s.ycK8f : s.ycA8f) : (void*)(mat == 0 ? s.ycK8 : s.ycA8);
      // the kept nodes must be a box, numbered like the compact rows
      const std::vector<int>& map = mat == 0 ? hs.mapK : hs.mapA;
      if (m.n > 0) {
        const int q0 = map[0] / 3, q1 = map[m.n - 1] / 3;
        m.ia = q0 / s.nyn;
        m.ja = q0 % s.nyn;
        m.nic = q1 / s.nyn - m.ia + 1;
        m.njc = q1 % s.nyn - m.ja + 1;
        good = m.nic > 0 && m.njc > 0 && 3 * m.nic * m.njc == m.n;
        for (int r = 0; r < m.n && good; ++r) {
          const int p = r / 3;
          good = map[r] == 3 * ((m.ia + p / m.njc) * s.nyn + m.ja + p % m.njc) + r % 3;
        }
      }
      if (mat == 0 && s.floating) {
        m.pinned = 1;
        for (int i = 0; i < 6; ++i) {
          m.pin[i] = -1;
          if (s.pin[i] < 0) continue;
          good = good && s.pin[i] < 3 * s.npl;   // the pins sit in layer 0
          if (good) m.pin[i] = hs.invK[s.pin[i]];
        }
      }
      bmax = std::max(bmax, m.b);
      f->mats.push_back(m);
    }
  }
  // rows of at most 6 KiB: eight per stage (in FP64 those layers all take the digit products)
  f->rs = h->mixed && bmax * es <= 6144 ? 8 : 4;
  // two stages of the widest layer and its vectors must fit with the widest cluster
  InvForm::Solve probe;
  for (int i = 0; i < (int)f->mats.size(); ++i)
    if (f->mats[i].n > 0) probe.list.push_back(i);
  if (good && !h->mixed && !probe.list.empty()) {
    f->digits = true;
    f->digits = solve_layout(h, *f, probe, 8, 1) <= INV_SMEM && (size_t)16 * (bmax + 2) * 8 <= (size_t)INV_SMEM;
  }
  good = good && (f->digits || solve_layout(h, *f, probe, 8, 2) <= INV_SMEM);
  if (!good) {
    delete f;
    return false;
  }
  h->inv = f;
  return true;
}

void inv_destroy(msgfem* h) {
  delete h->inv;
  h->inv = nullptr;
}

// Task lists of every wave (after the waves' storage has been placed).
msgfem_status inv_build(msgfem* h) {
  InvForm& f = *h->inv;
  // shared-memory limits (of the current device)
  for (bool back : {false, true})
    for (const void* k : {solve_kernel_ptr<float, 8>(back), solve_kernel_ptr<float, 4>(back), solve_kernel_ptr<double, 4>(back)})
      CK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, INV_SMEM));
  CK(cudaFuncSetAttribute(k_inv_step<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, inv_step_smem<double>()));
  CK(cudaFuncSetAttribute(k_inv_step<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, inv_step_smem<float>()));
  for (const void* k : {(const void*)k_inv_solve_f32<false>, (const void*)k_inv_solve_f32<true>})
    CK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, INV_SMEM));
  for (const void* k : {(const void*)k_inv_solve_fx<false>, (const void*)k_inv_solve_fx<true>})
    CK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, INV_SMEM));
  CK(cudaFuncSetAttribute(k_inv_digits, cudaFuncAttributeMaxDynamicSharedMemorySize, INV_SMEM));
  void* p = nullptr;
  TRY(dev_alloc_bytes(h, &p, f.mats.size() * sizeof(InvMat)));
  f.d_mats = static_cast<InvMat*>(p);
  CK(cudaMemcpy(f.d_mats, f.mats.data(), f.mats.size() * sizeof(InvMat), cudaMemcpyHostToDevice));
  TRY(dev_alloc_bytes(h, &p, 2 * (size_t)h->N * sizeof(int)));
  f.d_cond = static_cast<int*>(p);
  TRY(kerr_ensure(h));
  f.waves.resize(h->waves.size());
  for (size_t w = 0; w < h->waves.size(); ++w) {
    InvForm::Wave& wv = f.waves[w];
    for (int j : h->waves[w].members)
      for (int mat = 0; mat < 2; ++mat)
        if (f.mats[2 * j + mat].n > 0) {
          wv.all.push_back(2 * j + mat);
          wv.solve[mat].list.push_back(2 * j + mat);
        }
    int Tmax = 1;
    for (int i : wv.all) Tmax = std::max(Tmax, f.mats[i].b / TILE);
    const long long per = 2LL * Tmax + 6;
    const int ng = std::max(1, std::min(h->ngroup_factor, (int)wv.all.size()));
    std::vector<std::map<long long, std::vector<InvTask>>> keys(ng);
    for (size_t c = 0; c < wv.all.size(); ++c) {
      auto& fk = keys[c % ng];
      const int mi = wv.all[c];
      const InvMat& m = f.mats[mi];
      const int T = m.b / TILE, nbk = (m.n / 3 + NBLK - 1) / NBLK;
      auto schur = [&](long long key, int l, int dk) {
        for (int i = 0; i < nbk; ++i)
          for (int j = 0; j * TILE < m.n; ++j) fk[key].push_back({IV_SCHUR_A, mi, l, dk, i, j});
      };
      auto schur_add = [&](long long key, int l, int dk) {
        for (int i = 0; i < nbk; ++i)
          for (int j = 0; j * TILE <= 3 * (i * NBLK + NBLK - 1) + 2 && j * TILE < m.n; ++j)
            fk[key].push_back({IV_SCHUR_B, mi, l, dk, i, j});
      };
      auto sweep = [&](long long key, int l) {
        fk[key].push_back({IV_PIVOT, mi, l, 0, 0, 0});
        for (int k = 0; k < T; ++k) {
          for (int i = 0; i < T; ++i) fk[key + 1 + 2 * k].push_back({IV_PANEL, mi, l, k, i, 0});
          auto& up = fk[key + 2 + 2 * k];
          if (k + 1 < T) up.push_back({IV_UPDATE, mi, l, k, k + 1, k + 1});   // swept next: first
          for (int i = 0; i < T; ++i)
            for (int j = 0; j <= i; ++j)
              if (i != k && j != k && !(i == k + 1 && j == k + 1)) up.push_back({IV_UPDATE, mi, l, k, i, j});
        }
      };
      int tmid = 0;
      for (int half = 0; half < 2; ++half) {
        const int nch = half ? m.nL - 1 - m.mid : m.mid;
        tmid = std::max(tmid, nch);
        for (int t = 0; t < nch; ++t) {
          const int l = half ? m.nL - 1 - t : t, dk = half ? 1 : -1;
          if (t > 0) {
            schur(t * per, l, dk);
            schur_add(t * per + 1, l, dk);
          }
          sweep(t * per + 3, l);
        }
      }
      for (int dk : {-1, 1}) {
        if (m.mid + dk < 0 || m.mid + dk >= m.nL) continue;
        schur(tmid * per, m.mid, dk);
        schur_add(tmid * per + (dk < 0 ? 1 : 2), m.mid, dk);
      }
      sweep(tmid * per + 3, m.mid);
    }
    std::vector<InvTask> tasks;
    wv.steps.assign(ng, {});
    for (int g = 0; g < ng; ++g)
      for (auto& kv : keys[g]) {
        if (kv.second.empty()) continue;
        // tasks that sweep a pivot tile first: they are the longest
        std::stable_partition(kv.second.begin(), kv.second.end(), [](const InvTask& t) {
          return t.type == IV_PIVOT || (t.type == IV_UPDATE && t.i == t.j && t.i == t.k + 1);
        });
        wv.steps[g].push_back({(int)tasks.size(), (int)kv.second.size()});
        tasks.insert(tasks.end(), kv.second.begin(), kv.second.end());
      }
    TRY(dev_alloc_bytes(h, &p, std::max<size_t>(tasks.size(), 1) * sizeof(InvTask)));
    wv.d_tasks = static_cast<InvTask*>(p);
    CK(cudaMemcpy(wv.d_tasks, tasks.data(), tasks.size() * sizeof(InvTask), cudaMemcpyHostToDevice));
    for (InvForm::Solve& s : wv.solve) {
      if (s.list.empty()) continue;
      std::stable_sort(s.list.begin(), s.list.end(), [&](int x, int y) {
        return (double)f.mats[x].n * f.mats[x].n * f.mats[x].nL > (double)f.mats[y].n * f.mats[y].n * f.mats[y].nL;
      });
      choose_solve(h, f, s);
      if (s.rows32)
        for (int i : s.list) f.mats[i].sg = s.G;
      TRY(dev_alloc_bytes(h, &p, s.list.size() * sizeof(int)));
      s.d_list = static_cast<int*>(p);
      CK(cudaMemcpy(s.d_list, s.list.data(), s.list.size() * sizeof(int), cudaMemcpyHostToDevice));
    }
  }
  CK(cudaMemcpy(f.d_mats, f.mats.data(), f.mats.size() * sizeof(InvMat), cudaMemcpyHostToDevice));   // with sg
  return MSGFEM_OK;
}

// Launches of the factorisation of wave w on st (stream groups of h->gs).
template <typename T>
static void inv_factor_t(msgfem* h, int w, cudaStream_t st) {
  const InvForm& f = *h->inv;
  const InvForm::Wave& wv = f.waves[w];
  const int ng = (int)wv.steps.size();
  const bool multi = ng > 1;
  if (multi) {
    cudaEventRecord(h->gs.fork, st);
    for (int g = 0; g < ng; ++g) cudaStreamWaitEvent(h->gs.s[g], h->gs.fork, 0);
  }
  size_t maxlen = 0;
  for (const auto& v : wv.steps) maxlen = std::max(maxlen, v.size());
  for (size_t k = 0; k < maxlen; ++k)
    for (int g = 0; g < ng; ++g) {
      if (k >= wv.steps[g].size()) continue;
      const SchedStep& s = wv.steps[g][k];
      k_inv_step<T><<<s.count, 256, inv_step_smem<T>(), multi ? h->gs.s[g] : st>>>(wv.d_tasks + s.first, f.d_mats,
                                                                                h->d_flags, h->d_notspd);
      ++g_launch_count;
    }
  if (multi)
    for (int g = 0; g < ng; ++g) {
      cudaEventRecord(h->gs.join[g], h->gs.s[g]);
      cudaStreamWaitEvent(st, h->gs.join[g], 0);
    }
  // inactive subdomains (other waves) are skipped by the kernels below (the matrices, two
  // per subdomain, lie along x: the other grid dimensions end at 65,535)
  int maxl = 1;
  for (int i : wv.all) maxl = std::max(maxl, f.mats[i].nL);
  cudaMemsetAsync(f.d_cond, 0, 2 * (size_t)h->N * sizeof(int), st);
  k_inv_condition<T><<<dim3((int)f.mats.size(), maxl), 128, 0, st>>>(f.d_mats, h->d_flags, h->d_notspd, f.d_cond);
  ++g_launch_count;
  // packed couplings, over the sweep's scratch
  k_inv_pack<T><<<dim3((int)f.mats.size(), maxl), 256, 0, st>>>(f.d_mats, h->d_flags);
  ++g_launch_count;
  if (sizeof(T) == 4) {
    int kmax = 0;
    for (int i : wv.all)
      if (f.mats[i].sg > 0) kmax = std::max(kmax, (f.mats[i].n + 31) / 32);
    for (int last = 0; last < 2 && kmax > 0; ++last) {
      k_inv_pack_f32<<<dim3((int)f.mats.size(), last ? 1 : maxl, kmax), 256, 0, st>>>(f.d_mats, h->d_flags, last);
      ++g_launch_count;
    }
  }
  if (f.digits) {
    int bmax = 0, kmax = 0;
    for (int i : wv.all) {
      bmax = std::max(bmax, f.mats[i].b);
      kmax = std::max(kmax, (f.mats[i].n + 15) / 16);
    }
    k_inv_digits<<<dim3((int)f.mats.size(), maxl, kmax), 256, 16 * (bmax + 2) * 8, st>>>(f.d_mats, h->d_flags);
    ++g_launch_count;
  }
}

void inv_factor(msgfem* h, int w, cudaStream_t st) {
  if (h->mixed) inv_factor_t<float>(h, w, st);
  else inv_factor_t<double>(h, w, st);
}

msgfem_status inv_sound(msgfem* h, int w, bool* sound) {
  const InvForm& f = *h->inv;
  std::vector<float> g(2 * (size_t)h->N);
  CK(cudaMemcpyAsync(g.data(), f.d_cond, g.size() * sizeof(float), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  *sound = true;
  for (int i : f.waves[w].all) {
    const InvMat& m = f.mats[i];
    *sound = *sound && g[2 * m.sub + m.mat] <= (h->mixed ? INV_COND_F32 : m.mat == 0 ? INV_COND_K : INV_COND_A11);
  }
  return MSGFEM_OK;
}

// X = M^{-1} B for K (mat 0) or A11 (mat 1) of the current wave, the first ncols columns
// (in groups of KB) of blocks of `width`.
void inv_solve(msgfem* h, int mat, int src, int dst, int neg, int width, int add, int ncols) {
  const InvForm& f = *h->inv;
  const InvForm::Solve& s = f.waves[h->cur].solve[mat];
  if (s.list.empty()) return;
  for (int c0 = 0; c0 < std::min(width, ncols); c0 += KB) {
    InvSolveArgs a = {};
    a.mats = f.d_mats;
    a.list = s.d_list;
    a.subs = h->d_sub;
    a.active = h->d_flags;
    a.src = src;
    a.dst = dst;
    a.stride = width;
    a.coloff = c0;
    a.neg = neg;
    a.add = add;
    a.ring = s.ring;
    a.smem_z = s.smem_z;
    a.smem_u = s.smem_u;
    a.smem_c = s.smem_c;
    a.smem_r = s.smem_r;
    a.err = h->d_kerr;
    void* args[] = {&a};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * (int)s.list.size() * s.G);
    cfg.blockDim = dim3(solve_threads(f));
    cfg.dynamicSmemBytes = s.smem;
    cfg.stream = h->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = s.G;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    for (bool back : {false, true}) {
      cudaLaunchKernelExC(&cfg, solve_kernel(h, f, s, back), args);
      ++g_launch_count;
    }
  }
}

// The coarse matrix as one block: its sweep's tasks for the current NcPad, in place in
// d_AH, scratch in d_AHinv.  (The block Cholesky with its block inverse took T tile
// Cholesky steps and T inverse rows of up to T products on one CTA each: 6.6 ms at 10
// tiles, sweeps 1.1 ms.)
msgfem_status coarse_inv_build(msgfem* h) {
  InvForm& f = *h->inv;
  const int T = h->NcPad / TILE;
  dev_free_bytes(h, f.d_cmat);
  dev_free_bytes(h, f.d_ctasks);
  f.d_cmat = nullptr;
  f.d_ctasks = nullptr;
  InvMat m;
  memset(&m, 0, sizeof(m));
  m.sub = h->N;      // entry N of the flags: the coarse problem
  m.n = m.b = h->NcPad;
  m.nL = 1;
  m.D = h->d_AH;
  m.L = h->d_AHinv;
  std::vector<InvTask> tasks;
  f.csteps.clear();
  auto step = [&](size_t first) { f.csteps.push_back({(int)first, (int)(tasks.size() - first)}); };
  tasks.push_back({IV_PIVOT, 0, 0, 0, 0, 0});
  step(0);
  for (int k = 0; k < T; ++k) {
    size_t first = tasks.size();
    for (int i = 0; i < T; ++i) tasks.push_back({IV_PANEL, 0, 0, k, i, 0});
    step(first);
    first = tasks.size();
    if (k + 1 < T) tasks.push_back({IV_UPDATE, 0, 0, k, k + 1, k + 1});   // swept next: first
    for (int i = 0; i < T; ++i)
      for (int j = 0; j <= i; ++j)
        if (i != k && j != k && !(i == k + 1 && j == k + 1)) tasks.push_back({IV_UPDATE, 0, 0, k, i, j});
    if (tasks.size() > first) step(first);
  }
  void* p = nullptr;
  TRY(dev_alloc_bytes(h, &p, sizeof(InvMat)));
  f.d_cmat = static_cast<InvMat*>(p);
  TRY(dev_alloc_bytes(h, &p, tasks.size() * sizeof(InvTask)));
  f.d_ctasks = static_cast<InvTask*>(p);
  CK(cudaMemcpy(f.d_cmat, &m, sizeof(InvMat), cudaMemcpyHostToDevice));
  CK(cudaMemcpy(f.d_ctasks, tasks.data(), tasks.size() * sizeof(InvTask), cudaMemcpyHostToDevice));
  return MSGFEM_OK;
}

void coarse_inv_factor(msgfem* h) {
  const InvForm& f = *h->inv;
  for (const SchedStep& s : f.csteps) {
    k_inv_step<double><<<s.count, 256, inv_step_smem<double>(), h->stream>>>(f.d_ctasks + s.first, f.d_cmat, h->d_flags,
                                                                           h->d_notspd);
    ++g_launch_count;
  }
}

// flops of the inverse form: per layer the SPD inverse n^3 and the triple
// product 108 n^2 (executed: whole 64 x 64 tiles, both products of the triple product full width)
double inv_factor_flops(const msgfem* h, bool executed) {
  double fl = 0.0;
  for (const InvMat& m : h->inv->mats) {
    if (m.n == 0) continue;
    const double n = m.n, T = m.b / TILE, tile = 2.0 * TILE * TILE * TILE;
    if (!executed) fl += m.nL * (n * n * n + 108.0 * n * n);
    else fl += m.nL * (T * (T - 1.0 + 0.5 * T * (T - 1.0)) * tile + T * tile * 0.625 + 81.0 * n * n);
  }
  return fl;
}
