// Warm-start network: a multilayer perceptron with tanh hidden layers, its
// mean-squared-error gradient and Adam, all in FP32 on the GPU.
//
// Every layer is one tiled GEMM (32 x 32 output tile per CTA, 2 x 2 outputs per
// thread; 64 x 64 and 4 x 4 where enough of them fill the chip) with the bias, the
// tanh, the tanh derivative, the loss gradient and the bias gradient fused into it:
//   forward      Z_l = H_{l-1} W_l^T + b_l, H_l = tanh(Z_l) (linear output layer)
//   loss grad    G_L = 2 (Y - T) / (B d) in the output layer's epilogue
//   weight grad  dW_l = G_l^T H_{l-1}, db_l = column sums of G_l
//   data grad    G_{l-1} = (G_l W_l) * (1 - H_{l-1}^2)
// The products are mostly skinny: a hidden layer of 32 units is a handful of output tiles
// over an inner dimension of hundreds, so the time is latency, not arithmetic.
// Long inner dimensions are split over the CTAs of a thread-block cluster (one
// chunk of 64 each as far as 8 CTAs reach), whose partial tiles are summed in rank
// order through distributed shared memory.  128 x 672 -> 32 -> 1560 forward pass
// 55 -> 14 us, a training step at batch 64 245 -> 56 us (64 x 64 tiles, serial
// chunks of 16 before).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <vector>

#include "msgfem_warm.h"

extern long long g_launch_count;   // kernel launches issued by this library

struct msgfem_net {
  std::vector<int> sizes;
  int L = 0;                       // layers (weight matrices)
  int bmax = 0;
  long long np = 0;
  std::vector<long long> woff, boff;
  float* p = nullptr;              // parameters
  float* g = nullptr;              // gradient
  float* m = nullptr;              // Adam moments
  float* v = nullptr;
  std::vector<float*> act;         // act[l], l = 1..L-1: hidden outputs [bmax][sizes[l]]
  float* d1 = nullptr;             // back-propagated gradients [bmax][max width] (ping-pong)
  float* d2 = nullptr;
  double* part = nullptr;          // loss partial sums
  double* loss = nullptr;          // [1]
  int t = 0;                       // Adam step count
  cudaStream_t st = nullptr;
};

namespace {

enum { EPI_PLAIN = 0, EPI_BIAS_TANH = 1, EPI_BIAS = 2, EPI_DTANH = 3, EPI_MSE = 4 };

constexpr int GK = 64;    // K chunk of a rank, and of a partial sum

// C[m][n] = sum_k A(m, k) B(k, n) with A(m, k) = A[m lda + k] (or A[k lda + m]
// when AT) and B(k, n) = B[k ldb + n] (or B[n ldb + k] when BT), followed by
// the epilogue EPI.  H (EPI_DTANH: the hidden outputs, EPI_MSE: the targets) is read
// with the leading dimension of C.  EPI_PLAIN also writes the sums of A over k
// (the bias gradient) to gb; EPI_MSE stores scale (C + bias - H) and adds one
// partial sum of the squared differences per CTA to part.
// GT x GT output tiles, GT / 16 squared outputs per thread; tn tiles along n, all tiles
// along the grid's x (its other dimensions end at 65,535).
// A cluster of gridDim.z CTAs shares one output tile; rank z sums chunks
// [z, z + 1) per of the inner dimension.  Without a split a CTA of the larger tile adds
// the same chunks, in the same order (the same bits up to 8 chunks).
template <int GT, bool AT, bool BT, int EPI>
__global__ void __launch_bounds__(256)
k_gemm(int M, int N, int K, const float* __restrict__ A, int lda, const float* __restrict__ B, int ldb,
       float* __restrict__ C, int ldc, const float* __restrict__ bias, const float* __restrict__ H,
       float* __restrict__ gb, float scale, double* __restrict__ part, int tn) {
  namespace cg = cooperative_groups;
  constexpr int R = GT / 16;             // outputs per thread and dimension
  constexpr int KC = GT == 32 ? GK : 32;   // k staged at once
  constexpr int LD = GT * KC / 256;      // loads per thread and operand
  __shared__ float As[KC][GT + 1];
  __shared__ float Bs[KC][GT + 1];
  __shared__ float Cs[GT][GT + 1];   // partial tile of this rank
  __shared__ float Ss[GT];           // sums of A over its chunks (EPI_PLAIN)
  __shared__ double red[8];
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int bx = blockIdx.x % tn, m0 = blockIdx.x / tn * GT, n0 = bx * GT;
  const int nch = (K + GK - 1) / GK, per = (nch + gridDim.z - 1) / gridDim.z;
  const int c0 = blockIdx.z * per, c1 = min(c0 + per, nch);
  float acc[R][R] = {}, sum[R][R] = {};
  float asum = 0.f, atot = 0.f;
  auto stage = [&](int k0) {   // KC of k
    float ra[LD], rb[LD];
#pragma unroll
    for (int i = 0; i < LD; ++i) {   // every load in flight at once
      const int e = tid + 256 * i;
      const int am = AT ? e % GT : e / KC, ak = AT ? e / GT : e % KC;
      const int bn = BT ? e / KC : e % GT, bk = BT ? e % KC : e / GT;
      ra[i] = (m0 + am < M && k0 + ak < K)
                  ? (AT ? A[(size_t)(k0 + ak) * lda + m0 + am] : A[(size_t)(m0 + am) * lda + k0 + ak]) : 0.f;
      rb[i] = (n0 + bn < N && k0 + bk < K)
                  ? (BT ? B[(size_t)(n0 + bn) * ldb + k0 + bk] : B[(size_t)(k0 + bk) * ldb + n0 + bn]) : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < LD; ++i) {
      const int e = tid + 256 * i;
      if (AT) As[e / GT][e % GT] = ra[i]; else As[e % KC][e / KC] = ra[i];
      if (BT) Bs[e % KC][e / KC] = rb[i]; else Bs[e / GT][e % GT] = rb[i];
    }
    __syncthreads();
#pragma unroll 16
    for (int kk = 0; kk < KC; ++kk) {
      float a[R], b[R];
#pragma unroll
      for (int i = 0; i < R; ++i) {
        a[i] = As[kk][ty + 16 * i];
        b[i] = Bs[kk][tx + 16 * i];
      }
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (EPI == EPI_PLAIN && tid < GT)
      for (int kk = 0; kk < KC; ++kk) asum += As[kk][tid];
  };
  for (int c = c0; c < c1; ++c) {
    if constexpr (GT == 32) {
      stage(c * GK);
    } else {   // one CTA adds a long inner dimension: partial sums of GK terms
      for (int k0 = c * GK; k0 < min(c * GK + GK, K); k0 += KC) stage(k0);
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < R; ++j) {
          sum[i][j] += acc[i][j];
          acc[i][j] = 0.f;
        }
      atot += asum;
      asum = 0.f;
    }
  }
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int j = 0; j < R; ++j) Cs[ty + 16 * i][tx + 16 * j] = GT == 32 ? acc[i][j] : sum[i][j];
  if (EPI == EPI_PLAIN && tid < GT) Ss[tid] = GT == 32 ? asum : atot;
  // rank z finishes rows z, z + nr, ... of the tile
  cg::cluster_group cl = cg::this_cluster();
  const int nr = gridDim.z, z = blockIdx.z;
  if (nr > 1) cl.sync();
  else __syncthreads();
  double sq = 0.0;
  for (int e = tid; e < GT * GT; e += 256) {
    const int r = e / GT, cc = e % GT, gm = m0 + r, gn = n0 + cc;
    if (r % nr != z || gm >= M || gn >= N) continue;
    float v = 0.f;
    if (nr > 1) {
      for (int q = 0; q < nr; ++q) v += *cl.map_shared_rank(&Cs[r][cc], q);
    } else {
      v = Cs[r][cc];
    }
    if (EPI == EPI_BIAS_TANH) v = tanhf(v + bias[gn]);
    if (EPI == EPI_BIAS) v += bias[gn];
    if (EPI == EPI_DTANH) {
      const float h = H[(size_t)gm * ldc + gn];
      v *= 1.f - h * h;
    }
    if (EPI == EPI_MSE) {
      const float d = v + bias[gn] - H[(size_t)gm * ldc + gn];
      sq += (double)d * (double)d;
      v = scale * d;
    }
    C[(size_t)gm * ldc + gn] = v;
  }
  if (EPI == EPI_PLAIN && bx == 0 && z == 0 && tid < GT && m0 + tid < M) {
    float v = 0.f;
    for (int q = 0; q < nr; ++q) v += nr > 1 ? *cl.map_shared_rank(&Ss[tid], q) : Ss[tid];
    gb[m0 + tid] = v;
  }
  if (EPI == EPI_MSE) {
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if ((tid & 31) == 0) red[tid >> 5] = sq;
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < 8; ++w) t += red[w];
      part[(size_t)blockIdx.x * nr + z] = t;
    }
  }
  if (nr > 1) cl.sync();   // the partial tiles stay alive until every rank has read them
}

// loss = sum of the partials / n (fixed order: deterministic)
__global__ void k_loss_final(const double* __restrict__ part, int np, long long n, double* __restrict__ loss) {
  __shared__ double red[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < np; i += blockDim.x) s += part[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) loss[0] = red[0] / (double)n;
}

// Adam (Kingma and Ba 2015, Algorithm 1); c1 = 1 / (1 - beta1^t), c2 = 1 / (1 - beta2^t)
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, long long n, float lr, float b1, float b2, float eps, float c1,
                       float c2) {
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x) {
    const float ge = g[e];
    const float me = b1 * m[e] + (1.f - b1) * ge;
    const float ve = b2 * v[e] + (1.f - b2) * ge * ge;
    m[e] = me;
    v[e] = ve;
    p[e] -= lr * (me * c1) / (sqrtf(ve * c2) + eps);
  }
}

// Output tile, and CTAs that split the inner dimension, of an M x N x K product
struct GemmShape {
  int tile, split;
  long long tiles(int M, int N) const { return (long long)((M + tile - 1) / tile) * ((N + tile - 1) / tile); }
};

// 32 x 32 tiles, one chunk of the inner dimension per CTA of a cluster as far as 8 reach;
// from 128 tiles of 64 x 64 on those, without a split: four outputs per shared read instead
// of one, and the chip is full without it.  One layer's forward pass, us, 32 / 64: 128
// tiles with K = 512, 1,024, 4,096: 45 / 31, 78 / 56, 283 / 203; 256 with 64, 512, 1,024:
// 14.6 / 12.6, 82 / 51, 148 / 95; 512 with 4,096: 1,091 / 731; but 64 with 512: 27 / 31, 16
// with 1,024: 19 / 56.  Not where the larger tiles are half empty (65,536 x 32: 22.9 / 23.8).
GemmShape gemm_shape(int M, int N, int K) {
  const GemmShape small = {32, std::min(8, (K + GK - 1) / GK)}, large = {64, 1};
  return large.tiles(M, N) >= 128 && small.tiles(M, N) >= 3 * large.tiles(M, N) ? large : small;
}

template <int GT, bool AT, bool BT, int EPI>
void gemm_tile(cudaStream_t st, int split, int M, int N, int K, const float* A, int lda, const float* B, int ldb, float* C,
               int ldc, const float* bias, const float* H, float* gb, float scale, double* part) {
  const int tn = (N + GT - 1) / GT, tm = (M + GT - 1) / GT;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(tn * tm, 1, split);
  cfg.blockDim = dim3(256);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = split;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_gemm<GT, AT, BT, EPI>, M, N, K, A, lda, B, ldb, C, ldc, bias, H, gb, scale, part, tn);
  ++g_launch_count;
}

template <bool AT, bool BT, int EPI>
void gemm(cudaStream_t st, int M, int N, int K, const float* A, int lda, const float* B, int ldb, float* C, int ldc,
          const float* bias = nullptr, const float* H = nullptr, float* gb = nullptr, float scale = 0.f,
          double* part = nullptr) {
  const GemmShape g = gemm_shape(M, N, K);
  auto run = g.tile == 32 ? gemm_tile<32, AT, BT, EPI> : gemm_tile<64, AT, BT, EPI>;
  run(st, g.split, M, N, K, A, lda, B, ldb, C, ldc, bias, H, gb, scale, part);
}

// forward pass up to layer `layers`; the last layer's output goes to Y
void forward(msgfem_net* n, const float* X, int B, float* Y, int layers) {
  const float* h = X;
  for (int l = 0; l < layers; ++l) {
    const int in = n->sizes[l], out = n->sizes[l + 1];
    const float* W = n->p + n->woff[l];
    const float* b = n->p + n->boff[l];
    const bool last = l + 1 == n->L;
    float* o = last ? Y : n->act[l + 1];
    if (last) gemm<false, true, EPI_BIAS>(n->st, B, out, in, h, in, W, in, o, out, b);
    else gemm<false, true, EPI_BIAS_TANH>(n->st, B, out, in, h, in, W, in, o, out, b);
    h = o;
  }
}

// forward + backward into n->g; with want_loss the loss into n->loss[0]
void gradient(msgfem_net* n, const float* X, const float* T, int B, bool want_loss) {
  forward(n, X, B, nullptr, n->L - 1);
  const int dout = n->sizes[n->L], din = n->sizes[n->L - 1];
  const long long cnt = (long long)B * dout;
  const float* hl = n->L > 1 ? n->act[n->L - 1] : X;
  gemm<false, true, EPI_MSE>(n->st, B, dout, din, hl, din, n->p + n->woff[n->L - 1], din, n->d1, dout,
                             n->p + n->boff[n->L - 1], T, nullptr, 2.f / (float)cnt, n->part);
  if (want_loss) {
    const GemmShape g = gemm_shape(B, dout, din);
    const int np = (int)(g.tiles(B, dout) * g.split);
    k_loss_final<<<1, 256, 0, n->st>>>(n->part, np, cnt, n->loss);
    ++g_launch_count;
  }
  float* G = n->d1;
  float* Gn = n->d2;
  for (int l = n->L - 1; l >= 0; --l) {
    const int in = n->sizes[l], out = n->sizes[l + 1];
    const float* hin = l == 0 ? X : n->act[l];
    gemm<true, false, EPI_PLAIN>(n->st, out, in, B, G, out, hin, in, n->g + n->woff[l], in, nullptr, nullptr,
                                 n->g + n->boff[l]);
    if (l > 0) {
      gemm<false, false, EPI_DTANH>(n->st, B, in, out, G, out, n->p + n->woff[l], in, Gn, in, nullptr, n->act[l]);
      float* tmp = G;
      G = Gn;
      Gn = tmp;
    }
  }
}

bool ok(cudaError_t e) { return e == cudaSuccess; }

}  // namespace

extern "C" {

msgfem_status msgfem_net_create(int n_sizes, const int* sizes, int max_batch, const float* init_params, void* stream,
                                msgfem_net_h* out) {
  if (!out) return MSGFEM_EINVAL;
  *out = nullptr;
  if (n_sizes < 2 || !sizes || max_batch < 1) return MSGFEM_EINVAL;
  for (int i = 0; i < n_sizes; ++i)
    if (sizes[i] < 1) return MSGFEM_EINVAL;
  msgfem_net* n = new msgfem_net();
  n->sizes.assign(sizes, sizes + n_sizes);
  n->L = n_sizes - 1;
  n->bmax = max_batch;
  n->st = static_cast<cudaStream_t>(stream);
  long long off = 0;
  int wmax = 0;
  for (int l = 0; l < n->L; ++l) {
    n->woff.push_back(off);
    off += (long long)sizes[l + 1] * sizes[l];
    n->boff.push_back(off);
    off += sizes[l + 1];
  }
  for (int i = 0; i < n_sizes; ++i) wmax = sizes[i] > wmax ? sizes[i] : wmax;
  n->np = off;
  // partial sums of the loss: one per output-layer CTA, the most that a batch up to the
  // largest has (the smaller tiles and their split)
  const GemmShape small = {32, std::min(8, (sizes[n->L - 1] + GK - 1) / GK)};
  const size_t loss_parts = (size_t)small.tiles(max_batch, sizes[n->L]) * small.split;
  n->act.assign(n->L, nullptr);
  bool good = ok(cudaMalloc(&n->p, off * sizeof(float))) && ok(cudaMalloc(&n->g, off * sizeof(float))) &&
              ok(cudaMalloc(&n->m, off * sizeof(float))) && ok(cudaMalloc(&n->v, off * sizeof(float))) &&
              ok(cudaMalloc(&n->d1, (size_t)max_batch * wmax * sizeof(float))) &&
              ok(cudaMalloc(&n->d2, (size_t)max_batch * wmax * sizeof(float))) &&
              ok(cudaMalloc(&n->part, loss_parts * sizeof(double))) && ok(cudaMalloc(&n->loss, sizeof(double)));
  for (int l = 1; good && l < n->L; ++l) good = ok(cudaMalloc(&n->act[l], (size_t)max_batch * sizes[l] * sizeof(float)));
  if (!good) {
    msgfem_net_destroy(n);
    return MSGFEM_ENOMEM;
  }
  *out = n;
  if (init_params) return msgfem_net_set_params(n, init_params);
  if (!ok(cudaMemsetAsync(n->p, 0, off * sizeof(float), n->st)) || !ok(cudaMemsetAsync(n->m, 0, off * sizeof(float), n->st)) ||
      !ok(cudaMemsetAsync(n->v, 0, off * sizeof(float), n->st)))
    return MSGFEM_ECUDA;
  return MSGFEM_OK;
}

long long msgfem_net_param_count(msgfem_net_h n) { return n ? n->np : 0; }

msgfem_status msgfem_net_get_params(msgfem_net_h n, float* host_out) {
  if (!n || !host_out) return MSGFEM_EINVAL;
  if (!ok(cudaMemcpyAsync(host_out, n->p, n->np * sizeof(float), cudaMemcpyDeviceToHost, n->st)) ||
      !ok(cudaStreamSynchronize(n->st)))
    return MSGFEM_ECUDA;
  return MSGFEM_OK;
}

msgfem_status msgfem_net_set_params(msgfem_net_h n, const float* host_in) {
  if (!n || !host_in) return MSGFEM_EINVAL;
  if (!ok(cudaMemcpyAsync(n->p, host_in, n->np * sizeof(float), cudaMemcpyHostToDevice, n->st)) ||
      !ok(cudaMemsetAsync(n->m, 0, n->np * sizeof(float), n->st)) ||
      !ok(cudaMemsetAsync(n->v, 0, n->np * sizeof(float), n->st)) || !ok(cudaStreamSynchronize(n->st)))
    return MSGFEM_ECUDA;
  n->t = 0;
  return MSGFEM_OK;
}

msgfem_status msgfem_net_forward(msgfem_net_h n, const float* X, int batch, float* Y) {
  if (!n || !X || !Y || batch < 1 || batch > n->bmax) return MSGFEM_EINVAL;
  forward(n, X, batch, Y, n->L);
  return ok(cudaGetLastError()) ? MSGFEM_OK : MSGFEM_ECUDA;
}

msgfem_status msgfem_net_gradient(msgfem_net_h n, const float* X, const float* T, int batch, float* grad_out,
                                  double* loss_out) {
  if (!n || !X || !T || batch < 1 || batch > n->bmax) return MSGFEM_EINVAL;
  gradient(n, X, T, batch, loss_out != nullptr);
  if (!ok(cudaGetLastError())) return MSGFEM_ECUDA;
  if (grad_out && !ok(cudaMemcpyAsync(grad_out, n->g, n->np * sizeof(float), cudaMemcpyDeviceToHost, n->st)))
    return MSGFEM_ECUDA;
  if (loss_out && !ok(cudaMemcpyAsync(loss_out, n->loss, sizeof(double), cudaMemcpyDeviceToHost, n->st)))
    return MSGFEM_ECUDA;
  if ((grad_out || loss_out) && !ok(cudaStreamSynchronize(n->st))) return MSGFEM_ECUDA;
  return MSGFEM_OK;
}

msgfem_status msgfem_net_adam_step(msgfem_net_h n, const float* X, const float* T, int batch, float lr, float beta1,
                                   float beta2, float eps, double* loss_out) {
  if (!n || !X || !T || batch < 1 || batch > n->bmax) return MSGFEM_EINVAL;
  if (!(beta1 >= 0.f && beta1 < 1.f && beta2 >= 0.f && beta2 < 1.f && eps > 0.f)) return MSGFEM_EINVAL;
  gradient(n, X, T, batch, loss_out != nullptr);
  n->t += 1;
  double p1 = 1.0, p2 = 1.0;
  for (int i = 0; i < n->t; ++i) { p1 *= beta1; p2 *= beta2; }
  const float c1 = (float)(1.0 / (1.0 - p1)), c2 = (float)(1.0 / (1.0 - p2));
  k_adam<<<304, 256, 0, n->st>>>(n->p, n->g, n->m, n->v, n->np, lr, beta1, beta2, eps, c1, c2);
  ++g_launch_count;
  if (!ok(cudaGetLastError())) return MSGFEM_ECUDA;
  if (loss_out) {
    if (!ok(cudaMemcpyAsync(loss_out, n->loss, sizeof(double), cudaMemcpyDeviceToHost, n->st)) ||
        !ok(cudaStreamSynchronize(n->st)))
      return MSGFEM_ECUDA;
  }
  return MSGFEM_OK;
}

void msgfem_net_destroy(msgfem_net_h n) {
  if (!n) return;
  for (float* q : {n->p, n->g, n->m, n->v, n->d1, n->d2}) if (q) cudaFree(q);
  for (size_t l = 1; l < n->act.size(); ++l) if (n->act[l]) cudaFree(n->act[l]);
  if (n->part) cudaFree(n->part);
  if (n->loss) cudaFree(n->loss);
  delete n;
}

}  // extern "C"
