// Learned pair screener (rows a5 and a5' of the hot path; not in the paper, asked for by the
// benchmark configuration): a 3-layer MLP, width H, predicting log10|X_ab| from the two
// quasiparticle momentum sets, trained on exact elements of the Pfaffian path by the kernels of
// this file, and used to skip the Pfaffians of pairs predicted negligible.
//
// Features (D = 2Q + 4, Q = 8): k/pi of the NS state's modes (ascending, zero padded), k/pi of
// the R state's modes, M_a/Q, M_b/Q, 24/L, 1.  Target: log10|X| + (M_a + M_b)/2 log10(L/24),
// clipped at -30 (the 1/sqrt(L) normalisation of each quasiparticle taken out).
// Network: h1 = relu(W1 x + b1), h2 = relu(W2 h1 + b2), y = w3 . h2 + b3, MSE loss, Adam.
// Parameters (FP32) are stored flat as W1 [H][D], b1, W2 [H][H], b2, w3, b3.
//
// Training runs in FP32 on the CUDA cores (tiled SGEMM below).  Inference factors layer 1 into
// per-state partials, h1(a, b) = relu(A_a + B_b) with A_a = W1[:, NS part] x_a and
// B_b = W1[:, R part] x_b + b1, and runs layer 2 on the tensor cores (tcgen05 MMAs, BF16
// inputs, FP32 accumulation in tensor memory; screen_tc.cu), fused with the ReLU, the dot with
// w3, the threshold and the compaction of the kept pairs into per-size work lists.
#include <cuda_bf16.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <numeric>
#include <string>
#include <vector>

#include "tgba_internal.h"

namespace tgba {

constexpr int kQ = 8;
constexpr int kD = 2 * kQ + 4;

struct Screen {
  int H = 256;
  int64_t P = 0;
  float* theta = nullptr;   // parameters
  float* m = nullptr;       // Adam moments
  float* v = nullptr;
  __nv_bfloat16* W2b = nullptr;   // W2 in BF16 for inference, [H][H] row-major (output, input)
  bool w2b_valid = false;
  double margin = 1.0, val_rmse = 0, train_rmse = 0;
  int64_t adam_step = 0;
  int device = 0;
};

namespace {

// ----------------------------------------------------------------------------- SGEMM (FP32)
// C[M][N] = op(A) op(B), all row-major, on 64 x 64 tiles of 256 threads (4 x 4 each), K in steps of 16,
// the next step's global loads in flight during the current step's arithmetic.  op(A) is A [M][K] or,
// if TA, A^T with A stored [K][M]; op(B) is B [K][N] or, if TB, B^T with B stored [N][K].
// EPI: 0 plain; 1 C = max(C + bias[col], 0); 2 C = mask[row][col] > 0 ? C : 0 (the ReLU's derivative).
// SPLIT: K is cut into gridDim.z ranges of kz (a multiple of 16), range z's partial product at C + z M N: the
// weight gradients have M = N = 256 and K = the batch, 16 tiles for 152 SMs (the batch of 4096: 1.40 ms
// unsplit, of 1.48 ms for the whole gradient); sum_parts adds the ranges in order.
template <bool TA, bool TB, int EPI, bool SPLIT>
__global__ void __launch_bounds__(256) sgemm(int M, int N, int K, const float* __restrict__ A,
                                             const float* __restrict__ B, float* __restrict__ C,
                                             const float* __restrict__ aux, int kz) {
  __shared__ __align__(16) float As[2][16][68];
  __shared__ __align__(16) float Bs[2][16][68];
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  const int row0 = blockIdx.y * 64, col0 = blockIdx.x * 64;
  const int k_lo = SPLIT ? blockIdx.z * kz : 0, k_hi = SPLIT ? min(K, k_lo + kz) : K;
  float ra[4], rb[4];
  // a thread's four elements of a 16 x 64 operand step: consecutive threads along the contiguous index
  auto fetch = [&](int k0) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int q = threadIdx.x + 256 * e;
      const int ka = TA ? q / 64 : q % 16, ma = TA ? q % 64 : q / 16;
      const int kb = TB ? q % 16 : q / 64, nb = TB ? q / 16 : q % 64;
      const int r = row0 + ma, c = col0 + nb;
      ra[e] = (r < M && k0 + ka < k_hi) ? (TA ? A[(size_t)(k0 + ka) * M + r] : A[(size_t)r * K + k0 + ka]) : 0.f;
      rb[e] = (c < N && k0 + kb < k_hi) ? (TB ? B[(size_t)c * K + k0 + kb] : B[(size_t)(k0 + kb) * N + c]) : 0.f;
    }
  };
  auto stash = [&](int s) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int q = threadIdx.x + 256 * e;
      As[s][TA ? q / 64 : q % 16][TA ? q % 64 : q / 16] = ra[e];
      Bs[s][TB ? q % 16 : q / 64][TB ? q / 16 : q % 64] = rb[e];
    }
  };
  float acc[4][4] = {};
  fetch(k_lo);
  stash(0);
  __syncthreads();
  int s = 0;
  for (int k0 = k_lo; k0 < k_hi; k0 += 16, s ^= 1) {
    const bool more = k0 + 16 < k_hi;
    if (more) fetch(k0 + 16);
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      const float4 a4 = *(const float4*)&As[s][kk][ty * 4], b4 = *(const float4*)&Bs[s][kk][tx * 4];
      const float a[4] = {a4.x, a4.y, a4.z, a4.w}, b[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (more) stash(s ^ 1);
    __syncthreads();
  }
  float* out = SPLIT ? C + (size_t)blockIdx.z * M * N : C;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = row0 + ty * 4 + i, c = col0 + tx * 4 + j;
      if (r < M && c < N) {
        float v = acc[i][j];
        if (EPI == 1) v = fmaxf(v + aux[c], 0.f);
        if (EPI == 2) v = aux[(size_t)r * N + c] > 0.f ? v : 0.f;
        out[(size_t)r * N + c] = v;
      }
    }
}

template <bool TA, bool TB, int EPI>
void gemm(cudaStream_t st, int M, int N, int K, const float* A, const float* B, float* C, const float* aux) {
  dim3 grid((N + 63) / 64, (M + 63) / 64);
  sgemm<TA, TB, EPI, false><<<grid, 256, 0, st>>>(M, N, K, A, B, C, aux, 0);
}

// ranges of the split products and of the column sums for a batch: about 128 rows each, at most 32
int batch_parts(int64_t rows) { return (int)std::max<int64_t>(1, std::min<int64_t>(32, (rows + 127) / 128)); }

// C[M][N] = A^T B over `rows` rows (A [rows][M], B [rows][N]), the parts in `part` and then summed
__global__ void sum_parts(int64_t n, int parts, const float* __restrict__ part, float* __restrict__ out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float acc = 0.f;
    for (int z = 0; z < parts; ++z) acc += part[(size_t)z * n + i];
    out[i] = acc;
  }
}
void gemm_tn_split(cudaStream_t st, int M, int N, int64_t rows, const float* A, const float* B, float* C, float* part) {
  const int parts = batch_parts(rows), kz = (int)(((rows + parts - 1) / parts + 15) / 16 * 16);
  const int used = (int)((rows + kz - 1) / kz);
  dim3 grid((N + 63) / 64, (M + 63) / 64, used);
  sgemm<true, false, 0, true><<<grid, 256, 0, st>>>(M, N, (int)rows, A, B, part, nullptr, kz);
  sum_parts<<<(M * N + 255) / 256, 256, 0, st>>>((int64_t)M * N, used, part, C);
}

// y = H2 w3 + b3, r = y - t (per row), warp per row
__global__ void out_layer(int64_t rows, int H, const float* __restrict__ H2, const float* __restrict__ w3,
                          const float* __restrict__ b3, const float* __restrict__ t, float* __restrict__ y,
                          float* __restrict__ r) {
  const int lane = threadIdx.x & 31;
  for (int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < rows;
       row += ((int64_t)gridDim.x * blockDim.x) >> 5) {
    float acc = 0.f;
    for (int j = lane; j < H; j += 32) acc = fmaf(H2[row * H + j], w3[j], acc);
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) {
      const float yy = acc + b3[0];
      y[row] = yy;
      if (t) r[row] = yy - t[row];
    }
  }
}

// Per range of `per` rows (blockIdx.x) and column j: dZ2 = (dy w3^T) * (H2 > 0) with dy = scale r, and the
// range's sums for dw3 = H2^T dy, db2 = column sums of dZ2, db3 = sum dy: part [range][2 H + 1].
// One pass over H2 by all SMs (a thread per column over the whole batch took 0.37 ms and, for the two
// bias gradients, 0.47 ms).
__global__ void __launch_bounds__(256) back_out(int64_t rows, int per, const float* __restrict__ r,
                                                const float* __restrict__ w3, const float* __restrict__ H2, float scale,
                                                float* __restrict__ dZ2, float* __restrict__ part) {
  const int H = 256, j = threadIdx.x;
  const int64_t i0 = (int64_t)blockIdx.x * per, i1 = min(rows, i0 + per);
  const float w = w3[j];
  float gw = 0.f, gb = 0.f, gr = 0.f;
#pragma unroll 4
  for (int64_t i = i0; i < i1; ++i) {
    const float h = H2[i * H + j], dy = scale * r[i], d = h > 0.f ? dy * w : 0.f;
    dZ2[i * H + j] = d;
    gw = fmaf(h, dy, gw);
    gb += d;
    gr += dy;
  }
  float* p = part + (size_t)blockIdx.x * (2 * H + 1);
  p[j] = gw;
  p[H + j] = gb;
  if (j == 0) p[2 * H] = gr;
}

// the ranges' sums of back_out, in order
__global__ void back_out_sum(int parts, const float* __restrict__ part, float* __restrict__ dw3, float* __restrict__ db2,
                             float* __restrict__ db3) {
  const int H = 256, j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j > 2 * H) return;
  float acc = 0.f;
  for (int z = 0; z < parts; ++z) acc += part[(size_t)z * (2 * H + 1) + j];
  if (j < H) dw3[j] = acc;
  else if (j < 2 * H) db2[j - H] = acc;
  else db3[0] = acc;
}

// column sums of a rows x 256 matrix over ranges of `per` rows (blockIdx.x): part [range][256]
__global__ void __launch_bounds__(256) col_sum(int64_t rows, int per, const float* __restrict__ Mx, float* __restrict__ part) {
  const int j = threadIdx.x;
  const int64_t i0 = (int64_t)blockIdx.x * per, i1 = min(rows, i0 + per);
  float acc = 0.f;
#pragma unroll 8
  for (int64_t i = i0; i < i1; ++i) acc += Mx[i * 256 + j];
  part[(size_t)blockIdx.x * 256 + j] = acc;
}

__global__ void sum_squares(int64_t n, const float* __restrict__ r, double* __restrict__ out) {
  double acc = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    acc += (double)r[i] * r[i];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(out, acc);
}

__global__ void adam_kernel(int64_t n, float* __restrict__ th, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, float lr, float b1, float b2, float c1, float c2, float eps) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    th[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// features of explicit pairs of one sector (see the file header)
__global__ void pair_features(int64_t n, const int32_t* __restrict__ pairs, int64_t ns_off, int64_t r_off,
                              const int16_t* __restrict__ modes_ns, const int16_t* __restrict__ modes_r,
                              const uint8_t* __restrict__ M_ns, const uint8_t* __restrict__ M_r, int max_qp,
                              const int* __restrict__ nlab, int L, float* __restrict__ x) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    const int64_t a = ns_off + pairs[2 * q], b = r_off + pairs[2 * q + 1];
    float* xr = x + q * kD;
    for (int i = 0; i < kD; ++i) xr[i] = 0.f;
    const int ma = M_ns[a], mb = M_r[b];
    for (int i = 0; i < ma && i < kQ; ++i) xr[i] = (float)nlab[modes_ns[a * max_qp + i]] / L;
    for (int i = 0; i < mb && i < kQ; ++i) xr[kQ + i] = (float)nlab[L + modes_r[b * max_qp + i]] / L;
    xr[2 * kQ] = (float)ma / kQ;
    xr[2 * kQ + 1] = (float)mb / kQ;
    xr[2 * kQ + 2] = 24.f / L;
    xr[2 * kQ + 3] = 1.f;
  }
}

// training targets from exact X (complex, interleaved)
__global__ void pair_targets(int64_t n, const int32_t* __restrict__ pairs, int64_t ns_off, int64_t r_off,
                             const uint8_t* __restrict__ M_ns, const uint8_t* __restrict__ M_r,
                             const double* __restrict__ X, double log_l_ratio, float* __restrict__ t) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    const double ax = hypot(X[2 * q], X[2 * q + 1]);
    const int nq = M_ns[ns_off + pairs[2 * q]] + M_r[r_off + pairs[2 * q + 1]];
    double y = ax > 0 ? log10(ax) : -30.0;
    y = fmax(y + 0.5 * nq * log_l_ratio, -30.0);
    t[q] = (float)y;
  }
}

__global__ void gather_rows(int64_t n, int D, const int64_t* __restrict__ idx, const float* __restrict__ x,
                            const float* __restrict__ t, float* __restrict__ xb, float* __restrict__ tb) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n * D; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / D;
    const int c = (int)(i - r * D);
    xb[i] = x[idx[r] * D + c];
    if (c == 0) tb[r] = t[idx[r]];
  }
}

__global__ void to_bf16(int64_t n, const float* __restrict__ a, __nv_bfloat16* __restrict__ b) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    b[i] = __float2bfloat16_rn(a[i]);
}

// ----------------------------------------------------------------------------- inference
// Per-state layer-1 partials.  NS: A_a = W1[:, 0:Q] x_a + W1[:, 2Q] M_a/Q.
// R: B_b = W1[:, Q:2Q] x_b + W1[:, 2Q+1] M_b/Q + W1[:, 2Q+2] 24/L + W1[:, 2Q+3] + b1.
__global__ void state_partials(int64_t n_states, bool ns, const int16_t* __restrict__ modes,
                               const uint8_t* __restrict__ Mq, int max_qp, const int* __restrict__ nlab, int L, int H,
                               const float* __restrict__ W1, const float* __restrict__ b1, float* __restrict__ out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n_states * H; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = i / H;
    const int o = (int)(i - s * H);
    const int M = Mq[s];
    const float* w = W1 + (size_t)o * kD;
    float acc;
    if (ns) {
      acc = w[2 * kQ] * ((float)M / kQ);
      for (int q = 0; q < M && q < kQ; ++q) acc = fmaf(w[q], (float)nlab[modes[s * max_qp + q]] / L, acc);
    } else {
      acc = b1[o] + w[2 * kQ + 1] * ((float)M / kQ) + w[2 * kQ + 2] * (24.f / L) + w[2 * kQ + 3];
      for (int q = 0; q < M && q < kQ; ++q) acc = fmaf(w[kQ + q], (float)nlab[L + modes[s * max_qp + q]] / L, acc);
    }
    out[i] = acc;
  }
}

int blocks(int64_t work, int t = 256) {
  return (int)std::max<int64_t>(1, std::min<int64_t>((work + t - 1) / t, 152 * 16));
}

// SplitMix64 (Steele, Lea, Flood 2014): the counter-based generator of the training sample.
uint64_t splitmix64(uint64_t x) {
  x += 0x9e3779b97f4a7c15ull;
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return x ^ (x >> 31);
}

}  // namespace

// ----------------------------------------------------------------------------- host side
tgba_status screen_create(int H, const float* params, uint64_t seed, Screen** out) {
  Screen* s = new Screen();
  s->H = H;
  s->P = (int64_t)H * kD + H + (int64_t)H * H + H + H + 1;
  cudaGetDevice(&s->device);
  std::vector<float> th(s->P, 0.f);
  if (params) {
    std::copy(params, params + s->P, th.begin());
  } else {   // He-normal weights (Box-Muller on SplitMix64 draws), zero biases
    auto normal = [&](uint64_t k) {
      const double u1 = ((splitmix64(seed * 0x100000001b3ull + 2 * k) >> 11) + 1.0) / 9007199254740993.0;
      const double u2 = (splitmix64(seed * 0x100000001b3ull + 2 * k + 1) >> 11) / 9007199254740992.0;
      return std::sqrt(-2.0 * std::log(u1)) * std::cos(2.0 * M_PI * u2);
    };
    int64_t o = 0, k = 0;
    for (int64_t i = 0; i < (int64_t)H * kD; ++i) th[o++] = (float)(normal(k++) * std::sqrt(2.0 / kD));
    o += H;
    for (int64_t i = 0; i < (int64_t)H * H; ++i) th[o++] = (float)(normal(k++) * std::sqrt(2.0 / H));
    o += H;
    for (int64_t i = 0; i < H; ++i) th[o++] = (float)(normal(k++) * std::sqrt(1.0 / H));
  }
  if (cudaMalloc(&s->theta, s->P * 4) != cudaSuccess || cudaMalloc(&s->m, s->P * 4) != cudaSuccess ||
      cudaMalloc(&s->v, s->P * 4) != cudaSuccess || cudaMalloc(&s->W2b, (size_t)H * H * 2) != cudaSuccess) {
    cudaGetLastError();
    screen_free(s);
    return fail(TGBA_ENOMEM, "screen parameters");
  }
  TGBA_CUDA(cudaMemcpy(s->theta, th.data(), s->P * 4, cudaMemcpyHostToDevice));
  TGBA_CUDA(cudaMemset(s->m, 0, s->P * 4));
  TGBA_CUDA(cudaMemset(s->v, 0, s->P * 4));
  *out = s;
  return TGBA_OK;
}

void screen_free(Screen* s) {
  if (!s) return;
  if (s->theta) cudaFree(s->theta);
  if (s->m) cudaFree(s->m);
  if (s->v) cudaFree(s->v);
  if (s->W2b) cudaFree(s->W2b);
  delete s;
}

int64_t screen_nparams(const Screen* s) { return s->P; }

// Floats of scratch that forward_backward needs for a batch of B.
static int64_t batch_work(int64_t B) {
  const int64_t H = 256, parts = 32;
  return B * (3 * H + 2) + parts * (H * H) + 256 * (2 * H + 1) + 8;
}

// Forward and backward of one batch; loss (mean squared error) into *loss, gradient into grad.
// H1 and H2 hold the rectified layers; where H is positive the ReLU passes the gradient, so the layers'
// inputs are not kept.  For a batch of 4096 (FP32): 1.48 ms with plain products, separate bias, ReLU
// and mask passes and one thread per column for the sums over the batch.
static tgba_status forward_backward(Screen& s, const float* x, const float* t, int64_t B, float* grad, float* work,
                                    double* d_loss, cudaStream_t st) {
  const int H = s.H;
  const float* W1 = s.theta;
  const float* b1 = W1 + (int64_t)H * kD;
  const float* W2 = b1 + H;
  const float* b2 = W2 + (int64_t)H * H;
  const float* w3 = b2 + H;
  const float* b3 = w3 + H;
  float* H1 = work;
  float* H2 = H1 + B * H;
  float* dZ = H2 + B * H;
  float* y = dZ + B * H;
  float* r = y + B;
  float* part = r + B;                                          // split products
  float* sums = part + (int64_t)32 * H * H;                     // ranges' column sums
  gemm<false, true, 1>(st, (int)B, H, kD, x, W1, H1, b1);       // H1 = relu(X W1^T + b1)
  gemm<false, true, 1>(st, (int)B, H, H, H1, W2, H2, b2);       // H2 = relu(H1 W2^T + b2)
  out_layer<<<blocks(B * 32), 256, 0, st>>>(B, H, H2, w3, b3, t, y, r);
  if (d_loss) {
    TGBA_CUDA(cudaMemsetAsync(d_loss, 0, sizeof(double), st));
    sum_squares<<<blocks(B), 256, 0, st>>>(B, r, d_loss);
  }
  if (grad) {
    float* dW1 = grad;
    float* db1 = dW1 + (int64_t)H * kD;
    float* dW2 = db1 + H;
    float* db2 = dW2 + (int64_t)H * H;
    float* dw3 = db2 + H;
    float* db3 = dw3 + H;
    const float scale = 2.f / (float)B;                         // d(mean r^2)/dy = 2 r / B
    const int ranges = (int)std::max<int64_t>(1, std::min<int64_t>(256, (B + 15) / 16));
    const int per = (int)((B + ranges - 1) / ranges), used = (int)((B + per - 1) / per);
    back_out<<<used, 256, 0, st>>>(B, per, r, w3, H2, scale, dZ, sums);        // dZ2, and sums of its columns
    back_out_sum<<<3, 256, 0, st>>>(used, sums, dw3, db2, db3);
    gemm_tn_split(st, H, H, B, dZ, H1, dW2, part);              // dW2 = dZ2^T H1
    float* dZ1 = H2;                                            // H2 is dead after back_out
    gemm<false, false, 2>(st, (int)B, H, H, dZ, W2, dZ1, H1);   // dZ1 = (dZ2 W2) * (H1 > 0)
    gemm_tn_split(st, H, kD, B, dZ1, x, dW1, part);             // dW1 = dZ1^T X
    col_sum<<<used, 256, 0, st>>>(B, per, dZ1, sums);
    sum_parts<<<1, 256, 0, st>>>(H, used, sums, db1);
  }
  TGBA_CUDA(cudaGetLastError());
  return TGBA_OK;
}

tgba_status screen_grad(Screen& s, const float* x, const float* t, int64_t B, float* grad, double* loss,
                        cudaStream_t st) {
  float* work = nullptr;
  double* d_loss = nullptr;
  TGBA_CUDA(cudaMallocAsync(&work, (size_t)batch_work(B) * 4, st));
  TGBA_CUDA(cudaMallocAsync(&d_loss, sizeof(double), st));
  tgba_status r = forward_backward(s, x, t, B, grad, work, d_loss, st);
  double h = 0;
  if (r == TGBA_OK) {
    cudaMemcpyAsync(&h, d_loss, sizeof(double), cudaMemcpyDeviceToHost, st);
    cudaStreamSynchronize(st);
    *loss = h / (double)B;
  }
  cudaFreeAsync(work, st);
  cudaFreeAsync(d_loss, st);
  return r;
}

tgba_status screen_params(Screen& s, float* host) {
  TGBA_CUDA(cudaMemcpy(host, s.theta, s.P * 4, cudaMemcpyDeviceToHost));
  return TGBA_OK;
}

static tgba_status refresh_bf16(Screen& s, cudaStream_t st) {
  const float* W2 = s.theta + (int64_t)s.H * kD + s.H;
  to_bf16<<<blocks((int64_t)s.H * s.H), 256, 0, st>>>((int64_t)s.H * s.H, W2, s.W2b);
  TGBA_CUDA(cudaGetLastError());
  s.w2b_valid = true;
  return TGBA_OK;
}

// Layer-1 partials of every state of the basis (all sectors): part [n_ns_total + n_r_total][H],
// NS states first.  The caller frees *part (stream-ordered).
static tgba_status state_partials_all(Screen& s, Basis& b, float** part, cudaStream_t st) {
  const int H = s.H;
  const int64_t n_ns = (int64_t)b.ns.E.size(), n_r = (int64_t)b.r.E.size();
  TGBA_CUDA(cudaMallocAsync(part, (size_t)std::max<int64_t>(1, n_ns + n_r) * H * 4, st));
  const float* W1 = s.theta;
  const float* b1 = W1 + (int64_t)H * kD;
  if (n_ns > 0)
    state_partials<<<blocks(n_ns * H), 256, 0, st>>>(n_ns, true, b.d_modes_ns, b.d_M_ns, b.max_qp, b.d_nlab, b.L, H, W1,
                                                    b1, *part);
  if (n_r > 0)
    state_partials<<<blocks(n_r * H), 256, 0, st>>>(n_r, false, b.d_modes_r, b.d_M_r, b.max_qp, b.d_nlab, b.L, H, W1,
                                                   b1, *part + n_ns * H);
  TGBA_CUDA(cudaGetLastError());
  b.launches += 2;
  return TGBA_OK;
}

// Predicted y of every pair of sector `sidx`: pred float [n_ns][n_r].  Pairs outside the
// model (a state with more than Q quasiparticles) get 0.
tgba_status screen_score(Screen& s, Basis& b, int sidx, float* pred, cudaStream_t st) {
  if (s.H != 256) return fail(TGBA_EINVAL, "inference supports width 256");
  const Sector& sec = b.sectors[sidx];
  if (sec.n_ns == 0 || sec.n_r == 0) return TGBA_OK;
  if (!s.w2b_valid) {
    tgba_status r = refresh_bf16(s, st);
    if (r != TGBA_OK) return r;
  }
  std::vector<Rect> rects;
  for (const Rect& rc : b.rects)
    if (rc.ns0 >= sec.ns_off && rc.ns0 < sec.ns_off + sec.n_ns) rects.push_back(rc);
  float* part = nullptr;
  tgba_status r = state_partials_all(s, b, &part, st);
  if (r != TGBA_OK) return r;
  const int H = s.H;
  const float* b2 = s.theta + (int64_t)H * kD + H + (int64_t)H * H;
  TGBA_CUDA(cudaMemsetAsync(pred, 0, (size_t)sec.n_ns * sec.n_r * 4, st));
  r = score_rects_tc(b, rects, part, part + (int64_t)b.ns.E.size() * H, s.W2b, b2, b2 + H, b2 + 2 * H, 0.f, 0.f,
                     pred, sec.x_off, nullptr, nullptr, nullptr, st);
  cudaFreeAsync(part, st);
  return r;
}

// The screened element stage (after the contraction table): P = 0, the pairs with n <= 14 scored and
// the kept ones compacted into per-size lists, their elements from the lists, and the larger
// sizes without screening.  *kept: pairs evaluated.
tgba_status screen_pfaffians(Screen& s, Basis& b, double tau, double hx, int64_t* kept, cudaStream_t st) {
  if (s.H != 256) return fail(TGBA_EINVAL, "inference supports width 256");
  if (!s.w2b_valid) {
    tgba_status r = refresh_bf16(s, st);
    if (r != TGBA_OK) return r;
  }
  const int H = s.H;
  constexpr int kSizes = 8;                                     // n = 0, 2, ..., 14
  std::vector<int64_t> off(kSizes + 1, 0);
  const std::vector<Rect> small(b.rects.begin() + b.big_rects, b.rects.end());
  for (const Rect& rc : small) off[rc.n / 2 + 1] += (int64_t)rc.rows * rc.w;
  for (int i = 0; i < kSizes; ++i) off[i + 1] += off[i];
  TGBA_CUDA(cudaMemsetAsync(b.d_P, 0, (size_t)std::max<int64_t>(1, b.n_elements) * sizeof(double), st));
  void* lb = nullptr;
  const size_t list_bytes = (size_t)std::max<int64_t>(1, off[kSizes]) * sizeof(PairEntry);
  TGBA_CUDA(cudaMallocAsync(&lb, list_bytes + 64 * sizeof(int64_t), st));
  PairEntry* lists = (PairEntry*)lb;
  int64_t* d_off = (int64_t*)((char*)lb + list_bytes);
  unsigned* d_cnt = (unsigned*)(d_off + 16);
  TGBA_CUDA(cudaMemcpyAsync(d_off, off.data(), kSizes * sizeof(int64_t), cudaMemcpyHostToDevice, st));
  TGBA_CUDA(cudaMemsetAsync(d_cnt, 0, kSizes * sizeof(unsigned), st));
  float* part = nullptr;
  tgba_status r = state_partials_all(s, b, &part, st);
  if (r != TGBA_OK) { cudaFreeAsync(lb, st); return r; }
  const float* b2 = s.theta + (int64_t)H * kD + H + (int64_t)H * H;
  // keep iff y - (n/2) log10(L/24) + log10(L hx) >= log10(tau) - margin
  const float half_log_l = (float)(0.5 * std::log10(b.L / 24.0));
  const float shift = (float)(std::log10(b.L * std::fabs(hx)) - std::log10(tau) + s.margin);
  r = score_rects_tc(b, small, part, part + (int64_t)b.ns.E.size() * H, s.W2b, b2, b2 + H, b2 + 2 * H, shift,
                     half_log_l, nullptr, 0, d_cnt, d_off, lists, st);
  if (r == TGBA_OK) r = run_element_lists(b, d_cnt, d_off, kSizes, lists, st);
  if (r == TGBA_OK) r = run_elements_big(b, st);
  unsigned hc[kSizes] = {};
  if (r == TGBA_OK) {
    TGBA_CUDA(cudaMemcpyAsync(hc, d_cnt, sizeof(hc), cudaMemcpyDeviceToHost, st));
  }
  cudaFreeAsync(part, st);
  cudaFreeAsync(lb, st);
  if (r != TGBA_OK) return r;
  TGBA_CUDA(cudaStreamSynchronize(st));
  int64_t k = b.n_elements - off[kSizes];                       // sizes n >= 16: all evaluated
  for (int i = 0; i < kSizes; ++i) k += hc[i];
  *kept = k;
  return TGBA_OK;
}

// Train on n_samples pairs drawn uniformly from all NS x R pairs of the given bases.
tgba_status screen_train(Basis** sets, int n_sets, int64_t n_samples, uint64_t seed, int H, int epochs, Screen** out,
                         double* stats, cudaStream_t st) {
  auto t_start = std::chrono::steady_clock::now();
  Screen* s = nullptr;
  tgba_status r = screen_create(H, nullptr, seed, &s);
  if (r != TGBA_OK) return r;
  // 1. sample: global element index -> (set, sector, a, b), grouped by (set, sector)
  std::vector<std::pair<int, int>> groups;
  std::vector<int64_t> cum;
  int64_t total = 0;
  for (int k = 0; k < n_sets; ++k)
    for (size_t q = 0; q < sets[k]->sectors.size(); ++q) {
      const Sector& sec = sets[k]->sectors[q];
      if (sec.n_ns * sec.n_r == 0) continue;
      groups.emplace_back(k, (int)q);
      cum.push_back(total);
      total += sec.n_ns * sec.n_r;
    }
  if (total == 0) { screen_free(s); return fail(TGBA_EINVAL, "training bases have no pairs"); }
  std::vector<std::vector<int32_t>> gp(groups.size());
  for (int64_t i = 0; i < n_samples; ++i) {
    const int64_t e = (int64_t)(splitmix64(seed ^ (0x5bd1e995ull * (uint64_t)(i + 1))) % (uint64_t)total);
    const size_t gi = std::upper_bound(cum.begin(), cum.end(), e) - cum.begin() - 1;
    const Sector& sec = sets[groups[gi].first]->sectors[groups[gi].second];
    const int64_t loc = e - cum[gi];
    gp[gi].push_back((int32_t)(loc / sec.n_r));
    gp[gi].push_back((int32_t)(loc % sec.n_r));
  }
  // 2. exact labels and features, group by group
  float *X = nullptr, *T = nullptr;
  TGBA_CUDA(cudaMalloc(&X, (size_t)n_samples * kD * 4));
  TGBA_CUDA(cudaMalloc(&T, (size_t)n_samples * 4));
  int64_t o = 0;
  for (size_t gi = 0; gi < groups.size(); ++gi) {
    const int64_t n = (int64_t)gp[gi].size() / 2;
    if (n == 0) continue;
    Basis& bb = *sets[groups[gi].first];
    const int sidx = groups[gi].second;
    const Sector& sec = bb.sectors[sidx];
    int32_t* dp = nullptr;
    double* dx = nullptr;
    TGBA_CUDA(cudaMalloc(&dp, n * 8));
    TGBA_CUDA(cudaMalloc(&dx, n * 16));
    TGBA_CUDA(cudaMemcpy(dp, gp[gi].data(), n * 8, cudaMemcpyHostToDevice));
    if (!bb.table_valid) {
      if ((r = build_table(bb, st)) != TGBA_OK) return r;
    }
    if ((r = run_element_pairs(bb, sidx, dp, n, dx, st)) != TGBA_OK) return r;
    pair_features<<<blocks(n), 256, 0, st>>>(n, dp, sec.ns_off, sec.r_off, bb.d_modes_ns, bb.d_modes_r, bb.d_M_ns,
                                             bb.d_M_r, bb.max_qp, bb.d_nlab, bb.L, X + o * kD);
    pair_targets<<<blocks(n), 256, 0, st>>>(n, dp, sec.ns_off, sec.r_off, bb.d_M_ns, bb.d_M_r, dx,
                                            std::log10(bb.L / 24.0), T + o);
    TGBA_CUDA(cudaGetLastError());
    TGBA_CUDA(cudaStreamSynchronize(st));
    cudaFree(dp);
    cudaFree(dx);
    o += n;
  }
  // 3. Adam on mini-batches; the last 5 % (in sample order) are held out for validation
  const int64_t n_val = std::max<int64_t>(1, n_samples / 20), n_tr = n_samples - n_val;
  const int64_t Bsz = 4096;
  float *work = nullptr, *grad = nullptr, *xb = nullptr, *tb = nullptr;
  int64_t* idx = nullptr;
  double* d_loss = nullptr;
  const int64_t wrows = std::max(Bsz, n_val);
  TGBA_CUDA(cudaMalloc(&work, (size_t)batch_work(wrows) * 4));
  TGBA_CUDA(cudaMalloc(&grad, s->P * 4));
  TGBA_CUDA(cudaMalloc(&xb, Bsz * kD * 4));
  TGBA_CUDA(cudaMalloc(&tb, Bsz * 4));
  TGBA_CUDA(cudaMalloc(&idx, Bsz * 8));
  TGBA_CUDA(cudaMalloc(&d_loss, 8));
  std::vector<int64_t> perm(n_tr);
  std::iota(perm.begin(), perm.end(), 0);
  const float b1 = 0.9f, b2 = 0.999f;
  const int64_t steps_per_epoch = (n_tr + Bsz - 1) / Bsz;
  const int64_t total_steps = steps_per_epoch * epochs;
  double tr_sum = 0;
  int64_t tr_cnt = 0;
  for (int ep = 0; ep < epochs; ++ep) {
    for (int64_t i = n_tr - 1; i > 0; --i) {          // Fisher-Yates with SplitMix64
      const int64_t j = (int64_t)(splitmix64(seed + 7919ull * (uint64_t)ep + 104729ull * (uint64_t)i) % (uint64_t)(i + 1));
      std::swap(perm[i], perm[j]);
    }
    tr_sum = 0;
    tr_cnt = 0;
    for (int64_t k = 0; k < steps_per_epoch; ++k) {
      const int64_t bn = std::min(Bsz, n_tr - k * Bsz);
      TGBA_CUDA(cudaMemcpyAsync(idx, perm.data() + k * Bsz, bn * 8, cudaMemcpyHostToDevice, st));
      gather_rows<<<blocks(bn * kD), 256, 0, st>>>(bn, kD, idx, X, T, xb, tb);
      if ((r = forward_backward(*s, xb, tb, bn, grad, work, d_loss, st)) != TGBA_OK) return r;
      ++s->adam_step;
      // cosine-decayed learning rate from 2e-3
      const double frac = (double)(s->adam_step - 1) / std::max<int64_t>(1, total_steps);
      const float lr = (float)(2e-3 * 0.5 * (1.0 + std::cos(M_PI * frac)) + 1e-5);
      const float c1 = 1.f - std::pow(b1, (float)s->adam_step), c2 = 1.f - std::pow(b2, (float)s->adam_step);
      adam_kernel<<<blocks(s->P), 256, 0, st>>>(s->P, s->theta, grad, s->m, s->v, lr, b1, b2, c1, c2, 1e-8f);
      if (ep == epochs - 1) {
        double h = 0;
        TGBA_CUDA(cudaMemcpyAsync(&h, d_loss, 8, cudaMemcpyDeviceToHost, st));
        TGBA_CUDA(cudaStreamSynchronize(st));
        tr_sum += h;
        tr_cnt += bn;
      }
    }
  }
  TGBA_CUDA(cudaGetLastError());
  // validation RMSE -> margin (three standard errors)
  if ((r = forward_backward(*s, X + n_tr * kD, T + n_tr, n_val, nullptr, work, d_loss, st)) != TGBA_OK) return r;
  double vl = 0;
  TGBA_CUDA(cudaMemcpyAsync(&vl, d_loss, 8, cudaMemcpyDeviceToHost, st));
  TGBA_CUDA(cudaStreamSynchronize(st));
  s->val_rmse = std::sqrt(vl / n_val);
  s->train_rmse = tr_cnt ? std::sqrt(tr_sum / tr_cnt) : 0;
  s->margin = 3.0 * s->val_rmse;
  cudaFree(X); cudaFree(T); cudaFree(work); cudaFree(grad); cudaFree(xb); cudaFree(tb); cudaFree(idx); cudaFree(d_loss);
  if ((r = refresh_bf16(*s, st)) != TGBA_OK) return r;
  TGBA_CUDA(cudaStreamSynchronize(st));
  if (stats) {
    stats[0] = s->train_rmse;
    stats[1] = s->val_rmse;
    stats[2] = s->margin;
    stats[3] = std::chrono::duration<double>(std::chrono::steady_clock::now() - t_start).count();
  }
  *out = s;
  return TGBA_OK;
}

}  // namespace tgba
