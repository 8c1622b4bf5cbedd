// Effective Hamiltonian (row a6; Eq. 2 and Eq. S4):
//   H = diag(E^(0)) - L h_x [[0, X], [X^H, 0]],  X_ab = C0 (-i)^{(M_a+M_b)/2} P_ab.
// With the diagonal unitary G = diag(g), g_a = (-i)^{M_a/2} on NS states and
// g_b = i^{M_b/2} e^{-i arg C0} on R states, G^H H G is real symmetric with off-diagonal block
// -L h_x |C0| P; the eigen solver and the spectral sums work in that gauge (eigenvalues and
// |<psi|sigma|psi'>| are unchanged).
#include "tgba_internal.h"

namespace tgba {

constexpr int kHeffTile = 64;

namespace {

// X_ab from P_ab
__device__ __forceinline__ double2 xval(const double* c0, double p, int n) {
  const double re = c0[0] * p, im = c0[1] * p;
  switch ((n >> 1) & 3) {
    case 0: return make_double2(re, im);
    case 1: return make_double2(im, -re);
    case 2: return make_double2(-re, -im);
    default: return make_double2(-im, re);
  }
}

// Column-major complex H of every sector in one launch.  A block of 256 threads owns one kHeffTile
// square tile: of the X block (P read once, coalesced, and written to both off-diagonal blocks of H, the
// transposed one through shared memory) or of a diagonal block (zeros and the energies).  Bound: the
// HBM write of 16 B per entry.  Measured: L = 24, all sectors (1.39 GB) 257 us, L = 80, M <= 10 (1.70 GB) 311 us,
// 5.4 TB/s; 504 and 754 us with complex products, see phased.
// C0 is real (elements.cu), so an entry -L h_x X is v (-i)^{n/2}, v = -L h_x C0 P: one FP64
// multiplication per pair, the phase and the conjugate by moving v to the real or imaginary part and
// flipping its sign bit as an integer.  (General complex products, four FP64 multiplications per pair,
// held the kernel at 2.8 to 3.5 TB/s whatever its tile and store hints.)
__device__ __forceinline__ double2 phased(double v, int n, bool conj) {
  const int k = (n >> 1) & 3;                       // (-i)^k
  const bool im = k & 1, neg = k == 2 || (im && ((k == 1) != conj));
  const long long b = __double_as_longlong(v) ^ (neg ? (long long)0x8000000000000000ull : 0ll);
  return make_double2(__longlong_as_double(im ? 0ll : b), __longlong_as_double(im ? b : 0ll));
}

__global__ void __launch_bounds__(256) heff_kernel(const HeffSector* __restrict__ secs, int n_sec,
                                                   const double* __restrict__ E_ns, const double* __restrict__ E_r,
                                                   const uint8_t* __restrict__ M_ns, const uint8_t* __restrict__ M_r,
                                                   const double* __restrict__ P, const double* __restrict__ c0,
                                                   double scale, double2* __restrict__ Hall) {
  constexpr int T = kHeffTile, W = T / 32;            // W: lanes' columns per warp row
  __shared__ double t[T][T + 1];
  __shared__ uint8_t s_m[T], s_mr[T];
  int lo = 0, hi = n_sec - 1;                         // the sector holding this tile
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (secs[mid].tile0 <= (int64_t)blockIdx.x) lo = mid;
    else hi = mid - 1;
  }
  const HeffSector sc = secs[lo];
  const int n_ns = (int)sc.n_ns, n_r = (int)sc.n_r;
  const int64_t n = sc.n_ns + sc.n_r;
  const int tn = (n_ns + T - 1) / T, tr = (n_r + T - 1) / T;
  int q = (int)((int64_t)blockIdx.x - sc.tile0);
  double2* H = Hall + sc.h_off;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  if (q < tn * tr) {
    const int a0 = (q / tr) * T, b0 = (q % tr) * T;
    const double* Ps = P + sc.x_off + (int64_t)a0 * n_r + b0;
    if (threadIdx.x < T) {
      s_m[threadIdx.x] = a0 + (int)threadIdx.x < n_ns ? M_ns[sc.ns_off + a0 + threadIdx.x] : 0;
      s_mr[threadIdx.x] = b0 + (int)threadIdx.x < n_r ? M_r[sc.r_off + b0 + threadIdx.x] : 0;
    }
    const int na = min(T, n_ns - a0), nb = min(T, n_r - b0);
    const double cs = scale * c0[0];
#pragma unroll
    for (int y = ty; y < T; y += 8)
#pragma unroll
      for (int w = 0; w < W; ++w)
        if (y < na && tx + 32 * w < nb) t[y][tx + 32 * w] = cs * Ps[(int64_t)y * n_r + tx + 32 * w];
    __syncthreads();
#pragma unroll 4
    for (int y = ty; y < na; y += 8)
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const int b = tx + 32 * w;
        if (b < nb) H[(int64_t)(a0 + y) * n + n_ns + b0 + b] = phased(t[y][b], s_m[y] + s_mr[b], true);   // R row, NS column
      }
#pragma unroll 4
    for (int y = ty; y < nb; y += 8)
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const int a = tx + 32 * w;
        if (a < na) H[(int64_t)(n_ns + b0 + y) * n + a0 + a] = phased(t[a][y], s_m[a] + s_mr[y], false);
      }
    return;
  }
  q -= tn * tr;
  const bool ns = q < tn * tn;
  if (!ns) q -= tn * tn;
  const int nt = ns ? tn : tr, m = ns ? n_ns : n_r, o = ns ? 0 : n_ns;
  const double* E = ns ? E_ns + sc.ns_off : E_r + sc.r_off;
  const int col0 = (q / nt) * T, row0 = (q % nt) * T;
#pragma unroll 4
  for (int y = ty; y < T; y += 8)
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const int col = col0 + y, row = row0 + tx + 32 * w;
      if (col < m && row < m) H[(int64_t)(o + col) * n + o + row] = make_double2(row == col ? E[row] : 0.0, 0.0);
    }
}

// Real-gauge H~ (column-major, n_k x n_k) of a subset of a sector's states.
__global__ void heff_real_kernel(int64_t kn, int64_t kr, const int32_t* __restrict__ idx_ns,
                                 const int32_t* __restrict__ idx_r, int64_t n_r, const double* __restrict__ E_ns,
                                 const double* __restrict__ E_r, const double* __restrict__ P,
                                 const double* __restrict__ c0, double scale, double* __restrict__ A) {
  const int64_t n = kn + kr;
  const double c = scale * sqrt(c0[0] * c0[0] + c0[1] * c0[1]);
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n * n; idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t col = idx / n, row = idx - col * n;
    double v = 0.0;
    if (row == col) {
      v = row < kn ? E_ns[idx_ns ? idx_ns[row] : row] : E_r[idx_r ? idx_r[row - kn] : row - kn];
    } else if (row < kn && col >= kn) {
      const int64_t a = idx_ns ? idx_ns[row] : row, b = idx_r ? idx_r[col - kn] : col - kn;
      v = c * P[a * n_r + b];
    } else if (row >= kn && col < kn) {
      const int64_t a = idx_ns ? idx_ns[col] : col, b = idx_r ? idx_r[row - kn] : row - kn;
      v = c * P[a * n_r + b];
    }
    A[idx] = v;
  }
}

__global__ void export_kernel(int64_t n_ns, int64_t n_r, const uint8_t* __restrict__ M_ns,
                              const uint8_t* __restrict__ M_r, const double* __restrict__ P,
                              const double* __restrict__ c0, double2* __restrict__ X) {
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n_ns * n_r; idx += (int64_t)gridDim.x * blockDim.x) {
    const int64_t a = idx / n_r, b = idx - a * n_r;
    X[idx] = xval(c0, P[idx], M_ns[a] + M_r[b]);
  }
}

int grid_for(int64_t work, int threads) {
  int64_t g = (work + threads - 1) / threads;
  return (int)(g < 152 * 32 ? (g < 1 ? 1 : g) : 152 * 32);
}

}  // namespace

std::vector<HeffSector> heff_sectors(const Basis& b, int64_t* tiles) {
  std::vector<HeffSector> v;
  int64_t t = 0;
  for (const Sector& sec : b.sectors) {
    if (sec.n_ns + sec.n_r == 0) continue;
    v.push_back(HeffSector{sec.n_ns, sec.n_r, sec.ns_off, sec.r_off, sec.x_off, sec.h_off, t});
    const int64_t tn = (sec.n_ns + kHeffTile - 1) / kHeffTile, tr = (sec.n_r + kHeffTile - 1) / kHeffTile;
    t += tn * tr + tn * tn + tr * tr;
  }
  *tiles = t;
  return v;
}

tgba_status assemble_heff(Basis& b, double h_x, double* heff, cudaStream_t st) {
  if (b.heff_tiles == 0) return TGBA_OK;
  if (b.heff_tiles > 0x7fffffff) return fail(TGBA_ELIMIT, "too many tiles of H_eff");
  heff_kernel<<<(unsigned)b.heff_tiles, 256, 0, st>>>(b.d_heff_secs, b.n_heff_secs, b.d_E_ns, b.d_E_r, b.d_M_ns,
                                                      b.d_M_r, b.d_P, b.d_c0, -b.L * h_x, (double2*)heff);
  TGBA_CUDA(cudaGetLastError());
  ++b.launches;
  return TGBA_OK;
}

tgba_status export_x(Basis& b, int s, double* x, cudaStream_t st) {
  const Sector& sec = b.sectors[s];
  const int64_t work = sec.n_ns * sec.n_r;
  if (work == 0) return TGBA_OK;
  export_kernel<<<grid_for(work, 256), 256, 0, st>>>(sec.n_ns, sec.n_r, b.d_M_ns + sec.ns_off, b.d_M_r + sec.r_off,
                                                     b.d_P + sec.x_off, b.d_c0, (double2*)x);
  TGBA_CUDA(cudaGetLastError());
  ++b.launches;
  return TGBA_OK;
}

tgba_status build_real_heff(Basis& b, int s, double h_x, double* a, const int32_t* idx_ns, int64_t kn,
                            const int32_t* idx_r, int64_t kr, cudaStream_t st) {
  const Sector& sec = b.sectors[s];
  const int64_t n = kn + kr;
  if (n == 0) return TGBA_OK;
  heff_real_kernel<<<grid_for(n * n, 256), 256, 0, st>>>(kn, kr, idx_ns, idx_r, sec.n_r, b.d_E_ns + sec.ns_off,
                                                         b.d_E_r + sec.r_off, b.d_P + sec.x_off, b.d_c0,
                                                         -b.L * h_x, a);
  TGBA_CUDA(cudaGetLastError());
  ++b.launches;
  return TGBA_OK;
}

}  // namespace tgba
