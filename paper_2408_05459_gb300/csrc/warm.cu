// Learned warm start (an addition to the paper's method: an MLP predicts the
// initial n x k block instead of InitBCM).
//
//   features   A = [U | P_N U], U the unit rows of X (a zero row stays zero),
//              P_N the topology walk (Eqs. rw-hg, rw-ag, rw-mg), BF16, row
//              length kp = round_up(2d, 64), zero-padded;
//   forward    Z1 = A W1 + b1 on the tensor cores (tcgen05, BF16 operands,
//              FP32 accumulation), H = GELU(Z1), W = H W2 + b2 (CUDA cores);
//   loss       L = k - tr(G^-1 M^T M) + lam ||G/n - I||_F^2 with G = W^T W and
//              M = Q_t^T W (Q_t the target's k orthonormal columns): it
//              depends on W only through span(W) and its scale; dL/dW =
//              W C1 + Q_t C2 with C1 = 2 S + (4 lam / n)(G/n - I),
//              C2 = -2 M G^-1, S = G^-1 M^T M G^-1;
//   backward   dW2 = H^T dW, db2 = 1^T dW, dZ1 = (dW W2^T) * GELU'(Z1),
//              db1 = 1^T dZ1, dW1 = A^T dZ1 on the tensor cores (A^T and dZ1
//              in BF16, split over the node range);
//   update     Adam with FP32 master weights; W1^T refreshed in BF16.
// Reductions over nodes use float-float partial sums in a fixed order.
#include <algorithm>
#include <cmath>
#include <vector>

#include "common.cuh"

namespace ancka {

namespace {

constexpr int kHidden = 256;
constexpr int kWarmMaxK = 64;

__global__ void k_unit_rows(const float* __restrict__ X, int64_t n, int d, int ld, float* __restrict__ U) {
  const int lane = threadIdx.x & 31;
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (i >= n) return;
  const float* x = X + i * d;
  float s = 0.f;
  for (int c = lane; c < d; c += 32) s = fmaf(x[c], x[c], s);
  s = warp_sum(s);
  const float inv = s > 0.f ? 1.f / sqrtf(s) : 0.f;
  for (int c = lane; c < ld; c += 32) U[i * ld + c] = c < d ? x[c] * inv : 0.f;
}

// A[i, :] = [U_i | PU_i | 0] in BF16 (n_rows x kp, zero for i >= n) and, when
// requested, At = A^T (kp x n_pad): 64 x 64 tiles through shared memory, so
// that the features are read once and both copies are written in 128-byte
// rows.  Bound by HBM (820 MB at n = 200,000, d = 256); a thread per element
// with its own divisions, then a transpose, took 0.51 ms there.
__global__ void __launch_bounds__(256)
k_pack_features(const float* __restrict__ U, const float* __restrict__ PU, int64_t n, int d, int ld, int kp,
                int64_t n_pad, __nv_bfloat16* __restrict__ A, __nv_bfloat16* __restrict__ At) {
  __shared__ __nv_bfloat16 tile[64][66];
  const int64_t r0 = (int64_t)blockIdx.x * 64;
  const int c0 = blockIdx.y * 64, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int ca = c0 + lane, cb = ca + 32;
  float v[8][2];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int64_t i = r0 + w + 8 * q;
    const float* u = U + i * ld;
    const float* pu = PU + i * ld - d;
    v[q][0] = i < n && ca < 2 * d ? (ca < d ? u[ca] : pu[ca]) : 0.f;
    v[q][1] = i < n && cb < 2 * d ? (cb < d ? u[cb] : pu[cb]) : 0.f;
  }
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    tile[w + 8 * q][lane] = __float2bfloat16_rn(v[q][0]);
    tile[w + 8 * q][lane + 32] = __float2bfloat16_rn(v[q][1]);
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int r = w + 8 * q;
    const __nv_bfloat162 p = __halves2bfloat162(tile[r][2 * lane], tile[r][2 * lane + 1]);
    *reinterpret_cast<__nv_bfloat162*>(A + (r0 + r) * kp + c0 + 2 * lane) = p;
  }
  if (!At || r0 >= n_pad) return;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int c = w + 8 * q;
    const __nv_bfloat162 p = __halves2bfloat162(tile[2 * lane][c], tile[2 * lane + 1][c]);
    *reinterpret_cast<__nv_bfloat162*>(At + (int64_t)(c0 + c) * n_pad + r0 + 2 * lane) = p;
  }
}

// W = H W2 + b2, one warp per row, rows grid-stride.  A lane sums its 8 hidden
// units into 32 outputs, then five levels each halve the outputs a lane keeps
// (the additions of a butterfly per output, 31 shuffles instead of 160), which
// leaves output c in lane c.  W2 is kept transposed in shared memory (its
// rows, k floats apart, collided on the banks) and loaded once per CTA, not
// once per 8 rows: 0.54 ms before at n = 200,000, k = 20.
__global__ void __launch_bounds__(256)
k_mlp_out(const float* __restrict__ H, int64_t n, const float* __restrict__ W2, const float* __restrict__ b2, int k,
          float* __restrict__ W, int ldw) {
  extern __shared__ float w2s[];  // k x kHidden
  for (int e = threadIdx.x; e < kHidden * k; e += blockDim.x) w2s[(e % k) * kHidden + e / k] = W2[e];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t step = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t i = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); i < n; i += step) {
    float h[kHidden / 32];
#pragma unroll
    for (int j = 0; j < kHidden / 32; ++j) h[j] = H[i * kHidden + lane + 32 * j];
    for (int c0 = 0; c0 < k; c0 += 32) {
      float v[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        v[c] = 0.f;
        if (c0 + c < k) {
#pragma unroll
          for (int j = 0; j < kHidden / 32; ++j) v[c] = fmaf(h[j], w2s[(c0 + c) * kHidden + lane + 32 * j], v[c]);
        }
      }
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) {
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int c = 0; c < off; ++c) {
          const float send = up ? v[c] : v[c + off], keep = up ? v[c + off] : v[c];
          v[c] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
      }
      if (c0 + lane < k) W[i * ldw + c0 + lane] = v[0] + b2[c0 + lane];
    }
  }
}

// (hi, lo) += (bh, bl): float-float addition
__device__ __forceinline__ void ffa(float& hi, float& lo, float bh, float bl) {
  float s, e;
  two_sum(hi, bh, s, e);
  e = __fadd_rn(e, __fadd_rn(lo, bl));
  hi = __fadd_rn(s, e);
  lo = __fsub_rn(e, __fsub_rn(hi, s));
}

// partial[blk][a][b] = sum over the CTA's rows of X[r, a] Y[r, b] (X null:
// ones, p = 1), FP32 within 32-row tiles, float-float across tiles.  A thread
// owns N blocks of one row a and four columns of the result (block e: a = e mod
// p, columns 4 (e / p) ..), whose tile values are one load of X and one
// 16-byte load of Y per row; a tile is staged once for all columns.  (A thread
// per row a with 16 columns at a time left 236 of 256 threads idle for the
// k x k products and staged H twice: 1.6 ms for the four products of a step at
// n = 200,000, k = 20.)
constexpr int kXtyRows = 32;
template <int N>
__global__ void __launch_bounds__(256, 2)
k_xty_partial(const float* __restrict__ X, int ldx, const float* __restrict__ Y, int ldy, int64_t n, int p, int q,
              int stage_rows, float2* __restrict__ partial) {
  // stage_rows (a multiple of kXtyRows) x q4 float4 of Y, then as many rows of p floats of X
  extern __shared__ float4 xty_smem[];
  const int q4 = (q + 3) / 4;
  float4* ys4 = xty_smem;
  float* ys = reinterpret_cast<float*>(xty_smem);
  float* xs = ys + stage_rows * 4 * q4;
  const int64_t per = ceil_div(n, (int64_t)gridDim.x);
  const int64_t r0 = (int64_t)blockIdx.x * per;
  const int64_t r1 = (r0 + per < n) ? r0 + per : n;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int base = 0; base < p * q4; base += 256 * N) {
    int ea[N], eg[N];
    float hi[N][4], lo[N][4];
#pragma unroll
    for (int m = 0; m < N; ++m) {
      const int e = base + threadIdx.x + 256 * m;
      ea[m] = e % p;
      eg[m] = e < p * q4 ? e / p : 0;  // past the last block: a valid one, not written
#pragma unroll
      for (int c = 0; c < 4; ++c) hi[m][c] = lo[m][c] = 0.f;
    }
    for (int64_t rb = r0; rb < r1; rb += stage_rows) {
      const int rows = (int)((r1 - rb) < stage_rows ? (r1 - rb) : stage_rows);
      __syncthreads();
#pragma unroll 4
      for (int r = warp; r < rows; r += 8) {
        if (X) {
#pragma unroll 8
          for (int c = lane; c < p; c += 32) xs[r * p + c] = X[(rb + r) * ldx + c];
        } else if (lane == 0) {
          xs[r] = 1.f;
        }
        for (int c = lane; c < 4 * q4; c += 32) ys[r * 4 * q4 + c] = c < q ? Y[(rb + r) * ldy + c] : 0.f;
      }
      __syncthreads();
      for (int t0 = 0; t0 < rows; t0 += kXtyRows) {
        const int t1 = min(rows, t0 + kXtyRows);
        float acc[N][4];
#pragma unroll
        for (int m = 0; m < N; ++m)
#pragma unroll
          for (int c = 0; c < 4; ++c) acc[m][c] = 0.f;
#pragma unroll 2
        for (int r = t0; r < t1; ++r) {
#pragma unroll
          for (int m = 0; m < N; ++m) {
            const float xa = xs[r * p + ea[m]];
            const float4 y = ys4[r * q4 + eg[m]];
            acc[m][0] = fmaf(xa, y.x, acc[m][0]);
            acc[m][1] = fmaf(xa, y.y, acc[m][1]);
            acc[m][2] = fmaf(xa, y.z, acc[m][2]);
            acc[m][3] = fmaf(xa, y.w, acc[m][3]);
          }
        }
#pragma unroll
        for (int m = 0; m < N; ++m)
#pragma unroll
          for (int c = 0; c < 4; ++c) ffa(hi[m][c], lo[m][c], acc[m][c], 0.f);
      }
    }
#pragma unroll
    for (int m = 0; m < N; ++m) {
      if (base + threadIdx.x + 256 * m >= p * q4) continue;
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (4 * eg[m] + c < q)
          partial[((int64_t)blockIdx.x * p + ea[m]) * q + 4 * eg[m] + c] = make_float2(hi[m][c], lo[m][c]);
    }
  }
}

// sum over blocks of entry t of m entries per block by eight neighbouring
// lanes: lane u adds blocks u, u + 8, ... in order, then the lanes' sums are
// combined in a fixed order (one thread per entry, one load in flight, took
// 44 us for 304 blocks)
constexpr int kSumLanes = 8;
__device__ __forceinline__ void sum_partials(const float2* __restrict__ part, int nblk, int64_t m, int64_t t, float& hi,
                                             float& lo) {
  hi = 0.f;
  lo = 0.f;
  const int u = threadIdx.x % kSumLanes;
#pragma unroll 8
  for (int b = u; b < nblk; b += kSumLanes) {
    const float2 v = t < m ? part[(int64_t)b * m + t] : make_float2(0.f, 0.f);
    ffa(hi, lo, v.x, v.y);
  }
#pragma unroll
  for (int off = 1; off < kSumLanes; off <<= 1) {
    const float h2 = __shfl_xor_sync(0xffffffffu, hi, off), l2 = __shfl_xor_sync(0xffffffffu, lo, off);
    if (u & off) {  // the lower lane's sum first in both
      float h = h2, l = l2;
      ffa(h, l, hi, lo);
      hi = h;
      lo = l;
    } else {
      ffa(hi, lo, h2, l2);
    }
  }
}

// out[a][b] = sum over blocks (in order) of the partials, as double
__global__ void k_xty_reduce(const float2* __restrict__ partial, int nblk, int p, int q, double* __restrict__ out) {
  const int t = (blockIdx.x * blockDim.x + threadIdx.x) / kSumLanes;
  float hi, lo;
  sum_partials(partial, nblk, (int64_t)p * q, t, hi, lo);
  if (t < p * q && threadIdx.x % kSumLanes == 0) out[t] = (double)hi + (double)lo;
}

int xty_blocks(int64_t n) { return (int)std::min<int64_t>(304, std::max<int64_t>(1, ceil_div(n, 256))); }

ancka_status xty(Workspace& ws, const float* X, int ldx, const float* Y, int ldy, int64_t n, int p, int q,
                 double* out, cudaStream_t s) {
  const int nb = xty_blocks(n);
  float2* part;
  ANCKA_TRY(ws.alloc(&part, (size_t)nb * p * q));
  const int blocks = p * ((q + 3) / 4);
  // as many 32-row tiles staged at a time as 47 KB hold, eight at most (one at
  // p = 256, eight for the k x k products at k = 20, which waited for memory
  // at every tile: 88 us each with one); p <= kHidden and q <= 64: 41 KB a tile
  // at most
  const size_t tile = (size_t)kXtyRows * (p + 4 * ((q + 3) / 4)) * sizeof(float);
  const int tiles = (int)std::max<size_t>(1, std::min<size_t>(8, 47 * 1024 / tile));
  const int sr = tiles * kXtyRows;
  const size_t smem = tiles * tile;
  if (blocks <= 256)
    k_xty_partial<1><<<nb, 256, smem, s>>>(X, ldx, Y, ldy, n, p, q, sr, part);
  else if (blocks <= 1024)
    k_xty_partial<4><<<nb, 256, smem, s>>>(X, ldx, Y, ldy, n, p, q, sr, part);
  else  // six blocks fill the registers two CTAs an SM leave a thread
    k_xty_partial<6><<<nb, 256, smem, s>>>(X, ldx, Y, ldy, n, p, q, sr, part);
  ANCKA_LAUNCHED();
  k_xty_reduce<<<(unsigned)ceil_div((int64_t)p * q * kSumLanes, 128), 128, 0, s>>>(part, nb, p, q, out);
  ANCKA_LAUNCHED();
  return ANCKA_OK;
}

// One CTA, FP64: from G = W^T W and M = Q_t^T W (k x k), the loss and the
// coefficient matrices of dL/dW = W C1 + Q_t C2.  G = L L^T by a right-looking
// Cholesky and, in the same steps, Y = L^-1 by Gauss-Jordan elimination on
// [L | I], so that a step is one reciprocal root and a few dependent FP64
// operations across the CTA (with serial pivots, divisions and a thread per
// column of the back substitution the kernel took 240 us at k = 20); G^-1 =
// Y^T Y.  A non-positive pivot sets *status.
constexpr int kCoeffThreads = 512;
__global__ void __launch_bounds__(kCoeffThreads)
k_warm_coeffs(const double* __restrict__ G, const double* __restrict__ M, int k, double n, double lam,
              float* __restrict__ C1, float* __restrict__ C2, double* __restrict__ loss,
              int32_t* __restrict__ status) {
  extern __shared__ double sm[];
  double* R = sm;               // k x k: G's trailing block, then the columns of L (row j: column j of L)
  double* Gi = R + k * k;       // G^-1
  double* T1 = Gi + k * k;      // M^T M
  double* T2 = T1 + k * k;      // Y = L^-1, then G^-1 M^T M
  double* Sm = T2 + k * k;      // S
  __shared__ double rinv;
  const int kk = k * k;
  for (int e = threadIdx.x; e < kk; e += blockDim.x) {
    R[e] = G[e];
    T2[e] = e / k == e % k ? 1.0 : 0.0;
  }
  __syncthreads();
  for (int j = 0; j < k; ++j) {
    if (threadIdx.x == 0) {
      double d = R[j * k + j];
      if (!(d > 0.0)) {
        *status = 1;
        d = 1e-300;
      }
      rinv = 1.0 / sqrt(d);
    }
    __syncthreads();
    const double ri = rinv;
    // row j of L^T (columns > j) and of Y (columns <= j) times 1 / L_jj
    for (int c = threadIdx.x; c < k; c += blockDim.x) {
      if (c > j) R[j * k + c] *= ri;
      else T2[j * k + c] *= ri;
    }
    __syncthreads();
    const int m = k - j - 1;  // later rows
    for (int e = threadIdx.x; e < m * k; e += blockDim.x) {
      const int i = j + 1 + e / k, c = e % k;
      const double lij = R[j * k + i];
      if (c <= j) T2[i * k + c] = fma(-lij, T2[j * k + c], T2[i * k + c]);
      else if (c >= i) R[i * k + c] = fma(-lij, R[j * k + c], R[i * k + c]);
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < kk; e += blockDim.x) {
    const int a = e / k, b = e % k;
    double v = 0.0;
    for (int m = max(a, b); m < k; ++m) v += T2[m * k + a] * T2[m * k + b];
    Gi[e] = v;
    double w = 0.0;
    for (int m = 0; m < k; ++m) w += M[m * k + a] * M[m * k + b];
    T1[e] = w;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < kk; e += blockDim.x) {
    const int a = e / k, b = e % k;
    double v = 0.0;
    for (int m = 0; m < k; ++m) v += Gi[a * k + m] * T1[m * k + b];
    T2[e] = v;  // G^-1 M^T M
  }
  __syncthreads();
  for (int e = threadIdx.x; e < kk; e += blockDim.x) {
    const int a = e / k, b = e % k;
    double v = 0.0, u = 0.0;
    for (int m = 0; m < k; ++m) {
      v += T2[a * k + m] * Gi[m * k + b];   // S = G^-1 M^T M G^-1
      u += M[a * k + m] * Gi[m * k + b];    // M G^-1
    }
    Sm[e] = v;
    const double pen = G[e] / n - (a == b ? 1.0 : 0.0);
    T1[e] = pen * pen;
    C1[e] = (float)(2.0 * v + 4.0 * lam / n * pen);
    C2[e] = (float)(-2.0 * u);
  }
  __syncthreads();
  if (threadIdx.x < 32) {  // a lane's entries in order, then a butterfly
    double tr = 0.0, pen = 0.0;
    for (int a = threadIdx.x; a < k; a += 32) tr += T2[a * k + a];
    for (int e = threadIdx.x; e < kk; e += 32) pen += T1[e];
    tr = warp_sum_d(tr);
    pen = warp_sum_d(pen);
    if (threadIdx.x == 0) *loss = (double)k - tr + lam * pen;
  }
}

// dW[i, c] = sum_a W[i, a] C1[a, c] + Qt[i, a] C2[a, c]
__global__ void k_grad_w(const float* __restrict__ W, int ldw, const float* __restrict__ Qt, int ldq, int64_t n, int k,
                         const float* __restrict__ C1, const float* __restrict__ C2, float* __restrict__ dW) {
  extern __shared__ float cs[];  // C1, C2
  for (int e = threadIdx.x; e < 2 * k * k; e += blockDim.x) cs[e] = e < k * k ? C1[e] : C2[e - k * k];
  __syncthreads();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * k) return;
  const int64_t i = t / k;
  const int c = (int)(t % k);
  float acc = 0.f;
  for (int a = 0; a < k; ++a) {
    acc = fmaf(W[i * ldw + a], cs[a * k + c], acc);
    acc = fmaf(Qt[i * ldq + a], cs[k * k + a * k + c], acc);
  }
  dW[i * ldw + c] = acc;
}

__device__ __forceinline__ float gelu_grad_f(float z) {
  return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.3989422804014327f * expf(-0.5f * z * z);
}

// dZ1 = (dW W2^T) * GELU'(Z1) in tiles of 32 rows (a CTA takes tiles
// blockIdx.x, blockIdx.x + gridDim.x, ...), thread j = hidden unit; written
// transposed in BF16 (dZ1t: kHidden x n_pad) and summed per CTA for db1
// (float-float partials).  KQ: 16-byte groups of a row of dW (4 KQ >= k, zero
// padded), so that a row costs KQ loads of dW and 4 KQ FMAs instead of 64
// predicated ones of each; eight rows' Z1 are loaded ahead.
constexpr int kDzRows = 32;
template <int KQ>
__global__ void __launch_bounds__(kHidden, 2)
k_dz1(const float* __restrict__ dW, int ldw, const float* __restrict__ Z1, const float* __restrict__ W2, int k,
      int64_t n, int64_t n_pad, __nv_bfloat16* __restrict__ dZ1t, float2* __restrict__ db1_part) {
  __shared__ float4 dws[kDzRows][KQ];
  __shared__ __nv_bfloat162 tile[kHidden][kDzRows / 2 + 1];
  const int j = threadIdx.x;
  float w2[4 * KQ];
#pragma unroll
  for (int c = 0; c < 4 * KQ; ++c) w2[c] = c < k ? W2[j * k + c] : 0.f;
  float hi = 0.f, lo = 0.f;
  const int64_t ntiles = ceil_div(n_pad, (int64_t)kDzRows);
  for (int64_t tl = blockIdx.x; tl < ntiles; tl += gridDim.x) {
    const int64_t r0 = tl * kDzRows;
    __syncthreads();
    for (int e = threadIdx.x; e < kDzRows * 4 * KQ; e += blockDim.x) {
      const int r = e / (4 * KQ), c = e % (4 * KQ);
      reinterpret_cast<float*>(dws)[e] = (c < k && r0 + r < n) ? dW[(r0 + r) * ldw + c] : 0.f;
    }
    __syncthreads();
#pragma unroll 1
    for (int rb = 0; rb < kDzRows; rb += 8) {
      float z[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) z[u] = r0 + rb + u < n ? Z1[(r0 + rb + u) * kHidden + j] : 0.f;
      float dz[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        float dh = 0.f;
#pragma unroll
        for (int g = 0; g < KQ; ++g) {
          const float4 v = dws[rb + u][g];
          dh = fmaf(v.x, w2[4 * g], dh);
          dh = fmaf(v.y, w2[4 * g + 1], dh);
          dh = fmaf(v.z, w2[4 * g + 2], dh);
          dh = fmaf(v.w, w2[4 * g + 3], dh);
        }
        dz[u] = r0 + rb + u < n ? dh * gelu_grad_f(z[u]) : 0.f;
        ffa(hi, lo, dz[u], 0.f);
      }
#pragma unroll
      for (int u = 0; u < 8; u += 2) tile[j][(rb + u) / 2] = __floats2bfloat162_rn(dz[u], dz[u + 1]);
    }
    __syncthreads();
    // row jj of dZ1t: 32 consecutive nodes (n_pad is a multiple of 64)
    for (int e = threadIdx.x; e < kHidden * kDzRows / 2; e += blockDim.x) {
      const int jj = e / (kDzRows / 2), r = e % (kDzRows / 2);
      *reinterpret_cast<__nv_bfloat162*>(dZ1t + (int64_t)jj * n_pad + r0 + 2 * r) = tile[jj][r];
    }
  }
  db1_part[(int64_t)blockIdx.x * kHidden + j] = make_float2(hi, lo);
}

__global__ void k_reduce_f2(const float2* __restrict__ part, int nblk, int m, float* __restrict__ out) {
  const int t = (blockIdx.x * blockDim.x + threadIdx.x) / kSumLanes;
  float hi, lo;
  sum_partials(part, nblk, m, t, hi, lo);
  if (t < m && threadIdx.x % kSumLanes == 0) out[t] = hi + lo;
}

__global__ void k_d2f(const double* __restrict__ a, int64_t m, float* __restrict__ b) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < m) b[t] = (float)a[t];
}

// Adam (bias-corrected): p -= lr * (m / c1) / (sqrt(v / c2) + eps), for
// m rows x cols of g with row stride ldg (p, m, v contiguous)
__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, int64_t rows, int cols, int ldg,
                       float* __restrict__ m, float* __restrict__ v, float lr, float b1, float b2, float c1, float c2,
                       float eps) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= rows * cols) return;
  const float gv = g[(t / cols) * ldg + (t % cols)];
  const float mv = b1 * m[t] + (1.f - b1) * gv;
  const float vv = b2 * v[t] + (1.f - b2) * gv * gv;
  m[t] = mv;
  v[t] = vv;
  p[t] -= lr * (mv / c1) / (sqrtf(vv / c2) + eps);
}

// W1^T in BF16 (kHidden x kp) from W1 (d_in x kHidden FP32), zero-padded
__global__ void k_w1t(const float* __restrict__ W1, int d_in, int kp, __nv_bfloat16* __restrict__ W1t) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)kHidden * kp) return;
  const int j = (int)(t / kp), c = (int)(t % kp);
  W1t[t] = __float2bfloat16_rn(c < d_in ? W1[(int64_t)c * kHidden + j] : 0.f);
}

}  // namespace

int warm_kp(int d) { return (int)round_up(2 * (int64_t)d, 64); }

// A (round_up(n, 128) x kp BF16, rows >= n zero) and, if At is not null, At
// (round_up(kp, 128) x n_pad BF16, n_pad = round_up(n, 64), zero outside
// kp x n) for a topology and its attributes
ancka_status warm_features(Workspace& ws, const Walk& w, const float* X, int d, __nv_bfloat16* A,
                           __nv_bfloat16* At, cudaStream_t s) {
  const int64_t n = w.n;
  const int ld = (int)round_up(d, 4);
  const int kp = warm_kp(d);
  const int64_t n_pad = round_up(n, 64);
  if (At && kp % 128 != 0)  // the rows past kp; the kernel writes the rest
    ANCKA_CUDA(cudaMemsetAsync(At + (int64_t)kp * n_pad, 0, sizeof(__nv_bfloat16) * (round_up(kp, 128) - kp) * n_pad, s));
  float *U, *PU;
  ANCKA_TRY(ws.alloc(&U, (size_t)n * ld));
  ANCKA_TRY(ws.alloc(&PU, (size_t)n * ld));
  k_unit_rows<<<(unsigned)ceil_div(n * 32, 256), 256, 0, s>>>(X, n, d, ld, U);
  ANCKA_LAUNCHED();
  ANCKA_TRY(apply_topology(ws, w, U, ld, PU, s));
  const dim3 grid((unsigned)(round_up(n, 128) / 64), (unsigned)(kp / 64));
  k_pack_features<<<grid, 256, 0, s>>>(U, PU, n, d, ld, kp, n_pad, A, At);
  ANCKA_LAUNCHED();
  return ANCKA_OK;
}

// W = GELU(A W1 + b1) W2 + b2 (n x k, row stride ldw); Z1 and H (n x 256)
// are kept for a backward pass when the caller passes them
ancka_status warm_forward(Workspace& ws, const __nv_bfloat16* A, int64_t n, int kp, const __nv_bfloat16* W1t,
                          const float* b1, const float* W2, const float* b2, int k, float* W, int ldw, float* Z1,
                          float* H, int32_t* err, cudaStream_t s) {
  if (!Z1) ANCKA_TRY(ws.alloc(&Z1, (size_t)n * kHidden));
  if (!H) ANCKA_TRY(ws.alloc(&H, (size_t)n * kHidden));
  ANCKA_TRY(gemm_bias_gelu(A, n, kp, W1t, b1, Z1, H, kHidden, err, s));
  const size_t smem = (size_t)kHidden * k * sizeof(float);
  // (limits are the process's: those of k = 64, as other threads' calls may need them)
  ANCKA_CUDA(cudaFuncSetAttribute(k_mlp_out, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)(kHidden * kWarmMaxK * sizeof(float))));
  // six CTAs an SM at most; at k = 64 three fit (64 KB each), so two waves
  k_mlp_out<<<(unsigned)std::min<int64_t>(ceil_div(n, 8), 152 * 6), 256, smem, s>>>(H, n, W2, b2, k, W, ldw);
  ANCKA_LAUNCHED();
  return ANCKA_OK;
}

ancka_status warm_refresh_w1t(const float* W1, int d_in, int kp, __nv_bfloat16* W1t, cudaStream_t s) {
  k_w1t<<<(unsigned)ceil_div((int64_t)kHidden * kp, 256), 256, 0, s>>>(W1, d_in, kp, W1t);
  ANCKA_LAUNCHED();
  return ANCKA_OK;
}

// One training step on one graph: forward, loss, backward and Adam.  The
// model tensors (FP32) and their Adam moments are updated in place; *loss_dev
// receives the loss before the update.
ancka_status warm_train_step(Workspace& ws, const WarmStepArgs& a, cudaStream_t s) {
  const int64_t n = a.n;
  const int k = a.k;
  const int ldw = (int)round_up(k, 4);
  float *W, *Z1, *H, *dW, *C1, *C2, *dW2, *db2, *db1, *dW1;
  double *G, *M, *dW2d, *db2d;
  __nv_bfloat16* dZ1t;
  ANCKA_TRY(ws.alloc(&W, (size_t)n * ldw));
  ANCKA_TRY(ws.alloc(&Z1, (size_t)n * kHidden));
  ANCKA_TRY(ws.alloc(&H, (size_t)n * kHidden));
  ANCKA_TRY(ws.alloc(&dW, (size_t)n * ldw));
  ANCKA_TRY(ws.alloc(&C1, (size_t)k * k));
  ANCKA_TRY(ws.alloc(&C2, (size_t)k * k));
  ANCKA_TRY(ws.alloc(&G, (size_t)k * k));
  ANCKA_TRY(ws.alloc(&M, (size_t)k * k));
  ANCKA_TRY(ws.alloc(&dW2d, (size_t)kHidden * k));
  ANCKA_TRY(ws.alloc(&db2d, (size_t)k));
  ANCKA_TRY(ws.alloc(&dW2, (size_t)kHidden * k));
  ANCKA_TRY(ws.alloc(&db2, (size_t)k));
  ANCKA_TRY(ws.alloc(&db1, (size_t)kHidden));
  ANCKA_TRY(ws.alloc(&dW1, (size_t)round_up(a.kp, 128) * kHidden));
  const int64_t n_pad = round_up(n, 64);
  ANCKA_TRY(ws.alloc(&dZ1t, (size_t)kHidden * n_pad));
  // forward
  ANCKA_TRY(warm_forward(ws, a.A, n, a.kp, a.W1t, a.b1, a.W2, a.b2, k, W, ldw, Z1, H, a.err, s));
  // loss and dL/dW
  ANCKA_TRY(xty(ws, W, ldw, W, ldw, n, k, k, G, s));
  ANCKA_TRY(xty(ws, a.Qt, a.ldq, W, ldw, n, k, k, M, s));
  const size_t csm = (size_t)5 * k * k * sizeof(double);
  ANCKA_CUDA(cudaFuncSetAttribute(k_warm_coeffs, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)(5 * kWarmMaxK * kWarmMaxK * sizeof(double))));
  k_warm_coeffs<<<1, kCoeffThreads, csm, s>>>(G, M, k, (double)n, (double)a.lam, C1, C2, a.loss_dev, a.status);
  ANCKA_LAUNCHED();
  k_grad_w<<<(unsigned)ceil_div(n * k, 256), 256, (size_t)2 * k * k * sizeof(float), s>>>(W, ldw, a.Qt, a.ldq, n, k,
                                                                                           C1, C2, dW);
  ANCKA_LAUNCHED();
  // backward
  ANCKA_TRY(xty(ws, H, kHidden, dW, ldw, n, kHidden, k, dW2d, s));
  ANCKA_TRY(xty(ws, nullptr, 0, dW, ldw, n, 1, k, db2d, s));
  k_d2f<<<(unsigned)ceil_div((int64_t)kHidden * k, 256), 256, 0, s>>>(dW2d, (int64_t)kHidden * k, dW2);
  ANCKA_LAUNCHED();
  k_d2f<<<1, 64, 0, s>>>(db2d, k, db2);
  ANCKA_LAUNCHED();
  const int nb = (int)std::min<int64_t>(304, ceil_div(n_pad, (int64_t)kDzRows));
  float2* db1p;
  ANCKA_TRY(ws.alloc(&db1p, (size_t)nb * kHidden));
  // Five widths bound what the zero columns cost: at n = 200,000 (the kernel
  // alone) k = 4: 183 us, 174 with an instance of its own width; k = 9: 227 and
  // 202; k = 16: 228 and 215; k = 24: 244 and 238; k = 33: 305 and 259; k = 36:
  // 306 and 258; k = 52: 333 and 320.  That is 1.5% of a step (3.1 ms at
  // d = 256, k = 20) at most; all 16 widths would triple the kernel's code.
  auto dz1 = k <= 8 ? k_dz1<2> : k <= 20 ? k_dz1<5> : k <= 32 ? k_dz1<8> : k <= 48 ? k_dz1<12> : k_dz1<16>;
  dz1<<<nb, kHidden, 0, s>>>(dW, ldw, Z1, a.W2, k, n, n_pad, dZ1t, db1p);
  ANCKA_LAUNCHED();
  k_reduce_f2<<<(unsigned)(kHidden * kSumLanes / 128), 128, 0, s>>>(db1p, nb, kHidden, db1);
  ANCKA_LAUNCHED();
  ANCKA_TRY(gemm_at_b(ws, a.At, a.kp, n_pad, dZ1t, dW1, a.err, s));
  if (a.grads) {  // gradients out (tests)
    ANCKA_CUDA(cudaMemcpyAsync(a.grads->W1, dW1, sizeof(float) * a.d_in * kHidden, cudaMemcpyDeviceToDevice, s));
    ANCKA_CUDA(cudaMemcpyAsync(a.grads->b1, db1, sizeof(float) * kHidden, cudaMemcpyDeviceToDevice, s));
    ANCKA_CUDA(cudaMemcpyAsync(a.grads->W2, dW2, sizeof(float) * kHidden * k, cudaMemcpyDeviceToDevice, s));
    ANCKA_CUDA(cudaMemcpyAsync(a.grads->b2, db2, sizeof(float) * k, cudaMemcpyDeviceToDevice, s));
  }
  // Adam
  const double c1 = 1.0 - std::pow(0.9, (double)a.t), c2 = 1.0 - std::pow(0.999, (double)a.t);
  struct T {
    float* p;
    const float* g;
    int64_t rows;
    int cols;
    float* m;
    float* v;
  } ts[4] = {{a.W1, dW1, a.d_in, kHidden, a.mW1, a.vW1},
             {a.b1, db1, 1, kHidden, a.mb1, a.vb1},
             {a.W2, dW2, kHidden, k, a.mW2, a.vW2},
             {a.b2, db2, 1, k, a.mb2, a.vb2}};
  for (const T& q : ts) {
    k_adam<<<(unsigned)ceil_div(q.rows * q.cols, 256), 256, 0, s>>>(q.p, q.g, q.rows, q.cols, q.cols, q.m, q.v,
                                                                      a.lr, 0.9f, 0.999f, (float)c1, (float)c2, 1e-8f);
    ANCKA_LAUNCHED();
  }
  return warm_refresh_w1t(a.W1, a.d_in, a.kp, a.W1t, s);
}

}  // namespace ancka
