// k_leaf_simt.cu -- CUDA-core leaves: out = X Y^T mod p in exact int64
// arithmetic, independent of the digit planes of the tensor-core leaf.
// leaf_simt_kernel is the check path for the recursion (AAT_LEAF_SIMT), slow
// and simple; leaf_small_kernel computes small products in one launch.
#include <algorithm>

#include "common.cuh"

namespace aat {

namespace {

constexpr int TS = 32;  // output tile TS x TS, 32 x 8 threads, 4 rows each
constexpr int TK = 32;

__global__ void leaf_simt_kernel(const int32_t *__restrict__ X, int64_t ldx,
                                 const int32_t *__restrict__ Y, int64_t ldy, int64_t M,
                                 int64_t N, int64_t K, int32_t *out, int64_t ldo, int lower,
                                 Lin lin, ModP m) {
  __shared__ int32_t xs[TS][TK + 1];
  __shared__ int32_t ys[TS][TK + 1];
  const int64_t r0 = (int64_t)blockIdx.y * TS, c0 = (int64_t)blockIdx.x * TS;
  if (lower && c0 > r0 + TS - 1) return;
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  int32_t acc[4] = {0, 0, 0, 0};  // balanced partial sums
  for (int64_t k0 = 0; k0 < K; k0 += TK) {
    for (int yy = ty; yy < TS; yy += 8) {
      int64_t r = r0 + yy, c = c0 + yy, kk = k0 + tx;
      xs[yy][tx] = (r < M && kk < K) ? bal(X[r * ldx + kk], m) : 0;
      ys[yy][tx] = (c < N && kk < K) ? bal(Y[c * ldy + kk], m) : 0;
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < TK; ++kk) {
      const int32_t yv = ys[tx][kk];
      for (int q = 0; q < 4; ++q) {
        // |acc| <= p/2, |x y| <= p^2 / 4 < 2^60: the sum stays below 2^62
        acc[q] = red_s64((int64_t)acc[q] + (int64_t)xs[ty + 8 * q][kk] * yv, m);
      }
    }
    __syncthreads();
  }
  for (int q = 0; q < 4; ++q) {
    int64_t r = r0 + ty + 8 * q, c = c0 + tx;
    if (r >= M || c >= N) continue;
    if (lower && c > r) continue;
    const int32_t old = lin.beta.w ? out[r * ldo + c] : 0;
    out[r * ldo + c] = (int32_t)lin_apply(acc[q], old, lin, m);
  }
}

// Small products in one launch: no digit planes, no tensor-core pipeline to
// fill, and the strict upper triangle cleared on the way (zero).  The
// tensor-core path needs a split, a leaf and a clearing launch, ~13 us on the
// GPU however little there is to compute.  16 x 16 outputs per block so that
// small products still spread over the chip; four slices of K per block
// (two warps each) and 2 x 2 outputs per thread, so 16 multiply-adds go with
// four 16-byte shared-memory loads.  Bound by latency, then by 64-bit
// multiply-adds and shared-memory bandwidth.  Per call, host included, against
// the tensor-core path: 96 x 160 mod 65521 19 -> 14 us, 256 x 1024 mod 2^31 - 1
// 38 -> 17, 64 x 2048 mod 2^31 - 1 54 -> 29.
// FOLD: the int64 sums are brought back to |acc| <= 2^61 + p after every four
// products (|x y| < 2^60 each); else K ((p - 1) / 2)^2 stays below 2^62.
constexpr int kSmT = 16, kSmK = 128, kSmLd = kSmK + 4;

template <bool FOLD>
__global__ void __launch_bounds__(256)
    leaf_small_kernel(const int32_t *__restrict__ X, int64_t ldx, const int32_t *__restrict__ Y,
                      int64_t ldy, int64_t M, int64_t N, int64_t K, int32_t *out, int64_t ldo,
                      int lower, int zero, Lin lin, ModP m) {
  __shared__ __align__(16) int32_t xs[kSmT][kSmLd], ys[kSmT][kSmLd];
  __shared__ int32_t part[4][kSmT][kSmT + 1];
  int64_t I, J;
  if (lower) {
    tri_index(blockIdx.x, I, J);
  } else {
    const int64_t tn = (N + kSmT - 1) / kSmT;
    I = blockIdx.x / tn;
    J = blockIdx.x - I * tn;
  }
  const int64_t r0 = I * kSmT, c0 = J * kSmT;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int slice = threadIdx.x >> 6, tr = (threadIdx.x >> 3) & 7, tc = threadIdx.x & 7;
  // rows warp and warp + 8 of both tiles, four columns of the chunk per lane;
  // balanced only when stored, so that nothing waits for the next chunk's loads
  // while this one is multiplied
  int32_t pre[4][4];
  auto fetch = [&](int64_t k0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int64_t r = (i < 2 ? r0 : c0) + warp + 8 * (i & 1), lim = i < 2 ? M : N;
      const int32_t *row = i < 2 ? X + r * ldx : Y + r * ldy;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int64_t k = k0 + lane + 32 * j;
        pre[i][j] = (r < lim && k < K) ? __ldg(row + k) : 0;
      }
    }
  };
  int64_t acc[2][2] = {{0, 0}, {0, 0}};
  fetch(0);
  for (int64_t k0 = 0; k0 < K; k0 += kSmK) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        (i < 2 ? xs : ys)[warp + 8 * (i & 1)][lane + 32 * j] = bal(pre[i][j], m);
    __syncthreads();
    if (k0 + kSmK < K) fetch(k0 + kSmK);
#pragma unroll
    for (int q = 0; q < kSmK / 16; ++q) {
      const int k = 32 * slice + 4 * q;
      int4 xv[2], yv[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        xv[i] = *reinterpret_cast<const int4 *>(&xs[tr + 8 * i][k]);
        yv[i] = *reinterpret_cast<const int4 *>(&ys[tc + 8 * i][k]);
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          int64_t a = acc[i][j];
          a += (int64_t)xv[i].x * yv[j].x;
          a += (int64_t)xv[i].y * yv[j].y;
          a += (int64_t)xv[i].z * yv[j].z;
          a += (int64_t)xv[i].w * yv[j].w;
          if constexpr (FOLD) {
            constexpr int64_t lim = (int64_t)1 << 61;
            if (a > lim) a -= (int64_t)m.off;
            else if (a < -lim) a += (int64_t)m.off;
          }
          acc[i][j] = a;
        }
    }
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) part[slice][tr + 8 * i][tc + 8 * j] = red_s64(acc[i][j], m);
  __syncthreads();
  const int rr = threadIdx.x >> 4, cc = threadIdx.x & 15;
  const int64_t r = r0 + rr, c = c0 + cc;
  if (r < M && c < N && (!lower || c <= r)) {
    const int64_t s = (int64_t)part[0][rr][cc] + part[1][rr][cc] + part[2][rr][cc] + part[3][rr][cc];
    const int32_t old = lin.beta.w ? out[r * ldo + c] : 0;
    out[r * ldo + c] = (int32_t)lin_apply(red_s64(s, m), old, lin, m);
  }
  // the mirrored tile's entries above the diagonal
  const int64_t zr = c0 + rr, zc = r0 + cc;
  if (zero && zr < N && zc < M && zc > zr) out[zr * ldo + zc] = 0;
}

}  // namespace

// Whether the one-launch kernel beats the tensor-core path's launches: by the
// 16 x 16 x K blocks of work there are (both paths measured per call, small
// kernel first, mod 65521 and 2^31 - 1, n x k lower: 400 x 400, 130 k units,
// 16 / 19 and 21 / 27 us; 512 x 512, 270 k, 21 / 19 and 26 / 30; 700 x 300,
// 297 k, 26 / 19 and 32 / 27) and by the serial chain over K (64 x 2048:
// 21 / 25 and 29 / 54 us).
bool leaf_small_pays(int64_t M, int64_t N, int64_t K, int lower) {
  const double tm = (double)((M + kSmT - 1) / kSmT), tn = (double)((N + kSmT - 1) / kSmT);
  const double blocks = lower ? 0.5 * tm * (tm + 1.0) : tm * tn;
  return blocks * (double)std::max<int64_t>(K, kSmK) <= 180e3 && K <= 2048;
}

cudaError_t launch_leaf_small(const int32_t *X, int64_t ldx, const int32_t *Y, int64_t ldy,
                              int64_t M, int64_t N, int64_t K, int32_t *out, int64_t ldo,
                              int lower, bool zero, const Lin &lin, const ModP &m,
                              cudaStream_t st) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  const int64_t tm = (M + kSmT - 1) / kSmT, tn = (N + kSmT - 1) / kSmT;
  const int64_t blocks = lower ? tm * (tm + 1) / 2 : tm * tn;
  if ((lower && M != N) || blocks > INT32_MAX) return cudaErrorInvalidValue;
  const double macs = lower ? 0.5 * (double)M * (double)(M + 1) * K : (double)M * N * K;
  ProfScope prof(AAT_K_LEAF_SIMT, st, 2.0 * macs);
  const bool fold = (double)K * (double)m.half * (double)m.half >= 4.0e18;
  if (fold)
    leaf_small_kernel<true><<<(unsigned)blocks, 256, 0, st>>>(X, ldx, Y, ldy, M, N, K, out, ldo,
                                                              lower, zero, lin, m);
  else
    leaf_small_kernel<false><<<(unsigned)blocks, 256, 0, st>>>(X, ldx, Y, ldy, M, N, K, out, ldo,
                                                               lower, zero, lin, m);
  return cudaGetLastError();
}

cudaError_t launch_leaf_simt(const int32_t *X, int64_t ldx, const int32_t *Y, int64_t ldy,
                             int64_t M, int64_t N, int64_t K, int32_t *out, int64_t ldo,
                             int lower, const Lin &lin, const ModP &m, cudaStream_t st) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  dim3 grid((unsigned)((N + TS - 1) / TS), (unsigned)((M + TS - 1) / TS));
  const double macs = lower ? 0.5 * (double)M * (double)(M + 1) * K : (double)M * N * K;
  ProfScope prof(AAT_K_LEAF_SIMT, st, 2.0 * macs);
  leaf_simt_kernel<<<grid, 256, 0, st>>>(X, ldx, Y, ldy, M, N, K, out, ldo, lower, lin, m);
  return cudaGetLastError();
}

}  // namespace aat
