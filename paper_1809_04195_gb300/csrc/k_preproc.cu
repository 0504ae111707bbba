// Pre-processing in front of the per-slice solve (Sec. III.A), from a sparse array of
// fully sampled readout lines: line j holds the channels [Ctot][Nx] of phase encode
// (ky_j, kz_j) at echo t_j.  The host groups the lines by phase encode (pixel) ky nz + kz with a
// counting sort: order[off[pixel]] .. order[off[pixel + 1] - 1]; every kernel works on that table.
//
//   coil compression: the central win^3 window averaged over the echoes of each (ky, kz)
//     (k_calib), its channel Gram matrix G = X^H X (k_gram), eigenvectors of G by a
//     float64 cyclic Jacobi in one CTA, decreasing eigenvalue, canonical phase (k_eig):
//     W [Ctot][C];
//   decoupling: y_v = y W per line, then the centred unitary inverse DFT along x
//     (k_compress_readout): yhat [n][C][Nx];
//   re-sort and project: ytil[x][c][k][ky][kz] = sum_{j at (ky, kz)} Phi[t_j][k] yhat[j][c][x]
//     (k_project_lines) and the masks mask[t_j][ky_j][kz_j] = 1 (k_mark_mask).
#include "t2sh_device.cuh"
#include "two_radix.h"

namespace t2sh {

namespace {

constexpr int kPpThreads = 256;

// calibration rows X[p][c], p = (sampled phase encode in the window, kx in the window); off: first
// line of each phase encode in `order`, wpix: the sampled phase encodes of the window
__global__ void __launch_bounds__(kPpThreads) k_calib(const float2* __restrict__ lines, int ctot, int nx,
                                                    const int* __restrict__ order, const int* __restrict__ off,
                                                    const int* __restrict__ wpix, int nwpix, int win,
                                                    float2* __restrict__ X) {
  const int x0 = nx / 2 - win / 2;
  const long long total = (long long)nwpix * win * ctot;
  for (long long e = blockIdx.x * (long long)kPpThreads + threadIdx.x; e < total; e += (long long)gridDim.x * kPpThreads) {
    const int c = (int)(e % ctot);
    const long long p = e / ctot;
    const int xw = (int)(p % win), si = (int)(p / win);
    const int j0 = off[wpix[si]], j1 = off[wpix[si] + 1];
    float2 acc = make_float2(0.f, 0.f);
    for (int j = j0; j < j1; ++j) {
      const float2 v = lines[((long long)order[j] * ctot + c) * nx + x0 + xw];
      acc.x += v.x;
      acc.y += v.y;
    }
    const float inv = 1.f / (float)(j1 - j0);
    X[p * ctot + c] = make_float2(acc.x * inv, acc.y * inv);
  }
}

// G[c1][c2] += sum_p conj(X[p][c1]) X[p][c2] over this CTA's chunk of rows (float64 atomics)
__global__ void __launch_bounds__(kPpThreads) k_gram(const float2* __restrict__ X, long long npts, int ctot,
                                                   int chunk, double* G) {
  const long long p0 = (long long)blockIdx.x * chunk;
  const long long p1 = p0 + chunk < npts ? p0 + chunk : npts;
  for (int pr = threadIdx.x; pr < ctot * ctot; pr += kPpThreads) {
    const int c1 = pr / ctot, c2 = pr - c1 * ctot;
    float re = 0.f, im = 0.f;
    for (long long p = p0; p < p1; ++p) {
      const float2 a = X[p * ctot + c1], b = X[p * ctot + c2];
      re += a.x * b.x + a.y * b.y;
      im += a.x * b.y - a.y * b.x;
    }
    atomicAdd(&G[2 * pr], (double)re);
    atomicAdd(&G[2 * pr + 1], (double)im);
  }
}

// Eigenvectors of the Hermitian G (interleaved re/im, ctot <= kMaxChan) by Jacobi in float64, sorted
// by decreasing eigenvalue, each column rotated so that its entry of largest magnitude (first such
// index) is real positive; W [ctot][ncomp].  One CTA; each sweep is n - 1 rounds of n / 2 disjoint
// rotations (round-robin pairs), whose parameters come from the matrix before the round and which
// all threads apply together: on one thread the chain of dependent float64 operations took 21.3 ms
// for 16 channels, here 0.43 ms.
constexpr int kEigLd = kMaxChan + 1;
struct EigRot {
  int a, b;  // b < 0: no rotation
  double c, s, dr, di;
};
__global__ void __launch_bounds__(kPpThreads) k_eig(const double* G, int ctot, int ncomp, float2* W, int* err) {
  __shared__ double ar[kMaxChan][kEigLd], ai[kMaxChan][kEigLd], vr[kMaxChan][kEigLd], vi[kMaxChan][kEigLd];
  __shared__ EigRot rot[kMaxChan / 2];
  __shared__ double part[2][kPpThreads / 32];
  __shared__ int ord[kMaxChan];
  const int n = ctot, tid = threadIdx.x, m = n + (n & 1), h = m / 2;
  for (int e = tid; e < n * n; e += kPpThreads) {
    const int i = e / n, j = e - i * n;
    // symmetrised: the float partial sums are Hermitian only to rounding
    ar[i][j] = 0.5 * (G[2 * (i * n + j)] + G[2 * (j * n + i)]);
    ai[i][j] = i == j ? 0.0 : 0.5 * (G[2 * (i * n + j) + 1] - G[2 * (j * n + i) + 1]);
    vr[i][j] = i == j ? 1.0 : 0.0;
    vi[i][j] = 0.0;
  }
  __syncthreads();
  bool converged = n == 1;
  for (int sweep = 0; sweep < 60 && !converged; ++sweep) {
    double off = 0.0, diag = 0.0;
    for (int e = tid; e < n * n; e += kPpThreads) {
      const int i = e / n, j = e - i * n;
      if (i == j) diag += ar[i][i] * ar[i][i];
      else if (i < j) off += ar[i][j] * ar[i][j] + ai[i][j] * ai[i][j];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_xor_sync(0xffffffffu, off, o);
      diag += __shfl_xor_sync(0xffffffffu, diag, o);
    }
    if ((tid & 31) == 0) {
      part[0][tid >> 5] = off;
      part[1][tid >> 5] = diag;
    }
    __syncthreads();
    off = diag = 0.0;
    for (int i = 0; i < kPpThreads / 32; ++i) {
      off += part[0][i];
      diag += part[1][i];
    }
    converged = !(off > 1e-30 * diag);  // the same sums in every thread
    __syncthreads();
    if (converged) break;
    for (int rd = 0; rd < m - 1; ++rd) {
      if (tid < h) {  // pair tid of the round: i + j = rd (mod m - 1), the fixed point meets m - 1
        const int i0 = (int)((long long)rd * h % (m - 1));
        int a = tid == 0 ? i0 : (i0 + tid) % (m - 1);
        int b = tid == 0 ? m - 1 : (i0 - tid + m - 1) % (m - 1);
        if (a > b) {
          const int t = a;
          a = b;
          b = t;
        }
        EigRot r{a, -1, 1.0, 0.0, 1.0, 0.0};
        if (b < n) {
          const double xr = ar[a][b], xi = ai[a][b], r2 = xr * xr + xi * xi;
          if (r2 > 1e-290) {
            const double ir = rsqrt(r2);  // column b *= d = conj(a_ab) / |a_ab|
            const double theta = (ar[b][b] - ar[a][a]) * (0.5 * ir), u = theta * theta + 1.0;
            double t = fabs(theta) > 1e100 ? 0.5 / fabs(theta) : 1.0 / (fabs(theta) + u * rsqrt(u));
            if (theta < 0.0) t = -t;
            r.b = b;
            r.dr = xr * ir;
            r.di = -xi * ir;
            r.c = rsqrt(t * t + 1.0);
            r.s = t * r.c;
          }
        }
        rot[tid] = r;
      }
      __syncthreads();
      for (int e = tid; e < 2 * n * h; e += kPpThreads) {  // columns of A and of V
        const int k = (e >> 1) % n;
        const EigRot r = rot[(e >> 1) / n];
        if (r.b < 0) continue;
        double(*pr)[kEigLd] = (e & 1) ? vr : ar;
        double(*pi)[kEigLd] = (e & 1) ? vi : ai;
        const double xr = pr[k][r.a], xi = pi[k][r.a];
        const double yr = pr[k][r.b] * r.dr - pi[k][r.b] * r.di, yi = pr[k][r.b] * r.di + pi[k][r.b] * r.dr;
        pr[k][r.a] = r.c * xr - r.s * yr;
        pi[k][r.a] = r.c * xi - r.s * yi;
        pr[k][r.b] = r.s * xr + r.c * yr;
        pi[k][r.b] = r.s * xi + r.c * yi;
      }
      __syncthreads();
      for (int e = tid; e < n * h; e += kPpThreads) {  // rows of A
        const int k = e % n;
        const EigRot r = rot[e / n];
        if (r.b < 0) continue;
        const double xr = ar[r.a][k], xi = ai[r.a][k];
        const double yr = ar[r.b][k] * r.dr + ai[r.b][k] * r.di, yi = ai[r.b][k] * r.dr - ar[r.b][k] * r.di;
        const bool pa = k == r.a, pb = k == r.b;  // the pivot is zero, the diagonal real
        ar[r.a][k] = pb ? 0.0 : r.c * xr - r.s * yr;
        ai[r.a][k] = pa || pb ? 0.0 : r.c * xi - r.s * yi;
        ar[r.b][k] = pa ? 0.0 : r.s * xr + r.c * yr;
        ai[r.b][k] = pa || pb ? 0.0 : r.s * xi + r.c * yi;
      }
      __syncthreads();
    }
  }
  if (!converged && err && tid == 0) atomicExch(err, 1);
  if (tid == 0) {  // order by decreasing eigenvalue (stable selection)
    for (int i = 0; i < n; ++i) ord[i] = i;
    for (int i = 0; i < n; ++i) {
      int best = i;
      for (int j = i + 1; j < n; ++j)
        if (ar[ord[j]][ord[j]] > ar[ord[best]][ord[best]]) best = j;
      const int t = ord[i];
      ord[i] = ord[best];
      ord[best] = t;
    }
  }
  __syncthreads();
  for (int c = tid; c < ncomp; c += kPpThreads) {
    const int col = ord[c];
    int im = 0;
    double mm = -1.0;
    for (int k = 0; k < n; ++k) {
      const double m2 = vr[k][col] * vr[k][col] + vi[k][col] * vi[k][col];
      if (m2 > mm) {
        mm = m2;
        im = k;
      }
    }
    const double a = sqrt(mm);
    const double pr = a > 0.0 ? vr[im][col] / a : 1.0, pi = a > 0.0 ? -vi[im][col] / a : 0.0;  // conj phase
    for (int k = 0; k < n; ++k)
      W[k * ncomp + c] = make_float2((float)(vr[k][col] * pr - vi[k][col] * pi), (float)(vr[k][col] * pi + vi[k][col] * pr));
  }
}

// y_v = y W for line blockIdx.x, then the centred unitary inverse DFT along x:
// x[n] = s (-1)^n / sqrt(Nx) * IDFT((-1)^k X[k])[n], s = (-1)^(Nx/2).
template <bool R13>
__global__ void __launch_bounds__(kPpThreads) k_compress_readout(const float2* __restrict__ lines,
                                                               const float2* __restrict__ W, int ctot, int ncomp,
                                                               int nx, FftPlan px, const float2* __restrict__ tw_g,
                                                               int cb, float2* __restrict__ yh) {
  extern __shared__ float2 smem[];
  const int ld = nx + 1;
  float2* tw = smem;
  float2* ws = tw + ((nx + 1) & ~1);         // [ctot][ncomp]
  float2* buf = ws + ctot * ncomp;           // [cb][ld]
  const long long j = blockIdx.x;
  for (int i = threadIdx.x; i < nx; i += kPpThreads) tw[i] = tw_g[i];
  for (int i = threadIdx.x; i < ctot * ncomp; i += kPpThreads) ws[i] = W[i];
  const float scale = ((nx / 2) & 1 ? -1.f : 1.f) * rsqrtf((float)nx);
  for (int c0 = 0; c0 < ncomp; c0 += cb) {
    const int nc = min(cb, ncomp - c0);
    __syncthreads();
    for (int e = threadIdx.x; e < nc * nx; e += kPpThreads) {
      const int cl = e / nx, x = e - cl * nx;
      float2 v = make_float2(0.f, 0.f);
      for (int c = 0; c < ctot; ++c) cfma(v, lines[(j * ctot + c) * nx + x], ws[c * ncomp + c0 + cl]);
      buf[cl * ld + x] = (x & 1) ? make_float2(-v.x, -v.y) : v;
    }
    __syncthreads();
    fft_lines<true, R13>(buf, ld, nc, px, tw);
    for (int e = threadIdx.x; e < nc * nx; e += kPpThreads) {
      const int cl = e / nx, x = e - cl * nx;
      const float sg = (x & 1) ? -scale : scale;
      const float2 v = buf[cl * ld + x];
      yh[(j * ncomp + c0 + cl) * nx + x] = make_float2(sg * v.x, sg * v.y);
    }
  }
}

// The same for lengths nx = RA RB with two radices (run-time choice, fully unrolled butterflies).
// One thread per x reads each channel once and forms up to eight components in registers; the
// transform of a component is two register stages in place, an item per thread: A, DFT_RA over q of
// x = j + RB q; B, twiddle and DFT_RB over j, straight to global memory at x = k1 + RA k2 (runs of
// RA values).  RB values take an odd run in shared memory, so both stages are conflict free.
// Table I scan (35,777 lines, 16 channels to 7, nx = 288): 2.05 ms with per-value contractions
// and Stockham passes, 0.51 here (1.9 GB in and out: 0.28).
template <int R>
__device__ __forceinline__ void line_a(float2* b, int stride) {
  float2 v[R];
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = b[q * stride];
  dft_r<R, true>(v);
#pragma unroll
  for (int q = 0; q < R; ++q) b[q * stride] = v[q];
}
template <int R>
__device__ __forceinline__ void line_b(const float2* b, const float2* tw, int k1, float2* out, int ostride, float s0,
                                       float s1) {
  float2 v[R];
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = b[q];
#pragma unroll
  for (int q = 1; q < R; ++q) v[q] = twiddle_mul<true>(v[q], tw[q * k1]);
  dft_r<R, true>(v);
#pragma unroll
  for (int q = 0; q < R; ++q) out[q * ostride] = cscale(v[q], q & 1 ? s1 : s0);
}
constexpr int kTwoThreads = 160;  // 80 registers, five CTAs: 0.51 ms; 320 threads at 64 registers 0.56, at 96 0.62
__global__ void __launch_bounds__(kTwoThreads, 5) k_compress_two(const float2* __restrict__ lines, const float2* __restrict__ W,
                                                     int ctot, int ncomp, int nx, int RA, int RB, int qs,
                                                     const float2* __restrict__ tw_g, float2* __restrict__ yh) {
  extern __shared__ float2 smem[];
  const int ld = RA * qs;
  float2* tw = smem;
  float2* ws = tw + nx;             // [ctot][8]: the components of this pass
  float2* buf = ws + ctot * 8;      // [8][ld]
  const long long j = blockIdx.x;
  for (int i = threadIdx.x; i < nx; i += blockDim.x) tw[i] = tw_g[i];
  const float scale = ((nx / 2) & 1 ? -1.f : 1.f) * rsqrtf((float)nx);
  for (int c0 = 0; c0 < ncomp; c0 += 8) {
    const int nc = min(8, ncomp - c0);
    __syncthreads();
    for (int i = threadIdx.x; i < ctot * 8; i += blockDim.x)
      ws[i] = (i & 7) < nc ? W[(i >> 3) * ncomp + c0 + (i & 7)] : make_float2(0.f, 0.f);
    __syncthreads();
    for (int x = threadIdx.x; x < nx; x += blockDim.x) {
      const float2* lp = lines + j * ctot * nx + x;
      float2 v[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = make_float2(0.f, 0.f);
#pragma unroll 8
      for (int c = 0; c < ctot; ++c) {
        const float2 a = lp[(long long)c * nx];
#pragma unroll
        for (int i = 0; i < 8; ++i) cfma(v[i], a, ws[c * 8 + i]);
      }
      const int q = x / RB;
      float2* b = buf + q * qs + (x - q * RB);
#pragma unroll
      for (int i = 0; i < 8; ++i)
        if (i < nc) b[i * ld] = (x & 1) ? make_float2(-v[i].x, -v[i].y) : v[i];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nc * RB; i += blockDim.x) {
      const int l = i / RB;
      float2* b = buf + l * ld + (i - l * RB);
      switch (RA) {
#define X(R) case R: line_a<R>(b, qs); break;
        T2SH_RADICES(X)
#undef X
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nc * RA; i += blockDim.x) {
      const int l = i / RA, k1 = i - l * RA;
      const float s0 = (k1 & 1) ? -scale : scale, s1 = (RA & 1) ? -s0 : s0;  // (-1)^(k1 + RA k2)
      float2* o = yh + (j * ncomp + c0 + l) * nx + k1;
      switch (RB) {
#define X(R) case R: line_b<R>(buf + l * ld + k1 * qs, tw, k1, o, RA, s0, s1); break;
        T2SH_RADICES(X)
#undef X
      }
    }
  }
}

// ytil[x][c][k][pixel] = sum_{j in pixel} Phi[t_j][k] yhat[j][c][x], zero where no line falls: every
// value of the output is written once, so no clearing pass precedes it.  A CTA owns 32 pixels x
// 32 x of one component: a warp reads runs of 32 x of the lines of its pixels, the tile is turned in
// shared memory and written as runs of 32 pixels (256 bytes).  Writing each pixel's values where
// they were formed (8 bytes every ncomp K N values) after clearing 4.0 GB took 3.9 + 0.6 ms for the
// Table I scan; this takes 0.89 ms, bound by the writes.
constexpr int kProjTile = 32, kProjOrder = 256;
template <int KC>
__global__ void __launch_bounds__(kPpThreads) k_project_lines(const float2* __restrict__ yh, int ncomp, int nx,
                                                            const int* __restrict__ order, const int* __restrict__ tj,
                                                            const int* __restrict__ off, const float* __restrict__ phi,
                                                            int K, long long N, float2* __restrict__ ytil) {
  extern __shared__ float2 tile[];  // [K][32 x][33]
  __shared__ int soff[kProjTile + 1], sord[kProjOrder], stj[kProjOrder];
  const long long pix0 = (long long)blockIdx.x * kProjTile;
  const int x0 = blockIdx.y * kProjTile, c = blockIdx.z;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, x = x0 + lane;
  if (threadIdx.x <= kProjTile) soff[threadIdx.x] = off[min(pix0 + (long long)threadIdx.x, N)];
  __syncthreads();
  const int q0 = soff[0], nq = soff[kProjTile] - q0;
  for (int i = threadIdx.x; i < min(nq, kProjOrder); i += kPpThreads) {
    sord[i] = order[q0 + i];
    stj[i] = tj[q0 + i];
  }
  __syncthreads();
  for (int p = warp; p < kProjTile; p += kPpThreads / 32) {
    float2 acc[KC];
#pragma unroll
    for (int k = 0; k < KC; ++k) acc[k] = make_float2(0.f, 0.f);
    const int e1 = soff[p + 1] - q0;
#pragma unroll 2
    for (int i = soff[p] - q0; i < e1; ++i) {
      const int j = i < kProjOrder ? sord[i] : order[q0 + i], t = i < kProjOrder ? stj[i] : tj[q0 + i];
      const float2 v = x < nx ? yh[((long long)j * ncomp + c) * nx + x] : make_float2(0.f, 0.f);
      const float* ph = phi + (long long)t * K;
#pragma unroll
      for (int k = 0; k < KC; ++k)
        if (k < K) {
          acc[k].x = fmaf(ph[k], v.x, acc[k].x);
          acc[k].y = fmaf(ph[k], v.y, acc[k].y);
        }
    }
#pragma unroll
    for (int k = 0; k < KC; ++k)
      if (k < K) tile[(k * kProjTile + lane) * (kProjTile + 1) + p] = acc[k];
  }
  __syncthreads();
  if (pix0 + lane >= N) return;
  for (int r = warp; r < K * kProjTile; r += kPpThreads / 32) {
    const int k = r / kProjTile, xx = r - k * kProjTile;
    if (x0 + xx < nx)
      __stcs(ytil + (((long long)(x0 + xx) * ncomp + c) * K + k) * N + pix0 + lane,
             tile[(k * kProjTile + xx) * (kProjTile + 1) + lane]);
  }
}

__global__ void k_mark_mask(const int* __restrict__ t, const int* __restrict__ ky, const int* __restrict__ kz, int n,
                            int ny, int nz, uint8_t* mask) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < n) mask[((long long)t[j] * ny + ky[j]) * nz + kz[j]] = 1;
}

int grid_for(long long total) {
  const long long b = (total + kPpThreads - 1) / kPpThreads;
  return (int)(b < 65535LL * 16 ? (b > 0 ? b : 1) : 65535LL * 16);
}

}  // namespace

cudaError_t launch_calib(const float2* lines, int ctot, int nx, const int* order, const int* off, const int* wpix,
                         int nwpix, int win, float2* X, cudaStream_t st) {
  const long long total = (long long)nwpix * win * ctot;
  if (total == 0) return cudaSuccess;
  k_calib<<<grid_for(total), kPpThreads, 0, st>>>(lines, ctot, nx, order, off, wpix, nwpix, win, X);
  return cudaGetLastError();
}

cudaError_t launch_gram_eig(const float2* X, long long npts, int ctot, int ncomp, double* G, float2* W, int* err,
                            cudaStream_t st) {
  if (ctot > kMaxChan) return cudaErrorInvalidValue;
  const int chunk = 256;
  const long long nb = (npts + chunk - 1) / chunk;
  cudaError_t e = cudaMemsetAsync(G, 0, sizeof(double) * 2 * ctot * ctot, st);
  if (e != cudaSuccess) return e;
  if (nb > 0) k_gram<<<(unsigned)nb, kPpThreads, 0, st>>>(X, npts, ctot, chunk, G);
  k_eig<<<1, kPpThreads, 0, st>>>(G, ctot, ncomp, W, err);
  return cudaGetLastError();
}

cudaError_t launch_compress_readout(const float2* lines, const float2* W, int nlines, int ctot, int ncomp,
                                    const FftPlan& px, const float2* tw_x, float2* yh, cudaStream_t st) {
  const int nx = px.n;
  int RA = 0, RB = 0;
  if (two_radices(nx, kMaxRadix, false, &RA, &RB)) {
    const int qs = RB | 1, threads = std::min(kTwoThreads, (nx + 31) / 32 * 32);
    const size_t sm = sizeof(float2) * ((size_t)nx + 8 * ctot + 8 * (size_t)RA * qs);
    const cudaError_t e = smem_optin((const void*)k_compress_two, 64 * 1024);
    if (e != cudaSuccess) return e;
    k_compress_two<<<nlines, threads, sm, st>>>(lines, W, ctot, ncomp, nx, RA, RB, qs, tw_x, yh);
    return cudaGetLastError();
  }
  int cb = (kStage * kPpThreads) / nx;
  if (cb < 1) return cudaErrorInvalidValue;
  if (cb > ncomp) cb = ncomp;
  const size_t sm = sizeof(float2) * (((nx + 1) & ~1) + (size_t)ctot * ncomp + (size_t)cb * (nx + 1));
  if (sm > 200 * 1024) return cudaErrorInvalidValue;
  if (plan_has13(px)) {
    {
      const cudaError_t e = smem_optin((const void*)k_compress_readout<true>, 200 * 1024);
      if (e != cudaSuccess) return e;
    }
    k_compress_readout<true><<<nlines, kPpThreads, sm, st>>>(lines, W, ctot, ncomp, nx, px, tw_x, cb, yh);
  } else {
    {
      const cudaError_t e = smem_optin((const void*)k_compress_readout<false>, 200 * 1024);
      if (e != cudaSuccess) return e;
    }
    k_compress_readout<false><<<nlines, kPpThreads, sm, st>>>(lines, W, ctot, ncomp, nx, px, tw_x, cb, yh);
  }
  return cudaGetLastError();
}

cudaError_t launch_project_lines(const float2* yh, int ncomp, int nx, const int* order, const int* tj, const int* off,
                                 const float* phi, int K, int ny, int nz, float2* ytil, cudaStream_t st) {
  const long long N = (long long)ny * nz;
  dim3 grid((unsigned)((N + kProjTile - 1) / kProjTile), (nx + kProjTile - 1) / kProjTile, ncomp);
  const size_t sm = sizeof(float2) * (size_t)K * kProjTile * (kProjTile + 1);
  const void* kern = K <= 4 ? (const void*)k_project_lines<4> : (const void*)k_project_lines<8>;
  const cudaError_t e = smem_optin(kern, 72 * 1024);
  if (e != cudaSuccess) return e;
  if (K <= 4)
    k_project_lines<4><<<grid, kPpThreads, sm, st>>>(yh, ncomp, nx, order, tj, off, phi, K, N, ytil);
  else
    k_project_lines<8><<<grid, kPpThreads, sm, st>>>(yh, ncomp, nx, order, tj, off, phi, K, N, ytil);
  return cudaGetLastError();
}

cudaError_t launch_mark_mask(const int* t, const int* ky, const int* kz, int n, int ny, int nz, uint8_t* mask,
                             cudaStream_t st) {
  k_mark_mask<<<(n + 255) / 256, 256, 0, st>>>(t, ky, kz, n, ny, nz, mask);
  return cudaGetLastError();
}

}  // namespace t2sh
