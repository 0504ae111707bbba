// Row and column passes for any line length that is a product of two radices (nearly every even
// product of 2, 3, 5 and 13 up to 400), any number of basis images, radices chosen at run time.
//
// Layout of t: t[s][c][y][z / W][k][z % W] with W = 4 columns per chunk (W = 2 where nz is not a
// multiple of 4); for K = 4, W = 4 that is the layout of k_col_il.cuh without its slot rotation, so
// its row passes and these column passes combine.  A column tile is N rows of one chunk (K W
// values); consecutive threads take consecutive values of a chunk, so global and shared accesses
// are contiguous whatever K is.
//
// Every line is transformed in two register stages in place (decimation in frequency, frequencies
// left where they fall; decimation in time back), as in k_col_il.cuh, with the radix of a stage
// selected by a block-uniform switch over fully unrolled butterflies.  Bound by instruction issue:
// run-time strides and radices cost 167 instructions per value in the column pass against 73 in the
// specialised one, so four images on the lengths of k_col_il.cuh / k_row_il.cuh go there
// (180x144, C = 10, 48 slices: 358 us; here 714; 2246 with the Stockham passes of k_fft.cu, one pass
// per prime power with its own index divisions and two block-wide barriers).  256x160 with six
// images, 16 slices: 1246 -> 619 us.  The Stockham passes stay for lengths that need three stages.
#include <algorithm>

#define T2SH_PACKED_ADD 1
#include "launch.h"
#include "t2sh_device.cuh"
#include "two_radix.h"

namespace t2sh {

namespace {

constexpr int kColThreads = 256, kRowThreads = 192;  // most threads of a column / row CTA
constexpr int kMaxImage = 16;  // largest image-side radix of a row pass (its values stay in registers)

#define T2SH_IMAGE_RADICES(X) X(2) X(3) X(4) X(5) X(6) X(8) X(9) X(10) X(12) X(13) X(15) X(16)

// ------------------------------------------------------------------------------------------
// Column pass
// ------------------------------------------------------------------------------------------
// DFT_R of buf[base + q stride] in place; PRE: times w^(q m) first (forward stage B); POST: times
// conj(w^(q m)) after (inverse stage B)
template <int R, bool INV, bool PRE, bool POST>
__device__ __forceinline__ void any_stage(float2* buf, int base, int stride, const float2* tw, int m) {
  float2 v[R];
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = buf[base + q * stride];
  if (PRE) {
#pragma unroll
    for (int q = 1; q < R; ++q) v[q] = twiddle_mul<false>(v[q], tw[q * m]);
  }
  dft_r<R, INV>(v);
  if (POST) {
#pragma unroll
    for (int q = 1; q < R; ++q) v[q] = twiddle_mul<true>(v[q], tw[q * m]);
  }
#pragma unroll
  for (int q = 0; q < R; ++q) buf[base + q * stride] = v[q];
}
// IDFT_R of buf[base + q stride] to out[q ostride]
template <int R>
__device__ __forceinline__ void any_store(const float2* buf, int base, int stride, float2* out, long long ostride) {
  float2 v[R];
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = buf[base + q * stride];
  dft_r<R, true>(v);
#pragma unroll
  for (int q = 0; q < R; ++q) out[q * ostride] = v[q];
}

struct AnyCol {
  int RA, RB;  // N = RA RB
  int W;       // columns per chunk
  int mode;    // IlPass
  int qs;      // shared-memory stride of RB rows, congruent to one row modulo 16 values: consecutive
               // items of stage B then start on consecutive banks
  int psi_sm;  // Psi of the tile's columns kept in shared memory (up to four images)
};

// Threads of a column CTA: whole items of LK threads, in as few equal rounds as kColThreads allows.
constexpr int col_threads(int LK, int items) {
  const int at_once = kColThreads / LK, rounds = (items + at_once - 1) / at_once;
  return (LK * ((items + rounds - 1) / rounds) + 31) / 32 * 32;
}
constexpr bool col_threads_fit() {
  for (int k = 1; k <= kMaxK; ++k)
    for (int w = 2; w <= 4; w += 2)
      for (int items = 2; items <= kMaxRadix; ++items) {
        const int t = col_threads(k * w, items);
        if (t < k * w || t > kColThreads) return false;
      }
  return true;
}
static_assert(col_threads_fit(), "every column CTA within its launch bounds");

// Persistent CTAs over contiguous runs of the (column chunk, slice x coil) list, column-chunk major:
// Psi of a chunk's columns is copied to shared memory once per run.  The next tile streams in by
// cp.async while the current one is transformed.  FWD: the passes that begin with the forward transform;
// the others take k-space (compiled apart, so that neither costs the other registers).
template <int KC, bool FWD>
__global__ void __launch_bounds__(kColThreads, KC == 4 ? 3 : 2)
    k_col_any(Geom g, AnyCol a, const float2* __restrict__ tw_g, const float* __restrict__ psi, const float2* in,
              float2* out, int nsc, int ntiles) {
  extern __shared__ float2 smem[];
  const int nz = g.nz, N = g.ny, K = g.K, RA = a.RA, RB = a.RB, W = a.W, LK = K * W, QS = a.qs;
  const int wl = W == 4 ? 2 : 1;
  const long long NN = (long long)N * nz;
  const int rowlen = K * nz;  // values of one row of t
  float2* tw = smem;  // [N]
  float2* bufs = smem + ((N + 1) & ~1);
  const int ts = (RA * QS + 1) & ~1;
  int* ftab = reinterpret_cast<int*>(bufs + (FWD ? 2 : 1) * ts);  // position -> place << 10 | frequency
  float* ps = reinterpret_cast<float*>(ftab + N);                 // [entry][position][w]
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    const int k1 = i / RB, k2 = i - k1 * RB;
    tw[i] = tw_g[i];
    ftab[i] = (k1 * QS + k2 * LK) << 10 | (k1 + RA * k2);
  }
  // thread = (item, value of the chunk); nitem items at a time
  const int nitem = blockDim.x / LK, item0 = threadIdx.x / LK, e = threadIdx.x - item0 * LK;
  const bool act = item0 < nitem;
  // copies: thread = (row, 16 bytes of the chunk)
  const int h = LK / 2, nrow = blockDim.x / h, row0 = threadIdx.x / h, ce = 2 * (threadIdx.x - row0 * h);
  const float scale = g.gsign * g.inv_sqrt_n;
  const int lo = (int)((long long)ntiles * blockIdx.x / gridDim.x),
            hi = (int)((long long)ntiles * (blockIdx.x + 1) / gridDim.x);
  auto issue = [&](int tile, float2* dst) {
    const int zt = tile / nsc, sc = tile - zt * nsc;
    const float2* src = in + (long long)sc * N * rowlen + (long long)zt * LK + ce;
    if (row0 < nrow) {
      int q = row0 / RB, j = row0 - q * RB;
      for (int y = row0; y < N; y += nrow) {
        cp_async16(dst + q * QS + j * LK + ce, src + (long long)y * rowlen);
        j += nrow;
        while (j >= RB) {
          j -= RB;
          ++q;
        }
      }
    }
  };
  pdl_wait();
  pdl_trigger();
  if (FWD && lo < hi) issue(lo, bufs);
  cp_async_commit();
  int have = -1;  // column chunk whose Psi is in shared memory
  for (int tile = lo; tile < hi; ++tile) {
    const int zt = tile / nsc, sc = tile - zt * nsc, z0 = zt * W;
    const long long tbase = (long long)sc * N * rowlen + (long long)zt * LK;
    float2* buf = bufs + (FWD ? ((tile - lo) & 1) * ts : 0);
    cp_async_wait<0>();
    __syncthreads();  // tables and this tile are here; the previous tile is done
    if constexpr (FWD) {
      if (tile + 1 < hi) issue(tile + 1, bufs + ((tile + 1 - lo) & 1) * ts);
      cp_async_commit();
      if (a.psi_sm && have != zt) {
        for (int i = threadIdx.x; i < N * W; i += blockDim.x) {
          const float* pp = psi + (long long)(ftab[i >> wl] & 1023) * nz + z0 + (i & (W - 1));
          for (int q = 0; q < g.P; ++q) ps[q * N * W + i] = pp[q * NN];
        }
        have = zt;  // read after at least two barriers
      }
    } else {  // k-space, centred and scaled, to the places where stage B leaves it
      // More than four images: eight loads in flight per thread (the compiler keeps one behind the other's
      // shared-memory store, which the array could alias): A^H from projected k-space, 240x128, K = 5, C = 15,
      // 16 slices 925 -> 539 us.  Up to four images, with more items per round: 240x108, K = 2 35 -> 49 us.
      constexpr int B = KC == 4 ? 1 : 8;
      const int k = e >> wl, w = e & (W - 1);
      const float2* src = a.mode == IL_ADJ ? in + tbase + e : in + ((long long)sc * K + k) * NN + z0 + w;
      const int fstep = a.mode == IL_ADJ ? rowlen : nz;
      for (int p = item0; act && p < N; p += B * nitem) {
        float2 v[B];
        int ft[B];
#pragma unroll
        for (int u = 0; u < B; ++u) {
          ft[u] = p + u * nitem < N ? ftab[p + u * nitem] : -1;
          if (ft[u] >= 0) v[u] = src[(ft[u] & 1023) * fstep];
        }
#pragma unroll
        for (int u = 0; u < B; ++u)
          if (ft[u] >= 0) buf[(ft[u] >> 10) + e] = cscale(v[u], scale * parity_sign((ft[u] & 1023) + w));  // z0 is even
      }
      __syncthreads();
    }
    if constexpr (FWD) {
      for (int j = item0; act && j < RB; j += nitem) {
        switch (RA) {
#define X(R) case R: any_stage<R, false, false, false>(buf, j * LK + e, QS, tw, 0); break;
          T2SH_RADICES(X)
#undef X
        }
      }
      __syncthreads();
      for (int j = item0; act && j < RA; j += nitem) {
        switch (RB) {
#define X(R) case R: any_stage<R, false, true, false>(buf, j * QS + e, LK, tw, j); break;
          T2SH_RADICES(X)
#undef X
        }
      }
      __syncthreads();
      // pointwise: Psi of the normal operator in place, or the scaled results to memory
      for (int i = threadIdx.x; i < N * W; i += blockDim.x) {
        const int w = i & (W - 1), ft = ftab[i >> wl], f = ft & 1023;
        float2* b = buf + (ft >> 10) + w;
        float2 v[KC], u[KC];
        const float sg = a.mode == IL_NORMAL ? 1.f : scale * parity_sign(f + w);
#pragma unroll
        for (int k = 0; k < KC; ++k) {
          v[k] = k < K ? cscale(b[k * W], sg) : make_float2(0.f, 0.f);
          u[k] = make_float2(0.f, 0.f);
        }
        if (a.mode == IL_FWD_RAW) {
#pragma unroll
          for (int k = 0; k < KC; ++k)
            if (k < K) out[tbase + (long long)f * rowlen + k * W + w] = v[k];
          continue;
        }
        const float pscale = a.mode == IL_FWD_PROJ ? (float)NN : 1.f;
        const float* pp = a.psi_sm ? ps + i : psi + (long long)f * nz + z0 + w;
        const long long pstep = a.psi_sm ? N * W : NN;
        int q = 0;
#pragma unroll
        for (int k = 0; k < KC; ++k)
#pragma unroll
          for (int l = k; l < KC; ++l)
            if (l < K) {
              const float c = pp[(q++) * pstep] * pscale;
              u[k].x = fmaf(c, v[l].x, u[k].x);
              u[k].y = fmaf(c, v[l].y, u[k].y);
              if (l != k) {
                u[l].x = fmaf(c, v[k].x, u[l].x);
                u[l].y = fmaf(c, v[k].y, u[l].y);
              }
            }
#pragma unroll
        for (int k = 0; k < KC; ++k)
          if (k < K) {
            if (a.mode == IL_NORMAL) b[k * W] = u[k];
            else out[((long long)sc * K + k) * NN + (long long)f * nz + z0 + w] = u[k];
          }
      }
      if (a.mode != IL_NORMAL) continue;
      __syncthreads();
    }
    for (int j = item0; act && j < RA; j += nitem) {
      switch (RB) {
#define X(R) case R: any_stage<R, true, false, true>(buf, j * QS + e, LK, tw, j); break;
        T2SH_RADICES(X)
#undef X
      }
    }
    __syncthreads();
    for (int j = item0; act && j < RB; j += nitem) {
      float2* o = out + tbase + (long long)j * rowlen + e;
      switch (RA) {
#define X(R) case R: any_store<R>(buf, j * LK + e, QS, o, (long long)RB * rowlen); break;
        T2SH_RADICES(X)
#undef X
      }
    }
  }
  cp_async_wait<0>();
}

// ------------------------------------------------------------------------------------------
// Row pass: CTA = (slice, band of rows), coil loop inside, image values in registers, as in
// k_row_il.cuh.  N = RI RT: RT items of radix RI on the image side, RI items of radix RT on the
// side of t; thread = (item, line), line = (row, k) with k fastest.
// ------------------------------------------------------------------------------------------
struct AnyRow {
  int RI, RT, W, rows;
  int trb;  // slot rotation of k_col_il.cuh (K = 4, W = 4), or 0
  int xs;   // exchange stride of an item of the t side, congruent to its lines modulo 16 values
};

// forward image side: products with the maps and DFT_RI, to ex[k1 xs]
template <int R, int MC>
__device__ __forceinline__ void row_image_fwd(const float2 (&xr)[MC][kMaxImage], const float2* mrow, int mplane, int mstep,
                                              float2* ex, int xs) {
  float2 v[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
    v[q] = make_float2(0.f, 0.f);
#pragma unroll
    for (int m = 0; m < MC; ++m) cfma(v[q], mrow[m * mplane + q * mstep], xr[m][q]);
  }
  dft_r<R, false>(v);
#pragma unroll
  for (int q = 0; q < R; ++q) ex[q * xs] = v[q];
}
// adjoint image side: twiddle, IDFT_RI, conj(map) and the sum over coils
template <int R, int MC>
__device__ __forceinline__ void row_image_adj(float2 (&acc)[MC][kMaxImage], const float2* mrow, int mplane, int mstep,
                                              const float2* ex, int xs, const float2* tw, int j) {
  float2 v[R];
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = ex[q * xs];
#pragma unroll
  for (int q = 1; q < R; ++q) v[q] = twiddle_mul<true>(v[q], tw[q * j]);
  dft_r<R, true>(v);
#pragma unroll
  for (int m = 0; m < MC; ++m)
#pragma unroll
    for (int q = 0; q < R; ++q) cfmac(acc[m][q], mrow[m * mplane + q * mstep], v[q]);
}
// offset in a row of t of column z
__device__ __forceinline__ int any_off(int z, int wl, int LK) { return (z >> wl) * LK + (z & ((1 << wl) - 1)); }
// side of t, forward: twiddle, DFT_RT, store; adjoint: load, IDFT_RT, to ex
template <int R>
__device__ __forceinline__ void row_t_fwd(const float2* ex, int xs, const float2* tw, int i, float2* t, int zs, int wl,
                                          int LK, bool on) {
  float2 v[R];
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = ex[q * xs];
#pragma unroll
  for (int q = 1; q < R; ++q) v[q] = twiddle_mul<false>(v[q], tw[q * i]);
  dft_r<R, false>(v);
  if (on) {
#pragma unroll
    for (int q = 0; q < R; ++q) t[any_off(i + q * zs, wl, LK)] = v[q];
  }
}
// (the loads are issued before the barrier `sync`, which every thread takes: A^H A of 50 slices of 100x160,
// K = 6, M = 2 784 -> 760 us; not those of radix 25, which the registers do not hold across it; in: the thread
// has an item)
template <int R, typename Sync>
__device__ __forceinline__ void row_t_adj(float2* ex, int xs, int i, const float2* t, int zs, int wl, int LK, bool on,
                                          bool in, Sync sync) {
  if constexpr (R > 20) sync();
  float2 v[R];
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = on ? t[any_off(i + q * zs, wl, LK)] : make_float2(0.f, 0.f);
  if constexpr (R <= 20) sync();
  if (!in) return;
  dft_r<R, true>(v);
#pragma unroll
  for (int q = 0; q < R; ++q) ex[q * xs] = v[q];
}

template <int MODE, int MC>
__global__ void __launch_bounds__(kRowThreads, MC == 1 ? 3 : 2)
    k_row_any(Geom g, AnyRow a, const float2* __restrict__ tw_g, const float2* __restrict__ maps,
              const float2* x, float2* t, float2* __restrict__ out) {
  extern __shared__ float2 smem[];
  const int N = g.nz, K = g.K, RI = a.RI, RT = a.RT, rows = a.rows, nl = K * rows, LK = K * a.W, xs = a.xs;
  const int wl = a.W == 4 ? 2 : 1;
  const long long NN = (long long)g.ny * N;
  const int s = blockIdx.y, y0 = blockIdx.x * rows, rb = min(rows, g.ny - y0);
  const int item = threadIdx.x / nl, line = threadIdx.x - item * nl, r = line / K, k = line - r * K;
  const bool in_i = item < RT, in_t = item < RI;
  const bool on_i = in_i && r < rb, on_t = in_t && r < rb;
  float2* tw = smem;
  float2* ex = tw + N;             // [k1][j][line]
  float2* mst = ex + ((RI * xs + 1) & ~1);  // map rows x2 [MC][rows][N]
  for (int i = threadIdx.x; i < N; i += blockDim.x) tw[i] = tw_g[i];
  auto issue = [&](int c, int buf) {
    const int h = N / 2;
    const float2* mp = maps + (long long)(s * g.C + c) * MC * NN + (long long)y0 * N;
    float2* md = mst + buf * MC * rows * N;
#pragma unroll
    for (int m = 0; m < MC; ++m)
      for (int i = threadIdx.x; i < rb * h; i += blockDim.x)  // the band's rows are contiguous
        cp_async16(md + m * rows * N + 2 * i, mp + (long long)m * NN + 2 * i);
  };
  issue(0, 0);  // the plan's maps
  cp_async_commit();
  pdl_wait();
  pdl_trigger();
  const int y = y0 + r;
  const int slot = a.trb ? (k + y % a.trb + y / a.trb) & 3 : k;
  float2* tp = t + ((long long)s * g.C * g.ny + y) * (K * N) + slot * a.W;
  const long long tcoil = K * NN;
  const long long img = ((long long)s * MC * K + k) * NN + (long long)y * N + item;
  float2* ex_i = ex + item * nl + line;  // image side: k1 at stride xs
  float2* ex_t = ex + item * xs + line;  // side of t: j at stride nl
  float2 val[MC][kMaxImage];                  // forward: x; adjoint: the sums
#pragma unroll
  for (int m = 0; m < MC; ++m)
#pragma unroll
    for (int q = 0; q < kMaxImage; ++q)
      val[m][q] = MODE == ROW_FWD && on_i && q < RI ? x[img + (long long)m * K * NN + q * RT] : make_float2(0.f, 0.f);
  for (int c = 0; c < g.C; ++c) {
    const int buf = c & 1;
    auto next_coil = [&] {
      cp_async_wait<0>();
      __syncthreads();  // coil c's maps are here, and nobody is in the previous coil any more
      if (c + 1 < g.C) issue(c + 1, buf ^ 1);
      cp_async_commit();
    };
    if (MODE == ROW_FWD) next_coil();
    const float2* mrow = mst + (buf * MC * rows + r) * N + item;
    if (MODE == ROW_FWD) {
      if (in_i) {
        switch (RI) {
#define X(R) case R: row_image_fwd<R, MC>(val, mrow, rows * N, RT, ex_i, xs); break;
          T2SH_IMAGE_RADICES(X)
#undef X
        }
      }
      __syncthreads();
      if (in_t) {
        switch (RT) {
#define X(R) case R: row_t_fwd<R>(ex_t, nl, tw, item, tp, RI, wl, LK, on_t); break;
          T2SH_RADICES(X)
#undef X
        }
      }
    } else {
      switch (RT) {
#define X(R) case R: row_t_adj<R>(ex_t, nl, item, tp, RI, wl, LK, on_t, in_t, next_coil); break;
        T2SH_RADICES(X)
#undef X
      }
      __syncthreads();
      if (in_i) {
        switch (RI) {
#define X(R) case R: row_image_adj<R, MC>(val, mrow, rows * N, RT, ex_i, xs, tw, item); break;
          T2SH_IMAGE_RADICES(X)
#undef X
        }
      }
    }
    tp += tcoil;
  }
  if (MODE == ROW_ADJ && on_i) {
#pragma unroll
    for (int m = 0; m < MC; ++m)
#pragma unroll
      for (int q = 0; q < kMaxImage; ++q)
        if (q < RI) out[img + (long long)m * K * NN + q * RT] = val[m][q];
  }
  cp_async_wait<0>();
}

// n rounded up to m modulo 16
int padded(int n, int m) { return n + ((m - n) % 16 + 16) % 16; }

// radices, strides and shared memory of a column pass; false where it has none
bool col_any_plan(const Geom& g, int W, IlPass pass, AnyCol* a, size_t* smem) {
  if (!two_radices(g.ny, kMaxRadix, false, &a->RA, &a->RB)) return false;
  const int LK = g.K * W;
  const bool fwd = pass == IL_NORMAL || pass == IL_FWD_PROJ || pass == IL_FWD_RAW;
  a->W = W;
  a->mode = pass;
  a->qs = padded(a->RB * LK, LK);
  a->psi_sm = g.K <= 4 && (pass == IL_NORMAL || pass == IL_FWD_PROJ);
  const size_t ts = ((size_t)a->RA * a->qs + 1) & ~(size_t)1;
  *smem = sizeof(float2) * (((size_t)g.ny + 1) / 2 * 2 + (fwd ? 2 : 1) * ts) + sizeof(int) * g.ny +
          (a->psi_sm ? sizeof(float) * g.P * g.ny * W : 0);
  return *smem <= 220 * 1024;
}
// radices and rows per band of a row pass: about eight lines, at most kRowThreads threads
bool row_any_plan(const Geom& g, AnyRow* a) {
  if (g.M > 2 || !two_radices(g.nz, kMaxImage, true, &a->RI, &a->RT)) return false;
  const int items = std::max(a->RI, a->RT);
  a->rows = std::max(1, std::min(8 / g.K, kRowThreads / (items * g.K)));
  const int nl = g.K * a->rows;
  a->xs = padded(a->RT * nl, nl);
  return items * nl <= kRowThreads;
}
size_t row_any_smem(const Geom& g, const AnyRow& a) {
  return sizeof(float2) * (g.nz + (((size_t)a.RI * a.xs + 1) & ~(size_t)1) + 2 * (size_t)g.M * a.rows * g.nz);
}

}  // namespace

bool any_col_supported(const Geom& g) {
  AnyCol a{};
  size_t sm = 0;
  const long long nsc = (long long)g.S * g.C;
  return nsc * (g.nz / 2) < 0x7fffffffLL && col_any_plan(g, g.nz % 4 ? 2 : 4, IL_NORMAL, &a, &sm);
}
bool any_row_supported(const Geom& g) {
  AnyRow a{};
  return row_any_plan(g, &a) && row_any_smem(g, a) <= 200 * 1024;
}

cudaError_t launch_col_any(const Geom& g, int W, IlPass pass, const float2* tw_y, const float* psi, const float2* in,
                           float2* out, cudaStream_t st) {
  AnyCol a{};
  size_t sm = 0;
  if (!col_any_plan(g, W, pass, &a, &sm)) return cudaErrorNotSupported;
  const int threads = col_threads(g.K * W, std::max(a.RA, a.RB));
  const long long nsc = (long long)g.S * g.C, ntiles = nsc * (g.nz / W);
  const bool fwd = pass == IL_NORMAL || pass == IL_FWD_PROJ || pass == IL_FWD_RAW;
  auto kern = g.K <= 4 ? (fwd ? k_col_any<4, true> : k_col_any<4, false>) : (fwd ? k_col_any<8, true> : k_col_any<8, false>);
  int nsm = 0, per = 0;
  cudaError_t e = smem_optin((const void*)kern, 220 * 1024);
  if (e == cudaSuccess) e = sm_count(&nsm);
  if (e == cudaSuccess) e = ctas_per_sm((const void*)kern, threads, sm, &per);
  if (e != cudaSuccess) return e;
  const int grid = (int)std::min<long long>(ntiles, (long long)nsm * per);
  return launch_pdl(kern, dim3(grid), threads, sm, st, g, a, tw_y, psi, in, out, (int)nsc, (int)ntiles);
}

template <int MODE, int MC>
static cudaError_t row_any_go(const Geom& g, const AnyRow& a, const float2* tw, const float2* maps, const float2* x,
                              float2* t, float2* out, cudaStream_t st) {
  const cudaError_t e = smem_optin((const void*)k_row_any<MODE, MC>, 200 * 1024);
  if (e != cudaSuccess) return e;
  const int threads = (g.K * a.rows * std::max(a.RI, a.RT) + 31) / 32 * 32;
  dim3 grid((g.ny + a.rows - 1) / a.rows, g.S);
  return launch_pdl(k_row_any<MODE, MC>, grid, threads, row_any_smem(g, a), st, g, a, tw, maps, x, t, out);
}

cudaError_t launch_row_any(const Geom& g, RowMode mode, int W, int trb, const float2* tw_z, const float2* maps,
                           const float2* x, float2* t, float2* out, cudaStream_t st) {
  AnyRow a{};
  a.W = W;
  a.trb = trb;
  if (!row_any_plan(g, &a)) return cudaErrorNotSupported;
  if (mode == ROW_FWD)
    return g.M == 1 ? row_any_go<ROW_FWD, 1>(g, a, tw_z, maps, x, t, out, st)
                    : row_any_go<ROW_FWD, 2>(g, a, tw_z, maps, x, t, out, st);
  return g.M == 1 ? row_any_go<ROW_ADJ, 1>(g, a, tw_z, maps, x, t, out, st)
                  : row_any_go<ROW_ADJ, 2>(g, a, tw_z, maps, x, t, out, st);
}

}  // namespace t2sh
