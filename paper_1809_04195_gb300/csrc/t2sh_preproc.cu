// Host side of the pre-processing entry points (t2sh_coil_compression, t2sh_preprocess):
// argument checks, the table of the sparse lines by phase encode, stream-ordered scratch.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/t2sh.h"
#include "t2sh_plan.h"

namespace t2sh {
bool fft_plan_for(int n, FftPlan& p);
void set_last_error(const char* msg);
}  // namespace t2sh

using namespace t2sh;

namespace {

t2sh_status fail(t2sh_status s, const char* msg) {
  set_last_error(msg);
  return s;
}

#define PP_CK(call)                                                   \
  do {                                                                \
    cudaError_t e_ = (call);                                          \
    if (e_ != cudaSuccess) return fail(T2SH_ECUDA, cudaGetErrorString(e_)); \
  } while (0)

t2sh_status check_sparse(const t2sh_sparse* sp) {
  if (!sp || !sp->t || !sp->ky || !sp->kz) return fail(T2SH_EINVAL, "sparse description or index array is NULL");
  if (sp->nlines < 1 || sp->nchan < 1 || sp->nx < 2 || sp->ny < 1 || sp->nz < 1 || sp->nechoes < 1)
    return fail(T2SH_EINVAL, "nlines, nchan, nx, ny, nz, nechoes must be positive (nx >= 2)");
  if (sp->nchan > kMaxChan) return fail(T2SH_EINVAL, "nchan must be <= 32");
  if ((long long)sp->nechoes * sp->ny * sp->nz > (1LL << 31)) return fail(T2SH_EINVAL, "mask too large");
  for (int j = 0; j < sp->nlines; ++j)
    if (sp->t[j] < 0 || sp->t[j] >= sp->nechoes || sp->ky[j] < 0 || sp->ky[j] >= sp->ny || sp->kz[j] < 0 ||
        sp->kz[j] >= sp->nz)
      return fail(T2SH_EINVAL, "a line's (t, ky, kz) index is out of range");
  return T2SH_OK;
}

// The lines grouped (stably) by phase encode ky nz + kz: pixel p owns order[off[p]] ..
// order[off[p + 1] - 1].  A counting sort: two passes over the lines (a comparison sort of the
// Table I scan's 35,777 lines took 2 ms of host time per call).
struct Groups {
  std::vector<int> order, t_sorted, off;
};
// the window [y0, y0 + ny) x [z0, z0 + nz) of phase encodes; lines outside it are left out
void build_groups(const t2sh_sparse* sp, int y0, int z0, int ny, int nz, Groups& s) {
  const int n = sp->nlines;
  const size_t N = (size_t)ny * nz;
  auto pixel = [&](int j, size_t* p) {
    const int y = sp->ky[j] - y0, z = sp->kz[j] - z0;
    *p = (size_t)y * nz + z;
    return y >= 0 && y < ny && z >= 0 && z < nz;
  };
  size_t p;
  s.off.assign(N + 1, 0);
  for (int j = 0; j < n; ++j)
    if (pixel(j, &p)) ++s.off[p + 1];
  for (size_t i = 0; i < N; ++i) s.off[i + 1] += s.off[i];
  std::vector<int> next(s.off.begin(), s.off.end() - 1);
  s.order.resize(s.off[N]);
  s.t_sorted.resize(s.off[N]);
  for (int j = 0; j < n; ++j)
    if (pixel(j, &p)) {
      const int q = next[p]++;
      s.order[q] = j;
      s.t_sorted[q] = sp->t[j];
    }
}

// Stream-ordered scratch, freed in stream order.  The first kKeepScratch bytes of a call come from the
// library's pool, which keeps them for the next call or plan (t2sh_release_cached returns them), so that
// most calls map no fresh pages: the Table I scan (0.6 GB) 2.3 ms, 3.6 with the device's default pool, which
// gives its memory back at the next synchronisation.  What goes beyond comes from that one, so a call leaves no
// more than that behind.  Host tables are packed into one buffer and cross in one copy.
constexpr size_t kKeepScratch = (size_t)1 << 30;
struct Scratch {
  cudaStream_t st;
  size_t kept = 0;
  std::vector<void*> ptrs;
  std::vector<unsigned char> host;
  unsigned char* dev = nullptr;
  explicit Scratch(cudaStream_t s) : st(s) { ptrs.reserve(8); }
  template <typename T>
  cudaError_t alloc(T** p, size_t n) {
    void* q = nullptr;
    const size_t b = n ? n * sizeof(T) : 16;
    cudaMemPool_t pool = b <= kKeepScratch - kept ? library_pool() : nullptr;
    cudaError_t e = pool ? cudaMallocFromPoolAsync(&q, b, pool, st) : cudaMallocAsync(&q, b, st);
    if (e != cudaSuccess && pool) {  // hand the pool's unused memory back and try once more
      cudaGetLastError();
      cudaStreamSynchronize(st);
      cudaMemPoolTrimTo(pool, 0);
      e = cudaMallocFromPoolAsync(&q, b, pool, st);
    }
    if (e == cudaSuccess) {
      if (pool) kept += b;
      ptrs.push_back(q);
      *p = static_cast<T*>(q);
    } else {
      cudaGetLastError();  // reported here: not to be met again by the next launch
    }
    return e;
  }
  // place of n values in the packed tables
  template <typename T>
  size_t add(const T* v, size_t n) {
    const size_t at = (host.size() + 255) / 256 * 256;
    host.resize(at + n * sizeof(T));
    if (n) std::memcpy(host.data() + at, v, n * sizeof(T));
    return at;
  }
  cudaError_t upload() {
    cudaError_t e = alloc(&dev, host.size());
    if (e == cudaSuccess) e = cudaMemcpyAsync(dev, host.data(), host.size(), cudaMemcpyHostToDevice, st);
    return e;
  }
  template <typename T>
  const T* table(size_t at) const {
    return reinterpret_cast<const T*>(dev + at);
  }
  ~Scratch() {
    for (void* q : ptrs) cudaFreeAsync(q, st);
  }
};

bool fft_size_ok(int n) {
  if (n % 2) return false;
  for (int p : {2, 3, 5, 13})
    while (n % p == 0) n /= p;
  return n == 1;
}

}  // namespace

extern "C" {

t2sh_status t2sh_coil_compression(const t2sh_sparse* sp, const void* lines, int32_t window, int32_t ncomp,
                                  void* w_out, void* stream) {
  t2sh_status s = check_sparse(sp);
  if (s != T2SH_OK) return s;
  if (!lines || !w_out) return fail(T2SH_EINVAL, "NULL argument");
  if (ncomp < 1 || ncomp > sp->nchan) return fail(T2SH_EINVAL, "ncomp must be in [1, nchan]");
  if (window < 1 || window > sp->nx || window > sp->ny || window > sp->nz)
    return fail(T2SH_EINVAL, "window must be in [1, min(nx, ny, nz)]");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  try {
    Groups sg;
    build_groups(sp, sp->ny / 2 - window / 2, sp->nz / 2 - window / 2, window, window, sg);
    std::vector<int> wpix;  // sampled phase encodes of the window
    for (int p = 0; p < window * window; ++p)
      if (sg.off[p + 1] > sg.off[p]) wpix.push_back(p);
    if (wpix.empty()) return fail(T2SH_EINVAL, "no line falls in the calibration window");
    Scratch sc(st);
    int* err = nullptr;
    float2* X = nullptr;
    double* G = nullptr;
    const long long npts = (long long)wpix.size() * window;
    const size_t a_order = sc.add(sg.order.data(), sg.order.size()), a_off = sc.add(sg.off.data(), sg.off.size()),
                 a_w = sc.add(wpix.data(), wpix.size());
    PP_CK(sc.upload());
    PP_CK(sc.alloc(&X, (size_t)npts * sp->nchan));
    PP_CK(sc.alloc(&G, 2 * (size_t)sp->nchan * sp->nchan));
    PP_CK(sc.alloc(&err, 1));
    PP_CK(cudaMemsetAsync(err, 0, sizeof(int), st));
    PP_CK(launch_calib(static_cast<const float2*>(lines), sp->nchan, sp->nx, sc.table<int>(a_order),
                       sc.table<int>(a_off), sc.table<int>(a_w), (int)wpix.size(), window, X, st));
    PP_CK(launch_gram_eig(X, npts, sp->nchan, ncomp, G, static_cast<float2*>(w_out), err, st));
    int herr = 0;
    PP_CK(cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, st));
    PP_CK(cudaStreamSynchronize(st));
    if (herr) return fail(T2SH_ECUDA, "the channel eigendecomposition did not converge");
  } catch (const std::bad_alloc&) {
    return fail(T2SH_ENOMEM, "host allocation failed");
  }
  return T2SH_OK;
}

t2sh_status t2sh_preprocess(const t2sh_sparse* sp, const void* lines, const void* w, int32_t ncomp, const float* phi,
                            int32_t nbasis, void* ytil_out, uint8_t* mask_out, void* stream) {
  t2sh_status s = check_sparse(sp);
  if (s != T2SH_OK) return s;
  if (!lines || !w || !phi || !ytil_out || !mask_out) return fail(T2SH_EINVAL, "NULL argument");
  if (ncomp < 1 || ncomp > sp->nchan) return fail(T2SH_EINVAL, "ncomp must be in [1, nchan]");
  if (nbasis < 1 || nbasis > kMaxK || nbasis > sp->nechoes) return fail(T2SH_EINVAL, "nbasis must be in [1, min(8, nechoes)]");
  if (!fft_size_ok(sp->nx) || sp->nx > 8192) return fail(T2SH_EINVAL, "nx must be even, a product of 2, 3, 5 and 13, <= 8192");
  FftPlan px{};
  if (!fft_plan_for(sp->nx, px)) return fail(T2SH_EINVAL, "no radix plan for nx");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  try {
    Groups sg;
    build_groups(sp, 0, 0, sp->ny, sp->nz, sg);
    std::vector<float2> tw(sp->nx);
    for (int m = 0; m < sp->nx; ++m) {
      const double a = -2.0 * 3.14159265358979323846 * m / sp->nx;
      tw[m] = make_float2((float)std::cos(a), (float)std::sin(a));
    }
    Scratch sc(st);
    float2* yh = nullptr;
    const size_t n = sp->nlines;
    const size_t a_order = sc.add(sg.order.data(), n), a_ts = sc.add(sg.t_sorted.data(), n),
                 a_off = sc.add(sg.off.data(), sg.off.size()), a_t = sc.add(sp->t, n), a_ky = sc.add(sp->ky, n),
                 a_kz = sc.add(sp->kz, n), a_tw = sc.add(tw.data(), tw.size());
    PP_CK(sc.upload());
    PP_CK(sc.alloc(&yh, (size_t)sp->nlines * ncomp * sp->nx));
    PP_CK(cudaMemsetAsync(mask_out, 0, (size_t)sp->nechoes * sp->ny * sp->nz, st));
    PP_CK(launch_compress_readout(static_cast<const float2*>(lines), static_cast<const float2*>(w), sp->nlines,
                                  sp->nchan, ncomp, px, sc.table<float2>(a_tw), yh, st));
    PP_CK(launch_project_lines(yh, ncomp, sp->nx, sc.table<int>(a_order), sc.table<int>(a_ts), sc.table<int>(a_off),
                               phi, nbasis, sp->ny, sp->nz, static_cast<float2*>(ytil_out), st));
    PP_CK(launch_mark_mask(sc.table<int>(a_t), sc.table<int>(a_ky), sc.table<int>(a_kz), sp->nlines, sp->ny, sp->nz,
                           mask_out, st));
  } catch (const std::bad_alloc&) {
    return fail(T2SH_ENOMEM, "host allocation failed");
  }
  return T2SH_OK;
}

}  // extern "C"
