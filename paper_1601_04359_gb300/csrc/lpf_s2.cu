// Two-point probability function of a periodic image (Sec. 2.1), the
// baseline descriptor the paper compares the lineal path function with:
//   S2_p(x, y) = 1/(W H) * IDFT( DFT(chi_p) * conj(DFT(chi_p)) )(x, y)
// with chi_p the indicator of phase p and IDFT normalised by 1/(W H); this
// equals the direct autocorrelation sum of Eq. (S2dis), a whole number over
// W H.
//
// That whole number is computed exactly, by number-theoretic transforms: the
// DFT over the integers mod p = 119 * 2^23 + 1, whose roots of unity have
// every power-of-two order up to 2^23 (Pollard, "The fast Fourier transform
// in a finite field", 1971); counts are below 2^26 < p, so the result mod p is
// the result.  Extents that are powers of two are transformed as they are;
// others are padded with zeros to at least twice their length, and the linear
// correlation is folded onto the period.  Three kernels:
//   rows     indicator and row transforms (decimation in frequency, so the
//            spectrum stays in bit-reversed order and nothing is permuted)
//   columns  a block takes the columns kx and -kx: transforms along y, the
//            products F(ky, kx) F(-ky, -kx), one inverse transform (that of
//            column -kx is its mirror image), the fold along y, rows 0 .. H/2
//   back     inverse row transforms of those rows, fold along x, division,
//            and the point-mirrored half
// Everything stays in 32-bit integers at the full integer rate; double
// precision runs at 1/64 of it on this chip, and cuFFT's transforms took 120
// of 139 us at 512x512 in seven launches.  Measured, 512x512: 139 -> 28.7 us
// (rows 5.7, columns 9.3, back 9.2; bound by the latency of the 9 to 18
// butterfly stages, 40e6 integer operations over 1.5 MB in L2).
//
// Large images take cuFFT's double-precision real-to-complex / complex-to-real FFTs; the
// indicator, the power spectrum and the scaling are this library's kernels,
// plans and the spectrum buffer are cached per device and image size.
#include <cufft.h>

#include <algorithm>
#include <atomic>
#include <mutex>
#include <vector>

#include "../../include/lpf.h"
#include "lpf_state.hpp"

namespace lpf {

// ---- arithmetic mod p (Montgomery form, factor 2^32) -----------------------

constexpr uint32_t kP = 998244353u;          // 119 * 2^23 + 1, primitive root 3
constexpr uint64_t mod_pow(uint64_t b, uint64_t e) {
  uint64_t r = 1;
  for (; e; e >>= 1, b = b * b % kP)
    if (e & 1) r = r * b % kP;
  return r;
}
constexpr uint32_t neg_inverse() {           // -1 / p mod 2^32 (Newton steps double the correct bits)
  uint32_t x = 1;
  for (int i = 0; i < 5; ++i) x *= 2u - kP * x;
  return 0u - x;
}
constexpr uint32_t kNegInv = neg_inverse();
constexpr uint32_t kOne = (uint32_t)((uint64_t(1) << 32) % kP);
constexpr int kMaxLog = 12;                  // transforms of up to 4096
// Roots of unity of order 2^m, m = 0 .. kMaxLog, in Montgomery form.
struct Roots {
  uint32_t w[kMaxLog + 1];
};
constexpr Roots make_roots() {
  Roots r{};
  for (int m = 0; m <= kMaxLog; ++m) r.w[m] = (uint32_t)((mod_pow(3, (kP - 1) >> m) << 32) % kP);
  return r;
}
__constant__ Roots c_roots = make_roots();

// a b / 2^32 mod p, in [0, p).
__device__ __forceinline__ uint32_t mont_mul(uint32_t a, uint32_t b) {
  const uint32_t lo = a * b, hi = __umulhi(a, b);
  // lo + (lo kNegInv) p is 0 mod 2^32: its low words cancel, with a carry unless lo = 0
  const uint32_t u = hi + __umulhi(lo * kNegInv, kP) + (lo != 0u);
  return u >= kP ? u - kP : u;
}
__device__ __forceinline__ uint32_t mod_add(uint32_t a, uint32_t b) {
  const uint32_t c = a + b;
  return c >= kP ? c - kP : c;
}
__device__ __forceinline__ uint32_t mod_sub(uint32_t a, uint32_t b) { return a >= b ? a - b : a + kP - b; }

// tw[k] = w^k, k < n / 2, w the root of order n = 2^lg; every thread calls it.
__device__ __forceinline__ void make_twiddles(uint32_t* tw, int lg) {
  for (int k = threadIdx.x; k < (1 << lg) >> 1; k += blockDim.x) {
    uint32_t r = kOne;
    for (int b = 0; b < lg - 1; ++b)
      if ((k >> b) & 1) r = mont_mul(r, c_roots.w[lg - b]);
    tw[k] = r;
  }
}

// Forward transforms of n_seq sequences of 2^lg values (natural order in,
// bit-reversed out), and back (bit-reversed in, natural out, unscaled; the
// sequences 2^(lg + gap) apart).  Every thread of the block calls them, after
// a barrier; they end with one.
__device__ __forceinline__ void forward_transforms(uint32_t* x, int n_seq, int lg, const uint32_t* tw) {
  const int half = (1 << lg) >> 1;
  for (int s = 0; s < lg; ++s) {
    const int ll = lg - 1 - s;  // log2 of the butterfly distance
    for (int t = threadIdx.x; t < n_seq * half; t += blockDim.x) {
      const int j = t & ((1 << ll) - 1), i0 = ((t >> ll) << (ll + 1)) + j;
      const uint32_t u = x[i0], v = x[i0 + (1 << ll)];
      x[i0] = mod_add(u, v);
      x[i0 + (1 << ll)] = mont_mul(mod_sub(u, v), tw[j << s]);
    }
    __syncthreads();
  }
}
__device__ __forceinline__ void inverse_transforms(uint32_t* x, int n_seq, int lg, int gap, const uint32_t* tw) {
  const int half = (1 << lg) >> 1;
  for (int s = lg - 1; s >= 0; --s) {
    const int ll = lg - 1 - s;
    for (int t = threadIdx.x; t < n_seq * half; t += blockDim.x) {
      const int seq = t >> (lg - 1), in = t & (half - 1), j = in & ((1 << ll) - 1);
      const int i0 = (seq << (lg + gap)) + ((in >> ll) << (ll + 1)) + j;
      const int e = j << s;  // w^-e = -w^(n/2 - e)
      const uint32_t u = x[i0], v = x[i0 + (1 << ll)];
      const uint32_t m = e ? mont_mul(v, kP - tw[half - e]) : v;
      x[i0] = mod_add(u, m);
      x[i0 + (1 << ll)] = mod_sub(u, m);
    }
    __syncthreads();
  }
}

// Bit-reversed position of frequency -k, for position i of frequency k.
__device__ __forceinline__ int mirrored_position(int i, int lg) {
  if (lg == 0) return 0;
  const uint32_t k = __brev((uint32_t)i) >> (32 - lg);
  return (int)(__brev((0u - k) & ((1u << lg) - 1u)) >> (32 - lg));
}

constexpr int kNttThreads = 256;

// A[y][.] = transform of row y's indicator, padded to 2^lgw (n_seq rows per block).
__global__ void __launch_bounds__(kNttThreads) s2_rows_kernel(const uint8_t* __restrict__ img, int H, int W, int phase,
                                                              int lgw, int n_seq, uint32_t* __restrict__ A) {
  extern __shared__ uint32_t sx[];
  const int P = 1 << lgw, y0 = blockIdx.x * n_seq;
  uint32_t* tw = sx + n_seq * P;
  make_twiddles(tw, lgw);
  for (int t = threadIdx.x; t < n_seq * P; t += blockDim.x) {
    const int y = y0 + (t >> lgw), x = t & (P - 1);
    sx[t] = y < H && x < W && (img[(size_t)y * W + x] != 0) == (phase != 0) ? kOne : 0u;
  }
  __syncthreads();
  forward_transforms(sx, n_seq, lgw, tw);
  for (int t = threadIdx.x; t < n_seq * P; t += blockDim.x)
    if (y0 + (t >> lgw) < H) A[(size_t)y0 * P + t] = sx[t];
}

// Column pair q (0 .. P_W / 2) of the bit-reversed spectrum: positions i and
// of -k (equal for k = 0 and P_W / 2).  Positions in [2^m, 2^(m+1)) mirror
// onto 3 * 2^m - 1 - i.
__device__ __forceinline__ void column_pair(int q, int& i, int& j) {
  if (q < 2) { i = j = q; return; }
  const int m = 32 - __clz(q - 1);  // floor(log2(q - 1)) + 1
  i = (1 << m) + (q - 1 - (1 << (m - 1)));
  j = 3 * (1 << m) - 1 - i;
}

// B[y][.], y = 0 .. H / 2: the correlation along y of every column of the
// spectrum (n_pair column pairs per block).
__global__ void __launch_bounds__(kNttThreads) s2_columns_kernel(const uint32_t* __restrict__ A, int H, int lgw,
                                                                 int lgh, int n_pair, uint32_t* __restrict__ B) {
  extern __shared__ uint32_t sx[];
  const int PW = 1 << lgw, PH = 1 << lgh, n_q = PW / 2 + 1;
  uint32_t* tw = sx + 2 * n_pair * PH;
  make_twiddles(tw, lgh);
  for (int t = threadIdx.x; t < 2 * n_pair * PH; t += blockDim.x) {
    const int c = t % (2 * n_pair), y = t / (2 * n_pair);  // columns fastest: neighbours in memory
    const int q = blockIdx.x * n_pair + (c >> 1);
    uint32_t v = 0u;
    if (q < n_q && y < H) {
      int i, j;
      column_pair(q, i, j);
      v = A[(size_t)y * PW + ((c & 1) ? j : i)];
    }
    sx[c * PH + y] = v;
  }
  __syncthreads();
  forward_transforms(sx, 2 * n_pair, lgh, tw);
  // F(k) F(-k), in place of the first column of each pair
  for (int t = threadIdx.x; t < n_pair * PH; t += blockDim.x) {
    const int c = t >> lgh, r = t & (PH - 1);
    sx[2 * c * PH + r] = mont_mul(sx[2 * c * PH + r], sx[(2 * c + 1) * PH + mirrored_position(r, lgh)]);
  }
  __syncthreads();
  inverse_transforms(sx, n_pair, lgh, 1, tw);
  const bool fold = H != PH;
  for (int t = threadIdx.x; t < 2 * n_pair * (H / 2 + 1); t += blockDim.x) {
    const int c = t % (2 * n_pair), y = t / (2 * n_pair);
    const int q = blockIdx.x * n_pair + (c >> 1);
    if (q >= n_q) continue;
    int i, j;
    column_pair(q, i, j);
    if ((c & 1) && i == j) continue;
    const uint32_t* g = sx + (c & ~1) * PH;
    const int s = (c & 1) ? -y : y;  // column -kx is the mirror image along y
    uint32_t v = g[s & (PH - 1)];
    if (fold) v = mod_add(v, g[((c & 1) ? H - y : y - H) & (PH - 1)]);
    B[(size_t)y * PW + ((c & 1) ? j : i)] = v;
  }
}

// S2 rows y and H - y, y = 0 .. H / 2: inverse row transforms, fold, scale.
// unscale = 1 / (P_W P_H) mod p (not in Montgomery form: multiplying by it
// also takes the value out of it).
__global__ void __launch_bounds__(kNttThreads) s2_back_kernel(const uint32_t* __restrict__ B, int H, int W, int lgw,
                                                              int n_seq, uint32_t unscale, float* __restrict__ s2) {
  extern __shared__ uint32_t sx[];
  const int P = 1 << lgw, y0 = blockIdx.x * n_seq, rows = H / 2 + 1;
  uint32_t* tw = sx + n_seq * P;
  make_twiddles(tw, lgw);
  for (int t = threadIdx.x; t < n_seq * P; t += blockDim.x)
    sx[t] = y0 + (t >> lgw) < rows ? B[(size_t)y0 * P + t] : 0u;
  __syncthreads();
  inverse_transforms(sx, n_seq, lgw, 0, tw);
  const double N = (double)H * (double)W;
  const bool fold = W != P;
  for (int t = threadIdx.x; t < n_seq * W; t += blockDim.x) {
    const int r = t / W, x = t - r * W, y = y0 + r;
    if (y >= rows) continue;
    const uint32_t* g = sx + (r << lgw);
    uint32_t v = g[x];
    if (fold) v = mod_add(v, g[(x - W) & (P - 1)]);
    const float f = (float)((double)mont_mul(v, unscale) / N);
    s2[(size_t)y * W + x] = f;
    // C(-d) = C(d): row H - y (for y = 0 and H / 2 the mirrored row is the row itself)
    if (y > 0 && 2 * y < H) s2[(size_t)(H - y) * W + (x ? W - x : 0)] = f;
  }
}

// The 1x1 image: S2(0) = chi (three launches and a work area took 13 us, this 8).
__global__ void s2_single_kernel(const uint8_t* __restrict__ img, int phase, float* __restrict__ s2) {
  *s2 = (*img != 0) == (phase != 0) ? 1.0f : 0.0f;
}

// ---- cuFFT path -------------------------------------------------------------

__global__ void s2_indicator_kernel(const uint8_t* __restrict__ img, int64_t n, int phase, double* __restrict__ x) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] = (img[i] != 0) == (phase != 0) ? 1.0 : 0.0;
}

// X <- |X|^2 (imaginary part 0), in place.
__global__ void s2_power_kernel(cufftDoubleComplex* __restrict__ X, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const cufftDoubleComplex z = X[i];
    X[i] = make_cuDoubleComplex(z.x * z.x + z.y * z.y, 0.0);
  }
}

// s2 = x * scale, double -> float.
__global__ void s2_scale_kernel(const double* __restrict__ x, int64_t n, double scale, float* __restrict__ s2) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    s2[i] = (float)(x[i] * scale);
}

namespace {
struct S2Plan {
  int dev = -1, H = 0, W = 0;
  cufftHandle fwd = 0, inv = 0;
  double* x = nullptr;                 // [H][W]
  cufftDoubleComplex* X = nullptr;     // [H][W/2+1]
};
std::mutex g_s2_mu;
std::vector<S2Plan> g_s2_plans;

int s2_plan(int dev, int H, int W, S2Plan*& out) {
  for (S2Plan& p : g_s2_plans)
    if (p.dev == dev && p.H == H && p.W == W) { out = &p; return LPF_OK; }
  S2Plan p;
  p.dev = dev;
  p.H = H;
  p.W = W;
  // a single row or column is a 1-D transform of the other extent
  const int n1 = H == 1 ? W : H;
  const bool one_d = H == 1 || W == 1;
  if (one_d) {
    if (cufftPlan1d(&p.fwd, n1, CUFFT_D2Z, 1) != CUFFT_SUCCESS) return LPF_ECUDA;
    if (cufftPlan1d(&p.inv, n1, CUFFT_Z2D, 1) != CUFFT_SUCCESS) { cufftDestroy(p.fwd); return LPF_ECUDA; }
  } else {
    if (cufftPlan2d(&p.fwd, H, W, CUFFT_D2Z) != CUFFT_SUCCESS) return LPF_ECUDA;
    if (cufftPlan2d(&p.inv, H, W, CUFFT_Z2D) != CUFFT_SUCCESS) { cufftDestroy(p.fwd); return LPF_ECUDA; }
  }
  cudaError_t e = cudaMalloc(&p.x, sizeof(double) * (size_t)H * W);
  if (e == cudaSuccess) e = cudaMalloc(&p.X, sizeof(cufftDoubleComplex) * (size_t)(one_d ? n1 / 2 + 1 : H * (W / 2 + 1)));
  if (e != cudaSuccess) {
    cufftDestroy(p.fwd);
    cufftDestroy(p.inv);
    cudaFree(p.x);
    return set_cuda_error(e);
  }
  g_s2_plans.push_back(p);
  out = &g_s2_plans.back();
  return LPF_OK;
}

// The transforms' work area: stream-ordered allocations from a pool of the
// library's own per device, which keeps at most 32 MiB between calls (so calls
// on several threads and streams never share a buffer, and none is mapped
// anew on each call).
constexpr uint64_t kNttPoolBytes = uint64_t(32) << 20;
std::mutex g_ntt_mu;
cudaMemPool_t g_ntt_pool[64] = {};

int ntt_pool(int dev, cudaMemPool_t* out) {
  if (dev < 0 || dev >= 64) return LPF_EUNSUPPORTED;
  std::lock_guard<std::mutex> lock(g_ntt_mu);
  if (!g_ntt_pool[dev]) {
    cudaMemPoolProps props = {};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool;
    cudaError_t e = cudaMemPoolCreate(&pool, &props);
    if (e != cudaSuccess) return set_cuda_error(e);
    uint64_t keep = kNttPoolBytes;
    e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e != cudaSuccess) { cudaMemPoolDestroy(pool); return set_cuda_error(e); }
    g_ntt_pool[dev] = pool;
  }
  *out = g_ntt_pool[dev];
  return LPF_OK;
}

// log2 of the transform length for an extent: itself if a power of two, else
// the next one from twice the extent (room for every lag of either sign).
int ntt_log(int n) {
  int lg = 0;
  while ((1 << lg) < n) ++lg;
  if ((1 << lg) != n) ++lg;
  return lg;
}

// A call recorded into a graph takes an area of its own, which the graph holds
// (as a user object: so do its copies and the executables made from it, while
// they run too): two recorded calls may run side by side, from two graphs or
// on two branches of one.  An allocation in stream order would become a node of
// the graph, which then could not be copied or instantiated twice; so the area
// comes from the pool on a stream of the library's own and goes back there with
// the first call after the last graph that held it.
struct NttArea {
  uint32_t* p = nullptr;
  std::atomic<bool> idle{false};  // set by the runtime's thread, which must not call CUDA
};
struct NttRecorded {
  cudaStream_t stream = nullptr;
  std::vector<NttArea*> areas;
};
NttRecorded g_ntt_recorded[64];

// Areas that no graph holds any more back to the pool (g_ntt_mu held).
void give_back_areas(NttRecorded& r) {
  for (size_t i = 0; i < r.areas.size();) {
    if (r.areas[i]->idle.load(std::memory_order_acquire)) {
      cudaFreeAsync(r.areas[i]->p, r.stream);
      delete r.areas[i];
      r.areas[i] = r.areas.back();
      r.areas.pop_back();
    } else {
      ++i;
    }
  }
}

cudaError_t new_recorded_area(NttRecorded& r, cudaMemPool_t pool, cudaGraph_t graph, size_t bytes, uint32_t** out) {
  cudaError_t e = cudaSuccess;
  if (!r.stream && (e = cudaStreamCreateWithFlags(&r.stream, cudaStreamNonBlocking)) != cudaSuccess) return e;
  give_back_areas(r);
  uint32_t* p = nullptr;
  if ((e = cudaMallocFromPoolAsync(reinterpret_cast<void**>(&p), bytes, pool, r.stream)) != cudaSuccess) return e;
  NttArea* area = new NttArea;
  area->p = p;
  cudaUserObject_t held = nullptr;
  e = cudaStreamSynchronize(r.stream);  // (the graph's kernels run on other streams)
  if (e == cudaSuccess)
    e = cudaUserObjectCreate(&held, area, [](void* a) { static_cast<NttArea*>(a)->idle.store(true, std::memory_order_release); },
                             1, cudaUserObjectNoDestructorSync);
  if (e != cudaSuccess) {
    cudaFreeAsync(p, r.stream);
    delete area;
    return e;
  }
  r.areas.push_back(area);
  if ((e = cudaGraphRetainUserObject(graph, held, 1, cudaGraphUserObjectMove)) != cudaSuccess)
    cudaUserObjectRelease(held, 1);  // (idle then)
  *out = p;
  return e;
}

int recorded_area(int dev, cudaStream_t s, size_t bytes, uint32_t** out) {
  cudaMemPool_t pool;
  if (int rc = ntt_pool(dev, &pool)) return rc;
  cudaStreamCaptureStatus cap;
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamGetCaptureInfo(s, &cap, nullptr, &graph);
  if (e != cudaSuccess) return set_cuda_error(e);
  if (cap != cudaStreamCaptureStatusActive) return set_cuda_error(cudaErrorStreamCaptureInvalidated);
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;  // (allocating is not part of what is recorded)
  if ((e = cudaThreadExchangeStreamCaptureMode(&mode)) != cudaSuccess) return set_cuda_error(e);
  {
    std::lock_guard<std::mutex> lock(g_ntt_mu);
    e = new_recorded_area(g_ntt_recorded[dev], pool, graph, bytes, out);
  }
  (void)cudaThreadExchangeStreamCaptureMode(&mode);
  return set_cuda_error(e);
}

int s2_ntt(int dev, const uint8_t* img, int H, int W, int phase, float* s2, cudaStream_t s) {
  const int lgw = ntt_log(W), lgh = ntt_log(H), PW = 1 << lgw, PH = 1 << lgh, rows = H / 2 + 1;
  const size_t bytes = sizeof(uint32_t) * (size_t)PW * (H + rows);
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(s, &cap);
  if (e != cudaSuccess) return set_cuda_error(e);
  const bool recorded = cap != cudaStreamCaptureStatusNone;
  uint32_t* A = nullptr;
  if (recorded) {
    if (int rc = recorded_area(dev, s, bytes, &A)) return rc;
  } else {
    cudaMemPool_t pool;
    if (int rc = ntt_pool(dev, &pool)) return rc;
    {
      std::lock_guard<std::mutex> lock(g_ntt_mu);
      give_back_areas(g_ntt_recorded[dev]);
    }
    e = cudaMallocFromPoolAsync(reinterpret_cast<void**>(&A), bytes, pool, s);
    if (e != cudaSuccess) return set_cuda_error(e);
  }
  uint32_t* B = A + (size_t)PW * H;
  (void)cudaGetLastError();
  // 1024 values per block where there are enough blocks, at least one
  // sequence (16 KB and its twiddles at 4096)
  const int n_seq = std::max(1, 1024 / PW), n_pair = std::max(1, 512 / PH);
  const size_t row_smem = ((size_t)n_seq * PW + PW / 2 + 1) * 4, col_smem = ((size_t)2 * n_pair * PH + PH / 2 + 1) * 4;
  s2_rows_kernel<<<(H + n_seq - 1) / n_seq, kNttThreads, row_smem, s>>>(img, H, W, phase, lgw, n_seq, A);
  s2_columns_kernel<<<(PW / 2 + n_pair) / n_pair, kNttThreads, col_smem, s>>>(A, H, lgw, lgh, n_pair, B);
  const uint32_t unscale = (uint32_t)mod_pow((uint64_t)PW * PH % kP, kP - 2);
  s2_back_kernel<<<(rows + n_seq - 1) / n_seq, kNttThreads, row_smem, s>>>(B, H, W, lgw, n_seq, unscale, s2);
  e = cudaGetLastError();
  if (!recorded) cudaFreeAsync(A, s);
  return set_cuda_error(e);
}
}  // namespace

}  // namespace lpf

extern "C" int s2_fft(const uint8_t* img_dev, int32_t H, int32_t W, int32_t phase, float* s2_dev,
                      lpf_stream_t stream) {
  if (!img_dev || !s2_dev || H < 1 || W < 1 || (int64_t)H * W > (1 << 26) || (phase != 0 && phase != 1))
    return LPF_EINVAL;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return lpf::set_cuda_error(e);
  if (H == 1 && W == 1) {
    (void)cudaGetLastError();
    lpf::s2_single_kernel<<<1, 1, 0, (cudaStream_t)stream>>>(img_dev, phase, s2_dev);
    return lpf::set_cuda_error(cudaGetLastError());
  }
  // up to 4096 per extent (one transform in shared memory) and 4 Mi values
  const int lgw = lpf::ntt_log(W), lgh = lpf::ntt_log(H);
  if (std::max(lgw, lgh) <= lpf::kMaxLog && lgw + lgh <= 22)
    return lpf::s2_ntt(dev, img_dev, H, W, phase, s2_dev, (cudaStream_t)stream);
  std::lock_guard<std::mutex> lock(lpf::g_s2_mu);
  lpf::S2Plan* p = nullptr;
  int rc = lpf::s2_plan(dev, H, W, p);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  if (cufftSetStream(p->fwd, s) != CUFFT_SUCCESS || cufftSetStream(p->inv, s) != CUFFT_SUCCESS) return LPF_ECUDA;
  const int64_t n = (int64_t)H * W;
  const int64_t nc = (H == 1 || W == 1) ? n / 2 + 1 : (int64_t)H * (W / 2 + 1);
  const int blocks = (int)std::min<int64_t>((n + 255) / 256, 4096);
  (void)cudaGetLastError();
  lpf::s2_indicator_kernel<<<blocks, 256, 0, s>>>(img_dev, n, phase, p->x);
  if (cufftExecD2Z(p->fwd, p->x, p->X) != CUFFT_SUCCESS) return LPF_ECUDA;
  lpf::s2_power_kernel<<<(int)std::min<int64_t>((nc + 255) / 256, 4096), 256, 0, s>>>(p->X, nc);
  if (cufftExecZ2D(p->inv, p->X, p->x) != CUFFT_SUCCESS) return LPF_ECUDA;
  // cuFFT's inverse is unnormalised: IDFT = Z2D / (W H); S2 = IDFT / (W H).
  const double scale = 1.0 / ((double)n * (double)n);
  lpf::s2_scale_kernel<<<blocks, 256, 0, s>>>(p->x, n, scale, s2_dev);
  return lpf::set_cuda_error(cudaGetLastError());
}
