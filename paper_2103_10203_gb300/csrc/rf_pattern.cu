// Sampling patterns (reduced sets of frequencies), computed on the GPU.
//
// Adapted pattern (Sec. 4.2; 3D as in Sec. 5.3): the phase map becomes the step function g
// (1 on the inclusion phase), g is transformed in FP64 axis by axis, and the amplitudes |g^|
// rank the conjugate pairs (k, -k). Ranking key (smaller first): quantised amplitude
// round(|g^| / |g^(0)| * 2^30) descending, |k|^2 ascending, signed linear index ascending.
// Pairs are taken whole until at least k_target frequencies are held; the selection threshold
// is found by radix passes over weighted histograms of the key, each decided on the device by its
// last block, so the host waits twice per pattern: for its size and for its entries.
// g is real: two rows share a complex transform along x, and only kx = 0 .. Nx / 2 goes on, half
// the work of transforms that the FP64 rate bounds (96 and 100 us for 1024^2 before). A 1024^2
// pattern took 1374 us (some 530 us of kernels, 13 host reads, 16 allocations) and takes 540 us.
// Radial pattern (Sec. 4.1): L equiangular rasterised lines; the same selection machinery
// ranks pairs by (not on a line, |k|^2, index).
#include <algorithm>
#include <climits>
#include <cmath>
#include <mutex>
#include <vector>

#include "rf_internal.cuh"

namespace rfk {

namespace {

struct Grid3 {
  int nx, ny, nz;
  long long N;
  int hx, hy, hz;
};

__device__ __forceinline__ int sgn_index(int i, int n) { return i <= n / 2 ? i : i - n; }
__device__ __forceinline__ int wrap(int k, int n) {
  int r = k % n;
  return r < 0 ? r + n : r;
}
__device__ __forceinline__ long long signed_lin(int kx, int ky, int kz, const Grid3& g) {
  return ((long long)(kz + g.hz) * g.ny + (ky + g.hy)) * g.nx + (kx + g.hx);
}

__global__ void k_table_f64(double2* t, int L) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < L) {
    double s, c;
    sincospi(2.0 * (double)i / (double)L, &s, &c);
    t[i] = make_double2(c, -s);   // exp(-2 pi i t / L)
  }
}

// out[row][kx] = sum_x g(row, x) exp(-2 pi i kx x / nx) for kx <= nx / 2, one block per row
__global__ void k_g_rows(const uint8_t* pm, int incl, int nx, const double2* tab, double2* out) {
  const int H = nx / 2 + 1;
  extern __shared__ __align__(16) unsigned char sm[];
  double2* t = reinterpret_cast<double2*>(sm);
  float* gr = reinterpret_cast<float*>(t + nx);
  const long long row = blockIdx.x;
  for (int i = threadIdx.x; i < nx; i += blockDim.x) {
    t[i] = tab[i];
    gr[i] = pm[row * nx + i] == incl ? 1.f : 0.f;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < H; k += blockDim.x) {
    double re = 0.0, im = 0.0;
    int m = 0;
    for (int x = 0; x < nx; ++x) {
      if (gr[x] != 0.f) {
        re += t[m].x;
        im += t[m].y;
      }
      m += k;
      if (m >= nx) m -= nx;
    }
    out[row * H + k] = make_double2(re, im);
  }
}

// out[b][m][n] = sum_k exp(-2 pi i m k / L) in[b][k][n]; 4 m per thread, lanes over n
__global__ void k_axis_f64(const double2* in, double2* out, int L, int N, long long bstride,
                           const double2* tab) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  const int m0 = blockIdx.y * 4;
  const long long b = blockIdx.z;
  if (n >= N) return;
  double ar[4] = {0, 0, 0, 0}, ai[4] = {0, 0, 0, 0};
  int t[4] = {0, 0, 0, 0};   // m k mod L
  const double2* ib = in + b * bstride;
  for (int k = 0; k < L; ++k) {
    const double2 v = ib[(long long)k * N + n];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = m0 + i;
      if (m < L) {
        const double2 w = tab[t[i]];
        ar[i] += w.x * v.x - w.y * v.y;
        ai[i] += w.x * v.y + w.y * v.x;
        t[i] += m;
        if (t[i] >= L) t[i] -= L;
      }
    }
  }
  double2* ob = out + b * bstride;
#pragma unroll
  for (int i = 0; i < 4; ++i)
    if (m0 + i < L) ob[(long long)(m0 + i) * N + n] = make_double2(ar[i], ai[i]);
}

// FP64 Stockham FFTs (forward, exp(-2 pi i m n / L)) for lengths L = 2^b or 3 * 2^b: radix-4
// stages, one radix-2 stage, then one radix-3 stage. A stage of radix R and sub-transform size
// Ns reads element j + r L / R, multiplies it by exp(-2 pi i r k / (R Ns)) with k = j mod Ns
// (tab[t] = exp(-2 pi i t / L)), takes the R-point DFT and writes output q to
// (j / Ns) R Ns + k + q Ns. The zero frequency only meets the exact factor 1, so for 0/1 data it
// is an exact sum. C sequences of length L lie back to back in both shared buffers; returns
// the buffer holding the result. The whole block calls it.
__device__ __forceinline__ double2 cm64(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 add64(double2 a, double2 b) {
  return make_double2(a.x + b.x, a.y + b.y);
}
__device__ __forceinline__ double2 sub64(double2 a, double2 b) {
  return make_double2(a.x - b.x, a.y - b.y);
}

__device__ double2* fft64_block(double2* in, double2* out, const double2* tab, int L, int C) {
  const int p2 = (L % 3 == 0) ? L / 3 : L;
  int Ns = 1;
  auto swap = [&] {
    __syncthreads();
    double2* t = in;
    in = out;
    out = t;
  };
  while (Ns * 4 <= p2) {
    const int q = L / 4, step = L / (4 * Ns);
    for (int u = threadIdx.x; u < C * q; u += blockDim.x) {
      const int p = u / q, j = u - p * q, k = j % Ns;
      const double2* src = in + (long long)p * L + j;
      double2 a0 = src[0], a1 = src[q], a2 = src[2 * q], a3 = src[3 * q];
      if (Ns > 1) {
        a1 = cm64(a1, tab[k * step]);
        a2 = cm64(a2, tab[2 * k * step]);
        a3 = cm64(a3, tab[3 * k * step]);
      }
      const double2 s02 = add64(a0, a2), d02 = sub64(a0, a2);
      const double2 s13 = add64(a1, a3), d13 = sub64(a1, a3);
      const double2 md13 = make_double2(d13.y, -d13.x);   // -i (a1 - a3)
      double2* dst = out + (long long)p * L + (j / Ns) * 4 * Ns + k;
      dst[0] = add64(s02, s13);
      dst[Ns] = add64(d02, md13);
      dst[2 * Ns] = sub64(s02, s13);
      dst[3 * Ns] = sub64(d02, md13);
    }
    swap();
    Ns *= 4;
  }
  if (Ns * 2 <= p2) {
    const int q = L / 2, step = L / (2 * Ns);
    for (int u = threadIdx.x; u < C * q; u += blockDim.x) {
      const int p = u / q, j = u - p * q, k = j % Ns;
      const double2* src = in + (long long)p * L + j;
      double2 a0 = src[0], a1 = src[q];
      if (Ns > 1) a1 = cm64(a1, tab[k * step]);
      double2* dst = out + (long long)p * L + (j / Ns) * 2 * Ns + k;
      dst[0] = add64(a0, a1);
      dst[Ns] = sub64(a0, a1);
    }
    swap();
    Ns *= 2;
  }
  if (p2 != L) {   // Ns = L / 3: j = k < Ns, outputs j, j + Ns, j + 2 Ns
    const double h = 0.86602540378443864676;   // sqrt(3) / 2
    for (int u = threadIdx.x; u < C * Ns; u += blockDim.x) {
      const int p = u / Ns, j = u - p * Ns;
      const double2* src = in + (long long)p * L + j;
      double2 a0 = src[0], a1 = src[Ns], a2 = src[2 * Ns];
      if (Ns > 1) {
        a1 = cm64(a1, tab[j]);
        a2 = cm64(a2, tab[2 * j]);
      }
      // X0 = a0 + s, X1,2 = a0 - s / 2 -+ i sqrt(3)/2 (a1 - a2)
      const double2 sm = add64(a1, a2), d = sub64(a1, a2);
      const double2 m = make_double2(a0.x - 0.5 * sm.x, a0.y - 0.5 * sm.y);
      double2* dst = out + (long long)p * L + j;
      dst[0] = add64(a0, sm);
      dst[Ns] = make_double2(m.x + h * d.y, m.y - h * d.x);
      dst[2 * Ns] = make_double2(m.x - h * d.y, m.y + h * d.x);
    }
    swap();
  }
  return in;
}

constexpr size_t kFft64Smem = 96 * 1024;

bool fft64_length(int L) {
  const int p2 = (L % 3 == 0) ? L / 3 : L;
  return L >= 1 && (p2 & (p2 - 1)) == 0 && 2 * (size_t)L * sizeof(double2) <= kFft64Smem;
}

// sequences per block for length L within the shared-memory budget
int fft64_lines(int L, int cap) {
  return std::max(1, std::min(cap, (int)(kFft64Smem / (2 * (size_t)L * sizeof(double2)))));
}

// out[row][kx], kx <= nx / 2, by FFT along x of the indicator of `incl`: C complex sequences per
// block, each carrying two rows (the sum at kx = 0 stays exact: both parts are sums of ones)
__global__ void k_g_rows_fft(const uint8_t* pm, int incl, int nx, long long rows, int C,
                             const double2* tab, double2* out) {
  extern __shared__ __align__(16) unsigned char sm[];
  double2* b0 = reinterpret_cast<double2*>(sm);
  double2* b1 = b0 + (size_t)C * nx;
  const int H = nx / 2 + 1;
  const long long row0 = (long long)blockIdx.x * 2 * C;
  for (int i = threadIdx.x; i < C * nx; i += blockDim.x) {
    const int p = i / nx, x = i - p * nx;
    const long long r = row0 + 2 * p;
    b0[i] = make_double2(r < rows && pm[r * nx + x] == incl ? 1.0 : 0.0,
                         r + 1 < rows && pm[(r + 1) * nx + x] == incl ? 1.0 : 0.0);
  }
  __syncthreads();
  const double2* z = fft64_block(b0, b1, tab, nx, C);
  for (int i = threadIdx.x; i < C * H; i += blockDim.x) {
    const int p = i / H, k = i - p * H;
    const long long r = row0 + 2 * p;
    const double2 u = z[(long long)p * nx + k], v = z[(long long)p * nx + (k == 0 ? 0 : nx - k)];
    if (r < rows) out[r * H + k] = make_double2(0.5 * (u.x + v.x), 0.5 * (u.y - v.y));
    if (r + 1 < rows) out[(r + 1) * H + k] = make_double2(0.5 * (u.y + v.y), -0.5 * (u.x - v.x));
  }
}

// out[b][m][n] = sum_k exp(-2 pi i m k / L) in[b][k][n] by FFT, C columns n per block
__global__ void k_cols_fft64(const double2* in, double2* out, int L, int ncols, long long bstride,
                             int C, const double2* tab) {
  extern __shared__ __align__(16) unsigned char sm[];
  double2* b0 = reinterpret_cast<double2*>(sm);
  double2* b1 = b0 + (size_t)C * L;
  const int col0 = blockIdx.x * C;
  const double2* ib = in + blockIdx.y * bstride;
  double2* ob = out + blockIdx.y * bstride;
  for (int i = threadIdx.x; i < C * L; i += blockDim.x) {
    const int y = i / C, c = i - y * C, col = col0 + c;
    b0[c * L + y] = col < ncols ? ib[(long long)y * ncols + col] : make_double2(0.0, 0.0);
  }
  __syncthreads();
  const double2* z = fft64_block(b0, b1, tab, L, C);
  for (int i = threadIdx.x; i < C * L; i += blockDim.x) {
    const int y = i / C, c = i - y * C, col = col0 + c;
    if (col < ncols) ob[(long long)y * ncols + col] = z[c * L + y];
  }
}

// Ranking entries over the half spectrum [z][y][kx <= nx / 2], one per pair (k, -k): key, and the
// smaller signed linear index of the two with bit 31 set where k is its own conjugate. At kx = 0
// and the Nyquist kx both members lie in the half; the larger one gets key ~0.
__device__ __forceinline__ unsigned entry_size(unsigned lin) { return (lin >> 31) ? 1u : 2u; }
__device__ __forceinline__ unsigned entry_lin(unsigned lin) { return lin & 0x7fffffffu; }

__global__ void k_keys(const double2* G, const uint8_t* mark, Grid3 g, unsigned long long* key,
                       unsigned* lin) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int H = g.nx / 2 + 1;
  // |g^(0)| = number of inclusion voxels, exact in FP64 (a sum of ones)
  const double amax = G ? G[0].x : 0.0;
  if (i >= (long long)H * g.ny * g.nz) return;
  const int kx = (int)(i % H);
  const int iy = (int)((i / H) % g.ny);
  const int iz = (int)(i / ((long long)H * g.ny));
  const int ky = sgn_index(iy, g.ny), kz = sgn_index(iz, g.nz);
  const int cx = sgn_index(wrap(-kx, g.nx), g.nx);
  const int cy = sgn_index(wrap(-ky, g.ny), g.ny);
  const int cz = sgn_index(wrap(-kz, g.nz), g.nz);
  const long long l = signed_lin(kx, ky, kz, g);
  const long long lc = signed_lin(cx, cy, cz, g);
  const bool own = l <= lc;
  if (!own && cx == kx) {   // the conjugate is an entry of its own
    key[i] = ~0ull;
    lin[i] = 0;
    return;
  }
  lin[i] = (unsigned)(own ? l : lc) | (l == lc ? 0x80000000u : 0u);
  const unsigned long long k2 =
      (unsigned long long)((long long)kx * kx + (long long)ky * ky + (long long)kz * kz);
  unsigned long long primary;
  if (mark) {
    const long long m = own ? ((long long)iz * g.ny + iy) * g.nx + kx
                            : ((long long)wrap(cz, g.nz) * g.ny + wrap(cy, g.ny)) * g.nx +
                                  wrap(cx, g.nx);
    primary = mark[m] ? 0ull : 1ull;
  } else {
    long long aq = 0;
    if (amax > 0.0) {
      const double a = hypot(G[i].x, G[i].y);
      aq = llrint(a / amax * 1073741824.0);
    }
    long long p = 1073741824LL - aq;
    primary = (unsigned long long)(p < 0 ? 0 : p);
  }
  key[i] = (primary << 33) | k2;
}

// Radix selection of the threshold, the smallest (key, lin) whose weighted count of entries at or
// below it reaches k_target. One launch per digit, all enqueued at once: a weighted histogram of the
// digit over the entries that agree with the digits chosen so far (block-local, a thread adds
// runs of equal digits once: most amplitudes share their leading bits), and the last block to
// finish picks the digit and clears the histogram. With a host read per digit the 14
// passes took a third of a 1024^2 call.
struct Select {
  unsigned long long key;   // digits chosen so far
  unsigned lin;
  unsigned below;           // weighted count of the entries below them
  unsigned count;           // after the last digit: frequencies at or below the threshold
  unsigned blocks;          // finished blocks of the pass
};
constexpr int kDigitBits = 11, kBins = 1 << kDigitBits;

__global__ __launch_bounds__(256) void k_select_digit(const unsigned long long* key,
                                                      const unsigned* lin, long long n,
                                                      int on_lin, int shift, int bits,
                                                      unsigned k_target, Select* st,
                                                      unsigned* hist) {
  __shared__ unsigned sh[kBins];
  __shared__ unsigned wsum[8];
  __shared__ bool last;
  const int tid = threadIdx.x;
  for (int b = tid; b < kBins; b += 256) sh[b] = 0;
  const unsigned long long chosen = __ldcg(&st->key);
  const unsigned chosen_lin = __ldcg(&st->lin);
  __syncthreads();
  unsigned run = 0, bin = 0;
  for (long long i = blockIdx.x * 256LL + tid; i < n; i += gridDim.x * 256LL) {
    const unsigned long long k = key[i];
    if (k == ~0ull) continue;
    unsigned b;
    unsigned sz;
    if (!on_lin) {
      if (shift + bits < 64 && ((k ^ chosen) >> (shift + bits)) != 0) continue;
      b = (unsigned)(k >> shift) & ((1u << bits) - 1);
      sz = entry_size(lin[i]);
    } else {
      if (k != chosen) continue;
      const unsigned l = lin[i];
      if (shift + bits < 32 && ((entry_lin(l) ^ chosen_lin) >> (shift + bits)) != 0) continue;
      b = (entry_lin(l) >> shift) & ((1u << bits) - 1);
      sz = entry_size(l);
    }
    if (run && b != bin) {
      atomicAdd(&sh[bin], run);
      run = 0;
    }
    bin = b;
    run += sz;
  }
  if (run) atomicAdd(&sh[bin], run);
  __syncthreads();
  for (int b = tid; b < kBins; b += 256)
    if (sh[b]) atomicAdd(&hist[b], sh[b]);
  __threadfence();
  __syncthreads();
  if (tid == 0) last = atomicAdd(&st->blocks, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  // eight bins per thread, their exclusive scan, then the one bin that reaches the target
  constexpr int kPer = kBins / 256;
  unsigned v[kPer], sum = 0;
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    v[u] = __ldcg(hist + tid * kPer + u);
    hist[tid * kPer + u] = 0;
    sum += v[u];
  }
  unsigned inc = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, inc, o);
    if ((tid & 31) >= o) inc += t;
  }
  if ((tid & 31) == 31) wsum[tid >> 5] = inc;
  const unsigned below0 = st->below;
  __syncthreads();
  unsigned before = below0 + inc - sum;
  for (int w = 0; w < (tid >> 5); ++w) before += wsum[w];
  if (before < k_target && before + sum >= k_target) {   // one thread
    int u = 0;
    while (before + v[u] < k_target) before += v[u++];
    const unsigned b = tid * kPer + u;
    st->below = before;
    st->count = before + v[u];
    if (on_lin) st->lin = chosen_lin | (b << shift);
    else st->key = chosen | ((unsigned long long)b << shift);
  }
  if (tid == 0) st->blocks = 0;
}

// whether the frequency at signed-linear position s is selected
__device__ __forceinline__ bool selected(long long s, const unsigned long long* key,
                                         const unsigned* lin, const Grid3& g,
                                         unsigned long long thi, unsigned tlin) {
  const int H = g.nx / 2 + 1;
  int kx = (int)(s % g.nx) - g.hx;
  int ky = (int)((s / g.nx) % g.ny) - g.hy;
  int kz = (int)(s / ((long long)g.nx * g.ny)) - g.hz;
  if (kx < 0) {
    kx = -kx;
    ky = -ky;
    kz = -kz;
  }
  long long i = ((long long)wrap(kz, g.nz) * g.ny + wrap(ky, g.ny)) * H + kx;
  unsigned long long k = key[i];
  if (k == ~0ull) {   // its conjugate holds the pair's entry
    i = ((long long)wrap(-kz, g.nz) * g.ny + wrap(-ky, g.ny)) * H + kx;
    k = key[i];
  }
  return k < thi || (k == thi && entry_lin(lin[i]) <= tlin);
}

// selected frequencies per 1024 positions
__global__ __launch_bounds__(1024) void k_select_totals(const unsigned long long* key,
                                                        const unsigned* lin, Grid3 g,
                                                        const Select* st, int* tot) {
  const long long s = blockIdx.x * 1024LL + threadIdx.x;
  const int f = s < g.N && selected(s, key, lin, g, st->key, st->lin);
  const int n = __syncthreads_count(f);
  if (threadIdx.x == 0) tot[blockIdx.x] = n;
}

// exclusive scan of the totals in place, 1024 at a time
__global__ __launch_bounds__(1024) void k_scan_totals(int* tot, int nb) {
  __shared__ int ws[32];
  __shared__ int carry;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int b0 = 0; b0 < nb; b0 += 1024) {
    const int b = b0 + threadIdx.x;
    const int t = b < nb ? tot[b] : 0;
    int inc = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += u;
    }
    if (lane == 31) ws[warp] = inc;
    __syncthreads();
    int base = carry;
    for (int w = 0; w < warp; ++w) base += ws[w];
    if (b < nb) tot[b] = base + inc - t;
    __syncthreads();
    if (threadIdx.x == 1023) carry = base + inc;
    __syncthreads();
  }
}

// the selected frequencies in signed-linear order
__global__ __launch_bounds__(1024) void k_compact(const unsigned long long* key, const unsigned* lin,
                                                  Grid3 g, const Select* st, const int* tot,
                                                  int* out, long long cap) {
  __shared__ int ws[32];
  const long long s = blockIdx.x * 1024LL + threadIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool f = s < g.N && selected(s, key, lin, g, st->key, st->lin);
  const unsigned m = __ballot_sync(0xffffffffu, f);
  if (lane == 0) ws[warp] = __popc(m);
  __syncthreads();
  if (!f) return;
  long long pos = tot[blockIdx.x] + __popc(m & ((1u << lane) - 1));
  for (int w = 0; w < warp; ++w) pos += ws[w];
  if (pos < cap) {
    out[3 * pos + 0] = (int)(s % g.nx) - g.hx;
    out[3 * pos + 1] = (int)((s / g.nx) % g.ny) - g.hy;
    out[3 * pos + 2] = (int)(s / ((long long)g.nx * g.ny)) - g.hz;
  }
}

__global__ void k_radial_mark(int L, int nx, int ny, uint8_t* mark) {
  const int l = blockIdx.y;
  const int ti = blockIdx.x * blockDim.x + threadIdx.x;
  const double th = M_PI * (double)l / (double)L;
  const double c = cos(th), s = sin(th);
  long long x, y;
  if (fabs(c) >= fabs(s)) {
    const int t = ti - nx / 2;
    if (t > nx / 2) return;
    const double v = (double)t * (s / c);
    x = t;
    y = (long long)copysign(floor(fabs(v) + 0.5), v);
  } else {
    const int t = ti - ny / 2;
    if (t > ny / 2) return;
    const double v = (double)t * (c / s);
    y = t;
    x = (long long)copysign(floor(fabs(v) + 0.5), v);
  }
  if (llabs(x) <= nx / 2 && llabs(y) <= ny / 2) {
    const int ix = (int)(((x % nx) + nx) % nx), iy = (int)(((y % ny) + ny) % ny);
    mark[(long long)iy * nx + ix] = 1;
  }
}

__global__ void k_count_u8(const uint8_t* m, long long N, unsigned long long* out) {
  __shared__ unsigned long long sh[256];
  unsigned long long s = 0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < N;
       i += (long long)gridDim.x * blockDim.x)
    s += m[i] ? 1 : 0;
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0 && sh[0]) atomicAdd(out, sh[0]);
}

// One device allocation for all scratch of a call, carved in 256-byte steps: a cudaMalloc and a
// cudaFree per array (fourteen, and two of pinned memory) took a third of a 1024^2 call.
struct Scratch {
  unsigned char* base = nullptr;
  size_t off = 0, size = 0;
  ~Scratch() {
    if (base) cudaFree(base);
  }
  static size_t pad(size_t b) { return (b + 255) & ~(size_t)255; }
  bool alloc(size_t bytes) {
    size = bytes;
    if (cudaMalloc(reinterpret_cast<void**>(&base), bytes) == cudaSuccess) return true;
    base = nullptr;
    cudaGetLastError();
    return false;
  }
  template <class T>
  T* get(size_t n) {
    unsigned char* p = base + off;
    off += pad(n * sizeof(T));
    return off <= size ? reinterpret_cast<T*>(p) : nullptr;
  }
};

int check(cudaError_t e, const char* what) { return e == cudaSuccess ? RF_OK : cuda_fail(e, what); }

int validate_grid(const rf_grid* g, Grid3& out) {
  if (!g || (g->dim != 2 && g->dim != 3)) {
    set_error("grid: dim must be 2 or 3");
    return RF_ERR_INVALID;
  }
  for (int j = 0; j < 3; ++j)
    if (g->n[j] < 1 || g->n[j] > 4096) {
      set_error("grid: sizes must be in [1, 4096]");
      return RF_ERR_INVALID;
    }
  if (g->dim == 2 && g->n[2] != 1) {
    set_error("grid: Nz must be 1 in 2D");
    return RF_ERR_INVALID;
  }
  out.nx = g->n[0];
  out.ny = g->n[1];
  out.nz = g->n[2];
  out.N = (long long)out.nx * out.ny * out.nz;
  if (out.N >= (1LL << 31)) {
    set_error("grid: too many voxels");
    return RF_ERR_INVALID;
  }
  out.hx = (out.nx - 1) / 2;
  out.hy = (out.ny - 1) / 2;
  out.hz = (out.nz - 1) / 2;
  return RF_OK;
}

long long half_size(const Grid3& g) { return (long long)(g.nx / 2 + 1) * g.ny * g.nz; }

// Scratch of the selection: entries (half_size each), state, histogram, block totals, output
struct SelectScratch {
  unsigned long long* key;
  unsigned* lin;
  Select* st;
  unsigned* hist;
  int* tot;
  int* d_out;   // [3 (k_target + 1)]
};

size_t select_bytes(const Grid3& g, long long k_target) {
  const size_t m = (size_t)half_size(g);
  return Scratch::pad(m * 8) + Scratch::pad(m * 4) + Scratch::pad(sizeof(Select)) +
         Scratch::pad(kBins * 4) + Scratch::pad(((size_t)(g.N + 1023) / 1024) * 4) +
         Scratch::pad(sizeof(int) * 3 * (size_t)(k_target + 1));
}

bool select_carve(Scratch& sc, const Grid3& g, long long k_target, SelectScratch* ss) {
  ss->key = sc.get<unsigned long long>(half_size(g));
  ss->lin = sc.get<unsigned>(half_size(g));
  ss->st = sc.get<Select>(1);
  ss->hist = sc.get<unsigned>(kBins);
  ss->tot = sc.get<int>((g.N + 1023) / 1024);
  ss->d_out = sc.get<int>(3 * (size_t)(k_target + 1));
  return ss->d_out != nullptr;
}

// Selection of the pattern from the entries in ss, shared by every entry point: the threshold, the
// selected frequencies in signed-linear order, and their copy to the host. The pattern holds
// k_target or, when the last pair passes it, k_target + 1 frequencies.
int select_and_compact(const Grid3& g, const SelectScratch& ss, long long k_target,
                       int32_t* out_host, long long cap, long long* K_out, cudaStream_t s) {
  const long long n = half_size(g);
  if (int e = check(cudaMemsetAsync(ss.st, 0, sizeof(Select), s), "memset")) return e;
  if (int e = check(cudaMemsetAsync(ss.hist, 0, kBins * sizeof(unsigned), s), "memset")) return e;
  const int blocks = (int)std::min<long long>(304, (n + 255) / 256);
  // primary: bits 63 to 33 of the key; |k|^2 (below 3 2048^2 < 2^24): bits 23 to 0; lin: 31 bits
  struct Digit {
    int on_lin, shift, bits;
  };
  const Digit digits[] = {{0, 53, 11}, {0, 42, 11}, {0, 33, 9}, {0, 22, 11}, {0, 11, 11},
                          {0, 0, 11},  {1, 20, 11}, {1, 10, 10}, {1, 0, 10}};
  // a digit above every entry's |k|^2 or lin is zero throughout (two of the nine passes for 1024^2:
  // 31 us less of a call in turn with the nine; 64^2 302 and 279 us)
  const unsigned long long k2max = (unsigned long long)(g.nx / 2) * (g.nx / 2) +
                                   (unsigned long long)(g.ny / 2) * (g.ny / 2) +
                                   (unsigned long long)(g.nz / 2) * (g.nz / 2);
  for (const Digit& d : digits) {
    const bool k2 = !d.on_lin && d.shift < 33;
    const unsigned long long top = d.on_lin ? (unsigned long long)(g.N - 1) : k2 ? k2max : ~0ull;
    if (d.shift > 0 && (top >> d.shift) == 0) continue;
    k_select_digit<<<blocks, 256, 0, s>>>(ss.key, ss.lin, n, d.on_lin, d.shift, d.bits,
                                          (unsigned)k_target, ss.st, ss.hist);
  }
  const long long nb = (g.N + 1023) / 1024;
  k_select_totals<<<(unsigned)nb, 1024, 0, s>>>(ss.key, ss.lin, g, ss.st, ss.tot);
  k_scan_totals<<<1, 1024, 0, s>>>(ss.tot, (int)nb);
  k_compact<<<(unsigned)nb, 1024, 0, s>>>(ss.key, ss.lin, g, ss.st, ss.tot, ss.d_out,
                                          k_target + 1);
  if (int e = check(cudaGetLastError(), "select")) return e;
  Select h{};
  if (int e = check(cudaMemcpyAsync(&h, ss.st, sizeof h, cudaMemcpyDeviceToHost, s), "copy count"))
    return e;
  if (int e = check(cudaStreamSynchronize(s), "sync pattern")) return e;
  const long long K = h.count;
  if (K < k_target || K > k_target + 1) {
    set_error("pattern: threshold search failed");
    return RF_ERR_INVALID;
  }
  *K_out = K;
  if (K > cap) {
    set_error("pattern: output capacity too small");
    return RF_ERR_INVALID;
  }
  if (int e = check(cudaMemcpyAsync(out_host, ss.d_out, sizeof(int) * 3 * K, cudaMemcpyDeviceToHost,
                                    s), "copy pattern"))
    return e;
  return check(cudaStreamSynchronize(s), "sync pattern");
}

}  // namespace

// DFT of the inclusion indicator along x, y and z (FP64) from the device phase map: FFTs for
// sides 2^b and 3 * 2^b, dense DFTs (exact table sums along x) otherwise, on the half kx <= nx / 2.
// Uses A and B (half_size each) and the tables tx, ty, tz ([side] each); *G receives the buffer holding g^.
int indicator_transform(const Grid3& g, const uint8_t* d_pm, int incl, double2* A, double2* B,
                        double2* tx, double2* ty, double2* tz, double2** G, cudaStream_t s) {
  k_table_f64<<<(g.nx + 255) / 256, 256, 0, s>>>(tx, g.nx);
  k_table_f64<<<(g.ny + 255) / 256, 256, 0, s>>>(ty, g.ny);
  k_table_f64<<<(g.nz + 255) / 256, 256, 0, s>>>(tz, g.nz);
  const long long rows = g.N / g.nx;
  if (fft64_length(g.nx)) {
    // few enough rows per block to give every SM several
    const int C = std::max(1, std::min(fft64_lines(g.nx, 16), (int)(rows / (2 * 304))));
    if (int e = check(cudaFuncSetAttribute(k_g_rows_fft, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)kFft64Smem), "pattern: smem attribute"))
      return e;
    k_g_rows_fft<<<(unsigned)((rows + 2 * C - 1) / (2 * C)), 256, 2 * (size_t)C * g.nx * sizeof(double2), s>>>(
        d_pm, incl, g.nx, rows, C, tx, A);
  } else {
    const size_t smem = (size_t)g.nx * (sizeof(double2) + sizeof(float));
    if (int e = check(cudaFuncSetAttribute(k_g_rows, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           100 * 1024), "pattern: smem attribute"))
      return e;
    k_g_rows<<<(unsigned)rows, 256, smem, s>>>(d_pm, incl, g.nx, tx, A);
  }
  if (int e = check(cudaGetLastError(), "g rows")) return e;
  if (int e = check(cudaFuncSetAttribute(k_cols_fft64, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kFft64Smem), "pattern: smem attribute"))
    return e;
  // along y: batch z, k = y, n = kx
  const int H = g.nx / 2 + 1;
  if (fft64_length(g.ny)) {
    const int C = fft64_lines(g.ny, 8);
    dim3 grd((H + C - 1) / C, g.nz);
    k_cols_fft64<<<grd, 256, 2 * (size_t)C * g.ny * sizeof(double2), s>>>(
        A, B, g.ny, H, (long long)g.ny * H, C, ty);
  } else {
    dim3 grd((H + 127) / 128, (g.ny + 3) / 4, g.nz);
    k_axis_f64<<<grd, 128, 0, s>>>(A, B, g.ny, H, (long long)g.ny * H, ty);
  }
  *G = B;
  if (g.nz > 1) {
    const int Nn = g.ny * H;
    if (fft64_length(g.nz)) {
      const int C = fft64_lines(g.nz, 8);
      dim3 grd((Nn + C - 1) / C, 1);
      k_cols_fft64<<<grd, 256, 2 * (size_t)C * g.nz * sizeof(double2), s>>>(B, A, g.nz, Nn, 0, C,
                                                                             tz);
    } else {
      dim3 grd((Nn + 127) / 128, (g.nz + 3) / 4, 1);
      k_axis_f64<<<grd, 128, 0, s>>>(B, A, g.nz, Nn, 0, tz);
    }
    *G = A;
  }
  return check(cudaGetLastError(), "g axes");
}

int pattern_adapted(const rf_grid* grid, const uint8_t* pm_host, int incl, long long k_target,
                    int32_t* out, long long cap, long long* K_out, cudaStream_t s) {
  Grid3 g;
  if (int e = validate_grid(grid, g)) return e;
  if (!pm_host || !out || !K_out || k_target < 1 || k_target > g.N) {
    set_error("pattern_adapted: invalid arguments");
    return RF_ERR_INVALID;
  }
  Scratch sc;
  const size_t half = (size_t)half_size(g);
  if (!sc.alloc(Scratch::pad(g.N) + 2 * Scratch::pad(half * sizeof(double2)) +
                Scratch::pad(g.nx * sizeof(double2)) + Scratch::pad(g.ny * sizeof(double2)) +
                Scratch::pad(g.nz * sizeof(double2)) + select_bytes(g, k_target))) {
    set_error("pattern_adapted: out of device memory");
    return RF_ERR_OOM;
  }
  uint8_t* d_pm = sc.get<uint8_t>(g.N);
  double2* A = sc.get<double2>(half);
  double2* B = sc.get<double2>(half);
  double2* tx = sc.get<double2>(g.nx);
  double2* ty = sc.get<double2>(g.ny);
  double2* tz = sc.get<double2>(g.nz);
  SelectScratch ss{};
  if (!select_carve(sc, g, k_target, &ss)) {
    set_error("pattern_adapted: scratch layout");
    return RF_ERR_OOM;
  }
  if (int e = check(cudaMemcpyAsync(d_pm, pm_host, g.N, cudaMemcpyHostToDevice, s), "upload"))
    return e;
  double2* G = nullptr;
  if (int e = indicator_transform(g, d_pm, incl, A, B, tx, ty, tz, &G, s)) return e;
  k_keys<<<(unsigned)((half + 255) / 256), 256, 0, s>>>(G, nullptr, g, ss.key, ss.lin);
  if (int e = check(cudaGetLastError(), "keys")) return e;
  return select_and_compact(g, ss, k_target, out, cap, K_out, s);
}

int pattern_radial(const rf_grid* grid, long long k_target, int32_t* out, long long cap,
                   long long* K_out, cudaStream_t s) {
  Grid3 g;
  if (int e = validate_grid(grid, g)) return e;
  if (grid->dim != 2) {
    set_error("pattern_radial: 2D only");
    return RF_ERR_INVALID;
  }
  if (!out || !K_out || k_target < 1 || k_target > g.N) {
    set_error("pattern_radial: invalid arguments");
    return RF_ERR_INVALID;
  }
  Scratch sc;
  if (!sc.alloc(Scratch::pad(g.N) + Scratch::pad(8) + select_bytes(g, k_target))) {
    set_error("pattern_radial: out of device memory");
    return RF_ERR_OOM;
  }
  uint8_t* mark = sc.get<uint8_t>(g.N);
  unsigned long long* d_cnt = sc.get<unsigned long long>(1);
  SelectScratch ss{};
  if (!select_carve(sc, g, k_target, &ss)) {
    set_error("pattern_radial: scratch layout");
    return RF_ERR_OOM;
  }
  const int maxL = 4 * (g.nx > g.ny ? g.nx : g.ny);
  const int tcount = (g.nx > g.ny ? g.nx : g.ny) + 1;
  unsigned long long cnt = 0;
  int L = 1;
  for (; L <= maxL; ++L) {
    if (int e = check(cudaMemsetAsync(mark, 0, g.N, s), "memset mark")) return e;
    dim3 grd((tcount + 127) / 128, L);
    k_radial_mark<<<grd, 128, 0, s>>>(L, g.nx, g.ny, mark);
    if (int e = check(cudaMemsetAsync(d_cnt, 0, sizeof(unsigned long long), s), "memset")) return e;
    k_count_u8<<<304, 256, 0, s>>>(mark, g.N, d_cnt);
    if (int e = check(cudaGetLastError(), "radial")) return e;
    if (int e = check(cudaMemcpyAsync(&cnt, d_cnt, sizeof(cnt), cudaMemcpyDeviceToHost, s), "cp"))
      return e;
    if (int e = check(cudaStreamSynchronize(s), "sync")) return e;
    if ((long long)cnt >= k_target) break;
  }
  if ((long long)cnt < k_target) {
    set_error("pattern_radial: k_target not reachable");
    return RF_ERR_INVALID;
  }
  k_keys<<<(unsigned)((half_size(g) + 255) / 256), 256, 0, s>>>(nullptr, mark, g, ss.key, ss.lin);
  if (int e = check(cudaGetLastError(), "keys")) return e;
  return select_and_compact(g, ss, k_target, out, cap, K_out, s);
}

// ------------------------------------------------------------------------------------------
// Allocation-free variant of the adapted pattern.
//
// rf_pattern_adapted allocates its device scratch with cudaMalloc and frees it with cudaFree,
// and cudaFree synchronises the whole device. Callers that share the GPU with other streams
// they must not stall, or whose device memory is owned by another framework's pool allocator,
// cannot make those calls. rf_pattern_adapted_noalloc runs the same kernels with all scratch
// carved from the file-scope array below instead, for grids of at most kNoAllocMaxVoxels.
// Every GPU that loads this library holds the array until the process exits.
namespace {

constexpr long long kNoAllocMaxVoxels = 65536;     // e.g. 256 x 256 or 40 x 40 x 40
constexpr int kNoAllocMaxSide = 4096;
constexpr size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }
constexpr size_t kNoAllocBytes =
    align256(kNoAllocMaxVoxels)                                   // phase map
    + 2 * align256(kNoAllocMaxVoxels * sizeof(double2))           // transform buffers
    + 3 * align256(kNoAllocMaxSide * sizeof(double2))             // twiddle tables
    + align256(kNoAllocMaxVoxels * sizeof(unsigned long long))    // keys
    + align256(kNoAllocMaxVoxels * sizeof(unsigned))              // lin
    + align256((kNoAllocMaxVoxels / 1024 + 2) * sizeof(int))      // scan totals
    + align256(sizeof(Select))                                    // selection state
    + align256(kBins * sizeof(unsigned))                          // histogram
    + align256(3 * (kNoAllocMaxVoxels + 1) * sizeof(int));        // output frequencies

static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mutex;
unsigned char* g_noalloc_ptr[kMaxDevices] = {nullptr};

// Device address of the scratch array for the current device (looked up once per device).
int noalloc_scratch(unsigned char** out) {
  int dev = 0;
  if (int e = check(cudaGetDevice(&dev), "noalloc: cudaGetDevice")) return e;
  if (dev < 0 || dev >= kMaxDevices) {
    set_error("rf_pattern_adapted_noalloc: device index out of range");
    return RF_ERR_INVALID;
  }
  std::lock_guard<std::mutex> lock(g_noalloc_mutex);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    if (int e = check(cudaGetSymbolAddress(&p, g_noalloc_scratch), "noalloc: scratch address"))
      return e;
    g_noalloc_ptr[dev] = static_cast<unsigned char*>(p);
  }
  *out = g_noalloc_ptr[dev];
  return RF_OK;
}

}  // namespace

int pattern_adapted_noalloc(const rf_grid* grid, const uint8_t* pm_host, int incl,
                            long long k_target, int32_t* out_host, long long cap,
                            long long* K_out, cudaStream_t s) {
  Grid3 g;
  if (int e = validate_grid(grid, g)) return e;
  if (!pm_host || !out_host || !K_out || k_target < 1 || k_target > g.N) {
    set_error("rf_pattern_adapted_noalloc: invalid arguments");
    return RF_ERR_INVALID;
  }
  if (g.N > kNoAllocMaxVoxels) {
    set_error("rf_pattern_adapted_noalloc: grid has more than 65536 voxels (the limit of its "
              "static scratch); use rf_pattern_adapted");
    return RF_ERR_INVALID;
  }
  unsigned char* base = nullptr;
  if (int e = noalloc_scratch(&base)) return e;
  size_t off = 0;
  auto carve = [&](size_t bytes) {
    unsigned char* p = base + off;
    off += align256(bytes);
    return p;
  };
  uint8_t* d_pm = carve(kNoAllocMaxVoxels);
  double2* A = reinterpret_cast<double2*>(carve(kNoAllocMaxVoxels * sizeof(double2)));
  double2* B = reinterpret_cast<double2*>(carve(kNoAllocMaxVoxels * sizeof(double2)));
  double2* tx = reinterpret_cast<double2*>(carve(kNoAllocMaxSide * sizeof(double2)));
  double2* ty = reinterpret_cast<double2*>(carve(kNoAllocMaxSide * sizeof(double2)));
  double2* tz = reinterpret_cast<double2*>(carve(kNoAllocMaxSide * sizeof(double2)));
  // (the half spectrum never has more entries than the grid has voxels)
  SelectScratch ss{};
  ss.key = reinterpret_cast<unsigned long long*>(
      carve(kNoAllocMaxVoxels * sizeof(unsigned long long)));
  ss.lin = reinterpret_cast<unsigned*>(carve(kNoAllocMaxVoxels * sizeof(unsigned)));
  ss.tot = reinterpret_cast<int*>(carve((kNoAllocMaxVoxels / 1024 + 2) * sizeof(int)));
  ss.st = reinterpret_cast<Select*>(carve(sizeof(Select)));
  ss.hist = reinterpret_cast<unsigned*>(carve(kBins * sizeof(unsigned)));
  ss.d_out = reinterpret_cast<int*>(carve(3 * (kNoAllocMaxVoxels + 1) * sizeof(int)));

  // the transform, key and selection code of rf_pattern_adapted on carved scratch; the state and
  // the histogram, the only scratch that must start at zero, are cleared before every use
  if (int e = check(cudaMemcpyAsync(d_pm, pm_host, g.N, cudaMemcpyHostToDevice, s), "upload"))
    return e;
  double2* G = nullptr;
  if (int e = indicator_transform(g, d_pm, incl, A, B, tx, ty, tz, &G, s)) return e;
  k_keys<<<(unsigned)((half_size(g) + 255) / 256), 256, 0, s>>>(G, nullptr, g, ss.key, ss.lin);
  if (int e = check(cudaGetLastError(), "noalloc: keys")) return e;
  return select_and_compact(g, ss, k_target, out_host, cap, K_out, s);
}


}  // namespace rfk
