// Pruned DFTs of the default transform mode (any grid size, FP32): the row pass (inverse along x,
// law, forward along x) and the transforms along y and z, on the pattern's distinct frequencies.
//
// They are small real matrix products (a 375 x 250 cell with K = 5 %: 47 MFMA along x, 13 + 13
// along y, a few microseconds at the FP32 rate), so what counts is to cover the chip and to
// feed the multipliers:
//   - points x and L - x share their twiddles: with A = sum Re(T) cos and B = sum Im(T) sin the
//     values are A - B and A + B, and a forward transform takes the sums and differences of the
//     two points. That halves the products of both directions.
//   - a thread holds two pairs (or two frequencies) of six lines (two rows of three components, or
//     one of six): each twiddle is loaded once for twelve products, each line value, the same
//     for a whole warp, once for four.
//   - the sums of a pair are split over several threads where a cell has too few rows to fill the
//     chip, and added up in a fixed order.
// A row block used to stage five rows of such a cell (50 blocks on 152 SMs) and look the twiddles
// up by a modulo per product: 134 us per pass; the y transforms ran on 32 blocks, 28 and 23 us.
// Now 16 us, and 11 and 13 us (traced); the whole update 184 -> 35 us (75 x 90 x 66: 126 -> 65 us).
#include <algorithm>
#include <vector>

#include "rf_internal.cuh"
#include "rf_law.cuh"

namespace rfk {
namespace dftk {

constexpr int kThreads = 384;    // row pass
constexpr int kMaxX = 4 * kThreads - 2;   // two pairs per thread cover the row

struct RowDftArgs {
  const float2* T;      // [rows][NC][Kx]
  float2* Tout;
  const uint8_t* phase;
  float* state;
  const float* fac;     // [Kx] weight / N
  const float2* Wi;     // [Kx][np] (cos, sin) of 2 pi k x / Nx, x = 0 .. Nx / 2
  const float2* Wf;     // [np][Kx]
  int Nx, Kx, rows, np, PT, U, SJ, JT;   // np pairs, PT threads per unit, U units per block
  long long N;
  LawParams law;
  float* eps_out;
  float* sig_out;
  float* alpha_out;
  double* sbar_part;
  double* viol_part;
  int commit;
  const int* done;
  int early;            // let the next kernel start its prologue
};

// shared memory: line values [U][Kx][6], sums and differences [U][np][12], partial sums
__host__ __device__ inline size_t row_dft_smem(int U, int Kx, int np) {
  return sizeof(float) * ((size_t)U * Kx * 12 + (size_t)U * np * 12 + 24 * kThreads);
}

template <int NC, bool PLASTIC, bool FINAL>
__global__ __launch_bounds__(kThreads, 2) void k_row_dft(const __grid_constant__ RowDftArgs a) {
  constexpr int RPU = NC == 3 ? 2 : 1, NL = 6;   // a unit: six lines
  extern __shared__ __align__(16) float d_smem[];
  __shared__ DevPhase phs[kMaxPhases];
  __shared__ double red[32];
  const int tid = threadIdx.x, Kx = a.Kx, np = a.np, PT = a.PT, L = a.Nx;
  float* Ts = d_smem;
  float* UV = Ts + a.U * Kx * 12;
  float* Pp = UV + a.U * np * 12;
  for (int i = tid; i < kMaxPhases; i += kThreads) phs[i] = a.law.ph[i];
  const int unit0 = blockIdx.x * a.U, units = (a.rows + RPU - 1) / RPU;
  const int nu = min(a.U, units - unit0);
  if (a.early) grid_dep_launch();
  grid_dep_wait();
  if (!FINAL && a.done && __ldcg(a.done)) return;   // the same flag value for every thread
  // line values, scaled, a frequency's six lines together; loads in batches
  {
    const float2* src = a.T + (long long)unit0 * NL * Kx;
    const int lines = min(nu * NL, (a.rows - unit0 * RPU) * NC);   // an odd last row leaves half a unit
    const int tot = nu * NL * Kx;
    for (int i0 = tid; i0 < tot; i0 += 8 * kThreads) {
      float2 v[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const int i = i0 + m * kThreads;
        v[m] = make_float2(0.f, 0.f);
        if (i < lines * Kx) v[m] = __ldcg(src + i);
      }
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const int i = i0 + m * kThreads;
        if (i >= tot) break;
        const int l = i / Kx, j = i - l * Kx, uu = l / NL;
        const float f = a.fac[j];
        reinterpret_cast<float2*>(Ts)[(uu * Kx + j) * NL + l - uu * NL] =
            make_float2(f * v[m].x, f * v[m].y);
      }
    }
  }
  __syncthreads();
  const int CW = a.U * PT;
  {
    const int s = tid / CW, cw = tid - s * CW, uu = cw / PT, p = cw - uu * PT;
    if (s < a.SJ && uu < nu) {
      float A[2][NL], B[2][NL];
#pragma unroll
      for (int l = 0; l < NL; ++l) A[0][l] = A[1][l] = B[0][l] = B[1][l] = 0.f;
      const bool two = p + PT < np;
      const float2* w = a.Wi + p;
      const float4* t4 = reinterpret_cast<const float4*>(Ts) + uu * Kx * 3;
      const int x1 = two ? PT : 0;
#pragma unroll 4
      for (int j = s; j < Kx; j += a.SJ) {
        const float2 w0 = __ldg(w + (long long)j * np), w1 = __ldg(w + (long long)j * np + x1);
        const float4 t0 = t4[j * 3], t1 = t4[j * 3 + 1], t2 = t4[j * 3 + 2];
        const float re[6] = {t0.x, t0.z, t1.x, t1.z, t2.x, t2.z};
        const float im[6] = {t0.y, t0.w, t1.y, t1.w, t2.y, t2.w};
#pragma unroll
        for (int l = 0; l < NL; ++l) {
          A[0][l] = fmaf(re[l], w0.x, A[0][l]);
          B[0][l] = fmaf(im[l], w0.y, B[0][l]);
          A[1][l] = fmaf(re[l], w1.x, A[1][l]);
          B[1][l] = fmaf(im[l], w1.y, B[1][l]);
        }
      }
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int l = 0; l < NL; ++l) {
          Pp[(s * 24 + (q * NL + l) * 2) * CW + cw] = A[q][l];
          Pp[(s * 24 + (q * NL + l) * 2 + 1) * CW + cw] = B[q][l];
        }
    }
  }
  __syncthreads();
  // the law at the two voxels of a pair, one row of a unit per item
  double sb[6] = {0, 0, 0, 0, 0, 0}, vmax = 0.0;
  const float lam0 = a.law.lam0, mu0 = a.law.mu0;
  for (int it = tid; it < CW * 2 * RPU; it += kThreads) {
    const int cb = it / CW, cw = it - cb * CW, q = cb & 1, r = cb >> 1;
    const int uu = cw / PT, p = cw - uu * PT, x = p + q * PT;
    const int row = (unit0 + uu) * RPU + r;
    if (uu >= nu || x >= np) continue;
    float tau[2][NC];
    const bool self = x == 0 || 2 * x == L;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int c = 0; c < NC; ++c) tau[h][c] = 0.f;
    if (row < a.rows) {
      float sa[NC], sbm[NC];
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const float* pa = Pp + (q * NL + r * NC + c) * 2 * CW + cw;
        float va = 0.f, vb = 0.f;
        for (int s = 0; s < a.SJ; ++s) {
          va += pa[s * 24 * CW];
          vb += pa[s * 24 * CW + CW];
        }
        sa[c] = va;
        sbm[c] = vb;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (h == 1 && self) break;
        const long long g = (long long)row * L + (h == 0 ? x : L - x);
        float e[NC], e6[6];
#pragma unroll
        for (int c = 0; c < NC; ++c) e[c] = h == 0 ? sa[c] - sbm[c] : sa[c] + sbm[c];
        comp_to6<NC>(e, e6);
        const DevPhase& ph = phs[a.phase[g]];
        float ep[6] = {0, 0, 0, 0, 0, 0};
        float alpha = 0.f;
        if (PLASTIC) load_state<NC>(a.state, a.N, g, ep, alpha);
        LawOut o;
        stress6<PLASTIC>(e6, ph, ep, alpha, o);
        if (!FINAL) {
          const float tr = e6[0] + e6[1] + e6[2];
          float t6[6];
#pragma unroll
          for (int i = 0; i < 3; ++i) t6[i] = o.s[i] - (lam0 * tr + 2.f * mu0 * e6[i]);
#pragma unroll
          for (int i = 3; i < 6; ++i) t6[i] = o.s[i] - 2.f * mu0 * e6[i];
#pragma unroll
          for (int c = 0; c < NC; ++c) tau[h][c] = t6[comp6<NC>(c)];
        } else {
#pragma unroll
          for (int i = 0; i < 6; ++i) {
            sb[i] += (double)o.s[i];
            if (a.eps_out) a.eps_out[i * a.N + g] = e6[i];
            if (a.sig_out) a.sig_out[i * a.N + g] = o.s[i];
          }
          if (PLASTIC) {
            if (a.commit) store_state<NC>(a.state, a.N, g, o.ep, o.alpha);
            if (a.alpha_out) a.alpha_out[g] = o.alpha;
            if (o.yielded) {
              // FP64 consistency check of the FP32 return map: sigma_eq(sigma) = sy + H alpha
              const double s0 = o.s[0], s1 = o.s[1], s2 = o.s[2];
              const double pmd = (s0 + s1 + s2) / 3.0;
              const double d0 = s0 - pmd, d1 = s1 - pmd, d2 = s2 - pmd;
              const double qq = d0 * d0 + d1 * d1 + d2 * d2 +
                                2.0 * ((double)o.s[3] * o.s[3] + (double)o.s[4] * o.s[4] +
                                       (double)o.s[5] * o.s[5]);
              const double yl = (double)ph.sy + (double)ph.H * (double)o.alpha;
              vmax = fmax(vmax, fabs(sqrt(1.5 * qq) - yl) / (double)ph.sy);
            }
          } else if (a.alpha_out) {
            a.alpha_out[g] = 0.f;
          }
        }
      }
    }
    if (!FINAL) {
      // sums and differences (a point of its own: its value and zero)
      float2* d = reinterpret_cast<float2*>(UV) + (uu * np + x) * NL + r * NC;
#pragma unroll
      for (int c = 0; c < NC; ++c)
        d[c] = self ? make_float2(tau[0][c], 0.f)
                    : make_float2(tau[0][c] + tau[1][c], tau[0][c] - tau[1][c]);
    }
  }
  if (FINAL) {
    for (int i = 0; i < 6; ++i) {
      const double t = block_sum_d(sb[i], red);
      if (tid == 0) a.sbar_part[blockIdx.x * 6 + i] = t;
    }
    const double vm = block_max_d(vmax, red);
    if (tid == 0) a.viol_part[blockIdx.x] = vm;
    return;
  }
  __syncthreads();
  // forward: two frequencies of six lines per thread, the pairs split over SX threads
  const int FW = a.U * a.JT;
  const int fwn = min(FW, kThreads), SX = kThreads / fwn;
  for (int f0 = 0; f0 < FW; f0 += fwn) {
    const int s = tid / fwn, fl = tid - s * fwn, fw = f0 + fl;
    const int uu = fw / a.JT, jt = fw - uu * a.JT;
    if (s < SX && fw < FW && uu < nu) {
      float re[2][NL], im[2][NL];
#pragma unroll
      for (int l = 0; l < NL; ++l) re[0][l] = re[1][l] = im[0][l] = im[1][l] = 0.f;
      const int j1 = jt + a.JT < Kx ? a.JT : 0;
      const float2* w = a.Wf + jt;
      const float4* u4 = reinterpret_cast<const float4*>(UV) + uu * np * 3;
#pragma unroll 4
      for (int x = s; x < np; x += SX) {
        const float2 w0 = __ldg(w + (long long)x * Kx), w1 = __ldg(w + (long long)x * Kx + j1);
        const float4 t0 = u4[x * 3], t1 = u4[x * 3 + 1], t2 = u4[x * 3 + 2];
        const float u[6] = {t0.x, t0.z, t1.x, t1.z, t2.x, t2.z};
        const float v[6] = {t0.y, t0.w, t1.y, t1.w, t2.y, t2.w};
#pragma unroll
        for (int l = 0; l < NL; ++l) {
          re[0][l] = fmaf(u[l], w0.x, re[0][l]);
          im[0][l] = fmaf(v[l], w0.y, im[0][l]);
          re[1][l] = fmaf(u[l], w1.x, re[1][l]);
          im[1][l] = fmaf(v[l], w1.y, im[1][l]);
        }
      }
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int l = 0; l < NL; ++l) {
          Pp[(s * 24 + (q * NL + l) * 2) * fwn + fl] = re[q][l];
          Pp[(s * 24 + (q * NL + l) * 2 + 1) * fwn + fl] = im[q][l];
        }
    }
    __syncthreads();
    for (int o = tid; o < fwn * 2 * NL; o += kThreads) {
      const int ql = o / fwn, k = o - ql * fwn, f = f0 + k;
      const int u2 = f / a.JT, q = ql / NL, l = ql - q * NL, j = f - u2 * a.JT + q * a.JT;
      const int row = (unit0 + u2) * RPU + l / NC;
      if (f >= FW || u2 >= nu || j >= Kx || row >= a.rows) continue;
      float vr = 0.f, vi = 0.f;
      for (int s2 = 0; s2 < SX; ++s2) {
        vr += Pp[(s2 * 24 + ql * 2) * fwn + k];
        vi += Pp[(s2 * 24 + ql * 2 + 1) * fwn + k];
      }
      a.Tout[((long long)(unit0 + u2) * NL + l) * Kx + j] = make_float2(vr, -vi);
    }
    __syncthreads();
  }
}

// Wi[j][x] and Wf[x][j] from the row's table exp(+2 pi i t / Nx)
__global__ void k_row_tables(const float2* tab, const int* kx, int Nx, int Kx, int np, float2* Wi,
                             float2* Wf) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < np * Kx; i += gridDim.x * blockDim.x) {
    const int j = i / np, x = i - j * np;
    const float2 w = tab[(int)(((long long)kx[j] * x) % Nx)];
    Wi[i] = w;
    Wf[(long long)x * Kx + j] = w;
  }
}

struct AxisDftArgs {
  const float2* in;
  float2* out;
  long long in_bstride, out_bstride;
  int L, N, S;          // length, columns, sparse rows
  const int* vals;      // [S] frequency (mod L) of each sparse row
  const float2* table;  // exp(+2 pi i t / L)
  FastDiv dL;
  const int* done;
  int early;
  int ranks;            // blocks of one cluster (along the grid's z) that share a transform's sum
};

// Transform along one axis of [batch][rows][N]: FWD dense rows -> the S sparse ones (exp(-)),
// otherwise sparse -> dense (exp(+)). A block takes 32 columns; each of its four warps MP dense
// pairs (y, L - y) or MP sparse rows, over chunks of kC rows staged in shared memory. Where a long
// sum meets few results (2000 x 7, one frequency: 1001 pairs on one block; update 37 -> 17 us), the
// blocks of a cluster take a share of the chunks each and add up their sums in rank order.
constexpr int kC = 64;

// Sum of `splits` arrays of n values, `stride` apart (the row passes over slices of x): every block
// of a transform reads all its lines, so adding them up on the way in read each slice once per
// block of rows (1024^2 with every kx, split BF16, eight slices: 3550 us per update, so 907).
__global__ __launch_bounds__(256) void k_sum_slices(const float2* in, int splits, long long stride,
                                                    long long n, float2* out, const int* done) {
  grid_dep_wait();
  if (done && __ldcg(done)) return;
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += gridDim.x * 256LL) {
    float2 v = __ldcg(in + i);
#pragma unroll 4
    for (int s = 1; s < splits; ++s) {
      const float2 u = __ldcg(in + s * stride + i);
      v.x += u.x;
      v.y += u.y;
    }
    out[i] = v;
  }
}

template <int MP, bool FWD>
__global__ __launch_bounds__(128) void k_axis_dft(const __grid_constant__ AxisDftArgs a) {
  __shared__ float4 xs4[FWD ? kC * 32 : kC * 16];
  __shared__ float2 ws[kC][4 * MP];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n0 = blockIdx.x * 32, m0 = blockIdx.y * 4 * MP, L = a.L, np = L / 2 + 1;
  const int n = n0 + lane;
  const int bz = blockIdx.z / a.ranks, rank = blockIdx.z - bz * a.ranks;
  const float2* in = a.in + (long long)bz * a.in_bstride;
  float2* out = a.out + (long long)bz * a.out_bstride;
  float2* xs2 = reinterpret_cast<float2*>(xs4);
  const int K = FWD ? np : a.S, M = FWD ? a.S : np, chunks = (K + kC - 1) / kC;
  // this block's rows of the sum
  const int kbeg = chunks * rank / a.ranks * kC, kend = min(K, chunks * (rank + 1) / a.ranks * kC);
  float ar[MP], ai[MP], br[MP], bi[MP];
#pragma unroll
  for (int i = 0; i < MP; ++i) ar[i] = ai[i] = br[i] = bi[i] = 0.f;
  if (a.early) grid_dep_launch();
  // twiddles of a chunk: pair y (dense) and frequency v (sparse) meet at t = y v mod L
  auto twiddles = [&](int k0) {
    const int kn = min(kC, kend - k0);
    for (int i = tid; i < kn * 4 * MP; i += 128) {
      const int kk = i / (4 * MP), mm = i - kk * 4 * MP, m = m0 + mm;
      float2 w = make_float2(0.f, 0.f);
      if (m < M) {
        const int y = FWD ? k0 + kk : m, v = FWD ? a.vals[m] : a.vals[k0 + kk];
        const int t = y * v;
        w = __ldg(a.table + t - fdiv(t, a.dL) * L);
      }
      ws[kk][mm] = w;
    }
  };
  twiddles(kbeg);   // the pattern's alone
  grid_dep_wait();
  if (a.done && __ldcg(a.done)) return;   // the same flag value for every thread
  for (int k0 = kbeg; k0 < kend; k0 += kC) {
    const int kn = min(kC, kend - k0);
    if (k0 > kbeg) twiddles(k0);
    for (int r0 = warp; r0 < kn; r0 += 4 * 8) {
      float2 p[8], q[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int r = r0 + 4 * u, y = k0 + r;
        p[u] = q[u] = make_float2(0.f, 0.f);
        if (r < kn && n < a.N) {
          p[u] = __ldcg(in + (long long)y * a.N + n);
          if (FWD && y > 0 && 2 * y != L) q[u] = __ldcg(in + (long long)(L - y) * a.N + n);
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int r = r0 + 4 * u, y = k0 + r;
        if (r >= kn) break;
        if (FWD) {
          const bool self = y == 0 || 2 * y == L;
          xs4[r * 32 + lane] = self ? make_float4(p[u].x, p[u].y, 0.f, 0.f)
                                    : make_float4(p[u].x + q[u].x, p[u].y + q[u].y,
                                                  p[u].x - q[u].x, p[u].y - q[u].y);
        } else {
          xs2[r * 32 + lane] = p[u];
        }
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int kk = 0; kk < kn; ++kk) {
      if (FWD) {
        const float4 x = xs4[kk * 32 + lane];
#pragma unroll
        for (int i = 0; i < MP; ++i) {
          const float2 w = ws[kk][warp * MP + i];
          ar[i] = fmaf(x.x, w.x, ar[i]);
          ai[i] = fmaf(x.y, w.x, ai[i]);
          br[i] = fmaf(x.w, w.y, br[i]);
          bi[i] = fmaf(x.z, w.y, bi[i]);
        }
      } else {
        const float2 x = xs2[kk * 32 + lane];
#pragma unroll
        for (int i = 0; i < MP; ++i) {
          const float2 w = ws[kk][warp * MP + i];
          ar[i] = fmaf(x.x, w.x, ar[i]);
          ai[i] = fmaf(x.y, w.x, ai[i]);
          br[i] = fmaf(x.y, w.y, br[i]);
          bi[i] = fmaf(x.x, w.y, bi[i]);
        }
      }
    }
    __syncthreads();
  }
  auto put = [&](int m, int col, float vr, float vi, float wr, float wi) {
    if (m >= M || col >= a.N) return;
    if (FWD) {
      // (s.x c + d.y s, s.y c - d.x s)
      out[(long long)m * a.N + col] = make_float2(vr + wr, vi - wi);
    } else {
      // x c - y s, y c + x s at m; the conjugate twiddle at L - m
      out[(long long)m * a.N + col] = make_float2(vr - wr, vi + wi);
      if (m > 0 && 2 * m != L)
        out[(long long)(L - m) * a.N + col] = make_float2(vr + wr, vi - wi);
    }
  };
  if (a.ranks == 1) {
#pragma unroll
    for (int i = 0; i < MP; ++i) put(m0 + warp * MP + i, n, ar[i], ai[i], br[i], bi[i]);
    return;
  }
  // [4 MP][128 threads] partial sums in place of the staged rows, which every warp has read
  float* part = reinterpret_cast<float*>(xs4);
#pragma unroll
  for (int i = 0; i < MP; ++i) {
    part[(4 * i) * 128 + tid] = ar[i];
    part[(4 * i + 1) * 128 + tid] = ai[i];
    part[(4 * i + 2) * 128 + tid] = br[i];
    part[(4 * i + 3) * 128 + tid] = bi[i];
  }
  cluster_sync();
  const int per = 128 / a.ranks;   // this block adds up the sums of that many threads
  for (int q = tid; q < per * MP; q += 128) {
    const int i = q / per, t = rank * per + q - i * per;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    for (int r = 0; r < a.ranks; ++r)
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] += ld_cluster(part + (4 * i + k) * 128 + t, r);
    put(m0 + (t >> 5) * MP + i, n0 + (t & 31), v[0], v[1], v[2], v[3]);
  }
  __syncwarp();
  cluster_sync();   // no block leaves while another still reads its sums
}

}  // namespace dftk

using namespace dftk;

static int sm_count(const rf_ctx* c) {
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->dev);
  return sms;
}

static int dft_check(rf_ctx* c, cudaError_t e, const char* what) {
  if (e != cudaSuccess) return cuda_fail(e, what);
  c->launches += 1;
  e = cudaGetLastError();
  return e == cudaSuccess ? RF_OK : cuda_fail(e, what);
}

// Tables and block shape of the row pass for the current pattern (rows beyond kMaxX voxels keep the
// general row kernel).
int dft_setup(rf_ctx* c) {
  c->dft_U = 0;
  if (c->nx > kMaxX) return RF_OK;
  const int np = c->nx / 2 + 1, PT = (np + 1) / 2;
  const int sms = sm_count(c);
  const int units = c->nc == 3 ? (c->rows + 1) / 2 : c->rows;
  // two blocks per SM where the rows reach that far, then as many units as the threads hold
  int U = std::max(1, std::min((units + 2 * sms - 1) / (2 * sms), kThreads / PT));
  while (U > 1 && row_dft_smem(U, c->Kx, np) > 100 * 1024) --U;
  if (row_dft_smem(U, c->Kx, np) > 200 * 1024) return RF_OK;
  if (int e = palloc(c, &c->d_Wi, (size_t)np * c->Kx, "row tables")) return e;
  if (int e = palloc(c, &c->d_Wf, (size_t)np * c->Kx, "row tables")) return e;
  const int grid = (int)std::min<long long>(((long long)np * c->Kx + 255) / 256, 4096);
  k_row_tables<<<grid, 256, 0, c->stream>>>(c->d_twx, c->d_kx, c->nx, c->Kx, np, c->d_Wi, c->d_Wf);
  if (int e = dft_check(c, cudaGetLastError(), "row tables")) return e;
  c->dft_U = U;
  return RF_OK;
}

template <int NC, bool PL, bool FIN>
static int row_dft(rf_ctx* c, const RowDftArgs& a, int blocks, size_t smem) {
  if (FIN) {
    k_row_dft<NC, PL, FIN><<<blocks, kThreads, smem, c->stream>>>(a);
    return dft_check(c, cudaGetLastError(), "row");
  }
  return dft_check(c, launch_pdl(k_row_dft<NC, PL, FIN>, dim3(blocks), dim3(kThreads), smem,
                                 c->stream, a), "row");
}

// the row pass, or the final pass (its number of blocks to *blocks)
int launch_row_dft(rf_ctx* c, const int* done, bool final_pass, int commit, int* blocks) {
  RowDftArgs a{};
  a.T = c->d_T1;
  a.Tout = c->d_T1p;
  a.phase = c->d_phase;
  a.state = c->d_state;
  a.fac = c->d_fac;
  a.Wi = c->d_Wi;
  a.Wf = c->d_Wf;
  a.Nx = c->nx;
  a.Kx = c->Kx;
  a.rows = c->rows;
  a.np = c->nx / 2 + 1;
  a.PT = (a.np + 1) / 2;
  a.U = c->dft_U;
  a.SJ = std::max(1, std::min(8, kThreads / (a.U * a.PT)));
  a.JT = (c->Kx + 1) / 2;
  a.N = c->N;
  a.law = c->law;
  a.commit = commit;
  a.done = done;
  if (final_pass) {
    a.eps_out = c->d_eps;
    a.sig_out = c->d_sig;
    a.alpha_out = c->d_alpha;
    a.sbar_part = c->d_sbar_part;
    a.viol_part = c->d_viol_part;
  }
  const int units = c->nc == 3 ? (c->rows + 1) / 2 : c->rows;
  const int nb = (units + a.U - 1) / a.U;
  if (blocks) *blocks = nb;
  const size_t smem = row_dft_smem(a.U, a.Kx, a.np);
  // beside a grid of a few blocks the next kernel's prologue is free: up to 1 us per update (16 x 16,
  // 50 x 97), and no cell of 5 to 2000 a side was slower
  a.early = nb <= 32;
  const bool pl = c->has_plastic;
  if (c->nc == 3) {
    if (final_pass) return pl ? row_dft<3, true, true>(c, a, nb, smem) : row_dft<3, false, true>(c, a, nb, smem);
    return pl ? row_dft<3, true, false>(c, a, nb, smem) : row_dft<3, false, false>(c, a, nb, smem);
  }
  if (final_pass) return pl ? row_dft<6, true, true>(c, a, nb, smem) : row_dft<6, false, true>(c, a, nb, smem);
  return pl ? row_dft<6, true, false>(c, a, nb, smem) : row_dft<6, false, false>(c, a, nb, smem);
}

// sign +1: S sparse rows -> L dense ones, -1: the reverse (of `splits` partial sums); N columns,
// `batch` arrays
int launch_axis_dft(rf_ctx* c, const float2* in, int splits, long long split_stride,
                    long long in_bs, float2* out, long long out_bs, int L, int N, int S, int batch,
                    const int* vals, const float2* table, int sign, const int* done) {
  if (splits > 1) {   // partial sums of the row pass, which leaves its other output free
    const long long n = split_stride;
    const int grid = (int)std::min<long long>((n + 255) / 256, 8LL * sm_count(c));
    const cudaError_t e = launch_pdl(k_sum_slices, dim3(grid), dim3(256), 0, c->stream, in, splits,
                                     split_stride, n, c->d_T1p, done);
    if (int r = dft_check(c, e, "sum of slices")) return r;
    in = c->d_T1p;
  }
  AxisDftArgs a{};
  a.in = in;
  a.out = out;
  a.in_bstride = in_bs;
  a.out_bstride = out_bs;
  a.L = L;
  a.N = N;
  a.S = S;
  a.vals = vals;
  a.table = table;
  a.dL = make_fastdiv((unsigned)L);
  a.done = done;
  const int M = sign < 0 ? S : L / 2 + 1;
  const int sms = sm_count(c);
  // four rows per warp reuse a staged value twice as often; two where the grid would not give
  // every SM several blocks
  const long long b4 = (long long)((N + 31) / 32) * ((M + 15) / 16) * batch;
  const bool wide = b4 >= 4LL * sms;
  dim3 grid((N + 31) / 32, wide ? (M + 15) / 16 : (M + 7) / 8, batch);
  const long long blocks = (long long)grid.x * grid.y * batch;
  const int chunks = ((sign < 0 ? L / 2 + 1 : S) + kC - 1) / kC;
  a.ranks = 1;
  while (a.ranks < 8 && blocks * 2 * a.ranks <= sms && 2 * a.ranks <= chunks) a.ranks *= 2;
  grid.z *= a.ranks;
  // as in the row pass: 1 to 2 us per update of cells up to 200 x 190, none slower
  a.early = blocks * a.ranks <= 64;
  const auto kern = wide ? (sign < 0 ? k_axis_dft<4, true> : k_axis_dft<4, false>)
                         : (sign < 0 ? k_axis_dft<2, true> : k_axis_dft<2, false>);
  const cudaError_t e =
      launch_pdl_cluster(kern, grid, dim3(128), dim3(1, 1, a.ranks), 0, c->stream, a);
  return dft_check(c, e, "dft axis");
}

void init_attributes_dft() {
  const int s = 200 * 1024;
  for (const void* k : {(const void*)k_row_dft<3, false, false>, (const void*)k_row_dft<3, false, true>,
                        (const void*)k_row_dft<3, true, false>, (const void*)k_row_dft<3, true, true>,
                        (const void*)k_row_dft<6, false, false>, (const void*)k_row_dft<6, false, true>,
                        (const void*)k_row_dft<6, true, false>, (const void*)k_row_dft<6, true, true>})
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, s);
  cudaGetLastError();
}

}  // namespace rfk
