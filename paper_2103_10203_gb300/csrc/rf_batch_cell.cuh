// Cell-resident batched solve for RVEs of any sides (pruned DFTs): a block takes an RVE from a
// largest-first queue and runs all of its updates and its final pass with every array of the
// iteration in its shared memory. Included by rf_batch.cu inside its namespaces.
//
// A small RVE's update (85^2, K = 5 %: 0.9 MFMA, 33 KB of line transforms) is too little for a
// sweep of the grid: swept, 128 such RVEs took five launches and 110 us per update, with a
// modulo per twiddle and every stage's data through L2. Here only block barriers separate the
// stages, twiddles come from shared tables, points x and L - x share their products, and a
// thread holds two pairs (or two frequencies) of the six lines of two rows, as in the single-RVE
// pruned DFT. Blocks wait for nobody. What bounds it: instruction issue of one block per SM,
// and the largest RVE of the last wave. 128 RVEs with sides of 50 to 120: 3190 -> 1550 us a solve.

constexpr int kCellThreads = 512;
constexpr size_t kCellSmemMax = 220 * 1024;

// shared-memory layout of one RVE, in bytes
struct CellLayout {
  int np, npy, px, py, PT, units, U, JT, SX;
  int o_tl, o_er, o_out, o_wx, o_wy, o_uv, o_en, o_ei, o_fac, o_ph;
  size_t bytes;
};

__host__ __device__ inline CellLayout cell_layout(int nx, int ny, int Kx, int Ky, int Kh) {
  CellLayout c;
  c.np = nx / 2 + 1;
  c.npy = ny / 2 + 1;
  c.px = c.np | 1;    // odd pitches: neighbouring rows of a table on different banks
  c.py = c.npy | 1;
  c.PT = (c.np + 1) / 2;
  c.units = (ny + 1) / 2;
  c.U = kCellThreads / c.PT < c.units ? kCellThreads / c.PT : c.units;
  if (c.U < 1) c.U = 1;
  c.JT = (Kx + 1) / 2;
  c.SX = 1;
  while (c.SX < 8 && c.U * c.JT * 2 * c.SX <= kCellThreads) c.SX *= 2;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o += (bytes + 15) & ~(size_t)15;
    return (int)at;
  };
  c.o_tl = take((size_t)c.units * Kx * 6 * sizeof(float2));   // lines [unit][j][2 rows][3]
  c.o_er = take((size_t)Ky * Kx * 3 * sizeof(float2));        // coefficients [ky][j][3]
  c.o_out = take((size_t)Ky * Kx * 3 * sizeof(float2));
  c.o_wx = take((size_t)Kx * c.px * sizeof(float2));
  c.o_wy = take((size_t)Ky * c.py * sizeof(float2));
  c.o_uv = take((size_t)c.U * c.np * 12 * sizeof(float));
  c.o_en = take((size_t)Kh * sizeof(float4));
  c.o_ei = take((size_t)Kh * sizeof(int));
  c.o_fac = take((size_t)Kx * sizeof(float));
  c.o_ph = take((size_t)nx * ny);
  c.bytes = o;
  return c;
}

extern __shared__ __align__(16) unsigned char cell_smem[];

template <class T>
__device__ __forceinline__ T* cell_at(int off) {
  return reinterpret_cast<T*>(cell_smem + off);
}

// Row phase over all units of the RVE. FINAL: stress sums only.
template <bool FINAL>
__device__ __forceinline__ void cell_rows(const BDesc& d, const CellLayout& c, const DevPhase* phs,
                                          double* sb) {
  const int tid = threadIdx.x, Kx = d.Kx, np = c.np, PT = c.PT, L = d.nx;
  float2* TL = cell_at<float2>(c.o_tl);
  float* UV = cell_at<float>(c.o_uv);
  const float2* Wx = cell_at<float2>(c.o_wx);
  const uint8_t* ph8 = cell_at<uint8_t>(c.o_ph);
  for (int u0 = 0; u0 < c.units; u0 += c.U) {
    const int nu = min(c.U, c.units - u0);
    {
      const int uu = tid / PT, p = tid - uu * PT;
      if (uu < nu) {
        float A[2][6], B[2][6];
#pragma unroll
        for (int l = 0; l < 6; ++l) A[0][l] = A[1][l] = B[0][l] = B[1][l] = 0.f;
        const int x1 = p + PT < np ? PT : 0;
        const float2* w = Wx + p;
        const float4* t4 = reinterpret_cast<const float4*>(TL + (u0 + uu) * Kx * 6);
#pragma unroll 2
        for (int j = 0; j < Kx; ++j) {
          const float2 w0 = w[j * c.px], w1 = w[j * c.px + x1];
          const float4 t0 = t4[j * 3], t1 = t4[j * 3 + 1], t2 = t4[j * 3 + 2];
          const float re[6] = {t0.x, t0.z, t1.x, t1.z, t2.x, t2.z};
          const float im[6] = {t0.y, t0.w, t1.y, t1.w, t2.y, t2.w};
#pragma unroll
          for (int l = 0; l < 6; ++l) {
            A[0][l] = fmaf(re[l], w0.x, A[0][l]);
            B[0][l] = fmaf(im[l], w0.y, B[0][l]);
            A[1][l] = fmaf(re[l], w1.x, A[1][l]);
            B[1][l] = fmaf(im[l], w1.y, B[1][l]);
          }
        }
        // the law at the points x and L - x of both pairs, both rows
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int x = p + q * PT;
          if (x >= np) continue;
          const bool self = x == 0 || 2 * x == L;
          float2* uv = reinterpret_cast<float2*>(UV + (uu * np + x) * 12);
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const int row = 2 * (u0 + uu) + r;
            float tau[2][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
            if (row < d.ny) {
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                if (h == 1 && self) break;
                const DevPhase& ph = phs[ph8[row * L + (h ? L - x : x)]];
                float e6[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                  const float va = A[q][3 * r + i], vb = B[q][3 * r + i];
                  e6[comp6<3>(i)] = h ? va + vb : va - vb;
                }
                const float ep[6] = {0, 0, 0, 0, 0, 0};
                LawOut o;
                stress6<false>(e6, ph, ep, 0.f, o);
                if (FINAL) {
#pragma unroll
                  for (int i = 0; i < 6; ++i) sb[i] += (double)o.s[i];
                } else {
                  const float lt = d.lam0 * (e6[0] + e6[1]);
                  tau[h][0] = o.s[0] - (lt + 2.f * d.mu0 * e6[0]);
                  tau[h][1] = o.s[1] - (lt + 2.f * d.mu0 * e6[1]);
                  tau[h][2] = o.s[5] - 2.f * d.mu0 * e6[5];
                }
              }
            }
            if (!FINAL) {
#pragma unroll
              for (int i = 0; i < 3; ++i)
                uv[3 * r + i] = self ? make_float2(tau[0][i], 0.f)
                                     : make_float2(tau[0][i] + tau[1][i], tau[0][i] - tau[1][i]);
            }
          }
        }
      }
    }
    if (FINAL) continue;
    __syncthreads();
    {
      // two frequencies of six lines per thread, the pairs split over SX neighbouring lanes
      const int s = tid & (c.SX - 1), f = tid / c.SX;
      const int uu = f / c.JT, jt = f - uu * c.JT;
      const bool on = uu < nu;
      float re[2][6], im[2][6];
#pragma unroll
      for (int l = 0; l < 6; ++l) re[0][l] = re[1][l] = im[0][l] = im[1][l] = 0.f;
      const bool two = jt + c.JT < Kx;
      if (on) {
        const float2* w0p = Wx + jt * c.px;
        const float2* w1p = w0p + (two ? c.JT * c.px : 0);
        const float4* u4 = reinterpret_cast<const float4*>(UV) + uu * np * 3;
#pragma unroll 2
        for (int x = s; x < np; x += c.SX) {
          const float2 w0 = w0p[x], w1 = w1p[x];
          const float4 t0 = u4[x * 3], t1 = u4[x * 3 + 1], t2 = u4[x * 3 + 2];
          const float u[6] = {t0.x, t0.z, t1.x, t1.z, t2.x, t2.z};
          const float v[6] = {t0.y, t0.w, t1.y, t1.w, t2.y, t2.w};
#pragma unroll
          for (int l = 0; l < 6; ++l) {
            re[0][l] = fmaf(u[l], w0.x, re[0][l]);
            im[0][l] = fmaf(v[l], w0.y, im[0][l]);
            re[1][l] = fmaf(u[l], w1.x, re[1][l]);
            im[1][l] = fmaf(v[l], w1.y, im[1][l]);
          }
        }
      }
      for (int o = 1; o < c.SX; o <<= 1)
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int l = 0; l < 6; ++l) {
            re[q][l] += __shfl_xor_sync(0xffffffffu, re[q][l], o);
            im[q][l] += __shfl_xor_sync(0xffffffffu, im[q][l], o);
          }
      if (on && s == 0) {
        float2* o = TL + ((u0 + uu) * Kx + jt) * 6;
#pragma unroll
        for (int l = 0; l < 6; ++l) o[l] = make_float2(re[0][l], -im[0][l]);
        if (two)
#pragma unroll
          for (int l = 0; l < 6; ++l) o[c.JT * 6 + l] = make_float2(re[1][l], -im[1][l]);
      }
    }
    __syncthreads();
  }
}

// forward along y: lines -> OUT on the pattern's ky rows, four of them per task
__device__ __forceinline__ void cell_fwd_y(const BDesc& d, const CellLayout& c) {
  constexpr int MP = 4;
  const int NCK = 3 * d.Kx, Kx6 = d.Kx * 6, L = d.ny;
  const float2* TL = cell_at<float2>(c.o_tl);
  const float2* Wy = cell_at<float2>(c.o_wy);
  float2* OUT = cell_at<float2>(c.o_out);
  const int tasks = NCK * ((d.Ky + MP - 1) / MP);
  for (int t = threadIdx.x; t < tasks; t += kCellThreads) {
    const int g = t / NCK, n = t - g * NCK, j = n / 3, i = n - 3 * j;
    const float2* col = TL + j * 6 + i;
    float ar[MP], ai[MP], br[MP], bi[MP];
    const float2* w[MP];
#pragma unroll
    for (int m = 0; m < MP; ++m) {
      ar[m] = ai[m] = br[m] = bi[m] = 0.f;
      w[m] = Wy + min(g * MP + m, d.Ky - 1) * c.py;
    }
#pragma unroll 2
    for (int y = 0; y < c.npy; ++y) {
      float2 p = col[(y >> 1) * Kx6 + (y & 1) * 3], q = make_float2(0.f, 0.f);
      if (y > 0 && 2 * y != L) {
        const int z = L - y;
        const float2 v = col[(z >> 1) * Kx6 + (z & 1) * 3];
        q = make_float2(p.x - v.x, p.y - v.y);
        p = make_float2(p.x + v.x, p.y + v.y);
      }
#pragma unroll
      for (int m = 0; m < MP; ++m) {
        const float2 e = w[m][y];
        ar[m] = fmaf(p.x, e.x, ar[m]);
        ai[m] = fmaf(p.y, e.x, ai[m]);
        br[m] = fmaf(q.y, e.y, br[m]);
        bi[m] = fmaf(q.x, e.y, bi[m]);
      }
    }
#pragma unroll
    for (int m = 0; m < MP; ++m)
      if (g * MP + m < d.Ky)
        OUT[(g * MP + m) * NCK + n] = make_float2(ar[m] + br[m], ai[m] - bi[m]);
  }
}

// inverse along y: coefficients -> lines (scaled by weight / N for the transform along x), four
// pairs (y, L - y) per task
__device__ __forceinline__ void cell_inv_y(const BDesc& d, const CellLayout& c) {
  constexpr int MP = 4;
  const int NCK = 3 * d.Kx, Kx6 = d.Kx * 6, L = d.ny;
  float2* TL = cell_at<float2>(c.o_tl);
  const float2* Wy = cell_at<float2>(c.o_wy);
  const float2* ER = cell_at<float2>(c.o_er);
  const float* fac = cell_at<float>(c.o_fac);
  const int tasks = NCK * ((c.npy + MP - 1) / MP);
  for (int t = threadIdx.x; t < tasks; t += kCellThreads) {
    const int g = t / NCK, n = t - g * NCK, j = n / 3, i = n - 3 * j;
    float ar[MP], ai[MP], br[MP], bi[MP];
    int y[MP];
#pragma unroll
    for (int m = 0; m < MP; ++m) {
      ar[m] = ai[m] = br[m] = bi[m] = 0.f;
      y[m] = min(g * MP + m, c.npy - 1);
    }
#pragma unroll 2
    for (int k = 0; k < d.Ky; ++k) {
      const float2 x = ER[k * NCK + n];
      const float2* w = Wy + k * c.py;
#pragma unroll
      for (int m = 0; m < MP; ++m) {
        const float2 e = w[y[m]];
        ar[m] = fmaf(x.x, e.x, ar[m]);
        ai[m] = fmaf(x.y, e.x, ai[m]);
        br[m] = fmaf(x.y, e.y, br[m]);
        bi[m] = fmaf(x.x, e.y, bi[m]);
      }
    }
    float2* col = TL + j * 6 + i;
    const float f = fac[j];
#pragma unroll
    for (int m = 0; m < MP; ++m) {
      const int p = g * MP + m;
      if (p >= c.npy) break;
      col[(p >> 1) * Kx6 + (p & 1) * 3] = make_float2(f * (ar[m] - br[m]), f * (ai[m] + bi[m]));
      if (p > 0 && 2 * p != L) {
        const int z = L - p;
        col[(z >> 1) * Kx6 + (z & 1) * 3] = make_float2(f * (ar[m] + br[m]), f * (ai[m] - bi[m]));
      }
    }
  }
}

__global__ __launch_bounds__(kCellThreads, 1) void kb_cell(BArgs a, const int* order, int n,
                                                           unsigned* queue) {
  __shared__ BDesc d;
  __shared__ DevPhase phs[kMaxPhases];
  __shared__ double red[32];
  __shared__ double ebar[6];
  __shared__ int s_rve, s_done;
  const int tid = threadIdx.x;
  for (int i = tid; i < kMaxPhases; i += kCellThreads) phs[i] = a.law.ph[i];
  for (;;) {
    __syncthreads();   // the previous RVE's reads are done
    if (tid == 0) {
      const unsigned q = atomicAdd(queue, 1u);
      s_rve = q < (unsigned)n ? order[q] : -1;
      if (s_rve >= 0) d = a.d[s_rve];
    }
    __syncthreads();
    const int rve = s_rve;
    if (rve < 0) return;
    const CellLayout c = cell_layout(d.nx, d.ny, d.Kx, d.Ky, d.Kh);
    BStat& st = a.st[rve];
    const int Kx = d.Kx, NCK = 3 * Kx;
    float2* ER = cell_at<float2>(c.o_er);
    const float2* OUT = cell_at<float2>(c.o_out);
    float4* en = cell_at<float4>(c.o_en);
    int* ei = cell_at<int>(c.o_ei);
    // tables, phase ids, entries and the start coefficients
    for (int i = tid; i < Kx * c.np; i += kCellThreads) {
      const int j = i / c.np, x = i - j * c.np;
      cell_at<float2>(c.o_wx)[j * c.px + x] =
          a.tab[d.tab_x + (int)(((long long)a.kx[d.off_kx + j] * x) % d.nx)];
    }
    for (int i = tid; i < d.Ky * c.npy; i += kCellThreads) {
      const int k = i / c.npy, y = i - k * c.npy;
      cell_at<float2>(c.o_wy)[k * c.py + y] =
          a.tab[d.tab_y + (int)(((long long)a.kym[d.off_ky + k] * y) % d.ny)];
    }
    for (int i = tid; i < d.nx * d.ny; i += kCellThreads)
      cell_at<uint8_t>(c.o_ph)[i] = a.phase[d.off_phase + i];
    for (int i = tid; i < d.Kh; i += kCellThreads) {
      const HIdx hi = a.hidx[d.off_h + i];
      en[i] = a.hn[d.off_h + i];
      ei[i] = (hi.iy * Kx + hi.j) | (hi.kind << 28);
    }
    for (int i = tid; i < Kx; i += kCellThreads) cell_at<float>(c.o_fac)[i] = a.fac[d.off_kx + i];
    for (int i = tid; i < d.Ky * NCK; i += kCellThreads) {
      const int iy = i / NCK, m = i - iy * NCK, q = m / Kx, j = m - q * Kx;   // [iy][c][j]
      ER[iy * NCK + j * 3 + q] = a.ER[d.off_er + i];
    }
    // an odd last row has no partner: its unit's second row stays zero through the transforms
    for (int i = tid; i < c.units * Kx * 6; i += kCellThreads)
      cell_at<float2>(c.o_tl)[i] = make_float2(0.f, 0.f);
    if (tid < 6) ebar[tid] = st.ebar[tid];
    int iters = 0;
    double rmin = 0.0, last_r = 0.0;
    int nonfinite = 0, diverged = 0;
    if (tid == 0) {
      iters = st.iters;
      rmin = st.rmin;
    }
    __syncthreads();
    cell_inv_y(d, c);
    __syncthreads();
    for (;;) {
      cell_rows<false>(d, c, phs, nullptr);
      cell_fwd_y(d, c);
      __syncthreads();
      double dsum = 0.0;
      for (int e = tid; e < d.Kh; e += kCellThreads) {
        const int code = ei[e], kind = (unsigned)code >> 28, base = (code & 0x0fffffff) * 3;
        const float4 nv = en[e];
        float2 tv[3], old[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          tv[q] = OUT[base + q];
          old[q] = ER[base + q];
        }
        float er[3], em[3];
        green_update<3>(kind, nv, tv, ebar, (double)d.N, d.inv2mu0, d.cgam, er, em);
        float diff = 0.f;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const float dr = er[q] - old[q].x, di = em[q] - old[q].y;
          const float wc = comp6<3>(q) >= 3 ? 2.f : 1.f;
          diff = fmaf(nv.w * wc, dr * dr + di * di, diff);
          ER[base + q] = make_float2(er[q], em[q]);
        }
        dsum += (double)diff;
      }
      const double s = block_sum_d(dsum, red);   // its barriers order the coefficients
      if (tid == 0) {
        double r = sqrt(s * st.inv_n2);
        if (st.enorm > 0.0) r /= st.enorm;
        iters += 1;
        last_r = r;
        rmin = fmin(rmin, r);
        int done = 0;
        if (!isfinite(r)) nonfinite = done = 1;
        else if (r > kDivergeRatio * rmin && r > kDivergeFloor) diverged = done = 1;
        else if (r < st.tol || iters >= st.max_iter) done = 1;
        s_done = done;
      }
      cell_inv_y(d, c);
      __syncthreads();
      if (s_done) break;
    }
    double sb[6] = {0, 0, 0, 0, 0, 0};
    cell_rows<true>(d, c, phs, sb);
    for (int q = 0; q < 6; ++q) {
      const double t = block_sum_d(sb[q], red);
      if (tid == 0) st.sbar[q] = t / (double)d.N;
    }
    for (int i = tid; i < d.Ky * NCK; i += kCellThreads) {
      const int iy = i / NCK, m = i - iy * NCK, q = m / Kx, j = m - q * Kx;
      a.ER[d.off_er + i] = ER[iy * NCK + j * 3 + q];
    }
    if (tid == 0) {
      st.iters = iters;
      st.last_r = last_r;
      st.rmin = rmin;
      st.nonfinite = nonfinite;
      st.diverged = diverged;
      st.done = 1;
      atomicAdd(a.n_done, 1);
    }
  }
}
