// Host side of the 3D updates on team FFTs (rf_fft3.cuh).
#include <vector>

#include "rf_fft3.cuh"

namespace rfk {

using namespace fft3;

namespace {

constexpr int kSmem3 = 200 * 1024;

struct Shape3 {
  int lanes, tw, cols, kx;   // threads per sequence, twiddles, and what a block takes
};

bool shape_of(int L, Shape3* s) {
  switch (L) {
#define X(L_, R, M)                                                                              \
  case L_:                                                                                       \
    *s = Shape3{R * M, Plan<R, M>::kTw, cols_per_block<R, M>(), kx_per_block<R, M>()};           \
    return true;
    RF_TEAM_SIDES(X)
#undef X
  }
  return false;
}

int even_span(int L) { return (L + L / 16 + 2) & ~1; }
int odd_pitch(int L) { return (L + L / 16 + 2) | 1; }

// blocks that fill the device once, at most `want`
int fill(const rf_ctx* c, const void* k, int threads, size_t smem, long long want) {
  int sms = 152, occ = 1;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, threads, smem) != cudaSuccess) {
    cudaGetLastError();
    occ = 1;
  }
  return (int)std::max(1LL, std::min<long long>(want, (long long)std::max(1, occ) * sms));
}

int done3(rf_ctx* c, cudaError_t e, const char* what) {
  if (e != cudaSuccess) return cuda_fail(e, what);
  c->launches += 1;
  e = cudaGetLastError();
  return e == cudaSuccess ? RF_OK : cuda_fail(e, what);
}

}  // namespace

bool fft3_yz_ok(const rf_ctx* c) {
  Shape3 s;
  return c->dim == 3 && c->nc == 6 && shape_of(c->ny, &s) && shape_of(c->nz, &s) && c->d_zrange;
}

bool fft3_ok(const rf_ctx* c) {
  Shape3 s;
  return fft3_yz_ok(c) && c->opt.transform == RF_TRANSFORM_FFT && shape_of(c->nx, &s);
}

// Pattern tables: first half-pattern entry and count of every (ky, kx) (the half pattern is sorted
// by kx, ky, kz), and the rectangle row of each position along y.
int fft3_setup(rf_ctx* c, const int* kym) {
  Shape3 s;
  if (c->dim != 3 || !shape_of(c->ny, &s) || !shape_of(c->nz, &s)) return RF_OK;
  std::vector<int2> range((size_t)c->Ky * c->Kx, make_int2(0, 0));
  for (long long h = 0; h < c->Kh; ++h) {
    int2& r = range[(size_t)c->h_hidx[h].iy * c->Kx + c->h_hidx[h].j];
    if (r.y == 0) r.x = (int)h;
    r.y += 1;
  }
  std::vector<short> ymap(c->ny, -1);
  for (int i = 0; i < c->Ky; ++i) ymap[kym[i]] = (short)i;
  if (int e = palloc(c, &c->d_zrange, range.size(), "pattern")) return e;
  if (int e = palloc(c, &c->d_ymap, ymap.size(), "pattern")) return e;
  // (the second copy waits for both)
  cudaError_t e = cudaMemcpyAsync(c->d_zrange, range.data(), sizeof(int2) * range.size(),
                                  cudaMemcpyHostToDevice, c->stream);
  if (e == cudaSuccess) e = upload(c->d_ymap, ymap.data(), sizeof(short) * ymap.size(), c->stream);
  return e == cudaSuccess ? RF_OK : cuda_fail(e, "pattern");
}

void init_attributes_fft3() {
#define X(L, R, M)                                                                               \
  for (const void* k : {(const void*)row_kernel_elastic(L, false),                               \
                        (const void*)row_kernel_elastic(L, true),                                \
                        (const void*)row_kernel_plastic(L, false),                               \
                        (const void*)row_kernel_plastic(L, true), (const void*)col_kernel(L, 1), \
                        (const void*)col_kernel(L, -1), (const void*)z_kernel(L)})               \
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem3);
  RF_TEAM_SIDES(X)
#undef X
  cudaGetLastError();
}

int launch_fft3_row(rf_ctx* c, const int* done, bool final_pass, int commit, int* blocks) {
  Shape3 s;
  shape_of(c->nx, &s);
  RowArgs3 a{};
  a.T = c->d_T1;
  a.Tout = c->d_T1p;
  a.phase = c->d_phase;
  a.state = c->d_state;
  a.kx = c->d_kx;
  a.table = c->d_twx;
  a.Kx = c->Kx;
  a.rows = c->rows;
  a.teams = row_teams(s.lanes);
  a.groups = (c->rows + a.teams - 1) / a.teams;
  a.N = c->N;
  a.invN = (float)(1.0 / (double)c->N);
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
  RowKernel k = c->has_plastic ? row_kernel_plastic(c->nx, final_pass)
                               : row_kernel_elastic(c->nx, final_pass);
  const int threads = row_threads(s.lanes);
  const size_t smem = sizeof(float2) * (((s.tw + 1) & ~1) + (size_t)a.teams * 3 * even_span(c->nx)) +
                      sizeof(int) * c->Kx + sizeof(short) * (c->nx / 2 + 1) + 16;
  const int grid = fill(c, (const void*)k, threads, smem, a.groups);
  if (blocks) *blocks = grid;
  if (final_pass) {
    k<<<grid, threads, smem, c->stream>>>(a);
    return done3(c, cudaGetLastError(), "3D final pass");
  }
  return done3(c, launch_pdl(k, dim3(grid), dim3(threads), smem, c->stream, a), "3D row pass");
}

// sign +1: T2 -> T1 (sparse rows in), -1: T1p (or `splits` partial sums at `in`) -> T2f (sparse rows
// out)
int launch_fft3_y(rf_ctx* c, int sign, const int* done, const float2* in, int splits,
                  long long split_stride) {
  Shape3 s;
  shape_of(c->ny, &s);
  const int NCK = c->nc * c->Kx;
  const long long sparse = (long long)c->Ky * NCK, dense = (long long)c->ny * NCK;
  ColArgs3 a{};
  a.in = sign > 0 ? c->d_T2 : in ? in : c->d_T1p;
  a.splits = splits;
  a.split_stride = split_stride;
  a.out = sign > 0 ? c->d_T1 : c->d_T2f;
  a.in_bstride = sign > 0 ? sparse : dense;
  a.out_bstride = sign > 0 ? dense : sparse;
  a.map = c->d_ymap;
  a.table = c->d_twy;
  a.ncols = NCK;
  a.cgroups = (NCK + s.cols - 1) / s.cols;
  a.total = a.cgroups * c->nz;
  a.done = done;
  ColKernel k = col_kernel(c->ny, sign);
  const int threads = s.cols * s.lanes;
  const size_t smem = sizeof(float2) * (s.tw + 2 * (size_t)s.cols * odd_pitch(c->ny)) +
                      sizeof(short) * c->ny + 16;
  const int grid = fill(c, (const void*)k, threads, smem, a.total);
  return done3(c, launch_pdl(k, dim3(grid), dim3(threads), smem, c->stream, a), "3D y transform");
}

// full = false: only the inverse along z of the held coefficients (ER -> T2)
int launch_fft3_z(rf_ctx* c, bool full, const int* done) {
  Shape3 s;
  shape_of(c->nz, &s);
  ZArgs a{};
  a.in = c->d_T2f;
  a.out = c->d_T2;
  a.ER = c->d_ER;
  a.range = c->d_zrange;
  a.hidx = c->d_hidx;
  a.hn = c->d_hn;
  a.kzm = c->d_kzm;
  a.table = c->d_twz;
  a.Kx = c->Kx;
  a.Ky = c->Ky;
  a.jgroups = (c->Kx + s.kx - 1) / s.kx;
  a.inv2mu0 = (float)(0.5 / c->mu0);
  a.cgam = (float)((c->lam0 + c->mu0) / (c->mu0 * (c->lam0 + 2.0 * c->mu0)));
  a.Nd = (double)c->N;
  a.st = c->d_status;
  a.counter = c->d_counter;
  a.part = c->d_part;
  a.done = done;
  a.cond = c->while_cond;
  a.use_cond = c->capturing_while ? 1 : 0;
  a.full = full ? 1 : 0;
  ZKernel k = z_kernel(c->nz);
  const int threads = 6 * s.kx * s.lanes;
  const size_t smem = sizeof(float2) * (s.tw + 2 * (size_t)(6 * s.kx) * odd_pitch(c->nz)) + 16;
  const dim3 grid((unsigned)(c->Ky * a.jgroups));
  return done3(c, launch_pdl(k, grid, dim3(threads), smem, c->stream, a), "3D z phase");
}

}  // namespace rfk
