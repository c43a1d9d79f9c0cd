// Host side of the persistent 2D solve on team FFTs (rf_team.cuh), and its final pass.
#include "rf_team.cuh"

namespace rfk {
namespace team {

// Final pass: fields, homogenised-stress partials, commit; nothing after a solve that failed.
template <bool PLASTIC>
__global__ __launch_bounds__(kMaxWorkers) void k_team_final(const __grid_constant__ Args a) {
  __shared__ double red[kMaxWorkers / 32][8];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  double sb[7] = {0, 0, 0, 0, 0, 0, 0};   // stresses, violation
  if (!(a.st->nonfinite || a.st->diverged || a.st->timeout)) {   // the same for every thread
    fill_rows(a);
    __syncthreads();
    rows<0, PLASTIC, true>(a, sb);
  }
  auto add = [](int i, double x, double y) { return i < 6 ? x + y : fmax(x, y); };
  // fixed orders throughout: lanes, warps, then blocks
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < 7; ++i) sb[i] = add(i, sb[i], __shfl_down_sync(0xffffffffu, sb[i], o));
  if (lane == 0)
#pragma unroll
    for (int i = 0; i < 7; ++i) red[warp][i] = sb[i];
  __syncthreads();
  if (threadIdx.x < 7) {
    double s = red[0][threadIdx.x];
    for (int w = 1; w < nw; ++w) s = add(threadIdx.x, s, red[w][threadIdx.x]);
    a.fin_part[blockIdx.x * 8 + threadIdx.x] = s;
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(a.fin_count, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  // the last block: component i of the blocks r, r + rows, ... per thread 8 r + i
  __threadfence();
  const int i = threadIdx.x & 7, r = threadIdx.x >> 3, rows = blockDim.x >> 3;
  double s = 0.0;
  if (i < 7)
    for (int b = r; b < (int)gridDim.x; b += rows) s = add(i, s, __ldcg(a.fin_part + b * 8 + i));
  s = add(i, s, __shfl_down_sync(0xffffffffu, s, 16));
  s = add(i, s, __shfl_down_sync(0xffffffffu, s, 8));
  if (lane < 8) red[warp][lane] = s;
  __syncthreads();
  if (threadIdx.x < 7) {
    double t = red[0][i];
    for (int w = 1; w < nw; ++w) t = add(i, t, red[w][i]);
    if (i < 6) t /= a.Nd;
    a.sbar_dev[i] = t;
    a.sbar_host[i] = t;
  }
  if (threadIdx.x == 0) *a.fin_count = 0u;
  // the status as the solve left it, for the host to read after its wait
  for (int w = threadIdx.x; w < (int)(sizeof(Status) / 4); w += blockDim.x)
    reinterpret_cast<int*>(a.st_host)[w] = reinterpret_cast<const int*>(a.st)[w];
}

// ------------------------------------------------------------------------------------------
// host side
namespace {

constexpr size_t kSmemMax = 220 * 1024;

// threads of one sequence (0: the side is not handled) and twiddles of its passes
int lanes_of(int L) {
  switch (L) {
#define X(L_, R, M) \
  case L_: return R * M;
    RF_TEAM_SIDES_2D(X)
#undef X
  }
  return 0;
}
int twiddles_of(int L) {
  switch (L) {
#define X(L_, R, M) \
  case L_: return Plan<R, M>::kTw;
    RF_TEAM_SIDES_2D(X)
#undef X
  }
  return 0;
}

Kernel solve_kernel(const rf_ctx* c) {
  const int side = c->nx == c->ny ? c->nx : 0;
  Kernel k = side ? (c->has_plastic ? kernel_plastic(side) : kernel_elastic(side)) : nullptr;
  return k ? k : kernel_any(c->has_plastic);
}

// Block shape of a launch on G blocks with `W` workers at most: teams per block, rounds, shared
// memory; false if a round's teams or the shared memory do not fit.
bool shape_with(const rf_ctx* c, int G, bool final_pass, bool stream, Args& a, size_t* smem) {
  // the kernels of long square cells carry three sequences per thread of the row phase
  const bool three = !final_pass && c->nx == c->ny && three_in_one(c->nx);
  const int cap = three ? kMaxWorkers3 : kMaxWorkers;
  const int gx = (three ? 1 : 3) * lanes_of(c->nx), gy = 3 * lanes_of(c->ny);
  const int units = c->ny / 2;
  const int ux = (units + G - 1) / G, uy = (c->Kx + G - 1) / G;   // per block, at most
  auto teams = [cap](int want, int g) { return std::max(1, std::min(want, cap / g)); };
  a.Px = teams(ux, gx);
  a.Py = final_pass ? 1 : teams(uy, gy);
  a.rounds_x = (ux + a.Px - 1) / a.Px;
  a.rounds_y = (uy + a.Py - 1) / a.Py;
  const int w = std::max(a.Px * gx, final_pass ? 0 : a.Py * gy);
  a.W = (w + 31) & ~31;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t at = o;
    o += (bytes + 15) & ~(size_t)15;
    return (int)at;
  };
  a.o_ph = take(sizeof(DevPhase) * kMaxPhases);
  a.o_twx = take(sizeof(float2) * twiddles_of(c->nx));
  a.o_kx = take(sizeof(int) * c->Kx);
  a.o_jmap = take(sizeof(short) * (c->nx / 2 + 1));
  const size_t bx = (size_t)a.Px * (three ? 3 : 6) * (c->nx + c->nx / 16 + 2);
  const size_t by = final_pass ? 0 : (size_t)a.Py * 6 * (c->ny + c->ny / 16 + 2);
  a.o_buf = take(sizeof(float2) * std::max(bx, by));
  if (!final_pass) {
    // (a square cell's transforms share the table)
    a.o_twy = c->nx == c->ny ? a.o_twx : take(sizeof(float2) * twiddles_of(c->ny));
    a.o_red = take(sizeof(double) * a.W);
    a.o_eb = take(sizeof(double) * 8);
    const int nslot = a.Py * a.rounds_y;
    a.o_w = take(sizeof(float2) * 3 * (size_t)nslot * c->ny);
    a.o_slot = take(sizeof(int) * (nslot + 1));
    a.entries_cap = 0;
    for (int b = 0; b < G && b < c->Kx; ++b) {
      int n = 0;
      for (int j = b; j < c->Kx; j += G) n += c->h_jcount[j];
      a.entries_cap = std::max(a.entries_cap, n);
    }
    a.o_en = take(sizeof(float4) * a.entries_cap);
    a.o_ep = take(sizeof(int) * a.entries_cap);
    a.st_stream = stream;
    a.o_p8 = take((size_t)a.Px * a.rounds_x * 2 * c->nx);
    const int held = stream ? (three ? 0 : 1) : a.rounds_x;   // row pairs of a team
    a.o_st = take(!c->has_plastic ? 0 : (size_t)a.Px * held * 2 * c->nx * 16);
    if (a.cluster) {
      a.o_ts = take(sizeof(float4) * 3 * (size_t)a.Px * a.rounds_x * c->Kx);
      a.o_tp = take(sizeof(float2) * 3 * (size_t)nslot * c->ny);
    }
  }
  *smem = o;
  // (the long square cells have no cluster form)
  return gx <= cap && gy <= cap && o <= kSmemMax && !(three && a.cluster);
}

bool shape(const rf_ctx* c, int G, bool final_pass, Args& a, size_t* smem) {
  return shape_with(c, G, final_pass, c->team_stream, a, smem);
}

Args make_args(rf_ctx* c) {
  Args a{};
  a.T1 = c->d_T1;
  a.T1p = c->d_T1p;
  a.ER = c->d_ER;
  a.phase = c->d_phase;
  a.state = c->d_state;
  a.kx = c->d_kx;
  a.twx = c->d_twx;
  a.twy = c->d_twy;
  a.jptr = c->d_jptr;
  a.jent = c->d_jent;
  a.jn = c->d_jn;
  a.kym = c->d_kym;
  a.Nx = c->nx;
  a.Ny = c->ny;
  a.Kx = c->Kx;
  a.N = c->N;
  a.invN = (float)(1.0 / (double)c->N);
  a.law = c->law;
  a.inv2mu0 = (float)(0.5 / c->mu0);
  a.cgam = (float)((c->lam0 + c->mu0) / (c->mu0 * (c->lam0 + 2.0 * c->mu0)));
  a.Nd = (double)c->N;
  a.st = c->d_status;
  a.part = c->d_part;
  a.fin_part = c->d_fin;
  a.fin_count = c->d_bar + 2;   // (the other persistent solves leave a generation in the second word)
  a.sbar_dev = c->d_sbar;
  a.sbar_host = c->h_sbar;
  a.st_host = c->h_status;
  a.bar = c->d_bar;
  a.bar_limit = 1L << 26;
  return a;
}

int sm_count(const rf_ctx* c) {
  int sms = 152;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, c->dev);
  return sms;
}

}  // namespace
}  // namespace team

using namespace team;

// Whether the team solve takes this pattern at all (sides of the plans, plane strain).
bool team_ok(const rf_ctx* c) {
  return c->dim == 2 && c->nc == 3 && c->d_jptr && c->d_bar && lanes_of(c->nx) > 0 &&
         lanes_of(c->ny) > 0 && !c->h_jcount.empty();
}

// Chooses the launch: cluster = 0, a co-resident grid with one row pair per block as far as the
// device holds it; else one cluster of that many blocks. False if it does not fit.
bool team_geometry(rf_ctx* c, int cluster) {
  if (!team_ok(c)) return false;
  const void* k = (const void*)solve_kernel(c);
  Args a{};
  size_t smem = 0;
  const int units = c->ny / 2;
  c->team_stream = false;
  if (cluster > 0) {
    a.cluster = 1;
    if (cluster > units || !shape(c, cluster, false, a, &smem)) return false;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster);
    cfg.blockDim = dim3(a.W + 32);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess || n < 1) {
      cudaGetLastError();
      return false;
    }
    c->team_G = cluster;
    c->team_threads = a.W;
  } else {
    const int sms = sm_count(c);
    bool found = false;
    // as many blocks per SM as it takes to give each a row pair of its own; internal variables
    // held where that leaves room for them, else streamed
    for (int q = 0; q < 8 && !found; ++q) {
      const int per = 4 - q / 2;
      c->team_stream = q & 1;
      if (c->team_stream && !c->has_plastic) continue;
      const int G = std::min(units, per * sms);
      if (per > 1 && G <= (per - 1) * sms) continue;   // fewer blocks per SM hold it
      int occ = 0;
      if (!shape(c, G, false, a, &smem)) continue;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k, a.W + 32, smem) != cudaSuccess) {
        cudaGetLastError();
        continue;
      }
      if ((long long)occ * sms < G) continue;
      c->team_G = G;
      c->team_threads = a.W;
      found = true;
    }
    if (!found) return false;
  }
  c->team_cluster = cluster;
  return true;
}

void init_attributes_team() {
  std::vector<Kernel> all = {kernel_any(true), kernel_any(false)};
#define X(L, R, M) \
  all.push_back(kernel_plastic(L)); \
  all.push_back(kernel_elastic(L));
  RF_TEAM_SIDES_2D(X)
#undef X
  for (Kernel k : all) {
    cudaFuncSetAttribute((const void*)k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
    cudaFuncSetAttribute((const void*)k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  }
  for (const void* k : {(const void*)k_team_final<true>, (const void*)k_team_final<false>})
    cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
  cudaGetLastError();   // a refused attribute only narrows the geometries that fit
}

// What a solve starts from in one launch: the status, the arrivals of the grid barrier, and (plain
// start, mode 0) zeroed coefficients with the zero frequency at N v; mode 1 adds N v there, mode 2
// leaves the coefficients.
__global__ __launch_bounds__(256) void k_team_begin(Status s, Status* st, unsigned* bar, float2* ER,
                                                    long long rect, long long base0, int Kx,
                                                    double Nd, double v0, double v1, double v2,
                                                    int mode) {
  const long long i0 = blockIdx.x * 256LL + threadIdx.x;
  if (mode == 0)
    for (long long i = i0; i < rect; i += gridDim.x * 256LL) {
      float2 v = make_float2(0.f, 0.f);
      const long long d = i - base0;
      if (d >= 0 && d <= 2LL * Kx && d % Kx == 0)
        v.x = (float)(Nd * (d == 0 ? v0 : d == Kx ? v1 : v2));
      ER[i] = v;
    }
  if (blockIdx.x == 0) {
    if (mode == 1 && threadIdx.x < 3) {
      float2* p = ER + base0 + (long long)threadIdx.x * Kx;
      p->x = (float)((double)p->x + Nd * (threadIdx.x == 0 ? v0 : threadIdx.x == 1 ? v1 : v2));
    }
    if (threadIdx.x == 32) *bar = 0u;
    if (threadIdx.x == 64) *st = s;
  }
}

// One launch: the start's inverse along y, then updates until the decision ends the solve.
int launch_team_solve(rf_ctx* c, unsigned long long* trace, int trace_cap) {
  Args a = make_args(c);
  size_t smem = 0;
  a.cluster = c->team_cluster > 0;
  if (!shape(c, c->team_G, false, a, &smem)) {
    set_error("team solve: the launch does not fit");
    return RF_ERR_INVALID;
  }
  a.trace = trace;
  a.trace_cap = trace_cap;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(c->team_G);
  cfg.blockDim = dim3(a.W + 32);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = c->stream;
  cudaLaunchAttribute at[1];
  if (a.cluster) {
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = c->team_G;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  } else {
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
  }
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, solve_kernel(c), a);
  c->launches += 1;
  return e == cudaSuccess ? RF_OK : cuda_fail(e, "team solve");
}

// mode as k_team_begin's; macro: the six components of the start or of the increment
int launch_team_begin(rf_ctx* c, const double* macro, int mode) {
  const int blocks = mode == 0 ? (int)std::min<long long>((c->rect + 255) / 256, sm_count(c)) : 1;
  k_team_begin<<<blocks, 256, 0, c->stream>>>(*c->h_status, c->d_status, c->d_bar, c->d_ER, c->rect,
                                              c->zero_base_idx, c->Kx, (double)c->N, macro[0],
                                              macro[1], macro[5], mode);
  c->launches += 1;
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? RF_OK : cuda_fail(e, "team solve: start");
}

// Final pass over the strain lines that the solve left: as many blocks as row pairs, up to two
// per SM. The sums (d_sbar, h_sbar) and the status (h_status) are there after a wait.
int launch_team_final(rf_ctx* c, int commit) {
  Args a = make_args(c);
  a.commit = commit;
  a.eps_out = c->d_eps;
  a.sig_out = c->d_sig;
  a.alpha_out = c->d_alpha;
  const int G = std::min(c->ny / 2, 2 * sm_count(c));
  size_t smem = 0;
  if (!shape(c, G, true, a, &smem)) {
    set_error("team final pass: the launch does not fit");
    return RF_ERR_INVALID;
  }
  if (c->has_plastic) k_team_final<true><<<G, a.W, smem, c->stream>>>(a);
  else k_team_final<false><<<G, a.W, smem, c->stream>>>(a);
  c->launches += 1;
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? RF_OK : cuda_fail(e, "team final pass");
}

}  // namespace rfk
