// 3D updates of the FFT transform mode on team FFTs (FP32): four kernels per update,
//   inverse y     T2 -> T1, only the pattern's ky rows are read
//   row pass      inverse along x, law, forward along x (T1 -> T1p), a team of G threads per grid
//                 row: its six lines are three packed complex sequences
//   forward y     T1p -> T2f, only the pattern's ky rows are written
//   z phase       per (ky, kx): forward along z, Green operator and decision, inverse along z
//                 (T2f -> T2), all six components of a few neighbouring kx in one block
// (steps a-d of Sec. 4 and the convergence decision of Sec. 3). The general kernels bound a 128^3
// update by instructions (run-time radices and index divisions, staging through shared memory) and
// by six launches; here the sizes are compile-time constants, every transform's first pass
// reads global memory straight into registers and its last pass writes it straight back (sparse
// sides through a position map), and the frequencies of one (ky, kx) never leave the block between
// the two transforms along z. 128^3, K = 2 %: row 81 -> 36 us, y 30 + 30 -> 17 + 17, z and Green
// 20 + 15 + 20 -> 31 us (traced), 175 -> 86 us per update.
#pragma once

#include <algorithm>

#include "rf_internal.cuh"
#include "rf_law.cuh"
#include "rf_teamfft.cuh"

namespace rfk {
namespace fft3 {

using team::Plan;
using fftc::sw;

extern __shared__ __align__(16) unsigned char z_smem[];

// Row pass: teams of `lanes` threads per block, and the block's threads. Whole warps (252 and 240
// threads of teams of 12, 24 and 48 make 256): the final pass sums its stresses with shuffles of
// all 32 lanes, and a lane that does not exist hands over no defined value.
__host__ __device__ constexpr int row_teams(int lanes) { return 256 / lanes; }
__host__ __device__ constexpr int row_threads(int lanes) {
  return (row_teams(lanes) * lanes + 31) / 32 * 32;
}

struct RowArgs3 {
  const float2* T;      // [rows][6][Kx]
  float2* Tout;
  const uint8_t* phase;
  float* state;
  const int* kx;
  const float2* table;  // exp(+2 pi i t / Nx)
  int Kx, rows, teams, groups;
  long long N;
  float invN;
  LawParams law;
  float* eps_out;       // final pass
  float* sig_out;
  float* alpha_out;
  double* sbar_part;
  double* viol_part;
  int commit;
  const int* done;
};

// One row pass over all rows: a block of `teams` teams of G threads takes groups of that many rows
// in turn. A thread carries its points of all three sequences, so the law runs on registers and
// only the passes of the transforms cross shared memory, with warp barriers up to 256 points (3 G
// threads per row, the strains and polarizations staged through shared memory: 44 us at 128^3; so:
// 36 us).
template <int R, int M, bool PLASTIC, bool FINAL>
__global__ __launch_bounds__(256, 2) void k_row3(const __grid_constant__ RowArgs3 a) {
  using P = Plan<R, M>;
  constexpr int L = P::L, G = P::G;
  constexpr int span = (L + L / 16 + 2) & ~1;
  static_assert(row_threads(G) % 32 == 0 && row_threads(G) <= 256, "whole warps");
  __shared__ DevPhase phs[kMaxPhases];
  __shared__ double red[32];
  float2* tw = reinterpret_cast<float2*>(z_smem);
  float2* bufs = tw + ((P::kTw + 1) & ~1);
  int* kxs = reinterpret_cast<int*>(bufs + a.teams * 3 * span);
  short* jmap = reinterpret_cast<short*>(kxs + a.Kx);
  const int tid = threadIdx.x;
  const int team = tid / G, t = tid - team * G;
  const int Kx = a.Kx;
  P::twiddles(a.table, tw);
  for (int i = tid; i <= L / 2; i += blockDim.x) jmap[i] = -1;
  for (int i = tid; i < kMaxPhases; i += blockDim.x) phs[i] = a.law.ph[i];
  __syncthreads();
  for (int j = tid; j < Kx; j += blockDim.x) {
    const int k = a.kx[j];
    kxs[j] = k;
    jmap[k] = (short)j;
  }
  grid_dep_wait();
  if (!FINAL && a.done && __ldcg(a.done)) return;   // the same flag value for every thread
  __syncthreads();
  // (threads beyond the last team only take part in the block's barriers and sums)
  float2* b = bufs + min(team, a.teams - 1) * 3 * span;
  const float lam0 = a.law.lam0, mu0 = a.law.mu0;
  double sb[6] = {0, 0, 0, 0, 0, 0}, vmax = 0.0;
  for (int g = blockIdx.x; g < a.groups; g += gridDim.x) {
    const int row = g * a.teams + team;
    const bool on = team < a.teams && row < a.rows;
    float2 v[3][R];
    uint8_t pid[R];
    if (on) {
      const float2* s0 = a.T + (long long)row * 6 * Kx;
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const int p = t + G * q;
        const int j = jmap[p <= L / 2 ? p : L - p];
        float2 c[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) {
          c[i] = make_float2(0.f, 0.f);
          if (j >= 0) c[i] = __ldcg(s0 + i * Kx + j);
        }
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          float2 x = c[2 * s], y = c[2 * s + 1];
          if (p == 0 || 2 * p == L) x.y = y.y = 0.f;   // self-conjugate positions of real lines
          v[s][q] = 2 * p <= L ? make_float2(x.x - y.y, x.y + y.x) : make_float2(x.x + y.y, y.x - x.y);
        }
      }
      if (!FINAL) {
#pragma unroll
        for (int q = 0; q < R; ++q) pid[q] = a.phase[(long long)row * L + t + G * q];
      }
      P::template first3<+1>(v, b, span, t);
    }
    P::sync(team);
    if (M > 1) {
      if (on) P::template middle3<+1>(b, span, tw, t);
      P::sync(team);
    }
    if (on) P::template last3<+1>(b, span, v, tw, t);
    P::sync(team);
    if (FINAL) {
      // one voxel per step (this code runs once per solve, so its instructions come from memory)
      if (on) {
#pragma unroll
        for (int q = 0; q < R; ++q)
#pragma unroll
          for (int s = 0; s < 3; ++s) b[s * span + P::pt(t, q)] = v[s][q];
      }
      P::sync(team);
#pragma unroll 1
      for (int x = t; on && x < L; x += G) {
        const float2* z = b + sw(x);
        const float2 z0 = z[0], z1 = z[span], z2 = z[2 * span];
        const float e6[6] = {z0.x * a.invN, z0.y * a.invN, z1.x * a.invN,
                             z1.y * a.invN, z2.x * a.invN, z2.y * a.invN};
        const long long gv = (long long)row * L + x;
        float ep[6] = {0, 0, 0, 0, 0, 0};
        float alpha = 0.f;
        if (PLASTIC) load_state<6>(a.state, a.N, gv, ep, alpha);
        const DevPhase& ph = phs[a.phase[gv]];
        LawOut o;
        stress6<PLASTIC>(e6, ph, ep, alpha, o);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          sb[q] += (double)o.s[q];
          a.eps_out[q * a.N + gv] = e6[q];
          a.sig_out[q * a.N + gv] = o.s[q];
        }
        if (PLASTIC) {
          if (a.commit) store_state<6>(a.state, a.N, gv, o.ep, o.alpha);
          a.alpha_out[gv] = o.alpha;
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
        } else {
          a.alpha_out[gv] = 0.f;
        }
      }
      P::sync(team);
      continue;
    }
    if (on) {
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const float e6[6] = {v[0][q].x * a.invN, v[0][q].y * a.invN, v[1][q].x * a.invN,
                             v[1][q].y * a.invN, v[2][q].x * a.invN, v[2][q].y * a.invN};
        float ep[6] = {0, 0, 0, 0, 0, 0};
        float alpha = 0.f;
        if (PLASTIC) load_state<6>(a.state, a.N, (long long)row * L + t + G * q, ep, alpha);
        LawOut o;
        stress6<PLASTIC>(e6, phs[pid[q]], ep, alpha, o);
        const float lt = lam0 * (e6[0] + e6[1] + e6[2]);
        v[0][q] = make_float2(o.s[0] - (lt + 2.f * mu0 * e6[0]), o.s[1] - (lt + 2.f * mu0 * e6[1]));
        v[1][q] = make_float2(o.s[2] - (lt + 2.f * mu0 * e6[2]), o.s[3] - 2.f * mu0 * e6[3]);
        v[2][q] = make_float2(o.s[4] - 2.f * mu0 * e6[4], o.s[5] - 2.f * mu0 * e6[5]);
      }
      P::template first3<-1>(v, b, span, t);
    }
    P::sync(team);
    if (M > 1) {
      if (on) P::template middle3<-1>(b, span, tw, t);
      P::sync(team);
    }
    if (on) P::template last3<-1>(b, span, v, tw, t);
    P::sync(team);
    if (on) {
#pragma unroll
      for (int q = 0; q < R; ++q)
#pragma unroll
        for (int s = 0; s < 3; ++s) b[s * span + P::pt(t, q)] = v[s][q];
    }
    P::sync(team);
    if (on) {
      float2* o = a.Tout + (long long)row * 6 * Kx;
      for (int j = t; j < Kx; j += G) {
        const int k = kxs[j];
        const int ik = sw(k), im = sw(k == 0 ? 0 : L - k);
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          const float2 zk = b[s * span + ik], zm = b[s * span + im];
          o[(2 * s) * Kx + j] = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
          o[(2 * s + 1) * Kx + j] = make_float2(0.5f * (zk.y + zm.y), -0.5f * (zk.x - zm.x));
        }
      }
    }
    P::sync(team);
  }
  if (FINAL) {
    for (int i = 0; i < 6; ++i) {
      const double s = block_sum_d(sb[i], red);
      if (tid == 0) a.sbar_part[blockIdx.x * 6 + i] = s;
    }
    const double vm = block_max_d(vmax, red);
    if (tid == 0) a.viol_part[blockIdx.x] = vm;
  }
}

struct ColArgs3 {
  const float2* in;
  float2* out;
  long long in_bstride, out_bstride;
  int splits;            // S = -1: partial sums to add up (row passes over slices of x), ...
  long long split_stride;
  const short* map;      // [L] row of each position on the sparse side, -1: not in the pattern
  const float2* table;
  int ncols, cgroups, total;   // column groups per batch entry, groups in all
  const int* done;
};

template <int R, int M>
constexpr int cols_per_block() {
  constexpr int G = R * M;
  return G <= 8 ? 32 : G <= 16 ? 16 : 8;
}

// Transforms along one axis of a [batch][L rows][ncols] array: S = +1 reads only the mapped rows,
// S = -1 writes only those. A block takes neighbouring columns, G threads each; neighbouring
// threads hold neighbouring columns (whole sectors of global memory, and an odd buffer pitch keeps
// them on different banks).
template <int R, int M, int S>
__global__ __launch_bounds__(512) void k_cols3(const __grid_constant__ ColArgs3 a) {
  using P = Plan<R, M>;
  constexpr int L = P::L, G = P::G, C = cols_per_block<R, M>();
  constexpr int pitch = (L + L / 16 + 2) | 1;
  float2* tw = reinterpret_cast<float2*>(z_smem);
  float2* bufs = tw + P::kTw;
  short* map = reinterpret_cast<short*>(bufs + 2 * C * pitch);
  const int tid = threadIdx.x, t = tid / C, cc = tid - t * C;
  P::twiddles(a.table, tw);
  for (int i = tid; i < L; i += blockDim.x) map[i] = a.map[i];
  float2* b0 = bufs + cc * pitch;
  float2* b1 = b0 + C * pitch;
  grid_dep_wait();
  if (a.done && __ldcg(a.done)) return;
  __syncthreads();
  for (int g = blockIdx.x; g < a.total; g += gridDim.x) {
    const int b = g / a.cgroups, col = (g - b * a.cgroups) * C + cc;
    const bool on = col < a.ncols;
    const float2* in = a.in + b * a.in_bstride + col;
    float2* out = a.out + b * a.out_bstride + col;
    float2 v[R];
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int p = t + G * q;
      const int r = S > 0 ? map[p] : p;
      v[q] = make_float2(0.f, 0.f);
      if (on && r >= 0) v[q] = __ldcg(in + (long long)r * a.ncols);
    }
    if (S < 0 && on)
      for (int s = 1; s < a.splits; ++s) {
        const float2* is = in + s * a.split_stride;
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const float2 u = __ldcg(is + (long long)(t + G * q) * a.ncols);
          v[q].x += u.x;
          v[q].y += u.y;
        }
      }
    P::template first<S>(v, b0, t);
    __syncthreads();
    if (M > 1) {
      P::template middle<S>(b0, b1, tw, t);
      __syncthreads();
    }
    P::template last<S>(M == 1 ? b0 : b1, v, tw, t);
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int p = t + G * q;
      const int r = S < 0 ? map[p] : p;
      if (on && r >= 0) out[(long long)r * a.ncols] = v[q];
    }
    if (M == 1) __syncthreads();   // the one buffer is rewritten next
  }
}

struct ZArgs {
  const float2* in;      // [L][Ky][6][Kx]
  float2* out;           // [L][Ky][6][Kx]
  float2* ER;            // [Kz][Ky][6][Kx]
  const int2* range;     // [Ky][Kx] first half-pattern entry and count
  const HIdx* hidx;
  const float4* hn;
  const int* kzm;
  const float2* table;
  int Kx, Ky, jgroups;
  float inv2mu0, cgam;
  double Nd;
  Status* st;
  unsigned* counter;
  double* part;          // [gridDim.x]
  const int* done;
  cudaGraphConditionalHandle cond;
  int use_cond;
  int full;              // 0: only the inverse of the held coefficients (the start of a solve)
};

template <int R, int M>
constexpr int kx_per_block() {
  constexpr int G = R * M;   // 6 G times this is a multiple of 32 and at most 384
  return G <= 8 ? 8 : G <= 16 ? 4 : G <= 32 ? 2 : 1;
}

template <int R, int M>
__global__ __launch_bounds__(384, 2) void k_zphase(const __grid_constant__ ZArgs a) {
  using P = Plan<R, M>;
  constexpr int L = P::L, G = P::G, CX = kx_per_block<R, M>(), C = 6 * CX, NC = 6;
  constexpr int pitch = (L + L / 16 + 2) | 1;
  __shared__ double red[12];
  __shared__ double sh[32];
  __shared__ bool last;
  __shared__ int2 rng[CX];
  float2* tw = reinterpret_cast<float2*>(z_smem);
  float2* bufs = tw + P::kTw;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int t = tid / C, col = tid - t * C, c = col / CX, jj = col - c * CX;
  const int iy = blockIdx.x / a.jgroups, j0 = (blockIdx.x - iy * a.jgroups) * CX;
  const int j = j0 + jj;
  P::twiddles(a.table, tw);
  if (tid < CX) rng[tid] = j0 + tid < a.Kx ? a.range[iy * a.Kx + j0 + tid] : make_int2(0, 0);
  float2* b0 = bufs + col * pitch;
  float2* b1 = b0 + C * pitch;
  float2* const Z = M == 1 ? b1 : b0;   // tau^ along z, then scratch of the inverse
  float2* const W = M == 1 ? b0 : b1;   // the new coefficients in zeroed columns
  __syncthreads();
  // entry data of this thread's first frequency before the wait (pattern only)
  const int ej = tid % CX, e0 = tid / CX, estep = nt / CX;
  const int2 er0 = rng[ej];
  const bool has = tid < estep * CX && e0 < er0.y;
  HIdx hi{0, 0, 0, 2};
  float4 n = make_float4(0.f, 0.f, 0.f, 0.f);
  int pos = 0;
  if (has) {
    hi = a.hidx[er0.x + e0];
    n = a.hn[er0.x + e0];
    pos = a.kzm[hi.iz];
  }
  bool any = false;
#pragma unroll
  for (int i = 0; i < CX; ++i) any = any || rng[i].y > 0;
  grid_dep_wait();
  if (a.done && __ldcg(a.done)) return;
  const bool on = j < a.Kx;
  const long long NCK = (long long)NC * a.Kx;
  const long long cbase = iy * NCK + (long long)c * a.Kx + j, zs = a.Ky * NCK;
  double diff = 0.0;
  float2 v[R];
  if (any || !a.full) {   // no frequency of the pattern: the zeros of the start stay
    if (a.full) {
#pragma unroll
      for (int q = 0; q < R; ++q) {
        v[q] = make_float2(0.f, 0.f);
        if (on) v[q] = __ldcg(a.in + cbase + (t + G * q) * zs);
      }
      P::template first<-1>(v, b0, t);
      __syncthreads();
      if (M > 1) {
        P::template middle<-1>(b0, b1, tw, t);
        __syncthreads();
      }
      P::template last<-1>(M == 1 ? b0 : b1, v, tw, t);
#pragma unroll
      for (int q = 0; q < R; ++q) Z[P::pt(t, q)] = v[q];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < R; ++q) W[P::pt(t, q)] = make_float2(0.f, 0.f);
    __syncthreads();
    const float2* zc = bufs + (M == 1 ? C * pitch : 0);   // column cc of Z at zc + cc pitch
    float2* wc = bufs + (M == 1 ? 0 : C * pitch);
    for (int e = e0; tid < estep * CX && e < er0.y; e += estep) {
      if (e != e0) {
        hi = a.hidx[er0.x + e];
        n = a.hn[er0.x + e];
        pos = a.kzm[hi.iz];
      }
      const long long base = ((long long)(hi.iz * a.Ky + iy) * NC) * a.Kx + j0 + ej;
      float2 old[NC];
#pragma unroll
      for (int i = 0; i < NC; ++i) old[i] = a.ER[base + (long long)i * a.Kx];
      if (!a.full) {
#pragma unroll
        for (int i = 0; i < NC; ++i) wc[(i * CX + ej) * pitch + sw(pos)] = old[i];
        continue;
      }
      float2 tv[NC];
#pragma unroll
      for (int i = 0; i < NC; ++i) tv[i] = zc[(i * CX + ej) * pitch + sw(pos)];
      const double* eb = a.st->ebar;
      double em[6];
      if (hi.kind == 1 && a.st->mixed) {   // the one zero-frequency thread of the update
        mixed_macro<NC>(tv, a.Nd, a.st, em);
        for (int i = 0; i < 6; ++i) a.st->ebar[i] = em[i];
        eb = em;
      }
      float er[NC], ei[NC];
      green_update<NC>(hi.kind, n, tv, eb, a.Nd, a.inv2mu0, a.cgam, er, ei);
      float d = 0.f;
#pragma unroll
      for (int i = 0; i < NC; ++i) {
        const float dr = er[i] - old[i].x, di = ei[i] - old[i].y;
        const float wt = i >= 3 ? 2.f : 1.f;   // Frobenius: shear counted twice
        d = fmaf(n.w * wt, dr * dr + di * di, d);
        const float2 nv = make_float2(er[i], ei[i]);
        a.ER[base + (long long)i * a.Kx] = nv;
        wc[(i * CX + ej) * pitch + sw(pos)] = nv;
      }
      diff += (double)d;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < R; ++q) v[q] = W[P::pt(t, q)];
    P::template first<+1>(v, Z, t);
    __syncthreads();
    if (M > 1) {
      P::template middle<+1>(Z, W, tw, t);
      __syncthreads();
    }
    P::template last<+1>(M == 1 ? Z : W, v, tw, t);
    if (on) {
#pragma unroll
      for (int q = 0; q < R; ++q) a.out[cbase + (t + G * q) * zs] = v[q];
    }
  }
  if (!a.full) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) diff += __shfl_down_sync(0xffffffffu, diff, o);
  if ((tid & 31) == 0) red[tid >> 5] = diff;
  __syncthreads();
  if (tid == 0) {
    double s = 0.0;
    for (int i = 0; i < (nt + 31) >> 5; ++i) s += red[i];
    a.part[blockIdx.x] = s;
    __threadfence();
    last = (atomicAdd(a.counter, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (last) {
    __threadfence();
    decide(a.part, gridDim.x, a.st, sh);
    if (tid == 0) {
      *a.counter = 0u;
      // the only call site of the loop condition in this mode: one thread of one block
      if (a.use_cond && a.st->done) cudaGraphSetConditional(a.cond, 0u);
    }
  }
}

// kernels by side, each set compiled on its own
using RowKernel = void (*)(RowArgs3);
using ColKernel = void (*)(ColArgs3);
using ZKernel = void (*)(ZArgs);
RowKernel row_kernel_elastic(int side, bool final_pass);
RowKernel row_kernel_plastic(int side, bool final_pass);
ColKernel col_kernel(int side, int sign);
ZKernel z_kernel(int side);

}  // namespace fft3
}  // namespace rfk
