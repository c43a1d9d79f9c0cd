// Persistent 2D solve on team FFTs (FFT transform mode, FP32, plane strain): every update of one
// solve (Sec. 4, steps a-d, and the convergence decision of Sec. 3) in one launch, for sides
// whose transforms fit a thread team with at most eight points per thread.
//
// What bounds it: nothing but latency. A 256^2 update moves about a megabyte through L2 and
// takes some 10 MFLOP; its time is the chain row phase - barrier - column phase - barrier, each
// phase a chain of dependent loads, transform passes and block barriers. So the layout keeps
// every chain short:
//   - a team of 3 G threads carries the three packed complex sequences of two grid rows (row
//     phase: 11 + i 22 of each row and 12 of both rows) or the three component columns of one kx
//     (column phase). L = R M R points, G = R M threads per sequence: passes of radix R, M, R
//     (R = 8 or 4, M = 1 for none) with R points per thread in the outer passes. The last pass
//     of the inverse transform leaves each thread the points that its first forward pass
//     needs, so the law runs on registers in between; only line 12 crosses shared memory.
//   - the first inverse pass reads its points straight from the kx >= 0 coefficients (a map from
//     position to kx index, most positions empty): no zeroed buffer, no scatter, and one load
//     latency. The reduced coefficients of a kx stay in the shared memory of the block that owns
//     it for the whole solve (dense along y, zeros outside the pattern), as do the phase ids and
//     internal variables of its rows (of large J2 cells the internal variables are fetched by
//     asynchronous copies behind the inverse transform of their rows).
//   - the decision of update u (the same in every block, from block partials in a fixed order)
//     is taken by a warp of its own while the other warps already run the row phase of update
//     u + 1, which writes only scratch; a finished solve leaves after that phase.
//   - one arrival and one poll per grid barrier on a counter that only grows; or, for small
//     cells, the whole grid is one thread-block cluster: its hardware barrier, and the line
//     transforms are written straight into the shared memory of the block that reads them.
// Line transforms in global memory lie as their reader takes them, the strain lines by row pair,
// [u][3][Kx][2 rows], the polarization lines by column, [(c Kx + j) Ny + y]: whole sectors are read
// and 16 bytes written at a time (both by column, the row phase of a 512^2 update took 6.9 us, so
// 6.2 us, and of a 1024^2 update 35 us, so 23 us). Data of other blocks is read through L2. A
// second kernel runs the final pass.
#pragma once

#include <algorithm>
#include <vector>

#include "rf_fftcore.cuh"
#include "rf_internal.cuh"
#include "rf_law.cuh"
#include "rf_teamfft.cuh"

namespace rfk {
namespace team {

constexpr int kMaxWorkers = 384;   // threads of all teams of a block, ...
constexpr int kMaxWorkers3 = 512;  // ... and where a thread of the row phase carries three sequences
// Square cells of these sides have several row pairs per block: their row phase is row_phase3.
__host__ __device__ constexpr bool three_in_one(int side) { return side > 512; }
__host__ __device__ constexpr int max_workers(int side) {
  return three_in_one(side) ? kMaxWorkers3 : kMaxWorkers;
}

struct Args {
  float2* T1;            // strain lines, [u][3][Kx][2 rows]
  float2* T1p;           // polarization lines, [(c Kx + j) Ny + y]
  float2* ER;            // [Ky][NC][Kx]
  const uint8_t* phase;
  float* state;
  const int* kx;         // [Kx]
  const float2* twx;     // exp(+2 pi i t / Nx)
  const float2* twy;     // exp(+2 pi i t / Ny)
  const int* jptr;       // [Kx + 1] entries of each kx
  const int2* jent;      // per entry: rectangle row iy, frequency kind
  const float4* jn;      // per entry: unit wave vector, multiplicity
  const int* kym;        // [Ky] ky mod Ny
  int Nx, Ny, Kx;
  int W;                 // worker threads (a multiple of 32); one more warp decides
  int Px, Py;            // teams per block in the row and the column phase
  int rounds_x, rounds_y;   // row pairs and kx of one team, at most
  int cluster;           // the grid is one cluster
  int st_stream;         // internal variables copied per row pair instead of held
  int entries_cap;       // pattern entries a block holds, at most
  // shared-memory offsets in bytes
  int o_twx, o_twy, o_buf, o_w, o_en, o_ep, o_jmap, o_kx, o_slot, o_st, o_p8, o_ph, o_red, o_eb;
  int o_ts, o_tp;        // cluster: strain lines [slot][3][Kx][2 rows], polarization [slot][3][Ny]
  long long N;
  float invN;
  LawParams law;
  float inv2mu0, cgam;
  double Nd;
  Status* st;
  double* part;          // [min(grid, Kx)] squared-increment partials of the blocks
  // final pass: block partials [grid][8] (six stresses, violation), finished blocks (left zero),
  // and where the last block leaves its sums and the status (pinned host memory)
  double* fin_part;
  unsigned* fin_count;
  double* sbar_dev;
  double* sbar_host;
  Status* st_host;
  unsigned* bar;         // arrivals (zeroed before the launch)
  long bar_limit;
  int commit;
  float* eps_out;
  float* sig_out;
  float* alpha_out;
  unsigned long long* trace;
  int trace_cap;
};

extern __shared__ __align__(16) unsigned char t_smem[];

template <class T>
__device__ __forceinline__ T* at(int off) {
  return reinterpret_cast<T*>(t_smem + off);
}

// stores into the same shared-memory offset of another block of the cluster
__device__ __forceinline__ unsigned remote(const void* p, int rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;"
      : "=r"(r)
      : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_remote(unsigned addr, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y),
               "f"(v.z), "f"(v.w)
               : "memory");
}
__device__ __forceinline__ void st_remote(unsigned addr, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y)
               : "memory");
}

__device__ __forceinline__ void workers_sync(int W) {
  asm volatile("bar.sync 1, %0;" ::"r"(W) : "memory");
}

// Final pass of one row pair by the nt threads of its team (index w): the strains in space at z (11
// + i 22 of the rows, then 12 + i 12, ld entries apart), fields, commit, and the sums sb (six
// stresses, the violation of the yield surface). One voxel per step and no unrolling: this code
// runs once per solve, so its instructions come from memory; unrolled eight times it took 40 us
// on a 256^2 J2 cell.
template <int L, bool PLASTIC>
__device__ __forceinline__ void final_voxels(const Args& a, const float2* z, int ld, int row0,
                                             int w, int nt, const DevPhase* phs, double* sb) {
#pragma unroll 1
  for (int i = w; i < 2 * L; i += nt) {
    const int r = i >= L ? 1 : 0, x = i - r * L;
    const long long g = (long long)(row0 + r) * L + x;
    const float2 za = z[r * ld + sw(x)], zc = z[2 * ld + sw(x)];
    const float e6[6] = {za.x * a.invN, za.y * a.invN, 0.f, 0.f, 0.f, (r ? zc.y : zc.x) * a.invN};
    const DevPhase& ph = phs[a.phase[g]];
    float ep[6] = {0, 0, 0, 0, 0, 0};
    float alpha = 0.f;
    if (PLASTIC) load_state<3>(a.state, a.N, g, ep, alpha);
    LawOut o;
    stress6<PLASTIC>(e6, ph, ep, alpha, o);
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      sb[q] += (double)o.s[q];
      a.eps_out[q * a.N + g] = e6[q];
      a.sig_out[q * a.N + g] = o.s[q];
    }
    if (PLASTIC) {
      if (a.commit) store_state<3>(a.state, a.N, g, o.ep, o.alpha);
      a.alpha_out[g] = o.alpha;
      if (o.yielded) {
        // FP64 consistency check of the FP32 return map: sigma_eq(sigma) = sy + H alpha
        const double s0 = o.s[0], s1 = o.s[1], s2 = o.s[2];
        const double pmd = (s0 + s1 + s2) / 3.0;
        const double d0 = s0 - pmd, d1 = s1 - pmd, d2 = s2 - pmd;
        const double qq = d0 * d0 + d1 * d1 + d2 * d2 +
                          2.0 * ((double)o.s[3] * o.s[3] + (double)o.s[4] * o.s[4] +
                                 (double)o.s[5] * o.s[5]);
        const double yl = (double)ph.sy + (double)ph.H * (double)o.alpha;
        sb[6] = fmax(sb[6], fabs(sqrt(1.5 * qq) - yl) / (double)ph.sy);
      }
    } else {
      a.alpha_out[g] = 0.f;
    }
  }
}

// Row phase of a block: its teams' row pairs u = block + grid (team + Px round). FINAL: fields,
// homogenised-stress sums (sb) and the commit instead of the forward transform.
template <int R, int M, bool PLASTIC, bool FINAL>
__device__ __forceinline__ void row_phase(const Args& a, double* sb) {
  using P = Plan<R, M>;
  constexpr int L = P::L, G = P::G;
  const int team = threadIdx.x / (3 * G), w = threadIdx.x - team * 3 * G;
  const int seq = w / G, t = w - seq * G;
  const int Kx = a.Kx, Ny = a.Ny, units = a.Ny / 2;
  const float2* tw = at<float2>(a.o_twx);
  const short* jmap = at<short>(a.o_jmap);
  const int* kxs = at<int>(a.o_kx);
  constexpr int span = L + L / 16 + 2;
  float2* base = at<float2>(a.o_buf) + (long long)min(team, a.Px - 1) * 6 * span;
  float2* b0 = base + seq * 2 * span;
  float2* b1 = b0 + span;
  // the buffer that carries line 12 across the law, the other one, and where a finished
  // transform goes
  float2* const X2 = base + 4 * span + (M == 1 ? span : 0);
  float2* Y = M == 1 ? b0 : b1;
  float2* Xo = M == 1 ? b1 : b0;
  const float lam0 = a.law.lam0, mu0 = a.law.mu0;
  const DevPhase* phs = at<DevPhase>(a.o_ph);
  for (int rd = 0; rd < a.rounds_x; ++rd) {
    if ((int)blockIdx.x + (int)gridDim.x * a.Px * rd >= units) break;   // no team has a row pair
    const int u = blockIdx.x + gridDim.x * (team + a.Px * rd);
    const bool on = team < a.Px && u < units;
    const int row0 = 2 * u;
    if (PLASTIC && !FINAL && a.st_stream && on) {
      // the pair's internal variables, plane by plane [4][2 L], 16 bytes per copy
      float* sd = at<float>(a.o_st) + team * 8 * L;
      constexpr int per = 2 * L / 4;
      for (int i = w; i < 4 * per; i += 3 * G) {
        const int p = i / per, o = 4 * (i - p * per);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                         (unsigned)__cvta_generic_to_shared(sd + p * 2 * L + o)),
                     "l"(a.state + p * a.N + (long long)row0 * L + o)
                     : "memory");
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    float2 v[R];
    const int slot = team + a.Px * rd;
    if (on) {
      // points t + G q of the sequence's spectrum from the coefficients at kx = min(p, L - p)
      float2 ca[R], cb[R];
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const int p = t + G * q;
        const int j = jmap[p <= L / 2 ? p : L - p];
        ca[q] = cb[q] = make_float2(0.f, 0.f);
        // the pair's lines [3][Kx][2 rows]
        const int o = ((seq < 2 ? 0 : 2) * Kx + j) * 2;
        if (j >= 0 && !FINAL && a.cluster) {
          const float2* s = at<float2>(a.o_ts) + slot * 6 * Kx + o;
          if (seq < 2) {
            ca[q] = s[seq];
            cb[q] = s[2 * Kx + seq];
          } else {
            ca[q] = s[0];
            cb[q] = s[1];
          }
        } else if (j >= 0) {
          const float2* s = a.T1 + (long long)u * 6 * Kx + o;
          if (seq < 2) {
            ca[q] = __ldcg(s + seq);
            cb[q] = __ldcg(s + 2 * Kx + seq);
          } else {
            const float4 f = __ldcg(reinterpret_cast<const float4*>(s));
            ca[q] = make_float2(f.x, f.y);
            cb[q] = make_float2(f.z, f.w);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const int p = t + G * q;
        float2 x = ca[q], y = cb[q];
        if (p == 0 || 2 * p == L) x.y = y.y = 0.f;   // self-conjugate positions of real lines
        // x + i y below L / 2, conj(x) + i conj(y) above
        v[q] = 2 * p <= L ? make_float2(x.x - y.y, x.y + y.x) : make_float2(x.x + y.y, y.x - x.y);
      }
      P::template first<+1>(v, b0, t);
    }
    workers_sync(a.W);
    if (M > 1) {
      if (on) P::template middle<+1>(b0, b1, tw, t);
      workers_sync(a.W);
    }
    if (on) {
      P::template last<+1>(M == 1 ? b0 : b1, v, tw, t);
      if (FINAL || seq == 2) {
        float2* x = M == 1 ? b1 : b0;   // X2 of the third sequence
#pragma unroll
        for (int q = 0; q < R; ++q) x[P::pt(t, q)] = v[q];
      }
    }
    if (PLASTIC && !FINAL && a.st_stream) asm volatile("cp.async.wait_all;" ::: "memory");
    workers_sync(a.W);
    if (FINAL) {
      if (on) final_voxels<L, PLASTIC>(a, base + (M == 1 ? span : 0), 2 * span, row0, w, 3 * G, phs, sb);
      workers_sync(a.W);   // the buffers are reused by the next round
      continue;
    }
    if (on && seq < 2) {
      const uint8_t* ph8 = at<uint8_t>(a.o_p8);
      const float4* st4 = at<float4>(a.o_st);
      const float* sd = at<float>(a.o_st) + team * 8 * L + seq * L;
      const int rs = (slot * 2 + seq) * L;
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const int x = t + G * q;
        float2* x2 = X2 + sw(x);
        const float e12 = (seq ? x2->y : x2->x) * a.invN;
        const float e6[6] = {v[q].x * a.invN, v[q].y * a.invN, 0.f, 0.f, 0.f, e12};
        float ep[6] = {0, 0, 0, 0, 0, 0};
        float alpha = 0.f;
        if (PLASTIC) {
          const float4 s = a.st_stream ? make_float4(sd[x], sd[2 * L + x], sd[4 * L + x], sd[6 * L + x])
                                       : st4[rs + x];
          ep[0] = s.x;
          ep[1] = s.y;
          ep[5] = s.z;
          ep[2] = -(ep[0] + ep[1]);
          alpha = s.w;
        }
        LawOut o;
        stress6<PLASTIC>(e6, phs[ph8[rs + x]], ep, alpha, o);
        const float tr = e6[0] + e6[1];
        v[q] = make_float2(o.s[0] - (lam0 * tr + 2.f * mu0 * e6[0]),
                           o.s[1] - (lam0 * tr + 2.f * mu0 * e6[1]));
        const float t12 = o.s[5] - 2.f * mu0 * e6[5];
        if (seq) x2->y = t12;
        else x2->x = t12;
      }
    }
    workers_sync(a.W);
    if (on) {
      if (seq == 2) {
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = X2[P::pt(t, q)];
      }
      P::template first<-1>(v, Y, t);
    }
    workers_sync(a.W);
    if (M > 1) {
      if (on) P::template middle<-1>(Y, Xo, tw, t);
      workers_sync(a.W);
    }
    if (on) {
      P::template last<-1>(M == 1 ? Y : Xo, v, tw, t);
      float2* z = M == 1 ? Xo : Y;
#pragma unroll
      for (int q = 0; q < R; ++q) z[P::pt(t, q)] = v[q];
    }
    workers_sync(a.W);
    if (on) {
      // the pattern's columns of both rows: 11 and 22 of a row from its sequence's even and odd
      // parts, 12 of the two rows from those of the third
      const float2* z = base + span;   // sequence 0's result; the others 2 span further each
      for (int j = w; j < Kx; j += 3 * G) {
        const int k = kxs[j];
        const int ik = sw(k), im = sw(k == 0 ? 0 : L - k);
        float2 re[3], od[3];
#pragma unroll
        for (int s = 0; s < 3; ++s) {
          const float2 zk = z[s * 2 * span + ik], zm = z[s * 2 * span + im];
          re[s] = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
          od[s] = make_float2(0.5f * (zk.y + zm.y), -0.5f * (zk.x - zm.x));
        }
        const float4 o0 = make_float4(re[0].x, re[0].y, re[1].x, re[1].y);
        const float4 o1 = make_float4(od[0].x, od[0].y, od[1].x, od[1].y);
        const float4 o2 = make_float4(re[2].x, re[2].y, od[2].x, od[2].y);
        if (a.cluster) {
          const int js = j / (int)gridDim.x;   // the owner's slot of this kx
          const unsigned d = remote(at<float2>(a.o_tp) + js * 3 * Ny + row0, j - js * gridDim.x);
          st_remote(d, o0);
          st_remote(d + 8 * Ny, o1);
          st_remote(d + 16 * Ny, o2);
        } else {
          float4* d = reinterpret_cast<float4*>(a.T1p + (long long)j * Ny + row0);
          const long long cs = (long long)Kx * Ny / 2;
          __stcg(d, o0);
          __stcg(d + cs, o1);
          __stcg(d + 2 * cs, o2);
        }
      }
    }
    workers_sync(a.W);   // the buffers are reused by the next round or phase
  }
}

// Row phase of long square cells: a team of G threads per row pair, all three sequences in each
// thread. With several row pairs per block the phase is bound by instructions and by the block's
// barriers, no longer by one pair's latency: addresses, twiddles and barriers are shared by three
// sequences, both rows' laws run on registers (the internal variables of a point come straight
// from L2, fetched one point ahead), and the pairs of a block run independently of one another,
// four at a time instead of one. A 1024^2 J2 load path (3365 updates): 182 -> 158 ms.
template <int R, int M, bool PLASTIC>
__device__ __forceinline__ void row_phase3(const Args& a) {
  using P = Plan<R, M>;
  constexpr int L = P::L, G = P::G, span = L + L / 16 + 2;
  static_assert(G % 32 == 0, "a team has a barrier of its own");
  const int team = threadIdx.x / G, t = threadIdx.x - team * G;
  if (team >= a.Px) return;
  const int Kx = a.Kx, Ny = a.Ny, units = a.Ny / 2;
  const float2* tw = at<float2>(a.o_twx);
  const short* jmap = at<short>(a.o_jmap);
  const int* kxs = at<int>(a.o_kx);
  float2* b = at<float2>(a.o_buf) + (long long)team * 3 * span;
  const float lam0 = a.law.lam0, mu0 = a.law.mu0;
  const DevPhase* phs = at<DevPhase>(a.o_ph);
  for (int rd = 0; rd < a.rounds_x; ++rd) {
    const int slot = team + a.Px * rd;
    const int u = blockIdx.x + gridDim.x * slot;
    if (u >= units) break;
    const int row0 = 2 * u;
    float2 v[3][R];
    {
      // points t + G q of the spectra from the coefficients at kx = min(p, L - p)
      const float4* s = reinterpret_cast<const float4*>(a.T1) + (long long)u * 3 * Kx;
#pragma unroll
      for (int q = 0; q < R; ++q) {
        const int p = t + G * q;
        const int j = jmap[p <= L / 2 ? p : L - p];
        float4 f[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          f[i] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (j >= 0) f[i] = __ldcg(s + i * Kx + j);   // line i of both rows
        }
        if (p == 0 || 2 * p == L) {   // self-conjugate positions of real lines
#pragma unroll
          for (int i = 0; i < 3; ++i) f[i].y = f[i].w = 0.f;
        }
        // x + i y below L / 2, conj(x) + i conj(y) above: 11 + i 22 of each row, 12 of both
        const float sg = 2 * p <= L ? 1.f : -1.f;
        v[0][q] = make_float2(fmaf(-sg, f[1].y, f[0].x), fmaf(sg, f[0].y, f[1].x));
        v[1][q] = make_float2(fmaf(-sg, f[1].w, f[0].z), fmaf(sg, f[0].w, f[1].z));
        v[2][q] = make_float2(fmaf(-sg, f[2].w, f[2].x), fmaf(sg, f[2].y, f[2].z));
      }
    }
    P::template first3<+1>(v, b, span, t);
    P::sync(team);
    P::template middle3<+1>(b, span, tw, t);
    const float4* st4 = at<float4>(a.o_st) + (long long)slot * 2 * L;
    const float* sg = a.state + (long long)row0 * L;
    auto fetch = [&](int q, float4 (&s)[2]) {   // internal variables of point t + G q of both rows
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int x = r * L + t + G * q;
        if (a.st_stream)
          s[r] = make_float4(__ldcg(sg + x), __ldcg(sg + a.N + x), __ldcg(sg + 2 * a.N + x),
                             __ldcg(sg + 3 * a.N + x));
        else
          s[r] = st4[x];
      }
    };
    float4 sn[2];
    if (PLASTIC) fetch(0, sn);
    P::sync(team);
    P::template last3<+1>(b, span, v, tw, t);
    const uint8_t* ph8 = at<uint8_t>(a.o_p8) + slot * 2 * L + t;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      float4 sc[2];
      if (PLASTIC) {
        sc[0] = sn[0];
        sc[1] = sn[1];
        if (q + 1 < R) fetch(q + 1, sn);
      }
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float& c12 = r ? v[2][q].y : v[2][q].x;
        const float e6[6] = {v[r][q].x * a.invN, v[r][q].y * a.invN, 0.f, 0.f, 0.f, c12 * a.invN};
        float ep[6] = {0, 0, 0, 0, 0, 0};
        float alpha = 0.f;
        if (PLASTIC) {
          ep[0] = sc[r].x;
          ep[1] = sc[r].y;
          ep[5] = sc[r].z;
          ep[2] = -(ep[0] + ep[1]);
          alpha = sc[r].w;
        }
        LawOut o;
        stress6<PLASTIC>(e6, phs[ph8[r * L + G * q]], ep, alpha, o);
        const float tr = e6[0] + e6[1];
        v[r][q] = make_float2(o.s[0] - (lam0 * tr + 2.f * mu0 * e6[0]),
                              o.s[1] - (lam0 * tr + 2.f * mu0 * e6[1]));
        c12 = o.s[5] - 2.f * mu0 * e6[5];
      }
    }
    P::sync(team);
    P::template first3<-1>(v, b, span, t);
    P::sync(team);
    P::template middle3<-1>(b, span, tw, t);
    P::sync(team);
    P::template last3<-1>(b, span, v, tw, t);
    P::sync(team);
#pragma unroll
    for (int q = 0; q < R; ++q)
#pragma unroll
      for (int s = 0; s < 3; ++s) b[s * span + P::pt(t, q)] = v[s][q];
    P::sync(team);
    // the pattern's columns of both rows: 11 and 22 of a row from its sequence's even and odd
    // parts, 12 of the two rows from those of the third
    for (int j = t; j < Kx; j += G) {
      const int k = kxs[j];
      const int ik = sw(k), im = sw(k == 0 ? 0 : L - k);
      float2 re[3], od[3];
#pragma unroll
      for (int s = 0; s < 3; ++s) {
        const float2 zk = b[s * span + ik], zm = b[s * span + im];
        re[s] = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
        od[s] = make_float2(0.5f * (zk.y + zm.y), -0.5f * (zk.x - zm.x));
      }
      float4* d = reinterpret_cast<float4*>(a.T1p + (long long)j * Ny + row0);
      const long long cs = (long long)Kx * Ny / 2;
      __stcg(d, make_float4(re[0].x, re[0].y, re[1].x, re[1].y));
      __stcg(d + cs, make_float4(od[0].x, od[0].y, od[1].x, od[1].y));
      __stcg(d + 2 * cs, make_float4(re[2].x, re[2].y, od[2].x, od[2].y));
    }
    P::sync(team);   // the buffers are reused by the next round
  }
}

// Column phase of a block: its teams' kx, j = block + grid (team + Py round). full = false: only
// the inverse transform of the held coefficients (the start of a solve). Leaves each thread's
// FP64 squared-increment sum in the block's array and arrives at barrier 2.
template <int R, int M>
__device__ __forceinline__ void col_phase(const Args& a, bool full) {
  using P = Plan<R, M>;
  constexpr int L = P::L, G = P::G, NC = 3;
  const int team = threadIdx.x / (3 * G), w = threadIdx.x - team * 3 * G;
  const int c = w / G, t = w - c * G;
  const int Kx = a.Kx;
  const float2* tw = at<float2>(a.o_twy);
  constexpr int span = L + L / 16 + 2;
  float2* base = at<float2>(a.o_buf) + (long long)min(team, a.Py - 1) * 6 * span;
  float2* b0 = base + c * 2 * span;
  float2* b1 = b0 + span;
  const float4* en = at<float4>(a.o_en);
  const int* ep = at<int>(a.o_ep);
  const int* slot0 = at<int>(a.o_slot);
  double* eb0 = at<double>(a.o_eb);   // macroscopic strain, mixed control
  double dsum = 0.0;
  for (int rd = 0; rd < a.rounds_y; ++rd) {
    if ((int)blockIdx.x + (int)gridDim.x * a.Py * rd >= Kx) break;
    const int slot = team + a.Py * rd;
    const int j = blockIdx.x + gridDim.x * slot;
    const bool on = team < a.Py && j < Kx;
    float2* Wc = at<float2>(a.o_w) + (long long)slot * 3 * L;   // [3][L] held coefficients
    float2 v[R];
    if (full) {
      if (on) {
        if (a.cluster) {
          const float2* s = at<float2>(a.o_tp) + (slot * 3 + c) * L + t;
#pragma unroll
          for (int q = 0; q < R; ++q) v[q] = s[G * q];
        } else {
          const float2* s = a.T1p + (long long)(c * Kx + j) * L + t;
#pragma unroll
          for (int q = 0; q < R; ++q) v[q] = __ldcg(s + G * q);
        }
        P::template first<-1>(v, b0, t);
      }
      workers_sync(a.W);
      if (M > 1) {
        if (on) P::template middle<-1>(b0, b1, tw, t);
        workers_sync(a.W);
      }
      if (on) {
        P::template last<-1>(M == 1 ? b0 : b1, v, tw, t);
        float2* z = M == 1 ? b1 : b0;
#pragma unroll
        for (int q = 0; q < R; ++q) z[P::pt(t, q)] = v[q];
      }
      workers_sync(a.W);
      if (on) {
        const float2* z = base + (M == 1 ? span : 0);
        for (int e = slot0[slot] + w; e < slot0[slot + 1]; e += 3 * G) {
          const float4 n = en[e];
          const int pk = ep[e], pos = pk & 0xffff, kind = pk >> 16;
          const bool mixed0 = kind == 1 && eb0[6] != 0.0;
          float2 tv[NC], old[NC];
#pragma unroll
          for (int i = 0; i < NC; ++i) {
            tv[i] = (kind == 0 || mixed0) ? z[i * 2 * span + sw(pos)] : make_float2(0.f, 0.f);
            old[i] = Wc[i * L + pos];
          }
          if (mixed0) {
            mixed_macro<NC>(tv, a.Nd, a.st, eb0);
            for (int i = 0; i < 6; ++i) a.st->ebar[i] = eb0[i];
          }
          float er[NC], ei[NC];
          green_update<NC>(kind, n, tv, eb0, a.Nd, a.inv2mu0, a.cgam, er, ei);
          float diff = 0.f;
#pragma unroll
          for (int i = 0; i < NC; ++i) {
            const float dr = er[i] - old[i].x, di = ei[i] - old[i].y;
            const float wc = (comp6<NC>(i) >= 3) ? 2.f : 1.f;   // Frobenius: shear counted twice
            diff = fmaf(n.w * wc, dr * dr + di * di, diff);
            Wc[i * L + pos] = make_float2(er[i], ei[i]);
          }
          dsum += (double)diff;
        }
      }
      workers_sync(a.W);
    }
    if (on) {
#pragma unroll
      for (int q = 0; q < R; ++q) v[q] = Wc[c * L + t + G * q];
      P::template first<+1>(v, M == 1 ? b0 : b1, t);
    }
    workers_sync(a.W);
    if (M > 1) {
      if (on) P::template middle<+1>(b1, b0, tw, t);
      workers_sync(a.W);
    }
    if (on) {
      P::template last<+1>(b0, v, tw, t);
      if (a.cluster) {
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const int y = t + G * q, u = y >> 1, us = u / (int)gridDim.x;   // the owner's slot
          st_remote(remote(at<float2>(a.o_ts) + ((us * 3 + c) * Kx + j) * 2 + (y & 1),
                           u - us * gridDim.x),
                    v[q]);
        }
      } else {
        float2* d = a.T1 + (c * Kx + j) * 2;
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const int y = t + G * q;
          __stcg(d + (long long)(y >> 1) * 6 * Kx + (y & 1), v[q]);
        }
      }
    }
    if (full && ((int)blockIdx.x + (int)gridDim.x * a.Py * (rd + 1) >= Kx || rd + 1 == a.rounds_y)) {
      // the deciding warp sums these while the barrier collects the blocks
      at<double>(a.o_red)[threadIdx.x] = dsum;
      asm volatile("bar.arrive 2, %0;" ::"r"(a.W + 32) : "memory");
    }
    workers_sync(a.W);
  }
}

// SIDE > 0: the kernel is compiled for square cells of that side; 0: any of the sides
template <int SIDE, bool PLASTIC, bool FINAL>
__device__ __forceinline__ void rows(const Args& a, double* sb) {
  if constexpr (three_in_one(SIDE) && !FINAL) {
    if constexpr (SIDE == 768) row_phase3<8, 12, PLASTIC>(a);
    else row_phase3<8, 16, PLASTIC>(a);
    return;
  }
  switch (SIDE ? SIDE : a.Nx) {
#define X(L, R, M) \
  case L: row_phase<R, M, PLASTIC, FINAL>(a, sb); break;
    RF_TEAM_SIDES_2D(X)
#undef X
  }
}

template <int SIDE>
__device__ __forceinline__ void cols(const Args& a, bool full) {
  switch (SIDE ? SIDE : a.Ny) {
#define X(L, R, M) \
  case L: col_phase<R, M>(a, full); break;
    RF_TEAM_SIDES_2D(X)
#undef X
  }
}

__device__ inline void fill_twiddles(int L, const float2* tab, float2* tw) {
  switch (L) {
#define X(L_, R, M) \
  case L_: Plan<R, M>::twiddles(tab, tw); break;
    RF_TEAM_SIDES_2D(X)
#undef X
  }
}

// what both kernels read from shared memory in the row phase
__device__ inline void fill_rows(const Args& a) {
  fill_twiddles(a.Nx, a.twx, at<float2>(a.o_twx));
  short* jmap = at<short>(a.o_jmap);
  int* kxs = at<int>(a.o_kx);
  DevPhase* phs = at<DevPhase>(a.o_ph);
  for (int i = threadIdx.x; i <= a.Nx / 2; i += blockDim.x) jmap[i] = -1;
  for (int i = threadIdx.x; i < kMaxPhases; i += blockDim.x) phs[i] = a.law.ph[i];
  __syncthreads();
  for (int j = threadIdx.x; j < a.Kx; j += blockDim.x) {
    const int k = a.kx[j];
    kxs[j] = k;
    jmap[k] = (short)j;
  }
}

__device__ __forceinline__ unsigned long long stamp() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Barrier over the grid (all blocks co-resident); false if the wait ran out.
__device__ __forceinline__ bool grid_barrier(const Args& a, unsigned target, int* s_flag) {
  if (a.cluster) {
    cluster_sync();
    return true;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    // release and acquire are cumulative: they order the whole block's accesses through the block
    // barriers on both sides
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.bar) : "memory");
    unsigned v;
    long it = 0;
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.bar) : "memory");
      if ((int)(v - target) >= 0) break;
      if (++it > a.bar_limit) {
        ok = 0;
        break;
      }
    }
    *s_flag = ok;
  }
  __syncthreads();
  return *s_flag != 0;
}

template <int SIDE, bool PLASTIC>
__global__ __launch_bounds__(max_workers(SIDE) + 32, 1) void k_team2d(const __grid_constant__ Args a) {
  __shared__ int s_flag, s_done;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
  const bool worker = tid < a.W;
  const bool items = (int)blockIdx.x < a.Kx;   // this block owns a kx
  fill_rows(a);
  fill_twiddles(a.Ny, a.twy, at<float2>(a.o_twy));
  // this block's kx: entry offsets, entries, and their held coefficients in zeroed columns
  const int nslot = items ? (a.Kx - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
  int* slot0 = at<int>(a.o_slot);
  if (tid == 0) {
    int s = 0;
    for (int i = 0; i < nslot; ++i) {
      const int j = blockIdx.x + gridDim.x * i;
      slot0[i] = s;
      s += a.jptr[j + 1] - a.jptr[j];
    }
    slot0[nslot] = s;
  }
  float2* Wb = at<float2>(a.o_w);
  for (int i = tid; i < nslot * 3 * a.Ny; i += nt) Wb[i] = make_float2(0.f, 0.f);
  // phase ids and internal variables of this block's row pairs
  {
    const int units = a.Ny / 2, L = a.Nx;
    const int nu = (int)blockIdx.x < units ? (units - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    uint8_t* ph8 = at<uint8_t>(a.o_p8);
    float4* st4 = at<float4>(a.o_st);
    for (int i = tid; i < nu * 2 * L; i += nt) {
      const int s = i / (2 * L), r = i - s * 2 * L;
      const long long g = (long long)2 * (blockIdx.x + gridDim.x * s) * L + r;
      ph8[i] = a.phase[g];
      if (PLASTIC && !a.st_stream)
        st4[i] = make_float4(a.state[g], a.state[a.N + g], a.state[2 * a.N + g], a.state[3 * a.N + g]);
    }
  }
  __syncthreads();
  for (int s = 0; s < nslot; ++s) {
    const int j = blockIdx.x + gridDim.x * s, e0 = a.jptr[j], n = slot0[s + 1] - slot0[s];
    for (int i = tid; i < n; i += nt) {
      const int2 q = a.jent[e0 + i];
      const int pos = a.kym[q.x];
      at<float4>(a.o_en)[slot0[s] + i] = a.jn[e0 + i];
      at<int>(a.o_ep)[slot0[s] + i] = pos | (q.y << 16);
      for (int c = 0; c < 3; ++c)
        Wb[(s * 3 + c) * a.Ny + pos] = a.ER[((long long)q.x * 3 + c) * a.Kx + j];
    }
  }
  // the deciding warp's running values
  int iters = 0;
  double rmin = 0.0, tol = 0.0, enorm = 0.0, inv_n2 = 0.0;
  int max_iter = 0;
  if (!worker) {
    iters = a.st->iters;
    rmin = a.st->rmin;
    tol = a.st->tol;
    enorm = a.st->enorm;
    inv_n2 = a.st->inv_n2;
    max_iter = a.st->max_iter;
  }
  const int nparts = min((int)gridDim.x, a.Kx);
  unsigned target = 0;
  unsigned long long t_upd = 0, t_row = 0;   // trace stamps (block 0, thread 0)
  const bool tracer = a.trace && blockIdx.x == 0 && tid == 0;
  if (tid < 6) at<double>(a.o_eb)[tid] = a.st->ebar[tid];
  if (tid == 6) at<double>(a.o_eb)[6] = a.st->mixed ? 1.0 : 0.0;
  if (tid == 0) s_done = 0;
  __syncthreads();
  if (a.cluster) cluster_sync();   // every block runs before another writes its shared memory
  for (int u = 0;; ++u) {
    // column phase of update u (u = 0: the strain lines of the start coefficients)
    if (items) {
      if (worker) {
        cols<SIDE>(a, u > 0);
      } else if (u > 0) {
        asm volatile("bar.sync 2, %0;" ::"r"(a.W + 32) : "memory");
        double s = 0.0;
        for (int i = lane; i < a.W; i += 32) s += at<double>(a.o_red)[i];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) a.part[blockIdx.x] = s;
        __syncwarp();
      }
    }
    target += gridDim.x;
    if (!grid_barrier(a, target, &s_flag)) {
      if (tid == 0) atomicExch(&a.st->timeout, 1);
      return;
    }
    if (tracer) {
      const unsigned long long t_col = stamp();
      if (u > 0 && u <= a.trace_cap) {
        a.trace[3 * (u - 1)] = t_upd;
        a.trace[3 * (u - 1) + 1] = t_row;
        a.trace[3 * (u - 1) + 2] = t_col;
      }
      t_upd = t_col;
    }
    // row phase of update u + 1; meanwhile the decision on update u
    if (worker) {
      rows<SIDE, PLASTIC, false>(a, nullptr);
    } else if (u > 0) {
      double s = 0.0;
      for (int i = lane; i < nparts; i += 32) s += __ldcg(a.part + i);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
      if (lane == 0) {
        double r = sqrt(s * inv_n2);
        if (enorm > 0.0) r /= enorm;
        iters += 1;
        rmin = fmin(rmin, r);
        int done = 0, nonfinite = 0, diverged = 0;
        if (!isfinite(r)) nonfinite = done = 1;
        else if (r > kDivergeRatio * rmin && r > kDivergeFloor) diverged = done = 1;
        else if (r < tol || iters >= max_iter) done = 1;
        if (done && blockIdx.x == 0) {
          a.st->iters = iters;
          a.st->last_r = r;
          a.st->rmin = rmin;
          a.st->nonfinite = nonfinite;
          a.st->diverged = diverged;
          a.st->done = 1;
        }
        s_done = done;
      }
      __syncwarp();
    }
    __syncthreads();
    if (s_done) break;
    target += gridDim.x;
    if (!grid_barrier(a, target, &s_flag)) {
      if (tid == 0) atomicExch(&a.st->timeout, 1);
      return;
    }
    if (tracer) t_row = stamp();
  }
  if (a.cluster) {
    // no block leaves while another still writes into it; the strain lines to global memory for
    // the final pass
    cluster_sync();
    const int units = a.Ny / 2;
    const int nu = (int)blockIdx.x < units ? (units - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    for (int i = tid; i < nu * 3 * a.Kx; i += nt) {
      const int s = i / (3 * a.Kx), q = i - s * 3 * a.Kx;   // q = c Kx + j
      reinterpret_cast<float4*>(a.T1)[(long long)(blockIdx.x + gridDim.x * s) * 3 * a.Kx + q] =
          at<float4>(a.o_ts)[i];
    }
  }
  // the coefficients of the last update back to the rectangle
  for (int s = 0; s < nslot; ++s) {
    const int j = blockIdx.x + gridDim.x * s, e0 = a.jptr[j], n = slot0[s + 1] - slot0[s];
    for (int i = tid; i < n; i += nt) {
      const int iy = a.jent[e0 + i].x, pos = at<int>(a.o_ep)[slot0[s] + i] & 0xffff;
      for (int c = 0; c < 3; ++c)
        a.ER[((long long)iy * 3 + c) * a.Kx + j] = Wb[(s * 3 + c) * a.Ny + pos];
    }
  }
}

using Kernel = void (*)(Args);

// the solve kernels for square cells of a side, for elastic phases and with a J2 phase (null: not a
// side of the plans), and for any sides of the plans (side 0): each compiled on its own
Kernel kernel_elastic(int side);
Kernel kernel_plastic(int side);
Kernel kernel_any(bool plastic);

}  // namespace team
}  // namespace rfk
