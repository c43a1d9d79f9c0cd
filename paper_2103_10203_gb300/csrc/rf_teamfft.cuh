// Team FFTs (FP32): complex transforms of L = R M R points by G = R M threads, R points per thread
// in the outer passes, in three passes (two for M = 1) over shared memory, with every size known
// at compile time. Shared by the persistent 2D solve and the 3D transforms. Element i of a
// sequence lies at sw(i) = i + i / 16 of its buffer.
#pragma once

#include "rf_fftcore.cuh"

namespace rfk {
namespace team {

using fftc::cmul;
using fftc::span_of;
using fftc::sw;

// ---- DFTs of N points in registers, natural order in and out, kernel exp(S 2 pi i n q / N)
template <int N, int S>
struct Dft;

template <int S>
struct Dft<1, S> {
  static __device__ __forceinline__ void run(float2*) {}
};
template <int S>
struct Dft<2, S> {
  static __device__ __forceinline__ void run(float2* v) {
    const float2 a = v[0], b = v[1];
    v[0] = make_float2(a.x + b.x, a.y + b.y);
    v[1] = make_float2(a.x - b.x, a.y - b.y);
  }
};
template <int S>
struct Dft<3, S> {
  static __device__ __forceinline__ void run(float2* v) {
    const float hs = 0.86602540378443865f * (float)S;
    const float2 s = make_float2(v[1].x + v[2].x, v[1].y + v[2].y);
    const float2 d = make_float2(v[1].x - v[2].x, v[1].y - v[2].y);
    const float2 m = make_float2(v[0].x - 0.5f * s.x, v[0].y - 0.5f * s.y);
    v[0] = make_float2(v[0].x + s.x, v[0].y + s.y);
    v[1] = make_float2(m.x - hs * d.y, m.y + hs * d.x);
    v[2] = make_float2(m.x + hs * d.y, m.y - hs * d.x);
  }
};
template <int S>
struct Dft<4, S> {
  static __device__ __forceinline__ void run(float2* v) {
    fftc::dft4(v[0], v[1], v[2], v[3], S);
  }
};
template <int S>
struct Dft<6, S> {   // 2 x 3: n = 2 a + b, q = q3 + 3 q2
  static __device__ __forceinline__ void run(float2* v) {
    float2 e[3] = {v[0], v[2], v[4]}, o[3] = {v[1], v[3], v[5]};
    Dft<3, S>::run(e);
    Dft<3, S>::run(o);
    const float h = 0.86602540378443865f * (float)S;   // exp(S 2 pi i q / 6)
    o[1] = cmul(o[1], make_float2(0.5f, h));
    o[2] = cmul(o[2], make_float2(-0.5f, h));
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      v[q] = make_float2(e[q].x + o[q].x, e[q].y + o[q].y);
      v[q + 3] = make_float2(e[q].x - o[q].x, e[q].y - o[q].y);
    }
  }
};
template <int S>
struct Dft<8, S> {   // 2 x 4
  static __device__ __forceinline__ void run(float2* v) {
    float2 e[4] = {v[0], v[2], v[4], v[6]}, o[4] = {v[1], v[3], v[5], v[7]};
    Dft<4, S>::run(e);
    Dft<4, S>::run(o);
    const float h = 0.70710678118654752f, s = (float)S;
    // exp(S 2 pi i q / 8): (h, s h), (0, s), (-h, s h)
    o[1] = make_float2(h * (o[1].x - s * o[1].y), h * (o[1].y + s * o[1].x));
    o[2] = make_float2(-s * o[2].y, s * o[2].x);
    o[3] = make_float2(h * (-o[3].x - s * o[3].y), h * (-o[3].y + s * o[3].x));
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      v[q] = make_float2(e[q].x + o[q].x, e[q].y + o[q].y);
      v[q + 4] = make_float2(e[q].x - o[q].x, e[q].y - o[q].y);
    }
  }
};

template <int S>
struct Dft<12, S> {   // 4 x 3: n = 4 a + b, q = q3 + 3 q4
  static __device__ __forceinline__ void run(float2* v) {
    float2 w[4][3];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
#pragma unroll
      for (int a = 0; a < 3; ++a) w[b][a] = v[4 * a + b];
      Dft<3, S>::run(w[b]);
    }
    // exp(S 2 pi i b q3 / 12)
    const float h = 0.86602540378443865f, s = (float)S;
    w[1][1] = cmul(w[1][1], make_float2(h, 0.5f * s));
    w[1][2] = cmul(w[1][2], make_float2(0.5f, h * s));
    w[2][1] = cmul(w[2][1], make_float2(0.5f, h * s));
    w[2][2] = cmul(w[2][2], make_float2(-0.5f, h * s));
    w[3][1] = make_float2(-s * w[3][1].y, s * w[3][1].x);
    w[3][2] = make_float2(-w[3][2].x, -w[3][2].y);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      float2 u[4] = {w[0][q], w[1][q], w[2][q], w[3][q]};
      Dft<4, S>::run(u);
#pragma unroll
      for (int k = 0; k < 4; ++k) v[q + 3 * k] = u[k];
    }
  }
};
template <int S>
struct Dft<16, S> {
  static __device__ __forceinline__ void run(float2* v) {
    fftc::dft16(v, S);
    float2 u[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) u[q] = v[4 * (q & 3) + (q >> 2)];
#pragma unroll
    for (int q = 0; q < 16; ++q) v[q] = u[q];
  }
};

// ---- the three passes of a sequence of L = R M R points, thread t < G = R M of its team
template <int R, int M>
struct Plan {
  static constexpr int L = R * R * M, G = R * M;

  // sw(t + G q). Where G is no multiple of 16 the pad does not grow evenly with q; written so, the
  // R places of a thread come from a few bases (two for G = 24) instead of an address each (which
  // the passes of sides 96 and 192 spilled).
  static __device__ __forceinline__ int pt(int t, int q) {
    const int n = G * q, r = n & 15;
    return sw(t + r) + (n - r) + (n - r) / 16;
  }

  // stage-major twiddles: (M - 1) R of the middle pass, then (R - 1) G of the last
  static constexpr int kTw2 = (M - 1) * R, kTw = kTw2 + (R - 1) * G;

  static __device__ void twiddles(const float2* tab, float2* tw) {
    for (int i = threadIdx.x; i < kTw; i += blockDim.x) {
      if (i < kTw2) {
        const int q = 1 + i / R, k = i - (q - 1) * R;
        tw[i] = tab[q * k * R];
      } else {
        const int u = i - kTw2, q = 1 + u / G, k = u - (q - 1) * G;
        tw[i] = tab[q * k];
      }
    }
  }
  // first pass: v = points t + G q -> b
  template <int S>
  static __device__ __forceinline__ void first(float2* v, float2* b, int t) {
    Dft<R, S>::run(v);
    float2* d = b + sw(t * R);   // R consecutive entries inside one 16-entry block
#pragma unroll
    for (int q = 0; q < R; ++q) d[q] = v[q];
  }
  // middle pass: b -> o
  template <int S>
  static __device__ __forceinline__ void middle(const float2* b, float2* o, const float2* tw,
                                                int t) {
    constexpr int T = R * R, pq = T + T / 16;   // T tasks; T is a multiple of 16
#pragma unroll 1
    for (int j = t; j < T; j += G) {
      const int k = j % R;
      const float2* s = b + sw(j);
      float2 v[M];
#pragma unroll
      for (int q = 0; q < M; ++q) v[q] = s[q * pq];
#pragma unroll
      for (int q = 1; q < M; ++q) {
        float2 w = tw[(q - 1) * R + k];
        if (S < 0) w.y = -w.y;
        v[q] = cmul(v[q], w);
      }
      Dft<M, S>::run(v);
      const int base = (j / R) * (R * M) + k;
#pragma unroll
      for (int q = 0; q < M; ++q) o[sw(base + q * R)] = v[q];
    }
  }
  // last pass: b -> v = points t + G q
  template <int S>
  static __device__ __forceinline__ void last(const float2* b, float2* v, const float2* tw, int t) {
#pragma unroll
    for (int q = 0; q < R; ++q) v[q] = b[pt(t, q)];
#pragma unroll
    for (int q = 1; q < R; ++q) {
      float2 w = tw[kTw2 + (q - 1) * G + t];
      if (S < 0) w.y = -w.y;
      v[q] = cmul(v[q], w);
    }
    Dft<R, S>::run(v);
  }

  // ---- three sequences per thread, `ld` entries apart, each in one buffer: the middle pass leaves
  // output q of task j in the places that the task read (place(q), which keeps the last pass's
  // reads on different banks where M allows it); a team sync between passes and before the next
  // first pass. Addresses, twiddles and barriers are shared by the three sequences, and the law
  // runs on registers between the transforms.
  static __host__ __device__ constexpr int place(int q) {
    return M % 4 == 0 ? (q & ~3) | ((q & 1) << 1) | ((q >> 1) & 1) : q;
  }
  template <int S>
  static __device__ __forceinline__ void first3(float2 (&v)[3][R], float2* b, int ld, int t) {
#pragma unroll
    for (int s = 0; s < 3; ++s) first<S>(v[s], b + s * ld, t);
  }
  template <int S>
  static __device__ __forceinline__ void middle3(float2* b, int ld, const float2* tw, int t) {
    constexpr int T = R * R, pq = T + T / 16;
#pragma unroll 1
    for (int i = t; i < 3 * T; i += G) {
      const int s = i / T, j = i - s * T, k = j % R;
      float2* d = b + s * ld + sw(j);
      float2 v[M];
#pragma unroll
      for (int q = 0; q < M; ++q) v[q] = d[q * pq];
#pragma unroll
      for (int q = 1; q < M; ++q) {
        float2 w = tw[(q - 1) * R + k];
        if (S < 0) w.y = -w.y;
        v[q] = cmul(v[q], w);
      }
      Dft<M, S>::run(v);
#pragma unroll
      for (int q = 0; q < M; ++q) d[place(q) * pq] = v[q];
    }
  }
  template <int S>
  static __device__ __forceinline__ void last3(const float2* b, int ld, float2 (&v)[3][R],
                                               const float2* tw, int t) {
    constexpr int pq = R * R + R * R / 16;
    const float2* d = b + place(t / R) * pq;
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int o = sw(q * R + t % R);
#pragma unroll
      for (int s = 0; s < 3; ++s) v[s][q] = d[s * ld + o];
    }
#pragma unroll
    for (int q = 1; q < R; ++q) {
      float2 w = tw[kTw2 + (q - 1) * G + t];
      if (S < 0) w.y = -w.y;
#pragma unroll
      for (int s = 0; s < 3; ++s) v[s][q] = cmul(v[s][q], w);
    }
#pragma unroll
    for (int s = 0; s < 3; ++s) Dft<R, S>::run(v[s]);
  }
  // barrier of the G threads of one team of a block whose threads are teams 0, 1, ... in order:
  // within a warp, or a barrier of its own, or (teams that share warps unevenly) the whole block
  static constexpr bool kOwnSync = G % 32 == 0 || 32 % G == 0;
  static __device__ __forceinline__ void sync(int team) {
    if constexpr (32 % G == 0) __syncwarp();
    else if constexpr (G % 32 == 0)
      asm volatile("bar.sync %0, %1;" ::"r"(3 + team), "n"(G) : "memory");
    else
      __syncthreads();
  }
};

// sides with a plan: L, R, M
#define RF_TEAM_SIDES(X) \
  X(32, 4, 2) X(48, 4, 3) X(64, 8, 1) X(96, 4, 6) X(128, 8, 2) X(192, 8, 3) X(256, 8, 4) \
  X(384, 8, 6) X(512, 8, 8)

// ... and the longer ones that only the persistent 2D solve takes
#define RF_TEAM_SIDES_2D(X) RF_TEAM_SIDES(X) X(768, 8, 12) X(1024, 8, 16)

}  // namespace team
}  // namespace rfk
