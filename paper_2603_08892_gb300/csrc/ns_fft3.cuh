// ns_fft3.cuh -- register-to-register stages of the compile-time transforms.
//
// The transforms of ns_fft2.cuh keep every stage's inputs and outputs in shared memory.  The
// kernels built on this header keep the first stage's inputs and the last stage's outputs in
// registers (they come from and go to global memory, or feed a pointwise operation), so a
// two-stage transform passes through shared memory once instead of three times.  Radix plans
// are chosen per kernel by a search over ordered factorisations (radix_plan).
#pragma once

#include "ns_fft2.cuh"

namespace ns {

// a + b, a - b: packed in FP32 (ns_fft.cuh)
template <typename T>
__device__ __forceinline__ cpx<T> cadd(cpx<T> a, cpx<T> b) {
  if constexpr (sizeof(T) == 4 && NS_PACKED_F32) return padd(a, b);
  else return a + b;
}
template <typename T>
__device__ __forceinline__ cpx<T> csub(cpx<T> a, cpx<T> b) {
  if constexpr (sizeof(T) == 4 && NS_PACKED_F32) return psub(a, b);
  else return a - b;
}

// ---- 1-, 6-, 9- and 12-point DFTs (s = -1 forward, +1 inverse) --------------------------
template <typename T>
struct DFT<T, 1> {
  static __device__ __forceinline__ void run(cpx<T>*, T) {}
};
// 3-point DFT of (a, b, c) with the products by sqrt(3)/2 fused into the additions
template <typename T>
__device__ __forceinline__ void dft3(cpx<T>& a, cpx<T>& b, cpx<T>& c, T s) {
  const T h = s * T(0.86602540378443864676);  // s sqrt(3) / 2
  const cpx<T> p = cadd(b, c), d = csub(b, c);
  const cpx<T> m = mk<T>(fma1(T(-0.5), p.x, a.x), fma1(T(-0.5), p.y, a.y));
  a = cadd(a, p);
  b = mk<T>(fma1(-h, d.y, m.x), fma1(h, d.x, m.y));
  c = mk<T>(fma1(h, d.y, m.x), fma1(-h, d.x, m.y));
}

// 6 = 2 x 3 (coprime: no internal twiddles): n = 3 n1 + 2 n2 (mod 6), k = 3 k1 + 4 k2 (mod 6)
template <typename T>
struct DFT<T, 6> {
  static __device__ __forceinline__ void run(cpx<T>* v, T s) {
    cpx<T> a0 = v[0], a1 = v[2], a2 = v[4], b0 = v[3], b1 = v[5], b2 = v[1];
    dft3(a0, a1, a2, s);
    dft3(b0, b1, b2, s);
    v[0] = cadd(a0, b0);
    v[3] = csub(a0, b0);
    v[4] = cadd(a1, b1);
    v[1] = csub(a1, b1);
    v[2] = cadd(a2, b2);
    v[5] = csub(a2, b2);
  }
};

// 12 = 4 x 3 (coprime): n = 3 n1 + 4 n2 (mod 12), k = 9 k1 + 4 k2 (mod 12)
template <typename T>
struct DFT<T, 12> {
  static __device__ __forceinline__ void run(cpx<T>* v, T s) {
    cpx<T> t[3][4];
#pragma unroll
    for (int n2 = 0; n2 < 3; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < 4; ++n1) t[n2][n1] = v[(3 * n1 + 4 * n2) % 12];
      DFT<T, 4>::run(t[n2], s);
    }
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
      dft3(t[0][k1], t[1][k1], t[2][k1], s);
#pragma unroll
      for (int k2 = 0; k2 < 3; ++k2) v[(9 * k1 + 4 * k2) % 12] = t[k2][k1];
    }
  }
};

// 9 = 3 x 3: n = n1 + 3 n2, k = 3 k1 + k2, internal twiddles W9^(n1 k2)
template <typename T>
struct DFT<T, 9> {
  static __device__ __forceinline__ void run(cpx<T>* v, T s) {
    const T c1 = T(0.76604444311897803520), s1 = T(0.64278760968653932632);  // 2 pi / 9
    const T c2 = T(0.17364817766693034885), s2 = T(0.98480775301220805937);  // 4 pi / 9
    const T c4 = T(-0.93969262078590838405), s4 = T(0.34202014332566873304);  // 8 pi / 9
#pragma unroll
    for (int n1 = 0; n1 < 3; ++n1) dft3(v[n1], v[n1 + 3], v[n1 + 6], s);  // v[n1 + 3 k2]
    v[4] = cmul_fixed(v[4], mk<T>(c1, s * s1));
    v[7] = cmul_fixed(v[7], mk<T>(c2, s * s2));
    v[5] = cmul_fixed(v[5], mk<T>(c2, s * s2));
    v[8] = cmul_fixed(v[8], mk<T>(c4, s * s4));
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) dft3(v[3 * k2], v[3 * k2 + 1], v[3 * k2 + 2], s);  // [3 k2 + k1]
    cpx<T> t;  // v[3 k2 + k1] -> v[3 k1 + k2]
    t = v[1]; v[1] = v[3]; v[3] = t;
    t = v[2]; v[2] = v[6]; v[6] = t;
    t = v[5]; v[5] = v[7]; v[7] = t;
  }
};

// ---- radix plans ------------------------------------------------------------------------
// No radix of a plan exceeds the first (f).  Where the last one (l) divides it, as in every plan of
// radix_plan (those of cplan need not: 8.2.3 at 48), the set of f elements j + (N/f) r of a first-stage
// butterfly is also what K = f / l last-stage butterflies hold together: p = j + (N/f) i, i < K, element
// p + (N/l) r = j + (N/f) (i + K r).  A thread that runs those K butterflies at the end of one
// transform has in registers what the first stage of the next one (same plan) reads.
constexpr int kRadices[] = {16, 12, 9, 8, 6, 4, 3, 2};
struct PlanSearch {
  CPlan best{0, {0, 0, 0, 0, 0, 0, 0, 0}};
  int score = 1 << 30;
};
constexpr void plan_search(PlanSearch& s, CPlan p, int m, int cap) {
  if (m == 1) {
    const int f = p.r[0], l = p.r[p.nst - 1];
    if (p.nst < 2 || f % l) return;
    const int sc = 100 * p.nst + 4 * (f - l) + f;
    if (sc < s.score) {
      s.score = sc;
      s.best = p;
    }
    return;
  }
  if (p.nst == 5) return;
  for (int r : kRadices)
    if (r <= cap && m % r == 0 && (p.nst == 0 || r <= p.r[0])) {
      CPlan q = p;
      q.r[q.nst++] = r;
      plan_search(s, q, m / r, cap);
    }
}
// Fewest stages with radices <= cap whose last radix divides the first (one pass through shared
// memory per stage costs most; then the spread of the end radices, then registers).
__host__ __device__ constexpr CPlan radix_plan(int n, int cap) {
  PlanSearch s;
  plan_search(s, CPlan{0, {0, 0, 0, 0, 0, 0, 0, 0}}, n, cap);
  return s.best;
}
// FP32 transforms of 24 points and more keep the plans of cplan (radix cap mr), so that results
// recorded in FP64 from FP32 runs (energies, spectra, fields) stay the same to the last bit;
// FP64 ones, whose arithmetic bounds them, take the plan with the fewest stages of radices <= cap64.
template <typename T>
__host__ __device__ constexpr CPlan fplan(int n, int mr, int cap64) {
  return sizeof(T) == 4 && n >= 24 ? cplan(n, mr) : radix_plan(n, sizeof(T) == 4 ? 8 : cap64);
}
__host__ __device__ constexpr int plan_before(CPlan p, int s) {  // product of the radices before stage s
  int m = 1;
  for (int i = 0; i < s; ++i) m *= p.r[i];
  return m;
}

// ---- twiddles and stages ----------------------------------------------------------------
// Twiddles w[r] = W_{NS R}^{p r} of the stage's direction (DIR -1: as the table, +1:
// conjugated) from the padded shared-memory table of W_n: FP32 as stage_twiddles (few reads,
// products for the rest), FP64 every one read (its products cost 1/64 of the FP32 rate).
template <typename T, int n, int R, int NS, int DIR>
__device__ __forceinline__ void reg_twiddles(cpx<T>* w, const cpx<T>* __restrict__ tws, int p) {
  constexpr int TSTEP = n / (NS * R);
  if constexpr (sizeof(T) == 4) {
    stage_twiddles<T, R>(w, tws, p * TSTEP, T(-DIR));
  } else {
#pragma unroll
    for (int r = 1; r < R; ++r) {
      w[r] = tws[tw_pad(r * p * TSTEP)];
      if (DIR > 0) w[r].y = -w[r].y;
    }
  }
}
template <typename T, int R>
__device__ __forceinline__ void twiddle_dft(cpx<T>* v, const cpx<T>* w, T s) {
#pragma unroll
  for (int r = 1; r < R; ++r) v[r] = tw_mul(v[r], w[r]);
  DFT<T, R>::run(v, s);
}

// Exchange tile of W lines of length n in shared memory, written by a first stage of radix R0:
// element e of a line sits in row e + (e / R0) PAD.  COL: [row][line] (a row of W lines), else
// [line][row] with line stride LS.  PAD = 1 for even R0 makes the R0-strided rows that a warp's
// first-stage butterflies write start in different banks (COL: only needed when a row is
// narrower than the 32 banks); LS = 8 (mod 16) puts the next line half a bank period away.
template <typename T, int n, int R0, int W, bool COL>
struct Xchg {
  static constexpr int PAD = (R0 % 2 == 0 && (!COL || W * (int)sizeof(cpx<T>) < 128)) ? 1 : 0;
  static constexpr int ROWS = n + (n / R0) * PAD;
  static constexpr int LS = COL ? 1 : ROWS + (8 + 16 - ROWS % 16) % 16;
  static constexpr int ES = COL ? W : 1;  // stride of a row
  static constexpr int elems = COL ? ROWS * W : LS * W;
  // index of element e of a line
  static __device__ __forceinline__ int at(int line, int e) {
    return (e + (PAD ? e / R0 : 0)) * ES + line * LS;
  }
  // index step of d elements, d a multiple of R0
  static constexpr int step(int d) { return (d + d / R0 * PAD) * ES; }
};

// Middle stage S of plan P in place on NC tiles (tile c at buf + c * ts): every input is read
// before a barrier, then the outputs are written.  All threads of the block call it; threads
// >= NT only pass the barrier.  The caller places the barriers before and after.
template <typename T, int n, class PL, int S, int DIR, class X, int NLINES, int NC, int NT, bool COL>
__device__ __forceinline__ void mid_stage(cpx<T>* buf, int ts, const cpx<T>* __restrict__ tws) {
  constexpr int R = PL::P.r[S], NS = plan_before(PL::P, S), NB = n / R;
  constexpr int TOT = NB * NLINES, KB = (TOT + NT - 1) / NT;
  const int tid = threadIdx.x;
  cpx<T> v[KB][NC][R];
#pragma unroll
  for (int k = 0; k < KB; ++k) {
    const int b = tid + k * NT;
    if (tid < NT && (TOT % NT == 0 || b < TOT)) {
      const int line = COL ? b % NLINES : b / NB, j = COL ? b / NLINES : b % NB;
      const int i0 = X::at(line, j);
      cpx<T> w[R];
      reg_twiddles<T, n, R, NS, DIR>(w, tws, j % NS);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
#pragma unroll
        for (int r = 0; r < R; ++r) v[k][c][r] = buf[c * ts + i0 + r * X::step(NB)];
        twiddle_dft<T, R>(v[k][c], w, T(DIR));
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < KB; ++k) {
    const int b = tid + k * NT;
    if (tid < NT && (TOT % NT == 0 || b < TOT)) {
      const int line = COL ? b % NLINES : b / NB, j = COL ? b / NLINES : b % NB;
      const int o0 = X::at(line, (j / NS) * NS * R + j % NS);
#pragma unroll
      for (int c = 0; c < NC; ++c)
#pragma unroll
        for (int r = 0; r < R; ++r) buf[c * ts + o0 + r * X::step(NS)] = v[k][c][r];
    }
  }
}
// stages S .. END - 1 of plan PL::P in place, each followed by a barrier
template <typename T, int n, class PL, int S, int END, int DIR, class X, int NLINES, int NC, int NT, bool COL>
__device__ __forceinline__ void mid_stages(cpx<T>* buf, int ts, const cpx<T>* __restrict__ tws) {
  if constexpr (S < END) {
    mid_stage<T, n, PL, S, DIR, X, NLINES, NC, NT, COL>(buf, ts, tws);
    __syncthreads();
    mid_stages<T, n, PL, S + 1, END, DIR, X, NLINES, NC, NT, COL>(buf, ts, tws);
  }
}

}  // namespace ns
