// ns_kernels.cuh -- the CUDA kernels of one pseudo-spectral Navier-Stokes evaluation.
//
// Data layout in HBM (complex values of type cpx<T>, T = float or double):
//   state / acc   [3][kz][ky][kx]      spectral, kx = 0..N/2-1 contiguous
//   mixed         [5][z][ky][kx]       after the inverse z transform: u_x, u_y, u_z,
//                                      d_z u_x, d_z u_y (phase shift already applied)
//   Ft            [3][z][ky][kx]       FFT_xy of u x omega (mixed space)
//   scratch       [6][g][y][kx]        y-transformed planes of the current plane group
//                                      (L2-resident for small groups; the group size is
//                                      autotuned and may be the whole grid)
// One evaluation of the nonlinear term = slab pass over all planes (k_yinv -> k_xrow ->
// k_yfwd per plane group) followed by one pencil pass (k_pencil) that ends the forward
// transform and applies the whole spectral stage of Sec. 4 in the same HBM pass.
#pragma once

#include "ns_fft.cuh"

namespace ns {

// Layouts of the mixed fields and of Ft.  pairs = 0: each field by itself, [f][z][ky][kx].
// pairs = 1 (the compile-time kernels): fields 0 and 1 interleaved mode by mode, then field 2,
// then (mixed) fields 3 and 4 interleaved: a pencil tile of 8 columns reads and writes 128
// contiguous bytes per plane of a pair in FP32 instead of 64.
__host__ __device__ __forceinline__ size_t ft_index(int pairs, int f, size_t g, size_t fs) {
  return pairs && f < 2 ? 2 * g + f : f * fs + g;
}
__host__ __device__ __forceinline__ size_t mixed_index(int pairs, int f, size_t g, size_t fs) {
  return pairs && f >= 3 ? 3 * fs + 2 * g + (f - 3) : ft_index(pairs, f, g, fs);
}

enum PencilMode {
  MODE_INIT = 0,     // S_next = S0 (state)
  MODE_RK2_1 = 1,    // S_next = (S0 + dt/2 N) E_{dt/2}
  MODE_RK2_2 = 2,    // S = S0 E_dt + dt E_{dt/2} N -> state;      S_next = S
  MODE_RK4_1 = 3,    // acc = S0 E_dt + dt/6 E_dt N;               S_next = (S0 + dt/2 N) E_{dt/2}
  MODE_RK4_2 = 4,    // acc += dt/3 E_{dt/2} N;                    S_next = S0 E_{dt/2} + dt/2 N
  MODE_RK4_3 = 5,    // acc += dt/3 E_{dt/2} N;                    S_next = S0 E_dt + dt E_{dt/2} N
  MODE_RK4_4 = 6,    // S = acc + dt/6 N -> state;                 S_next = S
  MODE_ROG_1 = 7,    // A = S0 E_dt + dt/2 E_{dt/2} N -> state;    S_next = (S0 + dt N) E_dt
  MODE_ROG_2 = 8,    // S = A + dt/2 E_{dt/2} N -> state;          S_next = S
  MODE_NL = 9,       // acc = N
  MODE_PROJECT = 10  // state = N (input is a velocity: truncation + projection only)
};

// XMODE_ADJ_WR / XMODE_ADJ_RU: adjoint slab passes, u x omega replaced by omega x r and
// r x u (r: the mixed fields of the cotangent, in SlabArgs::mixedB)
enum XMode { XMODE_NONLINEAR = 0, XMODE_C2R = 1, XMODE_R2C = 2, XMODE_ADJ_WR = 3, XMODE_ADJ_RU = 4 };
__host__ __device__ __forceinline__ bool xmode_cross(int m) {
  return m == XMODE_NONLINEAR || m == XMODE_ADJ_WR || m == XMODE_ADJ_RU;
}

enum ErrBits { ERR_FFT_SHAPE = 1, ERR_LAUNCH_SHAPE = 2 };

__device__ __forceinline__ int kof(int i, int N) { return i < (N >> 1) ? i : i - N; }

// ----------------------------------------------------------------------------------------
// Tables (FP64 arithmetic, rounded to T)
// ----------------------------------------------------------------------------------------
// Truncation mask T at mode k (Sec. 3.2; Sec. 4.2 for the double aliases).  trunc 1, cubic:
// max_i |k_i| <= Kimax.  Otherwise spherical: |k|^2 <= K2max; trunc 2 also drops the modes a
// double alias can reach: |k + N e|^2 <= 4 K2max for some e with exactly one zero component,
// whose closest member gives (N - |k_i|)^2 + (N - |k_j|)^2 + k_l^2 for the pair (i, j).
__device__ __forceinline__ bool trunc_keep(int trunc, int kx, int ky, int kz, int N, int K2max, int Kimax) {
  if (trunc == 1) return max(abs(kx), max(abs(ky), abs(kz))) <= Kimax;
  const long long x2 = (long long)kx * kx, y2 = (long long)ky * ky, z2 = (long long)kz * kz;
  if (x2 + y2 + z2 > (long long)K2max) return false;
  if (trunc != 2) return true;
  const long long ax = N - abs(kx), ay = N - abs(ky), az = N - abs(kz), m4 = 4LL * K2max;
  return ax * ax + ay * ay + z2 > m4 && ax * ax + az * az + y2 > m4 && ay * ay + az * az + x2 > m4;
}

// Columns (kx, ky) that hold modes of the truncation or of the forcing table, |k_i| <= box (box < 0:
// none); for a given ky an interval of kx from 0.  Outside them the nonlinear term and the forcing
// vanish (the no-double-alias mask lies inside the sphere).  A state that vanishes there too stays
// so: the passes then leave these columns alone, 21 % of them at kmax = N/2 and 56 to 65 % at N/3.
// Per pass of 8 steps at most, all columns -> kept ones: 384^3 RK4 (N/3) 18490 -> 12060 us, 256^3
// random 4170 -> 4075, 512^3 split 21320 -> 20580.
__host__ __device__ __forceinline__ bool column_kept(int trunc, int K2max, int Kimax, int box, int kx, int ky) {
  const int ay = ky < 0 ? -ky : ky;
  const bool in = trunc == 1 ? (kx <= Kimax && ay <= Kimax) : kx * kx + ky * ky <= K2max;
  return in || (kx <= box && ay <= box);
}

// true (to some threads at least false otherwise) when the modes of S [3][N][N][M] in the columns
// (kx, ky = kof(iy)) that are not kept vanish.  One block of 256 threads per ky and part (of
// `parts`); reads only those modes (21 % of the state at C_t = 1), 16 bytes a load, four in flight.
// A row is given the next power of two of threads, so that no index needs a division.
template <typename T>
__device__ __forceinline__ bool cut_clean(const cpx<T>* S, int N, int trunc, int K2max, int Kimax, int box, int iy,
                                          int part, int parts) {
  constexpr int PER = 16 / (int)sizeof(cpx<T>);  // modes of a load
  const int M = N / 2, ky = kof(iy, N);
  int lo = 0;  // the first kx that is not kept (the kept ones are an interval from 0)
  for (int k0 = 0; k0 < M; k0 += blockDim.x) {
    const int k = k0 + threadIdx.x;
    lo += __syncthreads_count(k < M && column_kept(trunc, K2max, Kimax, box, k, ky));
  }
  if (lo == M) return true;
  const int c0 = lo / PER, nch = M / PER - c0;  // loads of a row
  const int lw = nch > 1 ? 32 - __clz(nch - 1) : 0, rows = blockDim.x >> lw;
  const int ch = threadIdx.x & ((1 << lw) - 1), r1 = threadIdx.x >> lw, kx = (c0 + ch) * PER;
  bool nz = false;
  if (ch < nch)
    for (int r0 = part * 4 * rows + r1; r0 < 3 * N; r0 += parts * 4 * rows) {
      cpx<T> v[4][PER];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = r0 + q * rows;  // component and kz
#pragma unroll
        for (int i = 0; i < PER; ++i) v[q][i] = mk<T>(0, 0);
        if (r < 3 * N) {
          const float4 w = *reinterpret_cast<const float4*>(&S[((size_t)r * N + iy) * M + kx]);
          memcpy(v[q], &w, 16);
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int i = 0; i < PER; ++i) nz = nz || (kx + i >= lo && (!(v[q][i].x == T(0)) || !(v[q][i].y == T(0))));
    }
  return !nz;
}
// *flag = 0 (it is 1 before) where they do not; *next = 1, the flag of the next check
template <typename T>
__global__ void __launch_bounds__(256) k_cut_check(const cpx<T>* S, int N, int trunc, int K2max, int Kimax, int box,
                                                   int* flag, int* next) {
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *next = 1;
  if (!cut_clean(S, N, trunc, K2max, Kimax, box, blockIdx.x, blockIdx.y, gridDim.y)) *flag = 0;
}

template <typename T>
__global__ void k_twiddle(cpx<T>* tw, int N) {
  int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= N) return;
  double s, c;
  sincospi(2.0 * (double)k / (double)N, &s, &c);
  tw[k] = mk<T>((T)c, (T)(-s));
}

// out[j * N + i] = exp(-nu k(i)^2 tau_j), j = 0, 1
template <typename T>
__global__ void k_ifac(T* out, int N, double nu, double tau0, double tau1) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  double k = (double)kof(i, N);
  out[i] = (T)exp(-nu * k * k * tau0);
  out[N + i] = (T)exp(-nu * k * k * tau1);
}

// out[(s * 3 + d) * N + i] = exp(i k(i) delta[s][d])  (Sec. 4.2, Eq. shift_operator_3d)
template <typename T>
__global__ void k_shift_tables(cpx<T>* out, int N, const double* __restrict__ delta, int nshift) {
  int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= nshift * 3 * N) return;
  int i = idx % N, sd = idx / N;
  double a = (double)kof(i, N) * delta[sd];
  double s, c;
  sincos(a, &s, &c);
  out[idx] = mk<T>((T)c, (T)s);
}

// ----------------------------------------------------------------------------------------
// Pencil pass: z transforms + spectral stage
// ----------------------------------------------------------------------------------------
template <typename T>
struct PencilArgs {
  int N, M, TX, LX;  // LX: columns transformed at a time (the run-time kernels)
  FastDiv dTX, dLX;
  FFTPlan pz;
  const cpx<T>* tw;
  int nF;                // number of nonlinear inputs (0, 1, 2)
  const cpx<T>* F[2];    // [3][N][N][M]
  const cpx<T>* dsh[2];  // shift tables of the inputs ([3][N]) or null (no shift)
  T wF[2];               // weights of the inputs (1/N^3 or 1/(2 N^3))
  int mode;
  T dt;
  const T* ifac;         // [2][N]: tau = dt, dt/2
  cpx<T>* state;
  cpx<T>* acc;
  const cpx<T>* src;     // MODE_INIT source (state or a temporary)
  int trunc, K2max, Kimax;
  const cpx<T>* force;   // [3][D] dense table of the forcing term, or null
  cpx<T>* shell;         // [3][D] S_next at the forcing table's modes, or null
  int fK;                // forcing table half-width (D = (2fK+1)^2 (fK+1))
  int nOut;
  const cpx<T>* osh[2];  // shift tables of the outputs
  cpx<T>* out[2];        // [5][N][N][M]
  int* err;
  double* epart;         // [tiles][2]: sums of w |S|^2 and w k^2 |S|^2 of the written state, or null
  int iy0;               // first ky row of the launch (rank-range passes; 0 for a whole field)
  int pairs;             // layout of F and out: mixed_index, ft_index
  // device flag, or null (as 0): not 0 when the state (src for INIT) vanishes outside the kept
  // columns (column_kept with box = cutK): tiles without one are then left alone, outputs included
  const int* cut;
  int cutK;
};

template <typename T>
__device__ __forceinline__ cpx<T> phase3(const cpx<T>* tab, int N, int ix, int iy, int iz) {
  return (ldg(&tab[ix]) * ldg(&tab[N + iy])) * ldg(&tab[2 * N + iz]);
}

// Run-time sizes: one block per ky row and TX columns.  The z transforms' first stages read global
// memory (or form the shifted values) and their last ones write it: only the stages between them
// go through shared memory.  Bound by issue (index arithmetic, radix-8 and radix-3 stages).  216^3 FP32,
// one in and one out: 394 us a launch, 834 with the tiles loaded and stored whole; a step 3240 us, 6180
// with that, run-time divisions, six-tile y passes and 15 values a thread.
template <typename T>
__global__ void __launch_bounds__(384, sizeof(T) == 4 ? 2 : 1) k_pencil(const __grid_constant__ PencilArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<T>* buf = reinterpret_cast<cpx<T>*>(smem_raw);
  const int N = a.N, M = a.M, TX = a.TX;
  const int ntx = M / TX;
  const int iy = a.iy0 + blockIdx.x / ntx;
  const int x0 = (blockIdx.x % ntx) * TX;
  const int tile = N * TX;
  const size_t fstride = (size_t)N * N * M;
  const int ky = kof(iy, N);
  const LineBatch lb = {a.LX, TX / a.LX, TX, 1, (int)threadIdx.x, (int)blockDim.x, true, a.dLX};
  cpx<T>* sxy = buf + 4 * tile;  // [4][16]: x and y factors of the shifts' phases (phase3's association)
  const size_t gz = (size_t)N * M;  // z stride
  const size_t g0 = (size_t)iy * M + x0;
  if (threadIdx.x < 64) {
    const int i = threadIdx.x >> 4, x = threadIdx.x & 15;
    const cpx<T>* tab = i < 2 ? (i < a.nF ? a.dsh[i] : nullptr) : (i - 2 < a.nOut ? a.osh[i - 2] : nullptr);
    if (tab && x < TX) sxy[threadIdx.x] = ldg(&tab[x0 + x]) * ldg(&tab[N + iy]);
  }
  __syncthreads();

  // 1) forward z transforms of the nonlinear inputs, de-shift, weights
#pragma unroll 1
  for (int c = 0; c < (a.nF > 0 ? 3 : 0); ++c) {
    cpx<T>* bc = buf + c * tile;
    const cpx<T>* F0 = a.F[0] + c * fstride + g0;
    fft_lines(bc, a.pz, lb, false, a.tw, T(-1), a.err, [&](int x, int z) { return F0[z * gz + x]; },
              [&](int x, int z, cpx<T> v) {
                if (a.dsh[0]) v = mul_conj(v, sxy[x] * ldg(&a.dsh[0][2 * N + z]));
                bc[z * TX + x] = a.wF[0] * v;
              });
    if (a.nF > 1) {
      const cpx<T>* F1 = a.F[1] + c * fstride + g0;
      fft_lines(buf + 3 * tile, a.pz, lb, false, a.tw, T(-1), a.err, [&](int x, int z) { return F1[z * gz + x]; },
                [&](int x, int z, cpx<T> w) {
                  if (a.dsh[1]) w = mul_conj(w, sxy[16 + x] * ldg(&a.dsh[1][2 * N + z]));
                  bc[z * TX + x] = bc[z * TX + x] + a.wF[1] * w;
                });
    }
  }
  __syncthreads();

  // 2) pointwise: N(0) = 0, truncation T, projection P, forcing, stage combine
  const T dt = a.dt, hdt = T(0.5) * a.dt;
  const int D1 = 2 * a.fK + 1;
  const int D = D1 * D1 * (a.fK + 1);
  for (int e = threadIdx.x; e < tile; e += blockDim.x) {
    const int iz = fdiv(e, a.dTX), x = e - iz * TX;
    const int kx = x0 + x, kz = kof(iz, N);
    const size_t g = ((size_t)iz * N + iy) * M + kx;
    cpx<T> nv[3];
    if (a.nF > 0) {
      const int k2 = kx * kx + ky * ky + kz * kz;
      const bool keep = trunc_keep(a.trunc, kx, ky, kz, N, a.K2max, a.Kimax) && (k2 != 0);
      if (keep) {
        cpx<T> v0 = buf[e], v1 = buf[tile + e], v2 = buf[2 * tile + e];
        const T fx = (T)kx, fy = (T)ky, fz = (T)kz;
        const T ik2 = T(1) / (T)k2;
        cpx<T> kd = mk<T>(fx * v0.x + fy * v1.x + fz * v2.x, fx * v0.y + fy * v1.y + fz * v2.y);
        nv[0] = v0 - (fx * ik2) * kd;
        nv[1] = v1 - (fy * ik2) * kd;
        nv[2] = v2 - (fz * ik2) * kd;
      } else {
        nv[0] = nv[1] = nv[2] = mk<T>(0, 0);
      }
      if (a.force && kx <= a.fK && abs(ky) <= a.fK && abs(kz) <= a.fK) {
        const int fi = ((kz + a.fK) * D1 + (ky + a.fK)) * (a.fK + 1) + kx;
#pragma unroll
        for (int c = 0; c < 3; ++c) nv[c] = nv[c] + a.force[c * D + fi];
      }
    }
    T E1 = 1, Eh = 1;
    if (a.mode != MODE_INIT && a.mode != MODE_NL && a.mode != MODE_PROJECT) {
      E1 = a.ifac[kx] * a.ifac[iy] * a.ifac[iz];
      Eh = a.ifac[N + kx] * a.ifac[N + iy] * a.ifac[N + iz];
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const size_t gi = g + c * fstride;
      cpx<T> sn = mk<T>(0, 0);
      switch (a.mode) {
        case MODE_INIT:
          sn = a.src[gi];
          break;
        case MODE_RK2_1: {
          cpx<T> s0 = a.state[gi];
          sn = Eh * (s0 + hdt * nv[c]);
        } break;
        case MODE_RK2_2: {
          cpx<T> s0 = a.state[gi];
          sn = E1 * s0 + (dt * Eh) * nv[c];
          a.state[gi] = sn;
        } break;
        case MODE_RK4_1: {
          cpx<T> s0 = a.state[gi];
          a.acc[gi] = E1 * s0 + (dt / T(6) * E1) * nv[c];
          sn = Eh * (s0 + hdt * nv[c]);
        } break;
        case MODE_RK4_2: {
          cpx<T> s0 = a.state[gi];
          a.acc[gi] = a.acc[gi] + (dt / T(3) * Eh) * nv[c];
          sn = Eh * s0 + hdt * nv[c];
        } break;
        case MODE_RK4_3: {
          cpx<T> s0 = a.state[gi];
          a.acc[gi] = a.acc[gi] + (dt / T(3) * Eh) * nv[c];
          sn = E1 * s0 + (dt * Eh) * nv[c];
        } break;
        case MODE_RK4_4: {
          sn = a.acc[gi] + (dt / T(6)) * nv[c];
          a.state[gi] = sn;
        } break;
        case MODE_ROG_1: {
          cpx<T> s0 = a.state[gi];
          a.state[gi] = E1 * s0 + (hdt * Eh) * nv[c];
          sn = E1 * (s0 + dt * nv[c]);
        } break;
        case MODE_ROG_2: {
          sn = a.state[gi] + (hdt * Eh) * nv[c];
          a.state[gi] = sn;
        } break;
        case MODE_NL:
          a.acc[gi] = nv[c];
          break;
        case MODE_PROJECT:
          a.state[gi] = nv[c];
          break;
      }
      buf[c * tile + e] = sn;
      if (a.shell && kx <= a.fK && abs(ky) <= a.fK && abs(kz) <= a.fK) {
        const int fi = ((kz + a.fK) * D1 + (ky + a.fK)) * (a.fK + 1) + kx;
        a.shell[c * D + fi] = sn;
      }
    }
  }
  __syncthreads();

  // 3) outputs: shift, z-derivatives, inverse z transforms
#pragma unroll 1
  for (int o = 0; o < a.nOut; ++o) {
    const cpx<T>* osh = a.osh[o];
#pragma unroll 1
    for (int f = 0; f < 5; ++f) {
      const cpx<T>* S = buf + (f < 3 ? f : f - 3) * tile;
      cpx<T>* dst = a.out[o] + f * fstride + g0;
      fft_lines(buf + 3 * tile, a.pz, lb, false, a.tw, T(1), a.err,
                [&](int x, int z) {
                  cpx<T> v = S[z * TX + x];
                  if (osh) v = v * (sxy[32 + 16 * o + x] * ldg(&osh[2 * N + z]));
                  if (f >= 3) v = mul_si(v, (T)kof(z, N));  // i kz v
                  return v;
                },
                [&](int x, int z, cpx<T> v) { dst[z * gz + x] = v; });
    }
  }
}

// ----------------------------------------------------------------------------------------
// Slab pass: y transforms and the x rows with the real-space cross product
// ----------------------------------------------------------------------------------------
template <typename T>
struct SlabArgs {
  int N, M, z0, G;
  int LY;              // columns transformed at a time (the run-time kernels)
  FastDiv dLY, dNP;    // dNP: M / 2 + 1
  FFTPlan py, px;
  const cpx<T>* tw;
  const cpx<T>* mixed;  // [5][N][N][M]
  const cpx<T>* mixedB; // [5][N][N][M] cotangent fields r (adjoint modes; first 3 used)
  cpx<T>* scr;          // [6][G][N][M]
  cpx<T>* Ft;           // [3][N][N][M]
  T* rio;               // physical rows [3][N][N][N] (C2R output / R2C input)
  int TY, RX, xmode;
  int* err;
  void* umax;           // or null: max_x |u_i(x)| of the velocity rows, i = 0..2, folded in
                        // with atomicMax on the IEEE bits (unsigned / unsigned long long [3])
  // skip: the compile-time kernels leave the products of columns (kx, ky) unwritten that are not
  // kept (column_kept with box = fK; kxn: the first kx none of whose columns is kept): no pencil
  // pass uses them.  cut: device flag, or null (as 0): not 0 when the mixed fields of such
  // columns are zero (and left unwritten)
  int skip, trunc, K2max, Kimax, fK, kxn;
  const int* cut;
  int pairs;             // layout of mixed, mixedB and Ft: mixed_index, ft_index
};

// Block maxima m0..m2 (non-negative) folded into umax[0..2], one atomic per value per block:
// the bit patterns of non-negative IEEE numbers order like the numbers, so an unsigned
// atomicMax is a max of the values.  scratch: 3 (blockDim.x / 32) values of shared memory
// that are free during the call; every thread of the block calls it (blockDim.x is a
// multiple of 32).
template <typename T>
__device__ void block_max3(T m0, T m1, T m2, T* scratch, void* umax) {
  for (int o = 16; o > 0; o >>= 1) {
    m0 = fmax(m0, __shfl_xor_sync(0xffffffffu, m0, o));
    m1 = fmax(m1, __shfl_xor_sync(0xffffffffu, m1, o));
    m2 = fmax(m2, __shfl_xor_sync(0xffffffffu, m2, o));
  }
  const int w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    scratch[3 * w] = m0;
    scratch[3 * w + 1] = m1;
    scratch[3 * w + 2] = m2;
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    T m = T(0);
    for (int i = 0; i < nw; ++i) m = fmax(m, scratch[3 * i + threadIdx.x]);
    if (sizeof(T) == 4)
      atomicMax(static_cast<unsigned*>(umax) + threadIdx.x, __float_as_uint((float)m));
    else
      atomicMax(static_cast<unsigned long long*>(umax) + threadIdx.x,
                (unsigned long long)__double_as_longlong((double)m));
  }
  __syncthreads();
}

// Inverse y transforms of one field per block: the velocity, or omega = i k x u formed from the
// mixed fields as they are read.  grid (M/TY, G, fields).  One field per block reads some mixed
// fields twice (from L2) and needs one tile of shared memory instead of six, so that enough blocks
// are resident to cover the loads: 216^3 FP32, per 100 planes: 160 us, 400 to 435 with six tiles (8 warps
// an SM).  The products are fused in writing: the compiler merges the branches' subtractions otherwise.
template <typename T>
__global__ void __launch_bounds__(384, sizeof(T) == 4 ? 2 : 1) k_yinv(const __grid_constant__ SlabArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<T>* buf = reinterpret_cast<cpx<T>*>(smem_raw);
  const int N = a.N, M = a.M, TY = a.TY;
  const int x0 = blockIdx.x * TY, zg = blockIdx.y, z = a.z0 + zg;
  const int f = blockIdx.z, c = f < 3 ? f : f - 3;
  const size_t fstride = (size_t)N * N * M;
  // fields 0..2 and 3..5: the pair whose cross product the x rows form (u, omega, or the cotangent r)
  enum { U, W, RB };
  int kind = f < 3 ? U : W;
  if (a.xmode == XMODE_ADJ_WR) kind = f < 3 ? W : RB;
  if (a.xmode == XMODE_ADJ_RU) kind = f < 3 ? RB : U;
  const LineBatch lb = {a.LY, TY / a.LY, TY, 1, (int)threadIdx.x, (int)blockDim.x, true, a.dLY};
  cpx<T>* dst = a.scr + f * (size_t)a.G * N * M + (size_t)zg * N * M + x0;
  fft_lines(buf, a.py, lb, false, a.tw, T(1), a.err,
            [&](int x, int iy) {
              const size_t g = ((size_t)z * N + iy) * M + x0 + x;
              auto mx = [&](const cpx<T>* m, int i) { return m[mixed_index(a.pairs, i, g, fstride)]; };
              if (kind == RB) return mx(a.mixedB, c);
              if (kind == U) return mx(a.mixed, c);
              const T kx = (T)(x0 + x), ky = (T)kof(iy, N);
              if (c == 0) {  // w_x = i ky uz - dz uy
                const cpx<T> uz = mx(a.mixed, 2), d = mx(a.mixed, 4);
                return mk<T>(fma1(-ky, uz.y, -d.x), fma1(ky, uz.x, -d.y));
              }
              if (c == 1) {  // w_y = dz ux - i kx uz
                const cpx<T> uz = mx(a.mixed, 2), d = mx(a.mixed, 3);
                return mk<T>(fma1(kx, uz.y, d.x), fma1(-kx, uz.x, d.y));
              }
              const cpx<T> uy = mx(a.mixed, 1), ux = mx(a.mixed, 0);  // w_z = i kx uy - i ky ux
              return mk<T>(fma1(ky, ux.y, -(kx * uy.y)), fma1(kx, uy.x, -(ky * ux.x)));
            },
            [&](int x, int iy, cpx<T> v) { dst[(size_t)iy * M + x] = v; });
}

// forward y transforms of one component of the x-transformed product.  grid (M/TY, G, 3)
template <typename T>
__global__ void __launch_bounds__(384, sizeof(T) == 4 ? 2 : 1) k_yfwd(const __grid_constant__ SlabArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<T>* buf = reinterpret_cast<cpx<T>*>(smem_raw);
  const int N = a.N, M = a.M, TY = a.TY;
  const int x0 = blockIdx.x * TY, zg = blockIdx.y, z = a.z0 + zg, f = blockIdx.z;
  const size_t fstride = (size_t)N * N * M;
  const LineBatch lb = {a.LY, TY / a.LY, TY, 1, (int)threadIdx.x, (int)blockDim.x, true, a.dLY};
  const cpx<T>* src = a.scr + f * (size_t)a.G * N * M + (size_t)zg * N * M + x0;
  fft_lines(buf, a.py, lb, false, a.tw, T(-1), a.err, [&](int x, int iy) { return src[(size_t)iy * M + x]; },
            [&](int x, int iy, cpx<T> v) {
              a.Ft[ft_index(a.pairs, f, ((size_t)z * N + iy) * M + x0 + x, fstride)] = v;
            });
}

// Hermitian half spectrum X_0..X_{M-1} (X_M = 0; x(i) reads X_i) -> Z'_k whose inverse M-point DFT
// is the packed real row z_m = x_{2m} + i x_{2m+1}, x_j = sum_{k=0}^{N-1} X_k exp(2 pi i jk/N).
template <typename T, class X>
__device__ __forceinline__ cpx<T> c2r_pre(X x, int M, const cpx<T>* __restrict__ tw, int k) {
  const int km = k ? M - k : 0;
  const bool low = k < km;
  const cpx<T> Xk = x(k), Xm = x(km);
  const cpx<T> A = Xk + conjg(Xm), B = Xk - conjg(Xm);
  cpx<T> w = ldg(&tw[low ? k : km]);
  if (low) w.y = -w.y;  // e^{+2 pi i k / N}; above M/2 it is -e^{-2 pi i (M-k)/N}
  const cpx<T> z = A + mul_si(w * B, low ? T(1) : T(-1));
  return k ? z : mk<T>(Xk.x, Xk.x);
}

// Z_k (row: forward M-point DFT of the packed real row) -> X_k = sum_j x_j e^{-2 pi i jk/N}, k < M:
// out[k] and out[M - k]
template <typename T>
__device__ __forceinline__ void r2c_post(cpx<T>* out, const cpx<T>* row, int M, const cpx<T>* __restrict__ tw,
                                         int k) {
  if (k == 0) {
    const cpx<T> Z = row[0];
    out[0] = mk<T>(Z.x + Z.y, T(0));
    if (M % 2 == 0 && M > 1) {
      // k = M/2: W^k = e^{-i pi/2} = -i
      cpx<T> Zk = row[M / 2];
      cpx<T> A = Zk + conjg(Zk), B = Zk - conjg(Zk);
      // X = A/2 - i/2 (-i) B = A/2 - B/2
      out[M / 2] = T(0.5) * (A - B);
    }
    return;
  }
  const int km = M - k;
  cpx<T> Zk = row[k], Zm = row[km];
  cpx<T> W = ldg(&tw[k]);  // e^{-2 pi i k/N}
  cpx<T> A = Zk + conjg(Zm), B = Zk - conjg(Zm);
  out[k] = T(0.5) * (A - mul_si(W * B, T(1)));
  // W^{M-k} = -conj(W)
  cpx<T> A2 = Zm + conjg(Zk), B2 = Zm - conjg(Zk);
  out[km] = T(0.5) * (A2 + mul_si(conjg(W) * B2, T(1)));
}

// x rows: c2r of 6 fields, u x omega, r2c of 3 fields (nonlinear mode); c2r of 3 fields to
// physical rows (C2R); r2c of 3 physical rows (R2C).  grid ceil(G*N / RX).  The block's threads form
// six groups that each transform the rows of one field at a time, so that the fields share the
// barriers of a stage; first stages read global memory (with c2r_pre's combination).
template <typename T>
__global__ void __launch_bounds__(384, sizeof(T) == 4 ? 2 : 1) k_xrow(const __grid_constant__ SlabArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<T>* buf = reinterpret_cast<cpx<T>*>(smem_raw);
  const int N = a.N, M = a.M, RX = a.RX;
  const int rows_total = a.G * N;
  const int r0 = blockIdx.x * RX;
  const int nr = min(RX, rows_total - r0);
  if (nr <= 0) return;
  const int tile = RX * M;
  const size_t sstride = (size_t)a.G * N * M;
  const int nin = xmode_cross(a.xmode) ? 6 : 3;
  constexpr int XG = 6;
  const int gt = blockDim.x / XG;  // threads of a group
  const int grp = threadIdx.x / gt, t0 = threadIdx.x - grp * gt;
  auto real_row = [&](int f, int r) {
    const int rr = r0 + r, zg = rr / N, y = rr - zg * N;
    return a.rio + ((size_t)f * N + a.z0 + zg) * N * N + (size_t)y * N;
  };
  // the group's field when nf fields are transformed, and its rows from l0 on (a field's rows are shared
  // by two groups when the groups are twice the fields); nl = 0: nothing to do, but the barriers of it
  auto batch = [&](int nf, int& f, int& l0) {
    const bool halves = XG == 2 * nf && RX % 2 == 0;
    f = grp % nf;
    l0 = halves && grp >= nf ? RX / 2 : 0;
    const int nl = halves ? RX / 2 : grp < nf ? RX : 0;
    return LineBatch{nl, 1, 1, M, t0, gt, false, FastDiv{1, 0}};
  };

  if (a.xmode != XMODE_R2C) {
    int f, l0;
    const LineBatch lb = batch(nin, f, l0);
    const cpx<T>* src = a.scr + f * sstride + (size_t)(r0 + l0) * M;
    cpx<T>* fb = buf + f * tile + l0 * M;
    const bool phys = a.xmode == XMODE_C2R;
    fft_lines(fb, a.px, lb, false, a.tw, T(1), a.err,
              [&](int l, int k) {
                if (l0 + l >= nr) return mk<T>(0, 0);
                return c2r_pre<T>([&](int i) { return src[(size_t)l * M + i]; }, M, a.tw, k);
              },
              [&](int l, int k, cpx<T> v) {
                if (!phys) {
                  fb[l * M + k] = v;
                } else if (l0 + l < nr) {
                  T* dst = real_row(f, l0 + l);
                  dst[2 * k] = v.x;
                  dst[2 * k + 1] = v.y;
                }
              });
    if (phys) return;
    __syncthreads();
  }

  if (xmode_cross(a.xmode)) {
    // (fields 0..2) x (fields 3..5) on the packed real rows, written over fields 0..2
    T* re = reinterpret_cast<T*>(buf);
    const int rt = 2 * tile;  // reals per field
    T m0 = 0, m1 = 0, m2 = 0;
    for (int e = threadIdx.x; e < 2 * nr * M; e += blockDim.x) {
      const T u0 = re[e], u1 = re[rt + e], u2 = re[2 * rt + e];
      const T w0 = re[3 * rt + e], w1 = re[4 * rt + e], w2 = re[5 * rt + e];
      m0 = fmax(m0, fabs(u0));
      m1 = fmax(m1, fabs(u1));
      m2 = fmax(m2, fabs(u2));
      re[e] = fma1(u1, w2, -(u2 * w1));
      re[rt + e] = fma1(u2, w0, -(u0 * w2));
      re[2 * rt + e] = fma1(u0, w1, -(u1 * w0));
    }
    __syncthreads();
    // CFL: max |u_i| of the rows (omega, fields 3..5, is no longer needed: scratch)
    if (a.umax && a.xmode == XMODE_NONLINEAR) block_max3<T>(m0, m1, m2, re + 3 * rt, a.umax);
  }

  // forward r2c of fields 0..2
  {
    int f, l0;
    const LineBatch lb = batch(3, f, l0);
    cpx<T>* fb = buf + f * tile + l0 * M;
    fft_lines(fb, a.px, lb, a.xmode != XMODE_R2C, a.tw, T(-1), a.err,
              [&](int l, int k) {
                if (l0 + l >= nr) return mk<T>(0, 0);
                const T* src = real_row(f, l0 + l);
                return mk<T>(src[2 * k], src[2 * k + 1]);
              },
              [&](int l, int k, cpx<T> v) { fb[l * M + k] = v; });
  }
  __syncthreads();
  const int npair = a.dNP.d;
  for (int f = 0; f < 3; ++f) {
    cpx<T>* dst = a.scr + f * sstride + (size_t)r0 * M;
    for (int e = threadIdx.x; e < nr * npair; e += blockDim.x) {
      const int r = fdiv(e, a.dNP), k = e - r * npair;
      if (k == 0 || k < M - k) r2c_post(dst + (size_t)r * M, buf + f * tile + r * M, M, a.tw, k);
    }
  }
}

// ----------------------------------------------------------------------------------------
// Forcing amplitude (Sec. 2 / 6.1; reading: an Euler step of the forcing injects eps*dt)
// ----------------------------------------------------------------------------------------
template <typename T>
__global__ void k_force_coef(const cpx<double>* __restrict__ pj, const cpx<double>* __restrict__ pj1,
                             double theta, const cpx<T>* __restrict__ shell, int fK, double dt,
                             double eps, cpx<T>* force, double* coef_out) {
  __shared__ double sb[256], sc[256];
  const int D1 = 2 * fK + 1, D = D1 * D1 * (fK + 1);
  double b = 0, c = 0;
  for (int i = threadIdx.x; i < D; i += blockDim.x) {
    const int kx = i % (fK + 1);
    const double w = kx == 0 ? 1.0 : 2.0;
    for (int comp = 0; comp < 3; ++comp) {
      cpx<double> p0 = pj[comp * D + i], p1 = pj1[comp * D + i];
      double fx = (1.0 - theta) * p0.x + theta * p1.x;
      double fy = (1.0 - theta) * p0.y + theta * p1.y;
      cpx<T> s = shell[comp * D + i];
      b += w * ((double)s.x * fx + (double)s.y * fy);
      c += w * (fx * fx + fy * fy);
    }
  }
  sb[threadIdx.x] = b;
  sc[threadIdx.x] = c;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      sb[threadIdx.x] += sb[threadIdx.x + s];
      sc[threadIdx.x] += sc[threadIdx.x + s];
    }
    __syncthreads();
  }
  const double B = sb[0], C = 0.5 * dt * sc[0];
  const double q = sqrt(B * B + 4.0 * C * eps);
  const double amp = (B >= 0.0) ? 2.0 * eps / (B + q) : 2.0 * eps / (B - q);
  for (int i = threadIdx.x; i < D; i += blockDim.x) {
    for (int comp = 0; comp < 3; ++comp) {
      cpx<double> p0 = pj[comp * D + i], p1 = pj1[comp * D + i];
      double fx = (1.0 - theta) * p0.x + theta * p1.x;
      double fy = (1.0 - theta) * p0.y + theta * p1.y;
      force[comp * D + i] = mk<T>((T)(amp * fx), (T)(amp * fy));
    }
  }
  if (threadIdx.x == 0 && coef_out) coef_out[0] = amp;
}

// ----------------------------------------------------------------------------------------
// Reductions (FP64 across threads and blocks; per thread FP64, or compensated FP32 for FP32
// states; fixed-order tree: bitwise reproducible)
// ----------------------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) k_energy(const cpx<T>* __restrict__ S, int N, double nu,
                                                double* partial) {
  __shared__ double se[256], sd[256];
  const int M = N / 2;
  const size_t nmode = (size_t)N * N * M;
  double e = 0, d = 0;
  if constexpr (sizeof(T) == 4) {
    // FP32 state: the terms in FP32 and each thread's share (about a hundred modes) summed
    // with compensated (Kahan) FP32 additions, then the partial sums reduced in FP64 (FP64
    // arithmetic per mode is ALU-bound on this GPU)
    float es = 0.f, ec = 0.f, ds = 0.f, dc = 0.f;
    auto kahan = [](float& sum, float& comp, float x) {
      const float y = x - comp;
      const float t = sum + y;
      comp = (t - sum) - y;
      sum = t;
    };
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nmode;
         i += (size_t)gridDim.x * blockDim.x) {
      const int kx = (int)(i % M);
      const size_t r = i / M;
      const int iy = (int)(r % N), iz = (int)(r / N);
      const int ky = kof(iy, N), kz = kof(iz, N);
      float a2 = 0.f;
      for (int c = 0; c < 3; ++c) {
        const cpx<T> v = S[i + c * nmode];
        a2 = fmaf((float)v.x, (float)v.x, fmaf((float)v.y, (float)v.y, a2));
      }
      const float te = (kx == 0 ? 1.f : 2.f) * a2;
      kahan(es, ec, te);
      kahan(ds, dc, te * (float)(kx * kx + ky * ky + kz * kz));
    }
    e = (double)es - (double)ec;
    d = (double)ds - (double)dc;
  } else {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nmode;
         i += (size_t)gridDim.x * blockDim.x) {
      const int kx = (int)(i % M);
      const size_t r = i / M;
      const int iy = (int)(r % N), iz = (int)(r / N);
      const int ky = kof(iy, N), kz = kof(iz, N);
      const double w = kx == 0 ? 1.0 : 2.0;
      double a2 = 0;
      for (int c = 0; c < 3; ++c) {
        cpx<T> v = S[i + c * nmode];
        a2 += (double)v.x * (double)v.x + (double)v.y * (double)v.y;
      }
      e += w * a2;
      d += w * (double)(kx * kx + ky * ky + kz * kz) * a2;
    }
  }
  se[threadIdx.x] = e;
  sd[threadIdx.x] = d;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      se[threadIdx.x] += se[threadIdx.x + s];
      sd[threadIdx.x] += sd[threadIdx.x + s];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    partial[2 * blockIdx.x] = 0.5 * se[0];
    partial[2 * blockIdx.x + 1] = nu * sd[0];
  }
}

// out = (f0 * sum_i partial[2i], f1 * sum_i partial[2i+1]) in a fixed order (one block)
static __global__ void k_sum_pairs(const double* partial, int nblk, double* out, double f0 = 1.0,
                                   double f1 = 1.0) {
  __shared__ double s0[256], s1[256];
  double a = 0, b = 0;
  for (int i = threadIdx.x; i < nblk; i += blockDim.x) {
    a += partial[2 * i];
    b += partial[2 * i + 1];
  }
  s0[threadIdx.x] = a;
  s1[threadIdx.x] = b;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      s0[threadIdx.x] += s0[threadIdx.x + s];
      s1[threadIdx.x] += s1[threadIdx.x + s];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = f0 * s0[0];
    out[1] = f1 * s1[0];
  }
}

// spectrum partials: block b accumulates its modes into smem bins, writes partial[b][bin]
// Binned quadratic forms of the half spectrum, weights 1/2 at kx = 0 and 1 elsewhere (so a
// bin holds half the full-spectrum sum): q = 0, |S|^2 (energy spectrum); q = 1, 2 Re(S* . B)
// (nonlinear transfer T(k) for B = N); q = 2, 2 nu k^2 |S|^2 (dissipation spectrum).
template <typename T>
__global__ void __launch_bounds__(256) k_spectrum(const cpx<T>* __restrict__ S, int N, int kind,
                                                  int nbins, double* partial, int q = 0,
                                                  const cpx<T>* __restrict__ B = nullptr,
                                                  double nu = 0.0) {
  extern __shared__ double bins[];
  for (int i = threadIdx.x; i < nbins; i += blockDim.x) bins[i] = 0.0;
  __syncthreads();
  const int M = N / 2;
  const size_t nmode = (size_t)N * N * M;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nmode;
       i += (size_t)gridDim.x * blockDim.x) {
    const int kx = (int)(i % M);
    const size_t r = i / M;
    const int iy = (int)(r % N), iz = (int)(r / N);
    const int ky = kof(iy, N), kz = kof(iz, N);
    double a2 = 0;
    for (int c = 0; c < 3; ++c) {
      const cpx<T> v = S[i + c * nmode];
      if (q == 1) {
        const cpx<T> b = B[i + c * nmode];
        a2 += 2.0 * ((double)v.x * (double)b.x + (double)v.y * (double)b.y);
      } else {
        a2 += (double)v.x * (double)v.x + (double)v.y * (double)v.y;
      }
    }
    if (q == 2) a2 *= 2.0 * nu * (double)(kx * kx + ky * ky + kz * kz);
    if (a2 == 0.0) continue;
    const double w = kx == 0 ? 0.5 : 1.0;
    int bin;
    if (kind == 0) {
      bin = (int)floor(sqrt((double)(kx * kx + ky * ky + kz * kz)) + 0.5);
    } else if (kind == 1) {
      bin = kx;
    } else if (kind == 2) {
      bin = abs(ky);
    } else {
      bin = abs(kz);
    }
    if (bin < nbins) atomicAdd(&bins[bin], w * a2);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nbins; i += blockDim.x) partial[(size_t)blockIdx.x * nbins + i] = bins[i];
}

static __global__ void k_spectrum_final(const double* partial, int nblk, int nbins, double* out) {
  int bin = blockIdx.x * blockDim.x + threadIdx.x;
  if (bin >= nbins) return;
  double s = 0;
  for (int b = 0; b < nblk; ++b) s += partial[(size_t)b * nbins + bin];
  out[bin] = s;
}

// ----------------------------------------------------------------------------------------
// Adjoint step building blocks (pointwise on [3][N][N][M] spectral arrays)
// ----------------------------------------------------------------------------------------
enum EwOp {
  EW_ROG_S1 = 0,   // o = E_dt (x + dt y)                         (S1 = E(S0 + dt N0))
  EW_ROG_SN = 1,   // o = E_dt x + dt/2 E_{dt/2} (y + z)          (S = E S0 + dt/2 Eh (N0 + N1))
  EW_RHO = 2,      // o = dt/2 E_{dt/2} x
  EW_SIGMA = 3,    // o = dt E_dt x
  EW_LAMBDA = 4,   // o = E_dt (x + y) + z
  EW_ADD = 5,      // o = x + y
  EW_LOSS = 6,     // o = 2 nu k^2 x        (gradient of eps = nu <S, k^2 S>_w)
  EW_SCALE = 7,    // o = c x
  EW_CURL_ADD = 8  // o = x + i k x y
};

template <typename T>
__global__ void k_elementwise(int op, int N, T dt, T c, const T* __restrict__ ifac,
                              const cpx<T>* x, const cpx<T>* y, const cpx<T>* z, cpx<T>* o) {
  const int M = N / 2;
  const size_t nmode = (size_t)N * N * M;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nmode;
       i += (size_t)gridDim.x * blockDim.x) {
    const int kx = (int)(i % M);
    const size_t r = i / M;
    const int iy = (int)(r % N), iz = (int)(r / N);
    const T E1 = ifac[kx] * ifac[iy] * ifac[iz];
    const T Eh = ifac[N + kx] * ifac[N + iy] * ifac[N + iz];
    const T fx = (T)kx, fy = (T)kof(iy, N), fz = (T)kof(iz, N);
    if (op == EW_CURL_ADD) {
      const cpx<T> y0 = y[i], y1 = y[i + nmode], y2 = y[i + 2 * nmode];
      o[i] = x[i] + mul_si(fy * y2 - fz * y1, T(1));
      o[i + nmode] = x[i + nmode] + mul_si(fz * y0 - fx * y2, T(1));
      o[i + 2 * nmode] = x[i + 2 * nmode] + mul_si(fx * y1 - fy * y0, T(1));
      continue;
    }
    for (int q = 0; q < 3; ++q) {
      const size_t j = i + q * nmode;
      cpx<T> v;
      switch (op) {
        case EW_ROG_S1: v = E1 * (x[j] + dt * y[j]); break;
        case EW_ROG_SN: v = E1 * x[j] + (T(0.5) * dt * Eh) * (y[j] + z[j]); break;
        case EW_RHO: v = (T(0.5) * dt * Eh) * x[j]; break;
        case EW_SIGMA: v = (dt * E1) * x[j]; break;
        case EW_LAMBDA: v = E1 * (x[j] + y[j]) + z[j]; break;
        case EW_ADD: v = x[j] + y[j]; break;
        case EW_LOSS: v = (T(2) * c * (fx * fx + fy * fy + fz * fz)) * x[j]; break;
        default: v = c * x[j]; break;
      }
      o[j] = v;
    }
  }
}

// dense forcing table [3][D] <-> spectral array at the table's modes
template <typename T>
__global__ void k_shell_gather(const cpx<T>* __restrict__ S, int N, int fK, cpx<T>* shell) {
  const int D1 = 2 * fK + 1, D = D1 * D1 * (fK + 1), M = N / 2;
  const size_t nmode = (size_t)N * N * M;
  for (int i = threadIdx.x; i < D; i += blockDim.x) {
    const int kx = i % (fK + 1), ky = (i / (fK + 1)) % D1 - fK, kz = i / ((fK + 1) * D1) - fK;
    const size_t g = ((size_t)((kz + N) % N) * N + (size_t)((ky + N) % N)) * M + kx;
    for (int c = 0; c < 3; ++c) shell[c * D + i] = S[g + c * nmode];
  }
}
template <typename T>
__global__ void k_shell_add(cpx<T>* S, int N, int fK, const cpx<T>* __restrict__ tab) {
  const int D1 = 2 * fK + 1, D = D1 * D1 * (fK + 1), M = N / 2;
  const size_t nmode = (size_t)N * N * M;
  for (int i = threadIdx.x; i < D; i += blockDim.x) {
    const int kx = i % (fK + 1), ky = (i / (fK + 1)) % D1 - fK, kz = i / ((fK + 1) * D1) - fK;
    const size_t g = ((size_t)((kz + N) % N) * N + (size_t)((ky + N) % N)) * M + kx;
    for (int c = 0; c < 3; ++c) S[g + c * nmode] = S[g + c * nmode] + tab[c * D + i];
  }
}

// adjoint of S -> a(S) f at one stage applied to rho: table = (da/db) Re<f, rho>_w f with
// da/db = -|a| / sqrt(b^2 + 4 c eps), b = Re<S, f>_w, c = dt/2 <f, f>_w
template <typename T>
__global__ void k_force_vjp(const cpx<double>* __restrict__ pj, const cpx<double>* __restrict__ pj1,
                            double theta, const cpx<T>* __restrict__ shS,
                            const cpx<T>* __restrict__ shR, int fK, double dt, double eps,
                            cpx<T>* tab) {
  __shared__ double sb[256], sc[256], sr[256];
  const int D1 = 2 * fK + 1, D = D1 * D1 * (fK + 1);
  double b = 0, c = 0, r = 0;
  for (int i = threadIdx.x; i < D; i += blockDim.x) {
    const double w = (i % (fK + 1)) == 0 ? 1.0 : 2.0;
    for (int q = 0; q < 3; ++q) {
      const cpx<double> p0 = pj[q * D + i], p1 = pj1[q * D + i];
      const double fx = (1.0 - theta) * p0.x + theta * p1.x, fy = (1.0 - theta) * p0.y + theta * p1.y;
      const cpx<T> s = shS[q * D + i], x = shR[q * D + i];
      b += w * ((double)s.x * fx + (double)s.y * fy);
      c += w * (fx * fx + fy * fy);
      r += w * ((double)x.x * fx + (double)x.y * fy);
    }
  }
  sb[threadIdx.x] = b;
  sc[threadIdx.x] = c;
  sr[threadIdx.x] = r;
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      sb[threadIdx.x] += sb[threadIdx.x + s];
      sc[threadIdx.x] += sc[threadIdx.x + s];
      sr[threadIdx.x] += sr[threadIdx.x + s];
    }
    __syncthreads();
  }
  const double B = sb[0], C = 0.5 * dt * sc[0], R = sr[0];
  const double q = sqrt(B * B + 4.0 * C * eps);
  const double amp = (B >= 0.0) ? 2.0 * eps / (B + q) : 2.0 * eps / (B - q);
  const double coef = -fabs(amp) / q * R;
  for (int i = threadIdx.x; i < D; i += blockDim.x) {
    for (int k = 0; k < 3; ++k) {
      const cpx<double> p0 = pj[k * D + i], p1 = pj1[k * D + i];
      const double fx = (1.0 - theta) * p0.x + theta * p1.x, fy = (1.0 - theta) * p0.y + theta * p1.y;
      tab[k * D + i] = mk<T>((T)(coef * fx), (T)(coef * fy));
    }
  }
}

// Block [lo, lo + n) of axis 0 (z or kz) or 1 (ky) of a buffer of F fields in layout `pairs`
// (mixed_index serves Ft as well: it has fields 0 .. 2 only) <-> contiguous [F][...] staging
template <typename T>
__global__ void k_block_copy(cpx<T>* buf, cpx<T>* stg, int F, int N, int axis, int lo, int n, int pairs, int to_buf) {
  const int M = N / 2;
  const size_t fs = (size_t)N * N * M, per = (size_t)n * N * M;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < F * per; i += (size_t)gridDim.x * blockDim.x) {
    const int f = (int)(i / per), kx = (int)(i % M);
    const size_t r = (i % per) / M;  // axis 0: z N + y of the block; axis 1: z n + y
    const size_t z = axis == 0 ? lo + r / N : r / n, y = axis == 0 ? r % N : lo + r % n;
    cpx<T>* p = buf + mixed_index(pairs, f, (z * N + y) * M + kx, fs);
    if (to_buf) *p = stg[i];
    else stg[i] = *p;
  }
}

// convert between the working precision and FP64 (state transfers)
template <typename T>
__global__ void k_to_double(const cpx<T>* __restrict__ in, cpx<double>* out, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    cpx<T> v = in[i];
    out[i] = mk<double>((double)v.x, (double)v.y);
  }
}
template <typename T>
__global__ void k_from_double(const cpx<double>* __restrict__ in, cpx<T>* out, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    cpx<double> v = in[i];
    out[i] = mk<T>((T)v.x, (T)v.y);
  }
}
template <typename T>
__global__ void k_real_to_double(const T* __restrict__ in, double* out, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    out[i] = (double)in[i];
}
template <typename T>
__global__ void k_real_from_double(const double* __restrict__ in, T* out, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    out[i] = (T)in[i];
}

}  // namespace ns
