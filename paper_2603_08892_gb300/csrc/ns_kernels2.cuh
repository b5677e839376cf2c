// ns_kernels2.cuh -- the hot kernels specialised on the grid size N (compile-time FFTs).
//
// Same passes, layouts and arithmetic as the generic kernels of ns_kernels.cuh (see there
// for the data layout): k2_pencil = z transforms + spectral stage of Sec. 4 / 6.1,
// k2_yinv / k2_xrow / k2_yfwd = slab pass (y transforms, x rows with u x omega), and
// k2_slabpipe = the slab pass as one persistent pipelined launch.  What changes is how the
// transforms run: the first stage's inputs and the last stage's outputs are in registers, which
// global memory or a pointwise operation fills and takes (ns_fft3.cuh), the stages between them go
// through shared memory, every index is a compile-time expression, and the butterflies are of
// radix 2 to 16 (per kernel and size, K2Cfg).
#pragma once

#include "ns_fft3.cuh"
#include "ns_kernels.cuh"

namespace ns {

__host__ __device__ constexpr int cmin(int a, int b) { return a < b ? a : b; }
__host__ __device__ constexpr int cmax(int a, int b) { return a > b ? a : b; }
__host__ __device__ constexpr int pick_div(int m, int target, int cap) {
  int t = cmin(cmax(target, 1), cap);
  for (int d = t; d >= 1; --d)
    if (m % d == 0) return d;
  return 1;
}
__host__ __device__ constexpr int cgcd(int a, int b) { return b == 0 ? a : cgcd(b, a % b); }
// thread count: >= t, >= 64, a multiple of the warp size and of w (each thread keeps one line)
__host__ __device__ constexpr int round_lines(int t, int w) {
  const int l = 32 / cgcd(32, w) * w;
  const int v = cmax(t, 64);
  return (v + l - 1) / l * l;
}

// two modes side by side in memory (16 bytes in FP32): the fields that share a line of the x rows
template <typename T>
struct alignas(16) cpair {
  cpx<T> a, b;
};

// Global-memory access policy.  MemNC: data written by earlier launches (read-only path).
// MemCG: data written by other blocks of the same launch (persistent kernel): loads and
// stores go to L2 (.cg) so a block never sees a stale line in its own L1.
struct MemNC {
  template <typename T>
  static __device__ __forceinline__ cpx<T> ld(const cpx<T>* p) { return ldg(p); }
  template <typename T>
  static __device__ __forceinline__ cpx<T> ldw(const cpx<T>* p) { return *p; }
  template <typename T>
  static __device__ __forceinline__ void st(cpx<T>* p, cpx<T> v) { *p = v; }
  static __device__ __forceinline__ void ldp(const cpair<float>* p, cpx<float>& a, cpx<float>& b) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    a = mk<float>(v.x, v.y);
    b = mk<float>(v.z, v.w);
  }
  static __device__ __forceinline__ void ldp(const cpair<double>* p, cpx<double>& a, cpx<double>& b) {
    a = p->a;
    b = p->b;
  }
  static __device__ __forceinline__ void stp(cpair<float>* p, cpx<float> a, cpx<float> b) {
    *reinterpret_cast<float4*>(p) = make_float4(a.x, a.y, b.x, b.y);
  }
  static __device__ __forceinline__ void stp(cpair<double>* p, cpx<double> a, cpx<double> b) {
    p->a = a;
    p->b = b;
  }
};
struct MemCG {
  static __device__ __forceinline__ cpx<float> ld(const cpx<float>* p) {
    const float2 v = __ldcg(reinterpret_cast<const float2*>(p));
    return mk<float>(v.x, v.y);
  }
  static __device__ __forceinline__ cpx<double> ld(const cpx<double>* p) {
    const double2 v = __ldcg(reinterpret_cast<const double2*>(p));
    return mk<double>(v.x, v.y);
  }
  template <typename T>
  static __device__ __forceinline__ cpx<T> ldw(const cpx<T>* p) { return ld(p); }
  static __device__ __forceinline__ void st(cpx<float>* p, cpx<float> v) {
    __stcg(reinterpret_cast<float2*>(p), make_float2(v.x, v.y));
  }
  static __device__ __forceinline__ void st(cpx<double>* p, cpx<double> v) {
    __stcg(reinterpret_cast<double2*>(p), make_double2(v.x, v.y));
  }
  static __device__ __forceinline__ void ldp(const cpair<float>* p, cpx<float>& a, cpx<float>& b) {
    const float4 v = __ldcg(reinterpret_cast<const float4*>(p));
    a = mk<float>(v.x, v.y);
    b = mk<float>(v.z, v.w);
  }
  static __device__ __forceinline__ void ldp(const cpair<double>* p, cpx<double>& a, cpx<double>& b) {
    a = ld(&p->a);
    b = ld(&p->b);
  }
  static __device__ __forceinline__ void stp(cpair<float>* p, cpx<float> a, cpx<float> b) {
    __stcg(reinterpret_cast<float4*>(p), make_float4(a.x, a.y, b.x, b.y));
  }
  static __device__ __forceinline__ void stp(cpair<double>* p, cpx<double> a, cpx<double> b) {
    st(&p->a, a);
    st(&p->b, b);
  }
};

// The alternative width of a tile (lines per tile): twice the default where that divides
// the half length m within the cap, else half (down to minw), else the default.
__host__ __device__ constexpr int alt_width(int w, int m, int cap, int minw) {
  return (m % (2 * w) == 0 && 2 * w <= cap) ? 2 * w : ((w / 2 >= minw && m % (w / 2) == 0) ? w / 2 : w);
}

// columns of a tile of `per` threads per column: 64-byte rows (128 bytes for an interleaved pair),
// fewer where that makes more than `lim` threads or, on small grids, fewer than a block for each of the
// 152 SMs; twice as many where that fills the warps and leaves 128 blocks (a step of 48^3 FP64 217 us
// with 8 columns, 96 threads, and 234 with 4).  wide (single FP32 grids of N <= 64): 128-byte rows, however
// few the blocks (fewer, fuller warps; a step at 24^3 48.0 us and 52.3 with 6 columns in the y passes, 32^3 51.1 and
// 52.5; at 48^3 with two other grids stepping 26.9 and 28.3, at 64^3 29.0 and 30.2).
__host__ __device__ constexpr int y_cols(int n, int per, int minw, int lim, bool wide) {
  int w = pick_div(n / 2, (wide ? 4 : 2) * minw, 16);
  while (w > minw && w % 2 == 0 && (w * per > lim || (!wide && n / 2 / w * n < 152 && w / 2 * per >= 32))) w /= 2;
  if (!wide && w * per % 32 && 2 * w * per % 32 == 0 && n / 2 % (2 * w) == 0 && n / (4 * w) * n >= 128) w *= 2;
  return w;
}

// Radix plans of the z, y and x transforms.  FP32: the x rows and both y passes with radix 16,
// except where that keeps a radix-2 stage that radix 8 avoids on N <= 128 (N = 32, 96).
__host__ __device__ constexpr bool plan_has_radix2(int n, int mr) {
  const CPlan p = cplan(n, mr);
  for (int i = 0; i < p.nst; ++i)
    if (p.r[i] == 2) return true;
  return false;
}
__host__ __device__ constexpr int slab_radix(int n) {
  return n <= 128 && plan_has_radix2(n, 16) && !plan_has_radix2(n, 8) ? 8 : 16;
}
// FP64 from N = 16 to 96: radix 4.  The FP64 pipes bound these grids, and an SM needs several full
// warps to keep its share of them busy: radix 4 gives 2 to 3 times the threads of radix 8 and 12 (a y
// tile of 48^3 has 48 instead of 16).  Steps with radix 4 and with 8 or 12, us: 16^3 133 and 138,
// 48^3 235 and 325, 64^3 389 and 403, 96^3 1260 and 1540; 128^3 2616 and 2578, 192^3 9740 and 9590.
// (24 and 32 were set to radix 4 before: 32^3 161 and 268.)
// The x rows of sizes whose FP32 tiles of x_rows rows do not divide the planes (192, 384) have no
// reproducible pairing of rows to keep and take the plan with the fewest stages.
__host__ __device__ constexpr bool small64(int n) { return n >= 16 && n <= 96; }
__host__ __device__ constexpr int x_rows(int n, int cs) { return cmin(cmax(8192 / (n / 2 * cs), 1), 16); }
template <typename T, int N>
struct ZPlan { static constexpr CPlan P = fplan<T>(N, 8, small64(N) ? 4 : 8); };
template <typename T, int N>
struct YPlan { static constexpr CPlan P = fplan<T>(N, slab_radix(N), small64(N) ? 4 : 12); };
template <typename T, int N>
struct XPlan {
  // (a pass holds every plane up to N = 96, groups of whole planes beyond)
  static constexpr bool FREE = sizeof(T) == 8 || (N < 128 ? N * N : N) % x_rows(N, (int)sizeof(cpx<T>)) != 0;
  static constexpr CPlan P = FREE ? radix_plan(N, sizeof(T) == 4 ? 16 : small64(N) ? 4 : 12) : fplan<T>(N, slab_radix(N), 12);
};

// Tile shapes of size N.  V selects compiled alternatives for the autotuner, one bit per
// kernel family: bit 0 the pencil width TX, bit 1 the inverse-y width TYI, bit 3 the forward-y
// width TY (V = 0: the defaults).  Bit 2: a single grid of N <= 64, whose launches put one or two
// blocks of a few warps on an SM and last for as long as one thread's loads and stages follow one
// another: the pencil may take every register and loads the state before the first transform
// (pencil_tile, EARLY), the x rows take twice the threads of their products for the stages, which
// have more lines than that.  A step at 48^3 FP32 64.0 us (70.6 without, 66.7 with the kernels that
// staged every tile), 24^3 47.3 (52.6, 56.6); 24^3 FP64 164 (177).
template <typename T, int N, int V = 0>
struct K2Cfg {
  static constexpr int M = N / 2;
  static constexpr int CS = (int)sizeof(cpx<T>);
  static constexpr int MINW = 32 / CS;  // 32-byte global segments
  static constexpr bool F32 = sizeof(T) == 4;
  static constexpr bool FEW = (V & 4) && N <= 64;  // bit 2
  // pencil: TX columns of N, three tiles in shared memory, one thread per column and first-stage
  // butterfly (radix f); registers hold 3 f modes
  static constexpr int ZF = ZPlan<T, N>::P.r[0], ZNB = N / ZF;
  // FP32 energy sums: the grouping of the modes that one thread adds in FP32 (N / 8, except on the
  // small grids whose N / 8 threads per column are not whole warps), kept as it was recorded with;
  // a wide tile needs a thread for each of its groups (not so at N = 24)
  static constexpr int EDX = pick_div(M, cmax(16384 / (N * CS), MINW), 16);
  static constexpr int EDZ = F32 && N >= 24 ? round_lines(EDX * N / 8, EDX) / EDX : ZNB;
  static constexpr int TXW = y_cols(N, ZNB, MINW, 512, true);
  static constexpr bool ZWIDE = FEW && F32 && (EDZ == ZNB || TXW * EDZ <= (TXW * ZNB + 31) / 32 * 32);
  static constexpr int TX0 = ZWIDE ? TXW : y_cols(N, ZNB, MINW, 512, false);
  static constexpr int TX = (V & 1) ? alt_width(TX0, M, 512 / ZNB, MINW) : TX0;
  static constexpr int NTP = (TX * ZNB + 31) / 32 * 32;  // (whole warps: the energy sums shuffle)
  static constexpr int PTS = Xchg<T, N, ZF, TX, true>::elems;
  static constexpr int p_elems = 3 * PTS + tw_elems(N);
  // blocks per SM the register budget must allow
  static constexpr int PREGS = FEW ? 255 : F32 ? 128 : 168;
  static constexpr int p_blocks(int regs) {
    return cmax(1, cmin(cmin(16, 65536 / (NTP * regs)), (227 * 1024) / (p_elems * CS + 1024)));
  }
  static constexpr int MINB_P = p_blocks(PREGS);
  static constexpr int MINB_P2 = p_blocks(F32 && !FEW ? 168 : 255);  // two inputs and outputs
  // y passes: tiles of TYI / TY columns, three in shared memory, one thread per column and
  // last-stage butterfly
  static constexpr CPlan YP = YPlan<T, N>::P;
  static constexpr int YNB = N / YP.r[0];
  static constexpr int TY0 = y_cols(N, YNB, MINW, 192, FEW && F32), TYI0 = TY0;
  static constexpr int TY = (V & 8) ? alt_width(TY0, M, 512 / YNB, MINW) : TY0;
  static constexpr int TYI = (V & 2) ? alt_width(TYI0, M, 512 / YNB, MINW) : TYI0;
  static constexpr int NTY = TY * YNB, NTYI = TYI * YNB;
  static constexpr int y_elems(int w) { return 3 * (N + N / YP.r[0]) * w + tw_elems(N); }
  static constexpr int y_blocks(int w, int regs) {
    return cmax(1, cmin(cmin(16, 65536 / ((w * YNB + 31) / 32 * 32 * regs)), (227 * 1024) / (y_elems(w) * CS + 1024)));
  }
  static constexpr int YIREGS = F32 ? 160 : 168, YFREGS = F32 ? 144 : 168;
  static constexpr int MINB_YI = y_blocks(TYI, YIREGS);
  static constexpr int MINB_Y = y_blocks(TY, YFREGS);
  // x rows: tiles of RX rows in pairs (q, q + RXH), whose third products share a line; N / f
  // threads per row.  Two-stage plans whose threads of some pairs make one warp run warp by warp
  // (XWP pairs each), without block barriers; the others take twice the threads when FEW.
  static constexpr CPlan XP = XPlan<T, N>::P;
  static constexpr int XF0 = XP.r[0], XNB = N / XF0;
  static constexpr int RXT = x_rows(N, CS);
  static constexpr int RX0 = !XPlan<T, N>::FREE ? RXT : small64(N) ? 4 : cmax(2, RXT / 2 * 2);
  static constexpr bool XWARP = XP.nst == 2 && XF0 % XP.r[XP.nst - 1] == 0 && RX0 % 2 == 0 && 2 * XNB <= 32 &&
                                32 % (2 * XNB) == 0 && (RX0 * XNB) % 32 == 0;
  static constexpr int RX = RX0, RXH = (RX0 + 1) / 2;
  static constexpr int XWP = XWARP ? 32 / (2 * XNB) : RXH;       // pairs of a group
  static constexpr int XNG = XWARP ? RXH / XWP : 1;              // groups of a tile
  static constexpr int XGT = XWARP ? 32 : (2 * RXH * XNB * (FEW ? 2 : 1) + 31) / 32 * 32;  // threads of a group
  static constexpr int NTX = XNG * XGT;
  static constexpr int XGEL = Xchg<T, N, XF0, 6 * XWP, false>::elems;
  static constexpr int XELEMS = XNG * XGEL + 32;                 // and the scratch of the block's maxima
  static constexpr int XREGS = F32 ? 144 : 168;
  static constexpr int MINB_X = cmax(1, cmin(cmin(16, 65536 / (NTX * XREGS)),
                                             (227 * 1024) / ((XELEMS + tw_elems(N)) * CS + 1024)));
};

// ---- accessors ------------------------------------------------------------------------
template <typename T, int W>
struct SmTile {  // shared [e][line]
  cpx<T>* p;
  __device__ __forceinline__ cpx<T> get(int line, int e) const { return p[lf_idx<T, W>(e, line)]; }
  __device__ __forceinline__ void put(int line, int e, cpx<T> v) const { p[lf_idx<T, W>(e, line)] = v; }
};
// 1 / k^2 of the projection: FP32 uses the fast division intrinsic (within 2 ulp, far below
// the FP32 path's per-step error), FP64 the correctly rounded division.
template <typename T>
__device__ __forceinline__ T recip_k2(int k2);
template <>
__device__ __forceinline__ float recip_k2<float>(int k2) { return __fdividef(1.0f, (float)k2); }
template <>
__device__ __forceinline__ double recip_k2<double>(int k2) { return 1.0 / (double)k2; }

template <int I>
struct IntC { static constexpr int v = I; };

// Sums of products in one fixed rounding order (the kernels of a pass have many instances, each
// of which the compiler could contract in its own way): a x + b y, its first product fused
// (x, the state, is the large term), and x + b y
template <typename T>
__device__ __forceinline__ cpx<T> lin2(T a, cpx<T> x, T b, cpx<T> y) {
  return mk<T>(fma1(a, x.x, b * y.x), fma1(a, x.y, b * y.y));
}
template <typename T>
__device__ __forceinline__ cpx<T> lin1(cpx<T> x, T b, cpx<T> y) {
  return mk<T>(fma1(b, y.x, x.x), fma1(b, y.y, x.y));
}

// ---- spectral stage at one mode (Sec. 4.1, 4.2, 6.1) ----------------------------------
// nv: de-shifted, weighted transform of u x omega at the mode: N(0) = 0, truncation T,
// Leray projection P, then the forcing term O (added on the modes of the forcing table).
template <typename T>
__device__ __forceinline__ void project_point(const PencilArgs<T>& a, int kx, int ky, int kz,
                                              cpx<T> nv[3]) {
  const int k2 = kx * kx + ky * ky + kz * kz;
  const bool keep = trunc_keep(a.trunc, kx, ky, kz, a.N, a.K2max, a.Kimax) && (k2 != 0);
  if (keep) {
    const cpx<T> v0 = nv[0], v1 = nv[1], v2 = nv[2];
    const T fx = (T)kx, fy = (T)ky, fz = (T)kz;
    const T ik2 = recip_k2<T>(k2);
    const cpx<T> kd = mk<T>(fma1(fz, v2.x, fma1(fx, v0.x, fy * v1.x)), fma1(fz, v2.y, fma1(fx, v0.y, fy * v1.y)));
    nv[0] = v0 - (fx * ik2) * kd;
    nv[1] = v1 - (fy * ik2) * kd;
    nv[2] = v2 - (fz * ik2) * kd;
  } else {
    nv[0] = nv[1] = nv[2] = mk<T>(0, 0);
  }
  if (a.force && kx <= a.fK && abs(ky) <= a.fK && abs(kz) <= a.fK) {
    const int D1 = 2 * a.fK + 1, D = D1 * D1 * (a.fK + 1);
    const int fi = ((kz + a.fK) * D1 + (ky + a.fK)) * (a.fK + 1) + kx;
#pragma unroll
    for (int c = 0; c < 3; ++c) nv[c] = nv[c] + a.force[c * D + fi];
  }
}

// RK stage combine of component c at one mode (modes of PencilMode).  s0: the value read
// from src (INIT), acc (RK4_4) or state (all other modes); s1: acc for RK4_2 / RK4_3.
// Performs the mode's global writes and returns S_next.
// mode: the pencil's stage (a.mode, or a compile-time constant in the specialised kernels)
template <typename T, class MP>
__device__ __forceinline__ cpx<T> stage_combine(const PencilArgs<T>& a, int c, size_t g, cpx<T> n,
                                                cpx<T> s0, cpx<T> s1, T E1, T Eh, int mode) {
  const T dt = a.dt, hdt = T(0.5) * a.dt;
  (void)c;
  switch (mode) {
    case MODE_INIT:
      return s0;
    case MODE_RK2_1:
      return Eh * lin1(s0, hdt, n);
    case MODE_RK2_2: {
      const cpx<T> s = lin2(E1, s0, dt * Eh, n);
      MP::st(&a.state[g], s);
      return s;
    }
    case MODE_RK4_1:
      MP::st(&a.acc[g], lin2(E1, s0, dt / T(6) * E1, n));
      return Eh * lin1(s0, hdt, n);
    case MODE_RK4_2:
      MP::st(&a.acc[g], lin1(s1, dt / T(3) * Eh, n));
      return lin2(Eh, s0, hdt, n);
    case MODE_RK4_3:
      MP::st(&a.acc[g], lin1(s1, dt / T(3) * Eh, n));
      return lin2(E1, s0, dt * Eh, n);
    case MODE_RK4_4: {
      const cpx<T> s = lin1(s0, dt / T(6), n);
      MP::st(&a.state[g], s);
      return s;
    }
    case MODE_ROG_1:
      MP::st(&a.state[g], lin2(E1, s0, hdt * Eh, n));
      return E1 * lin1(s0, dt, n);
    case MODE_ROG_2: {
      const cpx<T> s = lin1(s0, hdt * Eh, n);
      MP::st(&a.state[g], s);
      return s;
    }
    case MODE_NL:
      MP::st(&a.acc[g], n);
      return mk<T>(0, 0);
    default:  // MODE_PROJECT
      MP::st(&a.state[g], n);
      return mk<T>(0, 0);
  }
}

// S_next of component c at the modes of the forcing table (the forcing amplitude of the
// next stage needs Re<S_next, f>)
template <typename T, class MP>
__device__ __forceinline__ void shell_record(const PencilArgs<T>& a, int c, int kx, int ky, int kz,
                                             cpx<T> sn) {
  if (a.shell && kx <= a.fK && abs(ky) <= a.fK && abs(kz) <= a.fK) {
    const int D1 = 2 * a.fK + 1, D = D1 * D1 * (a.fK + 1);
    const int fi = ((kz + a.fK) * D1 + (ky + a.fK)) * (a.fK + 1) + kx;
    MP::st(&a.shell[c * D + fi], sn);
  }
}

// ---- pencil pass --------------------------------------------------------------------
// One tile: TX consecutive kx at one ky, all kz; 3 shared tiles and the twiddle table.
//
// Bound by HBM (ROG stages: 3 + 3 fields read, 3 + 5 written) and, where every stage passes
// through it, by shared memory.  The forward transforms' first stage reads Ft, the inverse ones'
// last stage writes the mixed fields, and in between a thread holds the f modes kz(j + (N/f) r)
// of its column for all three components in registers: the outputs of its K = f / l last forward
// butterflies and the inputs of its first inverse one (see radix plans; where l does not divide f
// the last forward stage goes through shared memory), so de-shift, N(0) = 0, truncation,
// projection, forcing, the stage combine, the shift and i kz never touch shared memory.  Measured,
// one Rogallo stage, FP32: 256^3 201 us (214 with every stage through shared memory), 512^3 1941
// (2278), 128^3 26.9 (30.6).  From 384^3 on the pattern itself limits it: a copy with 64-byte
// segments per plane and array reaches 3.3 TB/s at 512^3, with 128-byte ones 6.5 TB/s, hence the
// interleaved pairs of fields (5.1 TB/s with the state still in 64-byte segments).

// True when every mode of a pencil tile (kx in [x0, x0 + TX), this ky, every kz) lies outside
// the truncation and none is in the forcing table: the truncated nonlinear term and the
// forcing vanish there, so the tile's forward transforms are skipped (Sec. 2, truncation).
template <typename T, int TX>
__device__ __forceinline__ bool pencil_tile_truncated(const PencilArgs<T>& a, int x0, int ky) {
  bool out;  // the no-double-alias mask lies inside the sphere: the spherical test is safe
  if (a.trunc == 1)
    out = x0 > a.Kimax || abs(ky) > a.Kimax;
  else
    out = (long long)x0 * x0 + (long long)ky * ky > (long long)a.K2max;
  const bool forced = (a.force != nullptr || a.shell != nullptr) && x0 <= a.fK && abs(ky) <= a.fK;
  return out && !forced;
}

// Zero columns of the outputs of a tile whose S_next vanishes (the inverse transforms of zero);
// in either layout of the fields a pair of them takes the bytes of two
template <typename T, int N, int TX, int NT, class MP>
__device__ __forceinline__ void pencil_zero_outputs(const PencilArgs<T>& a, int nOut, int iy, int x0) {
  constexpr int M = N / 2;
  const size_t fstride = (size_t)N * N * M;
  if (threadIdx.x >= NT) return;
  for (int o = 0; o < nOut; ++o)
    for (int i = threadIdx.x; i < N * TX; i += NT) {
      const size_t g = ((size_t)(i / TX) * N + iy) * M + x0 + i % TX;
      for (int f = 0; f < 5; f += f == 2 ? 1 : 2) {
        cpx<T>* p = a.out[o] + f * fstride;
        if (f == 2) {
          MP::st(p + g, mk<T>(0, 0));
        } else {
          MP::st(p + (a.pairs ? 2 * g : g), mk<T>(0, 0));
          MP::st(p + (a.pairs ? 2 * g + 1 : g + fstride), mk<T>(0, 0));
        }
      }
    }
}

// Energy and dissipation sums of the state a final-stage pencil tile writes (Sec. 3.4: E =
// 1/2 sum w |S|^2, eps = nu sum w k^2 |S|^2, w = 1 at kx = 0 and 2 elsewhere): each thread's
// sums (in T, a few modes each) are reduced across the block in FP64 and stored as the
// tile's pair; a fixed-order sum over the tiles follows.  Every thread of the block calls it.
template <typename T>
__device__ __forceinline__ void tile_energy_store(double* epart, T e, T d) {
  __shared__ double red[2][32];
  double a = (double)e, b = (double)d;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) {
    red[0][w] = a;
    red[1][w] = b;
  }
  __syncthreads();
  if (w == 0) {
    const int nw = (int)(blockDim.x + 31) >> 5;
    a = l < nw ? red[0][l] : 0.0;
    b = l < nw ? red[1][l] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_down_sync(0xffffffffu, a, o);
      b += __shfl_down_sync(0xffffffffu, b, o);
    }
    if (l == 0) {
      epart[2 * blockIdx.x] = a;
      epart[2 * blockIdx.x + 1] = b;
    }
  }
}

// NFC, NOC: the number of inputs and outputs (NOC -1: a.nOut, at most one: the persistent ensemble's
// last pass, which has an output but in the last step); MC: the stage mode.  (1, 1) is every RK2,
// Rogallo and RK4 stage, (2, 2) and (0, 2) the exact scheme's, (0, 1) INIT, (1, 0) NL and PROJECT.
// EP: the tile's energy sums are stored (NOC = 2: whenever a.epart is set).
template <typename T, int N, class MP, int NFC, int NOC, bool EP, int MC, int V = 0>
__device__ __forceinline__ void pencil_tile(const PencilArgs<T>& a, int tile_id, cpx<T>* buf) {
  using C = K2Cfg<T, N, V>;
  using PL = ZPlan<T, N>;
  constexpr int nst = PL::P.nst, f = PL::P.r[0], l = PL::P.r[nst - 1], NB0 = N / f, NBL = N / l;
  constexpr bool FUSE = f % l == 0;                    // last forward butterflies held by their thread
  constexpr int K = FUSE ? f / l : (f + l - 1) / l;    // last-stage butterflies per thread
  constexpr int M = N / 2, TX = C::TX, NT = TX * NB0, TS = C::PTS;
  using X = Xchg<T, N, f, TX, true>;
  static_assert(NT <= C::NTP, "one first-stage butterfly per thread");
  constexpr int ED = C::EDZ;  // the energy sums add a column's modes iz = i (mod ED) in T, then in FP64
  const int nF = NFC, nOut = NOC >= 0 ? NOC : a.nOut;
  constexpr int mode = MC;
  cpx<T>* tws = buf + 3 * TS;
  constexpr int ntx = M / TX;
  const int iy = a.iy0 + tile_id / ntx;  // (iy0: first ky row of a rank-range launch)
  const int x0 = (tile_id % ntx) * TX;
  const size_t fstride = (size_t)N * N * M;
  const int ky = kof(iy, N);
  const int tid = threadIdx.x, line = tid % TX, j = tid / TX, kx = x0 + line;
  const bool act = tid < NT;
  const size_t gj = ((size_t)j * N + iy) * M + kx;  // element (kz index j, iy, kx) of a field
  constexpr size_t ZS = (size_t)N * M;              // one plane
  // the state is loaded first, in one piece, where registers hold it beside the transforms' values
  constexpr bool EARLY = C::FEW && f * sizeof(cpx<T>) <= 64 && NFC == 1 && MC != MODE_NL && MC != MODE_PROJECT;
  const bool tt = pencil_tile_truncated<T, TX>(a, x0, ky);  // N = 0 on the whole tile
  // the state vanishes there too: nothing to do (NL and PROJECT write their zeros)
  if (tt && a.cut && mode != MODE_NL && mode != MODE_PROJECT &&
      !column_kept(a.trunc, a.K2max, a.Kimax, a.cutK, x0, ky) && *a.cut) {
    if constexpr (EP || NOC == 2)
      if ((EP || a.epart) && tid == 0) a.epart[2 * blockIdx.x] = a.epart[2 * blockIdx.x + 1] = 0.0;
    return;
  }
  const int nFe = tt ? 0 : nF;                              // inputs that are transformed
  // the twiddle table, on its way while the first inputs are loaded
  constexpr int KT = (N + NT - 1) / NT;
  cpx<T> twr[KT];
#pragma unroll
  for (int c = 0; c < KT; ++c) twr[c] = act && tid + c * NT < N ? ldg(&a.tw[tid + c * NT]) : mk<T>(0, 0);
  auto put_tw = [&] {
#pragma unroll
    for (int c = 0; c < KT; ++c)
      if (act && tid + c * NT < N) tws[tw_pad(tid + c * NT)] = twr[c];
  };

  const bool rd0 = mode != MODE_NL && mode != MODE_PROJECT;
  const cpx<T>* base0 = (mode == MODE_INIT ? a.src : (mode == MODE_RK4_4 ? a.acc : a.state)) + gj;
  cpx<T> s0e[3][f];
  if constexpr (EARLY)
    if (act)
#pragma unroll
      for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int r = 0; r < f; ++r) s0e[c][r] = MP::ldw(base0 + c * fstride + r * NB0 * ZS);

  // 1) forward z transforms of the inputs: de-shifted by e^{-i k.delta} and weighted (products in
  //    one fixed rounding order, as the compiler may contract them differently in each instance)
  cpx<T> v[3][f];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int r = 0; r < f; ++r) v[c][r] = mk<T>(0, 0);
  if constexpr (NFC != 0) {
    for (int q = 0; q < nFe; ++q) {
      if (act) {
        cpx<T> u[3][f];
        const cpx<T>* src = a.F[q] + gj;
        if (a.pairs) {
          const cpair<T>* src01 = reinterpret_cast<const cpair<T>*>(a.F[q]) + gj;
#pragma unroll
          for (int r = 0; r < f; ++r) MP::ldp(src01 + r * NB0 * ZS, u[0][r], u[1][r]);
        } else {
#pragma unroll
          for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int r = 0; r < f; ++r) u[c][r] = MP::ld(src + c * fstride + r * NB0 * ZS);
        }
#pragma unroll
        for (int r = 0; r < f; ++r) u[2][r] = MP::ld(src + 2 * fstride + r * NB0 * ZS);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          DFT<T, f>::run(u[c], T(-1));
          const int o = c * TS + X::at(line, j * f);
#pragma unroll
          for (int r = 0; r < f; ++r) buf[o + r * TX] = u[c][r];
        }
      }
      if (q == 0) put_tw();
      __syncthreads();
      mid_stages<T, N, PL, 1, FUSE ? nst - 1 : nst, -1, X, TX, 3, NT, true>(buf, TS, tws);
      if (act) {
        const cpx<T>* sh = a.dsh[q];
        cpx<T> cxy = mk<T>(1, 0);
        if (sh) cxy = cmul_fixed(MP::ld(&sh[kx]), MP::ld(&sh[N + iy]));
        auto take = [&](int c, int r, cpx<T> t, cpx<T> s) {  // element j + NB0 r of component c
          if (sh) t = mul_conj_fixed(t, s);
          if constexpr (NFC == 2) {
            if (q == 0) v[c][r] = t;
            else v[c][r] = mk<T>(fma1(a.wF[0], v[c][r].x, a.wF[1] * t.x), fma1(a.wF[0], v[c][r].y, a.wF[1] * t.y));
          } else {
            v[c][r] = a.wF[q] * t;
          }
        };
        if constexpr (FUSE) {
#pragma unroll
          for (int i = 0; i < K; ++i) {
            const int p = j + NB0 * i;
            cpx<T> w[l], s[l];
            reg_twiddles<T, N, l, NBL, -1>(w, tws, p);
            if (sh)
#pragma unroll
              for (int r = 0; r < l; ++r) s[r] = cmul_fixed(cxy, MP::ld(&sh[2 * N + p + r * NBL]));
#pragma unroll
            for (int c = 0; c < 3; ++c) {
              cpx<T> t[l];
              const int o = c * TS + X::at(line, p);
#pragma unroll
              for (int r = 0; r < l; ++r) t[r] = buf[o + r * X::step(NBL)];
              twiddle_dft<T, l>(t, w, T(-1));
#pragma unroll
              for (int r = 0; r < l; ++r) take(c, i + K * r, t[r], s[r]);
            }
          }
        } else {
#pragma unroll
          for (int r = 0; r < f; ++r) {
            cpx<T> s = cxy;
            if (sh) s = cmul_fixed(cxy, MP::ld(&sh[2 * N + j + r * NB0]));
            const int o = X::at(line, j + r * NB0);
#pragma unroll
            for (int c = 0; c < 3; ++c) take(c, r, buf[c * TS + o], s);
          }
        }
      }
      __syncthreads();
    }
  }
  if (nFe == 0) put_tw();  // (its first reader is past the barrier of the first output batch)

  // 2) spectral stage: every mode's N(0) = 0, truncation, projection and forcing, then the RK
  //    stage combine; v becomes S_next, shifted for the output when there is one
  const bool pre = nOut == 1 && a.osh[0] != nullptr;
  const bool ep = EP || (NOC == 2 && a.epart != nullptr);  // the same for the whole block
  T eacc = 0, dacc = 0;  // energy sums of the written state
  bool nz = false;
  if (act) {
    cpx<T> oxy = mk<T>(1, 0);
    if (pre) oxy = cmul_fixed(MP::ld(&a.osh[0][kx]), MP::ld(&a.osh[0][N + iy]));
    const bool useE = mode != MODE_INIT && mode != MODE_NL && mode != MODE_PROJECT;
    T e1xy = 1, ehxy = 1;
    if (useE) {
      e1xy = a.ifac[kx] * a.ifac[iy];
      ehxy = a.ifac[N + kx] * a.ifac[N + iy];
    }
    const bool rd1 = mode == MODE_RK4_2 || mode == MODE_RK4_3;
    // modes whose loads are in flight together (the stores of a chunk hold back the next one's)
    constexpr int CHK = EARLY ? f : f % 4 == 0 ? 4 : (f % 3 == 0 ? 3 : 2);
#pragma unroll
    for (int r0 = 0; r0 < f; r0 += CHK) {
      cpx<T> s0[3][CHK], s1[3][CHK];
#pragma unroll
      for (int i = 0; i < CHK; ++i)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          s0[c][i] = s1[c][i] = mk<T>(0, 0);
          if constexpr (EARLY) s0[c][i] = s0e[c][r0 + i];
          else if (rd0) s0[c][i] = MP::ldw(base0 + c * fstride + (r0 + i) * NB0 * ZS);
          if (rd1) s1[c][i] = MP::ldw(&a.acc[c * fstride + gj + (r0 + i) * NB0 * ZS]);
        }
      T e1z[CHK], ehz[CHK];
      cpx<T> oz[CHK];
#pragma unroll
      for (int i = 0; i < CHK; ++i) {
        const int iz = j + (r0 + i) * NB0;
        e1z[i] = ehz[i] = 1;
        if (useE) {
          e1z[i] = a.ifac[iz];
          ehz[i] = a.ifac[N + iz];
        }
        oz[i] = mk<T>(1, 0);
        if (pre) oz[i] = MP::ld(&a.osh[0][2 * N + iz]);
      }
#pragma unroll
      for (int i = 0; i < CHK; ++i) {
        const int r = r0 + i, iz = j + r * NB0, kz = kof(iz, N);
        const size_t g = gj + r * NB0 * ZS;
        cpx<T> nv[3] = {v[0][r], v[1][r], v[2][r]};
        if (nFe > 0) project_point(a, kx, ky, kz, nv);
        T E1 = 1, Eh = 1;
        if (useE) {
          E1 = e1xy * e1z[i];
          Eh = ehxy * ehz[i];
        }
        cpx<T> shz = oxy;
        if (pre) shz = cmul_fixed(oxy, oz[i]);
        T m2 = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          cpx<T> sn = stage_combine<T, MP>(a, c, c * fstride + g, nv[c], s0[c][i], s1[c][i], E1, Eh, mode);
          shell_record<T, MP>(a, c, kx, ky, kz, sn);
          if (ep) m2 += sn.x * sn.x + sn.y * sn.y;
          nz = nz || sn.x != T(0) || sn.y != T(0);
          v[c][r] = pre ? cmul_fixed(sn, shz) : sn;
        }
        if (ep) {
          const T wm = (kx == 0 ? T(1) : T(2)) * m2;
          if constexpr (ED == NB0) {
            eacc += wm;
            dacc += wm * (T)(kx * kx + ky * ky + kz * kz);
          } else {
            // the tiles are free here, until the barriers that follow the sums
            reinterpret_cast<T*>(buf)[iz * TX + line] = wm;
          }
        }
      }
    }
  }
  if constexpr (EP || NOC == 2) {
    if (ep) {
      if constexpr (ED != NB0) {
        __syncthreads();
        for (int i = tid; i < TX * ED; i += blockDim.x) {
          T e = 0, d = 0;
          for (int iz = i / TX; iz < N; iz += ED) {
            const int kz = kof(iz, N), k1 = x0 + i % TX;
            const T wm = reinterpret_cast<const T*>(buf)[iz * TX + i % TX];
            e += wm;
            d += wm * (T)(k1 * k1 + ky * ky + kz * kz);
          }
          eacc += e;
          dacc += d;
        }
      }
      tile_energy_store<T>(a.epart, eacc, dacc);
      if constexpr (ED != NB0) __syncthreads();
    }
  }
  if (tt) {  // S_next vanishing on the whole tile (a truncated state): zero outputs, no transforms
    if (!__syncthreads_or(nz)) {
      pencil_zero_outputs<T, N, TX, NT, MP>(a, nOut, iy, x0);
      return;
    }
  }

  // 3) inverse z transforms of S_next and of i kz S_next (x and y components) per output
  if constexpr (NOC != 0) {
    for (int o = 0; o < nOut; ++o) {
      cpx<T> oxy = mk<T>(1, 0);
      const cpx<T>* sh = pre ? nullptr : a.osh[o];
      if (sh && act) oxy = cmul_fixed(MP::ld(&sh[kx]), MP::ld(&sh[N + iy]));
      // `cnt` fields f0 .. through the tiles: first stage of each from the registers, then the rest
      auto batch = [&](auto f0c, auto cntc) {
        constexpr int f0 = decltype(f0c)::v, cnt = decltype(cntc)::v;
        if (act) {
#pragma unroll
          for (int q = 0; q < cnt; ++q) {
            cpx<T> t[f];
#pragma unroll
            for (int r = 0; r < f; ++r) {
              t[r] = v[f0 + q < 3 ? f0 + q : f0 + q - 3][r];
              if (NOC == 2 && sh) t[r] = cmul_fixed(t[r], cmul_fixed(oxy, MP::ld(&sh[2 * N + j + r * NB0])));
              if (f0 >= 3) t[r] = mul_si(t[r], (T)kof(j + r * NB0, N));
            }
            DFT<T, f>::run(t, T(1));
            const int i = q * TS + X::at(line, j * f);
#pragma unroll
            for (int r = 0; r < f; ++r) buf[i + r * TX] = t[r];
          }
        }
        __syncthreads();
        mid_stages<T, N, PL, 1, nst - 1, 1, X, TX, cnt, NT, true>(buf, TS, tws);
#pragma unroll
        for (int i = 0; i < K; ++i) {
          const int p = j + NB0 * i;  // last-stage butterfly
          if (!act || (!FUSE && p >= NBL)) break;
          cpx<T> w[l], t[2][l];
          reg_twiddles<T, N, l, NBL, 1>(w, tws, p);
          auto last = [&](cpx<T>* u, int q) {
            const int o = q * TS + X::at(line, p);
#pragma unroll
            for (int r = 0; r < l; ++r) u[r] = buf[o + r * X::step(NBL)];
            twiddle_dft<T, l>(u, w, T(1));
          };
          const size_t g = ((size_t)p * N + iy) * M + kx;
          last(t[0], 0);
          last(t[1], 1);
          if (a.pairs) {
            cpair<T>* dst = reinterpret_cast<cpair<T>*>(a.out[o] + f0 * fstride) + g;
#pragma unroll
            for (int r = 0; r < l; ++r) MP::stp(dst + r * NBL * ZS, t[0][r], t[1][r]);
          } else {
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
              for (int r = 0; r < l; ++r) MP::st(a.out[o] + (f0 + q) * fstride + g + r * NBL * ZS, t[q][r]);
          }
          if (cnt == 3) {
            last(t[0], 2);
#pragma unroll
            for (int r = 0; r < l; ++r) MP::st(a.out[o] + 2 * fstride + g + r * NBL * ZS, t[0][r]);
          }
        }
        __syncthreads();
      };
      batch(IntC<0>{}, IntC<3>{});
      batch(IntC<3>{}, IntC<2>{});
    }
  }
}

// EP: the one-input variant that also stores the tile's energy sums (a.epart non-null)
// MC: the stage mode; V: tile variant
template <typename T, int N, int NFC, int NOC, bool EP, int MC, int V = 0>
__global__ void __launch_bounds__(K2Cfg<T, N, V>::NTP, NFC == 2 ? K2Cfg<T, N, V>::MINB_P2 : K2Cfg<T, N, V>::MINB_P)
    k2_pencil(PencilArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pencil_tile<T, N, MemNC, NFC, NOC, EP, MC, V>(a, blockIdx.x, reinterpret_cast<cpx<T>*>(smem_raw));
}

// ---- slab pass: y transforms --------------------------------------------------------
// Scratch of the slab pass (SlabArgs::scr), per plane group: three arrays [plane][y][kx] of
// pairs of modes, (u_x, u_y), (u_z, omega_x), (omega_y, omega_z), the pairs that share a line of
// the x rows, so the x rows load and store 16 bytes (FP32) per mode.  The x rows leave the
// products (f_0, f_1) in the first array and f_2 in the first half of each row of the second.
// One tile: W consecutive kx of plane zg.  Inverse y transforms of u and omega = i k x u, formed
// in registers from the mixed fields (u_x, u_y, u_z, d_z u_x, d_z u_y; interleaved layout).
// Bound by HBM (5 fields read, 6 written).  The first stage reads global memory and the last
// one writes it, so each line passes through shared memory once per middle stage and once
// between them; two batches of three lines share three tiles and one set of twiddles.  Measured,
// 128 planes, FP32: 256^3 59.6 us = 6.2 TB/s (68.7 with the inputs staged in shared memory), 512^3
// 279 (380), 384^3 145 (181).
template <typename T, int N, class MP, int W>
__device__ __forceinline__ void yinv_tile(const SlabArgs<T>& a, int tx, int zg, cpx<T>* buf) {
  using PL = YPlan<T, N>;
  constexpr int M = N / 2, nst = PL::P.nst, f = PL::P.r[0], l = PL::P.r[nst - 1], NB0 = N / f, NBL = N / l;
  constexpr int NT = W * NB0, K = (f + l - 1) / l;  // K last-stage butterflies p = j + NB0 i per thread
  using X = Xchg<T, N, f, W, true>;
  constexpr int TS = X::elems;
  cpx<T>* tws = buf + 3 * TS;
  const int tid = threadIdx.x, line = tid % W, j = tid / W;
  const int x0 = tx * W, kx = x0 + line, z = a.z0 + zg;
  const size_t fs = (size_t)N * N * M;
  const bool act = tid < NT;
  const T fx = (T)kx;
  auto ky = [&](int r) { return (T)kof(j + r * NB0, N); };
  auto stage0 = [&](cpx<T>* v, int t) {  // radix-f butterfly into tile t
    DFT<T, f>::run(v, T(1));
    const int o = t * TS + X::at(line, j * f);
#pragma unroll
    for (int r = 0; r < f; ++r) buf[o + r * W] = v[r];
  };
  const size_t sstride = (size_t)a.G * N * M;
  cpair<T>* dst = reinterpret_cast<cpair<T>*>(a.scr) + (size_t)zg * N * M + kx;
  // columns that are not kept are zero, and unwritten, when *a.cut; the flag is waited for only
  // after the loads of the kept ones are on their way
  const bool cutp = a.cut != nullptr;
  const int cutv = cutp ? *a.cut : 0;
  if (cutp && x0 >= a.kxn && cutv) return;
  unsigned km = 0;  // bit r: mode (kx, j + r NB0) is in a kept column
#pragma unroll
  for (int r = 0; r < f; ++r)
    km |= (unsigned)(!cutp || column_kept(a.trunc, a.K2max, a.Kimax, a.fK, kx, kof(j + r * NB0, N))) << r;
  constexpr unsigned KALL = (1u << f) - 1;
  auto load = [&](auto&& get) {  // get(r): loads mode r of the thread
#pragma unroll
    for (int r = 0; r < f; ++r)
      if (km >> r & 1) get(r);
    if (km != KALL && !cutv) {
#pragma unroll
      for (int r = 0; r < f; ++r)
        if (!(km >> r & 1)) get(r);
    }
  };
  auto load2 = [&](cpx<T>* va, cpx<T>* vb, int c) {  // two interleaved fields
    const cpair<T>* p = reinterpret_cast<const cpair<T>*>(a.mixed + c * fs) + ((size_t)z * N + j) * M + kx;
#pragma unroll
    for (int r = 0; r < f; ++r) va[r] = vb[r] = mk<T>(0, 0);
    load([&](int r) { MP::ldp(p + (size_t)r * NB0 * M, va[r], vb[r]); });
  };
  // last stage of the lines in the tiles: pair `pr` from tiles 0 and 1, and tile 2 into wz (pr = 0)
  // or, with wz, pair 2 (pr = 1)
  cpx<T> wz[K][l];
  auto last = [&](int pr) {
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const int p = j + NB0 * i;
      if (!act || (f % l != 0 && p >= NBL)) break;
      cpx<T> w[l], va[l], vb[l];
      reg_twiddles<T, N, l, NBL, 1>(w, tws, p);
      auto line_of = [&](cpx<T>* v, int t) {
        const int o = t * TS + X::at(line, p);
#pragma unroll
        for (int r = 0; r < l; ++r) v[r] = buf[o + r * X::step(NBL)];
        twiddle_dft<T, l>(v, w, T(1));
      };
      line_of(va, 0);
      line_of(vb, 1);
      cpair<T>* d = dst + pr * sstride + (size_t)p * M;
#pragma unroll
      for (int r = 0; r < l; ++r) MP::stp(d + (size_t)r * NBL * M, va[r], vb[r]);
      if (pr == 0) {
        line_of(wz[i], 2);
      } else {
        line_of(va, 2);
#pragma unroll
        for (int r = 0; r < l; ++r) MP::stp(d + sstride + (size_t)r * NBL * M, va[r], wz[i][r]);
      }
    }
  };

  cpx<T> ux[f], uy[f];
  if (act) load2(ux, uy, 0);
  for (int i = tid; i < N; i += blockDim.x) tws[tw_pad(i)] = ldg(&a.tw[i]);
  if (act) {
    cpx<T> v[f];
#pragma unroll
    for (int r = 0; r < f; ++r) v[r] = mul_si(uy[r], fx) - mul_si(ux[r], ky(r));  // i kx u_y - i ky u_x
    stage0(ux, 0);
    stage0(uy, 1);
    stage0(v, 2);
  }
  __syncthreads();
  mid_stages<T, N, PL, 1, nst - 1, 1, X, W, 3, NT, true>(buf, TS, tws);
  cpx<T> uz[f], dx[f], dy[f];
  if (act) {
    const cpx<T>* src = a.mixed + 2 * fs + ((size_t)z * N + j) * M + kx;
#pragma unroll
    for (int r = 0; r < f; ++r) uz[r] = mk<T>(0, 0);
    load([&](int r) { uz[r] = MP::ld(src + (size_t)r * NB0 * M); });
    load2(dx, dy, 3);
  }
  last(0);
  __syncthreads();
  if (act) {
#pragma unroll
    for (int r = 0; r < f; ++r) {
      const T k = ky(r);
      dy[r] = mk<T>(fma1(-k, uz[r].y, -dy[r].x), fma1(k, uz[r].x, -dy[r].y));  // i ky u_z - d_z u_y
      dx[r] = mk<T>(fma1(fx, uz[r].y, dx[r].x), fma1(-fx, uz[r].x, dx[r].y));  // d_z u_x - i kx u_z
    }
    stage0(uz, 0);
    stage0(dy, 1);
    stage0(dx, 2);
  }
  __syncthreads();
  mid_stages<T, N, PL, 1, nst - 1, 1, X, W, 3, NT, true>(buf, TS, tws);
  last(1);
}

template <typename T, int N, int V = 0>
__global__ void __launch_bounds__(K2Cfg<T, N, V>::NTYI, K2Cfg<T, N, V>::MINB_YI) k2_yinv(SlabArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  yinv_tile<T, N, MemNC, K2Cfg<T, N, V>::TYI>(a, blockIdx.x, blockIdx.y, reinterpret_cast<cpx<T>*>(smem_raw));
}

// One tile: W consecutive kx of plane zg.  Forward y transforms of the three products, the
// first stage from the scratch, the last one into Ft, where a mode is stored unless its column
// is outside the truncation (a.skip: no pencil pass uses it).  Bound by HBM.
template <typename T, int N, class MP, int W>
__device__ __forceinline__ void yfwd_tile(const SlabArgs<T>& a, int tx, int zg, cpx<T>* buf) {
  using PL = YPlan<T, N>;
  constexpr int M = N / 2, nst = PL::P.nst, f = PL::P.r[0], l = PL::P.r[nst - 1], NB0 = N / f, NBL = N / l;
  constexpr int NT = W * NB0, K = (f + l - 1) / l;
  using X = Xchg<T, N, f, W, true>;
  constexpr int TS = X::elems;
  cpx<T>* tws = buf + 3 * TS;
  const int tid = threadIdx.x, line = tid % W, j = tid / W;
  const int x0 = tx * W, kx = x0 + line, z = a.z0 + zg;
  const size_t sstride = (size_t)a.G * N * M, fs = (size_t)N * N * M;
  const bool act = tid < NT;
  if (a.skip && x0 >= a.kxn) return;  // no column of the tile is kept
  if (act) {
    cpx<T> v[3][f];
    const cpair<T>* src = reinterpret_cast<const cpair<T>*>(a.scr) + ((size_t)zg * N + j) * M + kx;
    const cpx<T>* src2 = reinterpret_cast<const cpx<T>*>(reinterpret_cast<const cpair<T>*>(a.scr) + sstride) +
                         ((size_t)zg * N + j) * 2 * M + kx;
#pragma unroll
    for (int r = 0; r < f; ++r) {
      MP::ldp(src + (size_t)r * NB0 * M, v[0][r], v[1][r]);
      v[2][r] = MP::ldw(src2 + (size_t)r * NB0 * 2 * M);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      DFT<T, f>::run(v[c], T(-1));
      const int o = c * TS + X::at(line, j * f);
#pragma unroll
      for (int r = 0; r < f; ++r) buf[o + r * W] = v[c][r];
    }
  }
  for (int i = tid; i < N; i += blockDim.x) tws[tw_pad(i)] = ldg(&a.tw[i]);
  __syncthreads();
  mid_stages<T, N, PL, 1, nst - 1, -1, X, W, 3, NT, true>(buf, TS, tws);
#pragma unroll
  for (int i = 0; i < K; ++i) {
    const int p = j + NB0 * i;  // last-stage butterfly
    if (!act || (f % l != 0 && p >= NBL)) break;
    cpx<T> w[l], v[2][l];
    reg_twiddles<T, N, l, NBL, -1>(w, tws, p);
    bool keep[l];
#pragma unroll
    for (int r = 0; r < l; ++r) keep[r] = !a.skip || column_kept(a.trunc, a.K2max, a.Kimax, a.fK, kx, kof(p + r * NBL, N));
    const size_t g = ((size_t)z * N + p) * M + kx;
    auto last = [&](cpx<T>* u, int c) {
      const int o = c * TS + X::at(line, p);
#pragma unroll
      for (int r = 0; r < l; ++r) u[r] = buf[o + r * X::step(NBL)];
      twiddle_dft<T, l>(u, w, T(-1));
    };
    last(v[0], 0);
    last(v[1], 1);
    cpair<T>* dst = reinterpret_cast<cpair<T>*>(a.Ft) + g;
#pragma unroll
    for (int r = 0; r < l; ++r)
      if (keep[r]) MP::stp(dst + (size_t)r * NBL * M, v[0][r], v[1][r]);
    last(v[0], 2);
#pragma unroll
    for (int r = 0; r < l; ++r)
      if (keep[r]) MP::st(a.Ft + 2 * fs + g + (size_t)r * NBL * M, v[0][r]);
  }
}

template <typename T, int N, int V = 0>
__global__ void __launch_bounds__(K2Cfg<T, N, V>::NTY, K2Cfg<T, N, V>::MINB_Y) k2_yfwd(SlabArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  yfwd_tile<T, N, MemNC, K2Cfg<T, N, V>::TY>(a, blockIdx.x, blockIdx.y, reinterpret_cast<cpx<T>*>(smem_raw));
}

// ---- slab pass: x rows --------------------------------------------------------------
// One tile: RX consecutive rows (plane, y) of the group.  Each row holds the half spectra
// (kx < N/2, the Nyquist mode zero) of 6 real fields, and two real rows share one complex line
// of length N: the line of fields a and b is z = a + i b, whose full spectrum is
// Z[k] = A[k] + i B[k] and Z[N - k] = conj(A[k]) + i conj(B[k]) (A[0], B[0] real).  Inverse
// lines per row: (u_x, u_y), (u_z, w_x), (w_y, w_z); the products come back as lines (f_0, f_1)
// of every row and (f_2 of row q, f_2 of row q + RXH), whose forward transforms P split into
// F_a[k] = (P[k] + conj(P[N - k])) / 2 and F_b[k] = (P[k] - conj(P[N - k])) / (2 i).  All
// transforms are unnormalised, as the r2c / c2r pair they replace.
//
// What bounds it: shared memory, when every stage goes through it (27 accesses per line element
// in six passes).  Here a thread takes the two first-stage butterflies j and N/f - j together:
// their inputs are closed under k -> N - k, so the lines are formed from the modes in registers;
// the last inverse butterflies, the products and the first forward butterfly of the points
// x = j + (N/f) r share registers (see radix plans); and the pair (p, N/l - p) of the last forward
// stage holds P[k] and P[N - k], which it splits and stores.  Shared memory sees each line once
// per transform and middle stage.  The two rows of a pair sit in neighbouring lanes, and the even
// lane takes the partner's third products.  One thread per row and N/f points; where a pair's
// threads fit a warp, the warps do not wait for one another.  Measured on GB300, 128 planes, FP32:
// 256^3 71.0 us (86.3 with every stage through shared memory), 512^3 293 (418), 384^3 195 (270),
// 128^3 18.6 (22.6).  156 registers and 12 warps per SM beat 124 and 16 (71 against 80 us): the
// loads in flight per thread hide more than further warps do.
template <typename T, int N, class MP, int V = 0>
__device__ __forceinline__ void xrow_tile(const SlabArgs<T>& a, int tile_id, cpx<T>* smem) {
  using C = K2Cfg<T, N, V>;
  using PL = XPlan<T, N>;
  constexpr int nst = PL::P.nst, f = PL::P.r[0], l = PL::P.r[nst - 1];  // outer and inner radix
  constexpr int M = N / 2, NB0 = N / f, NBL = N / l, H = f / 2, IP0 = (NB0 + 1) / 2, IPL = NBL / 2;
  constexpr bool ODD0 = NB0 % 2;  // (then j = 0 has no second self-mirrored butterfly)
  constexpr bool FUSE = f % l == 0;
  constexpr int K = f / l;                                      // last-stage butterflies per thread (FUSE)
  constexpr int NP = C::XWP, NT = C::XGT, ROWS = 2 * NP;         // pairs, threads and rows of a group
  constexpr int NLI = 3 * ROWS, NLF = ROWS + NP;                 // its inverse and forward lines
  using X = Xchg<T, N, f, NLI, false>;
  static_assert(f % 2 == 0 && NBL % 2 == 0, "modes k and N - k pair up");
  cpx<T>* tws = smem + C::XELEMS;
  // the twiddle table, on its way while the modes are loaded
  constexpr int KT = (N + C::NTX - 1) / C::NTX;
  cpx<T> twr[KT];
#pragma unroll
  for (int c = 0; c < KT; ++c) {
    const int i = threadIdx.x + c * C::NTX;
    twr[c] = (int)threadIdx.x < C::NTX && i < N ? ldg(&a.tw[i]) : mk<T>(0, 0);
  }
  const int grp = C::XWARP ? threadIdx.x / NT : 0, tid = C::XWARP ? threadIdx.x % NT : threadIdx.x;
  const bool in = C::XWARP ? grp < C::XNG : true;  // (a wider block's other warps only pass barriers)
  cpx<T>* buf = smem + (in ? grp : 0) * C::XGEL;
  auto sync = [] {
    if constexpr (C::XWARP) __syncwarp();
    else __syncthreads();
  };
  // local row 2 q + h is row grp NP + q + h RXH of the tile (the last pair of an odd tile has one)
  const int r0 = tile_id * C::RX, nr = in ? min(C::RX, a.G * N - r0) : 0;
  auto row_of = [&](int lr) {
    const int row = grp * NP + (lr >> 1) + (lr & 1) * C::RXH;
    return row < nr && (lr & 1 ? row < C::RX : row < C::RXH) ? row : -1;
  };
  const size_t sstride = (size_t)a.G * N * M;

  // modes kx >= kxn are zero, and unwritten, when *a.cut
  const bool cutp = a.cut != nullptr && a.kxn < M;
  const int cutv = cutp ? *a.cut : 0, kxl = cutp ? a.kxn : M, kxs = a.skip ? a.kxn : M;

  // 1) item (line p ROWS + row, pair h): the modes of both butterflies, their radix-f transforms
  for (int i = tid; i < NLI * IP0 && tid < NT && in; i += NT) {
    const int line = i / IP0, h = i % IP0, p = line / ROWS, row = row_of(line % ROWS);
    const int j0 = h, j1 = h == 0 ? (ODD0 ? 0 : NB0 / 2) : NB0 - h;
    cpx<T> v0[f], v1[f], m0[H], m1[H], b0[H], b1[H];
    const cpair<T>* src = reinterpret_cast<const cpair<T>*>(a.scr) + p * sstride + (size_t)(r0 + row) * M;
#pragma unroll
    for (int r = 0; r < H; ++r) {
      v0[r] = v1[r] = b0[r] = b1[r] = mk<T>(0, 0);
      if (row >= 0) {
        if (j0 + r * NB0 < kxl) MP::ldp(src + j0 + r * NB0, v0[r], b0[r]);
        if (j1 + r * NB0 < kxl) MP::ldp(src + j1 + r * NB0, v1[r], b1[r]);
      }
    }
    if (kxl < M && !cutv && row >= 0) {
#pragma unroll
      for (int r = 0; r < H; ++r) {
        if (j0 + r * NB0 >= kxl) MP::ldp(src + j0 + r * NB0, v0[r], b0[r]);
        if (j1 + r * NB0 >= kxl) MP::ldp(src + j1 + r * NB0, v1[r], b1[r]);
      }
    }
#pragma unroll
    for (int r = 0; r < H; ++r) {
      const cpx<T> A = v0[r], B = b0[r], D = v1[r], E = b1[r];
      v0[r] = mk<T>(A.x - B.y, A.y + B.x);  // A + i B
      m0[r] = mk<T>(A.x + B.y, B.x - A.y);  // conj(A) + i conj(B)
      if (r == 0 && h == 0) v0[0] = mk<T>(A.x, B.x);
      v1[r] = mk<T>(D.x - E.y, D.y + E.x);
      m1[r] = mk<T>(D.x + E.y, E.x - D.y);
    }
#pragma unroll
    for (int r = 0; r < H; ++r) {  // the mirrored halves: from each other, or (h = 0) from themselves
      const cpx<T> s = r == 0 ? mk<T>(0, 0) : m0[H - r];
      v0[H + r] = h == 0 ? s : m1[H - 1 - r];
      v1[H + r] = h == 0 ? m1[H - 1 - r] : m0[H - 1 - r];
    }
    DFT<T, f>::run(v0, T(1));
    const int o0 = X::at(line, j0 * f);
#pragma unroll
    for (int r = 0; r < f; ++r) buf[o0 + r] = v0[r];
    if (!ODD0 || h > 0) {
      DFT<T, f>::run(v1, T(1));
      const int o1 = X::at(line, j1 * f);
#pragma unroll
      for (int r = 0; r < f; ++r) buf[o1 + r] = v1[r];
    }
  }
#pragma unroll
  for (int c = 0; c < KT; ++c) {
    const int i = threadIdx.x + c * C::NTX;
    if ((int)threadIdx.x < C::NTX && i < N) tws[tw_pad(i)] = twr[c];
  }
  __syncthreads();
  mid_stages<T, N, PL, 1, FUSE ? nst - 1 : nst, 1, X, NLI, 1, NT, false>(buf, 0, tws);

  // 2) item (row 2 q + h, points x = j + NB0 r): last inverse stage of the row's 3 lines, the
  //    products, first forward stage of (f_0, f_1) and (even lane) of the pair's f_2 line
  const bool act = in && tid < ROWS * NB0;  // (the other lanes of its last warp repeat its last pair)
  const int it = act ? tid : ROWS * NB0 - 2 + (tid & 1);
  const int h = it & 1, j = (it >> 1) % NB0, q = (it >> 1) / NB0, lr = 2 * q + h;
  T um[3] = {T(0), T(0), T(0)};  // max |u_i| over the rows (CFL), padding rows are zero
  cpx<T> g[f], y[f];
  if (in && tid < (ROWS * NB0 + 31) / 32 * 32) {
    cpx<T> z0[f], z1[f], z2[f];
    if constexpr (FUSE) {
#pragma unroll
      for (int i = 0; i < K; ++i) {
        const int p = j + NB0 * i;
        cpx<T> w[l];
        reg_twiddles<T, N, l, NBL, 1>(w, tws, p);
        const int o = X::at(lr, p);
        auto last = [&](cpx<T>* z, int line0) {
          cpx<T> t[l];
#pragma unroll
          for (int r = 0; r < l; ++r) t[r] = buf[o + line0 * X::LS + r * X::step(NBL)];
          twiddle_dft<T, l>(t, w, T(1));
#pragma unroll
          for (int r = 0; r < l; ++r) z[i + K * r] = t[r];
        };
        last(z0, 0);
        last(z1, ROWS);
        last(z2, 2 * ROWS);
      }
    } else {
#pragma unroll
      for (int r = 0; r < f; ++r) {
        const int o = X::at(lr, j + r * NB0);
        z0[r] = buf[o];
        z1[r] = buf[o + ROWS * X::LS];
        z2[r] = buf[o + 2 * ROWS * X::LS];
      }
    }
#pragma unroll
    for (int r = 0; r < f; ++r) {
      const T ux = z0[r].x, uy = z0[r].y, uz = z1[r].x, wx = z1[r].y, wy = z2[r].x, wz = z2[r].y;
      um[0] = fmax(um[0], fabs(ux));
      um[1] = fmax(um[1], fabs(uy));
      um[2] = fmax(um[2], fabs(uz));
      g[r] = mk<T>(fma1(uy, wz, -(uz * wy)), fma1(uz, wx, -(ux * wz)));
      const T f2 = fma1(ux, wy, -(uy * wx));
      y[r] = mk<T>(f2, __shfl_xor_sync(0xffffffffu, f2, 1));
    }
    DFT<T, f>::run(g, T(-1));
    if (h == 0) DFT<T, f>::run(y, T(-1));
  }
  sync();
  if (act) {
    const int o0 = X::at(lr, j * f), o1 = X::at(ROWS + q, j * f);
#pragma unroll
    for (int r = 0; r < f; ++r) buf[o0 + r] = g[r];
    if (h == 0)
#pragma unroll
      for (int r = 0; r < f; ++r) buf[o1 + r] = y[r];
  }
  sync();
  if (a.umax) block_max3<T>(um[0], um[1], um[2], reinterpret_cast<T*>(smem + C::XNG * C::XGEL), a.umax);
  mid_stages<T, N, PL, 1, nst - 1, -1, X, NLF, 1, NT, false>(buf, 0, tws);

  // 3) item (line, pair hh): last forward stage of both butterflies, split and stored
  for (int i = tid; i < NLF * IPL && tid < NT && in; i += NT) {
    const int line = i / IPL, hh = i % IPL;
    const int p0 = hh, p1 = hh == 0 ? NBL / 2 : NBL - hh;
    const bool own = line < ROWS;  // (f_0, f_1) of a row, else f_2 of a pair's rows
    const int ra = row_of(own ? line : 2 * (line - ROWS)), rb = own ? -1 : row_of(2 * (line - ROWS) + 1);
    cpx<T> v0[l], v1[l];
    {
      cpx<T> w[l];
      reg_twiddles<T, N, l, NBL, -1>(w, tws, p0);
      const int i0 = X::at(line, p0), i1 = X::at(line, p1);
#pragma unroll
      for (int r = 0; r < l; ++r) v0[r] = buf[i0 + r * X::step(NBL)];
      twiddle_dft<T, l>(v0, w, T(-1));
      reg_twiddles<T, N, l, NBL, -1>(w, tws, p1);
#pragma unroll
      for (int r = 0; r < l; ++r) v1[r] = buf[i1 + r * X::step(NBL)];
      twiddle_dft<T, l>(v1, w, T(-1));
    }
    cpair<T>* d01 = reinterpret_cast<cpair<T>*>(a.scr) + (size_t)r0 * M;
    cpx<T>* d2 = reinterpret_cast<cpx<T>*>(d01 + sstride);
    auto put = [&](int k, cpx<T> P, cpx<T> Q) {  // P = P[k], Q = P[N - k]
      if (k >= kxs) return;
      const cpx<T> A = mk<T>(T(0.5) * (P.x + Q.x), T(0.5) * (P.y - Q.y));
      const cpx<T> B = mk<T>(T(0.5) * (P.y + Q.y), T(0.5) * (Q.x - P.x));
      if (own) {
        if (ra >= 0) MP::stp(d01 + (size_t)ra * M + k, A, B);
      } else {
        if (ra >= 0) MP::st(d2 + (size_t)ra * 2 * M + k, A);
        if (rb >= 0) MP::st(d2 + (size_t)rb * 2 * M + k, B);
      }
    };
#pragma unroll
    for (int r = 0; r < (l + 1) / 2; ++r) {  // (elements r > l / 2 have k >= N / 2)
      put(p0 + r * NBL, v0[r], hh == 0 ? v0[(l - r) % l] : v1[l - 1 - r]);
      put(p1 + r * NBL, v1[r], hh == 0 ? v1[l - 1 - r] : v0[l - 1 - r]);
    }
  }
}

template <typename T, int N, int V = 0>
__global__ void __launch_bounds__(K2Cfg<T, N, V>::NTX, K2Cfg<T, N, V>::MINB_X) k2_xrow(SlabArgs<T> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  xrow_tile<T, N, MemNC, V>(a, blockIdx.x, reinterpret_cast<cpx<T>*>(smem_raw));
}

// ---- slab pipeline: the three slab kernels as one persistent launch -------------------
__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Control block of a pipeline launch (zeroed by the host before each launch).
struct PipeCtl {
  unsigned long long* next;  // ticket counter
  int* done;                 // [3][N]: finished y-inverse, x-row and y-forward tiles per plane
  int* abort;                // set when a wait gives up: every block leaves its loop
  long long spin_limit;      // polls before a wait gives up (then bit PIPE_ERR_TIMEOUT in err)
  int ring, lag;             // scratch planes in the ring; slots between the three stages
  int stall;                 // test hook: added to every awaited count (waits cannot succeed)
};
constexpr int PIPE_ERR_TIMEOUT = 0x100;
#ifndef NS_PIPE_MINB
#define NS_PIPE_MINB 3  // resident blocks per SM the register allocation must allow
#endif

// Work items of plane z: y-inverse tiles of 4 columns, x-row tiles of RX rows, y-forward
// tiles; tickets in slot order, slot s = [y-inverse(s), x rows(s - lag), y-forward(s - 2 lag)].
template <typename T, int N>
struct PipeCfg {
  using C = K2Cfg<T, N>;
  static constexpr int M = N / 2;
  static constexpr int TYP = 4;
  static constexpr int NTYP = TYP * C::YNB;
  static constexpr int nYI = M / TYP, nX = N / C::RX, nYF = M / C::TY;
  static constexpr int per_slot = nYI + nX + nYF;
  static constexpr int NT = (cmax(cmax(NTYP, C::NTX), C::NTY) + 31) / 32 * 32;
  static constexpr bool ok = N % C::RX == 0 && M % TYP == 0 && TYP % C::MINW == 0;
  static constexpr size_t smem = sizeof(cpx<T>) *
      cmax(cmax(C::y_elems(TYP), C::y_elems(C::TY)), C::XELEMS + tw_elems(N));
};

// One slab pass over all N planes with the scratch as a ring of `ring` planes: every item
// waits (bounded) for the items it reads: x rows(z) for y-inverse(z), y-forward(z) for
// x rows(z), y-inverse(z) for y-forward(z - ring) (the ring slot it overwrites).  Each waits on
// an earlier ticket, held by a running block, so the pipeline progresses whatever the number
// of resident blocks.  Data written in the launch is read through L2 (MemCG).
// the y-pass tile bodies as separate functions (the union of the three bodies in one
// allocation spilled); the x-row body stays inline
template <typename T, int N>
__device__ __noinline__ void pipe_yinv(const SlabArgs<T>& b, int tile, int zs, cpx<T>* smem) {
  yinv_tile<T, N, MemCG, PipeCfg<T, N>::TYP>(b, tile, zs, smem);
}
template <typename T, int N>
__device__ __noinline__ void pipe_yfwd(const SlabArgs<T>& b, int tile, int zs, cpx<T>* smem) {
  yfwd_tile<T, N, MemCG, K2Cfg<T, N>::TY>(b, tile, zs, smem);
}

template <typename T, int N>
__global__ void __launch_bounds__(PipeCfg<T, N>::NT, NS_PIPE_MINB)
    k2_slabpipe(SlabArgs<T> a, PipeCtl c) {
  using P = PipeCfg<T, N>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cpx<T>* smem = reinterpret_cast<cpx<T>*>(smem_raw);
  __shared__ long long s_t;
  __shared__ int s_go;
  const long long total = (long long)(N + 2 * c.lag) * P::per_slot;
  for (;;) {
    if (threadIdx.x == 0) s_t = (long long)atomicAdd(c.next, 1ull);
    __syncthreads();
    const long long tk = s_t;
    __syncthreads();
    if (tk >= total) break;
    const int slot = (int)(tk / P::per_slot), r = (int)(tk % P::per_slot);
    int type, z, tile;
    if (r < P::nYI) {
      type = 0; z = slot; tile = r;
    } else if (r < P::nYI + P::nX) {
      type = 1; z = slot - c.lag; tile = r - P::nYI;
    } else {
      type = 2; z = slot - 2 * c.lag; tile = r - P::nYI - P::nX;
    }
    if (z < 0 || z >= N) continue;
    const int wtype = type == 0 ? 2 : type - 1;
    const int wz = type == 0 ? z - c.ring : z;
    const int wcnt = (type == 0 ? P::nYF : type == 1 ? P::nYI : P::nX) + c.stall;
    if (threadIdx.x == 0) {
      int ok = 1;
      if (wz >= 0) {
        long long it = 0;
        while (ld_acquire(&c.done[wtype * N + wz]) < wcnt) {
          if (*(volatile int*)c.abort || ++it > c.spin_limit) {
            ok = 0;
            atomicOr(a.err, PIPE_ERR_TIMEOUT);
            atomicExch(c.abort, 1);
            break;
          }
          __nanosleep(64);
        }
      }
      s_go = ok;
    }
    __syncthreads();
    if (!s_go) break;
    const int zs = z % c.ring;
    SlabArgs<T> b = a;
    b.z0 = z - zs;
    if (type == 0)
      pipe_yinv<T, N>(b, tile, zs, smem);
    else if (type == 1)
      xrow_tile<T, N, MemCG>(b, zs * P::nX + tile, smem);  // inline: it needs every register
    else
      pipe_yfwd<T, N>(b, tile, zs, smem);
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      atomicAdd(&c.done[type * N + z], 1);
    }
  }
}

}  // namespace ns

#include "ns_slabcl.cuh"

namespace ns {

// ---- registry entry of one size ------------------------------------------------------
template <typename T>
struct K2Entry {
  int N = 0;
  void (*pencil01)(PencilArgs<T>) = nullptr; // no input, one output (INIT)
  void (*pencil10[2])(PencilArgs<T>) = {};   // one input, no output: NL, PROJECT
  void (*pencil1[MODE_ROG_2 + 1])(PencilArgs<T>) = {};  // one input, one output, by stage mode
  void (*pencil1e[MODE_ROG_2 + 1])(PencilArgs<T>) = {}; // same for the final stages, also storing the energy sums
  void (*pencil2[2])(PencilArgs<T>) = {};    // two inputs, two outputs: RK2_1, RK2_2
  void (*pencil02)(PencilArgs<T>) = nullptr; // no input, two outputs (INIT of the exact scheme)
  void (*yinv)(SlabArgs<T>) = nullptr;
  void (*yfwd)(SlabArgs<T>) = nullptr;
  void (*xrow)(SlabArgs<T>) = nullptr;
  void (*slabpipe)(SlabArgs<T>, PipeCtl) = nullptr;  // null when the size has no pipeline
  int NTPIPE = 0;
  size_t smPIPE = 0;
  // the slab pass in thread-block clusters of CLS CTAs (null when the size has none), two
  // thread counts: variant v has NTCL[v] threads
  void (*slabcl[2])(CUtensorMap, cpx<T>*, const cpx<T>*, ClArgs) = {nullptr, nullptr};
  int CLS = 0, NTCL[2] = {0, 0}, CLKC = 0, CLPL = 1;
  size_t smCL = 0;
  int TX = 0, NTP = 0, TY = 0, NTY = 0, TYI = 0, NTYI = 0, RX = 0, NTX = 0;
  size_t smP = 0, smY = 0, smYI = 0, smX = 0;
  // the autotuner's compiled alternatives (K2Cfg variant 15: every family's other width; the x
  // rows have none); has_alt false when the size has none
  struct Alt {
    void (*pencil1r[2])(PencilArgs<T>) = {nullptr, nullptr};
    void (*yinv)(SlabArgs<T>) = nullptr;
    void (*yfwd)(SlabArgs<T>) = nullptr;
    int TX = 0, NTP = 0, TY = 0, NTY = 0, TYI = 0, NTYI = 0;
    size_t smP = 0, smY = 0, smYI = 0;
  } alt;
  bool has_alt = false;
};

// sizes with compiled alternatives: the FP32 grids of 128^3 and larger
template <typename T, int N>
__host__ __device__ constexpr bool k2_has_alt() { return sizeof(T) == 4 && N >= 128; }

template <typename T, int N>
K2Entry<T> make_k2_entry() {
  constexpr int FV = N <= 64 ? 4 : 0;  // (a single grid: FEW)
  using C = K2Cfg<T, N, FV>;
  K2Entry<T> e;
  e.N = N;
  e.pencil01 = k2_pencil<T, N, 0, 1, false, MODE_INIT, FV>;
  e.pencil10[0] = k2_pencil<T, N, 1, 0, false, MODE_NL, FV>;
  e.pencil10[1] = k2_pencil<T, N, 1, 0, false, MODE_PROJECT, FV>;
  e.pencil1[MODE_RK2_1] = k2_pencil<T, N, 1, 1, false, MODE_RK2_1, FV>;
  e.pencil1[MODE_RK2_2] = k2_pencil<T, N, 1, 1, false, MODE_RK2_2, FV>;
  e.pencil1[MODE_RK4_1] = k2_pencil<T, N, 1, 1, false, MODE_RK4_1, FV>;
  e.pencil1[MODE_RK4_2] = k2_pencil<T, N, 1, 1, false, MODE_RK4_2, FV>;
  e.pencil1[MODE_RK4_3] = k2_pencil<T, N, 1, 1, false, MODE_RK4_3, FV>;
  e.pencil1[MODE_RK4_4] = k2_pencil<T, N, 1, 1, false, MODE_RK4_4, FV>;
  e.pencil1[MODE_ROG_1] = k2_pencil<T, N, 1, 1, false, MODE_ROG_1, FV>;
  e.pencil1[MODE_ROG_2] = k2_pencil<T, N, 1, 1, false, MODE_ROG_2, FV>;
  e.pencil1e[MODE_RK2_2] = k2_pencil<T, N, 1, 1, true, MODE_RK2_2, FV>;
  e.pencil1e[MODE_RK4_4] = k2_pencil<T, N, 1, 1, true, MODE_RK4_4, FV>;
  e.pencil1e[MODE_ROG_2] = k2_pencil<T, N, 1, 1, true, MODE_ROG_2, FV>;
  e.pencil2[0] = k2_pencil<T, N, 2, 2, false, MODE_RK2_1, FV>;
  e.pencil2[1] = k2_pencil<T, N, 2, 2, false, MODE_RK2_2, FV>;
  e.pencil02 = k2_pencil<T, N, 0, 2, false, MODE_INIT, FV>;
  e.yinv = k2_yinv<T, N, FV>;
  e.yfwd = k2_yfwd<T, N, FV>;
  e.xrow = k2_xrow<T, N, FV>;
  if constexpr (ClCfg<T, N>::ok) {
    e.slabcl[0] = k2_slabcl<T, N, 384>;
    e.slabcl[1] = k2_slabcl<T, N, 768>;
    e.NTCL[0] = 384;
    e.NTCL[1] = 768;
    e.CLS = ClCfg<T, N>::CS;
    e.CLKC = ClCfg<T, N>::KC;
    e.CLPL = ClCfg<T, N>::PL;
    e.smCL = ClCfg<T, N>::smem;
  }
  if constexpr (PipeCfg<T, N>::ok) {
    e.slabpipe = k2_slabpipe<T, N>;
    e.NTPIPE = PipeCfg<T, N>::NT;
    e.smPIPE = PipeCfg<T, N>::smem;
  }
  e.TX = C::TX; e.NTP = C::NTP; e.TY = C::TY; e.NTY = C::NTY; e.RX = C::RX; e.NTX = C::NTX;
  e.TYI = C::TYI; e.NTYI = C::NTYI;
  e.smYI = (size_t)C::y_elems(C::TYI) * sizeof(cpx<T>);
  e.smP = (size_t)C::p_elems * sizeof(cpx<T>);
  e.smY = (size_t)C::y_elems(C::TY) * sizeof(cpx<T>);
  e.smX = ((size_t)C::XELEMS + tw_elems(N)) * sizeof(cpx<T>);
  if constexpr (k2_has_alt<T, N>()) {
    using A = K2Cfg<T, N, 15>;
    e.has_alt = true;
    e.alt.pencil1r[0] = k2_pencil<T, N, 1, 1, false, MODE_ROG_1, 15>;
    e.alt.pencil1r[1] = k2_pencil<T, N, 1, 1, false, MODE_ROG_2, 15>;
    e.alt.yinv = k2_yinv<T, N, 15>;
    e.alt.yfwd = k2_yfwd<T, N, 15>;
    e.alt.TX = A::TX; e.alt.NTP = A::NTP; e.alt.TY = A::TY; e.alt.NTY = A::NTY;
    e.alt.TYI = A::TYI; e.alt.NTYI = A::NTYI;
    e.alt.smYI = (size_t)A::y_elems(A::TYI) * sizeof(cpx<T>);
    e.alt.smP = (size_t)A::p_elems * sizeof(cpx<T>);
    e.alt.smY = (size_t)A::y_elems(A::TY) * sizeof(cpx<T>);
  }
  return e;
}

}  // namespace ns
