// Finite-difference Runge-Kutta stage: 4th-order centred first derivatives and
// 6th-difference Kreiss-Oliger dissipation (paper Sec. I and Sec. IV: FD4
// with KO dissipation; KO normalisation sigma/(64 dx) is the r = 3 form):
//   L(Q) = -sum_d B_d(Q) dQ/dx_d + S(Q) + sigma/(64 dx) sum_d delta6_d Q
//   dQ/dx  = [(Q_-2 - Q_+2) + 8 (Q_+1 - Q_-1)] / (12 dx)
//   delta6 = Q_-3 - 6 Q_-2 + 15 Q_-1 - 20 Q_0 + 15 Q_+1 - 6 Q_+2 + Q_+3
//   out = a q0 + b qs + g dt L ; acc += d dt L
// Constant states stay bitwise constant (the weights of every stencil sum to zero, and equal
// terms cancel exactly).
//
// Kernel design: a CTA owns an 8x8x4 tile of one patch, one voxel per thread.  The FP64 pipe
// (2 lanes per clock and SM) was the bound of this stage when the stencils were FP64 sums: 23 operations
// for the sixth differences of a variable and 3 per derivative, of 160 (wave) and 2400 (GW59) a
// voxel.  They are now sums in 64-bit fixed point on the integer pipe (dh_fixed.cuh, fd_stencil),
// which the FP64 operations of the products and of the update run beside: 19 and 627 FP64
// adds, products and FMAs a voxel are left, and a conversion for every sum.
// Each variable with the tile's three-voxel face halos (edges and corners are never read by the
// axis-aligned stencils) is brought into a padded 14x14x10 box of shared memory by asynchronous
// copies, several variables ahead of its use (FdRing), so one split barrier per variable is all the
// waiting there is; halo voxels outside the patch come from the face neighbours.  A variable's
// update is written after the next variable's staging: its chain of FP64 operations (64 clocks each)
// is then issued among the integer operations of the next stencil.
// Measured per RK4 step: the wave system on 8.4 M voxels 17.9 -> 4.43 ms (0.9 ms would be the
// memory's), GW59 on 3.9 M voxels 97 -> 29.0 ms.  With the sums in FP64 and every variable staged by plain
// loads: 12 and 75 ms at best.  Against one alignment for all sums whatever its loss (two guard bits, derivatives
// of steep fields short of up to all their bits): 4.05 and 27.4.  That form with the boxes loaded a group of five
// at a time: 5.7 and 36.9; with TMA copies of dense boxes (no padding, so every neighbour's address takes
// selects): 5.2 for the wave system, kept as a variant for it.
// GW59 goes variable by variable (lapse and shift first, then the 11 scalar-wave fields), keeping
// per voxel only the coupling quantities (alpha, beta, grad alpha, phi_b Pi_b, source sums) in registers.
#include <cuda.h>

#include <cstring>
#include <type_traits>

#include "dh_fixed.cuh"
#include "dh_internal.cuh"
#include "dh_pde.cuh"

namespace dh {

// Tensor-map descriptor as a kernel parameter (opaque 128 bytes).
struct alignas(64) TmaDesc {
  unsigned long long v[16];
};

constexpr int FD_MAX_LEVELS = 8;
enum { TMA_INT = 0, TMA_XS = 1, TMA_YS = 2, TMA_ZS = 3 };

struct FdArgs {
  TmaDesc maps[FD_MAX_LEVELS][4];  // per level: interior, x-slab, y-slab, z-slab boxes of qs
  const dh_patch* patches;
  const FdWork* work;
  const int2* lvl;                 // per patch: (level, index within the level)
  const double* qs;
  const double* q0;
  double* out;
  double* acc;
  const double* acc_in;            // acc = acc_in + d dt L (acc itself, or the state the sum starts from)
  double* acc_copy;                // NULL, or a second array that receives the new acc
  const double* mat;
  const double* dt_dev;
  double a, b, g, d;
  int a1, b1, b0;                  // a == 1, b == 1, b == 0 (host side: a comparison is an FP64 operation)
  double sigma;
  double* lam_out;
  unsigned long long* red;
  unsigned int* err;               // error flags (bit 0: a TMA wait gave up)
  int debug_no_issue;              // test hook: arm the barrier but issue no copy
  int64_t vs;
  DevParams P;
};

// Plain FP64 adds, subtractions and products.  (Issuing them as FMAs with
// run-time 1/-1/0 operands, as the FV stage does, measured 7% slower here.)
__device__ __forceinline__ double PADD(const DevParams&, double a, double b) { return a + b; }
__device__ __forceinline__ double PSUB(const DevParams&, double a, double b) { return a - b; }
__device__ __forceinline__ double PMUL(const DevParams&, double a, double b) { return a * b; }

constexpr int FTX = 8, FTY = 8, FTZ = 4, FH = 3;
constexpr int FBX = FTX + 2 * FH, FBY = FTY + 2 * FH, FBZ = FTZ + 2 * FH;
constexpr int FBOX = FBX * FBY * FBZ;                                               // 1960
constexpr int FNSLOT = FTX * FTY * FTZ + 2 * FH * (FTY * FTZ + FTX * FTZ + FTX * FTY);  // 1024
constexpr int FNT = FTX * FTY * FTZ;                                                // 256 threads
constexpr int GV = 5;                                                               // variables per group

// TMA staging buffer of one group (doubles): dense boxes, each 128-byte aligned.
//   interior [5][4][8][8], x-slabs [5][4][8][4] (x rounded out to 16-byte
//   alignment: the slab starts one voxel further out), y-slabs [5][4][3][8],
//   z-slabs [5][3][8][8].
constexpr int TI = 0;
constexpr int TXM = TI + GV * 4 * 8 * 8;   // 1280
constexpr int TXP = TXM + GV * 4 * 8 * 4;  // 1920
constexpr int TYM = TXP + GV * 4 * 8 * 4;  // 2560
constexpr int TYP = TYM + GV * 4 * 3 * 8;  // 3040
constexpr int TZM = TYP + GV * 4 * 3 * 8;  // 3520
constexpr int TZP = TZM + GV * 3 * 8 * 8;  // 4480
constexpr int TBUF = TZP + GV * 3 * 8 * 8;  // 5440 doubles = 43,520 bytes
constexpr unsigned TBYTES = TBUF * 8;
static_assert((TXM * 8) % 128 == 0 && (TXP * 8) % 128 == 0 && (TYM * 8) % 128 == 0 && (TYP * 8) % 128 == 0 &&
                  (TZM * 8) % 128 == 0 && (TZP * 8) % 128 == 0 && (TBUF * 8) % 128 == 0,
              "TMA destinations must be 128-byte aligned");

__device__ __forceinline__ int64_t fd_vox_index(const dh_patch* __restrict__ P, int k, int p, int x, int y, int z) {
  if (x < 0) { k = P[k].nbr[0]; x += p; }
  else if (x >= p) { k = P[k].nbr[1]; x -= p; }
  else if (y < 0) { k = P[k].nbr[2]; y += p; }
  else if (y >= p) { k = P[k].nbr[3]; y -= p; }
  else if (z < 0) { k = P[k].nbr[4]; z += p; }
  else if (z >= p) { k = P[k].nbr[5]; z -= p; }
  return P[k].offset + ((int64_t)z * p + y) * p + x;
}

// Slot s of the tile-plus-face-halo set -> tile-relative (x, y, z).
__device__ __forceinline__ void fd_slot(int s, int& x, int& y, int& z) {
  if (s < FNT) { x = s % FTX; y = (s / FTX) % FTY; z = s / (FTX * FTY); return; }
  int r = s - FNT;
  if (r < 2 * FH * FTY * FTZ) {  // x slabs
    const int side = r / (FH * FTY * FTZ), rr = r % (FH * FTY * FTZ);
    const int h = rr % FH;
    y = (rr / FH) % FTY; z = rr / (FH * FTY);
    x = side == 0 ? -FH + h : FTX + h;
    return;
  }
  r -= 2 * FH * FTY * FTZ;
  if (r < 2 * FH * FTX * FTZ) {  // y slabs
    const int side = r / (FH * FTX * FTZ), rr = r % (FH * FTX * FTZ);
    x = rr % FTX; const int h = (rr / FTX) % FH; z = rr / (FTX * FH);
    y = side == 0 ? -FH + h : FTY + h;
    return;
  }
  r -= 2 * FH * FTX * FTZ;  // z slabs
  const int side = r / (FH * FTX * FTY), rr = r % (FH * FTX * FTY);
  x = rr % FTX; y = (rr / FTX) % FTY; const int h = rr / (FTX * FTY);
  z = side == 0 ? -FH + h : FTZ + h;
}

__device__ __forceinline__ int fd_box(int x, int y, int z) { return ((z + FH) * FBY + (y + FH)) * FBX + (x + FH); }

// ------------------------------------------------------------- stencils
// Read access to one staged variable in a padded box (the variable index is not used: the box
// holds one) ...
struct BoxAcc {
  const double* c;  // this voxel's slot
  __device__ double val(int) const { return *c; }
  template <int D>
  __device__ double nb(int, int o) const {
    constexpr int st = D == 0 ? 1 : (D == 1 ? FBX : FBX * FBY);
    return c[o * st];
  }
};

// ... or the TMA staging buffer (dense interior box plus face slabs).
struct TmaAcc {
  const double* b;
  int lx, ly, lz;
  __device__ double val(int v) const { return b[TI + ((v * 4 + lz) * 8 + ly) * 8 + lx]; }
  template <int D>
  __device__ double nb(int v, int o) const {
    if (D == 0) {
      const int x = lx + o;
      if (x < 0) return b[TXM + ((v * 4 + lz) * 8 + ly) * 4 + (x + 4)];
      if (x >= 8) return b[TXP + ((v * 4 + lz) * 8 + ly) * 4 + (x - 8)];
      return b[TI + ((v * 4 + lz) * 8 + ly) * 8 + x];
    } else if (D == 1) {
      const int y = ly + o;
      if (y < 0) return b[TYM + ((v * 4 + lz) * 3 + (y + 3)) * 8 + lx];
      if (y >= 8) return b[TYP + ((v * 4 + lz) * 3 + (y - 8)) * 8 + lx];
      return b[TI + ((v * 4 + lz) * 8 + y) * 8 + lx];
    } else {
      const int z = lz + o;
      if (z < 0) return b[TZM + ((v * 3 + (z + 3)) * 8 + ly) * 8 + lx];
      if (z >= 4) return b[TZP + ((v * 3 + (z - 4)) * 8 + ly) * 8 + lx];
      return b[TI + ((v * 4 + z) * 8 + ly) * 8 + lx];
    }
  }
};

// The linear stencils of one variable at one voxel: the sum of the sixth differences and the
// unscaled derivatives (q_-2 - q_+2) + 8 (q_+1 - q_-1) along x, y, z.
struct Stencil {
  double ko, d[3];
};

// In FP64 operations, for values that the fixed-point form does not take (infinite, NaN, or beyond
// its exponents); x[d]: the values at -3, -2, -1, +1, +2, +3 along d.  The sixth differences are
// grouped by distance,
//   sum_d delta6_d = T3 - 6 T2 + 15 T1,   T_r = S_r - 6c,
//   S_r = ((Q_-r + Q_+r)_x + (Q_-r + Q_+r)_y) + (Q_-r + Q_+r)_z,
// with 6c formed as ((2c + 2c) + 2c) -- the very additions S_r performs on constant data -- so
// every T_r is exactly 0 on constants (23 FP64 operations).  A stencil of zeros, common in fields
// that start from rest, gives zeros at once.
template <int DM>
__device__ __forceinline__ Stencil fd_stencil_fp64(double c, const double (&x)[3][6]) {
  long long any = __double_as_longlong(c);
#pragma unroll
  for (int d = 0; d < 3; ++d)
#pragma unroll
    for (int i = 0; i < 6; ++i) any |= __double_as_longlong(x[d][i]);
  Stencil R{0.0, {0.0, 0.0, 0.0}};
  if ((any & 0x7fffffffffffffffll) == 0) return R;
  const double two = 2.0 * c, six = (two + two) + two;
  double T[3];
#pragma unroll
  for (int r = 1; r <= 3; ++r)
    T[r - 1] = (((x[0][3 - r] + x[0][2 + r]) + (x[1][3 - r] + x[1][2 + r])) + (x[2][3 - r] + x[2][2 + r])) - six;
  R.ko = fma(15.0, T[0], fma(-6.0, T[1], T[2]));
#pragma unroll
  for (int d = 0; d < 3; ++d)
    if (DM & (1 << d)) R.d[d] = fma(8.0, x[d][3] - x[d][2], x[d][1] - x[d][4]);
  return R;
}

// One unscaled derivative in FP64 operations, its values read again.  Not inlined: in GW59's nine
// stencils the code for a few warps in a hundred took 0.6 ms of an RK4 step of 29.0 (3.9 M voxels).
template <int D, class Acc>
__device__ __noinline__ double fd_derivative(const Acc& S, int v) {
  return fma(8.0, S.template nb<D>(v, 1) - S.template nb<D>(v, -1), S.template nb<D>(v, -2) - S.template nb<D>(v, 2));
}

// In fixed point (dh_fixed.cuh): the 19 values are aligned once, with five guard bits, and serve all
// four sums, in integer instructions and one conversion per sum instead of 23 FP64 operations and 3 per
// derivative: bound by the integer pipe, which the FP64 operations of the terms run beside.  The units that complemented terms lack are counted, so sums of terms that fit are exact
// (odd or linear data give sixth differences of exactly 0, as in FP64).  The sixth differences are
// T_3 - 6 T_2 + 15 T_1 with T_r = S_r - 6c, the grouping of the FP64 form: the T_r need four bits above the
// terms and are exact sums; only where T_1 or T_2 is large are all three shifted by three bits to make
// room for the weights (22 units of a quarter ulp of the largest value at most).
// Terms far below the largest of the 19 lose bits.  For the sixth differences, which read all of them,
// the error stays below that of the FP64 form; a derivative, which reads four, takes its three FP64
// operations where both neighbours along its direction lie more than four binades below the largest
// (a field steep along another direction: its four values may be the small ones).
// Mean error, this over the FP64 form: smooth fields at 16 to 128 voxels a wave 0.00-0.09 (sixth differences)
// and 0.62-0.95 (derivatives); a Gaussian pulse of 6.4 voxels 2, 8, 12 and 20 widths from its centre 0.00, 0.05,
// 0.36, 0.83 and 0.94, 0.56, 0.84, 1.00; white noise 0.45 and 1.00.
// DM: bit d for the derivative along d.  KEEP: the values stay in registers for the FP64 derivatives, which
// in the tails of a pulse most voxels take (RK4 step of the wave system, 8.4 M voxels, nearly all
// in the tails: 4.43 ms, 4.83 with calls of fd_derivative; GW59 without registers to spare 32.4 and 29.0).
template <int DM, bool KEEP, class Acc>
__device__ __forceinline__ Stencil fd_stencil(const Acc& S, int v) {
  constexpr int SH = 5;
  double x[3][6];  // values at -3, -2, -1, +1, +2, +3
  const double c = S.val(v);
  int e = fx_exp(c), nd[3];
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    const int o = i < 3 ? i - 3 : i - 2;
    x[0][i] = S.template nb<0>(v, o);
    x[1][i] = S.template nb<1>(v, o);
    x[2][i] = S.template nb<2>(v, o);
#pragma unroll
    for (int d = 0; d < 3; ++d)
      if (i != 2 && i != 3) e = max(e, fx_exp(x[d][i]));
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    nd[d] = max(fx_exp(x[d][2]), fx_exp(x[d][3]));
    e = max(e, nd[d]);
  }
  if (!fx_ok(e)) return fd_stencil_fp64<DM>(c, x);
  const int low = e - (4 << 20);
  long long s[3] = {0, 0, 0};  // S_1, S_2, S_3
  int n[3] = {0, 0, 0};        // minus their complemented terms
  Stencil R{0.0, {0.0, 0.0, 0.0}};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    long long m[6];
    int g[6];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      m[i] = fx_align<SH>(x[d][i], e);
      g[i] = fx_neg(x[d][i]);
    }
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      s[r] += m[2 - r] + m[3 + r];
      n[r] += g[2 - r] + g[3 + r];
    }
    if (DM & (1 << d)) {
      if (KEEP && nd[d] < low) R.d[d] = fma(8.0, x[d][3] - x[d][2], x[d][1] - x[d][4]);
      else R.d[d] = fx_value<SH>(((m[3] - m[2]) << 3) + (m[1] - m[4]) - (((g[3] - g[2]) << 3) + (g[1] - g[4])), e);
    }
  }
  const long long c6 = 6 * fx_align<SH>(c, e);
  const int n6 = 6 * fx_neg(c);
#pragma unroll
  for (int r = 0; r < 3; ++r) s[r] -= c6;  // T_r, up to the units in n
  int ek = e;
  long long t;
  if ((unsigned)((int)(s[0] >> 32) + (1 << 25)) >= (1u << 26) || (unsigned)((int)(s[1] >> 32) + (1 << 26)) >= (1u << 27)) {
    // |T_1| >= 2^57 or |T_2| >= 2^58: 15 |T_1| + 6 |T_2| + |T_3| < 25.5 x 2^58 below these
#pragma unroll
    for (int r = 0; r < 3; ++r) s[r] = (s[r] - (n[r] - n6) + 4) >> 3;
    t = (s[2] - 6 * s[1]) + 15 * s[0];
    ek += 3 << 20;
  } else {
    t = (s[2] - 6 * s[1]) + 15 * s[0] - ((n[2] - 6 * n[1]) + (15 * n[0] - 10 * n6));
  }
  R.ko = fx_value<SH>(t, ek);
  if constexpr (DM != 0 && !KEEP) {
    int least = low;
#pragma unroll
    for (int d = 0; d < 3; ++d)
      if (DM & (1 << d)) least = min(least, nd[d]);
    if (least < low) {
      if ((DM & 1) && nd[0] < low) R.d[0] = fd_derivative<0>(S, v);
      if ((DM & 2) && nd[1] < low) R.d[1] = fd_derivative<1>(S, v);
      if ((DM & 4) && nd[2] < low) R.d[2] = fd_derivative<2>(S, v);
    }
  }
  return R;
}

// ------------------------------------------------------------- staging
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// One TMA tensor copy (5-D tile) into shared memory, completing on `bar`.
__device__ __forceinline__ void tma_load5(void* dst, const TmaDesc* map, int c0, int c1, int c2, int c3, int c4,
                                          uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::
          "r"(smem_u32(dst)), "l"((unsigned long long)map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4),
      "r"(smem_u32(bar))
      : "memory");
}

// Bounded wait for phase `parity` of `bar`: gives up after ~2^27 SM clocks
// (about 65 ms) and returns false.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  const long long t0 = clock64();
  while (true) {
    uint32_t done;
    asm volatile(
        "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (done) return true;
    if (clock64() - t0 > (1ll << 27)) return false;
  }
}

// Issue the seven copies of group v0 (variables v0..v0+4) of tile w into buffer `buf`.
__device__ void tma_issue(const FdArgs& A, const FdWork& w, int p, double* buf, uint64_t* bar, int v0) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(TBYTES) : "memory");
  if (A.debug_no_issue) return;
  const int2 me = A.lvl[w.patch];
  const TmaDesc* M = A.maps[me.x];
  const dh_patch& pt = A.patches[w.patch];
  const int x0 = w.x0, y0 = w.y0, z0 = w.z0, kl = me.y;
  tma_load5(buf + TI, &M[TMA_INT], x0, y0, z0, kl, v0, bar);
  // x slabs (4 wide, 16-byte aligned start), from this patch or the x neighbours
  if (x0 > 0) tma_load5(buf + TXM, &M[TMA_XS], x0 - 4, y0, z0, kl, v0, bar);
  else tma_load5(buf + TXM, &M[TMA_XS], p - 4, y0, z0, A.lvl[pt.nbr[0]].y, v0, bar);
  if (x0 + 8 < p) tma_load5(buf + TXP, &M[TMA_XS], x0 + 8, y0, z0, kl, v0, bar);
  else tma_load5(buf + TXP, &M[TMA_XS], 0, y0, z0, A.lvl[pt.nbr[1]].y, v0, bar);
  if (y0 > 0) tma_load5(buf + TYM, &M[TMA_YS], x0, y0 - 3, z0, kl, v0, bar);
  else tma_load5(buf + TYM, &M[TMA_YS], x0, p - 3, z0, A.lvl[pt.nbr[2]].y, v0, bar);
  if (y0 + 8 < p) tma_load5(buf + TYP, &M[TMA_YS], x0, y0 + 8, z0, kl, v0, bar);
  else tma_load5(buf + TYP, &M[TMA_YS], x0, 0, z0, A.lvl[pt.nbr[3]].y, v0, bar);
  if (z0 > 0) tma_load5(buf + TZM, &M[TMA_ZS], x0, y0, z0 - 3, kl, v0, bar);
  else tma_load5(buf + TZM, &M[TMA_ZS], x0, y0, p - 3, A.lvl[pt.nbr[4]].y, v0, bar);
  if (z0 + 4 < p) tma_load5(buf + TZP, &M[TMA_ZS], x0, y0, z0 + 4, kl, v0, bar);
  else tma_load5(buf + TZP, &M[TMA_ZS], x0, y0, 0, A.lvl[pt.nbr[5]].y, v0, bar);
}

// CTA-uniform wait; on a timeout every thread records it, waits once more
// (bounded) for copies still in flight, and the caller abandons the tile.
__device__ bool tma_wait_all(const FdArgs& A, uint64_t* bar, uint32_t parity) {
  const bool ok = mbar_wait(bar, parity);
  if (__syncthreads_or(!ok)) {
    if (threadIdx.x == 0) atomicOr(A.err, 1u);
    mbar_wait(bar, parity);
    return false;
  }
  return true;
}

// Ring of NB padded boxes, one variable each: while variable i is computed, the copies of the
// next NB - 2 variables are in flight (asynchronous 8-byte copies global -> shared, one commit
// group per variable; every thread copies the same four of the 1024 slots of every variable, so
// their indexes are formed once per tile).  One barrier per variable, split in two: a warp arrives for
// variable i + 1 when it begins variable i (its copies of i + 1 have landed, its reads of i - 1 are done) and
// waits for the other warps' arrival only when it needs i + 1, so that warps may be a variable apart, some
// in integer stencils while others issue FP64 updates.  The box that new copies overwrite is that
// of variable i - 2.  With __syncthreads for every variable (all warps in the same phase, one variable more
// in flight) an RK4 step took 30.6 ms against 27.8 (GW59) and 4.36 against 3.98 (wave system), with the
// stencils of two guard bits.
static_assert(FNSLOT == 4 * FNT, "four slots per thread");
template <int NB>
struct FdRing {
  static constexpr int AHEAD = NB - 2;  // variables issued ahead of the current one
  double* box;         // NB x FBOX doubles of shared memory
  uint64_t* bars;      // two barriers of one arrival per warp, used in turn
  unsigned int* err;
  const double* qs;
  int64_t vs, e[4];    // arena elements of this thread's slots within a variable
  int c[4];            // their slots in a box
  int centre;

  __device__ __forceinline__ FdRing(const FdArgs& A, const FdWork& w, int p, double* smem, uint64_t* b)
      : box(smem), bars(b), err(A.err), qs(A.qs), vs(A.vs) {
    if (threadIdx.x < 2) mbar_init(&bars[threadIdx.x], FNT / 32);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      int x, y, z;
      fd_slot(threadIdx.x + k * FNT, x, y, z);
      e[k] = fd_vox_index(A.patches, w.patch, p, w.x0 + x, w.y0 + y, w.z0 + z);
      c[k] = fd_box(x, y, z);
    }
    centre = c[0];  // slot 0 of a thread is its own voxel
  }
  // The copies of variable v into box b (v < 0: an empty group, so that the count of groups in
  // flight stays the same to the end).
  __device__ __forceinline__ void issue(int v, int b) {
    if (v >= 0) {
      const double* src = qs + (int64_t)v * vs;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(box + b * FBOX + c[k])),
                     "l"(src + e[k])
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  // This warp is ready for variable i: its copies of it have landed (all groups but the NB - 3 after it).
  __device__ __forceinline__ void ready(int i) {
    asm volatile("cp.async.wait_group %0;" ::"n"(NB - 3) : "memory");
    __syncwarp();
    if ((threadIdx.x & 31) == 0)
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bars[i & 1])) : "memory");
  }
  // After this, variable i of the sequence is in its box and every warp has left the box of variable
  // i - 2.  Bounded by a number of tries, not by the clock, which runs on while a CTA is preempted;
  // every warp arrives for every variable, so it does not run out.
  __device__ __forceinline__ void wait(int i) {
    for (int n = 0; n < (1 << 20); ++n) {
      uint32_t done;
      asm volatile(
          "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2; selp.u32 %0, 1, 0, p; }"
          : "=r"(done)
          : "r"(smem_u32(&bars[i & 1])), "r"((uint32_t)(i >> 1) & 1u)
          : "memory");
      if (done) return;
    }
    atomicOr(err, 1u);
  }
  __device__ __forceinline__ BoxAcc acc(int b) const { return BoxAcc{box + b * FBOX + centre}; }
};

// What the update of one variable reads from memory, loaded ahead of its use.
struct FdOld {
  double q0, acc;
};
__device__ __forceinline__ FdOld fd_old(const FdArgs& A, int64_t ev) {
  FdOld o{0.0, 0.0};
  if (A.out && A.q0) o.q0 = __ldg(A.q0 + ev);
  if (A.acc && A.acc_in != A.qs) o.acc = A.acc_in[ev];
  return o;
}

// out / acc update of one variable; returns the new value of the result.
__device__ __forceinline__ double fd_combine(const FdArgs& A, int64_t ev, const FdOld& o, double qsv, double L, double gdt,
                                             double ddt) {
  double res = 0.0;
  if (A.out) {
    double base;
    if (A.q0 && A.b0 && A.a1) {
      base = o.q0;
    } else {
      base = A.b1 ? qsv : PMUL(A.P, A.b, qsv);
      if (A.q0) base = fma(A.a, o.q0, base);
    }
    res = fma(gdt, L, base);
  }
  if (A.acc) {
    const double r = fma(ddt, L, A.acc_in == A.qs ? qsv : o.acc);
    A.acc[ev] = r;
    if (A.acc_copy) A.acc_copy[ev] = r;
    if (!A.out) res = r;
  }
  if (A.out) A.out[ev] = res;
  return res;
}

// The tile's scalars, formed once per CTA (a division takes about nine FP64 operations).
struct FdScalars {
  double r12, ko, gdt, ddt;  // 1/(12 dx), sigma/(64 dx), g dt, d dt
};
__device__ __forceinline__ void fd_scalars(const FdArgs& A, double dx, FdScalars* s) {
  if (threadIdx.x == 0) {
    const double dt = *A.dt_dev;
    s->r12 = 1.0 / (12.0 * dx);
    s->ko = A.sigma / (64.0 * dx);
    s->gdt = A.g * dt;
    s->ddt = A.d * dt;
  }
}

// ------------------------------------------------------------- generic (N <= 5)
// Stencils of all variables of a system by its B (dq: derivatives times 1/(12 dx) where a column
// of B_d reads them), then the update.
template <class PDE>
__device__ __forceinline__ void fd_finish_generic(const FdArgs& A, const double* q, const double* ko, double (&dq)[3][PDE::N],
                                                  int64_t e, const FdScalars& C, double& lam_thread) {
  constexpr int N = PDE::N, NV = PDE::N + PDE::M;
  double L[N], W[1], D[N], res[NV];
  if (PDE::SRC) PDE::source(q, W, A.P, L);
  else {
#pragma unroll
    for (int v = 0; v < N; ++v) L[v] = 0.0;
  }
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    PDE::ncp(d, q, dq[d], A.P, D);
#pragma unroll
    for (int v = 0; v < N; ++v) L[v] = PSUB(A.P, L[v], D[v]);
  }
#pragma unroll
  for (int v = 0; v < N; ++v)
    res[v] = fd_combine(A, (int64_t)v * A.vs + e, fd_old(A, (int64_t)v * A.vs + e), q[v], fma(C.ko, ko[v], L[v]),
                        C.gdt, C.ddt);
  if (A.lam_out) {
#pragma unroll
    for (int v = N; v < NV; ++v) res[v] = q[v];
    double l = fmax(fmax(PDE::speed(0, res, W, A.P), PDE::speed(1, res, W, A.P)), PDE::speed(2, res, W, A.P));
    lam_thread = fmax(lam_thread, l);
  }
}

// The wave system written out (same operator as the generic path with PdeWave's B and S): the
// 1/(12 dx) of the derivatives is folded into the FMAs that consume them.
//   L_phi   = Pi + KO,   L_Pi = c^2 r12 (Dx psi_x + Dy psi_y + Dz psi_z) - damp Pi + KO,
//   L_psi_d = r12 Dd Pi + KO,   Dd q = (q_-2 - q_+2) + 8 (q_+1 - q_-1) along d.
// `stage(v)` gives access to variable v once it is staged; it is called once per variable, in the
// order 1, 2, 3, 4, 0.
// A variable's update stands after the staging of the next one, so that its FP64 operations can be
// issued among the integer operations of the next stencil.
template <class Stage>
__device__ __forceinline__ void fd_voxel_wave(const FdArgs& A, Stage stage, int64_t e, const FdScalars& C, double& lam_thread) {
  const DevParams& P = A.P;
  const double c = __ldg(A.mat + e);
  const int64_t vs = A.vs;
  Stencil sp, s1, s2, s3;
  double Pi, q1, q2, q3, div;
  const FdOld o1 = fd_old(A, vs + e);
  {
    const auto S = stage(1);
    Pi = S.val(1);
    sp = fd_stencil<7, true>(S, 1);
  }
  const FdOld o2 = fd_old(A, 2 * vs + e);
  {
    const auto S = stage(2);
    q1 = S.val(2);
    s1 = fd_stencil<1, true>(S, 2);
  }
  const FdOld o3 = fd_old(A, 3 * vs + e);
  {
    const auto S = stage(3);
    fd_combine(A, 2 * vs + e, o2, q1, fma(C.ko, s1.ko, PMUL(P, C.r12, sp.d[0])), C.gdt, C.ddt);
    q2 = S.val(3);
    s2 = fd_stencil<2, true>(S, 3);
    div = PADD(P, s1.d[0], s2.d[1]);
  }
  const FdOld o4 = fd_old(A, 4 * vs + e);
  {
    const auto S = stage(4);
    fd_combine(A, 3 * vs + e, o3, q2, fma(C.ko, s2.ko, PMUL(P, C.r12, sp.d[1])), C.gdt, C.ddt);
    q3 = S.val(4);
    s3 = fd_stencil<4, true>(S, 4);
    div = PADD(P, div, s3.d[2]);
  }
  const FdOld o0 = fd_old(A, e);
  {
    const auto S = stage(0);
    fd_combine(A, 4 * vs + e, o4, q3, fma(C.ko, s3.ko, PMUL(P, C.r12, sp.d[2])), C.gdt, C.ddt);
    fd_combine(A, vs + e, o1, Pi, fma(C.ko, sp.ko, fma(PMUL(P, PMUL(P, c, c), C.r12), div, PMUL(P, -P.damp, Pi))), C.gdt, C.ddt);
    fd_combine(A, e, o0, S.val(0), fma(C.ko, fd_stencil<0, true>(S, 0).ko, Pi), C.gdt, C.ddt);
  }
  if (A.lam_out) lam_thread = fmax(lam_thread, c);
}

// Systems of at most five variables.  NB: boxes of the ring (the TMA-staged variants of the wave
// system bring all five variables in one dense buffer instead).
template <class PDE, bool TMA, int NB>
__device__ void fd_tile_generic(const FdArgs& A, const FdWork& w, double* smem, uint64_t* bars, double& lam_thread) {
  static_assert(PDE::N <= GV, "generic FD path stages one group of at most five variables");
  constexpr int N = PDE::N;
  constexpr bool WAVE = std::is_same<PDE, PdeWave>::value;
  static_assert(!TMA || WAVE, "TMA staging is compiled for the wave system");
  const dh_patch& pt = A.patches[w.patch];
  const int p = pt.p;
  const int t = threadIdx.x;
  const int lx = t % FTX, ly = (t / FTX) % FTY, lz = t / (FTX * FTY);
  const int64_t e = pt.offset + ((int64_t)(w.z0 + lz) * p + (w.y0 + ly)) * p + (w.x0 + lx);
  __shared__ FdScalars C;
  if constexpr (TMA) {
    if (t == 0) tma_issue(A, w, p, smem, &bars[0], 0);
    fd_scalars(A, pt.dx, &C);
    if (!tma_wait_all(A, &bars[0], 0)) return;
    fd_voxel_wave(A, [&](int) { return TmaAcc{smem, lx, ly, lz}; }, e, C, lam_thread);
  } else {
    FdRing<NB> R(A, w, p, smem, bars);
    auto var = [](int i) { return i >= N ? -1 : (WAVE ? (i + 1) % N : i); };  // order of the variables
#pragma unroll
    for (int i = 0; i < R.AHEAD; ++i) R.issue(var(i), i);
    fd_scalars(A, pt.dx, &C);
    R.ready(0);
    auto stage = [&](int i) {  // i-th variable of the order
      R.wait(i);
      R.issue(var(i + R.AHEAD), (i + R.AHEAD) % NB);
      R.ready(i + 1);
      return R.acc(i % NB);
    };
    if constexpr (WAVE) {
      fd_voxel_wave(A, [&](int v) { return stage(v == 0 ? 4 : v - 1); }, e, C, lam_thread);
    } else {
      double q[N + PDE::M], ko[N], dq[3][N];
#pragma unroll
      for (int v = 0; v < PDE::M; ++v) q[N + v] = __ldg(A.mat + (int64_t)v * A.vs + e);
#pragma unroll
      for (int v = 0; v < N; ++v) {
        const BoxAcc S = stage(v);
        q[v] = S.val(v);
        const Stencil s = fd_stencil<7, true>(S, v);
        ko[v] = s.ko;
#pragma unroll
        for (int d = 0; d < 3; ++d) dq[d][v] = PDE::needs_grad(d, v) ? PMUL(A.P, s.d[d], C.r12) : 0.0;
      }
      fd_finish_generic<PDE>(A, q, ko, dq, e, C, lam_thread);
    }
  }
}

// ------------------------------------------------------------- GW59
struct Gw59State {
  double al, bx, by, bz, dal0, dal1, dal2, ko_ab[4], u[11], sumPi2, bs0, bs1, bs2;
  double alr, bxr, byr, bzr;  // alpha and beta times 1/(12 dx): the field derivatives stay unscaled
};

__device__ __forceinline__ void gw59_finish(const FdArgs& A, int64_t e, double gdt, double ddt, const Gw59State& G,
                                            double& lam_thread) {
  const DevParams& P = A.P;
  const int64_t vs = A.vs;
  const double Lal = fma(PMUL(P, -P.kappa, PMUL(P, G.al, G.al)), G.sumPi2, G.ko_ab[0]);
  const double ra = fd_combine(A, 55 * vs + e, fd_old(A, 55 * vs + e), G.al, Lal, gdt, ddt);
  const double r0 = fd_combine(A, 56 * vs + e, fd_old(A, 56 * vs + e), G.bx, fma(0.75, G.bs0, G.ko_ab[1]), gdt, ddt);
  const double r1 = fd_combine(A, 57 * vs + e, fd_old(A, 57 * vs + e), G.by, fma(0.75, G.bs1, G.ko_ab[2]), gdt, ddt);
  const double r2 = fd_combine(A, 58 * vs + e, fd_old(A, 58 * vs + e), G.bz, fma(0.75, G.bs2, G.ko_ab[3]), gdt, ddt);
  if (A.lam_out) lam_thread = fmax(lam_thread, PADD(P, ra, fmax(fmax(fabs(r0), fabs(r1)), fabs(r2))));
}

// Variables in the order lapse, shift x, y, z, then per field Pi, psi_x, psi_y, psi_z, phi: each is
// read from its box once, while the next ones stream in.
template <int NB>
__device__ void fd_tile_gw59(const FdArgs& A, const FdWork& w, double* smem, uint64_t* bars, double& lam_thread) {
  const DevParams& P = A.P;
  const int64_t vs = A.vs;
  const dh_patch& pt = A.patches[w.patch];
  const int p = pt.p;
  __shared__ FdScalars C;
  FdRing<NB> R(A, w, p, smem, bars);
  const int64_t e = R.e[0];
  auto var = [](int i) {  // i-th variable of the order
    if (i < 4) return 55 + i;
    if (i >= 59) return -1;
    const int a = (i - 4) / 5, j = (i - 4) - 5 * a;
    return 5 * a + (j == 4 ? 0 : j + 1);
  };
#pragma unroll
  for (int i = 0; i < R.AHEAD; ++i) R.issue(var(i), i);
  fd_scalars(A, pt.dx, &C);
  R.ready(0);
  int cur = 0, buf = 0;  // current variable of the order, its box
  auto stage = [&]() {
    R.wait(cur);
    R.issue(var(cur + R.AHEAD), buf >= NB - R.AHEAD ? buf + R.AHEAD - NB : buf + R.AHEAD);
    R.ready(cur + 1);
    ++cur;
    const BoxAcc S = R.acc(buf);
    buf = buf == NB - 1 ? 0 : buf + 1;
    return S;
  };
  Gw59State G;
  // phi_b Pi_b at this voxel for the source coupling
#pragma unroll
  for (int bb = 0; bb < 11; ++bb)
    G.u[bb] = PMUL(P, __ldg(A.qs + (int64_t)(5 * bb) * vs + e), __ldg(A.qs + (int64_t)(5 * bb + 1) * vs + e));
  G.sumPi2 = 0.0; G.bs0 = 0.0; G.bs1 = 0.0; G.bs2 = 0.0;
  {
    const BoxAcc S = stage();
    const double r12 = C.r12;
    G.al = S.val(0);
    const Stencil s = fd_stencil<7, false>(S, 0);
    G.dal0 = PMUL(P, s.d[0], r12);
    G.dal1 = PMUL(P, s.d[1], r12);
    G.dal2 = PMUL(P, s.d[2], r12);
    G.ko_ab[0] = PMUL(P, C.ko, s.ko);
    G.alr = PMUL(P, G.al, r12);
  }
#pragma unroll
  for (int v = 1; v < 4; ++v) {
    const BoxAcc S = stage();
    const double b = S.val(0);
    (v == 1 ? G.bx : v == 2 ? G.by : G.bz) = b;
    (v == 1 ? G.bxr : v == 2 ? G.byr : G.bzr) = PMUL(P, b, C.r12);
    G.ko_ab[v] = PMUL(P, C.ko, fd_stencil<0, false>(S, 0).ko);
  }
  const double ko = C.ko, gdt = C.gdt, ddt = C.ddt;
  const double al = G.al, bx = G.bx, by = G.by, bz = G.bz, alr = G.alr, bxr = G.bxr, byr = G.byr, bzr = G.bzr;
  double phi = 0.0, Lphi = 0.0;  // the field before: its phi and L_phi, updated in the next field's first step
  FdOld op{0.0, 0.0};
#pragma unroll 1
  for (int a = 0; a < 11; ++a) {
    const int64_t eb = (int64_t)(5 * a) * vs + e;
    // Pi: alpha div psi + beta . grad Pi + alpha cs;  psi_i: alpha d_i Pi + Pi d_i alpha + beta . grad psi_i
    // (unscaled derivatives: the 1/(12 dx) sits in alr, bxr, byr, bzr).  A variable's update stands
    // after the staging of the next one, so that its FP64 operations can be issued among the
    // integer operations of the next stencil.
    double Pi, LPi, div = 0.0, ps = 0.0;
    Stencil sP, s;
    FdOld oP = fd_old(A, eb + vs), o;
    {
      const BoxAcc S = stage();
      if (a > 0) fd_combine(A, eb - 5 * vs, op, phi, Lphi, gdt, ddt);
      Pi = S.val(0);
      sP = fd_stencil<7, false>(S, 0);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {  // psi_x, psi_y, psi_z, phi
      const FdOld on = fd_old(A, eb + (i < 3 ? 2 + i : 0) * vs);
      const BoxAcc S = stage();
      if (i == 0) {
        Lphi = PMUL(P, al, Pi);
        G.sumPi2 = fma(Pi, Pi, G.sumPi2);
        // coupling sum_b C_ab phi_b Pi_b
        double cs = PMUL(P, P.C[11 * a], G.u[0]);
#pragma unroll
        for (int bb = 1; bb < 11; ++bb) cs = fma(P.C[11 * a + bb], G.u[bb], cs);
        LPi = fma(ko, sP.ko, fma(bxr, sP.d[0], fma(byr, sP.d[1], fma(bzr, sP.d[2], PMUL(P, al, cs)))));
      } else {
        const int j = i - 1;
        div = j == 0 ? s.d[0] : PADD(P, div, s.d[j]);
        Lphi = fma(j == 0 ? bx : j == 1 ? by : bz, ps, Lphi);
        double& bs = j == 0 ? G.bs0 : j == 1 ? G.bs1 : G.bs2;
        bs = fma(ps, Pi, bs);
        const double L = fma(alr, sP.d[j], fma(Pi, j == 0 ? G.dal0 : j == 1 ? G.dal1 : G.dal2,
                                               fma(bxr, s.d[0], fma(byr, s.d[1], PMUL(P, bzr, s.d[2])))));
        fd_combine(A, eb + (2 + j) * vs, o, ps, fma(ko, s.ko, L), gdt, ddt);
      }
      if (i == 3) {
        fd_combine(A, eb + vs, oP, Pi, fma(alr, div, LPi), gdt, ddt);
        phi = S.val(0);
        op = on;
        Lphi = fma(ko, fd_stencil<0, false>(S, 0).ko, Lphi);
      } else {
        ps = S.val(0);
        o = on;
        s = fd_stencil<7, false>(S, 0);
      }
    }
  }
  fd_combine(A, 50 * vs + e, op, phi, Lphi, gdt, ddt);
  gw59_finish(A, e, gdt, ddt, G, lam_thread);
}

__device__ __forceinline__ double fd_warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__device__ void fd_publish_lambda(double lam, double* lam_out, unsigned long long* red) {
  __shared__ double wmax[FNT / 32];
  __shared__ bool last;
  lam = fd_warp_max(lam);
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = lam;
  __syncthreads();
  if (threadIdx.x == 0) {
    double m = 0.0;
    for (int i = 0; i < FNT / 32; ++i) m = fmax(m, wmax[i]);
    atomicMax(red, (unsigned long long)__double_as_longlong(m));
    __threadfence();
    last = atomicAdd(red + 1, 1ull) == gridDim.x - 1;
  }
  __syncthreads();
  if (last && threadIdx.x == 0) {
    __threadfence();
    *lam_out = __longlong_as_double((long long)atomicAdd(red, 0ull));
    red[0] = 0ull;
    red[1] = 0ull;
    __threadfence();
  }
}

// Kernel variants (chosen per plan by the autotuner):
//   VAR bit 1: at most 128 registers so that two CTAs fit on an SM, five boxes (else 80 registers
//              and four boxes for three CTAs); GW59 has the first form only;
//   VAR bit 2: TMA staging of all variables in one dense buffer instead of the ring (wave system);
//   VAR bit 3 / bit 4: with TMA staging, register caps for three / four CTAs per SM (80 / 64
//              registers; the buffer takes 43.6 KB).
template <class PDE, int VAR>
constexpr int fd_min_blocks() {
  return (VAR & 16) ? 4 : (VAR & 8) ? 3 : (VAR & 2) ? 2 : (VAR & 4) ? 1 : 3;
}
// Boxes of the ring: as many as fit beside the other CTAs of the SM, at most the variables.
template <class PDE, int VAR>
constexpr int fd_ring() {
  return PDE::N == 59 ? 6 : (VAR & 2) ? 5 : 4;
}

template <class PDE, int VAR>
__global__ void __launch_bounds__(FNT, (fd_min_blocks<PDE, VAR>())) k_fd_stage(const __grid_constant__ FdArgs A) {
  extern __shared__ __align__(128) double fd_smem[];
  __shared__ __align__(8) uint64_t bars[2];
  constexpr bool TMA = (VAR & 4) != 0;
  constexpr int NB = fd_ring<PDE, VAR>();
  const FdWork w = A.work[blockIdx.x];
  double lam = 0.0;
  if constexpr (TMA) {
    // TMA destinations start on a 128-byte boundary (the launch adds 128 bytes of slack)
    double* smem = reinterpret_cast<double*>((reinterpret_cast<uintptr_t>(fd_smem) + 127) & ~(uintptr_t)127);
    if (threadIdx.x == 0) {
      mbar_init(&bars[0], 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    fd_tile_generic<PDE, true, NB>(A, w, smem, bars, lam);
  } else if constexpr (PDE::N == 59) {
    fd_tile_gw59<NB>(A, w, fd_smem, bars, lam);
  } else {
    fd_tile_generic<PDE, false, NB>(A, w, fd_smem, bars, lam);
  }
  if (A.lam_out) fd_publish_lambda(lam, A.lam_out, A.red);
}

template <class PDE, int VAR>
static dh_status fd_launch_var(dh_plan* plan, const FdArgs& A, cudaStream_t stream) {
  constexpr size_t smem = (VAR & 4) ? (size_t)TBYTES + 128 : sizeof(double) * fd_ring<PDE, VAR>() * FBOX;
  static int configured_device = -1;
  if (configured_device != plan->device) {
    cudaError_t e = cudaFuncSetAttribute(k_fd_stage<PDE, VAR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute(k_fd_stage)");
    configured_device = plan->device;
  }
  k_fd_stage<PDE, VAR><<<plan->n_fdwork, FNT, smem, stream>>>(A);
  return cuda_error(cudaGetLastError(), "k_fd_stage launch");
}

// The TMA-staged variants are compiled for the wave system; the others run the ring for them.
template <class PDE>
static dh_status fd_launch(dh_plan* plan, const FdArgs& A, cudaStream_t stream) {
  if constexpr (std::is_same<PDE, PdeWave>::value) {
    switch (plan->fd_var) {
      case 4: return fd_launch_var<PDE, 4>(plan, A, stream);
      case 6: return fd_launch_var<PDE, 6>(plan, A, stream);
      case 12: return fd_launch_var<PDE, 12>(plan, A, stream);
      case 20: return fd_launch_var<PDE, 20>(plan, A, stream);
      default: break;
    }
  }
  if constexpr (PDE::N == 59) {
    return fd_launch_var<PDE, 2>(plan, A, stream);
  } else {
    if (plan->fd_var & 2) return fd_launch_var<PDE, 2>(plan, A, stream);
    return fd_launch_var<PDE, 0>(plan, A, stream);
  }
}

// ------------------------------------------------------------- tensor maps
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}

// 5-D maps over qs for every level: (x, y, z, patch, variable), four box shapes.
static dh_status encode_maps(dh_plan* plan, const double* qs, FdArgs& A) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) { set_error("patch_update_fd_ko: cuTensorMapEncodeTiled is unavailable"); return DH_EUNSUPPORTED; }
  static const cuuint32_t boxes[4][5] = {{8, 8, 4, 1, GV}, {4, 8, 4, 1, GV}, {8, 3, 4, 1, GV}, {8, 8, 3, 1, GV}};
  for (int l = 0; l < plan->n_lvl; ++l) {
    const uint64_t p = (uint64_t)plan->lvl_p[l];
    const cuuint64_t dims[5] = {p, p, p, (cuuint64_t)plan->lvl_K[l], (cuuint64_t)plan->nq};
    const cuuint64_t strides[4] = {p * 8, p * p * 8, p * p * p * 8, (cuuint64_t)plan->var_stride * 8};
    const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    void* base = (void*)(qs + plan->lvl_off[l]);
    for (int bt = 0; bt < 4; ++bt) {
      CUtensorMap m;
      CUresult r = fn(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 5, base, dims, strides, boxes[bt], estr,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (r != CUDA_SUCCESS) {
        set_error("patch_update_fd_ko: cuTensorMapEncodeTiled failed (%d) for level %d", (int)r, l);
        return DH_ECUDA;
      }
      static_assert(sizeof(TmaDesc) == sizeof(CUtensorMap), "tensor map size");
      std::memcpy(&A.maps[l][bt], &m, sizeof(CUtensorMap));
    }
  }
  return DH_OK;
}

dh_status launch_fd_stage(dh_plan* plan, const double* qs, const double* q0, double* out, double* acc,
                          const double* mat, const double* dt_dev, double a, double b, double g, double d,
                          double sigma, double* lam_out, cudaStream_t stream, const double* acc_in,
                          double* acc_copy) {
  FdArgs A;
  std::memset(&A.maps, 0, sizeof(A.maps));
  A.patches = plan->d_patches;
  A.work = plan->d_fdwork;
  A.lvl = plan->d_lvl;
  A.qs = qs; A.q0 = q0; A.out = out; A.acc = acc; A.mat = mat; A.dt_dev = dt_dev;
  A.acc_in = acc_in ? acc_in : acc;
  A.acc_copy = acc_copy;
  A.a = a; A.b = b; A.g = g; A.d = d; A.sigma = sigma;
  A.a1 = a == 1.0; A.b1 = b == 1.0; A.b0 = b == 0.0;
  A.lam_out = lam_out;
  A.red = plan->d_red;
  A.err = reinterpret_cast<unsigned int*>(plan->d_red + 2);
  A.debug_no_issue = plan->debug_flags & 1;
  A.vs = plan->var_stride;
  A.P = plan->params;
  if ((plan->fd_var & 4) && plan->pde == DH_PDE_WAVE3D) {  // (the others run the ring, which reads no maps)
    if (!plan->tma_ok) { set_error("patch_update_fd_ko: the TMA variant needs contiguous levels (see dh_plan_create)"); return DH_EUNSUPPORTED; }
    dh_status st = encode_maps(plan, qs, A);
    if (st != DH_OK) return st;
  }
  switch (plan->pde) {
    case DH_PDE_ADV_NCP: return fd_launch<PdeAdvNcp>(plan, A, stream);
    case DH_PDE_WAVE3D: return fd_launch<PdeWave>(plan, A, stream);
    case DH_PDE_GW59: return fd_launch<PdeGW59>(plan, A, stream);
    default:
      set_error("patch_update_fd_ko: PDE %d not supported by the FD stage", plan->pde);
      return DH_EUNSUPPORTED;
  }
}

}  // namespace dh
