// Second-order finite-volume Runge-Kutta stage over all patches in one launch:
// MUSCL reconstruction with the minmod limiter feeding the Rusanov flux (the
// face-state step of the face-flux operator, Sec. II-A Eq. 3, where a state on
// each side of a face comes from a linear stencil over neighbouring voxels),
// for conservative systems (B = 0):
//   sigma_i = minmod(Q_i - Q_{i-1}, Q_{i+1} - Q_i)            (per component)
//   minmod(a, b) = 0 if a, b differ in sign, else the one of smaller magnitude
//   QL = Q_{f-1} + sigma_{f-1}/2,  QR = Q_f - sigma_f/2         (face f)
//   F^ = (F_d(QL) + F_d(QR))/2 - s/2 (QR - QL),  s = max(lambda_d(QL), lambda_d(QR))
//   L(Q)_i = -(1/dx) sum_d [F^_{i+1/2} - F^_{i-1/2}] + S(Q_i)
//   out = a q0 + b qs + g dt L ; acc += d dt L
// A face state carries the material parameters of the voxel it comes from.
//
// Kernel design (the FP64 pipe is the bottleneck, so every slope, face state
// and face value is computed once):
//   * A CTA owns an 8x8x4 tile of one patch (one voxel per thread) and stages
//     its N (+M) quantities with two-voxel face halos into shared memory by
//     plain coalesced loads; halo voxels outside the patch come from the face
//     neighbours (edges and corners are never read and not loaded).
//   * Directions are processed one at a time.  Phase 1: each thread computes the limited slope of
//     its voxel along d and its two face states (+ and -), each with its velocity and speed along
//     d and its pressure; the - state goes to shared memory, the + state stays in registers;
//     further threads compute the inward face state of each halo voxel next to the tile.
//     Phase 2: each thread forms its + face from its own + state and the stored - state of the
//     voxel beyond; the faces before the first voxels are formed by the threads that hold the
//     halo's + states.  Twice the flux of a face is Q_L (u_L + s) + Q_R (u_R - s) plus the
//     pressure terms: 15 FP64 operations (25 with the two fluxes formed apart).
//   * The faces of all directions stay in shared memory, and the sum over a voxel's six faces is
//     formed in fixed point on the integer pipe (fx_sum); -1/(2 dx) carries the factor 1/2.
//   * minmod and all speed maxima run on the integer pipe (sign bits and
//     magnitude bits of the doubles).  (The slopes themselves stay in FP64: aligned to the largest
//     of their three values, a small state beside a large one would lose its low bits.)
//   * lambda_max of the result: warp shuffles, one atomicMax per CTA on the
//     bit pattern, last CTA publishes (no spin waits).
// One SSP-RK3 step of 2.6 M voxels: 5.83 -> 4.92 ms with the face values and the fixed-point sums (308
// FP64 instructions a voxel and stage, 386 before; the pipe is 85% busy).  A z-march of whole columns,
// which needs no halo states along z, took 4% longer than the tiles before these (128 registers with
// spills) and is gone.
#include <algorithm>

#include "dh_fixed.cuh"
#include "dh_internal.cuh"
#include "dh_pde.cuh"

namespace dh {
namespace {

constexpr int MX = 8, MY = 8, MZ = 4, MH = 2;
constexpr int MBX = MX + 2 * MH, MBY = MY + 2 * MH, MBZ = MZ + 2 * MH;
constexpr int MBOX = MBX * MBY * MBZ;                                          // 1152 slots per quantity
constexpr int MNT = MX * MY * MZ;                                              // 256 threads
constexpr int MSLOT = MNT + 2 * MH * (MY * MZ + MX * MZ + MX * MY);            // tile + face halos: 768
constexpr int MFS = (MZ + 1) * MX * MY;                                        // 320 >= (T_d + 1) * area

struct Fv2Args {
  const dh_patch* patches;
  const FdWork* work;
  const double* qs;
  const double* q0;
  double* out;
  double* acc;
  const double* mat;
  const double* dt_dev;
  double a, b, g, d;
  double* lam_out;
  unsigned long long* red;
  int64_t vs;
  DevParams P;
};

__device__ __forceinline__ int mbox(int x, int y, int z) { return ((z + MH) * MBY + (y + MH)) * MBX + (x + MH); }

// Arena index of voxel (x, y, z) of patch k; at most one coordinate outside [0, p).
__device__ __forceinline__ int64_t m_vox(const dh_patch* __restrict__ P, int k, int p, int x, int y, int z) {
  if (x < 0) { k = P[k].nbr[0]; x += p; }
  else if (x >= p) { k = P[k].nbr[1]; x -= p; }
  else if (y < 0) { k = P[k].nbr[2]; y += p; }
  else if (y >= p) { k = P[k].nbr[3]; y -= p; }
  else if (z < 0) { k = P[k].nbr[4]; z += p; }
  else if (z >= p) { k = P[k].nbr[5]; z -= p; }
  return P[k].offset + ((int64_t)z * p + y) * p + x;
}

// Slot s of the tile-plus-face-halo set -> tile-relative (x, y, z).
__device__ __forceinline__ void m_slot(int s, int& x, int& y, int& z) {
  if (s < MNT) { x = s % MX; y = (s / MX) % MY; z = s / (MX * MY); return; }
  int r = s - MNT;
  if (r < 2 * MH * MY * MZ) {
    const int side = r / (MH * MY * MZ), rr = r % (MH * MY * MZ);
    const int h = rr % MH;
    y = (rr / MH) % MY; z = rr / (MH * MY);
    x = side == 0 ? -MH + h : MX + h;
    return;
  }
  r -= 2 * MH * MY * MZ;
  if (r < 2 * MH * MX * MZ) {
    const int side = r / (MH * MX * MZ), rr = r % (MH * MX * MZ);
    x = rr % MX; const int h = (rr / MX) % MH; z = rr / (MX * MH);
    y = side == 0 ? -MH + h : MY + h;
    return;
  }
  r -= 2 * MH * MX * MZ;
  const int side = r / (MH * MX * MY), rr = r % (MH * MX * MY);
  x = rr % MX; y = (rr / MX) % MY; const int h = rr / (MX * MY);
  z = side == 0 ? -MH + h : MZ + h;
}

// minmod on the integer pipe: 0 if the signs differ, else the argument of smaller magnitude.
__device__ __forceinline__ double minmod(double a, double b) {
  const long long ia = __double_as_longlong(a), ib = __double_as_longlong(b);
  if ((ia ^ ib) < 0) return 0.0;
  return (ia & 0x7fffffffffffffffll) < (ib & 0x7fffffffffffffffll) ? a : b;
}

template <class PDE>
struct Fv2Tile {
  static constexpr int N = PDE::N, NV = PDE::N + PDE::M, NW = PDE::NW;
  static constexpr bool HYDRO = PDE::HYDRO;
  static constexpr int NS = N + 3;  // a stored face state: Q (N), velocity, pressure, speed
  static constexpr size_t SMEM = sizeof(double) * ((size_t)NV * MBOX + (size_t)(NS + 3 * N) * MFS);
  static_assert(!PDE::SRC && !PDE::NCP, "conservative systems without a source term");

  // A face state: its quantities, and velocity, pressure and speed along the face's direction.
  struct State {
    double q[N], u, p, lam;
  };
  template <bool WIDE>
  __device__ static State state(const DevParams& P, int d, const double* q, const double* sig, double h) {
    State S;
    double w[NV];
#pragma unroll
    for (int v = 0; v < N; ++v) w[v] = fma(h, sig[v], q[v]);
#pragma unroll
    for (int v = N; v < NV; ++v) w[v] = q[v];
    PDE::template edge<WIDE>(d, w, P, S.u, S.p, S.lam);
#pragma unroll
    for (int v = 0; v < N; ++v) S.q[v] = w[v];
    return S;
  }
  // The voxel at box index c and its limited slope along d (box stride st).
  __device__ static void slope(const DevParams& P, const double* box, int c, int st, double* q, double* sig) {
#pragma unroll
    for (int v = 0; v < N; ++v) {
      const double qm = box[v * MBOX + c - st], qp = box[v * MBOX + c + st];
      q[v] = box[v * MBOX + c];
      sig[v] = minmod(SUB(P, q[v], qm), SUB(P, qp, q[v]));
    }
#pragma unroll
    for (int v = N; v < NV; ++v) q[v] = box[v * MBOX + c];
  }
  __device__ static void store(double* SM, int i, const State& S) {
#pragma unroll
    for (int v = 0; v < N; ++v) SM[v * MFS + i] = S.q[v];
    SM[N * MFS + i] = S.u;
    if (HYDRO) SM[(N + 1) * MFS + i] = S.p;
    SM[(N + 2) * MFS + i] = S.lam;
  }
  // Twice the Rusanov flux along d between a left state in registers and the stored right state
  // at slot f, into the face array H of that direction.
  __device__ static void face(const DevParams& P, int d, const State& L, const double* SM, double* H, int f) {
    const double uR = SM[N * MFS + f], pR = HYDRO ? SM[(N + 1) * MFS + f] : 0.0;
    const double s = max_nn(L.lam, SM[(N + 2) * MFS + f]);
    const double a = ADD(P, L.u, s), b = SUB(P, uR, s);
    double pp = 0.0, pu = 0.0;
    if (HYDRO) {
      pp = ADD(P, L.p, pR);
      pu = fma(L.p, L.u, MUL(P, pR, uR));
    }
#pragma unroll
    for (int v = 0; v < N; ++v) {
      const double cell = HYDRO && v == N - 1 ? pu : (HYDRO && v == 1 + d ? pp : P.zero);
      H[v * MFS + f] = fma(SM[v * MFS + f], b, fma(L.q[v], a, cell));
    }
  }

  __device__ static void run(const Fv2Args& A, const FdWork& w, double* smem, double& lam_thread) {
    double* box = smem;
    double* SM = smem + NV * MBOX;  // - states of one direction
    double* H = SM + NS * MFS;      // faces [direction][N]
    const DevParams& P = A.P;
    const dh_patch pt = A.patches[w.patch];
    const int p = pt.p;
    const int t = threadIdx.x;
    const int tx = t % MX, ty = (t / MX) % MY, tz = t / (MX * MY);
    const int64_t e = pt.offset + ((int64_t)(w.z0 + tz) * p + (w.y0 + ty)) * p + (w.x0 + tx);
    // g dt and d dt times -1/(2 dx), formed once per CTA (faces hold twice the flux)
    __shared__ double sc[2];
    if (t == 0) {
      const double dt = *A.dt_dev, cL = -0.5 / pt.dx;
      sc[0] = A.g * dt * cL;
      sc[1] = A.d * dt * cL;
    }
    // what the update reads is brought into L2 meanwhile
#pragma unroll
    for (int v = 0; v < N; ++v) {
      if (A.q0) asm volatile("prefetch.global.L2 [%0];" ::"l"(A.q0 + (int64_t)v * A.vs + e));
      if (A.acc) asm volatile("prefetch.global.L2 [%0];" ::"l"(A.acc + (int64_t)v * A.vs + e));
    }
    // stage the tile and its two-voxel face halos; whether density and energy of every voxel (and so of
    // the limited states between them) are in the range where momenta can be squared: decided once for
    // the tile, with the loop over the directions compiled for both cases (a test in every edge state
    // took the 2.6 M voxel step from 5.0 to 5.6 ms)
    bool mid = true;
    for (int s = t; s < MSLOT; s += MNT) {
      int x, y, z;
      m_slot(s, x, y, z);
      const int64_t es = m_vox(A.patches, w.patch, p, w.x0 + x, w.y0 + y, w.z0 + z);
      const int c = mbox(x, y, z);
#pragma unroll
      for (int v = 0; v < N; ++v) box[v * MBOX + c] = __ldg(A.qs + (int64_t)v * A.vs + es);
#pragma unroll
      for (int v = 0; v < PDE::M; ++v) box[(N + v) * MBOX + c] = __ldg(A.mat + (int64_t)v * A.vs + es);
      if (HYDRO) mid = mid && mid_range(box[c]) && mid_range(box[(N - 1) * MBOX + c]);
    }
    mid = __syncthreads_and(mid);
    const int me = mbox(tx, ty, tz);
    // state slot of face j (along d) of line o: x faces line by line (consecutive threads, which
    // differ in x, then touch consecutive slots), y and z faces plane by plane (where consecutive
    // threads differ in o)
    auto slot = [&](int d, int area, int j, int o) { return d == 0 ? o * (MX + 1) + j : j * area + o; };
    auto directions = [&](auto wide) {
      constexpr bool WIDE = decltype(wide)::value;
#pragma unroll 1
      for (int d = 0; d < 3; ++d) {
        const int T = d == 0 ? MX : (d == 1 ? MY : MZ);
        const int area = MNT / T;
        const int st = d == 0 ? 1 : (d == 1 ? MBX : MBX * MBY);
        const int a = d == 0 ? tx : (d == 1 ? ty : tz);                          // along d
        const int o = d == 0 ? tz * MY + ty : (d == 1 ? tz * MX + tx : ty * MX + tx);  // across d
        // phase 1: face f lies between voxels f-1 and f along d, so this voxel's + state is the left
        // state of face a+1 and its - state the right state of face a.  Halo voxels next to the tile:
        // the + state of the voxel at -1 (left state of face 0) and the - state of the voxel at T
        // (right state of face T); taken by the last warps along x and z and by warps 4 and 5 along y,
        // so that the extra work of x and y falls on different SM sub-partitions.
        State L, L0;
        {
          double q[NV], sig[N];
          slope(P, box, me, st, q, sig);
          L = state<WIDE>(P, d, q, sig, -P.half);
          store(SM, slot(d, area, a, o), L);
          L = state<WIDE>(P, d, q, sig, P.half);
        }
        const int ht = t - (d == 1 ? 4 * 32 : MNT - 2 * area);
        const bool halo = ht >= 0 && ht < 2 * area;
        const int side = halo ? ht / area : 1, oo = halo ? ht % area : 0;
        if (halo) {
          int hx, hy, hz;
          if (d == 0) { hx = side == 0 ? -1 : MX; hy = oo % MY; hz = oo / MY; }
          else if (d == 1) { hy = side == 0 ? -1 : MY; hx = oo % MX; hz = oo / MX; }
          else { hz = side == 0 ? -1 : MZ; hx = oo % MX; hy = oo / MX; }
          double q[NV], sig[N];
          slope(P, box, mbox(hx, hy, hz), st, q, sig);
          L0 = state<WIDE>(P, d, q, sig, side == 0 ? P.half : -P.half);
          if (side == 1) store(SM, slot(d, area, T, oo), L0);
        }
        __syncthreads();
        // phase 2: every face along d once
        double* Hd = H + d * N * MFS;
        face(P, d, L, SM, Hd, slot(d, area, a + 1, o));
        if (side == 0) face(P, d, L0, SM, Hd, slot(d, area, 0, oo));
        __syncthreads();
      }
    };
    if (HYDRO && !mid) directions(std::true_type{});
    else directions(std::false_type{});
    // update
    const double cS = sc[0], cA = sc[1];
    const bool b1 = A.b == 1.0;
    const int fm[3] = {slot(0, MNT / MX, tx, tz * MY + ty), slot(1, MNT / MY, ty, tz * MX + tx),
                       slot(2, MNT / MZ, tz, ty * MX + tx)};
    const int fp[3] = {fm[0] + 1, fm[1] + MNT / MY, fm[2] + MNT / MZ};
    double q[NV], res[NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) q[v] = box[v * MBOX + me];
    for_n<N>([&](auto vc) {
      constexpr int v = decltype(vc)::value;
      const int64_t ev = (int64_t)v * A.vs + e;
      // the faces along a momentum's own direction hold the pressure: one term, so that nearly equal pressures
      // far above the momentum cancel exactly (fx_sum)
      constexpr int own = HYDRO && v >= 1 && v <= 3 ? v - 1 : -1;
      double tp[3], tm[own >= 0 ? 2 : 3];
      int n = 0;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const double hi = H[(d * N + v) * MFS + fp[d]], lo = H[(d * N + v) * MFS + fm[d]];
        if (d == own) {
          tp[2] = SUB(P, hi, lo);
        } else {
          tp[n] = hi;
          tm[n++] = lo;
        }
      }
      const double sum = fx_sum(tp, tm);
      if (A.out) {
        double base = b1 ? q[v] : MUL(P, A.b, q[v]);
        if (A.q0) base = fma(A.a, __ldg(A.q0 + ev), base);
        res[v] = fma(cS, sum, base);
      }
      if (A.acc) {
        const double r = fma(cA, sum, A.acc[ev]);
        A.acc[ev] = r;
        if (!A.out) res[v] = r;
      }
      if (A.out) A.out[ev] = res[v];
    });
    if (A.lam_out) {
#pragma unroll
      for (int v = N; v < NV; ++v) res[v] = q[v];
      double W[NW > 0 ? NW : 1];
      PDE::prims(res, P, W);
      const double l = max_nn(max_nn(PDE::speed(0, res, W, P), PDE::speed(1, res, W, P)), PDE::speed(2, res, W, P));
      lam_thread = max_nn(lam_thread, l);
    }
  }
};

__device__ void m_publish_lambda(double lam, double* lam_out, unsigned long long* red) {
  __shared__ double wmax[MNT / 32];
  __shared__ bool last;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) lam = max_nn(lam, __shfl_xor_sync(0xffffffffu, lam, o));
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = lam;
  __syncthreads();
  if (threadIdx.x == 0) {
    double m = 0.0;
    for (int i = 0; i < MNT / 32; ++i) m = max_nn(m, wmax[i]);
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

template <class PDE>
__global__ void __launch_bounds__(MNT, 2) k_fv2_stage(const __grid_constant__ Fv2Args A) {
  extern __shared__ __align__(16) double m_smem[];
  const FdWork w = A.work[blockIdx.x];
  double lam = 0.0;
  const Fv2Args R = with_reg_params(A);
  Fv2Tile<PDE>::run(R, w, m_smem, lam);
  if (A.lam_out) m_publish_lambda(lam, A.lam_out, A.red);
}

template <class PDE>
dh_status m_launch(dh_plan* plan, const Fv2Args& A, cudaStream_t s) {
  static int configured_device = -1;
  if (configured_device != plan->device) {
    cudaError_t e = cudaFuncSetAttribute(k_fv2_stage<PDE>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)Fv2Tile<PDE>::SMEM);
    if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute(k_fv2_stage)");
    configured_device = plan->device;
  }
  k_fv2_stage<PDE><<<plan->n_fdwork, MNT, Fv2Tile<PDE>::SMEM, s>>>(A);
  return cuda_error(cudaGetLastError(), "k_fv2_stage launch");
}

}  // namespace

dh_status launch_fv2_stage(dh_plan* plan, const double* qs, const double* q0, double* out, double* acc,
                           const double* mat, const double* dt_dev, double a, double b, double g, double d,
                           double* lam_out, cudaStream_t stream) {
  Fv2Args A;
  A.patches = plan->d_patches;
  A.work = plan->d_fdwork;
  A.qs = qs; A.q0 = q0; A.out = out; A.acc = acc; A.mat = mat; A.dt_dev = dt_dev;
  A.a = a; A.b = b; A.g = g; A.d = d;
  A.lam_out = lam_out;
  A.red = plan->d_red;
  A.vs = plan->var_stride;
  A.P = plan->params;
  switch (plan->pde) {
    case DH_PDE_ADV_FLUX: return m_launch<PdeAdvFlux>(plan, A, stream);
    case DH_PDE_EULER3D: return m_launch<PdeEuler3>(plan, A, stream);
    default:
      set_error("patch_update_fv_muscl: PDE %d not supported (conservative 3-D systems: ADV_FLUX, EULER3D)",
                plan->pde);
      return DH_EUNSUPPORTED;
  }
}

}  // namespace dh
