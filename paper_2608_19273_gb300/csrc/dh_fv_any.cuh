// First-order FV stage for plans with patch sizes that are not multiples of 8 (the paper's
// typical 3^3 and 6^3 cells, Sec. IV): the same operator as the z-marching stage (Rusanov face
// flux and non-conservative product of Sec. II-A Eq. 3, the stage combination and the lambda
// epilogue), in a simpler tiling that fits any p.
//
// A CTA of 256 threads takes one work item: up to eight whole small patches of equal p (each
// patch a group), a 2x2x2 block of face-adjacent 3^3 patches as one 6^3 box, or one box of a
// larger patch (6x6x6, 7x7x4 or 8x8x3 voxels in 3D, 16x15 or 15x16 in 2D, smaller at the patch's
// upper ends).  One voxel per thread.  Every item keeps within the limits below (checked on the
// host when the plan is made).
//   1. Every cell of the box and its one-voxel face halo (edges and corners are never read) is
//      loaded into shared memory with its velocity, pressure and sound speed (from the W arena of
//      the stage input, or computed; SRHD: the speeds of the directions it is used in).
//   2. After a barrier every face of all directions is formed once, one per thread and direction
//      (rusanov, the two-sided part of twice the flux), into the face arrays.
//   3. After another barrier every voxel sums its faces and its neighbours' cell terms in fixed
//      point (fx_sum); the stage combination, W of the result and lambda of the result as in the
//      marching stage.
// Shared memory: box cells x (N quantities, velocity, pressure, sound speed or speeds), faces x N
// and direction; 71.7 KB for the Euler equations in 3D, three CTAs per SM.
// Bound by the FP64 pipe: 81 instructions a voxel, 144 when every line cell's flux was formed (the
// face halo of a 6^3 box is as many cells as the box), direction after direction with two barriers
// each, and every face sum was FP64; a box whose W is at hand is copied asynchronously, all of it in flight
// at once (0.36 ms less than loads cell after cell).  16,384 patches of 6^3, two SSP-RK3 steps: 6.71 -> 4.67 ms (the FP64
// instructions alone: 3.4); 4096 of 3^3: 0.23 ms.
#pragma once

namespace dh {

constexpr int ANY_NT = 256;      // threads per CTA; voxels per item at most
constexpr int ANY_SLOTS = 512;   // box cells with halo (all groups) per item
constexpr int ANY_FACES = 256;   // faces of one direction per item (one per thread)

// Integer division by a run-time divisor without the integer divide sequence: for
// 0 <= n < 2^15 and 1 <= d < 2^24, (n + 1/2)/d is never an integer and lies at least 1/(2n + 1)
// (relative) from one, while (n + 1/2) * fl(1/d) in float errs by at most 2^-23 (relative):
// truncation gives floor(n/d) exactly.  Every cell, face and group index here is below 2^10.
struct ADiv {
  int d;
  float r;
  __device__ explicit ADiv(int d_) : d(d_), r(1.0f / (float)d_) {}  // IEEE-rounded quotient
  __device__ int q(int n) const { return (int)(((float)n + 0.5f) * r); }
};

template <class PDE>
struct FvAny {
  static constexpr int N = PDE::N, NV = PDE::N + PDE::M, NW = PDE::NW > 0 ? PDE::NW : 1, DIM = PDE::DIM;
  static constexpr bool HYDRO = PDE::HYDRO;
  // speeds: SRHD keeps the three of a cell (a square root each), Euler its sound speed (one addition
  // per use; with three arrays more only two CTAs fit), advection has them from the velocity
  static constexpr bool SRHD = std::is_same<PDE, PdeSRHD>::value;
  static constexpr int NL = SRHD ? 3 : (HYDRO ? 1 : 0);
  static constexpr int NC = N + DIM + (HYDRO ? 1 : 0) + NL;  // values kept per cell
  static constexpr int NF = PDE::NCP ? 2 : 1;  // face arrays: flux (and non-conservative product)
  static constexpr size_t SMEM =
      sizeof(double) * ((size_t)ANY_SLOTS * NC + (size_t)ANY_FACES * NF * N * DIM);
  static constexpr int CTAS = SMEM <= 74 * 1024 ? 3 : 2;

  template <int WM>
  __device__ static void run(const FvArgs& A, const AnyWork& w, double* smem, double& lam_thread) {
    double* Q = smem;                      // [N][ANY_SLOTS]: box cells
    double* U = Q + N * ANY_SLOTS;         // [DIM][ANY_SLOTS]: velocity (advection: the material)
    double* Pr = U + DIM * ANY_SLOTS;      // [ANY_SLOTS]: pressure (HYDRO)
    double* L = Pr + (HYDRO ? ANY_SLOTS : 0);  // [NL][ANY_SLOTS]
    double* H = L + NL * ANY_SLOTS;        // [DIM][N][ANY_FACES]: face values
    double* Dn = H + DIM * N * ANY_FACES;  // [DIM][N][ANY_FACES]: non-conservative products (NCP systems)
    __shared__ double sc[3];               // the item's -1/(2 dx) (faces hold twice the flux), g dt and d dt times it
    const DevParams& P = A.P;
    const int bx = w.bx, by = w.by, bz = DIM == 3 ? w.bz : 1, ng = w.ng;
    const int SX = bx + 2, SY = by + 2, SZ = DIM == 3 ? bz + 2 : 1;
    const int SG = SX * SY * SZ;  // cells per group
    const int nvg = bx * by * bz;  // voxels per group
    const int tid = threadIdx.x;
    const int g = tid / nvg, li = tid % nvg;
    const bool act = g < ng;
    const int lx = li % bx, ly = (li / bx) % by, lz = li / (bx * by);
    const int p = A.patches[w.patch[0]].p;  // every group or block member of an item has the same p
    if (tid == 0) {
      const double dt = *A.dt_dev;  // read before the lambda epilogue may rewrite it
      sc[0] = -0.5 / A.patches[w.patch[0]].dx;  // (every patch of an item has the same dx)
      sc[1] = A.g * dt * sc[0];
      sc[2] = A.d * dt * sc[0];
    }

    // this voxel's element; what its update reads of the earlier stages is brought into L2 meanwhile
    int64_t e = 0;
    if (act) {
      int k, x, y, z;
      if (w.mp > 0) {
        const int mx = lx >= w.mp, my = ly >= w.mp, mz = lz >= w.mp;
        k = __ldg(w.patch + mx + 2 * my + 4 * mz);
        x = lx - mx * w.mp; y = ly - my * w.mp; z = lz - mz * w.mp;
      } else {
        k = __ldg(w.patch + g);
        x = w.x0 + lx; y = w.y0 + ly; z = DIM == 3 ? w.z0 + lz : 0;
      }
      const int pk = w.mp > 0 ? w.mp : p;
      e = A.patches[k].offset + ((int64_t)z * pk + y) * pk + x;
#pragma unroll
      for (int v = 0; v < N; ++v) {
        if (A.q0) prefetch_l2(A.q0 + v * A.vs + e);
        if (A.acc && A.form != 1) prefetch_l2(A.acc + v * A.vs + e);
      }
    }

    // 1. the box and its face halo, with W: the cells that are read, enumerated group by group as
    //    the box (x fastest), then the two halo layers across x, y and z (edges and corners are
    //    never read and never visited)
    const int HX = by * bz, HY = bx * bz, HZ = DIM == 3 ? bx * by : 0;
    const int CG = nvg + 2 * (HX + HY + HZ);  // cells read per group
    const ADiv dCG(CG), dBX(bx), dBXY(bx * by), dBY(by), dHX(HX), dHY(HY), dHZ(HZ > 0 ? HZ : 1);
    // slot, arena element and halo direction of the j-th cell that is read
    auto cell = [&](int j, int& s, int64_t& e, int& hd) {
      const int gg = dCG.q(j);
      int r = j - gg * CG, cx, cy, cz;
      hd = -1;  // a halo cell's direction
      if (r < nvg) {
        cz = DIM == 3 ? dBXY.q(r) : 0;
        const int rxy = r - cz * bx * by;
        cy = dBX.q(rxy);
        cx = rxy - cy * bx;
      } else if ((r -= nvg) < 2 * HX) {
        const int side = dHX.q(r), t = r - side * HX;
        hd = 0;
        cx = side ? bx : -1;
        cz = dBY.q(t);
        cy = t - cz * by;
      } else if ((r -= 2 * HX) < 2 * HY) {
        const int side = dHY.q(r), t = r - side * HY;
        hd = 1;
        cy = side ? by : -1;
        cz = dBX.q(t);
        cx = t - cz * bx;
      } else {
        r -= 2 * HY;
        const int side = dHZ.q(r), t = r - side * HZ;
        hd = 2;
        cz = side ? bz : -1;
        cy = dBX.q(t);
        cx = t - cy * bx;
      }
      s = gg * SG + ((DIM == 3 ? cz + 1 : 0) * SY + (cy + 1)) * SX + (cx + 1);
      if (w.mp > 0) {
        // a 2x2x2 block of mp^3 patches: the member holding the cell, and the cell's
        // coordinates in it (at most one outside [0, mp): a face neighbour of that member)
        const int mx = cx >= w.mp, my = cy >= w.mp, mz = cz >= w.mp;
        e = vox_index(A.patches, nullptr, __ldg(w.patch + mx + 2 * my + 4 * mz), w.mp, cx - mx * w.mp,
                      cy - my * w.mp, cz - mz * w.mp);
      } else {
        e = vox_index(A.patches, nullptr, __ldg(w.patch + gg), p, w.x0 + cx, w.y0 + cy, DIM == 3 ? w.z0 + cz : 0);
      }
    };
    if constexpr ((WM & 1) && PDE::M == 0) {
      // the state and its W are copied as they are (velocity, pressure and sound speed lie in the
      // order of W), asynchronously: every copy of the item is in flight at once
      static_assert(NC == N + NW, "velocity, pressure and sound speed are W");
#pragma unroll
      for (int it = 0; it < ANY_SLOTS / ANY_NT; ++it) {
        const int j = tid + it * ANY_NT;
        if (j < ng * CG) {
          int s, hd;
          int64_t e;
          cell(j, s, e, hd);
#pragma unroll
          for (int v = 0; v < NC; ++v) {
            const double* src = v < N ? A.qs + v * A.vs + e : A.w_in + (v - N) * A.vs + e;
            asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"((uint32_t)__cvta_generic_to_shared(Q + v * ANY_SLOTS + s)),
                         "l"(src)
                         : "memory");
          }
        }
      }
      asm volatile("cp.async.wait_all;" ::: "memory");
    } else {
      for (int j = tid; j < ng * CG; j += ANY_NT) {
        int s, hd;
        int64_t e;
        cell(j, s, e, hd);
        double q[NV], W[NW];
#pragma unroll
        for (int v = 0; v < N; ++v) q[v] = __ldg(A.qs + v * A.vs + e);
#pragma unroll
        for (int v = 0; v < PDE::M; ++v) q[N + v] = __ldg(A.mat + v * A.vs + e);
        if (WM & 1) {
#pragma unroll
          for (int i = 0; i < NW; ++i) W[i] = __ldg(A.w_in + i * A.vs + e);
        } else {
          PDE::prims(q, P, W);
        }
#pragma unroll
        for (int v = 0; v < N; ++v) Q[v * ANY_SLOTS + s] = q[v];
#pragma unroll
        for (int d = 0; d < DIM; ++d) U[d * ANY_SLOTS + s] = PDE::vel(d, q, W);
        if constexpr (HYDRO) Pr[s] = PDE::press(W);
        if constexpr (SRHD) {
#pragma unroll
          for (int d = 0; d < DIM; ++d)
            if (hd < 0 || hd == d) L[d * ANY_SLOTS + s] = PDE::speed(d, q, W, P);
        } else if constexpr (HYDRO) {
          L[s] = W[DIM + 1];
        }
      }
    }
    __syncthreads();

    // 2. every face once, one per thread and direction, in x-fastest order (consecutive threads touch
    //    consecutive cells: no shared-memory bank conflicts in any direction).  The face grid of a
    //    direction is the voxel grid with one more layer along it: the face at c_d = pos lies
    //    between the cells at pos - 1 and pos (pos = 0 and pos = b_d take a halo cell).
    const int cst[3] = {1, SX, SX * SY};  // box cells along x, y, z
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      const int FX = bx + (d == 0), FY = by + (d == 1), FZ = DIM == 3 ? bz + (d == 2) : 1;
      const int FG = FX * FY * FZ;  // faces per group
      if (tid < ng * FG) {
        const ADiv dFG(FG), dFX(FX), dFY(FY);
        const int gg = dFG.q(tid), r = tid - gg * FG, t = dFX.q(r), cz = dFY.q(t);
        const int cx = r - t * FX, cy = t - cz * FY;
        const int cR = gg * SG + ((DIM == 3 ? cz + 1 : 0) * SY + (cy + 1)) * SX + (cx + 1), cLf = cR - cst[d];
        double qL[N], qR[N], h[N];
#pragma unroll
        for (int v = 0; v < N; ++v) { qL[v] = Q[v * ANY_SLOTS + cLf]; qR[v] = Q[v * ANY_SLOTS + cR]; }
        const double uL = U[d * ANY_SLOTS + cLf], uR = U[d * ANY_SLOTS + cR];
        double lL = abs_int(uL), lR = abs_int(uR);
        if constexpr (SRHD) { lL = L[d * ANY_SLOTS + cLf]; lR = L[d * ANY_SLOTS + cR]; }
        else if constexpr (HYDRO) { lL = ADD(P, lL, L[cLf]); lR = ADD(P, lR, L[cR]); }
        rusanov<PDE>(P, qL, uL, lL, qR, uR, lR, h);
#pragma unroll
        for (int v = 0; v < N; ++v) H[(d * N + v) * ANY_FACES + tid] = h[v];
        if constexpr (PDE::NCP) {
          double qb[NV], dq[N], Dv[N];
#pragma unroll
          for (int v = 0; v < N; ++v) { dq[v] = SUB(P, qR[v], qL[v]); qb[v] = MUL(P, 0.5, ADD(P, qL[v], qR[v])); }
#pragma unroll
          for (int v = 0; v < PDE::M; ++v) qb[N + v] = MUL(P, 0.5, ADD(P, U[v * ANY_SLOTS + cLf], U[v * ANY_SLOTS + cR]));
          PDE::ncp(d, qb, dq, P, Dv);
#pragma unroll
          for (int v = 0; v < N; ++v) Dn[(d * N + v) * ANY_FACES + tid] = Dv[v];
        }
      }
    }
    __syncthreads();

    // 3. stage combination, W and lambda of the result
    if (!act) return;
    const double cS = sc[1], cA = sc[2];
    const bool b1 = A.b == 1.0;
    const int me = g * SG + ((DIM == 3 ? lz + 1 : 0) * SY + (ly + 1)) * SX + (lx + 1);
    double Qk[NV], res[NV];
#pragma unroll
    for (int v = 0; v < N; ++v) Qk[v] = Q[v * ANY_SLOTS + me];
#pragma unroll
    for (int v = 0; v < PDE::M; ++v) Qk[N + v] = HYDRO ? __ldg(A.mat + v * A.vs + e) : U[v * ANY_SLOTS + me];
    static_assert(!PDE::SRC, "systems without a source term");
    // this voxel's faces in the face arrays: below along x, y, z, and the steps to those above
    int fm[DIM], fs[DIM];
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      const int FX = bx + (d == 0), FY = by + (d == 1), FZ = DIM == 3 ? bz + (d == 2) : 1;
      fm[d] = g * FX * FY * FZ + ((DIM == 3 ? lz : 0) * FY + ly) * FX + lx;
      fs[d] = d == 0 ? 1 : (d == 1 ? FX : FX * FY);
    }
    for_n<N>([&](auto vc) {
      constexpr int v = decltype(vc)::value;
      // the terms as in the marching stage: faces, cell terms of the neighbours, the raw sum R
      constexpr bool MOM = HYDRO && v >= 1 && v <= DIM, EN = HYDRO && v == N - 1;
      constexpr int NT = DIM + (EN ? DIM : 0);
      constexpr int NPT = NT + (MOM ? 1 : 0) + (PDE::NCP ? 2 * DIM : 0) + 1;
      const int64_t ev = v * A.vs + e;
      double tp[NPT], tm[NT];
#pragma unroll
      for (int d = 0; d < DIM; ++d) {
        const double* Hv = H + (d * N + v) * ANY_FACES + fm[d];
        tp[d] = Hv[fs[d]]; tm[d] = Hv[0];
        if constexpr (PDE::NCP) {
          const double* Dv = Dn + (d * N + v) * ANY_FACES + fm[d];
          tp[NT + 2 * d] = Dv[fs[d]]; tp[NT + 2 * d + 1] = Dv[0];
        }
        if constexpr (EN) {
          const int cp = me + cst[d], cm = me - cst[d];
          const double up = U[d * ANY_SLOTS + cp], um = U[d * ANY_SLOTS + cm];
          if constexpr (SRHD) {
            tp[DIM + d] = PdeSRHD::cross(Q[cp], Q[(1 + d) * ANY_SLOTS + cp], up);
            tm[DIM + d] = PdeSRHD::cross(Q[cm], Q[(1 + d) * ANY_SLOTS + cm], um);
          } else {
            tp[DIM + d] = MUL(P, Pr[cp], up);
            tm[DIM + d] = MUL(P, Pr[cm], um);
          }
        }
      }
      if constexpr (MOM) tp[DIM] = SUB(P, Pr[me + cst[v - 1]], Pr[me - cst[v - 1]]);
      const double R = A.acc && A.form != 1 ? A.acc[ev] : 0.0;
      tp[NPT - 1] = A.form == 2 ? R : 0.0;
      const double s = fx_sum(tp, tm);
      if (A.form != 0) {
        double o;
        if (A.form == 1) o = fma(cS, s, Qk[v]);
        else if (A.form == 2) o = fma(cS, s, __ldg(A.q0 + ev));
        else o = fma(cS, s, fma(cA, R, __ldg(A.q0 + ev)));
        if (A.form != 3) A.acc[ev] = s;
        res[v] = o;
        A.out[ev] = o;
        return;
      }
      if (A.out) {
        double base = b1 ? Qk[v] : MUL(P, A.b, Qk[v]);
        if (A.q0) base = fma(A.a, __ldg(A.q0 + ev), base);
        res[v] = fma(cS, s, base);
      }
      if (A.acc) {
        const double r = fma(cA, s, R);
        A.acc[ev] = r;
        if (!A.out) res[v] = r;
      }
      if (A.out) A.out[ev] = res[v];
    });
    if (A.lam_out || (WM & 2)) {
#pragma unroll
      for (int v = N; v < NV; ++v) res[v] = Qk[v];
      double Wr[NW];
      PDE::prims(res, P, Wr);
      if (WM & 2) {
#pragma unroll
        for (int i = 0; i < NW; ++i) A.w_out[i * A.vs + e] = Wr[i];
      }
      if (A.lam_out) {
        double l = max_nn(PDE::speed(0, res, Wr, P), PDE::speed(1, res, Wr, P));
        if (DIM == 3) l = max_nn(l, PDE::speed(2, res, Wr, P));
        lam_thread = max_nn(lam_thread, l);
      }
    }
  }
};

template <class PDE, int WM>
__global__ void __launch_bounds__(ANY_NT, FvAny<PDE>::CTAS) k_fv_any(const __grid_constant__ FvArgs A, const AnyWork* __restrict__ work) {
  extern __shared__ __align__(128) double smem[];
  double lam = 0.0;
  const FvArgs R = with_reg_params(A);
  FvAny<PDE>::template run<WM>(R, work[blockIdx.x], smem, lam);
  if (A.lam_out) publish_lambda(lam, A.lam_out, A.red, A.dt_next, A.cfl, A.dx_dim);
}

template <class PDE, int WM>
static dh_status launch_any_wm(dh_plan* plan, const FvArgs& A, cudaStream_t stream) {
  constexpr size_t smem = FvAny<PDE>::SMEM;
  static int configured_device = -1;
  if (configured_device != plan->device) {
    cudaError_t e = cudaFuncSetAttribute(k_fv_any<PDE, WM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute(k_fv_any)");
    configured_device = plan->device;
  }
  if (plan->n_any <= 0) return DH_OK;
  k_fv_any<PDE, WM><<<plan->n_any, ANY_NT, smem, stream>>>(A, plan->d_any);
  return cuda_error(cudaGetLastError(), "k_fv_any launch");
}

template <class PDE>
static dh_status launch_any(dh_plan* plan, const FvArgs& A, int wmode, cudaStream_t stream) {
  if constexpr (std::is_same<PDE, PdeEuler2>::value || std::is_same<PDE, PdeEuler3>::value) {
    switch (wmode & 3) {
      case 1: return launch_any_wm<PDE, 1>(plan, A, stream);
      case 2: return launch_any_wm<PDE, 2>(plan, A, stream);
      case 3: return launch_any_wm<PDE, 3>(plan, A, stream);
      default: break;
    }
  }
  return launch_any_wm<PDE, 0>(plan, A, stream);
}

}  // namespace dh
