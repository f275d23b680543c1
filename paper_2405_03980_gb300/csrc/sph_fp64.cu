// FP64 form of the two-fluid spin-SPH step: every stored field in double
// precision; the neighbour passes in 62-bit fixed point where that is at least
// as exact (sph_fixed.cuh), everything else in double precision.
//
// Model (Sec. 2.1, Eqs. 1, 2, 4; Algorithm 1; Sec. 3 boundary set-up):
//   density   rho_i = sum_j m_j W_ij (self included), Wendland C2, support 2h,
//             for fluid and inner-wall particles; outer walls keep rho0;
//   pressure  Eq. 4, P = p0 (rho/rho0)^alpha_P - beta_P;
//   pair pass per neighbour j of a fluid particle i, r_ij = r_i - r_j,
//             F = -(1/r) dW/dr, V = m/rho, e = r_ij / r:
//     pressure      m_i m_j (P_i/rho_i^2 + P_j/rho_j^2) F r_ij
//     interfacial   C_T V_i V_j F (x_ij, y_ij, 0)        unlike species only
//     shear         -10 (eta - 0.6 eta_r) V_i V_j F (e.v_ij) e  neither inviscid
//     rotational    -4 eta_r V_i V_j F (I - ee) u_ij,       neither inviscid
//                   u_ij = v_ij + 1/2 r_ij x (w_i + w_j)
//     F_sn          -C_l V_i V_j W u_ij                    unlike species only
//     spin torque   -1/2 r_ij x (rotational + F_sn), I_i dw_i/dt = tau_i;
//   integrator kick-drift-kick velocity Verlet, rigid walls rotating at Omega,
//   periodic z (slip top/bottom).  Walls count as the viscous species.
#include <math.h>

#include <type_traits>

#include "sph_kernels.h"
#include "sph_partition.cuh"

namespace sphgb {
namespace {

using fx::u64;

__device__ __forceinline__ void latch(uint32_t* err, uint32_t bit) {
  if ((*(volatile uint32_t*)err & bit) == 0u) atomicOr(err, bit);
}

__device__ __forceinline__ bool finite3(double a, double b, double c) {
  return isfinite(a) && isfinite(b) && isfinite(c);
}

// Cell of a position.  A particle outside the interior cell range (or with a
// non-finite coordinate) is clamped into it and ERR_ESCAPED is latched, so
// every later access stays inside the cell arrays.
__device__ __forceinline__ uint32_t cell_key(const InstDev& P, double x, double y, double z,
                                             int sp, uint32_t* err) {
  int c[3];
  const double r[3] = {x, y, z};
  bool bad = false;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const double t = floor((r[a] - P.lo[a]) * P.inv_cell[a]);
    if (a == 2 && P.periodic_z) {
      // z was wrapped into [lo, lo + Hz); rounding may give nz for z just
      // below the top, which belongs to the last cell
      bad |= !(r[a] >= P.lo[a] && r[a] < P.lo[a] + P.Hz);
      c[a] = (t >= 0.0) ? ((t <= (double)(P.nz - 1)) ? (int)t : P.nz - 1) : 0;
    } else if (t >= (double)P.clo[a] && t <= (double)P.chi[a]) {
      c[a] = (int)t;
    } else {
      bad = true;
      c[a] = (t > (double)P.chi[a]) ? P.chi[a] : P.clo[a];  // NaN -> clo
    }
  }
  if (bad) latch(err, ERR_ESCAPED);
  // parts of a cell: the inviscid particles in two x-slabs (short runs for the
  // sort inside a part), the viscous ones, the walls
  int part = sp < 2 ? 2 : 3;
  if (sp == 0) part = (r[0] - P.lo[0]) * P.inv_cell[0] - (double)c[0] < 0.5 ? 0 : 1;
  return (uint32_t)(P.cell_base +
                    ((int64_t)c[0] + (int64_t)P.nx * (c[1] + (int64_t)P.ny * c[2])) * P.slabs +
                    part);
}

inline int grid_for(int64_t n, int threads, int sm_count, int per_sm) {
  int64_t g = (n + threads - 1) / threads;
  int64_t cap = (int64_t)sm_count * per_sm;
  if (g > cap) g = cap;
  return (int)(g < 1 ? 1 : g);
}

// ---------------------------------------------------------------- integrator

__global__ void k_kick_drift_fp64(int64_t n, Fp64Buf b, Fp64Fields f,
                                  const InstDev* __restrict__ inst,
                                  const InstState* __restrict__ ist, CellWs cw,
                                  uint32_t* err, int mode) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t k = b.inst[i];
    const InstDev& P = inst[k];
    dvec4 p = b.pos[i];
    dvec4 v = b.vel[i];
    dvec4 w = b.spin[i];
    const int sp = (int)p.w;
    if (sp < 2) {
      if (mode == 1) {
        const dvec4 a = f.acc[i];
        const dvec4 al = f.dspin[i];
        v.x += P.hdt * a.x;
        v.y += P.hdt * a.y;
        v.z += P.hdt * a.z;
        w.x += P.hdt * al.x;
        w.y += P.hdt * al.y;
        w.z += P.hdt * al.z;
        p.x += P.dt * v.x;
        p.y += P.dt * v.y;
        p.z += P.dt * v.z;
        if (P.periodic_z) {
          if (p.z >= P.Hz + P.lo[2]) p.z -= P.Hz;
          else if (p.z < P.lo[2]) p.z += P.Hz;
        }
        b.vel[i] = v;
        b.spin[i] = w;
        b.pos[i] = p;
      }
      if (!finite3(p.x, p.y, p.z) || !finite3(v.x, v.y, v.z) || !finite3(w.x, w.y, w.z))
        latch(err, ERR_NONFINITE);
    } else {
      // rigid vessel: phase theta_n (mode 0) or theta_n + Omega dt (mode 1)
      double th = ist[k].theta;
      if (mode == 1) th = __dadd_rn(th, __dmul_rn(P.Omega, P.dt));
      double s, c;
      sincos(th, &s, &c);
      const dvec2 r0 = b.ref[i];
      p.x = __dsub_rn(__dmul_rn(c, r0.x), __dmul_rn(s, r0.y));
      p.y = __dadd_rn(__dmul_rn(s, r0.x), __dmul_rn(c, r0.y));
      v.x = -P.Omega * p.y;
      v.y = P.Omega * p.x;
      v.z = 0.0;
      w.x = 0.0;
      w.y = 0.0;
      w.z = P.Omega;
      b.pos[i] = p;
      b.vel[i] = v;
      b.spin[i] = w;
    }
    const uint32_t key = cell_key(P, p.x, p.y, p.z, sp, err);
    cw.key[i] = key;
    cw.slot[i] = atomicAdd(&cw.count[key], 1u);
  }
}

__global__ void k_kick_fp64(int64_t n, Fp64Buf b, Fp64Fields f,
                            const InstDev* __restrict__ inst) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double spw = b.pos[i].w;
    if (spw >= 2.0) continue;
    const double hdt = inst[b.inst[i]].hdt;
    const dvec4 a = f.acc[i];
    const dvec4 al = f.dspin[i];
    dvec4 v = b.vel[i];
    dvec4 w = b.spin[i];
    v.x += hdt * a.x;
    v.y += hdt * a.y;
    v.z += hdt * a.z;
    w.x += hdt * al.x;
    w.y += hdt * al.y;
    w.z += hdt * al.z;
    b.vel[i] = v;
    b.spin[i] = w;
  }
}

// -------------------------------------------------------------------- reorder

__global__ void k_reorder_fp64(int64_t n, Fp64Buf src, Fp64Buf dst, CellWs cw, NbrWs nw,
                               const InstDev* __restrict__ inst) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t j = checked_index(cw.slot[k], n, cw.err);
    const dvec4 p = src.pos[j];
    dst.pos[k] = p;
    dst.vel[k] = src.vel[j];
    dst.spin[k] = src.spin[j];
    dst.ref[k] = src.ref[j];
    dst.id[k] = src.id[j];
    dst.inst[k] = src.inst[j];
    cw.skey[k] = cw.key[j];
    nw.posf[k] = make_float4((float)p.x, (float)p.y, (float)p.z, (float)p.w);
    const fx::Unit U = inst[src.inst[j]].fx_unit;
    QPos q;
    q.x = fx::to_fixed(p.x, U);
    q.y = fx::to_fixed(p.y, U);
    q.z = fx::to_fixed(p.z, U);
    q.tag = (uint32_t)p.w;
    q.exps = 0u;
    nw.posq[k] = q;
    // a wall placed from a non-finite reference (fluid is tested at its drift)
    if (!finite3(p.x, p.y, p.z)) latch(cw.err, ERR_NONFINITE);
  }
}

// Species and wrap tests without FP64 instructions (the FP64 pipe is the
// bottleneck of this form): the species codes 0..3 are stored as doubles, so
// the high word orders them (0.0 -> 0, 1.0 -> 0x3ff00000, 2.0 -> 0x40000000,
// 3.0 -> 0x40080000).
__device__ __forceinline__ bool inviscid(double w) { return __double2hiint(w) == 0; }
__device__ __forceinline__ bool is_wall(double w) { return __double2hiint(w) >= 0x40000000; }
// Species classes and wall-row zeroing of the FP64 state, for the partition.
struct Fp64Species {
  const uint32_t* skey;
  Fp64Fields f;
  __device__ __forceinline__ int cls(int64_t i) const {  // 0 inviscid, 1 viscous, 2 wall
    const int part = (int)(skey[i] & (uint32_t)(kSlabs - 1));  // (a cell's parts: cell_key)
    return part < 2 ? 0 : part - 1;
  }
  __device__ __forceinline__ void zero(int64_t i) const {
    const dvec4 z = {0.0, 0.0, 0.0, 0.0};
    f.acc[i] = z;
    f.dspin[i] = z;
    f.tw[i] = z;
  }
};

// z period crossed by the pair (i, j): +1 if j's image lies one period above
// i's cell row (i in the bottom row, cell code dz + 1 = 2), -1 if below (i in
// the top row, code 0), else 0.  The code is c_i - c_j + 1 per axis.
__device__ __forceinline__ int z_wrap(uint32_t ent, int cz_i, int nz) {
  const uint32_t cz = ent >> (kNbrIndexBits + 4);
  return (cz_i == 0 && cz == 2u) ? 1 : ((cz_i == nz - 1 && cz == 0u) ? -1 : 0);
}

// Lanes that share a particle's list in the density pass.
constexpr int kLanes = 4;

// -------------------------------------------------------------------- density

__device__ __forceinline__ double ipow(double x, int e) {
  double r = 1.0;
  for (int t = 0; t < e; ++t) r *= x;
  return r;
}

// A QPos record in one 256-bit load.
__device__ __forceinline__ QPos ld_qpos(const QPos* q) {
  unsigned long long x, y, z, s;
  asm("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];" : "=l"(x), "=l"(y), "=l"(z), "=l"(s) : "l"(q));
  QPos r;
  r.x = (int64_t)x;
  r.y = (int64_t)y;
  r.z = (int64_t)z;
  r.tag = (uint32_t)s;
  r.exps = (uint32_t)(s >> 32);
  return r;
}

// What decides a pair in fixed point, and the z code and period of a
// neighbour across the periodic boundary, for particle i in z cell cz.
struct PairRange {
  uint64_t near2, width, far2;  // r^2 - near2 < width: neighbour; r^2 >= far2: not
  uint32_t wrap_code;
  int64_t wrap;
  bool bottom;
};
__device__ __forceinline__ PairRange pair_range(const InstDev& P, int cz) {
  PairRange R;
  R.near2 = P.fx_near;
  R.width = P.fx_width;
  R.far2 = P.fx_far;
  R.bottom = cz == 0;
  R.wrap_code = !P.periodic_z ? 3u : (R.bottom ? 2u : (cz == P.nz - 1 ? 0u : 3u));
  R.wrap = R.bottom ? P.fx_Hz : -P.fx_Hz;
  return R;
}
__device__ __forceinline__ int z_cell(const InstDev& P, uint32_t skey) {
  const int64_t g = (int64_t)skey / P.slabs;  // grid cell
  return (int)((g - P.cell_base / P.slabs) / ((int64_t)P.nx * P.ny));
}
// The pair vector of particle q and neighbour o by entry ent, in halves.
struct PairVec {
  fx::Half d[3];
  bool across;
};
__device__ __forceinline__ PairVec pair_vec(const QPos& q, const QPos& o, uint32_t ent,
                                            const PairRange& R) {
  PairVec v;
  v.across = (ent >> (kNbrIndexBits + 4)) == R.wrap_code;
  uint64_t dz = (uint64_t)q.z - (uint64_t)o.z;
  if (v.across) dz += (uint64_t)R.wrap;
  v.d[0] = fx::split((int64_t)((uint64_t)q.x - (uint64_t)o.x));
  v.d[1] = fx::split((int64_t)((uint64_t)q.y - (uint64_t)o.y));
  v.d[2] = fx::split((int64_t)dz);
  return v;
}

// The exact test of a pair, r^2 < (2h)^2 without fused multiply-adds, strict
// <, in FP64; across: the pair meets across the z period.
__device__ __forceinline__ double exact_r2(const dvec4& a, const dvec4& b, bool across,
                                           const PairRange& R, const InstDev& P) {
  const double dx = __dsub_rn(a.x, b.x), dy = __dsub_rn(a.y, b.y);
  double dz = __dsub_rn(a.z, b.z);
  if (across) dz = R.bottom ? __dadd_rn(dz, P.Hz) : __dsub_rn(dz, P.Hz);
  return __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
}

// The list of a particle whose prefiltered neighbours exceed the list's
// capacity, by one lane with the exact test: returns their number (those past
// the capacity are dropped) and the entries of the first two classes.
__device__ __noinline__ uint32_t exact_list(int64_t n, int64_t i, uint32_t K, uint32_t end0,
                                            uint32_t end1, const uint32_t* tab, const dvec4* pos,
                                            const InstDev* P, const NbrWs* nw, const PairRange* R,
                                            uint32_t* parts) {
  uint32_t have = 0, c0 = 0, c1 = 0;
  const dvec4 a = pos[i];
  for (uint32_t k = 0; k < K; ++k)
    for (uint32_t m = nw->mask[(int64_t)k * n + i]; m; m &= m - 1u) {
      const uint32_t q = (k << 5) + (uint32_t)__ffs(m) - 1u, ent = tab[q];
      const bool across = (ent >> (kNbrIndexBits + 4)) == R->wrap_code;
      if (!(exact_r2(a, pos[ent & kNbrIndexMask], across, *R, *P) < P->cut2)) continue;
      if (have < (uint32_t)nw->cap) {
        nw->list[nbr_slot(n, i, have)] = ent;
        c0 += q < end0 ? 1u : 0u;
        c1 += q < end1 ? 1u : 0u;
      }
      ++have;
    }
  *parts = c0 | ((c1 - c0) << 11);
  return have;
}

// The FP64 route of the candidate pairs that fixed point does not decide
// (within rounding of the cutoff, or nearly coincident), after the common
// loop has passed over them: the exact test and the W shape t^4 (2q + 1).  A
// pair beyond 2h gets an entry that names i itself.
template <bool kFilter>
__device__ __noinline__ void density_exact(int64_t n, int64_t i, uint32_t t0, uint32_t na,
                                           uint32_t cnt, const dvec4* pos, const InstDev* Pp,
                                           const NbrWs* nwp, const PairRange* Rp, fx::Sum96* sums,
                                           uint32_t* dead) {
  const InstDev& P = *Pp;
  const NbrWs& nw = *nwp;
  const QPos pi = nw.posq[i];
  for (uint32_t t = t0; t < cnt; t += kLanes) {
    const int64_t at = nbr_slot(n, i, t);
    const uint32_t ent = nw.list[at], j = ent & kNbrIndexMask;
    if ((int64_t)j == i) continue;  // found beyond 2h before
    const PairVec v = pair_vec(pi, nw.posq[j], ent, *Rp);
    const uint64_t r2q = fx::norm2(v.d[0], v.d[1], v.d[2]);
    if (r2q - Rp->near2 < Rp->width || r2q >= Rp->far2) continue;
    const double r2 = exact_r2(pos[i], pos[j], v.across, *Rp, P);
    double W = 0.0;
    if (r2 < P.cut2) {
      const double t1 = fma(-0.5 * P.inv_h, sqrt(r2), 1.0), t2 = t1 * t1;
      W = t2 * t2 * fma(2.0 * P.inv_h, sqrt(r2), 1.0);
      sums[t < na ? 0 : 1].add(__double2ull_rn(W * 2305843009213693952.0));  // 2^61
    } else {
      nw.list[at] = (uint32_t)i | (21u << kNbrIndexBits);
      ++*dead;
    }
    if (kFilter) nw.wsh_d[at] = W;
  }
}

// The density of a particle that weighs little against a neighbour's own term
// (species masses far apart): its sum hangs on W shapes far below one, where
// the fixed-point step of 2^-61 shows.  Its list once more in FP64, with the
// filter's shapes.
template <bool kFilter>
__device__ __noinline__ double density_light(int64_t n, int64_t i, uint32_t na, uint32_t skey,
                                             const dvec4* pos, const InstDev* Pp,
                                             const NbrWs* nwp, double m_i) {
  const InstDev& P = *Pp;
  const NbrWs& nw = *nwp;
  const PairRange R = pair_range(P, z_cell(P, skey));
  const dvec4 a = pos[i];
  const uint32_t cnt = nw.count[i];
  double S[2] = {0.0, 0.0};
  for (uint32_t t = 0; t < cnt; ++t) {
    const int64_t at = nbr_slot(n, i, t);
    const uint32_t ent = nw.list[at], j = ent & kNbrIndexMask;
    if ((int64_t)j == i) continue;
    const bool across = (ent >> (kNbrIndexBits + 4)) == R.wrap_code;
    const double r = sqrt(exact_r2(a, pos[j], across, R, P));
    const double t1 = fma(-0.5 * P.inv_h, r, 1.0), t2 = t1 * t1;
    const double W = t2 * t2 * fma(2.0 * P.inv_h, r, 1.0);
    S[t < na ? 0 : 1] += W;
    if (kFilter) nw.wsh_d[at] = W;
  }
  return fma(P.m_s * P.aD, S[0], fma(P.m_n * P.aD, S[1], m_i * P.aD));
}

// Density and Tait pressure (Eq. 4).  kLanes lanes first turn the particle's
// candidate mask (the search's FP32 prefilter; words dealt out to the lanes)
// into its list, inviscid neighbours, then viscous ones, then walls, in shared
// memory; then they walk the list, test every entry, sum the neighbours' W
// shapes and write it out for the pair pass; one thread per particle forms rho
// and P.  An entry beyond 2h is replaced by one that names i itself, which the
// pair pass and the read-outs skip.  (With the bits walked and the pairs
// evaluated in one loop, a thread per particle, 22 of 32 lanes were active.)
//
// The pair geometry is in fixed point (sph_fixed.cuh): about 120 integer
// instructions per entry in place of 20 FP64 ones, each of which holds the
// FP64 pipe for 64 issue slots.  A W shape is within 7.5e-18, in units of the
// self term's (an FP64 evaluation within a few 1.1e-16 of itself), and the sum
// over a list is exact.  20.1M particles: 64.5 ms with FP64 arithmetic, 19.6 ms in fixed
// point with a thread per particle, 14.3 ms now (bound by issue, 68 %, and the
// ALU).  Lists written by the search instead took 10.5 ms here but 7.2 ms more
// there.  kFilter: some instance uses the pressure filter; the kernel shape of
// every list entry is then stored beside the list (nw.wsh_d).
constexpr uint32_t kStaged = 168;  // entries of a list staged in shared memory; a longer one is
                                   // written out and read back
template <int BLOCK, bool kFilter>
__global__ void __launch_bounds__(BLOCK)
k_density_fp64(int64_t n, Fp64Buf b, Fp64Fields f, const InstDev* __restrict__ inst, CellWs cw,
               NbrWs nw, uint32_t* err) {
  constexpr int kRows = BLOCK / kLanes;
  __shared__ uint32_t staged[kRows][kStaged + 1];
  __shared__ double sums[kRows][2];
  __shared__ uint32_t gone[kRows];
  const int64_t first = (int64_t)blockIdx.x * kRows;
  const int row = threadIdx.x / kLanes, lane = threadIdx.x % kLanes;
  const bool live = first + row < n;
  const int64_t i = live ? first + row : n - 1;
  const InstDev& P = inst[b.inst[i]];
  const QPos pi = ld_qpos(nw.posq + i);
  const int64_t g = (int64_t)cw.skey[i] / P.slabs;  // grid cell
  PairRange R = pair_range(P, z_cell(P, cw.skey[i]));
  // ---- the list: word k of the mask by lane k % kLanes
  const bool lists = live && (pi.tag & 0xFFFFu) != 3u;  // outer-wall particles keep none
  const uint32_t K = lists ? (nw.ncand[2 * g] + 31u) >> 5 : 0u;
  const uint32_t ends = lists ? nw.ncand[2 * g + 1] : 0u, end0 = ends & 0xFFFFu, end1 = ends >> 16;
  const uint32_t* __restrict__ tab = nw.cand + g * kMaxCand;
  uint32_t cnt = 0, part0 = 0, part1 = 0;
  const uint32_t rounds = __reduce_max_sync(~0u, (K + kLanes - 1) / kLanes);
  for (uint32_t r = 0; r < rounds; ++r) {
    const uint32_t k = r * kLanes + (uint32_t)lane;
    uint32_t m = k < K ? nw.mask[(int64_t)k * n + i] : 0u;
    uint32_t incl = (uint32_t)__popc(m);  // inclusive scan over the lanes
    const uint32_t own = incl;
#pragma unroll
    for (int o = 1; o < kLanes; o <<= 1) {
      const uint32_t v = __shfl_up_sync(~0u, incl, o, kLanes);
      if (lane >= o) incl += v;
    }
    uint32_t at = cnt + incl - own;
    cnt += __shfl_sync(~0u, incl, kLanes - 1, kLanes);
    // the bits of the first two classes (positions before their ends)
    const uint32_t q0 = k << 5;
    const uint32_t d0 = end0 > q0 ? end0 - q0 : 0u, d1 = end1 > q0 ? end1 - q0 : 0u;
    part0 += (uint32_t)__popc(d0 >= 32u ? m : m & ((1u << d0) - 1u));
    part1 += (uint32_t)__popc(d1 >= 32u ? m : m & ((1u << d1) - 1u));
    for (; m; m &= m - 1u, ++at) {
      const uint32_t ent = tab[q0 + (uint32_t)__ffs(m) - 1u];
      if (at < kStaged) staged[row][at] = ent;
      if (cnt > kStaged && at < (uint32_t)nw.cap) nw.list[nbr_slot(n, i, at)] = ent;
    }
  }
#pragma unroll
  for (int o = 1; o < kLanes; o <<= 1) {
    part0 += __shfl_xor_sync(~0u, part0, o);
    part1 += __shfl_xor_sync(~0u, part1, o);
  }
  uint32_t parts = part0 | ((part1 - part0) << 11);
  bool in_memory = cnt > kStaged;  // the list, past the staging
  __syncwarp();
  // rounds before the staging filled up wrote to it alone (a list past the
  // capacity is written anew below, by one lane)
  if (in_memory && cnt <= (uint32_t)nw.cap) {
    for (uint32_t t = (uint32_t)lane; t < kStaged; t += kLanes)
      nw.list[nbr_slot(n, i, t)] = staged[row][t];
  }
  if (cnt > (uint32_t)nw.cap) {
    uint32_t have = 0;
    if (lane == 0) {
      have = exact_list(n, i, K, end0, end1, tab, b.pos, &P, &nw, &R, &parts);
      if (have > (uint32_t)nw.cap) latch(err, ERR_NEIGHBORS);
    }
    const uint32_t group = ((1u << kLanes) - 1u) << (threadIdx.x & 31 & ~(kLanes - 1));
    cnt = min(__shfl_sync(group, have, 0, kLanes), (uint32_t)nw.cap);
    parts = __shfl_sync(group, parts, 0, kLanes);
    in_memory = true;
  }
  __syncwarp();
  if (live && lane == 0) nw.count[i] = cnt;
  // ---- the sum
  const uint32_t na = part_inv(parts), nab = na + part_vis(parts);
  fx::Sum96 sum[2];  // the inviscid neighbours, the others
  uint32_t bits[3] = {0u, 0u, 0u};  // high halves of the t of each class, joined: the highest bit
                                    // is the largest t's
  uint32_t dead = 0;
  bool undecided = false;
  const auto entry = [&](uint32_t t) {
    return in_memory ? nw.list[nbr_slot(n, i, t)] : staged[row][t];
  };
  if (lane < (int)cnt) {
    uint32_t ent_n = entry((uint32_t)lane);  // the next record is loaded one entry ahead
    QPos q_n = ld_qpos(nw.posq + checked_index(ent_n & kNbrIndexMask, n, err));
    for (uint32_t t = (uint32_t)lane; t < cnt; t += kLanes) {
      uint32_t ent = ent_n;
      const QPos q = q_n;
      if (t + kLanes < cnt) {
        ent_n = entry(t + kLanes);
        q_n = ld_qpos(nw.posq + checked_index(ent_n & kNbrIndexMask, n, err));
      }
      const PairVec v = pair_vec(pi, q, ent, R);
      const uint64_t r2 = fx::norm2(v.d[0], v.d[1], v.d[2]);
      uint64_t w8 = 0;
      if (r2 - R.near2 < R.width) {
        const uint64_t tt = fx::shape_t(r2);
        w8 = fx::shape_w8(tt, fx::mulhi(tt, tt));
        const uint32_t hi = (uint32_t)(tt >> 32);
        if (t < na) {
          sum[0].add(w8);
          bits[0] |= hi;
        } else {
          sum[1].add(w8);
          bits[1] |= t < nab ? hi : 0u;
          bits[2] |= t < nab ? 0u : hi;
        }
      } else if (r2 >= R.far2) {
        ent = (uint32_t)i | (21u << kNbrIndexBits);
        ++dead;
      } else {
        undecided = true;
      }
      const int64_t at = nbr_slot(n, i, t);
      nw.list[at] = ent;
      if (kFilter) nw.wsh_d[at] = (double)w8 * 4.336808689942017736e-19;  // 2^-61
    }
    if (undecided)
      density_exact<kFilter>(n, i, (uint32_t)lane, na, cnt, b.pos, &P, &nw, &R, sum, &dead);
  }
  __syncwarp();
  uint32_t lead = (uint32_t)(__clz((int)bits[0]) | (__clz((int)bits[1]) << 8) |
                             (__clz((int)bits[2]) << 16));
#pragma unroll
  for (int o = 1; o < kLanes; o <<= 1) {
    lead = __vminu4(lead, __shfl_xor_sync(~0u, lead, o));
    dead += __shfl_xor_sync(~0u, dead, o);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const uint32_t x = __shfl_xor_sync(~0u, sum[k].w0, o), y = __shfl_xor_sync(~0u, sum[k].w1, o),
                     z = __shfl_xor_sync(~0u, sum[k].w2, o);
      sum[k].add((uint64_t)y << 32 | x);
      sum[k].w2 += z;
    }
  }
  if (lane < 2) sums[row][lane] = lane == 0 ? sum[0].shape_sum() : sum[1].shape_sum();
  if (live && lane == 0) nw.lead[i] = lead | (P.fx_pairs ? 0u : 1u << 31);
  if (lane == 0) gone[row] = parts | (min(dead, 1023u) << 22);
  __syncthreads();
  // ---- rho and P, one thread per particle
  const int64_t io = first + threadIdx.x;
  if (threadIdx.x >= kRows || io >= n) return;
  const InstDev& Q = inst[b.inst[io]];
  const int sp = (int)(nw.posq[io].tag & 0xFFFFu);
  const double m_i = sp == 0 ? Q.m_s : Q.m_n;
  // rho_i = aD (m_i + m_s sum_s W/aD + m_n sum_n W/aD), the self term W(0) = aD;
  // outer walls keep rho0
  double rho = Q.rho0;
  if (sp != 3)
    rho = fma(Q.m_s * Q.aD, sums[threadIdx.x][0],
              fma(Q.m_n * Q.aD, sums[threadIdx.x][1], m_i * Q.aD));
  if (rho < Q.rho_light && sp != 3)
    rho = density_light<kFilter>(n, io, part_inv(gone[threadIdx.x]), cw.skey[io], b.pos, &Q, &nw,
                                 m_i);
  nw.parts[io] = gone[threadIdx.x];
  const double Pres = Q.p0 * ipow(rho * Q.inv_rho0, Q.alphaP) - Q.beta_P;
  f.rho[io] = rho;
  f.P[io] = Pres;
  const double V = m_i / rho;
  b.vel[io].w = V;
  b.spin[io].w = Pres / (rho * rho);
  if (Q.flags & SPH_PFILTER) f.vp[io] = sp == 3 ? dvec2{0.0, 0.0} : dvec2{V, V * Pres};
  if (!isfinite(rho) || !isfinite(Pres)) latch(err, ERR_NONFINITE);
}

// ------------------------------------------------------------ pressure filter

// Pressure filter of Algorithm 1 (its formula is not printed; read as the
// zeroth-order kernel average): P_i <- sum_j V_j P_j W_ij / sum_j V_j W_ij
// over i itself and its neighbour list, for fluid and inner-wall particles of
// the instances that enable it.  The inputs (V, P) come from the density
// pass's separate array, as (V, V P), and the outputs go to f.P and spin.w,
// so rows never read a value another row writes.  W enters through its shape
// t^4 (2q + 1) (the constant aD cancels), which the density pass stored for
// every list entry: the pass streams the list and the shapes and gathers
// (V, V P) only, leaving two FP64 fused multiply-adds per neighbour (the FP64
// pipe, not memory, bounds it).
template <int BLOCK>
__global__ void __launch_bounds__(BLOCK)
k_pfilter_fp64(int64_t n, Fp64Buf b, Fp64Fields f, const InstDev* __restrict__ inst, NbrWs nw,
               uint32_t* err) {
  const int64_t i = (int64_t)blockIdx.x * BLOCK + threadIdx.x;
  if (i >= n) return;
  const InstDev& P = inst[b.inst[i]];
  if (!(P.flags & SPH_PFILTER) || b.pos[i].w == 3.0) return;  // outer walls keep P
  const dvec2 own = f.vp[i];
  double num = own.y, den = own.x;  // self term, W(0) / aD = 1
  const uint32_t cnt = checked_count(nw.count[i], nw.cap, err);
  const uint4* __restrict__ groups = reinterpret_cast<const uint4*>(nw.list);
  const dvec2* __restrict__ shapes = reinterpret_cast<const dvec2*>(nw.wsh_d);
  for (uint32_t t0 = 0; t0 < cnt; t0 += 8) {
    const int64_t g = (int64_t)(t0 >> 3) * n + i;
    const uint4 ga = groups[2 * g], gb = groups[2 * g + 1];
    const uint32_t e[8] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w};
    const uint32_t m = cnt - t0 < 8u ? cnt - t0 : 8u;
    dvec2 w2[4];
#pragma unroll
    for (uint32_t q = 0; q < 4; ++q)
      if (2 * q < m) w2[q] = shapes[4 * g + q];
#pragma unroll
    for (uint32_t u = 0; u < 8; ++u) {
      if (u >= m) break;
      const dvec2 vj = f.vp[checked_index(e[u] & kNbrIndexMask, n, err)];
      const double w = (u & 1) ? w2[u >> 1].y : w2[u >> 1].x;
      num = fma(w, vj.y, num);
      den = fma(w, vj.x, den);
    }
  }
  const double Pf = num / den;
  const double rho = f.rho[i];
  f.P[i] = Pf;
  b.spin[i].w = Pf / (rho * rho);
  if (!isfinite(Pf)) latch(err, ERR_NONFINITE);
}

// ------------------------------------------------------------------ pair pass

// The pair terms a neighbour brings depend on the species of the pair
// (walls count as viscous): two inviscid particles exchange the pressure
// term alone; unlike species the pressure, interfacial and local-interaction
// terms (and the latter's spin torque); two viscous particles the pressure,
// shear and rotational terms and the rotational torque.  The density pass
// lists a fluid particle's inviscid neighbours first (part_inv of them), and
// the pair pass runs over the fluid particles in species order (all inviscid
// ones, then all viscous ones), so that each warp walks the two parts of its
// lists with one specialised loop each: kPathII, kPathIX, kPathVV.
enum { kPathII = 1, kPathIX = 2, kPathVV = 3 };

// Per-particle constants of the pair pass, with the term switches, V_i and
// the kernel constants folded in.
struct PairCtx {
  dvec4 pi, vi, wi;          // own records: position+species, velocity+V, spin+P/rho^2
  double cP0, cP1;           // pressure coefficient for an inviscid / other j
  double cT0, cT1;           // interfacial, j inviscid / other (zero for like species)
  double cBA1, cB1;          // shear - rotational along r, rotational along u (j other)
  double cN0, cN1;           // local interaction (zero for like species)
  double half_inv_h, two_inv_h;
  double hwx, hwy, hwz;      // half the own spin
  long long col2b;           // collision distance^2 bits (0: off)
  int si, cz_i;
  bool hproj, literal, per;
};

struct PairSums {
  double fx = 0.0, fy = 0.0, fz = 0.0;  // force
  double tx = 0.0, ty = 0.0, tz = 0.0;  // spin torque (times -2)
  double wx = 0.0, wy = 0.0, wz = 0.0;  // torque of the walls on the particle
};

// Entries t_begin .. t_end of particle i's list, one 32-byte group at a time.
template <int kPath, int kOpt>
__device__ __forceinline__ void pair_loop(const PairCtx& C, const InstDev& P, const Fp64Buf& b,
                                          const NbrWs& nw, int64_t n, int64_t i,
                                          uint32_t t_begin, uint32_t t_end, uint32_t* err,
                                          PairSums& S) {
  const uint4* __restrict__ groups = reinterpret_cast<const uint4*>(nw.list);
  const dvec4 pi = C.pi, vi = C.vi, wi = C.wi;
  for (uint32_t t = t_begin; t < t_end;) {
    const uint32_t g0 = t >> 3;
    const int64_t gi = 2 * ((int64_t)g0 * n + i);
    const uint4 ga = groups[gi], gb = groups[gi + 1];
    const uint32_t e[8] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w};
    const uint32_t u0 = t & 7u;
    const uint32_t u1 = t_end - (g0 << 3) < 8u ? t_end - (g0 << 3) : 8u;
    t = (g0 + 1) << 3;
#pragma unroll
    for (uint32_t u = 0; u < 8; ++u) {
      if (u < u0) continue;
      if (u >= u1) break;
      const uint32_t j = checked_index(e[u] & kNbrIndexMask, n, err);
      const dvec4 pj = b.pos[j];
      const double dx = pi.x - pj.x, dy = pi.y - pj.y;
      double dz = pi.z - pj.z;
      if (C.per) {  // minimum image across the z period
        const int wz = z_wrap(e[u], C.cz_i, P.nz);
        if (wz > 0) dz += P.Hz;
        else if (wz < 0) dz -= P.Hz;
      }
      const double r2 = dx * dx + dy * dy + dz * dz;
      // coincident particles (r2 = 0) count for the density only; r2 > 0 is
      // tested on the bits (r2 >= 0 or NaN)
      const long long r2b = __double_as_longlong(r2);
      if (!(r2b > 0 && r2b <= 0x7ff0000000000000LL)) continue;
      const double inv_r = rsqrt(r2);
      const double r = r2 * inv_r;
      const double t1 = fma(-C.half_inv_h, r, 1.0);  // 1 - q/2
      const double t2 = t1 * t1;
      const double F = t2 * t1;                      // F / cF
      if (kPath == kPathII) {
        // two inviscid particles: the pressure term alone (and a collision);
        // j is fluid, so no wall torque
        const double Prj = b.spin[j].w;
        double al = C.cP0 * (wi.w + Prj) * F;
        if (kOpt & kOptCollision) {
          const dvec4 vj = b.vel[j];
          const double dv = dx * (vi.x - vj.x) + dy * (vi.y - vj.y) + dz * (vi.z - vj.z);
          if (r2b < C.col2b && __double2hiint(dv) < 0) al += P.cC[0] * dv * (inv_r * inv_r);
        }
        S.fx = fma(al, dx, S.fx);
        S.fy = fma(al, dy, S.fy);
        S.fz = fma(al, dz, S.fz);
        continue;
      }
      const dvec4 vj = b.vel[j];
      const dvec4 wj = b.spin[j];
      // whether j is viscous (or a wall): fixed by the list part (unlike
      // species: j is viscous iff i is not)
      const bool vis_j = kPath == kPathVV || C.si == 0;
      // relative velocity v_ij and spin-corrected u_ij = v_ij + 1/2 r_ij x (w_i + w_j),
      // with s = (w_i + w_j) / 2
      const double vx = vi.x - vj.x, vy = vi.y - vj.y, vz = vi.z - vj.z;
      const double sx = fma(0.5, wj.x, C.hwx), sy = fma(0.5, wj.y, C.hwy),
                   sz = fma(0.5, wj.z, C.hwz);
      const double ux = fma(dy, sz, fma(-dz, sy, vx));
      const double uy = fma(dz, sx, fma(-dx, sz, vy));
      const double uz = fma(dx, sy, fma(-dy, sx, vz));
      // The five pair terms collected along r_ij and u_ij (and v_ij for the
      // literal F_sn): shear -A V_iV_j F (e.v) e = -A V_iV_j F dv/r^2 r_ij,
      // rotational -B V_iV_j F (u - (e.u) e) = -B V_iV_j F u + B V_iV_j F dv/r^2 r_ij
      // (r_ij . u_ij = r_ij . v_ij: the spin part of u_ij is normal to r_ij).
      const double VF = vj.w * F;
      double aP, aT = 0.0, aV = 0.0, bR = 0.0, bN = 0.0, dv = 0.0;
      const bool need_dv = kPath != kPathIX || (kOpt & kOptCollision);
      if (need_dv) dv = dx * vx + dy * vy + dz * vz;  // r_ij . v_ij
      if (kPath == kPathIX) {  // unlike species: pressure, interfacial, F_sn
        const double W = t2 * t2 * fma(C.two_inv_h, r, 1.0);  // W / aD
        aP = (vis_j ? C.cP1 : C.cP0) * (wi.w + wj.w) * F;
        aT = (vis_j ? C.cT1 : C.cT0) * VF;
        bN = (vis_j ? C.cN1 : C.cN0) * vj.w * W;
      } else {  // like viscous species: pressure, shear, rotational
        aP = C.cP1 * (wi.w + wj.w) * F;
        aV = VF * (inv_r * inv_r) * (C.cBA1 * dv);
        bR = C.cB1 * VF;
      }
      // (a class loop adds only the terms its class carries: no FP64 addition
      // of a zero term, as the FP64 pipe bounds this loop)
      double base = kPath == kPathIX ? aP : aP + aV;  // the z component drops aT
      // collision of an approaching pair closer than col_dist: the central
      // force m_i dv_i / dt = -(1 + e) mu_ij (r_ij . v_ij) / (r^2 dt) r_ij;
      // both tests on the bits (dv < 0: its sign bit; -0 adds nothing)
      if ((kOpt & kOptCollision) && r2b < C.col2b && __double2hiint(dv) < 0)
        base += P.cC[C.si + (vis_j ? 1 : 0)] * dv * (inv_r * inv_r);
      const double al = kPath == kPathVV ? base : base + aT;
      const double alz = C.hproj ? base : al;
      // coefficient of u_ij
      const double bu = kPath == kPathIX ? (C.literal ? 0.0 : bN) : bR;
      // The pair force al r_ij + bu u_ij (+ bN v_ij) goes into the sums one
      // fused multiply-add per term, and so does the spin torque
      // -1/2 r_ij x (f_rot + f_sn) = -1/2 bu (r_ij x u_ij), whose factor
      // -1/2 (exact) is applied to the sums: the FP64 pipe bounds this loop.
      const double cx = dy * uz - dz * uy, cy = dz * ux - dx * uz, cz = dx * uy - dy * ux;
      S.fx = fma(al, dx, fma(bu, ux, S.fx));
      S.fy = fma(al, dy, fma(bu, uy, S.fy));
      S.fz = fma(alz, dz, fma(bu, uz, S.fz));
      if ((kOpt & kOptLiteral) && C.literal) {  // coefficient bN of v_ij
        S.fx = fma(bN, vx, S.fx);
        S.fy = fma(bN, vy, S.fy);
        S.fz = fma(bN, vz, S.fz);
      }
      S.tx = fma(bu, cx, S.tx);
      S.ty = fma(bu, cy, S.ty);
      S.tz = fma(bu, cz, S.tz);
      if (is_wall(pj.w)) {  // torque exerted by the wall on particle i
        double pfx = al * dx + bu * ux;
        double pfy = al * dy + bu * uy;
        double pfz = alz * dz + bu * uz;
        if ((kOpt & kOptLiteral) && C.literal) {
          pfx += bN * vx;
          pfy += bN * vy;
          pfz += bN * vz;
        }
        S.wx += fma(-0.5, bu * cx, pi.y * pfz - pi.z * pfy);
        S.wy += fma(-0.5, bu * cy, pi.z * pfx - pi.x * pfz);
        S.wz += fma(-0.5, bu * cz, pi.x * pfy - pi.y * pfx);
      }
    }
  }
}

// kOpt: kOptLiteral if some instance uses the literal F_sn (coefficient of
// v_ij), kOptCollision if some instance uses the collision model; the
// default form (0) has neither and drops both at compile time.  Thread t
// takes the fluid particle order[t]: t < n_inv are the inviscid ones, and
// the threads from the fluid count on (the grid covers all n) return, as do
// those of the instances that k_forces_fx takes.
template <int BLOCK, int kOpt>
__global__ void __launch_bounds__(BLOCK, kOpt ? 512 / BLOCK : 0)
k_forces_fp64(int64_t n, Fp64Buf b, Fp64Fields f, const InstDev* __restrict__ inst, CellWs cw,
              NbrWs nw, uint32_t* err, int64_t part_totals) {
  const int64_t t = (int64_t)blockIdx.x * BLOCK + threadIdx.x;
  if (t >= (int64_t)nw.part[part_totals + 1]) return;
  const int64_t n_inv = nw.part[part_totals];
  const int64_t i = checked_index(nw.order[t], n, err);
  PairCtx C;
  C.pi = b.pos[i];
  const int sp_i = (int)C.pi.w;
  const InstDev& P = inst[b.inst[i]];
  if (P.fx_pairs) return;  // by k_forces_fx
  C.vi = b.vel[i];   // w = V_i
  C.wi = b.spin[i];  // w = P_i / rho_i^2
  const double m_i = sp_i == 0 ? P.m_s : P.m_n;
  const double inv_I = sp_i == 0 ? P.inv_I_s : P.inv_I_n;
  const uint32_t fl = P.flags;
  const double cP = (fl & SPH_TERM_P) ? m_i : 0.0;
  const double cT = (fl & SPH_TERM_T) ? P.C_T * C.vi.w : 0.0;
  const double cA = (fl & SPH_TERM_SH) ? P.A * C.vi.w : 0.0;
  const double cB = (fl & SPH_TERM_ROT) ? P.B * C.vi.w : 0.0;
  const double cN = (fl & SPH_TERM_SN) ? P.C_l * C.vi.w : 0.0;
  C.literal = (kOpt & kOptLiteral) && (fl & SPH_SN_LITERAL) != 0;
  const bool inv_i = sp_i == 0;
  // collision model: the bits of col_dist^2 (0 when off; r^2 > 0 orders like
  // its bits); its coefficient -(1 + e) mu_ij / dt is read, for the rare
  // colliding pair only, from the table indexed by the species sum, so both
  // sides of a pair read one value
  C.col2b = (kOpt & kOptCollision) ? __double_as_longlong(P.col2) : 0ll;
  C.si = inv_i ? 0 : 1;
  // The species factors of the pair terms depend on j only through whether
  // j is inviscid (suffix 0) or not (suffix 1): mX = 1 for unlike species
  // (interfacial force, F_sn), mV = 1 for two viscous particles (shear,
  // rotational); walls count as viscous.
  const double mX0 = inv_i ? 0.0 : 1.0, mX1 = inv_i ? 1.0 : 0.0;
  const double mV1 = inv_i ? 0.0 : 1.0;
  // The kernel constants cF (in F) and aD (in W) are folded in here, so
  // that the pair loop forms only the shapes t^3 and t^4 (2q + 1).
  C.cP0 = cP * P.m_s * P.cF;
  C.cP1 = cP * P.m_n * P.cF;
  C.cT0 = cT * mX0 * P.cF;
  C.cT1 = cT * mX1 * P.cF;
  C.cBA1 = mV1 != 0.0 ? (cB - cA) * P.cF : 0.0;
  C.cB1 = -cB * mV1 * P.cF;
  C.cN0 = -cN * mX0 * P.aD;
  C.cN1 = -cN * mX1 * P.aD;
  C.hproj = (fl & SPH_HPROJ) != 0;
  C.half_inv_h = 0.5 * P.inv_h;
  C.two_inv_h = 2.0 * P.inv_h;
  C.hwx = 0.5 * C.wi.x;
  C.hwy = 0.5 * C.wi.y;
  C.hwz = 0.5 * C.wi.z;
  const int64_t g = (int64_t)cw.skey[i] / P.slabs;  // grid cell
  C.cz_i = (int)((g - P.cell_base / P.slabs) / ((int64_t)P.nx * P.ny));
  C.per = P.periodic_z != 0;
  PairSums S;
  const uint32_t cnt = checked_count(nw.count[i], nw.cap, err);
  const uint32_t ca = part_inv(nw.parts[i]);
  const uint32_t na = ca < cnt ? ca : cnt;
  // the inviscid neighbours, then the others: the warp's particles are of
  // one species except at the boundary of the two parts of the order
  if (t < n_inv) {
    pair_loop<kPathII, kOpt>(C, P, b, nw, n, i, 0u, na, err, S);
    pair_loop<kPathIX, kOpt>(C, P, b, nw, n, i, na, cnt, err, S);
  } else {
    pair_loop<kPathIX, kOpt>(C, P, b, nw, n, i, 0u, na, err, S);
    pair_loop<kPathVV, kOpt>(C, P, b, nw, n, i, na, cnt, err, S);
  }
  const double inv_m = 1.0 / m_i;
  f.acc[i] = dvec4{S.fx * inv_m, S.fy * inv_m, S.fz * inv_m, 0.0};
  const double tx = -0.5 * S.tx, ty = -0.5 * S.ty, tz = -0.5 * S.tz;
  f.dspin[i] = dvec4{tx * inv_I, ty * inv_I, tz * inv_I, 0.0};
  f.tw[i] = dvec4{S.wx, S.wy, S.wz, 0.0};
  if (!finite3(S.fx, S.fy, S.fz) || !finite3(tx, ty, tz)) latch(err, ERR_NONFINITE);
}

// ----------------------------------------------- pair pass in fixed point
//
// The pair pass of the instances with neither the literal F_sn nor the
// collision model, whose species masses are within a factor of eight
// (InstDev::fx_pairs; the others take the class loops above).  An FP64
// operation holds its pipe for 64 issue slots on this part (two thread
// operations per SM and clock), so the class loops, 23 to 79 of them per pair,
// run 89 % FP64-pipe busy.  Here a pair's vectors are 64-bit fixed point and
// the sums 96-bit, on the integer pipe; FP64 is left to the coefficients of
// the finished sums.
//
// Scales.  The geometry is in units of 2h (sph_fixed.cuh).  Velocities,
// h times the spins and P / rho^2 come as mantissas at each particle's own
// exponent; a first walk over i's list takes the largest exponents of its
// neighbours, and the largest |v_ij| in FP32, which give the power of two
// 2^E2 above every |u_ij|.  u_ij is then rounded at 2^-60 of that (an FP64
// evaluation rounds each operation at 2^-53 of its own value).  The shapes t^3
// and t^4 (5 - 4t) are formed from t 2^lead, which the largest t of the
// neighbours' class brings into [1/2, 1) (found by the density pass), so they
// keep their 60 bits where all neighbours of a class stand near the cutoff
// and t is small (from t itself the force of one neighbour at t = 0.001 was off
// by 1.6e-8, its torque by 1.9e-7).  The coefficient V_j F or V_j W of u_ij is
// shifted up to 62 bits and the product added that much lower in a 96-bit
// sum; a pressure term is rounded at 2^-58 of the largest pressure and F.  A
// sum is exact: it does not depend on the order of the list or on the number
// of lanes.
//
// kL lanes take a particle's entries in turn, two to eight of them (warps of 16
// or 8 particles diverge less than warps of 32, and small vessels spread over
// more warps; see kPairLanes4); their sums are added by shuffles and the
// block's first threads finish one particle each, so the FP64 instructions of
// the end are issued by full warps.  The wall neighbours stand at the end of
// the list and are summed by themselves: their force and torque give the wall
// torque.  A pair that fixed point does not resolve (see fx_near; two viscous
// particles closer than 2h / 8) and every pair of a list that the scales do
// not cover (velocities more than 2^10 apart, overflow, NaN) is evaluated in
// FP64 by slow_walk.
//
// Measured against a 64-bit-mantissa evaluation (vessels of 10,800 to 33,280
// particles: lattices, up to 300 steps, jitter of 0.3 dx at f_v = 0.01, starts
// from rest): largest error per particle relative to its pair terms, of the
// acceleration 1.2e-15 to 7.9e-15 (FP64 loops 5.4e-15 to 5.9e-14), of the spin
// change 3.5e-16 to 1.5e-14 (1.0e-15 to 2.7e-11), of the density 2.4e-16 to
// 3.0e-16 (1.4e-15 to 2.4e-15).  20.1M particles: 134.3 ms in FP64, 39.5 ms
// here (38.2 ms with positions jittered by 0.3 dx).  Nothing is saturated: at
// 15.3 warps per SM (128 registers) issue is 52 % busy, the ALU 48 %, the FMA
// pipe's multiplier 45 %, L1 51 %; the warps wait on their chains of integer
// products (2.0 warps per issue) and on their gathers (1.7).

// Particles below which eight and four lanes take a list, else two: more lanes
// fill the GPU sooner, fewer spend less on adding up (pair pass with 8 / 4 / 2
// lanes: 10,800 particles 59 / 78 / 120 us, 132,000 331 / 303 / 312 us, 169,000
// 421 / 379 / 385 us, 335,000 838 / 722 / 702 us, 2.6M 6.59 / 5.44 / 4.98 ms).
constexpr int64_t kPairLanes8 = 1 << 15;
constexpr int64_t kPairLanes4 = 1 << 18;
constexpr u64 kNearVV = 1ull << 54;  // (2h / 8)^2, the range of fx::recip
constexpr int kSlots = 48;           // per particle: 3 phases x 12 sums, 12 of the FP64 route

__global__ void k_pair_records(int64_t n, Fp64Buf b, const InstDev* __restrict__ inst, NbrWs nw) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const InstDev& P = inst[b.inst[i]];
    const dvec4 v = b.vel[i], w = b.spin[i];
    const double hx = P.h * w.x, hy = P.h * w.y, hz = P.h * w.z;
    const int ev = max(fx::exponent_of(v.x), max(fx::exponent_of(v.y), fx::exponent_of(v.z)));
    const int eh = max(fx::exponent_of(hx), max(fx::exponent_of(hy), fx::exponent_of(hz)));
    const int ep = fx::exponent_of(w.w);
    PairRec r;
    r.v[0] = fx::mantissa_at(v.x, ev);
    r.v[1] = fx::mantissa_at(v.y, ev);
    r.v[2] = fx::mantissa_at(v.z, ev);
    const double V = v.w * P.aD * 4611686018427387904.0;  // 2^62
    r.V = V < 4611686018427387904.0 ? (uint64_t)__double2ll_rn(V) : (1ull << 62) - 1ull;
    r.h[0] = fx::mantissa_at(hx, eh);
    r.h[1] = fx::mantissa_at(hy, eh);
    r.h[2] = fx::mantissa_at(hz, eh);
    r.P = fx::mantissa_at(w.w, ep);
    nw.prec[i] = r;
    nw.pvel[i] = make_float4((float)v.x, (float)v.y, (float)v.z, 0.f);
    QPos* q = nw.posq + i;
    q->tag = (q->tag & 0xFFFFu) | ((uint32_t)(ev + 1022) << 16);
    q->exps = (uint32_t)(eh + 1022) | ((uint32_t)(ep + 1022) << 16);
  }
}

// One pair in FP64: the force and the spin torque of j on i.  Returns 0 for
// coincident particles (density only), 2 if j is a wall, else 1.
__device__ __noinline__ int slow_pair(const Fp64Buf* b, const InstDev* Pp, uint32_t i, uint32_t j,
                                      int wz, double* f) {
  const InstDev& P = *Pp;
  const dvec4 pi = b->pos[i], vi = b->vel[i], wi = b->spin[i];
  const dvec4 pj = b->pos[j], vj = b->vel[j], wj = b->spin[j];
  const double dx = pi.x - pj.x, dy = pi.y - pj.y;
  double dz = pi.z - pj.z;
  if (wz > 0) dz += P.Hz;
  else if (wz < 0) dz -= P.Hz;
  const double r2 = dx * dx + dy * dy + dz * dz;
  if (!(r2 > 0.0)) return 0;
  const double inv_r = rsqrt(r2), r = r2 * inv_r;
  const double t1 = fma(-0.5 * P.inv_h, r, 1.0), t2 = t1 * t1;
  const double F = P.cF * (t2 * t1), W = P.aD * (t2 * t2 * fma(2.0 * P.inv_h, r, 1.0));
  const bool inv_i = inviscid(pi.w), inv_j = inviscid(pj.w);
  const uint32_t fl = P.flags;
  const double VV = vi.w * vj.w;
  const double mm = (inv_i ? P.m_s : P.m_n) * (inv_j ? P.m_s : P.m_n);
  double al = (fl & SPH_TERM_P) ? mm * (wi.w + wj.w) * F : 0.0, aT = 0.0, bu = 0.0;
  const double vx = vi.x - vj.x, vy = vi.y - vj.y, vz = vi.z - vj.z;
  if (inv_i != inv_j) {
    if (fl & SPH_TERM_T) aT = P.C_T * VV * F;
    if (fl & SPH_TERM_SN) bu = -P.C_l * VV * W;
  } else if (!inv_i) {
    const double A = (fl & SPH_TERM_SH) ? P.A : 0.0, B = (fl & SPH_TERM_ROT) ? P.B : 0.0;
    al += (B - A) * VV * F * (dx * vx + dy * vy + dz * vz) * (inv_r * inv_r);
    bu = -B * VV * F;
  }
  const double sx = 0.5 * (wi.x + wj.x), sy = 0.5 * (wi.y + wj.y), sz = 0.5 * (wi.z + wj.z);
  const double ux = vx + (dy * sz - dz * sy), uy = vy + (dz * sx - dx * sz),
               uz = vz + (dx * sy - dy * sx);
  f[0] = (al + aT) * dx;
  f[1] = (al + aT) * dy;
  f[2] = (al + ((fl & SPH_HPROJ) ? 0.0 : aT)) * dz;
  f[3] = f[4] = f[5] = 0.0;
  if (inv_i != inv_j || !inv_i) {  // (two inviscid particles do not see the velocities)
    f[0] += bu * ux;
    f[1] += bu * uy;
    f[2] += bu * uz;
    f[3] = -0.5 * bu * (dy * uz - dz * uy);
    f[4] = -0.5 * bu * (dz * ux - dx * uz);
    f[5] = -0.5 * bu * (dx * uy - dy * ux);
  }
  return is_wall(pj.w) ? 2 : 1;
}

__device__ __forceinline__ int64_t shr(int64_t v, int s) { return v >> (s < 63 ? s : 63); }
__device__ __forceinline__ int64_t sub64(int64_t a, int64_t b) {
  return (int64_t)((uint64_t)a - (uint64_t)b);
}

// What the loops over a particle's entries need.
struct FxCtx {
  QPos q;                       // own position
  int64_t v[3], h[3], P;        // own values at the common scales
  int Ev, Eh, EP;               // shifts of a neighbour's mantissas: E - e (biased)
  int L;                        // left shift of v_ij to the scale of u
  PairRange R;                  // (width 0: fixed point never)
  uint64_t width_vv;            // the same above kNearVV, for two viscous particles
};

// The entries that fixed point does not resolve, in FP64, after the common
// loops have passed over them: each lane's pair by itself, added up in the
// list's order (so that the sums do not depend on the number of lanes), every
// lane left with them: force and torque in out[0..5], the walls' again in
// out[6..11].  Viscous i: the pairs from vv on are of two viscous particles.
template <int kL>
__device__ __noinline__ void slow_walk(int64_t n, int64_t i, uint32_t cnt, uint32_t vv,
                                       const Fp64Buf* b, const InstDev* P, const NbrWs* nw,
                                       const FxCtx* C, double* out) {
  const uint32_t lane = threadIdx.x % kL;
  const uint32_t group = ((1u << kL) - 1u) << (threadIdx.x & 31u & ~(uint32_t)(kL - 1));
  for (uint32_t t0 = 0; t0 < cnt; t0 += kL) {
    const uint32_t t = t0 + lane;
    double f[6];
    int kind = 0;
    if (t < cnt) {
      const uint32_t ent = nw->list[nbr_slot(n, i, t)], j = ent & kNbrIndexMask;
      const PairVec v = pair_vec(C->q, nw->posq[j], ent, C->R);
      const uint64_t r2 = fx::norm2(v.d[0], v.d[1], v.d[2]);
      const bool done = t >= vv ? r2 - kNearVV < C->width_vv : r2 - C->R.near2 < C->R.width;
      if (!done && (int64_t)j != i)  // (an entry that names i is beyond 2h)
        kind = slow_pair(b, P, (uint32_t)i, j, v.across ? (C->R.bottom ? 1 : -1) : 0, f);
    }
    if (!__any_sync(group, kind)) continue;
    for (int l = 0; l < kL; ++l) {
      const int k_l = __shfl_sync(group, kind, l, kL);
      if (!k_l) continue;
      for (int k = 0; k < 6; ++k) {
        const double v = __shfl_sync(group, f[k], l, kL);
        out[k] += v;
        if (k_l == 2) out[6 + k] += v;
      }
    }
  }
}

// Entries t0, t0 + kL, ... of particle i below t1, all of one class; lead:
// the leading zeros of the class's largest t, from which its scale follows.
template <int kPath, int kL>
__device__ __forceinline__ void fx_loop(const FxCtx& C, const NbrWs& nw, int64_t n, int64_t i,
                                        uint32_t t0, uint32_t t1, uint32_t lead,
                                        uint32_t* err,
                                        fx::Acc96 (&acc)[12], bool& any_slow) {
  using fx::Half;
  using fx::mul;
  using fx::split;
  // the next entry's position record is loaded one entry ahead, the entry
  // after it two ahead
  if (t0 >= t1) return;
  uint32_t ent_n = nw.list[nbr_slot(n, i, t0)];
  QPos q_n = ld_qpos(nw.posq + checked_index(ent_n & kNbrIndexMask, n, err));
  uint32_t ent_nn = t0 + kL < t1 ? nw.list[nbr_slot(n, i, t0 + kL)] : ent_n;
  for (uint32_t t = t0; t < t1; t += kL) {
    const uint32_t ent = ent_n;
    const uint32_t j = checked_index(ent & kNbrIndexMask, n, err);
    const QPos q = q_n;
    ent_n = ent_nn;
    q_n = ld_qpos(nw.posq + checked_index(ent_n & kNbrIndexMask, n, err));
    if (t + 2 * kL < t1) ent_nn = nw.list[nbr_slot(n, i, t + 2 * kL)];
    const PairRec* __restrict__ rec = nw.prec + j;
    const PairVec pv = pair_vec(C.q, q, ent, C.R);
    const Half(&d)[3] = pv.d;
    const uint64_t r2 = fx::norm2(d[0], d[1], d[2]);
    if (kPath == kPathVV ? r2 - kNearVV >= C.width_vv : r2 - C.R.near2 >= C.R.width) {
      any_slow |= (int64_t)j != i;  // (an entry beyond 2h names i, and adds nothing)
      continue;
    }
    const int64_t rho = fx::root(r2);
    const uint64_t tt = (uint64_t)((1ll << 62) - rho) << 2;  // t in units of 2^-64
    const uint64_t T = fx::scaled_t(tt, lead);
    const uint64_t Tq = fx::mulhi(T, T);
    const uint64_t F = fx::mulhi(Tq, T);                     // F shape t^3 2^(3 lead)
    // pressure: (P_i / rho_i^2 + P_j / rho_j^2) F r_ij
    const int64_t g = C.P + shr(rec->P, C.EP - (int)(q.exps >> 16));
    const Half gF = split(mul(split(g), split((int64_t)(F >> 2))) << 2);
#pragma unroll
    for (int a = 0; a < 3; ++a) acc[a].add(mul(gF, d[a]));
    if (kPath == kPathII) continue;
    // u_ij = v_ij + r_ij x (w_i + w_j) / 2
    const int sv = C.Ev - (int)(q.tag >> 16), sh = C.Eh - (int)(q.exps & 0xFFFFu);
    int64_t v[3];
    Half s[3], u[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      v[a] = sub64(C.v[a], shr(rec->v[a], sv)) << C.L;
      s[a] = split(C.h[a] + shr(rec->h[a], sh));
    }
    u[0] = split(v[0] + fx::mul_sub(d[1], s[2], d[2], s[1]));
    u[1] = split(v[1] + fx::mul_sub(d[2], s[0], d[0], s[2]));
    u[2] = split(v[2] + fx::mul_sub(d[0], s[1], d[1], s[0]));
    const uint64_t V = rec->V << 2;
    const uint64_t VF = fx::mulhi(V, F);
    uint64_t c;  // the coefficient of u: V_j W / 8 (unlike species) or V_j F (two viscous), 2^-64
    if (kPath == kPathIX) {
      // interfacial: V_j F r_ij
      const Half VFh = split((int64_t)(VF >> 2));
#pragma unroll
      for (int a = 0; a < 3; ++a) acc[3 + a].add(mul(VFh, d[a]));
      c = fx::mulhi(V, fx::shape_w8(tt, Tq));
    } else {
      c = VF;
    }
    const int lz = (int)min(fx::lead32(c), 24u), up = 24 - lz;
    const Half ch = split((int64_t)((c << lz) >> 2));  // 2^lz c in 62 bits
    if (kPath == kPathVV) {
      // the part along e_ij: V_j F (e_ij . v_ij) e_ij
      const Half z = split(fx::recip(rho));
      Half e[3], vh[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        e[a] = split(mul(d[a], z) << 5);
        vh[a] = split(v[a]);
      }
      const Half ev = split(mul(ch, split(fx::dot3(e, vh) << 2)) << 2);
#pragma unroll
      for (int a = 0; a < 3; ++a) acc[3 + a].add_shifted(mul(ev, e[a]), up);
    }
    int64_t p[3];
    Half ph[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      p[a] = mul(ch, u[a]);
      acc[6 + a].add_shifted(p[a], up);
      ph[a] = split(p[a] << 3);
    }
    acc[9].add_shifted(fx::mul_sub(d[1], ph[2], d[2], ph[1]), up);
    acc[10].add_shifted(fx::mul_sub(d[2], ph[0], d[0], ph[2]), up);
    acc[11].add_shifted(fx::mul_sub(d[0], ph[1], d[1], ph[0]), up);
  }
}

// Adds another lane's sum.
__device__ __forceinline__ void add_lane(fx::Acc96& a, const fx::Acc96& give, int mask) {
  const uint32_t x = __shfl_xor_sync(~0u, give.w0, mask);
  const uint32_t y = __shfl_xor_sync(~0u, give.w1, mask);
  const uint32_t z = __shfl_xor_sync(~0u, give.w2, mask);
  a.add3(x, y, z);
}

// The kL lanes' twelve sums added, lane l left with sums m l .. m (l + 1) - 1,
// m = 12 / kL, in acc[0 .. m - 1]: each exchange halves what a lane holds.
template <int kL>
__device__ __forceinline__ void reduce12(fx::Acc96 (&acc)[12]) {
#pragma unroll
  for (int o = kL / 2, m = 6; o > 0; o >>= 1, m >>= 1) {
    if (m == 1) {  // eight lanes: three sums are added up by both lanes of a pair
#pragma unroll
      for (int k = 0; k < 3; ++k) add_lane(acc[k], acc[k], o);
      break;
    }
    const bool up = (threadIdx.x & o) != 0;
#pragma unroll
    for (int k = 0; k < m; ++k) {
      const fx::Acc96 give = up ? acc[k] : acc[k + m];
      acc[k] = up ? acc[k + m] : acc[k];
      add_lane(acc[k], give, o);
    }
  }
}

template <int BLOCK, int kL>
__global__ void __launch_bounds__(BLOCK, 512 / BLOCK)
k_forces_fx(int64_t n, Fp64Buf b, Fp64Fields f, const InstDev* __restrict__ inst, CellWs cw,
            NbrWs nw, uint32_t* err, int64_t part_totals) {
  constexpr int kRows = BLOCK / kL, kKeep = kL == 8 ? 3 : 12 / kL;
  __shared__ double sums[kRows][kSlots + 1];
  const int64_t n_fluid = nw.part[part_totals + 1], n_inv = nw.part[part_totals];
  const int64_t first = (int64_t)blockIdx.x * kRows;
  if (first >= n_fluid) return;
  const int row = threadIdx.x / kL, lane = threadIdx.x % kL;
  const int part = kL == 8 ? lane >> 1 : lane;  // which of the sums the lane keeps
  const bool live = first + row < n_fluid;
  const bool inv_i = first + row < n_inv;
  const int64_t i = live ? checked_index(nw.order[first + row], n, err) : 0;
  const InstDev& P = inst[b.inst[i]];
  uint32_t cnt = 0, na = 0, nb = 0, leads = 0;
  FxCtx C;
  C.q = ld_qpos(nw.posq + i);
  if (live) {
    cnt = checked_count(nw.count[i], nw.cap, err);
    const uint32_t parts = nw.parts[i];
    na = min(part_inv(parts), cnt);
    nb = min(part_vis(parts), cnt - na);
    leads = nw.lead[i];
    if (leads >> 31) cnt = na = nb = 0;  // an instance of k_forces_fp64's
  }
  // first walk: the largest exponents, and the largest |v_ij|
  const uint32_t u0 = inv_i ? na : 0u;  // from here on the entries see the velocities
  uint32_t eP = C.q.exps >> 16, ev = C.q.tag >> 16, eh = C.q.exps & 0xFFFFu;
  const uint32_t own = max(ev, eh);
  uint32_t em = 4095u;  // the smallest exponent of a pair (at rest too: the products of a zero
                        // come out as a unit)
  float dv = 0.f;
  const float4 vi = nw.pvel[i];
  for (uint32_t t0 = lane; t0 < cnt; t0 += 4 * kL) {  // four entries' loads in flight
    uint32_t j[4];
    uint2 m[4];
    float4 vj[4];
#pragma unroll
    for (uint32_t u = 0; u < 4; ++u) {
      const uint32_t t = t0 + u * kL;
      j[u] = t < cnt ? checked_index(nw.list[nbr_slot(n, i, t)] & kNbrIndexMask, n, err)
                     : (uint32_t)i;
    }
#pragma unroll
    for (uint32_t u = 0; u < 4; ++u) {
      m[u] = *reinterpret_cast<const uint2*>(&nw.posq[j[u]].tag);
      if (t0 + u * kL >= u0) vj[u] = nw.pvel[j[u]];
    }
#pragma unroll
    for (uint32_t u = 0; u < 4; ++u) {
      eP = max(eP, m[u].y >> 16);
      if (t0 + u * kL >= u0) {
        ev = max(ev, m[u].x >> 16);
        eh = max(eh, m[u].y & 0xFFFFu);
        const uint32_t e = max(own, max(m[u].x >> 16, m[u].y & 0xFFFFu));
        em = min(em, j[u] != (uint32_t)i ? e : 4095u);
        const float x = fabsf(vi.x - vj[u].x), y = fabsf(vi.y - vj[u].y),
                    z = fabsf(vi.z - vj[u].z);
        dv = fmaxf(dv, fmaxf(x, fmaxf(y, z)));
      }
    }
  }
#pragma unroll
  for (int o = 1; o < kL; o <<= 1) {
    eP = max(eP, __shfl_xor_sync(~0u, eP, o));
    ev = max(ev, __shfl_xor_sync(~0u, ev, o));
    eh = max(eh, __shfl_xor_sync(~0u, eh, o));
    em = min(em, __shfl_xor_sync(~0u, em, o));
    dv = fmaxf(dv, __shfl_xor_sync(~0u, dv, o));
  }
  // 2^E2 above |v_ij| + |r_ij x s| in every component: |v_ij| from its FP32
  // value (off by at most 2^-22 of the largest velocity), |s| <= 2 sqrt(3) 2^Eh
  const int E_v = (int)ev - 1022, E_h = (int)eh - 1022, E_P = (int)eP - 1022;
  const float bound = fmaf(3.5f, ldexpf(1.f, E_h), fmaf(1.0001f, dv, ldexpf(1.f, E_v - 22)));
  // (nothing moves or spins: the products' half units come out as zero)
  const bool still = (ev | eh) == 0u;
  const int E2 = still ? -1020 : max((int)(__float_as_uint(bound) >> 23) - 126, E_h + 2);
  const int E_v1 = max(E_v, E2);
  // values the scales do not cover: overflow, NaN, FP32 underflow of v_ij,
  // pairs a thousand times slower than the fastest (at that ratio the errors
  // are those of FP64; at 1e10, 1.5e-7 of a particle's pair terms)
  const bool covered = eP < 2047u && ev < 2047u && eh < 2047u && bound < 1e30f &&
                       (still || (bound > 1e-30f && E2 - ((int)em - 1022) <= 10));
  {
    C.R = pair_range(P, z_cell(P, cw.skey[i]));
    if (!covered) C.R.width = 0u;
    C.width_vv = C.R.width ? C.R.width - (kNearVV - C.R.near2) : 0u;
    const PairRec r = nw.prec[i];
    C.Ev = E_v1 + 1022;
    C.Eh = E2 - 2 + 1022;
    C.EP = (int)eP;
    C.L = E_v1 - E2;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      C.v[a] = shr(r.v[a], C.Ev - (int)(C.q.tag >> 16));
      C.h[a] = shr(r.h[a], C.Eh - (int)(C.q.exps & 0xFFFFu));
    }
    C.P = shr(r.P, C.EP - (int)(C.q.exps >> 16));
  }
  bool any_slow = false;
  // the inviscid neighbours, the viscous ones, the walls
  const uint32_t end[4] = {0u, na, na + nb, cnt};
  const int phases = __syncthreads_or(live && cnt > na + nb) ? 3 : 2;
  for (int ph = 0; ph < phases; ++ph) {
    fx::Acc96 acc[12];
    const uint32_t t0 = ph == 0 ? end[0] : (ph == 1 ? end[1] : end[2]);
    const uint32_t t1 = ph == 0 ? end[1] : (ph == 1 ? end[2] : end[3]);
    const uint32_t lead = (leads >> (8 * ph)) & 0xFFu;
    const int s3 = 3 * (int)lead, s4 = 4 * (int)lead;  // the scales of F and W
    if (!__any_sync(~0u, t0 < t1)) {  // none for this warp's particles
#pragma unroll
      for (int k = 0; k < kKeep; ++k) sums[row][12 * ph + kKeep * part + k] = 0.0;
      continue;
    }
    if (inv_i) {
      if (ph == 0)
        fx_loop<kPathII, kL>(C, nw, n, i, t0 + lane, t1, lead, err, acc, any_slow);
      else
        fx_loop<kPathIX, kL>(C, nw, n, i, t0 + lane, t1, lead, err, acc, any_slow);
    } else {
      if (ph == 0)
        fx_loop<kPathIX, kL>(C, nw, n, i, t0 + lane, t1, lead, err, acc, any_slow);
      else
        fx_loop<kPathVV, kL>(C, nw, n, i, t0 + lane, t1, lead, err, acc, any_slow);
    }
    __syncwarp();
    if (ph == 0 && __all_sync(~0u, inv_i)) {  // pairs of inviscid particles: pressure alone
#pragma unroll
      for (int k = 0; k < 3; ++k) {
#pragma unroll
        for (int o = 1; o < kL; o <<= 1) add_lane(acc[k], acc[k], o);
      }
#pragma unroll
      for (int k = 0; k < 3; k += kL) {  // sum k + lane
        fx::Acc96 mine = acc[k];
#pragma unroll
        for (int q = 1; q < kL && k + q < 3; ++q)
          if (lane == q) mine = acc[k + q];
        if (k + lane < 3) sums[row][k + lane] = mine.value(E_P - 59 - s3);
      }
      continue;
    }
    reduce12<kL>(acc);
    // the units of the sums: the pressure's, the interfacial force's (unlike
    // species) or the part along e_ij's, that along u_ij's, the torque's
    const bool unlike = inv_i ? ph > 0 : ph == 0;
    const int eu = unlike ? E2 - 80 - s4 : E2 - 83 - s3;
#pragma unroll
    for (int k = 0; k < kKeep; ++k) {
      const int q = kKeep * part + k;
      const int e = q < 3 ? E_P - 59 - s3 : (q < 6 ? (unlike ? -60 - s3 : eu) : (q < 9 ? eu : eu - 1));
      sums[row][12 * ph + q] = acc[k].value(e);
    }
  }
#pragma unroll
  for (int k = 0; k < kKeep; ++k) sums[row][36 + kKeep * part + k] = 0.0;
  __syncwarp();
  if (__any_sync(~0u, any_slow)) {  // the FP64 route
#pragma unroll
    for (int o = 1; o < kL; o <<= 1) any_slow |= __shfl_xor_sync(~0u, (int)any_slow, o) != 0;
    if (any_slow) {  // (the same in all lanes of the row)
      double slow[12];
      for (int k = 0; k < 12; ++k) slow[k] = 0.0;
      slow_walk<kL>(n, i, cnt, inv_i ? cnt : na, &b, &P, &nw, &C, slow);
      if (lane == 0)
        for (int k = 0; k < 12; ++k) sums[row][36 + k] = slow[k];
    }
  }
  __syncthreads();
  // one thread per particle: the coefficients of the sums
  if (threadIdx.x >= kRows || first + threadIdx.x >= n_fluid) return;
  const double* S = sums[threadIdx.x];
  const int64_t io = checked_index(nw.order[first + threadIdx.x], n, err);
  const bool inv_o = first + threadIdx.x < n_inv;
  const InstDev& Q = inst[b.inst[io]];
  if (!Q.fx_pairs) return;
  const uint32_t fl = Q.flags;
  const double m_i = inv_o ? Q.m_s : Q.m_n, V_i = b.vel[io].w, two_h = 2.0 * Q.h;
  const double mc = (fl & SPH_TERM_P) ? m_i * Q.cF * two_h : 0.0;
  const double cPs = mc * Q.m_s, cPn = mc * Q.m_n;
  const double VF = V_i * Q.cF / Q.aD;  // V_i cF over the unit of the stored volumes
  const double A = (fl & SPH_TERM_SH) ? Q.A : 0.0, B = (fl & SPH_TERM_ROT) ? Q.B : 0.0;
  const double cX = (fl & SPH_TERM_T) ? Q.C_T * VF * two_h : 0.0;
  const double cXz = (fl & SPH_HPROJ) ? 0.0 : cX;
  const double cN = (fl & SPH_TERM_SN) ? -Q.C_l * V_i : 0.0;
  const double cE = (B - A) * VF, cB = -B * VF;
  double F[3], T[3], Fw[3] = {0.0, 0.0, 0.0}, Tw[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    F[a] = S[36 + a];
    T[a] = S[39 + a];
    if (inv_o) {
      F[a] = fma(cPs, S[a], F[a]);
    } else {
      F[a] = fma(cPs, S[a], fma(a < 2 ? cX : cXz, S[3 + a], fma(cN, S[6 + a], F[a])));
      T[a] = fma(-Q.h * cN, S[9 + a], T[a]);
    }
    // the viscous neighbours, then the walls
    const double c3 = inv_o ? (a < 2 ? cX : cXz) : cE, c6 = inv_o ? cN : cB;
    F[a] = fma(cPn, S[12 + a], fma(c3, S[15 + a], fma(c6, S[18 + a], F[a])));
    T[a] = fma(-Q.h * c6, S[21 + a], T[a]);
    if (phases == 3) {
      Fw[a] = fma(cPn, S[24 + a], fma(c3, S[27 + a], c6 * S[30 + a]));
      Tw[a] = -Q.h * c6 * S[33 + a];
      F[a] += Fw[a];
      T[a] += Tw[a];
    }
    Fw[a] += S[42 + a];
    Tw[a] += S[45 + a];
  }
  const double inv_m = 1.0 / m_i, inv_I = inv_o ? Q.inv_I_s : Q.inv_I_n;
  const dvec4 x = b.pos[io];
  f.acc[io] = dvec4{F[0] * inv_m, F[1] * inv_m, F[2] * inv_m, 0.0};
  f.dspin[io] = dvec4{T[0] * inv_I, T[1] * inv_I, T[2] * inv_I, 0.0};
  f.tw[io] = dvec4{x.y * Fw[2] - x.z * Fw[1] + Tw[0], x.z * Fw[0] - x.x * Fw[2] + Tw[1],
                   x.x * Fw[1] - x.y * Fw[0] + Tw[2], 0.0};
  if (!finite3(F[0], F[1], F[2]) || !finite3(T[0], T[1], T[2])) latch(err, ERR_NONFINITE);
}

// ----------------------------------------------------------- load / unload

__global__ void k_load_fp64(int64_t n, Fp64Buf b, const double* __restrict__ pos,
                            const double* __restrict__ vel, const double* __restrict__ spin,
                            const uint8_t* __restrict__ sp, const InstDev* __restrict__ inst,
                            int32_t n_inst) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double s = (double)sp[i];
    b.pos[i] = dvec4{pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], s};
    b.vel[i] = dvec4{vel[3 * i], vel[3 * i + 1], vel[3 * i + 2], 0.0};
    b.spin[i] = dvec4{spin[3 * i], spin[3 * i + 1], spin[3 * i + 2], 0.0};
    b.ref[i] = dvec2{pos[3 * i], pos[3 * i + 1]};
    b.id[i] = (uint32_t)i;
    b.inst[i] = instance_of(inst, n_inst, i);
  }
}

__global__ void k_unsort_fp64(int64_t n, Fp64Buf b, Fp64Fields f, double* pos, double* vel,
                              double* spin, double* rho, double* P, double* acc,
                              double* dspin) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t o = b.id[k];
    if (pos) {
      const dvec4 p = b.pos[k];
      pos[3 * o] = p.x;
      pos[3 * o + 1] = p.y;
      pos[3 * o + 2] = p.z;
    }
    if (vel) {
      const dvec4 v = b.vel[k];
      vel[3 * o] = v.x;
      vel[3 * o + 1] = v.y;
      vel[3 * o + 2] = v.z;
    }
    if (spin) {
      const dvec4 w = b.spin[k];
      spin[3 * o] = w.x;
      spin[3 * o + 1] = w.y;
      spin[3 * o + 2] = w.z;
    }
    if (rho) rho[o] = f.rho[k];
    if (P) P[o] = f.P[k];
    if (acc) {
      const dvec4 a = f.acc[k];
      acc[3 * o] = a.x;
      acc[3 * o + 1] = a.y;
      acc[3 * o + 2] = a.z;
    }
    if (dspin) {
      const dvec4 a = f.dspin[k];
      dspin[3 * o] = a.x;
      dspin[3 * o + 1] = a.y;
      dspin[3 * o + 2] = a.z;
    }
  }
}

}  // namespace

cudaError_t launch_kick_drift_fp64(int64_t n, const Fp64Buf& b, const Fp64Fields& f,
                                   const InstDev* inst, const InstState* ist,
                                   const CellWs& cw, uint32_t* err, int mode,
                                   cudaStream_t s, const LaunchCfg& lc, int* launches) {
  k_kick_drift_fp64<<<grid_for(n, 256, lc.sm_count, 32), 256, 0, s>>>(n, b, f, inst, ist, cw,
                                                                       err, mode);
  if (launches) ++*launches;
  return cudaGetLastError();
}

cudaError_t launch_reorder_fp64(int64_t n, const Fp64Buf& src, const Fp64Buf& dst,
                                const CellWs& cw, const NbrWs& nw, const InstDev* inst,
                                cudaStream_t s, const LaunchCfg& lc, int* launches) {
  k_reorder_fp64<<<grid_for(n, 256, lc.sm_count, 32), 256, 0, s>>>(n, src, dst, cw, nw, inst);
  if (launches) ++*launches;
  return cudaGetLastError();
}

cudaError_t launch_density_fp64(int64_t n, const Fp64Buf& b, const Fp64Fields& f,
                                const InstDev* inst, const CellWs& cw, const NbrWs& nw,
                                uint32_t* err, cudaStream_t s, const LaunchCfg& lc,
                                int* launches) {
  const auto blocks = [&](int t) { return (unsigned)((n * kLanes + t - 1) / t); };
  auto go = [&](auto filter) {
    constexpr bool F = decltype(filter)::value;
    if (lc.block_density == 32)
      k_density_fp64<32, F><<<blocks(32), 32, 0, s>>>(n, b, f, inst, cw, nw, err);
    else if (lc.block_density == 64)
      k_density_fp64<64, F><<<blocks(64), 64, 0, s>>>(n, b, f, inst, cw, nw, err);
    else
      k_density_fp64<128, F><<<blocks(128), 128, 0, s>>>(n, b, f, inst, cw, nw, err);
  };
  if (lc.any_filter)
    go(std::true_type());
  else
    go(std::false_type());
  if (launches) ++*launches;
  return cudaGetLastError();
}

cudaError_t launch_forces_fp64(int64_t n, const Fp64Buf& b, const Fp64Fields& f,
                               const InstDev* inst, const CellWs& cw, const NbrWs& nw,
                               uint32_t* err, cudaStream_t s, const LaunchCfg& lc,
                               int* launches) {
  // the species partition of the fluid particles, then the pair pass over it
  const int64_t nt = part_tiles(n);
  cudaError_t e = launch_partition(n, Fp64Species{cw.skey, f}, nw, s, launches);
  if (e != cudaSuccess) return e;
  const unsigned g256 = (unsigned)((n + 255) / 256), g128 = (unsigned)((n + 127) / 128),
                 g64 = (unsigned)((n + 63) / 64);
  // each instance's pairs by one of the two passes, by its own parameters (so
  // that a batched instance's bits equal its solo run's)
  if (lc.any_fixed) {
    k_pair_records<<<grid_for(n, 256, lc.sm_count, 32), 256, 0, s>>>(n, b, inst, nw);
    auto fixed = [&](auto lanes) {
      constexpr int L = decltype(lanes)::value;
      const auto blocks = [&](int t) { return (unsigned)((n * L + t - 1) / t); };
      if (lc.block_forces == 256)
        k_forces_fx<256, L><<<blocks(256), 256, 0, s>>>(n, b, f, inst, cw, nw, err, 2 * nt);
      else if (lc.block_forces == 64)
        k_forces_fx<64, L><<<blocks(64), 64, 0, s>>>(n, b, f, inst, cw, nw, err, 2 * nt);
      else
        k_forces_fx<128, L><<<blocks(128), 128, 0, s>>>(n, b, f, inst, cw, nw, err, 2 * nt);
    };
    if (n < kPairLanes8)
      fixed(std::integral_constant<int, 8>());
    else if (n < kPairLanes4)
      fixed(std::integral_constant<int, 4>());
    else
      fixed(std::integral_constant<int, 2>());
    if (launches) *launches += 2;
  }
  if (lc.any_loops) {
    auto go = [&](auto kopt) {
      constexpr int O = decltype(kopt)::value;
      if (lc.block_forces == 256)
        k_forces_fp64<256, O><<<g256, 256, 0, s>>>(n, b, f, inst, cw, nw, err, 2 * nt);
      else if (lc.block_forces == 64)
        k_forces_fp64<64, O><<<g64, 64, 0, s>>>(n, b, f, inst, cw, nw, err, 2 * nt);
      else
        k_forces_fp64<128, O><<<g128, 128, 0, s>>>(n, b, f, inst, cw, nw, err, 2 * nt);
    };
    // the loops carry only the options some instance uses
    const int opt = (lc.any_literal ? kOptLiteral : 0) | (lc.any_collision ? kOptCollision : 0);
    if (opt == 0)
      go(std::integral_constant<int, 0>());
    else if (opt == kOptCollision)
      go(std::integral_constant<int, kOptCollision>());
    else  // the literal F_sn, with or without collisions
      go(std::integral_constant<int, kOptLiteral | kOptCollision>());
    if (launches) ++*launches;
  }
  return cudaGetLastError();
}

cudaError_t launch_pfilter_fp64(int64_t n, const Fp64Buf& b, const Fp64Fields& f,
                                const InstDev* inst, const NbrWs& nw, uint32_t* err,
                                cudaStream_t s, int* launches) {
  k_pfilter_fp64<128><<<(unsigned)((n + 127) / 128), 128, 0, s>>>(n, b, f, inst, nw, err);
  if (launches) ++*launches;
  return cudaGetLastError();
}

cudaError_t launch_kick_fp64(int64_t n, const Fp64Buf& b, const Fp64Fields& f,
                             const InstDev* inst, cudaStream_t s, const LaunchCfg& lc,
                             int* launches) {
  k_kick_fp64<<<grid_for(n, 256, lc.sm_count, 32), 256, 0, s>>>(n, b, f, inst);
  if (launches) ++*launches;
  return cudaGetLastError();
}

cudaError_t launch_unsort_fp64(int64_t n, const Fp64Buf& b, const Fp64Fields& f,
                               double* pos, double* vel, double* spin, double* rho,
                               double* P, double* acc, double* dspin, cudaStream_t s,
                               const LaunchCfg& lc) {
  k_unsort_fp64<<<grid_for(n, 256, lc.sm_count, 32), 256, 0, s>>>(n, b, f, pos, vel, spin, rho,
                                                                   P, acc, dspin);
  return cudaGetLastError();
}

cudaError_t launch_load_fp64(int64_t n, const Fp64Buf& b, const double* pos,
                             const double* vel, const double* spin, const uint8_t* sp,
                             const InstDev* inst, int32_t n_inst, cudaStream_t s,
                             const LaunchCfg& lc) {
  k_load_fp64<<<grid_for(n, 256, lc.sm_count, 32), 256, 0, s>>>(n, b, pos, vel, spin, sp, inst,
                                                                 n_inst);
  return cudaGetLastError();
}

}  // namespace sphgb
