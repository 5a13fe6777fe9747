// The fused stream/collide kernel of one population storage format and
// number of nodes per thread.  This file is compiled once per format
// (LBM_COLLIDE_STORAGE = LBM_FP32, LBM_FP16_SHIFT, LBM_BF16_SHIFT) and nodes
// per thread (LBM_COLLIDE_NODES = 1, 2), so that the instances of the kernel
// (species count, walls, charge, diagnostics) build in parallel; each object
// defines collide_dispatch<LBM_COLLIDE_STORAGE, LBM_COLLIDE_NODES>.
#include "lbm_lattice.cuh"

#if !defined(LBM_COLLIDE_STORAGE) || !defined(LBM_COLLIDE_NODES)
#error "compile with -DLBM_COLLIDE_STORAGE=<storage code> -DLBM_COLLIDE_NODES=<1 or 2>"
#endif

namespace lbm_gb300 {
namespace {

// ---------------------------------------------------------------------------
// Fused stream + collide, all S species of a thread's nodes in registers.
//   1. pull the 19*S populations f_p^alpha(r, t), as deviations from
//      w_p n_ref                                            (Eq. latboeq, lhs)
//   2. n^alpha, bare u^alpha = sum c f / n, barycentric u   (Sec. 3 definitions)
//   3. F^alpha = F_el + F_drag: electric z(-c_s^2 grad psi + E) and the drag
//      -omega_drag sum_beta (n_beta/n)(u^a - u^b) on velocities shifted by
//      half the electric acceleration                       (Sec. 2)
//   4. f* = f - omega_visc (f - phi_perp) + g_p              (Eq. latboeq, rhs)
//      phi_perp in its reduced form n w [1 + 3 a + 4.5 a^2 - 1.5 |u^a|^2],
//      a = u^a . c (algebraically equal to the Appendix expression);
//      g_p = n w [3 F.c + 9 (F.c)(u.c) - 3 F.u]             (Eq. ourforc)
//   5. store f* at r.
//   6. (DIAG) FP64 diagnostics of the state after the step (Sec. 3: species
//      continuity, total momentum): every stored value is pulled by exactly
//      one fluid node at the next step (by r + c_p, or by r itself in the
//      opposite direction when r + c_p is a wall node), so the sums of the
//      stored values give the next state's species masses, and the stored
//      values signed by the direction they are pulled in give its momentum.
//      Per CTA: the deviation sums (FP32 over 32 nodes, FP64 over more) and
//      a count of densities (of a node and species) entering the step that
//      were not finite and positive, written to a[blockIdx.x * DIAG_NQ + k].
// ---------------------------------------------------------------------------
// NV nodes per thread (V<NV>, lbm_lattice.cuh): one in FP32, two consecutive
// x nodes in the 16-bit formats when nx is even.  The 16-bit kernel is bound
// by instruction issue and by the latency between its instructions, not by
// HBM: with two nodes the arithmetic issues packed FP32 instructions, the
// populations wait in registers as packed pairs, addresses are formed once
// per pair and directions without an x component move as one word
// (ternary 128^3, FP16: 1.10e8 -> 6.7e7 warp instructions, 122.6 -> 106 us a
// launch; with wall planes 153 -> 124 us).  In FP32 two nodes
// per thread need over 200 registers: 8 warps per SM instead of 16, 234 us
// against 180, and a form that landed the next tile in shared memory behind
// the arithmetic 223 us, so FP32 keeps one node.
//
// Charge scatter: the target of a stored population h*_p(r) is r + c_p
// (it is pulled there at the next step).  Targets are grouped by their row
// offset (dy, dz) = (c_y, c_z), nine groups; GRP numbers them.  Five groups
// also hold directions with an x component (dy = 0 or dz = 0); XGRP numbers
// those.  Per node: q0[GRP] sums the contributions to (x, y + dy, z + dz),
// qp[XGRP] those to x + 1, qm[XGRP] those to x - 1.
__host__ __device__ __forceinline__ constexpr int GRP(int p) { return (CZ(p) + 1) * 3 + (CY(p) + 1); }
__host__ __device__ __forceinline__ constexpr int XGRP_OF(int dy, int dz) {
  return dz == 0 ? (dy == 0 ? 0 : (dy == 1 ? 1 : 2)) : (dz == 1 ? 3 : 4);
}
__host__ __device__ __forceinline__ constexpr int XGRP(int p) { return XGRP_OF(CY(p), CZ(p)); }
// group of XGRP j
__host__ __device__ __forceinline__ constexpr int GRP_OF_X(int j) {
  return j == 0 ? 4 : (j == 1 ? 5 : (j == 2 ? 3 : (j == 3 ? 7 : 1)));
}

struct Scat {
  float q0[9], qp[5], qm[5];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int g = 0; g < 9; ++g) q0[g] = 0.f;
#pragma unroll
    for (int g = 0; g < 5; ++g) qp[g] = qm[g] = 0.f;
  }
  // (p is a constant once the direction loops are unrolled, so the sums stay
  // in registers)
  __device__ __forceinline__ void add(int p, float kw, float h) {
    float& q = CX(p) == 0 ? q0[GRP(p)] : (CX(p) == 1 ? qp[XGRP(p)] : qm[XGRP(p)]);
    q = fmaf(kw, h, q);
  }
};

// A warp holds 32 consecutive nodes of one x row (nx is a multiple of 32).
// Per target group (dy, dz) a lane adds the contributions that reach its own
// x: its own ones with c_x = 0, those of lane - 1 with c_x = +1 and of
// lane + 1 with c_x = -1 (register shuffles); rows of one warp wrap inside
// the warp, and for wider rows the first and last lane send the
// contributions that cross into the neighbouring warp themselves.  Each
// sum goes to the next step's source with one 64-bit integer atomic per
// target (exact, so the order in which warps add does not matter; the
// FP32 sums are formed in a fixed order, so every run gives the same
// source).  The node's own target also receives the reference part of the
// source, once per node.  (x, y, z): the lane's node.
__device__ __forceinline__ void scatter_charge(const StepArgs& a, int x, int y, int z, Scat& c) {
  const int lane = threadIdx.x & 31;
  const int nx = a.nx, ny = a.ny, nz = a.nz;
  const bool one = nx == 32;  // the row is this warp: the shuffles wrap it
#pragma unroll
  for (int j = 0; j < 5; ++j) {
    const float fl = __shfl_sync(0xffffffffu, c.qp[j], (lane + 31) & 31);  // lane - 1 sends to x
    const float fr = __shfl_sync(0xffffffffu, c.qm[j], (lane + 1) & 31);   // lane + 1 sends to x
    if (one || lane != 0) c.q0[GRP_OF_X(j)] += fl;
    if (one || lane != 31) c.q0[GRP_OF_X(j)] += fr;
  }
  unsigned long long* acc = reinterpret_cast<unsigned long long*>(a.scat_acc);
  const int ym = y == 0 ? ny - 1 : y - 1, yp = y == ny - 1 ? 0 : y + 1;
  const int zm = z == 0 ? nz - 1 : z - 1, zp = z == nz - 1 ? 0 : z + 1;
  const int64_t nxy = (int64_t)nx * ny;
  const int64_t rowz[3] = {(int64_t)zm * nxy, (int64_t)z * nxy, (int64_t)zp * nxy};
  const int rowy[3] = {ym * nx, y * nx, yp * nx};
#pragma unroll
  for (int g = 0; g < 9; ++g) {
    unsigned long long q = scat_fixed(c.q0[g]);
    if (g == 4) q += (unsigned long long)a.src_ref;
    atomicAdd(acc + rowz[g / 3] + rowy[g % 3] + x, q);
  }
  if (!one && (lane == 0 || lane == 31)) {
    // the contributions that cross into the neighbouring warp of the row
    const int xt = lane == 0 ? (x == 0 ? nx - 1 : x - 1) : (x == nx - 1 ? 0 : x + 1);
#pragma unroll
    for (int j = 0; j < 5; ++j)
      atomicAdd(acc + rowz[GRP_OF_X(j) / 3] + rowy[GRP_OF_X(j) % 3] + xt,
                scat_fixed(lane == 0 ? c.qm[j] : c.qp[j]));
  }
}

// r + x, node by node: the packed form of r + r * y comes out fused.
template <int NV>
__device__ __forceinline__ V<NV> add_scalar(float r, const V<NV>& x) {
  V<NV> v;
#pragma unroll
  for (int k = 0; k < NV; ++k) v.set(k, __fadd_rn(r, x.get(k)));
  return v;
}

// x * y, formed here even if it was formed before: for one node per thread a
// value kept from the moments to the update would hold a register in the
// part of the kernel that has none to spare (ternary 128^3, FP32 with the
// charge scatter: 172 us a launch with the product kept, 162 with it formed
// again).
__device__ __forceinline__ V<1> mul_here(V<1> x, V<1> y) {
  float r;
  asm volatile("mul.rn.f32 %0, %1, %2;" : "=f"(r) : "f"(x.a), "f"(y.a));
  return r;
}
__device__ __forceinline__ V<2> mul_here(V<2> x, V<2> y) { return x * y; }

// c . v for the direction p (a constant once unrolled): additions only.
template <int NV>
__device__ __forceinline__ V<NV> cdot(int p, const V<NV>& x, const V<NV>& y, const V<NV>& z) {
  const int c[3] = {CX(p), CY(p), CZ(p)};
  const V<NV>* v[3] = {&x, &y, &z};
  V<NV> r;
  bool first = true;
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    if (c[d] == 0) continue;
    // every odd p has its first non-zero component positive or its pair has
    if (first) r = c[d] > 0 ? *v[d] : V<NV>(0.f) - *v[d];
    else r = c[d] > 0 ? r + *v[d] : r - *v[d];
    first = false;
  }
  return r;
}

// Deviation sums of the state after the step over a thread's nodes.
template <int S>
struct Sums {
  float m[S], jx, jy, jz, bad;
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int s = 0; s < S; ++s) m[s] = 0.f;
    jx = jy = jz = bad = 0.f;
  }
};

// The pulled populations of a thread as they came from memory: floats, or
// for two nodes of a 16-bit format the packed pair (half the registers of
// the unpacked ones; unpacked where it is used, once for the moments and
// once for the update).
template <int ST, int NV>
struct Raw {
  V<NV> v;
  __device__ __forceinline__ V<NV> get() const { return v; }
  __device__ __forceinline__ void clear(int k) { v.set(k, 0.f); }
};
template <>
struct Raw<LBM_FP16_SHIFT, 2> {
  uint32_t v;
  __device__ __forceinline__ V<2> get() const { return Fmt<LBM_FP16_SHIFT>::unpack(v); }
  __device__ __forceinline__ void clear(int k) { v &= k ? 0x0000ffffu : 0xffff0000u; }
};
template <>
struct Raw<LBM_BF16_SHIFT, 2> {
  uint32_t v;
  __device__ __forceinline__ V<2> get() const { return Fmt<LBM_BF16_SHIFT>::unpack(v); }
  __device__ __forceinline__ void clear(int k) { v &= k ? 0x0000ffffu : 0xffff0000u; }
};

// Population (s, p): the base address is the same for the whole warp, the
// node's byte offset one 32-bit number (a plane of 2^30 nodes is at most
// 2^32 bytes).
template <class T>
__device__ __forceinline__ const T* pop_at(const void* base, int64_t plane, uint32_t off) {
  return reinterpret_cast<const T*>(static_cast<const char*>(base) + plane * (int64_t)sizeof(T) + off);
}

// Gradient of psi along one axis at a node: mean of the two face gradients,
// each an exact integer difference, rounded once (a step of psi up to 2^11
// per face).  At a wall face the node's own value takes the neighbour's
// place and the Neumann value of the surface-charge condition is in the wall
// part w (k_wall_gradient).  The conversions issue on the FP64 pipe, six per
// node: the difference over two nodes, rounded once, would need three (128^3
// with wall planes 165 -> 155 us a launch), but rounds otherwise and wraps at
// half the step; joining two exact 32-bit pieces instead (157 us there) was
// slower without walls (with the scatter 166 against 162 us, FP16 114
// against 106).
template <bool WALLS>
__device__ __forceinline__ float axis_gradient(int64_t c, int64_t m, int64_t p, uint32_t wm, uint32_t wp,
                                               float w) {
  if (WALLS) {
    p = wp ? c : p;
    m = wm ? c : m;
  }
  return fmaf((float)(p - c) + (float)(c - m), 0.5f * PSI_INV_SCALE_F, w);
}

// Potential of NV consecutive nodes.
template <int NV>
__device__ __forceinline__ void ld_psi(const int64_t* __restrict__ p, int64_t (&v)[NV]) {
  if constexpr (NV == 1) {
    v[0] = *p;
  } else {
    const longlong2 w = *reinterpret_cast<const longlong2*>(p);
    v[0] = w.x;
    v[1] = w.y;
  }
}

// (link: a node of the warp has a wall node beside it)
template <int NV, bool WALLS>
__device__ __forceinline__ void psi_gradient_v(const StepArgs& a, uint32_t i, const Nbr& o,
                                               const uint32_t (&lk)[NV], bool link, V<NV>& gx,
                                               V<NV>& gy, V<NV>& gz) {
  const int64_t* __restrict__ ps = a.psi + i;
  int64_t c[NV] = {}, yp[NV], ym[NV], zp[NV], zm[NV];
  ld_psi<NV>(ps, c);
  ld_psi<NV>(ps + o.dyp, yp);
  ld_psi<NV>(ps + o.dym, ym);
  ld_psi<NV>(ps + o.dzp, zp);
  ld_psi<NV>(ps + o.dzm, zm);
  const int64_t xl = ps[o.dxm], xr = ps[NV - 1 + o.dxp];
  V<NV> w[3] = {0.f, 0.f, 0.f};
  if (WALLS && link && a.wallg) {
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
      for (int k = 0; k < NV; ++k) w[d].set(k, a.wallg[(int64_t)d * a.N + i + k]);
  }
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    // bit 2: r + x is a wall node; bit 1: r - x; 4: +y; 3: -y; 6: +z; 5: -z
    const uint32_t l = lk[k];
    const int64_t m = k == 0 ? xl : c[0], p = k == NV - 1 ? xr : c[NV - 1];
    gx.set(k, axis_gradient<WALLS>(c[k], m, p, l & 2u, l & 4u, w[0].get(k)));
    gy.set(k, axis_gradient<WALLS>(c[k], ym[k], yp[k], l & 8u, l & 16u, w[1].get(k)));
    gz.set(k, axis_gradient<WALLS>(c[k], zm[k], zp[k], l & 32u, l & 64u, w[2].get(k)));
  }
}

// The step's roundings are all written out (no multiplication and addition
// that the compiler may or may not contract), so that one and two nodes per
// thread and every instance round alike, and so that runs repeat the results
// of earlier versions of the library bit for bit: near the tolerance of the
// Poisson solve one rounding decides how many applications a step takes,
// which the records hold.  Three places keep a contraction that only some
// instances had:
//   total    the densities in the sum over species, charged beside walls
//   density  the fourth species' density, neutral and periodic in FP32
//   drag     the mean velocity of a single species in its own drag
template <int S, bool WALLS, bool CHARGED, int ST, bool DIAG, bool PAIR>
struct Fused {
  static constexpr bool total = S > 1 && WALLS && CHARGED && !DIAG && !PAIR;
  static constexpr bool density3 = S == 4 && ST == LBM_FP32 && !WALLS && !CHARGED && !DIAG && !PAIR;
  static constexpr bool drag = S == 1 && !(WALLS && CHARGED);
};

// The collision of a thread's NV nodes from i on (plane z) and the stores:
// f the pulled h_p, (gx, gy, gz) the potential's gradient, lk the link words
// and act the fluid flags of the nodes.
template <int S, int NV, bool WALLS, bool CHARGED, int ST, bool DIAG, bool PAIR, bool SCAT>
__device__ __forceinline__ void collide_nodes(const StepArgs& a, uint32_t i, int z,
                                              const uint32_t (&lk)[NV], const bool (&act)[NV],
                                              const Raw<ST, NV> (&f)[S][Q], const V<NV>& gx,
                                              const V<NV>& gy, const V<NV>& gz, Scat& sc,
                                              Sums<S>& q) {
  using T = typename Fmt<ST>::T;
  using F = V<NV>;
  using FU = Fused<S, WALLS, CHARGED, ST, DIAG, PAIR>;
  T* __restrict__ fout = static_cast<T*>(a.fout) + i;
  const int64_t N = a.N;
  // n = n_ref (1 + sum w h), j = n_ref sum c w h  (sum w = 1, sum w c = 0),
  // summed per weight class (faces p = 1..6, edges 7..18) so that each
  // population costs additions only
  F mh[S], n[S], jx[S], jy[S], jz[S], ntot;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    F h[Q];
#pragma unroll
    for (int p = 0; p < Q; ++p) h[p] = f[s][p].get();
    F sf = h[1], se = h[7];
#pragma unroll
    for (int p = 2; p <= 6; ++p) sf = sf + h[p];
#pragma unroll
    for (int p = 8; p < Q; ++p) se = se + h[p];
    // edges with an x, y or z component, in the order of the directions
    const F xe = ((((((h[7] - h[8]) + h[9]) - h[10]) + h[11]) - h[12]) + h[13]) - h[14];
    const F ye = ((((((h[7] - h[8]) - h[9]) + h[10]) + h[15]) - h[16]) + h[17]) - h[18];
    const F ze = ((((((h[11] - h[12]) - h[13]) + h[14]) + h[15]) - h[16]) - h[17]) + h[18];
    mh[s] = vfma(F(WT(0)), h[0], vfma(F(WT(1)), sf, F(WT(7)) * se));
    const float r = a.nref[s];
    const F nf = vfma(F(r), mh[s], F(r));
    n[s] = FU::density3 && s == 3 ? nf : add_scalar<NV>(r, F(r) * mh[s]);
    const F nt = FU::total ? nf : n[s];
    ntot = s == 0 ? nt : ntot + nt;
    jx[s] = F(r) * vfma(F(WT(1)), h[1] - h[2], F(WT(7)) * xe);
    jy[s] = F(r) * vfma(F(WT(1)), h[3] - h[4], F(WT(7)) * ye);
    jz[s] = F(r) * vfma(F(WT(1)), h[5] - h[6], F(WT(7)) * ze);
    if (DIAG) {
#pragma unroll
      for (int k = 0; k < NV; ++k)
        if (act[k] && (!(n[s].get(k) > 0.f) || !isfinite(n[s].get(k)))) q.bad += 1.f;
    }
  }

  F Jx = jx[0], Jy = jy[0], Jz = jz[0];
#pragma unroll
  for (int s = 1; s < S; ++s) {
    Jx = Jx + jx[s];
    Jy = Jy + jy[s];
    Jz = Jz + jz[s];
  }
  const F inv_ntot = vrcp(ntot);
  // barycentric velocity (equal masses: mass-weighted = number-weighted)
  const F ux = Jx * inv_ntot, uy = Jy * inv_ntot, uz = Jz * inv_ntot;

  // field: applied minus c_s^2 grad psi
  F Ex(a.eext[0]), Ey(a.eext[1]), Ez(a.eext[2]);
  if (CHARGED) {
    Ex = vfma(F(-CS2), gx, Ex);
    Ey = vfma(F(-CS2), gy, Ey);
    Ez = vfma(F(-CS2), gz, Ez);
  }

  // number-weighted mean of the drag velocities u^a + F_el^a / 2
  F zn = F(a.valence[0]) * n[0];
#pragma unroll
  for (int s = 1; s < S; ++s) zn = vfma(F(a.valence[s]), n[s], zn);
  const F hzn = F(0.5f) * zn;
  const F vpx = vfma(hzn, Ex, Jx), vpy = vfma(hzn, Ey, Jy), vpz = vfma(hzn, Ez, Jz);
  const F vbx = vpx * inv_ntot, vby = vpy * inv_ntot, vbz = vpz * inv_ntot;
  // pair frequencies: the fractions x_b and x_b v_b of every species
  F px[PAIR ? S : 1], pxv[PAIR ? S : 1][3];
  if (PAIR) {
#pragma unroll
    for (int b = 0; b < S; ++b) {
      px[b] = n[b] * inv_ntot;
      const F hz = F(0.5f * a.valence[b]) * n[b];
      pxv[b][0] = vfma(hz, Ex, jx[b]) * inv_ntot;
      pxv[b][1] = vfma(hz, Ey, jy[b]) * inv_ntot;
      pxv[b][2] = vfma(hz, Ez, jz[b]) * inv_ntot;
    }
  }

  const float om = a.omega_visc;
  const float omd = a.omega_drag_z ? a.omega_drag_z[z] : a.omega_drag;
  uint32_t rnd[NV];
  if (ST != LBM_FP32) {
    const uint32_t st = mix32(a.step_dev ? *a.step_dev : a.step);
#pragma unroll
    for (int k = 0; k < NV; ++k) rnd[k] = mix32((i + k) * 0x9E3779B9u ^ st);
  }
  auto next = [&](int k) -> uint32_t { return ST != LBM_FP32 ? lcg_next(rnd[k]) : 0u; };
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const F inv_n = vrcp(n[s]);
    const F usx = jx[s] * inv_n, usy = jy[s] * inv_n, usz = jz[s] * inv_n;
    // force per unit mass (Sec. 2): the electric acceleration and the drag
    // on the velocities shifted by half of it
    const F zs(a.valence[s]);
    F Fx, Fy, Fz;
    {
      const F ex = zs * Ex, ey = zs * Ey, ez = zs * Ez, half(0.5f);
      const F vx = vfma(half, ex, usx), vy = vfma(half, ey, usy), vz = vfma(half, ez, usz);
      if (PAIR) {
        // F_drag^a = -(W v_a - M), W = sum_b omega^{ab} x_b,
        // M = sum_b omega^{ab} x_b v_b (omega^{aa} = 0)
        F W(0.f), Mx(0.f), My(0.f), Mz(0.f);
#pragma unroll
        for (int b = 0; b < S; ++b) {
          const F w(a.pair[s][b]);
          W = vfma(w, px[b], W);
          Mx = vfma(w, pxv[b][0], Mx);
          My = vfma(w, pxv[b][1], My);
          Mz = vfma(w, pxv[b][2], Mz);
        }
        Fx = ex + vfma(F(0.f) - W, vx, Mx);
        Fy = ey + vfma(F(0.f) - W, vy, My);
        Fz = ez + vfma(F(0.f) - W, vz, Mz);
      } else {
        Fx = vfma(F(omd), FU::drag ? vfma(vpx, inv_ntot, F(0.f) - vx) : vbx - vx, ex);
        Fy = vfma(F(omd), FU::drag ? vfma(vpy, inv_ntot, F(0.f) - vy) : vby - vy, ey);
        Fz = vfma(F(omd), FU::drag ? vfma(vpz, inv_ntot, F(0.f) - vz) : vbz - vz, ez);
      }
    }
    const F usq = vfma(usz, usz, vfma(usx, usx, usy * usy));
    const F Fu = vfma(Fz, uz, vfma(Fx, ux, Fy * uy));
    // In deviations, d*_p = (1 - omega) d_p + [omega phi_p + g_p - omega w_p n_ref]
    // with, per weight w_p,
    //   omega phi_p + g_p - omega w_p n_ref
    //     = w_p [omega dn + n (-1.5 omega |u^a|^2 - 3 F.u
    //                          + 4.5 omega a^2 + 9 (F.c)(u.c))]      (even in c)
    //     + w_p n 3 (omega a + F.c)                                 (odd in c)
    // a = u^a.c (phi_perp in its reduced form, the Appendix expression;
    // g_p of Eq. ourforc).  Divided by w_p n_ref this updates the stored
    // h = d / (w_p n_ref) directly: h*_p = (1 - omega) h_p + (even' +/- odd') / n_ref,
    // with the bracket values even', odd' free of w_p.  Every term is of
    // the size of the deviations.
    const float inr = 1.0f / a.nref[s];
    // the per-species factors of the bracket values, once per species:
    // even' = Ce + Ae a^2 + Be (F.c)(u.c), odd' = Dom a + Do F.c
    const F nin = n[s] * F(inr);
    const F Ae = nin * F(4.5f * om), Be = nin * F(9.0f), Do = nin * F(3.0f), Dom = Do * F(om);
    const F dn = mul_here(F(a.nref[s]), mh[s]), base = vfma(F(-1.5f * om), usq, F(-3.0f) * Fu);
    const F Ce = F(inr) * (PAIR ? vfma(n[s], base, F(om) * dn) : vfma(F(om), dn, n[s] * base));
    // moving populations first; the rest population then takes
    // d*_0 = dn - sum_{p>0} d*_p over the stored (rounded) moving values,
    // i.e. h*_0 = (sum w h - sum_{p>0} w h*_p) / w_0, which holds exactly
    // in real arithmetic (phi_perp carries mass n, g_p none) and keeps the
    // rounding of the weights and of 16-bit stores from drifting the
    // species mass.
    // Directions come in opposite pairs (p, p+1), c_{p+1} = -c_p: a = u^a.c,
    // F.c and u.c flip sign, so each pair shares the even part and takes
    // +/- the odd part.
    const F omm(1.0f - om);
    F moved(0.f);  // stored values, weighted and summed
    float mjx = 0.f, mjy = 0.f, mjz = 0.f;
#pragma unroll
    for (int p = 1; p < Q; p += 2) {
      const F av = cdot<NV>(p, usx, usy, usz);
      const F fc = cdot<NV>(p, Fx, Fy, Fz);
      const F uc = cdot<NV>(p, ux, uy, uz);
      const F even = vfma(Ae, av * av, vfma(Be, fc * uc, Ce));
      const F odd = vfma(Dom, av, Do * fc);
      F ha = vfma(omm, f[s][p].get(), even + odd), hb = vfma(omm, f[s][p + 1].get(), even - odd);
      T* pa = fout + (int64_t)(s * Q + p) * N;
      if constexpr (NV == 2) {
        Fmt<ST>::sth_sr22(pa, ha.a, pa + N, hb.a, next(0), next(1));
      } else {
        const float2 hs = Fmt<ST>::sth_sr2(pa, ha.a, pa + N, hb.a, next(0));
        ha = hs.x;
        hb = hs.y;
      }
      moved = vfma(F(WT(p)), ha + hb, moved);  // same weight for p and p + 1
      if constexpr (SCAT) {
        // charge these stored values carry to r + c_p and r - c_p
        // (zero for a neutral species)
        const float kw = a.scat_k[s] * WT(p);
        sc.add(p, kw, ha.a);
        sc.add(p + 1, kw, hb.a);
      }
      // momentum carried by the pair at the next step: h*_p moves along
      // c_p unless r + c_p is a wall node (bit p+1), then it is pulled
      // back along -c_p; h*_{p+1} likewise with bit p
      if (DIAG) {
        float mj = 0.f;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          if (WALLS) {
            if (act[k])
              mj += (((lk[k] >> (p + 1)) & 1u) ? -ha.get(k) : ha.get(k)) -
                    (((lk[k] >> p) & 1u) ? -hb.get(k) : hb.get(k));
          } else {
            mj += ha.get(k) - hb.get(k);
          }
        }
        if (CX(p)) mjx += CX(p) * WT(p) * mj;
        if (CY(p)) mjy += CY(p) * WT(p) * mj;
        if (CZ(p)) mjz += CZ(p) * WT(p) * mj;
      }
    }
    F h0 = (mh[s] - moved) * F(INV_WT(0));
    T* p0 = fout + (int64_t)(s * Q) * N;
    if constexpr (NV == 2) Fmt<ST>::sth_sr_pair(p0, h0.a, next(0), next(1));
    else h0 = Fmt<ST>::sth_sr(p0, h0.a, next(0));
    if constexpr (SCAT) sc.add(0, a.scat_k[s] * WT(0), h0.a);
    if (DIAG) {
      const float r = a.nref[s];
#pragma unroll
      for (int k = 0; k < NV; ++k)
        if (act[k]) q.m[s] += r * fmaf(WT(0), h0.get(k), moved.get(k));
      q.jx += r * mjx;
      q.jy += r * mjy;
      q.jz += r * mjz;
    }
  }
}

// The diagnostics sums of a thread as the DIAG_NQ quantities of the partials.
template <int S>
__device__ __forceinline__ void diag_quantities(const StepArgs& a, const Sums<S>& q,
                                                float (&v)[DIAG_NQ]) {
#pragma unroll
  for (int k = 0; k < DIAG_NQ; ++k) v[k] = 0.f;
  float qc = 0.f;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    v[s] = q.m[s];
    qc += a.valence[s] * q.m[s];
  }
  v[MAX_SPECIES + 0] = q.jx;
  v[MAX_SPECIES + 1] = q.jy;
  v[MAX_SPECIES + 2] = q.jz;
  v[MAX_SPECIES + 3] = qc;
  v[MAX_SPECIES + 4] = q.bad;
}

// Registers: up to 128 per thread (16 warps per SM), 255 for four species.
// Two nodes per thread of three species: 168 (12 warps); in a sweep ternary
// 128^3 FP16 took 102 us with 168 in ncu, 123 with 128 (spills), 108 with 144;
// 64 slits 271 us with 168, 331 with 200, 322 with 255.  One node per
// thread of three species in 16 bits (odd nx), bound by instruction issue
// and not by HBM: 92, 20 warps in CTAs of 128 threads (127x128x128 FP16:
// 120 us a launch, 124.5 with 128, 126.7 with 96, 120.6 with 88; beside
// wall planes 128, 137 with 128; neutral 115, 118.5; BF16 120, 124.5).
template <int S, int NV, int ST>
constexpr int collide_maxnreg() {
  return S >= 4 ? 255 : (S < 3 ? 128 : (NV == 2 ? 168 : (ST == LBM_FP32 ? 128 : 92)));
}

template <int S, int NV, bool WALLS, bool CHARGED, int ST, bool DIAG, bool PAIR, bool SCAT>
__global__ void __launch_bounds__(256) __maxnreg__((collide_maxnreg<S, NV, ST>()))
    k_stream_collide(const StepArgs a) {
  using T = typename Fmt<ST>::T;
  // neutral lattices, whose launch need not wait for the previous kernel to
  // end (launch_one): nothing is touched before all of it is visible, and the
  // next launch may come up from here on
  if constexpr (!CHARGED) {
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
  }
  // a speculative launch the step has decided against (same for every
  // thread of the grid)
  if (a.skip && *a.skip) return;
  const uint32_t i = (blockIdx.x * blockDim.x + threadIdx.x) * NV;
  Sums<S> q;
  q.clear();
  Scat sc;  // (SCAT) charge sent to the next step's source
  if constexpr (SCAT) sc.clear();
  const bool inrange = i < (uint32_t)a.N;
  uint32_t lk[NV];
  bool act[NV], work = inrange, mixed = false;
#pragma unroll
  for (int k = 0; k < NV; ++k) lk[k] = 0u;
  if (WALLS) {
    // The class of the warp's nodes (a byte per 32 nodes, from the caches)
    // tells whether the link words matter: warps without wall nodes or wall
    // neighbours pull at once, warps of wall nodes only do nothing, and only
    // the others wait for their link words, which choose the addresses of
    // the pulls.  Wall nodes in a warp with fluid nodes run the same
    // instructions and store what they computed from zeros into their own
    // slots (which no pull reads): every store of the warp then covers whole
    // sectors, so the L2 need not fetch the rest of a sector a partial write
    // leaves (measured on the porous box: about 130 MB of DRAM reads per
    // launch at 128^3).
    const uint32_t g = (i - (threadIdx.x & 31) * NV) >> 5, gl = (uint32_t)((a.N - 1) >> 5);
    uint8_t c = a.wcls[min(g, gl)];
    if (NV == 2) {
      const uint8_t c1 = a.wcls[min(g + 1, gl)];
      c = c == c1 ? c : (uint8_t)WCLS_MIXED;
    }
    work = inrange && c != WCLS_SOLID;
    mixed = c == WCLS_MIXED;
    if (work && mixed) {
      if constexpr (NV == 2) {
        const uint2 w = *reinterpret_cast<const uint2*>(a.links + i);
        lk[0] = w.x;
        lk[1] = w.y;
      } else {
        lk[0] = a.links[i];
      }
    }
  }
#pragma unroll
  for (int k = 0; k < NV; ++k) act[k] = work && !(lk[k] & LINK_SOLID);
  if (work) {
    int x, y, z;
    site_xyz(i, a.nx, a.ny, x, y, z);
    Nbr o = neighbours(x, y, z, a.nx, a.ny, a.nz);
    if (NV == 2) o.dxp = x + 2 == a.nx ? -(a.nx - 1) : 1;  // from the second node
    const int64_t N = a.N;
    // stored h_p = (f_p - w_p n_ref) / (w_p n_ref) of every species, pulled
    // from r - c_p, or where that is a wall node from the node's own reversed
    // population (halfway bounce-back)
    Raw<ST, NV> f[S][Q];
    auto pull_all = [&]() {
#pragma unroll
      for (int p = 0; p < Q; ++p) {
        const int d = (CY(p) == 1 ? o.dym : (CY(p) == -1 ? o.dyp : 0)) +
                      (CZ(p) == 1 ? o.dzm : (CZ(p) == -1 ? o.dzp : 0));
        // upstream nodes of the thread's (first) node and of its second one
        const uint32_t o0 = (uint32_t)((int)i + d + (CX(p) == 1 ? o.dxm : (CX(p) == -1 ? (NV == 2 ? 1 : o.dxp) : 0))) *
                            (uint32_t)sizeof(T);
        const uint32_t o1 = (uint32_t)((int)i + d + (CX(p) == 1 ? 0 : 1 + (CX(p) == -1 ? o.dxp : 0))) *
                            (uint32_t)sizeof(T);
#pragma unroll
        for (int s = 0; s < S; ++s) {
          const int64_t pl = (int64_t)(s * Q + p) * N;
          if constexpr (NV == 1) {
            f[s][p].v = Fmt<ST>::ldh(pop_at<T>(a.fin, pl, o0));
          } else if (CX(p) == 0) {
            f[s][p].v = *reinterpret_cast<const uint32_t*>(pop_at<T>(a.fin, pl, o0));
          } else {
            f[s][p].v = (uint32_t)*reinterpret_cast<const unsigned short*>(pop_at<T>(a.fin, pl, o0)) |
                        (uint32_t)*reinterpret_cast<const unsigned short*>(pop_at<T>(a.fin, pl, o1)) << 16;
          }
        }
      }
    };
    // the same with the link word choosing the address: one round trip, where
    // pulls followed by the bounce-back loads took two
    auto pull_linked = [&]() {
      if constexpr (NV == 1) {
        const uint32_t wb = act[0] ? (lk[0] & ~LINK_SOLID) : 0u;
#pragma unroll
        for (int p = 0; p < Q; ++p) {
          const bool bb = p > 0 && ((wb >> p) & 1u);
          const int64_t e = bb ? (int64_t)OPP(p) * N + i
                               : (int64_t)p * N + (uint32_t)((int)i + upstream(o, p));
          const T* ptr = static_cast<const T*>(a.fin) + e;
#pragma unroll
          for (int s = 0; s < S; ++s) {
            const float h = Fmt<ST>::ldh(ptr + (int64_t)(s * Q) * N);
            f[s][p].v = V<NV>(act[0] ? h : 0.f);
          }
        }
      }
    };
    if (WALLS && NV == 1 && mixed) pull_linked();
    else pull_all();
    if constexpr (WALLS && NV == 2) {
      if (mixed) {
        // reversed values of the pair where a node is next to a wall node;
        // wall nodes compute from zeros
        const uint32_t w0 = act[0] ? (lk[0] & ~LINK_SOLID) : 0u, w1 = act[1] ? (lk[1] & ~LINK_SOLID) : 0u;
#pragma unroll
        for (int p = 1; p < Q; ++p)
          if (((w0 | w1) >> p) & 1u) {
            const uint32_t m = ((w0 >> p) & 1u ? 0x0000ffffu : 0u) | ((w1 >> p) & 1u ? 0xffff0000u : 0u);
#pragma unroll
            for (int s = 0; s < S; ++s) {
              const uint32_t r = *reinterpret_cast<const uint32_t*>(
                  static_cast<const T*>(a.fin) + (int64_t)(s * Q + OPP(p)) * N + i);
              f[s][p].v = (f[s][p].v & ~m) | (r & m);
            }
          }
#pragma unroll
        for (int k = 0; k < NV; ++k)
          if (!act[k]) {
#pragma unroll
            for (int s = 0; s < S; ++s)
#pragma unroll
              for (int p = 0; p < Q; ++p) f[s][p].clear(k);
          }
      }
    }
    V<NV> gx(0.f), gy(0.f), gz(0.f);
    if (CHARGED) psi_gradient_v<NV, WALLS>(a, i, o, lk, mixed, gx, gy, gz);
    collide_nodes<S, NV, WALLS, CHARGED, ST, DIAG, PAIR, SCAT>(a, i, z, lk, act, f, gx, gy, gz, sc, q);
    if constexpr (SCAT) scatter_charge(a, x, y, z, sc);
  }

  // per-CTA partial sums of the diagnostics (inactive threads add zeros)
  if (DIAG) {
    float v[DIAG_NQ];
    diag_quantities<S>(a, q, v);
    // 32 nodes are added in FP32, by the LANES lanes that hold them, the rest
    // in FP64
    constexpr int LANES = 32 / NV;
    __shared__ float red[256 / LANES][DIAG_NQ];
#pragma unroll
    for (int k = 0; k < DIAG_NQ; ++k) {
      if (k >= S && k < MAX_SPECIES) continue;
#pragma unroll
      for (int off = LANES / 2; off > 0; off >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], off);
      if (threadIdx.x % LANES == 0) red[threadIdx.x / LANES][k] = v[k];
    }
    __syncthreads();
    if (threadIdx.x < DIAG_NQ) {
      const int k = threadIdx.x;
      double tot = 0.0;
      if (k < S || k >= MAX_SPECIES)
        for (int w = 0; w < (int)blockDim.x / LANES; ++w) tot += (double)red[w][k];
      a.diag[(int64_t)blockIdx.x * DIAG_NQ + k] = tot;
    }
  }
}

template <int S, bool W, bool C, int ST, bool SC, bool DIAG, bool PAIR>
cudaError_t launch_one(const StepArgs& a, cudaStream_t st, int threads, int64_t* ctas) {
  constexpr int NV = LBM_COLLIDE_NODES;
  *ctas = nblocks(a.N / NV, threads);
  // A step of a neutral lattice is this one kernel.  Programmatic
  // serialisation brings up the next step's CTAs beside the last ones of this
  // step, which shortens small boxes (32^3 binary, 256 CTAs, 100 steps: 248 ->
  // 231 us); grids of more than one wave gain nothing (97x61x45, four
  // species, about seven waves: 598 against 601 us) and keep the plain launch.
  // One wave: what the registers of an SM (65536) hold at the kernel's cap.
  const int64_t one_wave = (int64_t)a.sms * (65536 / (collide_maxnreg<S, NV, ST>() * threads));
  if (!C && *ctas <= one_wave) {
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)*ctas);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_stream_collide<S, NV, W, C, ST, DIAG, PAIR, SC>, a);
  }
  k_stream_collide<S, NV, W, C, ST, DIAG, PAIR, SC><<<(unsigned)*ctas, threads, 0, st>>>(a);
  return cudaGetLastError();
}

template <int S, bool W, bool C, int ST, bool SC>
cudaError_t launch_nv(const StepArgs& a, cudaStream_t st, int threads, bool diag,
                      int64_t* ctas) {
  // the pair-frequency drag exists for three or more species (a binary
  // depends on its one cross frequency, which the host passes as omega_drag)
  constexpr bool CAN_PAIR = S >= 3;
  if (CAN_PAIR && a.pair_on)
    return diag ? launch_one<S, W, C, ST, SC, true, CAN_PAIR>(a, st, threads, ctas)
                : launch_one<S, W, C, ST, SC, false, CAN_PAIR>(a, st, threads, ctas);
  return diag ? launch_one<S, W, C, ST, SC, true, false>(a, st, threads, ctas)
              : launch_one<S, W, C, ST, SC, false, false>(a, st, threads, ctas);
}

// The charge scatter: a.scat_acc is set by the host only for charged FP32
// lattices without walls whose nx is a multiple of 32.
template <int S, bool W, bool C, int ST>
cudaError_t launch_sc(const StepArgs& a, cudaStream_t st, int threads, bool diag,
                      int64_t* ctas) {
  if constexpr (!W && C && ST == LBM_FP32) {
    if (a.scat_acc) return launch_nv<S, W, C, ST, true>(a, st, threads, diag, ctas);
  }
  return launch_nv<S, W, C, ST, false>(a, st, threads, diag, ctas);
}

template <int S, int ST>
cudaError_t dispatch_wc(const StepArgs& a, bool w, bool c, cudaStream_t st, int t, bool d,
                        int64_t* n) {
  if (w)
    return c ? launch_sc<S, true, true, ST>(a, st, t, d, n) : launch_sc<S, true, false, ST>(a, st, t, d, n);
  return c ? launch_sc<S, false, true, ST>(a, st, t, d, n) : launch_sc<S, false, false, ST>(a, st, t, d, n);
}

}  // namespace

template <>
cudaError_t collide_dispatch<LBM_COLLIDE_STORAGE, LBM_COLLIDE_NODES>(const StepArgs& a, int S, bool w,
                                                                     bool c, cudaStream_t st,
                                                                     int threads, bool d,
                                                                     int64_t* ctas) {
  constexpr int ST = LBM_COLLIDE_STORAGE;
  switch (S) {
    case 1: return dispatch_wc<1, ST>(a, w, c, st, threads, d, ctas);
    case 2: return dispatch_wc<2, ST>(a, w, c, st, threads, d, ctas);
    case 3: return dispatch_wc<3, ST>(a, w, c, st, threads, d, ctas);
    case 4: return dispatch_wc<4, ST>(a, w, c, st, threads, d, ctas);
  }
  return cudaErrorInvalidValue;
}

}  // namespace lbm_gb300
