// Heun step of Q alone, on the padded mirrors: lattices with the flow off, and
// the Q update of Gauss-Seidel coupling (with the new velocity u^{n+1}).
//
//   k_heun<CORRECT = false>  Q^n, u       -> Q* = Q + R(Q, u)
//   k_heun<CORRECT = true>   Q*, Q^n, u   -> Q^{n+1} = (Q + Q* + R(Q*, u)) / 2
// (Sec. 2.1 Eq. Qevolution, mat_der; u = 0 with the flow off)
//
// A thread owns one (x, y) position and marches through the planes of its
// z-chunk: the site and its z neighbours stay in registers, so that a site costs
// five vector loads of the stencil field (its z + 1 neighbour and the four in its
// plane, through L1) instead of seven.  Positions of a plane are taken linearly,
// so ragged widths leave no lanes idle, and H is formed in each launch instead of
// stored between them.  96^3 FP32 without flow: 21 us per step, against 39 us on
// the generic kernels (which store H and read scalars); 200^3: 176 us, 0.67 of
// the copy bandwidth on the 100 B a site moves; 32^3: 3.6 us.  The corrector adds
// in the order of the generic kernels: (Q + Q*) + R; with Q + (Q* + R) the FP64
// result was 2.7 times as far from the exact one after 40 steps.  186 instructions
// a site put the issue floor at 4.3 us per launch at 96^3; what is above it is
// the latency of the loads, which the fetch of the next plane covers in part
// (24 -> 21 us).  Tiles of 2-D neighbourhoods in place of linear positions and
// one plane per thread were no faster.
#include <algorithm>

#include "common.cuh"
#include "kernels.h"
#include "runtime.h"
#include "tma.cuh"
#include "zm.cuh"

namespace lcbp {

namespace {

// FP64: the pipe (half a lane per SM sub-partition) is the bound, so what counts is
// an even spread of warps: CTAs of one warp, one plane each.  Against 128 threads
// and several planes: 24^3 15.5 -> 10.4 us a step, 32^3 31.5 -> 17.5, 40^3 59.0 ->
// 35.8, 64^3 143 -> 117 (the generic kernels: 16.6, 23.8, 58.6, 127).
template <typename real>
constexpr int heun_threads() {
  return sizeof(real) == 8 ? 32 : 128;
}

// LINEAR: threads take the positions of all chunks in one sequence, so that planes
// much smaller than a CTA leave no lanes idle (4 x 4 x 16384 FP32 37.5 -> 17.3 us a
// step, 17 x 8 x 5000 31.0 -> 21.7; FP64 223 -> 119, 6 x 6 x 4000 117 -> 70).  Else a
// CTA keeps to one chunk, whose planes are then the same for all of its threads:
// FP32 21.6 us at 96^3 against 23.3.
template <typename real, bool FLOW, bool WALLS, bool CORRECT, bool LINEAR>
__global__ void __launch_bounds__(heun_threads<real>())
    k_heun(ZmGeom G, Model<real> m, const real* S, const real* Qn, const real* U, real* out, Sym5<real> qw) {
  grid_wait();
  const int nx = G.nx, ny = G.ny, nz = G.nz, nxm = G.nxm;
  const int np = nx * ny, t = (LINEAR ? blockIdx.x : blockIdx.x % G.tiles_x) * heun_threads<real>() + threadIdx.x;
  const int chunk = LINEAR ? t / np : blockIdx.x / G.tiles_x;
  const int p = LINEAR ? t - chunk * np : t;
  if (LINEAR ? chunk >= G.tiles_z : p >= np) return;
  const int y = p / nx, x = p - y * nx;
  const int z0 = chunk * G.zc, z1 = min(z0 + G.zc, nz);
  // periodic neighbours in the plane, as offsets in sites
  const int dxm = x == 0 ? nx - 1 : -1, dxp = x == nx - 1 ? 1 - nx : 1;
  const int dym = y == 0 ? (ny - 1) * nxm : -nxm, dyp = y == ny - 1 ? (1 - ny) * nxm : nxm;
  const int cq4 = 4 * (int)G.cq;
  auto oq = [&](int z) { return (z * G.nyq + y + 2) * nxm + x + kZmMirX; };
  auto ou = [&](int z) { return (z * G.nyu + y + 1) * nxm + x + kZmMirX; };
  auto below = [&](int z) { return z == 0 ? nz - 1 : z - 1; };
  auto above = [&](int z) { return z == nz - 1 ? 0 : z + 1; };
  auto vel = [&](int o, real u[3]) {  // of the [rho - 1, u_x, u_y, u_z] vector at site o
    real v[4];
    ld4(U, 4 * o, v);
    u[0] = v[1], u[1] = v[2], u[2] = v[3];
  };
  Stencil7<real> st;
  st.zm = WALLS && z0 == 0 ? qw : qmirror_at(S, cq4, oq(below(z0)));
  st.c = qmirror_at(S, cq4, oq(z0));
  real u[3] = {}, ulo[3] = {}, uhi[3] = {};
  if constexpr (FLOW) {
    vel(ou(below(z0)), ulo);
    vel(ou(z0), u);
  }
  // a plane's loads, issued before the arithmetic of the plane before it
  Stencil7<real> next;
  Sym5<real> next_q0;
  auto fetch = [&](int z) {
    const int o = oq(z);
    next.zp = WALLS && z == nz - 1 ? qw : qmirror_at(S, cq4, oq(above(z)));
    next.xm = qmirror_at(S, cq4, o + dxm);
    next.xp = qmirror_at(S, cq4, o + dxp);
    next.ym = qmirror_at(S, cq4, o + dym);
    next.yp = qmirror_at(S, cq4, o + dyp);
    if constexpr (CORRECT) next_q0 = qmirror_at(Qn, cq4, o);
  };
  fetch(z0);
  for (int z = z0; z < z1; ++z) {
    const int o = oq(z);
    st.zp = next.zp;
    st.xm = next.xm;
    st.xp = next.xp;
    st.ym = next.ym;
    st.yp = next.yp;
    const Sym5<real> q0 = next_q0;
    if (z + 1 < z1) fetch(z + 1);
    Sym5<real> dq[3];
    const Sym5<real> h = molecular_field<true>(st, m, dq);
    real w[3][3] = {};
    if constexpr (FLOW) {
      const int a = ou(z);
      real up[3], um[3];
      vel(ou(above(z)), uhi);
      vel(a + dxp, up);
      vel(a + dxm, um);
#pragma unroll
      for (int k = 0; k < 3; ++k) w[k][0] = up[k] - um[k];  // twice the central derivatives
      vel(a + dyp, up);
      vel(a + dym, um);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        w[k][1] = up[k] - um[k];
        // no slip half a spacing beyond a wall
        w[k][2] = (WALLS && z == nz - 1 ? -u[k] : uhi[k]) - (WALLS && z == 0 ? -u[k] : ulo[k]);
      }
    }
    const Sym5<real> r = be_rate<true>(st.c, h, dq, u, w, m, FLOW);
    if constexpr (CORRECT) {
      const real half = real(0.5);
      const Sym5<real> q1 = {half * (q0.xx + st.c.xx + r.xx), half * (q0.xy + st.c.xy + r.xy),
                             half * (q0.xz + st.c.xz + r.xz), half * (q0.yy + st.c.yy + r.yy),
                             half * (q0.yz + st.c.yz + r.yz)};
      // the state's mirror: its periodic images too
      mirror_positions(kZmMirX, 2, nx, ny, x, y, [&](int X, int Y) {
        const int i = (z * G.nyq + Y) * nxm + X;
        st4(out + 4 * i, q1.xx, q1.xy, q1.xz, q1.yy);
        out[cq4 + i] = q1.yz;
      });
    } else {
      const Sym5<real> q1 = {st.c.xx + r.xx, st.c.xy + r.xy, st.c.xz + r.xz, st.c.yy + r.yy, st.c.yz + r.yz};
      st4(out + 4 * o, q1.xx, q1.xy, q1.xz, q1.yy);
      out[cq4 + o] = q1.yz;
    }
    st.zm = st.c;
    st.c = st.zp;
    if constexpr (FLOW) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        ulo[k] = u[k];
        u[k] = uhi[k];
      }
    }
  }
}

// CTAs of the kernel that the chip holds at once
template <typename real, typename K>
long long heun_slots(K kernel) {
  int per_sm = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, heun_threads<real>(), 0);
  return (long long)sm_count() * std::max(1, per_sm);
}

template <typename real, bool FLOW, bool WALLS, bool LINEAR>
cudaError_t launch_as(const HeunArgs& a, ZmGeom G, cudaStream_t s) {
  G.tiles_z = (a.nz + G.zc - 1) / G.zc;
  const int T = heun_threads<real>();
  const int grid = LINEAR ? (a.nx * a.ny * G.tiles_z + T - 1) / T : G.tiles_x * G.tiles_z;
  const Model<real> m = *static_cast<const Model<real>*>(a.model);
  Sym5<real> qw{};
  if (WALLS) qw = {(real)a.q_wall[0], (real)a.q_wall[1], (real)a.q_wall[2], (real)a.q_wall[3], (real)a.q_wall[4]};
  const real *q = static_cast<const real*>(a.q), *u = static_cast<const real*>(a.u);
  real *qs = static_cast<real*>(a.qs), *out = static_cast<real*>(a.q);
  launch_dependent(k_heun<real, FLOW, WALLS, false, LINEAR>, grid, T, 0, s, G, m, q, nullptr, u, qs, qw);
  if (a.mid) cudaEventRecord(a.mid, s);
  launch_dependent(k_heun<real, FLOW, WALLS, true, LINEAR>, grid, T, 0, s, G, m, qs, q, u, out, qw);
  return cudaGetLastError();
}

// Planes per thread: FP64 one (above); FP32 as many as let the grid fill the
// resident CTAs once (fewer loads per site), at most 16.  FP64 is always LINEAR (no
// shape of 24 lost by it); FP32 where planes would fill less than 0.6 of their CTAs'
// lanes, in more CTAs than the chip holds at once (above 0.6 it gave 0.87-1.01 of the
// other's speed, below 0.98-2.16; 4 x 4 x 500, which fits at once, 0.91).
template <typename real, bool FLOW, bool WALLS>
cudaError_t launch(const HeunArgs& a, cudaStream_t s) {
  ZmGeom G{};
  G.nx = a.nx;
  G.ny = a.ny;
  G.nz = a.nz;
  G.nxm = zm_mirror_nx(a.nx);
  G.nyq = a.ny + 4;
  G.nyu = a.ny + 2;
  G.cq = (long long)G.nxm * G.nyq * a.nz;
  const int T = heun_threads<real>(), np = a.nx * a.ny;
  G.tiles_x = (np + T - 1) / T;
  if constexpr (sizeof(real) == 8) {
    G.zc = 1;
    return launch_as<real, FLOW, WALLS, true>(a, G, s);
  } else {
    const long long slots = heun_slots<real>(k_heun<real, FLOW, WALLS, true, false>);
    const long long ctas = (long long)G.tiles_x * a.nz;
    const bool linear = np < 0.6 * G.tiles_x * T && ctas > slots;
    const long long all = linear ? ((long long)np * a.nz + T - 1) / T : ctas;
    G.zc = (int)std::min<long long>(16, std::max<long long>(1, (all + slots - 1) / slots));
    return linear ? launch_as<real, FLOW, WALLS, true>(a, G, s) : launch_as<real, FLOW, WALLS, false>(a, G, s);
  }
}

}  // namespace

template <typename real>
cudaError_t launch_heun(const HeunArgs& a, cudaStream_t s) {
  if (a.u) return a.q_wall ? launch<real, true, true>(a, s) : launch<real, true, false>(a, s);
  return a.q_wall ? launch<real, false, true>(a, s) : launch<real, false, false>(a, s);
}
template cudaError_t launch_heun<float>(const HeunArgs&, cudaStream_t);
template cudaError_t launch_heun<double>(const HeunArgs&, cudaStream_t);

}  // namespace lcbp
