// Adjoint of the level-set passes of a step with a MOVING interface (the paper
// has no adjoint; the forward passes are Sec. 2.2 and Eq. hyperbolicExtension).
// Within a window without phase changes, a step maps (f, phi, u~) smoothly:
//   u~ on interface cells = mean u_I of their cut links (moments of f_n, q(phi_n)),
//   n_ext first-order upwind extension sweeps on the other band cells, velocity
//   S(phi) n(phi); TVD-RK3 transport with the fifth-order upwind-biased stencil;
//   one TVD-RK3 pseudo step of the constrained HJ-WENO5 reinitialisation.
// The discrete choices (band, frozen cells, upwind sides, Godunov branch) are
// those of the forward step.  The kernels below apply the transposes of these
// passes as scatter-adds (FP32 atomics): a stencil point that is not updated by
// the pass keeps the pass input's value, so its adjoint goes straight to the
// adjoint of that input.  The lattice Boltzmann part of the step reuses the
// frozen-interface kernels with the geometry of phi_n.
#include "lsb_kernels.h"
#include "lsb_lspass.cuh"

#ifndef LSA_MINB
#define LSA_MINB 2  // CTAs of 512 threads per SM k_lsa_levelset is built for
#endif

namespace lsb {

namespace {

// The seven points at offsets -3..+3 along axis a of a cell of band block gb (global id) at
// level offset c: offsets from the cell (walls clamp, periodic axes wrap) and which of them
// lie in the band.  Inside the box a point's membership is its own block's (in the band) or
// that of the face neighbour it falls into.
struct Line7 {
  int off[7];
  unsigned band;
};
template <int D>
__device__ __forceinline__ Line7 line7(const Ctx &C, const LevelDev &L, const BlockShape &S, int gb, int x, int y, int z,
                                       long long c, int a) {
  Line7 r;
  const int crd[3] = {x, y, z};
  const int q = a == 0 ? x : (a == 1 ? y : z);
  const int str = a == 0 ? 1 : (a == 1 ? L.p[0] : L.p[0] * L.p[1]);
  r.band = 0;
  if (q >= 3 && q + 3 < L.n[a] && S.bs[a] >= 4) {
    const int s0 = (q >> S.lg[a]) << S.lg[a], s1 = s0 + S.bs[a];
    const int bstr = a == 0 ? 1 : (a == 1 ? L.nb[0] : L.nb[0] * L.nb[1]);
    const bool fm = q - 3 < s0 && (C.bflag[gb - bstr] & BF_BAND) != 0;
    const bool fp = q + 3 >= s1 && (C.bflag[gb + bstr] & BF_BAND) != 0;
#pragma unroll
    for (int m = 0; m < 7; ++m) {
      r.off[m] = (m - 3) * str;
      const int v = q + m - 3;
      if (v < s0 ? fm : (v >= s1 ? fp : true)) r.band |= 1u << m;
    }
  } else {
#pragma unroll
    for (int m = 0; m < 7; ++m) {
      int p[3] = {crd[0], crd[1], crd[2]};
      p[a] = clampwrap(L, a, q + m - 3);
      r.off[m] = (int)(cidx(L, p[0], p[1], p[2]) - c);
      if (in_band(C, L, S, p[0], p[1], p[2])) r.band |= 1u << m;
    }
  }
  return r;
}

// HJ-WENO5 value and its partial derivatives in the five differences (Jiang & Peng).
__device__ __forceinline__ float weno5_grad(const float v[5], float g[5]) {
  const float eps = 1e-6f;
  const float e[3][5] = {{1.f / 3.f, -7.f / 6.f, 11.f / 6.f, 0.f, 0.f},
                         {0.f, -1.f / 6.f, 5.f / 6.f, 1.f / 3.f, 0.f},
                         {0.f, 0.f, 1.f / 3.f, 5.f / 6.f, -1.f / 6.f}};
  const float b[3][5] = {{1.f, -2.f, 1.f, 0.f, 0.f}, {0.f, 1.f, -2.f, 1.f, 0.f}, {0.f, 0.f, 1.f, -2.f, 1.f}};
  const float c[3][5] = {{1.f, -4.f, 3.f, 0.f, 0.f}, {0.f, 1.f, 0.f, -1.f, 0.f}, {0.f, 0.f, 3.f, -4.f, 1.f}};
  const float gam[3] = {0.1f, 0.6f, 0.3f};
  float d[3], a[3], bv[3], cv[3], sk[3];
  float A = 0.f, num = 0.f;
  for (int k = 0; k < 3; ++k) {
    d[k] = bv[k] = cv[k] = 0.f;
    for (int m = 0; m < 5; ++m) {
      d[k] += e[k][m] * v[m];
      bv[k] += b[k][m] * v[m];
      cv[k] += c[k][m] * v[m];
    }
    sk[k] = 13.f / 12.f * bv[k] * bv[k] + 0.25f * cv[k] * cv[k];
    a[k] = gam[k] / ((sk[k] + eps) * (sk[k] + eps));
    A += a[k];
    num += a[k] * d[k];
  }
  const float val = num / A;
  for (int m = 0; m < 5; ++m) g[m] = 0.f;
  for (int k = 0; k < 3; ++k) {
    const float wk = a[k] / A;
    const float dak = -2.f * gam[k] / ((sk[k] + eps) * (sk[k] + eps) * (sk[k] + eps));
    const float r = (d[k] - val) / A * dak;
    for (int m = 0; m < 5; ++m)
      g[m] += wk * e[k][m] + r * (13.f / 6.f * bv[k] * b[k][m] + 0.5f * cv[k] * c[k][m]);
  }
  return val;
}

}  // namespace

// ------------------------------------------------------------------ forward replay: interface velocity
// u~ on interface cells = mean over cut links of (1 - q) u(x) + q u(y), with the
// pre-collision moments of the stored state F (= f_n) and q from C.phi (= phi_n):
// the values d_ext_init writes from the collide kernel's moments.
template <int Q>
__global__ void k_lsa_init(Ctx C, int glevel, const float *__restrict__ F, float *U0) {
  using LT = Lat<Q>;
  constexpr int D = LT::D;
  const int n = min(C.counters[glevel * NCOUNT + 1], (int)C.list_cap);
  const int2 *lst = C.iface_list + (long long)glevel * C.list_cap;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const int2 it = lst[e];
    const LevelDev &L = C.lds[it.x];
    const long long c = it.y;
    int x, y, z;
    cell_xyz(L, c, x, y, z);
    const long long fo = L.fine_off, NF = C.nfine, N = L.ncell;
    const float *Fl = F + L.cell_off * Q;
    const uint32_t m = C.cmask[fo + c];
    float f[Q], rx, ux[3];
#pragma unroll
    for (int j = 0; j < Q; ++j) f[j] = Fl[j * N + c];
    lb_moments<Q>(f, rx, ux);
    const float phx = C.phi[fo + c];
    float acc[3] = {0.f, 0.f, 0.f};
    int cnt = 0;
    for (int k = 0; k < Q; ++k) {
      if (!(m & (1u << k))) continue;
      const int i = LT::opp(k);
      int yx = x + LT::cx(i), yy = y + LT::cy(i), yz = z + LT::cz(i);
      wrap(L, 0, yx); wrap(L, 1, yy); if (D == 3) wrap(L, 2, yz);
      const long long cy_ = cidx(L, yx, yy, yz);
      const float q = phx / (phx - C.phi[fo + cy_]);
      float fy[Q], ry, uy[3];
#pragma unroll
      for (int j = 0; j < Q; ++j) fy[j] = Fl[j * N + cy_];
      lb_moments<Q>(fy, ry, uy);
      for (int a = 0; a < D; ++a) acc[a] += (1.0f - q) * ux[a] + q * uy[a];
      ++cnt;
    }
    for (int a = 0; a < D; ++a) U0[a * NF + fo + c] = acc[a] / (float)cnt;
  }
}

// ------------------------------------------------------------------ transpose of the interface velocity
// For interface cell x with cnt cut links: lu = LS0(x) / cnt per link; the moment
// adjoints go to the macro buffer's u slots of x and y (carried to the populations
// by k_adj_macro), the q adjoint to phi(x), phi(y); LS0(x) is then cleared (the
// pass overwrote u~ there).
template <int Q>
__global__ void k_lsa_init_T(Ctx C, int glevel, const float *__restrict__ F, float *LS0, float *MA, float *LPHI) {
  using LT = Lat<Q>;
  constexpr int D = LT::D;
  const int n = min(C.counters[glevel * NCOUNT + 1], (int)C.list_cap);
  const int2 *lst = C.iface_list + (long long)glevel * C.list_cap;
  const long long NF = C.nfine;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n; e += gridDim.x * blockDim.x) {
    const int2 it = lst[e];
    const LevelDev &L = C.lds[it.x];
    const long long c = it.y;
    int x, y, z;
    cell_xyz(L, c, x, y, z);
    const long long fo = L.fine_off, N = L.ncell;
    const float *Fl = F + L.cell_off * Q;
    const uint32_t m = C.cmask[fo + c];
    const int cnt = __popc(m);
    float lu[3] = {0.f, 0.f, 0.f};
    for (int a = 0; a < D; ++a) {
      lu[a] = LS0[a * NF + fo + c] / (float)cnt;
      LS0[a * NF + fo + c] = 0.f;
    }
    float f[Q], rx, ux[3];
#pragma unroll
    for (int j = 0; j < Q; ++j) f[j] = Fl[j * N + c];
    lb_moments<Q>(f, rx, ux);
    const float phx = C.phi[fo + c];
    float mx[3] = {0.f, 0.f, 0.f}, lphx = 0.f;
    for (int k = 0; k < Q; ++k) {
      if (!(m & (1u << k))) continue;
      const int i = LT::opp(k);
      int yx = x + LT::cx(i), yy = y + LT::cy(i), yz = z + LT::cz(i);
      wrap(L, 0, yx); wrap(L, 1, yy); if (D == 3) wrap(L, 2, yz);
      const long long cy_ = cidx(L, yx, yy, yz);
      const float phy = C.phi[fo + cy_];
      const float q = phx / (phx - phy);
      float fy[Q], ry, uy[3];
#pragma unroll
      for (int j = 0; j < Q; ++j) fy[j] = Fl[j * N + cy_];
      lb_moments<Q>(fy, ry, uy);
      float lq = 0.f;
      for (int a = 0; a < D; ++a) {
        mx[a] += (1.0f - q) * lu[a];
        atomicAdd(MA + (1 + a) * NF + fo + cy_, q * lu[a]);
        lq += lu[a] * (uy[a] - ux[a]);
      }
      const float den = (phx - phy) * (phx - phy);
      lphx += -lq * phy / den;
      atomicAdd(LPHI + fo + cy_, lq * phx / den);
    }
    for (int a = 0; a < D; ++a) atomicAdd(MA + (1 + a) * NF + fo + c, mx[a]);
    atomicAdd(LPHI + fo + c, lphx);
  }
}

// ------------------------------------------------------------------ transposed stages
// Shu-Osher stages p1 = p0 + R(p0), p2 = 3/4 p0 + 1/4 (p1 + R(p1)), p3 = 1/3 p0 + 2/3 (p2 +
// R(p2)) on the updated cells (band cells; without the frozen ones for the reinitialisation).
// LP holds the adjoint of p3 and becomes, in place, that of p0; L2 and L1 collect those of p2
// and p1 (zero before, and left zero).  Transposed stage st (3, 2, 1 in this order) takes the
// stage's adjoint m at its cell,
//   st 3: m = LP, LP = m / 3,      L2 += 2/3 m, mu = 2/3 m;
//   st 2: m = L2, LP += 3/4 m,     L1 += 1/4 m, mu = 1/4 m;
//   st 1: m = L1, LP += m,         mu = m,
// and scatters mu times R's Jacobian: stencil points that the stage's input holds as updated
// values get their part in L2 (st 3) or L1 (st 2), all others, and every point for st 1, in LP.
// The cell's own shares go by atomics wherever other cells may scatter to it in the pass.
__device__ __forceinline__ float stage_adjoint(int st, long long fc, float *LP, float *L1, float *L2) {
  if (st == 3) {
    const float m = LP[fc];  // an updated cell: no point of this pass scatters to LP here
    LP[fc] = m / 3.0f;
    atomicAdd(L2 + fc, 2.0f / 3.0f * m);
    return 2.0f / 3.0f * m;
  }
  if (st == 2) {
    const float m = L2[fc];
    LP[fc] += 0.75f * m;
    atomicAdd(L1 + fc, 0.25f * m);
    return 0.25f * m;
  }
  const float m = L1[fc];
  atomicAdd(LP + fc, m);
  L1[fc] = 0.f;  // nothing scatters to L1, L2 in this pass
  L2[fc] = 0.f;
  return m;
}

// Transposed reinitialisation stage: R(p) = -dtau S0 (|grad p|_G - 1) with Godunov's
// Hamiltonian on HJ-WENO5 one-sided differences; the stage value p is pin at updated points
// and C.phi (= phi*) elsewhere.  LS0 collects d/dS0 over the stages; stage 1 adds its share
// S'(phi*) = (phi*^2 + 1)^(-3/2) to LP.
template <int D>
__device__ __forceinline__ void d_lsa_reinit(const Ctx &C, const BlockShape &S, int glevel, int st, const float *pin,
                                             float *LP, float *L1, float *L2, float *LS0) {
  const int nl = min(C.counters[glevel * NCOUNT + 3], C.band_cap);
  const int *lst = C.band_list + (long long)glevel * C.band_cap;
  float *Lt = st == 3 ? L2 : L1;
  for (int w = blockIdx.x; w < nl; w += gridDim.x) {
    int x, y, z;
    const LevelDev &L = band_cell(C, S, glevel, w, threadIdx.x, x, y, z);
    if (x >= L.n[0] || y >= L.n[1] || z >= L.n[2]) continue;
    const long long c = cidx(L, x, y, z), fc = L.fine_off + c;
    if (C.frozen[fc]) continue;
    const float mu = stage_adjoint(st, fc, LP, L1, L2);
    float ls0 = st == 3 ? 0.f : LS0[fc];
    if (mu != 0.f) {
      const int gb = lst[w];
      const float s0 = C.s0[fc];
      // per axis: the chosen side's derivative terms (mirrored for the right-biased side)
      float gd[D][5], dga[D], g2 = 0.f;
      bool left[D];
      unsigned upd[D];
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const Line7 ln = line7<D>(C, L, S, gb, x, y, z, c, a);
        float P[7];
        upd[a] = 0;
#pragma unroll
        for (int m = 0; m < 7; ++m) {
          const long long cc = fc + ln.off[m];
          const bool u = st > 1 && ((ln.band >> m) & 1u) && !C.frozen[cc];
          if (u) upd[a] |= 1u << m;
          P[m] = u ? pin[cc] : C.phi[cc];
        }
        const float vm[5] = {P[1] - P[0], P[2] - P[1], P[3] - P[2], P[4] - P[3], P[5] - P[4]};
        const float vp[5] = {P[6] - P[5], P[5] - P[4], P[4] - P[3], P[3] - P[2], P[2] - P[1]};
        float gm[5], gp[5];
        const float dm = weno5_grad(vm, gm), dp = weno5_grad(vp, gp);
        const float am = s0 > 0.f ? fmaxf(dm, 0.f) : fminf(dm, 0.f), ap = s0 > 0.f ? fminf(dp, 0.f) : fmaxf(dp, 0.f);
        left[a] = am * am >= ap * ap;
        g2 += left[a] ? am * am : ap * ap;
        dga[a] = 2.f * (left[a] ? am : ap);
#pragma unroll
        for (int m = 0; m < 5; ++m) gd[a][m] = left[a] ? gm[m] : gp[m];
      }
      const float sq = sqrtf(g2), dt = L.dtau_reinit;
      ls0 += mu * (-dt * (sq - 1.0f));
      const float lg2 = sq > 0.f ? mu * (-dt * s0 / (2.0f * sq)) : 0.f;
      if (lg2 != 0.f) {
#pragma unroll
        for (int a = 0; a < D; ++a) {
          // left: difference m is P[m+1] - P[m]; right: P[6-m] - P[5-m]
          const float wg = lg2 * dga[a];
          float lp[7] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
          if (left[a]) {
#pragma unroll
            for (int m = 0; m < 5; ++m) {
              lp[m + 1] += wg * gd[a][m];
              lp[m] -= wg * gd[a][m];
            }
          } else {
#pragma unroll
            for (int m = 0; m < 5; ++m) {
              lp[6 - m] += wg * gd[a][m];
              lp[5 - m] -= wg * gd[a][m];
            }
          }
          const Line7 ln = line7<D>(C, L, S, gb, x, y, z, c, a);
#pragma unroll
          for (int m = 0; m < 7; ++m)
            if (lp[m] != 0.f) atomicAdd(((upd[a] >> m) & 1u ? Lt : LP) + fc + ln.off[m], lp[m]);
        }
      }
    }
    if (st > 1) {
      LS0[fc] = ls0;
    } else {
      const float p = C.phi[fc], d = p * p + 1.0f;
      atomicAdd(LP + fc, ls0 / (d * sqrtf(d)));
    }
  }
}

// Transposed transport stage: R(p) = -sum_a u~_a d_a(p) with the fifth-order upwind-biased
// stencil on the side of sign(u~_a) (C.ut0 = the committed u~ of the step).  Stage value:
// pin at band points, C.phi (= phi_n) elsewhere.  LU (adjoint of u~) gets -mu d_a(p).  With
// restore set, stage 3 also writes phi_n back into C.phi at its cell (no stage before the
// first reads C.phi in the band).
template <int D>
__device__ __forceinline__ void d_lsa_adv(const Ctx &C, const BlockShape &S, int glevel, int st, const float *pin,
                                          const float *restore, float *LP, float *L1, float *L2, float *LU) {
  const float wm[7] = {-2.f / 60.f, 15.f / 60.f, -60.f / 60.f, 20.f / 60.f, 30.f / 60.f, -3.f / 60.f, 0.f};
  const int nl = min(C.counters[glevel * NCOUNT + 3], C.band_cap);
  const int *lst = C.band_list + (long long)glevel * C.band_cap;
  const long long NF = C.nfine;
  float *Lt = st == 3 ? L2 : L1;
  for (int w = blockIdx.x; w < nl; w += gridDim.x) {
    int x, y, z;
    const LevelDev &L = band_cell(C, S, glevel, w, threadIdx.x, x, y, z);
    if (x >= L.n[0] || y >= L.n[1] || z >= L.n[2]) continue;
    const long long c = cidx(L, x, y, z), fc = L.fine_off + c;
    if (st == 3 && restore) C.phi[fc] = restore[fc];
    const float mu = stage_adjoint(st, fc, LP, L1, L2);
    if (mu == 0.0f) continue;
    const int gb = lst[w];
    for (int a = 0; a < D; ++a) {
      const Line7 ln = line7<D>(C, L, S, gb, x, y, z, c, a);
      const float ua = C.ut0[a * NF + fc];
      float da = 0.f;
#pragma unroll
      for (int m = 0; m < 7; ++m) {
        // d5m: weights wm on points 0..5; d5p: -wm mirrored onto points 6..1
        const float cw = ua >= 0.f ? wm[m] : -wm[6 - m];
        if (cw == 0.f) continue;
        const long long cc = fc + ln.off[m];
        const bool upd = st > 1 && ((ln.band >> m) & 1u);
        da += cw * (upd ? pin[cc] : C.phi[cc]);
        atomicAdd((upd ? Lt : LP) + cc, -ua * cw * mu);
      }
      LU[a * NF + fc] += -mu * da;
    }
  }
}

// ------------------------------------------------------------------ transpose of an extension sweep
// Forward sweep k on band cells that are not interface cells:
//   u_{k+1}(c) = u_k(c) - dtau sum_a v_a (v_a > 0 ? u_k(c) - u_k(c - e_a) : u_k(c + e_a) - u_k(c)),
// v = S(phi) n(phi) (central n), a neighbour outside the band read from S0 (= the
// committed u~ of the previous step, which the sweeps leave alone).  Lin holds the adjoint of
// u_{k+1} at band cells (cleared as it is read, unless it is LU itself), Lout (zero before)
// collects that of u_k; a neighbour outside the band gets its part in LU.  LV(a, c)
// accumulates d/dv_a over the sweeps.  Cleared where there is something to clear: a store of zero
// right behind the load of the same word made a sweep over 2.2 M band cells take 325 us instead of
// 80 (and the reverse of a step on 384 x 384 x 48 cells 7.8 ms instead of 5.4).
template <int D>
__device__ __forceinline__ void d_lsa_ext_T(const Ctx &C, const BlockShape &S, int glevel, const float *Sk,
                                            const float *S0, float *Lin, float *Lout, float *LU, float *LV) {
  const int nl = min(C.counters[glevel * NCOUNT + 3], C.band_cap);
  const long long NF = C.nfine;
  for (int w = blockIdx.x; w < nl; w += gridDim.x) {
    int x, y, z;
    const LevelDev &L = band_cell(C, S, glevel, w, threadIdx.x, x, y, z);
    if (x >= L.n[0] || y >= L.n[1] || z >= L.n[2]) continue;
    const long long fo = L.fine_off, c = cidx(L, x, y, z);
    float lc[3] = {0.f, 0.f, 0.f};
    for (int b = 0; b < D; ++b) {
      lc[b] = Lin[b * NF + fo + c];
      if (Lin != LU && lc[b] != 0.f) Lin[b * NF + fo + c] = 0.f;
    }
    const uint8_t pf = C.plan_f[fo + c];
    if (pf & 64) {  // interface cell: carried over
      for (int b = 0; b < D; ++b)
        if (lc[b] != 0.f) atomicAdd(Lout + b * NF + fo + c, lc[b]);
      continue;
    }
    const float dt = L.dtau_ext;
    float own[3] = {lc[0], lc[1], lc[2]};
    for (int a = 0; a < D; ++a) {
      // the replay's plan: v_a, its side and whether the neighbour lies in the band
      const float va = C.plan_v[a * NF + fo + c];
      const int dir = (pf >> a) & 1 ? -1 : 1;
      long long cn;
      if (pf & 128) {
        int nb[3] = {x, y, z};
        nb[a] = clampwrap(L, a, nb[a] + dir);
        cn = cidx(L, nb[0], nb[1], nb[2]);
      } else {
        cn = c + dir * (a == 0 ? 1LL : (a == 1 ? (long long)L.p[0] : (long long)L.p[0] * L.p[1]));
      }
      const bool inb = (pf >> (3 + a)) & 1;
      const float *src = inb ? Sk : S0;
      float lva = 0.f;
      for (int b = 0; b < D; ++b) {
        const float u0 = Sk[b * NF + fo + c], un = src[b * NF + fo + cn];
        lva += lc[b] * (-dt * (va > 0.f ? (u0 - un) : (un - u0)));
        if (lc[b] == 0.f || va == 0.f) continue;
        own[b] += lc[b] * (va > 0.f ? -dt * va : dt * va);
        atomicAdd((inb ? Lout : LU) + b * NF + fo + cn, lc[b] * (va > 0.f ? dt * va : -dt * va));
      }
      LV[a * NF + fo + c] += lva;
    }
    for (int b = 0; b < D; ++b)
      if (own[b] != 0.f) atomicAdd(Lout + b * NF + fo + c, own[b]);
  }
}

// d/dphi of the extension velocity v = S(phi) n, n = g / |g|, g_a = (phi(c + e_a) - phi(c - e_a)) / 2,
// S(phi) = phi / sqrt(phi^2 + 1), from LV (summed over the sweeps); LV is cleared.  Lin, the
// adjoint of the sweeps' input at band cells, moves to LU and is cleared.
template <int D>
__device__ __forceinline__ void d_lsa_ext_v(const Ctx &C, const BlockShape &S, int glevel, float *Lin, float *LU,
                                            float *LV, float *LPHI) {
  const int nl = min(C.counters[glevel * NCOUNT + 3], C.band_cap);
  const long long NF = C.nfine;
  for (int w = blockIdx.x; w < nl; w += gridDim.x) {
    int x, y, z;
    const LevelDev &L = band_cell(C, S, glevel, w, threadIdx.x, x, y, z);
    if (x >= L.n[0] || y >= L.n[1] || z >= L.n[2]) continue;
    const long long fo = L.fine_off;
    const long long c = cidx(L, x, y, z);
    for (int b = 0; b < D; ++b) {
      const float l = Lin[b * NF + fo + c];
      LU[b * NF + fo + c] = l;
      if (l != 0.f) Lin[b * NF + fo + c] = 0.f;
    }
    if (C.plan_f[fo + c] & 64) continue;
    float lv[3] = {0.f, 0.f, 0.f};
    bool any = false;
    for (int a = 0; a < D; ++a) {
      lv[a] = LV[a * NF + fo + c];
      if (lv[a] != 0.f) {
        LV[a * NF + fo + c] = 0.f;
        any = true;
      }
    }
    if (!any) continue;
    const int crd[3] = {x, y, z};
    long long ip[3], im[3];
    float nv[3], gm = 0.f;
    for (int a = 0; a < D; ++a) {
      int p[3] = {x, y, z}, m[3] = {x, y, z};
      p[a] = clampwrap(L, a, crd[a] + 1);
      m[a] = clampwrap(L, a, crd[a] - 1);
      ip[a] = fo + cidx(L, p[0], p[1], p[2]);
      im[a] = fo + cidx(L, m[0], m[1], m[2]);
      nv[a] = 0.5f * (C.phi[ip[a]] - C.phi[im[a]]);
      gm += nv[a] * nv[a];
    }
    gm = sqrtf(gm);
    if (!(gm > 0.f)) continue;
    const float ph = C.phi[fo + c];
    const float d = ph * ph + 1.0f;
    const float sg = ph / sqrtf(d);
    float ls = 0.f, dot = 0.f;
    for (int a = 0; a < D; ++a) {
      ls += lv[a] * nv[a] / gm;
      dot += nv[a] / gm * sg * lv[a];
    }
    atomicAdd(LPHI + fo + c, ls / (d * sqrtf(d)));
    for (int a = 0; a < D; ++a) {
      const float lg = (sg * lv[a] - nv[a] / gm * dot) / gm;
      atomicAdd(LPHI + ip[a], 0.5f * lg);
      atomicAdd(LPHI + im[a], -0.5f * lg);
    }
  }
}

// ------------------------------------------------------------------ the level-set part of a reverse sub-step
// Everything between the interface velocity's replay and its transpose in one cooperative
// launch, a CTA per band block and a grid barrier between passes: the replay of the n_ext
// extension sweeps, the transport and the first two reinitialisation stages of the step from
// (phi_n, u~_n), then the transposes of the reinitialisation, the transport and the sweeps.
// As launches these were 41 per sub-step beside 20 dense copies and fills; now 28 passes that
// touch band cells only.  A window of 8 steps on 64 x 96 cells (two levels) and its reverse
// sweep 10.4 -> 7.9 ms, 4 steps on 96 x 96 x 128 (two levels) 31.4 -> 25.4 ms; the launch
// itself takes 130 us there in 2D (a CTA per band block) and 0.61 ms in 3D (442 k band cells;
// 0.82 before the sweeps' accumulators were cleared only where they hold something).  Two CTAs of
// 512 threads per SM: 0.82 ms per sub-step then, against 0.99 with one (more chains in flight) and
// 0.84 with three (spills).  As a launch per pass, 2.2 M band cells: within 1%.
// The adjoints LP (of phi) and LU (of u~) change in place; phi_n is overwritten by phi* on the
// band while the reinitialisation is transposed and written back from PB.
// A: scratch of the sweep (LsaScratch); rein: the step reinitialised.
template <int Q, int MODE>  // MODE of the barriers
__global__ void __launch_bounds__(512, LSA_MINB) k_lsa_levelset(Ctx C, BlockShape S, int glevel, int n_ext, int rein,
                                                                LsaScratch A, unsigned *bar, unsigned limit) {
  constexpr int D = Lat<Q>::D;
  const long long NF = C.nfine;
  unsigned target = 0;
  __shared__ unsigned wait_limit;
  if (threadIdx.x == 0) wait_limit = limit;
  float *const phi_n = C.phi;
  auto Sk = [&](int k) { return k == 0 ? A.S0 : A.S + (long long)(k - 1) * D * NF; };
  // ---- replay: extension (E: the committed field outside the band is u~_n with the
  // interface cells' new values), transport, reinitialisation
  Ctx E = C;
  E.ut0 = A.S0;
  for (int k = 0; k < n_ext; ++k) {
    d_ext_iter<D>(E, S, glevel, Sk(k), Sk(k + 1), k == 0 ? 2 : 3);
    if (!lsf_barrier<MODE>(bar, target, C.err, &wait_limit)) return lsf_leave<MODE>(bar);
  }
  Ctx T = C;
  T.p1 = A.A1;
  T.p2 = A.A2;
  T.ut0 = Sk(n_ext);  // the committed u~ (read at the cells themselves only)
  d_adv_stage<D>(T, S, glevel, 1);
  if (!lsf_barrier<MODE>(bar, target, C.err, &wait_limit)) return lsf_leave<MODE>(bar);
  d_adv_stage<D>(T, S, glevel, 2);
  if (!lsf_barrier<MODE>(bar, target, C.err, &wait_limit)) return lsf_leave<MODE>(bar);
  if (rein) {
    const int nl = min(C.counters[glevel * NCOUNT + 3], C.band_cap);
    for (int w = blockIdx.x; w < nl; w += gridDim.x) {  // phi_n of the band, kept
      int x, y, z;
      const LevelDev &L = band_cell(C, S, glevel, w, threadIdx.x, x, y, z);
      if (x >= L.n[0] || y >= L.n[1] || z >= L.n[2]) continue;
      const long long fc = L.fine_off + cidx(L, x, y, z);
      A.PB[fc] = phi_n[fc];
    }
    d_adv_stage<D>(T, S, glevel, 3);  // phi* into phi_n (each cell by the thread that kept it)
    if (!lsf_barrier<MODE>(bar, target, C.err, &wait_limit)) return lsf_leave<MODE>(bar);
    Ctx R = C;
    R.p1 = A.R1;
    R.p2 = A.R2;
    R.frozen = A.FR;
    R.s0 = A.SS;
    d_reinit_prep<Q>(R, S, glevel);
    d_reinit_stage<D>(R, S, glevel, 1);  // reads only its own cell's frozen flag and S(phi*)
    if (!lsf_barrier<MODE>(bar, target, C.err, &wait_limit)) return lsf_leave<MODE>(bar);
    d_reinit_stage<D>(R, S, glevel, 2);
    if (!lsf_barrier<MODE>(bar, target, C.err, &wait_limit)) return lsf_leave<MODE>(bar);
    for (int st = 3; st >= 1; --st) {
      d_lsa_reinit<D>(R, S, glevel, st, st == 3 ? A.R2 : A.R1, A.LP, A.L1, A.L2, A.LS0);
      if (!lsf_barrier<MODE>(bar, target, C.err, &wait_limit)) return lsf_leave<MODE>(bar);
    }
  }
  for (int st = 3; st >= 1; --st) {
    d_lsa_adv<D>(T, S, glevel, st, st == 3 ? A.A2 : A.A1, rein ? A.PB : nullptr, A.LP, A.L1, A.L2, A.LU);
    if (!lsf_barrier<MODE>(bar, target, C.err, &wait_limit)) return lsf_leave<MODE>(bar);
  }
  if (n_ext > 0) {
    float *Lin = A.LU;
    for (int k = n_ext - 1; k >= 0; --k) {
      float *out = Lin == A.LK0 ? A.LK1 : A.LK0;
      d_lsa_ext_T<D>(E, S, glevel, Sk(k), A.S0, Lin, out, A.LU, A.LV);
      if (!lsf_barrier<MODE>(bar, target, C.err, &wait_limit)) return lsf_leave<MODE>(bar);
      Lin = out;
    }
    d_lsa_ext_v<D>(E, S, glevel, Lin, A.LU, A.LV, A.LP);
  }
  lsf_leave<MODE>(bar);
}

// ------------------------------------------------------------------ launchers
#define LSA_Q(kern, ...)                                                          \
  do {                                                                            \
    if (Q == 9) kern<9><<<L.grid, L.block, 0, L.stream>>>(__VA_ARGS__);           \
    else kern<19><<<L.grid, L.block, 0, L.stream>>>(__VA_ARGS__);                 \
    return cudaGetLastError();                                                    \
  } while (0)
cudaError_t run_lsa_init(int Q, Launch L, Ctx C, int glevel, const float *F, float *U0) {
  LSA_Q(k_lsa_init, C, glevel, F, U0);
}
cudaError_t run_lsa_init_T(int Q, Launch L, Ctx C, int glevel, const float *F, float *LS0, float *MA, float *LPHI) {
  LSA_Q(k_lsa_init_T, C, glevel, F, LS0, MA, LPHI);
}
// grid: at most the resident CTAs (a cooperative launch needs them all)
template <int Q, int MODE>
cudaError_t lsa_levelset_launch(Launch L, Ctx C, BlockShape S, int glevel, int n_ext, int rein, LsaScratch A,
                                unsigned *bar, unsigned limit) {
  int per_sm = 0, dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_lsa_levelset<Q, MODE>, L.block, 0);
  if (e != cudaSuccess) return e;
  const int grid = L.grid < per_sm * sms ? L.grid : per_sm * sms;
  void *args[] = {&C, &S, &glevel, &n_ext, &rein, &A, &bar, &limit};
  return cudaLaunchCooperativeKernel((const void *)k_lsa_levelset<Q, MODE>, dim3(grid), dim3(L.block), args, 0, L.stream);
}
cudaError_t run_lsa_levelset(int Q, Launch L, Ctx C, BlockShape S, int glevel, int n_ext, int rein, LsaScratch A,
                             unsigned *bar, unsigned limit) {
  if (limit == kDefaultWait)
    return Q == 9 ? lsa_levelset_launch<9, 2>(L, C, S, glevel, n_ext, rein, A, bar, limit)
                  : lsa_levelset_launch<19, 2>(L, C, S, glevel, n_ext, rein, A, bar, limit);
  return Q == 9 ? lsa_levelset_launch<9, 1>(L, C, S, glevel, n_ext, rein, A, bar, limit)
                : lsa_levelset_launch<19, 1>(L, C, S, glevel, n_ext, rein, A, bar, limit);
}

}  // namespace lsb

namespace lsb {

// Latch whether the last classification of level glevel listed flipped cells.
__global__ void k_lsa_flipflag(const int *counters, int glevel, int *flag) {
  if (threadIdx.x == 0 && blockIdx.x == 0 && counters[glevel * NCOUNT + 2] > 0) *flag = 1;
}

cudaError_t run_lsa_flipflag(Launch L, const int *counters, int glevel, int *flag) {
  k_lsa_flipflag<<<1, 32, 0, L.stream>>>(counters, glevel, flag);
  return cudaGetLastError();
}

}  // namespace lsb
