// Passes of the level-set update over the band work list, shared by the launches of the
// forward step (lsb_ls.cu) and the replay inside the reverse sweep (lsb_adj_ls.cu): the
// per-pass forms with a band lookup per stencil point, and the barriers between the passes of
// one launch.
#pragma once
#include "lsb_device.cuh"

namespace lsb {

__device__ __forceinline__ bool in_band(const Ctx &C, const LevelDev &L, const BlockShape &S, int x, int y, int z) {
  return (C.bflag[L.block_off + block_of(L, x, y, z, S)] & BF_BAND) != 0;
}

// One Jacobi sweep of first-order upwind extension on the band (interface cells
// copy their value).  Neighbours outside the band read the committed field ut0.
// mode 2: the first sweep, which stores the plan (velocity S(phi) n, upwind side and
// band membership of each upwind neighbour, interface / boundary bits) that phi
// fixes for all sweeps of a step; 3: a sweep from the plan; 1: copy uin into ut0 on
// the band (commit).
template <int D>
__device__ __forceinline__ void d_ext_iter(const Ctx &C, BlockShape S, int glevel, const float *uin, float *uout, int mode) {
  const int nl = min(C.counters[glevel * NCOUNT + 3], C.band_cap);
  const int *lst = C.band_list + (long long)glevel * C.band_cap;
  for (int w = blockIdx.x; w < nl; w += gridDim.x) {
    const int gb = lst[w];
    int x, y, z;
    const LevelDev &L = band_cell(C, S, glevel, w, threadIdx.x, x, y, z);
    if (!L.ls_active) continue;  // frozen level set in this case
    if (x >= L.n[0] || y >= L.n[1] || z >= L.n[2]) continue;
    const long long fo = L.fine_off, NF = C.nfine;
    const long long c = cidx(L, x, y, z);
    if (mode == 1) {
      for (int a = 0; a < D; ++a) C.ut0[a * NF + fo + c] = uin[a * NF + fo + c];
      continue;
    }
    const int crd[3] = {x, y, z};
    const int str[3] = {1, L.p[0], L.p[0] * L.p[1]};
    if (mode == 3) {
      // sweep from the plan of the first sweep: same values, no normal, no band lookups
      const uint8_t pf = C.plan_f[fo + c];
      if (pf & 64) {
        for (int a = 0; a < D; ++a) uout[a * NF + fo + c] = uin[a * NF + fo + c];
        continue;
      }
      float u0[3];
      for (int b = 0; b < D; ++b) u0[b] = uin[b * NF + fo + c];
      float acc[3] = {0.f, 0.f, 0.f};
      for (int a = 0; a < D; ++a) {
        const float va = C.plan_v[a * NF + fo + c];
        const int dir = (pf >> a) & 1 ? -1 : 1;
        long long cn;
        if (pf & 128) {
          int nb[3] = {x, y, z};
          nb[a] = clampwrap(L, a, crd[a] + dir);
          cn = cidx(L, nb[0], nb[1], nb[2]);
        } else {
          cn = c + dir * str[a];
        }
        const float *src = (pf >> (3 + a)) & 1 ? uin : C.ut0;
        for (int b = 0; b < D; ++b) {
          const float un = src[b * NF + fo + cn];
          acc[b] += va * (va > 0.f ? (u0[b] - un) : (un - u0[b]));
        }
      }
      for (int b = 0; b < D; ++b) uout[b * NF + fo + c] = u0[b] - L.dtau_ext * acc[b];
      continue;
    }
    const uint8_t tg = C.tag[L.cell_off + c];
    if (tg & TAG_IFACE) {
      for (int a = 0; a < D; ++a) uout[a * NF + fo + c] = uin[a * NF + fo + c];
      C.plan_f[fo + c] = 64;
      continue;
    }
    // interior: all +-1 neighbours inside the box (direct offsets, face-neighbour band flags)
    bool inner = true;
    for (int a = 0; a < D; ++a) inner = inner && crd[a] >= 1 && crd[a] + 1 < L.n[a];
    const float *phiL = C.phi + fo;
    float nvec[3], gm = 0.f;
    uint8_t pf = inner ? 0 : 128;
    for (int a = 0; a < D; ++a) {
      if (inner) {
        nvec[a] = 0.5f * (phiL[(unsigned)c + str[a]] - phiL[(unsigned)c - str[a]]);
      } else {
        int p[3] = {x, y, z}, m[3] = {x, y, z};
        p[a] = clampwrap(L, a, crd[a] + 1);
        m[a] = clampwrap(L, a, crd[a] - 1);
        nvec[a] = 0.5f * (phiL[cidx(L, p[0], p[1], p[2])] - phiL[cidx(L, m[0], m[1], m[2])]);
      }
      gm += nvec[a] * nvec[a];
    }
    gm = sqrtf(gm);
    const float ph = phiL[c];
    const float sg = ph / sqrtf(ph * ph + 1.0f);
    float u0[3];
    for (int b = 0; b < D; ++b) u0[b] = uin[b * NF + fo + c];
    float acc[3] = {0.f, 0.f, 0.f};
    for (int a = 0; a < D; ++a) {
      const float va = gm > 0.f ? sg * nvec[a] / gm : 0.f;
      const int dir = va > 0.f ? -1 : 1;
      long long cn;
      bool inb;
      if (inner) {
        cn = c + dir * str[a];
        const int s0 = (crd[a] >> S.lg[a]) << S.lg[a];
        const int q = crd[a] + dir;
        if (q >= s0 && q < s0 + S.bs[a]) {
          inb = true;  // own block (a band block)
        } else {
          const int bstr = a == 0 ? 1 : (a == 1 ? L.nb[0] : L.nb[0] * L.nb[1]);
          inb = (C.bflag[gb + dir * bstr] & BF_BAND) != 0;
        }
      } else {
        int nb[3] = {x, y, z};
        nb[a] = clampwrap(L, a, crd[a] + dir);
        cn = cidx(L, nb[0], nb[1], nb[2]);
        inb = in_band(C, L, S, nb[0], nb[1], nb[2]);
      }
      const float *src = inb ? uin : C.ut0;
      for (int b = 0; b < D; ++b) {
        const float un = src[b * NF + fo + cn];
        acc[b] += va * (va > 0.f ? (u0[b] - un) : (un - u0[b]));
      }
      C.plan_v[a * NF + fo + c] = va;
      pf |= (dir < 0 ? 1 : 0) << a;
      pf |= (inb ? 1 : 0) << (3 + a);
    }
    for (int b = 0; b < D; ++b) uout[b * NF + fo + c] = u0[b] - L.dtau_ext * acc[b];
    C.plan_f[fo + c] = pf;
  }
}
// ------------------------------------------------------------------ transport
// Gather phi along axis a at offsets -3..+3; points in the band (and, for the
// reinitialisation, not frozen) read the stage array, others the committed phi.
template <int D>
__device__ __forceinline__ void gather7(const Ctx &C, const LevelDev &L, const BlockShape &S, const float *pin,
                                        bool use_frozen, int x, int y, int z, int a, float v[7]) {
  const int crd[3] = {x, y, z};
  for (int m = 0; m < 7; ++m) {
    int p[3] = {x, y, z};
    p[a] = clampwrap(L, a, crd[a] + m - 3);
    const long long cc = L.fine_off + cidx(L, p[0], p[1], p[2]);
    bool upd = pin != C.phi && in_band(C, L, S, p[0], p[1], p[2]);
    if (upd && use_frozen) upd = !C.frozen[cc];
    v[m] = upd ? pin[cc] : C.phi[cc];
  }
}

// gather7 for a cell of band block gb (global id) at level offset c.  When the
// seven points lie inside the box on axis a (no clamping or wrapping), they are
// read at direct offsets, and a point's band membership is its own block's
// (always in the band) or that of the face neighbour it falls into; otherwise the
// general path above.  Same values as gather7.
template <int D>
__device__ __forceinline__ void gather7f(const Ctx &C, const LevelDev &L, const BlockShape &S, int gb,
                                         const float *pin, bool use_frozen, int x, int y, int z, unsigned c, int a,
                                         float v[7]) {
  const int crd = a == 0 ? x : (a == 1 ? y : z);
  if (crd < 3 || crd + 3 >= L.n[a] || S.bs[a] < 4) {  // the fast path assumes at most one block crossed
    gather7<D>(C, L, S, pin, use_frozen, x, y, z, a, v);
    return;
  }
  const float *phiL = C.phi + L.fine_off;
  const float *pinL = pin + L.fine_off;
  const uint8_t *frzL = C.frozen + L.fine_off;
  const bool merged = pin != C.phi;
  const int str = a == 0 ? 1 : (a == 1 ? L.p[0] : L.p[0] * L.p[1]);
  const int s0 = (crd >> S.lg[a]) << S.lg[a], s1 = s0 + S.bs[a];
  const int bstr = a == 0 ? 1 : (a == 1 ? L.nb[0] : L.nb[0] * L.nb[1]);
  bool fm = false, fp = false;
  if (merged) {
    if (crd - 3 < s0) fm = (C.bflag[gb - bstr] & BF_BAND) != 0;
    if (crd + 3 >= s1) fp = (C.bflag[gb + bstr] & BF_BAND) != 0;
  }
#pragma unroll
  for (int m = 0; m < 7; ++m) {
    const int q = crd + m - 3;
    const unsigned off = c + (m - 3) * str;
    bool upd = merged && (q < s0 ? fm : (q >= s1 ? fp : true));
    if (upd && use_frozen) upd = !frzL[off];
    const float *src = upd ? pinL : phiL;  // one load from the selected array
    v[m] = src[off];
  }
}

__device__ __forceinline__ float d5m(const float v[7]) {  // left-biased, offsets -3..+2
  return (-2.f * v[0] + 15.f * v[1] - 60.f * v[2] + 20.f * v[3] + 30.f * v[4] - 3.f * v[5]) / 60.f;
}
__device__ __forceinline__ float d5p(const float v[7]) {  // mirror image
  return -(-2.f * v[6] + 15.f * v[5] - 60.f * v[4] + 20.f * v[3] + 30.f * v[2] - 3.f * v[1]) / 60.f;
}

// TVD-RK3 stage of d phi/dt = -u~ . grad phi on the band (dt = 1):
// stage 1: p1 = phi + L(phi); 2: p2 = 3/4 phi + 1/4 (p1 + L(p1)); 3: phi = 1/3 phi + 2/3 (p2 + L(p2)).
template <int D>
__device__ __forceinline__ void d_adv_stage(const Ctx &C, BlockShape S, int glevel, int stage) {
  const int nl = min(C.counters[glevel * NCOUNT + 3], C.band_cap);
  const float *pin = stage == 1 ? C.phi : (stage == 2 ? C.p1 : C.p2);
  for (int w = blockIdx.x; w < nl; w += gridDim.x) {
    int x, y, z;
    const LevelDev &L = band_cell(C, S, glevel, w, threadIdx.x, x, y, z);
    if (!L.ls_active) continue;  // frozen level set in this case
    if (x >= L.n[0] || y >= L.n[1] || z >= L.n[2]) continue;
    const long long fc = L.fine_off + cidx(L, x, y, z);
    float rhs = 0.f;
    for (int a = 0; a < D; ++a) {
      float v[7];
      gather7<D>(C, L, S, pin, false, x, y, z, a, v);  // measured faster here than gather7f
      const float ua = C.ut0[a * C.nfine + fc];
      rhs -= ua * (ua >= 0.f ? d5m(v) : d5p(v));
    }
    const float p0 = C.phi[fc];
    if (stage == 1) C.p1[fc] = p0 + rhs;
    else if (stage == 2) C.p2[fc] = 0.75f * p0 + 0.25f * (C.p1[fc] + rhs);
    else C.phi[fc] = p0 / 3.0f + (2.0f / 3.0f) * (C.p2[fc] + rhs);
  }
}
// ------------------------------------------------------------------ reinitialisation
// Frozen cells (sign change to any lattice neighbour in the box) and S(phi0).
template <int Q>
__device__ __forceinline__ void d_reinit_prep(const Ctx &C, BlockShape S, int glevel) {
  using LT = Lat<Q>;
  constexpr int D = LT::D;
  const int nl = min(C.counters[glevel * NCOUNT + 3], C.band_cap);
  for (int w = blockIdx.x; w < nl; w += gridDim.x) {
    int x, y, z;
    const LevelDev &L = band_cell(C, S, glevel, w, threadIdx.x, x, y, z);
    if (!L.ls_active) continue;  // frozen level set in this case
    if (x >= L.n[0] || y >= L.n[1] || z >= L.n[2]) continue;
    const long long fc = L.fine_off + cidx(L, x, y, z);
    const float p = C.phi[fc];
    const bool g = p >= 0.f;
    bool fr = false;
    const bool inner = x >= 1 && x + 1 < L.n[0] && y >= 1 && y + 1 < L.n[1] && (D == 2 || (z >= 1 && z + 1 < L.n[2]));
    if (inner) {  // every lattice neighbour inside the box: direct offsets
      const int p0 = L.p[0], p01 = L.p[0] * L.p[1];
#pragma unroll
      for (int i = 0; i < Q; ++i) {
        if (i == LT::REST) continue;
        if ((C.phi[fc + LT::cx(i) + LT::cy(i) * p0 + LT::cz(i) * p01] >= 0.f) != g) fr = true;
      }
    } else {
      for (int i = 0; i < Q; ++i) {
        if (i == LT::REST) continue;
        int tx = x + LT::cx(i), ty = y + LT::cy(i), tz = z + LT::cz(i);
        if (!(wrap(L, 0, tx) && wrap(L, 1, ty) && (D == 2 || wrap(L, 2, tz)))) continue;
        if ((C.phi[L.fine_off + cidx(L, tx, ty, tz)] >= 0.f) != g) fr = true;
      }
    }
    C.frozen[fc] = fr ? 1 : 0;
    C.s0[fc] = p / sqrtf(p * p + 1.0f);
  }
}
// HJ-WENO5 one-sided derivative (Jiang & Peng 2000) from the five differences: the three
// candidates, and their weighted mean.  Constant divisions are multiplications by the
// reciprocals, and the three weights gamma_k / (s_k + eps)^2 are formed as gamma_k
// prod_{j != k} (s_j + eps)^2 (the same normalised weights, one division instead of four).
__device__ __forceinline__ void weno5_candidates(float v1, float v2, float v3, float v4, float v5, float d[3]) {
  const float r3 = 1.f / 3.f, r6 = 1.f / 6.f;
  d[0] = v1 * r3 - 7.f * r6 * v2 + 11.f * r6 * v3;
  d[1] = -v2 * r6 + 5.f * r6 * v3 + v4 * r3;
  d[2] = v3 * r3 + 5.f * r6 * v4 - v5 * r6;
}
__device__ __forceinline__ float weno5_mean(float v1, float v2, float v3, float v4, float v5, const float d[3]) {
  const float eps = 1e-6f;
  const float b1 = v1 - 2.f * v2 + v3, c1 = v1 - 4.f * v2 + 3.f * v3;
  const float b2 = v2 - 2.f * v3 + v4, c2 = v2 - v4;
  const float b3 = v3 - 2.f * v4 + v5, c3 = 3.f * v3 - 4.f * v4 + v5;
  const float t1 = 13.f / 12.f * b1 * b1 + 0.25f * c1 * c1 + eps;
  const float t2 = 13.f / 12.f * b2 * b2 + 0.25f * c2 * c2 + eps;
  const float t3 = 13.f / 12.f * b3 * b3 + 0.25f * c3 * c3 + eps;
  const float q1 = t1 * t1, q2 = t2 * t2, q3 = t3 * t3;
  const float a1 = 0.1f * q2 * q3, a2 = 0.6f * q1 * q3, a3 = 0.3f * q1 * q2;
  return (a1 * d[0] + a2 * d[1] + a3 * d[2]) / (a1 + a2 + a3);
}

// Godunov's |grad phi|^2 along one axis from the seven values v at offsets -3..+3, for the
// sign of s0: max(max(d-, 0)^2, min(d+, 0)^2) for s0 > 0, the other signs otherwise, with the
// left- and right-biased derivatives d-, d+.  A derivative is a weighted mean of its
// candidates: where all three have the sign that Godunov's choice drops, the side's square
// is exactly zero and its weights are not formed (one side always in smooth regions).
__device__ __forceinline__ float godunov_axis(const float v[7], float s0) {
  const float D0 = v[1] - v[0], D1 = v[2] - v[1], D2 = v[3] - v[2], D3 = v[4] - v[3], D4 = v[5] - v[4], D5 = v[6] - v[5];
  float m[3], p[3];
  weno5_candidates(D0, D1, D2, D3, D4, m);
  weno5_candidates(D5, D4, D3, D2, D1, p);
  const bool pos = s0 > 0.f;
  const bool um = pos ? fmaxf(fmaxf(m[0], m[1]), m[2]) > 0.f : fminf(fminf(m[0], m[1]), m[2]) < 0.f;
  const bool up = pos ? fminf(fminf(p[0], p[1]), p[2]) < 0.f : fmaxf(fmaxf(p[0], p[1]), p[2]) > 0.f;
  float gm = 0.f, gp = 0.f;
  if (um) {
    const float dm = weno5_mean(D0, D1, D2, D3, D4, m), d = pos ? fmaxf(dm, 0.f) : fminf(dm, 0.f);
    gm = d * d;
  }
  if (up) {
    const float dp = weno5_mean(D5, D4, D3, D2, D1, p), d = pos ? fminf(dp, 0.f) : fmaxf(dp, 0.f);
    gp = d * d;
  }
  return fmaxf(gm, gp);
}

// TVD-RK3 stage of phi_tau = -S(phi0)(|grad phi|_G - 1) on band cells that are not frozen.
template <int D>
__device__ __forceinline__ void d_reinit_stage(const Ctx &C, BlockShape S, int glevel, int stage) {
  const int nl = min(C.counters[glevel * NCOUNT + 3], C.band_cap);
  const int *lst = C.band_list + (long long)glevel * C.band_cap;
  const float *pin = stage == 1 ? C.phi : (stage == 2 ? C.p1 : C.p2);
  for (int w = blockIdx.x; w < nl; w += gridDim.x) {
    const int gb = lst[w];
    int x, y, z;
    const LevelDev &L = band_cell(C, S, glevel, w, threadIdx.x, x, y, z);
    if (!L.ls_active) continue;  // frozen level set in this case
    if (x >= L.n[0] || y >= L.n[1] || z >= L.n[2]) continue;
    const unsigned cl = (unsigned)cidx(L, x, y, z);
    const long long fc = L.fine_off + cl;
    if (C.frozen[fc]) continue;
    const float s0 = C.s0[fc];
    float g2 = 0.f;
    for (int a = 0; a < D; ++a) {
      float v[7];
      gather7f<D>(C, L, S, gb, pin, true, x, y, z, cl, a, v);
      g2 += godunov_axis(v, s0);
    }
    const float rhs = L.dtau_reinit * (-s0 * (sqrtf(g2) - 1.0f));
    const float p0 = C.phi[fc];
    if (stage == 1) C.p1[fc] = p0 + rhs;
    else if (stage == 2) C.p2[fc] = 0.75f * p0 + 0.25f * (C.p1[fc] + rhs);
    else C.phi[fc] = p0 / 3.0f + (2.0f / 3.0f) * (C.p2[fc] + rhs);
  }
}
// ------------------------------------------------------------------ barriers between passes of a launch
// MODE 0: the grid is one thread-block cluster and the barrier is the hardware's, without a limit;
// 1: a cooperative launch (bar[0] counts arrivals).  *limit: reads of the count before the wait
// gives up (the handle's wait limit; 0 gives up at once unless the CTA is alone), in shared memory
// and written by thread 0: as a kernel parameter it had left the constant cache by the next barrier
// and cost each 0.13 us (3D bubble, 28 of them: step 691 -> 695 us).  false: it gave up, ERR_TIMEOUT
// is set, and the CTA has to leave: it arrives at no later barrier, so no CTA gets past the next
// one either.
// 2: a cooperative launch with the default limit, a constant: the reverse sweep's launch (28
// barriers) is built for it too, where a limit read from memory costs 1% (2D window 7.56 and 7.64
// ms).
constexpr unsigned kGaveUp = 1u << 16;  // (more than a cooperative grid's CTAs)
template <int MODE>
__device__ __forceinline__ bool lsf_barrier(unsigned *bar, unsigned &target, int *err, const unsigned *limit) {
  if (MODE == 0) {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    return true;
  }
  __shared__ int gave_up;
  target += gridDim.x;
  __syncthreads();
  if (MODE == 2 && threadIdx.x == 0) {
    gave_up = 0;
    unsigned v, reads = 0;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if (++reads > kDefaultWait) {
        gave_up = 1;
        atomicOr(err, ERR_TIMEOUT);
        break;
      }
    } while ((int)(v - target) < 0);
  } else if (threadIdx.x == 0) {
    gave_up = 0;
    unsigned v, left = *limit;
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    do {
      if (left-- == 0) {
        if (gridDim.x == 1) break;
        gave_up = 1;
        atomicOr(err, ERR_TIMEOUT);
        __threadfence();  // the arrival, which no read has seen yet, before the marks in bar[1]
        atomicAdd(bar + 1, kGaveUp);
        break;
      }
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
    } while ((int)(v - target) < 0);
  }
  __syncthreads();
  return gave_up == 0;
}

// Every CTA of a MODE 1 or 2 launch passes here once, last: bar[1] counts them (and, from kGaveUp
// up, those that gave up with an arrival not read back), and the last one clears both words for
// the next launch.
template <int MODE>
__device__ __forceinline__ void lsf_leave(unsigned *bar) {
  if (threadIdx.x != 0) return;
  const unsigned out = atomicAdd(bar + 1, 1u);
  if ((MODE == 2 ? out : out % kGaveUp) == gridDim.x - 1) {
    if (MODE != 2 && out >= kGaveUp) __threadfence();  // (1 us of the launch where it is not needed)
    bar[0] = 0;
    bar[1] = 0;
  }
}

}  // namespace lsb
