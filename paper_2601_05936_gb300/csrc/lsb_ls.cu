// Level-set kernels on the finest level (Sec. 2.2): phase classification and
// cut links (Sec. 2.3 radiation theorem), the narrow band, float64
// least-squares geometry, hyperbolic velocity extension (Eq.
// hyperbolicExtension), upwind-5 / TVD-RK3 transport, constrained
// reinitialisation (HJ-WENO5 Godunov, interface cells frozen), refill of cells
// that change phase (Sec. 2.4) and the refinement sensor (Sec. 2.6, 3.2.2).
//
// The narrow band is block granular: finest-level blocks holding an interface
// cell and their 3^D neighbours (active blocks only).  phi, the RK stage
// arrays and the extension velocity are dense finest-level arrays; stencil
// points outside the band read the committed fields.
#include <cooperative_groups.h>

#include <map>
#include <mutex>

#include "lsb_kernels.h"
#include "lsb_lspass.cuh"

namespace lsb {

// ------------------------------------------------------------------ classification
// A cell that changed phase: into the flip list, and the blocks around it that the previous
// band does not hold into the check list (the band flags tested here are those of the
// previous classification, which no thread of the phase pass changes).
template <int Q>
__device__ __forceinline__ void list_flip(const Ctx &C, const LevelDev &L, const BlockShape &S, int glevel, int ld,
                                       long long c, int x, int y, int z) {
  using LT = Lat<Q>;
  constexpr int D = LT::D;
  int e = atomicAdd(&C.counters[glevel * NCOUNT + 2], 1);
  if (e < C.list_cap) C.flip_list[(long long)glevel * C.list_cap + e] = make_int2(ld, (int)c);
  else atomicOr(C.err, ERR_LIST_OVF);
  for (int k = 0; k < Q; ++k) {
    int sx = x + LT::cx(k), sy = y + LT::cy(k), sz = z + LT::cz(k);
    if (!(wrap(L, 0, sx) && wrap(L, 1, sy) && (D == 2 || wrap(L, 2, sz)))) continue;
    const int nb = L.block_off + block_of(L, sx, sy, sz, S);
    // set BF_CHECK once per block (compare-and-swap on the flag's word) and list it
    unsigned *wp = reinterpret_cast<unsigned *>(C.bflag + (nb & ~3));
    const int sh = (nb & 3) * 8;
    unsigned old = *reinterpret_cast<volatile unsigned *>(wp);
    while (!(((old >> sh) & 0xffu) & (BF_BAND | BF_CHECK))) {
      const unsigned seen = atomicCAS(wp, old, old | ((unsigned)BF_CHECK << sh));
      if (seen == old) {
        const int slot = atomicAdd(&C.counters[glevel * NCOUNT + 4], 1);
        if (slot < C.band_cap) C.check_list[(long long)glevel * C.band_cap + slot] = nb;
        else atomicOr(C.err, ERR_BAND_OVF);
        break;
      }
      old = seen;
    }
  }
}

// Pass 1: phase of every leaf cell from phi (liquid iff phi < 0); flipped cells
// are listed.  init = 1 (after creation or regrid): all blocks, no flips,
// previous = current.  Otherwise only blocks of the previous band (they keep the band
// flag the previous band pass set until the link pass rewrites the flags), and every
// block next to a flipped cell (or holding one) that is not in that band gets BF_CHECK
// and a place in the check list.
template <int Q>
__global__ void k_classify_phase(Ctx C, BlockShape S, const int *list, int nlist, int glevel, int init) {
  LSB_GRID_WAIT();
  using LT = Lat<Q>;
  constexpr int D = LT::D;
  // phi changes only on band cells, so outside the previous band no phase (and no stale
  // flip bit: flips happen next to the interface, inside the band) can change: unless
  // init, the blocks are those of the previous band list
  if (!init) {
    nlist = min(C.counters[glevel * NCOUNT + 5], C.band_cap);
    list = C.band_list + (long long)glevel * C.band_cap;
    // the band count starts again for the band pass (no pass before it reads it)
    if (blockIdx.x == 0 && threadIdx.x == 0) C.counters[glevel * NCOUNT + 3] = 0;
  }
  for (int w = blockIdx.x; w < nlist; w += gridDim.x) {
    const int gb = list[w];
    int x, y, z;
    const LevelDev &L = blk_cell(C, S, gb, threadIdx.x, x, y, z);
    if (x >= L.n[0] || y >= L.n[1] || z >= L.n[2]) continue;
    const long long c = cidx(L, x, y, z);
    const uint8_t tg = C.tag[L.cell_off + c];
    if (!(tg & TAG_LEAF)) continue;
    const float ph = C.phi[L.fine_off + c];
    // the transport and reinitialisation stages of this update wrote p1, p2 on band
    // cells: back to phi, as the mirrored passes expect outside the next band
    C.p1[L.fine_off + c] = ph;
    C.p2[L.fine_off + c] = ph;
    const int gas = ph >= 0.0f ? 1 : 0;
    const int prev = init ? gas : (tg & TAG_GAS);
    const bool flip = !init && (gas != prev);
    uint8_t nt = (tg & (TAG_LEAF | TAG_RLAYER | TAG_GHOST)) | (gas ? TAG_GAS : 0) | (prev ? TAG_PREVGAS : 0) |
                 (flip ? TAG_FLIP : 0);
    C.tag[L.cell_off + c] = nt;
    if (flip) list_flip<Q>(C, L, S, glevel, C.blk_ld[gb], c, x, y, z);
  }
}

// Offsets from a cell to its neighbours at -1 and +1 along each axis (wrapped on periodic
// axes), and a mask of the sides that lie behind a wall (bit 2 a: -1, bit 2 a + 1: +1).
struct NearOff {
  int m[3], p[3];
  unsigned wall;
};
template <int D>
__device__ __forceinline__ NearOff near_off(const int crd[3], const int n[3], unsigned per, unsigned p0, unsigned p01) {
  NearOff o;
  o.wall = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    o.m[a] = o.p[a] = 0;
    if (a >= D) continue;
    const int str = a == 0 ? 1 : (int)(a == 1 ? p0 : p01);
    const bool w = (per >> a) & 1u;
    o.m[a] = crd[a] > 0 ? -str : (n[a] - 1) * str;
    o.p[a] = crd[a] < n[a] - 1 ? str : -(n[a] - 1) * str;
    if (!w && crd[a] == 0) o.wall |= 1u << (2 * a);
    if (!w && crd[a] == n[a] - 1) o.wall |= 2u << (2 * a);
  }
  return o;
}
// The offset to the neighbour in direction (x, y, z); out: it lies behind a wall.
__device__ __forceinline__ int off_to(const NearOff &o, int x, int y, int z, bool &out) {
  const unsigned need = (x < 0 ? 1u : (x > 0 ? 2u : 0u)) | (y < 0 ? 4u : (y > 0 ? 8u : 0u)) | (z < 0 ? 16u : (z > 0 ? 32u : 0u));
  out = (o.wall & need) != 0;
  return (x < 0 ? o.m[0] : (x > 0 ? o.p[0] : 0)) + (y < 0 ? o.m[1] : (y > 0 ? o.p[1] : 0)) +
         (z < 0 ? o.m[2] : (z > 0 ? o.p[2] : 0));
}
__device__ __forceinline__ unsigned per_mask(const LevelDev &L) {
  return (L.per[0] ? 1u : 0u) | (L.per[1] ? 2u : 0u) | (L.per[2] ? 4u : 0u);
}

// Cut mask of a cell with tag tg (tag pointer tc at the cell): bit k set when the source
// x - c_k is a leaf of the other phase (no source through a wall).
template <int Q>
__device__ __forceinline__ uint32_t cut_mask(const uint8_t *tc, uint8_t tg, const NearOff &o) {
  using LT = Lat<Q>;
  uint32_t m = 0;
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    if (k == LT::REST) continue;
    bool out;
    const int off = off_to(o, -LT::cx(k), -LT::cy(k), -LT::cz(k), out);
    const uint8_t ts = tc[out ? 0 : off];  // a cell is never of the other phase to itself
    if ((ts & TAG_LEAF) && ((ts ^ tg) & TAG_GAS)) m |= 1u << k;
  }
  return m;
}

// The same for a cell with every source in the box.
template <int Q>
__device__ __forceinline__ uint32_t cut_mask_inner(const uint8_t *tc, uint8_t tg, long long p0, long long p01) {
  using LT = Lat<Q>;
  uint32_t m = 0;
#pragma unroll
  for (int k = 0; k < Q; ++k) {
    if (k == LT::REST) continue;
    const uint8_t ts = tc[-(LT::cx(k) + LT::cy(k) * p0 + LT::cz(k) * p01)];
    if ((ts & TAG_LEAF) && ((ts ^ tg) & TAG_GAS)) m |= 1u << k;
  }
  return m;
}

// Slots of a warp's cut links and interface cells in the lists (one atomic pair per warp;
// every lane of the warp calls this), then the entries, the link base and TAG_IFACE of the
// cell (ld, c) with cut mask m; fc and tc: its finest-level and tag indices.
__device__ __forceinline__ void list_links(const Ctx &C, int glevel, uint32_t m, int ld, int c, long long fc,
                                           long long tc, uint8_t tg) {
  const int lane = threadIdx.x & 31;
  const unsigned wcells = __ballot_sync(0xffffffffu, m != 0);
  if (!wcells) return;
  const int np = __popc(m);
  int incl = np;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const int wlinks = __shfl_sync(0xffffffffu, incl, 31);
  int lbase = 0, cbase0 = 0;
  if (lane == 0) {
    lbase = atomicAdd(&C.counters[glevel * NCOUNT + 0], wlinks);
    cbase0 = atomicAdd(&C.counters[glevel * NCOUNT + 1], __popc(wcells));
  }
  lbase = __shfl_sync(0xffffffffu, lbase, 0);
  cbase0 = __shfl_sync(0xffffffffu, cbase0, 0);
  if (!m) return;
  const int base = lbase + incl - np;
  if ((long long)base + np > C.link_cap) atomicOr(C.err, ERR_LINK_OVF);
  C.cbase[fc] = base;
  // the link list: one entry per cut link, in link-buffer order
  const int2 cell = make_int2(ld, c);
  uint32_t mm = m;
  for (int r = 0; mm; ++r) {
    const int k = __ffs(mm) - 1;
    mm &= mm - 1u;
    if ((long long)base + r < C.link_cap) {
      C.link_cell[C.link_list_off[glevel] + base + r] = cell;
      C.link_dir[C.link_list_off[glevel] + base + r] = (uint8_t)k;
    }
  }
  C.tag[tc] = tg | TAG_IFACE;
  const int e = cbase0 + __popc(wcells & ((1u << lane) - 1u));
  if (e < C.list_cap) C.iface_list[(long long)glevel * C.list_cap + e] = cell;
  else atomicOr(C.err, ERR_LIST_OVF);
}

// Pass 2: cut mask of every leaf cell (bit k: source x - c_k is a leaf of the
// other phase), link base, interface list, block interface flag.  Unless full,
// only blocks of the previous band and blocks next to a flipped cell are
// examined: phi changes only on band cells, so a cut link elsewhere would need a
// neighbour that flipped; every other block has no cut link now and, having left
// the band with none, an all-zero mask already.
template <int Q>
__global__ void k_classify_links(Ctx C, BlockShape S, const int *list, int nlist, int glevel, int full) {
  LSB_GRID_WAIT();
  using LT = Lat<Q>;
  constexpr int D = LT::D;
  // unless full: the previous band list, then the check list (every other block keeps
  // flag 0 and an all-zero mask)
  int nband = nlist;
  if (!full) {
    nband = min(C.counters[glevel * NCOUNT + 5], C.band_cap);
    nlist = nband + min(C.counters[glevel * NCOUNT + 4], C.band_cap);
    list = C.band_list + (long long)glevel * C.band_cap;
  }
  const int *chk = C.check_list + (long long)glevel * C.band_cap;
  for (int w = blockIdx.x; w < nlist; w += gridDim.x) {
    const int gb = w < nband ? list[w] : chk[w - nband];
    const bool work = full || (C.bflag[gb] & (BF_BAND | BF_CHECK));
    __syncthreads();  // every thread has read the flags before thread 0 rewrites them
    if (!work) {
      if (threadIdx.x == 0) C.bflag[gb] = 0;
      continue;
    }
    int x, y, z;
    const LevelDev &L = blk_cell(C, S, gb, threadIdx.x, x, y, z);
    uint32_t m = 0;
    long long c = 0;
    uint8_t tg = 0;
    if (x < L.n[0] && y < L.n[1] && z < L.n[2]) {
      c = cidx(L, x, y, z);
      tg = C.tag[L.cell_off + c];
      if (tg & TAG_LEAF) {
        const int crd[3] = {x, y, z};
        m = cut_mask<Q>(C.tag + L.cell_off + c, tg,
                        near_off<D>(crd, L.n, per_mask(L), (unsigned)L.p[0], (unsigned)(L.p[0] * L.p[1])));
        C.cmask[L.fine_off + c] = m;
      }
    }
    list_links(C, glevel, m, C.blk_ld[gb], (int)c, L.fine_off + c, L.cell_off + c, tg);
    const bool any = __syncthreads_or(m != 0);
    if (threadIdx.x == 0) C.bflag[gb] = any ? BF_IFACE : 0;
  }
}

// Pass 3: band flag of every active finest block (itself or a 3^D neighbour
// holds an interface cell); band blocks are listed.  One warp per block, lane k
// reading the flags of neighbour k, so the 3^D loads are in flight together.
// On the CTAs [b0, b0 + nb) of the launch.
template <int Q>
__device__ __forceinline__ void d_band(const Ctx &C, const int *list, int nlist, int glevel, int b0, int nb) {
  constexpr int D = Lat<Q>::D;
  constexpr int NN = D == 3 ? 27 : 9;
  const int lane = threadIdx.x & 31;
  const int wpb = blockDim.x >> 5;
  for (int w = ((int)blockIdx.x - b0) * wpb + (threadIdx.x >> 5); w < nlist; w += nb * wpb) {
    const int gb = list[w];
    const LevelDev &L = C.lds[C.blk_ld[gb]];
    bool hot = false;
    if (lane < NN) {
      const int lb = gb - L.block_off;
      int nb3[3] = {lb % L.nb[0] + lane % 3 - 1, (lb / L.nb[0]) % L.nb[1] + (lane / 3) % 3 - 1,
                    lb / (L.nb[0] * L.nb[1]) + (D == 3 ? lane / 9 - 1 : 0)};
      bool ok = true;
      for (int a = 0; a < D; ++a) {
        if (nb3[a] < 0 || nb3[a] >= L.nb[a]) {
          if (L.per[a]) nb3[a] = (nb3[a] + L.nb[a]) % L.nb[a];
          else ok = false;
        }
      }
      if (ok) hot = (C.bflag[L.block_off + nb3[0] + L.nb[0] * (nb3[1] + L.nb[1] * nb3[2])] & BF_IFACE) != 0;
    }
    const bool band = __any_sync(0xffffffffu, hot);
    if (lane == 0 && band && C.bstat[gb] == BLK_LEAF) {
      C.bflag[gb] = C.bflag[gb] | BF_BAND;
      const int e = atomicAdd(&C.counters[glevel * NCOUNT + 3], 1);
      if (e < C.band_cap) {
        C.band_list[(long long)glevel * C.band_cap + e] = gb;
        C.band_info[(long long)glevel * C.band_cap + e] = C.blk_info[gb];
      } else {
        atomicOr(C.err, ERR_BAND_OVF);
      }
    }
  }
}

// ------------------------------------------------------------------ geometry (float64)
// Unweighted least-squares quadratic over the 3^D stencil.  With offsets in
// {-1,0,1}^D the odd basis functions decouple: grad_a = sum(o_a phi)/sum(o_a^2),
// H_ab = sum(o_a o_b phi)/sum(o_a^2 o_b^2) (a != b); the constant and pure
// quadratic coefficients solve the 1 + D even normal equations in closed form.
// n = g/|g|, kappa = (|g|^2 tr H - g.H.g)/|g|^3.
// The fit from the stencil sums (exact integers in units of 2^-30): n and kappa.
// The fit's coefficients are fixed rational combinations of the stencil sums.  In 2D
// (9 points: sum o^2 = 6, sum o_x^2 o_y^2 = 4, sum o^4 = 6) g_a = S_a / 6, H_aa =
// (3 S_aa - 2 P) / 3, H_xy = S_xy / 4; in 3D (27 points: 18, 12, 18) g_a = S_a / 18,
// H_aa = (3 S_aa - 2 P) / 9, H_ab = S_ab / 12.  In the unit 1 / (12 * 2^30) (2D) or
// 1 / (36 * 2^30) (3D) both read g = 2 G and H = K with the integers G_a = S_a,
// K_aa = 4 (3 S_aa - 2 P), K_ab = 3 S_ab, and kappa, homogeneous of degree zero in
// (g, H), is (|G|^2 tr K - G.K.G) / (2 |G|^3): float64 from exact integers, one
// square root and two divisions.
template <int D>
__device__ __forceinline__ void fit_from_sums(long long iP, const long long isx[3], const long long isxx[3],
                                              const long long isxy[3], float n[3], float &kappa) {
  double G[3] = {0, 0, 0}, K[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
  for (int a = 0; a < D; ++a) {
    G[a] = (double)isx[a];
    K[a][a] = (double)(4 * (3 * isxx[a] - 2 * iP));
  }
  K[0][1] = K[1][0] = (double)(3 * isxy[0]);
  if (D == 3) {
    K[0][2] = K[2][0] = (double)(3 * isxy[1]);
    K[1][2] = K[2][1] = (double)(3 * isxy[2]);
  }
  double g2 = 0, tr = 0, gKg = 0;
  for (int a = 0; a < D; ++a) {
    g2 += G[a] * G[a];
    tr += K[a][a];
    for (int b = 0; b < D; ++b) gKg += G[a] * K[a][b] * G[b];
  }
  const double mag = sqrt(g2);
  n[0] = n[1] = n[2] = 0.f;
  kappa = 0.f;
  // |grad phi| = |G| / (6 or 18) / 2^30
  if (mag > 1e-12 * (D == 2 ? 6.0 : 18.0) * 1073741824.0) {
    const double inv = 1.0 / mag;
    for (int a = 0; a < D; ++a) n[a] = (float)(G[a] * inv);
    kappa = (float)((g2 * tr - gKg) / (2.0 * g2 * mag));
  }
}
// phi in fixed point with 30 fraction bits (exact for |phi| >= 2^-6, within 2^-31 below): the
// stencil sums are exact in 64-bit integers, so the float64 work of the fit is its closed form
// only (GB300 runs float64 at a small fraction of its integer rate).
__device__ __forceinline__ long long phi_fixed(float p) { return __float2ll_rn(p * 1073741824.0f); }

// The interface cells, one thread each, on the CTAs [b0, b0 + nb) of the launch.
template <int D>
__device__ __forceinline__ void d_geometry(const Ctx &C, int glevel, int b0, int nb) {
  const int ni = min(C.counters[glevel * NCOUNT + 1], (int)C.list_cap);
  const int2 *li = C.iface_list + (long long)glevel * C.list_cap;
  for (int e = ((int)blockIdx.x - b0) * blockDim.x + threadIdx.x; e < ni; e += nb * blockDim.x) {
    const int2 it = li[e];
    const LevelDev &L = C.lds[it.x];
    const long long c = it.y;
    int x, y, z;
    cell_xyz(L, c, x, y, z);
    long long iP = 0, isx[3] = {0, 0, 0}, isxx[3] = {0, 0, 0}, isxy[3] = {0, 0, 0};
    // cells whose 3^D stencil lies inside the box read it at direct offsets
    const bool inner = x >= 1 && x + 1 < L.n[0] && y >= 1 && y + 1 < L.n[1] && (D == 2 || (z >= 1 && z + 1 < L.n[2]));
    const long long p0 = L.p[0], p01 = (long long)L.p[0] * L.p[1];
#pragma unroll
    for (int oz = (D == 3 ? -1 : 0); oz <= (D == 3 ? 1 : 0); ++oz)
#pragma unroll
      for (int oy = -1; oy <= 1; ++oy)
#pragma unroll
        for (int ox = -1; ox <= 1; ++ox) {
          long long cc;
          if (inner) {
            cc = c + ox + oy * p0 + oz * p01;
          } else {
            const int xx = clampwrap(L, 0, x + ox), yy = clampwrap(L, 1, y + oy);
            const int zz = D == 3 ? clampwrap(L, 2, z + oz) : 0;
            cc = cidx(L, xx, yy, zz);
          }
          const long long v = phi_fixed(C.phi[L.fine_off + cc]);
          const int o[3] = {ox, oy, oz};
          iP += v;
          for (int a = 0; a < D; ++a) {
            isx[a] += o[a] > 0 ? v : (o[a] < 0 ? -v : 0);
            isxx[a] += o[a] != 0 ? v : 0;
          }
          isxy[0] += ox * oy > 0 ? v : (ox * oy < 0 ? -v : 0);
          if (D == 3) {
            isxy[1] += ox * oz > 0 ? v : (ox * oz < 0 ? -v : 0);
            isxy[2] += oy * oz > 0 ? v : (oy * oz < 0 ? -v : 0);
          }
        }
    float n[3], kap;
    fit_from_sums<D>(iP, isx, isxx, isxy, n, kap);
    const long long fc = L.fine_off + c;
    for (int a = 0; a < D; ++a) C.nvec[a * C.nfine + fc] = n[a];
    C.kappa[fc] = kap;
  }
}
template <int D>
__global__ void k_geometry(Ctx C, int glevel) {
  LSB_GRID_WAIT();
  d_geometry<D>(C, glevel, 0, gridDim.x);
}

// ------------------------------------------------------------------ forward passes on mirrored stage arrays
// The forward step keeps the stage arrays equal to the committed fields at every finest
// cell outside the band when a level-set update starts: p1 = p2 = phi, and both sweep
// buffers = ut0.  Band cells restore this during each update (u~ in the first transport
// stage, which also commits the extension; phi in the phase pass of the classification),
// and the host fills the arrays in full after creation and after every restore of phi or
// u~.  A stencil point then reads the stage array wherever it lies, so the passes below
// need no band or frozen-cell lookups; frozen cells of the reinitialisation write phi into
// the stage arrays their neighbours read.  The arithmetic and its order are those of the
// passes above, so the results are the same bit for bit.

// seven values of the stage array along axis a at offsets -3..+3 (clamped or
// wrapped at the box faces like gather7)
__device__ __forceinline__ void gather7m(const LevelDev &L, const float *pinL, int x, int y, int z, unsigned c, int a,
                                         float v[7]) {
  const int crd = a == 0 ? x : (a == 1 ? y : z);
  if (crd >= 3 && crd + 3 < L.n[a]) {
    const int str = a == 0 ? 1 : (a == 1 ? L.p[0] : L.p[0] * L.p[1]);
#pragma unroll
    for (int m = 0; m < 7; ++m) v[m] = pinL[c + (m - 3) * str];
  } else {
#pragma unroll
    for (int m = 0; m < 7; ++m) {
      int p[3] = {x, y, z};
      p[a] = clampwrap(L, a, crd + m - 3);
      v[m] = pinL[cidx(L, p[0], p[1], p[2])];
    }
  }
}

// The forward step's sweep buffers hold u~ interleaved (a vector per cell, so that a
// neighbour is one load): two floats in 2D, four in 3D.
template <int D> struct UVec;
template <> struct UVec<2> { using T = float2; };
template <> struct UVec<3> { using T = float4; };
__device__ __forceinline__ void u_get(const float2 &v, float u[3]) { u[0] = v.x; u[1] = v.y; }
__device__ __forceinline__ void u_get(const float4 &v, float u[3]) { u[0] = v.x; u[1] = v.y; u[2] = v.z; }
__device__ __forceinline__ void u_put(float2 &v, const float u[3], float) { v = make_float2(u[0], u[1]); }
__device__ __forceinline__ void u_put(float4 &v, const float u[3], float w) { v = make_float4(u[0], u[1], u[2], w); }

// First extension sweep at one band cell (mode 2 of d_ext_iter): sweep from ut0 into the
// buffer uout and store the plan (S(phi) n, upwind sides, interface and box-boundary bits).
template <int D>
__device__ __forceinline__ void ext_first_cell(const Ctx &C, const LevelDev &L, int x, int y, int z,
                                               typename UVec<D>::T *uout) {
  const long long fo = L.fine_off, NF = C.nfine;
  const long long c = cidx(L, x, y, z);
  float u0[3];
  for (int b = 0; b < D; ++b) u0[b] = C.ut0[b * NF + fo + c];
  if (C.tag[L.cell_off + c] & TAG_IFACE) {
    u_put(uout[fo + c], u0, 0.f);
    C.plan_f[fo + c] = 64;
    return;
  }
  const int crd[3] = {x, y, z};
  const int str[3] = {1, L.p[0], L.p[0] * L.p[1]};
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
  float acc[3] = {0.f, 0.f, 0.f};
  for (int a = 0; a < D; ++a) {
    const float va = gm > 0.f ? sg * nvec[a] / gm : 0.f;
    const int dir = va > 0.f ? -1 : 1;
    long long cn;
    if (inner) {
      cn = c + dir * str[a];
    } else {
      int nb[3] = {x, y, z};
      nb[a] = clampwrap(L, a, crd[a] + dir);
      cn = cidx(L, nb[0], nb[1], nb[2]);
    }
    for (int b = 0; b < D; ++b) {
      const float un = C.ut0[b * NF + fo + cn];
      acc[b] += va * (va > 0.f ? (u0[b] - un) : (un - u0[b]));
    }
    C.plan_v[a * NF + fo + c] = va;
    pf |= (dir < 0 ? 1 : 0) << a;
  }
  for (int b = 0; b < D; ++b) u0[b] = u0[b] - L.dtau_ext * acc[b];
  u_put(uout[fo + c], u0, 0.f);
  C.plan_f[fo + c] = pf;
}

// A later extension sweep at one band cell, from the stored plan.
template <int D>
__device__ __forceinline__ void ext_sweep_cell(const Ctx &C, const LevelDev &L, int x, int y, int z,
                                               const typename UVec<D>::T *uin, typename UVec<D>::T *uout) {
  const long long NF = C.nfine, c = cidx(L, x, y, z);
  const typename UVec<D>::T *ui = uin + L.fine_off;
  const uint8_t pf = C.plan_f[L.fine_off + c];
  float u0[3];
  u_get(ui[c], u0);
  if (!(pf & 64)) {
    float acc[3] = {0.f, 0.f, 0.f};
    for (int a = 0; a < D; ++a) {
      const float va = C.plan_v[a * NF + L.fine_off + c];
      const int dir = (pf >> a) & 1 ? -1 : 1;
      long long cn;
      if (pf & 128) {  // box-boundary cell: the neighbour clamped or wrapped
        int nb[3] = {x, y, z};
        nb[a] = clampwrap(L, a, nb[a] + dir);
        cn = cidx(L, nb[0], nb[1], nb[2]);
      } else {
        cn = c + dir * (a == 0 ? 1LL : (a == 1 ? (long long)L.p[0] : (long long)L.p[0] * L.p[1]));
      }
      float un[3];
      u_get(ui[cn], un);
      for (int b = 0; b < D; ++b) acc[b] += va * (va > 0.f ? (u0[b] - un[b]) : (un[b] - u0[b]));
    }
    for (int b = 0; b < D; ++b) u0[b] = u0[b] - L.dtau_ext * acc[b];
  }
  u_put(uout[L.fine_off + c], u0, 0.f);
}

// TVD-RK3 transport stage at one band cell (as d_adv_stage).  Stage 1 takes u~ from the
// last extension sweep (ufin; nullptr: ut0, no sweeps) and commits it to ut0; stage 2 also to
// both sweep buffers at the cell.
template <int D>
__device__ __forceinline__ void adv_cell(const Ctx &C, const LevelDev &L, int x, int y, int z, int stage,
                                         const typename UVec<D>::T *ufin, typename UVec<D>::T *ub1,
                                         typename UVec<D>::T *ub2) {
  const float *pin = stage == 1 ? C.phi : (stage == 2 ? C.p1 : C.p2);
  const long long NF = C.nfine;
  const unsigned c = (unsigned)cidx(L, x, y, z);
  const long long fc = L.fine_off + c;
  float ua[3];
  if (stage == 1 && ufin) u_get(ufin[fc], ua);
  else
    for (int a = 0; a < D; ++a) ua[a] = C.ut0[a * NF + fc];
  if (stage == 1)
    for (int a = 0; a < D; ++a) C.ut0[a * NF + fc] = ua[a];
  if (stage == 2) {  // (not in stage 1, beside which the last sweep may still run)
    u_put(ub1[fc], ua, 0.f);
    u_put(ub2[fc], ua, 0.f);
  }
  const float *pinL = pin + L.fine_off;
  float rhs = 0.f;
  for (int a = 0; a < D; ++a) {
    float v[7];
    gather7m(L, pinL, x, y, z, c, a, v);
    rhs -= ua[a] * (ua[a] >= 0.f ? d5m(v) : d5p(v));
  }
  const float p0 = C.phi[fc];
  if (stage == 1) C.p1[fc] = p0 + rhs;
  else if (stage == 2) C.p2[fc] = 0.75f * p0 + 0.25f * (C.p1[fc] + rhs);
  else C.phi[fc] = p0 / 3.0f + (2.0f / 3.0f) * (C.p2[fc] + rhs);
}

// Whether the level set changes sign between a cell (value p0, at phi) and a lattice neighbour.
template <int Q>
__device__ __forceinline__ bool sign_change(const float *phi, float p0, const NearOff &o) {
  using LT = Lat<Q>;
  const bool g = p0 >= 0.f;
  bool fr = false;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    if (i == LT::REST) continue;
    bool out;
    const int off = off_to(o, LT::cx(i), LT::cy(i), LT::cz(i), out);
    if ((phi[out ? 0 : off] >= 0.f) != g) fr = true;
  }
  return fr;
}

// The same for a cell with every neighbour in the box.
template <int Q>
__device__ __forceinline__ bool sign_change_inner(const float *phi, float p0, long long q0, long long q01) {
  using LT = Lat<Q>;
  const bool g = p0 >= 0.f;
  bool fr = false;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    if (i == LT::REST) continue;
    if ((phi[LT::cx(i) + LT::cy(i) * q0 + LT::cz(i) * q01] >= 0.f) != g) fr = true;
  }
  return fr;
}

// Reinitialisation stage at one band cell (as d_reinit_stage); with prep set (first stage
// of the first pseudo step) it also finds the frozen cells and S(phi0) as d_reinit_prep
// does.  Frozen cells leave phi as it is and write it into the stage array of stages 1, 2.
template <int Q>
__device__ __forceinline__ void reinit_cell(const Ctx &C, const LevelDev &L, int x, int y, int z, int stage, int prep) {
  constexpr int D = Lat<Q>::D;
  const float *pin = stage == 1 ? C.phi : (stage == 2 ? C.p1 : C.p2);
  const unsigned cl = (unsigned)cidx(L, x, y, z);
  const long long fc = L.fine_off + cl;
  const float p0 = C.phi[fc];
  bool fr;
  float s0;
  if (prep) {
    const int crd[3] = {x, y, z};
    fr = sign_change<Q>(C.phi + fc, p0, near_off<D>(crd, L.n, per_mask(L), (unsigned)L.p[0], (unsigned)(L.p[0] * L.p[1])));
    s0 = p0 / sqrtf(p0 * p0 + 1.0f);
    C.frozen[fc] = fr ? 1 : 0;
    C.s0[fc] = s0;
  } else {
    fr = C.frozen[fc] != 0;
    s0 = C.s0[fc];
  }
  if (fr) {
    if (stage == 1) C.p1[fc] = p0;
    else if (stage == 2) C.p2[fc] = p0;
    return;
  }
  const float *pinL = pin + L.fine_off;
  float g2 = 0.f;
  for (int a = 0; a < D; ++a) {
    float v[7];
    gather7m(L, pinL, x, y, z, cl, a, v);
    g2 += godunov_axis(v, s0);
  }
  const float rhs = L.dtau_reinit * (-s0 * (sqrtf(g2) - 1.0f));
  if (stage == 1) C.p1[fc] = p0 + rhs;
  else if (stage == 2) C.p2[fc] = 0.75f * p0 + 0.25f * (C.p1[fc] + rhs);
  else C.phi[fc] = p0 / 3.0f + (2.0f / 3.0f) * (C.p2[fc] + rhs);
}

// ------------------------------------------------------------------ the level-set update in one launch
// Everything the level set does in a finest sub-step after the interface pass, in one
// launch: n_ext extension sweeps, three transport stages, the reinitialisation, and the
// phase and cut-link passes of the classification (16 passes by default), with a barrier
// between them but for two places where a pass needs its own cells' values only: the first
// transport stage behind the last sweep, and the phases behind the last stage (barriers there
// cost 3 us of the launch's 47 over the 2D ensemble, 6 of 157 on the 3D bubble).  As launches of their own the passes are bound by their chains: ~1 us
// for the launch, then band count, band entry, level descriptor, plan, neighbours, one L2
// round trip each.  Here a CTA's cells stay its own for all passes: each thread sets up
// its band cells once (slots) and keeps their offsets, flags, extension velocity and
// current values in shared memory, so a pass is one round of neighbour loads and stores.
//
// MODE 0: the grid is one thread-block cluster and the barrier is the cluster's.
// MODE 1: a cooperative launch; the barrier counts arrivals in bar[0] (one release-add per
// CTA, polled up to the handle's wait limit; a barrier that gives up sets ERR_TIMEOUT and ends
// the CTA).  bar[1] counts CTAs that left: the last one clears both words for the next launch.
// Measured per pass, one store and two neighbour loads per thread: a launch of its own in a
// captured graph 3.8 us, grid barrier 1.4 us (152 CTAs), cluster barrier 0.6 - 1.0 us
// (16 CTAs of 256 - 1024 threads).
//
// Slots: a sweep of the grid covers gridDim.x * blockDim.x cells = GB whole band blocks
// (blockDim.x is a multiple of the block's cells); slot k of a thread is its cell in the
// k-th such group.  The first kcap slots live in shared memory; cells beyond (the band grew
// since the launch was sized) take the passes' per-cell functions above, with the plan in
// global memory.  The arithmetic and its order are those functions', so the results are
// the same bit for bit.  No load here may go through the read-only path: every array
// changes during the launch.
struct __align__(16) LsfGeo {  // what the passes need of a level descriptor
  int p0, p01;          // strides
  float dte, dtr;
  int n[3];
  unsigned per;         // periodic axes; bit 3: the case's level set moves
  long long tag_delta;  // tag index of a cell - its finest-level index
  unsigned fo;          // offset in the finest-level arrays
};
__device__ __forceinline__ LsfGeo lsf_geo(const LevelDev &L) {
  LsfGeo g;
  g.p0 = L.p[0];
  g.p01 = L.p[0] * L.p[1];
  g.fo = (unsigned)L.fine_off;
  for (int a = 0; a < 3; ++a) g.n[a] = L.n[a];
  g.per = per_mask(L) | (L.ls_active ? 8u : 0u);
  g.dte = L.dtau_ext;
  g.dtr = L.dtau_reinit;
  g.tag_delta = L.cell_off - L.fine_off;
  return g;
}
constexpr int kLsfGeo = 192;              // level descriptors with an entry in shared memory
enum : unsigned {  // slot flags
  SL_NEAR = 1,      // << axis: a stencil point three cells along the axis lies outside the box
  SL_IFACE = 8,     // interface cell: keeps its u~
  SL_EDGE = 16,     // a lattice neighbour lies outside the box
  SL_CELL = 32,     // a cell of the box
  SL_LIVE = 64,     // ... of a case whose level set moves
  SL_FROZEN = 128,  // reinitialisation: frozen
  SL_DIST = 8,      // 12 bits from here: lsf_dist
  SL_LD = 20        // the bits above: the cell's level descriptor
};
constexpr int kLsfMaxLd = 1 << (32 - SL_LD);  // more level descriptors: a launch per pass
// How far a cell lies from the box faces, up to three cells: per axis 2 bits towards the low
// face, 2 towards the high one.
template <int D>
__device__ __forceinline__ unsigned lsf_dist(const int crd[3], const int n[3]) {
  unsigned d = 0;
#pragma unroll
  for (int a = 0; a < D; ++a) d |= (unsigned)(min(crd[a], 3) | (min(n[a] - 1 - crd[a], 3) << 2)) << (4 * a);
  return d;
}
// The step d along axis a kept in the box: clamped at walls, wrapped on periodic axes.
__device__ __forceinline__ int lsf_step(const LsfGeo &g, unsigned dist, int a, int d) {
  const int lo = (int)((dist >> (4 * a)) & 3u), hi = (int)((dist >> (4 * a + 2)) & 3u);
  if ((g.per >> a) & 1u) {
    // lo, hi are exact where d reaches past them (|d| <= 3)
    if (d < -lo) {
      do d += g.n[a]; while (d < -lo);
    } else if (d > hi) {
      do d -= g.n[a]; while (d > hi);
    }
    return d;
  }
  return min(max(d, -lo), hi);
}
// The offsets of near_off from the distances.
template <int D>
__device__ __forceinline__ NearOff lsf_near(const LsfGeo &g, unsigned dist) {
  int crd[3] = {0, 0, 0}, n[3] = {1, 1, 1};
  // stands in for the coordinate: only its being 0 or n - 1 counts, beside n itself
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const unsigned lo = (dist >> (4 * a)) & 3u, hi = (dist >> (4 * a + 2)) & 3u;
    n[a] = g.n[a];
    crd[a] = lo == 0 ? 0 : (hi == 0 ? n[a] - 1 : 1);
  }
  return near_off<D>(crd, n, g.per, (unsigned)g.p0, (unsigned)g.p01);
}

// A slot in shared memory: kcap planes of 1024 threads of each field (constant strides, so
// a slot's fields sit at constant offsets).  v: S(phi) n during the sweeps, then phi and the
// last stage value in its first two words; u: u~, then S(phi0) of the reinitialisation in
// its first word.
template <int D> struct LsfSlot {
  using V = typename UVec<D>::T;
  V v[1024], u[1024];
  unsigned fc[1024], fl[1024];  // finest-level index, flags
};
template <int Q, int MODE>
__global__ void __launch_bounds__(1024, 1) k_levelset_fused(Ctx C, BlockShape S, int glevel, int n_ext, int n_re, int nld,
                                                            int kcap, unsigned *bar, unsigned limit) {
  constexpr int D = Lat<Q>::D;
  using V = typename UVec<D>::T;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  extern __shared__ __align__(16) unsigned char lsf_sm[];
  __shared__ LsfGeo geo[kLsfGeo];
  __shared__ int hot[32];  // link pass: a cut link in each of the CTA's blocks
  __shared__ unsigned wait_limit;
  LsfSlot<D> *const SM = reinterpret_cast<LsfSlot<D> *>(lsf_sm);
  const int T = blockDim.x, tid = threadIdx.x;
  if (tid == 0) wait_limit = limit;
  const int lgnt = S.lg[0] + S.lg[1] + S.lg[2];
  const int t = tid & ((1 << lgnt) - 1);
  const int GB = (int)((gridDim.x * (unsigned)T) >> lgnt);         // band blocks per sweep of the grid
  const int w0 = (int)((blockIdx.x * (unsigned)T + tid) >> lgnt);  // this thread's block in the first
  const long long NF = C.nfine;
  V *const ub1 = reinterpret_cast<V *>(C.ut1), *const ub2 = reinterpret_cast<V *>(C.ut2);
  int *cnt = C.counters + glevel * NCOUNT;
  const int4 *info = C.band_info + (long long)glevel * C.band_cap;
  // the first band entry is fetched beside the band count, not after it
  int4 bi = info[min(w0, C.band_cap - 1)];
  const int nl = min(cnt[3], C.band_cap);
  const int kn = (nl + GB - 1) / GB, ks = min(kn, kcap);
  unsigned target = 0;
  for (int i = tid; i < min(nld, kLsfGeo); i += T) geo[i] = lsf_geo(C.lds[i]);
  auto geo_of = [&](unsigned ld) { return ld < (unsigned)kLsfGeo ? geo[ld] : lsf_geo(C.lds[ld]); };
  // a cell beyond the slots: its level descriptor and coordinates (ok: a live cell of the box)
  auto beyond = [&](int k, int &x, int &y, int &z, bool &ok) -> const LevelDev & {
    const int w = w0 + k * GB;
    ok = w < nl;
    const LevelDev &L = band_cell_at(C, S, ok ? info[w] : info[0], t, x, y, z);
    ok = ok && L.ls_active && x < L.n[0] && y < L.n[1] && z < L.n[2];
    return L;
  };
  auto leave = [&]() {
    if (MODE == 1) lsf_leave<MODE>(bar);
  };
  __syncthreads();
  // ---- slots, and the first extension sweep with the plan
  for (int k = 0; k < ks; ++k) {
    const int w = w0 + k * GB;
    const int4 b = bi;
    if (w + GB < nl) bi = info[w + GB];
    unsigned fl = 0;
    if (w < nl) {
      const LsfGeo g = geo_of((unsigned)b.x);
      const int crd[3] = {(b.y << S.lg[0]) + (t & (S.bs[0] - 1)), (b.z << S.lg[1]) + ((t >> S.lg[0]) & (S.bs[1] - 1)),
                          (b.w << S.lg[2]) + (t >> (S.lg[0] + S.lg[1]))};
      if (crd[0] < g.n[0] && crd[1] < g.n[1] && crd[2] < g.n[2]) {
        const unsigned fc = g.fo + (unsigned)crd[0] + (unsigned)(g.p0 * crd[1] + g.p01 * crd[2]);
        const unsigned dist = lsf_dist<D>(crd, g.n);
        fl = SL_CELL | ((g.per & 8u) ? SL_LIVE : 0u) | (dist << SL_DIST) | ((unsigned)b.x << SL_LD);
        bool edge = false;
#pragma unroll
        for (int a = 0; a < D; ++a) {
          edge = edge || crd[a] < 1 || crd[a] + 1 >= g.n[a];
          if (crd[a] < 3 || crd[a] + 3 >= g.n[a]) fl |= SL_NEAR << a;
        }
        if (edge) fl |= SL_EDGE;
        SM[k].fc[tid] = fc;
        if (fl & SL_LIVE) {
          // one round of loads: the cell's tag, phi around it, its u~
          const uint8_t tg = C.tag[(long long)fc + g.tag_delta];
          int om[3], op[3];
          float u0[3] = {0.f, 0.f, 0.f}, pm[3], pp[3], va[3] = {0.f, 0.f, 0.f};
#pragma unroll
          for (int a = 0; a < D; ++a) {
            const int str = a == 0 ? 1 : (a == 1 ? g.p0 : g.p01);
            om[a] = -str;
            op[a] = str;
            if (edge) {
              om[a] = lsf_step(g, dist, a, -1) * str;
              op[a] = lsf_step(g, dist, a, 1) * str;
            }
            pm[a] = C.phi[fc + (unsigned)om[a]];
            pp[a] = C.phi[fc + (unsigned)op[a]];
            u0[a] = C.ut0[a * NF + fc];
          }
          const float ph = C.phi[fc];
          if (tg & TAG_IFACE) {
            fl |= SL_IFACE;
            if (n_ext > 0) u_put(ub1[fc], u0, 0.f);
          } else if (n_ext > 0) {
            float nvec[3], gm = 0.f, un[D][3];
#pragma unroll
            for (int a = 0; a < D; ++a) {
              nvec[a] = 0.5f * (pp[a] - pm[a]);
              gm += nvec[a] * nvec[a];
            }
            gm = sqrtf(gm);
            const float sg = ph / sqrtf(ph * ph + 1.0f);
#pragma unroll
            for (int a = 0; a < D; ++a) {
              va[a] = gm > 0.f ? sg * nvec[a] / gm : 0.f;
              const unsigned cn = fc + (unsigned)(va[a] > 0.f ? om[a] : op[a]);
#pragma unroll
              for (int b = 0; b < D; ++b) un[a][b] = C.ut0[b * NF + cn];
            }
            float acc[3] = {0.f, 0.f, 0.f};
#pragma unroll
            for (int a = 0; a < D; ++a)
#pragma unroll
              for (int b = 0; b < D; ++b) acc[b] += va[a] * (va[a] > 0.f ? (u0[b] - un[a][b]) : (un[a][b] - u0[b]));
#pragma unroll
            for (int b = 0; b < D; ++b) u0[b] = u0[b] - g.dte * acc[b];
            u_put(ub1[fc], u0, 0.f);
          }
          u_put(SM[k].v[tid], va, 0.f);
          u_put(SM[k].u[tid], u0, 0.f);
        }
      }
    }
    SM[k].fl[tid] = fl;
  }
  for (int k = ks; k < kn; ++k) {
    int x, y, z;
    bool ok;
    const LevelDev &L = beyond(k, x, y, z, ok);
    if (ok && n_ext > 0) ext_first_cell<D>(C, L, x, y, z, ub1);
  }
  const V *uin = n_ext > 0 ? ub1 : nullptr;
  if (!lsf_barrier<MODE>(bar, target, C.err, &wait_limit)) return leave();
  // start the classification's counters (every CTA has read the band count; the lists are
  // filled after the next barriers): the band count into the previous-band slot
  if (blockIdx.x == 0 && tid == 0) {
    cnt[5] = nl;
    cnt[0] = cnt[1] = cnt[2] = cnt[3] = cnt[4] = 0;
  }
  // ---- the other sweeps
  for (int it = 1; it < n_ext; ++it) {
    V *const uout = (it & 1) ? ub2 : ub1;
    for (int k = 0; k < ks; ++k) {
      const unsigned fl = SM[k].fl[tid];
      if (!(fl & SL_LIVE)) continue;
      const unsigned fc = SM[k].fc[tid];
      if (fl & SL_IFACE) {  // after two sweeps both buffers hold the value
        if (it == 1) uout[fc] = SM[k].u[tid];
        continue;
      }
      const LsfGeo g = geo_of(fl >> SL_LD);
      float va[3], u0[3], un[D][3], acc[3] = {0.f, 0.f, 0.f};
      u_get(SM[k].v[tid], va);
      int dn[3];
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const int str = a == 0 ? 1 : (a == 1 ? g.p0 : g.p01);
        dn[a] = va[a] > 0.f ? -str : str;
      }
      if (fl & SL_EDGE) {
        const unsigned dist = fl >> SL_DIST;
#pragma unroll
        for (int a = 0; a < D; ++a)
          dn[a] = lsf_step(g, dist, a, va[a] > 0.f ? -1 : 1) * (a == 0 ? 1 : (a == 1 ? g.p0 : g.p01));
      }
#pragma unroll
      for (int a = 0; a < D; ++a) u_get(uin[fc + (unsigned)dn[a]], un[a]);
      u_get(SM[k].u[tid], u0);
      // va (u0 - un) upwind, -va (u0 - un) downwind: |va| (u0 - un) on both sides
#pragma unroll
      for (int a = 0; a < D; ++a)
#pragma unroll
        for (int b = 0; b < D; ++b) acc[b] += fabsf(va[a]) * (u0[b] - un[a][b]);
#pragma unroll
      for (int b = 0; b < D; ++b) u0[b] = u0[b] - g.dte * acc[b];
      V r;
      u_put(r, u0, 0.f);
      uout[fc] = r;
      SM[k].u[tid] = r;
    }
    for (int k = ks; k < kn; ++k) {
      int x, y, z;
      bool ok;
      const LevelDev &L = beyond(k, x, y, z, ok);
      if (ok) ext_sweep_cell<D>(C, L, x, y, z, uin, uout);
    }
    uin = uout;
    // (the first transport stage reads phi and its own cells' u~: no barrier before it)
    if (it < n_ext - 1 && !lsf_barrier<MODE>(bar, target, C.err, &wait_limit)) return leave();
  }
  // values around a cell (at pc) along axis a at offsets -3..+3, or mirrored; last: the
  // highest index wanted
  auto gather = [&](const float *pc, const LsfGeo &g, unsigned fl, int a, bool back, float v[7], int last) {
    const int str = a == 0 ? 1 : (a == 1 ? g.p0 : g.p01);
    if (!(fl & (SL_NEAR << a))) {
      const long long s = back ? -str : str;
      const float *q = pc - 3 * s;
#pragma unroll
      for (int m = 0; m < 7; ++m)
        if (m <= last) v[m] = q[m * s];
    } else {
      const unsigned dist = fl >> SL_DIST;
#pragma unroll
      for (int m = 0; m < 7; ++m)
        if (m <= last) v[m] = pc[(long long)lsf_step(g, dist, a, back ? 3 - m : m - 3) * str];
    }
  };
  // ---- transport
  for (int stage = 1; stage <= 3; ++stage) {
    const float *pin = stage == 1 ? C.phi : (stage == 2 ? C.p1 : C.p2);
    for (int k = 0; k < ks; ++k) {
      const unsigned fl = SM[k].fl[tid];
      if (!(fl & SL_LIVE)) continue;
      const unsigned fc = SM[k].fc[tid];
      const LsfGeo g = geo_of(fl >> SL_LD);
      float ua[3], v[D][7];
      u_get(SM[k].u[tid], ua);
      const float p0 = stage == 1 ? C.phi[fc] : SM[k].v[tid].x;
#pragma unroll
      for (int a = 0; a < D; ++a)  // upwind side by the sign of u~: the mirrored stencil is the same sum negated
        gather(pin + fc, g, fl, a, !(ua[a] >= 0.f), v[a], 5);
      // commit u~ (the buffer of the last sweep holds it; the other one's old values are read
      // until the barrier behind stage 1)
      if (stage == 1) {
#pragma unroll
        for (int a = 0; a < D; ++a) C.ut0[a * NF + fc] = ua[a];
      } else if (stage == 2) {
        if (uin != ub1) u_put(ub1[fc], ua, 0.f);
        if (uin != ub2) u_put(ub2[fc], ua, 0.f);
      }
      float rhs = 0.f;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const float d = d5m(v[a]);
        rhs -= ua[a] * (ua[a] >= 0.f ? d : -d);
      }
      float r;
      if (stage == 1) {
        r = p0 + rhs;
        C.p1[fc] = r;
        SM[k].v[tid].x = p0;
        SM[k].v[tid].y = r;
      } else if (stage == 2) {
        r = 0.75f * p0 + 0.25f * (SM[k].v[tid].y + rhs);
        C.p2[fc] = r;
        SM[k].v[tid].y = r;
      } else {
        r = p0 / 3.0f + (2.0f / 3.0f) * (SM[k].v[tid].y + rhs);
        C.phi[fc] = r;
        SM[k].v[tid].x = r;
      }
    }
    for (int k = ks; k < kn; ++k) {
      int x, y, z;
      bool ok;
      const LevelDev &L = beyond(k, x, y, z, ok);
      if (ok) adv_cell<D>(C, L, x, y, z, stage, uin, ub1, ub2);
    }
    // (the phases read their own cells' phi and leave p2, which the last stage's neighbours
    // read, as it is: no barrier between them)
    if ((stage < 3 || n_re > 0) && !lsf_barrier<MODE>(bar, target, C.err, &wait_limit)) return leave();
  }
  // ---- reinitialisation
  for (int r = 0; r < n_re; ++r)
    for (int stage = 1; stage <= 3; ++stage) {
      const float *pin = stage == 1 ? C.phi : (stage == 2 ? C.p1 : C.p2);
      const bool prep = r == 0 && stage == 1;
      for (int k = 0; k < ks; ++k) {
        unsigned fl = SM[k].fl[tid];
        if (!(fl & SL_LIVE)) continue;
        const unsigned fc = SM[k].fc[tid];
        const LsfGeo g = geo_of(fl >> SL_LD);
        const float p0 = SM[k].v[tid].x;
        if (prep) {
          if ((fl & SL_EDGE) ? sign_change<Q>(C.phi + fc, p0, lsf_near<D>(g, fl >> SL_DIST))
                             : sign_change_inner<Q>(C.phi + fc, p0, g.p0, g.p01))
            fl |= SL_FROZEN;
          SM[k].fl[tid] = fl;
          SM[k].u[tid].x = p0 / sqrtf(p0 * p0 + 1.0f);
        }
        if (fl & SL_FROZEN) {
          if (stage == 1) C.p1[fc] = p0;
          else if (stage == 2) C.p2[fc] = p0;
          continue;
        }
        const float s0 = SM[k].u[tid].x;
        float g2 = 0.f, v[D][7];
#pragma unroll
        for (int a = 0; a < D; ++a) gather(pin + fc, g, fl, a, false, v[a], 6);
#pragma unroll
        for (int a = 0; a < D; ++a) g2 += godunov_axis(v[a], s0);
        const float rhs = g.dtr * (-s0 * (sqrtf(g2) - 1.0f));
        float q;
        if (stage == 1) {
          q = p0 + rhs;
          C.p1[fc] = q;
          SM[k].v[tid].y = q;
        } else if (stage == 2) {
          q = 0.75f * p0 + 0.25f * (SM[k].v[tid].y + rhs);
          C.p2[fc] = q;
          SM[k].v[tid].y = q;
        } else {
          q = p0 / 3.0f + (2.0f / 3.0f) * (SM[k].v[tid].y + rhs);
          C.phi[fc] = q;
          SM[k].v[tid].x = q;
        }
      }
      for (int k = ks; k < kn; ++k) {
        int x, y, z;
        bool ok;
        const LevelDev &L = beyond(k, x, y, z, ok);
        if (ok) reinit_cell<Q>(C, L, x, y, z, stage, prep);
      }
      if ((stage < 3 || r < n_re - 1) && !lsf_barrier<MODE>(bar, target, C.err, &wait_limit)) return leave();
    }
  // ---- phases (k_classify_phase without init): p1 (p2 below) back to phi, tags, flips
  for (int k = 0; k < kn; ++k) {
    const int w = w0 + k * GB;
    unsigned fc;
    long long tc;
    float ph;
    int ld;
    if (k < ks) {
      const unsigned fl = SM[k].fl[tid];
      if (!(fl & SL_CELL)) continue;
      fc = SM[k].fc[tid];
      ld = (int)(fl >> SL_LD);
      tc = (long long)fc + geo_of((unsigned)ld).tag_delta;
      ph = (fl & SL_LIVE) ? SM[k].v[tid].x : C.phi[fc];
    } else {
      if (w >= nl) continue;
      int x, y, z;
      const int4 b = info[w];
      const LevelDev &L = band_cell_at(C, S, b, t, x, y, z);
      if (x >= L.n[0] || y >= L.n[1] || z >= L.n[2]) continue;
      fc = (unsigned)(L.fine_off + cidx(L, x, y, z));
      ld = b.x;
      tc = (long long)fc + L.cell_off - L.fine_off;
      ph = C.phi[fc];
    }
    const uint8_t tg = C.tag[tc];
    if (!(tg & TAG_LEAF)) continue;
    C.p1[fc] = ph;
    const int gas = ph >= 0.0f ? 1 : 0, prev = tg & TAG_GAS;
    C.tag[tc] = (tg & (TAG_LEAF | TAG_RLAYER | TAG_GHOST)) | (gas ? TAG_GAS : 0) | (prev ? TAG_PREVGAS : 0) |
                (gas != prev ? TAG_FLIP : 0);
    if (gas != prev) {
      const LevelDev &L = C.lds[ld];
      int x, y, z;
      cell_xyz(L, fc - L.fine_off, x, y, z);
      list_flip<Q>(C, L, S, glevel, ld, fc - L.fine_off, x, y, z);
    }
  }
  if (!lsf_barrier<MODE>(bar, target, C.err, &wait_limit)) return leave();
  // ---- cut links (k_classify_links without full): the previous band, then the check list
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int *lst = C.band_list + (long long)glevel * C.band_cap, *chk = C.check_list + (long long)glevel * C.band_cap;
  const int nb2 = nl + min(cnt[4], C.band_cap);
  const int hb = tid >> lgnt;
  for (int k = 0; k * GB < nb2; ++k) {
    const int w = w0 + k * GB;
    if (t == 0) hot[hb] = 0;
    __syncthreads();
    int gb = 0;
    if (w < nb2) {
      uint32_t m = 0;
      unsigned fc = 0, dist = 0;
      uint8_t tg = 0;
      int ld = 0;
      bool cell, edge;
      float ph = 0.f;
      gb = w < nl ? lst[w] : chk[w - nl];
      if (k < ks && w < nl) {
        const unsigned fl = SM[k].fl[tid];
        ph = SM[k].v[tid].x;
        ld = (int)(fl >> SL_LD);
        cell = (fl & SL_CELL) != 0;
        edge = (fl & SL_EDGE) != 0;
        dist = fl >> SL_DIST;
        if (cell) fc = SM[k].fc[tid];
        if (cell && !(fl & SL_LIVE)) ph = C.phi[fc];
      } else {
        const int4 b = C.blk_info[gb];
        ld = b.x;
        const int crd[3] = {(b.y << S.lg[0]) + (t & (S.bs[0] - 1)), (b.z << S.lg[1]) + ((t >> S.lg[0]) & (S.bs[1] - 1)),
                            (b.w << S.lg[2]) + (t >> (S.lg[0] + S.lg[1]))};
        const LsfGeo g = geo_of((unsigned)ld);
        cell = crd[0] < g.n[0] && crd[1] < g.n[1] && crd[2] < g.n[2];
        edge = true;
        if (cell) {
          fc = g.fo + (unsigned)crd[0] + (unsigned)(g.p0 * crd[1] + g.p01 * crd[2]);
          dist = lsf_dist<D>(crd, g.n);
          if (w < nl) ph = C.phi[fc];
        }
      }
      const LsfGeo g = geo_of((unsigned)ld);
      const long long tc = (long long)fc + g.tag_delta;
      if (cell) {
        tg = C.tag[tc];
        if (tg & TAG_LEAF) {
          if (w < nl) C.p2[fc] = ph;
          m = edge ? cut_mask<Q>(C.tag + tc, tg, lsf_near<D>(g, dist)) : cut_mask_inner<Q>(C.tag + tc, tg, g.p0, g.p01);
          C.cmask[fc] = m;
        }
      }
      list_links(C, glevel, m, ld, (int)(fc - g.fo), fc, tc, tg);
      if (m) hot[hb] = 1;
    }
    __syncthreads();
    if (t == 0 && w < nb2) C.bflag[gb] = hot[hb] ? BF_IFACE : 0;
  }
  leave();
}

// ------------------------------------------------------------------ a launch per pass
// One pass of the update over the band list, for bands so large that most cells lie beyond the
// slots of the launch above: there every pass loads a cell's descriptor and plan again on 1024
// threads per SM, here on 1536, and the launches and their chains (~4 us each, 14 of them) weigh
// little.  A layer of 16 M band cells (1024 x 1024 x 64): 7418 -> 6499 us a step.  The
// reinitialisation is built for two CTAs of 512 threads per SM: with three (its stages 873
// instead of 934 us there) the compiler contracts its arithmetic otherwise, an ulp in one of 500
// cells, and the shape of the launch changes no result.  The counters are started by the
// classification (no pass here touches them).
enum { LS_EXT_FIRST, LS_EXT_SWEEP, LS_ADVECT, LS_REINIT };
template <int Q, int PASS>
__global__ void __launch_bounds__(512, PASS == LS_REINIT ? 2 : 3) k_levelset_pass(Ctx C, BlockShape S, int glevel, int stage, int prep,
                                                          const void *uin_, void *uout_) {
  LSB_GRID_WAIT();
  constexpr int D = Lat<Q>::D;
  using V = typename UVec<D>::T;
  const V *uin = static_cast<const V *>(uin_);
  V *uout = static_cast<V *>(uout_);
  const int nl = min(C.counters[glevel * NCOUNT + 3], C.band_cap);
  // the next entry of the band list is loaded while this one is processed
  const int4 *info = C.band_info + (long long)glevel * C.band_cap;
  int4 next = (int)blockIdx.x < nl ? __ldg(info + blockIdx.x) : make_int4(0, 0, 0, 0);
  for (int w = blockIdx.x; w < nl; w += gridDim.x) {
    const int4 bi = next;
    if (w + (int)gridDim.x < nl) next = __ldg(info + w + gridDim.x);
    int x, y, z;
    const LevelDev &L = band_cell_at(C, S, bi, threadIdx.x, x, y, z);
    if (!L.ls_active || x >= L.n[0] || y >= L.n[1] || z >= L.n[2]) continue;
    if constexpr (PASS == LS_EXT_FIRST) ext_first_cell<D>(C, L, x, y, z, uout);
    else if constexpr (PASS == LS_EXT_SWEEP) ext_sweep_cell<D>(C, L, x, y, z, uin, uout);
    else if constexpr (PASS == LS_ADVECT)
      adv_cell<D>(C, L, x, y, z, stage, uin, reinterpret_cast<V *>(C.ut1), reinterpret_cast<V *>(C.ut2));
    else reinit_cell<Q>(C, L, x, y, z, stage, prep);
  }
}

// Both sweep buffers from ut0 at every finest cell (their state between updates).
template <int D>
__global__ void k_ut_pack(const float *__restrict__ ut0, typename UVec<D>::T *ub1, typename UVec<D>::T *ub2,
                          long long n) {
  LSB_GRID_WAIT();
  for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n; c += (long long)gridDim.x * blockDim.x) {
    float u[3];
    for (int a = 0; a < D; ++a) u[a] = ut0[a * n + c];
    u_put(ub1[c], u, 0.f);
    u_put(ub2[c], u, 0.f);
  }
}

// ------------------------------------------------------------------ persistent level-set phase
// The whole level-set update of a finest level (extension, transport,
// reinitialisation: up to 16 dependent passes over the band list) as one
// cooperative launch, with a grid barrier between passes.  The barrier spins
// with an iteration limit: on expiry the block sets ERR_TIMEOUT and returns, so
// a barrier that cannot complete ends the kernel instead of hanging it (the
// cooperative launch makes every CTA resident, so this does not happen in
// normal operation).  bar: two words, arrival count and generation, zero at rest
// (cleared before every launch).  limit: sleeps of ~64 ns before giving up (the
// handle's wait limit, 2^22 ~ 0.3 s by default; 0 gives up at the first wait).
__device__ __forceinline__ bool grid_barrier(unsigned *bar, int *err, long long limit) {
  __shared__ int abort_flag;
  __syncthreads();
  if (threadIdx.x == 0) {
    abort_flag = 0;
    volatile unsigned *vgen = bar + 1;
    const unsigned gen = *vgen;
    __threadfence();
    const unsigned arrived = atomicAdd(bar, 1u) + 1u;
    if (arrived == gridDim.x) {
      atomicExch(bar, 0u);
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      long long it = 0;
      while (*vgen == gen) {
        if (++it > limit) {
          atomicOr(err, ERR_TIMEOUT);
          abort_flag = 1;
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return abort_flag == 0;
}

template <int Q>
__global__ void k_levelset_persistent(Ctx C, BlockShape S, int glevel, int n_ext, int reinit, int n_reinit,
                                      unsigned *bar, long long limit) {
  LSB_GRID_WAIT();
  constexpr int D = Lat<Q>::D;
  d_ext_init<Q>(C, glevel, 0, gridDim.x);
  if (!grid_barrier(bar, C.err, limit)) return;
  const float *uin = C.ut0;
  for (int it = 0; it < n_ext; ++it) {
    float *uout = (it & 1) ? C.ut2 : C.ut1;
    d_ext_iter<D>(C, S, glevel, uin, uout, it == 0 ? 2 : 3);
    if (!grid_barrier(bar, C.err, limit)) return;
    uin = uout;
  }
  if (n_ext > 0) {
    d_ext_iter<D>(C, S, glevel, uin, nullptr, 1);
    if (!grid_barrier(bar, C.err, limit)) return;
  }
  for (int st = 1; st <= 3; ++st) {
    d_adv_stage<D>(C, S, glevel, st);
    if (!grid_barrier(bar, C.err, limit)) return;
  }
  if (reinit) {
    d_reinit_prep<Q>(C, S, glevel);
    if (!grid_barrier(bar, C.err, limit)) return;
    for (int r = 0; r < n_reinit; ++r)
      for (int st = 1; st <= 3; ++st) {
        d_reinit_stage<D>(C, S, glevel, st);
        if (!grid_barrier(bar, C.err, limit)) return;
      }
  }
}

// ------------------------------------------------------------------ refill (Sec. 2.4)
template <int Q>
__device__ __forceinline__ float feq_q(int i, float drho, const float u[3]) {
  using LT = Lat<Q>;
  const float cu = LT::cx(i) * u[0] + LT::cy(i) * u[1] + LT::cz(i) * u[2];
  const float usq = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
  return LT::w(i) * (drho + (1.0f + drho) * (3.0f * cu + 4.5f * cu * cu - 1.5f * usq));
}

// The flipped cells, one warp each, on the CTAs [b0, b0 + nb) of the launch: the curvature fit
// (lane k takes stencil point k; integer sums, so the order does not matter) and, with refill
// set, the refill (lane i takes direction i).  A launch that flips a cell waits for that cell's
// whole chain, so it is spread over lanes and kept short: as one thread per cell after its fit
// it was ~25 us of loops over the directions (3D bubble, ~5 flips per sub-step; unrolled to
// issue its loads together it took longer still, all of it instruction fetch).
template <int Q, typename T>
__device__ __forceinline__ void d_flipped(const Ctx &C, int glevel, int refill, int b0, int nb) {
  using LT = Lat<Q>;
  constexpr int D = LT::D, NS = D == 3 ? 27 : 9;
  const unsigned all = 0xffffffffu;
  const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  const int nf = min(C.counters[glevel * NCOUNT + 2], (int)C.list_cap);
  const int2 *lf = C.flip_list + (long long)glevel * C.list_cap;
  for (int e = ((int)blockIdx.x - b0) * wpb + (threadIdx.x >> 5); e < nf; e += nb * wpb) {
    const int2 it = lf[e];
    const LevelDev &L = C.lds[it.x];
    const long long c = it.y, fo = L.fine_off;
    int x, y, z;
    cell_xyz(L, c, x, y, z);
    // ---- fit
    const int ox = lane % 3 - 1, oy = (lane / 3) % 3 - 1, oz = D == 3 ? lane / 9 - 1 : 0;
    long long v = 0;
    if (lane < NS)
      v = phi_fixed(C.phi[fo + cidx(L, clampwrap(L, 0, x + ox), clampwrap(L, 1, y + oy),
                                    D == 3 ? clampwrap(L, 2, z + oz) : 0)]);
    auto sum = [&](int s) {  // sum of s v over the stencil, s = -1, 0, 1
      long long r = s > 0 ? v : (s < 0 ? -v : 0);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(all, r, o);
      return r;
    };
    const long long iP = sum(1), isx[3] = {sum(ox), sum(oy), sum(oz)}, isxx[3] = {sum(ox * ox), sum(oy * oy), sum(oz * oz)},
                    isxy[3] = {sum(ox * oy), sum(ox * oz), sum(oy * oz)};
    float n[3], kap;
    fit_from_sums<D>(iP, isx, isxx, isxy, n, kap);
    if (lane < D) C.nvec[lane * C.nfine + fo + c] = lane == 0 ? n[0] : (lane == 1 ? n[1] : n[2]);
    if (lane == 0) C.kappa[fo + c] = kap;
    if (!refill) continue;
    // ---- refill
    const long long N = L.ncell;
    T *Bf = fB<T, Q>(C, L);
    const uint8_t *tagL = C.tag + L.cell_off;
    const uint8_t tg = tagL[c];
    const int Pn = tg & TAG_GAS;
    const int Po = (tg & TAG_PREVGAS) ? 1 : 0;
    const float sg = Pn == 0 ? 1.0f : -1.0f;
    auto valid_new = [&](int tx, int ty, int tz, long long &ct) -> bool {
      if (!(wrap(L, 0, tx) && wrap(L, 1, ty) && (D == 2 || wrap(L, 2, tz)))) return false;
      ct = cidx(L, tx, ty, tz);
      const uint8_t tt = tagL[ct];
      return (tt & TAG_LEAF) && (tt & TAG_GAS) == Pn && ((tt & TAG_PREVGAS) ? 1 : 0) == Pn;
    };
    // e_min: the largest e.m / |e|, m = the normal into the new phase; ties to the lowest index
    const int i = lane < Q ? lane : LT::REST;
    const int ci = LT::cx(i), cj = LT::cy(i), ck = LT::cz(i);
    long long ct = c;
    float bv = -1e30f;
    int best = Q;
    if (i != LT::REST && valid_new(x + ci, y + cj, z + ck, ct)) {
      const float mvec[3] = {-sg * n[0], -sg * n[1], D == 3 ? -sg * n[2] : 0.f};
      const float nrm = sqrtf((float)(ci * ci + cj * cj + ck * ck));
      const float w = (ci * mvec[0] + cj * mvec[1] + ck * mvec[2]) / nrm;
      if (w > bv) {
        bv = w;
        best = i;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float ov = __shfl_xor_sync(all, bv, o);
      const int ob = __shfl_xor_sync(all, best, o);
      if (ov > bv || (ov == bv && ob < best)) {
        bv = ov;
        best = ob;
      }
    }
    if (best >= Q) {
      if (lane < Q) Store<T>::st(Bf + i * N + c, 0.0f, C.fp16_scale);
      continue;
    }
    const int ex = LT::cx(best), ey = LT::cy(best), ez = LT::cz(best);
    const long long c1 = __shfl_sync(all, ct, best);
    long long c2 = c;
    const bool quad = valid_new(x + 2 * ex, y + 2 * ey, z + 2 * ez, c2);
    const float phr = C.phi[fo + c];
    float q = 0.5f;
    {
      int bx = x - ex, by = y - ey, bz = z - ez;
      if (wrap(L, 0, bx) && wrap(L, 1, by) && (D == 2 || wrap(L, 2, bz))) {
        const long long cb = cidx(L, bx, by, bz);
        if ((tagL[cb] & TAG_GAS) != Pn) q = phr / (phr - C.phi[fo + cb]);
      }
    }
    float w0, w1, w2;
    if (quad) {
      w0 = 2.0f / ((q + 1.0f) * (q + 2.0f));
      w1 = 2.0f * q / (q + 1.0f);
      w2 = -q / (q + 2.0f);
    } else {
      w0 = 1.0f / (1.0f + q);
      w1 = q / (1.0f + q);
      w2 = 0.0f;
    }
    const float f_old = Store<T>::ld(Bf + i * N + c, C.fp16_inv), f_1 = Store<T>::ld(Bf + i * N + c1, C.fp16_inv);
    const float f_2 = Store<T>::ld(Bf + i * N + c2, C.fp16_inv);
    // moments of the three cells, summed in the order of the populations
    float d[3] = {0.f, 0.f, 0.f}, jx[3] = {0.f, 0.f, 0.f}, jy[3] = {0.f, 0.f, 0.f}, jz[3] = {0.f, 0.f, 0.f};
#pragma unroll 1
    for (int k = 0; k < Q; ++k) {
      const float a = (float)LT::cx(k), b = (float)LT::cy(k), g = (float)LT::cz(k);
      const float fk[3] = {__shfl_sync(all, f_old, k), __shfl_sync(all, f_1, k), __shfl_sync(all, f_2, k)};
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        d[m] += fk[m];
        jx[m] += a * fk[m];
        jy[m] += b * fk[m];
        jz[m] += g * fk[m];
      }
    }
    float u_old[3], u1[3], u2[3];
    auto velocity = [&](int m, float u[3]) {
      const float inv = 1.0f / (1.0f + d[m]);
      u[0] = jx[m] * inv; u[1] = jy[m] * inv; u[2] = jz[m] * inv;
    };
    velocity(0, u_old);
    velocity(1, u1);
    const float p_gamma = L.rho_phys[Po] * CS2 * d[0] + L.sigma * sg * kap;
    const float r_g = p_gamma / (L.rho_phys[Pn] * CS2);
    float rr = w0 * r_g + w1 * d[1];
    float ur[3];
    for (int a = 0; a < 3; ++a) ur[a] = w0 * u_old[a] + w1 * u1[a];
    if (quad) {
      velocity(2, u2);
      rr += w2 * d[2];
      for (int a = 0; a < 3; ++a) ur[a] += w2 * u2[a];
    }
    if (lane < Q)
      Store<T>::st(Bf + i * N + c, feq_q<Q>(i, rr, ur) + (f_1 - feq_q<Q>(i, d[1], u1)), C.fp16_scale);
  }
}

// The classification's last passes in one launch, which read nothing of each other's: the
// flipped cells (CTAs [0, kFlipCtas), a warp per cell: the longest chain, scheduled first), the
// curvature fit of the interface cells (the next gg) and the band (the rest, a warp per finest
// block).  The refill reads the fit at its own cell, and neighbours of the new phase that did
// not flip; a cell on both lists gets the same fit twice.
constexpr int kFlipCtas = 16;
template <int Q, typename T>
__global__ void k_post_classify(Ctx C, const int *list, int nlist, int glevel, int gg, int refill) {
  LSB_GRID_WAIT();
  constexpr int D = Lat<Q>::D;
  const int b = (int)blockIdx.x;
  if (b < kFlipCtas) d_flipped<Q, T>(C, glevel, refill, 0, kFlipCtas);
  else if (b < kFlipCtas + gg) d_geometry<D>(C, glevel, kFlipCtas, gg);
  else d_band<Q>(C, list, nlist, glevel, kFlipCtas + gg, (int)gridDim.x - gg - kFlipCtas);
}

// ------------------------------------------------------------------ refinement sensor
// Per listed coarse block: min |phi| (mode 0) or max phi (mode 1) over the
// finest cells under it.
__global__ void k_sensor(Ctx C, BlockShape S, const int *list, int nlist, int mode, float *out) {
  LSB_GRID_WAIT();
  __shared__ float red[32];
  for (int w = blockIdx.x; w < nlist; w += gridDim.x) {
    const int gb = list[w];
    const LevelDev &L = C.lds[C.blk_ld[gb]];
    const LevelDev &F = C.lds[L.fine_ld];
    const int lb = gb - L.block_off;
    const int b[3] = {lb % L.nb[0], (lb / L.nb[0]) % L.nb[1], lb / (L.nb[0] * L.nb[1])};
    int lo[3], hi[3];
    for (int a = 0; a < 3; ++a) {
      lo[a] = b[a] * S.bs[a] * L.scale;
      hi[a] = min((b[a] + 1) * S.bs[a], L.n[a]) * L.scale;
      hi[a] = min(hi[a], F.n[a]);
    }
    const long long cnt = (long long)(hi[0] - lo[0]) * (hi[1] - lo[1]) * (hi[2] - lo[2]);
    float acc = mode == 0 ? 3.0e38f : -3.0e38f;
    for (long long e = threadIdx.x; e < cnt; e += blockDim.x) {
      const int sx = hi[0] - lo[0], sy = hi[1] - lo[1];
      const int x = lo[0] + (int)(e % sx);
      const int y = lo[1] + (int)((e / sx) % sy);
      const int z = lo[2] + (int)(e / ((long long)sx * sy));
      const float p = C.phi[F.fine_off + cidx(F, x, y, z)];
      acc = mode == 0 ? fminf(acc, fabsf(p)) : fmaxf(acc, p);
    }
    for (int off = 16; off > 0; off >>= 1) {
      const float o = __shfl_down_sync(0xffffffffu, acc, off);
      acc = mode == 0 ? fminf(acc, o) : fmaxf(acc, o);
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      float r = red[0];
      for (int k = 1; k < (int)(blockDim.x + 31) / 32; ++k) r = mode == 0 ? fminf(r, red[k]) : fmaxf(r, red[k]);
      out[w] = r;
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ host launchers
#define LQ(kern, ...)                                                          \
  do {                                                                         \
    if (Q == 9) launcher(kern<9>, L, 0)(__VA_ARGS__);        \
    else if (Q == 19) launcher(kern<19>, L, 0)(__VA_ARGS__); \
    else launcher(kern<27>, L, 0)(__VA_ARGS__);              \
    return cudaGetLastError();                                                 \
  } while (0)
#define LD(kern, ...)                                                          \
  do {                                                                         \
    if (D == 2) launcher(kern<2>, L, 0)(__VA_ARGS__);        \
    else launcher(kern<3>, L, 0)(__VA_ARGS__);               \
    return cudaGetLastError();                                                 \
  } while (0)
// CTAs of a kernel resident at once (SMs x CTAs per SM for this block size), at most want: a
// cooperative launch walks its list with that many.
template <typename K>
int resident_grid(K kern, int block, int want) {
  static std::mutex mu;
  static std::map<std::pair<const void *, int>, int> cache;  // (kernel, block) -> resident CTAs
  const std::pair<const void *, int> key{reinterpret_cast<const void *>(kern), block};
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find(key);
  if (it == cache.end()) {
    int n = 1, dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, block, 0) != cudaSuccess || n < 1) n = 1;
    it = cache.emplace(key, n * sms).first;
  }
  return want < it->second ? want : it->second;
}

cudaError_t run_classify_phase(int Q, Launch L, Ctx C, BlockShape S, const int *list, int n, int glevel, int init) {
  LQ(k_classify_phase, C, S, list, n, glevel, init);
}
cudaError_t run_classify_links(int Q, Launch L, Ctx C, BlockShape S, const int *list, int n, int glevel, int full) {
  LQ(k_classify_links, C, S, list, n, glevel, full);
}
cudaError_t run_geometry(int D, Launch L, Ctx C, int glevel) { LD(k_geometry, C, glevel); }
// Shared memory of the one-launch level-set update.
size_t lsf_smem(int D, int kcap) { return (D == 2 ? sizeof(LsfSlot<2>) : sizeof(LsfSlot<3>)) * (size_t)kcap; }
cudaError_t run_ut_pack(int D, Launch L, const float *ut0, float *ut1, float *ut2, long long n) {
  if (D == 2) launcher(k_ut_pack<2>, L, 0)(ut0, (float2 *)ut1, (float2 *)ut2, n);
  else launcher(k_ut_pack<3>, L, 0)(ut0, (float4 *)ut1, (float4 *)ut2, n);
  return cudaGetLastError();
}
template <int Q>
cudaError_t lsf_prepare(LsfLimits *out) {
  constexpr int D = Lat<Q>::D;
  int dev = 0, sms = 0, optin = 0, coop = 0, nb = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  cudaFuncAttributes fa;
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k_levelset_fused<Q, 1>);
  if (e != cudaSuccess) return e;
  out->kmax = (int)(((size_t)optin - fa.sharedSizeBytes - 1024) / lsf_smem(D, 1));
  const int smem = (int)lsf_smem(D, out->kmax);
  e = cudaFuncSetAttribute(k_levelset_fused<Q, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_levelset_fused<Q, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_levelset_fused<Q, 0>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  out->max_ld = kLsfMaxLd;
  // what fits on a device is asked once per device, not for every handle (64 x 32 channel: a handle's
  // creation 0.55 ms; 0.53 without this launch to prepare at all)
  constexpr int kDevs = 64;
  static std::mutex mu;
  static LsfLimits known[kDevs];  // (grid, cluster; cluster 0: not asked yet)
  std::lock_guard<std::mutex> lock(mu);
  if (dev < kDevs && known[dev].cluster) {
    out->grid = known[dev].grid;
    out->cluster = known[dev].cluster;
    return cudaSuccess;
  }
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_levelset_fused<Q, 1>, 1024, smem);
  if (e != cudaSuccess) return e;
  out->grid = coop && nb > 0 ? sms : 0;
  out->cluster = 8;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = 16;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.gridDim = dim3(16);
  cfg.blockDim = dim3(1024);
  cfg.dynamicSmemBytes = lsf_smem(D, 2);
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  int nc = 0;
  if (cudaOccupancyMaxActiveClusters(&nc, k_levelset_fused<Q, 0>, &cfg) == cudaSuccess && nc > 0) out->cluster = 16;
  else cudaGetLastError();
  if (dev < kDevs) known[dev] = *out;
  return cudaSuccess;
}
cudaError_t prepare_levelset_fused(int Q, LsfLimits *out) {
  return Q == 9 ? lsf_prepare<9>(out) : (Q == 19 ? lsf_prepare<19>(out) : lsf_prepare<27>(out));
}
template <int Q>
cudaError_t lsf_launch(const Launch &L, const LsfPlan &P, Ctx C, BlockShape S, int glevel, int n_ext, int n_re, int nld,
                       unsigned *bar, unsigned limit) {
  cudaLaunchAttribute at[3];
  unsigned na = 0;
  if (P.form == LSF_GRID) {
    at[na].id = cudaLaunchAttributeCooperative;
    at[na++].val.cooperative = 1;
  } else {
    at[na].id = cudaLaunchAttributeClusterDimension;
    at[na].val.clusterDim.x = (unsigned)P.grid;
    at[na].val.clusterDim.y = at[na].val.clusterDim.z = 1;
    ++na;
  }
  // a cooperative launch is no programmatic dependent: launched early it loses the guarantee
  // that its CTAs become resident together (steps of 1 to 80 ms seen beside a side stream's
  // collide, 0.77 without)
  if (L.pdl && P.form != LSF_GRID) {
    at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[na++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (L.prio) {
    at[na].id = cudaLaunchAttributePriority;
    at[na++].val.priority = L.prio;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)P.grid);
  cfg.blockDim = dim3((unsigned)P.threads);
  cfg.dynamicSmemBytes = lsf_smem(Lat<Q>::D, P.kcap);
  cfg.stream = L.stream;
  cfg.attrs = at;
  cfg.numAttrs = na;
  if (P.form == LSF_GRID) return cudaLaunchKernelEx(&cfg, k_levelset_fused<Q, 1>, C, S, glevel, n_ext, n_re, nld, P.kcap, bar, limit);
  return cudaLaunchKernelEx(&cfg, k_levelset_fused<Q, 0>, C, S, glevel, n_ext, n_re, nld, P.kcap, bar, limit);
}
cudaError_t run_levelset_fused(int Q, Launch L, LsfPlan P, Ctx C, BlockShape S, int glevel, int n_ext, int n_re, int nld,
                               unsigned *bar, unsigned limit) {
  if (Q == 9) return lsf_launch<9>(L, P, C, S, glevel, n_ext, n_re, nld, bar, limit);
  if (Q == 19) return lsf_launch<19>(L, P, C, S, glevel, n_ext, n_re, nld, bar, limit);
  return lsf_launch<27>(L, P, C, S, glevel, n_ext, n_re, nld, bar, limit);
}
template <int PASS>
cudaError_t pass_launch(int Q, Launch L, Ctx C, BlockShape S, int glevel, int stage, int prep, const void *uin,
                        void *uout) {
  if (Q == 9) launcher(k_levelset_pass<9, PASS>, L, 0)(C, S, glevel, stage, prep, uin, uout);
  else if (Q == 19) launcher(k_levelset_pass<19, PASS>, L, 0)(C, S, glevel, stage, prep, uin, uout);
  else launcher(k_levelset_pass<27, PASS>, L, 0)(C, S, glevel, stage, prep, uin, uout);
  return cudaGetLastError();
}
cudaError_t run_ext_pass(int Q, Launch L, Ctx C, BlockShape S, int glevel, const void *uin, void *uout) {
  return uin ? pass_launch<LS_EXT_SWEEP>(Q, L, C, S, glevel, 0, 0, uin, uout)
             : pass_launch<LS_EXT_FIRST>(Q, L, C, S, glevel, 0, 0, uin, uout);
}
cudaError_t run_adv_pass(int Q, Launch L, Ctx C, BlockShape S, int glevel, int stage, const void *ufin) {
  return pass_launch<LS_ADVECT>(Q, L, C, S, glevel, stage, 0, ufin, nullptr);
}
cudaError_t run_reinit_pass(int Q, Launch L, Ctx C, BlockShape S, int glevel, int stage, int prep) {
  return pass_launch<LS_REINIT>(Q, L, C, S, glevel, stage, prep, nullptr, nullptr);
}
cudaError_t run_post_classify(int Q, int st, Launch L, Ctx C, const int *list, int n, int glevel, int gg,
                              int refill) {
  L.grid += kFlipCtas;
  if (Q == 9) {
    if (st == 0) launcher(k_post_classify<9, float>, L, 0)(C, list, n, glevel, gg, refill);
    else launcher(k_post_classify<9, __half>, L, 0)(C, list, n, glevel, gg, refill);
  } else if (Q == 19) {
    if (st == 0) launcher(k_post_classify<19, float>, L, 0)(C, list, n, glevel, gg, refill);
    else launcher(k_post_classify<19, __half>, L, 0)(C, list, n, glevel, gg, refill);
  } else {
    if (st != 0) return cudaErrorInvalidValue;  // D3Q27: FP32 storage only
    launcher(k_post_classify<27, float>, L, 0)(C, list, n, glevel, gg, refill);
  }
  return cudaGetLastError();
}
cudaError_t run_sensor(Launch L, Ctx C, BlockShape S, const int *list, int n, int mode, float *out) {
  launcher(k_sensor, L, 0)(C, S, list, n, mode, out);
  return cudaGetLastError();
}

// One cooperative launch of the level-set phase; grid = resident CTAs (required
// for a cooperative launch, which fails rather than oversubscribe).
cudaError_t run_levelset_persistent(int Q, Launch L, Ctx C, BlockShape S, int glevel, int n_ext, int reinit,
                                    int n_reinit, unsigned *bar, long long limit) {
  void *args[] = {&C, &S, &glevel, &n_ext, &reinit, &n_reinit, &bar, &limit};
  if (Q == 9) {
    const int grid = resident_grid(k_levelset_persistent<9>, L.block, L.grid);
    return cudaLaunchCooperativeKernel((const void *)k_levelset_persistent<9>, grid, L.block, args, 0, L.stream);
  }
  if (Q == 19) {
    const int grid = resident_grid(k_levelset_persistent<19>, L.block, L.grid);
    return cudaLaunchCooperativeKernel((const void *)k_levelset_persistent<19>, grid, L.block, args, 0, L.stream);
  }
  const int grid = resident_grid(k_levelset_persistent<27>, L.block, L.grid);
  return cudaLaunchCooperativeKernel((const void *)k_levelset_persistent<27>, grid, L.block, args, 0, L.stream);
}

}  // namespace lsb
