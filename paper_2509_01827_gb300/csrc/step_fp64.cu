// step_fp64.cu -- FP64 explicit step kernels (compiled with -fmad=false).
//
// One step of the explicit MCT-2D-CEM (see include/cem.h):
//   k_pieces64   internal force of every split-element piece (Eq. 6 with the
//                piece area), own strain at each edge point (smoothing off);
//   k_main64     one CTA per tile of real nodes: ES-FEM edge strains
//                (Eqs. 1, 2, 4) of the intact elements around the tile,
//                stresses, the node gather of intact and piece forces in
//                increasing element id, and the central-difference update
//                with lumped mass, Neumann and Dirichlet loads;
//   k_phantom64  the same gather and update for phantom nodes;
//   k_eval64     energy release rate of the candidate paths of every
//                free-surface point (Sec. 2.2) and the Q4 cracking rule; the
//                proposals are appended with a warp ballot.
#include <cuda_runtime.h>

#include <cfloat>

#include "cem_internal.h"
#include "q4_fp64.cuh"
#include "eval_common.cuh"

namespace cem {

namespace {

constexpr int NT = 256;  // threads of a node-update CTA (its tile shape: tile64_shape)

__device__ __forceinline__ double dot3(const double e[3], const double s[3]) {
  return e[0] * s[0] + e[1] * s[1] + e[2] * s[2];
}

// Block-wide sum of two values into e_part[blockIdx * 2 + {0,1}] (fixed tree).
__device__ void block_sum2(double a, double b, double *out) {
  __shared__ double wa[32], wb[32];
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, o);
    b += __shfl_down_sync(0xffffffffu, b, o);
  }
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  if (lane == 0) { wa[w] = a; wb[w] = b; }
  __syncthreads();
  if (w == 0) {
    a = lane < nw ? wa[lane] : 0.0;
    b = lane < nw ? wb[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_down_sync(0xffffffffu, a, o);
      b += __shfl_down_sync(0xffffffffu, b, o);
    }
    if (lane == 0) { out[0] = a; out[1] = b; }
  }
}

__device__ __forceinline__ bool finite64(double x) {
  return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000;  // an integer test: FP64 compares share the FP64 pipe
}

__device__ __forceinline__ void load_factors(const DevState &d, double &lamN, double &lamD) {
  int idx = d.cnt->step - d.cnt->lam_base;
  lamN = d.lamN[idx];
  lamD = d.lamD[idx];
}

// Central-difference update of one node (real or phantom); mirrors the
// oracle's expression order exactly.  Returns its kinetic energy on record
// steps; the mean velocity that needs is formed only there and at nodes with
// a load or a prescribed velocity.
__device__ __forceinline__ double update_node(const DevState &d, int N, int cur, bool first,
                                              double fintx, double finty, uint8_t nf, bool energy) {
  const double dt = d.mat.dt;
  const double dtv = first ? 0.5 * dt : dt;
  double fex = 0.0, fey = 0.0, lamN = 0.0, lamD = 0.0;
  if (nf) load_factors(d, lamN, lamD);
  const bool loaded = (nf & NF_LOADED) != 0;
  if (loaded) {
    fex = lamN * d.Fx[N];
    fey = lamN * d.Fy[N];
  }
  double minv = d.minv[N];
  double ax = (loaded ? fex - fintx : -fintx) * minv;
  double ay = (loaded ? fey - finty : -finty) * minv;
  double vxo = d.vx[N], vyo = d.vy[N];
  double vxn = vxo + dtv * ax;
  double vyn = vyo + dtv * ay;
  if (nf & NF_DIRX) vxn = lamD * d.Vx[N];
  if (nf & NF_DIRY) vyn = lamD * d.Vy[N];
  double ke = 0.0;
  if (nf || energy) {
    double vbx = first ? vxo : 0.5 * (vxo + vxn);
    double vby = first ? vyo : 0.5 * (vyo + vyn);
    if (loaded) d.Wn[N] = d.Wn[N] + dt * (fex * vbx + fey * vby);
    if (nf & (NF_DIRX | NF_DIRY)) {
      double m = d.m[N];
      double Rx = m * ((vxn - vxo) / dtv) - (fex - fintx);
      double Ry = m * ((vyn - vyo) / dtv) - (fey - finty);
      double w = 0.0;
      if (nf & NF_DIRX) w = w + Rx * vbx;
      if (nf & NF_DIRY) w = w + Ry * vby;
      d.Wd[N] = d.Wd[N] + dt * w;
    }
    if (energy) ke = 0.5 * (d.m[N] * (vbx * vbx + vby * vby));
  }
  d.vx[N] = vxn;
  d.vy[N] = vyn;
  // a non-finite velocity (NaN or Inf) is reported through the status word
  if (!finite64(vxn) || !finite64(vyn)) atomicOr(&d.cnt->status, STAT_NONFINITE);
  d.ux[cur ^ 1][N] = d.ux[cur][N] + dt * vxn;
  d.uy[cur ^ 1][N] = d.uy[cur][N] + dt * vyn;
  return ke;
}

// ------------------------------------------------------------------ pieces
__device__ __forceinline__ void pieces64(const DevState &d, VBlk vb, int cur, int energy,
                                         int part_off) {
  const int n = 2 * d.cnt->n_ck;
  double se = 0.0;
  for (int t = vb.x * blockDim.x + threadIdx.x; t < n; t += vb.gx * blockDim.x) {
    int c = t >> 1, p = t & 1;
    double u[4], v[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      int N = d.ck_node[c * 8 + p * 4 + a];
      u[a] = d.ux[cur][N];
      v[a] = d.uy[cur][N];
    }
    double s[4][3], e[4][3];
    strain64<0>(d.g, u, v, e[0]);
    strain64<1>(d.g, u, v, e[1]);
    strain64<2>(d.g, u, v, e[2]);
    strain64<3>(d.g, u, v, e[3]);
#pragma unroll
    for (int k = 0; k < 4; ++k) stress64(d.mat, e[k], s[k]);
    double qA = d.ck_Ap[c * 2 + p] * 0.25;
    double *f = d.pf + c * 16 + p * 8;
    node_force64<0>(d.g, s, qA, f[0], f[1]);
    node_force64<1>(d.g, s, qA, f[2], f[3]);
    node_force64<2>(d.g, s, qA, f[4], f[5]);
    node_force64<3>(d.g, s, qA, f[6], f[7]);
    if (energy) {
      double acc = 0.0;
#pragma unroll
      for (int k = 0; k < 4; ++k) acc = acc + 0.5 * (qA * dot3(e[k], s[k]));
      se += acc;
    }
  }
  if (energy) block_sum2(0.0, se, d.e_part + 2 * (part_off + vb.x));
}

__global__ void k_pieces64(DevState d, int cur, int energy, int part_off) {
  wait_for_predecessors();
  release_dependents();  // the node update waits where it first reads a piece force
  pieces64(d, hw_vblk(), cur, energy, part_off);
}

// -------------------------------------------------------------- main tile
// The node update is bound by the FP64 pipe (about 0.5 T instructions/s on
// the whole GPU, 1/74 of FP32), so it is built to issue as few FP64
// instructions as the definition allows while keeping every rounding:
//   - each node's products with 1/h are formed once and every difference and
//     sum that two edges, two sides or two elements share is formed once;
//   - with both sides of an edge intact the tangential derivative is the same
//     on both sides, and 0.5 a + 0.5 b is formed as 0.5 (a + b), the halving
//     and the doubling 1/(2h) -> 1/h by an exponent step in integer
//     registers.  These are exact unless a value is subnormal or close to
//     overflow: a CTA whose products leave [2^-800, 2^800] (other than zero)
//     takes the plain formulas instead (a CTA-wide vote);
//   - the bracketed pairs of Eq. 6's sum are formed per edge, up to a sign,
//     not per element and node.
// About 120 instead of 309 FP64 instructions per node: 2683 -> 1095 us on the
// 2048 x 2048 plate, 58 -> 26 us on 400 x 160, 36 -> 10 us on 100 x 40.
// The tile shape follows the mesh (tile64_shape): a small mesh is cut finer so
// that every SM gets a share.
struct Tile64 {
  int tx, ty;    // nodes [i0, i0+tx) x [j0, j0+ty)
  int nw, nh;    // nodes [i0-2, i0+tx+1] x [j0-2, j0+ty+1]
  int ew, eh;    // elements [i0-2, i0+tx] x [j0-2, j0+ty]
  int hw, hh;    // horizontal edges [i0-1, i0+tx) x [j0-1, j0+ty]
  int vw, vh;    // vertical edges [i0-1, i0+tx] x [j0-1, j0+ty)
  __host__ __device__ Tile64(int tx_, int ty_)
      : tx(tx_), ty(ty_), nw(tx_ + 4), nh(ty_ + 4), ew(tx_ + 3), eh(ty_ + 3), hw(tx_ + 1),
        hh(ty_ + 2), vw(tx_ + 2), vh(ty_ + 1) {}
  __host__ __device__ int nodes() const { return nw * nh; }
  __host__ __device__ int elems() const { return ew * eh; }
  __host__ __device__ int hedges() const { return hw * hh; }
  __host__ __device__ int vedges() const { return vw * vh; }
  // node products (4, or 2 of square elements), element sums (4), edge terms (6)
  // and, on record steps, eps.sigma; then the element states
  __host__ __device__ size_t bytes(bool energy, bool square) const {
    return 8 * ((square ? 2 : 4) * (size_t)nodes() + 4 * (size_t)elems() +
                (energy ? 7 : 6) * (size_t)(hedges() + vedges())) + elems();
  }
};

// FP64 instructions of one tile, in warp instructions
inline double tile64_cost(const Tile64 &t) {
  auto w = [](int n) { return (double)((n + 31) / 32); };
  return 4 * w(t.nodes()) + 12 * w(t.elems()) + 21 * w(t.hedges() + t.vedges()) +
         52 * w(t.tx * t.ty);
}

__device__ __forceinline__ void prefetch_l1(const void *p) {
  asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}

// x / 2 and 2 x of a normal number or zero, by its exponent field
__device__ __forceinline__ double half64(double x) {
  const int h = __double2hiint(x);
  return __hiloint2double(h - ((h & 0x7ff00000) ? 0x00100000 : 0), __double2loint(x));
}
__device__ __forceinline__ double twice64(double x) {
  const int h = __double2hiint(x);
  return __hiloint2double(h + ((h & 0x7ff00000) ? 0x00100000 : 0), __double2loint(x));
}
// zero, or within [2^-800, 2^800]
__device__ __forceinline__ bool mid_range64(double x) {
  const unsigned e = ((unsigned)__double2hiint(x) >> 20) & 0x7ff;
  return e - (1023u - 800u) <= 1600u || (e == 0 && ((__double2hiint(x) << 1) | __double2loint(x)) == 0);
}

__device__ __forceinline__ void main64_tile(const DevState &d, VBlk vb, int cur, int first,
                                            int energy, double *sm) {
  const Geo &g = d.g;
  const Tile64 T(d.t64x, d.t64y);
  const int i0 = vb.x * T.tx, j0 = vb.y * T.ty;
  const int tid = threadIdx.x;
  const double *uxc = d.ux[cur], *uyc = d.uy[cur];
  const int nn = T.nodes(), ne = T.elems(), nhe = T.hedges(), nve = T.vedges();
  // node products u/(2hx), v/(2hx), u/(2hy), v/(2hy) (u, v themselves on the plain path)
  double *pa = sm, *pb = pa + nn;
  const bool square = g.rxh == g.ryh;
  double *pc = square ? pa : pb + nn, *pd = square ? pb : pc + nn;
  // element sums: half the normal derivatives that enter exx (vertical edges)
  // and eyy (horizontal edges), and the whole ones that enter gxy
  double *eX = pd + nn, *eN = eX + ne, *eXv = eN + ne, *eNu = eXv + ne;
  // edge terms, planes of nhe (nve) values: see edge_terms
  const int planes = energy ? 7 : 6;
  double *H = eNu + ne, *V = H + planes * nhe;
  uint8_t *sst = reinterpret_cast<uint8_t *>(V + planes * nve);

  int ok = 1;
  for (int q = tid; q < nn; q += NT) {
    const int li = q % T.nw, lj = q / T.nw, i = i0 - 2 + li, j = j0 - 2 + lj;
    double a = 0.0, b = 0.0;
    if (i >= 0 && j >= 0 && i <= g.nx && j <= g.ny) {
      const int N = j * (g.nx + 1) + i;
      a = uxc[N];
      b = uyc[N];
    }
    const double a1 = g.rxh * a, b1 = g.rxh * b;
    pa[q] = a1;
    pb[q] = b1;
    ok &= (int)(mid_range64(a1) && mid_range64(b1));
    if (!square) {
      const double a2 = g.ryh * a, b2 = g.ryh * b;
      pc[q] = a2;
      pd[q] = b2;
      ok &= (int)(mid_range64(a2) && mid_range64(b2));
    }
  }
  for (int q = tid; q < ne; q += NT) {
    const int li = q % T.ew, lj = q / T.ew, i = i0 - 2 + li, j = j0 - 2 + lj;
    uint8_t s = ST_OUT;
    if (i >= 0 && j >= 0 && i < g.nx && j < g.ny) s = d.estate[j * g.nx + i];
    sst[q] = s;
  }
  // what the node updates at the end read besides, on its way into L1
  for (int q = tid; q < T.tx * T.ty; q += NT) {
    const int i = i0 + q % T.tx, j = j0 + q / T.tx;
    if (i > g.nx || j > g.ny) continue;
    const int N = j * (g.nx + 1) + i;
    prefetch_l1(d.vx + N);
    prefetch_l1(d.vy + N);
    prefetch_l1(d.minv + N);
    prefetch_l1(d.nflag + N);
  }
  ok = __syncthreads_and(ok);

  if (ok) {
    for (int q = tid; q < ne; q += NT) {
      if (sst[q] != ST_INTACT) continue;
      const int li = q % T.ew, lj = q / T.ew;
      const int n0 = lj * T.nw + li, n1 = n0 + 1, n3 = n0 + T.nw, n2 = n3 + 1;
      eX[q] = half64(((pa[n1] - pa[n0]) + pa[n2]) - pa[n3]);
      eXv[q] = ((pb[n1] - pb[n0]) + pb[n2]) - pb[n3];
      eN[q] = half64((pd[n2] - (pd[n0] + pd[n1])) + pd[n3]);
      eNu[q] = (pc[n2] - (pc[n0] + pc[n1])) + pc[n3];
    }
  } else {
    // plain path: the displacements themselves
    pc = pa;
    pd = pb;
    for (int q = tid; q < nn; q += NT) {
      const int li = q % T.nw, lj = q / T.nw, i = i0 - 2 + li, j = j0 - 2 + lj;
      const bool in = i >= 0 && j >= 0 && i <= g.nx && j <= g.ny;
      const int N = j * (g.nx + 1) + i;
      pa[q] = in ? uxc[N] : 0.0;
      pb[q] = in ? uyc[N] : 0.0;
    }
  }
  __syncthreads();

  // every edge of the tile: the strain its intact sides use (with both intact
  // the average of theirs), the stress, and the terms the node sums take
  // from it.  Both sides take the same terms, so one set per edge is kept.
  for (int q = tid; q < nhe + nve; q += NT) {
    const bool hor = q < nhe;
    const int p = hor ? q : q - nhe, w = hor ? T.hw : T.vw;
    const int li = p % w, lj = p / w;
    // the elements below and above (left and right) of the edge, the node at its start
    const int eb = hor ? lj * T.ew + li + 1 : (lj + 1) * T.ew + li;
    const int ea = hor ? eb + T.ew : eb + 1;
    const int n0 = (lj + 1) * T.nw + li + 1;
    const bool ib = sst[eb] == ST_INTACT, ia = sst[ea] == ST_INTACT;
    if (!ib && !ia) continue;
    double e[3];
    if (ok) {
      const int es = ib ? eb : ea;  // the (or one) intact side
      if (hor) {
        e[0] = twice64(pa[n0 + 1] - pa[n0]);
        const double t = twice64(pb[n0 + 1] - pb[n0]);
        if (ib && ia) {
          e[1] = eN[eb] + eN[ea];
          e[2] = half64((eNu[eb] + t) + (eNu[ea] + t));
        } else {
          e[1] = twice64(eN[es]);
          e[2] = eNu[es] + t;
        }
      } else {
        e[1] = twice64(pd[n0 + T.nw] - pd[n0]);
        const double t = twice64(pc[n0 + T.nw] - pc[n0]);
        if (ib && ia) {
          e[0] = eX[eb] + eX[ea];
          e[2] = half64((t + eXv[eb]) + (t + eXv[ea]));
        } else {
          e[0] = twice64(eX[es]);
          e[2] = t + eXv[es];
        }
      }
    } else {
      double eB[3], eA[3], u[4], v[4];
      auto gather = [&](int el) {
        const int m0 = (el / T.ew) * T.nw + el % T.ew;
        u[0] = pa[m0];            v[0] = pb[m0];
        u[1] = pa[m0 + 1];        v[1] = pb[m0 + 1];
        u[2] = pa[m0 + T.nw + 1]; v[2] = pb[m0 + T.nw + 1];
        u[3] = pa[m0 + T.nw];     v[3] = pb[m0 + T.nw];
      };
      if (ib) {
        gather(eb);
        if (hor) strain64<2>(g, u, v, eB); else strain64<1>(g, u, v, eB);
      }
      if (ia) {
        gather(ea);
        if (hor) strain64<0>(g, u, v, eA); else strain64<3>(g, u, v, eA);
      }
#pragma unroll
      for (int c = 0; c < 3; ++c)
        e[c] = ib && ia ? 0.5 * eB[c] + 0.5 * eA[c] : ib ? eB[c] : eA[c];
    }
    double s[3];
    stress64(d.mat, e, s);
    // horizontal: x sum 1/hx sxx (k), 1/(2hy) sxy (m); y sum 1/(2hy) syy (l), 1/hx sxy (n)
    // vertical:   x sum 1/(2hx) sxx (k), 1/hy sxy (m); y sum 1/hy syy (l), 1/(2hx) sxy (n)
    double *o = hor ? H + q : V + p;
    const int st = hor ? nhe : nve;
    const double rk = hor ? g.rx : g.rxh, rm = hor ? g.ryh : g.ry;
    const double k = rk * s[0], m = rm * s[2], l = rm * s[1], n = rk * s[2];
    o[0] = k + m;
    o[st] = k - m;
    o[2 * st] = l + n;
    o[3 * st] = n - l;
    o[4 * st] = hor ? m : k;
    o[5 * st] = hor ? l : n;
    if (energy) o[6 * st] = dot3(e, s);
  }
  __syncthreads();

  // only the node sums read what the kernel before this one (the piece forces)
  // writes: the strains and stresses above run beside it
  wait_for_predecessors();
  double ke = 0.0, se = 0.0;
  const double qA = g.A * 0.25;
  for (int q = tid; q < T.tx * T.ty; q += NT) {
    const int tx = q % T.tx, ty = q / T.tx;
    const int i = i0 + tx, j = j0 + ty;
    if (i > g.nx || j > g.ny) continue;
    const int N = j * (g.nx + 1) + i;
    double fx = 0.0, fy = 0.0;
    // adjacent elements in increasing id: (i-1,j-1) a=2, (i,j-1) a=3, (i-1,j) a=1, (i,j) a=0
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int di = (r & 1) - 1, dj = (r >> 1) - 1;
      constexpr int kLocal[4] = {2, 3, 1, 0};
      const int a = kLocal[r];
      const int st = sst[(ty + 2 + dj) * T.ew + tx + 2 + di];
      if (st == ST_INTACT) {
        // bottom, top, left and right edge of the element
        const double *hb = H + (ty + 1 + dj) * T.hw + tx + 1 + di, *ht = hb + T.hw;
        const double *vl = V + (ty + 1 + dj) * T.vw + tx + 1 + di, *vr = vl + 1;
        double sx, sy;
        if (a == 2) {
          sx = ((hb[4 * nhe] + vr[0]) + ht[0]) + vl[4 * nve];
          sy = ((hb[5 * nhe] + vr[2 * nve]) + ht[2 * nhe]) + vl[5 * nve];
        } else if (a == 3) {
          sx = ((hb[4 * nhe] - vr[4 * nve]) - ht[nhe]) - vl[nve];
          sy = ((hb[5 * nhe] - vr[5 * nve]) - ht[3 * nhe]) - vl[3 * nve];
        } else if (a == 1) {
          sx = ((hb[nhe] + vr[nve]) - ht[4 * nhe]) + vl[4 * nve];
          sy = ((hb[3 * nhe] + vr[3 * nve]) - ht[5 * nhe]) + vl[5 * nve];
        } else {
          sx = -(((hb[0] + vr[4 * nve]) + ht[4 * nhe]) + vl[0]);
          sy = -(((hb[2 * nhe] + vr[5 * nve]) + ht[5 * nhe]) + vl[2 * nve]);
        }
        fx = fx + sx * qA;
        fy = fy + sy * qA;
      } else if (st == ST_CRACKED) {
        const int e = (j + dj) * g.nx + i + di;
        const int c = d.crack_of[e];
        const int side = (d.ck_info[c] >> (4 + a)) & 1;
        fx = fx + d.pf[c * 16 + side * 8 + 2 * a];
        fy = fy + d.pf[c * 16 + side * 8 + 2 * a + 1];
      }
    }
    ke += update_node(d, N, cur, first != 0, fx, fy, d.nflag[N], energy != 0);
    if (energy && i < g.nx && j < g.ny && sst[(ty + 2) * T.ew + tx + 2] == ST_INTACT) {
      const double *hb = H + 6 * nhe + (ty + 1) * T.hw + tx + 1, *ht = hb + T.hw;
      const double *vl = V + 6 * nve + (ty + 1) * T.vw + tx + 1, *vr = vl + 1;
      const double dk[4] = {*hb, *vr, *ht, *vl};
      double acc = 0.0;
#pragma unroll
      for (int k = 0; k < 4; ++k) acc = acc + 0.5 * (qA * dk[k]);
      se += acc;
    }
  }
  if (energy) {
    int b = vb.y * vb.gx + vb.x;
    block_sum2(ke, se, d.e_part + 2 * b);
  }
}

__global__ void __launch_bounds__(NT) k_main64(DevState d, int cur, int first, int energy) {
  // a programmatic dependent of the piece forces (7 us, most of it latency), which
  // start after the previous step's split writes have completed: it runs beside
  // them and waits where main64_tile first needs them
  release_dependents();
  extern __shared__ double sm64[];
  main64_tile(d, hw_vblk(), cur, first, energy, sm64);
}

// ---------------------------------------------------------------- phantoms
__device__ __forceinline__ void phantom64(const DevState &d, VBlk vb, int cur, int first,
                                          int energy, int part_off) {
  const int n = d.cnt->n_ph;
  double ke = 0.0;
  for (int t = vb.x * blockDim.x + threadIdx.x; t < n; t += vb.gx * blockDim.x) {
    int N = d.g.nn + t;
    // users' piece-force indices in increasing element id, -1 unused
    const int4 uf = reinterpret_cast<const int4 *>(d.ph_upf)[t];
    const int us[4] = {uf.x, uf.y, uf.z, uf.w};
    double fx = 0.0, fy = 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (us[q] < 0) break;
      fx = fx + d.pf[us[q]];
      fy = fy + d.pf[us[q] + 1];
    }
    ke += update_node(d, N, cur, first != 0, fx, fy, 0, energy != 0);
  }
  if (energy) block_sum2(ke, 0.0, d.e_part + 2 * (part_off + vb.x));
}

__global__ void k_phantom64(DevState d, int cur, int first, int energy, int part_off) {
  phantom64(d, hw_vblk(), cur, first, energy, part_off);
}

// Surface evaluation, 32 points per block of four warps: warp k forms the
// candidate of local edge k (every lane of a warp then runs the same
// formulas), warp 0 applies the rule.  Bound by the FP64 pipe of the SMs that
// hold points, so few points per SM: a block of 256 threads, one point each,
// took 36 us for 380 points (two SMs busy) on the 100 x 40 plate, this 7 us;
// 43 and 13 us for the 9,008 points of the 2048 x 2048 plate.
constexpr int kEvalPts = 32, kEvalTB = 4 * kEvalPts;

__device__ __forceinline__ void eval64(const DevState &d, VBlk vb, int cur) {
  __shared__ double sG[4][kEvalPts];
  const int n = d.cnt->n_S;
  const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
  const U64 U{d.ux[cur], d.uy[cur]};
  for (int base = vb.x * kEvalPts; base < n; base += vb.gx * kEvalPts) {
    const int i = base + lane;
    int key = 0, edge = -1;
    if (i < n) edge = d.S[i];
    bool live = edge >= 0;
    if (live) {
      key = d.S_info[i];
      live = d.mat.scope != 2 || is_tip_edge(d, key >> 2, key & 3);
    }
    if (live) sG[k][lane] = eval_G64_k(d, U, key >> 2, key & 3, k);
    __syncthreads();
    if (k == 0) {
      bool has = false;
      int kk = -1;
      double Gk = 0.0;
      if (live) {
        const double G[4] = {sG[0][lane], sG[1][lane], sG[2][lane], sG[3][lane]};
        double gm = -1.0;
        for (int c = 0; c < 4; ++c) gm = fmax(gm, G[c]);
        d.S_G[i] = gm;
        kk = q4_rule(d, key >> 2, key & 3, G);
        if (kk >= 0) { has = true; Gk = G[kk]; }
      }
      append_proposal(d, has, key, edge, kk, Gk);
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kEvalTB) k_eval64(DevState d, int cur) {
  wait_for_predecessors();
  release_dependents();
  eval64(d, hw_vblk(), cur);
}

// ---------------------------------------------------------------- batched
// One launch per kernel kind for every member of a batch (persistent grids
// walking the work lists; 1-D items are (member, block, energy-partial
// offset, member's grid size)).
__global__ void __launch_bounds__(NT) k_main64_batch(BatchDev b, int first, int energy) {
  extern __shared__ double sm64[];
  __shared__ DevState sd;
  int held = -1, w0, w1;
  const int n = *b.bstep;
  block_range(b.n_main, w0, w1);
  for (int w = w0; w < w1; ++w) {
    const int4 it = b.w_main[w];
    stage_member(b.ds, it.x, sd, held);
    if (!member_active(sd, n)) continue;
    main64_tile(sd, item_vblk(it), member_cur(sd, n), first, energy, sm64);
    __syncthreads();
  }
}

__global__ void k_pieces64_batch(BatchDev b, int energy) {
  release_dependents();
  __shared__ DevState sd;
  int held = -1, w0, w1;
  const int n = *b.bstep;
  block_range(b.n_pieces, w0, w1);
  for (int w = w0; w < w1; ++w) {
    const int4 it = b.w_pieces[w];
    stage_member(b.ds, it.x, sd, held);
    if (!member_active(sd, n)) continue;
    pieces64(sd, VBlk{it.y, 0, it.w, 1}, member_cur(sd, n), energy, it.z);
    __syncthreads();
  }
}

__global__ void k_phantom64_batch(BatchDev b, int first, int energy) {
  __shared__ DevState sd;
  int held = -1, w0, w1;
  const int n = *b.bstep;
  block_range(b.n_ph, w0, w1);
  for (int w = w0; w < w1; ++w) {
    const int4 it = b.w_ph[w];
    stage_member(b.ds, it.x, sd, held);
    if (!member_active(sd, n)) continue;
    phantom64(sd, VBlk{it.y, 0, it.w, 1}, member_cur(sd, n), first, energy, it.z);
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kEvalTB) k_eval64_batch(BatchDev b) {
  __shared__ DevState sd;
  int held = -1, w0, w1;
  const int n = *b.bstep;
  block_range(b.n_eval, w0, w1);
  for (int w = w0; w < w1; ++w) {
    const int4 it = b.w_eval[w];
    stage_member(b.ds, it.x, sd, held);
    if (!member_active(sd, n)) continue;
    eval64(sd, VBlk{it.y, 0, it.w, 1}, member_cur(sd, n));
    __syncthreads();
  }
}

// ------------------------------------------------------------- init masses
__global__ void k_init_masses(DevState d) {
  const Geo &g = d.g;
  for (int N = blockIdx.x * blockDim.x + threadIdx.x; N < g.nn; N += gridDim.x * blockDim.x) {
    int r = g.nx + 1, i = N % r, j = N / r;
    const int di[4] = {-1, 0, -1, 0}, dj[4] = {-1, -1, 0, 0};
    double acc = 0.0;
    for (int q = 0; q < 4; ++q) {
      int ei = i + di[q], ej = j + dj[q];
      if (ei < 0 || ej < 0 || ei >= g.nx || ej >= g.ny) continue;
      if (d.estate[ej * g.nx + ei] == ST_INTACT) acc = acc + d.mat.rho * g.A * 0.25;
    }
    d.m[N] = acc;
    d.minv[N] = acc > 0.0 ? 1.0 / acc : 0.0;
  }
}

int grid_for(int n, int block, int maxb) {
  int b = (n + block - 1) / block;
  return b < 1 ? 1 : (b > maxb ? maxb : b);
}

}  // namespace

int energy_parts_fp32(const DevState &d);

// Tile shape of a mesh's FP64 node update: of the shapes below, the one with
// the fewest FP64 instructions on the busiest SM, tiles being dealt evenly to
// the 152 SMs, plus a constant for a tile's load and barrier latency (about
// 60 warp instructions' time; it matters for small meshes only).  On the 100 x
// 40 plate that is 16 x 2 nodes (10 us; 32 x 8 takes 36), on 400 x 160 32 x 8,
// on large meshes 32 x 12, of which three CTAs share an SM where the elements are
// square, two elsewhere (launch_step_fp64).
void tile64_shape(int nx, int ny, int &tx, int &ty) {
  constexpr int kTx[] = {32, 16}, kTy[] = {12, 8, 6, 4, 3, 2, 1}, kSms = 152;
  double best = 0.0;
  tx = 0;
  for (int x : kTx)
    for (int y : kTy) {
      const long n = (long)((nx + 1 + x - 1) / x) * ((ny + 1 + y - 1) / y);
      const double c = (double)((n + kSms - 1) / kSms) * (tile64_cost(Tile64(x, y)) + 60.0);
      if (tx == 0 || c < best) {
        best = c;
        tx = x;
        ty = y;
      }
    }
}

void grid_main64(const DevState &d, int &gx, int &gy) {
  gx = (d.g.nx + 1 + d.t64x - 1) / d.t64x;
  gy = (d.g.ny + 1 + d.t64y - 1) / d.t64y;
}

int tiles_fp64(const DevState &d) {
  int gx, gy;
  grid_main64(d, gx, gy);
  return gx * gy;
}

// piece blocks of kPieceTB threads (one per piece): small blocks, so that
// the pieces of a small crack set spread over the SMs' FP64 pipes (100 x 40
// plate, 5,700 pieces: 15 -> 8 us against blocks of 256)
constexpr int kPieceTB = 64;
int grid_pieces64(const DevState &d) { return grid_for(2 * d.ck_cap, kPieceTB, 608); }

// evaluation blocks: 32 surface points each
int grid_eval64(const DevState &d) { return grid_for(d.list_cap, kEvalPts, 608); }

namespace {
// The FP64 step's kernels ask for one shared-memory split (see
// match_tile_carveout), so that the surface evaluation's blocks do not keep
// the node update off their SMs.
cudaError_t fp64_attrs() {
  static PerDevice attrs;
  return attrs.once([] {
    const int most = (int)Tile64(32, 12).bytes(true, false);
    cudaError_t e = cudaFuncSetAttribute(k_main64, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_main64_batch, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
    if (e == cudaSuccess) e = match_tile_carveout(k_main64);
    if (e == cudaSuccess) e = match_tile_carveout(k_main64_batch);
    if (e == cudaSuccess) e = match_tile_carveout(k_pieces64);
    if (e == cudaSuccess) e = match_tile_carveout(k_pieces64_batch);
    if (e == cudaSuccess) e = match_tile_carveout(k_phantom64);
    if (e == cudaSuccess) e = match_tile_carveout(k_phantom64_batch);
    if (e == cudaSuccess) e = match_tile_carveout(k_eval64);
    if (e == cudaSuccess) e = match_tile_carveout(k_eval64_batch);
    return e;
  });
}
}  // namespace

int energy_parts_needed(const DevState &d) {
  if (d.precision == 1) return energy_parts_fp32(d);
  return tiles_fp64(d) + 2 * 1216 + 8;
}

int energy_parts_step_fp32(const DevState &d, int tile_rows);
int march_rows_solo(const DevState &d);

int energy_parts_step(const DevState &d) {
  if (d.precision == 1) return energy_parts_step_fp32(d, march_rows_solo(d));
  return tiles_fp64(d) + grid_pieces64(d) + grid_phantoms(d);
}

cudaError_t launch_init_masses(const DevState &d, cudaStream_t st) {
  k_init_masses<<<grid_for(d.g.nn, 256, 4096), 256, 0, st>>>(d);
  return cudaGetLastError();
}

cudaError_t launch_step_fp64(const DevState &d, int cur, bool first, bool energy,
                             const StepStreams &ss, cudaEvent_t *marks) {
  cudaError_t e = fp64_attrs();
  if (e != cudaSuccess) return e;
  int gx, gy;
  grid_main64(d, gx, gy);
  const dim3 grid(gx, gy);
  int tiles = gx * gy;
  // Three CTAs of 32 x 12 square elements (70 KB each) feed the FP64 pipe better than
  // two (2048 x 2048: 1136 -> 1097 us, the pipe 80% busy with two; 1000 x 1000: 295 ->
  // 281), if the SM gives them all of its memory.  Meshes of few waves keep the side
  // kernels' split, as an SM changes it only when it is empty (100 x 40: 18.7 us a
  // step, 19.7 otherwise), and two CTAs, as a third on some SMs leaves others idle
  // (400 x 160: 32.7 and 37.9).
  const bool large = tiles >= 3 * 3 * 152;
  const size_t smem = Tile64(d.t64x, d.t64y).bytes(energy, large && d.g.rxh == d.g.ryh);
  int gp = grid_pieces64(d);
  int gph = grid_phantoms(d);
  const int ge = grid_eval64(d);
  cudaStream_t st = ss.main;
  if (marks) {
    k_pieces64<<<gp, kPieceTB, 0, st>>>(d, cur, energy ? 1 : 0, tiles);
    cudaEventRecord(marks[0], st);
    k_main64<<<grid, NT, smem, st>>>(d, cur, first ? 1 : 0, energy ? 1 : 0);
    cudaEventRecord(marks[1], st);
    k_phantom64<<<gph, 256, 0, st>>>(d, cur, first ? 1 : 0, energy ? 1 : 0, tiles + gp);
    cudaEventRecord(marks[2], st);
    k_eval64<<<ge, kEvalTB, 0, st>>>(d, cur);
    return cudaGetLastError();
  }
  cudaEventRecord(ss.fork, st);
  cudaStreamWaitEvent(ss.aux2, ss.fork, 0);
  launch_dependent(k_eval64, ge, kEvalTB, 0, ss.aux2, d, cur);
  launch_select(d, TRACK_STEP, ss.aux2);
  launch_dependent(k_pieces64, gp, kPieceTB, 0, st, d, cur, energy ? 1 : 0, tiles);
  cudaEventRecord(ss.fork, st);
  cudaStreamWaitEvent(ss.aux1, ss.fork, 0);
  k_phantom64<<<gph, 256, 0, ss.aux1>>>(d, cur, first ? 1 : 0, energy ? 1 : 0, tiles + gp);
  launch_dependent_carveout(large ? 100 : 0, k_main64, grid, NT, smem, st, d, cur, first ? 1 : 0, energy ? 1 : 0);
  cudaEventRecord(ss.join1, ss.aux1);
  cudaEventRecord(ss.join2, ss.aux2);
  cudaStreamWaitEvent(st, ss.join1, 0);
  cudaStreamWaitEvent(st, ss.join2, 0);
  return cudaGetLastError();
}

// The same fork/join as launch_step_fp64, one launch per kernel kind for all
// members of the batch.
cudaError_t launch_step_fp64_batch(const BatchDev &b, bool first, bool energy, int grid_main,
                                   const StepStreams &ss) {
  cudaError_t e = fp64_attrs();
  if (e != cudaSuccess) return e;
  const int gm = grid_main < 1 ? 1 : grid_main;
  // four times the piece blocks of 256 threads that the SMs hold, as these have 64: 64 specimens
  // of 50 x 20 to 100 x 40 elements, most of them split, 409 us a step with 1216, 318 so
  const int gp = grid_for(b.n_pieces, 1, 4 * 1216), gph = grid_for(b.n_ph, 1, 1216);
  const int ge = grid_for(b.n_eval, 1, 1216);
  cudaStream_t st = ss.main;
  cudaEventRecord(ss.fork, st);
  cudaStreamWaitEvent(ss.aux2, ss.fork, 0);
  k_eval64_batch<<<ge, kEvalTB, 0, ss.aux2>>>(b);
  e = launch_select_batch(b, ss.aux2);
  if (e != cudaSuccess) return e;
  k_pieces64_batch<<<gp, kPieceTB, 0, st>>>(b, energy ? 1 : 0);
  cudaEventRecord(ss.fork, st);
  cudaStreamWaitEvent(ss.aux1, ss.fork, 0);
  k_phantom64_batch<<<gph, 256, 0, ss.aux1>>>(b, first ? 1 : 0, energy ? 1 : 0);
  launch_dependent(k_main64_batch, gm, NT, Tile64(32, 12).bytes(energy, false), st, b, first ? 1 : 0, energy ? 1 : 0);
  cudaEventRecord(ss.join1, ss.aux1);
  cudaEventRecord(ss.join2, ss.aux2);
  cudaStreamWaitEvent(st, ss.join1, 0);
  cudaStreamWaitEvent(st, ss.join2, 0);
  return cudaGetLastError();
}

const void *phantom64_kernel() { return reinterpret_cast<const void *>(&k_phantom64); }

}  // namespace cem
