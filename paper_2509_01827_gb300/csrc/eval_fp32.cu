// eval_fp32.cu -- surface-point evaluation of the FP32-mixed mode
// (compiled with -fmad=false so that its FP64 re-check uses the same
// operation order as the FP64 mode).
//
// Each free-surface point computes the energy release rate of its three
// candidate paths (Sec. 2.2) in FP32 from the compensated displacement.  If
// any candidate lies within 1e-3 of G_c (|G/G_c - 1| < 1e-3) the point is
// re-evaluated in FP64, so that the threshold decision is the FP64 one.  The
// Q4 cracking rule then runs on the (FP64-widened) values and proposals are
// appended with a warp ballot.
#include <cuda_runtime.h>

#include "cem_internal.h"
#include "eval_common.cuh"
#include "q4_fp64.cuh"

namespace cem {

namespace {

__device__ __forceinline__ float df_diff(float ah, float al, float bh, float bl) {
  return (bh - ah) + (bl - al);
}

// Own FP32 strain of an intact element at its edge k (Eq. 4 at the edge
// point), from its four nodes' displacement pairs in local order.
__device__ __forceinline__ void own_strain32(const Geo &g, const float4 (&q)[4], int k,
                                             float eps[3]) {
  const float rx = g.rxf, ry = g.ryf, hx2 = 0.5f * rx, hy2 = 0.5f * ry;
  // differences along the edges: a bottom, b top, c left, e right
  const float au = df_diff(q[0].x, q[0].y, q[1].x, q[1].y), bu = df_diff(q[3].x, q[3].y, q[2].x, q[2].y);
  const float cu = df_diff(q[0].x, q[0].y, q[3].x, q[3].y), eu = df_diff(q[1].x, q[1].y, q[2].x, q[2].y);
  const float av = df_diff(q[0].z, q[0].w, q[1].z, q[1].w), bv = df_diff(q[3].z, q[3].w, q[2].z, q[2].w);
  const float cv = df_diff(q[0].z, q[0].w, q[3].z, q[3].w), ev = df_diff(q[1].z, q[1].w, q[2].z, q[2].w);
  if (k & 1) {
    eps[0] = hx2 * (au + bu);
    eps[1] = ry * (k == 1 ? ev : cv);
    eps[2] = ry * (k == 1 ? eu : cu) + hx2 * (av + bv);
  } else {
    eps[0] = rx * (k == 0 ? au : bu);
    eps[1] = hy2 * (cv + ev);
    eps[2] = hy2 * (cu + eu) + rx * (k == 0 ? av : bv);
  }
}

// G of the candidate path of local edge k != k0 of surface point (e, k0), and
// G_c of e.  Everything it reads (the nodes of e and of the element across
// edge k, that element's state, G_c) is loaded in one level.
__device__ __forceinline__ float eval_G32_k(const DevState &d, const float4 *u, int e, int k0, int k,
                                            float &gc) {
  const Geo &g = d.g;
  const int i = e % g.nx, j = e / g.nx, r = g.nx + 1, n0 = j * r + i;
  const int di = k == 1 ? 1 : k == 3 ? -1 : 0, dj = k == 2 ? 1 : k == 0 ? -1 : 0;
  const bool in = i + di >= 0 && i + di < g.nx && j + dj >= 0 && j + dj < g.ny;
  const int m0 = in ? n0 + dj * r + di : n0;  // node 0 of the element across edge k
  const float4 q[4] = {u[n0], u[n0 + 1], u[n0 + r + 1], u[n0 + r]};
  const float4 f[4] = {u[m0], u[m0 + 1], u[m0 + r + 1], u[m0 + r]};
  const bool both = in && d.estate[e + (in ? dj * g.nx + di : 0)] == ST_INTACT;
  gc = d.gc[e];
  const float DX = g.DXf[k0], DY = g.DYf[k0];
  float4 P1 = q[0], P2 = q[1];
#pragma unroll
  for (int a = 1; a < 4; ++a)
    if (a == k0) { P1 = q[a]; P2 = q[(a + 1) & 3]; }
  const float dux = df_diff(P1.x, P1.y, P2.x, P2.y);
  const float duy = df_diff(P1.z, P1.w, P2.z, P2.w);
  // |x_N2 - x_N1|^2 - |X_N2 - X_N1|^2 without cancellation
  const float stretch = 2.f * (DX * dux + DY * duy) + (dux * dux + duy * duy);
  const float H = stretch > 0.f ? 1.f : 0.f;
  const float ddx = dux * H, ddy = duy * H;
  // the stress used at edge k: smoothed with an intact neighbour
  float e1[3], e2[3];
  own_strain32(g, q, k, e1);
  own_strain32(g, f, (k + 2) & 3, e2);
#pragma unroll
  for (int c = 0; c < 3; ++c) e1[c] = both ? 0.5f * (e1[c] + e2[c]) : e1[c];
  const Mat &m = d.mat;
  const float s0 = m.D11f * e1[0] + m.D12f * e1[1];
  const float s1 = m.D12f * e1[0] + m.D11f * e1[1];
  const float s2 = m.D33f * e1[2];
  const float nx = g.nxf[k0][k], ny = g.nyf[k0][k];
  const float tx = s0 * nx + s2 * ny;
  const float ty = s2 * nx + s1 * ny;
  return 0.5f * (ddx * tx + ddy * ty);
}

// FP64 work of the rare point, out of line so that it is not predicated into
// (and its code not fetched for) every point's evaluation: the candidate's
// energy release rate, and the cracking rule.
__device__ __noinline__ double recheck64(const DevState &d, const float4 *u, int e, int k0, int k) {
  const U32x2 U{u};
  return eval_G64_k(d, U, e, k0, k);
}
__device__ __noinline__ int rule64(const DevState &d, int e, int k0, const double *G) {
  const double g4[4] = {G[0], G[1], G[2], G[3]};
  return q4_rule(d, e, k0, g4);
}

// 32 points per block of four warps, warp k forms the candidate of local edge
// k, warp 0 applies the rule.  Bound by latency (the selection and the split
// writes wait for it): the list entries are read beside its length, a
// candidate's inputs in one level, and FP64 is left to points near the
// threshold or above it.  With one thread a point, 256 a block, the three
// candidates, their re-check and the FP64 rule came one after another: 6.4 us for
// the 1,700 points of a notched 400 x 160 plate, now 4.0; 9.9 and 6.7 us for the
// 6,400 of a breaking 1024 x 1024 one, 8.1 and 4.3 us for 9,008 intact ones.
constexpr int kEvalPts = 32, kEvalTB = 4 * kEvalPts;

__device__ __forceinline__ void eval32(const DevState &d, VBlk vb, int cur) {
  __shared__ float sG[4][kEvalPts];
  __shared__ double sD[4][kEvalPts];
  __shared__ unsigned s_near[4];
  const int n = d.cnt->n_S;
  const int lane = threadIdx.x & 31, k = threadIdx.x >> 5;
  const float4 *u = d.u4[cur];
  for (int base = vb.x * kEvalPts; base < d.list_cap; base += vb.gx * kEvalPts) {
    const int i = base + lane;
    int edge = -1, key = 0;
    if (i < d.list_cap) {
      edge = d.S[i];
      key = d.S_info[i];
    }
    if (base >= n) break;
    const int e = key >> 2, k0 = key & 3;
    bool live = i < n && edge >= 0;
    if (live && d.mat.scope == 2) live = is_tip_edge(d, e, k0);
    float G = -1.f, gc = 0.f;
    bool near = false;
    if (live && k != k0) {
      G = eval_G32_k(d, u, e, k0, k, gc);
      near = fabsf(G / gc - 1.f) < 1e-3f;
    }
    sG[k][lane] = G;
    const unsigned nm = __ballot_sync(0xffffffffu, near);
    if (lane == 0) s_near[k] = nm;
    __syncthreads();
    // FP64 re-check of every candidate of a point near the threshold
    const unsigned nears = s_near[0] | s_near[1] | s_near[2] | s_near[3];
    if (nears) {
      if ((nears >> lane) & 1) sD[k][lane] = recheck64(d, u, e, k0, k);
      __syncthreads();
    }
    if (k == 0) {
      int kk = -1;
      double Gk = 0.0;
      if (live) {
        double g4[4];
        double gm;
        bool above;
        if ((nears >> lane) & 1) {
          gm = -1.0;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            g4[c] = sD[c][lane];
            gm = fmax(gm, g4[c]);
          }
          above = true;
        } else {
          float m = -1.f;
#pragma unroll
          for (int c = 0; c < 4; ++c) m = fmaxf(m, sG[c][lane]);
          gm = (double)m;
          above = m > d.gc[e];  // otherwise no candidate is, and the rule proposes nothing
          if (above) {
#pragma unroll
            for (int c = 0; c < 4; ++c) g4[c] = (double)sG[c][lane];
          }
        }
        d.S_G[i] = gm;
        if (above) {
          kk = rule64(d, e, k0, g4);
          if (kk >= 0) Gk = kk == 0 ? g4[0] : kk == 1 ? g4[1] : kk == 2 ? g4[2] : g4[3];
        }
      }
      append_proposal(d, kk >= 0, key, edge, kk, Gk);
    }
    if (base + vb.gx * kEvalPts < n) __syncthreads();  // read before the next points' values
  }
}

__global__ void __launch_bounds__(kEvalTB) k_eval32(DevState d, int cur) {
  wait_for_predecessors();
  release_dependents();
  eval32(d, hw_vblk(), cur);
}

// Everything the FP32 evaluation of surface point (e, k0) reads, loaded in
// one level: the displacement pairs of e's nodes, the states of its four
// neighbours, the two far nodes of each neighbour inside the mesh (across
// the edges other than k0) and G_c of e.
struct EvalPatch {
  float4 ue[4];     // e's nodes, local order
  float4 far[4][2]; // neighbour across edge k: its two nodes not on edge k
  int st[4];        // neighbour states (ST_OUT outside the mesh)
  float gc;
};

__device__ __forceinline__ void load_patch(const DevState &d, const U32x2 &U, int e, int k0,
                                           EvalPatch &P) {
  const Geo &g = d.g;
  const int i = e % g.nx, j = e / g.nx, r = g.nx + 1;
  const int n0 = j * r + i, n1 = n0 + 1, n2 = n0 + r + 1, n3 = n0 + r;
  const int nd[4] = {n0, n1, n2, n3};
  // far nodes of the neighbour below, right, above, left
  const int fa[4][2] = {{n0 - r, n1 - r}, {n1 + 1, n2 + 1}, {n2 + r, n3 + r}, {n0 - 1, n3 - 1}};
#pragma unroll
  for (int a = 0; a < 4; ++a) P.ue[a] = U.u[nd[a]];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int f = elem_neighbor(g, e, k);
    P.st[k] = estatus(d, f);
    const bool use = f >= 0 && k != k0;
    P.far[k][0] = use ? U.u[fa[k][0]] : make_float4(0.f, 0.f, 0.f, 0.f);
    P.far[k][1] = use ? U.u[fa[k][1]] : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  P.gc = d.gc[e];
}

// The neighbour across edge k in its own local node order.
__device__ __forceinline__ void neighbour_nodes(const EvalPatch &P, int k, float4 (&q)[4]) {
  switch (k) {
    case 0: q[0] = P.far[0][0]; q[1] = P.far[0][1]; q[2] = P.ue[1]; q[3] = P.ue[0]; break;
    case 1: q[0] = P.ue[1]; q[1] = P.far[1][0]; q[2] = P.far[1][1]; q[3] = P.ue[2]; break;
    case 2: q[0] = P.ue[3]; q[1] = P.ue[2]; q[2] = P.far[2][0]; q[3] = P.far[2][1]; break;
    default: q[0] = P.far[3][0]; q[1] = P.ue[0]; q[2] = P.ue[3]; q[3] = P.far[3][1]; break;
  }
}

__device__ __forceinline__ void used_stress32(const DevState &d, const EvalPatch &P, int k,
                                              float s[3]) {
  float e1[3];
  own_strain32(d.g, P.ue, k, e1);
  if (P.st[k] == ST_INTACT) {
    float4 q[4];
    neighbour_nodes(P, k, q);
    float e2[3];
    own_strain32(d.g, q, (k + 2) & 3, e2);
    for (int c = 0; c < 3; ++c) e1[c] = 0.5f * (e1[c] + e2[c]);
  }
  const Mat &m = d.mat;
  s[0] = m.D11f * e1[0] + m.D12f * e1[1];
  s[1] = m.D12f * e1[0] + m.D11f * e1[1];
  s[2] = m.D33f * e1[2];
}

__device__ __forceinline__ void eval_G32(const DevState &d, const EvalPatch &P, int k0,
                                         float G[4]) {
  const Geo &g = d.g;
  const float DX = g.DXf[k0], DY = g.DYf[k0];
  float4 P1 = P.ue[0], P2 = P.ue[1];
#pragma unroll
  for (int a = 1; a < 4; ++a)
    if (a == k0) { P1 = P.ue[a]; P2 = P.ue[(a + 1) & 3]; }
  float dux = df_diff(P1.x, P1.y, P2.x, P2.y);
  float duy = df_diff(P1.z, P1.w, P2.z, P2.w);
  // |x_N2 - x_N1|^2 - |X_N2 - X_N1|^2 without cancellation
  float stretch = 2.f * (DX * dux + DY * duy) + (dux * dux + duy * duy);
  float H = stretch > 0.f ? 1.f : 0.f;
  float ddx = dux * H, ddy = duy * H;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (k == k0) { G[k] = -1.f; continue; }
    const float nx = g.nxf[k0][k], ny = g.nyf[k0][k];
    float s[3];
    used_stress32(d, P, k, s);
    float tx = s[0] * nx + s[2] * ny;
    float ty = s[2] * nx + s[1] * ny;
    G[k] = 0.5f * (ddx * tx + ddy * ty);
  }
}

// Large meshes: a thread per point, its candidates one after another, one
// block of 256 threads per SM.  There the node update sets the step, or the piece
// forces once much is broken, and this form takes less from them: an intact
// 2048 x 2048 plate's step is 55.0 us, 57.5 with the split above, one with 1.1
// million split elements 245 and 322 us (between, after 400 to 9000 steps of a breaking
// plate, both take as long within 2%).  On a 1024 x 1024 plate, whose step is the chain
// of evaluation, selection and split writes, the split is the better one (40 us
// while it breaks, 45 with this form).
constexpr int kLargeMesh = 1 << 21;  // nodes
__device__ __forceinline__ void eval32_points(const DevState &d, VBlk vb, int cur) {
  const int n = d.cnt->n_S;
  const U32x2 U{d.u4[cur]};
  for (int base = vb.x * blockDim.x; base < n; base += vb.gx * blockDim.x) {
    int i = base + threadIdx.x;
    bool has = false;
    int key = 0, edge = 0, kk = -1;
    double Gk = 0.0;
    if (i < n) {
      edge = d.S[i];
      const int info = d.S_info[i];
      if (edge >= 0) {
        key = info;
        int e = key >> 2, k0 = key & 3;
        if (d.mat.scope != 2 || is_tip_edge(d, e, k0)) {
          EvalPatch P;
          load_patch(d, U, e, k0, P);
          float G32[4];
          eval_G32(d, P, k0, G32);
          float gc = P.gc;
          bool near = false;
          for (int k = 0; k < 4; ++k)
            if (k != k0 && fabsf(G32[k] / gc - 1.f) < 1e-3f) near = true;
          double G[4];
          if (near) {
            // FP64 re-check near the threshold
            for (int k = 0; k < 4; ++k) G[k] = recheck64(d, d.u4[cur], e, k0, k);
          } else {
            for (int k = 0; k < 4; ++k) G[k] = (double)G32[k];
          }
          double gm = -1.0;
          for (int k = 0; k < 4; ++k) gm = fmax(gm, G[k]);
          d.S_G[i] = gm;
          kk = rule64(d, e, k0, G);
          if (kk >= 0) { has = true; Gk = G[kk]; }
        }
      }
    }
    append_proposal(d, has, key, edge, kk, Gk);
  }
}

__global__ void __launch_bounds__(256, 4) k_eval32_points(DevState d, int cur) {
  eval32_points(d, hw_vblk(), cur);
}

__global__ void __launch_bounds__(kEvalTB) k_eval32_batch(BatchDev b) {
  __shared__ DevState sd;
  int held = -1, w0, w1;
  const int n = *b.bstep;
  block_range(b.n_eval, w0, w1);
  for (int w = w0; w < w1; ++w) {
    const int4 it = b.w_eval[w];
    stage_member(b.ds, it.x, sd, held);
    if (!member_active(sd, n)) continue;
    eval32(sd, VBlk{it.y, 0, it.w, 1}, member_cur(sd, n));
    __syncthreads();  // this item's shared values are read before the next one's (39 members on: two a block)
  }
}

int grid_for(int n, int block, int maxb) {
  int b = (n + block - 1) / block;
  return b < 1 ? 1 : (b > maxb ? maxb : b);
}

}  // namespace

int grid_eval(const DevState &d) { return grid_for(d.list_cap, kEvalPts, 608); }

// k_eval32 asks for no shared-memory split.  With the node update's (164 KB) an SM that
// runs it keeps little L1 for the piece forces beside it, which gather nodes: a
// 1024 x 1024 plate with 590,000 split elements took 141 us a step so, 116 without; with
// 59,000 of them 40 and 37, and as long with few.
cudaError_t eval32_carveouts() {
  static PerDevice attrs;
  return attrs.once([] {
    cudaError_t e = match_tile_carveout(k_eval32_batch);
    if (e == cudaSuccess) e = match_tile_carveout(k_eval32_points);
    return e;
  });
}

cudaError_t launch_eval32(const DevState &d, int cur, cudaStream_t st) {
  cudaError_t e = eval32_carveouts();
  if (e != cudaSuccess) return e;
  if (d.g.nn > kLargeMesh) {
    k_eval32_points<<<grid_for(d.list_cap, 256, 152), 256, 0, st>>>(d, cur);
    return cudaGetLastError();
  }
  return launch_dependent(k_eval32, grid_eval(d), kEvalTB, 0, st, d, cur);
}

cudaError_t launch_eval32_batch(const BatchDev &b, cudaStream_t st) {
  cudaError_t e = eval32_carveouts();
  if (e != cudaSuccess) return e;
  k_eval32_batch<<<grid_for(b.n_eval, 1, 1216), kEvalTB, 0, st>>>(b);
  return cudaGetLastError();
}

}  // namespace cem
