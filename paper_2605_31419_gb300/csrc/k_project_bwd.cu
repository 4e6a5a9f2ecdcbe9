// k_project_bwd.cu -- chain rule from the per-face screen-space sums to the map and the pose.
//
// Closed form per visible (view, face), from the 22 sums the raster backward accumulated (26 with the side array):
//   * interpolants with vertex values w (colour channels, camera depth): dL/dw_k is the sum
//     itself, and moving vertex k moves the interpolant's plane: dL/dq_k -= dL/dw_k * grad f;
//   * edge functions E_i = s_i lambda_{i+2} with s_i = perimeter / |e_i| (Eq. 2-3 normalised
//     by phi(s), the inradius): the same plane term plus the chain through the edge lengths;
//   * o_F = (o_i + o_j + o_k) / 3 (Sec. 3.1): each vertex opacity gets a third;
//   * with TS_FLAG_NORMALS, the face normal of the normal map (Eq. 12) through the cross product
//     of the camera-space edge vectors; with TS_FLAG_FACE_SIGMA, dL/dsigma_F (a sum the raster
//     backward already formed) is summed over views;
//   * the pinhole (Eq. 1) to camera space, R^T to world space, and the left-perturbation pose
//     Jacobian [I, -[v_C]x] (Eq. 7): dL/dtau += [g_C ; v_C x g_C].
//
// Gradient slots are face-major (slot = face * V + view) and cleared by the projection pass for
// the visible ones; each is read once, in full, and nothing is written back.  Two forms:
//   * with map gradients, a warp takes 32 faces at a time (2 to 16 of a small map or for many views): it stages
//     the faces' vertices in shared memory, lists their visible entries face by face with views in order, and
//     runs the chain rule on 32 entries at a time; each entry leaves its 20 map words in a shared row, the words
//     are summed over each face's rows in view order, and the sums are added to the map gradient, consecutive
//     vertices by consecutive lanes.  Pose terms are added to per-view sums in face order;
//   * without map gradients (tracking), warps walk one view's faces, queue the visible ones and run the
//     chain rule on full warps, each lane keeping its own pose sums.
// In both, a lane's next slot crosses into shared memory (cp.async) while the current one is worked on.
// Every sum runs in a fixed order, so the gradients are deterministic given the slots.  The pose sums
// leave per-block partials, which a last kernel adds in a fixed order.  (The two forms' orders differ, and with
// map gradients the order depends on the number of views as well as on the map's size.)
//
// Both are bound by the latency of their loads and by issue (37 % issue active, 16 warps per SM; the chain
// rule is about 550 instructions a batch).  With 4 faces a warp, each lane gathering its entry's vertices,
// view and slot itself, and a separate two-pass form below 8 views, the map form took 484 us of 12 views of 320 x
// 240 of 1M faces (now 267), 163 of 20 views of 300k (127), 117 of 6 (59), 16.9 of 3 views of 30k (8.7); the pose
// alone, 64 tracking views of 150k faces, 151 (138).  Two buffers of staged vertices cost the fourth resident block
// and a second wave: 263 us on the 20-view room.

#include <algorithm>

#include "ts_internal.cuh"

namespace {

struct PBArgs {
  const TsView* views;
  const ts_pose* poses;
  int V;
  long long M;
  const uint32_t* count;
  float* grad;
  const float4* aux;  // per (view, face) normal and sigma_F (TS_FLAG_NORMALS / TS_FLAG_FACE_SIGMA)
  bool normals;
  float* dst_sigma;  // dL/dsigma_F per face (TS_FLAG_FACE_SIGMA), may be null
  const TsDevHeader* hdr;
  float* dst[7];  // gpx, gpy, gpz, gcr, gcg, gcb, gop
  bool min_opacity;  // o_F = min of the vertex opacities: dL/do_F to the first minimal vertex
  float* part;       // per (view, block): the pose sums
  int part_stride;   // blocks the workspace has room for
  uint32_t* part_n;  // receives the blocks used
  int unit;          // without map gradients: consecutive faces per warp (a multiple of 32)
};

__device__ __forceinline__ long long face_vertex(const TsDevHeader* h, long long m, int k) {
  long long j = h->faces ? (long long)h->faces[3 * m + k] : 3 * m + k;
  return (j >= 0 && j < h->n_vertices) ? j : 0;
}

// A slot's sums in registers: G as numbered by G_E .. G_O, dL/dn_F and dL/dsigma_F.
struct SlotSums {
  float G[22], n[3], sig;
};
// A lane's slot copy in shared memory: its eight 16-byte groups in an order of the lane's own, so that the
// lanes of a quarter warp read distinct banks.
__device__ __forceinline__ int group_place(int i) { return (i ^ (threadIdx.x & 7)) * 4; }

// This lane copies a slot into its place `dst`; wait_slot waits for the lane's own copies only.
__device__ __forceinline__ void fetch_slot(const PBArgs& a, float* dst, long long slot) {
  const float* src = a.grad + slot * TS_GRAD_WORDS;
#pragma unroll
  for (int i = 0; i < 8; ++i) ts_cp_async16(dst + group_place(i), src + 4 * i);
  ts_cp_async_commit();
}
__device__ __forceinline__ void wait_slot(const float* src, SlotSums& s) {
  ts_cp_async_wait_all();
#pragma unroll
  for (int i = 0; i < 7; ++i) {
    const float4 q = *reinterpret_cast<const float4*>(src + group_place(i));
    s.G[3 * i] = q.x; s.G[3 * i + 1] = q.y; s.G[3 * i + 2] = q.z;
    if (i < 3) s.n[i] = q.w;
    if (i == 3) s.sig = q.w;
  }
  s.G[G_O] = src[group_place(7)];
}

// 4-byte asynchronous copy of one value.
__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(ts_smem_u32(dst)), "l"(src) : "memory");
}
// Copy vertex j as vertex k of a staged face (positions at d + 3k, colours at d + 9 + 3k); the copies
// join the group committed next.
__device__ __forceinline__ void fetch_vertex(const TsDevHeader* h, float* d, int k, long long j) {
  d += 3 * k;
  cp_async4(d, h->px + j);
  cp_async4(d + 1, h->py + j);
  cp_async4(d + 2, h->pz + j);
  cp_async4(d + 9, h->cr + j);
  cp_async4(d + 10, h->cg + j);
  cp_async4(d + 11, h->cb + j);
}

// A view's intrinsics and pose as 16 floats: fx, fy, cx, cy, R, t.  VP is odd, so that lanes with
// different views read distinct banks.
constexpr int VP = 17;
__device__ __forceinline__ void stage_view(const PBArgs& a, float* d, int v) {
  d[0] = a.views[v].fx;
  d[1] = a.views[v].fy;
  d[2] = a.views[v].cx;
  d[3] = a.views[v].cy;
#pragma unroll
  for (int i = 0; i < 9; ++i) d[4 + i] = a.poses[v].R[i];
#pragma unroll
  for (int i = 0; i < 3; ++i) d[13 + i] = a.poses[v].t[i];
}

// The same values from global memory, four 16-byte loads.
__device__ __forceinline__ void load_view(const PBArgs& a, float* d, int v) {
  static_assert(sizeof(TsView) % 16 == 0 && sizeof(ts_pose) == 48, "16-byte loads of a view and its pose");
  const float4 k = *reinterpret_cast<const float4*>(a.views + v);
  d[0] = k.x; d[1] = k.y; d[2] = k.z; d[3] = k.w;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const float4 q = reinterpret_cast<const float4*>(a.poses + v)[i];
    d[4 + 4 * i] = q.x; d[5 + 4 * i] = q.y; d[6 + 4 * i] = q.z; d[7 + 4 * i] = q.w;
  }
}

// What the chain rule of one visible (view, face) gives: the world-space vertex-position
// gradients, the pose terms, and the slot's colour, opacity and sigma_F sums passed through.
struct SlotTerms {
  float out[9];  // dL/dp of vertex k, coordinate c at 3k + c
  float tau[6];  // [g_C ; v_C x g_C] summed over the vertices
  float gc[9];   // dL/dc of vertex k, channel ch at 3 ch + k (the raster sums)
  float go;      // dL/do_F
  float gsig;    // dL/dsigma_F (TS_FLAG_FACE_SIGMA)
};

// The chain rule of one visible (view, face) from its slot's sums; X holds the face's world positions
// (vertex k, coordinate c at 3k + c) and then its vertex colours, vp its view (stage_view).
__device__ __forceinline__ void chain_terms(const PBArgs& a, int v, long long m, const SlotSums& sl, const float* X,
                                            const float* vp, SlotTerms& t) {
  const float(&G)[22] = sl.G;
  TsView vw;
  vw.fx = vp[0];
  vw.fy = vp[1];
  vw.cx = vp[2];
  vw.cy = vp[3];
  ts_pose P;
#pragma unroll
  for (int i = 0; i < 9; ++i) P.R[i] = vp[4 + i];
#pragma unroll
  for (int i = 0; i < 3; ++i) P.t[i] = vp[13 + i];
  // The projection, edge vectors, lengths and area are recomputed in the forward record's fixed
  // operation order, so the chain rule sees bit-identical values; for slivers the area is a
  // cancelling difference and a one-ulp change of a vertex would move the gradient visibly.
  float xc[3], yc[3], zc[3], u[3], w[3], col[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    ts_rigid_f32(P, X[3 * k], X[3 * k + 1], X[3 * k + 2], xc[k], yc[k], zc[k]);
    ts_pinhole_f32(vw, xc[k], yc[k], zc[k], u[k], w[k]);
    col[k][0] = X[9 + 3 * k]; col[k][1] = X[10 + 3 * k]; col[k][2] = X[11 + 3 * k];
  }
  float ex[3], ey[3], len[3], il[3];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int j = (i + 1) % 3;
    ex[i] = u[j] - u[i];
    ey[i] = w[j] - w[i];
    len[i] = __fsqrt_rn(__fadd_rn(__fmul_rn(ex[i], ex[i]), __fmul_rn(ey[i], ey[i])));
    il[i] = 1.0f / len[i];
  }
  const float per = __fadd_rn(__fadd_rn(len[0], len[1]), len[2]);
  const float D2 = __fsub_rn(__fmul_rn(__fsub_rn(u[1], u[0]), __fsub_rn(w[2], w[0])),
                             __fmul_rn(__fsub_rn(u[2], u[0]), __fsub_rn(w[1], w[0])));
  const float invD = 1.0f / D2;
  float A[3], B[3];  // gradient of the barycentric lambda_k
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int k1 = (k + 1) % 3, k2 = (k + 2) % 3;
    A[k] = (w[k1] - w[k2]) * invD;
    B[k] = (u[k2] - u[k1]) * invD;
  }
  float fa[3], fb[3];  // colour-field gradients
#pragma unroll
  for (int ch = 0; ch < 3; ++ch) {
    fa[ch] = col[0][ch] * A[0] + col[1][ch] * A[1] + col[2][ch] * A[2];
    fb[ch] = col[0][ch] * B[0] + col[1][ch] * B[1] + col[2][ch] * B[2];
  }
  const float za = zc[0] * A[0] + zc[1] * A[1] + zc[2] * A[2];
  const float zb = zc[0] * B[0] + zc[1] * B[1] + zc[2] * B[2];
  float gu[3], gv[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    float su = G[G_Z + k] * za, sv = G[G_Z + k] * zb;
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      su += G[G_C + 3 * ch + k] * fa[ch];
      sv += G[G_C + 3 * ch + k] * fb[ch];
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
      const int o = (i + 2) % 3;
      const float si = per * il[i];
      su += G[G_E + 3 * i + k] * si * A[o];
      sv += G[G_E + 3 * i + k] * si * B[o];
    }
    gu[k] = -su;
    gv[k] = -sv;
  }
  // edge lengths through s_i = per / len_i: dL/dlen_j = sum_i dL/ds_i / len_i - dL/ds_j per / len_j^2
  float ds[3], sum_ds_len = 0.f;
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    ds[i] = G[G_E + 3 * i + (i + 2) % 3];
    sum_ds_len += ds[i] * il[i];
  }
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const float dlen = sum_ds_len - ds[j] * per * il[j] * il[j];
    const float cx = dlen * ex[j] * il[j], cy = dlen * ey[j] * il[j];
    const int j1 = (j + 1) % 3;
    gu[j1] += cx; gv[j1] += cy;
    gu[j] -= cx; gv[j] -= cy;
  }
  // normal map (Eq. 12): dL/dn_F through n = s u / |u|, u = e1 x e2 with
  // e1 = v1 - v0, e2 = v2 - v0 in camera space and s = +-1 the camera-facing turn of the forward:
  // dL/du = s (g - n (n . g)) / |u|, dL/de1 = e2 x dL/du, dL/de2 = dL/du x e1
  float ng[3][3] = {{0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}, {0.f, 0.f, 0.f}};
  if (a.normals) {
    const float gn[3] = {sl.n[0], sl.n[1], sl.n[2]};
    if (gn[0] != 0.f || gn[1] != 0.f || gn[2] != 0.f) {
      const float4 nn = a.aux[(long long)v * a.M + m];
      const float e1[3] = {xc[1] - xc[0], yc[1] - yc[0], zc[1] - zc[0]};
      const float e2[3] = {xc[2] - xc[0], yc[2] - yc[0], zc[2] - zc[0]};
      const float uu[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
      const float il2 = rsqrtf(uu[0] * uu[0] + uu[1] * uu[1] + uu[2] * uu[2]);
      const float sg = (nn.x * uu[0] + nn.y * uu[1] + nn.z * uu[2]) < 0.f ? -1.f : 1.f;
      const float n[3] = {sg * uu[0] * il2, sg * uu[1] * il2, sg * uu[2] * il2};
      const float ndg = n[0] * gn[0] + n[1] * gn[1] + n[2] * gn[2];
      float du[3];
#pragma unroll
      for (int r = 0; r < 3; ++r) du[r] = sg * il2 * (gn[r] - n[r] * ndg);
      const float d1[3] = {e2[1] * du[2] - e2[2] * du[1], e2[2] * du[0] - e2[0] * du[2], e2[0] * du[1] - e2[1] * du[0]};
      const float d2[3] = {du[1] * e1[2] - du[2] * e1[1], du[2] * e1[0] - du[0] * e1[2], du[0] * e1[1] - du[1] * e1[0]};
#pragma unroll
      for (int r = 0; r < 3; ++r) {
        ng[1][r] = d1[r];
        ng[2][r] = d2[r];
        ng[0][r] = -(d1[r] + d2[r]);
      }
    }
  }
  float* out = t.out;
  float* tau = t.tau;
#pragma unroll
  for (int i = 0; i < 6; ++i) tau[i] = 0.f;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float iz = 1.0f / zc[k];
    const float gxp = gu[k] * vw.fx * iz;
    const float gyp = gv[k] * vw.fy * iz;
    const float gz = -(gxp * xc[k] + gyp * yc[k]) * iz + G[G_Z + k] + ng[k][2];  // pinhole + depth + normal
    const float gx = gxp + ng[k][0], gy = gyp + ng[k][1];
    out[3 * k + 0] = P.R[0] * gx + P.R[3] * gy + P.R[6] * gz;  // R^T g_C
    out[3 * k + 1] = P.R[1] * gx + P.R[4] * gy + P.R[7] * gz;
    out[3 * k + 2] = P.R[2] * gx + P.R[5] * gy + P.R[8] * gz;
    tau[0] += gx; tau[1] += gy; tau[2] += gz;
    tau[3] += yc[k] * gz - zc[k] * gy;
    tau[4] += zc[k] * gx - xc[k] * gz;
    tau[5] += xc[k] * gy - yc[k] * gx;
  }
#pragma unroll
  for (int i = 0; i < 9; ++i) t.gc[i] = G[G_C + i];
  t.go = G[G_O];
  t.gsig = sl.sig;
}

constexpr int PB_WARPS = 4;
constexpr int PB_T = 32 * PB_WARPS;
constexpr int PB_RS = 21;   // floats per entry row (positions 9, colours 9, opacity, sigma; odd: no bank conflicts)
constexpr int PB_FS = 19;   // floats per staged face (positions 9, colours 9)
constexpr int PB_PS = 6;    // floats per view's pose sums
// Faces of a batch up to which lane w sums word w over each face's rows.  3 / 5 / 8: 342 / 329 / 329 us for 64 views of
// 300k faces (354 without), 59 / 59 / 60 for 6 views, where a batch holds more.
constexpr int PB_FEW = 5;

// Shared floats of one warp (a multiple of 4): slot copies, entry rows, staged faces, per-face sums,
// per-view pose sums, entry list.
__host__ __device__ constexpr int pbwd_warp_floats(int V, int faces) {
  return (32 * TS_GRAD_WORDS + 32 * PB_RS + faces * (PB_FS + PB_RS) + V * PB_PS + (faces * V + 1) / 2 + 3) & ~3;
}

// With map gradients: FPW faces per warp iteration, 32 / FPW lanes looking up each face's views.  STAGED: the views'
// constants in shared memory, else each entry loads its view's.
template <int FPW, bool STAGED>
__global__ void __launch_bounds__(PB_T, 4) k_pbwd_map(PBArgs a) {
  constexpr int LPF = 32 / FPW, ROUNDS = (3 * FPW + 31) / 32;
  extern __shared__ __align__(16) float pv[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const TsDevHeader* h = a.hdr;
  const int per_warp = pbwd_warp_floats(a.V, FPW);
  float* views = pv + (size_t)PB_WARPS * per_warp;  // [V][VP]
  float* slots = pv + (size_t)warp * per_warp;
  float* rows = slots + 32 * TS_GRAD_WORDS;
  float* fdat = rows + 32 * PB_RS;
  float* fsum = fdat + FPW * PB_FS;
  float* my = fsum + FPW * PB_RS;
  uint16_t* list = reinterpret_cast<uint16_t*>(my + a.V * PB_PS);  // face * 256 + view
  float* slot_here = slots + lane * TS_GRAD_WORDS;
  if (STAGED)
    for (int v = threadIdx.x; v < a.V; v += PB_T) stage_view(a, views + v * VP, v);
  for (int i = lane; i < a.V * PB_PS; i += 32) my[i] = 0.f;
  __syncthreads();
  const bool indexed = h->faces != nullptr;
  const int f = lane / LPF;
  const long long stride = (long long)gridDim.x * PB_WARPS * FPW;
  for (long long m0 = ((long long)blockIdx.x * PB_WARPS + warp) * FPW; m0 < a.M; m0 += stride) {
#pragma unroll
    for (int i0 = 0; i0 < 3 * FPW; i0 += 32) {
      const int i = i0 + lane, fi = i / 3, k = i - 3 * fi;
      if (i < 3 * FPW && m0 + fi < a.M) fetch_vertex(h, fdat + fi * PB_FS, k, face_vertex(h, m0 + fi, k));
    }
    ts_cp_async_commit();
    for (int i = lane; i < FPW * PB_RS; i += 32) fsum[i] = 0.f;
    // this lane looks up views [va, vb) of face f: at most 64, a bit each (the launch sees to it)
    const int Q = (a.V + LPF - 1) / LPF;
    const int va = min((lane % LPF) * Q, a.V), vb = min(va + Q, a.V);
    unsigned long long bits = 0ull;
    {
      const uint32_t* cp = a.count + (long long)va * a.M + m0 + f;
      const int nv = m0 + f < a.M ? vb - va : 0;
#pragma unroll 8
      for (int i = 0; i < nv; ++i) bits |= (unsigned long long)(cp[(long long)i * a.M] != 0u) << i;
    }
    const int mine = __popcll(bits);
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    const unsigned seen = __ballot_sync(0xffffffffu, mine > 0);
    for (int k = incl - mine; bits; bits &= bits - 1) list[k++] = (uint16_t)(f * 256 + va + __ffsll(bits) - 1);
    // where this lane's vertices' faces have their entries: one round of lanes per 32 (face, vertex)s
    int e0[ROUNDS], e1[ROUNDS];
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
      const int fi = min((r * 32 + lane) / 3, FPW - 1);
      e1[r] = __shfl_sync(0xffffffffu, incl, fi * LPF + LPF - 1);
      e0[r] = __shfl_sync(0xffffffffu, incl - mine, fi * LPF);
      if (r * 32 + lane >= 3 * FPW) e1[r] = e0[r];
    }
    ts_cp_async_wait_all();  // this lane's share of the faces
    __syncwarp();
    int next = lane < total ? list[lane] : -1;
    if (next >= 0) fetch_slot(a, slot_here, (m0 + (next >> 8)) * a.V + (next & 255));
    for (int b0 = 0; b0 < total; b0 += 32) {
      const int ne = min(total - b0, 32);
      const bool act = lane < ne;
      const int code = act ? next : 0;
      const int fe = code >> 8, v = code & 255;
      SlotSums sl;
      if (act) wait_slot(slot_here, sl);
      next = b0 + 32 + lane < total ? list[b0 + 32 + lane] : -1;
      if (next >= 0) fetch_slot(a, slot_here, (m0 + (next >> 8)) * a.V + (next & 255));
      float tau[6];
      if (act) {
        SlotTerms t;
        if constexpr (STAGED) {
          chain_terms(a, v, m0 + fe, sl, fdat + fe * PB_FS, views + v * VP, t);
        } else {
          float vp[16];
          load_view(a, vp, v);
          chain_terms(a, v, m0 + fe, sl, fdat + fe * PB_FS, vp, t);
        }
        float* row = rows + lane * PB_RS;
#pragma unroll
        for (int i = 0; i < 9; ++i) row[i] = t.out[i];
#pragma unroll
        for (int i = 0; i < 9; ++i) row[9 + i] = t.gc[i];
        row[18] = t.go;
        row[19] = t.gsig;
#pragma unroll
        for (int i = 0; i < 6; ++i) tau[i] = t.tau[i];
      }
      // pose terms: the entries of one view, in face order, one after another
      const unsigned same = __match_any_sync(0xffffffffu, act ? v : 256 + lane);
      const int rank = __popc(same & ((1u << lane) - 1u));
      const int rounds = (int)__reduce_max_sync(0xffffffffu, (unsigned)rank) + 1;
      for (int r = 0; r < rounds; ++r) {
        if (act && rank == r) {
#pragma unroll
          for (int i = 0; i < 6; ++i) my[v * PB_PS + i] += tau[i];
        }
        __syncwarp();
      }
      // map words, views in order: where the batch holds many faces, the lane of each (face, vertex) sums its
      // words over the face's rows; where it holds few (faces seen by many views), lane w sums word w over
      // each face's rows, so that no lane walks all eight words of 32 rows.  The same sums either way.
      const int fprev = __shfl_up_sync(0xffffffffu, fe, 1);
      const unsigned firsts = __ballot_sync(0xffffffffu, act && (lane == 0 || fe != fprev));
      if (__popc(firsts) <= PB_FEW) {
        for (unsigned rem = firsts; rem; rem &= rem - 1) {
          const int lo = __ffs(rem) - 1, hi = rem & (rem - 1) ? __ffs(rem & (rem - 1)) - 1 : ne;
          const int face = __shfl_sync(0xffffffffu, fe, lo);
          if (lane < PB_RS - 1) {
            float sum = fsum[face * PB_RS + lane];
#pragma unroll 4
            for (int e = lo; e < hi; ++e) sum += rows[e * PB_RS + lane];
            fsum[face * PB_RS + lane] = sum;
          }
        }
      } else {
#pragma unroll
        for (int r = 0; r < ROUNDS; ++r) {
          const int lo = max(e0[r] - b0, 0), hi = min(e1[r] - b0, 32);
          if (lo < hi) {
            const int i = r * 32 + lane, k = i % 3;
            float* w = fsum + i / 3 * PB_RS;
            float sum[8];
#pragma unroll
            for (int c = 0; c < 3; ++c) sum[c] = w[3 * k + c];
#pragma unroll
            for (int c = 0; c < 3; ++c) sum[3 + c] = w[9 + 3 * c + k];
            sum[6] = w[18];
            sum[7] = w[19];
            for (int e = lo; e < hi; ++e) {
              const float* row = rows + e * PB_RS;
#pragma unroll
              for (int c = 0; c < 3; ++c) sum[c] += row[3 * k + c];
#pragma unroll
              for (int c = 0; c < 3; ++c) sum[3 + c] += row[9 + 3 * c + k];
              sum[6] += row[18];
              sum[7] += row[19];
            }
#pragma unroll
            for (int c = 0; c < 3; ++c) w[3 * k + c] = sum[c];
#pragma unroll
            for (int c = 0; c < 3; ++c) w[9 + 3 * c + k] = sum[3 + c];
            if (k == 0) {  // (the face's other two lanes drop these sums)
              w[18] = sum[6];
              w[19] = sum[7];
            }
          }
        }
      }
      __syncwarp();  // every lane has read the rows before the next batch writes them
    }
    // into the map gradient; a face seen by no view adds nothing
    for (int i = lane; i < 3 * FPW; i += 32) {
      const int fi = i / 3, k = i - 3 * fi;
      if (((seen >> (fi * LPF)) & ((1u << LPF) - 1u)) == 0u) continue;  // (a face past M has no view)
      const long long m = m0 + fi, j = face_vertex(h, m, k);
      const float* w = fsum + fi * PB_RS;
      float scale = 1.0f / 3.0f;
      if (a.min_opacity) {  // the first vertex, in face order, attaining the minimum
        const float o0 = __ldg(h->op + face_vertex(h, m, 0)), o1 = __ldg(h->op + face_vertex(h, m, 1));
        const float o2 = __ldg(h->op + face_vertex(h, m, 2));
        const int km = (o0 <= o1 && o0 <= o2) ? 0 : (o1 <= o2 ? 1 : 2);
        scale = k == km ? 1.0f : 0.0f;
      }
      float add[7];
#pragma unroll
      for (int c = 0; c < 7; ++c) add[c] = c < 3 ? w[3 * k + c] : (c < 6 ? w[9 + 3 * (c - 3) + k] : w[18] * scale);
      if (indexed) {
#pragma unroll
        for (int c = 0; c < 7; ++c)
          if (a.dst[c]) atomicAdd(a.dst[c] + j, add[c]);
      } else {
        float old[7];
#pragma unroll
        for (int c = 0; c < 7; ++c) old[c] = a.dst[c] ? a.dst[c][j] : 0.f;
#pragma unroll
        for (int c = 0; c < 7; ++c)
          if (a.dst[c]) a.dst[c][j] = old[c] + add[c];
      }
      if (k == 0 && a.dst_sigma) a.dst_sigma[m] += w[19];
    }
    __syncwarp();  // the next faces reuse the sums and the list
  }
  __syncthreads();
  for (int t = threadIdx.x; t < a.V * 6; t += PB_T) {
    const int v = t / 6, i = t - 6 * (t / 6);
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < PB_WARPS; ++w) sum += pv[(size_t)w * per_warp + (my - slots) + v * PB_PS + i];
    a.part[((long long)v * a.part_stride + blockIdx.x) * 6 + i] = sum;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.part_n = gridDim.x;
}

// Without map gradients: blocks (part of the faces, view), a.unit consecutive faces per warp.
__global__ void __launch_bounds__(PB_T, 4) k_pbwd_pose(PBArgs a) {
  extern __shared__ __align__(16) float pv[];  // [PB_T] slot copies, [PB_T] faces
  __shared__ uint32_t q[PB_WARPS][64];         // queued visible faces
  __shared__ float red[PB_WARPS][6], view[VP];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, v = blockIdx.y;
  const TsDevHeader* h = a.hdr;
  const uint32_t* cnt = a.count + (long long)v * a.M;
  float* slot_here = pv + threadIdx.x * TS_GRAD_WORDS;
  float* face_here = pv + PB_T * TS_GRAD_WORDS + threadIdx.x * PB_FS;
  if (threadIdx.x == 0) stage_view(a, view, v);
  __syncthreads();
  float tau[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  long long pend = -1;  // the face whose slot this lane fetched last
  // take up the pending face, after starting the copies of the next one's vertices and slot
  auto take = [&](long long m_next) {
    const long long m = pend;
    SlotSums sl;
    float X[18];
    if (m >= 0) {
      wait_slot(slot_here, sl);
#pragma unroll
      for (int i = 0; i < 18; ++i) X[i] = face_here[i];
    }
    if (m_next >= 0) {
#pragma unroll
      for (int k = 0; k < 3; ++k) fetch_vertex(h, face_here, k, face_vertex(h, m_next, k));
      fetch_slot(a, slot_here, m_next * a.V + v);
    }
    pend = m_next;
    if (m < 0) return;
    SlotTerms t;
    chain_terms(a, v, m, sl, X, view, t);
#pragma unroll
    for (int i = 0; i < 6; ++i) tau[i] += t.tau[i];
  };
  int qn = 0;
  const long long m_begin = ((long long)blockIdx.x * PB_WARPS + warp) * a.unit, m_end = min(m_begin + a.unit, a.M);
  uint32_t next = m_begin + lane < m_end ? cnt[m_begin + lane] : 0u;
  for (long long m0 = m_begin; m0 < m_end; m0 += 32) {
    const uint32_t cur = next;
    const long long mn = m0 + 32 + lane;
    next = mn < m_end ? cnt[mn] : 0u;  // the next 32 faces' counts are on their way
    const unsigned bal = __ballot_sync(0xffffffffu, cur > 0u);
    if (cur > 0u) q[warp][qn + __popc(bal & ((1u << lane) - 1u))] = (uint32_t)(m0 + lane);
    qn += __popc(bal);
    __syncwarp();
    if (qn >= 32) {
      take(q[warp][lane]);
      __syncwarp();
      if (lane < qn - 32) q[warp][lane] = q[warp][lane + 32];
      qn -= 32;
      __syncwarp();
    }
  }
  take(lane < qn ? (long long)q[warp][lane] : -1);
  take(-1);
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 6; ++i) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tau[i] += __shfl_xor_sync(0xffffffffu, tau[i], o);
    if (lane == 0) red[warp][i] = tau[i];
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < PB_WARPS; ++w) sum += red[w][threadIdx.x];
    a.part[((long long)v * a.part_stride + blockIdx.x) * 6 + threadIdx.x] = sum;
  }
  if (blockIdx.x == 0 && v == 0 && threadIdx.x == 0) *a.part_n = gridDim.x;
}

__global__ void __launch_bounds__(256) k_pose_reduce(const float* __restrict__ part, int part_stride,
                                                     const uint32_t* __restrict__ part_n, float* dtau) {
  __shared__ float red[256][6];
  const int v = blockIdx.x;
  const int nblocks = (int)min(*part_n, (uint32_t)part_stride);  // written by the backward
  float s[6] = {0, 0, 0, 0, 0, 0};
  for (int b = threadIdx.x; b < nblocks; b += 256) {
    const float* p = part + ((long long)v * part_stride + b) * 6;
#pragma unroll
    for (int i = 0; i < 6; ++i) s[i] += p[i];
  }
#pragma unroll
  for (int i = 0; i < 6; ++i) red[threadIdx.x][i] = s[i];
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
#pragma unroll
      for (int i = 0; i < 6; ++i) red[threadIdx.x][i] += red[threadIdx.x + o][i];
    }
    __syncthreads();
  }
  if (threadIdx.x < 6) dtau[v * 6 + threadIdx.x] = red[0][threadIdx.x];
}

}  // namespace

// The faces per warp and block fix the partial sums of the pose gradient and so its summation order: without
// map gradients they depend on the map's size alone, so that a tracked view's dtau is the same alone and
// among others, and on every GPU.
constexpr long long MAP_BLOCKS = 4 * TS_SMS;    // the resident blocks
constexpr long long POSE_BLOCKS = 16 * TS_SMS;  // most blocks per view of the form without map gradients
int ts_pose_blocks(long long M) {               // the most either form uses
  return (int)std::max<long long>(1, std::min<long long>((M + 7) / 8, POSE_BLOCKS));
}

namespace {
// Shared memory of a block of the form with map gradients, and whether four such blocks fit on a
// multiprocessor (228 KB, of which each block takes 1 KB more): up to 23 views of 32 faces, 68 of 16, 110 of 8, all of
// 2.  Four faces and fewer leave the views in global memory: a batch then holds many views of few faces.
constexpr bool pbwd_staged(int faces) { return faces > 4; }
constexpr int pbwd_smem(int V, int faces) {
  return (PB_WARPS * pbwd_warp_floats(V, faces) + (pbwd_staged(faces) ? V * VP : 0)) * (int)sizeof(float);
}
constexpr bool pbwd_four_blocks(int V, int faces) { return 4 * (pbwd_smem(V, faces) + 1024) <= 228 * 1024; }
static_assert(pbwd_four_blocks(23, 32) && !pbwd_four_blocks(65, 32) && pbwd_four_blocks(68, 16) &&
                  !pbwd_four_blocks(129, 16) && pbwd_four_blocks(TS_MAX_VIEWS, 2) && TS_MAX_VIEWS <= 256,
              "a lane looks up at most 64 views of its face, an entry holds its view in 8 bits");

template <int FPW>
cudaError_t launch_pbwd_map(const PBArgs& a, cudaStream_t s) {
  const int smem = pbwd_smem(a.V, FPW);  // at most 56 KB
  const cudaError_t e = ts_smem_limit((const void*)k_pbwd_map<FPW, pbwd_staged(FPW)>, smem);
  if (e != cudaSuccess) return e;
  const long long want = (a.M + PB_WARPS * FPW - 1) / (PB_WARPS * FPW);
  k_pbwd_map<FPW, pbwd_staged(FPW)><<<(unsigned)std::min(want, MAP_BLOCKS), PB_T, smem, s>>>(a);
  return cudaGetLastError();
}
}  // namespace

cudaError_t ts_launch_project_bwd(const TsPlanImpl* p, const TsWs& w, const ts_map_grad* g, cudaStream_t s) {
  if (p->M == 0) {
    return cudaMemsetAsync(w.pose_n, 0, 4, s);  // no partials
  }
  PBArgs a;
  a.views = w.views;
  a.poses = w.poses;
  a.V = p->V;
  a.M = p->M;
  a.count = w.count;
  a.grad = w.grad;
  a.aux = w.aux;
  a.normals = p->normals;
  a.dst_sigma = p->face_sigma ? g->gsigma : nullptr;
  a.hdr = w.hdr;
  a.dst[0] = g->gpx; a.dst[1] = g->gpy; a.dst[2] = g->gpz;
  a.dst[3] = g->gcr; a.dst[4] = g->gcg; a.dst[5] = g->gcb;
  a.dst[6] = g->gop;
  a.min_opacity = p->min_opacity;
  a.part = w.pose;
  a.part_stride = (int)p->n_pose_blocks;
  a.part_n = w.pose_n;
  a.unit = 0;
  bool map = a.dst_sigma != nullptr;
  for (int c = 0; c < 7; ++c) map = map || a.dst[c] != nullptr;
  if (!map) {
    // faces per warp: enough that full batches dominate, once every SM has warps.  One view is fastest with few (150k
    // faces: 6.4 us at 128, 8.3 at 256, 12.5 at 512), many views with many (64: 191, 162 and 148); at 128, 256 and 512
    // 7 views of 40k take 9.2, 10.6 and 14.2, 64 views 57, 51 and 53, 7 views of 65k 14.2, 11.7 and 15.1, 64 86, 77 and 74.
    const long long least = (p->M + PB_WARPS * POSE_BLOCKS - 1) / (PB_WARPS * POSE_BLOCKS);
    a.unit = p->M >= (1 << 16) ? (int)std::max<long long>(512, (least + 31) / 32 * 32)
                               : (p->M >= 3 << 14 ? 256 : (p->M >= 1 << 14 ? 128 : 32));
    const long long nb = (p->M + PB_WARPS * a.unit - 1) / (PB_WARPS * a.unit);
    const int smem = PB_T * (TS_GRAD_WORDS + PB_FS) * (int)sizeof(float);  // 26 KB
    k_pbwd_pose<<<dim3((unsigned)nb, (unsigned)p->V), PB_T, smem, s>>>(a);
    return cudaGetLastError();
  }
  // As many faces a warp as leave every warp of the grid some, and four blocks room on a multiprocessor (fewer leave the
  // grid a second wave); above 110 views two, which fill batches then.  300k faces take 141 us at 23 views of 32 faces
  // and 150 of 16, 332 at 64 views of 16 and 346 of 8; 30k faces 101 us at 128 views of 8 faces, 81 of 4 and 83 of 2, 10k
  // at 200 views 99, 68 and 59; 2000 faces of 64 views 25 us of 8, 18 of 4 and 13 of 2, 10k of 16 views 11 of 8 and 13
  // of 4.
  int faces = 32;
  while (faces > 2 && (!pbwd_four_blocks(p->V, std::max(faces, 8)) || p->M <= MAP_BLOCKS * PB_WARPS * (faces / 2)))
    faces /= 2;
  switch (faces) {
    case 32: return launch_pbwd_map<32>(a, s);
    case 16: return launch_pbwd_map<16>(a, s);
    case 8: return launch_pbwd_map<8>(a, s);
    case 4: return launch_pbwd_map<4>(a, s);
    default: return launch_pbwd_map<2>(a, s);
  }
}

cudaError_t ts_launch_pose_reduce(const TsPlanImpl* p, const TsWs& w, float* dtau, cudaStream_t s) {
  k_pose_reduce<<<p->V, 256, 0, s>>>(w.pose, (int)p->n_pose_blocks, w.pose_n, dtau);
  return cudaGetLastError();
}
