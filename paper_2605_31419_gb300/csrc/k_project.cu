// k_project.cu -- Eq. 1-3 per (view, face): projection, culling and the screen-space record.
//
// A warp takes 32 consecutive faces and a block of views: the vertices are loaded once for all of the
// block's views (coalesced), and per view the camera-space vertices decide with a few products whether the
// face can be seen (in front of the camera and, with margins above all rounding, not wholly beyond one side
// of the image).  The faces that can, a quarter of a room's, are queued in shared memory, and full warps of
// them run the exact tests and write the (view, face) outputs: the divisions, square roots and record
// stores run on 32 lanes instead of the quarter to third that a plain loop leaves active.  Bound by the
// stores of visible faces (256 + 16 bytes each; 20 views of 300k faces write 0.64 GB at 4.7 TB/s) and by
// issue (half of the slots): 170 -> 139 us there, 298 -> 237 for the 12-view window of 1M faces, 385 -> 282
// for 9 views of 2M, 213 -> 152 for 64 tracking views.
// The projection, area, perimeter, inradius, face opacity, pixel box and depth key follow one fixed FP32
// operation order (no FMA contraction, IEEE division and square root), so culling, tiles and depth keys are
// reproducible bit for bit; the margin test only leaves out faces that the exact box test culls.
#include <algorithm>

#include "ts_internal.cuh"

namespace {

struct MapArgs {
  const float *px, *py, *pz, *cr, *cg, *cb, *op;
  const int32_t* faces;
  long long n_vertices;
};

__global__ void k_setup(TsViewTable tab, int V, MapArgs map, const ts_pose* __restrict__ poses, TsDevHeader* hdr,
                        TsView* views, ts_pose* ws_poses, unsigned long long* ctr) {
  const int t = threadIdx.x;
  for (int v = t; v < V; v += blockDim.x) {
    views[v] = tab.v[v];
    ws_poses[v] = poses[v];
  }
  for (int i = t; i < TS_N_CTR * TS_CTR_SLOTS; i += blockDim.x) ctr[(size_t)i * TS_CTR_STRIDE] = 0ull;
  if (t == 0) {
    hdr->n_pairs = 0;
    hdr->n_visible = 0;
    hdr->fwd_contrib = 0;
    hdr->bwd_contrib = 0;
    hdr->indexed = map.faces ? 1u : 0u;
    hdr->px = map.px; hdr->py = map.py; hdr->pz = map.pz;
    hdr->cr = map.cr; hdr->cg = map.cg; hdr->cb = map.cb;
    hdr->op = map.op;
    hdr->faces = map.faces;
    hdr->n_vertices = map.n_vertices;
  }
}

// One 32-byte store (eight floats) to a 32-byte aligned global address.
__device__ __forceinline__ void st_v8(float* p, float a0, float a1, float a2, float a3, float a4, float a5, float a6,
                                      float a7) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(a0), "f"(a1), "f"(a2),
               "f"(a3), "f"(a4), "f"(a5), "f"(a6), "f"(a7)
               : "memory");
}

struct ProjArgs {
  MapArgs map;
  const TsView* views;
  const ts_pose* poses;
  long long M;
  int V;
  float z_near, r_min, alpha_min;
  bool min_opacity;
  int tile_w, tile_h;
  float4* frec;
  float4* aux;  // camera-space unit normal (TS_FLAG_NORMALS) and sigma_F in .w (TS_FLAG_FACE_SIGMA)
  bool normals;
  const float* sigma;  // per-face window exponents (TS_FLAG_FACE_SIGMA), else null
  uint32_t* cov;  // per (view, face) forward pixel coverage (TS_FLAG_STATS), else null
  float* grad;
  short4* rect;
  uint32_t* zbits;
  uint32_t* count;
  unsigned long long* ctr;
};

// Views' constants in shared memory: pose (R, t), fx, fy, cx, cy, the four cull offsets, W, H and the
// coordinates above which the margin test is not used (its products could overflow).
constexpr int PJ_T = 128;     // threads per block
constexpr int PJ_VIEWS = 8;   // most views per block
constexpr int PJ_VP = 24;     // words per view
constexpr int PJ_Q = 64;      // queue places per warp: below 32 waiting, up to 32 pushed at a time
constexpr int PJ_STEPS = 32;  // (32 faces, view) steps per warp of a large map
enum { V_T = 9, V_FX = 12, V_FY, V_CX, V_CY, V_LOX, V_HIX, V_LOY, V_HIY, V_W, V_H, V_LIM };

__device__ __forceinline__ void cp_async4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(ts_smem_u32(dst)), "l"(src) : "memory");
}

// One queued (view, face): the record and what the later passes read, or, where an exact test culls it, the
// marks of an invisible face.  c: the camera-space vertices; face m of view `view`, constants vp.
__device__ __forceinline__ bool project_face(const ProjArgs& a, long long m, int view, const float* vp,
                                             const float (&c)[9]) {
  const long long idx = (long long)view * a.M + m;
  long long vi[3];
  if (a.map.faces) {
    vi[0] = a.map.faces[3 * m]; vi[1] = a.map.faces[3 * m + 1]; vi[2] = a.map.faces[3 * m + 2];
  } else {
    vi[0] = 3 * m; vi[1] = 3 * m + 1; vi[2] = 3 * m + 2;
  }
  float o[3], col[3][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const long long j = vi[k];
    o[k] = __ldg(a.map.op + j);
    col[k][0] = __ldg(a.map.cr + j);
    col[k][1] = __ldg(a.map.cg + j);
    col[k][2] = __ldg(a.map.cb + j);
  }
  TsView vw;
  vw.fx = vp[V_FX]; vw.fy = vp[V_FY]; vw.cx = vp[V_CX]; vw.cy = vp[V_CY];
  float u[3], v[3], z[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    z[k] = c[3 * k + 2];
    ts_pinhole_f32(vw, c[3 * k], c[3 * k + 1], z[k], u[k], v[k]);
  }
  bool vis = true;
  float len[3];
  const float du1 = __fsub_rn(u[1], u[0]), dv1 = __fsub_rn(v[1], v[0]);
  const float du2 = __fsub_rn(u[2], u[0]), dv2 = __fsub_rn(v[2], v[0]);
  const float area2 = __fsub_rn(__fmul_rn(du1, dv2), __fmul_rn(du2, dv1));
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int j = (i + 1) % 3;
    const float ex = __fsub_rn(u[j], u[i]), ey = __fsub_rn(v[j], v[i]);
    len[i] = __fsqrt_rn(__fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)));
  }
  const float per = __fadd_rn(__fadd_rn(len[0], len[1]), len[2]);
  const float r = __fdiv_rn(fabsf(area2), per);
  if (!(r >= a.r_min)) vis = false;
  const float oF = a.min_opacity ? fminf(o[0], fminf(o[1], o[2])) : __fdiv_rn(__fadd_rn(__fadd_rn(o[0], o[1]), o[2]), 3.0f);
  if (oF < a.alpha_min) vis = false;
  int x0 = 0, x1 = 0, y0 = 0, y1 = 0;
  {
    const int W = __float_as_int(vp[V_W]), H = __float_as_int(vp[V_H]);
    const float umin = fminf(u[0], fminf(u[1], u[2])), umax = fmaxf(u[0], fmaxf(u[1], u[2]));
    const float vmin = fminf(v[0], fminf(v[1], v[2])), vmax = fmaxf(v[0], fmaxf(v[1], v[2]));
    const float fx0 = ceilf(__fsub_rn(umin, 0.5f)), fx1 = floorf(__fsub_rn(umax, 0.5f));
    const float fy0 = ceilf(__fsub_rn(vmin, 0.5f)), fy1 = floorf(__fsub_rn(vmax, 0.5f));
    const float Wm = (float)(W - 1), Hm = (float)(H - 1);
    if (!(fx0 <= fx1) || fx1 < 0.0f || fx0 > Wm) vis = false;
    if (!(fy0 <= fy1) || fy1 < 0.0f || fy0 > Hm) vis = false;
    if (vis) {
      x0 = fx0 < 0.0f ? 0 : (int)fx0;
      x1 = fx1 > Wm ? W - 1 : (int)fx1;
      y0 = fy0 < 0.0f ? 0 : (int)fy0;
      y1 = fy1 > Hm ? H - 1 : (int)fy1;
    }
  }
  if (!vis) {
    a.rect[idx] = make_short4(-1, -1, -1, -1);
    a.count[idx] = 0u;
    return false;
  }
  const float zk = __fdiv_rn(__fadd_rn(__fadd_rn(z[0], z[1]), z[2]), 3.0f);
  a.zbits[idx] = __float_as_uint(zk);
  // record: edge vectors, normalised edge-function scales s_i / D2, barycentric scale 1 / D2
  const float e0x = u[1] - u[0], e0y = v[1] - v[0];
  const float e1x = u[2] - u[1], e1y = v[2] - v[1];
  const float e2x = u[0] - u[2], e2y = v[0] - v[2];
  const float invD = 1.0f / area2;
  const float k0 = (per / len[0]) * invD, k1 = (per / len[1]) * invD, k2 = (per / len[2]) * invD;
  float* rec = reinterpret_cast<float*>(a.frec + idx * (TS_REC_WORDS / 4));
  st_v8(rec, u[0], u[1], u[2], v[0], v[1], v[2], e0x, e0y);
  st_v8(rec + 8, e1x, e1y, e2x, e2y, k0, k1, k2, invD);
  st_v8(rec + 16, oF, col[0][0], col[0][1], col[0][2], col[1][0], col[1][1], col[1][2], col[2][0]);
  // gradient slot of this (view, face), face-major so that a face's views are adjacent
  const long long slot = m * a.V + view;
  st_v8(rec + 24, col[2][1], col[2][2], z[0], z[1], z[2], __uint_as_float((uint32_t)x0 | ((uint32_t)x1 << 16)),
        __uint_as_float((uint32_t)y0 | ((uint32_t)y1 << 16)), __uint_as_float((uint32_t)slot));
  const int tx0 = x0 / a.tile_w, tx1 = x1 / a.tile_w, ty0 = y0 / a.tile_h, ty1 = y1 / a.tile_h;
  a.rect[idx] = make_short4((short)tx0, (short)ty0, (short)tx1, (short)ty1);
  a.count[idx] = (uint32_t)((tx1 - tx0 + 1) * (ty1 - ty0 + 1));
  if (a.cov) a.cov[idx] = 0u;
  if (a.aux) {
    float4 ax = make_float4(0.f, 0.f, 0.f, a.sigma ? __ldg(a.sigma + m) : 0.f);
    if (a.normals) {
      // unit normal (v1 - v0) x (v2 - v0), turned towards the camera.  The edge vectors are
      // taken in world space, where nearby float32 positions subtract almost exactly, and the
      // unit normal is then rotated by R: camera-space edges would be differences of
      // metre-sized coordinates and lose ~1e-5 of the normal for centimetre faces.
      float e1[3], e2[3];
      const float* const xyz[3] = {a.map.px, a.map.py, a.map.pz};
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float w0 = __ldg(xyz[d] + vi[0]);
        e1[d] = __ldg(xyz[d] + vi[1]) - w0;
        e2[d] = __ldg(xyz[d] + vi[2]) - w0;
      }
      const float wx = e1[1] * e2[2] - e1[2] * e2[1], wy = e1[2] * e2[0] - e1[0] * e2[2];
      const float wz = e1[0] * e2[1] - e1[1] * e2[0];
      const float inv = rsqrtf(wx * wx + wy * wy + wz * wz);
      float nc[3];
#pragma unroll
      for (int d = 0; d < 3; ++d) nc[d] = (vp[3 * d] * wx + vp[3 * d + 1] * wy + vp[3 * d + 2] * wz) * inv;
      const float facing = nc[0] * (c[0] + c[3] + c[6]) + nc[1] * (c[1] + c[4] + c[7]) + nc[2] * (z[0] + z[1] + z[2]);
      const float sg = facing > 0.f ? -1.f : 1.f;
      ax.x = sg * nc[0];
      ax.y = sg * nc[1];
      ax.z = sg * nc[2];
    }
    a.aux[idx] = ax;
  }
  return true;
}

// blockIdx.x: 4 warps' faces, `groups` times 32 consecutive faces per warp; blockIdx.y: block of views.
__global__ void __launch_bounds__(PJ_T, 6) k_project(ProjArgs a, int views_per_block, int groups) {
  __shared__ float vtab[PJ_VIEWS][PJ_VP];
  __shared__ float queue[PJ_T / 32][10][PJ_Q];  // camera-space vertices and (view << 16 | face of the warp)
  __shared__ float pos[PJ_T / 32][2][9][32];    // the faces' vertices, two groups of 32 faces
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int v0 = (int)blockIdx.y * views_per_block;
  const int nv = min(a.V - v0, views_per_block);
  if (threadIdx.x < nv) {
    float* vp = vtab[threadIdx.x];
    const TsView& vw = a.views[v0 + threadIdx.x];
    const ts_pose& P = a.poses[v0 + threadIdx.x];
#pragma unroll
    for (int i = 0; i < 9; ++i) vp[i] = P.R[i];
#pragma unroll
    for (int i = 0; i < 3; ++i) vp[V_T + i] = P.t[i];
    vp[V_FX] = vw.fx;
    vp[V_FY] = vw.fy;
    vp[V_CX] = vw.cx;
    vp[V_CY] = vw.cy;
    // margins of 0.01 px and 2e-6 of the offsets, above the rounding of u, v and of the test itself
    const float W = (float)vw.W, H = (float)vw.H;
    const float mx = 0.01f + 2e-6f * (fabsf(vw.cx) + W), my = 0.01f + 2e-6f * (fabsf(vw.cy) + H);
    vp[V_LOX] = vw.cx - 0.5f + mx;
    vp[V_HIX] = vw.cx - (W - 0.5f) - mx;
    vp[V_LOY] = vw.cy - 0.5f + my;
    vp[V_HIY] = vw.cy - (H - 0.5f) - my;
    vp[V_W] = __int_as_float(vw.W);
    vp[V_H] = __int_as_float(vw.H);
    vp[V_LIM] = a.z_near >= 1e-30f
                    ? 1e37f / fmaxf(fmaxf(fmaxf(vw.fx, vw.fy), 1.f), fmaxf(fabsf(vw.cx) + W, fabsf(vw.cy) + H))
                    : 0.f;
  }
  __syncthreads();
  const long long mw = ((long long)blockIdx.x * (PJ_T / 32) + warp) * groups * 32;  // the warp's first face
  float(*q)[PJ_Q] = queue[warp];
  int head = 0, nq = 0;
  unsigned seen = 0u;
  auto take = [&](int n) {  // the first n queued faces, one per lane
    __syncwarp();
    bool vis = false;
    long long slot = 0;
    if (lane < n) {
      const int i = (head + lane) & (PJ_Q - 1);
      float c[9];
#pragma unroll
      for (int k = 0; k < 9; ++k) c[k] = q[k][i];
      const int code = __float_as_int(q[9][i]);
      const long long m = mw + (code & 0xffff);
      slot = m * a.V + v0 + (code >> 16);
      vis = project_face(a, m, v0 + (code >> 16), vtab[code >> 16], c);
    }
    const unsigned bal = __ballot_sync(0xffffffffu, vis);
    seen += lane == 0 ? __popc(bal) : 0;
    if (a.grad) {  // null for a forward-only plan
      // the visible faces' gradient slots, cleared for the raster backward's atomics: four lanes per slot, so
      // that a store covers 8 lines instead of 32
      static_assert(TS_GRAD_WORDS == 32, "four lanes of eight words");
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int from = i * 8 + (lane >> 2);
        const long long sl = __shfl_sync(0xffffffffu, slot, from);
        if ((bal >> from) & 1u)
          st_v8(a.grad + sl * TS_GRAD_WORDS + (lane & 3) * 8, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f);
      }
    }
    head = (head + n) & (PJ_Q - 1);
    nq -= n;
    __syncwarp();  // every lane has read its places before the next faces are pushed into them
  };
  // this lane's copies of the vertices of face m into places b; not a face of the map, or an index outside it:
  // not a number, which every view culls
  auto load = [&](long long m, int b) {
    bool ok = m < a.M;
    long long vi[3] = {3 * m, 3 * m + 1, 3 * m + 2};
    if (ok && a.map.faces) {
#pragma unroll
      for (int k = 0; k < 3; ++k) vi[k] = a.map.faces[3 * m + k];
    }
#pragma unroll
    for (int k = 0; k < 3; ++k)
      if (vi[k] < 0 || vi[k] >= a.map.n_vertices) ok = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      if (ok) {
        cp_async4(&pos[warp][b][3 * k][lane], a.map.px + vi[k]);
        cp_async4(&pos[warp][b][3 * k + 1][lane], a.map.py + vi[k]);
        cp_async4(&pos[warp][b][3 * k + 2][lane], a.map.pz + vi[k]);
      } else {
        pos[warp][b][3 * k][lane] = pos[warp][b][3 * k + 1][lane] = pos[warp][b][3 * k + 2][lane] =
            __int_as_float(0x7fffffff);
      }
    }
    ts_cp_async_commit();
  };
  load(mw + lane, 0);
  for (int g = 0; g < groups && mw + g * 32 < a.M; ++g) {
    const long long m = mw + g * 32 + lane;
    ts_cp_async_wait_all();
    if (g + 1 < groups) load(m + 32, (g + 1) & 1);  // while this group's faces are projected
    const float(*wp)[32] = pos[warp][g & 1];
    for (int v = 0; v < nv; ++v) {
      const float* vp = vtab[v];
      ts_pose P;
#pragma unroll
      for (int i = 0; i < 9; ++i) P.R[i] = vp[i];
#pragma unroll
      for (int i = 0; i < 3; ++i) P.t[i] = vp[V_T + i];
      float c[9];
      bool in = true, left = true, right = true, above = true, below = true;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        ts_rigid_f32(P, wp[3 * k][lane], wp[3 * k + 1][lane], wp[3 * k + 2][lane], c[3 * k], c[3 * k + 1], c[3 * k + 2]);
        const float z = c[3 * k + 2];
        const float fx = vp[V_FX] * c[3 * k], fy = vp[V_FY] * c[3 * k + 1];
        in = in && z > a.z_near;
        left = left && fmaf(vp[V_LOX], z, fx) < 0.f;
        right = right && fmaf(vp[V_HIX], z, fx) > 0.f;
        above = above && fmaf(vp[V_LOY], z, fy) < 0.f;
        below = below && fmaf(vp[V_HIY], z, fy) > 0.f;
      }
      const float big = fmaxf(fmaxf(fmaxf(fabsf(c[0]), fabsf(c[1])), fmaxf(fabsf(c[3]), fabsf(c[4]))),
                              fmaxf(fmaxf(fabsf(c[6]), fabsf(c[7])), fmaxf(c[2], fmaxf(c[5], c[8]))));
      in = in && !((left || right || above || below) && big < vp[V_LIM]);
      if (!in && m < a.M) {
        const long long idx = (long long)(v0 + v) * a.M + m;
        a.rect[idx] = make_short4(-1, -1, -1, -1);
        a.count[idx] = 0u;
      }
      const unsigned bal = __ballot_sync(0xffffffffu, in);
      if (in) {
        const int i = (head + nq + __popc(bal & ((1u << lane) - 1u))) & (PJ_Q - 1);
#pragma unroll
        for (int k = 0; k < 9; ++k) q[k][i] = c[k];
        q[9][i] = __int_as_float((v << 16) | (g * 32 + lane));
      }
      nq += __popc(bal);
      const bool last = v + 1 == nv && (g + 1 == groups || mw + (g + 1) * 32 >= a.M);
      while (nq >= 32 || (last && nq > 0)) take(min(nq, 32));
    }
  }
  ts_count_add(a.ctr, TS_CTR_VISIBLE, seen);
}

}  // namespace

cudaError_t ts_launch_setup(const TsPlanImpl* p, const TsWs& w, const ts_map* map, const ts_pose* poses,
                            cudaStream_t s) {
  TsViewTable local;  // passed by value: capture-safe, no host-to-device copy
  for (int v = 0; v < p->V; ++v) local.v[v] = p->views[v];
  MapArgs m{map->px, map->py, map->pz, map->cr, map->cg, map->cb, map->op, map->faces, map->n_vertices};
  k_setup<<<1, 256, 0, s>>>(local, p->V, m, poses, w.hdr, w.views, w.poses, w.ctr);
  return cudaGetLastError();
}

cudaError_t ts_launch_project(const TsPlanImpl* p, const TsWs& w, const ts_map* map, cudaStream_t s) {
  const long long VM = (long long)p->V * p->M;
  if (VM == 0) return cudaSuccess;
  ProjArgs a;
  a.map = MapArgs{map->px, map->py, map->pz, map->cr, map->cg, map->cb, map->op, map->faces, map->n_vertices};
  a.views = w.views;
  a.poses = w.poses;
  a.M = p->M;
  a.z_near = p->prm.z_near;
  a.r_min = p->prm.r_min;
  a.alpha_min = p->prm.alpha_min;
  a.min_opacity = p->min_opacity;
  a.tile_w = p->prm.tile_w;
  a.tile_h = p->prm.tile_h;
  a.V = p->V;
  a.grad = w.grad;
  a.frec = w.frec;
  a.aux = w.aux;
  a.normals = p->normals;
  a.sigma = p->face_sigma ? map->sigma : nullptr;
  a.cov = w.cov;
  a.rect = w.rect;
  a.zbits = w.zbits;
  a.count = w.count;
  a.ctr = w.ctr;
  // views per block: up to PJ_VIEWS, so that a map is read once per block of views and full warps of faces collect, but
  // fewer where that leaves over half of the GPU's places (six blocks per multiprocessor) empty: 8 against 4 measured
  // 147 against 161 us at 20 views of 300k faces, 280 against 294 at 9 of 2M, 10.9 against 9.3 at 7 of 40k (one partly
  // filled wave there beats a full one and a bit: 784 blocks 7.7 us, 1568 9.9).  Steps per warp: up to PJ_STEPS once
  // every place has eight blocks to run.  One view leaves a step a quarter of a warp of faces to project, and takes up
  // to three of them as soon as the places are full: 1, 2, 3 and 4 steps 12.0, 10.2, 9.5 and 9.3 us for 300k faces, 38,
  // 29, 26 and 26 for 1M, 73, 53, 49 and 48 for 2M.
  const long long places = 6LL * ts_sm_count(), fg = (p->M + 31) / 32;
  int per = std::min(p->V, PJ_VIEWS);
  auto blocks_of = [&](int n) { return (fg + PJ_T / 32 - 1) / (PJ_T / 32) * ((p->V + n - 1) / n); };
  while (per > 1 && 2 * blocks_of(per) < places) per = (per + 1) / 2;
  const long long vb = (p->V + per - 1) / per;
  const long long steps = p->V == 1 ? std::min(3LL, (blocks_of(1) + places - 1) / places)
                                    : std::min<long long>(PJ_STEPS / per, blocks_of(per) / (8 * places));
  const int groups = (int)std::max(1LL, steps);
  const long long face_blocks = (fg + (long long)groups * (PJ_T / 32) - 1) / ((long long)groups * (PJ_T / 32));
  k_project<<<dim3((unsigned)face_blocks, (unsigned)vb), PJ_T, 0, s>>>(a, per, groups);
  return cudaGetLastError();
}

// The counters' slots summed into the header (read by ts_sync_status).
__global__ void __launch_bounds__(256) k_sum_counters(const unsigned long long* __restrict__ ctr, TsDevHeader* hdr) {
  __shared__ unsigned long long red[TS_N_CTR][256];
  for (int c = 0; c < TS_N_CTR; ++c) {
    unsigned long long s = 0;
    for (int i = threadIdx.x; i < TS_CTR_SLOTS; i += 256) s += ctr[((size_t)c * TS_CTR_SLOTS + i) * TS_CTR_STRIDE];
    red[c][threadIdx.x] = s;
  }
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o)
      for (int c = 0; c < TS_N_CTR; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    hdr->n_visible = red[TS_CTR_VISIBLE][0];
    hdr->fwd_contrib = red[TS_CTR_FWD][0];
    hdr->bwd_contrib = red[TS_CTR_BWD][0];
  }
}

cudaError_t ts_launch_sum_counters(const TsWs& w, cudaStream_t s) {
  k_sum_counters<<<1, 256, 0, s>>>(w.ctr, w.hdr);
  return cudaGetLastError();
}
