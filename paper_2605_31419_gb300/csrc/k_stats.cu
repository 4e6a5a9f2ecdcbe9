// k_stats.cu -- the map statistics that Sec. 3.4's map management reads from a render:
//   * pixel coverage per (view, face), counted by the forward blend (TS_FLAG_STATS): the number of
//     pixels at which the face was blended; densification splits faces whose coverage exceeds
//     theta_blur * H * W;
//   * projected area per (view, face): |D2| / 2 of the projected triangle, recomputed from the
//     record's vertices in the projection's fixed FP32 operation order (bit-identical to the
//     value culling saw); pruning removes faces above epsilon_a pixels;
//   * per-view visible-face bitsets and counts, and the co-visibility IoU between views that
//     keyframe selection compares.
#include "ts_internal.cuh"

static_assert(R_U0 == 0 && R_V0 == 3 && R_V1 == 4 && R_V2 == 5, "a record's first six words are its vertices");

namespace {

constexpr int ST_T = 256;

struct StatsArgs {
  const float4* frec;
  const uint32_t* count;
  const uint32_t* cov_in;
  long long M;
  int words;  // ceil(M / 32)
  uint32_t* coverage;
  float* area;
  uint32_t* visible;
  uint32_t* n_visible;
};

// grid (ceil(M / (256 ST_PER)), V): 256 ST_PER faces of view v per block, 256 at a time; a warp covers 32 faces of one view,
// so its ballot is one word of the view's bitset.  Bound by its 12 to 20 bytes per (view, face) and the
// visible records' sectors.  The visible counts are summed per block: one add per warp queued 9,375 adds on
// each view's address (8 views of 300k faces: 58 -> 23 us).  Maps that leave most multiprocessors without a block
// take a face per thread (ST_PER 1).
template <int ST_PER>
__global__ void __launch_bounds__(ST_T) k_face_stats(StatsArgs a) {
  __shared__ unsigned red[ST_T / 32];
  const int v = blockIdx.y;
  unsigned seen = 0u;
  const long long m0 = (long long)blockIdx.x * ST_PER * ST_T + threadIdx.x;
  const long long base = (long long)v * a.M;
  // all counts, then all coverages, then all records: the loads of one kind are in flight together
  bool proj[ST_PER];
  uint32_t cov[ST_PER];
#pragma unroll
  for (int k = 0; k < ST_PER; ++k) {
    const long long m = m0 + k * ST_T;
    proj[k] = m < a.M && a.count[base + m] > 0;
  }
#pragma unroll
  for (int k = 0; k < ST_PER; ++k) cov[k] = (proj[k] && a.cov_in) ? a.cov_in[base + m0 + k * ST_T] : 0u;
  if (a.area) {
    float4 q[ST_PER];  // u0, u1, u2, v0
    float2 p[ST_PER];  // v1, v2
#pragma unroll
    for (int k = 0; k < ST_PER; ++k) {
      const float4* r = a.frec + (base + m0 + k * ST_T) * (TS_REC_WORDS / 4);
      q[k] = proj[k] ? r[0] : make_float4(0.f, 0.f, 0.f, 0.f);
      p[k] = proj[k] ? *reinterpret_cast<const float2*>(r + 1) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int k = 0; k < ST_PER; ++k) {
      const float du1 = __fsub_rn(q[k].y, q[k].x), dv1 = __fsub_rn(p[k].x, q[k].w);
      const float du2 = __fsub_rn(q[k].z, q[k].x), dv2 = __fsub_rn(p[k].y, q[k].w);
      if (m0 + k * ST_T < a.M)
        a.area[base + m0 + k * ST_T] = 0.5f * fabsf(__fsub_rn(__fmul_rn(du1, dv2), __fmul_rn(du2, dv1)));
    }
  }
#pragma unroll
  for (int k = 0; k < ST_PER; ++k) {
    const long long m = m0 + k * ST_T;
    if (a.coverage && m < a.M) a.coverage[base + m] = cov[k];
    const unsigned bal = __ballot_sync(0xffffffffu, cov[k] > 0);
    seen += __popc(bal);
    if (a.visible && (threadIdx.x & 31) == 0 && m < a.M) a.visible[(long long)v * a.words + (m >> 5)] = bal;
  }
  if (!a.n_visible) return;
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = seen;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned s = 0u;
#pragma unroll
    for (int w = 0; w < ST_T / 32; ++w) s += red[w];
    if (s) atomicAdd(a.n_visible + v, s);
  }
}

// iou[i][j] = |S_i & S_j| / |S_i | S_j| over the views' bitsets (0 when both sets are empty)
__global__ void __launch_bounds__(ST_T) k_covis(const uint32_t* __restrict__ bits, int words, int V,
                                                float* __restrict__ iou) {
  __shared__ unsigned long long red[2][ST_T / 32];
  const int i = blockIdx.y, j = blockIdx.x;
  const uint32_t* a = bits + (long long)i * words;
  const uint32_t* b = bits + (long long)j * words;
  unsigned long long in = 0, un = 0;
  for (int k = threadIdx.x; k < words; k += ST_T) {
    const uint32_t x = a[k], y = b[k];
    in += __popc(x & y);
    un += __popc(x | y);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    in += __shfl_xor_sync(0xffffffffu, in, o);
    un += __shfl_xor_sync(0xffffffffu, un, o);
  }
  if ((threadIdx.x & 31) == 0) {
    red[0][threadIdx.x >> 5] = in;
    red[1][threadIdx.x >> 5] = un;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long si = 0, su = 0;
#pragma unroll
    for (int w = 0; w < ST_T / 32; ++w) {
      si += red[0][w];
      su += red[1][w];
    }
    iou[(long long)i * V + j] = su ? (float)((double)si / (double)su) : 0.f;
  }
}

}  // namespace

cudaError_t ts_launch_face_stats(const TsPlanImpl* p, const TsWs& w, uint32_t* coverage, float* area,
                                 uint32_t* visible, uint32_t* n_visible, cudaStream_t s) {
  if (n_visible) {
    cudaError_t e = cudaMemsetAsync(n_visible, 0, sizeof(uint32_t) * p->V, s);
    if (e != cudaSuccess) return e;
  }
  if (p->M == 0) return cudaSuccess;
  StatsArgs a;
  a.frec = w.frec;
  a.count = w.count;
  a.cov_in = w.cov;
  a.M = p->M;
  a.words = (int)((p->M + 31) / 32);
  a.coverage = coverage;
  a.area = area;
  a.visible = visible;
  a.n_visible = n_visible;
  const long long blocks = (p->M + 4 * ST_T - 1) / (4 * ST_T);
  if (blocks * p->V >= TS_SMS)
    k_face_stats<4><<<dim3((unsigned)blocks, (unsigned)p->V), ST_T, 0, s>>>(a);
  else
    k_face_stats<1><<<dim3((unsigned)((p->M + ST_T - 1) / ST_T), (unsigned)p->V), ST_T, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t ts_launch_covisibility(const TsPlanImpl* p, const uint32_t* visible, float* iou, cudaStream_t s) {
  const int words = (int)((p->M + 31) / 32);
  k_covis<<<dim3((unsigned)p->V, (unsigned)p->V), ST_T, 0, s>>>(visible, words, p->V, iou);
  return cudaGetLastError();
}
