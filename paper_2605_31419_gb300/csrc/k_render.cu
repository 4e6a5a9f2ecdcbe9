// k_render.cu -- Eq. 3-4 forward blend and its adjoint, one CTA per (view, tile) at a time.
//
// Staging: the tile's depth-sorted face ids select 128-byte records, of which the CTA copies seven of
// the eight 16-byte groups into shared memory with cp.async (two edge vectors are subtractions of the
// staged vertices, rounded as the projection rounds them); two buffers alternate so the next stage
// streams in while the current one is blended.  A staged record is 28 words long, so that 8 lanes
// reading the same group of 8 consecutive records hit distinct banks.  Each warp owns an 8 x 4 pixel
// sub-block of the tile.
//
// Forward: for 32 staged faces at a time, lane = face computes which of the warp's 32 pixels its face
// can cover (per pixel row the interval between its edges, widened: conservative); a 32 x 32 bit
// transpose gives every pixel the faces to visit, and then lane = pixel walks its own faces front to
// back: window (Eq. 3) from cancellation-free edge functions, alpha = min(alpha_max,
// o_F I), skip below alpha_min, stop before the face that would take T below T_min, accumulate colour,
// depth and opacity (Eq. 4).  A warp's cost is its longest pixel list instead of all the faces of its
// sub-block, each of which 5 of 32 pixels blend: issue-bound either way, the forward of 9 views of a
// 2M-face map went from 1182 to 688 us, of 64 tracking views from 878 to 687, and the fused step from
// 1893 to 1645 us (20-view room) and 1823 to 1441 (12-view window), images bit for bit.  (Two faces per
// pass leave half a pass idle at the end of every odd list, and their code is twice as long: one per pass
// takes the forward of 64 tracking views from 555 to 512 us at 40 registers, of 9 views of 2M faces from 697
// to 663, the fused step of the 12-view window from 1244 to 1199.)  The transpose of the blended bits gives,
// per face, the mask of the warp's pixels that blended it.  Writes C + T bg, D, A = 1 - T, per pixel T_final and the list position after the last
// contribution, and per sorted pair and warp that mask.
//
// Backward: per pixel, back to front from that position: recover T_n = T_{n+1} / (1 - alpha_n),
// keep the suffix sum S of later contributions (including the background term), form
// dL/dalpha_n = T_n v_n - S / (1 - alpha_n) with v_n = gC . c_n + gD z_n + gA, and chain into 22
// per-face sums (barycentric-weighted gradients of the edge, colour and depth interpolants, and of o_F;
// 26 with the side array: the face's normal and sigma_F).  The forward stores, per sorted pair and warp, the 32-bit
// mask of the warp's pixels that blended the face; the backward numbers those (face, pixel)
// entries back to front (a warp-wide scan of the masks' bit counts) and processes them 32 at a
// time, one per lane, so that no lane idles on a pixel the face does not cover.  Entries of
// one pixel are chained: each lane knows the lane of the entry before its own and how many there are, and
// in round r the lanes with r before them take up that lane's (T, S) -- the same products and sums, in the
// same order, as a per-pixel loop, in one short loop where replaying T and then S over all earlier entries
// took two long ones.  With 32-bit tile geometry, and masks of a one-stage list that stay in shared memory
// until the fused step's backward: fused step 1703 -> 1604 us (20-view room) and 1455 -> 1349 (12-view
// window), backward of 64 tracking views 780 -> 716.  Every
// per-face sum is over products of two per-entry factors: one of seven weighted gradients times one of
// three barycentrics (the gradient of o_F alone).  Each lane writes its entry's factors to a ring row in
// shared memory; then the 8 lanes of each quarter warp walk 8 rows, lane a accumulating factor a times the
// three barycentrics, and add them into the face's accumulator with one four-word reduction per lane where a
// face's run of rows ends: 8 unrolled steps a batch.  Odd quarters walk their rows the other way, so that a run
// across two quarters is left over in both and added once, and so is one from the first quarter into the last.
// (A reduction at every quarter's end gave the slot of a large face up to four times the additions, and its sums
// twice the rounding error: the colour gradients of two views of large faces were 1.26 times as far from their
// 64-bit values as those of a sum per batch, now 1.01.  Putting the quarters together cost 3 % of the fused pass,
// 1438 -> 1484 us for the 20-view room; with an entry's slot checked once, where its row is written, instead of at
// every reduction it takes 1433, the backward of 64 tracking views 709 for 688 before.)  The reductions themselves cost
// nothing measurable; the instructions do.  (A loop over the faces' runs, one word per lane: the backward of 64
// tracking views 1034 -> 918 us; testing every row's sums for zero and the slot in 64 bits: fused step 1321 ->
// 1244 us for the 12-view window, backward of 6 mapping views 172 -> 164.)
//
// Launch forms: one CTA per tile, or persistent CTAs (as many as fit on the GPU) that take tiles
// from a device counter.  The fused L1 step (ts_render_step_l1) runs a tile's forward, its loss
// and its backward in one CTA.
#include <algorithm>

#include "ts_internal.cuh"

namespace {

struct RenderArgs {
  const TsView* views;
  int V;
  long long M, VM;
  long long n_tiles;
  const float4* frec;
  const uint32_t* ids;
  const uint2* ranges;
  float* color;
  float* depth;
  float* alpha;
  float* tfin;
  int32_t* nlast;
  const float* dC;
  const float* dD;
  const float* dA;
  float* grad;
  float sigma, alpha_min, alpha_max, T_min;
  float bg0, bg1, bg2;
  int S;
  unsigned int* counter;
  uint32_t* lmask;
  const float4* aux;   // per (view, face): camera-space normal and, in .w, sigma_F; else null
  bool normals;        // TS_FLAG_NORMALS: composite the normal map
  bool face_sigma;     // TS_FLAG_FACE_SIGMA: each face's own window exponent
  float* normal;       // normal map output (may be null)
  const float* dN;     // gradient w.r.t. the normal map (may be null)
  uint32_t* cov;       // per (view, face) pixels blended by the forward (TS_FLAG_STATS), else null
  // fused L1 step (ts_render_step_l1): targets, depth weight, optional loss-gradient images and
  // the per-tile loss partials
  const float* tC;
  const float* tD;
  float lambda_dep;
  float* dC_out;
  float* dD_out;
  float* tloss;
  TsDevHeader* hdr;
  unsigned long long* ctr;  // counter slots (contributions)
};

constexpr unsigned FULL = 0xffffffffu;

// Register budgets of the raster kernels per thread, expressed as the minimum number of resident CTAs in the
// launch bounds.  More resident CTAs hide more latency until spills cost more.  16 x 8 tiles: 64 tracking views
// take the forward 512 us at 40 and 538 at 48, the backward 686 at 48, 669 at 56 and 768 at 64; with the side
// array, 6 mapping views take the forward 112 at 48 and 116 at 56, the backward 201 / 192 / 179 / 166 at 48 / 56 /
// 64 / 72; the fused step of the 12-view window takes 1247 / 1216 / 1260 at 48 / 56 / 64.  The forward of 8 x 8
// tiles, of which shared memory holds 14 at 64 faces a stage, spills at 40: 187 / 153 / 152 / 148 us at 40 / 48 /
// 56 / 72 for 16 views of 100k faces.
// With the side array the backward of CTAs of 256 threads takes 266 us at 72 (three CTAs) and 227 at 64 (four).
constexpr int REGS_FWD = 40, REGS_FWD_64 = 56, REGS_BWD = 56, REGS_STEP = 56, REGS_FWD_AUX = 48, REGS_BWD_AUX = 72;
constexpr int REGS_BWD_AUX_256 = 64;
// A quarter of a multiprocessor (16,384 registers) holds whole warps, so `regs` registers (a multiple of 8)
// leave 4 floor(16384 / (32 regs)) warps; in CTAs of `threads` the nearest number, halves down.  (Dividing 65,536 by
// threads x regs gave 8 x 8 tiles 32 registers for 40, and left CTAs of 512 threads one to a multiprocessor, with
// 108 registers, for 72: the side-array backward of 16 x 32 tiles took 421 us where it takes 271, 16 views of 100k.)
constexpr int raster_min_blocks(int threads, int regs) {
  const int resident = 4 * (16384 / (32 * regs)) * 32;
  return (2 * resident + threads - 1) / (2 * threads) > 0 ? (2 * resident + threads - 1) / (2 * threads) : 1;
}
constexpr int fwd_min_blocks(int threads, bool aux) {
  return raster_min_blocks(threads, aux ? REGS_FWD_AUX : (threads == 64 ? REGS_FWD_64 : REGS_FWD));
}
constexpr int bwd_min_blocks(int threads, bool aux) {
  return raster_min_blocks(threads, !aux ? REGS_BWD : (threads >= 256 ? REGS_BWD_AUX_256 : REGS_BWD_AUX));
}
// every tile shape gets its budget: 64 threads exactly, and 512 are not left with one CTA
static_assert(raster_min_blocks(64, 40) == 24 && raster_min_blocks(64, 48) == 20 && raster_min_blocks(128, 72) == 7 &&
                  raster_min_blocks(512, 72) == 2 && raster_min_blocks(512, 48) == 2 && raster_min_blocks(512, 40) == 3 &&
                  fwd_min_blocks(64, false) == 18 && fwd_min_blocks(128, false) == 12 &&
                  bwd_min_blocks(128, true) == 7 && bwd_min_blocks(256, true) == 4 && bwd_min_blocks(512, true) == 2,
              "resident CTAs of a register budget");

// Shared state of a render CTA.
struct RenderSmem {
  float lred[16][2];       // fused step: the warps' loss sums
  int lmax[16];            // fused step: the warps' largest last positions
  int4 geo;                // the tile's first pixel, W and H of its view
  long long pix_off;
  int view;
  int nmax;
  int next_tile;
};

// Forward only, TS_FLAG_STATS: per staged face, the number of the tile's pixels that blended it.
struct FwdMasks {
  uint32_t cv[2][128];
};

// What a tile's forward leaves for the backward of the fused step, per pixel (thread) and for the
// stage buffers: the last stage processed (in buffer st & 1), and whether the stage before it is still
// in the other buffer.
struct TileCarry {
  float T, C0, C1, C2, D;
  int nl;
  int st_last;
  bool prev_in;
};

// The backward's per-pixel inputs in the fused step: T_final and the loss gradients.
struct PixIn {
  float T, gC0, gC1, gC2, gD;
  int nl;
  int nmax;  // the same in every thread: the tile's largest nl
};

// Backward scratch per warp: the ring of one batch's rows and the pixels' back-to-front state.  Row words:
// 0-2 barycentrics l_k, 3 the face's gradient slot; 4-6 dm routed to the nearest edge (zero for the other
// two), 7-9 w gC_c, 10 w gD, 11 dL/do_F; with the side array 12-14 w gN_c and 15 dL/dsigma_F.  Rows are EW
// words apart, eight rows another 8, so that the quarter warps' rows and a row's words hit distinct banks.
constexpr int FMAX = 4;        // faces per lane when the backward numbers a stage's entries (128 / 32)
template <bool AUX>
struct Ring {
  static constexpr int EW = AUX ? 20 : 12;
  static constexpr int WORDS = 32 * EW + 4 * 8;
  static constexpr int BYTES_PER_WARP = WORDS * 4 + 32 * 8;
};

template <int TW, int TH>
struct TileGeom {
  static constexpr int NSBX = TW / 8;
  int view, x, y, W, H;
  bool inimg;
  float px, py;
  long long pix_off;
};

template <int TW, int TH>
__device__ __forceinline__ TileGeom<TW, TH> tile_geom(const RenderArgs& a, long long tile, RenderSmem& sm) {
  TileGeom<TW, TH> g;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp == 0) {  // the view owning the tile: one coalesced load and a ballot per 32 views
    int below = 0;
    for (int base = 0; base < a.V; base += 32) {
      const int v = base + lane;
      const unsigned b = __ballot_sync(FULL, v < a.V && a.views[v].tile_off <= tile);
      below += __popc(b);
      if (b != FULL) break;
    }
    if (lane == 0) {  // a tile of a view and its pixels fit 32 bits
      const TsView& vw = a.views[below - 1];
      const int lt = (int)(tile - vw.tile_off), ty = lt / vw.TX, tx = lt - ty * vw.TX;
      sm.geo = make_int4(tx * TW, ty * TH, vw.W, vw.H);
      sm.pix_off = vw.pix_off;
      sm.view = below - 1;
    }
  }
  __syncthreads();
  const int4 geo = sm.geo;
  g.view = sm.view;
  g.pix_off = sm.pix_off;
  g.W = geo.z;
  g.H = geo.w;
  g.x = geo.x + (warp % TileGeom<TW, TH>::NSBX) * 8 + (lane & 7);
  g.y = geo.y + (warp / TileGeom<TW, TH>::NSBX) * 4 + (lane >> 3);
  g.inimg = g.x < g.W && g.y < g.H;
  g.px = (float)g.x + 0.5f;
  g.py = (float)g.y + 0.5f;
  return g;
}

// 16-byte groups of a staged record: groups 0, 1 and 3..7 of the record (group 2 holds the edge vectors
// e1 and e2).
constexpr int SG = 7;

// Face id at place `at` of the sorted pair list.
__device__ __forceinline__ uint32_t list_id(const RenderArgs& a, uint32_t at) {
  const uint32_t id = __ldg(a.ids + at);
  if ((long long)id < a.M) return id;
  atomicOr(&a.hdr->error_bits, TS_ERRBIT_BOUNDS);  // never expected: record the fault, stage an in-bounds record
  return 0u;
}

// Every thread of the CTA copies 16-byte groups of stage `st` (records [st*S, st*S + cnt) of the
// tile's list) into buffer `b` with cp.async, SG groups per record and, with the side array, one more
// for the record's side entry (normal, sigma_F) after both record buffers; one commit group per stage.
template <bool AUX>
__device__ __forceinline__ void issue_stage(const RenderArgs& a, float4* smrec, int b, int st, uint32_t start,
                                            int n, const float4* vbase, const float4* nbase, int nthreads) {
  const int S = a.S;
  const int cnt = min(S, n - st * S);
  constexpr int PER = AUX ? SG + 1 : SG;
  for (int i = threadIdx.x; i < cnt * PER; i += nthreads) {
    const int j = i / PER, c = i - j * PER;
    const uint32_t id = list_id(a, start + (uint32_t)(st * S + j));
    if (!AUX || c < SG) {
      ts_cp_async16(smrec + ((size_t)b * S + j) * SG + c, vbase + (size_t)id * 8 + (c < 2 ? c : c + 1));
    } else {
      ts_cp_async16(smrec + (size_t)2 * S * SG + (size_t)b * S + j, nbase + id);
    }
  }
  ts_cp_async_commit();
}

// Wait for the stage issued last: each thread's copies (they always complete), then a barrier.
__device__ __forceinline__ void wait_stage() {
  ts_cp_async_wait_all();
  __syncthreads();
}

static_assert(R_U0 == 0 && R_V0 == 3 && R_V1 == 4 && R_E0X == 6 && R_E1X == 8 && R_E2X == 10 && R_K0 == 12 &&
                  R_INVD == 15 && R_OF == 16 && R_C0 == 17 && R_C1 == 20 && R_C2 == 23 && R_Z0 == 26 && R_Z2 == 28 &&
                  R_SLOT == 31,
              "record layout assumed by the staged groups");

// The edge evaluation (cross products, normalised edge functions, their minimum) from a staged
// record's groups 0..2: u, v, e0 and k, 1 / D2.  e1 and e2 are the projection's own subtractions.
__device__ __forceinline__ TsPix eval_edges(float4 q0, float4 q1, float4 qk, float px, float py) {
  TsPix o;
  o.cr0 = ts_det2(q1.z, q1.w, px - q0.x, py - q0.w);
  o.cr1 = ts_det2(__fsub_rn(q0.z, q0.y), __fsub_rn(q1.y, q1.x), px - q0.y, py - q1.x);
  o.cr2 = ts_det2(__fsub_rn(q0.x, q0.z), __fsub_rn(q0.w, q1.y), px - q0.z, py - q1.y);
  const float e0 = o.cr0 * qk.x, e1 = o.cr1 * qk.y, e2 = o.cr2 * qk.z;
  o.m = e0;
  o.arg = 0;
  if (e1 < o.m) { o.m = e1; o.arg = 1; }
  if (e2 < o.m) { o.m = e2; o.arg = 2; }
  return o;
}

// Conservative cover of one staged face in an 8 x 4 pixel block whose first pixel centre is (px, py):
// bit 8 r + c set when pixel (c, r) can have a positive window.  Per edge, the pixels inside satisfy
// f(c, r) = g + r a - c b > 0 (a, b the edge vector turned so that inside is positive, g the edge
// function at the block's first centre), i.e. c lies below or above (g + r a) / b; every row's interval
// is the intersection of its edges'.  g is widened by what moves the edge 0.01 px and by the rounding
// of its own terms (relevant for vertices far outside the image).
__device__ __forceinline__ unsigned block_cover(const float4* r4, float px, float py) {
  const float4 q0 = r4[0], q1 = r4[1];
  const float sg = r4[2].w > 0.f ? 1.f : -1.f;
  const float u[3] = {q0.x, q0.y, q0.z}, v[3] = {q0.w, q1.x, q1.y};
  // columns cut off at the right (hi) and at the left (lo) of each row
  float hi[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const int j = (i + 1) % 3;
    const float a = sg * (u[j] - u[i]), b = sg * (v[j] - v[i]);
    const float ya = a * (py - v[i]), xb = b * (px - u[i]);
    const float g = (ya - xb) + (0.01f * (fabsf(a) + fabsf(b)) + 1e-6f * (fabsf(ya) + fabsf(xb)));
    const float ib = ts_rcp_approx(fabsf(b));  // b = 0: infinite or NaN cuts, which cut nothing or everything
    const bool right = b > 0.f;
    // cut at the right: 7 - floor(t), at the left: ceil(t), t = (g + r a) / b; both -(g + r a) / |b| + a
    // constant, rounded to nearest below with 0.499 for the floor and the ceiling
    const float c0 = fmaf(-g, ib, right ? 7.499f : 0.499f), cs = -a * ib;
    if (right) {
      hi[0] = fmaxf(hi[0], c0);
#pragma unroll
      for (int r = 1; r < 4; ++r) hi[r] = fmaxf(hi[r], fmaf((float)r, cs, c0));
    } else {
      lo[0] = fmaxf(lo[0], c0);
#pragma unroll
      for (int r = 1; r < 4; ++r) lo[r] = fmaxf(lo[r], fmaf((float)r, cs, c0));
    }
  }
  constexpr float MAGIC = 12582912.f;  // 1.5 * 2^23: adding it rounds to an integer in the low bits
  unsigned cover = 0u;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const unsigned h = __float_as_uint(fminf(hi[r], 8.f) + MAGIC) & 15u;
    const unsigned l = __float_as_uint(fminf(lo[r], 8.f) + MAGIC) & 15u;
    cover |= ((0xffu >> h) & (0xffu << l)) << (8 * r);
  }
  return cover;
}

// Transpose of a 32 x 32 bit matrix, lane r holding row r: five exchanges of off-diagonal blocks.
__device__ __forceinline__ unsigned transpose32(unsigned x, int lane) {
#pragma unroll
  for (int j = 16; j > 0; j >>= 1) {
    const unsigned low = j == 16 ? 0x0000ffffu : j == 8 ? 0x00ff00ffu : j == 4 ? 0x0f0f0f0fu : j == 2 ? 0x33333333u : 0x55555555u;
    const unsigned y = __shfl_xor_sync(FULL, x, j);
    const bool upper = (lane & j) != 0;
    const unsigned take = upper ? low : ~low;  // the bits that come from the partner
    const unsigned rot = __funnelshift_l(y, y, upper ? 32 - j : j);
    x = (x & ~take) | (rot & take);
  }
  return x;
}

// Forward of one tile.  Stage st is staged in buffer st & 1.
template <int TW, int TH, bool AUX, bool FUSED = false>
__device__ __forceinline__ void fwd_tile(const RenderArgs& a, long long tile, float4* smrec, RenderSmem& sm,
                                         FwdMasks& fm, TileCarry* carry = nullptr,
                                         const TileGeom<TW, TH>* gin = nullptr, const uint2* rgin = nullptr,
                                         uint32_t* held = nullptr) {
  // (the list's range loads while the view is looked up)
  const uint2 rg = FUSED ? *rgin : a.ranges[tile];
  const TileGeom<TW, TH> g = FUSED ? *gin : tile_geom<TW, TH>(a, tile, sm);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = (int)(rg.y - rg.x);
  float T = 1.f, C0 = 0.f, C1 = 0.f, C2 = 0.f, D = 0.f;
  float N0 = 0.f, N1 = 0.f, N2 = 0.f;
  int nl = 0;
  bool done = !g.inimg;
  unsigned contrib = 0;
  int st_last = -1;
  bool prefetched = false;
  if (n > 0) {
    const int S = a.S;
    const int nst = (n + S - 1) / S;
    const float4* vbase = a.frec + (size_t)g.view * (size_t)a.M * 8;
    const float4* nbase = AUX ? a.aux + (size_t)g.view * (size_t)a.M : nullptr;
    const float bx = g.px - (float)(lane & 7), by = g.py - (float)(lane >> 3);  // the warp's first pixel centre
    issue_stage<AUX>(a, smrec, 0, 0, rg.x, n, vbase, nbase, TW * TH);
    if (a.cov)
      for (int j = threadIdx.x; j < 2 * 128; j += TW * TH) (&fm.cv[0][0])[j] = 0u;
    wait_stage();
    for (int st = 0; st < nst; ++st) {
      const int b = st & 1;
      const int cnt = min(S, n - st * S);
      st_last = st;
      // every warp is done with the other buffer (the barrier that ended the stage before)
      if (st + 1 < nst) issue_stage<AUX>(a, smrec, b ^ 1, st + 1, rg.x, n, vbase, nbase, TW * TH);
      const float4* rb = smrec + (size_t)b * S * SG;
      const float4* nb = smrec + (size_t)2 * S * SG + (size_t)b * S;
      for (int q = 0; q * 32 < cnt; ++q) {
        const int jq = q * 32 + lane;
        unsigned lm = 0;  // this warp's pixels that blended face jq
        if (!__all_sync(FULL, done)) {
          unsigned bits = jq < cnt ? block_cover(rb + jq * SG, bx, by) : 0u;
          if (__any_sync(FULL, bits != 0u)) {
            bits = transpose32(bits, lane);  // this pixel's faces
            if (done) bits = 0u;
            unsigned blended = 0u;
            while (bits) {
              const int j = __ffs(bits) - 1;
              bits &= bits - 1;
              const float4* r = rb + (q * 32 + j) * SG;
              const float4 kk = r[2];
              const TsPix e = eval_edges(r[0], r[1], kk, g.px, g.py);
              const float4 q4 = r[3];  // o_F, colour of vertex 0
              const float sig = (AUX && a.face_sigma) ? nb[q * 32 + j].w : a.sigma;
              // (the tests in one condition: where the window is not positive, alpha is not used)
              const float al = fminf(q4.x * ts_window(e.m, sig), a.alpha_max);
              const float Tn = T * (1.f - al);
              if (e.m > 0.f && al >= a.alpha_min) {
                if (Tn < a.T_min) {
                  done = true;
                  bits = 0u;
                } else {
                  const float invD = kk.w;
                  const float l0 = e.cr1 * invD, l1 = e.cr2 * invD, l2 = e.cr0 * invD;
                  const float w = al * T;
                  const float4 q5 = r[4], q6 = r[5];  // colours of vertices 1 and 2, depths z_0, z_1
                  C0 += w * (l0 * q4.y + l1 * q5.x + l2 * q5.w);
                  C1 += w * (l0 * q4.z + l1 * q5.y + l2 * q6.x);
                  C2 += w * (l0 * q4.w + l1 * q5.z + l2 * q6.y);
                  D += w * (l0 * q6.z + l1 * q6.w + l2 * r[6].x);
                  if (AUX && a.normals) {
                    const float4 nn = nb[q * 32 + j];
                    N0 += w * nn.x;
                    N1 += w * nn.y;
                    N2 += w * nn.z;
                  }
                  T = Tn;
                  nl = st * S + q * 32 + j + 1;
                  blended |= 1u << j;
                }
              }
            }
            contrib += __popc(blended);
            // the backward takes exactly these (face, pixel) contributions
            if (FUSED || a.lmask || a.cov) lm = transpose32(blended, lane);
            if (a.cov && lm) atomicAdd(&fm.cv[b][jq], (unsigned)__popc(lm));
          }
        }
        if (FUSED && jq < cnt) held[b * S + jq] = lm;
        // (a list of one stage stays in shared memory until the fused step's backward)
        if (a.lmask && jq < cnt && !(FUSED && nst == 1)) a.lmask[(size_t)(rg.x + (uint32_t)(st * S + jq)) * (TW * TH / 32) + warp] = lm;
      }
      if (st + 1 == nst && !a.cov) break;  // nothing reads the buffers or the counts after this stage
      ts_cp_async_wait_all();              // the next stage, published by the barrier
      const int alive = __syncthreads_count(!done);
      if (a.cov) {
        for (int j = threadIdx.x; j < cnt; j += TW * TH) {
          // the face from the list: other warps may already be copying the stage after next over this
          // stage's records, which nothing reads past the barrier
          if (fm.cv[b][j]) {
            const uint32_t id = list_id(a, rg.x + (uint32_t)(st * S + j));
            atomicAdd(a.cov + (long long)g.view * a.M + id, fm.cv[b][j]);
            fm.cv[b][j] = 0u;  // for the stage after next, a barrier away
          }
        }
      }
      if (alive == 0) {
        prefetched = st + 1 < nst;
        break;
      }
    }
  }
  ts_count_add(a.ctr, TS_CTR_FWD, contrib);
  if constexpr (FUSED) {
    carry->T = T;
    carry->C0 = C0;
    carry->C1 = C1;
    carry->C2 = C2;
    carry->D = D;
    carry->nl = nl;
    carry->st_last = st_last;
    carry->prev_in = st_last >= 1 && !prefetched;
  }
  if (g.inimg) {
    const int HW = g.W * g.H, pi = g.y * g.W + g.x;
    const long long o = g.pix_off + pi;
    if (a.color) {
      float* c = a.color + 3 * g.pix_off + pi;
      c[0] = C0 + T * a.bg0;
      c[HW] = C1 + T * a.bg1;
      c[2LL * HW] = C2 + T * a.bg2;
    }
    if (a.depth) a.depth[o] = D;
    if (a.alpha) a.alpha[o] = 1.f - T;
    if (AUX && a.normal) {
      float* q = a.normal + 3 * g.pix_off + pi;
      q[0] = N0;
      q[HW] = N1;
      q[2LL * HW] = N2;
    }
    if (!FUSED) {  // what ts_render_bwd needs; the fused step keeps them in registers
      a.tfin[o] = T;
      a.nlast[o] = nl;
    }
  }
}

// Add four floats to a 16-byte aligned global address, without a result.
__device__ __forceinline__ void red_add_v4(float* p, float a, float b, float c, float d) {
  asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c), "f"(d)
               : "memory");
}

template <int TW, int TH, bool AUX, bool FUSED = false>
__device__ __forceinline__ void bwd_tile(const RenderArgs& a, long long tile, float4* smrec, RenderSmem& sm,
                                         const PixIn* pin = nullptr, const TileCarry* carry = nullptr,
                                         const TileGeom<TW, TH>* gin = nullptr, const uint2* rgin = nullptr,
                                         const uint32_t* held = nullptr) {
  // (the list's range loads while the view is looked up)
  const uint2 rg = FUSED ? *rgin : a.ranges[tile];
  const TileGeom<TW, TH> g = FUSED ? *gin : tile_geom<TW, TH>(a, tile, sm);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int len = (int)(rg.y - rg.x);
  const float4* vbase = a.frec + (size_t)g.view * (size_t)a.M * 8;
  const float4* nbase = AUX ? a.aux + (size_t)g.view * (size_t)a.M : nullptr;
  float T = 0.f, Sacc = 0.f, gC0 = 0.f, gC1 = 0.f, gC2 = 0.f, gD = 0.f, gA = 0.f;
  float gN0 = 0.f, gN1 = 0.f, gN2 = 0.f;
  int nl = 0;
  if (FUSED) {  // the forward's state and the loss gradients, still in registers
    if (g.inimg) {
      T = pin->T;
      nl = pin->nl;
      gC0 = pin->gC0;
      gC1 = pin->gC1;
      gC2 = pin->gC2;
      gD = pin->gD;
      Sacc = T * (gC0 * a.bg0 + gC1 * a.bg1 + gC2 * a.bg2);
    }
  } else if (g.inimg) {
    const int HW = g.W * g.H, pi = g.y * g.W + g.x;
    const long long o = g.pix_off + pi;
    T = a.tfin[o];
    nl = a.nlast[o];
    const float* dc = a.dC + 3 * g.pix_off + pi;
    gC0 = dc[0];
    gC1 = dc[HW];
    gC2 = dc[2LL * HW];
    gD = a.dD ? a.dD[o] : 0.f;
    gA = a.dA ? a.dA[o] : 0.f;
    if (AUX && a.dN) {
      const float* dn = a.dN + 3 * g.pix_off + pi;
      gN0 = dn[0];
      gN1 = dn[HW];
      gN2 = dn[2LL * HW];
    }
    Sacc = T * (gC0 * a.bg0 + gC1 * a.bg1 + gC2 * a.bg2);
  }
  int nmax;
  if (FUSED) {
    nmax = pin->nmax;  // the tile's largest last position, reduced with the loss sums
  } else {
    if (threadIdx.x == 0) sm.nmax = 0;
    __syncthreads();
    {
      const int m = __reduce_max_sync(FULL, (unsigned)nl);
      if (lane == 0 && m) atomicMax(&sm.nmax, m);
    }
    __syncthreads();
    nmax = sm.nmax;
  }
  // positions come from the forward pass over the same lists; clamp in case the caller did not
  // run it after the last ts_bin
  const int n = min(nmax, len);
  unsigned contrib = 0;
  if (n > 0) {
    const int S = a.S;
    const int nst = (n + S - 1) / S;
    if (!FUSED) issue_stage<AUX>(a, smrec, (nst - 1) & 1, nst - 1, rg.x, n, vbase, nbase, TW * TH);
    constexpr int EW = Ring<AUX>::EW;
    unsigned char* wbase = reinterpret_cast<unsigned char*>(smrec + (size_t)2 * S * (AUX ? SG + 1 : SG)) +
                           (size_t)warp * Ring<AUX>::BYTES_PER_WARP;
    float* ring = reinterpret_cast<float*>(wbase);
    float2* pst = reinterpret_cast<float2*>(wbase + Ring<AUX>::WORDS * 4);  // per pixel lane: (T, S)
    pst[lane] = make_float2(T, Sacc);
    __syncwarp();  // read by other lanes; a stage that is still staged has no barrier before its first batch
    // this lane's entry's row (odd quarters' in falling order)
    float* row_here = ring + (lane ^ ((lane & 8) ? 7 : 0)) * EW + (lane >> 3) * 8;
    const float* row_sum = ring + (lane >> 3) * (8 * EW + 8);                  // its quarter warp's first row
    const int fa = lane & 7;                                                   // the factor it sums
    const uint32_t vm32 = (uint32_t)min(a.VM, 0xffffffffll);                   // slots
    const int xw = g.x - (lane & 7), yw = g.y - (lane >> 3);  // the warp's first pixel
    for (int k = 0; k < nst; ++k) {
      const int st = nst - 1 - k;
      int b = st & 1;
      const int cnt = min(S, n - st * S);
      // The forward's lane masks (positions below the tile's largest list position after a
      // contribution were all written by it) give, per face, the pixels of this warp that blended
      // it.  Lane L holds the masks of F = ceil(cnt / 32) faces, lane 0 the backmost; the stage's
      // (face, pixel) entries are numbered back to front, face by face, pixels in lane order, and
      // each batch of 32 consecutive numbers gives every lane one entry.  The masks load while
      // the stage's copies land.
      constexpr int NW = TW * TH / 32;
      const uint32_t* lmrow = a.lmask + (size_t)(rg.x + (uint32_t)(st * S)) * NW + warp;
      const int F = (cnt + 31) >> 5;  // faces per lane: lane L holds faces F * (32 - L) - 1 - i, i < F
      // the fused step: the forward's last stage, and the one before it unless a prefetch replaced it, are
      // still staged, their masks in shared memory; other stages are staged again
      const bool here = FUSED && (st == carry->st_last || (st == carry->st_last - 1 && carry->prev_in));
      unsigned lmk[FMAX];
#pragma unroll
      for (int i = 0; i < FMAX; ++i) {
        const int jf = F * (32 - lane) - 1 - i;
        lmk[i] = 0u;
        if (i < F && jf < cnt) lmk[i] = here ? held[b * S + jf] : lmrow[(size_t)jf * NW];
      }
      if (FUSED) {
        if (!here) {  // (all warps are done with both buffers)
          __syncthreads();
          b = 0;
          issue_stage<AUX>(a, smrec, b, st, rg.x, n, vbase, nbase, TW * TH);
          wait_stage();
        }
      } else {
        wait_stage();
        if (k + 1 < nst) issue_stage<AUX>(a, smrec, b ^ 1, st - 1, rg.x, n, vbase, nbase, TW * TH);
      }
      const float4* rb = smrec + (size_t)b * S * SG;
      const float4* nb = smrec + (size_t)2 * S * SG + (size_t)b * S;
      {
        // lane L's faces have popc of their masks entries; their numbers start at the exclusive
        // scan over the lanes, face by face within a lane
        int c = 0;
#pragma unroll
        for (int i = 0; i < FMAX; ++i) c += __popc(lmk[i]);
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int t = __shfl_up_sync(FULL, incl, o);
          if (lane >= o) incl += t;
        }
        const int total = __shfl_sync(FULL, incl, 31);
        const int excl = incl - c;
        for (int e0 = 0; e0 < total; e0 += 32) {
          const int ne = min(total - e0, 32);
          const bool act = lane < ne;
          const int ee = e0 + lane;
          // the entry's lane: the last lane whose first number is at most ee (binary search)
          int ow = 0;
#pragma unroll
          for (int w = 16; w > 0; w >>= 1) {
            const int ex = __shfl_sync(FULL, excl, (ow + w) & 31);
            if (ow + w < 32 && ex <= ee) ow += w;
          }
          int kk = ee - __shfl_sync(FULL, excl, ow);  // the entry's rank among that lane's pixels
          // the face among the lane's F faces, then its pixel: the kk-th set bit of its mask
          unsigned om = 0u;
          int fi = 0;
          bool found = false;
#pragma unroll
          for (int i = 0; i < FMAX; ++i) {
            if (i >= F) break;  // uniform
            const unsigned mi = __shfl_sync(FULL, lmk[i], ow);
            const int ci = __popc(mi);
            if (!found) {
              if (kk < ci) {
                om = mi;
                fi = i;
                found = true;
              } else {
                kk -= ci;
              }
            }
          }
          int pb = 0;
          unsigned mm = om;
#pragma unroll
          for (int w = 16; w > 0; w >>= 1) {
            const int cl = __popc(mm & ((1u << w) - 1u));
            if (kk >= cl) {
              kk -= cl;
              pb += w;
              mm >>= w;
            }
          }
          const int j = act ? F * (32 - ow) - 1 - fi : 0;
          const int p = act ? pb : lane;
          // -- one entry per lane: face j at pixel lane p ---------------------------------------
          const float4* r4 = rb + j * SG;
          const float px = (float)(xw + (p & 7)) + 0.5f, py = (float)(yw + (p >> 3)) + 0.5f;
          const float sig = (AUX && a.face_sigma) ? nb[j].w : a.sigma;
          const float4 q3 = r4[2];  // k_0, k_1, k_2, invD
          const TsPix e = eval_edges(r4[0], r4[1], q3, px, py);
          const float4 q4 = r4[3];  // o_F, colour of vertex 0
          const float oF = q4.x;
          const float I = act ? ts_window(e.m, sig) : 0.f;
          const float al = fminf(oF * I, a.alpha_max);
          const float ro = ts_rcp_approx(1.f - al);  // 1 - al >= 1 - alpha_max
          // entries of the same pixel, in entry (back-to-front) order: the one before this lane's, and how many
          // are
          const unsigned peers = __match_any_sync(FULL, act ? p : 32 + lane);
          const unsigned before = peers & ((1u << lane) - 1u);
          const int prev = before ? 31 - __clz(before) : lane, depth = __popc(before);
          const int K = (int)__reduce_max_sync(FULL, (unsigned)depth);
          const float2 st0 = pst[p];
          const float qC0 = __shfl_sync(FULL, gC0, p), qC1 = __shfl_sync(FULL, gC1, p);
          const float qC2 = __shfl_sync(FULL, gC2, p), qD = __shfl_sync(FULL, gD, p);
          const float qA = __shfl_sync(FULL, gA, p);
          float qN0 = 0.f, qN1 = 0.f, qN2 = 0.f;
          if constexpr (AUX) {
            qN0 = __shfl_sync(FULL, gN0, p);
            qN1 = __shfl_sync(FULL, gN1, p);
            qN2 = __shfl_sync(FULL, gN2, p);
          }
          const float invD = q3.w;
          const float l0 = e.cr1 * invD, l1 = e.cr2 * invD, l2 = e.cr0 * invD;
          const float4 q5 = r4[4], q6 = r4[5];  // colours of vertices 1 and 2, depths z_0, z_1
          const float4 q7 = r4[6];
          const float z2 = q7.x;
          const uint32_t slot = __float_as_uint(q7.w);
          const float c0 = l0 * q4.y + l1 * q5.x + l2 * q5.w;
          const float c1 = l0 * q4.z + l1 * q5.y + l2 * q6.x;
          const float c2 = l0 * q4.w + l1 * q5.z + l2 * q6.y;
          const float z = l0 * q6.z + l1 * q6.w + l2 * z2;
          float val = qC0 * c0 + qC1 * c1 + qC2 * c2 + qD * z + qA;
          if (AUX && a.normals) {
            const float4 nn = nb[j];
            val += qN0 * nn.x + qN1 * nn.y + qN2 * nn.z;
          }
          // the pixel's recurrences T <- T / (1 - alpha) and S <- S + (this face's term), entry after entry: in
          // round r the lanes with r entries of their pixel before them take up the state of the one before
          float Tn = st0.x * ro, Sn = st0.y;
          float add = val * al * Tn;  // this face's term of the suffix sum S seen by earlier faces
          for (int r = 1; r <= K; ++r) {
            const float Tb = __shfl_sync(FULL, Tn, prev), Sb = __shfl_sync(FULL, Sn + add, prev);
            if (depth == r) {
              Tn = Tb * ro;
              Sn = Sb;
              add = val * al * Tn;
            }
          }
          const float w = al * Tn;
          __syncwarp();  // every lane has read its pixel's state before the last entries replace it
          if (act && (peers >> lane) == 1u) pst[p] = make_float2(Tn, Sn + add);
          const float dal = val * Tn - Sn * ro;
          float go = 0.f, dm = 0.f, gs = 0.f;
          if (!(oF * I > a.alpha_max)) {
            go = dal * I;
            const float dI = dal * oF;
            // I >= alpha_min / o_F for a contributing entry, far from zero
            dm = (sig == 0.5f) ? dI * 0.5f * ts_rcp_approx(I) : dI * sig * I / e.m;
            if constexpr (AUX) {  // dL/dsigma_F = dL/dalpha o_F I ln(ratio)
              if (a.face_sigma) gs = dI * I * logf(e.m);
            }
          }
          float4* row = reinterpret_cast<float4*>(row_here);
          // (never expected: record the fault, add nothing)
          if (act && slot >= vm32) atomicOr(&a.hdr->error_bits, TS_ERRBIT_BOUNDS);
          if (act && slot < vm32) {
            row[0] = make_float4(l0, l1, l2, __uint_as_float(slot));
            row[1] = make_float4(e.arg == 0 ? dm : 0.f, e.arg == 1 ? dm : 0.f, e.arg == 2 ? dm : 0.f, qC0 * w);
            row[2] = make_float4(qC1 * w, qC2 * w, qD * w, go);
            if constexpr (AUX) row[3] = make_float4(qN0 * w, qN1 * w, qN2 * w, gs);
          } else {  // nothing to add
            row[0] = row[1] = row[2] = make_float4(0.f, 0.f, 0.f, 0.f);
            if constexpr (AUX) row[3] = make_float4(0.f, 0.f, 0.f, 0.f);
          }
          contrib += act ? 1u : 0u;
          // the batch's faces are runs of consecutive entries.  Even quarters take their rows upwards and add a run's
          // sums at its last row, odd quarters downwards (their rows lie in that order) and at its first: a run that
          // crosses from an even quarter into the next is then left in both, and put together
          const int jnext = __shfl_down_sync(FULL, j, 1);
          const unsigned ends = __ballot_sync(FULL, act && (lane == ne - 1 || j != jnext));
          const unsigned rows = (2u << (ne - 1)) - 1u;  // the active ones
          const unsigned firsts = ((ends << 1) | 1u) & rows;
          const unsigned stop = (lane & 8) ? __brev(firsts) >> (24 - (lane & 24)) : ends >> (lane & 24);
          const bool cross = ((~ends & (rows >> 1)) >> (lane & 16)) & 0x80u;  // into this lane's pair's odd quarter
          __syncwarp();
          float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
          uint32_t sl = 0u;
          auto to_slot = [&]() {
            if (fa == 7) s1 = s2 = 0.f;
            red_add_v4(a.grad + (size_t)sl * TS_GRAD_WORDS + 4 * fa, s0, s1, s2, s3);
          };
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float4 l = *reinterpret_cast<const float4*>(row_sum + i * EW);
            const float f = row_sum[i * EW + 4 + fa];
            s0 = fmaf(f, fa == 7 ? 1.f : l.x, s0);
            s1 = fmaf(f, l.y, s1);
            s2 = fmaf(f, l.z, s2);
            if (AUX && fa < 4) s3 += row_sum[i * EW + 12 + fa];
            sl = __float_as_uint(l.w);
            if (i < 7 && ((stop >> i) & 1u)) {
              to_slot();
              s0 = s1 = s2 = s3 = 0.f;
            }
          }
          const float t0 = __shfl_xor_sync(FULL, s0, 8), t1 = __shfl_xor_sync(FULL, s1, 8);
          const float t2 = __shfl_xor_sync(FULL, s2, 8), t3 = AUX ? __shfl_xor_sync(FULL, s3, 8) : 0.f;
          s0 += cross ? t0 : 0.f;
          s1 += cross ? t1 : 0.f;
          s2 += cross ? t2 : 0.f;
          if (AUX) s3 += cross ? t3 : 0.f;
          bool whole = cross ? !(lane & 8) : ((stop >> 7) & 1u) != 0u;
          if (ne > 24 && !(ends & 0x00ffff80u)) {  // uniform: one run from the first quarter into the last
            s0 += __shfl_xor_sync(FULL, s0, 16);
            s1 += __shfl_xor_sync(FULL, s1, 16);
            s2 += __shfl_xor_sync(FULL, s2, 16);
            if (AUX) s3 += __shfl_xor_sync(FULL, s3, 16);
            whole = lane < 8;
          }
          if (whole) to_slot();
          __syncwarp();
        }
      }
    }
  }
  ts_count_add(a.ctr, TS_CTR_BWD, contrib);
}

// The fused L1 step of one tile: the forward, the mean-L1 loss of its pixels (Eq. 8 L1 part with
// the depth term of Eq. 9: per pixel dL/dC = sign(C - Cbar) / (3HW) on the colour image with its
// background term, dL/dD = lambda_dep sign(D - Dbar) / (HW) where Dbar > 0), the tile's loss sums
// in a fixed order, and the backward from those gradients -- the same values ts_render_fwd,
// ts_l1_loss and ts_render_bwd give, without the images' round trip through memory.
template <int TW, int TH>
__device__ __forceinline__ void step_tile(const RenderArgs& a, long long tile, float4* smrec, RenderSmem& sm,
                                          FwdMasks& fm) {
  TileCarry c;
  // the warp's lane masks of the two stage buffers, after the rings
  uint32_t* held = reinterpret_cast<uint32_t*>(reinterpret_cast<unsigned char*>(smrec + (size_t)2 * a.S * SG) +
                                               (size_t)(TW * TH / 32) * Ring<false>::BYTES_PER_WARP) +
                   (size_t)(threadIdx.x >> 5) * 2 * a.S;
  const uint2 rg = a.ranges[tile];
  const TileGeom<TW, TH> g = tile_geom<TW, TH>(a, tile, sm);
  fwd_tile<TW, TH, false, true>(a, tile, smrec, sm, fm, &c, &g, &rg, held);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  PixIn pin{c.T, 0.f, 0.f, 0.f, 0.f, c.nl, 0};
  float lc = 0.f, ld = 0.f;
  if (g.inimg) {
    const int HW = g.W * g.H, pi = g.y * g.W + g.x;
    const long long o = g.pix_off + pi;
    const float ic = 1.0f / (3.0f * (float)HW), id = a.lambda_dep / (float)HW;
    const float col[3] = {c.C0 + c.T * a.bg0, c.C1 + c.T * a.bg1, c.C2 + c.T * a.bg2};  // the colour image
    float gc[3];
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) {
      const long long q = 3 * g.pix_off + (long long)ch * HW + pi;
      const float r = col[ch] - a.tC[q];
      lc += fabsf(r);
      gc[ch] = r > 0.f ? ic : (r < 0.f ? -ic : 0.f);
      if (a.dC_out) a.dC_out[q] = gc[ch];
    }
    const float t = a.tD[o];
    const float r = c.D - t;
    const bool valid = t > 0.f;
    if (valid) ld += fabsf(r);
    pin.gD = valid ? (r > 0.f ? id : (r < 0.f ? -id : 0.f)) : 0.f;
    if (a.dD_out) a.dD_out[o] = pin.gD;
    pin.gC0 = gc[0];
    pin.gC1 = gc[1];
    pin.gC2 = gc[2];
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lc += __shfl_xor_sync(FULL, lc, o);
    ld += __shfl_xor_sync(FULL, ld, o);
  }
  const int wmax = (int)__reduce_max_sync(FULL, (unsigned)c.nl);
  if (lane == 0) {
    sm.lred[warp][0] = lc;
    sm.lred[warp][1] = ld;
    sm.lmax[warp] = wmax;
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    float sum = 0.f;
#pragma unroll
    for (int w = 0; w < TW * TH / 32; ++w) sum += sm.lred[w][threadIdx.x];
    a.tloss[2 * tile + threadIdx.x] = sum;
  }
#pragma unroll
  for (int w = 0; w < TW * TH / 32; ++w) pin.nmax = max(pin.nmax, sm.lmax[w]);
  bwd_tile<TW, TH, false, true>(a, tile, smrec, sm, &pin, &c, &g, &rg, held);
}

// Next tile of a persistent CTA (the same value in every thread), or -1 when none is left.
__device__ __forceinline__ long long next_tile(const RenderArgs& a, RenderSmem& sm) {
  __syncthreads();
  if (threadIdx.x == 0) sm.next_tile = (int)atomicAdd(a.counter, 1u);
  __syncthreads();
  return sm.next_tile < a.n_tiles ? (long long)sm.next_tile : -1;
}

template <int TW, int TH, bool PERSIST, bool AUX>
__global__ void __launch_bounds__(TW * TH, fwd_min_blocks(TW * TH, AUX)) k_render_fwd(RenderArgs a) {
  extern __shared__ __align__(128) float4 smrec[];
  __shared__ RenderSmem sm;
  __shared__ FwdMasks fm;
  if constexpr (!PERSIST) {
    fwd_tile<TW, TH, AUX>(a, blockIdx.x, smrec, sm, fm);
  } else {
    for (long long t = next_tile(a, sm); t >= 0; t = next_tile(a, sm))
      fwd_tile<TW, TH, AUX>(a, t, smrec, sm, fm);
  }
}

template <int TW, int TH, bool PERSIST, bool AUX>
__global__ void __launch_bounds__(TW * TH, bwd_min_blocks(TW * TH, AUX)) k_render_bwd(RenderArgs a) {
  extern __shared__ __align__(128) float4 smrec[];
  __shared__ RenderSmem sm;
  if constexpr (!PERSIST) {
    bwd_tile<TW, TH, AUX>(a, blockIdx.x, smrec, sm);
  } else {
    for (long long t = next_tile(a, sm); t >= 0; t = next_tile(a, sm))
      bwd_tile<TW, TH, AUX>(a, t, smrec, sm);
  }
}

// The fused step kernel.  Its forward's coverage counts (TS_FLAG_STATS) live in the space of the
// backward's rings, which the forward does not use.
template <int TW, int TH, bool PERSIST>
__global__ void __launch_bounds__(TW * TH, raster_min_blocks(TW * TH, REGS_STEP)) k_render_step(RenderArgs a) {
  extern __shared__ __align__(128) float4 smrec[];
  __shared__ RenderSmem sm;
  static_assert(sizeof(FwdMasks) <= (TW * TH / 32) * Ring<false>::BYTES_PER_WARP, "coverage counts fit the rings");
  FwdMasks& fm = *reinterpret_cast<FwdMasks*>(smrec + (size_t)2 * a.S * SG);
  if constexpr (!PERSIST) {
    step_tile<TW, TH>(a, blockIdx.x, smrec, sm, fm);
  } else {
    for (long long t = next_tile(a, sm); t >= 0; t = next_tile(a, sm)) step_tile<TW, TH>(a, t, smrec, sm, fm);
  }
}

// Per view, the sum of its tiles' loss partials in a fixed order.
__global__ void __launch_bounds__(256) k_loss_tiles(const TsView* __restrict__ views, const float* __restrict__ tloss,
                                                    float lambda_dep, float* __restrict__ loss) {
  __shared__ float red[256][2];
  const TsView& vw = views[blockIdx.x];
  const long long t0 = vw.tile_off, nt = (long long)vw.TX * vw.TY;
  float x = 0.f, y = 0.f;
  for (long long t = threadIdx.x; t < nt; t += 256) {
    x += tloss[2 * (t0 + t)];
    y += tloss[2 * (t0 + t) + 1];
  }
  red[threadIdx.x][0] = x;
  red[threadIdx.x][1] = y;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      red[threadIdx.x][0] += red[threadIdx.x + o][0];
      red[threadIdx.x][1] += red[threadIdx.x + o][1];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double HW = (double)vw.W * vw.H;
    loss[blockIdx.x] = (float)((double)red[0][0] / (3.0 * HW) + (double)lambda_dep * (double)red[0][1] / HW);
  }
}

template <int TW, int TH>
cudaError_t launch_step(bool persist, const RenderArgs& a, cudaStream_t s) {
  const size_t smem = (size_t)2 * a.S * SG * 16 + (size_t)(TW * TH / 32) * (Ring<false>::BYTES_PER_WARP + 2 * a.S * 4);
  if (a.n_tiles == 0) return cudaSuccess;
  const void* f = persist ? (const void*)k_render_step<TW, TH, true> : (const void*)k_render_step<TW, TH, false>;
  cudaError_t e = ts_smem_limit(f, (int)smem);
  if (e != cudaSuccess) return e;
  if (!persist) {
    k_render_step<TW, TH, false><<<(unsigned)a.n_tiles, TW * TH, smem, s>>>(a);
    return cudaGetLastError();
  }
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_render_step<TW, TH, true>, TW * TH, smem);
  const long long grid = std::max(1LL, std::min<long long>(a.n_tiles, (long long)sms * std::max(per_sm, 1)));
  e = cudaMemsetAsync(a.counter, 0, sizeof(unsigned int), s);
  if (e != cudaSuccess) return e;
  k_render_step<TW, TH, true><<<(unsigned)grid, TW * TH, smem, s>>>(a);
  return cudaGetLastError();
}

// Dynamic shared memory: two stage buffers of S staged records, then (with the side array) two
// of S 16-byte side entries, then in the backward the warps' rings and their headers.
template <int TW, int TH, bool AUX>
cudaError_t launch_pair(bool fwd, bool persist, const RenderArgs& a, cudaStream_t s) {
  const size_t smem = (size_t)2 * a.S * (AUX ? SG + 1 : SG) * 16 + (fwd ? 0 : (size_t)(TW * TH / 32) * Ring<AUX>::BYTES_PER_WARP);
  if (a.n_tiles == 0) return cudaSuccess;
  {
    const void* f = fwd ? (persist ? (const void*)k_render_fwd<TW, TH, true, AUX> : (const void*)k_render_fwd<TW, TH, false, AUX>)
                        : (persist ? (const void*)k_render_bwd<TW, TH, true, AUX> : (const void*)k_render_bwd<TW, TH, false, AUX>);
    const cudaError_t e = ts_smem_limit(f, (int)smem);
    if (e != cudaSuccess) return e;
  }
  if (!persist) {
    if (fwd) k_render_fwd<TW, TH, false, AUX><<<(unsigned)a.n_tiles, TW * TH, smem, s>>>(a);
    else k_render_bwd<TW, TH, false, AUX><<<(unsigned)a.n_tiles, TW * TH, smem, s>>>(a);
    return cudaGetLastError();
  }
  int dev = 0, sms = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (fwd) cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_render_fwd<TW, TH, true, AUX>, TW * TH, smem);
  else cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_render_bwd<TW, TH, true, AUX>, TW * TH, smem);
  const long long grid = std::max(1LL, std::min<long long>(a.n_tiles, (long long)sms * std::max(per_sm, 1)));
  cudaError_t e = cudaMemsetAsync(a.counter, 0, sizeof(unsigned int), s);
  if (e != cudaSuccess) return e;
  if (fwd) k_render_fwd<TW, TH, true, AUX><<<(unsigned)grid, TW * TH, smem, s>>>(a);
  else k_render_bwd<TW, TH, true, AUX><<<(unsigned)grid, TW * TH, smem, s>>>(a);
  return cudaGetLastError();
}

template <bool AUX>
cudaError_t dispatch_tiles(bool fwd, const TsPlanImpl* p, const RenderArgs& a, cudaStream_t s) {
  const int tw = p->prm.tile_w, th = p->prm.tile_h;
  const bool persist = (p->prm.flags & TS_FLAG_PERSISTENT) != 0;
  if (tw == 16 && th == 8) return launch_pair<16, 8, AUX>(fwd, persist, a, s);
  if (tw == 16 && th == 16) return launch_pair<16, 16, AUX>(fwd, persist, a, s);
  if (tw == 8 && th == 8) return launch_pair<8, 8, AUX>(fwd, persist, a, s);
  if (tw == 32 && th == 8) return launch_pair<32, 8, AUX>(fwd, persist, a, s);
  if (tw == 16 && th == 32) return launch_pair<16, 32, AUX>(fwd, persist, a, s);
  if (tw == 32 && th == 16) return launch_pair<32, 16, AUX>(fwd, persist, a, s);
  return cudaErrorInvalidValue;
}

cudaError_t dispatch(bool fwd, const TsPlanImpl* p, const RenderArgs& a, cudaStream_t s) {
  return (p->normals || p->face_sigma) ? dispatch_tiles<true>(fwd, p, a, s) : dispatch_tiles<false>(fwd, p, a, s);
}

RenderArgs base_args(const TsPlanImpl* p, const TsWs& w) {
  RenderArgs a;
  a.views = w.views;
  a.V = p->V;
  a.M = p->M;
  a.VM = (long long)p->V * p->M;
  a.n_tiles = p->n_tiles;
  a.frec = w.frec;
  a.ids = w.vals[0];
  a.ranges = w.ranges;
  a.color = a.depth = a.alpha = nullptr;
  a.tfin = w.tfin;
  a.nlast = w.nlast;
  a.dC = a.dD = a.dA = nullptr;
  a.grad = w.grad;
  a.sigma = p->prm.sigma;
  a.alpha_min = p->prm.alpha_min;
  a.alpha_max = p->prm.alpha_max;
  a.T_min = p->prm.T_min;
  a.bg0 = p->prm.bg[0];
  a.bg1 = p->prm.bg[1];
  a.bg2 = p->prm.bg[2];
  a.S = p->prm.tris_per_stage;
  a.hdr = w.hdr;
  a.ctr = w.ctr;
  a.counter = &w.hdr->tile_counter;
  a.lmask = w.lmask;
  a.aux = w.aux;
  a.normals = p->normals;
  a.face_sigma = p->face_sigma;
  a.cov = w.cov;
  a.normal = nullptr;
  a.dN = nullptr;
  a.tC = a.tD = nullptr;
  a.lambda_dep = 0.f;
  a.dC_out = a.dD_out = nullptr;
  a.tloss = nullptr;
  return a;
}

}  // namespace

cudaError_t ts_launch_render_fwd(const TsPlanImpl* p, const TsWs& w, float* color, float* depth, float* alpha,
                                 float* normal, cudaStream_t s) {
  RenderArgs a = base_args(p, w);
  a.color = color;
  a.depth = depth;
  a.alpha = alpha;
  a.normal = normal;
  return dispatch(true, p, a, s);
}

cudaError_t ts_launch_render_bwd(const TsPlanImpl* p, const TsWs& w, const float* dC, const float* dD,
                                 const float* dA, const float* dN, cudaStream_t s) {
  RenderArgs a = base_args(p, w);
  a.dC = dC;
  a.dD = dD;
  a.dA = dA;
  a.dN = dN;
  return dispatch(false, p, a, s);
}

cudaError_t ts_launch_render_step(const TsPlanImpl* p, const TsWs& w, const float* tgt_color, const float* tgt_depth,
                                  float lambda_dep, float* color, float* depth, float* alpha, float* loss, float* dC,
                                  float* dD, cudaStream_t s) {
  RenderArgs a = base_args(p, w);
  a.color = color;
  a.depth = depth;
  a.alpha = alpha;
  a.tC = tgt_color;
  a.tD = tgt_depth;
  a.lambda_dep = lambda_dep;
  a.dC_out = dC;
  a.dD_out = dD;
  a.tloss = w.tloss;
  const int tw = p->prm.tile_w, th = p->prm.tile_h;
  const bool persist = (p->prm.flags & TS_FLAG_PERSISTENT) != 0;
  cudaError_t e;
  if (tw == 16 && th == 8) e = launch_step<16, 8>(persist, a, s);
  else if (tw == 16 && th == 16) e = launch_step<16, 16>(persist, a, s);
  else if (tw == 8 && th == 8) e = launch_step<8, 8>(persist, a, s);
  else if (tw == 32 && th == 8) e = launch_step<32, 8>(persist, a, s);
  else if (tw == 16 && th == 32) e = launch_step<16, 32>(persist, a, s);
  else if (tw == 32 && th == 16) e = launch_step<32, 16>(persist, a, s);
  else e = cudaErrorInvalidValue;
  if (e != cudaSuccess) return e;
  k_loss_tiles<<<p->V, 256, 0, s>>>(w.views, w.tloss, lambda_dep, loss);
  return cudaGetLastError();
}
