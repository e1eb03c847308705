// Transposed first product of Algorithm 2 (A1^T F1) from register tiles of
// output rows, with A1 stored for a fundamental set of sensor columns of the
// aperture's symmetry group.
//
// Tiles.  A gather-per-FMA product is bound by the L1 data pipe (one dense
// row fetched per entry).  A circle crossing a pixel usually crosses its
// neighbour too, so a warp owns a 2 x 2 tile of pixels (rows of A1^T) and
// walks the union of its rows' gathered rows: one record per gathered row,
// with four weights (zero, and skipped, where a pixel does not use it, so an
// infinite or NaN sample reaches only the pixels that do).  At 256^3 a record
// serves 2.0 entries on average.  (The same idea for A1 itself, 4
// consecutive radii of one column per warp, measured slower than the CSR
// row kernel: there the rows of a block already share their gathered pixels
// through L1, and the tiles lose that sharing.)
//
// Symmetry (Sec. 2's columns are equispaced around the axis).  Let
// rot(ix, iy) = (ms-1-iy, ix) (a quarter turn of the pixel grid) and
// D(ix, iy) = (iy, ix) (the mirror across the diagonal).  With q = n_phi/4,
// phi0 = 0 and the whole aperture, the quarter turn takes sensor column j to
// j + q and the mirror takes column t to q - t, and both map circles to
// circles, so for g = rot^s D^m
//   A1[(C_g(j), l), P_g(p)] = A1[(j, l), p],  C_g(j) = s q + (m ? q - j : j),
// P_g = rot^s after D^m.  Mode 2 (8-fold) stores the columns j = 0 .. q/2:
// column J = s q + t is stored column t (m = 0) for t <= q/2 and q - t
// (m = 1) otherwise.  Columns 0 and q/2 are fixed by a mirror, so in the
// transpose they count once per quarter turn, not twice: their records sit
// apart (list B) and only the unmirrored passes read them.  Mode 1 (4-fold)
// stores j < q; mode 0 stores every column.
//
// A1^T tile T: for each group element g, the stored tile Q = P_g^-1(T) (rot
// and D map aligned 2 x 2 tiles to aligned 2 x 2 tiles when ms is even),
// whose records (j, l), sorted by (list, j, l), gather row (C_g(j), l) of F1
// into the output pixel P_g(q_sigma) of T: a fixed permutation of the
// tile's four slots per g (with few slabs the warp's groups of lanes share
// the elements, k_a1t_split).  With every column stored (one pass) each pixel
// sums its entries in the CSR order of A1^T, ascending (j, l).  Every output
// row is one warp's FP32 sum, in a fixed order: no atomics, deterministic.
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "devutil.cuh"

namespace {

#ifdef SRT_CHECKS
__device__ unsigned long long g_viol;  // gathered rows outside their operand
#endif

// Records per group of the main loop; two groups alternate, as in tiles.cu.
// At 256^3 the L1 data pipe is 75% busy; what holds the rest of the time was
// not found (eight copies of the loop share 128 registers and reload 120 bytes
// of spills).  Blocks of four warps at 128 registers with the FMAs of a record
// under the test that the slot's weight is not zero (see tiles.cu) take A1^T
// from 1.391 to 1.263 ms there, and groups of five where 128 columns leave the registers free
// from 434 to 297 us at 128^3 (groups of three 346, four 328, six 307).
template <int CH>
constexpr int kH = CH == 2 ? 3 : 5;

template <typename W>
__device__ __forceinline__ void rec_w(const W* p, float w[4]);
template <>
__device__ __forceinline__ void rec_w<float4>(const float4* p, float w[4]) {
  const float4 v = __ldg(p);
  w[0] = v.x;
  w[1] = v.y;
  w[2] = v.z;
  w[3] = v.w;
}
template <>
__device__ __forceinline__ void rec_w<uint2>(const uint2* p, float w[4]) {
  const uint2 v = __ldg(p);  // four BF16 weights, w[0] in the low half of .x
  w[0] = __uint_as_float(v.x << 16);
  w[1] = __uint_as_float(v.x & 0xffff0000u);
  w[2] = __uint_as_float(v.y << 16);
  w[3] = __uint_as_float(v.y & 0xffff0000u);
}

__device__ __forceinline__ void fma4(float2 (&a)[2], float w, const float4& xv) {
  const float2 ww = make_float2(w, w);
  a[0] = __ffma2_rn(ww, make_float2(xv.x, xv.y), a[0]);
  a[1] = __ffma2_rn(ww, make_float2(xv.z, xv.w), a[1]);
}

// Slot (dx*2 + dy) of the stored tile's pixel -> slot of its image under
// g = rot^s D^m (rot: (dx, dy) -> (1-dy, dx); D: (dx, dy) -> (dy, dx)).
__host__ __device__ constexpr int sym_slot(int s, int m, int sg) {
  int dx = sg >> 1, dy = sg & 1;
  if (m) {
    const int t = dx;
    dx = dy;
    dy = t;
  }
  for (int k = 0; k < (s & 3); ++k) {
    const int t = dx;
    dx = 1 - dy;
    dy = t;
  }
  return dx * 2 + dy;
}

struct A1Args {
  const int32_t* ptr;  // record ranges (see the kernels)
  const int32_t* key;  // (j << 16 | l)
  int mode, q, ms, n_phi, n_ell, ntx;
  int G, R, S;         // block order
  int g0, g1;          // tile rows [g0, g1) (pixel rows 2 g0 .. 2 g1 - 1)
  int xrows;           // rows of the gathered operand (debug-build checks)
};


// Blocks of four warps own 2 x 2 tiles (4 x 4 pixels), of eight 4 x 2; which,
// launch_a1t says.
template <int NW>
constexpr int kTG = NW == 8 ? 4 : 2;

// Warp -> (group, index) as in spmm.cu's block_row: G groups of R, a block
// owning kTG groups x NW / kTG consecutive indices, chunk-major, or S x S
// super-tiles (S > 0).
template <int NW>
__device__ __forceinline__ bool warp_tile(const A1Args& A, int* g, int* i) {
  const int w = threadIdx.x >> 5;
  constexpr int TG = kTG<NW>, TI = NW / TG;
  if (A.S > 0) {
    const int per_row = A.S / TG, bpt = per_row * (A.S / TI);
    const int st = blockIdx.x / bpt, r = blockIdx.x - st * bpt;
    const int nsx = (A.G + A.S - 1) / A.S, sx = st % nsx, sy = st / nsx;
    const int tx = r % per_row, ty = r / per_row;
    *g = sx * A.S + tx * TG + w / TI;
    *i = sy * A.S + ty * TI + w % TI;
  } else {
    const int tiles = (A.G + TG - 1) / TG;
    const int c = blockIdx.x / tiles, t = blockIdx.x - c * tiles;
    *g = t * TG + w / TI;
    *i = c * TI + w % TI;
  }
  return *g < A.G && *i < A.R;
}

// ----------------------------------------------------------------- A1^T
// One group element's pass over the stored tile's records: list A
// (ptr[2t] .. ptr[2t+1]) always, list B (.. ptr[2t+2]) for unmirrored g.
template <typename W, int CH, int PS, int PM>
__device__ __forceinline__ void a1t_pass(const A1Args& A, const W* __restrict__ wt, int ta,
                                         int tb, const float* x0, int ldx, const bool (&in)[CH],
                                         float2 (&acc)[4][CH][2]) {
  int qa = ta, qb = tb;
#pragma unroll
  for (int k = 0; k < PS; ++k) {  // rot^-1 on tiles: (a, b) -> (b, ntx-1-a)
    const int t = qa;
    qa = qb;
    qb = A.ntx - 1 - t;
  }
  if (PM) {
    const int t = qa;
    qa = qb;
    qb = t;
  }
  const int64_t t2 = 2 * ((int64_t)qa * A.ntx + qb);
  const int e0 = A.ptr[t2], e1 = A.ptr[t2 + (PM ? 1 : 2)];
  // The stored tile's records are read by its 8 images' warps, far apart in
  // the launch, so they are mostly fetched from DRAM: request the pass's
  // lines at once rather than one miss per line as the walk reaches them
  // (A1^T 1.407 -> 1.374 ms at 256^3; the next pass's lines instead: 1.391,
  // every pass's at the kernel's start: 1.415).
  if (e1 > e0) {
    srt_prefetch_l2(A.key + e0, A.key + e1);
    srt_prefetch_l2(wt + e0, wt + e1);
  }
  const int base = PM ? (PS + 1) * A.q : PS * A.q;
  auto row_of = [&](int k) {  // gathered row (C_g(j), l)
    const int j = k >> 16, l = k & 0xffff;
    int J = PM ? base - j : base + j;
    if (J >= A.n_phi) J -= A.n_phi;
    int row = J * A.n_ell + l;
    SRT_CHECK_GATHER(0, row, A.xrows, g_viol);
    return row;
  };
  constexpr int H = kH<CH>;
  int oA[H], oB[H];
  float wA[H][4], wB[H][4];
  float4 vA[H][CH], vB[H][CH];
  // group of records eb .. eb + H - 1: gathered rows, then weights
  auto load = [&](int eb, int (&o)[H], float (&w)[H][4], float4 (&v)[H][CH]) {
#pragma unroll
    for (int u = 0; u < H; ++u) o[u] = row_of(__ldg(A.key + eb + u));
#pragma unroll
    for (int u = 0; u < H; ++u) {
      const float* xr = x0 + (int64_t)o[u] * ldx;
#pragma unroll
      for (int c = 0; c < CH; ++c)
        if (in[c]) v[u][c] = srt_ld_keep(xr + c * 128);
    }
#pragma unroll
    for (int u = 0; u < H; ++u) rec_w<W>(wt + eb + u, w[u]);
  };
  auto comp = [&](float (&w)[H][4], float4 (&v)[H][CH]) {
#pragma unroll
    for (int u = 0; u < H; ++u)
#pragma unroll
      for (int c = 0; c < CH; ++c)
#pragma unroll
        for (int sg = 0; sg < 4; ++sg)
          if (w[u][sg] != 0.f) fma4(acc[sym_slot(PS, PM, sg)][c], w[u][sg], v[u][c]);
  };
  int e = e0;
  const int groups = (e1 - e0) / H;
  if (groups >= 2) {  // two groups alternate: one's gathers fly while the other computes
    load(e, oA, wA, vA);
    int gi = 1;
#pragma unroll 1
    for (; gi + 1 < groups; gi += 2) {
      load(e + gi * H, oB, wB, vB);
      comp(wA, vA);
      load(e + (gi + 1) * H, oA, wA, vA);
      comp(wB, vB);
    }
    if (gi < groups) {
      load(e + gi * H, oB, wB, vB);
      comp(wA, vA);
      comp(wB, vB);
    } else {
      comp(wA, vA);
    }
    e += groups * H;
  }
#pragma unroll 1
  for (; e < e1; ++e) {
    const float* xr = x0 + (int64_t)row_of(__ldg(A.key + e)) * ldx;
    float w[4];
    rec_w<W>(wt + e, w);
    float4 v[CH];
#pragma unroll
    for (int c = 0; c < CH; ++c)
      if (in[c]) v[c] = srt_ld_keep(xr + c * 128);
#pragma unroll
    for (int sg = 0; sg < 4; ++sg)
      if (w[sg] != 0.f) {
#pragma unroll
        for (int c = 0; c < CH; ++c) fma4(acc[sym_slot(PS, PM, sg)][c], w[sg], v[c]);
      }
  }
}

// f[b][p][k] = sum_(J,l) A1[(J, l), p] F1[b][(J, l)][k] for the 2 x 2 pixel
// tile (ta, tb) with ta in [g0, g1); y points at pixel row 2 g0.
template <typename W, int CH, int NW>
__global__ void __launch_bounds__(NW * 32, 16 / NW)
    k_a1t_tile(A1Args A, const W* __restrict__ wt, const float* __restrict__ x, int ldx, int64_t bsx,
               float* __restrict__ y, int ldy, int64_t bsy, int ncols) {
  srt_in_order();
  const int lane = threadIdx.x & 31;
  int ga, tb;
  if (!warp_tile<NW>(A, &ga, &tb)) return;
  const int ta = A.g0 + ga;
  const int n0 = blockIdx.y * (128 * CH) + lane * 4;
  const float* x0 = x + blockIdx.z * bsx + n0;
  bool in[CH];
#pragma unroll
  for (int c = 0; c < CH; ++c) in[c] = n0 + c * 128 < ncols;
  float2 acc[4][CH][2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int c = 0; c < CH; ++c) acc[i][c][0] = acc[i][c][1] = make_float2(0.f, 0.f);
  a1t_pass<W, CH, 0, 0>(A, wt, ta, tb, x0, ldx, in, acc);
  if (A.mode == 2) a1t_pass<W, CH, 0, 1>(A, wt, ta, tb, x0, ldx, in, acc);
  if (A.mode) {
    a1t_pass<W, CH, 1, 0>(A, wt, ta, tb, x0, ldx, in, acc);
    if (A.mode == 2) a1t_pass<W, CH, 1, 1>(A, wt, ta, tb, x0, ldx, in, acc);
    a1t_pass<W, CH, 2, 0>(A, wt, ta, tb, x0, ldx, in, acc);
    if (A.mode == 2) a1t_pass<W, CH, 2, 1>(A, wt, ta, tb, x0, ldx, in, acc);
    a1t_pass<W, CH, 3, 0>(A, wt, ta, tb, x0, ldx, in, acc);
    if (A.mode == 2) a1t_pass<W, CH, 3, 1>(A, wt, ta, tb, x0, ldx, in, acc);
  }
  float* y0 = y + blockIdx.z * bsy;
#pragma unroll
  for (int sg = 0; sg < 4; ++sg) {
    const int ix = 2 * ga + (sg >> 1), iy = 2 * tb + (sg & 1);  // ix relative to row 2 g0
    float* yr = y0 + ((int64_t)ix * A.ms + iy) * ldy;
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      const int n = n0 + c * 128;
      if (n < ncols)
        *reinterpret_cast<float4*>(yr + n) =
            make_float4(acc[sg][c][0].x, acc[sg][c][0].y, acc[sg][c][1].x, acc[sg][c][1].y);
    }
  }
}

// One FP32 weight of a record (slot q).
__device__ __forceinline__ float rec_w1(const float4* p, int q) {
  return __ldg(reinterpret_cast<const float*>(p) + q);
}
__device__ __forceinline__ float rec_w1(const uint2* p, int q) {
  return srt_bf16_to_f32(__ldg(reinterpret_cast<const uint16_t*>(p) + q));
}

// A1^T with at most 64 slabs from a symmetric form: GL lanes cover the width
// and the warp's 32 / GL groups of lanes take the group elements of the same
// tile between them (the 8-fold form's 8 passes, the quarter turns' 4), so
// no lane idles and a tile's chain of gathers is 32 / GL times shorter.  Each
// group permutes a record's weights as it loads them, four 4-byte loads
// that cost the L1 data pipe no more than one 16-byte load, and the groups'
// sums are added at the end.  us, a whole warp to a pass before: 16^3 22.5 ->
// 10.2 (GL = 4), 48^3 38.9 -> 26.6, 64^3 63.5 -> 45.1 (GL = 16; GL = 8 with two
// chunks 45.1, 28.7 at 48^3).  With 96 or 128 slabs two chunks a lane leave
// too few registers for groups of five: 201 against 166 and 350 against 297
// us, so wider volumes keep a warp to a pass.
template <typename W, int CH, int GL>
__global__ void __launch_bounds__(128, 4)
    k_a1t_split(A1Args A, const W* __restrict__ wt, const float* __restrict__ x, int ldx,
                int64_t bsx, float* __restrict__ y, int ldy, int64_t bsy, int ncols) {
  srt_in_order();
  constexpr int NS = 32 / GL, H = kH<CH>;
  const int lane = threadIdx.x & 31, sub = lane / GL, sl = lane % GL;
  int ga, tb;
  if (!warp_tile<4>(A, &ga, &tb)) return;
  const int ta = A.g0 + ga;
  const int n0 = sl * 4;
  const float* x0 = x + blockIdx.z * bsx + n0;
  bool in[CH];
#pragma unroll
  for (int c = 0; c < CH; ++c) in[c] = n0 + c * (4 * GL) < ncols;
  float2 acc[4][CH][2];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int c = 0; c < CH; ++c) acc[i][c][0] = acc[i][c][1] = make_float2(0.f, 0.f);
  const int np = A.mode == 2 ? 8 : 4;
#pragma unroll 1
  for (int pi = 0; pi < np; pi += NS) {
    // this group's element g = rot^ps D^pm, its stored tile and its column map
    const int pg = pi + sub, ps = pg & 3, pm = pg >> 2;
    const int n = A.ntx - 1;
    int qa = ps == 0 ? ta : ps == 1 ? tb : ps == 2 ? n - ta : n - tb;
    int qb = ps == 0 ? tb : ps == 1 ? n - ta : ps == 2 ? n - tb : ta;
    if (pm) {
      const int t = qa;
      qa = qb;
      qb = t;
    }
    const int64_t t2 = 2 * ((int64_t)qa * A.ntx + qb);
    const int e0 = A.ptr[t2], e1 = pg < np ? A.ptr[t2 + (pm ? 1 : 2)] : e0;
    const int cnt = e1 - e0, most = (int)__reduce_max_sync(0xffffffffu, (unsigned)cnt);
    const int base = (ps + pm) * A.q, sign = pm ? -1 : 1;
    int from[4];  // stored slot that lands in slot d
#pragma unroll
    for (int sg = 0; sg < 4; ++sg) from[sg] = 0;
#pragma unroll
    for (int sg = 0; sg < 4; ++sg) {
      const int d = sym_slot(ps, pm, sg);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k == d) from[k] = sg;
    }
    {  // the pass's records from L2 at once, as in a1t_pass
      const char* kb = reinterpret_cast<const char*>(A.key + e0);
      for (int b = sl * 128; b < cnt * 4; b += GL * 128)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(kb + b));
      const char* wb = reinterpret_cast<const char*>(wt + e0);
      for (int b = sl * 128; b < cnt * (int)sizeof(W); b += GL * 128)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(wb + b));
    }
    float wA[H][4], wB[H][4];
    float4 vA[H][CH], vB[H][CH];
    // records eb .. eb + H - 1 of each group's own list; past its end the
    // last record again, with zero weights
    auto load = [&](int eb, float (&w)[H][4], float4 (&v)[H][CH]) {
      int o[H];
#pragma unroll
      for (int u = 0; u < H; ++u) {
        const int k = __ldg(A.key + max(0, e0 + min(eb + u, cnt - 1)));
        int J = base + sign * (k >> 16);
        if (J >= A.n_phi) J -= A.n_phi;
        o[u] = J * A.n_ell + (k & 0xffff);
        SRT_CHECK_GATHER(0, o[u], A.xrows, g_viol);
      }
#pragma unroll
      for (int u = 0; u < H; ++u) {
        const float* xr = x0 + (int64_t)o[u] * ldx;
#pragma unroll
        for (int c = 0; c < CH; ++c)
          if (in[c]) v[u][c] = srt_ld_keep(xr + c * (4 * GL));
      }
#pragma unroll
      for (int u = 0; u < H; ++u)
#pragma unroll
        for (int d = 0; d < 4; ++d)
          w[u][d] = eb + u < cnt ? rec_w1(wt + e0 + eb + u, from[d]) : 0.f;
    };
    auto comp = [&](float (&w)[H][4], float4 (&v)[H][CH]) {
#pragma unroll
      for (int u = 0; u < H; ++u)
#pragma unroll
        for (int c = 0; c < CH; ++c)
#pragma unroll
          for (int d = 0; d < 4; ++d)
            if (w[u][d] != 0.f) fma4(acc[d][c], w[u][d], v[u][c]);
    };
    if (most > 0) {
      load(0, wA, vA);
#pragma unroll 1
      for (int r = 0; r < most; r += 2 * H) {
        load(r + H, wB, vB);
        comp(wA, vA);
        load(r + 2 * H, wA, vA);
        comp(wB, vB);
      }
    }
  }
  // the groups' sums, added in a fixed tree
#pragma unroll
  for (int o = GL; o < 32; o <<= 1)
#pragma unroll
    for (int d = 0; d < 4; ++d)
#pragma unroll
      for (int c = 0; c < CH; ++c)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          acc[d][c][h].x += __shfl_xor_sync(0xffffffffu, acc[d][c][h].x, o);
          acc[d][c][h].y += __shfl_xor_sync(0xffffffffu, acc[d][c][h].y, o);
        }
  float* y0 = y + blockIdx.z * bsy;
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    if (d % NS != sub) continue;  // one group stores each slot
    const int ix = 2 * ga + (d >> 1), iy = 2 * tb + (d & 1);  // ix relative to row 2 g0
    float* yr = y0 + ((int64_t)ix * A.ms + iy) * ldy;
#pragma unroll
    for (int c = 0; c < CH; ++c)
      if (in[c])
        *reinterpret_cast<float4*>(yr + n0 + c * (4 * GL)) =
            make_float4(acc[d][c][0].x, acc[d][c][0].y, acc[d][c][1].x, acc[d][c][1].y);
  }
}

// ------------------------------------------------------------ records
struct TEnt {
  int64_t key;  // list << 40 | j << 16 | l
  int32_t slot;
  int64_t src;
};

template <typename T>
int upload(const std::vector<T>& h, T** d, int64_t* bytes) {
  SRT_TRY(srt_dmalloc(d, (int64_t)h.size(), bytes));
  if (!h.empty())
    SRT_CUDA_TRY(cudaMemcpy(*d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice));
  return SRT_OK;
}

}  // namespace

void srt_a1tiles_free(SrtA1Tiles* t) {
  cudaFree(t->aptr);
  cudaFree(t->akey);
  cudaFree(t->aw32);
  cudaFree(t->aw16);
  *t = SrtA1Tiles();
}

int srt_build_a1tiles(srt_plan_s* plan, int64_t* bytes) {
  const srt_geometry& g = plan->g;
  const SrtCsr& a = plan->a1;
  const int ms = g.ms, ne = g.n_ell, q = g.n_phi / 4;
  const int mode = plan->a1_rot;
  if (ms % 2 || ms >= (1 << 15) || ne >= (1 << 16)) return SRT_ERR_ARG;
  const int64_t ns = a.nnz;
  std::vector<int32_t> rp(a.rows + 1), cl(ns);
  std::vector<float> v32(a.v32 ? ns : 0);
  std::vector<uint16_t> v16(a.v16 ? ns : 0);
  SRT_CUDA_TRY(cudaMemcpy(rp.data(), a.rowptr, rp.size() * 4, cudaMemcpyDeviceToHost));
  if (ns) {
    SRT_CUDA_TRY(cudaMemcpy(cl.data(), a.col, ns * 4, cudaMemcpyDeviceToHost));
    if (a.v32) SRT_CUDA_TRY(cudaMemcpy(v32.data(), a.v32, ns * 4, cudaMemcpyDeviceToHost));
    if (a.v16) SRT_CUDA_TRY(cudaMemcpy(v16.data(), a.v16, ns * 2, cudaMemcpyDeviceToHost));
  }
  SrtA1Tiles& t = plan->a1tl;
  t.ntx = ms / 2;
  // A1^T: per 2 x 2 pixel tile, records (j, l) sorted by (list, j, l); list
  // B holds the mirror-fixed stored columns 0 and q/2 of the 8-fold form
  {
    const int64_t ntiles = (int64_t)t.ntx * t.ntx;
    std::vector<int64_t> cnt(ntiles + 1, 0);
    for (int64_t row = 0; row < a.rows; ++row)
      for (int64_t e = rp[row]; e < rp[row + 1]; ++e) {
        const int ix = cl[e] / ms, iy = cl[e] % ms;
        ++cnt[(int64_t)(ix / 2) * t.ntx + iy / 2 + 1];
      }
    for (int64_t i = 0; i < ntiles; ++i) cnt[i + 1] += cnt[i];
    std::vector<TEnt> ent(ns);
    std::vector<int64_t> at(cnt.begin(), cnt.end() - 1);
    for (int64_t row = 0; row < a.rows; ++row) {
      const int j = (int)(row / ne), l = (int)(row % ne);
      const int64_t list = (mode == 2 && (j == 0 || 2 * j == q)) ? 1 : 0;
      for (int64_t e = rp[row]; e < rp[row + 1]; ++e) {
        const int ix = cl[e] / ms, iy = cl[e] % ms;
        const int64_t tt = (int64_t)(ix / 2) * t.ntx + iy / 2;
        ent[at[tt]++] = TEnt{list << 40 | (int64_t)j << 16 | l, (ix & 1) * 2 + (iy & 1), e};
      }
    }
    std::vector<int32_t> ptr(2 * ntiles + 1), key;
    std::vector<float> w32;
    std::vector<uint16_t> w16;
    for (int64_t tt = 0; tt < ntiles; ++tt) {
      auto b0 = ent.begin() + cnt[tt], b1 = ent.begin() + cnt[tt + 1];
      std::stable_sort(b0, b1, [](const TEnt& x, const TEnt& y) { return x.key < y.key; });
      ptr[2 * tt] = (int32_t)key.size();
      ptr[2 * tt + 1] = -1;
      for (auto b = b0; b != b1;) {
        if ((b->key >> 40) && ptr[2 * tt + 1] < 0) ptr[2 * tt + 1] = (int32_t)key.size();
        float f[4] = {0.f, 0.f, 0.f, 0.f};
        uint16_t h[4] = {0, 0, 0, 0};
        auto c = b;
        for (; c != b1 && c->key == b->key; ++c) {
          if (!v32.empty()) f[c->slot] = v32[c->src];
          if (!v16.empty()) h[c->slot] = v16[c->src];
        }
        key.push_back((int32_t)(b->key & 0xffffffffll));
        if (!v32.empty()) w32.insert(w32.end(), f, f + 4);
        if (!v16.empty()) w16.insert(w16.end(), h, h + 4);
        b = c;
      }
      if (ptr[2 * tt + 1] < 0) ptr[2 * tt + 1] = (int32_t)key.size();
    }
    ptr.back() = (int32_t)key.size();
    if (key.size() >= ((size_t)1 << 31)) return SRT_ERR_GEOMETRY;
    t.na = (int64_t)key.size();
    SRT_TRY(upload(ptr, &t.aptr, bytes));
    SRT_TRY(upload(key, &t.akey, bytes));
    if (!w32.empty()) SRT_TRY(upload(w32, &t.aw32, bytes));
    if (!w16.empty()) SRT_TRY(upload(w16, &t.aw16, bytes));
  }
  return SRT_OK;
}

namespace {

// Blocks of the launch, NW warps each.
template <int NW>
int64_t a1t_blocks(const A1Args& A) {
  constexpr int TG = kTG<NW>, TI = NW / TG;
  if (A.S > 0)
    return (int64_t)((A.G + A.S - 1) / A.S) * ((A.R + A.S - 1) / A.S) * (A.S / TG) * (A.S / TI);
  return (int64_t)((A.R + TI - 1) / TI) * ((A.G + TG - 1) / TG);
}

template <typename W>
int launch_a1t(const A1Args& A, const W* w, const float* x, int64_t ldx, int64_t bsx, float* y,
               int64_t ldy, int64_t bsy, int ncols, int batch, cudaStream_t st) {
  const int CH = ncols > 128 ? 2 : 1;
  // More than 128 slabs, blocks of eight warps where the tiles' lists are short
  // or the launch is long: with four, the later parts of a long launch are
  // slower, and with few sensor columns the first as well (us, four and eight
  // warps: 256^3, 256 columns, 768 radii, batch 2 2576 and 2488, 4 5460 and 4902, 8
  // 11305 and 9754; 512^3 11787 and 9832; 384^2 x 256 3968 and 3750; 512^2 x 192
  // 7523 and 6452; 1024 radii, 64 columns, batch 1 481 and 453, 4 1973 and 1705; 4
  // x 192^3, 128 columns 2061 and 1832).  Fewer blocks: 2 x 192^3 1854 and 1893, 4 x
  // 64^2 x 160 234 and 254, 320^2 x 256 2615 and 2668, 256^3 1263 and 1290, 160^3 682
  // and 717, 128 columns of 224^2 x 192 in BF16 707 and 719; one chunk of slabs:
  // 128^3 303 and 322, 8 x 96^3 1207 and 1218.
  const int over = (ncols + 128 * CH - 1) / (128 * CH);
  const bool big = CH == 2 && a1t_blocks<8>(A) * over * batch >= (A.n_phi <= 64 ? 1024 : 4096);
  const int64_t gx = big ? a1t_blocks<8>(A) : a1t_blocks<4>(A);
  if (gx > 0x7fffffff || batch > 65535) return SRT_ERR_ARG;
  dim3 grid((unsigned)gx, over, batch);
#define SRT_A1T(K, NW)                                                                            \
  SRT_CUDA_TRY(srt_launch(3 * kSMs, K, grid, NW * 32, st, A, w, x, (int)ldx, bsx, y, (int)ldy, bsy, \
                          ncols))
  if (A.mode && ncols <= 64) {
    if (ncols <= 16 && A.mode == 2)  // 8 groups: one to each of the 8 passes
      SRT_A1T((k_a1t_split<W, 1, 4>), 4);
    else if (ncols <= 32)
      SRT_A1T((k_a1t_split<W, 1, 8>), 4);
    else
      SRT_A1T((k_a1t_split<W, 1, 16>), 4);
  } else if (big) {
    SRT_A1T((k_a1t_tile<W, 2, 8>), 8);
  } else if (CH == 2) {
    SRT_A1T((k_a1t_tile<W, 2, 4>), 4);
  } else {
    SRT_A1T((k_a1t_tile<W, 1, 4>), 4);
  }
#undef SRT_A1T
  SRT_CUDA_TRY(cudaGetLastError());
  return SRT_OK;
}

}  // namespace

int srt_a1tiles_apply(const srt_plan_s* plan, int g0, int g1, const float* x, int64_t ldx,
                      int64_t bsx, float* y, int64_t ldy, int64_t bsy, int ncols, int batch,
                      cudaStream_t st) {
  const srt_geometry& g = plan->g;
  const SrtA1Tiles& t = plan->a1tl;
  if (!t.aptr || ncols <= 0 || batch <= 0) return SRT_ERR_ARG;
  // float4 gathers and stores of 16-byte aligned rows
  if (ncols % 4 || ldx % 4 || ldy % 4 || bsx % 4 || bsy % 4 || (uintptr_t)x % 16 ||
      (uintptr_t)y % 16 || ldx > 0x7fffffff || ldy > 0x7fffffff)
    return SRT_ERR_ARG;
  if (g0 < 0 || g1 > t.ntx || g1 <= g0) return SRT_ERR_ARG;
  A1Args A{};
  A.ptr = t.aptr;
  A.key = t.akey;
  A.mode = plan->a1_rot;
  A.q = g.n_phi / 4;
  A.ms = g.ms;
  A.n_phi = g.n_phi;
  A.n_ell = g.n_ell;
  A.ntx = t.ntx;
  A.xrows = srt_checked_rows((int64_t)g.n_phi * g.n_ell);
  // tiles (ta, tb), ta in [g0, g1): blocks of 2 x 2 tiles (4 x 4 pixels)
  // walked in 16 x 16 tile (32 x 32 pixel) super-tiles where they fit, so
  // the rows gathered at any time belong to a compact patch (256^3: blocks of
  // 2 x 2 tiles 1.263 ms, of 4 x 1 1.266; 32 x 32 tiles 1.265, none 1.256, but
  // none 1.703 against 1.670 with 1024 radii; blocks of 4 x 2 tiles 1.290)
  A.g0 = g0;
  A.g1 = g1;
  A.G = g1 - g0;
  A.R = t.ntx;
  A.S = (A.G % 16 == 0 && A.R % 16 == 0) ? 16 : 0;
  if (g.weight_dtype == SRT_BF16) {
    const uint2* w = reinterpret_cast<const uint2*>(t.aw16);
    if (!w) return SRT_ERR_ARG;
    return launch_a1t<uint2>(A, w, x, ldx, bsx, y, ldy, bsy, ncols, batch, st);
  }
  const float4* w = reinterpret_cast<const float4*>(t.aw32);
  if (!w) return SRT_ERR_ARG;
  return launch_a1t<float4>(A, w, x, ldx, bsx, y, ldy, bsy, ncols, batch, st);
}

long long srt_checks_take_a1tiles() {
#ifdef SRT_CHECKS
  unsigned long long v = 0, z = 0;
  if (cudaMemcpyFromSymbol(&v, g_viol, sizeof(v)) != cudaSuccess) return -1;
  if (cudaMemcpyToSymbol(g_viol, &z, sizeof(z)) != cudaSuccess) return -1;
  return (long long)v;
#else
  return 0;
#endif
}
