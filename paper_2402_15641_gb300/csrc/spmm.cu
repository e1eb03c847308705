// Sparse-times-dense products of Algorithm 1 (A1 F, A2 Y) and Algorithm 2
// (A2^T Y, A1^T F') of the paper, in gather form: every output row is owned by
// one group of lanes, so no atomics are used and results are deterministic.
//
// y[b][r][n] = sum_{e in row r} A[e] * x[b][col[e]][n],  n < ncols.
// A group of lanes owns a row and its lanes consecutive dense columns, as
// many rows to a warp as the width leaves room for; a row's (column, value)
// pairs are loaded coalesced, staged in shared memory and read back one by
// one.  Entries are FP32 or BF16; accumulation is FP32.
//
// A1 by rotation (SrtRot): with n_phi a multiple of 4, sensor column
// j + n_phi/4 sees the image turned by 90 degrees about the axis, so
//   A1[(j + s n_phi/4, l), rot^s(p)] = A1[(j, l), p],
//   rot(ix, iy) = (ms-1-iy, ix),
// and only the rows of the first n_phi/4 columns are stored.  Mode 1 (A1):
// output row (j, l) walks stored row (j mod n_phi/4, l) and gathers pixel
// rot^s(p).  Mode 2 (A1^T): output row p walks, for s = 0..3, stored row
// rot^-s(p) of the stored transpose and gathers row (j + s n_phi/4, l): the
// same terms in the same order (ascending j, then l) as the full transpose.
#include "common.cuh"

namespace {

constexpr unsigned FULL = 0xffffffffu;
#ifdef SRT_CHECKS
__device__ unsigned long long g_viol;  // gathered rows outside their operand
#endif

template <typename V>
__device__ __forceinline__ float wval(V v);
template <>
__device__ __forceinline__ float wval<float>(float v) {
  return v;
}
template <>
__device__ __forceinline__ float wval<uint16_t>(uint16_t v) {
  return srt_bf16_to_f32(v);
}

// Pixel p = ix*ms + iy turned s quarter turns: rot(ix, iy) = (ms-1-iy, ix).
// ix = floor(p / ms) as (p * magic) >> 40 with magic = ceil(2^40 / ms), exact
// for p < 2^24 and ms < 2^16 (the quotient's error stays below 1/ms).
__device__ __forceinline__ int rot_pixel(int p, int s, int ms, uint64_t magic, bool m = false) {
  int ix = (int)(((uint64_t)(uint32_t)p * magic) >> 40), iy = p - ix * ms;
  if (m) {  // mirror across the diagonal first: (ix, iy) -> (iy, ix)
    const int t = ix;
    ix = iy;
    iy = t;
    p = ix * ms + iy;
  }
  switch (s & 3) {
    case 0: return p;
    case 1: return (ms - 1 - iy) * ms + ix;
    case 2: return (ms - 1 - ix) * ms + (ms - 1 - iy);
    default: return iy * ms + (ms - 1 - ix);
  }
}

// Block-to-rows order.  Rows come in G groups of R rows (r = g*R + i).  With
// G > 0 a block owns a tile of TG groups x RPB/TG consecutive i, and
// consecutive blocks take the same chunk of i in consecutive group tiles
// (chunk-major): all groups advance through i together, so the dense rows
// gathered by concurrently running blocks stay within a narrow band of the
// operand (L2 reuse), while a block's rows gather overlapping rows (L1
// reuse).  With G = 0 blocks take consecutive rows.  With S > 0 the G x R
// grid is walked in S x S super-tiles (S dividing G and R), tiles row-major
// inside each: the dense rows gathered by concurrently running blocks then
// belong to a compact patch instead of a band across all G groups (A1^T:
// pixels, whose circles through a 64 x 64 patch cover ~40% of the operand
// instead of most of it).  w: this row's place among the block's RPB rows.
template <int RPB>
__device__ __forceinline__ int block_row(int G, int R, int TG, int S, int w) {
  if (G <= 0) return blockIdx.x * RPB + w;
  const int TI = RPB / TG;
  if (S > 0) {
    const int per_row = S / TG, bpt = per_row * (S / TI);
    const int st = blockIdx.x / bpt, r = blockIdx.x - st * bpt;
    const int nsx = G / S, sx = st % nsx, sy = st / nsx;
    const int tx = r % per_row, ty = r / per_row;
    const int g = sx * S + tx * TG + w / TI, i = sy * S + ty * TI + w % TI;
    return (sy < R / S) ? g * R + i : -1;
  }
  const int chunks = (R + TI - 1) / TI, tiles = (G + TG - 1) / TG;
  const int bid = blockIdx.x;
  const int c = bid / tiles, t = bid - c * tiles;
  if (c >= chunks) return -1;
  const int g = t * TG + w / TI, i = c * TI + w % TI;
  return (g < G && i < R) ? g * R + i : -1;
}

struct Rows {
  int rows, r0;    // output rows of this launch, first output row
  int G, R, TG;    // block order
  int S;           // super-tile side of the block order (0: chunk-major bands)
  SrtRot rot;
  uint64_t magic;  // ceil(2^40 / rot.ms)
  int xrows;       // rows of the gathered operand (debug-build checks)
  int64_t ldn;     // > 0: reshape P1 fused, stride of Y1''s rows
};

// VW consecutive dense columns of a gathered row.
template <int VW>
__device__ __forceinline__ void ld_cols(const float* p, float (&v)[VW]) {
  if constexpr (VW == 4) {
    const float4 q = srt_ld_keep(p);
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
    v[3] = q.w;
  } else if constexpr (VW == 2) {
    const float2 q = srt_ld2(p);
    v[0] = q.x;
    v[1] = q.y;
  } else {
    v[0] = srt_ld1(p);
  }
}

// Warps of a block (four where a warp holds four rows or more: 8 x 64^3 224 ->
// 217 us, 96^3 185 -> 180).
template <int GL>
constexpr int kBlockWarps = GL > 8 ? 8 : 4;

// A group of GL lanes owns an output row, 32 / GL rows to a warp; a lane
// owns VW consecutive columns of each of CH chunks of VW GL columns.  The
// row's entries are loaded EB at a time by the group's lanes, the gathered
// row remapped there (MODE 1: A1 row (j, l) from stored row (j mod q, l),
// pixels turned j / q times, mirrored first where the stored column is a
// mirror image; MODE 2: A1^T row p from stored rows rot^-s(p), s = 0..3,
// gathered rows shifted by s q n_ell; MODE 3 and 4: A2 rows (h, m) and A2^T
// rows (l, k) from the Toeplitz taps, ms = mz slabs and q = n_zs rings, see
// toeplitz.cu), and put in shared memory as (row, value) pairs that the group
// then reads back.
//
// What bounds it.  A gathered operand feeds one FMA, so the L1 data pipe
// (128 B a cycle per SM) is the limit at full width: 93% busy at 256^3,
// where each entry takes 8 cycles for its 1 KB and 2 for broadcasting row
// and value by two shuffles.  The pair read back by one 8-byte shared load
// takes 1 (a load that all lanes read from one shared address costs half of
// what it writes to registers): A1 at 256^3 1.578 -> 1.526 ms, and 1.480 with
// each batch's entries requested before the batch before is gathered (8 x
// 64^3 218 -> 212 us, 128^3 346 -> 340, 192^3 1088 -> 1072).  Below 128
// columns a whole warp to a row leaves lanes idle and spends the same loop
// on fewer columns; with GL lanes to a row (measured, one box, FP32 entries,
// a warp to a row before): 8 x 64^3 446 -> 212 us, 128^3 416 -> 340, 192^3
// 1180 -> 1072.  U gathers are requested before their FMAs: two gain 4% at
// 128^3, at 54 registers and 32 warps per SM in the kernel of 256 columns (48 to
// 72 registers in the others); four, at 72 to 99 registers and 16 to 24 warps,
// cost 6% at 256^3 but win where the launch cannot fill the GPU.
// A row's entries are summed in the same order in every variant.
//
// TR (MODE 1, GL = 32, blocks of 4 sensor columns x 2 radii, G = n_phi, R =
// n_ell): the reshape P1 in the epilogue.  The block's 8 rows go through
// shared memory, 128 slabs at a time, and are written as Y1'[(l, k)][b G +
// j], row stride ldn, 16 bytes (4 sensor columns) per radius and slab.
template <typename V, int VW, int CH, int GL, int MODE, bool TR, int U>
__global__ void __launch_bounds__(kBlockWarps<GL> * 32, MODE == 2 && U == 1 ? 6 : 0)
    k_rows(int rows, int r0, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
           const V* __restrict__ val, const float* __restrict__ x, int64_t ldx, int64_t bsx,
           float* __restrict__ y, int64_t ldy, int64_t bsy, int ncols, int G, int R, int TG, int S,
           int ms, int n_ell, int q, int mirror, uint64_t magic, int xrows, int64_t ldn) {
  srt_in_order();
  constexpr int NR = 32 / GL, EB = GL == 32 ? 32 : 16;
  // 384 or 512 columns to a warp: the pairs stay in registers and go round
  // by shuffles, whose share of the row's time is small there, and the
  // shared loads' extra registers cost more (A2 as CSR at 3072 columns 244
  // us, 268 through shared memory; A2^T 249, 316)
  constexpr bool SH = GL == 32 && VW == 4 && CH > 2;
  __shared__ int2 stage[SH ? 1 : kBlockWarps<GL>][NR][EB + (NR > 1 ? 1 : 0)];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, sub = lane / GL, sl = lane % GL;
  const int lr = block_row<kBlockWarps<GL> * NR>(G, R, TG, S, w * NR + sub);
  const bool mine = lr >= 0 && lr < rows;
  if (!TR && NR == 1 && !mine) return;  // (otherwise every lane reaches the barriers)
  const int row = r0 + (mine ? lr : 0);
  // (the taps' dense width holds the whole batch; two additions kept out of the
  // wide loop: 4 x 256^3 A2 row by row 10.68 -> 10.60 ms, 4 x 192^3 6.82 -> 6.77)
  if (!SH || MODE < 3) {
    x += blockIdx.z * bsx;
    if (!TR) y += blockIdx.z * bsy;
  }
  const int n0 = blockIdx.y * (VW * GL * CH) + sl * VW;
  float acc[CH][VW];
#pragma unroll
  for (int k = 0; k < CH; ++k)
#pragma unroll
    for (int i = 0; i < VW; ++i) acc[k][i] = 0.f;
  int t = 0, sr = row, ca = 0;
  bool mir = false;
  if (MODE == 3) {  // taps of row (h, m): offsets nz-1-h .. of radius m, row l mz + h + q-(nz-1)
    const int h = row / n_ell, m = row - h * n_ell;
    sr = m * (ms + q - 1) + q - 1 - h;
    ca = h - (q - 1);
  }
  if (MODE == 4) {  // taps of row (l, k): row (k + e - (mz-1)) n_ell + m
    const int l = row / ms, k = row - l * ms;
    sr = l * (ms + q - 1) + ms - 1 - k;
    ca = k - (ms - 1);
  }
  if (MODE == 1) {
    const int j = row / n_ell, l = row - j * n_ell;
    t = j / q;
    int js = j - t * q;
    if (mirror && 2 * js > q) {  // 8-fold form: stored column q - js, mirrored
      js = q - js;
      mir = true;
    }
    sr = js * n_ell + l;
  }
  // gathered row of a stored column (a tap's key: index | offset << 16)
  auto remap = [&](int c, int off) {
    if (MODE == 1) return rot_pixel(c, t, ms, magic, mir);
    if (MODE == 2) return c + off;
    if (MODE == 3) return (c & 0xffff) * ms + ca + (c >> 16);
    if (MODE == 4) return (ca + (c >> 16)) * n_ell + (c & 0xffff);
    return c;
  };
  int2* st = stage[SH ? 0 : w][sub];
#pragma unroll 1
  for (int s = 0; s < (MODE == 2 ? 4 : 1); ++s) {
    if (MODE == 2) sr = rot_pixel(row, 4 - s, ms, magic);
    const int off = MODE == 2 ? s * q * n_ell : 0;
    // (unsigned: a batch asks past its row's end, where 2^31 may be passed)
    const uint32_t e0 = rowptr[sr];
    const uint32_t e1 = mine ? rowptr[sr + (MODE == 3 ? ms : MODE == 4 ? q : 1)] : e0;
    // batches run in step over the warp's rows (an exhausted row idles); the
    // next batch's entries are requested before this one's gathers
    const int len = NR > 1 ? (int)__reduce_max_sync(FULL, e1 - e0) : (int)(e1 - e0);
    constexpr int KE = EB / GL;
    // (short rows of single columns have too few gathers to cover the request)
    constexpr bool PF = !SH && !(VW == 1 && U == 4);
    int nc[KE];
    V nv[KE];
    auto ask = [&](uint32_t eb) {
#pragma unroll
      for (int k = 0; k < KE; ++k)
        if (srt_in_row(eb + sl + k * GL, e1)) {
          nc[k] = col[eb + sl + k * GL];
          nv[k] = val[eb + sl + k * GL];
        }
    };
    if (PF) ask(e0);
#pragma unroll 1
    for (int b = 0; b < len; b += EB) {
      const uint32_t eb = e0 + b;
      if constexpr (SH) {
        int c = 0;
        float v = 0.f;
        if (srt_in_row(eb + lane, e1)) {
          c = col[eb + lane];
          c = remap(c, off);
          SRT_CHECK_GATHER(0, c, xrows, g_viol);
          v = wval<V>(val[eb + lane]);
        }
        const int cnt = min(32, (int)(e1 - eb));
#pragma unroll 1
        for (int i = 0; i < cnt; ++i) {
          const int ci = __shfl_sync(FULL, c, i);
          const float vi = __shfl_sync(FULL, v, i);
          const float* xr = x + (int64_t)ci * ldx;
#pragma unroll
          for (int k = 0; k < CH; ++k) {
            const int n = n0 + k * (VW * GL);
            if (n < ncols) {
              float xv[VW];
              ld_cols<VW>(xr + n, xv);
#pragma unroll
              for (int u = 0; u < VW; ++u) acc[k][u] = fmaf(vi, xv[u], acc[k][u]);
            }
          }
        }
        continue;
      }
      if (!PF) ask(eb);
#pragma unroll
      for (int k = 0; k < KE; ++k)
        if (srt_in_row(eb + sl + k * GL, e1)) {
          int c = nc[k];
          c = remap(c, off);
          SRT_CHECK_GATHER(0, c, xrows, g_viol);
          st[sl + k * GL] = make_int2(c, __float_as_int(wval<V>(nv[k])));
        }
      if (PF) ask(eb + EB);
      __syncwarp();
      const int cnt = min(EB, (int)(e1 - eb));
      int i = 0;
#pragma unroll 1
      for (; i + U <= cnt; i += U) {
        float xv[U][CH][VW], vi[U];
#pragma unroll
        for (int h = 0; h < U; ++h) {
          const int2 en = st[i + h];
          vi[h] = __int_as_float(en.y);
          const float* xr = x + (int64_t)en.x * ldx;
#pragma unroll
          for (int k = 0; k < CH; ++k)
            if (n0 + k * (VW * GL) < ncols) ld_cols<VW>(xr + n0 + k * (VW * GL), xv[h][k]);
        }
#pragma unroll
        for (int h = 0; h < U; ++h)
#pragma unroll
          for (int k = 0; k < CH; ++k)
            if (n0 + k * (VW * GL) < ncols) {
#pragma unroll
              for (int u = 0; u < VW; ++u) acc[k][u] = fmaf(vi[h], xv[h][k][u], acc[k][u]);
            }
      }
#pragma unroll 1
      for (; i < cnt; ++i) {
        const int2 en = st[i];
        const float vi = __int_as_float(en.y);
        const float* xr = x + (int64_t)en.x * ldx;
#pragma unroll
        for (int k = 0; k < CH; ++k) {
          const int n = n0 + k * (VW * GL);
          if (n < ncols) {
            float xv[VW];
            ld_cols<VW>(xr + n, xv);
#pragma unroll
            for (int u = 0; u < VW; ++u) acc[k][u] = fmaf(vi, xv[u], acc[k][u]);
          }
        }
      }
      __syncwarp();
    }
  }
  if (!TR) {
    if (!mine) return;
    float* yr = y + (int64_t)lr * ldy;
#pragma unroll
    for (int k = 0; k < CH; ++k) {
      const int n = n0 + k * (VW * GL);
      if (n >= ncols) continue;
      if constexpr (VW == 4)
        *reinterpret_cast<float4*>(yr + n) = make_float4(acc[k][0], acc[k][1], acc[k][2], acc[k][3]);
      else if constexpr (VW == 2)
        *reinterpret_cast<float2*>(yr + n) = make_float2(acc[k][0], acc[k][1]);
      else
        yr[n] = acc[k][0];
    }
    return;
  }
  // fused P1: Sb[w][n] holds row w = 2 jl + il (column j0 + jl, radius
  // l0 + il) of the block, 128 slabs n; a thread then writes one radius and
  // slab of the 4 columns
  if constexpr (TR) {
    __shared__ __align__(16) float Sb[8 * 128];
    const int tiles = (G + 3) / 4;
    const int c = blockIdx.x / tiles, tt = blockIdx.x - c * tiles;
    const int il = threadIdx.x >> 7, nl = threadIdx.x & 127;
    const int l = 2 * c + il;
    const int64_t cb = (int64_t)blockIdx.z * G + 4 * tt;  // column b G + j0 of Y1'
#pragma unroll
    for (int k = 0; k < CH; ++k) {
      if (k) __syncthreads();  // the previous chunk's reads are done
      *reinterpret_cast<float4*>(Sb + w * 128 + lane * 4) =
          make_float4(acc[k][0], acc[k][1], acc[k][2], acc[k][3]);
      __syncthreads();
      const int n = blockIdx.y * (128 * CH) + k * 128 + nl;
      if (l < R && n < ncols && 4 * tt < G)
        *reinterpret_cast<float4*>(y + ((int64_t)l * ncols + n) * ldn + cb) =
            make_float4(Sb[il * 128 + nl], Sb[(2 + il) * 128 + nl], Sb[(4 + il) * 128 + nl],
                        Sb[(6 + il) * 128 + nl]);
    }
  }
}

// Columns of one launch: VW GL CH per group, blockIdx.y over the groups' widths.
template <typename V, int VW, int CH, int GL, int MODE, int U, bool TR = false>
int launch_as(const SrtCsr& A, const V* val, const Rows& W, const float* x, int64_t ldx,
              int64_t bsx, float* y, int64_t ldy, int64_t bsy, int ncols, int batch,
              cudaStream_t st) {
  constexpr int RPB = kBlockWarps<GL> * (32 / GL);
  const int TI = RPB / W.TG;
  const int S = W.S > 0 && W.S % TI == 0 ? W.S : 0;
  const int64_t gx = S > 0     ? (int64_t)(W.G / S) * (W.R / S) * (S / W.TG) * (S / TI)
                     : W.G > 0 ? (int64_t)((W.G + W.TG - 1) / W.TG) * ((W.R + TI - 1) / TI)
                               : ((int64_t)W.rows + RPB - 1) / RPB;
  const int wide = VW * GL * CH;
  if (gx > 0x7fffffff || (ncols + wide - 1) / wide > 65535 || batch > 65535) return SRT_ERR_ARG;
  dim3 grid((unsigned)gx, (ncols + wide - 1) / wide, batch);
  const SrtRot& r = W.rot;
  SRT_CUDA_TRY(srt_launch(12 * kSMs, k_rows<V, VW, CH, GL, MODE, TR, U>, grid,
                          kBlockWarps<GL> * 32, st, W.rows, W.r0, A.rowptr, A.col, val, x, ldx, bsx,
                          y, ldy, bsy, ncols, W.G, W.R, W.TG, S, r.ms, r.n_ell, r.q, r.mirror,
                          W.magic, W.xrows, W.ldn));
  SRT_CUDA_TRY(cudaGetLastError());
  return SRT_OK;
}

template <typename V, int VW, int MODE, int U>
int launch_width(const SrtCsr& A, const V* val, const Rows& W, const float* x, int64_t ldx,
                 int64_t bsx, float* y, int64_t ldy, int64_t bsy, int ncols, int batch,
                 cudaStream_t st) {
#define SRT_ROWS(CH, GL) \
  return launch_as<V, VW, CH, GL, MODE, U>(A, val, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, st)
  const int n = (ncols + VW - 1) / VW;  // vectors of a row
  // wide rows stored as they are: each entry's reuse over 512 columns wins
  // over more warps (at 1024 columns 10.6 against 11.1 ms for A2 of 256^3 as CSR)
  if constexpr (U == 1) {
    if (n > 96) SRT_ROWS(4, 32);
    SRT_ROWS(3, 32);
  } else {
    // rows wider than a part in equal parts (64 float4 vectors, 128 narrower
    // ones: what a warp covers in two chunks or in up to four light ones);
    // then the narrowest group that covers a part
    constexpr int P = VW == 4 ? 64 : 128;
    const int parts = (n + P - 1) / P, m = (n + parts - 1) / parts;
    // Too few rows for 32 warps per SM even with a half warp to a row: the
    // time is one row's chain of gathers, and packing more rows into a warp
    // only lengthens it to the longest of them (A1 at 32^3, 8 vectors: 13.5 us
    // with a half warp to a row, 17.9 with four lanes; at 64^3, 44.5 against 41.2
    // the other way round, half warps losing).
    if (m <= 8 && (int64_t)W.rows * batch * parts <= (int64_t)2 * 32 * kSMs) SRT_ROWS(2, 16);
    if (m <= 8) SRT_ROWS(2, 4);
    if (m <= 16) SRT_ROWS(2, 8);
    if constexpr (VW == 4)
      if (m <= 24) SRT_ROWS(3, 8);
    if (m <= 32) SRT_ROWS(2, 16);
    // (A1^T rows in two chunks of a whole warp, unless few: 192^3 by symmetry
    // 1368 -> 1195 us, 160^3 936 -> 881, 191^2 x 192 1370 -> 1226; A1 and A2 rows are
    // faster in three chunks of a half warp, A1 at 192^3 by 3%)
    if constexpr (VW == 4)
      if (m <= 48 && (U == 4 || parts > 1 || !(MODE == 2 || (MODE == 0 && W.S > 0)))) SRT_ROWS(3, 16);
    // (parts of 64 vectors instead: A2 of 191 columns at 126 slabs 959 us, 707 so;
    // A1^T of 187 slabs 1307, 1023)
    if constexpr (VW != 4) {
      if (m > 96) SRT_ROWS(4, 32);
      if (m > 64) SRT_ROWS(3, 32);
    }
    SRT_ROWS(2, 32);
  }
#undef SRT_ROWS
}

template <typename V, int MODE>
int launch(const SrtCsr& A, const V* val, const Rows& W, const float* x, int64_t ldx, int64_t bsx,
           float* y, int64_t ldy, int64_t bsy, int ncols, int batch, cudaStream_t st) {
  if constexpr (MODE == 1) {
    if (W.ldn > 0) {
      if (ncols > 128)
        return launch_as<V, 4, 2, 32, 1, 1, true>(A, val, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, st);
      return launch_as<V, 4, 1, 32, 1, 1, true>(A, val, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, st);
    }
  }
  const int64_t any = ncols | ldx | ldy | bsx | bsy;
  const uintptr_t at = (uintptr_t)x | (uintptr_t)y;
  // Four gathers in flight per row up to 128 warps' worth of rows per SM, five
  // to eight times what the registers of the variants leave room for at once
  // (75 x 75 x 53, 18090 rows: A1 44.8 -> 35.8 us, A1^T 47.1 -> 36.9; 32^3: 18.6 ->
  // 13.5), two above (96^3, 24576 warps of four rows: 207 us with four, 188 with
  // two).
  const int lanes = any % 4 == 0 && at % 16 == 0 ? 4 : any % 2 == 0 && at % 8 == 0 ? 2 : 1;
  const int64_t vecs = ((int64_t)ncols + lanes - 1) / lanes;
  const int64_t per_warp = vecs > 32 ? 1 : vecs > 16 ? 2 : 4;
  const bool few = (int64_t)W.rows * batch / per_warp <= (int64_t)128 * kSMs &&
                   vecs <= (lanes == 4 ? 64 : 128);
  if constexpr (MODE != 1 && MODE != 2)
    if (lanes == 4 && vecs > 64)
      return launch_width<V, 4, MODE, 1>(A, val, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, st);
  // A1^T rows by symmetry of more than 192 slabs walking super-tiles: one
  // gather at a time at 40 registers, 48 warps per SM, which suits that walk's
  // reuse in L2 better than two at 60 (256^3, 768 radii 1668 -> 1607 us, batch 4
  // 6473 -> 6166, 224^3 1727 -> 1648; with 1024 radii 2121 -> 2174; without
  // super-tiles 240^3 1922 -> 2063)
  if constexpr (MODE == 2)
    if (lanes == 4 && vecs > 48 && vecs <= 64 && !few && W.S > 0)
      return launch_as<V, 4, 2, 32, 2, 1>(A, val, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, st);
  // A1 whose part of the volume (256 slabs at most) is larger than L2 waits on
  // DRAM, and four gathers hide more of it (us, two and four: 512^3 15813 and
  // 15283, 512^2 x 256 10140 and 9819, 384^2 x 256 5026 and 4956; 320^2 x 256, which
  // L2 holds, 3238 and 3247, 512^2 x 160 in three chunks 7988 and 8364)
  if constexpr (MODE == 1) {
    const int64_t parts = (vecs + 63) / 64, m = (vecs + parts - 1) / parts;
    if (lanes == 4 && m > 48 && A.cols * 16 * m > (int64_t)128 << 20)
      return launch_width<V, 4, MODE, 4>(A, val, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, st);
  }
#define SRT_WIDTH(VW)                                                                          \
  return few ? launch_width<V, VW, MODE, 4>(A, val, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, \
                                            st)                                               \
             : launch_width<V, VW, MODE, 2>(A, val, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, \
                                            st)
  if (lanes == 4) SRT_WIDTH(4);
  if (lanes == 2) SRT_WIDTH(2);
  // Single columns of A1^T and of the taps: four gathers, many rows or few (us,
  // four and two: A2 of 191 columns at 126 slabs 707 and 799, of 171 at 187 2247
  // and 2560; A1^T of 187 slabs 1023 and 1072); pairs of columns gain nothing
  // there (A2 of 190 columns at 127 slabs 498 and 492).
  if constexpr (MODE >= 2)
    return launch_width<V, 1, MODE, 4>(A, val, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, st);
  else
    SRT_WIDTH(1);
#undef SRT_WIDTH
}

template <typename V>
int dispatch(const SrtCsr& A, const V* val, const Rows& W, const float* x, int64_t ldx,
             int64_t bsx, float* y, int64_t ldy, int64_t bsy, int ncols, int batch,
             cudaStream_t st) {
  switch (W.rot.mode) {
    case 1: return launch<V, 1>(A, val, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, st);
    case 2: return launch<V, 2>(A, val, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, st);
    case 3: return launch<V, 3>(A, val, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, st);
    case 4: return launch<V, 4>(A, val, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, st);
    default: return launch<V, 0>(A, val, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, st);
  }
}

}  // namespace

int srt_spmm(const SrtCsr& A, int wdt, const float* x, int64_t ldx, int64_t bsx, float* y,
             int64_t ldy, int64_t bsy, int ncols, int batch, cudaStream_t st, int G, int R,
             int TG, int64_t r0, int64_t rows, SrtRot rot, int S, int64_t ldn) {
  if (rows < 0) rows = A.rows - r0;
  if (rows <= 0) return SRT_OK;
  if (rows > 0x7fffffff || r0 + rows > 0x7fffffff) return SRT_ERR_ARG;
  uint64_t magic = 0;
  if (rot.mode == 1 || rot.mode == 2) {
    if (rot.q <= 0 || rot.ms <= 0 || rot.ms >= (1 << 16) || rot.n_ell <= 0 ||
        (int64_t)rot.ms * rot.ms >= (1 << 24))
      return SRT_ERR_ARG;
    magic = ((1ull << 40) + rot.ms - 1) / rot.ms;
  }
  if (G > 0 && (int64_t)G * R != rows) G = 0;
  if (TG != 1 && TG != 2 && TG != 4 && TG != 8) TG = 1;
  if (S > 0 && (G % S || R % S)) S /= 2;  // (160^3 891 -> 881 us, 224^3 1730 -> 1693)
  if (G <= 0 || S <= 0 || G % S || R % S || S % TG) S = 0;
  // gathered operand: A's columns, or for A1^T from the stored quarter
  // (mode 2) the rows (j, l) of every sensor column
  const int64_t xr = rot.mode == 2 ? (int64_t)4 * rot.q * rot.n_ell : A.cols;
  if (ldn > 0) {
    // fused P1: the rotated-rows kernel with blocks of 4 sensor columns x
    // 2 radii over all rows, 16-byte aligned pieces of Y1'
    if (rot.mode != 1 || G <= 0 || r0 != 0 || G % 4 || ncols % 4 || ldx % 4 || bsx % 4 ||
        ldn % 4 || (uintptr_t)x % 16 || (uintptr_t)y % 16 || (int64_t)batch * G > ldn)
      return SRT_ERR_ARG;
    TG = 4;
    S = 0;
  }
  const Rows W{(int)rows, (int)r0, G, R, TG, S, rot, magic, srt_checked_rows(xr), ldn};
  if (wdt == SRT_BF16) return dispatch<uint16_t>(A, A.v16, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, st);
  return dispatch<float>(A, A.v32, W, x, ldx, bsx, y, ldy, bsy, ncols, batch, st);
}

long long srt_checks_take_spmm() {
#ifdef SRT_CHECKS
  unsigned long long v = 0, z = 0;
  if (cudaMemcpyFromSymbol(&v, g_viol, sizeof(v)) != cudaSuccess) return -1;
  if (cudaMemcpyToSymbol(g_viol, &z, sizeof(z)) != cudaSuccess) return -1;
  return (long long)v;
#else
  return 0;
#endif
}
