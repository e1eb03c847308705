// Second product of Algorithms 1 and 2 through the Toeplitz structure of A2.
//
// When the sensor rings are spaced like the slabs (ring spacing dz, any
// number n_zs of rings, any offset), ring h sits at slab h + s plus a fixed
// fraction eps of a slab (offset of the ring range = s dz + eps), and the
// semicircle of ring h and radius l_m meets cell (radius bin l, slab k)
// exactly as the semicircle of ring h+1 meets cell (l, k+1):
//   A2[(h,m),(l,k)] = T[m, d = k - h - s, l],
// so all of A2 (and A2^T) is held by the master tensor T: a few "taps"
// (l, d, weight) per radius m instead of one row per (ring, radius).  T is
// assembled once for one ring at eps over the D = mz + n_zs - 1 slab offsets
// d = q - (n_zs - 1) - s, q < D, that some (ring, slab) pair takes.
//
// The taps are stored twice, grouped so that the entries of any output row
// form ONE contiguous range, which the product kernel then walks exactly like
// a CSR row (spmm.cu k_rows, modes 3 and 4):
//   forward  (rows (h, m) of A2):   sub-rows (m, q), each listing l
//     ascending; row (h, m) is sub-rows q = n_zs-1-h .. n_zs-2-h+mz, i.e.
//     every slab k = h + q - (n_zs-1) of the volume.  Entry key = l | q << 16;
//     gathered row l*mz + k.
//   adjoint (rows (l, k) of A2^T):  sub-rows (l, e = D - 1 - q), each listing
//     m ascending; row (l, k) is sub-rows e = mz-1-k .. mz-2-k+n_zs, i.e.
//     rings h = k + e - (mz-1) = 0 .. n_zs-1 in ascending order.  Entry key =
//     m | e << 16; gathered row h*n_ell + m.
// With the rings at the slab centres (n_zs = mz, s = eps = 0), D = 2 mz - 1.
// The adjoint visits its entries in the same order as the CSR form of A2^T
// (ascending (h, m)), the forward by ascending (d, l).  Every output row is
// owned by one group of lanes: no atomics.  The row kernel serves every dense
// width (us, A2 / A2^T, with the taps' own warp-per-row kernels before: 57
// columns at 65 slabs 61.5 / 50.2 -> 38.9 / 34.0, 63 at 128 317 / 283 -> 225 /
// 216; row by row at 256^3 2816 / 2818 -> 2614 / 2685).
#include <algorithm>
#include <cstdlib>
#include <vector>

#include "common.cuh"
#include "devutil.cuh"

namespace {

// Upload one grouped tap list (host vectors) into t.
int upload(const std::vector<int32_t>& rp, const std::vector<int32_t>& key,
           const std::vector<float>& w32, const std::vector<uint16_t>& w16, SrtTaps* t,
           int64_t* bytes) {
  t->nsub = (int64_t)rp.size() - 1;
  t->nent = (int64_t)key.size();
  SRT_TRY(srt_dmalloc(&t->rowptr, (int64_t)rp.size(), bytes));
  SRT_TRY(srt_dmalloc(&t->key, t->nent, bytes));
  SRT_CUDA_TRY(cudaMemcpy(t->rowptr, rp.data(), rp.size() * 4, cudaMemcpyHostToDevice));
  if (t->nent)
    SRT_CUDA_TRY(cudaMemcpy(t->key, key.data(), key.size() * 4, cudaMemcpyHostToDevice));
  if (!w32.empty()) {
    SRT_TRY(srt_dmalloc(&t->w32, t->nent, bytes));
    SRT_CUDA_TRY(cudaMemcpy(t->w32, w32.data(), w32.size() * 4, cudaMemcpyHostToDevice));
  }
  if (!w16.empty()) {
    SRT_TRY(srt_dmalloc(&t->w16, t->nent, bytes));
    SRT_CUDA_TRY(cudaMemcpy(t->w16, w16.data(), w16.size() * 2, cudaMemcpyHostToDevice));
  }
  return SRT_OK;
}

}  // namespace

void srt_taps_free(SrtTaps* t) {
  cudaFree(t->rowptr);
  cudaFree(t->key);
  cudaFree(t->w32);
  cudaFree(t->w16);
  *t = SrtTaps();
}

// T: rows m < n_ell, columns l*D + q (D = mz + n_zs - 1), ascending.
int srt_build_taps(srt_plan_s* plan, const SrtCsr& T, int64_t* nnz2, int64_t* bytes) {
  const srt_geometry& g = plan->g;
  const int mz = g.mz, nz = g.n_zs, n_ell = g.n_ell, D = mz + nz - 1;
  if (T.rows != n_ell || n_ell > 0xffff || D > 0x7fff) return SRT_ERR_ARG;
  const int64_t nt = T.nnz;
  std::vector<int32_t> rp(n_ell + 1), col(nt);
  std::vector<float> v32(T.v32 ? nt : 0);
  std::vector<uint16_t> v16(T.v16 ? nt : 0);
  SRT_CUDA_TRY(cudaMemcpy(rp.data(), T.rowptr, rp.size() * 4, cudaMemcpyDeviceToHost));
  if (nt) {
    SRT_CUDA_TRY(cudaMemcpy(col.data(), T.col, nt * 4, cudaMemcpyDeviceToHost));
    if (T.v32) SRT_CUDA_TRY(cudaMemcpy(v32.data(), T.v32, nt * 4, cudaMemcpyDeviceToHost));
    if (T.v16) SRT_CUDA_TRY(cudaMemcpy(v16.data(), T.v16, nt * 2, cudaMemcpyDeviceToHost));
  }
  // entries of A2: the tap in column q serves the rings h < nz whose slab
  // k = h + u, u = q - (nz - 1), lies in the volume
  int64_t n2 = 0;
  for (int64_t e = 0; e < nt; ++e) {
    const int u = col[e] % D - (nz - 1);
    const int h0 = std::max(0, -u), h1 = std::min(nz - 1, mz - 1 - u);
    n2 += h1 >= h0 ? h1 - h0 + 1 : 0;
  }
  *nnz2 = n2;
  // counting sorts, stable in T's (m, l, q) order
  const int64_t nsub = (int64_t)n_ell * D;
  std::vector<int32_t> fp(nsub + 1, 0), ap(nsub + 1, 0);
  for (int m = 0; m < n_ell; ++m)
    for (int e = rp[m]; e < rp[m + 1]; ++e) {
      const int l = col[e] / D, q = col[e] % D;
      ++fp[(int64_t)m * D + q + 1];
      ++ap[(int64_t)l * D + (D - 1 - q) + 1];
    }
  for (int64_t i = 0; i < nsub; ++i) {
    fp[i + 1] += fp[i];
    ap[i + 1] += ap[i];
  }
  std::vector<int32_t> fk(nt), ak(nt);
  std::vector<int32_t> fpos(fp.begin(), fp.end() - 1), apos(ap.begin(), ap.end() - 1);
  std::vector<float> f32(v32.size()), a32(v32.size());
  std::vector<uint16_t> f16(v16.size()), a16(v16.size());
  for (int m = 0; m < n_ell; ++m)
    for (int e = rp[m]; e < rp[m + 1]; ++e) {
      const int l = col[e] / D, q = col[e] % D, ee = D - 1 - q;
      const int64_t i = fpos[(int64_t)m * D + q]++, j = apos[(int64_t)l * D + ee]++;
      fk[i] = l | (q << 16);
      ak[j] = m | (ee << 16);
      if (!v32.empty()) f32[i] = a32[j] = v32[e];
      if (!v16.empty()) f16[i] = a16[j] = v16[e];
    }
  SRT_TRY(upload(fp, fk, f32, f16, &plan->tf, bytes));
  SRT_TRY(upload(ap, ak, a32, a16, &plan->ta, bytes));
  if (!(plan->g.flags & SRT_ROWWISE)) {
    SRT_TRY(srt_build_tiles(plan, rp, col, v32, v16, bytes));
    plan->tiles = 1;
  }
  return SRT_OK;
}

int srt_taps_apply(const srt_plan_s* plan, bool adjoint, int64_t r0, int64_t rows, int G, int R,
                   int TG, const float* x, int64_t ldx, float* y, int64_t ldy, int ncols,
                   cudaStream_t st) {
  const srt_geometry& g = plan->g;
  const SrtTaps& t = adjoint ? plan->ta : plan->tf;
  if (!t.rowptr || rows <= 0 || ncols <= 0) return SRT_ERR_ARG;
  if (g.weight_dtype == SRT_BF16 ? !t.w16 : !t.w32) return SRT_ERR_ARG;
  SrtCsr a;  // the taps as the row kernel reads them; every output row a range of them
  a.rows = adjoint ? g.n_ell * g.mz : g.n_zs * g.n_ell;
  a.cols = adjoint ? g.n_zs * g.n_ell : g.n_ell * g.mz;
  a.nnz = t.nent;
  a.rowptr = t.rowptr;
  a.col = t.key;
  a.v32 = t.w32;
  a.v16 = t.w16;
  SrtRot how;
  how.mode = adjoint ? 4 : 3;
  how.ms = g.mz;
  how.n_ell = g.n_ell;
  how.q = g.n_zs;
  return srt_spmm(a, g.weight_dtype, x, ldx, 0, y, ldy, 0, ncols, 1, st, G, R, TG, r0, rows, how);
}
