// What the star factorisation (starfact.cu) and the star solves (starsolve.cu) share: the
// layout of a star's factor blob, the elements of a star, and small warp sums.
#pragma once

#include <vector>

#include "spnet_internal.cuh"

namespace spnet {

__host__ __device__ inline int64_t align_up(int64_t x, int64_t a) { return (x + a - 1) / a * a; }

// A star's factor blob (FP64; packed into the solve's records, then released).  Header:
// dofs n, sparse levels nlev, off-diagonal entries nnz of the sparse part, and c, the nodes
// of the dense block whose inverse the solve applies (0: none).  With c > 0 the last c
// positions are the block's: rows list their entries outside the block only, the block has
// no columns and no levels.
struct BlobLayout {
  int64_t gidx, rowptr, colptr, lvl, perm, rowidx, colidx, c2r, rowval, colval, invd, total;
};

__host__ __device__ inline BlobLayout blob_layout(int n, int nlev, int nnz) {
  BlobLayout L;
  int64_t o = 16;  // header: n, nlev, nnz, c
  L.gidx = o;   o += 4ll * n;
  L.rowptr = o; o += 4ll * (n + 1);
  L.colptr = o; o += 4ll * (n + 1);
  L.lvl = o;    o += 2ll * (nlev + 1);
  L.perm = o;   o += 2ll * n;
  L.rowidx = o; o += 2ll * nnz;
  L.colidx = o; o += 2ll * nnz;
  o = align_up(o, 8);
  L.c2r = o;    o += 4ll * nnz;  // column entry -> row entry
  o = align_up(o, 8);
  L.rowval = o; o += 8ll * nnz;
  L.colval = o; o += 8ll * nnz;
  L.invd = o;   o += 8ll * n;    // 1 / L_vv
  L.total = align_up(o, 16);
  return L;
}

// a blob's arrays
struct Blob {
  int n, nlev, nnz, c;
  const int32_t* gidx;
  const uint32_t *rowptr, *colptr;
  const uint16_t *lvl, *perm, *rowidx, *colidx;
  const int32_t* c2r;
  double *rowv, *colv, *invd;
};
__device__ inline Blob blob_at(char* b) {
  Blob B;
  const int32_t* h = (const int32_t*)b;
  B.n = h[0];
  B.nlev = h[1];
  B.nnz = h[2];
  B.c = h[3];
  const BlobLayout L = blob_layout(B.n, B.nlev, B.nnz);
  B.gidx = (const int32_t*)(b + L.gidx);
  B.rowptr = (const uint32_t*)(b + L.rowptr);
  B.colptr = (const uint32_t*)(b + L.colptr);
  B.lvl = (const uint16_t*)(b + L.lvl);
  B.perm = (const uint16_t*)(b + L.perm);
  B.rowidx = (const uint16_t*)(b + L.rowidx);
  B.colidx = (const uint16_t*)(b + L.colidx);
  B.c2r = (const int32_t*)(b + L.c2r);
  B.rowv = (double*)(b + L.rowval);
  B.colv = (double*)(b + L.colval);
  B.invd = (double*)(b + L.invd);
  return B;
}

// the 2^d elements of a star, in c' order, with their offsets in the star
struct StarElems {
  int e[8];
  int off[9];
  int nc;
};

__device__ inline StarElems star_elems(const Mesh& m, int k, const int32_t* elem_ptr) {
  StarElems se;
  int km[3];
  mesh_multi(m, k, km);
  int o = 0;
  se.nc = m.nc;
  for (int cp = 0; cp < m.nc; ++cp) {
    int e = elem_around(m, km, cp);
    se.e[cp] = e;
    se.off[cp] = o;
    if (e >= 0) o += elem_ptr[e + 1] - elem_ptr[e];
  }
  se.off[m.nc] = o;
  return se;
}

__device__ inline int pc_of_local(const StarElems& se, const int32_t* elem_ptr, int t) {
  int cp = 0;
  while (cp + 1 < se.nc && se.off[cp + 1] <= t) ++cp;
  return elem_ptr[se.e[cp]] + (t - se.off[cp]);
}

// "support" patches: local dof t lies outside the open support of the star's basis
// function (its Q1 value there is zero).  The star's mesh node sits at corner
// nc - 1 - c' of the element in slot c'.
__device__ inline bool off_support(const StarElems& se, const int32_t* elem_ptr, const double* q1w,
                                   int64_t N, int t) {
  int cp = 0;
  while (cp + 1 < se.nc && se.off[cp + 1] <= t) ++cp;
  const int i = elem_ptr[se.e[cp]] + (t - se.off[cp]);
  return q1w[(int64_t)(se.nc - 1 - cp) * N + i] == 0.0;
}

__device__ inline int warp_min(int v) {
  for (int o = 16; o > 0; o >>= 1) v = min(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

__device__ inline int warp_sum(int v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ inline int warp_incl_scan(int v, int lane) {
  for (int o = 1; o < 32; o <<= 1) {
    int t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// starsolve.cu: the solve's records from the blobs (the sizes first, then the entries)
int star_records_plan(spnet_pc_s* pc, DevArena& tmp, const std::vector<int32_t>& lev,
                      const std::vector<int32_t>& nz, const int32_t* noinv);
int star_records_fill(spnet_pc_s* pc);

// where a star's dense-block inverse goes: records of `kc` columns (starsolve.cu), each
// [row block of 32][column group of V][row][V], V = 16 / sizeof(T); an entry's index in the
// block's area
template <class T>
__host__ __device__ inline int64_t core_slot(int c, int kc, int i, int j) {
  constexpr int V = 16 / (int)sizeof(T);
  const int cp = (c + 3) / 4 * 4;
  const int rec = j / kc, jj = j - rec * kc;
  const int kcr = cp - rec * kc < kc ? cp - rec * kc : kc;
  const int rb = i / 32, nr = c - rb * 32 < 32 ? c - rb * 32 : 32;
  return (int64_t)rec * kc * c + (int64_t)rb * 32 * kcr + ((int64_t)(jj / V) * nr + (i & 31)) * V + jj % V;
}

}  // namespace spnet
