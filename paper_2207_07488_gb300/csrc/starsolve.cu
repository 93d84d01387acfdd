// The star solves w_j = A_j^{-1} E_j^T r (Section 4.1, eq. defPj), one block per star, for one
// right-hand side or a block of them.
//
// With A_j = L L^T (starfact.cu) written as a unit triangle times a diagonal, and the dense
// block that ends the elimination kept as its inverse, a solve is
//   forward   y_v = r_v - sum_u l_vu y_u          level by level (l_vu = L_vu / L_uu),
//             the last "level" being the rows of the dense block,
//   block     z_c = S^{-1} y_c                     one product,
//   backward  z_v = y_v / L_vv^2 - sum_i l_iv z_i  levels in reverse.
// Rows of a level do not read one another: a lane takes a row, so a level of a few dozen
// rows costs one step of a few dozen instructions, with no scan across lanes.
//
// A star's data is a sequence of records, read in order:
//   forward records | block records | backward records.
// A forward or backward record holds steps; a step holds up to 16 groups of rows, and a
// barrier follows it.  Step: u16 groups, u16 size / 16, u32 1 in the record's last step;
// per group 8 B: u16 place / 16 in the step, u16 entries per row K, u8 rows, u8 flags
// (1: scaled by 1 / L_vv^2, 2: one row across the lanes).  Group: u16 row places, the scales,
// u16 columns [K][rows], coefficients [K][rows] (negated: a row is a chain of fused
// multiply-adds).  The rows of a level are sorted by their number of entries, so a group
// pads little, and rows with no forward entry are left out.
// A block record holds kc columns of S^{-1} (core_slot, star_blob.cuh): a lane takes a row
// and reads 16 bytes of coefficients at a time, the vector broadcast from shared memory.
//
// Records are fetched by bulk copies (cp.async.bulk, one mbarrier a slot) into a ring of
// slots in shared memory, from the first instruction on: they do not depend on the previous
// kernel, so under programmatic launch the first slots fill while it drains.
// Every sum is taken in an order fixed by the records: the result depends neither on the
// warps per block nor on the other right-hand sides.
#include <algorithm>
#include <atomic>

#include "star_blob.cuh"
#include "star_ring.cuh"

namespace spnet {

constexpr int STEP_GROUPS = 16;
constexpr int WIDE_K = 192;       // a row with more entries goes across the lanes
constexpr int SOLVE_SMEM = 227 * 1024;
constexpr int SOLVE_HEAD = 128;   // the slots' mbarriers

// Record size.  A block waits and synchronises once a record, so a record holds eight columns of
// the largest dense block where 16 KB allow it (a 16-byte column group, c * 16 bytes, always
// fits); small stars take small records, so that the slots of many blocks fit an SM's shared
// memory.  On the (2^9 + 1)^2 grid
// (FP64, blocks of up to 199 nodes) a 26-step solve takes 9.6 ms with 16 KB, 13.1 with 4 KB.
inline int record_size(int max_star, int cmax, int vb) {
  if ((int64_t)max_star * vb > STAR_HUGE) return 4096;  // blocks of at most 256 nodes then
  int r = max_star <= 1024 ? 4096 : 8192;
  while (r < 16384 && r < 8 * cmax * vb) r *= 2;
  return r;
}
constexpr int GF_SCALE = 1, GF_WIDE = 2;

// Headers and records lie in the order of the blocks: stars by cost, largest first.
struct StarHdr {
  int64_t sbase;   // byte offset of the star's records
  int64_t wbase;   // first slot of the star in w (star_ptr)
  int64_t rec0;    // its first entry in rec_off (offsets from sbase, 16 B units, one past the last)
  uint32_t off[SLOTS + 2];  // the first of those entries: the first copies wait for the header only
  uint32_t pad;
  int32_t n, ns;   // dofs; those outside the dense block
  int32_t c, kc;   // nodes of the block, columns of its inverse per record
  int32_t nf, nc, nb;  // records: forward, block, backward
  int32_t pad2;
  int32_t es[8];   // pc index of the first dof of each of the 2^d elements, -1 if absent
  uint16_t eo[8];  // local offset of each element's dofs within the star
};
static_assert(sizeof(StarHdr) == 128, "StarHdr layout");

__host__ __device__ inline int up4(int v) { return (v + 3) / 4 * 4; }
// the solve's vector: sparse dofs at 0.., the block's forward values at cb, its solution at zb
__host__ __device__ inline int place_cb(int ns) { return up4(ns); }
__host__ __device__ inline int place_zb(int ns, int c) { return up4(ns) + up4(c); }
__host__ __device__ inline int vec_len(int ns, int c) { return c > 0 ? place_zb(ns, c) + up4(c) : ns; }

__host__ __device__ inline int group_bytes(int rows, int K, bool scale, int vb) {
  const int b = (int)align_up(2 * rows, 8) + (scale ? vb * rows : 0) + (int)align_up(2 * rows * K, 8) + vb * rows * K;
  return (b + 15) / 16 * 16;
}
__host__ __device__ inline int step_head(int groups) { return (8 + 8 * groups + 15) / 16 * 16; }

// columns of the dense block's inverse per record
__host__ __device__ inline int core_cols(int c, int rec, int vb) {
  if (c == 0) return 0;
  const int v = 16 / vb;
  const int kc = rec / (c * vb) / v * v;
  return kc > up4(c) ? up4(c) : kc;
}

// ---------------------------------------------------------------------------
// the records of a star: one walk that sizes them (FILL = false, one thread) or writes them
// (FILL = true, one warp; every decision is the same in all lanes)
// ---------------------------------------------------------------------------
template <class T, bool FILL>
struct RecordWriter {
  int rec_size;
  int lane;
  char* base;        // the star's records
  uint32_t* off;     // the star's record offsets
  int rec = 0, fill = 0, last = -1;
  int64_t bytes = 0;
  Blob B;
  int ns, cb, zb;

  __device__ void close() {
    if (fill == 0) return;
    if (FILL && lane == 0) {
      ((uint32_t*)(base + bytes + last))[1] = 1u;
      off[rec + 1] = (uint32_t)((bytes + fill) / 16);
    }
    bytes += fill;
    ++rec;
    fill = 0;
  }
  __device__ char* step(int groups, int body) {
    const int size = step_head(groups) + body;
    if (fill + size > rec_size) close();
    char* p = base + bytes + fill;
    if (FILL && lane == 0) {
      ((uint32_t*)p)[0] = (uint32_t)groups | ((uint32_t)(size / 16) << 16);
      ((uint32_t*)p)[1] = 0u;
    }
    last = fill;
    fill += size;
    return p;
  }
  __device__ void desc(char* st, int g, int at, int K, int rows, int flags) {
    if (FILL && lane == 0)
      ((uint2*)(st + 8))[g] = make_uint2((uint32_t)(at / 16) | ((uint32_t)K << 16), (uint32_t)rows | ((uint32_t)flags << 8));
  }
};

struct SupportTest {  // which elimination positions of a star lie off its basis function's support
  int patch;
  StarElems se;
  const int32_t* elem_ptr;
  const double* q1w;
  int64_t N;
  const uint16_t* perm;  // elimination position -> local index
  __device__ bool off(int v) const {
    return patch == SPNET_PATCH_SUPPORT && off_support(se, elem_ptr, q1w, N, perm[v]);
  }
};

// entries k0..k1 of the rows ord[0..rows) as one group at gp
template <class T>
__device__ void fill_group(char* gp, const Blob& B, int ns, int cb, int zb, bool bwd, const uint16_t* ord, int rows,
                           int k0, int k1, bool scale, bool wide, int lane, const SupportTest& sup) {
  const uint32_t* ptr = bwd ? B.colptr : B.rowptr;
  const uint16_t* idx = bwd ? B.colidx : B.rowidx;
  const double* val = bwd ? B.colv : B.rowv;
  const int K = k1 - k0;
  uint16_t* rid = (uint16_t*)gp;
  char* p = gp + align_up(2 * rows, 8);
  T* dv = (T*)p;
  if (scale) p += sizeof(T) * rows;
  uint16_t* cols = (uint16_t*)p;
  T* co = (T*)(p + align_up(2ll * rows * K, 8));
  const int step = wide ? 1 : rows;
  for (int i = wide ? 0 : lane; i < rows; i += 32) {
    const int v = ord[i];
    const int place = v < ns ? v : cb + (v - ns);
    const double iv = bwd ? B.invd[v] : 0.0;
    if (!wide || lane == 0) {
      rid[i] = (uint16_t)place;
      // a dof off the star's support (support patches) is an isolated row: a zero scale
      // makes its value, and the star's contribution there, zero
      if (scale) dv[i] = sup.off(v) ? (T)0 : (T)(iv * iv);
    }
    const int q0 = (int)ptr[v], cnt = (int)ptr[v + 1] - q0;
    for (int k = k0 + (wide ? lane : 0); k < k1; k += wide ? 32 : 1) {
      int col = place;
      double a = 0.0;
      if (k < cnt) {
        const int u = idx[q0 + k];
        col = u < ns ? u : zb + (u - ns);
        a = -val[q0 + k] * (bwd ? iv : B.invd[u]);
      }
      cols[(k - k0) * step + i] = (uint16_t)col;
      co[(k - k0) * step + i] = (T)a;
    }
  }
}

// the rows ord[0..nr) (sorted by entries, most first) as steps; bwd: scaled columns
template <class T, bool FILL>
__device__ void write_level(RecordWriter<T, FILL>& w, const uint16_t* ord, int nr, bool bwd, const SupportTest& sup) {
  const Blob& B = w.B;
  const uint32_t* ptr = bwd ? B.colptr : B.rowptr;
  constexpr int vb = (int)sizeof(T);
  auto count = [&](int i) { return (int)(ptr[ord[i] + 1] - ptr[ord[i]]); };
  if (!bwd) {  // rows without forward entries stay as they are
    int lo = 0, hi = nr;
    while (lo < hi) {
      const int m = (lo + hi) >> 1;
      if (count(m) > 0) lo = m + 1;
      else hi = m;
    }
    nr = lo;
  }
  // rows of the group that starts at row i, and its K; at least two groups fit a record
  auto pick = [&](int i, int& rows, int& K) {
    K = count(i);
    rows = nr - i < 32 ? nr - i : 32;
    if (K > WIDE_K) {
      rows = 1;
      return;
    }
    while (rows > 4 && group_bytes(rows, K, bwd, vb) > (w.rec_size - 32) / 2) rows = (rows + 1) / 2;
  };
  int i = 0;
  while (i < nr) {
    int rows, K;
    pick(i, rows, K);
    const bool wide = K > WIDE_K;
    if (wide || step_head(1) + group_bytes(rows, K, bwd, vb) > w.rec_size) {
      // a long row: parts, each a step of its own (the barriers keep their order)
      int kp = K;
      while (step_head(1) + group_bytes(rows, kp, bwd, vb) > w.rec_size) kp = (kp + 1) / 2;
      for (int k0 = 0; k0 < K; k0 += kp) {
        const int k1 = k0 + kp < K ? k0 + kp : K;
        const bool scale = bwd && k0 == 0;
        char* st = w.step(1, group_bytes(rows, k1 - k0, scale, vb));
        w.desc(st, 0, step_head(1), k1 - k0, rows, (scale ? GF_SCALE : 0) | (wide ? GF_WIDE : 0));
        if (FILL)
          fill_group<T>(st + step_head(1), B, w.ns, w.cb, w.zb, bwd, ord + i, rows, k0, k1, scale, wide, w.lane, sup);
      }
      i += rows;
      continue;
    }
    // as many groups as the record has room for (all, if they fit a fresh one)
    int gr[STEP_GROUPS], gk[STEP_GROUPS];
    int ng = 0, body = 0, j = i;
    while (j < nr && ng < STEP_GROUPS) {
      pick(j, rows, K);
      if (K > WIDE_K) break;
      const int gb = group_bytes(rows, K, bwd, vb);
      const int room = w.rec_size - (ng == 0 && w.fill + step_head(1) + gb > w.rec_size ? 0 : w.fill);
      if (ng > 0 && step_head(ng + 1) + body + gb > room) {
        // the rest goes to another step; a fresh record first where that holds more of it
        if (w.fill > 0 && step_head(ng + 1) + body + gb <= w.rec_size && 2 * w.fill >= w.rec_size) {
          w.close();
          continue;
        }
        break;
      }
      if (ng == 0 && w.fill + step_head(1) + gb > w.rec_size) w.close();
      gr[ng] = rows;
      gk[ng] = K;
      body += gb;
      ++ng;
      j += rows;
    }
    char* st = w.step(ng, body);
    int at = step_head(ng);
    for (int g = 0; g < ng; ++g) {
      w.desc(st, g, at, gk[g], gr[g], bwd ? GF_SCALE : 0);
      if (FILL)
        fill_group<T>(st + at, B, w.ns, w.cb, w.zb, bwd, ord + i, gr[g], 0, gk[g], bwd, false, w.lane, sup);
      at += group_bytes(gr[g], gk[g], bwd, vb);
      i += gr[g];
    }
  }
}

// all records of a star; counts[0..2]: forward, block, backward records; *fbytes: bytes before the block's
template <class T, bool FILL>
__device__ void write_star(RecordWriter<T, FILL>& w, const uint16_t* ford, const uint16_t* bord, int kc, int* counts,
                           int64_t* fbytes, const SupportTest& sup) {
  const Blob& B = w.B;
  if (FILL && w.lane == 0) w.off[0] = 0;
  for (int l = 1; l < B.nlev; ++l)
    write_level<T, FILL>(w, ford + B.lvl[l], B.lvl[l + 1] - B.lvl[l], false, sup);
  if (B.c > 0) write_level<T, FILL>(w, ford + w.ns, B.c, false, sup);
  w.close();
  counts[0] = w.rec;
  *fbytes = w.bytes;
  for (int k0 = 0; k0 < up4(B.c); k0 += kc) {
    const int kcr = up4(B.c) - k0 < kc ? up4(B.c) - k0 : kc;
    w.bytes += (int64_t)B.c * kcr * sizeof(T);
    ++w.rec;
    if (FILL && w.lane == 0) w.off[w.rec] = (uint32_t)(w.bytes / 16);
  }
  counts[1] = w.rec - counts[0];
  for (int l = B.nlev - 1; l >= 0; --l)
    write_level<T, FILL>(w, bord + B.lvl[l], B.lvl[l + 1] - B.lvl[l], true, sup);
  w.close();
  counts[2] = w.rec - counts[0] - counts[1];
}

template <class T, bool FILL>
__device__ RecordWriter<T, FILL> make_writer(char* blob, int rec_size, int lane, char* base, uint32_t* off) {
  RecordWriter<T, FILL> w;
  w.rec_size = rec_size;
  w.lane = lane;
  w.base = base;
  w.off = off;
  w.B = blob_at(blob);
  w.ns = w.B.n - w.B.c;
  w.cb = place_cb(w.ns);
  w.zb = place_zb(w.ns, w.B.c);
  return w;
}

// rows [v0, v1) by their number of entries, most first (stable), by one warp
__device__ void sort_rows(const uint32_t* ptr, int v0, int v1, uint16_t* out, int lane) {
  constexpr unsigned FULL = 0xffffffffu;
  int want = 1 << 30, at = 0;
  while (at < v1 - v0) {
    int m = -1;  // the next smaller count present
    for (int v = v0 + lane; v < v1; v += 32) {
      const int c = (int)(ptr[v + 1] - ptr[v]);
      if (c < want) m = max(m, c);
    }
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(FULL, m, o));
    want = m;
    for (int b = v0; b < v1; b += 32) {
      const int v = b + lane;
      const bool hit = v < v1 && (int)(ptr[v + 1] - ptr[v]) == want;
      const unsigned bal = __ballot_sync(FULL, hit);
      if (hit) out[at + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)v;
      at += __popc(bal);
    }
  }
}

// warp per star: the rows of every level in the order the records take them
__global__ void __launch_bounds__(128) k_star_rows(int S, char* pool, const int64_t* __restrict__ star_off,
                                                   const int64_t* __restrict__ star_ptr, uint16_t* ford,
                                                   uint16_t* bord) {
  const int lane = threadIdx.x & 31;
  const int s = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  if (s >= S) return;
  const Blob B = blob_at(pool + star_off[s]);
  uint16_t *f = ford + star_ptr[s], *b = bord + star_ptr[s];
  for (int l = 0; l < B.nlev; ++l) {
    const int v0 = B.lvl[l], v1 = B.lvl[l + 1];
    if (l > 0) sort_rows(B.rowptr, v0, v1, f + v0, lane);
    sort_rows(B.colptr, v0, v1, b + v0, lane);
  }
  if (B.c > 0) sort_rows(B.rowptr, B.n - B.c, B.n, f + B.n - B.c, lane);
}

// thread per star: its record counts and bytes
template <class T>
__global__ void __launch_bounds__(128) k_record_sizes(int S, char* pool, const int64_t* __restrict__ star_off,
                                                      const int64_t* __restrict__ star_ptr,
                                                      const uint16_t* __restrict__ ford,
                                                      const uint16_t* __restrict__ bord, int rec_size,
                                                      const int32_t* __restrict__ place, int4* counts, int64_t* nrec,
                                                      int64_t* bytes, int64_t* fbytes) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= S) return;
  RecordWriter<T, false> w = make_writer<T, false>(pool + star_off[s], rec_size, 0, nullptr, nullptr);
  SupportTest sup{};
  int cnt[3];
  const int kc = core_cols(w.B.c, rec_size, (int)sizeof(T));
  write_star<T, false>(w, ford + star_ptr[s], bord + star_ptr[s], kc, cnt, &fbytes[s], sup);
  counts[s] = make_int4(cnt[0], cnt[1], cnt[2], kc);
  nrec[place[s]] = w.rec + 1;
  bytes[place[s]] = w.bytes;
}

// thread per star: where its inverse goes
__global__ void k_core_places(int S, const int32_t* __restrict__ place, const int4* __restrict__ counts,
                              const int64_t* __restrict__ sbase,
                              const int64_t* __restrict__ fbytes, int64_t* core_off, int32_t* core_kc) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= S) return;
  core_off[s] = sbase[place[s]] + fbytes[s];
  core_kc[s] = counts[s].w;
}

// warp per star: header, places and records
template <class T>
__global__ void __launch_bounds__(128) k_record_fill(int S, Mesh m, char* pool, const int64_t* __restrict__ star_off,
                                                     const int32_t* __restrict__ star_mesh,
                                                     const int32_t* __restrict__ elem_ptr,
                                                     const int64_t* __restrict__ star_ptr,
                                                     const uint16_t* __restrict__ ford,
                                                     const uint16_t* __restrict__ bord, int rec_size,
                                                     const int4* __restrict__ counts,
                                                     const int64_t* __restrict__ rec0,
                                                     const int64_t* __restrict__ sbase, StarHdr* __restrict__ hdr,
                                                     const int32_t* __restrict__ place,
                                                     uint16_t* __restrict__ iperm, char* recs, uint32_t* rec_off,
                                                     int patch, const double* __restrict__ q1w, int64_t N) {
  const int lane = threadIdx.x & 31;
  const int s = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  if (s >= S) return;
  const int at = place[s];
  RecordWriter<T, true> w =
      make_writer<T, true>(pool + star_off[s], rec_size, lane, recs + sbase[at], rec_off + rec0[at]);
  const Blob& B = w.B;
  const int64_t wb = star_ptr[s];
  SupportTest sup;
  sup.patch = patch;
  sup.se = star_elems(m, star_mesh[s], elem_ptr);
  sup.elem_ptr = elem_ptr;
  sup.q1w = q1w;
  sup.N = N;
  sup.perm = B.perm;
  const int4 cn = counts[s];
  for (int pos = lane; pos < B.n; pos += 32)
    iperm[wb + B.perm[pos]] = (uint16_t)(pos < w.ns ? pos : w.cb + (pos - w.ns));
  int cnt[3];
  int64_t fb;
  write_star<T, true>(w, ford + wb, bord + wb, cn.w, cnt, &fb, sup);
  if (lane == 0) {
    StarHdr h;
    h.sbase = sbase[at];
    h.wbase = wb;
    h.rec0 = rec0[at];
    for (int i = 0; i < SLOTS + 2; ++i) h.off[i] = i <= cn.x + cn.y + cn.z ? w.off[i] : 0;
    h.pad = 0;
    h.n = B.n;
    h.ns = w.ns;
    h.c = B.c;
    h.kc = cn.w;
    h.nf = cn.x;
    h.nc = cn.y;
    h.nb = cn.z;
    h.pad2 = 0;
    for (int cp = 0; cp < 8; ++cp) h.es[cp] = (cp < m.nc && sup.se.e[cp] >= 0) ? elem_ptr[sup.se.e[cp]] : -1;
    for (int cp = 0; cp < 8; ++cp) h.eo[cp] = (uint16_t)(sup.se.off[cp < m.nc ? cp : m.nc]);
    hdr[at] = h;
  }
}

template <class T>
static int records_plan_t(spnet_pc_s* pc, DevArena& tmp, const std::vector<int32_t>& sn,
                          const std::vector<int32_t>& lev, const std::vector<int32_t>& nz) {
  cudaStream_t s = pc->op->stream;
  const int S = pc->S;
  const unsigned g1 = (unsigned)((S + 127) / 128), gw = (unsigned)((S + 3) / 4);
  SPNET_TRY(tmp.get(&pc->ford, pc->sum_s > 0 ? pc->sum_s : 1));
  SPNET_TRY(tmp.get(&pc->bord, pc->sum_s > 0 ? pc->sum_s : 1));
  int4* counts = nullptr;
  int32_t* place = nullptr;
  int64_t *nrec = nullptr, *bytes = nullptr, *fbytes = nullptr, *rec0 = nullptr, *sbase = nullptr;
  SPNET_TRY(tmp.get(&counts, S));
  SPNET_TRY(tmp.get(&place, S));
  SPNET_TRY(tmp.get(&nrec, S + 1));
  SPNET_TRY(tmp.get(&bytes, S + 1));
  SPNET_TRY(tmp.get(&fbytes, S + 1));
  SPNET_TRY(tmp.get(&rec0, S + 1));
  SPNET_TRY(tmp.get(&sbase, S + 1));
  SPNET_TRY(tmp.get(&pc->core_off, S));
  SPNET_TRY(tmp.get(&pc->core_kc, S));
  // stars by cost, largest first: the order of the solve's blocks
  std::vector<double> cost(S);
  std::vector<int32_t> ord(S), rank(S);
  for (int i = 0; i < S; ++i) {
    const double c = pc->star_inv[i];
    cost[i] = 3.0 * (double)sn[i] + 2.0 * nz[i] + c * c + 64.0 * lev[i];
    ord[i] = i;
  }
  std::stable_sort(ord.begin(), ord.end(), [&](int a, int b) { return cost[a] > cost[b]; });
  for (int i = 0; i < S; ++i) rank[ord[i]] = i;
  SPNET_CUDA_TRY(cudaMemcpyAsync(place, rank.data(), sizeof(int32_t) * S, cudaMemcpyHostToDevice, s));
  note_launch();
  k_star_rows<<<gw, 128, 0, s>>>(S, pc->pool, pc->star_off, pc->star_ptr, pc->ford, pc->bord);
  note_launch();
  k_record_sizes<T><<<g1, 128, 0, s>>>(S, pc->pool, pc->star_off, pc->star_ptr, pc->ford, pc->bord, pc->rec_size,
                                       place, counts, nrec, bytes, fbytes);
  SPNET_CUDA_TRY(cudaGetLastError());
  SPNET_TRY(scan_exclusive64(nrec, rec0, S, s, tmp));
  SPNET_TRY(scan_exclusive64(bytes, sbase, S, s, tmp));
  int64_t total_rec = 0, total = 0;
  SPNET_CUDA_TRY(cudaMemcpyAsync(&total_rec, rec0 + S, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  SPNET_CUDA_TRY(cudaMemcpyAsync(&total, sbase + S, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  SPNET_CUDA_TRY(cudaStreamSynchronize(s));  // also: the host tables go out of scope
  SPNET_TRY(pc->mem.get(&pc->srec, total > 0 ? total : 16));
  SPNET_TRY(pc->mem.get(&pc->rec_off, total_rec));
  pc->srec_bytes = total;
  pc->rec_counts = counts;
  pc->rec_place = place;
  pc->rec_first = rec0;
  pc->rec_base = sbase;
  note_launch();
  k_core_places<<<g1, 128, 0, s>>>(S, place, counts, sbase, fbytes, pc->core_off, pc->core_kc);
  SPNET_CUDA_TRY(cudaGetLastError());
  return SPNET_OK;
}

// (lev and nz may still be on their way from the device: the wait below is theirs too)
int star_records_plan(spnet_pc_s* pc, DevArena& tmp, const std::vector<int32_t>& lev,
                      const std::vector<int32_t>& nz, const int32_t* noinv) {
  cudaStream_t s = pc->op->stream;
  const int S = pc->S;
  std::vector<int32_t> core(S), sn(S), no(S);
  SPNET_CUDA_TRY(cudaMemcpyAsync(no.data(), noinv, sizeof(int32_t) * S, cudaMemcpyDeviceToHost, s));
  SPNET_CUDA_TRY(cudaMemcpyAsync(core.data(), pc->star_core, sizeof(int32_t) * S, cudaMemcpyDeviceToHost, s));
  SPNET_CUDA_TRY(cudaMemcpyAsync(sn.data(), pc->star_n, sizeof(int32_t) * S, cudaMemcpyDeviceToHost, s));
  SPNET_CUDA_TRY(cudaStreamSynchronize(s));
  pc->star_inv.resize(S);
  int cmax = 0;
  pc->ylen = 4;
  for (int i = 0; i < S; ++i) {
    const int c = core[i] <= pc->core_inv && !no[i] ? core[i] : 0;
    pc->star_inv[i] = c;
    cmax = std::max(cmax, c);
    pc->ylen = std::max(pc->ylen, up4(vec_len(sn[i] - c, c)));
  }
  const int vb = pc->precision == SPNET_PREC_FP64 ? 8 : 4;
  pc->rec_size = record_size(pc->max_star, cmax, vb);
  return vb == 8 ? records_plan_t<double>(pc, tmp, sn, lev, nz) : records_plan_t<float>(pc, tmp, sn, lev, nz);
}

// ---------------------------------------------------------------------------
// the solve
// ---------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(unsigned bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_load(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// true once the phase of the given parity is complete; gives up after `limit` clocks (0: at once)
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, long long limit) {
  if (limit <= 0) return false;
  long long t0 = 0;
  for (int it = 0;; ++it) {
    unsigned ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if (it == 0) t0 = clock64();
    else if (clock64() - t0 > limit) return false;
  }
}

// JW consecutive values (16-byte vectors where they fill one)
template <class T, int JW>
__device__ __forceinline__ void ldv(const T* p, T (&v)[JW]) {
  if constexpr (sizeof(T) == 4 && JW == 4) {
    const float4 x = *reinterpret_cast<const float4*>(p);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w;
  } else if constexpr (sizeof(T) == 4 && JW == 2) {
    const float2 x = *reinterpret_cast<const float2*>(p);
    v[0] = x.x; v[1] = x.y;
  } else if constexpr (sizeof(T) == 8 && JW >= 2) {
#pragma unroll
    for (int i = 0; i < JW / 2; ++i) {
      const double2 x = reinterpret_cast<const double2*>(p)[i];
      v[2 * i] = x.x; v[2 * i + 1] = x.y;
    }
  } else {
    v[0] = p[0];
  }
}
template <class T, int JW>
__device__ __forceinline__ void stv(T* p, const T (&v)[JW]) {
  if constexpr (sizeof(T) == 4 && JW == 4) *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  else if constexpr (sizeof(T) == 4 && JW == 2) *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
  else if constexpr (sizeof(T) == 8 && JW >= 2) {
#pragma unroll
    for (int i = 0; i < JW / 2; ++i) reinterpret_cast<double2*>(p)[i] = make_double2(v[2 * i], v[2 * i + 1]);
  } else {
    p[0] = v[0];
  }
}

// one group of rows of a step (see the head of this file)
template <class T, int JW>
__device__ __forceinline__ void solve_group(const char* gp, uint2 d, T* __restrict__ y, int lane) {
  const int K = d.x >> 16, rows = d.y & 0xff;
  const bool scale = d.y & (GF_SCALE << 8);
  if (!(d.y & (GF_WIDE << 8))) {
    if (lane < rows) {
      const char* p = gp + ((2 * rows + 7) & ~7);
      T* yr = y + ((const uint16_t*)gp)[lane] * JW;
      T acc[JW];
      ldv<T, JW>(yr, acc);
      if (scale) {
        const T dv = ((const T*)p)[lane];
        p += sizeof(T) * rows;
#pragma unroll
        for (int j = 0; j < JW; ++j) acc[j] *= dv;
      }
      const uint16_t* cols = (const uint16_t*)p + lane;
      const T* co = (const T*)(p + ((2 * rows * K + 7) & ~7)) + lane;
      int k = K;
      for (; k >= 4; k -= 4) {
        int c[4];
        T a[4], v[4][JW];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          c[u] = *cols;
          a[u] = *co;
          cols += rows;
          co += rows;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) ldv<T, JW>(y + c[u] * JW, v[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int j = 0; j < JW; ++j) acc[j] = fma(a[u], v[u][j], acc[j]);
      }
      for (; k > 0; --k) {
        T v[JW];
        const T a = *co;
        ldv<T, JW>(y + *cols * JW, v);
        cols += rows;
        co += rows;
#pragma unroll
        for (int j = 0; j < JW; ++j) acc[j] = fma(a, v[j], acc[j]);
      }
      stv<T, JW>(yr, acc);
    }
    return;
  }
  // one row across the lanes
  const char* p = gp + 8;
  const int row = ((const uint16_t*)gp)[0];
  T dv = T(1);
  if (scale) {
    dv = ((const T*)p)[0];
    p += sizeof(T);
  }
  const uint16_t* cols = (const uint16_t*)p;
  const T* co = (const T*)(p + ((2 * K + 7) & ~7));
  T acc[JW];
#pragma unroll
  for (int j = 0; j < JW; ++j) acc[j] = T(0);
  for (int k = lane; k < K; k += 32) {
    T v[JW];
    const T a = co[k];
    ldv<T, JW>(y + cols[k] * JW, v);
#pragma unroll
    for (int j = 0; j < JW; ++j) acc[j] = fma(a, v[j], acc[j]);
  }
#pragma unroll
  for (int j = 0; j < JW; ++j)
    for (int o = 16; o > 0; o >>= 1) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
  if (lane == 0) {
    T v[JW];
    ldv<T, JW>(y + row * JW, v);
#pragma unroll
    for (int j = 0; j < JW; ++j) v[j] = fma(dv, v[j], acc[j]);
    stv<T, JW>(y + row * JW, v);
  }
}

// The warps that solve the same right-hand sides of a star: one, or the whole block (no named
// barriers: a kernel that may use them all is given a quarter of the SM's 64, four blocks).
__device__ __forceinline__ void team_sync(int wr) {
  if (wr == 1) __syncwarp();
  else __syncthreads();
}

// JW right-hand sides of dof g (of k), doubles
template <int JW>
__device__ __forceinline__ void load_rhs(const double* __restrict__ r, int64_t g, int k, int j0, bool vec,
                                         double (&v)[JW]) {
  const double* p = r + g * k + j0;
  if (JW >= 2 && vec) {  // k and j0 even: 16-byte aligned, and j0 + JW <= k
#pragma unroll
    for (int i = 0; i < JW / 2; ++i) {
      const double2 x = __ldg(reinterpret_cast<const double2*>(p) + i);
      v[2 * i] = x.x;
      v[2 * i + 1] = x.y;
    }
  } else {
#pragma unroll
    for (int j = 0; j < JW; ++j) v[j] = j0 + j < k ? __ldg(p + j) : 0.0;  // past k: zeros
  }
}

struct SolveArgs {
  const StarHdr* hdr;
  const char* recs;
  const uint32_t* rec_off;
  const uint16_t* iperm;
  int rec_size, ylen;
  int wr;                  // warps of a team
  long long wait;          // clocks a wait for a record may take (spnet_op_wait_limit)
  int* err;                // set where a wait ran out
};

// Block (star, teams x JW right-hand sides): a team of wr warps takes JW right-hand
// sides and its own vector; the rows of a step are dealt to its warps.  Teams of one warp
// share the ring; a team of several warps is the whole block.
// With q set (a PCG step of one right-hand side) the right-hand side is the new residual
// r - alpha q (alpha from the SpMV), formed exactly as the update forms it; otherwise r.
// r, w: [dofs][k].
template <class T, int JW>
__global__ void __launch_bounds__(256, JW == 1 ? 6 : 4) k_star_solve(SolveArgs A, const double* __restrict__ r,
                                                                     const double* __restrict__ q, const Scal* sc,
                                                                     const int* done, int k, int groups,
                                                                     T* __restrict__ w) {
  extern __shared__ __align__(128) char sm[];
  const int tid = threadIdx.x, lane = tid & 31, wr = A.wr;
  const int team = (tid >> 5) / wr, rw = (tid >> 5) % wr, teams = (int)(blockDim.x >> 5) / wr;
  const int j0 = ((int)(blockIdx.x % groups) * teams + team) * JW;
  const StarHdr* H = A.hdr + blockIdx.x / groups;
  const int n = H->n, ns = H->ns, c = H->c, kc = H->kc, nf = H->nf, nc = H->nc, nrec = nf + nc + H->nb;
  const int64_t wb = H->wbase;
  const int RS = A.rec_size;
  const unsigned bars = (unsigned)__cvta_generic_to_shared(sm);
  char* ring = sm + SOLVE_HEAD;
  T* y = (T*)(ring + SLOTS * RS) + team * A.ylen * JW;
  const char* src = A.recs + H->sbase;
  const uint32_t* off = A.rec_off + H->rec0;
  auto fetch = [&](int sl, unsigned o0, unsigned o1) {  // by thread 0
    const unsigned bytes = (o1 - o0) * 16;
    mbar_expect(bars + 8 * sl, bytes);
    bulk_load(bars + SOLVE_HEAD + sl * RS, src + (int64_t)o0 * 16, bytes, bars + 8 * sl);
  };
  // thread 0: the places of the next record to fetch, read a record ahead (the load's latency
  // would stall its warp)
  unsigned oa = 0, ob = 0;
  if (tid == 0) {
    for (int i = 0; i < SLOTS; ++i) mbar_init(bars + 8 * i);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
#pragma unroll
    for (int i = 0; i < SLOTS; ++i)
      if (i < nrec) fetch(i, H->off[i], H->off[i + 1]);
    oa = H->off[SLOTS];
    ob = H->off[SLOTS + 1];
  }
  __syncwarp();  // warp 0 polls the mbarriers that its first lane has initialised
  int eo[8], es[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    eo[e] = H->eo[e];
    es[e] = H->es[e] - eo[e];
  }
  pdl_wait();
  pdl_trigger();
  if (done && *done) {
    if (tid == 0)  // the copies in flight end before the block does
      for (int i = 0; i < SLOTS && i < nrec; ++i) mbar_wait(bars + 8 * i, 0u, WAIT_CLOCKS);
    return;
  }
  const double alpha = q ? sc->alpha : 0.0;
  const bool vec = k % 2 == 0 && j0 + JW <= k, wvec = k % JW == 0 && j0 + JW <= k;
  const int first = rw * 32 + lane, stride = wr * 32;
  const int cb = place_cb(ns), cpad = up4(c);
  // gather r over the star in local order (element ranges: coalesced), to its places
  constexpr int GU = 4;
  for (int t0 = first; t0 < n; t0 += stride * GU) {
    double rv[GU][JW];
    int pv[GU];
#pragma unroll
    for (int u = 0; u < GU; ++u) {
      const int t = t0 + u * stride;
      pv[u] = -1;
      if (t < n) {
        int base = es[0];
#pragma unroll
        for (int e = 1; e < 8; ++e) base = t >= eo[e] ? es[e] : base;
        pv[u] = __ldg(&A.iperm[wb + t]);
        load_rhs<JW>(r, base + t, k, j0, vec, rv[u]);
        if (JW == 1 && q) rv[u][0] = fma(-alpha, __ldg(&q[base + t]), rv[u][0]);
      }
    }
#pragma unroll
    for (int u = 0; u < GU; ++u)
      if (pv[u] >= 0) {
        T v[JW];
#pragma unroll
        for (int j = 0; j < JW; ++j) v[j] = (T)rv[u][j];
        stv<T, JW>(y + pv[u] * JW, v);
      }
  }
  if (first < (cpad - c) * JW) y[(cb + c) * JW + first] = T(0);
  int sl = 0, prev = SLOTS - 1;  // slots of this record and of the one before
  unsigned phase = 0;
  for (int rec = 0; rec < nrec; ++rec) {
    // one warp polls, the barrier tells the rest; it is also the barrier after the previous
    // record's last step (or the gather)
    const bool ok = tid >= 32 || mbar_wait(bars + 8 * sl, phase, A.wait);
    if (__syncthreads_or(!ok)) {
      if (tid == 0) {
        *A.err = 1;
        for (int i = rec; i < ring_issued(rec, nrec); ++i)  // every copy in flight
          mbar_wait(bars + 8 * (i % SLOTS), ring_parity(i), WAIT_CLOCKS);
      }
      return;
    }
    if (tid == 0 && rec > 0 && rec - 1 + SLOTS < nrec) {  // into the slot just freed
      fetch(prev, oa, ob);
      oa = ob;
      if (rec + SLOTS < nrec) ob = __ldg(off + rec + SLOTS + 1);
    }
    const char* p = ring + sl * RS;
    if (rec < nf || rec >= nf + nc) {
      for (;;) {
        const uint2 h = *(const uint2*)p;
        const int ng = h.x & 0xffff;
        for (int g = rw; g < ng; g += wr) {
          const uint2 d = *(const uint2*)(p + 8 + 8 * g);
          solve_group<T, JW>(p + 16 * (d.x & 0xffff), d, y, lane);
        }
        if (h.y) break;
        team_sync(wr);
        p += 16 * (h.x >> 16);
      }
    } else {  // kc columns of the dense block's inverse
      constexpr int V = 16 / (int)sizeof(T);
      const int k0 = (rec - nf) * kc, kcr = cpad - k0 < kc ? cpad - k0 : kc;
      const T* yc = y + (cb + k0) * JW;
      T* z = y + (cb + cpad) * JW;
      for (int rb = rw; rb * 32 < c; rb += wr) {
        const int nr = c - rb * 32 < 32 ? c - rb * 32 : 32;
        if (lane < nr) {
          const T* a = (const T*)p + rb * 32 * kcr + lane * V;
          T* zr = z + (rb * 32 + lane) * JW;
          // V partial sums: shorter chains, and less rounding than one sum over all columns
          T acc[V][JW];
#pragma unroll
          for (int u = 0; u < V; ++u)
#pragma unroll
            for (int j = 0; j < JW; ++j) acc[u][j] = T(0);
#pragma unroll 2
          for (int kk = 0; kk < kcr; kk += V) {
            T av[V];
            ldv<T, V>(a + kk * nr, av);
            if constexpr (JW == 1) {
              T v[V];
              ldv<T, V>(yc + kk, v);
#pragma unroll
              for (int u = 0; u < V; ++u) acc[u][0] = fma(av[u], v[u], acc[u][0]);
            } else {
#pragma unroll
              for (int u = 0; u < V; ++u) {
                T v[JW];
                ldv<T, JW>(yc + (kk + u) * JW, v);
#pragma unroll
                for (int j = 0; j < JW; ++j) acc[u][j] = fma(av[u], v[j], acc[u][j]);
              }
            }
          }
          T zv[JW];
          if (k0 > 0) ldv<T, JW>(zr, zv);
#pragma unroll
          for (int j = 0; j < JW; ++j) {
            T t = acc[0][j] + acc[1][j];
            if constexpr (V == 4) t += acc[2][j] + acc[3][j];
            zv[j] = k0 > 0 ? zv[j] + t : t;
          }
          stv<T, JW>(zr, zv);
        }
      }
    }
    prev = sl;
    if (++sl == SLOTS) {
      sl = 0;
      phase ^= 1u;
    }
  }
  team_sync(wr);
  for (int t = first; t < n; t += stride) {
    int pl = __ldg(&A.iperm[wb + t]);
    if (c > 0 && pl >= cb) pl += cpad;
    T v[JW];
    ldv<T, JW>(y + pl * JW, v);
    T* o = w + (wb + t) * k + j0;
    if (wvec) {
      stv<T, JW>(o, v);
    } else {
#pragma unroll
      for (int j = 0; j < JW; ++j)
        if (j0 + j < k) o[j] = v[j];
    }
  }
}

// shared memory of a block of `teams` teams of JW right-hand sides
static int64_t solve_smem(const spnet_pc_s* pc, int jw, int teams) {
  const int vb = pc->precision == SPNET_PREC_FP64 ? 8 : 4;
  return SOLVE_HEAD + (int64_t)SLOTS * pc->rec_size + align_up((int64_t)pc->ylen * vb * jw * teams, 16);
}
static bool solve_fits(const spnet_pc_s* pc, int jw, int teams) { return solve_smem(pc, jw, teams) <= SOLVE_SMEM; }

template <class T, int JW>
static int launch_solve_t(spnet_pc_s* pc, int wr, int teams, const double* r, const double* q, const Scal* sc, int* err,
                          const int* done, int k, T* w, cudaStream_t s) {
  if (!solve_fits(pc, JW, teams))
    return fail(SPNET_ERR_UNSUPPORTED, "star solves: the largest star's solve vector exceeds a block's shared memory");
  static std::atomic<bool> attr_set[64];  // per device (workers may race: setting twice is harmless)
  int dev = 0;
  SPNET_CUDA_TRY(cudaGetDevice(&dev));
  dev &= 63;
  if (!attr_set[dev]) {
    SPNET_CUDA_TRY(cudaFuncSetAttribute(k_star_solve<T, JW>, cudaFuncAttributeMaxDynamicSharedMemorySize, SOLVE_SMEM));
    attr_set[dev] = true;
  }
  const int groups = (k + JW * teams - 1) / (JW * teams);
  SolveArgs A{(const StarHdr*)pc->shdr, pc->srec, pc->rec_off, pc->iperm_star, pc->rec_size, pc->ylen, wr,
              pc->op->wait_clocks, err};
  launch_pdl(k_star_solve<T, JW>, (unsigned)(pc->S * groups), wr * teams * 32, (size_t)solve_smem(pc, JW, teams), s, A,
             r, q, sc, done, k, groups, w);
  return SPNET_OK;
}

void launch_star_solve(spnet_pc_s* pc, const double* r, const double* q, const Scal* sc, const int* done,
                       cudaStream_t s) {
  if (pc->S == 0) return;
  note_launch();
  ProfScope ps(KID_STARS, s);
  int* err = &pc->scal->err;
  if (pc->precision == SPNET_PREC_FP64)
    launch_solve_t<double, 1>(pc, pc->solve_wpb, 1, r, q, sc, err, done, 1, (double*)pc->w, s);
  else
    launch_solve_t<float, 1>(pc, pc->solve_wpb, 1, r, q, sc, err, done, 1, (float*)pc->w, s);
}

// Widest block of right-hand sides stepped together, from what jw columns of the largest star took
// in the solve's first layout (vectors, places and a few KB of factor data, in a block's shared
// memory).  A block takes solve_smem now, and fewer columns where that does not fit; the widths and
// the largest star (also in star_records_fill) are kept, so that the same stars are taken and the
// same right-hand sides stepped together.
static int64_t batch_bytes(const spnet_pc_s* pc, int jw) {
  const int64_t vb = pc->precision == SPNET_PREC_FP64 ? 8 : 4;
  return 8 * (80 + 32 * vb) + 80 + align_up(vb * pc->max_star * jw, 16) + align_up(2ll * pc->max_star, 16);
}
int star_batch_max_k(const spnet_pc_s* pc) {
  int kp = 32;
  while (kp > 1 && batch_bytes(pc, kp < 4 ? kp : 4) > SOLVE_SMEM) kp >>= 1;
  return kp;
}

template <class T>
static int launch_batch_t(spnet_pc_s* pc, const double* R, int k, T* W, int* err, const int* done, cudaStream_t s) {
  int jw = pc->batch_jw > 0 ? pc->batch_jw : 4;
  if (k < jw) jw = k < 2 ? 1 : 2;
  while (jw > 1 && !solve_fits(pc, jw, 1)) jw /= 2;
  // small stars: one warp a team, up to four teams on one ring; large ones: a team of eight warps
  const bool large = pc->max_star > 1024;
  const int wr = large ? 8 : 1;
  int teams = large ? 1 : 4;
  while (teams > 1 && (teams * jw / 2 >= k || !solve_fits(pc, jw, teams))) teams /= 2;
  switch (jw) {
    case 1: return launch_solve_t<T, 1>(pc, wr, teams, R, nullptr, nullptr, err, done, k, W, s);
    case 2: return launch_solve_t<T, 2>(pc, wr, teams, R, nullptr, nullptr, err, done, k, W, s);
    default: return launch_solve_t<T, 4>(pc, wr, teams, R, nullptr, nullptr, err, done, k, W, s);
  }
}

int launch_star_batch(spnet_pc_s* pc, const double* R, int k, void* W, int* err, const int* done, cudaStream_t s) {
  if (pc->S == 0) return SPNET_OK;
  if (k < 1 || k > 32) return fail(SPNET_ERR_BAD_INPUT, "star solves: 1..32 right-hand sides at once");
  if (batch_bytes(pc, 1) > SOLVE_SMEM)
    return fail(SPNET_ERR_UNSUPPORTED, "star solves: the largest star's solve vector for " + std::to_string(k) +
                                           " right-hand sides exceeds a block's shared memory");
  note_launch();
  ProfScope ps(KID_STARS, s);
  if (pc->precision == SPNET_PREC_FP64) return launch_batch_t<double>(pc, R, k, (double*)W, err, done, s);
  return launch_batch_t<float>(pc, R, k, (float*)W, err, done, s);
}

// Size class of the star solve: the solve precision, half-octaves of the star count, the
// largest star and the record bytes per star (the tuner's cache keeps the warps per star
// timed best for each, per device).
static TuneClass map_class(const spnet_pc_s* pc) {
  const int vb = pc->precision == SPNET_PREC_FP64 ? 8 : 4;
  return TuneClass{{vb, half_octave(pc->S), half_octave(pc->max_star), half_octave((double)pc->stream_bytes / pc->S)}};
}

// a cached choice; a loaded file may hold any number
static int known_warps(int v) { return v < 1 ? 1 : v > 8 ? 8 : v; }

// headers, places and records of all stars (the inverses are in place already)
int star_records_fill(spnet_pc_s* pc) {
  cudaStream_t s = pc->op->stream;
  const int S = pc->S;
  const int vb = pc->precision == SPNET_PREC_FP64 ? 8 : 4;
  SPNET_TRY(pc->mem.alloc(&pc->shdr, (size_t)S * sizeof(StarHdr)));
  SPNET_TRY(pc->mem.get(&pc->iperm_star, pc->sum_s > 0 ? pc->sum_s : 1));
  pc->stream_bytes = (int64_t)S * (int64_t)sizeof(StarHdr) + 2 * pc->sum_s + pc->srec_bytes;
  const unsigned gw = (unsigned)((S + 3) / 4);
  note_launch();
  auto fill = [&](auto kern) {
    kern<<<gw, 128, 0, s>>>(S, mesh_of_pc(pc), pc->pool, pc->star_off, pc->star_mesh, pc->elem_ptr, pc->star_ptr,
                            pc->ford, pc->bord, pc->rec_size, (const int4*)pc->rec_counts, pc->rec_first, pc->rec_base,
                            (StarHdr*)pc->shdr, pc->rec_place, pc->iperm_star, pc->srec, pc->rec_off, pc->star_rule,
                            pc->patch_w, pc->N);
  };
  if (vb == 8) fill(k_record_fill<double>);
  else fill(k_record_fill<float>);
  SPNET_CUDA_TRY(cudaGetLastError());
  pc->ford = pc->bord = nullptr;
  pc->core_off = nullptr;
  pc->core_kc = nullptr;
  pc->rec_counts = nullptr;
  pc->rec_place = nullptr;
  pc->rec_first = pc->rec_base = nullptr;
  // a vector of up to 200 KB less a few (the limit of star_batch_max_k's layout)
  if (8 * (80 + 32 * vb) + 80 + align_up((int64_t)vb * pc->max_star, 16) > 200 * 1024 || !solve_fits(pc, 1, 1))
    return fail(SPNET_ERR_UNSUPPORTED, "setup_preconditioner: a star too large for the solve's shared memory");
  // a block per star: with few stars per SM eight warps shorten the longest star
  int v = 0;
  if (pc->star_map > 0) pc->solve_wpb = pc->star_map;
  else if (S < 4 * num_sms()) pc->solve_wpb = 8;
  else pc->solve_wpb = tune_peek(TUNE_STAR_WARPS, map_class(pc), &v) ? known_warps(v) : 4;
  return SPNET_OK;
}

// SPNET_ERR_TIMEOUT where a wait of the solves just timed ran out: their times say nothing.  The
// flag is cleared, so that it is not charged to the first call on the preconditioner.
static int timed_waits(spnet_pc_s* pc) {
  cudaStream_t s = pc->op->stream;
  int err = 0;
  SPNET_CUDA_TRY(cudaMemcpyAsync(&err, &pc->scal->err, sizeof(int), cudaMemcpyDeviceToHost, s));
  SPNET_CUDA_TRY(cudaMemsetAsync(&pc->scal->err, 0, sizeof(int), s));
  SPNET_CUDA_TRY(cudaStreamSynchronize(s));
  return err ? fail(SPNET_ERR_TIMEOUT, "setup_preconditioner: a device wait of the timed star solves ran out") : SPNET_OK;
}

int star_map_tune(spnet_pc_s* pc) {
  if (pc->S == 0 || pc->star_map > 0) return SPNET_OK;  // fixed
  if (pc->S < 4 * num_sms()) return SPNET_OK;           // a few stars per SM: see star_records_fill
  const TuneClass key = map_class(pc);
  {
    int v = 0;
    if (tune_begin(TUNE_STAR_WARPS, key, &v)) {  // known
      pc->solve_wpb = known_warps(v);
      return SPNET_OK;
    }
  }
  cudaStream_t s = pc->op->stream;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaMemsetAsync(pc->vtmp, 0, sizeof(double) * pc->N, s) != cudaSuccess || cudaEventCreate(&e0) != cudaSuccess ||
      cudaEventCreate(&e1) != cudaSuccess) {
    if (e0) cudaEventDestroy(e0);
    tune_end(TUNE_STAR_WARPS, key, 0);
    return fail(SPNET_ERR_CUDA, "setup_preconditioner: timing the star solve failed");
  }
  int best = 4, rc = SPNET_OK;
  float best_ms = 0.0f;
  for (int w : {4, 2, 1, 8}) {
    pc->solve_wpb = w;
    launch_star_solve(pc, pc->vtmp, nullptr, nullptr, nullptr, s);  // warm-up
    cudaEventRecord(e0, s);
    for (int rep = 0; rep < 3; ++rep) launch_star_solve(pc, pc->vtmp, nullptr, nullptr, nullptr, s);
    cudaEventRecord(e1, s);
    float ms = 0.0f;
    if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
      rc = fail(SPNET_ERR_CUDA, "setup_preconditioner: timing the star solve failed");
      break;
    }
    if (w == 4 || ms < 0.97f * best_ms) {
      best = w;
      best_ms = ms;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc == SPNET_OK) rc = timed_waits(pc);
  pc->solve_wpb = best;
  tune_end(TUNE_STAR_WARPS, key, rc == SPNET_OK ? best : 0);
  return rc;
}

// Right-hand sides per block of the batched star solve (2 or 4), timed once per size class
// (precision and block width, half-octaves of the star count and the largest star, whether
// dense blocks are inverted) on the preconditioner's own stars, for the block width the
// preconditioner steps (batch_rhs).
int batch_jw_tune(spnet_pc_s* pc) {
  pc->batch_jw = 0;
  const int k = pc->batch_rhs < 32 ? pc->batch_rhs : 32;
  if (pc->S == 0 || k < 4 || !solve_fits(pc, 4, 1)) return SPNET_OK;
  const int kp = k <= 4 ? 4 : k <= 8 ? 8 : k <= 16 ? 16 : 32;
  const int vb = pc->precision == SPNET_PREC_FP64 ? 8 : 4;
  const TuneClass key{{vb * 64 + kp, half_octave(pc->S), half_octave(pc->max_star), pc->panel_stars > 0 ? 1 : 0}};
  int v = 0;
  if (tune_begin(TUNE_STAR_COLUMNS, key, &v)) {
    pc->batch_jw = v == 2 ? 2 : 4;  // whatever a loaded file holds
    return SPNET_OK;
  }
  cudaStream_t s = pc->op->stream;
  DevArena tmp;
  tmp.stream = s;
  struct Guard {
    DevArena& a;
    ~Guard() { a.free_all(); }
  } guard{tmp};
  const int64_t rbytes = 8ll * pc->N * k, wbytes = (int64_t)vb * pc->sum_s * k;
  int best = 4, rc = SPNET_OK;
  if (rbytes + wbytes > (2ll << 30)) {  // too large to time on the side: the default
    tune_end(TUNE_STAR_COLUMNS, key, best);
    pc->batch_jw = best;
    return SPNET_OK;
  }
  double* R = nullptr;
  void* W = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if ((rc = tmp.get(&R, (size_t)pc->N * k)) || (rc = tmp.alloc(&W, (size_t)wbytes)) ||
      cudaMemsetAsync(R, 0, (size_t)rbytes, s) != cudaSuccess || cudaEventCreate(&e0) != cudaSuccess ||
      cudaEventCreate(&e1) != cudaSuccess) {
    if (e0) cudaEventDestroy(e0);
    tune_end(TUNE_STAR_COLUMNS, key, 0);
    return rc ? rc : fail(SPNET_ERR_CUDA, "setup_preconditioner: timing the batched star solve failed");
  }
  float best_ms = 0.0f;
  for (int jw : {4, 2}) {
    pc->batch_jw = jw;
    rc = launch_star_batch(pc, R, k, W, &pc->scal->err, nullptr, s);  // warm-up
    cudaEventRecord(e0, s);
    for (int rep = 0; rep < 2 && rc == SPNET_OK; ++rep) rc = launch_star_batch(pc, R, k, W, &pc->scal->err, nullptr, s);
    cudaEventRecord(e1, s);
    float ms = 0.0f;
    if (rc != SPNET_OK || cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) {
      if (rc == SPNET_OK) rc = fail(SPNET_ERR_CUDA, "setup_preconditioner: timing the batched star solve failed");
      break;
    }
    if (jw == 4 || ms < 0.95f * best_ms) {  // the narrower one must beat four per block by 5 %
      best = jw;
      best_ms = ms;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc == SPNET_OK) rc = timed_waits(pc);
  tune_end(TUNE_STAR_COLUMNS, key, rc == SPNET_OK ? best : 0);
  pc->batch_jw = rc == SPNET_OK ? best : 0;
  return rc;
}

}  // namespace spnet
