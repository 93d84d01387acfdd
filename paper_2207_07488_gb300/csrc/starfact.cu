// Exact local solves on the stars (Section 4.1, eq. defPj): the factors of
//   A_j = E_j^T A E_j
// for every star j at once (the solves are in starsolve.cu).
//
// Each A_j is factored A_j = L_j L_j^T (sparse Cholesky) in an elimination order built in
// rounds: every round eliminates an independent set of nodes of small degree in the current
// elimination graph (their fill is added before the next round).  Nodes eliminated in one
// round do not couple in L, so a round is a level of the triangular solves.  When few nodes
// are left (tail_nodes), or the remaining graph gets dense, the rest becomes one dense block
// whose inverse is formed (k_star_core) and applied as a product.
//
// Pass 1 (symbolic) computes the order, levels and the structure of L in column form (for the
// backward solve) and in row form (forward solve) and places each star's blob in a pool; pass
// 2 (numeric) fills the values level by level, left-looking in FP64; pass 3 forms the blocks'
// inverses in FP64.  Everything is rounded to FP32 only when it is written into the solve's
// records of the mixed precision.
#include <algorithm>
#include <climits>
#include <atomic>
#include <cmath>

#include "star_blob.cuh"

namespace spnet {

// Adjacency slots per node during elimination: 32 (64 for planar networks with stars beyond
// 1024 dofs: their elimination would otherwise stop at blocks of 200 to 350 nodes, whose
// inverses take c^3 / 2 FP64 operations: 17.5 against 2.4 ms on a 119,000-node 2D network, for
// 12.7 instead of 7.3 ms of elimination), or for matrices with longer rows
// (the beam model couples a node with its neighbours' neighbours, up to ~60 entries
// a row) three times as many as the longest row holds off the diagonal, rounded up to
// a multiple of 32 and at most 192.  The rest of a star turns dense once the minimum
// degree passes three quarters of the capacity.  A node whose list overflows is frozen:
// it is kept for the dense block and the elimination goes on around it (its own list
// stays incomplete; every other list stays complete, and a fill pair is looked up in the
// list of a member that is not frozen).  On the beam model this shrinks the dense block of
// a 7,400-dof star from about 3,700 dofs to about 900.
constexpr int CAP_WIDE_STAR = 1024;
constexpr int CAP_MIN = 32;
constexpr int CAP_MAX = 192;
inline int adjacency_cap(int max_offdiag, int dim, int max_star) {
  if (max_offdiag <= 24) return dim == 2 && max_star > CAP_WIDE_STAR ? 2 * CAP_MIN : CAP_MIN;
  int c = (3 * max_offdiag + 31) / 32 * 32;
  return c < CAP_MAX ? c : CAP_MAX;
}
constexpr int ST_FROZEN = -2;  // elimination state of a frozen node (alive: -1; eliminated: position)
__host__ __device__ inline int switch_degree(int cap) { return cap - cap / 4; }
// Dense blocks of up to CORE_INV nodes are inverted at set-up (k_star_core) and applied as
// one product; larger ones (the beam model's largest stars) are eliminated a node a level.
constexpr int CORE_INV = 1024;
constexpr int CORE_FIRST = 256;  // capacity of the first attempt where blocks are not inverted
// Nodes left at which the elimination stops for the dense block.  Its inverse costs c^2
// coefficients a solve and c^3 / 2 FP64 operations at set-up, and saves the levels of the last c
// nodes, most of them of one or two rows.  One solve, 3D workload (341 dofs a star): 34 us with
// 8 to 16 nodes, 33 with 24, 32 with 32, 34 with 48; structural workload (2,419 dofs): 168 us
// with at most 64, 159 with 128, 170 with 192.
// At most 128 (tail_most); 64 for 3D networks of few stars, where a star has its SM to itself and the
// block's c^3 / 4 cycles are waited for, while the levels saved are few.  Set-up and one solve, 128 and
// 64: 1,333 dofs in one star 2.68, 2.52 ms; 5,356 in 8 stars 3.77, 3.34, in 20 stars 3.73, 3.36;
// 80,788 in 64 stars 21.2, 21.1; 110,699 in 125 stars 18.1, 18.5.  2D: 4,972 in 9 stars 6.35, 6.78.
__host__ __device__ inline int tail_nodes(int n, int most) {
  const int t = n / 8;
  return t < 32 ? 32 : t > most ? most : t;
}
inline int tail_most(int dim, int64_t stars, int sms) { return dim == 3 && 4 * stars <= sms ? 64 : 128; }

// One elimination round takes an independent set among the nodes of degree at most
// round_degree(md), md the least degree left.  A round is a level of the triangular
// solves, so few large rounds matter as much as little fill: taking nodes up to twice the
// least degree (two above it while that is small), and breaking ties between neighbours by
// a scrambled rank instead of the node number (on a grid the numbers order a round into
// wavefronts of one or two nodes), costs 0 to 5 % more entries for a third to a sixth of the
// levels: ahead of a dense block of 128 nodes 25 instead of 88 levels on the stars of a
// 330,000-node 2D network, 24 instead of 181 on the (2^9+1)^2 grid, 5 instead of 8 ahead of 32
// nodes on the 3D workload.
__host__ __device__ inline int round_degree(int md, int most) {
  const int t = md < 2 ? md + 2 : 2 * md;
  return t < most ? t : most;
}
// a bijection of 0..65535 (odd multipliers and xor-shifts): distinct nodes have distinct ranks
__host__ __device__ inline uint32_t node_rank(uint32_t t) {
  t = (t * 0x9E35u) & 0xffffu;
  t ^= t >> 7;
  t = (t * 0xC2B3u) & 0xffffu;
  return t ^ (t >> 9);
}

__host__ __device__ inline int64_t core_entries(int core_max) { return (int64_t)core_max * (core_max - 1) / 2; }

// The state of a star: its structure is to be built; built, the values are to come; done (every
// byte 1, as a memset sets it).
enum : int32_t { STAR_TODO = 0, STAR_BUILT = 2, STAR_DONE = 0x01010101 };

// What a pass over the stars counts.  Stars that did not fit their scratch or the pool, or whose
// dense block is too ill conditioned to be inverted, are left for another pass.
struct StarCount {
  int next;       // the queue of stars
  int left;       // stars left for another pass
  int need_core;  // the largest dense block among them
  int max_row;    // the longest row of K
  unsigned long long pool_more;  // bytes the stars left will take
  unsigned long long pool_top;   // bytes of the pool given out
};

struct StarArgs {
  Mesh m;
  int S;
  const int32_t* star_mesh;
  const int32_t* star_n;
  const int32_t* elem_ptr;
  const int32_t* elem_of;
  const int64_t* kptr;
  const int32_t* kcol;
  const double* kval;
  char* scratch;
  int64_t stride;  // global scratch bytes per warp
  int64_t hot;     // hot bytes per warp
  int hot_in_smem; // 1: degrees, states and marks in dynamic shared memory (k_star_symbolic_block)
  int nmax;
  int core_max;    // largest dense block the scratch holds
  char* pool;
  int64_t pool_cap;
  int64_t* star_off;
  int32_t* star_lev;
  int32_t* star_nnz;
  int32_t* star_core;
  int* flags;
  StarCount* cnt;
  int32_t* todo;   // [S] STAR_*
  int core_inv;    // largest dense block that is inverted (0: none)
  int tail_most;   // see tail_nodes
  const int32_t* noinv;  // [S] 1: a star whose block is not inverted (ill conditioned)
  int cap;            // adjacency slots per node (adjacency_cap)
  int patch;          // SPNET_PATCH_*
  const double* q1w;  // [nc][N] Q1 values (the support rule tests them against zero)
  int64_t N;
};

struct Scratch {
  int cap;
  uint16_t* nbr;     // [nmax*cap]
  uint16_t* colent;  // [nmax*cap + core_entries(core_max)]
  int32_t* deg;      // [nmax]
  int32_t* state;    // [nmax]: -1 alive, else elimination position
  int32_t* posnode;  // [nmax]
  int32_t* colstart; // [nmax+1]
  int32_t* lvl;      // [nmax+1]
  int32_t* rcnt;     // [nmax+1]
  int32_t* rstart;   // [nmax+1]
  uint8_t* sel;      // [nmax]
};

// hot arrays (adjacency, degrees, states, selection), touched in every round: in shared
// memory when they fit (k_star_symbolic), else behind the cold ones in global scratch
__host__ __device__ inline int64_t hot_bytes(int nmax, int cap) {
  return align_up(2ll * nmax * cap, 16) + align_up(8ll * nmax, 16) + align_up((int64_t)nmax, 16);
}

__host__ __device__ inline int64_t cold_bytes(int nmax, int core_max, int cap) {
  int64_t o = 2ll * ((int64_t)nmax * cap + core_entries(core_max));
  o = align_up(o, 8);
  o += 4ll * (nmax + 1) * 6;
  return align_up(o, 256);
}

__device__ inline Scratch carve(char* cold, char* hot, int nmax, int core_max, int cap) {
  Scratch s;
  s.cap = cap;
  int64_t o = 0;
  s.nbr = (uint16_t*)(hot + o);   o = align_up(o + 2ll * nmax * cap, 16);
  s.deg = (int32_t*)(hot + o);    o += 4ll * nmax;
  s.state = (int32_t*)(hot + o);  o = align_up(o + 4ll * nmax, 16);
  s.sel = (uint8_t*)(hot + o);
  o = 0;
  s.colent = (uint16_t*)(cold + o); o += 2ll * ((int64_t)nmax * cap + core_entries(core_max));
  o = align_up(o, 8);
  s.posnode = (int32_t*)(cold + o);  o += 4ll * (nmax + 1);
  s.colstart = (int32_t*)(cold + o); o += 4ll * (nmax + 1);
  s.lvl = (int32_t*)(cold + o);      o += 4ll * (nmax + 1);
  s.rcnt = (int32_t*)(cold + o);     o += 4ll * (nmax + 1);
  s.rstart = (int32_t*)(cold + o);   o += 4ll * (nmax + 1);
  return s;
}

// a star left for another pass: c nodes of its dense block as columns, of `nnz` entries the rest
// (or all: block_in)
__device__ inline void leave_star(const StarArgs& A, int flag, int n, int nlev, int nnz, int c, bool block_in = false) {
  atomicOr(A.flags, flag);
  atomicAdd(&A.cnt->left, 1);
  atomicMax(&A.cnt->need_core, c);
  atomicAdd(&A.cnt->pool_more,
            (unsigned long long)blob_layout(n, nlev, nnz + (block_in ? 0 : (int)core_entries(c))).total);
}

__device__ inline int local_of_pc(const Mesh& m, const StarElems& se, const int32_t* elem_ptr,
                                  const int32_t* elem_of, int k_multi0, int k_multi1, int k_multi2,
                                  int j) {
  int e = elem_of[j];
  int ex[3];
  elem_multi(m, e, ex);
  int km[3] = {k_multi0, k_multi1, k_multi2};
  int cp = 0;
  for (int a = 0; a < m.d; ++a) {
    int r = ex[a] - (km[a] - 1);
    if (r < 0 || r > 1) return -1;
    cp |= r << a;
  }
  return se.off[cp] + (j - elem_ptr[e]);
}

// remove the nodes eliminated by the current elimination step from the adjacency lists
// that hold them.
// Those are the lists of the round's column entries c0..c1 (the alive neighbours of the
// eliminated nodes; every other list holds alive nodes only), each marked once in sel
// (free after the round's selection) and compacted in order by the lane that meets it.
__device__ inline void compact_touched(const Scratch& W, int n, int lane, int c0, int c1) {
  for (int q = c0 + lane; q < c1; q += 32) W.sel[W.colent[q]] = 2;
  __syncwarp();
  for (int t = lane; t < n; t += 32) {
    if (W.sel[t] != 2) continue;
    W.sel[t] = 0;
    uint16_t* lst = W.nbr + (int64_t)t * W.cap;
    int c = 0, d = W.deg[t];
    for (int q = 0; q < d; ++q) {
      int u = lst[q];
      if (W.state[u] < 0) lst[c++] = (uint16_t)u;
    }
    W.deg[t] = c;
  }
  __syncwarp();
}

__global__ void __launch_bounds__(128) k_star_symbolic(StarArgs A) {
  extern __shared__ __align__(16) char sm_hot[];
  const int lane = threadIdx.x & 31;
  const int64_t wg = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  char* cold = A.scratch + wg * A.stride;
  char* hot = sm_hot + (threadIdx.x >> 5) * A.hot;
  const Scratch W = carve(cold, hot, A.nmax, A.core_max, A.cap);
  const int CAP = A.cap, SWITCH_DEG = switch_degree(A.cap);
  const unsigned FULL = 0xffffffffu;
  for (;;) {
    int s = 0;
    if (lane == 0) s = atomicAdd(&A.cnt->next, 1);
    s = __shfl_sync(FULL, s, 0);
    if (s >= A.S) break;
    if (A.todo[s] != STAR_TODO) continue;
    const int k = A.star_mesh[s];
    const int n = A.star_n[s];
    if (n > A.nmax || n > 65535) {
      if (lane == 0) atomicOr(A.flags, FLAG_STAR_BIG);
      continue;
    }
    const StarElems se = star_elems(A.m, k, A.elem_ptr);
    int km[3];
    mesh_multi(A.m, k, km);
    // adjacency of the star graph (with support patches a dof off the support is an
    // isolated node: its row of the local matrix is the identity, and its solve
    // coefficient is zero, so the star adds nothing there)
    for (int t = lane; t < n; t += 32) {
      int i = pc_of_local(se, A.elem_ptr, t);
      int cnt = 0;
      bool o = false;
      const bool tex = A.patch == SPNET_PATCH_SUPPORT && off_support(se, A.elem_ptr, A.q1w, A.N, t);
      for (int64_t q = tex ? A.kptr[i + 1] : A.kptr[i]; q < A.kptr[i + 1]; ++q) {
        int j = A.kcol[q];
        if (j == i) continue;
        int lt = local_of_pc(A.m, se, A.elem_ptr, A.elem_of, km[0], km[1], km[2], j);
        if (lt < 0) continue;
        if (A.patch == SPNET_PATCH_SUPPORT && off_support(se, A.elem_ptr, A.q1w, A.N, lt)) continue;
        if (cnt < CAP) W.nbr[(int64_t)t * CAP + cnt++] = (uint16_t)lt;
        else o = true;
      }
      W.deg[t] = cnt;
      W.state[t] = o ? ST_FROZEN : -1;
    }
    __syncwarp();
    int npos = 0, nlev = 0, ncol = 0;
    bool dense = false;
    const int core_inv = A.noinv[s] ? 0 : A.core_inv;
    const int tail = core_inv > 0 ? tail_nodes(n, A.tail_most) : 0;
    while (npos < n) {
      if (n - npos <= tail) {
        dense = true;
        break;
      }
      int md = 1 << 30;  // over the nodes that may still be eliminated
      for (int t = lane; t < n; t += 32)
        if (W.state[t] == -1) md = min(md, W.deg[t]);
      md = warp_min(md);
      if (md > SWITCH_DEG) {
        dense = true;
        break;
      }
      const int thr = round_degree(md, SWITCH_DEG);
      // independent set: candidates of degree <= thr that beat every candidate neighbour
      for (int t = lane; t < n; t += 32) {
        bool sl = false;
        if (W.state[t] == -1 && W.deg[t] <= thr) {
          sl = true;
          const int dt = W.deg[t];
          const uint32_t ht = node_rank(t);
          const uint16_t* lst = W.nbr + (int64_t)t * CAP;
          for (int q = 0; q < dt; ++q) {
            int u = lst[q];
            int du = W.deg[u];
            if (W.state[u] == -1 && du <= thr && (du < dt || (du == dt && node_rank(u) < ht))) {
              sl = false;
              break;
            }
          }
        }
        W.sel[t] = sl ? 1 : 0;
      }
      __syncwarp();
      // positions in ascending node order, columns = current neighbour lists
      const int lev_start = npos;
      W.lvl[nlev] = npos;
      for (int base = 0; base < n; base += 32) {
        int t = base + lane;
        bool sl = t < n && W.sel[t];
        unsigned b = __ballot_sync(FULL, sl);
        int dcount = sl ? W.deg[t] : 0;
        int incl = warp_incl_scan(dcount, lane);
        int tot = __shfl_sync(FULL, incl, 31);
        if (sl) {
          int pos = npos + __popc(b & ((1u << lane) - 1u));
          int cs = ncol + incl - dcount;
          W.posnode[pos] = t;
          W.colstart[pos] = cs;
          const uint16_t* lst = W.nbr + (int64_t)t * CAP;
          for (int q = 0; q < dcount; ++q) W.colent[cs + q] = lst[q];
          W.state[t] = pos;
        }
        npos += __popc(b);
        ncol += tot;
      }
      W.colstart[npos] = ncol;
      __syncwarp();
      compact_touched(W, n, lane, W.colstart[lev_start], ncol);
      // fill among the neighbours of each eliminated node: every pair (a, b) of
      // a column of this elimination step, 32 pairs at a time.  Lanes test adjacency in
      // parallel; pairs repeated inside a batch are merged; new list slots go
      // by rank among the lanes that extend the same list (deterministic).  A node
      // whose list would pass CAP entries is frozen.
      {
        int total = 0;  // pairs of the round; prefix per position in W.rstart
        for (int base = lev_start; base < npos; base += 32) {
          const int pos = base + lane;
          int c = 0;
          if (pos < npos) {
            const int d = W.colstart[pos + 1] - W.colstart[pos];
            c = d * (d - 1) / 2;
          }
          const int incl = warp_incl_scan(c, lane);
          if (pos < npos) W.rstart[pos - lev_start] = total + incl - c;
          total += __shfl_sync(FULL, incl, 31);
        }
        __syncwarp();
        const int nl = npos - lev_start;
        for (int p0 = 0; p0 < total; p0 += 32) {
          const int p = p0 + lane;
          int a = -1, b = -1;
          if (p < total) {
            int lo = 0, hi = nl - 1;  // position of pair p: last prefix <= p
            while (lo < hi) {
              const int mid = (lo + hi + 1) >> 1;
              if (W.rstart[mid] <= p) lo = mid;
              else hi = mid - 1;
            }
            const int pos = lev_start + lo;
            int l = p - W.rstart[lo];
            const int cs = W.colstart[pos], d = W.colstart[pos + 1] - cs;
            int ai = 0;
            while (l >= d - 1 - ai) {
              l -= d - 1 - ai;
              ++ai;
            }
            a = W.colent[cs + ai];
            b = W.colent[cs + ai + 1 + l];
            const bool fa = W.state[a] == ST_FROZEN, fb = W.state[b] == ST_FROZEN;
            if (fa && fb) {
              a = b = -1;  // both in the dense block, where every pair is coupled
            } else {
              const int c0 = fa ? b : a, c1 = fa ? a : b;  // look up in a complete list
              const int dc = W.deg[c0];
              bool found = false;
              for (int q = 0; q < dc; ++q) found |= W.nbr[(int64_t)c0 * CAP + q] == c1;
              if (found) a = b = -1;
            }
          }
          const unsigned key = a < 0 ? 0xffffffffu : ((unsigned)min(a, b) << 16) | (unsigned)max(a, b);
          const unsigned same = __match_any_sync(FULL, key);
          const bool ins = a >= 0 && __ffs(same) - 1 == lane;
#pragma unroll
          for (int side = 0; side < 2; ++side) {  // b into the list of a, then a into the list of b
            const int x = side == 0 ? a : b, y = side == 0 ? b : a;
            const bool insx = ins && W.state[x] != ST_FROZEN;  // a frozen list takes nothing more
            const unsigned grp = __match_any_sync(FULL, insx ? (unsigned)x : 0xffffffffu);
            const int rank = __popc(grp & ((1u << lane) - 1u));
            const int dx = insx ? W.deg[x] : 0;
            __syncwarp();
            if (insx) {
              if (dx + rank < CAP) W.nbr[(int64_t)x * CAP + dx + rank] = (uint16_t)y;
              else W.state[x] = ST_FROZEN;
              if (rank == 0) W.deg[x] = min(dx + __popc(grp), CAP);
            }
            __syncwarp();
          }
        }
      }
      nlev++;
    }
    if (dense && npos < n && A.patch == SPNET_PATCH_SUPPORT) {
      // dofs off the support still alive (all of them when the first adjacency
      // overflowed) are isolated: one level of their own ahead of the dense block,
      // so that the block couples none of them
      const int p0 = npos;
      for (int base = 0; base < n; base += 32) {
        int t = base + lane;
        bool al = t < n && W.state[t] < 0 && off_support(se, A.elem_ptr, A.q1w, A.N, t);
        unsigned b = __ballot_sync(FULL, al);
        if (al) {
          int pos = npos + __popc(b & ((1u << lane) - 1u));
          W.posnode[pos] = t;
          W.colstart[pos] = ncol;
          W.state[t] = pos;
        }
        npos += __popc(b);
      }
      if (npos > p0) {
        if (lane == 0) {
          W.lvl[nlev] = p0;
          W.colstart[npos] = ncol;  // nothing may be left for the dense block
        }
        nlev++;
      }
      __syncwarp();
    }
    int core_c = 0;      // nodes of the dense block
    bool inv = false;    // it is inverted: no columns, no levels
    if (dense && npos < n) {
      // the rest, in ascending node order, one node per level, columns dense
      const int core0 = npos;
      for (int base = 0; base < n; base += 32) {
        int t = base + lane;
        bool al = t < n && W.state[t] < 0;
        unsigned b = __ballot_sync(FULL, al);
        if (al) {
          int pos = npos + __popc(b & ((1u << lane) - 1u));
          W.posnode[pos] = t;
          W.state[t] = pos;
        }
        npos += __popc(b);
      }
      const int c = n - core0;
      core_c = c;
      inv = c <= core_inv;
      if (!inv && (c > A.core_max || ncol + core_entries(c) > (int64_t)A.nmax * CAP + core_entries(A.core_max))) {
        if (lane == 0) leave_star(A, FLAG_STAR_BIG, n, nlev + c, ncol, c);
        continue;
      }
      if (inv) {
        for (int q = lane; q <= c; q += 32) W.colstart[core0 + q] = ncol;
      }
      for (int q = 0; q < c && !inv; ++q) {
        W.lvl[nlev + q] = core0 + q;
        int cs = ncol + q * (c - 1) - q * (q - 1) / 2;
        if (lane == 0) W.colstart[core0 + q] = cs;
        for (int r = q + 1 + lane; r < c; r += 32) W.colent[cs + (r - q - 1)] = (uint16_t)W.posnode[core0 + r];
      }
      if (!inv) {
        nlev += c;
        ncol += c * (c - 1) / 2;
        if (lane == 0) W.colstart[n] = ncol;
      }
      __syncwarp();
    }
    if (lane == 0) W.lvl[nlev] = inv ? n - core_c : n;
    // column entries to positions; row counts
    for (int t = lane; t <= n; t += 32) W.rcnt[t] = 0;
    __syncwarp();
    for (int q = lane; q < ncol; q += 32) {
      int pos = W.state[W.colent[q]];
      W.colent[q] = (uint16_t)pos;
      atomicAdd(&W.rcnt[pos], 1);
    }
    __syncwarp();
    int carry = 0;
    for (int base = 0; base < n; base += 32) {
      int t = base + lane;
      int v = t < n ? W.rcnt[t] : 0;
      int incl = warp_incl_scan(v, lane);
      if (t < n) W.rstart[t] = carry + incl - v;
      carry += __shfl_sync(FULL, incl, 31);
    }
    if (lane == 0) W.rstart[n] = carry;
    for (int t = lane; t < n; t += 32) W.rcnt[t] = 0;
    __syncwarp();
    // place the blob
    const BlobLayout L = blob_layout(n, nlev, ncol);
    unsigned long long off = 0;
    if (lane == 0) off = atomicAdd(&A.cnt->pool_top, (unsigned long long)L.total);
    off = __shfl_sync(FULL, off, 0);
    if ((int64_t)off + L.total > A.pool_cap) {
      if (lane == 0) leave_star(A, FLAG_POOL, n, nlev, ncol, inv ? 0 : core_c, true);
      continue;
    }
    char* blob = A.pool + off;
    if (lane == 0) {
      int32_t* hdr = (int32_t*)blob;
      hdr[0] = n;
      hdr[1] = nlev;
      hdr[2] = ncol;
      hdr[3] = inv ? core_c : 0;
      A.star_off[s] = (int64_t)off;
      A.star_lev[s] = nlev + (inv ? 1 : 0);
      A.star_nnz[s] = ncol;
      A.star_core[s] = core_c;
      A.todo[s] = STAR_BUILT;
    }
    int32_t* gidx = (int32_t*)(blob + L.gidx);
    uint16_t* perm = (uint16_t*)(blob + L.perm);
    uint16_t* lvl = (uint16_t*)(blob + L.lvl);
    uint32_t* colptr = (uint32_t*)(blob + L.colptr);
    uint16_t* colidx = (uint16_t*)(blob + L.colidx);
    uint32_t* rowptr = (uint32_t*)(blob + L.rowptr);
    uint16_t* rowidx = (uint16_t*)(blob + L.rowidx);
    int32_t* c2r = (int32_t*)(blob + L.c2r);
    for (int pos = lane; pos < n; pos += 32) {
      int t = W.posnode[pos];
      gidx[pos] = pc_of_local(se, A.elem_ptr, t);
      perm[pos] = (uint16_t)t;
    }
    for (int q = lane; q <= nlev; q += 32) lvl[q] = (uint16_t)W.lvl[q];
    for (int q = lane; q <= n; q += 32) {
      colptr[q] = (uint32_t)W.colstart[q];
      rowptr[q] = (uint32_t)W.rstart[q];
    }
    for (int q = lane; q < ncol; q += 32) colidx[q] = W.colent[q];
    // row form: columns in ascending position, so every row lists its columns ascending
    for (int v = 0; v < n; ++v) {
      const int cs = W.colstart[v], ce = W.colstart[v + 1];
      for (int q = cs + lane; q < ce; q += 32) {
        int i = W.colent[q];
        int slot = W.rstart[i] + W.rcnt[i];
        W.rcnt[i] += 1;
        rowidx[slot] = (uint16_t)v;
        c2r[q] = slot;
      }
      __syncwarp();
    }
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// The same for stars whose adjacency lists do not fit shared memory: a block of four warps per
// star.  Lists lie in global scratch; degrees, states and marks in shared memory where they fit.
// The fill of a round is added list by list instead of pair by pair: a warp takes an alive
// neighbour of the eliminated nodes, drops those from its list and appends the entries of their
// columns that it does not hold yet, told by a bitmap of the star's nodes in shared memory.  A
// list has one writer and nothing is looked up in another node's list.  (A warp per star, a pair
// at a time with a search of one member's list, is bound by the latency of those searches: 12.7
// ms on a 119,000-node 2D network, 16.4 ms on the structural workload.)
// ---------------------------------------------------------------------------
constexpr int BT = 128;  // threads of a block

__host__ __device__ inline int64_t bitmap_bytes(int nmax) { return align_up((int64_t)(nmax + 31) / 32 * 4, 16); }
__host__ __device__ inline int64_t marks_bytes(int nmax) { return align_up(9ll * nmax, 16); }  // deg, state, sel

struct BlockScan {  // per-warp totals
  int a[BT / 32], b[BT / 32];
};

__global__ void __launch_bounds__(BT) k_star_symbolic_block(StarArgs A) {
  extern __shared__ __align__(16) char sm_hot[];
  __shared__ BlockScan bsc;
  __shared__ int sh_i[2];
  __shared__ unsigned long long sh_off;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  char* cold = A.scratch + (int64_t)blockIdx.x * A.stride;
  Scratch W = carve(cold, cold + cold_bytes(A.nmax, A.core_max, A.cap), A.nmax, A.core_max, A.cap);
  uint32_t* bm = (uint32_t*)(sm_hot + wid * bitmap_bytes(A.nmax));
  if (A.hot_in_smem) {
    char* p = sm_hot + (BT / 32) * bitmap_bytes(A.nmax);
    W.deg = (int32_t*)p;
    W.state = W.deg + A.nmax;
    W.sel = (uint8_t*)(W.state + A.nmax);
  }
  const int CAP = A.cap, SWITCH_DEG = switch_degree(A.cap);
  constexpr unsigned FULL = 0xffffffffu;
  for (int i = lane; i < (A.nmax + 31) / 32; i += 32) bm[i] = 0;
  // exclusive prefix over the block of (on ? 1 : 0, v), and the totals; every thread calls
  auto scan = [&](bool on, int v, int& before_n, int& before_v, int& tot_n, int& tot_v) {
    const unsigned b = __ballot_sync(FULL, on);
    const int incl = warp_incl_scan(v, lane);
    if (lane == 31) {
      bsc.a[wid] = __popc(b);
      bsc.b[wid] = incl;
    }
    __syncthreads();
    before_n = __popc(b & ((1u << lane) - 1u));
    before_v = incl - v;
    tot_n = tot_v = 0;
#pragma unroll
    for (int w = 0; w < BT / 32; ++w) {
      if (w < wid) {
        before_n += bsc.a[w];
        before_v += bsc.b[w];
      }
      tot_n += bsc.a[w];
      tot_v += bsc.b[w];
    }
    __syncthreads();
  };
  for (;;) {
    __syncthreads();  // the previous star's last reads of sh_i
    if (tid == 0) sh_i[0] = atomicAdd(&A.cnt->next, 1);
    __syncthreads();
    const int s = sh_i[0];
    if (s >= A.S) break;
    if (A.todo[s] != STAR_TODO) continue;
    const int k = A.star_mesh[s];
    const int n = A.star_n[s];
    const StarElems se = star_elems(A.m, k, A.elem_ptr);
    int km[3];
    mesh_multi(A.m, k, km);
    const bool sup = A.patch == SPNET_PATCH_SUPPORT;
    // adjacency of the star graph (off-support dofs are isolated nodes, as above)
    for (int t = tid; t < n; t += BT) {
      const int i = pc_of_local(se, A.elem_ptr, t);
      int cnt = 0;
      bool o = false;
      const bool tex = sup && off_support(se, A.elem_ptr, A.q1w, A.N, t);
      for (int64_t q = tex ? A.kptr[i + 1] : A.kptr[i]; q < A.kptr[i + 1]; ++q) {
        const int j = A.kcol[q];
        if (j == i) continue;
        const int lt = local_of_pc(A.m, se, A.elem_ptr, A.elem_of, km[0], km[1], km[2], j);
        if (lt < 0) continue;
        if (sup && off_support(se, A.elem_ptr, A.q1w, A.N, lt)) continue;
        if (cnt < CAP) W.nbr[(int64_t)t * CAP + cnt++] = (uint16_t)lt;
        else o = true;
      }
      W.deg[t] = cnt;
      W.state[t] = o ? ST_FROZEN : -1;
    }
    __syncthreads();
    int npos = 0, nlev = 0, ncol = 0;
    bool dense = false;
    const int core_inv = A.noinv[s] ? 0 : A.core_inv;
    const int tail = core_inv > 0 ? tail_nodes(n, A.tail_most) : 0;
    while (npos < n) {
      if (n - npos <= tail) {
        dense = true;
        break;
      }
      int md = 1 << 30;  // over the nodes that may still be eliminated
      for (int t = tid; t < n; t += BT)
        if (W.state[t] == -1) md = min(md, W.deg[t]);
      md = warp_min(md);
      if (lane == 0) bsc.a[wid] = md;
      __syncthreads();
      md = min(min(bsc.a[0], bsc.a[1]), min(bsc.a[2], bsc.a[3]));
      if (md > SWITCH_DEG) {
        dense = true;
        __syncthreads();
        break;
      }
      const int thr = round_degree(md, SWITCH_DEG);
      // independent set: candidates of degree <= thr that beat every candidate neighbour
      for (int t = tid; t < n; t += BT) {
        bool sl = false;
        if (W.state[t] == -1 && W.deg[t] <= thr) {
          sl = true;
          const int dt = W.deg[t];
          const uint32_t ht = node_rank(t);
          const uint16_t* lst = W.nbr + (int64_t)t * CAP;
          for (int q = 0; q < dt; ++q) {
            const int u = lst[q];
            const int du = W.deg[u];
            if (W.state[u] == -1 && du <= thr && (du < dt || (du == dt && node_rank(u) < ht))) {
              sl = false;
              break;
            }
          }
        }
        W.sel[t] = sl ? 1 : 0;
      }
      __syncthreads();
      // positions in ascending node order, columns = current neighbour lists
      const int lev_start = npos;
      if (tid == 0) W.lvl[nlev] = npos;
      for (int base = 0; base < n; base += BT) {
        const int t = base + tid;
        const bool sl = t < n && W.sel[t] == 1;
        const int dcount = sl ? W.deg[t] : 0;
        int bn, bv, tn, tv;
        scan(sl, dcount, bn, bv, tn, tv);
        if (sl) {
          const int pos = npos + bn, cs = ncol + bv;
          W.posnode[pos] = t;
          W.colstart[pos] = cs;
          const uint16_t* lst = W.nbr + (int64_t)t * CAP;
          for (int q = 0; q < dcount; ++q) W.colent[cs + q] = lst[q];
          W.state[t] = pos;
        }
        npos += tn;
        ncol += tv;
      }
      if (tid == 0) W.colstart[npos] = ncol;
      __syncthreads();
      // the alive neighbours of the eliminated nodes, each marked once
      for (int q = W.colstart[lev_start] + tid; q < ncol; q += BT) W.sel[W.colent[q]] = 2;
      __syncthreads();
      for (int base = wid * 32; base < n; base += BT) {
        const int t0 = base + lane;
        unsigned todo = __ballot_sync(FULL, t0 < n && W.sel[t0] == 2 && W.state[t0] == -1);
        while (todo) {
          const int a = base + __ffs(todo) - 1;
          todo &= todo - 1;
          uint16_t* lst = W.nbr + (int64_t)a * CAP;
          const int d = W.deg[a];
          constexpr int MB = CAP_MAX / 32;
          int ent[MB], est[MB];
#pragma unroll
          for (int b = 0; b < MB; ++b) {
            const int q = b * 32 + lane;
            ent[b] = q < d ? lst[q] : -1;
            est[b] = ent[b] >= 0 ? W.state[ent[b]] : -1;
          }
          __syncwarp();
          if (lane == 0) atomicOr(&bm[a >> 5], 1u << (a & 31));
          int cnt = 0;
#pragma unroll
          for (int b = 0; b < MB; ++b) {  // kept entries move up, in order
            const bool keep = ent[b] >= 0 && est[b] < 0;
            const unsigned bal = __ballot_sync(FULL, keep);
            if (keep) {
              lst[cnt + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)ent[b];
              atomicOr(&bm[ent[b] >> 5], 1u << (ent[b] & 31));
            }
            cnt += __popc(bal);
          }
          __syncwarp();
#pragma unroll
          for (int b = 0; b < MB; ++b) {  // the columns of the eliminated ones
            unsigned gone = __ballot_sync(FULL, ent[b] >= 0 && est[b] >= 0);
            while (gone) {
              const int src = __ffs(gone) - 1;
              gone &= gone - 1;
              const int pos = __shfl_sync(FULL, est[b], src);
              const int ce = W.colstart[pos + 1];
              for (int q0 = W.colstart[pos]; q0 < ce; q0 += 32) {
                const int u = q0 + lane < ce ? W.colent[q0 + lane] : -1;
                const bool add = u >= 0 && !((bm[u >> 5] >> (u & 31)) & 1u);
                const unsigned bal = __ballot_sync(FULL, add);
                if (add) {
                  const int at = cnt + __popc(bal & ((1u << lane) - 1u));
                  if (at < CAP) {
                    lst[at] = (uint16_t)u;
                    atomicOr(&bm[u >> 5], 1u << (u & 31));
                  }
                }
                cnt += __popc(bal);
                __syncwarp();
              }
            }
          }
          // a list past its slots: the node waits for the dense block (entries that did not fit
          // set no bit)
          if (lane == 0) {
            W.deg[a] = cnt < CAP ? cnt : CAP;
            if (cnt > CAP) W.state[a] = ST_FROZEN;
            bm[a >> 5] = 0;
          }
          const int dn = cnt < CAP ? cnt : CAP;
          for (int q = lane; q < dn; q += 32) bm[lst[q] >> 5] = 0;
          __syncwarp();
        }
      }
      __syncthreads();
      nlev++;
    }
    auto place_rest = [&](bool off_only) {
      for (int base = 0; base < n; base += BT) {
        const int t = base + tid;
        const bool al = t < n && W.state[t] < 0 && (!off_only || off_support(se, A.elem_ptr, A.q1w, A.N, t));
        int bn, bv, tn, tv;
        scan(al, 0, bn, bv, tn, tv);
        if (al) {
          W.posnode[npos + bn] = t;
          W.colstart[npos + bn] = ncol;
          W.state[t] = npos + bn;
        }
        npos += tn;
      }
    };
    if (dense && npos < n && sup) {  // off-support dofs left: a level of their own
      const int p0 = npos;
      place_rest(true);
      if (npos > p0) {
        if (tid == 0) {
          W.lvl[nlev] = p0;
          W.colstart[npos] = ncol;
        }
        nlev++;
      }
      __syncthreads();
    }
    int core_c = 0;    // nodes of the dense block
    bool inv = false;  // it is inverted: no columns, no levels
    if (dense && npos < n) {
      const int core0 = npos, c = n - core0;
      core_c = c;
      inv = c <= core_inv;
      if (!inv && (c > A.core_max || ncol + core_entries(c) > (int64_t)A.nmax * CAP + core_entries(A.core_max))) {
        if (tid == 0) leave_star(A, FLAG_STAR_BIG, n, nlev + c, ncol, c);
        continue;
      }
      place_rest(false);
      __syncthreads();
      if (inv) {
        if (tid == 0) W.colstart[n] = ncol;
      } else {
        for (int q = wid; q < c; q += BT / 32) {
          const int cs = ncol + q * (c - 1) - q * (q - 1) / 2;
          if (lane == 0) {
            W.lvl[nlev + q] = core0 + q;
            W.colstart[core0 + q] = cs;
          }
          for (int r = q + 1 + lane; r < c; r += 32) W.colent[cs + (r - q - 1)] = (uint16_t)W.posnode[core0 + r];
        }
        nlev += c;
        ncol += c * (c - 1) / 2;
        if (tid == 0) W.colstart[n] = ncol;
      }
    }
    if (tid == 0) W.lvl[nlev] = inv ? n - core_c : n;
    // column entries to positions; row counts and starts
    for (int t = tid; t <= n; t += BT) W.rcnt[t] = 0;
    __syncthreads();
    for (int q = tid; q < ncol; q += BT) {
      const int pos = W.state[W.colent[q]];
      W.colent[q] = (uint16_t)pos;
      atomicAdd(&W.rcnt[pos], 1);
    }
    __syncthreads();
    int carry = 0;
    for (int base = 0; base < n; base += BT) {
      const int t = base + tid;
      int bn, bv, tn, tv;
      scan(false, t < n ? W.rcnt[t] : 0, bn, bv, tn, tv);
      if (t < n) W.rstart[t] = carry + bv;
      carry += tv;
    }
    if (tid == 0) W.rstart[n] = carry;
    for (int t = tid; t < n; t += BT) W.rcnt[t] = 0;
    // place the blob
    const BlobLayout L = blob_layout(n, nlev, ncol);
    if (tid == 0) sh_off = atomicAdd(&A.cnt->pool_top, (unsigned long long)L.total);
    __syncthreads();
    const unsigned long long off = sh_off;
    if ((int64_t)off + L.total > A.pool_cap) {
      if (tid == 0) leave_star(A, FLAG_POOL, n, nlev, ncol, inv ? 0 : core_c, true);
      continue;
    }
    char* blob = A.pool + off;
    if (tid == 0) {
      int32_t* hdr = (int32_t*)blob;
      hdr[0] = n;
      hdr[1] = nlev;
      hdr[2] = ncol;
      hdr[3] = inv ? core_c : 0;
      A.star_off[s] = (int64_t)off;
      A.star_lev[s] = nlev + (inv ? 1 : 0);
      A.star_nnz[s] = ncol;
      A.star_core[s] = core_c;
      A.todo[s] = STAR_BUILT;
    }
    int32_t* gidx = (int32_t*)(blob + L.gidx);
    uint16_t* perm = (uint16_t*)(blob + L.perm);
    uint16_t* lvl = (uint16_t*)(blob + L.lvl);
    uint32_t* colptr = (uint32_t*)(blob + L.colptr);
    uint16_t* colidx = (uint16_t*)(blob + L.colidx);
    uint32_t* rowptr = (uint32_t*)(blob + L.rowptr);
    uint16_t* rowidx = (uint16_t*)(blob + L.rowidx);
    int32_t* c2r = (int32_t*)(blob + L.c2r);
    unsigned long long* put = (unsigned long long*)(blob + L.rowval);  // (column, entry) of a row, unordered
    for (int pos = tid; pos < n; pos += BT) {
      const int t = W.posnode[pos];
      gidx[pos] = pc_of_local(se, A.elem_ptr, t);
      perm[pos] = (uint16_t)t;
    }
    for (int q = tid; q <= nlev; q += BT) lvl[q] = (uint16_t)W.lvl[q];
    for (int q = tid; q <= n; q += BT) {
      colptr[q] = (uint32_t)W.colstart[q];
      rowptr[q] = (uint32_t)W.rstart[q];
    }
    for (int q = tid; q < ncol; q += BT) colidx[q] = W.colent[q];
    // row form: the entries of each row in any order, then by column (every row lists its
    // columns ascending)
    for (int v = wid; v < n; v += BT / 32)
      for (int q = W.colstart[v] + lane; q < W.colstart[v + 1]; q += 32) {
        const int i = W.colent[q];
        put[W.rstart[i] + atomicAdd(&W.rcnt[i], 1)] = ((unsigned long long)v << 32) | (unsigned)q;
      }
    __syncthreads();
    for (int i = wid; i < n; i += BT / 32) {
      const int r0 = W.rstart[i], r1 = W.rstart[i + 1];
      for (int q = r0 + lane; q < r1; q += 32) {
        const unsigned long long e = put[q];
        int rank = 0;
        for (int p = r0; p < r1; ++p) rank += put[p] < e;
        rowidx[r0 + rank] = (uint16_t)(e >> 32);
        c2r[(unsigned)e] = r0 + rank;
      }
    }
    __syncthreads();
  }
}

// the longest row of K (entries), for the adjacency capacity
__global__ void k_max_row(int64_t n, const int64_t* __restrict__ ptr, int* out) {
  int m = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    m = max(m, (int)(ptr[i + 1] - ptr[i]));
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

__device__ inline double k_entry(const int64_t* kptr, const int32_t* kcol, const double* kval, int row,
                                 int col) {
  int64_t lo = kptr[row], hi = kptr[row + 1] - 1;
  while (lo <= hi) {
    int64_t mid = (lo + hi) >> 1;
    int c = kcol[mid];
    if (c == col) return kval[mid];
    if (c < col) lo = mid + 1; else hi = mid - 1;
  }
  return 0.0;
}

// A group of TPS threads per star (a warp, four stars to a block; or the whole
// block of 128 when stars are large): a wide level gives a column to each
// thread, a narrow one (the dense block: one node per level) takes its columns
// in turn with their entries across the threads; a barrier ends each level.
constexpr int NT = 128;

template <int TPS>
__device__ __forceinline__ void group_sync() {
  if constexpr (TPS == 32) __syncwarp();
  else __syncthreads();
}

template <int TPS>
__global__ void __launch_bounds__(NT) k_star_numeric(int S, char* pool, const int64_t* star_off, const int32_t* todo,
                                                     const int64_t* kptr, const int32_t* kcol,
                                                     const double* kval, int* flags) {
  constexpr int GPB = NT / TPS;  // stars per block at a time
  const int tid = threadIdx.x % TPS;
  for (int64_t s = (int64_t)blockIdx.x * GPB + threadIdx.x / TPS; s < S; s += (int64_t)gridDim.x * GPB) {
    if (todo[s] != STAR_BUILT) continue;  // uniform over the group
    const Blob B = blob_at(pool + star_off[s]);
    const int nlev = B.nlev;
    const int32_t *gidx = B.gidx, *c2r = B.c2r;
    const uint16_t *lvl = B.lvl, *colidx = B.colidx, *rowidx = B.rowidx;
    const uint32_t *colptr = B.colptr, *rowptr = B.rowptr;
    double *rowv = B.rowv, *colv = B.colv, *invd = B.invd;
    bool bad = false;
    // L_iv = (K_iv - sum_k L_vk L_ik) / L_vv for the entries of column v: a
    // merge of the sparse rows v and i (only earlier levels meet there)
    auto entries = [&](int v, int gv, double inv, uint32_t q0, uint32_t q1, uint32_t dq) {
      const uint32_t rv0 = rowptr[v], rv1 = rowptr[v + 1];
      for (uint32_t q = q0; q < q1; q += dq) {
        const int i = colidx[q];
        double a = k_entry(kptr, kcol, kval, gv, gidx[i]);
        uint32_t kv = rv0, ki = rowptr[i];
        const uint32_t ki1 = rowptr[i + 1];
        while (kv < rv1 && ki < ki1) {
          const int uv = rowidx[kv], ui = rowidx[ki];
          if (uv == ui) {
            a -= rowv[kv] * rowv[ki];
            ++kv;
            ++ki;
          } else if (uv < ui) {
            ++kv;
          } else {
            ++ki;
          }
        }
        const double lval = a * inv;
        colv[q] = lval;
        rowv[c2r[q]] = lval;
      }
    };
    auto pivot = [&](int v, int gv) {
      double d = k_entry(kptr, kcol, kval, gv, gv);
      for (uint32_t q = rowptr[v]; q < rowptr[v + 1]; ++q) d -= rowv[q] * rowv[q];
      if (!(d > 0.0)) {
        bad = true;
        d = 1.0;
      }
      return 1.0 / sqrt(d);
    };
    for (int l = 0; l < nlev; ++l) {
      const int v0 = lvl[l], v1 = lvl[l + 1];
      if (v1 - v0 >= 32) {  // a wide level: a column per thread
        for (int v = v0 + tid; v < v1; v += TPS) {
          const int gv = gidx[v];
          const double inv = pivot(v, gv);
          invd[v] = inv;
          entries(v, gv, inv, colptr[v], colptr[v + 1], 1);
        }
      } else {  // a narrow level: its columns in turn, their entries across the threads
        for (int v = v0; v < v1; ++v) {
          const int gv = gidx[v];
          const double inv = pivot(v, gv);  // every thread the same sum
          if (tid == 0) invd[v] = inv;
          entries(v, gv, inv, colptr[v] + tid, colptr[v + 1], TPS);
        }
      }
      group_sync<TPS>();
    }
    const bool any_bad = TPS == 32 ? __any_sync(0xffffffffu, bad) : __syncthreads_or(bad);
    if (any_bad && tid == 0) atomicOr(flags, FLAG_NOT_SPD);
    group_sync<TPS>();
  }
}

// ---------------------------------------------------------------------------
// The inverse of the dense block that ends a star's elimination.  With S the Schur
// complement of the block (c x c, FP64), S_ij = K_ij - sum_u L_iu L_ju over the columns u
// outside it, the solve applies S^{-1} as one product: c^2 coefficients read once, where the
// two triangular solves read as many in 2c dependent steps.  S is swept in place (symmetric
// Gauss-Jordan on its lower triangle: pivot k maps S_ij -> S_ij - S_ik S_kj / S_kk, after c
// pivots S holds -S^{-1}; S is SPD, so no pivoting) and rounded to the solve's precision
// into the star's records.
// Bound by the FP64 pipe (c^3 / 2 multiply-adds at two a cycle and SM), so the rank-1
// updates from shared memory cost nothing extra; but a warp's FP64 instruction takes 16 cycles
// however few of its lanes matter, so the division is left to the warps that hold the column and
// the column is scaled once (every warp dividing and every row scaling its own factor cost more
// than the updates of a 42-node block: 1.42 ms on the 3D workload, 0.85 now).  A block of 256
// threads takes a star; the triangle lies in shared memory up to CORE_SMEM nodes, else in a slab of global memory.
// ---------------------------------------------------------------------------
constexpr int CORE_SMEM = 224;  // 224 * 225 / 2 * 8 B = 201,600 B
// The rounded inverse S^{-1} + E, |E| <= eps |S^{-1}|, keeps its stiff modes only while eps k
// is small, k = max_i S_ii (S^{-1})_ii (scale invariant; networks: 1e2 to 1e4).  Beyond these
// limits (the beam model, whose K spans 13 decades) the block is eliminated a node a level:
// the product of rounded triangular factors perturbs the soft modes instead, which a
// preconditioner bears.
constexpr double KAPPA32 = 1e5, KAPPA64 = 1e10;
constexpr int CORE_TC = 32;     // smallest block counted in spnet_pc_info.panel_stars

template <class T, bool SMEM>
__global__ void __launch_bounds__(256) k_star_core(int S, char* pool, const int64_t* __restrict__ star_off,
                                                   const int64_t* __restrict__ kptr, const int32_t* __restrict__ kcol,
                                                   const double* __restrict__ kval, const int64_t* __restrict__ coff,
                                                   const int32_t* __restrict__ ckc, char* __restrict__ recs,
                                                   double* slab, int64_t slab_n, int lo, int hi, int32_t* noinv,
                                                   int32_t* todo, StarCount* cnt) {
  extern __shared__ __align__(16) double sm_core[];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int s = blockIdx.x; s < S; s += gridDim.x) {
    const Blob B = blob_at(pool + star_off[s]);
    const int c = B.c;
    if (c <= lo || c > hi) continue;  // uniform over the block
    double* col = sm_core;            // the pivot's column
    double* dg = sm_core + c;         // S's diagonal
    double* uc = sm_core + 2 * c;     // -1 / pivot times the pivot's column
    double* A = SMEM ? sm_core + 3 * c : slab + (int64_t)blockIdx.x * slab_n;  // row i at i (i + 1) / 2
    const int core0 = B.n - c;
    const int64_t tri = (int64_t)c * (c + 1) / 2;
    for (int64_t e = tid; e < tri; e += 256) {
      int i = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);  // a guess
      while ((int64_t)i * (i + 1) / 2 > e) --i;
      while ((int64_t)(i + 1) * (i + 2) / 2 <= e) ++i;
      const int j = (int)(e - (int64_t)i * (i + 1) / 2);
      A[e] = k_entry(kptr, kcol, kval, B.gidx[core0 + i], B.gidx[core0 + j]);
    }
    __syncthreads();
    // S_i: -= L_iu L_ju over the entries u of row i, j those of column u in the block: a warp
    // per row, so every row has one writer and a fixed order (merging the rows of every pair
    // took most of this kernel: rows hold tens of entries, columns a handful in the block)
    for (int i = wid; i < c; i += 8) {
      double* row = A + (int64_t)i * (i + 1) / 2;
      const uint32_t p1 = B.rowptr[core0 + i + 1];
      for (uint32_t p = B.rowptr[core0 + i]; p < p1; ++p) {
        const int u = B.rowidx[p];
        const double l = -B.rowv[p];
        const uint32_t q1 = B.colptr[u + 1];
        for (uint32_t q = B.colptr[u] + lane; q < q1; q += 32) {
          const int j = (int)B.colidx[q] - core0;
          if (j >= 0 && j <= i) row[j] = fma(l, B.colv[q], row[j]);
        }
        __syncwarp();
      }
    }
    __syncthreads();
    for (int i = tid; i < c; i += 256) dg[i] = A[(int64_t)i * (i + 1) / 2 + i];
    bool bad = false;
    for (int k = 0; k < c; ++k) {
      if (tid < c) {
        double piv = A[(int64_t)k * (k + 1) / 2 + k];
        if (!(piv > 0.0)) {
          bad = true;
          piv = 1.0;
        }
        const double ip = 1.0 / piv;
        for (int i = tid; i < c; i += 256) {
          const int hi2 = i > k ? i : k, lo2 = i > k ? k : i;
          const double v = A[(int64_t)hi2 * (hi2 + 1) / 2 + lo2];
          col[i] = v;
          uc[i] = i == k ? -ip : -v * ip;
        }
      }
      __syncthreads();
      for (int i = wid; i < c; i += 8) {
        double* row = A + (int64_t)i * (i + 1) / 2;
        if (i == k) {
          for (int j = lane; j <= i; j += 32) row[j] = j == k ? uc[j] : -uc[j];
        } else {
          const double u = uc[i];
          for (int j = lane; j <= i; j += 32) row[j] = j == k ? -u : fma(u, col[j], row[j]);
        }
      }
      __syncthreads();
    }
    // a pivot lost to rounding (or a block that is not positive definite): the triangular factors
    // decide
    bool ill = bad;
    for (int i = tid; i < c; i += 256)
      ill |= !(dg[i] * -A[(int64_t)i * (i + 1) / 2 + i] <= (sizeof(T) == 4 ? KAPPA32 : KAPPA64));
    if (__syncthreads_or(ill) && tid == 0) {
      noinv[s] = 1;
      todo[s] = STAR_TODO;
      atomicAdd(&cnt->left, 1);
      atomicMax(&cnt->need_core, c);
      // (fewer where the elimination had stopped for the block: it goes on without one)
      atomicAdd(&cnt->pool_more, (unsigned long long)blob_layout(B.n, B.nlev + c, B.nnz + (int)core_entries(c)).total);
    }
    T* out = (T*)(recs + coff[s]);
    const int kc = ckc[s], cp = (c + 3) / 4 * 4;
    for (int64_t e = tid; e < (int64_t)c * cp; e += 256) {
      const int i = (int)(e % c), j = (int)(e / c);
      const int hi2 = i > j ? i : j, lo2 = i > j ? j : i;
      out[core_slot<T>(c, kc, i, j)] = j < c ? (T)-A[(int64_t)hi2 * (hi2 + 1) / 2 + lo2] : (T)0;
    }
    __syncthreads();
  }
}

// Bytes of the structures' scratch; and of the slabs below, which come when it has been given back.
constexpr int64_t SCRATCH_BUDGET = (int64_t)1 << 30, SLAB_BUDGET = (int64_t)2 << 30;

// Blocks of k_star_core with slabs of n doubles: four an SM (29,791 blocks of 339 nodes on
// average, 699 at most: set-up 5.9 s, 8.1 with two).
static int slab_blocks(int64_t stars, int64_t n, int sms) {
  int64_t g = 4ll * sms;
  if (g > stars) g = stars;
  if (g * n * 8 > SLAB_BUDGET) g = SLAB_BUDGET / (n * 8);
  return g < 1 ? 1 : (int)g;
}

template <class T>
static int core_inverses_t(spnet_pc_s* pc, DevArena& tmp, int32_t* noinv, int32_t* todo, StarCount* cnt) {
  cudaStream_t s = pc->op->stream;
  int cmax = 0, csm = 0, nbig = 0;  // largest block; largest that fits shared memory; blocks beyond
  for (int c : pc->star_inv) {
    cmax = c > cmax ? c : cmax;
    if (c <= CORE_SMEM) csm = c > csm ? c : csm;
    else ++nbig;
  }
  auto launch = [&](auto kern, int grid, size_t smem, double* slab, int64_t slab_n, int lo, int hi) -> int {
    SPNET_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    note_launch();
    kern<<<grid, 256, smem, s>>>(pc->S, pc->pool, pc->star_off, pc->K.ptr, pc->K.col, pc->K.val, pc->core_off,
                                 pc->core_kc, pc->srec, slab, slab_n, lo, hi, noinv, todo, cnt);
    SPNET_CUDA_TRY(cudaGetLastError());
    return SPNET_OK;
  };
  if (csm > 0)
    SPNET_TRY(launch(k_star_core<T, true>, pc->S, sizeof(double) * ((size_t)csm * (csm + 1) / 2 + 3 * csm), nullptr, 0, 0,
                     CORE_SMEM));
  if (nbig > 0) {
    const int64_t n = (int64_t)cmax * (cmax + 1) / 2;
    const int grid = slab_blocks(nbig, n, num_sms());
    double* slab = nullptr;
    SPNET_TRY(tmp.get(&slab, grid * n));
    SPNET_TRY(launch(k_star_core<T, false>, grid, sizeof(double) * 3 * cmax, slab, n, CORE_SMEM, CORE_INV));
  }
  return SPNET_OK;
}

static int core_inverses(spnet_pc_s* pc, DevArena& tmp, int32_t* noinv, int32_t* todo, StarCount* cnt) {
  return pc->precision == SPNET_PREC_FP64 ? core_inverses_t<double>(pc, tmp, noinv, todo, cnt)
                                          : core_inverses_t<float>(pc, tmp, noinv, todo, cnt);
}

// How the structures are spread over the GPU: a warp per star with everything in shared memory
// when four warps' worth fit in 200 KiB, else a block of four warps per star (its marks in shared
// memory while they fit).
struct StructurePlan {
  int nmax, acap, per_sm, hot_in_smem;
  bool per_warp;
  int64_t hot;
  size_t smem;
  StructurePlan(int nmax_, int acap_) : nmax(nmax_), acap(acap_), hot(hot_bytes(nmax_, acap_)) {
    per_warp = 4 * hot <= 200 * 1024;
    const int64_t marks = (BT / 32) * bitmap_bytes(nmax) + marks_bytes(nmax);
    hot_in_smem = per_warp || marks <= 200 * 1024 ? 1 : 0;
    smem = per_warp ? (size_t)(4 * hot) : (size_t)(hot_in_smem ? marks : (BT / 32) * bitmap_bytes(nmax));
    per_sm = (int)((200 * 1024) / (smem + 1024));  // blocks per SM
    per_sm = per_sm < 1 ? 1 : per_sm > (per_warp ? 4 : 8) ? (per_warp ? 4 : 8) : per_sm;
  }
  // scratch of a worker (a warp or a block), with room for the columns of a dense block of
  // core_max nodes where it is not inverted
  int64_t stride(int core_max) const {
    return cold_bytes(nmax, core_max, acap) + (per_warp ? 0 : align_up(hot, 256));
  }
  int64_t workers(int core_max, int64_t stars, int sms) const {
    int64_t w = (int64_t)(per_warp ? 4 : 1) * per_sm * sms;
    if (w * stride(core_max) > SCRATCH_BUDGET) w = SCRATCH_BUDGET / stride(core_max);
    if (w > stars) w = stars;
    if (w < 1) w = 1;
    return per_warp ? (w + 3) / 4 * 4 : w;
  }
};

// the largest dense block that is inverted
static int inverted_up_to(int panels, int max_star, int vb) {
  return !panels ? 0 : (int64_t)max_star * vb > STAR_HUGE ? 256 : CORE_INV;
}
// the pool at first: per dof 28 bytes + ~4 factor entries of 32 bytes, per star 64
static int64_t pool_first(int64_t dofs, int64_t stars) { return dofs * (28 + 4 * 32) + stars * 64 + (1 << 20); }

// Device bytes that the stars' factors take at the peak of the set-up, estimated from the stars'
// sizes; `cycles`: edges a node of the network beyond a tree's.  Not known before the elimination
// are the factor entries (measured: 1.1 to 2 a dof on 3D networks, 4 to 8 in 2D and on trusses;
// taken: 9) and the dense blocks (3D: the tail rule's up to 1000 dofs, beyond up to 0.05 n with 0.1
// cycles a node and 0.15 n with 0.46; 2D: up to 7.4 sqrt n; taken: the tail rule's or half of
// cycles * n in 3D, 8 sqrt n in 2D).  Peak over estimate of whole requests: 0.06 to 0.75, 0.38 for
// the 10.9M-node network.
int64_t star_bytes_estimate(const std::vector<int32_t>& sizes, int dim, int ndof, int max_row, double cycles, int vb,
                            int panels) {
  if (sizes.empty()) return 0;
  const int64_t S = (int64_t)sizes.size();
  int64_t sum = 0, nbig = 0, cbig = 0;
  int nmax = 0;
  for (int32_t n : sizes) {
    sum += n;
    nmax = n > nmax ? n : nmax;
  }
  const int core_inv = inverted_up_to(panels, nmax, vb);
  double blocks = 0.0;
  for (int32_t n : sizes) {
    double c = dim == 2 ? 8.0 * std::sqrt((double)ndof * n) : 0.5 * cycles * n;
    c = std::min(std::max(c, (double)tail_nodes(n, tail_most(dim, S, num_sms()))), (double)n);
    // c^2 coefficients as an inverse, else entries of the records and the blob
    blocks += c * c * (c <= core_inv ? vb : vb + 2 + 16);
    if (c > CORE_SMEM && c <= core_inv) {
      ++nbig;
      cbig = std::max(cbig, (int64_t)c);
    }
  }
  const StructurePlan P(nmax, adjacency_cap(max_row - 1, dim, nmax));
  const int64_t scratch = P.workers(0, S, num_sms()) * P.stride(0);
  const int64_t slab_n = cbig * (cbig + 1) / 2;
  const int64_t slab = nbig > 0 ? slab_blocks(nbig, slab_n, num_sms()) * slab_n * 8 : 0;
  const int64_t pool = pool_first(sum, S) + sum * (28 + 9 * 32);  // one that has grown, beside the old one
  const int64_t records = sum * (2 * 10 * (vb + 2) + 6) + S * 512 + (int64_t)blocks;
  return pool + std::max(scratch, records + slab);
}

// what the passes of the factorisation share
struct StarWork {
  int acap = 0;                // adjacency slots per node
  int core_max = 0;            // largest dense block the scratch takes as columns
  int left = 0;                // stars whose structure is to be built
  int32_t* noinv = nullptr;    // [S] 1: the dense block is not inverted
  int32_t* todo = nullptr;     // [S] STAR_*
  StarCount* cnt = nullptr;
};

// room for `more` bytes behind the first `used` (a multiple of 16, as blobs and the pool are) of
// the pool, which are kept
static int pool_room(spnet_pc_s* pc, const StarWork& W, int64_t used, int64_t more) {
  cudaStream_t s = pc->op->stream;
  more = align_up(more, 16);
  if (used + more > pc->pool_bytes) {
    char* p = nullptr;
    SPNET_TRY(pc->mem.get(&p, used + more));
    if (used > 0) SPNET_CUDA_TRY(cudaMemcpyAsync(p, pc->pool, used, cudaMemcpyDeviceToDevice, s));
    if (pc->pool) pc->mem.release(pc->pool);
    pc->pool = p;
    pc->pool_bytes = used + more;
  }
  if (used == 0) return SPNET_OK;  // the count is zero
  const unsigned long long top = (unsigned long long)used;
  SPNET_CUDA_TRY(cudaMemcpyAsync(&W.cnt->pool_top, &top, sizeof(top), cudaMemcpyHostToDevice, s));
  SPNET_CUDA_TRY(cudaStreamSynchronize(s));  // top goes out of scope
  return SPNET_OK;
}

// nothing left, nothing asked for; the pool as it is
static int clear_counts(const StarWork& W, cudaStream_t s) {
  SPNET_CUDA_TRY(cudaMemsetAsync(W.cnt, 0, offsetof(StarCount, pool_top), s));
  return SPNET_OK;
}

// the structures of the stars to do.  Stars that do not fit the scratch or the pool are
// counted, and the pass repeated for them alone with what they need.
static int star_structures(spnet_pc_s* pc, StarWork& W) {
  cudaStream_t s = pc->op->stream;
  DevArena tmp;
  tmp.stream = s;
  struct Guard {
    DevArena& a;
    ~Guard() { a.free_all(); }
  } guard{tmp};
  const int nmax = pc->max_star, acap = W.acap;
  const StructurePlan P(nmax, acap);
  {
    static std::atomic<bool> attr_set[64];  // per device
    int dev = 0;
    SPNET_CUDA_TRY(cudaGetDevice(&dev));
    dev &= 63;
    if (!attr_set[dev]) {
      SPNET_CUDA_TRY(cudaFuncSetAttribute(k_star_symbolic, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
      SPNET_CUDA_TRY(cudaFuncSetAttribute(k_star_symbolic_block, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
      attr_set[dev] = true;
    }
  }
  int* flags = pc->op->dflags;
  char* scratch = nullptr;
  for (int attempt = 0; attempt < 8; ++attempt) {
    const int64_t stride = P.stride(W.core_max), workers = P.workers(W.core_max, W.left, num_sms());
    if (scratch) tmp.release(scratch);
    scratch = nullptr;
    SPNET_TRY(tmp.get(&scratch, workers * stride));
    SPNET_TRY(clear_counts(W, s));
    SPNET_CUDA_TRY(cudaMemsetAsync(flags, 0, sizeof(int), s));
    StarArgs A;
    A.m = mesh_of_pc(pc);
    A.S = pc->S;
    A.star_mesh = pc->star_mesh;
    A.star_n = pc->star_n;
    A.elem_ptr = pc->elem_ptr;
    A.elem_of = pc->elem_of;
    A.kptr = pc->K.ptr;
    A.kcol = pc->K.col;
    A.kval = pc->K.val;
    A.scratch = scratch;
    A.stride = stride;
    A.hot = P.hot;
    A.hot_in_smem = P.hot_in_smem;
    A.nmax = nmax;
    A.core_max = W.core_max;
    A.pool = pc->pool;
    A.pool_cap = pc->pool_bytes;
    A.star_off = pc->star_off;
    A.star_lev = pc->star_lev;
    A.star_nnz = pc->star_nnz;
    A.star_core = pc->star_core;
    A.flags = flags;
    A.cnt = W.cnt;
    A.todo = W.todo;
    A.core_inv = pc->core_inv;
    A.tail_most = tail_most(pc->d, pc->S, num_sms());
    A.noinv = W.noinv;
    A.cap = acap;
    A.patch = pc->star_rule;
    A.q1w = pc->patch_w;
    A.N = pc->N;
    note_launch();
    {
      ProfScope ps(KID_STAR_SYMBOLIC, s);
      if (P.per_warp) k_star_symbolic<<<(unsigned)(workers / 4), 128, P.smem, s>>>(A);
      else k_star_symbolic_block<<<(unsigned)workers, BT, P.smem, s>>>(A);
    }
    SPNET_CUDA_TRY(cudaGetLastError());
    int h = 0;
    StarCount c;
    SPNET_CUDA_TRY(cudaMemcpyAsync(&h, flags, sizeof(int), cudaMemcpyDeviceToHost, s));
    SPNET_CUDA_TRY(cudaMemcpyAsync(&c, W.cnt, sizeof(c), cudaMemcpyDeviceToHost, s));
    SPNET_CUDA_TRY(cudaStreamSynchronize(s));
    if (h == 0) return SPNET_OK;
    if ((h & ~(FLAG_STAR_BIG | FLAG_POOL)) || c.left == 0) break;
    W.left = c.left;
    W.core_max = c.need_core > W.core_max ? c.need_core : W.core_max;
    // blobs lie below the first one that did not fit
    const int64_t used = h & FLAG_POOL ? pc->pool_bytes : (int64_t)c.pool_top;
    SPNET_TRY(pool_room(pc, W, used, (int64_t)c.pool_more));
  }
  return check_flags(flags, s, "setup_preconditioner (star structure)");
}

// Stars whose dense block turns out too ill conditioned to be inverted (k_star_core) are
// marked and done again, they alone; the others keep their factors.  (The mixed beam set-ups of
// Section 6.3 mark stars with blocks of up to 1024 nodes; the larger blocks, most of the numeric
// pass, are not inverted in the first place.  Every star done twice, the pull at H = 1/16 took
// 27.1 s in mixed precision, now 13.1; each pass over all stars until the scratch and the pool
// held the largest, 13.8 s in FP64, now 11.3.)
int pc_factor_stars(spnet_pc_s* pc) {
  if (pc->S == 0) return SPNET_OK;
  cudaStream_t s = pc->op->stream;
  if (pc->sum_s > INT32_MAX)
    return fail(SPNET_ERR_UNSUPPORTED, "setup_preconditioner: the stars hold more than 2^31-1 entries in total");
  if (pc->max_star > 65535)  // u16 places
    return fail(SPNET_ERR_UNSUPPORTED, "setup_preconditioner: a star holds more than 65535 dofs");
  DevArena tmp;
  tmp.stream = s;
  struct Guard {
    DevArena& a;
    ~Guard() { a.free_all(); }
  } guard{tmp};
  StarWork W;
  // counts and marks, all zero at first (STAR_TODO)
  char* zero = nullptr;
  const size_t zeros = sizeof(StarCount) + 2 * sizeof(int32_t) * (size_t)pc->S;
  SPNET_TRY(tmp.get(&zero, zeros));
  SPNET_CUDA_TRY(cudaMemsetAsync(zero, 0, zeros, s));
  W.cnt = (StarCount*)zero;
  W.noinv = (int32_t*)(zero + sizeof(StarCount));
  W.todo = W.noinv + pc->S;
  W.left = pc->S;
  int max_row = 0;
  note_launch();
  k_max_row<<<4 * num_sms(), 256, 0, s>>>(pc->N, pc->K.ptr, &W.cnt->max_row);
  SPNET_CUDA_TRY(cudaGetLastError());
  SPNET_CUDA_TRY(cudaMemcpyAsync(&max_row, &W.cnt->max_row, sizeof(int), cudaMemcpyDeviceToHost, s));
  SPNET_CUDA_TRY(cudaStreamSynchronize(s));
  W.acap = adjacency_cap(max_row - 1, pc->d, pc->max_star);
  const int vb = pc->precision == SPNET_PREC_FP64 ? 8 : 4;
  pc->core_inv = inverted_up_to(pc->panels, pc->max_star, vb);
  // without inverses room for a dense block from the start: a repeated pass costs a launch
  if (pc->core_inv == 0) {
    const int first = pc->max_star <= 4 * CORE_FIRST ? CORE_FIRST : 4 * CORE_FIRST;
    W.core_max = pc->max_star < first ? pc->max_star : first;
  }
  SPNET_TRY(pc->mem.get(&pc->star_off, pc->S));
  SPNET_TRY(pc->mem.get(&pc->star_lev, pc->S));
  SPNET_TRY(pc->mem.get(&pc->star_nnz, pc->S));
  SPNET_TRY(pc->mem.get(&pc->star_core, pc->S));
  SPNET_TRY(pool_room(pc, W, 0, pool_first(pc->sum_s, pc->S)));
  int* flags = pc->op->dflags;
  std::vector<int32_t> lev(pc->S), nz(pc->S);
  for (;;) {
    SPNET_TRY(star_structures(pc, W));
    note_launch();
    {
      ProfScope ps(KID_STAR_NUMERIC, s);
      // a warp per star, or a block per star when some star exceeds 1024 dofs
      if (pc->max_star > 1024)
        k_star_numeric<NT><<<pc->S, NT, 0, s>>>(pc->S, pc->pool, pc->star_off, W.todo, pc->K.ptr, pc->K.col, pc->K.val,
                                                flags);
      else
        k_star_numeric<32><<<(pc->S + NT / 32 - 1) / (NT / 32), NT, 0, s>>>(pc->S, pc->pool, pc->star_off, W.todo,
                                                                            pc->K.ptr, pc->K.col, pc->K.val, flags);
    }
    SPNET_CUDA_TRY(cudaGetLastError());
    SPNET_CUDA_TRY(cudaMemsetAsync(W.todo, STAR_DONE & 0xff, sizeof(int32_t) * pc->S, s));
    // the records of the solves: their sizes and places, the inverses of the dense blocks
    // (written into them), then the sparse entries; the set-up blobs are released
    SPNET_CUDA_TRY(cudaMemcpyAsync(lev.data(), pc->star_lev, sizeof(int32_t) * pc->S, cudaMemcpyDeviceToHost, s));
    SPNET_CUDA_TRY(cudaMemcpyAsync(nz.data(), pc->star_nnz, sizeof(int32_t) * pc->S, cudaMemcpyDeviceToHost, s));
    DevArena pass;
    pass.stream = s;
    Guard pass_guard{pass};
    SPNET_TRY(star_records_plan(pc, pass, lev, nz, W.noinv));
    StarCount c{};
    SPNET_TRY(clear_counts(W, s));
    SPNET_TRY(core_inverses(pc, pass, W.noinv, W.todo, W.cnt));
    SPNET_CUDA_TRY(cudaMemcpyAsync(&c, W.cnt, sizeof(c), cudaMemcpyDeviceToHost, s));
    SPNET_TRY(check_flags(flags, s, "setup_preconditioner (star factorisation)"));  // waits for the device
    if (c.left == 0) {
      // statistics
      pc->factor_nnz = 0;
      pc->total_levels = 0;
      pc->max_levels = 0;
      pc->panel_stars = 0;
      for (int i = 0; i < pc->S; ++i) {
        pc->factor_nnz += nz[i] + (int64_t)pc->star_inv[i] * (pc->star_inv[i] - 1) / 2;
        pc->total_levels += lev[i];
        pc->max_levels = lev[i] > pc->max_levels ? lev[i] : pc->max_levels;
        pc->panel_stars += pc->star_inv[i] >= CORE_TC && pc->batch_rhs >= 2 && pc->precision == SPNET_PREC_MIXED;
      }
      SPNET_TRY(star_records_fill(pc));
      pc->mem.release(pc->pool);
      pc->pool = nullptr;
      return SPNET_OK;
    }
    W.left = c.left;
    W.core_max = c.need_core > W.core_max ? c.need_core : W.core_max;
    pc->mem.release(pc->srec);
    pc->mem.release(pc->rec_off);
    SPNET_TRY(pool_room(pc, W, (int64_t)c.pool_top, (int64_t)c.pool_more));
  }
}

}  // namespace spnet
