// Restricted additive Schwarz with block ILU(0) subdomain solves: the
// R(A)^{-1} stages of CPR-FPF (Algorithm 2: the RAS solves that open and
// close it) of arXiv 1701.06254, with the local potential reordering of
// eqs. (30)-(32) applied inside each subdomain.  A subdomain is a column
// tile of tile_x x tile_y cells over all layers (a well goes with the tile
// of its first perforated cell); its local system is the owned rows plus
// every row within graph distance 1 or 2 of them (the overlap, Table 9).  Each subdomain maps to one thread
// block: the potential sort, the level sets of the reordered factors, the
// factorisation and both triangular solves run level by level inside that
// block.
#include "common.cuh"
#include <cuda_bf16.h>
#include <algorithm>
#include <cfloat>
#include <climits>
#include <type_traits>

// Streamed per-subdomain factors for the shared-memory apply.  One block
// solves one subdomain (one warp in FP32 / BF16, two in FP64): its local
// vector y lives in shared memory, and the factors, which each application
// reads exactly once and in a fixed order, stream through registers, a few
// groups ahead of the sweep.  A subdomain's stream is a list of groups: the
// rows of the L sweep (L levels 1.., level 0 has no entries), then the rows
// of the U sweep (U levels 0..), level by level, without the rows no owned
// row depends on (k_ras_levels); a level is split into groups of at most 32
// rows, in descending order of their entry counts.  A group is a sequence of
// pieces of 16 bytes per row (per row and component in FP64), each piece
// stored for the first n[p] rows only:
//   header    {row, col[0..5]} u16 (a missing column names the zero element
//             behind y)
//   blocks    U groups: the inverse diagonal block, then the entries; L
//             groups: the entries.  A piece holds two BF16 blocks, one FP32
//             block, or one component's half of an FP64 block
// Piece by piece the reads of a warp are contiguous, and there is little
// padding.  A row of more than RAS_K entries (a well's, a wide stencil's)
// takes part in several groups, with the identity for the inverse diagonal
// in all but the last.  The groups of each sweep are filled up to a multiple
// of ras_ahead with empty ones (one row, behind the zero element).
// A group's descriptor (64 bit): start / 16 (20 bits) | rows (6) | n[6] (6),
// n[1..5] (6 bits each); n[0] = rows.
#define RAS_SMEM_BUDGET (200 * 1024)
#define RAS_K 6                                  // entries of a row per group
#define RAS_START_MAX (1LL << 24)                // a stream's bytes: 20-bit starts in units of 16
#define RAS_NONFINITE (1 << 30)                  // with a subdomain's group count: its stream has Inf or NaN
// groups held in registers ahead of the sweep
template <class TB> __host__ __device__ constexpr int ras_ahead() { return sizeof(TB) == 2 ? 3 : 2; }
// stored bytes per 2x2 block
static int ras_block_bytes(int prec) { return prec == SIM_PREC_FP64 ? 32 : prec == SIM_PREC_MIXED_BF16 ? 8 : 16; }
__host__ __device__ inline int al16(int x) { return (x + 15) & ~15; }

// flag = 1 when some entry (i, c) of the pattern has no entry (c, i)
__global__ void k_pattern_asym(int nb, const int *rp, const int *ci, int *flag) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nb) return;
  for (int q = rp[i]; q < rp[i + 1]; q++) {
    int c = ci[q], lo = rp[c], hi = rp[c + 1];
    while (lo < hi) { int mid = (lo + hi) >> 1; if (ci[mid] < i) lo = mid + 1; else hi = mid; }
    if (lo >= rp[c + 1] || ci[lo] != i) *flag = 1;
  }
}

// ------------------------------------------------- static partition (host)
void ras_build_static(sim_ls_s *ls) {
  ras_data &R = ls->ras;
  int tx = ls->o.tile_x, ty = ls->o.tile_y;
  int ntx = (ls->nx + tx - 1) / tx, nty = (ls->ny + ty - 1) / ty;
  int nsub = ntx * nty, nb = ls->nb, n = ls->n;
  R.nsub = nsub;
  std::vector<int> owner(nb);
  for (int c = 0; c < n; c++) {
    int i = c % ls->nx, j = (c / ls->nx) % ls->ny;
    owner[c] = (i / tx) + ntx * (j / ty);
  }
  for (int w = 0; w < ls->nw; w++) owner[n + w] = owner[ls->h_wc0[w]];
  std::vector<std::vector<int>> own(nsub);
  for (int r = 0; r < nb; r++) own[owner[r]].push_back(r);
  std::vector<int> sub_ptr(nsub + 1, 0), ext, owned, ncell(nsub), lrp_ptr(nsub + 1, 0), lrlen, lrp, lci, lsrc;
  std::vector<int> mark(nb, 0), loc(nb, -1);
  R.max_ext = 0; R.max_nnz = 0;
  int maxcells = 0;
  for (int s = 0; s < nsub; s++) {
    std::vector<int> list;
    for (int g : own[s])
      if (!mark[g]) { mark[g] = 1; list.push_back(g); }
    // rings of graph neighbours, one per level of overlap (1, or 2: Table 9)
    int ov = ls->o.overlap == 2 ? 2 : 1;
    for (int lev = 0, r0 = 0, r1 = (int)list.size(); lev < ov; lev++, r0 = r1, r1 = (int)list.size())
      for (int a = r0; a < r1; a++) {
        int g = list[a];
        for (int q = ls->h_rp[g]; q < ls->h_rp[g + 1]; q++) {
          int c = ls->h_ci[q];
          if (!mark[c]) { mark[c] = 1; list.push_back(c); }
        }
      }
    std::sort(list.begin(), list.end());      // cells ascending, then wells ascending
    int m = (int)list.size(), base = (int)ext.size(), nc = 0;
    for (int a = 0; a < m; a++) {
      int g = list[a];
      mark[g] = 0; loc[g] = a;
      ext.push_back(g);
      owned.push_back(owner[g] == s);
      nc += g < n;
    }
    ncell[s] = nc;
    maxcells = std::max(maxcells, nc);
    int nnz0 = (int)lci.size();
    for (int a = 0; a < m; a++) {
      int g = list[a], len = 0;
      lrp.push_back((int)lci.size());
      for (int q = ls->h_rp[g]; q < ls->h_rp[g + 1]; q++) {
        int lc = loc[ls->h_ci[q]];
        if (lc < 0) continue;
        lci.push_back(lc); lsrc.push_back(q); len++;
      }
      lrlen.push_back(len);
    }
    for (int a = 0; a < m; a++) loc[list[a]] = -1;
    sub_ptr[s + 1] = base + m;
    lrp_ptr[s + 1] = (int)lci.size();
    R.max_ext = std::max(R.max_ext, m);
    const int nz = (int)lci.size() - nnz0;
    R.max_nnz = std::max(R.max_nnz, nz);
    for (int k = 0; k < 2; k++) {               // k_ras_levels' shared memory, without and with the pruned lists
      int cnt = (k ? 4 : 2) * (m + 1);
      R.lvl_smem[k] = std::max(R.lvl_smem[k], sizeof(int) * ((size_t)3 * m + 1 + nz + (nz >= cnt ? 0 : cnt)));
    }
  }
  cudaStream_t st = ls->st;
  h2d(R.sub_ptr, sub_ptr, st); h2d(R.ext, ext, st);
  std::vector<uint8_t> ow(owned.begin(), owned.end());
  h2d(R.owned, ow, st); h2d(R.ncell, ncell, st);
  h2d(R.lrp_ptr, lrp_ptr, st); h2d(R.lrlen, lrlen, st); h2d(R.lrp, lrp, st);
  h2d(R.lci, lci, st); h2d(R.lsrc, lsrc, st);
  size_t next_tot = ext.size(), nnz_tot = lci.size();
  R.perm.alloc(next_tot); R.ipos.alloc(next_tot); R.frp.alloc(next_tot + nsub);
  R.fci.alloc(nnz_tot); R.fdiag.alloc(next_tot);
  R.lvl.alloc(2 * next_tot); R.lvl_rows.alloc(2 * next_tot); R.nlev.alloc(2 * nsub);
  R.lvl_ptr.alloc(2 * (next_tot + nsub));
  if (ls->o.precision != SIM_PREC_FP64) { R.fval32.alloc(4 * nnz_tot); R.dinv32.alloc(4 * next_tot); }
  else { R.fval.alloc(4 * nnz_tot); R.dinv.alloc(4 * next_tot); }
  int m = 1;
  while (m < maxcells) m <<= 1;
  R.max_lvl_ptr = m;   // sort width (power of two >= most cells in a subdomain)
  // shared-memory apply: a bound on each subdomain's stream (the grouping
  // follows the level sets of each setup, the bound only rows and entries: a
  // row's parts have a header, an inverse diagonal block and a rounding each)
  {
    const int prec = ls->o.precision, vb = ras_block_bytes(prec);
    int yb = prec == SIM_PREC_FP64 ? 16 : 8;               // local vector: double2 or float2 per row
    std::vector<long long> boff(nsub + 1, 0);
    int mmax = 0;
    bool fits = true;
    for (int s2 = 0; s2 < nsub; s2++) {
      long long ms = sub_ptr[s2 + 1] - sub_ptr[s2], nz = lrp_ptr[s2 + 1] - lrp_ptr[s2], e = nz - ms;
      if (ms >= 65534) fits = false;                       // 16-bit rows, the zero element and one more
      long long bound = (2 * ms + e / RAS_K + 5) * (32 + vb) + e * vb;   // (up to two empty groups per sweep)
      if (bound >= RAS_START_MAX) fits = false;
      boff[s2 + 1] = boff[s2] + ((bound + 15) & ~15LL);
      mmax = std::max(mmax, (int)ms);
    }
    R.smem_bytes = ((size_t)mmax + 2) * yb;
    // k_ras_pack's tables: groups per level, then the groups' sizes
    R.pack_smem = (4 * (size_t)mmax + (size_t)R.max_nnz / RAS_K + 24) * sizeof(int);
    R.smem_path = fits && R.smem_bytes <= RAS_SMEM_BUDGET;
    if (R.smem_path) {
      // gather / scatter order: the owned rows first, each part in natural
      // order (runs of neighbouring cells share their sectors)
      std::vector<int> gidx(ext.size()), gord(ext.size()), nown(nsub, 0);
      for (int s2 = 0; s2 < nsub; s2++) {
        int at = sub_ptr[s2];
        for (int pass = 0; pass < 2; pass++)
          for (int a = sub_ptr[s2]; a < sub_ptr[s2 + 1]; a++)
            if ((owned[a] != 0) == (pass == 0)) { gidx[at] = ext[a]; gord[at] = a - sub_ptr[s2]; at++; nown[s2] += pass == 0; }
      }
      h2d(R.blob_off, boff, st); R.blob.alloc(boff[nsub]);
      h2d(R.gidx, gidx, st); h2d(R.gord, gord, st); h2d(R.nown, nown, st);
      R.gpos.alloc(ext.size()); R.ngrp.alloc(2 * (size_t)nsub);
      // the lists without unneeded rows rely on a symmetric pattern (which the
      // interface asks for); one that is not keeps every row
      dbuf<int> asym;
      asym.alloc(1);
      RS_CUDA(cudaMemsetAsync(asym.p, 0, sizeof(int), st));
      k_pattern_asym<<<grid_for(nb, 256), 256, 0, st>>>(nb, ls->rp.p, ls->ci.p, asym.p);
      RS_LAUNCHED(1);
      R.symmetric = d2h(asym.p, 1, st)[0] == 0;
      R.alvl_rows.alloc(2 * next_tot); R.alvl_ptr.alloc(2 * (next_tot + nsub));
      R.gdesc.alloc(2 * ext.size() + 8 * (size_t)nsub + nnz_tot / RAS_K + 1);
      if (R.pack_smem > RAS_SMEM_BUDGET) { R.pack_lv.alloc(2 * ext.size() + nsub); R.pack_gr.alloc(R.gdesc.n); }
      RS_CUDA(cudaStreamSynchronize(st));                  // the host vectors above go out of scope
    }
  }
  if ((size_t)m * 12 > 200 * 1024) RS_FAIL(SIM_ERR_ARG, "RAS: %d cells per subdomain is too many (reduce tile_x/tile_y)", maxcells);
  if ((size_t)R.max_ext * 16 > 200 * 1024) RS_FAIL(SIM_ERR_ARG, "RAS: subdomain too large");
}

// --------------------------------------------- potential ordering (eq. 30)
// Sort the cells of each subdomain by descending oil potential; equal keys
// keep ascending natural order (ext indices of cells ascend with the natural
// index).  Wells keep their place after the cells (eq. 32).
__global__ void k_ras_order(const int *sub_ptr, const int *ext, const int *ncell, const double *key, int reorder,
                            int *perm, int *ipos) {
  extern __shared__ unsigned char smem[];
  int s = blockIdx.x, base = sub_ptr[s], m = sub_ptr[s + 1] - base, nc = ncell[s];
  int w = 1;
  while (w < nc) w <<= 1;
  long long *k = reinterpret_cast<long long *>(smem);   // integer keys (dkey) of the potentials
  int *id = reinterpret_cast<int *>(k + w);
  if (reorder) {
    const long long kmin = dkey(-DBL_MAX);
    for (int i = threadIdx.x; i < w; i += blockDim.x) {
      if (i < nc) {
        double kv = key[ext[base + i]];
        k[i] = kv > -DBL_MAX ? dkey(kv) : kmin;   // NaN / -inf sort with the padding, before it
        id[i] = i;
      }
      else { k[i] = kmin; id[i] = INT_MAX; }
    }
    __syncthreads();
    for (int kk = 2; kk <= w; kk <<= 1)
      for (int j = kk >> 1; j > 0; j >>= 1) {
        for (int i = threadIdx.x; i < w; i += blockDim.x) {
          int ixj = i ^ j;
          if (ixj > i) {
            // "a before b": larger key first, then smaller index
            long long ka = k[i], kb = k[ixj]; int ia = id[i], ib = id[ixj];
            bool a_first = (ka > kb) || (ka == kb && ia < ib);
            bool up = (i & kk) == 0;
            if (a_first != up) { k[i] = kb; k[ixj] = ka; id[i] = ib; id[ixj] = ia; }
          }
        }
        __syncthreads();
      }
    for (int i = threadIdx.x; i < nc; i += blockDim.x) { perm[base + i] = id[i]; ipos[base + id[i]] = i; }
  } else {
    for (int i = threadIdx.x; i < nc; i += blockDim.x) { perm[base + i] = i; ipos[base + i] = i; }
  }
  for (int i = nc + threadIdx.x; i < m; i += blockDim.x) { perm[base + i] = i; ipos[base + i] = i; }
}

// ascending by key, both arrays carried along: Batcher's odd-even merge
// network for eight (Knuth, The Art of Computer Programming vol. 3, 5.2.2)
__device__ __forceinline__ void sort8(int *k, int *v) {
  const int P[19][2] = {{0, 1}, {2, 3}, {4, 5}, {6, 7}, {0, 2}, {1, 3}, {4, 6}, {5, 7}, {1, 2}, {5, 6},
                        {0, 4}, {1, 5}, {2, 6}, {3, 7}, {2, 4}, {3, 5}, {1, 2}, {3, 4}, {5, 6}};
#pragma unroll
  for (int t = 0; t < 19; t++) {
    const int a = P[t][0], b = P[t][1];
    const bool sw = k[a] > k[b];
    const int ka = sw ? k[b] : k[a], kb = sw ? k[a] : k[b], va = sw ? v[b] : v[a], vb = sw ? v[a] : v[b];
    k[a] = ka; k[b] = kb; v[a] = va; v[b] = vb;
  }
}

// Local pattern in position order, columns sorted by position (rows of at
// most eight entries in registers), and for the factorisation the index ftr
// of entry (k, i) for each entry (i, k) below the diagonal, with fgen[i] = 1
// where row i needs the general elimination: a row k < i of its pattern has a
// column j > k besides i that row i has too (the wells' columns; never among
// the cells of a 7-point stencil), or lacks column i.
__global__ void k_ras_pattern(const int *sub_ptr, const int *lrp_ptr, const int *lrp, const int *lrlen,
                              const int *lci, const int *lsrc, const int *perm, const int *ipos, int *frp, int *fci,
                              int *fdiag, int *fsrc, int *ftr, uint8_t *fgen) {
  __shared__ int warp_tot[32];
  __shared__ int carry;
  int s = blockIdx.x, base = sub_ptr[s], m = sub_ptr[s + 1] - base, pbase = lrp_ptr[s];
  int fbase = base + s;                   // frp segment has m + 1 entries
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int c0 = 0; c0 < m; c0 += blockDim.x) {
    int pos = c0 + threadIdx.x, len = pos < m ? lrlen[base + perm[base + pos]] : 0;
    int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, x = len;
    for (int o = 1; o < 32; o <<= 1) { int y = __shfl_up_sync(0xffffffffu, x, o); if (lane >= o) x += y; }
    if (lane == 31) warp_tot[wid] = x;
    __syncthreads();
    if (wid == 0) {
      int nw = blockDim.x >> 5, v = lane < nw ? warp_tot[lane] : 0, z = v;
      for (int o = 1; o < 32; o <<= 1) { int y = __shfl_up_sync(0xffffffffu, z, o); if (lane >= o) z += y; }
      if (lane < nw) warp_tot[lane] = z - v;
    }
    __syncthreads();
    int excl = carry + warp_tot[wid] + x - len;
    if (pos < m) frp[fbase + pos] = excl;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = excl + len;
    __syncthreads();
  }
  if (threadIdx.x == 0) frp[fbase + m] = carry;
  __syncthreads();
  for (int pos = threadIdx.x; pos < m; pos += blockDim.x) {
    int e = perm[base + pos], src0 = lrp[base + e], len = lrlen[base + e], o = pbase + frp[fbase + pos];
    if (len <= 8) {
      int c[8], q[8];
#pragma unroll
      for (int a = 0; a < 8; a++) {
        c[a] = a < len ? lci[src0 + a] : -1;
        q[a] = a < len ? lsrc[src0 + a] : 0;
      }
#pragma unroll
      for (int a = 0; a < 8; a++) c[a] = c[a] >= 0 ? ipos[base + c[a]] : INT_MAX;
      sort8(c, q);
#pragma unroll
      for (int a = 0; a < 8; a++)
        if (a < len) {
          fci[o + a] = c[a]; fsrc[o + a] = q[a];
          if (c[a] == pos) fdiag[base + pos] = o + a;
        }
      continue;
    }
    for (int a = 0; a < len; a++) {         // insertion by position
      int c = ipos[base + lci[src0 + a]], q = lsrc[src0 + a], b = o + a - 1;
      while (b >= o && fci[b] > c) { fci[b + 1] = fci[b]; fsrc[b + 1] = fsrc[b]; b--; }
      fci[b + 1] = c; fsrc[b + 1] = q;
    }
    for (int a = 0; a < len; a++) if (fci[o + a] == pos) fdiag[base + pos] = o + a;
  }
  __syncthreads();                          // the block's rows are complete
  for (int pos = threadIdx.x; pos < m; pos += blockDim.x) {
    const int r0 = pbase + frp[fbase + pos], r1 = pbase + frp[fbase + pos + 1];
    bool gen = false;
    for (int q = r0; q < r1; q++) {
      const int k = fci[q];
      if (k >= pos) break;
      // row k's columns beyond k: pos, and any that row pos shares
      int t = -1;
      for (int qk = pbase + frp[fbase + k]; qk < pbase + frp[fbase + k + 1]; qk++) {
        const int j = fci[qk];
        if (j <= k) continue;
        if (j == pos) { t = qk; continue; }
        for (int qi = q + 1; qi < r1; qi++) gen |= fci[qi] == j;
      }
      ftr[q] = t;
      gen |= t < 0;
    }
    fgen[base + pos] = gen;
  }
}

// Level sets of the subdomain's factors: L level of row i = 1 + the largest
// L level among its columns c < i (0 without such a column), U level the
// same over c > i; rows of a level in ascending position.  The levels are
// the longest paths of the two DAGs, computed for all rows in parallel from
// the pattern in shared memory, each row once its predecessors are done,
// then counted, scanned and filled by one warp each for L and U (ranks
// within a chunk of 32 rows by matching levels, so the fill keeps the
// ascending order).  Blocks
// whose pattern does not fit in shared memory take k_ras_levels_serial.
//
// The apply's own row lists (alvl_rows, alvl_ptr) leave out the rows whose
// solution no owned row depends on: only owned rows are written back, and
// row i of the U sweep is needed when i is owned or some needed row c < i
// has it in its U part (c's entry i; the pattern is symmetric, so i's entry
// c), row i of the L sweep when the U sweep needs it or some needed row
// c > i does.  Both closures follow the level recurrences, so the flags ride
// along with the levels (bit 0 of the stored value).
__global__ void __launch_bounds__(128) k_ras_levels(const int *sub_ptr, const int *lrp_ptr, const int *frp,
                                                    const int *fci, const int *perm, const uint8_t *owned, int *lvl,
                                                    int *lvl_rows, int *nlev, int *lvl_ptr, int *alvl_rows,
                                                    int *alvl_ptr, int *err) {   // alvl_rows NULL: no pruned lists
  extern __shared__ int lsm[];
  int s = blockIdx.x, base = sub_ptr[s], m = sub_ptr[s + 1] - base, pbase = lrp_ptr[s], fbase = base + s;
  int nnz = frp[fbase + m] - frp[fbase];
  const int *rpg = frp + fbase, *cig = fci + pbase + frp[fbase];
  // cnt (2 or 4 arrays of m + 1) takes the columns' place once the levels
  // are known, or the space behind them where the columns are fewer
  const int sets = alvl_rows ? 4 : 2;
  int *srp = lsm, *LvL = srp + (m + 1), *LvU = LvL + m, *sci = LvU + m;
  int *cnt = nnz >= sets * (m + 1) ? sci : sci + nnz;
  for (int k = threadIdx.x; k <= m; k += blockDim.x) srp[k] = rpg[k] - rpg[0];
  for (int k = threadIdx.x; k < nnz; k += blockDim.x) sci[k] = cig[k];
  for (int k = threadIdx.x; k < m; k += blockDim.x) { LvL[k] = -1; LvU[k] = -1; }
  __syncthreads();
  // L levels: thread t takes rows t, t + nt, ... ascending and waits (in
  // shared memory) for each column c < i to have its level; every wait is
  // on a lower row, taken earlier by its thread, so the waits end.  U levels
  // the same from the last row down.  Each wait is bounded: past the limit
  // the kernel records code 5 and takes 0 for that level.  Stored: 2 level +
  // needed (L pass: by the U sweep; U pass: by the L sweep).
  volatile int *vL = LvL, *vU = LvU;
  const int LIMIT = 1 << 22;
  bool bad = false;
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    int l = 0, need = owned[base + perm[base + i]] ? 1 : 0;
    for (int q = srp[i]; q < srp[i + 1]; q++) {
      int c = sci[q];
      if (c >= i) break;                            // columns ascending
      int v, spins = 0;
      while ((v = vL[c]) < 0 && ++spins < LIMIT) {}
      if (v < 0) { bad = true; v = 1; }
      l = max(l, (v >> 1) + 1);
      need |= v & 1;
    }
    vL[i] = 2 * l + need;
  }
  __syncthreads();
  for (int i = m - 1 - (int)threadIdx.x; i >= 0; i -= blockDim.x) {
    int u = 0, need = LvL[i] & 1;
    for (int q = srp[i + 1] - 1; q >= srp[i]; q--) {
      int c = sci[q];
      if (c <= i) break;
      int v, spins = 0;
      while ((v = vU[c]) < 0 && ++spins < LIMIT) {}
      if (v < 0) { bad = true; v = 1; }
      u = max(u, (v >> 1) + 1);
      need |= v & 1;
    }
    vU[i] = 2 * u + need;
  }
  if (bad) atomicExch(err, 5);
  __syncthreads();
  for (int k = threadIdx.x; k < sets * (m + 1); k += blockDim.x) cnt[k] = 0;
  __syncthreads();
  // counts per level, then per warp (0: L, 1: U, 2 and 3: L and U with the
  // needed rows only) the scan and the fill
  for (int i = threadIdx.x; i < m; i += blockDim.x) {
    int l = LvL[i], u = LvU[i];
    atomicAdd(&cnt[l >> 1], 1);
    atomicAdd(&cnt[(m + 1) + (u >> 1)], 1);
    if (sets == 4 && (u & 1)) atomicAdd(&cnt[2 * (m + 1) + (l >> 1)], 1);
    if (sets == 4 && (l & 1)) atomicAdd(&cnt[3 * (m + 1) + (u >> 1)], 1);
    lvl[2 * base + i] = l >> 1; lvl[2 * base + m + i] = u >> 1;
  }
  __syncthreads();
  int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (wid > 1 && !alvl_rows) return;
  const bool upper = wid & 1, some = wid > 1;
  const int *Lv = upper ? LvU : LvL, *Nd = upper ? LvL : LvU;   // a row's flag sits with the other level
  int *c = cnt + wid * (m + 1), *c0 = cnt + (upper ? m + 1 : 0);
  int *pp = (some ? alvl_ptr : lvl_ptr) + 2 * (base + s) + (upper ? m + 1 : 0);
  int *rr = (some ? alvl_rows : lvl_rows) + 2 * base + (upper ? m : 0);
  // number of levels: one past the last non-empty count (of all rows: the
  // counts become cursors below, so both warps of a triangle look first)
  int nl = 0;
  for (int k = lane; k < m; k += 32) if (c0[k]) nl = max(nl, k + 1);
  for (int o = 16; o > 0; o >>= 1) nl = max(nl, __shfl_xor_sync(0xffffffffu, nl, o));
  if (alvl_rows) __syncthreads(); else asm volatile("bar.sync 1, 64;" ::: "memory");
  // exclusive scan of the counts into pp[0..nl] and the cursors c[0..nl)
  int run = 0;
  for (int k0 = 0; k0 <= nl; k0 += 32) {
    int k = k0 + lane, v = k < nl ? c[k] : 0, x = v;
    for (int o = 1; o < 32; o <<= 1) { int y = __shfl_up_sync(0xffffffffu, x, o); if (lane >= o) x += y; }
    if (k <= nl) pp[k] = run + x - v;
    if (k < nl) c[k] = run + x - v;
    run += __shfl_sync(0xffffffffu, x, 31);
  }
  __syncwarp();
  for (int i0 = 0; i0 < m; i0 += 32) {
    int i = i0 + lane;
    bool in = i < m && (!some || (Nd[i] & 1));
    int lv = in ? Lv[i] >> 1 : -1 - lane;
    unsigned grp = __match_any_sync(0xffffffffu, lv);
    if (in) rr[c[lv] + __popc(grp & ((1u << lane) - 1u))] = i;
    __syncwarp();
    if (in && lane == __ffs(grp) - 1) c[lv] += __popc(grp);
    __syncwarp();
  }
  if (lane == 0 && !some) nlev[2 * s + (upper ? 1 : 0)] = nl;
}

// the same, one thread per triangle walking the rows serially from global
// memory (subdomains whose pattern does not fit in shared memory)
__global__ void k_ras_levels_serial(const int *sub_ptr, const int *lrp_ptr, const int *frp, const int *fci,
                                    int *lvl, int *lvl_rows, int *nlev, int *lvl_ptr) {
  int s = blockIdx.x, base = sub_ptr[s], m = sub_ptr[s + 1] - base, pbase = lrp_ptr[s], fbase = base + s;
  const int *rp_ = frp + fbase, *ci_ = fci + pbase;
  bool upper;
  if (threadIdx.x == 0) upper = false;
  else if (threadIdx.x == 32) upper = true;
  else return;
  int *Lv = lvl + 2 * base + (upper ? m : 0);
  int nl = 0;
  for (int t = 0; t < m; t++) {
    int i = upper ? m - 1 - t : t;
    int lv = 0;
    for (int q = rp_[i]; q < rp_[i + 1]; q++) {
      int c = ci_[q];
      if ((upper ? c > i : c < i) && Lv[c] + 1 > lv) lv = Lv[c] + 1;
    }
    Lv[i] = lv; if (lv + 1 > nl) nl = lv + 1;
  }
  nlev[2 * s + (upper ? 1 : 0)] = nl;
  int *pp = lvl_ptr + 2 * (base + s) + (upper ? m + 1 : 0);
  int *rr = lvl_rows + 2 * base + (upper ? m : 0);
  for (int l = 0; l <= nl; l++) pp[l] = 0;
  for (int i = 0; i < m; i++) pp[Lv[i] + 1]++;
  for (int l = 0; l < nl; l++) pp[l + 1] += pp[l];
  for (int i = 0; i < m; i++) rr[pp[Lv[i]]++] = i;       // counts reused as cursors
  for (int l = nl; l > 0; l--) pp[l] = pp[l - 1];
  pp[0] = 0;
}

// launch order of the apply: subdomains by descending L + U level count
// (a CTA's time grows with its levels; starting the longest first keeps them
// out of the last wave).  One block: counting sort on the clamped key; the
// order within a key is whatever the atomics give (each subdomain writes only
// its own rows, so the order changes no result).
#define RAS_KEYS 4096
__global__ void __launch_bounds__(1024) k_ras_lpt(int nsub, const int *nlev, int *order) {
  __shared__ int cnt[RAS_KEYS];
  for (int k = threadIdx.x; k < RAS_KEYS; k += blockDim.x) cnt[k] = 0;
  __syncthreads();
  for (int s = threadIdx.x; s < nsub; s += blockDim.x) {
    int key = min(nlev[2 * s] + nlev[2 * s + 1], RAS_KEYS - 1);
    atomicAdd(&cnt[RAS_KEYS - 1 - key], 1);                 // descending keys
  }
  __syncthreads();
  if (threadIdx.x == 0) {                                   // exclusive scan (4096 entries)
    int run = 0;
    for (int k = 0; k < RAS_KEYS; k++) { int c = cnt[k]; cnt[k] = run; run += c; }
  }
  __syncthreads();
  for (int s = threadIdx.x; s < nsub; s += blockDim.x) {
    int key = min(nlev[2 * s] + nlev[2 * s + 1], RAS_KEYS - 1);
    order[atomicAdd(&cnt[RAS_KEYS - 1 - key], 1)] = s;
  }
}

template <class T> __device__ __forceinline__ void inv2x2(const T *M, T *I) {
  T det = M[0] * M[3] - M[1] * M[2];
  T r = T(1) / det;
  I[0] = M[3] * r; I[1] = -M[1] * r; I[2] = -M[2] * r; I[3] = M[0] * r;
}

// Block ILU(0), level by level (IKJ form per row): for each k < i in the
// row, L_ik = A_ik U_kk^{-1}; A_ij -= L_ik U_kj for j > k present in row i.
// A level's rows are few (about 18), so a block's time is its level count
// times one row's dependent loads.  Where the only such j is i itself (fgen
// clear: all rows without a shared well column) a row is A_ii -= L_ik U_ki
// with the position of U_ki known (ftr), and RAS_FB entries' loads are in
// flight together: one dependent level of loads instead of a search through
// row k per entry.  Against that search everywhere, on the 1M-cell
// case in FP32: 1.23 -> 0.46 ms per launch.
// FP64: LPR = 2 lanes per row, one component row each (a warp instruction
// holds the FP64 pipe for 64 cycles whatever the active lanes).
#define RAS_FB 2
template <class T> __host__ __device__ constexpr int ras_lpr() { return sizeof(T) == 8 ? 2 : 1; }
template <class T> __host__ __device__ constexpr int ras_factor_threads() { return sizeof(T) == 8 ? 128 : 64; }
template <class T>
__global__ void __launch_bounds__(ras_factor_threads<T>(), sizeof(T) == 8 ? 5 : 20)
k_ras_factor(const int *sub_ptr, const int *lrp_ptr, const int *frp, const int *fci, const int *fdiag, const int *fsrc,
             const int *__restrict__ ftr, const uint8_t *__restrict__ fgen, const double *__restrict__ val,
             const int *lvl_rows, const int *nlev, const int *lvl_ptr, T *fv, T *dinv, const int *order) {
  constexpr int LPR = ras_lpr<T>(), BS = ras_factor_threads<T>();
  struct __align__(16) blk { T v[4]; };
  int s = order[blockIdx.x], base = sub_ptr[s], m = sub_ptr[s + 1] - base, pbase = lrp_ptr[s], fbase = base + s;
  int q0 = pbase + frp[fbase], q1 = pbase + frp[fbase + m];
  for (int q = q0 + threadIdx.x; q < q1; q += 4 * BS) {       // gather values in factor order
    int src[4];
    double2 a[4], b[4];
#pragma unroll
    for (int u = 0; u < 4; u++) src[u] = q + u * BS < q1 ? fsrc[q + u * BS] : -1;
#pragma unroll
    for (int u = 0; u < 4; u++)
      if (src[u] >= 0) {
        a[u] = reinterpret_cast<const double2 *>(val)[2 * (size_t)src[u]];
        b[u] = reinterpret_cast<const double2 *>(val)[2 * (size_t)src[u] + 1];
      }
#pragma unroll
    for (int u = 0; u < 4; u++)
      if (src[u] >= 0) {
        blk B;
        B.v[0] = (T)a[u].x; B.v[1] = (T)a[u].y; B.v[2] = (T)b[u].x; B.v[3] = (T)b[u].y;
        reinterpret_cast<blk *>(fv)[q + u * BS] = B;
      }
  }
  __syncthreads();
  const int *pL = lvl_ptr + 2 * (base + s), *rL = lvl_rows + 2 * base;
  const int nL = nlev[2 * s], c = threadIdx.x % LPR;
  for (int l = 0; l < nL; l++) {
    const int a0 = pL[l], a1 = pL[l + 1];
    for (int a = a0 + threadIdx.x / LPR; a < a1; a += BS / LPR) {
      const int i = rL[a], r0 = pbase + frp[fbase + i], qd = fdiag[base + i];
      const unsigned pair = 3u << (threadIdx.x & 30);
      if (!fgen[base + i]) {
        T d[4];                                                // this lane's rows of A_ii: LPR 1 both, LPR 2 row c
        const T *Ad = fv + 4 * (size_t)qd;
#pragma unroll
        for (int u = 0; u < 4 / LPR; u++) d[u] = Ad[2 * c + u];
        for (int qb = r0; qb < qd; qb += RAS_FB) {
          int k[RAS_FB], t[RAS_FB];
          T A[RAS_FB][4 / LPR];
          blk D[RAS_FB], U[RAS_FB];
#pragma unroll
          for (int u = 0; u < RAS_FB; u++)
            if (qb + u < qd) {
              k[u] = fci[qb + u]; t[u] = ftr[qb + u];
#pragma unroll
              for (int w = 0; w < 4 / LPR; w++) A[u][w] = fv[4 * (size_t)(qb + u) + 2 * c + w];
            }
#pragma unroll
          for (int u = 0; u < RAS_FB; u++)
            if (qb + u < qd) { D[u] = reinterpret_cast<const blk *>(dinv)[base + k[u]]; U[u] = reinterpret_cast<const blk *>(fv)[t[u]]; }
#pragma unroll
          for (int u = 0; u < RAS_FB; u++)
            if (qb + u < qd) {
              T *Aq = fv + 4 * (size_t)(qb + u);
#pragma unroll
              for (int w = 0; w < 2 / LPR; w++) {
                const T l0 = A[u][2 * w] * D[u].v[0] + A[u][2 * w + 1] * D[u].v[2];
                const T l1 = A[u][2 * w] * D[u].v[1] + A[u][2 * w + 1] * D[u].v[3];
                Aq[2 * (c + w)] = l0; Aq[2 * (c + w) + 1] = l1;
                d[2 * w] -= l0 * U[u].v[0] + l1 * U[u].v[2];
                d[2 * w + 1] -= l0 * U[u].v[1] + l1 * U[u].v[3];
              }
            }
        }
        T M[4], I[4];
        if constexpr (LPR == 2) {
          const T o0 = __shfl_xor_sync(pair, d[0], 1), o1 = __shfl_xor_sync(pair, d[1], 1);
          M[0] = c ? o0 : d[0]; M[1] = c ? o1 : d[1]; M[2] = c ? d[0] : o0; M[3] = c ? d[1] : o1;
        } else {
#pragma unroll
          for (int u = 0; u < 4; u++) M[u] = d[u];
        }
        inv2x2(M, I);
        if (c == 0) {
          blk B;
#pragma unroll
          for (int u = 0; u < 4; u++) B.v[u] = M[u];
          reinterpret_cast<blk *>(fv)[qd] = B;
#pragma unroll
          for (int u = 0; u < 4; u++) B.v[u] = I[u];
          reinterpret_cast<blk *>(dinv)[base + i] = B;
        }
      } else if (c == 0) {
        const int r1 = pbase + frp[fbase + i + 1];
        for (int q = r0; q < r1; q++) {
          int k = fci[q];
          if (k >= i) break;
          T *Aq = fv + 4 * (size_t)q;
          const T *Dk = dinv + 4 * (size_t)(base + k);
          T l0 = Aq[0] * Dk[0] + Aq[1] * Dk[2], l1 = Aq[0] * Dk[1] + Aq[1] * Dk[3];
          T l2 = Aq[2] * Dk[0] + Aq[3] * Dk[2], l3 = Aq[2] * Dk[1] + Aq[3] * Dk[3];
          Aq[0] = l0; Aq[1] = l1; Aq[2] = l2; Aq[3] = l3;
          int k1 = pbase + frp[fbase + k + 1];
          int qi = q + 1;
          for (int qk = fdiag[base + k] + 1; qk < k1; qk++) {
            int j = fci[qk];
            while (qi < r1 && fci[qi] < j) qi++;
            if (qi >= r1) break;
            if (fci[qi] != j) continue;
            const T *U = fv + 4 * (size_t)qk;
            T *A = fv + 4 * (size_t)qi;
            A[0] -= l0 * U[0] + l1 * U[2]; A[1] -= l0 * U[1] + l1 * U[3];
            A[2] -= l2 * U[0] + l3 * U[2]; A[3] -= l2 * U[1] + l3 * U[3];
          }
        }
        inv2x2(fv + 4 * (size_t)qd, dinv + 4 * (size_t)(base + i));
      }
    }
    __syncthreads();
  }
}

void ras_pack(sim_ls_s *ls);
void ras_setup(sim_ls_s *ls) {
  ras_data &R = ls->ras;
  cudaStream_t s = ls->st;
  int w = R.max_lvl_ptr;
  size_t smem = (size_t)w * 12;
  static bool attr = false;
  if (!attr) {
    RS_CUDA(cudaFuncSetAttribute(k_ras_order, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    attr = true;
  }
  k_ras_order<<<R.nsub, 512, smem, s>>>(R.sub_ptr.p, R.ext.p, R.ncell.p, ls->key.p, ls->o.reorder, R.perm.p, R.ipos.p);
  static thread_local dbuf<int> fsrc, ftr;
  static thread_local dbuf<uint8_t> fgen;
  fsrc.ensure(R.lci.n); ftr.ensure(R.lci.n); fgen.ensure(R.ext.n);
  k_ras_pattern<<<R.nsub, 256, 0, s>>>(R.sub_ptr.p, R.lrp_ptr.p, R.lrp.p, R.lrlen.p, R.lci.p, R.lsrc.p, R.perm.p,
                                       R.ipos.p, R.frp.p, R.fci.p, R.fdiag.p, fsrc.p, ftr.p, fgen.p);
  // level sets from shared memory when the largest pattern fits
  size_t lsmem = R.lvl_smem[1];
  static bool lattr = false;
  if (!lattr) {
    RS_CUDA(cudaFuncSetAttribute(k_ras_levels, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    lattr = true;
  }
  R.pruned = R.smem_path && R.symmetric && lsmem <= 200 * 1024;   // the apply's lists leave unneeded rows out
  if (!R.pruned) lsmem = R.lvl_smem[0];
  if (lsmem <= 200 * 1024)
    k_ras_levels<<<R.nsub, 128, lsmem, s>>>(R.sub_ptr.p, R.lrp_ptr.p, R.frp.p, R.fci.p, R.perm.p, R.owned.p, R.lvl.p,
                                            R.lvl_rows.p, R.nlev.p, R.lvl_ptr.p, R.pruned ? R.alvl_rows.p : nullptr,
                                            R.pruned ? R.alvl_ptr.p : nullptr, ls->errw_dev);
  else
    k_ras_levels_serial<<<R.nsub, 64, 0, s>>>(R.sub_ptr.p, R.lrp_ptr.p, R.frp.p, R.fci.p, R.lvl.p, R.lvl_rows.p,
                                              R.nlev.p, R.lvl_ptr.p);
  // longest subdomains first for the factorisation and the applies (their
  // CTAs' times grow with the level counts)
  R.order.ensure(R.nsub);
  k_ras_lpt<<<1, 1024, 0, s>>>(R.nsub, R.nlev.p, R.order.p);
#define RAS_FACTOR(T, FV, DI)                                                                                         \
  k_ras_factor<T><<<R.nsub, ras_factor_threads<T>(), 0, s>>>(R.sub_ptr.p, R.lrp_ptr.p, R.frp.p, R.fci.p, R.fdiag.p,   \
                                                             fsrc.p, ftr.p, fgen.p, ls->val.p, R.lvl_rows.p, R.nlev.p, \
                                                             R.lvl_ptr.p, FV, DI, R.order.p)
  if (ls->o.precision != SIM_PREC_FP64) RAS_FACTOR(float, R.fval32.p, R.dinv32.p);
  else RAS_FACTOR(double, R.fval.p, R.dinv.p);
#undef RAS_FACTOR
  // (measured: the same factorisation with the subdomain in shared memory
  // took 4.2 against 1.2 ms on the 1M-cell case: 94 KB per block left two
  // blocks per SM, and the level loop's time is not its loads')
  RS_LAUNCHED(5);
  ras_pack(ls);
  R.built = true;
  RS_CHECK_LAUNCH();
}

// x = R(A)^{-1} f: gather the local right-hand side in position order,
// forward solve with L (unit diagonal) level by level, backward solve with U,
// write back the owned rows only.
template <class T>
__global__ void k_ras_apply(const int *sub_ptr, const int *ext, const uint8_t *owned, const int *lrp_ptr,
                            const int *frp, const int *fci, const int *fdiag, const int *perm, const int *lvl_rows,
                            const int *nlev, const int *lvl_ptr, const T *fv, const T *dinv, const T *f, T *x) {
  extern __shared__ unsigned char smem_raw[];
  T *y = reinterpret_cast<T *>(smem_raw);
  int s = blockIdx.x, base = sub_ptr[s], m = sub_ptr[s + 1] - base, pbase = lrp_ptr[s], fbase = base + s;
  for (int pos = threadIdx.x; pos < m; pos += blockDim.x) {
    int g = ext[base + perm[base + pos]];
    y[2 * pos] = f[2 * (size_t)g]; y[2 * pos + 1] = f[2 * (size_t)g + 1];
  }
  __syncthreads();
  const int *pL = lvl_ptr + 2 * (base + s), *pU = pL + (m + 1);
  const int *rL = lvl_rows + 2 * base, *rU = rL + m;
  int nL = nlev[2 * s], nU = nlev[2 * s + 1];
  for (int l = 1; l < nL; l++) {                 // level 0 rows have no L entries
    for (int a = pL[l] + threadIdx.x; a < pL[l + 1]; a += blockDim.x) {
      int i = rL[a];
      T y0 = y[2 * i], y1 = y[2 * i + 1];
      for (int q = pbase + frp[fbase + i]; q < fdiag[base + i]; q++) {
        const T *B = fv + 4 * (size_t)q; int c = fci[q];
        T c0 = y[2 * c], c1 = y[2 * c + 1];
        y0 -= B[0] * c0 + B[1] * c1; y1 -= B[2] * c0 + B[3] * c1;
      }
      y[2 * i] = y0; y[2 * i + 1] = y1;
    }
    __syncthreads();
  }
  for (int l = 0; l < nU; l++) {
    for (int a = pU[l] + threadIdx.x; a < pU[l + 1]; a += blockDim.x) {
      int i = rU[a];
      T y0 = y[2 * i], y1 = y[2 * i + 1];
      int r1 = pbase + frp[fbase + i + 1];
      for (int q = fdiag[base + i] + 1; q < r1; q++) {
        const T *B = fv + 4 * (size_t)q; int c = fci[q];
        T c0 = y[2 * c], c1 = y[2 * c + 1];
        y0 -= B[0] * c0 + B[1] * c1; y1 -= B[2] * c0 + B[3] * c1;
      }
      const T *D = dinv + 4 * (size_t)(base + i);
      y[2 * i] = D[0] * y0 + D[1] * y1; y[2 * i + 1] = D[2] * y0 + D[3] * y1;
    }
    __syncthreads();
  }
  for (int pos = threadIdx.x; pos < m; pos += blockDim.x) {
    int e = perm[base + pos];
    if (owned[base + e]) {
      int g = ext[base + e];
      x[2 * (size_t)g] = y[2 * pos]; x[2 * (size_t)g + 1] = y[2 * pos + 1];
    }
  }
}

// values as they are stored in the streams
template <class TB> __device__ __forceinline__ TB to_blob(float v);
template <> __device__ __forceinline__ float to_blob<float>(float v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 to_blob<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }
template <class TB> __device__ __forceinline__ TB to_blob_d(double v) { return to_blob<TB>((float)v); }
template <> __device__ __forceinline__ double to_blob_d<double>(double v) { return v; }
// BF16 pairs of a stored block
__device__ __forceinline__ void blk4(unsigned u, unsigned w, float &b0, float &b1, float &b2, float &b3) {
  b0 = __uint_as_float(u << 16); b1 = __uint_as_float(u & 0xffff0000u);
  b2 = __uint_as_float(w << 16); b3 = __uint_as_float(w & 0xffff0000u);
}

// The groups of one subdomain are numbered from this entry of gdesc on.
__device__ __forceinline__ size_t ras_group0(int s, int base, int pbase) {
  return 2 * (size_t)base + 8 * (size_t)s + (size_t)(pbase / RAS_K);
}

// Packs the factors of each subdomain into its stream (one block of four
// warps per subdomain; T: factor type, TB: stored type).  A warp takes a
// level at a time, its lanes the next 32 rows of the level's list, which
// become one group, or several when a row has more than RAS_K entries.  The
// groups are counted, numbered, sized and placed, then filled one warp each.
// (The first version split each level with one thread walking its rows: 0.47
// ms per setup on the 1M-cell case, bound by that thread's dependent loads.)
// The groups' tables lie in shared memory, or for subdomains of more than some
// 10,000 rows (GT) in global memory: the setup alone reads them, so they must
// not decide where the streamed apply ends (24x24x360 cells, BF16, 208
// iterations: 380 ms per step, RAS 244 us per launch).
template <class T, class TB, bool GT>
__global__ void __launch_bounds__(128) k_ras_pack(const int *sub_ptr, const int *lrp_ptr, const int *frp,
                                                  const int *fci, const int *fdiag, const int *ipos, const int *gord,
                                                  uint16_t *gpos, const T *fv, const T *dinv, const int *lvl_rows,
                                                  const int *nlev, const int *lvl_ptr, const long long *blob_off,
                                                  unsigned char *blobs, uint2 *gdesc, int *ngrp, const int *order,
                                                  int *err, int *lv_tab, int *gr_tab) {
  const int s = order[blockIdx.x], base = sub_ptr[s], m = sub_ptr[s + 1] - base, pbase = lrp_ptr[s], fbase = base + s;
  const int *pL = lvl_ptr + 2 * (base + s), *pU = pL + (m + 1);
  const int *rL = lvl_rows + 2 * base, *rU = rL + m;
  const int nL = nlev[2 * s], nU = nlev[2 * s + 1];
  unsigned char *b = blobs + blob_off[s];
  uint2 *gd = gdesc + ras_group0(s, base, pbase);
  constexpr int BPP = sizeof(TB) == 2 ? 2 : 1;              // blocks per piece
  constexpr int PB = sizeof(TB) == 8 ? 32 : 16;             // bytes per row of a piece
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  constexpr int AH = ras_ahead<TB>();
  __shared__ int ngr, ngl, pad0, pad1;                      // groups, those of the L sweep, the empty ones' starts
  // per level its group count (then the first group's index), per group its
  // bytes (then its start); at most 2 m levels
  extern __shared__ int psm[];
  const int nLw = nL > 1 ? nL - 1 : 0, nlevels = nLw + nU;
  int *lgc = GT ? lv_tab + 2 * (size_t)base + s : psm, *gby = GT ? gr_tab + ras_group0(s, base, pbase) : psm + nlevels + 1;
  // positions in gather order
  for (int k = threadIdx.x; k < m; k += blockDim.x) gpos[base + k] = (uint16_t)ipos[base + gord[base + k]];
  // groups of one level of the sweep order (L levels 1..nL-1, then U levels):
  // emit(up, row, entries of the row, first entry, part) in every lane, lanes
  // beyond the level with entries -1
  auto split = [&](int lv, auto emit) {
    const bool up = lv >= nLw;
    const int l = up ? lv - nLw : lv + 1;
    const int *pp = up ? pU : pL, *rr = up ? rU : rL;
    const int a1 = pp[l + 1];
    for (int a = pp[l]; a < a1; a += 32) {
      int i = 0, ne = -1, q0 = 0;
      if (a + lane < a1) {
        i = rr[a + lane];
        const int d = fdiag[base + i] - pbase;
        if (up) { q0 = d + 1; ne = frp[fbase + i + 1] - d - 1; }
        else { q0 = frp[fbase + i]; ne = d - q0; }
      }
      const int kmax = __reduce_max_sync(0xffffffffu, ne);
      for (int p = 0; p == 0 || p * RAS_K < kmax; p++) emit(up, i, ne, q0, p);
    }
  };
  for (int lv = wid; lv < nlevels; lv += nwarps) {                   // groups per level
    int c = 0;
    split(lv, [&](bool, int, int, int, int) { c++; });
    if (lane == 0) lgc[lv] = c;
  }
  __syncthreads();
  auto scan = [&](int *v, int n) {                                   // exclusive, one warp; returns the total
    int run = 0;
    for (int k0 = 0; k0 < n; k0 += 32) {
      int k = k0 + lane, t = k < n ? v[k] : 0, x = t;
      for (int o = 1; o < 32; o <<= 1) { int y = __shfl_up_sync(0xffffffffu, x, o); if (lane >= o) x += y; }
      if (k < n) v[k] = run + x - t;
      run += __shfl_sync(0xffffffffu, x, 31);
    }
    return run;
  };
  // first group of each level; the L sweep's groups, then the U sweep's, are
  // filled up to a multiple of AH
  if (wid == 0) {
    const int nl = scan(lgc, nLw), padl = (AH - nl % AH) % AH;
    const int nu = scan(lgc + nLw, nU), padu = (AH - nu % AH) % AH;
    for (int k = nLw + lane; k < nlevels; k += 32) lgc[k] += nl + padl;
    if (lane == 0) {
      ngl = nl + padl; ngr = nl + padl + nu + padu;
      for (int k = 0; k < padl; k++) gby[nl + k] = 16 + PB;
      for (int k = 0; k < padu; k++) gby[nl + padl + nu + k] = 16 + PB;
      pad0 = nl; pad1 = nl + padl + nu;                      // where the empty ones start
    }
  }
  __syncthreads();
  // blocks of a row in part p: its entries from p RAS_K on (at most RAS_K),
  // after the inverse diagonal block of a U row
  auto blocks = [&](bool up, int ne, int p) { return ne < 0 || (p > 0 && ne <= p * RAS_K) ? 0 : min(ne - p * RAS_K, RAS_K) + (up ? 1 : 0); };
  for (int lv = wid; lv < nlevels; lv += nwarps) {                   // bytes of each group
    int g = lgc[lv];
    split(lv, [&](bool up, int, int ne, int, int p) {
      const int nb = blocks(up, ne, p);
      const bool in = p == 0 ? ne >= 0 : ne > p * RAS_K;
      const int by = __reduce_add_sync(0xffffffffu, in ? 16 + (nb + BPP - 1) / BPP * PB : 0);
      if (lane == 0) gby[g] = by;
      g++;
    });
  }
  __syncthreads();
  const int ng = ngr;
  if (wid == 0) {
    const int total = scan(gby, ng);
    // the stream must fit its bound (rows and entries only); never false by
    // construction, checked so that a violation is an error, not an overrun
    if (lane == 0) {
      const bool fits = total <= blob_off[s + 1] - blob_off[s];
      if (!fits) { atomicExch(err, 4); ngr = 0; gd[0] = make_uint2(0, 0); }
      ngrp[2 * s] = fits ? ngl : 0; ngrp[2 * s + 1] = fits ? ng : 0;
    }
  }
  __syncthreads();
  if (ngr == 0) return;
  if (wid == 0 && lane < 2 * (AH - 1)) {                             // empty groups: row m + 1, columns m
    const int g = lane < AH - 1 ? pad0 + lane : pad1 + lane - (AH - 1);
    if (g < (lane < AH - 1 ? ngl : ng)) {
      const unsigned mm = (unsigned)m | (unsigned)m << 16;
      uint4 *G = reinterpret_cast<uint4 *>(b + gby[g]);
      G[0] = make_uint4((unsigned)(m + 1) | (unsigned)m << 16, mm, mm, (unsigned)m);
      for (int k = 0; k < PB / 16; k++) G[1 + k] = make_uint4(0, 0, 0, 0);
      gd[g] = make_uint2((unsigned)(gby[g] >> 4) | 1u << 20, 0);
    }
  }
  bool bad = false;                                                  // a stored value is not finite
  for (int lv = wid; lv < nlevels; lv += nwarps) {
    int g = lgc[lv];
    split(lv, [&](bool up, int i, int ne, int q0, int p) {
      const bool in = p == 0 ? ne >= 0 : ne > p * RAS_K;
      const int nb = blocks(up, ne, p), key = in ? nb : -1;
      // rows by descending block count (equal counts in list order)
      int rank = 0, before = 0;
      for (int c = RAS_K + 1; c >= 0; c--) {
        const unsigned eq = __ballot_sync(0xffffffffu, key == c);
        if (key == c) rank = before + __popc(eq & ((1u << lane) - 1u));
        before += __popc(eq);
      }
      const int rows = before;
      unsigned char *G = b + gby[g];
      // header: the row and its columns, missing ones naming the zero element
      const int qe = pbase + q0 + p * RAS_K, n = in ? nb - (up ? 1 : 0) : 0;
      if (in) {
        unsigned c[RAS_K + 2];
        c[0] = (unsigned)i; c[RAS_K + 1] = 0;
#pragma unroll
        for (int k = 0; k < RAS_K; k++) c[k + 1] = k < n ? (unsigned)fci[qe + k] : (unsigned)m;
        reinterpret_cast<uint4 *>(G)[rank] = make_uint4(c[0] | c[1] << 16, c[2] | c[3] << 16, c[4] | c[5] << 16, c[6] | c[7] << 16);
      }
      unsigned char *at = G + 16 * rows;
      unsigned nlo = 0, nhi = 0;                         // n[6], n[1..5]
      const bool fin = ne <= (p + 1) * RAS_K;
#pragma unroll
      for (int q = 0; q * BPP <= RAS_K; q++) {
        const int cnt = __popc(__ballot_sync(0xffffffffu, key > q * BPP));
        if (key > q * BPP) {
          TB *dst = reinterpret_cast<TB *>(at + (size_t)PB * rank);
#pragma unroll
          for (int u = 0; u < BPP; u++) {
            const int k = q * BPP + u - (up ? 1 : 0);    // -1: the inverse diagonal block
            T v[4] = {0, 0, 0, 0};
            if (k < 0) {
              if (fin) for (int w = 0; w < 4; w++) v[w] = dinv[4 * (size_t)(base + i) + w];
              else v[0] = v[3] = T(1);
            } else if (k < n) {
              for (int w = 0; w < 4; w++) v[w] = fv[4 * (size_t)(qe + k) + w];
            }
            for (int w = 0; w < 4; w++) {
              const TB z = to_blob_d<TB>(v[w]);
              dst[4 * u + w] = z;
              bad |= !isfinite((T)z);
            }
          }
        }
        at += PB * cnt;
        if (q >= 1 && q <= 5) nhi |= (unsigned)cnt << (6 * (q - 1));
        if (q == 6) nlo = (unsigned)cnt;
      }
      if (lane == 0) gd[g] = make_uint2((unsigned)(gby[g] >> 4) | (unsigned)rows << 20 | nlo << 26, nhi);
      g++;
    });
  }
  if (bad) atomicOr(&ngrp[2 * s + 1], RAS_NONFINITE);
}

template <class T> struct v2_t;
template <> struct v2_t<float> { typedef float2 type; };
template <> struct v2_t<double> { typedef double2 type; };

// x = R(A)^{-1} f, one block per subdomain.  The right-hand side is gathered
// into y; then group after group, each lane subtracts its row's products in
// stored order, a = f_i - sum_k B_k y_{c_k} (U rows: times the inverse
// diagonal block), and stores y_i; at the end the owned rows are written (or
// added).  Groups depend on earlier ones, so a block's time is its group
// count (70 to 150 on the 1M-cell case) times one group's latency, which is
// mostly one warp's own instructions.  They are kept few and free of
// branches, so that the loads of a later group fill the waits of the current
// one (a uniform branch costs about as much as a block's product; the same
// sweep with a test per entry took 108 us per launch on the 1M-cell case): a
// group's pieces come straight from global memory into registers, ras_ahead
// groups early (every lane its own row; no ring, no waits), missing entries
// multiply the zero element, and what a lane or a group does not have keeps an
// earlier group's values, which only ever multiply that zero or are not
// stored.  A subdomain with a value that is not finite (a singular block)
// takes a copy of the sweeps that clears them, so that Inf and NaN stay in the
// rows that depend on it.  A bulk prefetch into L2 runs RAS_PF_BYTES ahead of
// the loads.  One lane per row, BF16: 20 blocks per SM (at most 96 registers),
// since with 113 the 2500 subdomains of the 1M-cell case needed a second wave
// (111 us); FP64 input spills 120 bytes at that limit and takes the same 85
// us.  FP32 factors take 124 registers, 16 blocks per SM; the 68 subdomains
// that then start late are the shortest (longest first): 84 us.
//
// Per launch in the solver, against the sweep it replaces (factors through a
// shared-memory ring, products by entry, then sums by row): 1M cells, BF16,
// 137 -> 84 us; 200k, FP32, 74 -> 44 us; 65k, BF16, 75 -> 36 us; 207k, FP64,
// 190 -> 98 us; 2,000 cells, FP64, 54 -> 34 us.
//
// FP64: the pipe takes 64 cycles per warp instruction whatever the number of
// active lanes (measured), so two lanes share a row, one component each, and
// a block has two warps: half the FP64 instructions in each warp's chain,
// and the four sub-partitions' pipes evenly used; slots that none of a warp's
// rows has are skipped.
// FP32 and BF16 use two lanes per row as well while all blocks are resident
// (RAS_W2_MAX): each lane issues half the products and shuffles of a group.
// Per launch, one against two lanes: 200k, FP32, 43 -> 37 us; 65k, BF16, 36 ->
// 28 us; 150k with overlap 2, 44 -> 39 us; 155k, 33 -> 29 us.  Beyond one wave
// the second warp's instructions compete with the other blocks' (1M cells:
// one lane, 84 us).  The rule counts subdomains only, since two lanes also win
// where the vectors of thick models leave fewer blocks resident (BF16, one
// against two lanes: 256 subdomains of 360 layers, two per SM, 381 -> 281 us;
// 576 of them 683 -> 498; 900 of 200 layers, four per SM, 396 -> 318).
#define RAS_PF_BYTES 8192
#define RAS_PF_STEP 2048
#define RAS_W2_MAX (152 * 8)
template <int NP> struct ras_group { uint2 d; uint4 h; uint4 p[NP]; };
template <class T, class Tin, bool ACC, class TB, int LPR>
__global__ void __launch_bounds__(32 * LPR, LPR == 2 ? 8 : sizeof(TB) == 2 ? 20 : 16)
k_ras_apply_stream(const long long *blob_off, const unsigned char *blobs, const int *gidx_all, const uint16_t *gpos_all,
                   const int *nown, const uint2 *gdesc, const int *ngrp, const int *lrp_ptr, const int *sub_ptr,
                   const int *order, const Tin *f, T *x) {
  constexpr bool D = sizeof(T) == 8, W2 = LPR == 2;    // W2: two lanes per row, one component each
  constexpr int BS = 32 * LPR, BPP = sizeof(TB) == 2 ? 2 : 1, NP = RAS_K / BPP + 1, AHEAD = ras_ahead<TB>();
  typedef typename v2_t<T>::type T2;
  typedef typename v2_t<Tin>::type Tin2;
  extern __shared__ uint4 sm4[];
  T2 *y = reinterpret_cast<T2 *>(sm4);
  const int tid = threadIdx.x, row_of = tid / LPR, comp = tid & 1;
  const int s = order[blockIdx.x], base = sub_ptr[s], m = sub_ptr[s + 1] - base, no = nown[s];
  const int ngl = ngrp[2 * s], ngw = ngrp[2 * s + 1], ng = ngw & ~RAS_NONFINITE;
  const int *gidx = gidx_all + base;
  const uint16_t *gpos = gpos_all + base;
  const unsigned char *st = blobs + blob_off[s];
  const uint4 *st_h = reinterpret_cast<const uint4 *>(st) + row_of, *st_b = reinterpret_cast<const uint4 *>(st) + (D ? tid : row_of);
  const uint2 *gd = gdesc + ras_group0(s, base, lrp_ptr[s]);
  const int bound = (int)(blob_off[s + 1] - blob_off[s]), glast = max(ng - 1, 0);
  auto sync = [&]() { if (W2) __syncthreads(); else __syncwarp(); };
  pdl_trigger();
  int pf = min(bound, RAS_PF_BYTES);                   // the stream is prefetched into L2 up to here
  if (tid == 0)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(st), "r"(pf) : "memory");
  ras_group<NP> S[AHEAD];
  const unsigned mm = (unsigned)m | (unsigned)m << 16;
#pragma unroll
  for (int k = 0; k < AHEAD; k++) {
    S[k].h = make_uint4(mm, mm, mm, mm);
#pragma unroll
    for (int q = 0; q < NP; q++) S[k].p[q] = make_uint4(0, 0, 0, 0);
  }
  // descriptors of the next groups to load, fetched two groups before their use
  int gq = 0;
  auto fetch_desc = [&]() { const uint2 d = __ldg(gd + min(gq, glast)); gq++; return d; };
  uint2 dq0 = fetch_desc(), dq1 = fetch_desc();
  // the next group into a register set; CLEAR: what the lane's row does not
  // have becomes zero
  auto load = [&](ras_group<NP> &G, auto clear_) {
    constexpr bool CLEAR = decltype(clear_)::value;
    const uint2 d = dq0;
    dq0 = dq1;
    dq1 = fetch_desc();
    const int rows = (d.x >> 20) & 63, start = d.x & 0xfffff;
    G.d = d;
    if (row_of < rows) {
      G.h = __ldg(st_h + start);
      G.p[0] = __ldg(st_b + (start + rows));
    }
    int q = start + (D ? 3 : 2) * rows;                // in units of 16 bytes
#pragma unroll
    for (int k = 1; k < NP; k++) {
      const int n = k < 6 ? (d.y >> (6 * (k - 1))) & 63 : d.x >> 26;
      if (row_of < n) G.p[k] = __ldg(st_b + q);
      else if (CLEAR) G.p[k] = make_uint4(0, 0, 0, 0);
      q += (D ? 2 : 1) * n;
    }
    // prefetch (thread 0) when the loads come within RAS_PF_BYTES of it
    const bool go = 16 * start + RAS_PF_BYTES > pf && pf < bound;
    const int len = min(bound - pf, RAS_PF_STEP);
    asm volatile("{\n .reg .pred p;\n setp.ne.s32 p, %2, 0;\n @p cp.async.bulk.prefetch.L2.global [%0], %1;\n}\n" ::"l"(
                     st + pf), "r"(len), "r"((int)(go && tid == 0)) : "memory");
    pf += go ? len : 0;
  };
  // gather the extended right-hand side, the first indices ahead of the wait
  // for the kernel that makes f (all other inputs are fixed between setups)
  const Tin2 *f2 = reinterpret_cast<const Tin2 *>(f);
  constexpr int GU = W2 ? 8 : 16;
  int gi[GU], pos[GU];
  auto indices = [&](int p0) {
#pragma unroll
    for (int u = 0; u < GU; u++)
      if (p0 + u * BS < m) { gi[u] = gidx[p0 + u * BS]; pos[u] = gpos[p0 + u * BS]; }
  };
  indices(tid);
  pdl_wait();
  for (int p0 = tid; p0 < m; p0 += GU * BS) {
    Tin2 v[GU];
    if (p0 != tid) indices(p0);
#pragma unroll
    for (int u = 0; u < GU; u++) if (p0 + u * BS < m) v[u] = f2[gi[u]];
#pragma unroll
    for (int u = 0; u < GU; u++)
      if (p0 + u * BS < m) { T2 t; t.x = (T)v[u].x; t.y = (T)v[u].y; y[pos[u]] = t; }
  }
#pragma unroll
  for (int k = 0; k < AHEAD; k++) load(S[k], std::false_type());      // (the sets are zero)
  if (tid < 2) { T2 z; z.x = 0; z.y = 0; y[m + tid] = z; }
  sync();
  // one group: blocks of piece k are k BPP .. ; in a U group block 0 is the
  // inverse diagonal and block b entry b - 1, in an L group block b entry b
  auto solve = [&](const ras_group<NP> &G, auto up_) {
    constexpr int UP = decltype(up_)::value;
    constexpr int NB = RAS_K + UP;                      // blocks at most
    const int rows = (G.d.x >> 20) & 63;
    auto n_of = [&](int k) { return k == 0 ? rows : (int)(k < 6 ? (G.d.y >> (6 * (k - 1))) & 63 : G.d.x >> 26); };
    auto col = [&](int e) {                             // entry e's column
      const unsigned w = e == 0 ? G.h.x : e <= 2 ? G.h.y : e <= 4 ? G.h.z : G.h.w;
      return (e & 1) == 0 ? w >> 16 : w & 0xffffu;
    };
    const int row = G.h.x & 0xffffu;
    const int wfirst = D ? (tid >> 5) * 16 : 0;         // FP64: the warp's first row
    T2 yc[RAS_K];
    T a0;
    [[maybe_unused]] T a1 = 0;
    if constexpr (W2) a0 = reinterpret_cast<const T *>(y + row)[comp];
    else { const T2 t = y[row]; a0 = t.x; a1 = t.y; }
#pragma unroll
    for (int e = 0; e < RAS_K; e++) yc[e] = y[col(e)];
#pragma unroll
    for (int k = 0; k * BPP < NB; k++) {
      if (D && n_of(k) <= wfirst) break;
#pragma unroll
      for (int u = 0; u < BPP; u++) {
        const int e = k * BPP + u - UP;
        if (e < 0 || e >= RAS_K) continue;
        if constexpr (D) {
          const double bx = __hiloint2double(G.p[k].y, G.p[k].x), by = __hiloint2double(G.p[k].w, G.p[k].z);
          a0 = __fma_rn(-bx, yc[e].x, a0);
          a0 = __fma_rn(-by, yc[e].y, a0);
        } else if constexpr (W2) {
          float bx, by;
          if constexpr (BPP == 2) {
            const unsigned w = u ? (comp ? G.p[k].w : G.p[k].z) : (comp ? G.p[k].y : G.p[k].x);
            bx = __uint_as_float(w << 16); by = __uint_as_float(w & 0xffff0000u);
          } else {
            bx = __uint_as_float(comp ? G.p[k].z : G.p[k].x); by = __uint_as_float(comp ? G.p[k].w : G.p[k].y);
          }
          a0 = __fsub_rn(a0, __fmaf_rn(bx, yc[e].x, __fmul_rn(by, yc[e].y)));
        } else {
          float b0, b1, b2, b3;
          if constexpr (BPP == 2) blk4(u ? G.p[k].z : G.p[k].x, u ? G.p[k].w : G.p[k].y, b0, b1, b2, b3);
          else { b0 = __uint_as_float(G.p[k].x); b1 = __uint_as_float(G.p[k].y); b2 = __uint_as_float(G.p[k].z); b3 = __uint_as_float(G.p[k].w); }
          // product first, then the subtraction: the same FP32 values as the
          // sweeps have always had, and a shorter chain than two FMAs per entry
          a0 = __fsub_rn(a0, __fmaf_rn(b0, yc[e].x, __fmul_rn(b1, yc[e].y)));
          a1 = __fsub_rn(a1, __fmaf_rn(b2, yc[e].x, __fmul_rn(b3, yc[e].y)));
        }
      }
    }
    if constexpr (UP) {
      if constexpr (D) {
        const double dx = __hiloint2double(G.p[0].y, G.p[0].x), dy = __hiloint2double(G.p[0].w, G.p[0].z);
        if (rows > wfirst) {
          const double o = __shfl_xor_sync(0xffffffffu, a0, 1);
          a0 = __fma_rn(comp ? dy : dx, a0, (comp ? dx : dy) * o);
        }
      } else if constexpr (W2) {
        float dx, dy;
        if constexpr (BPP == 2) {
          const unsigned w = comp ? G.p[0].y : G.p[0].x;
          dx = __uint_as_float(w << 16); dy = __uint_as_float(w & 0xffff0000u);
        } else {
          dx = __uint_as_float(comp ? G.p[0].z : G.p[0].x); dy = __uint_as_float(comp ? G.p[0].w : G.p[0].y);
        }
        const float o = __shfl_xor_sync(0xffffffffu, a0, 1), ax = comp ? o : a0, ay = comp ? a0 : o;
        a0 = dx * ax + dy * ay;
      } else {
        float d0, d1, d2, d3;
        if constexpr (BPP == 2) blk4(G.p[0].x, G.p[0].y, d0, d1, d2, d3);
        else { d0 = __uint_as_float(G.p[0].x); d1 = __uint_as_float(G.p[0].y); d2 = __uint_as_float(G.p[0].z); d3 = __uint_as_float(G.p[0].w); }
        const float t = d0 * a0 + d1 * a1;
        a1 = d2 * a0 + d3 * a1;
        a0 = t;
      }
    }
    if (row_of < rows) {
      if constexpr (W2) reinterpret_cast<T *>(y + row)[comp] = a0;
      else { T2 t; t.x = a0; t.y = a1; y[row] = t; }
    }
  };
  auto sweep = [&](int n, auto up_, auto clear_) {       // n groups, a multiple of AHEAD
    for (int g = 0; g < n; g += AHEAD) {
#pragma unroll
      for (int k = 0; k < AHEAD; k++) { solve(S[k], up_); load(S[k], clear_); sync(); }
    }
  };
  auto sweeps = [&](auto clear_) {
    sweep(ngl, std::integral_constant<int, 0>(), clear_);
    sweep(ng - ngl, std::integral_constant<int, 1>(), clear_);
  };
  if (ngw & RAS_NONFINITE) sweeps(std::true_type());
  else sweeps(std::false_type());
  for (int p0 = tid; p0 < no; p0 += 8 * BS) {            // the owned rows come first in gather order
    T2 v[8], w[8];
#pragma unroll
    for (int u = 0; u < 8; u++)
      if (p0 + u * BS < no) {
        gi[u] = gidx[p0 + u * BS];
        v[u] = y[gpos[p0 + u * BS]];
        if (ACC) w[u] = reinterpret_cast<const T2 *>(x)[gi[u]];
      }
#pragma unroll
    for (int u = 0; u < 8; u++)
      if (p0 + u * BS < no) {
        if (ACC) { v[u].x += w[u].x; v[u].y += w[u].y; }
        reinterpret_cast<T2 *>(x)[gi[u]] = v[u];
      }
  }
}

template <class T, class TB> static void ras_pack_go(sim_ls_s *ls, const T *fv, const T *dinv) {
  ras_data &R = ls->ras;
  auto go = [&](auto kern, size_t smem) {
    kern<<<R.nsub, 128, smem, ls->st>>>(R.sub_ptr.p, R.lrp_ptr.p, R.frp.p, R.fci.p, R.fdiag.p, R.ipos.p, R.gord.p,
                                        R.gpos.p, fv, dinv, R.pruned ? R.alvl_rows.p : R.lvl_rows.p, R.nlev.p,
                                        R.pruned ? R.alvl_ptr.p : R.lvl_ptr.p, R.blob_off.p, R.blob.p, R.gdesc.p,
                                        R.ngrp.p, R.order.p, ls->errw_dev, R.pack_lv.p, R.pack_gr.p);
  };
  if (R.pack_smem > RAS_SMEM_BUDGET) go(k_ras_pack<T, TB, true>, 0);
  else {
    static bool attr = false;
    if (!attr) {
      RS_CUDA(cudaFuncSetAttribute(k_ras_pack<T, TB, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, RAS_SMEM_BUDGET));
      attr = true;
    }
    go(k_ras_pack<T, TB, false>, R.pack_smem);
  }
  RS_LAUNCHED(1);
}
void ras_pack(sim_ls_s *ls) {
  ras_data &R = ls->ras;
  if (!R.smem_path) return;
  if (ls->o.precision == SIM_PREC_MIXED_BF16) ras_pack_go<float, __nv_bfloat16>(ls, R.fval32.p, R.dinv32.p);
  else if (ls->o.precision != SIM_PREC_FP64) ras_pack_go<float, float>(ls, R.fval32.p, R.dinv32.p);
  else ras_pack_go<double, double>(ls, R.fval.p, R.dinv.p);
}

template <class T, class Tin>
__global__ void k_cast_acc(size_t m, const Tin *a, T *b, bool acc) {
  size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i < m) b[i] = acc ? b[i] + (T)a[i] : (T)a[i];
}

template <class T, class Tin, class TB>
static void ras_apply_go(sim_ls_s *ls, const Tin *f, T *x, bool acc) {
  ras_data &R = ls->ras;
#define RAS_APPLY_ARGS R.blob_off.p, R.blob.p, R.gidx.p, R.gpos.p, R.nown.p, R.gdesc.p, R.ngrp.p, R.lrp_ptr.p, R.sub_ptr.p, R.order.p, f, x
  auto go = [&](auto kern, int lpr) { launch_pdl(kern, R.nsub, 32 * lpr, R.smem_bytes, ls->st, RAS_APPLY_ARGS); };
  if (sizeof(T) == 8 || R.nsub <= RAS_W2_MAX) {
    if (acc) go(k_ras_apply_stream<T, Tin, true, TB, 2>, 2); else go(k_ras_apply_stream<T, Tin, false, TB, 2>, 2);
  } else if constexpr (sizeof(T) == 4) {
    if (acc) go(k_ras_apply_stream<T, Tin, true, TB, 1>, 1); else go(k_ras_apply_stream<T, Tin, false, TB, 1>, 1);
  }
#undef RAS_APPLY_ARGS
}
template <class T, class Tin> static void ras_apply_launch(sim_ls_s *ls, const Tin *f, T *x, bool acc);
template <> void ras_apply_launch<double, double>(sim_ls_s *ls, const double *f, double *x, bool acc) {
  ras_apply_go<double, double, double>(ls, f, x, acc);
}
template <> void ras_apply_launch<float, float>(sim_ls_s *ls, const float *f, float *x, bool acc) {
  if (ls->o.precision == SIM_PREC_MIXED_BF16) ras_apply_go<float, float, __nv_bfloat16>(ls, f, x, acc);
  else ras_apply_go<float, float, float>(ls, f, x, acc);
}
template <> void ras_apply_launch<float, double>(sim_ls_s *ls, const double *f, float *x, bool acc) {
  if (ls->o.precision == SIM_PREC_MIXED_BF16) ras_apply_go<float, double, __nv_bfloat16>(ls, f, x, acc);
  else ras_apply_go<float, double, float>(ls, f, x, acc);
}

template <class T, class Tin> void ls_ras_apply(sim_ls_s *ls, const Tin *f, T *x, bool accumulate) {
  ras_data &R = ls->ras;
  cudaStream_t s = ls->st;
  if (R.smem_path) {
    static bool attr = false;
    if (!attr) {
#define RAS_ATTR(...)                                                                                              \
  RS_CUDA(cudaFuncSetAttribute(k_ras_apply_stream<__VA_ARGS__>, cudaFuncAttributeMaxDynamicSharedMemorySize, RAS_SMEM_BUDGET))
#define RAS_ATTR4(T, Tin, TB)                                                                                      \
  RAS_ATTR(T, Tin, false, TB, 2); RAS_ATTR(T, Tin, true, TB, 2); RAS_ATTR(T, Tin, false, TB, 1); RAS_ATTR(T, Tin, true, TB, 1)
      RAS_ATTR4(float, float, float); RAS_ATTR4(float, double, float);
      RAS_ATTR4(float, float, __nv_bfloat16); RAS_ATTR4(float, double, __nv_bfloat16);
      RAS_ATTR(double, double, false, double, 2); RAS_ATTR(double, double, true, double, 2);
#undef RAS_ATTR4
#undef RAS_ATTR
      attr = true;
    }
    rs_timed tm(ls, SIM_T_RAS);
    ras_apply_launch<T, Tin>(ls, f, x, accumulate);
    RS_LAUNCHED(1);
    return;
  }
  // global-memory path (subdomains too large for shared memory)
  size_t nu = 2 * (size_t)ls->nb;
  static thread_local dbuf<T> tin, tout;
  const T *fin = reinterpret_cast<const T *>(f);
  if (sizeof(Tin) != sizeof(T)) {
    tin.ensure(nu);
    k_cast_acc<T, Tin><<<grid_for(nu, 256), 256, 0, s>>>(nu, f, tin.p, false);
    RS_LAUNCHED(1);
    fin = tin.p;
  }
  T *xout = x;
  if (accumulate) { tout.ensure(nu); xout = tout.p; }
  size_t smem = (size_t)R.max_ext * 2 * sizeof(T);
  static bool attr2 = false;
  if (!attr2) {
    RS_CUDA(cudaFuncSetAttribute(k_ras_apply<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    RS_CUDA(cudaFuncSetAttribute(k_ras_apply<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    attr2 = true;
  }
  bool mixed = sizeof(T) == 4;
  {
    rs_timed tm(ls, SIM_T_RAS);
    k_ras_apply<T><<<R.nsub, 256, smem, s>>>(R.sub_ptr.p, R.ext.p, R.owned.p, R.lrp_ptr.p, R.frp.p, R.fci.p,
                                             R.fdiag.p, R.perm.p, R.lvl_rows.p, R.nlev.p, R.lvl_ptr.p,
                                             mixed ? (const T *)R.fval32.p : (const T *)R.fval.p,
                                             mixed ? (const T *)R.dinv32.p : (const T *)R.dinv.p, fin, xout);
    RS_LAUNCHED(1);
  }
  if (accumulate) {
    k_cast_acc<T, T><<<grid_for(nu, 256), 256, 0, s>>>(nu, xout, x, true);
    RS_LAUNCHED(1);
  }
}
template void ls_ras_apply<double, double>(sim_ls_s *, const double *, double *, bool);
template void ls_ras_apply<float, float>(sim_ls_s *, const float *, float *, bool);
template void ls_ras_apply<float, double>(sim_ls_s *, const double *, float *, bool);
