// FP64 pressure Poisson solve (Eq. pm_poisson) by CG on the Jacobi-scaled system (pcg_scaled.cu)
// with ONE grid barrier per iteration.
//
// Plainly, an iteration needs two device-wide barriers: one so that the stencil
// w = K~ r sees the neighbours' new residual, one for the dot products.  Here each block
// owns a 2-D tile of cells and computes the new residual of the one-cell ring around its tile
// itself, from the previous iteration's vectors:
//     r_{i+1} = r_i - alpha_i (w_i + beta_i s_{i-1})      (= r_i - alpha_i s_i),
// so the stencil needs no other block's work of the same iteration and only the reduction
// needs a barrier.
//
// Two kernels run this iteration: k_pcg_poisson_f1 (pcg_fused_global.cu) keeps the vectors in global
// memory; k_pcg_poisson_f2 here keeps its tile's x~, r, p, s and w in shared memory for the whole
// solve.  Per iteration, in each block of f2:
//   1. own cells: s_i, r_{i+1}; ring cells: r_{i+1}, in the frame of the tile's r (zero outside the
//      domain)
//   2. block barrier; own cells: w_{i+1} = K~ r_{i+1} and the sums; the grid barrier
//   3. every block forms the scalars from the same sums.
// With one barrier per iteration a block can publish the next iteration's partials while a
// slower block still reads this iteration's, so the partials alternate between two sets of
// rows by iteration parity.
// Tiles are TX x TY cells (TX a power of two, 32..512), one per block; the host picks the
// shape that makes the largest tile smallest (fused_plan.h).
//
// f2's ring needs one value per cell and iteration from the neighbours: w.  The ring's r and s are
// kept by the tile that reads them, updated with the same recurrences as their owner's (equal bit
// for bit), so a tile pushes the w of its perimeter into its neighbours' mailboxes (one 16-byte slot
// per ring cell holding the value and the iteration's number, double-buffered by parity) and reads
// its own mailbox.  The slot's tag says that the value is there, and the words of the reduction carry
// the sums, so no release or acquire, and no wait for outstanding stores, is left in the iteration.
//
// One further warp per block (the communication warp) sums the block's digits, adds them to the
// reduction's words, waits for the grid's and forms the scalars of the next iteration in integer
// arithmetic (pcg_scalar.cuh), while the other warps do the work that no other block reads:
// p = r_i + beta p and x~ += alpha p (r_i is kept beside r_{i+1} in a second framed copy,
// where the tile leaves room for it: otherwise p is formed in step 1 and only x~ waits), and the
// wait for the ring's next w.  The FP64 pipe (one warp instruction per 64 cycles on each
// sub-partition) stays with the vectors, and the serial chain beside it.
//
// The sums of the iterations (reductions 1, 2, ...) are exact fixed-point sums that travel
// with the grid barrier (pcg_fixed.cuh): the block's arrival adds its digit sums to words in
// global memory and the wait on those words ends with the grid's sums in hand, so neither the
// block sum nor the grid sum is a chain of FP64 additions.  Reduction 0 (phase 0) and the
// rare reduction whose values leave the fixed-point window take the FP64 sums.
//
// What bounds it: on 1024x512 the FP64 pipe (10 operations per cell: 8.4 us of the 10.9 us per
// iteration; 12.7 us with published r, w and s, release and acquire, and FP64 scalars), on small
// grids the chain of one iteration: step, stencil, digits, one L2 hop between SMs (907 cycles
// measured), scalars (128x64: 3.3 us per iteration against 4.3 us).
//
// Threads: NT = 128, 256 or 512 by the tile's cells (fused_threads), one to ten rows of the tile
// each, so that a small tile is not paced by the block sums and barriers of idle warps.
#include <algorithm>

#include "pcg_common.cuh"
#include "batch_common.cuh"
#include "pcg_scalar.cuh"

namespace ccm {

namespace {

// Shared memory of a block besides the tile (dynamic).
template <int NT>
struct FusedShared {
  double red[4][NT];
  double bsum[8];
  double gsum[8];
  double alpha, beta, rr, bb;
  double nn;  // singular systems: squared norm of the null vector, sum of d over the active cells
  int stop, lo, redo;
  // a wait that ran out: before the block barrier that ends step 1 (fail) and after it (late); each is read
  // behind the barrier that follows its waits and written again only behind the next one
  int fail, late;
  int scan[NT / 32 + 1];
  FxShared<NT> fx;
};

// Named barrier 2 hands the block's digits to the communication warp (which alone waits).
template <int NT>
__device__ __forceinline__ void digits_ready(bool wait) {
  if (wait) asm volatile("bar.sync 2, %0;" ::"n"(NT + 32) : "memory");
  else asm volatile("bar.arrive 2, %0;" ::"n"(NT + 32) : "memory");
}

// One tile of a solve: tile `tile` of the case's f.ntiles, one block of NT + 32 threads each.
template <int NT>
__device__ __forceinline__ void fused_body(const FusedSolve& f, const int tile, FusedShared<NT>& sh) {
  // dynamic shared memory: x~, p, s, w of the tile (TX*TY each), r~ of the tile in a one-cell
  // frame ((TX+2)*(TY+2), the frame holding the ring), with f.defer twice, then the ring's s
  // [W: TY][E: TY][S: TX][N: TX], then with f.dcache the five scaled coefficients of every cell,
  // with f.lcache those of the first NT listed cells, then the list
  extern __shared__ double dyn[];
  unsigned int target = 0;
  const ScaledSolve& a = f.a;
  const int nb = f.ntiles;
  const Geom& g = a.g;
  const int nx = g.nx, ny = g.ny, P = g.pitch;
  const int TX = f.TX, TY = f.TY;
  const int bx = tile % f.nbx, by = tile / f.nbx;
  const int i0 = bx * TX, j0 = by * TY;
  const int i1 = min(i0 + TX, nx), j1 = min(j0 + TY, ny);
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const bool comm = t >= NT;  // the communication warp
  const int tx = t % TX, ty0 = t / TX, RP = NT / TX;
  const int ci = i0 + tx;  // this thread's column
  const int TXY = TX * TY;
  // this thread's own cells: column ci, rows j0 + ty0 + q RP, q < nq; tile-local index t + q NT
  const int nq = !comm && ci < i1 && j0 + ty0 < j1 ? (j1 - j0 - ty0 + RP - 1) / RP : 0;
  const size_t k0 = g.idx(ci, j0 + ty0);  // of own cell 0 (used where nq > 0)
  const size_t kstep = (size_t)RP * P;
  double* const sx = dyn;
  double* const sp = dyn + TXY;
  double* const ss = dyn + 2 * TXY;
  double* const sw = dyn + 3 * TXY;
  // r~ of the tile with a one-cell frame that holds the ring, so that the stencil reads every
  // neighbour from one array without a branch; with defer two of them alternate
  const int TXP = TX + 2, FR = TXP * (TY + 2);
  const int lp0 = (ty0 + 1) * TXP + tx + 1, lpstep = RP * TXP;  // frame index of own cell 0, and step
  const bool defer = f.defer != 0;
  double* sr = dyn + 4 * TXY;                         // r_i
  double* srn = defer ? sr + FR : sr;                 // r_{i+1}
  double* const ring = dyn + 4 * TXY + (defer ? 2 : 1) * FR;
  double* const dcoef = ring + 2 * (TX + TY);
  double* const lcoef = dcoef + (f.dcache ? 5 * TXY : 0);
  int* const list = reinterpret_cast<int*>(lcoef + (f.lcache ? 5 * NT : 0));
  // index of cell (i, j) of the tile or its frame in the framed r~
  auto lpad = [&](int i, int j) -> int { return (j - j0 + 1) * TXP + (i - i0 + 1); };
  // ring cells: W and E columns, then S and N rows, taken by threads t, t + NT, ...
  const int nring = 2 * (j1 - j0) + 2 * (i1 - i0);
  // cell (ri, rj) of ring position q and its slot in `ring`; false outside the domain,
  // where the value is 0
  auto ring_cell = [&](int q, int& ri, int& rj, int& slot) -> bool {
    const int h = j1 - j0, w = i1 - i0;
    if (q < h) { ri = i0 - 1; rj = j0 + q; slot = q; }
    else if ((q -= h) < h) { ri = i1; rj = j0 + q; slot = TY + q; }
    else if ((q -= h) < w) { ri = i0 + q; rj = j0 - 1; slot = 2 * TY + q; }
    else { q -= w; ri = i0 + q; rj = j1; slot = 2 * TY + f.wx + q; }
    return ri >= 0 && ri < nx && rj >= 0 && rj < ny;
  };
  int my_ri = 0, my_rj = 0, my_slot = 0;
  const bool my_ring = !comm && t < nring;
  const bool my_in = my_ring && ring_cell(t, my_ri, my_rj, my_slot);
  const int my_lp = lpad(my_ri, my_rj);
  // the mailbox, f.mail[parity][tile][slot]; nslot slots per tile (f.wx: the tile's width
  // clipped to the grid's)
  const int nslot = 2 * (TY + f.wx);
  auto mailbox = [&](int parity, int q) -> ulonglong2* { return f.mail + ((size_t)parity * nb + q) * nslot; };
  // w~ of a perimeter cell to the ring of every neighbour that reads it: first slots of the
  // neighbours' rows (columns) that face this tile, -1 where there is no neighbour
  const bool sends = tile != a.bar.silent;
  const int slotW = sends && bx > 0 ? (tile - 1) * nslot + TY : -1, slotE = sends && i1 < nx ? (tile + 1) * nslot : -1;
  const int slotS = sends && by > 0 ? (tile - f.nbx) * nslot + 2 * TY + f.wx : -1;
  const int slotN = sends && j1 < ny ? (tile + f.nbx) * nslot + 2 * TY : -1;
  const int hi_ = i1 - i0 - 1, hj_ = j1 - j0 - 1;  // last column and row
  // (ir, jr): the cell within the tile
  auto push = [&](int parity, unsigned int tag, int ir, int jr, double wk) {
    ulonglong2* const m = mailbox(parity, 0);
    if (ir == 0 && slotW >= 0) tag_put(m + slotW + jr, wk, tag);
    if (ir == hi_ && slotE >= 0) tag_put(m + slotE + jr, wk, tag);
    if (jr == 0 && slotS >= 0) tag_put(m + slotS + ir, wk, tag);
    if (jr == hj_ && slotN >= 0) tag_put(m + slotN + ir, wk, tag);
  };
  const bool edge_col = tx == 0 || tx == hi_;
  const int8_t* __restrict__ kinds = a.kinds;
  const double* __restrict__ cus = a.cus;
  const double* __restrict__ cvs = a.cvs;
  const double* __restrict__ sd = a.sd;
  const double ax = a.ax, ay = a.ay, dreg = a.dreg;
  auto sync_grid = [&]() -> bool { return range_sync(a.bar, a.bar.count, (unsigned int)nb, target); };

  // r~ of own cell (i, j) and its neighbours after step 1
  auto gather = [&](int i, int j, double (&r)[5]) {
    const double* q = srn + lpad(i, j);
    r[0] = q[0]; r[1] = q[-1]; r[2] = q[1]; r[3] = q[-TXP]; r[4] = q[TXP];
  };
  // w~ of own cell (i, j), tile-local index l, into the tile, the perimeter's also to the neighbours
  auto wput = [&](int parity, unsigned int tag, int i, int j, int l, double wk) {
    sw[l] = wk;
    if (i == i0 || i == i1 - 1 || j == j0 || j == j1 - 1) push(parity, tag, i - i0, j - j0, wk);
  };
  // Rows of cut cells and rows next to a Neumann side (kind 2) are listed per tile, in a fixed
  // order, at the start.  The stencil pass applies the constant stencil to every own cell, so
  // no warp diverges (an FP64 warp instruction costs the same however few of its lanes are
  // active); a second pass, spread densely over the threads, computes the listed cells.
  // Inactive cells (identity rows, kind 0) get their exact solution x = b in phase 0 and zero
  // in every vector after it.  A tile takes the general row for every cell instead where that is
  // shorter: a warp then runs 8 FP64 operations per row instead of 6, and none of the 8 of each
  // round of listed cells (a stretched mesh, every row of which has coefficients of its own; a
  // small tile, of a few rows per thread, with any listed cell); and where the list does not hold
  // them.  (The scaled coefficient arrays hold the constants on uniform rows and zeros on inactive
  // ones.)
  unsigned int m_in = 0u, m_list = 0u;  // bit q: own cell q is inactive, is listed (nq <= 32)
  int nlist = 0;
  bool dense = false;
  {
    int mine = 0;
    for (int q = 0; q < nq; ++q) {
      const int8_t km = kinds[k0 + q * kstep];
      mine += km == 2;
      m_in |= (km == 0 ? 1u : 0u) << q;
      m_list |= (km == 2 ? 1u : 0u) << q;
    }
    // exclusive scan of the counts over the block (thread order)
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (!comm && lane == 31) sh.scan[wid] = incl;
    __syncthreads();
    if (t == 0) {
      int acc = 0;
      for (int q = 0; q < NT / 32; ++q) {
        const int c = sh.scan[q];
        sh.scan[q] = acc;
        acc += c;
      }
      sh.scan[NT / 32] = acc;
      sh.fail = sh.late = 0;
    }
    __syncthreads();
    nlist = sh.scan[NT / 32];
    const int rows = (j1 - j0 + RP - 1) / RP;
    dense = nlist > f.list_cap || 8 * rows < 6 * rows + 8 * ((nlist + NT - 1) / NT);
    if (!dense && mine > 0) {
      int at = sh.scan[wid] + incl - mine;
      for (int q = 0; q < nq; ++q)
        if (kinds[k0 + q * kstep] == 2) list[at++] = t + q * NT;
    }
    __syncthreads();
  }
  // Listed cell q is computed by thread NT - 1 - q (then NT - 1 - q + NT, ...): threads are
  // ordered by the first row they take, so the last threads have the fewest own rows (with
  // TY = 27 and 4 rows per pass, the last 128 threads take 6 rows and the others 7), and a
  // tile's listed cells fill those free slots before they lengthen any warp.  An FP64-bound
  // sub-partition's time is the sum over its warps, and the slowest tile sets every
  // iteration's barrier.
  const int myq = comm || dense ? nlist : NT - 1 - t;
  int q_l = -1, q_i = 0, q_j = 0;  // this thread's first listed cell
  if (myq < nlist) {
    q_l = list[myq];
    q_i = i0 + q_l % TX;
    q_j = j0 + q_l / TX;
  }
  // The coefficients that the solve reads in every iteration, cached: W, E, S, N and d - dreg
  auto coefs = [&](size_t k, double (&c)[5]) {
    c[0] = cus[k]; c[1] = cus[k + 1]; c[2] = cvs[k]; c[3] = cvs[k + P];
    const int8_t km = kinds[k];
    c[4] = (km == 1 ? dreg : (km == 2 ? sd[k] * sd[k] : 1.0)) - dreg;
  };
  {
    double c[5];
    if (dense && f.dcache)
      for (int q = 0, l = t; q < nq; ++q, l += NT) {
        coefs(k0 + q * kstep, c);
#pragma unroll
        for (int e = 0; e < 5; ++e) dcoef[e * TXY + l] = c[e];
      }
    else if (f.lcache && q_l >= 0) {
      coefs(g.idx(q_i, q_j), c);
#pragma unroll
      for (int e = 0; e < 5; ++e) lcoef[e * NT + t] = c[e];
    }
  }
  // the general row: w = K~ r from r and its neighbours, and the sums
  auto row = [&](const double (&r)[5], const double (&c)[5], double (&v)[4]) -> double {
    const double wk = r[0] - c[0] * r[1] - c[1] * r[2] - c[2] * r[3] - c[3] * r[4];
    const double r2 = r[0] * r[0];
    v[0] += r2;
    v[1] += c[4] * r2;
    v[2] += wk * r[0];
    return wk;
  };
  // step 2 on own cells: w = K~ r, sums into v
  auto stencil = [&](int parity, unsigned int tag, double (&v)[4]) {
    double r[5], c[5];
    if (dense) {
      for (int q = 0, l = t; q < nq; ++q, l += NT) {
        const int j = j0 + ty0 + q * RP;
        gather(ci, j, r);
        if (f.dcache) {
#pragma unroll
          for (int e = 0; e < 5; ++e) c[e] = dcoef[e * TXY + l];
        } else {
          coefs(k0 + q * kstep, c);
        }
        wput(parity, tag, ci, j, l, row(r, c, v));
      }
      return;
    }
    // the listed cells first: their chains of FP64 operations interleave with the other warps'
    // constant-stencil passes instead of trailing them
    if (q_l >= 0) {
      gather(q_i, q_j, r);
      if (f.lcache) {
#pragma unroll
        for (int e = 0; e < 5; ++e) c[e] = lcoef[e * NT + t];
      } else {
        coefs(g.idx(q_i, q_j), c);
      }
      wput(parity, tag, q_i, q_j, q_l, row(r, c, v));
    }
    for (int q = myq + NT; q < nlist; q += NT) {
      const int l = list[q], i = i0 + l % TX, j = j0 + l / TX;
      gather(i, j, r);
      coefs(g.idx(i, j), c);
      wput(parity, tag, i, j, l, row(r, c, v));
    }
    // constant stencil on every own cell; the listed ones add nothing to the sums and are not
    // stored (selects and predicates: a branch would run the FP64 instructions of both sides)
    const double* z = srn + lp0;
#pragma unroll 2
    for (int q = 0; q < nq; ++q, z += lpstep) {
      const bool listed = (m_list >> q) & 1u;
      const double rc = z[0];
      double wk = rc - ax * (z[-1] + z[1]) - ay * (z[-TXP] + z[TXP]);
      if ((m_in >> q) & 1u) wk = 0.0;
      const double rs = listed ? 0.0 : rc;
      v[0] += rs * rs;
      v[2] += wk * rs;
      if (!listed) {
        sw[t + q * NT] = wk;
        const int jr = ty0 + q * RP;
        if (edge_col || jr == 0 || jr == hj_) push(parity, tag, tx, jr, wk);
      }
    }
  };
  // FP64 sums of the computing threads' values over the block into rows[q * nb + tile] (all threads)
  auto reduce = [&](const double (&v)[4], int nv, double* rows) {
    if (!comm)
      for (int q = 0; q < nv; ++q) sh.red[q][t] = v[q];
    __syncthreads();
    if (wid < nv) {
      double s = 0.0;
#pragma unroll
      for (int m = 0; m < NT / 32; ++m) s += sh.red[wid][lane + 32 * m];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
      if (lane == 0) sh.bsum[wid] = s;
    }
    __syncthreads();
    if (t == 0)
      for (int q = 0; q < nv; ++q) rows[(size_t)q * nb + tile] = sh.bsum[q];
  };
  double* const rows0 = a.partials;              // reductions 0, 2, 4, ...
  double* const rows1 = a.partials + 4 * nb;     // reductions 1, 3, 5, ...

  // Phase 0: x~ = D^1/2 x, r_0 = D^-1/2 (b - K x) into R[0], s_{-1} = p_{-1} = 0.
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  {
    const KRow<double> K{a.cu, a.cv, a.dk, a.kind, a.creg_x, a.creg_y, a.dreg, (size_t)P};
    for (int q = 0; q < nq; ++q) {
      const size_t k = k0 + q * kstep;
      const double bk = a.b[k];
      const bool inactive = kinds[k] == 0;  // identity row: x = b exactly
      const double rk = inactive ? 0.0 : bk - K(a.x, k);
      const double x0 = inactive ? bk : sd[k] * a.x[k], r0 = a.isd[k] * rk;
      const int l = t + q * NT, jr = ty0 + q * RP;
      sx[l] = x0;
      srn[lp0 + q * lpstep] = r0;
      ss[l] = 0.0;
      sp[l] = 0.0;
      if (edge_col || jr == 0 || jr == hj_) f.R[0][k] = r0;  // the neighbours' first ring
      v[3] += bk * bk;
    }
  }
  // the fixed-point words and the mailboxes start at zero (they hold an earlier launch's); the
  // barriers of phase 0 order this before their first use
  if (tile == 0 && t < 2 * kFxWords) f.fxacc[(size_t)t * kFxStride] = 0ULL;
  for (int q = t; q < 2 * nslot; q += NT + 32)
    mailbox(q >= nslot, tile)[q >= nslot ? q - nslot : q] = make_ulonglong2(0ULL, 0ULL);
  bool ok = sync_grid();
  if (ok) {
    // w_0 = K~ r_0: every neighbour's r_0 is complete, read through the same ring path
    if (!comm)
      for (int q = t; q < nring; q += NT) {
        int ri, rj, slot;
        const bool in = ring_cell(q, ri, rj, slot);
        const double rv0 = in ? f.R[0][g.idx(ri, rj)] : 0.0;
        sr[lpad(ri, rj)] = srn[lpad(ri, rj)] = rv0;  // 0 outside the domain, in both frames, for good
        ring[slot] = 0.0;                            // s_{-1}
      }
    __syncthreads();
    stencil(0, 1u, v);
    reduce(v, 4, rows0);
    if (f.zero_mean) {
      double n[4] = {0.0, 0.0, 0.0, 0.0};
      for (int q = 0; q < nq; ++q) {
        const size_t k = k0 + q * kstep;
        if (kinds[k] != 0) n[0] += sd[k] * sd[k];
      }
      reduce(n, 1, rows1);
    }
    ok = sync_grid();
    if (ok && f.zero_mean) {
      double n[1];
      grid_sum<1>(rows1, nb, n, sh.gsum);
      if (t == 0) sh.nn = n[0];
    }
  }
  // The communication warp's state: the recurrence, and its lanes' words after their last use
  // (of the buffer next in turn and of the other).
  CgState st{};
  double thr = 0.0;  // tol^2 ||b||^2
  double alpha = 0.0, beta = 0.0;
  unsigned long long last = 0ULL, last2 = 0ULL;
  int it = 0;
  if (ok) {
    double s[4];
    grid_sum<4>(rows0, nb, s, sh.gsum);
    if (comm) {
      const double rr = dreg * s[0] + s[1];
      const int stop = (s[3] == 0.0 || rr <= a.tol * a.tol * s[3]) ? 1 : (a.max_iter <= 0 ? 2 : 0);
      const Scalar gamma = sc_of_double(s[0]);
      st.igamma = cg_inverse(gamma);
      st.den = sc_of_double(s[2]);
      alpha = sc_double(sc_mul(gamma, sc_recip(st.den)));
      thr = a.tol * a.tol * s[3];
      if (lane == 0) {
        sh.rr = rr;
        sh.bb = s[3];
        sh.stop = stop;
        sh.alpha = alpha;
        sh.beta = 0.0;
        sh.lo = fx_window(s[0], s[1], s[2]);
      }
    }
    __syncthreads();
  }
  // The scalars of the next iteration from the sums of reduction `red` (1, 2, ...), in lane 0 of
  // the communication warp: alpha and beta at once; then, while the other warps are in step 1
  // with them, the stopping test and the window (step 1 leaves x~ alone, so an iteration that
  // turns out to be one too many is dropped after it); 1 / gamma while they are in step 2.
  auto scalars_rest = [&](const Scalar (&s)[3], int red) {
    const double rr = dreg * sc_double(s[0]) + sc_double(s[1]);
    sh.rr = rr;
    sh.stop = rr <= thr ? 1 : (red >= a.max_iter ? 2 : 0);
    sh.lo = max(max(sc_log2(s[0]), sc_log2(s[1])), sc_log2(s[2])) + kFxMargin - kFxTop;
  };
  int cur = 0;
  double my_w = 0.0;  // w_i of this thread's first ring cell
  if (ok && sh.stop == 0 && my_in && !tag_wait(mailbox(0, tile) + my_slot, 1u, my_w, a.bar.budget, a.bar.err))
    sh.fail = 1;  // seen behind the next block barrier
  Scalar sums[3] = {};   // the last reduction's (communication warp)
  long long digit = 0;   // and this lane's digit sum of it
  bool rest = false;     // their stopping test is outstanding
  while (ok) {
    const int nxt = cur ^ 1;
    const int red = it + 1;                         // this iteration's reduction
    const unsigned int tag = (unsigned int)it + 1u; // of w_i
    const double al = sh.alpha, be = sh.beta;
    // every block takes the same branch: the overflow count is the grid's, and the test hook
    // depends on the reduction index only
    const bool forced = (f.fx_fallback_every > 0 && red % f.fx_fallback_every == 0) ||
                        (f.zero_mean != 0 && red % kZeroMeanEvery == 1);
    // the frame that received r_i becomes the current one
    if (defer) {
      double* const q = sr;
      sr = srn;
      srn = q;
    }
    v[0] = v[1] = v[2] = 0.0;
    if (comm) {
      if (rest && lane == 0) scalars_rest(sums, it);
    } else {
      // step 1: own cells
      if (defer) {
#pragma unroll 2
        for (int q = 0, l = t, lp = lp0; q < nq; ++q, l += NT, lp += lpstep) {
          const double sk = sw[l] + be * ss[l];
          ss[l] = sk;
          srn[lp] = sr[lp] - al * sk;
        }
      } else {
        for (int q = 0, l = t, lp = lp0; q < nq; ++q, l += NT, lp += lpstep) {
          const double sk = sw[l] + be * ss[l], pk = sr[lp] + be * sp[l];
          ss[l] = sk;
          sp[l] = pk;
          sr[lp] -= al * sk;
        }
      }
      // ring cells: r_{i+1} from the neighbours' w_i in the mailbox, r and s kept here (cells outside
      // the domain stay 0)
      const ulonglong2* const box = mailbox(cur, tile);
      auto ring_step = [&](int slot, int lp, double wv) {
        const double sk = wv + be * ring[slot];
        ring[slot] = sk;
        srn[lp] = sr[lp] - al * sk;
      };
      if (my_in) ring_step(my_slot, my_lp, my_w);
      for (int q = t + NT; q < nring; q += NT) {
        int ri, rj, slot;
        double wv = 0.0;
        if (!ring_cell(q, ri, rj, slot)) continue;
        if (!tag_wait(box + slot, tag, wv, a.bar.budget, a.bar.err)) sh.fail = 1;
        ring_step(slot, lpad(ri, rj), wv);
      }
    }
    __syncthreads();
    if (sh.stop != 0 || sh.fail) break;
    const int fx_lo = sh.lo;
    if (!comm) {
      stencil(nxt, tag + 1u, v);
      fx_block_digits<NT>(v, fx_lo, sh.fx);
      digits_ready<NT>(false);
      // the neighbours' w_{i+1} arrive about when their digits do: a first look now, its answer
      // used after the update
      ulonglong2* const box = mailbox(nxt, tile) + my_slot;
      bool here = true;
      if (my_in) here = tag_get(box, tag + 1u, my_w);
      // read by no other block and by nothing before the end
      if (defer) {
#pragma unroll 2
        for (int q = 0, l = t, lp = lp0; q < nq; ++q, l += NT, lp += lpstep) {
          const double pk = sr[lp] + be * sp[l];
          sp[l] = pk;
          sx[l] += al * pk;
        }
      } else {
        for (int q = 0, l = t; q < nq; ++q, l += NT) sx[l] += al * sp[l];
      }
      if (!here && !tag_wait(box, tag + 1u, my_w, a.bar.budget, a.bar.err)) sh.late = 1;
    } else {
      // The communication warp: arrive, wait, form the scalars.  Its code between the wait and the
      // barrier is on every block's critical path and runs once per iteration, with cold
      // instruction caches: so it runs twice, first on the previous reduction's digits while the
      // digits of this one are still being formed.
      if (rest && lane == 0) st.igamma = cg_inverse(sums[0]);
      int over = 0;
      bool got = true;
      CgState next = st;
#pragma unroll 1
      for (int pass = 0; pass < 2; ++pass) {
        if (pass == 1) {
          digits_ready<NT>(true);
          fx_arrive<NT, false>(f.fxacc, red & 1, tile == a.bar.absent, sh.fx);
          got = fx_wait<false>(f.fxacc, red & 1, nb, a.bar.budget, a.bar.err, last, digit);
        }
        fx_sums(digit, fx_lo, sums, &over);
        if (lane == 0) {
          next = st;
          cg_scalars(sums[0], sums[2], next, alpha, beta);
          // (pass 0 writes what no one reads before pass 1 has written)
          sh.alpha = alpha;
          sh.beta = beta;
        }
      }
      const unsigned long long q = last;
      last = last2;
      last2 = q;
      rest = got && !forced && over == 0;
      if (rest) st = next;
      if (lane == 0) {
        sh.redo = forced || over != 0;
        if (!got) sh.late = 1;
      }
    }
    __syncthreads();
    if (sh.late) { ok = false; break; }
    if (sh.redo) {
      // a value outside the window (every block sees the same count): this reduction again in
      // FP64 through the partial rows and the counter barrier
      double* const rows = (it & 1) ? rows0 : rows1;
      double d[4];
      if (f.zero_mean) {
        // ... with (n, r), n = D^1/2 1, and r -= n (n, r) / (n, n) on the tile and its ring
        v[3] = 0.0;
        for (int q = 0, lp = lp0; q < nq; ++q, lp += lpstep) v[3] += sd[k0 + q * kstep] * srn[lp];
        reduce(v, 4, rows);
        if (!sync_grid()) { ok = false; break; }
        grid_sum<4>(rows, nb, d, sh.gsum);
        const double c = d[3] / sh.nn;
        for (int q = 0, lp = lp0; q < nq; ++q, lp += lpstep) {
          const size_t k = k0 + q * kstep;
          if (kinds[k] != 0) srn[lp] = fma(-c, sd[k], srn[lp]);
        }
        if (!comm)
          for (int q = t; q < nring; q += NT) {
            int ri, rj, slot;
            if (!ring_cell(q, ri, rj, slot)) continue;
            const size_t k = g.idx(ri, rj);
            if (kinds[k] != 0) srn[lpad(ri, rj)] = fma(-c, sd[k], srn[lpad(ri, rj)]);
          }
        d[0] -= c * d[3];
      } else {
        reduce(v, 3, rows);
        if (!sync_grid()) { ok = false; break; }
        double d3[3];
        grid_sum<3>(rows, nb, d3, sh.gsum);
        d[0] = d3[0]; d[1] = d3[1]; d[2] = d3[2];
      }
      if (comm) {
        if (isfinite(d[0]) && isfinite(d[1]) && isfinite(d[2])) {
#pragma unroll
          for (int q = 0; q < 3; ++q) sums[q] = sc_of_double(d[q]);
          if (lane == 0) {
            cg_scalars(sums[0], sums[2], st, alpha, beta);
            sh.alpha = alpha;
            sh.beta = beta;
          }
          rest = true;
        } else if (lane == 0) {
          // not finite: nothing meets the tolerance any more
          sh.alpha = sh.beta = sh.rr = d[0] + d[1] + d[2];
          sh.stop = red >= a.max_iter ? 2 : 0;
        }
      }
      __syncthreads();
    }
    it = red;
    cur = nxt;
  }
  if (sh.fail) ok = false;  // (left behind step 1)
  // b = 0: the solution is 0, whatever the warm start was
  const bool none = ok && sh.bb == 0.0;
  for (int q = 0; q < nq; ++q) {
    const size_t k = k0 + q * kstep;
    a.x[k] = none ? 0.0 : a.isd[k] * sx[t + q * NT];
  }
  if (tile == 0 && t == 0) {
    const bool conv = ok && sh.stop == 1;
    a.out.iters[0] = ok ? it : 0;
    a.out.rr[0] = ok ? sh.rr : 0.0;
    a.out.bb[0] = ok ? sh.bb : 0.0;
    a.out.converged[0] = conv ? 1 : 0;
    if (a.out.total && ok) a.out.total[0] += it;
    if (!conv && a.out.nconv) a.out.nconv[0] += 1;
  }
}

// __grid_constant__: the body takes the parameter by reference without a local copy.  MINB:
// blocks per SM that must fit.
template <int NT, int MINB>
__global__ void __launch_bounds__(NT + 32, MINB) k_pcg_poisson_f2(const __grid_constant__ FusedSolve f) {
  __shared__ FusedShared<NT> sh;
  fused_body<NT>(f, blockIdx.x, sh);
}

// Many cases in one cooperative launch: block b serves a tile of case block_case[b], whose tiles
// pass barriers and words of their own, so every case iterates at its own pace and its blocks leave
// the launch when it has converged.
template <int NT, int MINB>
__global__ void __launch_bounds__(NT + 32, MINB) k_fused_batch(const FusedBatchEntry* __restrict__ cases,
                                                              const int* __restrict__ block_case) {
  __shared__ FusedShared<NT> sh;
  __shared__ __align__(16) unsigned char s_entry[sizeof(FusedBatchEntry)];
  const FusedBatchEntry& E = stage_entry(cases, block_case, s_entry);
  fused_body<NT>(E.f, (int)blockIdx.x - E.block0, sh);
}

}  // namespace

constexpr size_t kFusedSmemMax = 64 * 1024;  // f1: ring and list of non-uniform cells, per block

namespace {

int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

const void* fused_kernel(int nt, bool two) {
  if (nt == 128) return (const void*)k_pcg_poisson_f2<128, 2>;
  if (nt == 256) return two ? (const void*)k_pcg_poisson_f2<256, 2> : (const void*)k_pcg_poisson_f2<256, 1>;
  return two ? (const void*)k_pcg_poisson_f2<512, 2> : (const void*)k_pcg_poisson_f2<512, 1>;
}

// Shared memory of ntiles resident tiles of TX x TY cells, which must fit the GPU at once: with
// every cell's coefficients cached, with a second r frame (defer) and with the listed cells'
// coefficients cached where they fit too; 0 if nothing fits.
size_t resident_shape(int TX, int TY, int ntiles, FusedSolve* f) {
  const int sms = sm_count(), nt = fused_threads(TX, TY, ntiles, sms);
  if (ntiles < 1 || ntiles > 2 * sms || TX * TY > kFusedRows * nt) return 0;
  const void* kern = fused_kernel(nt, ntiles > sms);
  const size_t room = allow_most_smem(kern);
  for (int k = 7; k >= 0; --k) {
    const bool dc = (k & 4) != 0, df = (k & 2) != 0, lc = (k & 1) != 0;
    const size_t smem = resident_smem(TX, TY, nt, dc, df, lc);
    if (smem > room) continue;
    int per = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, nt + 32, smem) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    if (ntiles > sms * std::min(per, 2)) continue;
    if (f) {
      f->dcache = dc ? 1 : 0;
      f->defer = df ? 1 : 0;
      f->lcache = lc ? 1 : 0;
    }
    return smem;
  }
  return 0;
}

}  // namespace

int fused_blocks() {
  const void* kern = fused_global_kernel(512, true);
  int per = 0;
  allow_most_smem(kern);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, 512, kFusedSmemMax);
  per = per > 2 ? 2 : (per < 1 ? 1 : per);
  return sm_count() * per;
}

bool fused_resident_ok(int TX, int TY, int ntiles) { return resident_shape(TX, TY, ntiles, nullptr) != 0; }

// Batched launch: two blocks of 256 computing threads per SM.  Blocks of different cases share an
// SM, and one's vectors fill the FP64 pipe while the other waits for its reduction.
constexpr int kBatchNT = 256, kBatchPerSM = 2;

int fused_batch_blocks() { return kBatchPerSM * sm_count(); }

namespace {
// dynamic shared memory that each of the blocks of an SM can have
size_t batch_room() {
  int dev = 0, per_sm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  const size_t fixed = sizeof(FusedShared<kBatchNT>) + sizeof(FusedBatchEntry) + 1024 + 256;  // static and reserved
  return (size_t)per_sm / kBatchPerSM > fixed ? (size_t)per_sm / kBatchPerSM - fixed : 0;
}
}  // namespace

size_t fused_batch_cells() { return batch_room() / (5 * sizeof(double) + sizeof(int)) + 1; }

size_t fused_batch_plan(FusedSolve* f, int blocks) {
  f->ntiles = 0;
  fused_tiles(f->a.g.nx, f->a.g.ny, blocks, &f->TX, &f->TY, &f->nbx, &f->ntiles, kResidentCells, kBatchNT);
  if (f->ntiles < 1 || f->ntiles > blocks || f->TX * f->TY > kFusedRows * kBatchNT) return 0;
  if (f->mail_slots < fused_mail_slots(f->a.g.nx, f->TX, f->TY, f->ntiles)) return 0;
  f->resident = 1;
  f->wx = std::min(f->TX, f->a.g.nx);
  f->list_cap = f->TX * f->TY;
  const size_t room = batch_room();
  for (int k = 7; k >= 0; --k) {
    const size_t smem = resident_smem(f->TX, f->TY, kBatchNT, (k & 4) != 0, (k & 2) != 0, (k & 1) != 0);
    if (smem > room) continue;
    f->dcache = (k & 4) != 0;
    f->defer = (k & 2) != 0;
    f->lcache = (k & 1) != 0;
    return smem;
  }
  return 0;
}

cudaError_t run_fused_batch(const FusedBatchEntry* dev_cases, const int* dev_block_case, BatchControl ctl, int blocks,
                            size_t smem, cudaStream_t st) {
  if (!ctl.case_bar || ctl.ncases < 1) return cudaErrorInvalidValue;
  const void* kern = (const void*)k_fused_batch<kBatchNT, kBatchPerSM>;
  if (smem > allow_most_smem(kern)) return cudaErrorInvalidConfiguration;
  cudaMemsetAsync(ctl.case_bar, 0, sizeof(unsigned int) * kCaseBarStride * (size_t)ctl.ncases, st);
  void* params[] = {(void*)&dev_cases, (void*)&dev_block_case};
  return cudaLaunchCooperativeKernel(kern, blocks, kBatchNT + 32, params, smem, st);
}

cudaError_t run_poisson_fused(FusedSolve f, cudaStream_t st) {
  const int blocks = fused_blocks(), sms = sm_count();
  if (f.TX == 0) {
    // the built-in plan: resident tiles, one per SM, where they and their mailboxes fit, else two in
    // global memory
    fused_tiles(f.a.g.nx, f.a.g.ny, sms, &f.TX, &f.TY, &f.nbx, &f.ntiles, kResidentCells, 512,
                f.mail ? f.mail_slots : SIZE_MAX);
    const bool fits = f.mail && resident_shape(f.TX, f.TY, f.ntiles, nullptr) != 0;
    if (!fits && f.resident) return cudaErrorInvalidConfiguration;  // the caller has resident tiles only
    if (!fits) fused_tiles(f.a.g.nx, f.a.g.ny, blocks, &f.TX, &f.TY, &f.nbx, &f.ntiles);
    f.resident = fits ? 1 : 0;
  }
  if (f.ntiles < 1) return cudaErrorInvalidConfiguration;
  const int nt = fused_threads(f.TX, f.TY, f.ntiles, sms);
  const void* kernel = f.resident ? fused_kernel(nt, f.ntiles > sms) : fused_global_kernel(nt, f.zero_mean != 0);
  size_t smem = 0;
  f.wx = std::min(f.TX, f.a.g.nx);
  if (f.resident) {
    // the tile's vectors in shared memory: as many blocks as fit must hold every tile
    smem = resident_shape(f.TX, f.TY, f.ntiles, &f);
    if (smem == 0 || !f.mail || f.mail_slots < fused_mail_slots(f.a.g.nx, f.TX, f.TY, f.ntiles))
      return cudaErrorInvalidConfiguration;
    f.list_cap = f.TX * f.TY;
  } else {
    const size_t ring = sizeof(double) * 2 * ((size_t)f.TX + (size_t)f.TY);
    if (ring + sizeof(int) * 256 > kFusedSmemMax || f.ntiles > blocks) return cudaErrorInvalidConfiguration;
    // the list of non-uniform cells takes what is left, up to one entry per tile cell
    f.list_cap = (int)std::min<size_t>((kFusedSmemMax - ring) / sizeof(int), (size_t)f.TX * (size_t)f.TY);
    smem = ring + sizeof(int) * (size_t)f.list_cap;
    if (smem > allow_most_smem(kernel)) return cudaErrorInvalidConfiguration;
  }
  cudaMemsetAsync(f.a.bar.count, 0, sizeof(unsigned int) * kBarWords, st);
  void* params[] = {&f};
  return cudaLaunchCooperativeKernel(kernel, f.ntiles, f.resident ? nt + 32 : nt, params, smem, st);
}

}  // namespace ccm
