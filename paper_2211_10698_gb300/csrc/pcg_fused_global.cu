// The one-barrier FP64 solve of pcg_fused.cu on tiles whose vectors do not fit shared memory: x~, r, p, s
// and w live in global memory (L2, and beyond about 2 million cells HBM), and each block reads the ring
// around its tile from its neighbours' vectors.
//
// r, w and s are double-buffered by iteration parity: iteration i reads buffer i%2 everywhere and writes
// buffer (i+1)%2 for its own cells, so the ring cells a neighbouring block reads are never the ones being
// written.  Per iteration, in each block:
//   1. own cells: s_i, p_i, x~ += alpha p_i, r_{i+1} (written to the next buffers); ring cells: r_{i+1}
//      into shared memory (zero outside the domain)
//   2. block barrier; own cells: w_{i+1} = K~ r_{i+1} (neighbours inside the tile from the next buffer, on
//      the ring from shared memory) and the sums, in fixed point (pcg_fixed.cuh), added to the words in
//      global memory by the block's first warp; the wait for the grid's words is the grid barrier
//   3. the scalars in integer arithmetic (pcg_scalar.cuh), in three warps: alpha and beta, the stopping
//      test with the window, 1 / gamma.
// The vectors' traffic bounds it (about 96 B per cell and iteration), so the threads' loads in flight count,
// and with them the registers: 512 threads and two blocks per SM leave 64 each.  All of an own cell's vectors
// are read and written once, in step 1.  Measured per iteration on uniform grids, against a form that had the
// communication warp of the resident tiles (56 registers, 678 bytes of spills) and left p and x~ to a second
// pass behind the block's arrival: 1280x640 23.7 -> 22.0 us, 2048x1024 55.5 -> 51.1, 2560x1280 86.7 -> 81.5,
// 3072x1536 120.4 -> 118.9, 4096x2048 203 -> 204.
#include <algorithm>

#include "pcg_common.cuh"
#include "pcg_scalar.cuh"

namespace ccm {

namespace {

template <int NT>
struct GlobalShared {
  double red[4][NT];
  double bsum[8];
  double gsum[8];
  double alpha, beta, rr, bb, thr;  // thr: tol^2 ||b||^2
  double nn;                        // singular systems: sum of d over the active cells
  Scalar sums[3], den, igamma[2];   // the last reduction's sums; the recurrence, 1 / gamma by parity
  unsigned long long last[2][32];   // words of either buffer after their last use, by lane
  int stop, lo, over, got;
  int scan[NT / 32 + 1];
  FxShared<NT> fx;
};

// ZM: singular system
template <bool ZM, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_pcg_poisson_f1(const __grid_constant__ FusedSolve f) {
  __shared__ GlobalShared<NT> sh;
  // dynamic shared memory: the ring's r~ [W: TY][E: TY][S: TX][N: TX], then the list
  extern __shared__ double dyn[];
  unsigned int target = 0;
  const ScaledSolve& a = f.a;
  const int nb = gridDim.x;
  const Geom& g = a.g;
  const int nx = g.nx, ny = g.ny, P = g.pitch;
  const int TX = f.TX, TY = f.TY;
  const int bx = blockIdx.x % f.nbx, by = blockIdx.x / f.nbx;
  const int i0 = bx * TX, j0 = by * TY;
  const int i1 = min(i0 + TX, nx), j1 = min(j0 + TY, ny);
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  const int tx = t % TX, ty0 = t / TX, RP = NT / TX;
  const int ci = i0 + tx;  // this thread's column; its own cells are rows j0 + ty0, + RP, ... of it
  const bool col = ci < i1;
  double* const ring = dyn;
  int* const list = reinterpret_cast<int*>(ring + 2 * (TX + TY));
  // ring cells: W and E columns, then S and N rows, taken by threads t, t + NT, ...
  const int nring = 2 * (j1 - j0) + 2 * (i1 - i0);
  // cell (ri, rj) of ring position q and its slot in `ring`; false outside the domain, where the
  // value is 0
  auto ring_cell = [&](int q, int& ri, int& rj, int& slot) -> bool {
    const int h = j1 - j0, w = i1 - i0;
    if (q < h) { ri = i0 - 1; rj = j0 + q; slot = q; }
    else if ((q -= h) < h) { ri = i1; rj = j0 + q; slot = TY + q; }
    else if ((q -= h) < w) { ri = i0 + q; rj = j0 - 1; slot = 2 * TY + q; }
    else { q -= w; ri = i0 + q; rj = j1; slot = 2 * TY + TX + q; }
    return ri >= 0 && ri < nx && rj >= 0 && rj < ny;
  };
  const int8_t* __restrict__ kinds = a.kinds;
  const double* __restrict__ cus = a.cus;
  const double* __restrict__ cvs = a.cvs;
  const double* __restrict__ sd = a.sd;
  const double ax = a.ax, ay = a.ay, dreg = a.dreg;
  double* __restrict__ xs = a.xs;
  double* __restrict__ p = a.p;

  // r~ at neighbour (i, j) of an own cell after step 1: inside the tile from the next buffer, on the
  // ring from shared memory
  auto rnb = [&](const double* rn, int i, int j) -> double {
    if (i < i0) return ring[j - j0];
    if (i >= i1) return ring[TY + (j - j0)];
    if (j < j0) return ring[2 * TY + (i - i0)];
    if (j >= j1) return ring[2 * TY + TX + (i - i0)];
    return rn[g.idx(i, j)];
  };
  auto gather = [&](const double* rn, int i, int j, double (&r)[5]) {
    r[0] = rn[g.idx(i, j)];
    r[1] = rnb(rn, i - 1, j); r[2] = rnb(rn, i + 1, j); r[3] = rnb(rn, i, j - 1); r[4] = rnb(rn, i, j + 1);
  };
  // coefficients of a listed row: W, E, S, N and sqrt(d)
  auto coefs = [&](size_t k, double (&c)[5]) {
    c[0] = cus[k]; c[1] = cus[k + 1]; c[2] = cvs[k]; c[3] = cvs[k + P]; c[4] = sd[k];
  };
  auto row = [&](const double (&r)[5], const double (&c)[5], double (&v)[4]) -> double {
    const double wk = r[0] - c[0] * r[1] - c[1] * r[2] - c[2] * r[3] - c[3] * r[4];
    const double r2 = r[0] * r[0];
    v[0] += r2;
    v[1] += (c[4] * c[4] - dreg) * r2;
    v[2] += wk * r[0];
    return wk;
  };
  // Rows of kind 2 (cut cells, rows next to a Neumann side) are listed per tile, in a fixed order, and
  // computed by threads chosen for it before the constant stencil of the others; a tile takes the
  // general row for every cell where that is shorter, or where the list does not hold them (pcg_fused.cu
  // says why).  Inactive cells (identity rows, kind 0) get their exact solution x = b in phase 0 and zero
  // in every vector after it.
  int nlist = 0;
  bool dense = false;
  {
    int mine = 0;
    if (col)
      for (int j = j0 + ty0; j < j1; j += RP) mine += kinds[g.idx(ci, j)] == 2;
    // exclusive scan of the counts over the block (thread order)
    int incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) sh.scan[wid] = incl;
    __syncthreads();
    if (t == 0) {
      int acc = 0;
      for (int q = 0; q < NT / 32; ++q) {
        const int c = sh.scan[q];
        sh.scan[q] = acc;
        acc += c;
      }
      sh.scan[NT / 32] = acc;
    }
    __syncthreads();
    nlist = sh.scan[NT / 32];
    const int rows = (j1 - j0 + RP - 1) / RP;
    dense = nlist > f.list_cap || 8 * rows < 6 * rows + 8 * ((nlist + NT - 1) / NT);
    if (!dense && mine > 0) {
      int at = sh.scan[wid] + incl - mine;
      for (int j = j0 + ty0; j < j1; j += RP)
        if (kinds[g.idx(ci, j)] == 2) list[at++] = (j - j0) * TX + tx;
    }
    __syncthreads();
  }
  // listed cell q is computed by thread NT - 1 - q: the last threads have the fewest own rows
  const int myq = NT - 1 - t;
  // step 2 on own cells: w = K~ r, sums into v
  auto stencil = [&](const double* rn, double* wn, double (&v)[4]) {
    if (dense) {
      if (col)
        for (int j = j0 + ty0; j < j1; j += RP) {
          double r[5], c[5];
          const size_t k = g.idx(ci, j);
          gather(rn, ci, j, r);
          coefs(k, c);
          wn[k] = row(r, c, v);
        }
      return;
    }
    // the listed cells' sums come first, as on the resident tiles (both kernels then add the same values
    // in the same order)
    const int q0 = myq < nlist ? list[myq] : -1;
    int li = 0, lj = 0;
    double lr[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, lc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
    if (q0 >= 0) {
      li = i0 + q0 % TX;
      lj = j0 + q0 / TX;
      gather(rn, li, lj, lr);
      coefs(g.idx(li, lj), lc);
    }
    double lw = 0.0;
    if (q0 >= 0) lw = row(lr, lc, v);
    for (int q = myq + NT; q < nlist; q += NT) {
      const int l = list[q], i = i0 + l % TX, j = j0 + l / TX;
      double r[5], c[5];
      gather(rn, i, j, r);
      coefs(g.idx(i, j), c);
      wn[g.idx(i, j)] = row(r, c, v);
    }
    // constant stencil on every own cell but the listed ones, two rows of this thread at a time
    if (col)
      for (int j = j0 + ty0; j < j1; j += 2 * RP) {
        const bool two = j + RP < j1;
        const int jb = two ? j + RP : j;
        const size_t ka = g.idx(ci, j), kb = g.idx(ci, jb);
        const int8_t kma = kinds[ka], kmb = kinds[kb];
        const double rca = rn[ka], rwa = rnb(rn, ci - 1, j), rea = rnb(rn, ci + 1, j);
        const double rsa = rnb(rn, ci, j - 1), rqa = rnb(rn, ci, j + 1);
        const double rcb = rn[kb], rwb = rnb(rn, ci - 1, jb), reb = rnb(rn, ci + 1, jb);
        const double rsb = rnb(rn, ci, jb - 1), rqb = rnb(rn, ci, jb + 1);
        const double wa = kma == 0 ? 0.0 : rca - ax * (rwa + rea) - ay * (rsa + rqa);
        if (kma != 2) {
          wn[ka] = wa;
          v[0] += rca * rca;
          v[2] += wa * rca;
        }
        if (two) {
          const double wb = kmb == 0 ? 0.0 : rcb - ax * (rwb + reb) - ay * (rsb + rqb);
          if (kmb != 2) {
            wn[kb] = wb;
            v[0] += rcb * rcb;
            v[2] += wb * rcb;
          }
        }
      }
    if (q0 >= 0) wn[g.idx(li, lj)] = lw;
  };
  // FP64 sums over the block into rows[q * nb + block], in the order of the resident tiles
  auto reduce = [&](const double (&v)[4], int nv, double* rows) {
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
      for (int q = 0; q < nv; ++q) rows[(size_t)q * nb + blockIdx.x] = sh.bsum[q];
  };
  double* const rows0 = a.partials;           // reductions 0, 2, 4, ...
  double* const rows1 = a.partials + 4 * nb;  // reductions 1, 3, 5, ...

  // Phase 0: x~ = D^1/2 x, r_0 = D^-1/2 (b - K x) into R[0], s_{-1} = p_{-1} = 0.
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  if (col) {
    const KRow<double> K{a.cu, a.cv, a.dk, a.kind, a.creg_x, a.creg_y, a.dreg, (size_t)P};
    for (int j = j0 + ty0; j < j1; j += RP) {
      const size_t k = g.idx(ci, j);
      const double bk = a.b[k];
      const bool inactive = kinds[k] == 0;  // identity row: x = b exactly
      const double rk = inactive ? 0.0 : bk - K(a.x, k);
      xs[k] = inactive ? bk : sd[k] * a.x[k];
      f.R[0][k] = a.isd[k] * rk;
      f.S[0][k] = 0.0;
      p[k] = 0.0;
      v[3] += bk * bk;
    }
  }
  // the fixed-point words start at zero (they hold an earlier launch's); the barriers of phase 0 order
  // this before their first use
  if (blockIdx.x == 0 && t < 2 * kFxWords) f.fxacc[(size_t)t * kFxStride] = 0ULL;
  if (t < 64) sh.last[t >> 5][lane] = 0ULL;
  bool ok = grid_sync(a.bar, target);
  if (ok) {
    // w_0 = K~ r_0: every neighbour's r_0 is complete, read through the same ring path
    for (int q = t; q < nring; q += NT) {
      int ri, rj, slot;
      const bool in = ring_cell(q, ri, rj, slot);
      ring[slot] = in ? f.R[0][g.idx(ri, rj)] : 0.0;
    }
    __syncthreads();
    stencil(f.R[0], f.W[0], v);
    reduce(v, 4, rows0);
    if constexpr (ZM) {
      double n[4] = {0.0, 0.0, 0.0, 0.0};
      if (col)
        for (int j = j0 + ty0; j < j1; j += RP) {
          const size_t k = g.idx(ci, j);
          if (kinds[k] != 0) n[0] += sd[k] * sd[k];
        }
      reduce(n, 1, rows1);
    }
    ok = grid_sync(a.bar, target);
    if constexpr (ZM) {
      double n[1] = {0.0};
      if (ok) grid_sum<1>(rows1, nb, n, sh.gsum);
      if (t == 0) sh.nn = n[0];
    }
  }
  if (ok) {
    double s[4];
    grid_sum<4>(rows0, nb, s, sh.gsum);
    if (t == 0) {
      const Scalar gamma = sc_of_double(s[0]);
      sh.igamma[0] = cg_inverse(gamma);
      sh.den = sc_of_double(s[2]);
      sh.alpha = sc_double(sc_mul(gamma, sc_recip(sh.den)));
      sh.beta = 0.0;
      sh.rr = dreg * s[0] + s[1];
      sh.bb = s[3];
      sh.thr = a.tol * a.tol * s[3];
      sh.stop = (s[3] == 0.0 || sh.rr <= sh.thr) ? 1 : (a.max_iter <= 0 ? 2 : 0);
      sh.lo = fx_window(s[0], s[1], s[2]);
    }
    __syncthreads();
  }
  // The scalars of the next iteration from the sums of reduction `red` in sh.sums (all threads, between
  // block barriers): each of the three chains in a warp of its own.
  auto scalars = [&](int red) {
    if (t == 0) {
      CgState st{sh.igamma[(red & 1) ^ 1], sh.den};
      double alpha = sh.alpha, beta = sh.beta;
      cg_scalars(sh.sums[0], sh.sums[2], st, alpha, beta);
      sh.alpha = alpha;
      sh.beta = beta;
      sh.den = st.den;
    } else if (t == 32) {
      sh.rr = dreg * sc_double(sh.sums[0]) + sc_double(sh.sums[1]);
      sh.stop = sh.rr <= sh.thr ? 1 : (red >= a.max_iter ? 2 : 0);
      sh.lo = max(max(sc_log2(sh.sums[0]), sc_log2(sh.sums[1])), sc_log2(sh.sums[2])) + kFxMargin - kFxTop;
    } else if (t == 64) {
      sh.igamma[red & 1] = cg_inverse(sh.sums[0]);
    }
    __syncthreads();
  };
  int it = 0, cur = 0;
  while (ok && sh.stop == 0) {
    const int nxt = cur ^ 1, red = it + 1;
    const double al = sh.alpha, be = sh.beta;
    const int fx_lo = sh.lo;
    const double* __restrict__ rc_ = f.R[cur];
    const double* __restrict__ wc_ = f.W[cur];
    const double* __restrict__ sc_ = f.S[cur];
    double* __restrict__ rn_ = f.R[nxt];
    double* __restrict__ sn_ = f.S[nxt];
    // this thread's first ring cell: the neighbours' iteration-i values, published before the last
    // grid barrier, are loaded now so the L2 round trip overlaps step 1
    int pf_slot = 0;
    bool pf_in = false;
    double pf_r = 0.0, pf_w = 0.0, pf_s = 0.0;
    if (t < nring) {
      int ri, rj;
      pf_in = ring_cell(t, ri, rj, pf_slot);
      if (pf_in) {
        const size_t k = g.idx(ri, rj);
        pf_r = rc_[k];
        pf_w = wc_[k];
        pf_s = sc_[k];
      }
    }
    // step 1: two rows of this thread at a time with their loads in flight
    if (col)
      for (int j = j0 + ty0; j < j1; j += 2 * RP) {
        const bool two = j + RP < j1;
        const size_t ka = g.idx(ci, j), kb = two ? g.idx(ci, j + RP) : ka;
        const double r0 = rc_[ka], w0 = wc_[ka], s0 = sc_[ka], p0 = p[ka], x0 = xs[ka];
        const double r1 = rc_[kb], w1 = wc_[kb], s1 = sc_[kb], p1 = p[kb], x1 = xs[kb];
        {
          const double sk = w0 + be * s0, pk = r0 + be * p0;
          sn_[ka] = sk;
          p[ka] = pk;
          xs[ka] = x0 + al * pk;
          rn_[ka] = r0 - al * sk;
        }
        if (two) {
          const double sk = w1 + be * s1, pk = r1 + be * p1;
          sn_[kb] = sk;
          p[kb] = pk;
          xs[kb] = x1 + al * pk;
          rn_[kb] = r1 - al * sk;
        }
      }
    // ring cells: r_{i+1} from the neighbours' iteration-i vectors
    if (t < nring) ring[pf_slot] = pf_in ? pf_r - al * (pf_w + be * pf_s) : 0.0;
    for (int q = t + NT; q < nring; q += NT) {
      int ri, rj, slot;
      double rv = 0.0;
      if (ring_cell(q, ri, rj, slot)) {
        const size_t k = g.idx(ri, rj);
        rv = rc_[k] - al * (wc_[k] + be * sc_[k]);
      }
      ring[slot] = rv;
    }
    __syncthreads();
    v[0] = v[1] = v[2] = 0.0;
    stencil(rn_, f.W[nxt], v);
    fx_block_digits<NT>(v, fx_lo, sh.fx);
    __syncthreads();
    if (wid == 0) {
      const int buf = red & 1;
      fx_arrive<NT, true>(f.fxacc, buf, (int)blockIdx.x == a.bar.absent, sh.fx);
      long long digit = 0;
      const bool got = fx_wait<true>(f.fxacc, buf, nb, a.bar.budget, a.bar.err, sh.last[buf][lane], digit);
      Scalar s[3];
      int over = 0;
      fx_sums(digit, fx_lo, s, &over);
      if (lane == 0) {
#pragma unroll
        for (int q = 0; q < 3; ++q) sh.sums[q] = s[q];
        sh.over = over;
        sh.got = got;
      }
    }
    __syncthreads();
    if (!sh.got) { ok = false; break; }
    // every block takes the same branch: the overflow count is the grid's, and the test hook depends on
    // the reduction index only
    bool finite = true;
    if (sh.over != 0 || (f.fx_fallback_every > 0 && red % f.fx_fallback_every == 0) ||
        (ZM && red % kZeroMeanEvery == 1)) {
      // a value outside the window: this reduction again in FP64 through the partial rows and the
      // counter barrier
      double* const rows = (it & 1) ? rows0 : rows1;
      double d[4];
      if constexpr (ZM) {
        // ... with (n, r), n = D^1/2 1, and r -= n (n, r) / (n, n), which the neighbours' rings read next
        v[3] = 0.0;
        if (col)
          for (int j = j0 + ty0; j < j1; j += RP) v[3] += sd[g.idx(ci, j)] * rn_[g.idx(ci, j)];
        reduce(v, 4, rows);
        if (!grid_sync(a.bar, target)) { ok = false; break; }
        grid_sum<4>(rows, nb, d, sh.gsum);
        const double c = d[3] / sh.nn;
        if (col)
          for (int j = j0 + ty0; j < j1; j += RP) {
            const size_t k = g.idx(ci, j);
            if (kinds[k] != 0) rn_[k] = fma(-c, sd[k], rn_[k]);
          }
        if (!grid_sync(a.bar, target)) { ok = false; break; }
        d[0] -= c * d[3];
      } else {
        reduce(v, 3, rows);
        if (!grid_sync(a.bar, target)) { ok = false; break; }
        double d3[3];
        grid_sum<3>(rows, nb, d3, sh.gsum);
        d[0] = d3[0]; d[1] = d3[1]; d[2] = d3[2];
      }
      finite = isfinite(d[0]) && isfinite(d[1]) && isfinite(d[2]);
      if (t == 0) {
        if (finite) {
#pragma unroll
          for (int q = 0; q < 3; ++q) sh.sums[q] = sc_of_double(d[q]);
        } else {
          // nothing meets the tolerance any more
          sh.alpha = sh.beta = sh.rr = d[0] + d[1] + d[2];
          sh.stop = red >= a.max_iter ? 2 : 0;
        }
      }
      __syncthreads();
    }
    if (finite) scalars(red);
    it = red;
    cur = nxt;
  }
  // b = 0: the solution is 0, whatever the warm start was
  const bool none = ok && sh.bb == 0.0;
  if (col)
    for (int j = j0 + ty0; j < j1; j += RP) {
      const size_t k = g.idx(ci, j);
      a.x[k] = none ? 0.0 : a.isd[k] * xs[k];
    }
  if (blockIdx.x == 0 && t == 0) {
    const bool conv = ok && sh.stop == 1;
    a.out.iters[0] = ok ? it : 0;
    a.out.rr[0] = ok ? sh.rr : 0.0;
    a.out.bb[0] = ok ? sh.bb : 0.0;
    a.out.converged[0] = conv ? 1 : 0;
    if (a.out.total && ok) a.out.total[0] += it;
    if (!conv && a.out.nconv) a.out.nconv[0] += 1;
  }
}

}  // namespace

const void* fused_global_kernel(int nt, bool zero_mean) {
  if (zero_mean)
    return nt == 128 ? (const void*)k_pcg_poisson_f1<true, 128, 2>
                     : nt == 256 ? (const void*)k_pcg_poisson_f1<true, 256, 2> : (const void*)k_pcg_poisson_f1<true, 512, 2>;
  return nt == 128 ? (const void*)k_pcg_poisson_f1<false, 128, 2>
                   : nt == 256 ? (const void*)k_pcg_poisson_f1<false, 256, 2> : (const void*)k_pcg_poisson_f1<false, 512, 2>;
}

}  // namespace ccm
