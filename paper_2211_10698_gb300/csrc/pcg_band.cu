// Mixed-precision pressure Poisson solve (Eq. pm_poisson) on resident tiles with their band: the
// reliable-update CG of pcg_mixed.cu (FP32 single-reduction CG on the Jacobi-scaled correction
// equation, Jacobi or Chebyshev preconditioner of degree k, FP64 residual replacements) with one
// reduction per FP32 iteration and nothing of the solve in global memory but what neighbours
// exchange.
//
// Each block owns a tile of W x TY cells (W a multiple of 4) and a band around it: h = k rows (1
// for Jacobi), and h columns rounded up to whole quads.
// In shared memory lie the residual r and two Chebyshev iterates on the region (tile and band), in
// rows of 128 floats; in registers the direction's K~ p (s) on the region and the direction p on
// the tile (in global memory but around its update where a warp has many rows); the correction e,
// which no one else reads, in global memory.  One iteration:
//   1. region: s = w + beta s, r -= alpha s; tile: p = u + beta p.  The band's r and s
//      are kept here, updated with the same recurrences as their owner's, so only w = K~ u comes
//      from the neighbours.
//   2. the k - 1 Chebyshev steps on a region that shrinks by one cell per step, in shared memory:
//      z2 from r alone (z1 = r / theta is not stored), then two buffers in turn; u = M^-1 r is
//      exact on the tile and its one-cell ring.
//   3. tile: w = K~ u and the sums (r, u), (w, u), (r, r); the frame (cells within h of the tile's
//      edge) goes to global memory, value and number of the apply in one 64-bit word, which the
//      neighbours poll: no fence, no wait for outstanding stores.
//   4. the communication warp adds the warps' sums, posts them with the reduction's number in one
//      16-byte slot, polls every block's slot, adds them in a fixed order and forms alpha and beta;
//      meanwhile the other warps update e += alpha p and fetch the band's w.
// A warp owns RS consecutive rows of the region and a lane one quad of each, so a row's west and
// east neighbours come by shuffles, a stencil reads each row of a strip once, every access to
// shared memory is 16 bytes wide, and a lane's own quads of r, w, s, p need no barrier.  Cells
// outside the domain have coefficients 0 and hold 0 in every vector; a row of inner quads takes the
// constant stencil, any other the coefficients that each quad has in a slot of shared memory,
// without divergence (with a branch per cell in the rows of a Neumann side the two columns of tiles
// at the sides took 1.5 times the others' time, and every block waits for the slowest).
//
// A replacement (FP64 residual, rare) folds e into x, forms D^-1/2 (b - K x) in FP64 with its norms
// (one grid barrier), and restarts r from it, band included; then the preconditioner, the formed
// direction and its curvature, as in pcg_mixed.cu.  It is a function of its own between segments of
// iterations: inlined into their loop, its FP64 temporaries made the loop's registers spill (24 local
// loads and stores per warp and iteration; 13.3 us per iteration at 1024x512 with k = 3 instead of 6.7).
//
// What bounds it: the chain of one iteration, k + 1 block barriers, one L2 hop between SMs (907
// cycles measured) and the scalars; on large tiles the instructions of the k + 1 passes.  Measured per
// iteration against the best plan of pcg_mixed.cu and pcg_mixed1.cu: 1024x512, k = 3: 10.8 -> 7.4 us;
// 2048x1024, k = 3: about 28 -> 16.4 us; 701x333, Jacobi: 4.9 -> 4.1 us.
#include <algorithm>

#include "batch_common.cuh"
#include "pcg_cheb.cuh"
#include "pcg_quad.cuh"

namespace ccm {

namespace {

constexpr int kRow = 128;  // floats per region row: one quad per lane

template <int NW>
struct __align__(16) BandShared {
  double params[sizeof(BandSolve) / sizeof(double)];  // the kernel's parameter, for the functions that are called
  __device__ const BandSolve& solve() const { return *reinterpret_cast<const BandSolve*>(params); }
  float4 ctl;     // alpha, beta, flow (as bits), unused
  float4 ws[NW];  // the warps' sums
  double dred[3][NW + 1];
  double dsum[8];
  double sigma, rescale, rr, bb;
  int stop, fail, ncut;
};
constexpr int kReplace = 1, kKeep = 2, kLimit = 4, kFail = 8;

// The same value, of which the compiler keeps nothing derived from phase to phase: addresses and
// predicates of every row of a warp, kept over the iterations, would not fit the registers.
template <class T>
__device__ __forceinline__ T anew(T v) {
  asm volatile("" : "+r"(v));
  return v;
}

// A frame word: a value and the number of the apply it belongs to, written and read as one 64-bit
// access.  Words are indexed (j + 1) pitch + i, so that the quads of a tile are 32-byte aligned.
__device__ __forceinline__ unsigned long long word_of(float v, unsigned int tag) {
  return ((unsigned long long)tag << 32) | __float_as_uint(v);
}
__device__ __forceinline__ void slot_put(ulonglong2* p, float a, float b, float c, unsigned int tag) {
  const unsigned long long lo = ((unsigned long long)__float_as_uint(b) << 32) | __float_as_uint(a);
  const unsigned long long hi = ((unsigned long long)tag << 32) | __float_as_uint(c);
  const unsigned __int128 w = ((unsigned __int128)hi << 64) | lo;
  asm volatile("st.relaxed.gpu.global.b128 [%0], %1;" ::"l"(p), "q"(w) : "memory");
}
__device__ __forceinline__ bool slot_get(const ulonglong2* p, unsigned int tag, float& a, float& b, float& c) {
  unsigned __int128 w;
  asm volatile("ld.relaxed.gpu.global.b128 %0, [%1];" : "=q"(w) : "l"(p) : "memory");
  const unsigned long long lo = (unsigned long long)w, hi = (unsigned long long)(w >> 64);
  a = __uint_as_float((unsigned int)lo);
  b = __uint_as_float((unsigned int)(lo >> 32));
  c = __uint_as_float((unsigned int)hi);
  return (unsigned int)(hi >> 32) == tag;
}

// One tile and its place in shared memory: r and the iterates A and B (B only if cheb > 1), then per
// region row 32 slot numbers of its quads, then f.ncut slots of 16 coefficients (W, E, S and N faces
// of the four cells): 0 an inner quad's, 1 those of a quad outside the domain, the others of quads
// with cut cells.  A row of
// the strip loads may lie before the first or after the last row of a buffer: a guard row in front,
// and what follows the buffers behind.
struct BandTile {
  int i0, j0, Wt, Ht, h, hp, rows, live;  // live: lanes below it hold quads of the tile or its band
  int oR, oA, oB, oI, oCut;               // offsets in floats
  __device__ BandTile(const BandSolve& f, int tile) {
    const Geom& g = f.m.d.g;
    const int cheb = f.m.cheb > 1 ? f.m.cheb : 1;
    const int by = tile / f.nbx;
    h = cheb;
    hp = (h + 3) & ~3;
    i0 = (tile - by * f.nbx) * f.W;
    j0 = by * f.TY;
    Wt = min(f.W, g.nx - i0);
    Ht = min(f.TY, g.ny - j0);
    rows = Ht + 2 * h;
    live = (((Wt + 3) & ~3) + 2 * hp) / 4;
    const int all = f.TY + 2 * h, buf = all * kRow;
    oR = kRow;
    oA = oR + buf;
    oB = oA + buf;
    oI = oR + (cheb > 1 ? 3 : 2) * buf;
    oCut = oI + all * 16;
  }
};

// frame words, p and e: the quad of cells i .. i + 3 (i a multiple of 4) of row j starts at word i of a
// row of pitch >= nx + 3 words, 32-byte aligned; a last quad that reaches beyond nx stays in its row
__device__ __forceinline__ int word(const Geom& g, int i, int j) { return (j + 1) * g.pitch + i; }

// The row kind of cell k of the FP32 system: 0 identity, 1 the constant stencil, 2 its own coefficients.
// A row marked cut for the rounding of its FP64 coefficients alone (on a grid whose spacing is no
// dyadic fraction most are) has the constants in FP32, and so takes the constant stencil here.
__device__ __forceinline__ int kind32(const MixedSolve& a, size_t k, int P, float ax, float ay) {
  const int km = a.d.kinds[k];
  return km == 2 && a.cus32[k] == ax && a.cus32[k + 1] == ax && a.cvs32[k] == ay && a.cvs32[k + P] == ay ? 1 : km;
}

// Zeroes the tile's vectors, classifies its quads and copies the coefficients of those with cut cells
// (all threads).
template <int NW>
__device__ __noinline__ void band_init(const int tile, BandShared<NW>& sh) {
  const BandSolve& f = sh.solve();
  extern __shared__ __align__(16) float bdyn[];
  const MixedSolve& a = f.m;
  const Geom& g = a.d.g;
  const BandTile T(f, tile);
  const int t = threadIdx.x, nt = blockDim.x, P = g.pitch;
  const float ax = (float)a.d.ax, ay = (float)a.d.ay;
  unsigned short* const cidx = reinterpret_cast<unsigned short*>(bdyn + T.oI);
  const float4 z4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  for (int q = t; q < T.oI / 4; q += nt) reinterpret_cast<float4*>(bdyn)[q] = z4;
  if (t == 0) {
    sh.ctl = z4;
    sh.sigma = sh.rescale = sh.rr = sh.bb = 0.0;
    sh.stop = sh.fail = 0;
    sh.ncut = 2;
  }
  if (t < 32) bdyn[T.oCut + t] = t < 8 ? ax : t < 16 ? ay : 0.0f;
  __syncthreads();
  for (int q = t; q < T.rows * 32; q += nt) {
    const int ry = q >> 5, c = 4 * (q & 31) - T.hp, j = T.j0 - T.h + ry;
    const bool in = (q & 31) < T.live && j >= 0 && j < g.ny;
    const size_t k = g.idx(T.i0 + c, j);
    int km[4];
    int b = 0;
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int i = T.i0 + c + m;
      km[m] = in && i >= 0 && i < g.nx ? kind32(a, k + m, P, ax, ay) : 0;
      b |= (km[m] == 1 ? 1 : km[m] == 2 ? 16 : 0) << m;
    }
    // the quad's coefficients: slot 0 of inner cells, 1 of cells outside the domain, or one of its own:
    // W, E, S and N face of every cell, 0 for a cell outside
    int slot = b == 15 ? 0 : b == 0 ? 1 : atomicAdd(&sh.ncut, 1);
    if (slot >= f.ncut) slot = 0xffff;
    cidx[q] = (unsigned short)slot;
    if (b != 15 && b != 0 && slot != 0xffff) {
      float* const cf = bdyn + T.oCut + 16 * slot;
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        cf[m] = km[m] == 2 ? a.cus32[k + m] : km[m] == 1 ? ax : 0.0f;
        cf[4 + m] = km[m] == 2 ? a.cus32[k + m + 1] : km[m] == 1 ? ax : 0.0f;
        cf[8 + m] = km[m] == 2 ? a.cvs32[k + m] : km[m] == 1 ? ay : 0.0f;
        cf[12 + m] = km[m] == 2 ? a.cvs32[k + m + P] : km[m] == 1 ? ay : 0.0f;
      }
    }
  }
  const int W4 = (T.Wt + 3) & ~3;
  for (int q = t; q < T.Ht * kRow; q += nt) {
    const int jr = q / kRow, c = q % kRow;
    if (c >= W4) continue;
    const int k = word(g, T.i0 + c, T.j0 + jr);
    if (jr < T.h || jr >= T.Ht - T.h || c < T.hp || c >= W4 - T.hp) f.WT[0][k] = f.WT[1][k] = 0ULL;
    f.E[k] = 0.0f;
  }
  if (t < 2) f.part[(size_t)t * f.ntiles + tile] = make_ulonglong2(0ULL, 0ULL);
  __syncthreads();
}

// A start from the FP64 residual (all threads): x += D^-1/2 e / sigma and e = 0 on the tile (not the
// first time), r64 = D^-1/2 (b - K x) with its norm, that of b - K x and (the first time) b's, the new
// normalisation and the stopping test, r = sigma r64 on the region.  0: go on, 1: a barrier timed
// out, 2: stop (converged, or `last`).
template <int NW>
__device__ __noinline__ int band_restart(const int tile, BandShared<NW>& sh, const bool first, const bool last,
                                         unsigned int target) {
  const BandSolve& f = sh.solve();
  extern __shared__ __align__(16) float bdyn[];
  const ScaledSolve& d = f.m.d;
  const Geom& g = d.g;
  const BandTile T(f, tile);
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5, P = g.pitch, nb = f.ntiles;
  constexpr int NC = kRow / 32;  // cells of a row per lane, 32 apart
  if (!first) {
    const double isig = 1.0 / sh.sigma;
    for (int jr = wid; jr < T.Ht; jr += NW + 1) {
      const size_t k = g.idx(T.i0, T.j0 + jr);
      float* const e = f.E + word(g, T.i0, T.j0 + jr);
      float ev[NC];
      double x[NC], is[NC];
#pragma unroll
      for (int m = 0; m < NC; ++m) {
        const int c = lane + 32 * m;
        if (c < T.Wt) ev[m] = e[c], x[m] = d.x[k + c], is[m] = d.isd[k + c];
      }
#pragma unroll
      for (int m = 0; m < NC; ++m) {
        const int c = lane + 32 * m;
        if (c < T.Wt) d.x[k + c] = x[m] + is[m] * (double)ev[m] * isig, e[c] = 0.0f;
      }
    }
    if (!range_sync(d.bar, d.bar.count, (unsigned int)nb, target)) return 1;
  }
  const KRow<double> K{d.cu, d.cv, d.dk, d.kind, d.creg_x, d.creg_y, d.dreg, (size_t)P};
  double v[3] = {0.0, 0.0, 0.0};
  for (int jr = wid; jr < T.Ht; jr += NW + 1) {
    const size_t k0 = g.idx(T.i0, T.j0 + jr) + lane;
    double bk[NC], xc[NC], xw[NC], xe[NC], xs[NC], xn[NC], is[NC];
    int8_t km[NC];
#pragma unroll
    for (int m = 0; m < NC; ++m)
      if (lane + 32 * m < T.Wt) {
        const size_t k = k0 + 32 * m;
        bk[m] = d.b[k], is[m] = d.isd[k], km[m] = d.kind[k];
        xc[m] = __ldcg(&d.x[k]), xw[m] = __ldcg(&d.x[k - 1]), xe[m] = __ldcg(&d.x[k + 1]);
        xs[m] = __ldcg(&d.x[k - P]), xn[m] = __ldcg(&d.x[k + P]);
      }
#pragma unroll
    for (int m = 0; m < NC; ++m)
      if (lane + 32 * m < T.Wt) {
        const size_t k = k0 + 32 * m;
        double kx = xc[m];
        if (km[m] == 1) kx = K.dreg * xc[m] - K.cx * (xw[m] + xe[m]) - K.cy * (xs[m] + xn[m]);
        else if (km[m] == 2)
          kx = K.dk[k] * xc[m] - K.cu[k] * xw[m] - K.cu[k + 1] * xe[m] - K.cv[k] * xs[m] - K.cv[k + P] * xn[m];
        const double rk = bk[m] - kx, rs = is[m] * rk;
        d.r[k] = rs;
        v[0] += rs * rs;
        v[1] += rk * rk;
        if (first) v[2] += bk[m] * bk[m];
      }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
  if (lane == 0)
    for (int k = 0; k < 3; ++k) sh.dred[k][wid] = v[k];
  __syncthreads();
  if (t < 3) {
    double q = 0.0;
    for (int w = 0; w <= NW; ++w) q += sh.dred[t][w];
    d.partials[(size_t)t * nb + tile] = q;
  }
  if (!range_sync(d.bar, d.bar.count, (unsigned int)nb, target)) return 1;
  double r[3];
  grid_sum<3>(d.partials, nb, r, sh.dsum);
  if (t == 0) {
    if (first) sh.bb = r[2];
    sh.rr = r[1];
    const double old = sh.sigma;
    sh.sigma = r[0] > 0.0 ? 1.0 / sqrt(r[0]) : 1.0;
    sh.rescale = old > 0.0 ? sh.sigma / old : 0.0;
    if (sh.bb == 0.0 || sh.rr <= d.tol * d.tol * sh.bb) sh.stop = 1;
  }
  __syncthreads();
  // b = 0: x = 0, whatever the warm start was (every block has read x before the barrier above)
  if (sh.bb == 0.0)
    for (int q = t; q < T.Ht * kRow; q += (NW + 1) * 32)
      if (q % kRow < T.Wt) d.x[g.idx(T.i0 + q % kRow, T.j0 + q / kRow)] = 0.0;
  if (sh.stop != 0 || last) return 2;
  const double sig = sh.sigma;
  for (int ry = wid; ry < T.rows; ry += NW + 1) {
    const int j = T.j0 - T.h + ry;
    if (j < 0 || j >= g.ny) continue;
    const double* const r64 = d.r + g.idx(T.i0 - T.hp, j);
    double rv[NC];
#pragma unroll
    for (int m = 0; m < NC; ++m) {
      const int c = lane + 32 * m, i = T.i0 - T.hp + c;
      rv[m] = c < 4 * T.live && i >= 0 && i < g.nx ? __ldcg(&r64[c]) : 0.0;
    }
#pragma unroll
    for (int m = 0; m < NC; ++m) bdyn[T.oR + ry * kRow + lane + 32 * m] = (float)(sig * rv[m]);
  }
  __syncthreads();
  return 0;
}

// The computing warps' part of one segment: the start on the residual that band_restart left in shared
// memory, then iterations up to the next replacement (0), a failure (1) or the iteration limit (2).
// p and s live in registers here; between segments s is in the buffer A and p in global memory, so
// that the registers of the iterations and those of the restart are not live at once.
template <int NW, int RS>
__device__ __forceinline__ int band_segment(const BandSolve& f, const int tile, BandShared<NW>& sh, const bool first,
                                            unsigned int& tag) {
  constexpr int NT = NW * 32;
  extern __shared__ __align__(16) float bdyn[];
  // few rows: r and w of this lane's quads stay in registers (r in shared memory as well)
  constexpr bool REG = RS <= (NW <= 15 ? 2 : 1);
  // many rows: p is in global memory but from the wait for the sums to the update after it
  constexpr bool PG = RS > 2;
  const Geom& g = f.m.d.g;
  const BandTile T(f, tile);
  const int cheb = f.m.cheb > 1 ? f.m.cheb : 1;
  const int lane = threadIdx.x & 31, r0 = (threadIdx.x >> 5) * RS;  // the warp's first region row
  const int col = 4 * lane - T.hp;                                  // tile column of the lane's first cell
  // u = M^-1 r after the steps, and the buffer that then receives w
  const int oR = T.oR, oA = T.oA, oB = T.oB;
  const int oU = cheb == 1 ? oR : ((cheb & 1) ? oB : oA), oW = cheb == 1 ? oA : ((cheb & 1) ? oA : oB);
  const float ax = (float)f.m.d.ax, ay = (float)f.m.d.ay;
  constexpr float ith = (float)(1.0 / ChebCoef::theta);
  auto compute_sync = [&]() {
    __syncwarp();
    asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
  };
  // bits of the warp's rows [lo, hi) of the region
  auto bits = [&](int lo, int hi) -> unsigned int {
    lo = min(max(lo - r0, 0), RS);
    hi = min(max(hi - r0, 0), RS);
    return ((1u << hi) - 1u) & ~((1u << lo) - 1u);
  };
  const unsigned int rows_in = bits(max(0, T.h - T.j0), min(T.rows, g.ny - T.j0 + T.h));  // in the domain
  const unsigned int rows_own = bits(T.h, T.h + T.Ht);
  const bool sends = tile != f.m.d.bar.silent;
  const unsigned int rows_frame = sends ? rows_own & ~bits(2 * T.h, T.Ht) : 0u;
  const bool live = lane < T.live, own = col >= 0 && col < T.Wt;
  const bool frame_col = sends && (col < T.hp || col + 3 >= T.Wt - T.hp);
  const bool in_col = live && T.i0 + col >= 0 && T.i0 + col < g.nx;
  const int woff = word(g, T.i0 + col, T.j0 - T.h + r0);

  // The warp's rows (bits): plain, whose live quads are inner cells throughout (what the lanes beyond
  // the band compute then no needed cell reads), and slots, all of whose quads have theirs in shared memory.
  const unsigned short* const cidx = reinterpret_cast<const unsigned short*>(bdyn + T.oI) + r0 * 32 + lane;
  unsigned int plain = 0, slots = 0;
#pragma unroll
  for (int q = 0; q < RS; ++q) {
    const int slot = r0 + q < T.rows ? cidx[q * 32] : 1;
    if (__all_sync(0xffffffffu, slot == 0 || !live)) plain |= 1u << q;
    if (__all_sync(0xffffffffu, slot != 0xffff)) slots |= 1u << q;
  }

  // K~ z on this lane's quad of the warp's row q, with the rows south and north of it: the constant
  // stencil, and the one with coefficients
  auto krow_plain = [&](const float4& c, const float4& so, const float4& no) -> float4 {
    const float l = __shfl_up_sync(0xffffffffu, c.w, 1), r = __shfl_down_sync(0xffffffffu, c.x, 1);
    return make_float4(c.x - ax * (l + c.y) - ay * (so.x + no.x), c.y - ax * (c.x + c.z) - ay * (so.y + no.y),
                       c.z - ax * (c.y + c.w) - ay * (so.z + no.z), c.w - ax * (c.z + r) - ay * (so.w + no.w));
  };
  auto krow = [&](const float4& c, const float4& so, const float4& no, int q, unsigned int plainq) -> float4 {
    if ((plainq >> q) & 1u) return krow_plain(c, so, no);
    const float l = __shfl_up_sync(0xffffffffu, c.w, 1), r = __shfl_down_sync(0xffffffffu, c.x, 1);
    const int slot = cidx[q * 32];
    float4 cw, ce, cs, cn;
    if ((slots >> q) & 1u) {
      const float4* const cf = reinterpret_cast<const float4*>(bdyn + T.oCut + 16 * slot);
      cw = cf[0], ce = cf[1], cs = cf[2], cn = cf[3];
    } else if (slot != 0xffff) {
      const float4* const cf = reinterpret_cast<const float4*>(bdyn + T.oCut + 16 * slot);
      cw = cf[0], ce = cf[1], cs = cf[2], cn = cf[3];
    } else {
      const size_t k = (size_t)anew(woff) + q * g.pitch + 1;  // idx of the quad's first cell
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int km = T.i0 + col + m < g.nx ? kind32(f.m, k + m, g.pitch, ax, ay) : 0;
        put(cw, m, km == 2 ? f.m.cus32[k + m] : km == 1 ? ax : 0.0f);
        put(ce, m, km == 2 ? f.m.cus32[k + m + 1] : km == 1 ? ax : 0.0f);
        put(cs, m, km == 2 ? f.m.cvs32[k + m] : km == 1 ? ay : 0.0f);
        put(cn, m, km == 2 ? f.m.cvs32[k + m + g.pitch] : km == 1 ? ay : 0.0f);
      }
    }
    return make_float4(c.x - cw.x * l - ce.x * c.y - cs.x * so.x - cn.x * no.x,
                       c.y - cw.y * c.x - ce.y * c.z - cs.y * so.y - cn.y * no.y,
                       c.z - cw.z * c.y - ce.z * c.w - cs.z * so.z - cn.z * no.z,
                       c.w - cw.w * c.z - ce.w * r - cs.w * so.w - cn.w * no.w);
  };
  // this lane's quad of the warp's row q in the buffer at offset o
  float* const mine = bdyn + r0 * kRow + 4 * lane;
  auto ld = [&](int o, int q) -> float4 { return *reinterpret_cast<const float4*>(mine + o + q * kRow); };
  auto st = [&](int o, int q, const float4& v) { *reinterpret_cast<float4*>(mine + o + q * kRow) = v; };
  // many rows: no more loads in flight than the registers beside s hold
  auto row_end = [&]() {
    if (RS > 2) asm volatile("" ::: "memory");
  };
  // fn(q, K~ z, z) for the rows of `mask`: a window of three rows moves up, the next one in flight
  auto rows = [&](int z, unsigned int mask_, auto&& fn) {
    if (mask_ == 0) return;
    const unsigned int mask = anew(mask_), plainq = anew(plain);
    if (RS <= 2 && (mask & plainq) == (1u << RS) - 1u) {
      // without a branch between the rows
      float4 c[RS + 2];
#pragma unroll
      for (int q = 0; q < RS + 2; ++q) c[q] = ld(z, q - 1);
#pragma unroll
      for (int q = 0; q < RS; ++q) fn(q, krow_plain(c[q + 1], c[q], c[q + 2]), c[q + 1]);
      return;
    }
    float4 c0 = ld(z, -1), c1 = ld(z, 0), c2 = ld(z, 1);
#pragma unroll
    for (int q = 0; q < RS; ++q) {
      float4 c3 = c2;
      if (q + 1 < RS) c3 = ld(z, q + 2);
      if ((mask >> q) & 1u) fn(q, krow(c1, c0, c2, q, plainq), c1);
      c0 = c1;
      c1 = c2;
      c2 = c3;
      row_end();
    }
  };

  const float4 z4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  float4 s[RS], p[RS], rq[REG ? RS : 1], wq[REG ? RS : 1];
#pragma unroll
  for (int q = 0; q < RS; ++q) {
    const bool mine_p = own && ((rows_own >> q) & 1u);
    s[q] = !first && ((rows_in >> q) & 1u) ? ld(oA, q) : z4;
    if (!PG) p[q] = !first && mine_p ? *reinterpret_cast<const float4*>(f.m.p + (woff + q * g.pitch)) : z4;
    else if (first && mine_p) *reinterpret_cast<float4*>(f.m.p + (woff + q * g.pitch)) = z4;
    if (REG) {
      rq[REG ? q : 0] = (rows_in >> q) & 1u ? ld(oR, q) : z4;
      wq[REG ? q : 0] = z4;
    }
  }

  // this warp's sums v to the communication warp
  auto post_sums = [&](const float v0, const float v1, const float v2) {
    // v0 in lanes below 16 and v1 above, then v2 in lanes with bit 3
    float x = (lane & 16) ? v1 : v0, y = v2;
    x += __shfl_xor_sync(0xffffffffu, (lane & 16) ? v0 : v1, 16);
    y += __shfl_xor_sync(0xffffffffu, y, 16);
    const float z = __shfl_xor_sync(0xffffffffu, (lane & 8) ? x : y, 8);
    x = ((lane & 8) ? y : x) + z;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((lane & 7) == 0 && lane != 24) reinterpret_cast<float*>(&sh.ws[threadIdx.x >> 5])[lane == 0 ? 0 : lane == 16 ? 1 : 2] = x;
    __syncwarp();
    asm volatile("bar.arrive 2, %0;" ::"n"(NT + 32) : "memory");
  };

  bool fresh = true;
  float4 ct = z4;
  int end = 0;
#pragma unroll 1
  while (true) {
    if (!fresh) {
      // region: s = w + beta s, r -= alpha s; tile: p = u + beta p (s and p may be formed already)
      const float al = ct.x, be = ct.y;
      const bool keep = (__float_as_int(ct.z) & kKeep) != 0;
      if (live) {
        const unsigned int in = anew(rows_in), mo = anew(rows_own);
        const int wo = anew(woff);
#pragma unroll
        for (int q = 0; q < RS; ++q) {
          if (!((in >> q) & 1u)) continue;
          if (!keep) {
            if ((mo >> q) & 1u) {
              p[q] = axpy4(be, p[q], ld(oU, q));
              if (PG && own) *reinterpret_cast<float4*>(f.m.p + (wo + q * g.pitch)) = p[q];
            }
            s[q] = axpy4(be, s[q], REG ? wq[REG ? q : 0] : ld(oW, q));
          }
          const float4 v = axpy4(-al, s[q], REG ? rq[REG ? q : 0] : ld(oR, q));
          if (REG) rq[REG ? q : 0] = v;
          st(oR, q, v);
          row_end();
        }
      }
      compute_sync();
    }
    // Chebyshev steps on a region that shrinks by a cell per step
#pragma unroll 1
    for (int js = 1; js < cheb; ++js) {
      float c1, c2;
      cheb_step_coef(js, c1, c2);
      const unsigned int mask = bits(js, T.rows - js);
      if (js == 1) {
        // z1 = r / theta; z2 = z1 + c1 z1 + c2 (r - K~ z1)
        const float g1 = ith + c1 * ith + c2, g2 = -c2 * ith;
        rows(oR, mask, [&](int q, const float4& kz, const float4& c) {
          st(oA, q, make_float4(g1 * c.x + g2 * kz.x, g1 * c.y + g2 * kz.y, g1 * c.z + g2 * kz.z, g1 * c.w + g2 * kz.w));
        });
      } else {
        const int zin = (js & 1) ? oB : oA, zout = (js & 1) ? oA : oB;
        // z_{j-1}: r / theta at step 2, then what zout holds
        const int zp = js == 2 ? oR : zout;
        const float gp = js == 2 ? ith : 1.0f;
        const float g1 = 1.0f + c1, gm = -c1 * gp;
        rows(zin, mask, [&](int q, const float4& kz, const float4& c) {
          const float4 rv = REG ? rq[REG ? q : 0] : ld(oR, q), pv = ld(zp, q);
          st(zout, q, make_float4(g1 * c.x + gm * pv.x + c2 * (rv.x - kz.x), g1 * c.y + gm * pv.y + c2 * (rv.y - kz.y),
                                  g1 * c.z + gm * pv.z + c2 * (rv.z - kz.z), g1 * c.w + gm * pv.w + c2 * (rv.w - kz.w)));
        });
      }
      compute_sync();
    }
    // tile: w = K~ u, the frame to the neighbours, the sums
    ++tag;
    unsigned long long* const WT = ((tag & 1u) ? f.WT[1] : f.WT[0]);
    float v0 = 0.0f, v1 = 0.0f, v2 = 0.0f;
    const int wf = anew(woff);
    const unsigned int mf = anew(rows_frame);
    rows(oU, rows_own, [&](int q, const float4& w, const float4& u) {
      const float4 rv = REG ? rq[REG ? q : 0] : cheb == 1 ? u : ld(oR, q);
      if (own) {
        if (frame_col || ((mf >> q) & 1u)) {
          unsigned long long* const k = WT + (wf + q * g.pitch);
          asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(k), "l"(word_of(w.x, tag)), "l"(word_of(w.y, tag)) : "memory");
          asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(k + 2), "l"(word_of(w.z, tag)), "l"(word_of(w.w, tag)) : "memory");
        }
        if (REG) wq[REG ? q : 0] = w;
        else st(oW, q, w);
        v0 += rv.x * u.x + rv.y * u.y + rv.z * u.z + rv.w * u.w;
        v1 += w.x * u.x + w.y * u.y + w.z * u.z + w.w * u.w;
        v2 += rv.x * rv.x + rv.y * rv.y + rv.z * rv.z + rv.w * rv.w;
      }
    });
    post_sums(v0, v1, v2);
    // while the sums go round: e += alpha p of the update above, and the band's w
    const unsigned int in = anew(rows_in), mo = anew(rows_own);
    const int wo = anew(woff);
    auto correct = [&]() {
      if (PG) {
        // three rows' p and e in flight at a time
#pragma unroll
        for (int q0 = 0; q0 < RS; q0 += 3) {
          float4 ev[3];
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            const int q = q0 + m < RS ? q0 + m : RS - 1;
            if (q0 + m >= RS) continue;
            const bool mine_q = own && ((mo >> q) & 1u);
            p[q] = mine_q ? *reinterpret_cast<const float4*>(f.m.p + (wo + q * g.pitch)) : z4;
            ev[m] = mine_q && !fresh ? *reinterpret_cast<const float4*>(f.E + (wo + q * g.pitch)) : z4;
          }
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            const int q = q0 + m < RS ? q0 + m : RS - 1;
            if (q0 + m < RS && own && ((mo >> q) & 1u) && !fresh)
              *reinterpret_cast<float4*>(f.E + (wo + q * g.pitch)) = axpy4(ct.x, p[q], ev[m]);
          }
          row_end();
        }
      } else if (own && !fresh) {
#pragma unroll
        for (int q = 0; q < RS; ++q)
          if ((mo >> q) & 1u) {
            float4* const ek = reinterpret_cast<float4*>(f.E + (wo + q * g.pitch));
            *ek = axpy4(ct.x, p[q], *ek);
          }
      }
    };
    // (many rows: the band's words first, before p takes registers: 2048x1024, k = 3, 17.7 -> 16.4 us
    // per iteration; two or more rows' words in flight spill again, 17.3 us and more)
    if (!PG) correct();
#pragma unroll
    for (int q = 0; q < RS; ++q) {
      if (!((in >> q) & 1u) || !in_col || (own && ((mo >> q) & 1u))) continue;
      const unsigned long long* const k = WT + (wo + q * g.pitch);
      unsigned long long w[4];
      auto poll = [&]() {
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w[0]), "=l"(w[1]) : "l"(k) : "memory");
        asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(w[2]), "=l"(w[3]) : "l"(k + 2) : "memory");
      };
      poll();
      long long t0 = 0;
      while ((unsigned int)(w[0] >> 32) != tag || (unsigned int)(w[1] >> 32) != tag || (unsigned int)(w[2] >> 32) != tag ||
             (unsigned int)(w[3] >> 32) != tag) {
        if (t0 == 0) t0 = clock64();
        else if (clock64() - t0 > f.m.d.bar.budget) {
          atomicExch(f.m.d.bar.err, 1);
          sh.fail = 1;
          break;
        }
        poll();
      }
      const float4 v = make_float4(__uint_as_float((unsigned int)w[0]), __uint_as_float((unsigned int)w[1]),
                                   __uint_as_float((unsigned int)w[2]), __uint_as_float((unsigned int)w[3]));
      if (REG) wq[REG ? q : 0] = v;
      else st(oW, q, v);
    }
    if (PG) correct();
    __syncthreads();
    ct = sh.ctl;
    const int flow = __float_as_int(ct.z);
    if (flow & kFail) return 1;
    if (flow & kKeep) {
      // after a replacement: p = u + beta' p, s = w + beta' s, (p, s) to the communication warp
      const float be = ct.y;
      float v = 0.0f;
      if (live)
#pragma unroll
        for (int q = 0; q < RS; ++q) {
          if (!((rows_in >> q) & 1u)) continue;
          s[q] = axpy4(be, s[q], REG ? wq[REG ? q : 0] : ld(oW, q));
          if (own && ((rows_own >> q) & 1u)) {
            p[q] = axpy4(be, p[q], ld(oU, q));
            if (PG) *reinterpret_cast<float4*>(f.m.p + (woff + q * g.pitch)) = p[q];
            v += p[q].x * s[q].x + p[q].y * s[q].y + p[q].z * s[q].z + p[q].w * s[q].w;
          }
        }
      post_sums(0.0f, 0.0f, v);
      __syncthreads();
      ct = sh.ctl;
      if (__float_as_int(ct.z) & kFail) return 1;
    }
    if (flow & (kReplace | kLimit)) {
      end = (flow & kReplace) ? 0 : 2;
      break;
    }
    fresh = false;
  }
#pragma unroll
  for (int q = 0; q < RS; ++q) {
    if ((rows_in >> q) & 1u) st(oA, q, s[q]);
    if (!PG && own && ((rows_own >> q) & 1u)) *reinterpret_cast<float4*>(f.m.p + (woff + q * g.pitch)) = p[q];
  }
  return end;
}

// The computing warps' part of the solve.
template <int NW, int RS>
__device__ __forceinline__ void band_compute(const BandSolve& f, const int tile, BandShared<NW>& sh) {
  unsigned int tag = 0, target = 0;
  bool first = true, last = false;
#pragma unroll 1
  while (true) {
    if (band_restart<NW>(tile, sh, first, last, target)) return;
    target += (first ? 1u : 2u) * f.ntiles;
    int seg = tile;
    asm volatile("" : "+r"(seg));  // what a segment derives from its tile is derived anew, not kept
    const int end = band_segment<NW, RS>(f, seg, sh, first, tag);
    if (end == 1) return;
    last = end == 2;
    first = false;
  }
}

// The communication warp's part: the reductions, the scalars and the flow of the solve, the same
// values in every lane.
template <int NW>
__device__ __forceinline__ void band_communicate(const BandSolve& f, const int tile, BandShared<NW>& sh) {
  const ScaledSolve& d = f.m.d;
  const int lane = threadIdx.x & 31, nb = f.ntiles;
  const double tol2 = d.tol * d.tol;
  // reduction `red` (1, 2, ...) of the warps' sums over all blocks
  auto reduce = [&](unsigned int red, float (&v)[3]) -> bool {
    __syncwarp();
    asm volatile("bar.sync 2, %0;" ::"n"(NW * 32 + 32) : "memory");
    const float4 ws = lane < NW ? sh.ws[lane] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    v[0] = ws.x;
    v[1] = ws.y;
    v[2] = ws.z;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < 3; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    ulonglong2* const slots = f.part + (size_t)(red & 1) * nb;
    if (lane == 0 && tile != d.bar.absent) slot_put(slots + tile, v[0], v[1], v[2], red);
    v[0] = v[1] = v[2] = 0.0f;
    const long long t0 = clock64();
    bool ok = true;
    for (int b0 = 0; b0 < nb; b0 += 32 * 5) {
      float x[5][3];
      while (true) {
        bool here = true;
#pragma unroll
        for (int m = 0; m < 5; ++m) {
          const int b = b0 + lane + 32 * m;
          x[m][0] = x[m][1] = x[m][2] = 0.0f;
          if (b < nb) here = slot_get(slots + b, red, x[m][0], x[m][1], x[m][2]) && here;
        }
        if (__all_sync(0xffffffffu, here)) break;
        if (__shfl_sync(0xffffffffu, clock64() - t0 > d.bar.budget ? 1 : 0, 0)) {
          ok = false;
          break;
        }
      }
      if (!ok) break;
#pragma unroll
      for (int m = 0; m < 5; ++m)
#pragma unroll
        for (int k = 0; k < 3; ++k) v[k] += x[m][k];
    }
    if (!ok && lane == 0) {
      atomicExch(d.bar.err, 1);
      sh.fail = 1;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < 3; ++k) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    return ok;
  };
  unsigned int target = 0, red = 0;
  int it = 0, nrep = 0, rep_it = -1000;
  bool fresh = true, first = true, last = false, restart = false, ok = true;
  // rescaling of p and s, 1 / gamma and 1 / alpha of the last update, the replacement threshold
  float pscale = 1.0f, igamma = 1.0f, ialpha = 1.0f, thr = 0.0f;
#pragma unroll 1
  while (true) {
    if (fresh) {
      if (!first && !last) {
        nrep += 1;
        if (it - rep_it < 3) restart = true;  // replacements back to back: no progress
        rep_it = it;
      }
      const int e = band_restart<NW>(tile, sh, first, last, target);
      target += (first ? 1u : 2u) * nb;
      ok = e != 1;
      if (e) break;
      // directions and K~ p carried over are rescaled to the new normalisation
      const double c = sh.rescale;
      pscale = (float)c;
      igamma = (float)((double)igamma / (c * c + (c == 0.0)));
    }
    float v[3];
    ++red;
    ok = reduce(red, v);
    const float gamma = v[0], delta = v[1], rr32 = v[2];
    float alpha = 0.0f, beta = 0.0f, den = 1.0f;
    bool replace = false, keep = false, update = false;
    if (!fresh) {
      it += 1;
      // the residual fell by `drop`, or the estimate of the unscaled norm meets the tolerance
      replace = rr32 <= thr;
    }
    if (!replace) {
      if (!fresh) {
        // Chronopoulos-Gear: beta = gamma / gamma_old, alpha = gamma / (delta - beta gamma / alpha_old)
        beta = gamma * igamma;
        den = delta - beta * gamma * ialpha;
        update = den > 0.0f && den < INFINITY;
        if (!update) replace = restart = true;  // loss of positivity in FP32: replace and restart
      } else if ((it == 0 && nrep == 0) || restart) {
        // the first direction, or a restart after a breakdown or back-to-back replacements
        restart = false;
        den = delta;
        update = true;
      } else {
        // beta as usual, alpha = gamma / (p, K~ p) from the formed direction
        beta = gamma * igamma * pscale;
        keep = true;
      }
      if (update) alpha = gamma / den;
    }
    const bool limit = !replace && it >= d.max_iter;
    // (a wait for the band that ran out in another warp shows in sh.fail an iteration later)
    if (!ok || *(volatile int*)&sh.fail) ok = false;
    const int flow = (replace ? kReplace : 0) | (keep ? kKeep : 0) | (limit ? kLimit : 0) | (ok ? 0 : kFail);
    if (lane == 0) sh.ctl = make_float4(alpha, beta, __int_as_float(flow), 0.0f);
    __syncthreads();
    if (!ok) break;
    // what the next reduction needs, after the others went on
    if (update) {
      igamma = 1.0f / gamma;
      ialpha = den / gamma;
    }
    if (fresh) {
      // replace at rr32 <= drop^2 gref, or rr_ref rr32 / gref <= tol^2 bb
      const double gref = rr32, dr = f.m.drop * f.m.drop * gref, est = sh.rr > 0.0 ? tol2 * sh.bb * gref / sh.rr : 0.0;
      thr = gref > 0.0 ? (float)(dr > est ? dr : est) : -1.0f;
    }
    if (keep) {
      ++red;
      ok = reduce(red, v);
      // the third sum: it shares a 64-bit word with the reduction's number, so that the pair stays whole
      // where the compiler reads no more of a slot than is used
      ialpha = v[2] / gamma;
      igamma = 1.0f / gamma;
      if (lane == 0) {
        sh.ctl.x = gamma / v[2];
        if (!ok) sh.ctl.z = __int_as_float(flow | kFail);
      }
      __syncthreads();
      if (!ok) break;
    }
    first = false;
    last = limit;
    fresh = replace || limit;
  }
  if (tile == 0 && lane == 0) {
    const bool conv = ok && sh.stop == 1;
    d.out.iters[0] = ok ? it : 0;
    d.out.rr[0] = ok ? sh.rr : 0.0;
    d.out.bb[0] = ok ? sh.bb : 0.0;
    d.out.converged[0] = conv ? 1 : 0;
    if (d.out.total && ok) d.out.total[0] += it;
    if (!conv && d.out.nconv) d.out.nconv[0] += 1;
    if (f.m.replacements) f.m.replacements[0] = nrep;
  }
}

template <int NW, int RS>
__global__ void __launch_bounds__(NW * 32 + 32, 1) k_pcg_poisson_band(const __grid_constant__ BandSolve f) {
  __shared__ BandShared<NW> sh;
  if (threadIdx.x == 0) *reinterpret_cast<BandSolve*>(sh.params) = f;
  __syncthreads();
  band_init<NW>(blockIdx.x, sh);
  if (threadIdx.x < NW * 32) band_compute<NW, RS>(f, blockIdx.x, sh);
  else band_communicate<NW>(f, blockIdx.x, sh);
}

// Shapes of a block that has its SM to itself, by rising capacity: computing warps and region rows
// per warp.  Many warps with few rows hide the latency of each phase; tall tiles keep p and s in
// registers, which leaves 16 warps 128 each.
struct BandShape {
  int nw, rs;
  const void* kernel;
};
#define CCM_BAND(NW, RS) {NW, RS, (const void*)k_pcg_poisson_band<NW, RS>}
const BandShape kShapes[] = {CCM_BAND(15, 1), CCM_BAND(23, 1), CCM_BAND(15, 2), CCM_BAND(19, 2), CCM_BAND(23, 2), CCM_BAND(15, 5), CCM_BAND(15, 9)};
#undef CCM_BAND
constexpr int kShapeN = sizeof(kShapes) / sizeof(kShapes[0]);

// the first shape that holds `rows` region rows (-1: none)
int band_shape(int rows) {
  for (int k = 0; k < kShapeN; ++k)
    if (rows <= kShapes[k].nw * kShapes[k].rs) return k;
  return -1;
}

constexpr size_t kSlot = 16 * sizeof(float);

size_t band_smem(int TY, int cheb) {
  const int h = cheb > 1 ? cheb : 1;
  const size_t rows = (size_t)(TY + 2 * h), row = kRow * sizeof(float), tables = rows * 32 * sizeof(short);
  // a strip's loads reach up to RS rows beyond the last, which the tables cover where RS > 4
  return row + rows * row * (cheb > 1 ? 3 : 2) + std::max(tables, 4 * row) + 2 * kSlot;
}

}  // namespace

// Quads of a region that need slots: all on a stretched mesh, else those of a side of the box.
static size_t band_cut_quads(const Geom& g, int rows) { return g.xf || g.yf ? (size_t)rows * 32 : (size_t)rows + 32; }

// Slots for the coefficients of cut quads: those and a body's outline, as far as they fit (the rest is
// read from global memory; what is left of the SM's memory caches that).
static int band_cut_slots(const Geom& g, int TY, int cheb, size_t room) {
  const size_t used = band_smem(TY, cheb), rows = (size_t)(TY + 2 * (cheb > 1 ? cheb : 1));
  const size_t want = g.xf || g.yf ? rows * 32 : 2 * rows + 256;
  return 2 + (int)std::min((room - used) / kSlot, want);
}

// Tiles of a grid on at most `blocks` blocks with `room` bytes of shared memory: the smallest shape,
// then the fewest region rows (one per warp: then the fewest tiles).  Widths are even shares of the
// grid, at most what a region row holds beside the band.
static bool band_plan(BandSolve* f, int blocks, size_t room) {
  const Geom& g = f->m.d.g;
  const int cheb = f->m.cheb > 1 ? f->m.cheb : 1, h = cheb, hp = (h + 3) & ~3;
  const int wmax = kRow - 2 * hp;
  int best = -1, best_rows = 0, best_tiles = 0;
  for (int nbx = (g.nx + wmax - 1) / wmax; nbx <= blocks && nbx <= (g.nx + wmax - 1) / wmax + 3; ++nbx) {
    const int W = ((g.nx + nbx - 1) / nbx + 3) & ~3;
    if (W > wmax || (g.nx + W - 1) / W != nbx) continue;
    for (int nby = std::min(blocks / nbx, g.ny); nby >= 1; --nby) {
      const int TY = (g.ny + nby - 1) / nby, rows = TY + 2 * h, k = band_shape(rows);
      // taller tiles do not fit either
      if (k < 0 || band_smem(TY, cheb) + kSlot * band_cut_quads(g, rows) > room) break;
      const int tiles = nbx * ((g.ny + TY - 1) / TY), cost = kShapes[k].rs == 1 ? 0 : rows;
      if (best < 0 || k < best || (k == best && (cost < best_rows || (cost == best_rows && tiles < best_tiles)))) {
        best = k;
        best_rows = cost;
        best_tiles = tiles;
        f->W = W;
        f->TY = TY;
        f->nbx = nbx;
        f->ntiles = tiles;
      }
    }
  }
  f->shape = best;
  if (best >= 0) f->ncut = band_cut_slots(g, f->TY, cheb, room);
  return best >= 0;
}

bool band_fits(BandSolve* f) {
  int dev = 0, sms = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  const size_t fixed = sizeof(BandShared<23>) + 512;
  return f->m.cheb <= 8 && band_plan(f, std::min(sms, kBandTilesMax), (size_t)optin - fixed);
}

cudaError_t run_poisson_band(BandSolve f, cudaStream_t st) {
  if (!band_fits(&f)) return cudaErrorInvalidConfiguration;
  const BandShape& shape = kShapes[f.shape];
  const size_t smem = band_smem(f.TY, f.m.cheb) + kSlot * (size_t)(f.ncut - 2);
  if (smem > allow_most_smem(shape.kernel)) return cudaErrorInvalidConfiguration;
  cudaMemsetAsync(f.m.d.bar.count, 0, sizeof(unsigned int) * kBarWords, st);
  void* params[] = {&f};
  return cudaLaunchCooperativeKernel(shape.kernel, f.ntiles, shape.nw * 32 + 32, params, smem, st);
}

}  // namespace ccm
