// krylov2d.cuh - the restart cycle of the 2D GMRES: the operator with its per-cell
// preconditioner in one pass, Gram-Schmidt, the Givens rotations and the stopping test on the
// device (GB300, sm_103a).  Included by grte2d.cu inside namespace grte2.
//
// One Arnoldi step is three launches (binary64: five, of which the last two return at once
// unless the vector has to be orthogonalised again):
//   k2_op     w = D_w P^{-1} M D_w^{-1} V_j
//   k2_dot    h_i = w.V_i and w.w; the last block to finish sums the blocks' parts
//   k2_axpy   w -= sum h_i V_i and |w|^2; the last block rotates the Hessenberg column, decides
//             whether the cycle ends and hands that to the host through pinned memory
// The basis vectors are kept unnormalised with 1/|V_i| beside them (KState.inv), which saves
// a pass over each.  The host launches two steps ahead of the last decision that it has seen;
// a step launched past the end returns at its first instruction.

// Scalars of one restart cycle (device).
struct KState {
  int stop, kk, reorth;
  double beta;                       // |r| at the cycle's start
  double g[kMaxRestart2 + 1], cs[kMaxRestart2], sn[kMaxRestart2], y[kMaxRestart2];
  double rdiag[kMaxRestart2];        // 1/H[i][i]
  double inv[kMaxRestart2 + 1];      // 1/|V_i|
  double h[kMaxRestart2 + 2];        // Hessenberg column of the step
  double coef[kMaxRestart2 + 1];     // what k2_axpy subtracts: h_i inv_i
  double ww;                         // w.w before the orthogonalisation
  double H[kMaxRestart2 * kMaxRestart2];
};

// When a cycle ends (the tests of the residual estimate |g_{j+1}|).
struct KStop {
  double thr;       // where the estimate may stop (gmres2)
  double inner;     // binary32 cycles: the reduction they aim at (0: none)
  int mg;           // the multigrid stage's stagnation test
  int m;            // restart length
};

// What the host reads after a synchronisation (pinned, written by the kernels).
struct KPin {
  double r2;                     // |r|^2 of the restart
  int kk;                        // steps of the last cycle
  int status;                    // status2's copy of D.status
  int stop[kMaxRestart2 + 1];    // per step: the cycle ends after it
};

// ----------------------------------------------------------------------------- operator
// out = M z (PREC: D_w P^{-1} M z) or, with RES, of b - M z, for the prediction's (e, rho)
// matrix (PRED) or the correction's stacked A + G_k; z is read scaled by sc[c] (the Krylov
// unknowns) and by *inv.  P as in the per-cell block elimination: with g_k the diagonal of G_k
//   rho = [r_rho - sum_k w_k g_k r_k/(A+g_k)] / [alpha + sum_k w_k g_k (A - alpha)/(A+g_k)],
//   e_k = (r_k - (alpha + g_k) rho)/(A + g_k)         (correction: r_k/(A + g_k)).
//
// A block takes a tile of TX x TY cells through all pairs: the pair's cell values with a halo
// of one go to shared memory, the (TX+1) x (TY+1) vertex values O = -d D_k u are formed once
// from them, then every cell its streaming derivative; the rows r_k stay in shared memory until
// their weighted sum is complete and the preconditioner can be applied.  In terms of
// a = mu/(2dx) + eta/(2dy), b = mu/(2dx) - eta/(2dy) both stencils are four operations:
//   D_k u = a (u11 - u00) + b (u10 - u01)   (and the same over the vertices of a cell).
// A thread keeps to one cell, its lower left vertex, and (the first threads) one halo cell and
// one vertex of the tile's upper or right edge, so that every index is formed once per block.
// G groups of threads share the pairs of a tile, each with its own barrier.
// Bound: binary64 the FP64 pipe (about 22 operations per cell and pair; the separate vertex,
// cell, sum and preconditioner kernels took about 60), binary32 issue and L1; the vectors are
// read and written once.  512^2 cells, 20 pairs, prediction and correction: 49 and 34 us in
// binary32, 347 and 263 us in binary64 (the separate kernels 127 and 108, 560 and 480); 192^2 in
// binary64 56 and 52 us (105 and 101), 61 x 47 15 and 12 us (53 and 34).
template <typename S>
__host__ __device__ constexpr size_t op_smem(int K, int TX, int TY, int G, bool prec) {
  return sizeof(S) * ((size_t)(TY + 2) * (TX + 2) * G + (size_t)(TY + 1) * (TX + 1) * G + 7 * (size_t)K +
                      (size_t)2 * TX * TY * G + (prec ? (size_t)K * TX * TY : 0));
}

// Barrier of one group of NT threads (a multiple of a warp): its own hardware barrier, 0 being
// __syncthreads'.
template <int NT, int G>
__device__ __forceinline__ void group_sync(int gq) {
  if (NT == 32) __syncwarp();
  else if (G == 1) __syncthreads();
  else asm volatile("bar.sync %0, %1;" ::"r"(gq + 1), "n"(NT) : "memory");
}

// Blocks per SM that the registers have to leave room for: binary32 32 x 8 tiles live on many
// warps in flight, the 32 x 4 tiles of four groups must all be resident at once (a second,
// partial wave would double their time).
template <typename S, int TX, int TY, int G>
constexpr int op_min_blocks() { return TX == 8 ? 1 : G > 1 ? 2 : sizeof(S) == 4 ? 5 : 3; }

template <typename S, bool PRED, bool PREC, bool RES, int TX, int TY, int G>
__global__ void __launch_bounds__(TX * TY * G, op_min_blocks<S, TX, TY, G>())
    k2_op(D2 D, CV<S> cv, const S* __restrict__ z, const S* __restrict__ sc, const double* __restrict__ inv,
          const S* __restrict__ b, S* __restrict__ out, const int* __restrict__ stop) {
  if (stop && *stop) return;
  constexpr int NT = TX * TY;                       // threads of a group = cells of the tile
  constexpr int LC = TX + 2, LV = TX + 1;           // row lengths of the cell and vertex tiles
  constexpr int NC = (TY + 2) * LC, NV = (TY + 1) * LV;
  constexpr int NH = 2 * LC + 2 * TY, NE = LV + TY; // halo cells; vertices of the upper and right edge
  static_assert(NT % 32 == 0 && G < 16, "a group is whole warps, one hardware barrier each");
  static_assert(NH <= NT && NE <= NT, "one halo cell and one edge vertex per thread");
  extern __shared__ __align__(16) unsigned char op_raw[];
  const G2& g = D.g;
  const int K = g.K, nc = (int)g.nc;                // K nc < 2^31 (rows_fit) but not (K+1) nc:
  const int64_t rrow = rho_row(K, nc);              // the rho row's indices have 64 bits
  const int tid = threadIdx.x % NT, gq = threadIdx.x / NT, lx = tid % TX, ly = tid / TX;
  S* p = reinterpret_cast<S*>(op_raw);
  S* const tu = p + gq * NC;   p += G * NC;         // u of the group's pair
  S* const tv = p + gq * NV;   p += G * NV;         // its vertex values
  S* const ka = p;   p += K;
  S* const kb = p;   p += K;
  S* const kmu = p;  p += K;
  S* const keta = p; p += K;
  S* const kw = p;   p += K;
  S* const kex = p;  p += K;                        // |mu| (2/eps)/dx, |eta| (2/eps)/dy: a wall
  S* const key = p;  p += K;                        // side's coefficient of E_cell (cell_sides)
  S* const red = p;  p += 2 * NT * G;
  S* const rows = p;                                // [k][cell of the tile]
  const int p0 = blockIdx.x * TX, q0 = blockIdx.y * TY;
  const S iv = inv ? S(*inv) : S(1);
  for (int k = threadIdx.x; k < K; k += NT * G) {
    const S mu = cv.mu[k], eta = cv.eta[k];
    ka[k] = mu * cv.h2x + eta * cv.h2y;
    kb[k] = mu * cv.h2x - eta * cv.h2y;
    kmu[k] = mu;
    keta[k] = eta;
    kw[k] = cv.w[k];
    kex[k] = fabs(mu) * (cv.te * S(2) * cv.h2x);
    key[k] = fabs(eta) * (cv.te * S(2) * cv.h2y);
  }
  // the thread's cell: scale and scaled rho part, then what its row needs
  const int pc = p0 + lx, qc = q0 + ly;
  const bool live = pc < g.Nx && qc < g.Ny;
  const int oc = (ly + 1) * LC + lx + 1;            // in the tile
  // (past the domain: a halo cell of a live one, or on a periodic axis its image)
  const int c = live ? qc * g.Nx + pc : cell_of(g, pc, qc);
  const S fc = c >= 0 ? (sc ? sc[c] * iv : iv) : S(0);
  const S rc = PRED && c >= 0 ? z[rrow + c] * fc : S(0);
  const S A = live ? cv.A[c] : S(0), kc = live ? cv.kc[c] : S(0), al = PRED && live ? cv.alpha[c] : S(0);
  const S ws = PREC && live ? cv.wsc[c] : S(1), arc = al * rc;
  const bool xw = g.bcx == GRTE_BC_INFLOW, yw = g.bcy == GRTE_BC_INFLOW;
  // side weights of the general form (cell_sides), for tiles that touch an inflow wall
  const bool wl = xw && pc == 0, wr = xw && pc == g.Nx - 1, wb = yw && qc == 0, wt = yw && qc == g.Ny - 1;
  const S cL = cv.h2x * (wl ? S(0) : wr ? S(-2) : S(-1)), cR = cv.h2x * (wr ? S(0) : wl ? S(2) : S(1));
  const S cB = cv.h2y * (wb ? S(0) : wt ? S(-2) : S(-1)), cT = cv.h2y * (wt ? S(0) : wb ? S(2) : S(1));
  // its halo cell: lower row, upper row, left and right columns
  int hc = -1, ho = 0;
  S hf = S(0), hu = S(0);
  if (tid < NH) {
    const int hx = tid < 2 * LC ? tid % LC : (tid - 2 * LC) % 2 * (TX + 1);
    const int hy = tid < LC ? 0 : tid < 2 * LC ? TY + 1 : 1 + (tid - 2 * LC) / 2;
    ho = hy * LC + hx;
    hc = cell_of(g, p0 - 1 + hx, q0 - 1 + hy);
    if (hc >= 0) {
      hf = sc ? sc[hc] * iv : iv;
      if (PRED) hu = z[rrow + hc] * hf;
    }
  }
  // its vertices: the cell's lower left one, and one of the upper row or right column
  const int ov = ly * LV + lx, ex = tid < LV ? tid : TX, ey = tid < LV ? TY : tid - LV;
  auto vertex_kind = [&](int i, int j) { return i <= g.Nx && j <= g.Ny ? vkind(g, i, j) : -1; };
  auto vertex_d = [&](int i, int j) { return i <= g.Nx && j <= g.Ny ? cv.dv[(int64_t)j * (g.Nx + 1) + i] : S(0); };
  const S d0 = vertex_d(pc, qc), d1 = tid < NE ? vertex_d(p0 + ex, q0 + ey) : S(0);
  const int k0 = vertex_kind(pc, qc), k1 = tid < NE ? vertex_kind(p0 + ex, q0 + ey) : -1;
  // The tile's inflow-wall vertices (x walls: TY + 1 each, y walls: TX + 1 each; corners enter no
  // cell), one per thread from the first on: one or two warps take the wall expression instead
  // of every warp that has a wall cell.  The vertex, its wall and its inner vertex's coefficient:
  constexpr int NW = 2 * (LV + TY + 1);
  int wk = 0, wvx = 0, wvy = 0;
  S wd = S(0);
  for (int t = tid; t < NW && wk == 0; t += NT) {
    const bool x = t < 2 * (TY + 1);
    const int u = x ? t : t - 2 * (TY + 1), len = x ? TY + 1 : LV, r = u % len;
    const bool lo = u < len;
    const int i = x ? (lo ? 0 : g.Nx) : p0 + r, j = x ? q0 + r : (lo ? 0 : g.Ny);
    if (i < p0 || i > p0 + TX || j < q0 || j > q0 + TY || i > g.Nx || j > g.Ny) continue;
    if (vkind(g, i, j) != (x ? 2 : 3)) continue;
    wk = x ? (lo ? 1 : 2) : (lo ? 3 : 4);
    wvx = i - p0;
    wvy = j - q0;
    wd = cv.dv[(int64_t)(j + (x ? 0 : lo ? 1 : -1)) * (g.Nx + 1) + i + (x ? (lo ? 1 : -1) : 0)];
  }
  // a tile away from the inflow walls has node equations only (uniform over the block)
  const bool edge = (xw && (p0 == 0 || p0 + TX >= g.Nx)) || (yw && (q0 == 0 || q0 + TY >= g.Ny));
  if (edge)
    for (int e = tid; e < NV; e += NT) tv[e] = S(0);   // (corners, and past the grid)
  __syncthreads();
  // sum w_k kappa S_k, and the preconditioner's sum w_k g_k r_k/(A+g_k) (apart: at inflow walls
  // the first cancels against the right-hand side to a 1/eps-th of its terms)
  S st = S(0), sp = S(0);
  // the next pair's values are loaded while the current one is worked on
  S nz = S(0), nh = S(0), nb = S(0), ngd = S(0), ngi = S(0);
  auto fetch = [&](int k) {
    if (k >= K) return;
    const int o = k * nc;
    if (c >= 0) nz = z[o + c];
    if (hc >= 0) nh = z[o + hc];
    if (live) {
      if (RES) nb = b[o + c];
      if (PREC) ngi = cv.gdi[o + c];
      if (PREC && PRED) ngd = cv.gd[o + c];
    }
  };
  fetch(gq);
  for (int k = gq; k < K; k += G) {
    const S ec = nz * fc, uc = PRED ? fma(nz, fc, rc) : ec, bk = nb, gdk = ngd, gik = ngi;
    tu[oc] = uc;
    // (not over another thread's own cell: the halo is the ring around the tile)
    if (tid < NH) tu[ho] = PRED ? fma(nh, hf, hu) : nh * hf;
    group_sync<NT, G>(gq);
    fetch(k + G);
    const S a = ka[k], bb = kb[k];
    auto node = [&](int o, S d) {   // O at the vertex whose lower left cell is at o
      return -d * fma(a, tu[o + LC + 1] - tu[o], bb * (tu[o + 1] - tu[o + LC]));
    };
    S v00 = S(0);
    if (!edge) {
      v00 = node(oc - LC - 1, d0);
      tv[ov] = v00;
      if (tid < NE) tv[ey * LV + ex] = node(ey * LC + ex, d1);
    } else {
      if (k0 == 0) tv[ov] = node(oc - LC - 1, d0);
      if (tid < NE && k1 == 0) tv[ey * LV + ex] = node(ey * LC + ex, d1);
      if (wk != 0) {
        // Eq. bc-pre along the wall's normal with E the mean of the two wall cells
        const bool x = wk <= 2, lo = wk == 1 || wk == 3;
        const int o = wvy * LC + wvx, step = x ? (lo ? 1 : -1) : (lo ? LC : -LC);
        const int w0 = x ? (lo ? o + 1 : o) : (lo ? o + LC : o), w1 = w0 + (x ? LC : 1);
        const S comp = x ? kmu[k] : keta[k];
        const S ht = (lo ? comp > S(0) : comp < S(0)) ? S(-0.5) * cv.te : S(0.5) * cv.te;
        tv[wvy * LV + wvx] = fma(ht, tu[w0] + tu[w1], -node(o + step, wd));
      }
    }
    group_sync<NT, G>(gq);
    if (live) {
      const S v10 = tv[ov + 1], v01 = tv[ov + LV], v11 = tv[ov + LV + 1];
      if (edge) v00 = tv[ov];
      S div;
      if (!edge) {
        div = fma(a, v11 - v00, bb * (v10 - v01));
      } else {
        div = fma(kmu[k], fma(cL, v00 + v01, cR * (v10 + v11)), keta[k] * fma(cB, v00 + v10, cT * (v01 + v11)));
        const S ed = (wl || wr ? kex[k] : S(0)) + (wb || wt ? key[k] : S(0));
        div = fma(ed, uc, div);
      }
      S y = fma(kc, div, PRED ? fma(A, ec, arc) : A * ec);
      if (RES) y = bk - y;
      if (PRED) {
        st = fma(kw[k], kc * div, st);
        if (PREC) {
          sp = fma(kw[k] * gdk * gik, y, sp);
          rows[k * NT + tid] = y;
        }
      }
      if (!PREC) out[k * nc + c] = y;
      else if (!PRED) out[k * nc + c] = ws * y * gik;
    }
  }
  if (!PRED) return;
  // the rho row: the groups' sums in a fixed order
  if (G > 1) {
    red[gq * NT + tid] = st;
    red[(G + gq) * NT + tid] = sp;
    __syncthreads();
    st = red[tid];
    sp = red[G * NT + tid];
#pragma unroll
    for (int q = 1; q < G; ++q) {
      st += red[q * NT + tid];
      sp += red[(G + q) * NT + tid];
    }
  }
  if (!live) return;
  const int64_t orho = rrow + c;
  S rr = fma(al, rc, st);
  if (RES) rr = b[orho] - rr;
  if (!PREC) {
    if (gq == 0) out[orho] = rr;
    return;
  }
  const S rho = (rr - sp) * cv.pdi[c];
  if (gq == 0) out[orho] = ws * rho;
#pragma unroll 4
  for (int k = gq; k < K; k += G) {
    const int o = k * nc + c;
    out[o] = ws * fma(-(al + cv.gd[o]), rho, rows[k * NT + tid]) * cv.gdi[o];
  }
}

// ----------------------------------------------------------------------------- Gram-Schmidt
// Streaming kernels over the basis: 16-byte loads (the vectors start on 16-byte boundaries,
// a last partial group is done by single threads), one full wave of blocks.  Bound: HBM, or
// the L2 where the basis fits; on small grids the latency of a turn and of the block sums.
constexpr int kVecBlocks = 4 * 152;   // at most: block parts of a value

template <typename S> struct Vec16;
template <> struct Vec16<float> { using T = float4; static constexpr int N = 4; };
template <> struct Vec16<double> { using T = double2; static constexpr int N = 2; };
template <typename S>
__device__ __forceinline__ void load16(const S* __restrict__ p, S (&v)[Vec16<S>::N]) {
  *reinterpret_cast<typename Vec16<S>::T*>(v) = *reinterpret_cast<const typename Vec16<S>::T*>(p);
}

// The last block to arrive (the others' writes to global memory visible to it).
__device__ __forceinline__ bool last_block(unsigned* count) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    const unsigned t = atomicAdd(count, 1u);
    last = t == gridDim.x - 1;
    if (last) *count = 0;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// Block sums of C values per thread (C a power of two), within a warp in the vectors' type and
// across warps in binary64, to part[(i0 + t) * gridDim.x + block] for t < nv.  A warp leaves each
// lane one value's sum by
// halving the values it holds with every exchange (C - 1 + 5 - log2 C additions instead of
// 5 C: a binary64 warp addition holds its sub-partition's pipe for many cycles).
template <typename S, int C>
__device__ __forceinline__ void block_sums(S (&acc)[C], int nv, int i0, double* __restrict__ part) {
  __shared__ double red[kThreads / 32][C];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int base = 0, o = 16;
#pragma unroll
  for (int h = C / 2; h >= 1; h >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int s = 0; s < h; ++s) {
      const S send = up ? acc[s] : acc[s + h], keep = up ? acc[s + h] : acc[s];
      acc[s] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
    if (up) base += h;
  }
  for (; o >= 1; o >>= 1) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
  if ((lane & (32 / C - 1)) == 0) red[wid][base] = (double)acc[0];
  __syncthreads();
  if ((int)threadIdx.x < nv) {
    double u = 0.0;
#pragma unroll
    for (int q = 0; q < kThreads / 32; ++q) u += red[q][threadIdx.x];
    part[(int64_t)(i0 + threadIdx.x) * gridDim.x + blockIdx.x] = u;
  }
  __syncthreads();
}

// Sum of value i's block parts (one warp, fixed order); every lane gets it.
__device__ __forceinline__ double part_sum(const double* __restrict__ part, int i) {
  const int lane = threadIdx.x & 31;
  double s = 0.0;
  for (int q = lane; q < (int)gridDim.x; q += 32) s += __ldcg(part + (int64_t)i * gridDim.x + q);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// Dot products of w with the C - 1 vectors at V (loads past nv repeat the last one and are
// dropped) and w.w, U groups of 16 bytes per thread and turn.
template <typename S, int C, int U>
__device__ __forceinline__ void dot_chunk(const S* __restrict__ w, const S* __restrict__ V, int64_t ld, int nv,
                                          int64_t n, int i0, int iww, double* __restrict__ part) {
  constexpr int N = Vec16<S>::N, D1 = C - 1;
  S acc[C];
#pragma unroll
  for (int t = 0; t < C; ++t) acc[t] = S(0);
  const int64_t ng = n / N, nt = (int64_t)gridDim.x * blockDim.x;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < ng; q += nt * U) {
    S wv[U][N], v[U][D1][N];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t qu = q + u * nt;
      if (qu < ng) {
        load16(w + qu * N, wv[u]);
#pragma unroll
        for (int t = 0; t < D1; ++t) load16(V + (int64_t)max(min(t, nv - 1), 0) * ld + qu * N, v[u][t]);
      } else {
#pragma unroll
        for (int e = 0; e < N; ++e) wv[u][e] = S(0);
#pragma unroll
        for (int t = 0; t < D1; ++t)
#pragma unroll
          for (int e = 0; e < N; ++e) v[u][t][e] = S(0);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int e = 0; e < N; ++e) {
#pragma unroll
        for (int t = 0; t < D1; ++t) acc[t] = fma(wv[u][e], v[u][t][e], acc[t]);
        acc[D1] = fma(wv[u][e], wv[u][e], acc[D1]);
      }
  }
  if (blockIdx.x == 0 && (int64_t)threadIdx.x < n - ng * N) {
    const int64_t e = ng * N + threadIdx.x;
    const S wv = w[e];
#pragma unroll
    for (int t = 0; t < D1; ++t) acc[t] = fma(wv, V[(int64_t)max(min(t, nv - 1), 0) * ld + e], acc[t]);
    acc[D1] = fma(wv, wv, acc[D1]);
  }
  // value nv of the chunk: w.w (first chunk), beside the vectors' sums
  if (nv < D1) {
#pragma unroll
    for (int t = 0; t < D1; ++t)
      if (t == nv) acc[t] = acc[D1];
  }
  block_sums<S, C>(acc, iww >= 0 ? nv + 1 : nv, i0, part);
}

// h_i = (w.V_i)/|V_i| for i < nv (pass 1; pass 2 adds) and w.w, for k2_axpy.  nv = 0: the
// restart's |w|^2 for the host.
// C: one more than the vectors of a chunk (chosen by nv, so that few vectors leave room for
// more blocks and more loads of each in flight).
template <typename S, int C>
__global__ void __launch_bounds__(kThreads, C <= 4 ? 4 : C <= 8 ? 3 : 2)
    k2_dot(const S* __restrict__ w, const S* __restrict__ V, int64_t ld, int nv, int64_t n, double* __restrict__ part,
           KState* ks, unsigned* count, int pass, KPin* pin) {
  if (nv > 0 && (ks->stop || (pass == 2 && !ks->reorth))) return;
  constexpr int U = C <= 4 || (C <= 8 && sizeof(S) == 4) ? 2 : 1;
  // the last chunk first: it carries w.w in the slot after its vectors
  const int nch = nv > 0 ? (nv + C - 2) / (C - 1) : 1;
  for (int ch = nch - 1; ch >= 0; --ch) {
    const int i0 = ch * (C - 1), c = min(C - 1, nv - i0);
    dot_chunk<S, C, U>(w, nv > 0 ? V + (int64_t)i0 * ld : w, ld, max(c, 0), n, i0, ch == nch - 1 ? nv : -1, part);
  }
  if (!last_block(count)) return;
  for (int i = threadIdx.x >> 5; i <= nv; i += kThreads / 32) {
    const double s = part_sum(part, i);
    if ((threadIdx.x & 31) != 0) continue;
    if (i == nv) {
      ks->ww = s;
      if (nv == 0) {
        pin->r2 = s;
        pin->kk = ks->kk;
      }
    } else {
      const double h = s * ks->inv[i];
      ks->h[i] = pass == 1 ? h : ks->h[i] + h;
      ks->coef[i] = h * ks->inv[i];
    }
  }
}

// sqrt(q) and 1/sqrt(q) for q >= 0: a binary32 seed and two Newton-Raphson steps (relative error
// at binary64 rounding) instead of the square root, divide and hypot sequences, whose dependent
// binary64 operations cost ~70 cycles each on the one thread that runs them; outside the seed's
// range, and for 0, inf and NaN, the plain operations.
__device__ __forceinline__ void sqrt_pair(double q, double& r, double& ir) {
  if (!(q > 1e-36 && q < 1e36)) {
    r = sqrt(q);
    ir = 1.0 / r;
    return;
  }
  double y = (double)rsqrtf((float)q);
  y = y * fma(-0.5 * q, y * y, 1.5);
  y = y * fma(-0.5 * q, y * y, 1.5);
  r = q * y;
  ir = y;
}

// After step j's column h_0..h_j and |w|^2 = hn2 are final: rotations, residual estimate and
// the cycle's end (the last block; the operands of the serial chain come to shared memory
// first).
__device__ __forceinline__ void krylov_column(KState* ks, int j, double hn2, KStop sp, KPin* pin) {
  __shared__ double h[kMaxRestart2 + 1], cs[kMaxRestart2], sn[kMaxRestart2], gs[2];
  const int t = threadIdx.x;
  if (t <= j) h[t] = __ldcg(&ks->h[t]);
  if (t < j) {
    cs[t] = __ldcg(&ks->cs[t]);
    sn[t] = __ldcg(&ks->sn[t]);
  }
  if (t == 64) gs[0] = __ldcg(&ks->g[j]);
  if (t == 65) gs[1] = j >= 3 ? __ldcg(&ks->g[j - 3]) : 0.0;
  __syncthreads();
  if (t == 0) {
    double hn, ihn, rr, ir;
    sqrt_pair(hn2, hn, ihn);
    double r = h[0];
    for (int i = 0; i < j; ++i) {
      const double u = h[i + 1];
      h[i] = cs[i] * r + sn[i] * u;
      r = cs[i] * u - sn[i] * r;
    }
    sqrt_pair(fma(r, r, hn2), rr, ir);
    h[j] = rr;
    const double c = rr > 0.0 ? r * ir : 1.0, s = rr > 0.0 ? hn * ir : 0.0;
    const double gj = gs[0], gn = -s * gj, ga = fabs(gn);
    ks->rdiag[j] = ir;
    ks->cs[j] = c;
    ks->sn[j] = s;
    ks->g[j] = c * gj;
    ks->g[j + 1] = gn;
    ks->inv[j + 1] = hn > 0.0 ? ihn : 1.0;
    ks->kk = j + 1;
    bool stop = ga <= sp.thr || hn == 0.0 || j + 1 >= sp.m;
    if (sp.inner > 0.0 && ga <= sp.inner * ks->beta) stop = true;
    if (sp.mg && j >= 4 && ga <= 1e-6 * ks->beta && ga > 0.5 * fabs(gs[1])) stop = true;
    ks->stop = stop ? 1 : 0;
    pin->stop[j] = stop ? 1 : 0;
  }
  __syncthreads();
  if (t <= j) ks->H[t * kMaxRestart2 + j] = h[t];
}

// w -= sum_{i <= j} coef_i V_i and |w|^2.  Pass 1 decides whether w has to be orthogonalised
// again (binary64: when little of it is left, so that the rounding of the first pass weighs:
// |w|^2 <= 1e-2 |w before|^2, which takes the same steps to the same errors as a second pass
// always, on 192^2 and 61 x 47 cells 1.21x and 1.18x as fast; binary32 cycles, which only have to gain 1e5 and whose restarts
// are binary64, never); the last pass finishes the column.
// C: vectors of a chunk, loaded together (past the last one it is loaded again, with a zero
// coefficient); U groups of 16 bytes per thread and turn.
template <typename S, int C>
__global__ void __launch_bounds__(kThreads, C <= 4 ? 4 : C <= 8 ? 3 : 2)
    k2_axpy(S* __restrict__ w, const S* __restrict__ V, int64_t ld, int j, int64_t n, double* __restrict__ part,
            KState* ks, unsigned* count, int pass, KStop sp, KPin* pin) {
  if (ks->stop || (pass == 2 && !ks->reorth)) return;
  constexpr int N = Vec16<S>::N, U = C <= 4 || (C <= 8 && sizeof(S) == 4) ? 2 : 1;
  __shared__ S cf[kMaxRestart2 + 16];
  const int nv = j + 1;
  for (int i = threadIdx.x; i < kMaxRestart2 + 16; i += blockDim.x) cf[i] = i < nv ? S(-ks->coef[i]) : S(0);
  __syncthreads();
  S nrm = S(0);
  const int64_t ng = n / N, nt = (int64_t)gridDim.x * blockDim.x;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < ng; q += nt * U) {
    S a[U][N];
#pragma unroll
    for (int u = 0; u < U; ++u) load16(w + min(q + u * nt, ng - 1) * N, a[u]);
    for (int i0 = 0; i0 < nv; i0 += C) {
      S v[U][C][N];
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int t = 0; t < C; ++t)
          load16(V + (int64_t)min(i0 + t, nv - 1) * ld + min(q + u * nt, ng - 1) * N, v[u][t]);
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int e = 0; e < N; ++e) {   // two sums per element: shorter chains
          S s0 = S(0), s1 = S(0);
#pragma unroll
          for (int t = 0; t < C; t += 2) {
            s0 = fma(cf[i0 + t], v[u][t][e], s0);
            s1 = fma(cf[i0 + t + 1], v[u][t + 1][e], s1);
          }
          a[u][e] += s0 + s1;
        }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (q + u * nt >= ng) continue;
#pragma unroll
      for (int e = 0; e < N; ++e) nrm = fma(a[u][e], a[u][e], nrm);
      *reinterpret_cast<typename Vec16<S>::T*>(w + (q + u * nt) * N) = *reinterpret_cast<typename Vec16<S>::T*>(a[u]);
    }
  }
  if (blockIdx.x == 0 && (int64_t)threadIdx.x < n - ng * N) {
    const int64_t e = ng * N + threadIdx.x;
    S a = w[e];
    for (int i = 0; i < nv; ++i) a = fma(cf[i], V[(int64_t)i * ld + e], a);
    w[e] = a;
    nrm = fma(a, a, nrm);
  }
  S one[1] = {nrm};
  block_sums<S, 1>(one, 1, 0, part);
  if (!last_block(count)) return;
  const double hn2 = part_sum(part, 0);   // every warp the same
  const bool again = sizeof(S) == 8 && pass == 1 && hn2 <= 1e-2 * ks->ww;
  if (threadIdx.x == 0) ks->reorth = again ? 1 : 0;
  if (!again) krylov_column(ks, j, hn2, sp, pin);
}

// Start of a cycle from the residual in V_0 (its norm beta; inv0 its stored scale).
__global__ void k2_cycle_begin(KState* ks, double beta, double inv0) {
  ks->stop = 0;
  ks->kk = 0;
  ks->reorth = 0;
  ks->beta = beta;
  ks->g[0] = beta;
  ks->inv[0] = inv0;
}

// H y = g (upper triangular, kk columns), column by column with lane = row (the next column
// loaded ahead); y scaled by the vectors' 1/|V_i| for k2_update.
__global__ void k2_solve_y(KState* ks) {
  const int kk = ks->kk, lane = threadIdx.x;
  double g0 = lane < kk ? ks->g[lane] : 0.0, g1 = lane + 32 < kk ? ks->g[lane + 32] : 0.0;
  auto col = [&](int i, double& a, double& b, double& d, double& v) {
    a = i >= 0 && lane < i ? ks->H[lane * kMaxRestart2 + i] : 0.0;
    b = i >= 0 && lane + 32 < i ? ks->H[(lane + 32) * kMaxRestart2 + i] : 0.0;
    d = i >= 0 ? ks->rdiag[i] : 0.0;
    v = i >= 0 ? ks->inv[i] : 0.0;
  };
  double a, b, d, v;
  col(kk - 1, a, b, d, v);
  for (int i = kk - 1; i >= 0; --i) {
    double an, bn, dn, vn;
    col(i - 1, an, bn, dn, vn);
    const double y = __shfl_sync(0xffffffffu, i < 32 ? g0 : g1, i & 31) * d;
    g0 -= a * y;
    g1 -= b * y;
    if (lane == 0) ks->y[i] = y * v;
    a = an, b = bn, d = dn, v = vn;
  }
}

// x += D_w^{-1} V y (x binary64 and unscaled; a binary32 basis is combined in binary32 and
// added once): blockIdx.y = block of cells, so that the scale is read by cell.
template <typename S>
__global__ void __launch_bounds__(kThreads) k2_update(double* __restrict__ x, const S* __restrict__ V, int64_t ld,
                                                      int64_t nc, const double* __restrict__ iw,
                                                      const KState* __restrict__ ks) {
  __shared__ S cf[kMaxRestart2];
  const int kk = ks->kk;
  for (int i = threadIdx.x; i < kk; i += blockDim.x) cf[i] = S(ks->y[i]);
  __syncthreads();
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= nc) return;
  const int64_t o = blockIdx.y * nc + c;
  S t0 = S(0), t1 = S(0);
  int i = 0;
#pragma unroll 4
  for (; i + 2 <= kk; i += 2) {
    t0 = fma(cf[i], V[(int64_t)i * ld + o], t0);
    t1 = fma(cf[i + 1], V[(int64_t)(i + 1) * ld + o], t1);
  }
  if (i < kk) t0 = fma(cf[i], V[(int64_t)i * ld + o], t0);
  x[o] += iw[c] * (double)(t0 + t1);
}

// Krylov scale per cell from a magnitude field src: s = |src| + 1e-13 max|src| (uniform: s =
// max|src| for every cell), w = f/s (f = 1 in the prediction, eps in the correction, whose
// unknown E_J enters E as eps E_J), with binary32 copies for the binary32 cycles.
__global__ void k2_maxabs(const double* __restrict__ x, int64_t n, double* __restrict__ part, unsigned* count,
                          double* __restrict__ out) {
  __shared__ double red[kThreads / 32];
  auto block_max = [&](double t) {
    for (int o = 16; o > 0; o >>= 1) t = fmax(t, __shfl_xor_sync(0xffffffffu, t, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    double m = 0.0;
#pragma unroll
    for (int q = 0; q < kThreads / 32; ++q) m = fmax(m, red[q]);
    __syncthreads();
    return m;
  };
  double t = 0.0;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
    t = fmax(t, fabs(x[j]));
  const double m = block_max(t);
  if (threadIdx.x == 0) part[blockIdx.x] = m;
  if (!last_block(count)) return;
  t = 0.0;
  for (int q = threadIdx.x; q < (int)gridDim.x; q += blockDim.x) t = fmax(t, __ldcg(part + q));
  const double a = block_max(t);
  if (threadIdx.x == 0) *out = a;
}

__global__ void k2_weights(D2 D, const double* __restrict__ src, double f, const double* __restrict__ maxabs,
                           int uniform, float* __restrict__ w32, float* __restrict__ iw32) {
  const int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (c >= D.g.nc) return;
  const double m = *maxabs;
  const double s = (uniform ? m : fabs(src[c]) + 1e-13 * m) + 1e-300;
  const double w = f / s, iw = s / f;
  D.wsc[c] = w;
  D.iwsc[c] = iw;
  if (w32) {
    w32[c] = (float)w;
    iw32[c] = (float)iw;
  }
}
