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
// G groups of threads share the pairs of a tile, each with its own barrier.
// Bound: binary64 the FP64 pipe (about 23 operations per cell and pair; the separate vertex,
// cell, sum and preconditioner kernels took about 60), binary32 issue and L1; the vectors are
// read and written once.  512^2 cells, 20 pairs: 49 us (prediction) and 36 us (correction) in
// binary32, 398 and 325 us in binary64, against 127 and 108, and 560 and 480, of the separate
// kernels; 61 x 47 in binary64 19 and 15 us against 53 and 34.
template <typename S>
__host__ __device__ constexpr size_t op_smem(int K, int TX, int TY, int G, bool prec) {
  return sizeof(S) * ((size_t)(TY + 2) * (TX + 2) * (2 + G) + (size_t)(TY + 1) * (TX + 1) * G + 5 * (size_t)K +
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

template <typename S, bool PRED, bool PREC, bool RES, int TX, int TY, int G>
__global__ void __launch_bounds__(TX * TY * G) k2_op(D2 D, CV<S> cv, const S* __restrict__ z,
                                                     const S* __restrict__ sc, const double* __restrict__ inv,
                                                     const S* __restrict__ b, S* __restrict__ out,
                                                     const int* __restrict__ stop) {
  if (stop && *stop) return;
  constexpr int NT = TX * TY;                       // threads of a group = cells of the tile
  constexpr int LC = TX + 2, LV = TX + 1;           // row lengths of the cell and vertex tiles
  constexpr int NC = (TY + 2) * LC, NV = (TY + 1) * LV;
  constexpr int RC = (NC + NT - 1) / NT, RV = (NV + NT - 1) / NT;
  static_assert(NT % 32 == 0 && G < 16, "a group is whole warps, one hardware barrier each");
  extern __shared__ __align__(16) unsigned char op_raw[];
  const G2& g = D.g;
  const int K = g.K, nc = (int)g.nc;
  const int tid = threadIdx.x % NT, gq = threadIdx.x / NT, lx = tid % TX, ly = tid / TX;
  S* p = reinterpret_cast<S*>(op_raw);
  S* const sf = p;   p += NC;                       // scale of the tile's cells
  S* const su = p;   p += NC;                       // scaled rho part
  S* const tu = p + gq * NC;   p += G * NC;         // u of the group's pair
  S* const tv = p + gq * NV;   p += G * NV;         // its vertex values
  S* const ka = p;   p += K;
  S* const kb = p;   p += K;
  S* const kmu = p;  p += K;
  S* const keta = p; p += K;
  S* const kw = p;   p += K;
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
  }
  // this thread's cells of the haloed tile (the same for every pair) and its vertices
  int cc[RC];
#pragma unroll
  for (int r = 0; r < RC; ++r) {
    const int e = tid + r * NT;
    const int c = e < NC ? cell_of(g, p0 - 1 + e % LC, q0 - 1 + e / LC) : -1;
    cc[r] = c;
    if (e < NC && gq == 0) {
      const S f = c >= 0 ? (sc ? sc[c] * iv : iv) : S(0);
      sf[e] = f;
      su[e] = PRED && c >= 0 ? z[(int64_t)K * nc + c] * f : S(0);
    }
  }
  S dv[RV];
  int vk[RV];      // 0: node equation, 2/3: x/y wall, else nothing to form
#pragma unroll
  for (int r = 0; r < RV; ++r) {
    const int e = tid + r * NT, i = p0 + e % LV, j = q0 + e / LV;
    const bool in = e < NV && i <= g.Nx && j <= g.Ny;
    vk[r] = in ? vkind(g, i, j) : -1;
    dv[r] = in ? cv.dv[(int64_t)j * (g.Nx + 1) + i] : S(0);
  }
  const int pc = p0 + lx, qc = q0 + ly;
  const bool live = pc < g.Nx && qc < g.Ny;
  const int c = live ? qc * g.Nx + pc : 0;
  const bool wall = live && ((g.bcx == GRTE_BC_INFLOW && (pc == 0 || pc == g.Nx - 1)) ||
                             (g.bcy == GRTE_BC_INFLOW && (qc == 0 || qc == g.Ny - 1)));
  const S A = live ? cv.A[c] : S(0), kc = live ? cv.kc[c] : S(0), al = PRED && live ? cv.alpha[c] : S(0);
  const S ws = PREC && live ? cv.wsc[c] : S(1);
  __syncthreads();
  const int oc = (ly + 1) * LC + lx + 1;            // the thread's cell in the tile
  const S fc = sf[oc], rc = su[oc], arc = al * rc;
  // sum w_k kappa S_k, and the preconditioner's sum w_k g_k r_k/(A+g_k) (apart: at inflow walls
  // the first cancels against the right-hand side to a 1/eps-th of its terms)
  S st = S(0), sp = S(0);
  // the next pair's values are loaded while the current one is worked on
  S nx[RC], nz = S(0), nb = S(0), ngd = S(0), ngi = S(0);
  auto fetch = [&](int k) {
#pragma unroll
    for (int r = 0; r < RC; ++r) nx[r] = k < K && cc[r] >= 0 ? z[(int64_t)k * nc + cc[r]] : S(0);
    if (k < K && live) {
      const int64_t o = (int64_t)k * nc + c;
      nz = z[o];
      if (RES) nb = b[o];
      if (PREC) ngi = cv.gdi[o];
      if (PREC && PRED) ngd = cv.gd[o];
    }
  };
  fetch(gq);
  for (int k = gq; k < K; k += G) {
#pragma unroll
    for (int r = 0; r < RC; ++r) {
      const int e = tid + r * NT;
      if (e < NC) tu[e] = PRED ? fma(nx[r], sf[e], su[e]) : nx[r] * sf[e];
    }
    const S ec = nz * fc, bk = nb, gdk = ngd, gik = ngi;
    group_sync<NT, G>(gq);
    fetch(k + G);
    const S a = ka[k], bb = kb[k];
    auto node = [&](int o, S d) {   // O at the vertex whose lower left cell is at o
      return -d * fma(a, tu[o + LC + 1] - tu[o], bb * (tu[o + 1] - tu[o + LC]));
    };
#pragma unroll
    for (int r = 0; r < RV; ++r) {
      const int e = tid + r * NT, vx = e % LV, vy = e / LV, o = vy * LC + vx;
      if (e >= NV) continue;
      S v = S(0);
      if (vk[r] == 0) {
        v = node(o, dv[r]);
      } else if (vk[r] == 2 || vk[r] == 3) {
        // Eq. bc-pre along the wall's normal with E the mean of the two wall cells
        const int i = p0 + vx, j = q0 + vy;
        const bool xw = vk[r] == 2, lo = xw ? i == 0 : j == 0;
        const S comp = xw ? kmu[k] : keta[k];
        const S sg = (lo ? comp > S(0) : comp < S(0)) ? S(1) : S(-1);
        const int step = xw ? (lo ? 1 : -1) : (lo ? LC : -LC);
        const int64_t vin = (int64_t)(j + (xw ? 0 : (lo ? 1 : -1))) * (g.Nx + 1) + i + (xw ? (lo ? 1 : -1) : 0);
        const int w0 = xw ? (lo ? o + 1 : o) : (lo ? o + LC : o), w1 = w0 + (xw ? LC : 1);
        v = -sg * cv.te * (S(0.5) * (tu[w0] + tu[w1])) - node(o + step, cv.dv[vin]);
      }
      tv[e] = v;
    }
    group_sync<NT, G>(gq);
    if (live) {
      const int o = ly * LV + lx;
      const S v00 = tv[o], v10 = tv[o + 1], v01 = tv[o + LV], v11 = tv[o + LV + 1];
      S div;
      if (!wall) {
        div = fma(a, v11 - v00, bb * (v10 - v01));
      } else {
        // (E_cell not from tu: the next pair's values may be on their way into it)
        const CellSides<S> cs = cell_sides<S>(D, cv, k, pc, qc);
        div = kmu[k] * cv.h2x * (cs.wL * (v00 + v01) + cs.wR * (v10 + v11)) +
              keta[k] * cv.h2y * (cs.wB * (v00 + v10) + cs.wT * (v01 + v11)) + cs.ed() * (ec + rc);
      }
      const int64_t o2 = (int64_t)k * nc + c;
      S y = fma(kc, div, PRED ? fma(A, ec, arc) : A * ec);
      if (RES) y = bk - y;
      if (PRED) {
        st = fma(kw[k], kc * div, st);
        if (PREC) {
          sp = fma(kw[k] * gdk * gik, y, sp);
          rows[k * NT + tid] = y;
        }
      }
      if (!PREC) out[o2] = y;
      else if (!PRED) out[o2] = ws * y * gik;
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
  const int64_t orho = (int64_t)K * nc + c;
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
    const int64_t o2 = (int64_t)k * nc + c;
    out[o2] = ws * fma(-(al + cv.gd[o2]), rho, rows[k * NT + tid]) * cv.gdi[o2];
  }
}

// ----------------------------------------------------------------------------- Gram-Schmidt
// Streaming kernels over the basis: 16-byte loads (the vectors start on 16-byte boundaries,
// a last partial group is done by single threads), one full wave of blocks.  Bound: HBM, or
// the L2 where the basis fits; on small grids the fixed cost of the block sums, so the blocks
// are as few as leave every thread a few groups of 16 bytes (vec_blocks).
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

// Block sums of C values per thread (C a power of two), in binary64, to
// part[(i0 + t) * gridDim.x + block] for t < nv.  A warp leaves each lane one value's sum by
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
// |w|^2 <= 1e-2 |w before|^2; binary32 cycles, which only have to gain 1e5 and whose restarts
// are binary64, never); the last pass finishes the column.
template <typename S>
__global__ void __launch_bounds__(kThreads, 2) k2_axpy(S* __restrict__ w, const S* __restrict__ V, int64_t ld, int j,
                                                       int64_t n, double* __restrict__ part, KState* ks,
                                                       unsigned* count, int pass, KStop sp, KPin* pin) {
  if (ks->stop || (pass == 2 && !ks->reorth)) return;
  constexpr int N = Vec16<S>::N;
  __shared__ S cf[kMaxRestart2 + 1];
  const int nv = j + 1;
  for (int i = threadIdx.x; i < nv; i += blockDim.x) cf[i] = S(-ks->coef[i]);
  __syncthreads();
  S nrm = S(0);
  const int64_t ng = n / N;
  for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < ng; q += (int64_t)gridDim.x * blockDim.x) {
    S a[N], a2[N];
    load16(w + q * N, a);
#pragma unroll
    for (int e = 0; e < N; ++e) a2[e] = S(0);
    const S* Vq = V + q * N;
    int i = 0;
    for (; i + 8 <= nv; i += 8) {
      S v[8][N];
#pragma unroll
      for (int t = 0; t < 8; ++t) load16(Vq + (int64_t)(i + t) * ld, v[t]);
#pragma unroll
      for (int t = 0; t < 8; t += 2)
#pragma unroll
        for (int e = 0; e < N; ++e) {
          a[e] = fma(cf[i + t], v[t][e], a[e]);
          a2[e] = fma(cf[i + t + 1], v[t + 1][e], a2[e]);
        }
    }
    for (; i + 2 <= nv; i += 2) {
      S v[2][N];
      load16(Vq + (int64_t)i * ld, v[0]);
      load16(Vq + (int64_t)(i + 1) * ld, v[1]);
#pragma unroll
      for (int e = 0; e < N; ++e) {
        a[e] = fma(cf[i], v[0][e], a[e]);
        a2[e] = fma(cf[i + 1], v[1][e], a2[e]);
      }
    }
    if (i < nv) {
      S v[N];
      load16(Vq + (int64_t)i * ld, v);
#pragma unroll
      for (int e = 0; e < N; ++e) a[e] = fma(cf[i], v[e], a[e]);
    }
#pragma unroll
    for (int e = 0; e < N; ++e) {
      a[e] += a2[e];
      nrm = fma(a[e], a[e], nrm);
    }
    *reinterpret_cast<typename Vec16<S>::T*>(w + q * N) = *reinterpret_cast<typename Vec16<S>::T*>(a);
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
