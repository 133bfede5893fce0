// lbm_tile.cuh — several time steps per launch for channels whose columns fit
// in shared memory (FP32 storage).  Included by lbm_mix.cu inside its
// anonymous namespace, after the node arithmetic and the step kernel.
//
// What bounds a small channel is not memory or arithmetic but the length of
// one step: a launch per step, the CTA's wall prologue, and rows that a warp
// takes one after another.  lbm_step_kernel needs 9.0 us per step on a 320 x 16
// channel, 9.7 us on 700 x 20 and on 1280 x 64, whose state is 6 MB (14.5, 18 and
// 33 before it took rows and end strips by the channel's size); this kernel needs
// 2.2, 2.3 and 4.6 us in calls of 100 steps.  lbm_tile_kernel cuts the channel
// into tiles of W whole columns, one CTA each, loads a tile with
// a halo of k columns on both sides into shared memory and takes k steps
// there, the updated range shrinking by one column per side and step.  What a
// column needs besides its neighbours (r and tau_q of its walls) is inside
// the tile, because the tile holds all of its rows; the tiles that hold the
// columns next to an end recompute the density correction (Eq. rho2) from
// their own column sums.  So no CTA waits for another, and the redundant halo
// work (about (k - 1) columns per tile and step) is paid on SMs that a
// launch per step would leave idle.
//
// A tile's node p = c S + j (column c, row j) keeps its nine pairs side by
// side, as a strip row does in memory (72 bytes a node; 18 words and odd S
// keep a warp's accesses free of bank conflicts along rows and along columns
// alike), so that every access is at a fixed offset from p, p - S or p + S.
// Warps have one of three roles, so that none diverges: inner rows (one node
// per thread for the whole launch where they fit), wall rows, and 1/tau_q of
// every column's walls, beside the others' moments and rates.  One barrier
// hands 1/tau_q over, a second ends the step.  r of the next step's walls is
// formed where the wall node's populations are still in registers.
//
// Sums over a column's rows (diagnostics, and the ends' density correction)
// are taken by column_sum8, in an order that depends on N alone: neither the
// tile width, nor k, nor the other channels of a batch change a bit of the
// result.

constexpr int TILE_TAUQ = 64;      // threads of the 1/tau_q role
constexpr int TILE_WALL = 64;      // threads of the wall-row role
constexpr int TILE_INNER = 512;    // most threads of the inner-row role
constexpr int TILE_THREADS = TILE_INNER + TILE_WALL + TILE_TAUQ;
constexpr int TILE_KMAX = 15;      // most steps of one launch
constexpr int TILE_SMEM_MAX = 227 * 1024 - 1024;

// One channel's share of a launch.
struct TileInst {
  LatCore L;
  const float* fin;      // deviations of the first step's input (strip layout)
  float* fout;           // deviations after step k
  const float* refrho;
  const float* alpha;
  const double* cs_in;   // [4][Nx]; the columns next to the ends are read
  double* cs_out;        // [4][Nx] column sums after step k
  float2* hist;          // [records][4][Nx] column sums (pairs, column_sum8) of
                         // the launch's diagnostic steps, without N rhobar
  int W;                 // own columns per tile
  int diag_every, diag_phase;  // steps taken since the last multiple of diag_every
  int last;              // 1: step k ends the call (its sums are recorded)
};

template <int NI>
struct TileBatch {
  int k;                    // steps of this launch (all channels)
  int block0[NI + 1];       // first CTA of each channel
  TileInst inst[NI];
};

__host__ __device__ inline int tile_stride(int N) { return N | 1; }
// Shared memory of a tile of `cols` columns: two state buffers (nine pairs a
// node), two buffers of density and momentum pairs for the column sums, nine
// pairs of reference densities and wall quantities per column, psi's table.
__host__ __device__ inline size_t tile_smem(int N, int cols) {
  return sizeof(float2) * ((2 * 9 + 4) * (size_t)cols * tile_stride(N) + 9 * (size_t)cols) +
         sizeof(float) * 20 + sizeof(float4) * PSI_SEGMENTS;
}

// Pre-collision deviations of the tile node whose nine pairs start at f
// (column x, S rows of pairs from one column to the next): the arithmetic of
// pull_node.  E: kappa_in[2], kappa_out[2] and the ghost reference offsets of
// load_ends; inl, outl: the neighbour column is the inlet, outlet ghost.
// wall: -1 inner row, 0 bottom, 1 top (the same in all lanes of a warp but
// for the mix of 0 and 1); r: the wall's.
__device__ __forceinline__ void pull_tile(const float2* f, int S9, const LatCore& L, const float* E,
                                          float2 dl, float2 dr, bool inl, bool outl, int wall,
                                          float2 r, float2 g[9]) {
  // population i of the node at f + off, streamed from the column to its left
  // or right, in the deviations of its own column
  auto left = [&](int off, int i, float2 cw) -> float2 {
    const float2* q = f + off + i;
    float2 v = q[-S9];
    if (inl) {
      const float2 a = q[0], b = q[S9];
      const float2 e = make_float2(fmaf(2.0f, a.x, -b.x), fmaf(2.0f, a.y, -b.y));
      v = fma2(make_float2(E[0], E[1]), e, mul2(cw, make_float2(E[4], E[5])));
    }
    return fma2(cw, dl, v);
  };
  auto right = [&](int off, int i, float2 cw) -> float2 {
    const float2* q = f + off + i;
    float2 v = q[S9];
    if (outl) {
      const float2 a = q[0], b = q[-S9];
      const float2 e = make_float2(fmaf(2.0f, a.x, -b.x), fmaf(2.0f, a.y, -b.y));
      v = fma2(make_float2(E[2], E[3]), e, mul2(cw, make_float2(E[6], E[7])));
    }
    return fma2(cw, dr, v);
  };
  const float2 c1 = L.cw1_2, c5 = L.cw5_2;
  g[0] = f[0];
  g[1] = left(0, 1, c1);
  g[3] = right(0, 3, c1);
  if (wall < 0) {
    g[2] = f[2 - 9];
    g[5] = left(-9, 5, c5);
    g[6] = right(-9, 6, c5);
    g[4] = f[4 + 9];
    g[7] = right(9, 7, c5);
    g[8] = left(9, 8, c5);
    return;
  }
  // the wall row: normal u0 and diagonal u1, u2 populations it does not
  // receive, from the partners o0, o1, o2 that leave it (bottom: 2, 5, 6 from
  // 4, 7, 8; top: 4, 7, 8 from 2, 5, 6); those from the inside as above.  The
  // diagonals 5 and 8 come from the left column, 6 and 7 from the right one.
  const bool top = wall == 1;
  const int in = top ? -9 : 9;  // the neighbouring inner row
  const float2 o0 = f[top ? 2 : 4], o1 = f[top ? 5 : 7], o2 = f[top ? 6 : 8];
  const float2 i0 = f[in + (top ? 2 : 4)];
  const float2 il = left(in, top ? 5 : 8, c5), ir = right(in, top ? 6 : 7, c5);
  const float2 q = sub2(f2(1.0f), r);
  float2 u0, u1, u2;
  if (L.wall_mode == LBM_WALL_BSR) {
    // the mirror images leave the neighbour columns of this row
    const float2 ml = left(0, top ? 5 : 8, c5), mr = right(0, top ? 6 : 7, c5);
    u0 = o0;
    u1 = fma2(r, o1, mul2(q, top ? mr : ml));
    u2 = fma2(r, o2, mul2(q, top ? ml : mr));
  } else {
    const float2 t = mul2(r, add2(add2(o0, o1), o2)), t6 = mul2(t, f2(1.0f / 6.0f));
    u0 = fma2(q, o0, fma2(f2(-2.0f), t6, t));
    u1 = fma2(q, o1, t6);
    u2 = fma2(q, o2, t6);
  }
  g[2] = top ? i0 : u0;
  g[5] = top ? il : u1;
  g[6] = top ? ir : u2;
  g[4] = top ? u0 : i0;
  g[7] = top ? u1 : ir;
  g[8] = top ? u2 : il;
}

// r of a wall node from its post-collision deviations g(0) .. g(8): the sums
// of dbb_r.
template <typename G>
__device__ __forceinline__ float2 slip_tile(const LatCore& L, float2 rb, float cm, G&& g) {
  float2 acc = f2(0.0f);
#pragma unroll
  for (int i = 0; i < 9; ++i) acc = add2(acc, g(i));
  const float2 rho = add2(rb, acc);
  return slip_r(L, rho.x, rho.y, cm);
}

template <int NI>
__global__ void __launch_bounds__(TILE_THREADS, 1)
    lbm_tile_kernel(const __grid_constant__ TileBatch<NI> B) {
  extern __shared__ float2 tile_mem[];
  pdl_launch_dependents();
  const int ii = channel_of<NI>(B.block0, blockIdx.x);
  const TileInst& I = B.inst[ii];
  const LatCore& L = I.L;
  const int b = (int)blockIdx.x - B.block0[ii], k = B.k;
  const int N = L.N, Nx = L.Nx, S = tile_stride(N), S9 = 9 * S;
  const int T = (int)blockDim.x - TILE_WALL - TILE_TAUQ, tid = threadIdx.x;
  // own columns [xs, xs + own), tile columns [xl, xl + C)
  const bool open = !L.x_periodic;
  const int xfirst = open ? 1 : 0, nup = open ? Nx - 2 : Nx;
  const int xs = xfirst + b * I.W, own = min(I.W, xfirst + nup - xs);
  const int C = own + 2 * k, xl = xs - k, P = C * S;
  float2* const F0 = tile_mem;
  float2* const F1 = F0 + 9 * P;
  float2* const SD = F1 + 9 * P;  // [2][P] density deviations by step parity
  float2* const MX = SD + 2 * P;  // [2][P] x momenta
  float2* const RB = MX + 2 * P;  // [C] reference densities
  float2* const RW = RB + C;           // [2][2][C] r by step parity and wall
  float2* const A12 = RW + 4 * C;      // [2][C] (A1, A2) of Eq. A12
  float* const CM = (float*)(A12 + 2 * C);  // [2][C] c_m of Eq. R
  float* const OMQ = CM + 2 * C;       // [2][C] 1/tau_q
  float* const E = OMQ + 2 * C;        // [2][8] by step parity
  float4* const PT = (float4*)(((size_t)(E + 16) + 15) & ~(size_t)15);  // psi's table
  // column of the channel behind tile column c; < 0 where there is none
  auto column = [&](int c) -> int {
    int x = xl + c;
    if (!open) {
      x %= Nx;
      return x < 0 ? x + Nx : x;
    }
    return x < 0 || x >= Nx ? -1 : x;
  };
  // lanes of a warp along the columns of one (row, population) pair, the rest
  // of the warp on the next pairs: calls move(tile column, channel column,
  // pair index ji = 9 j + i) over columns [c0, c0 + n)
  auto sweep = [&](int c0, int n, auto&& move) {
    int lw = 1;
    while (lw < n && lw < 32) lw <<= 1;
    const int per = 32 / lw, sub = (tid & 31) / lw, lane = (tid & 31) & (lw - 1);
    const int step = per * ((int)blockDim.x >> 5);
    for (int c = lane; c < n; c += lw) {
      const int x = column(c0 + c);
      if (x < 0) continue;
      for (int ji = (tid >> 5) * per + sub; ji < 9 * N; ji += step) move(c0 + c, x, ji);
    }
  };
  load_psi_table(PT, tid, blockDim.x);
  pdl_wait();
  // the tile, by 8-byte asynchronous copies
  sweep(0, C, [&](int c, int x, int ji) {
    const float* src = I.fin + ((size_t)(x >> 5) * L.SS + 2 * (x & 31)) + (size_t)PS * ji;
    const unsigned dst = (unsigned)__cvta_generic_to_shared(F0 + c * S9 + ji);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
  });
  for (int c = tid; c < C; c += blockDim.x) {
    const int x = column(c);
    RB[c] = x < 0 ? f2(0.0f) : make_float2(I.refrho[x], I.refrho[Nx + x]);
    for (int w = 0; w < 2; ++w) {
      const float al = x < 0 ? 1.0f : I.alpha[w * Nx + x];
      A12[w * C + c] = slip_coefficients(al);
      CM[w * C + c] = slip_cm(L, al);
    }
  }
  // the ends whose density correction this tile needs at some step
  const bool has_in = open && xl < 1, has_out = open && xl + C - 1 > Nx - 2;
  // one lane per (end, species) for step 1
  const int er = (int)blockDim.x - 1 - tid;
  if (er < 4 && (er < 2 ? has_in : has_out)) {
    const int sp = er & 1, x0 = er < 2 ? 0 : Nx - 1, in = er < 2 ? 1 : -1;
    const double* cs = I.cs_in + (size_t)sp * Nx + x0;
    const float* ref = I.refrho + sp * Nx + x0;
    end_factors(L.end_mass[er >> 1][sp], split_double(cs[in]), split_double(cs[2 * in]), ref[0],
                ref[in], ref[2 * in], E[8 + er], E[12 + er]);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();

  const bool compute = tid < T + TILE_WALL, walls = compute && tid >= T;
  // the nodes of this thread's role: q = first, first + stride, ... < count;
  // inner rows column by column, wall rows wall by wall
  const int rows = walls ? C - 2 : max(N - 2, 1);  // q / rows: column or wall
  const int first = walls ? tid - T : tid, stride = walls ? TILE_WALL : T;
  const int count = walls ? 2 * (C - 2) : (C - 2) * (N - 2);
  const int first_d = first / rows, first_m = first - first_d * rows;
  const bool has_end = has_in || has_out;
  // every node is some thread's first
  const bool one_pass = (C - 2) * (N - 2) <= T && 2 * (C - 2) <= TILE_WALL;
  const int half = (N + 1) / 2;
  // r of wall w of column c (node p) at step t: left by step t - 1, for the
  // first step from the populations
  auto wall_r = [&](const float2* F, int p, int w, int c, int t) -> float2 {
    if (t > 1) return RW[(t & 1) * 2 * C + w * C + c];
    return slip_tile(L, RB[c], CM[w * C + c], [&](int i) { return F[9 * p + i]; });
  };
  int phase = I.diag_phase, rec = 0;
  for (int t = 1; t <= k; ++t) {
    const float2* Fc = (t & 1) ? F0 : F1;
    float2* Fn = (t & 1) ? F1 : F0;
    const float* Et = E + 8 * (t & 1);
    float2* sd = SD + (t & 1) * P;
    float2* mxs = MX + (t & 1) * P;
    float2* rw_next = RW + ((t + 1) & 1) * 2 * C;
    if (++phase == I.diag_every) phase = 0;
    const bool diag = phase == 0 || (I.last && t == k);
    const bool sums = diag || t == k;
    // columns [ca, cb) are updated in this step
    const int ca = max(t, open ? 1 - xl : 0), cb = min(C - t, open ? Nx - 1 - xl : C);
    if (compute) {
      bool waited = false;
      int d = first_d, e = first_m;
      for (int q = first;; q += stride) {
        if (q != first) {
          d = q / rows;
          e = q - d * rows;
        }
        const int c = 1 + (walls ? e : d), j = walls ? (d ? N - 1 : 0) : 1 + e;
        const int p = c * S + j, x = xl + c;
        const bool ok = q < count && c >= ca && c < cb;
        float2 g[9];
        Macro2 m;
        float om_s, om_d;
        if (ok) {
          const float2 rb = RB[c], rl = RB[c - 1], rr = RB[c + 1];
          float2 r = f2(0.0f);
          if (walls) r = wall_r(Fc, p, d, c, t);
          pull_tile(Fc + 9 * p, S9, L, Et, sub2(rl, rb), sub2(rr, rb), open && x == 1,
                    open && x == Nx - 2, walls ? d : -1, r, g);
          macro2(L, rb, g, m);
          if (sums || has_end) sd[p] = m.sd;
          rates2(L, PT, m, (float)j + 0.5f, om_s, om_d);
        }
        if (!waited) {
          asm volatile("bar.sync 1, %0;" ::"r"((int)blockDim.x) : "memory");
          waited = true;
        }
        if (ok) {
          const float om_q = OMQ[(j < half ? 0 : C) + c];
          const float2 mv = collide2(g, L, m, om_d, om_q, om_s);
          if (sums) mxs[p] = mv;
#pragma unroll
          for (int i = 0; i < 9; ++i) Fn[9 * p + i] = g[i];
          if (walls)  // r of the next step
            rw_next[d * C + c] = slip_tile(L, RB[c], CM[d * C + c], [&](int i) { return g[i]; });
        }
        if (q + stride >= count) break;
      }
    } else {
      // 1/tau_q of both walls of every column updated now
      const int wt = tid - T - TILE_WALL;
      for (int q = wt; q < 2 * (C - 2); q += TILE_TAUQ) {
        const int w = q >= C - 2 ? 1 : 0, c = 1 + q - w * (C - 2), x = xl + c;
        if (c < ca || c >= cb) continue;
        const int p = c * S + (w == 0 ? 0 : N - 1);
        const float2 rb = RB[c], rl = RB[c - 1], rr = RB[c + 1];
        // with DBB walls tau_q does not depend on r (see wall_task)
        const float2 r = L.wall_mode == LBM_WALL_BSR ? wall_r(Fc, p, w, c, t) : f2(0.0f);
        float2 g[9];
        pull_tile(Fc + 9 * p, S9, L, Et, sub2(rl, rb), sub2(rr, rb), open && x == 1,
                  open && x == Nx - 2, w, r, g);
        const float2 rho = add2(rb, density_sum(g));
        const float n = number_density(L, rho.x, rho.y), inv_n = rcp_fast(n);
        const float mx = mixture_mass(__fadd_rn(rho.x, rho.y), n, inv_n);
        OMQ[w * C + c] = inv_tau_q(L, PT, kDpsiTab, n, inv_n, mx, A12[w * C + c]);
      }
      __syncwarp();
      if (has_end)  // also waits: the ends' density sums are then complete
        asm volatile("bar.sync 1, %0;" ::"r"((int)blockDim.x) : "memory");
      else
        asm volatile("bar.arrive 1, %0;" ::"r"((int)blockDim.x) : "memory");
    }
    if (has_end && t < k) {
      // kappa of the next step (Eq. rho2) from this step's column sums: one
      // warp of the 1/tau_q role per end, eight lanes per (column, species)
      if (!one_pass) __syncthreads();
      if (!compute) {
        const int wt = tid - T - TILE_WALL, end = wt >> 5, lane = wt & 31;
        const int x1 = end == 0 ? 1 : Nx - 2, x2 = end == 0 ? 2 : Nx - 3;
        const int xc = (lane & 16) ? x2 : x1, c = xc - xl, sp = (lane >> 3) & 1;
        const bool need = end == 0 ? has_in : has_out;
        // both columns are in the range just updated whenever column x1 is
        // still to be updated at the next step
        const int cf = x1 - xl;
        if (need && cf >= t + 1 && cf < C - t - 1) {  // warp-uniform
          const float2 v = column_sum8(N, lane & 7, [&](int r) { return sp ? sd[c * S + r].y : sd[c * S + r].x; });
          const float2 cs = column_total(N, sp ? RB[c].y : RB[c].x, v);
          const float2 cs2 = make_float2(__shfl_down_sync(0xffffffffu, cs.x, 16),
                                         __shfl_down_sync(0xffffffffu, cs.y, 16));
          if (lane == 0 || lane == 8) {
            const int cg = cf + (end == 0 ? -1 : 1), c2 = cf + (end == 0 ? 1 : -1);
            const float r0 = sp ? RB[cg].y : RB[cg].x, r1 = sp ? RB[cf].y : RB[cf].x,
                        r2 = sp ? RB[c2].y : RB[c2].x;
            float* En = E + 8 * ((t + 1) & 1);
            end_factors(L.end_mass[end][sp], cs, cs2, r0, r1, r2, En[2 * end + sp],
                        En[4 + 2 * end + sp]);
          }
        }
      }
    }
    __syncthreads();
    const bool own_end = open && (xs <= 2 || xs + own > Nx - 3);
    if (diag || (t == k && own_end)) {
      // column sums of the own columns; one warp per column
      for (int it = tid; it < 32 * own; it += blockDim.x) {
        const int c = k + (it >> 5), q = (it >> 3) & 3;
        const float2* v = (q < 2 ? sd : mxs) + c * S;
        const float2 s =
            column_sum8(N, it & 7, [&](int r) { return (q & 1) ? v[r].y : v[r].x; });
        if ((it & 7) == 0) {
          const int x = xs + (it >> 5);
          if (diag) I.hist[((size_t)rec * 4 + q) * Nx + x] = s;
          if (t == k)
            I.cs_out[(size_t)q * Nx + x] =
                pair_value(q < 2 ? column_total(N, q == 0 ? RB[c].x : RB[c].y, s) : s);
        }
      }
      if (t == k && open && tid < 4) {
        if (xs == 1) I.cs_out[(size_t)tid * Nx] = 0.0;
        if (xs + own == Nx - 1) I.cs_out[(size_t)tid * Nx + Nx - 1] = 0.0;
      }
    }
    if (diag) ++rec;
  }
  // own columns out
  const float2* Fk = (k & 1) ? F1 : F0;
  sweep(k, own, [&](int c, int x, int ji) {
    float* dst = I.fout + ((size_t)(x >> 5) * L.SS + 2 * (x & 31)) + (size_t)PS * ji;
    *reinterpret_cast<float2*>(dst) = Fk[c * S9 + ji];
  });
}

// The diagnostic records of a call's steps from the column sums the tile
// kernel left in hist: C_l(x), CL, C~_l, the mean mass flows and the total
// masses, the formulas and reductions of column_epilogue.  Grid: blocks of
// columns x records x channels.  The FP64 work of 256 columns holds an SM for
// some 2.5 us, so a record has a block per 256 columns up to REC_BLOCKS, the
// last of which folds their partials in block order.  With one block per record
// a call of a single step took 82 us on 5000 x 64 and 441 on 40000 x 8 (54 and
// 79 now), a step with a record of its own, many to a launch, 27 and 121 (18
// and 32); 320 x 16 the same either way.
// The last record to finish advances the record counter.
constexpr int REC_BLOCKS = 128;
struct RecInst {
  int N, Nx, x_periodic, light;
  float s[2];
  double C_in, C_out;
  const float2* hist;
  const float* refrho;
  double* diag;
  unsigned long long* diag_count;
  unsigned* counter;
  double* clprof;
  double* part;      // [records][NPART][blocks]
  unsigned* rec_cnt; // [records] blocks finished
  int nrec, blocks;
};
template <int NI>
struct RecBatch {
  RecInst inst[NI];
};
inline int record_blocks(int Nx) {
  const int b = (Nx + 255) / 256;
  return b < REC_BLOCKS ? b : REC_BLOCKS;
}

template <int NI>
__global__ void __launch_bounds__(256) lbm_records_kernel(const __grid_constant__ RecBatch<NI> B) {
  // partials by warp, then of the block, then of the record: min C_l, its
  // column, sums of C_l - C_in, the momenta, the masses and the columns
  __shared__ double wpart[NPART][8], tot[NPART];
  __shared__ int last;
  pdl_wait();
  const RecInst &I = B.inst[NI > 1 ? blockIdx.z : 0], &L = I;
  const int r = blockIdx.y, b = blockIdx.x, nb = I.blocks, tid = threadIdx.x, Nx = L.Nx;
  if (r >= I.nrec || b >= nb) return;
  const unsigned long long cnt0 = *(volatile unsigned long long*)I.diag_count;
  const float2* h = I.hist + (size_t)r * 4 * Nx;
  const bool profile = r == I.nrec - 1;
  double vmin = INFINITY, sm[6] = {0, 0, 0, 0, 0, 0};
  int imin = 0x7fffffff;
  for (int x = 256 * b + tid; x < Nx; x += 256 * nb) {
    if (!L.x_periodic && (x < 1 || x > Nx - 2)) {
      if (profile) I.clprof[x] = x == 0 ? L.C_in : L.C_out;
      continue;
    }
    double c[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) c[q] = pair_value(h[(size_t)q * Nx + x]);
    c[0] += (double)L.N * (double)I.refrho[x];
    c[1] += (double)L.N * (double)I.refrho[Nx + x];
    const double na = c[0] * L.s[0], nb_ = c[1] * L.s[1];
    const double Cl = (L.light == 0 ? na : nb_) / (na + nb_);
    if (profile) I.clprof[x] = Cl;
    if (Cl < vmin) {
      vmin = Cl;
      imin = x;
    }
    sm[0] += Cl - L.C_in;
    sm[1] += c[2];
    sm[2] += c[3];
    sm[3] += c[0];
    sm[4] += c[1];
    sm[5] += 1.0;
  }
  warp_min(vmin, imin);
#pragma unroll
  for (int q = 0; q < 6; ++q) sm[q] = warp_sum(sm[q]);
  const int lane = tid & 31, wid = tid >> 5;
  if (lane == 0) {
    wpart[0][wid] = vmin;
    wpart[1][wid] = (double)imin;
#pragma unroll
    for (int q = 0; q < 6; ++q) wpart[2 + q][wid] = sm[q];
  }
  __syncthreads();
  // n partials get(q, k) of each quantity q folded by warp q, warp 0 the minimum
  // and its column; the result in tot
  static_assert(NPART == 8, "a warp per partial");
  auto fold = [&](int n, auto&& get) {
    if (wid == 0) {
      double v = INFINITY;
      int i = 0x7fffffff;
      for (int k = lane; k < n; k += 32) {
        const double w = get(0, k);
        const int iw = (int)get(1, k);
        if (w < v || (w == v && iw < i)) {
          v = w;
          i = iw;
        }
      }
      warp_min(v, i);
      if (lane == 0) {
        tot[0] = v;
        tot[1] = (double)i;
      }
    } else if (wid != 1) {
      double v = 0.0;
      for (int k = lane; k < n; k += 32) v += get(wid, k);
      v = warp_sum(v);
      if (lane == 0) tot[wid] = v;
    }
    __syncthreads();
  };
  fold(8, [&](int q, int k) { return wpart[q][k]; });
  if (nb > 1) {
    double* p = I.part + (size_t)r * NPART * nb;
    if (tid < NPART) {
      p[(size_t)tid * nb + b] = tot[tid];
      __threadfence();
    }
    __syncthreads();
    if (tid == 0) last = atomicAdd(I.rec_cnt + r, 1u) == (unsigned)nb - 1u;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (tid == 0) I.rec_cnt[r] = 0u;
    fold(nb, [&](int q, int k) { return __ldcg(p + (size_t)q * nb + k); });
  }
  if (tid >= NREC) return;
  double dev = tot[2];
  if (!L.x_periodic) dev += (L.C_out - L.C_in);  // the outlet boundary column
  const unsigned long long cnt = cnt0 + (unsigned long long)r + 1ull;
  // one division for all eight entries
  double num = 0.0, den = 1.0;
  switch (tid) {
    case 0: num = (double)cnt; break;
    case 1: num = L.C_in - tot[0], den = L.C_in; break;
    case 2: num = dev, den = (double)Nx * L.C_in; break;
    case 3: num = tot[3], den = tot[7]; break;
    case 4: num = tot[4], den = tot[7]; break;
    case 5: num = tot[1]; break;
    case 6: num = tot[5]; break;
    case 7: num = tot[6]; break;
  }
  I.diag[(size_t)((cnt - 1ull) % DIAG_CAP) * NREC + tid] = num / den;
  __syncwarp((1u << NREC) - 1u);
  if (tid != 0) return;
  __threadfence();
  if (atomicAdd(I.counter, 1u) == (unsigned)I.nrec - 1u) {
    *I.diag_count = cnt0 + (unsigned long long)I.nrec;
    *I.counter = 0u;
  }
}
