// step_split64.cuh -- the CTU step in FP64: included by step_fp64.cu inside
// namespace ctulbm.
//
// GB300 issues two FP64 lanes per clock and SM (a warp instruction takes the
// pipe 16 cycles), so the step in FP64 is bound by the number of FP64
// operations and nothing else: 32 x 8 bytes of traffic per node would allow 26.5
// G nodes/s, the ~480 operations of a node 1.2.  So it is laid out for the fewest
// operations, evenly spread, and memory traffic is not counted:
//
//  * two kernels, advection f^n -> f* and collision f* -> f^{n+1}, through global
//    memory (the second buffer holds f*, the result returns to the first): a
//    fused kernel advects 8 of every 64 columns and 8 rows of every row block
//    more than once; apart, advection repeats 4 of 32 columns and one row of a
//    block, and the collision's tiles repeat only the density of their halo;
//  * work is handed out per warp (advection: a half strip of one plane, and of a
//    row block as many rows as leave every SM a dozen warps) or per tile of 16 x 8
//    nodes (collision), small enough that lattices of 128^2 nodes use every SM.  An
//    SM needs about twelve warps to keep the FP64 pipe busy: one warp alone gets
//    an FP64 result every ~170 cycles however independent its operations are;
//  * comparisons, minima, absolute values and signs are integer operations on the
//    bit patterns; quarters and quadruples are folded into constants and exponents.
//
// Measured, us per step (advection + collision), against the fused kernel it
// replaces: 128^2 CTU2 233 -> 26, 362^2 CTU1 167 -> 100, 1024^2 CTU2 2175 -> 965 (419 +
// 546; the FP64 pipe 88 and 85 % busy).

// Four times the half-limited jump of Sec. II C 2 (see mc_half): the minmod of
// 4 R, 4 Ru and R + Ru, s = R + Ru given.  No FP64 operation: magnitudes compare
// as integers, 4 m is m with the exponent raised by two (a subnormal or zero m
// counts as zero).
// (mag64 hides the mask: written in C++ the compiler makes it an FP64 |x|.)
__device__ __forceinline__ unsigned long long mag64(double x) {
  unsigned long long m;
  asm("{\n .reg .b64 t;\n mov.b64 t, %1;\n and.b64 %0, t, 0x7fffffffffffffff;\n}\n" : "=l"(m) : "d"(x));
  return m;
}
template <int LIM>
__device__ __forceinline__ double mc_quad(double R, double Ru, double s) {
  if constexpr (LIM == 1) {
    return 0.0;
  } else if constexpr (LIM == 2) {
    return R + R;
  } else {
    constexpr unsigned long long ONE = 1ULL << 52;
    const unsigned long long m = min(mag64(R), mag64(Ru));
    const unsigned long long v = min(m >= ONE ? m + 2 * ONE : 0ULL, mag64(s));
    const int hr = __double2hiint(R);
    const bool opposed = (hr ^ __double2hiint(Ru)) < 0;
    return __hiloint2double(opposed ? 0 : (int)(v >> 32) | (hr & (int)0x80000000),
                            opposed ? 0 : (int)v);
  }
}

// ------------------------------------------------------------- advection
// A warp advects one plane over half a strip (28 columns; its 32 lanes hold two
// more on either side) and a block of rows, a lane one column, marching in the
// direction of xi_y with the lanes laid out in the direction of xi_x: upwind is
// always the lane and the row before, whatever the signs.  With (Sec. II C 2
// collected per node)
//   Z(j) = f - c_x (f - f_up) - ax [S^x(down) - S^x],
//   Q(j) = Z(j) + (1 - c_y) [(1 - c_x) S^y(j + 1) + c_x S^y_up(j + 1)],
//   f*(j) = Z(j) + c_y (Q(j - 1) - Q(j)):
// 11 FP64 operations per node.  Rows come in batches of four, by tensor copies
// (three slots per warp) or, at the lattice's edges and where the lattice has no
// tensor maps, by the lanes' loads.
constexpr int A64_WARPS = NT / 32, A64_SLOTS = 3, A64_COLS = 32, A64_OUT = TW / 2;

template <int ORDER, int LIM>
__global__ void __launch_bounds__(NT, 2)
    advect64_kernel(const __grid_constant__ StepArgs<double> P, const __grid_constant__ RowMaps maps) {
  __shared__ __align__(128) double stage[A64_WARPS][A64_SLOTS][RPI][A64_COLS];
  __shared__ unsigned long long bars[A64_WARPS][A64_SLOTS];
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  if (lane == 0) {
    for (int b = 0; b < A64_SLOTS; ++b) mbar_init(&bars[warp][b], 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncwarp();
  previous_step_done();
  const int Lx = P.Lx, Ly = P.Ly;
  unsigned phase = 0;
  bool dead = false;  // a staged batch did not arrive: the results are void, nothing more is staged
  const int sub = P.sub, sub_rows = (P.row_block + sub - 1) / sub;
  const long long tasks = P.items * 32 * sub, step = (long long)gridDim.x * A64_WARPS;
  for (long long t = blockIdx.x + (long long)gridDim.x * warp; t < tasks; t += step) {
    const unsigned part = (unsigned)(t >> 5), item = part / (unsigned)sub;
    const int k = (int)(t >> 1) & 15, half = (int)t & 1;
    const unsigned rb = item / (unsigned)P.nstrip;
    const int strip = (int)(item - rb * (unsigned)P.nstrip);
    const int xs = strip * TW + half * A64_OUT;  // first output column
    const int y0 = (int)rb * P.row_block, ys = y0 + (int)(part - item * sub) * sub_rows;
    const int ye = min(min(Ly, y0 + P.row_block), ys + sub_rows);
    if (xs >= Lx || ys >= ye) continue;
    const VelConst<double>& v = P.v[k];
    const bool right = v.xi_x > 0.0, up = v.xi_y > 0.0;
    const int j = right ? lane : A64_COLS - 1 - lane;  // the lane's staged column
    const int x = xs - 2 + j;
    const double ncx = -v.cx, nax = -0.25 * v.ax, cy = v.cy, b0 = 0.25 * v.qy0, b1 = 0.25 * v.qy1;
    const double* const plane = static_cast<const double*>(P.fin) + (long long)k * P.plane;
    const double* const col = plane + wrapi(x, Lx);
    double* const out = static_cast<double*>(P.fout) + (long long)k * P.plane + x;
    const bool store = j >= 2 && j < 2 + A64_OUT && x < Lx;
    const int start = up ? ys - 2 : ye + 1, dir = up ? 1 : -1;
    const int rows = ye - ys + 3, nb = (rows + RPI - 1) / RPI;
    const bool xin = P.tma_in && xs - 2 >= 0 && xs - 2 + A64_COLS <= Lx;
    // the rows of batch b, lowest first; staged by a tensor copy if inside
    const auto low = [&](int b) { return up ? start + RPI * b : start - RPI * b - (RPI - 1); };
    const auto staged = [&](int b) { return xin && low(b) >= 0 && low(b) + RPI <= Ly; };
    const auto arm = [&](int b) {
      if (b < nb && staged(b) && !dead && lane == 0) {
        unsigned long long* bar = &bars[warp][b % A64_SLOTS];
        mbar_arrive_expect_tx(bar, RPI * A64_COLS * 8);
        tma_load_tile(&stage[warp][b % A64_SLOTS][0][0], maps.m, xs - 2, k, low(b), bar);
      }
    };
    __syncwarp();  // the slots' previous rows have been read
    for (int b = 0; b < A64_SLOTS - 1; ++b) arm(b);
    double F = 0.0, Ry = 0.0, Z = 0.0, Q = 0.0;  // of the row before (Q: of the one before that)
    int m = 0;  // rows done
    for (int b = 0; b < nb; ++b) {
      double in[RPI];
      if (staged(b)) {
        const int s = b % A64_SLOTS;
        if (!dead && !mbar_wait_bounded(&bars[warp][s], phase >> s & 1, 1000000000ULL)) {
          dead = true;
          atomicOr(P.err, 2u);
        }
        phase ^= 1u << s;
#pragma unroll
        for (int i = 0; i < RPI; ++i) in[i] = stage[warp][s][up ? i : RPI - 1 - i][j];
      } else {
#pragma unroll
        for (int i = 0; i < RPI; ++i) {
          const int row = start + dir * (RPI * b + i);
          if (P.walls && (unsigned)row >= (unsigned)Ly)  // wall ghost rows
            in[i] = row < 0 ? v.gbot : v.gtop;
          else
            in[i] = col[(long long)wrap_row(row, Ly) * Lx];
        }
      }
      __syncwarp();  // slot (b + 2) % 3 was read with batch b - 1
      arm(b + A64_SLOTS - 1);
      // each row does what a later one needs of it and no more
#pragma unroll
      for (int i = 0; i < RPI; ++i, ++m) {
        if (m >= rows) break;
        const double f = in[i];
        double Sy = 0.0, Syu = 0.0;
        if constexpr (ORDER == 2) {
          const double r = f - F;
          if (m >= 2) {
            Sy = mc_quad<LIM>(r, Ry, r + Ry);
            Syu = shfl_up1(Sy);
          }
          Ry = r;
        }
        if (m >= 2) {
          // row m - 1's downwind face, and with it row m - 1 itself
          double q = Z;
          if constexpr (ORDER == 2) q = fma(b1, Syu, fma(b0, Sy, q));
          if (m >= 3) {
            const double o = fma(cy, Q - q, Z);
            if (store) out[(long long)(start + dir * (m - 1)) * Lx] = o;
          }
          Q = q;
        }
        if (m >= 1 && m < rows - 1) {
          const double R = f - shfl_up1(f);
          Z = fma(ncx, R, f);
          if constexpr (ORDER == 2) {
            const double Ru = shfl_up1(R);
            const double S = mc_quad<LIM>(R, Ru, R + Ru);
            Z = fma(nax, shfl_dn1(S) - S, Z);
          }
        }
        F = f;
      }
    }
  }
  // after a timed-out wait copies may still be in flight into this CTA's shared
  // memory: wait, bounded, for either phase of each slot
  if (dead)
    for (int b = 0; b < 2 * A64_SLOTS; ++b) mbar_wait_bounded(&bars[warp][b >> 1], b & 1, 1000000000ULL);
}

// ------------------------------------------------- moments and collision
// A block takes a tile of 16 x 8 nodes.  rho* - rho_ref and p^i - p^w of the tile and
// its halo of two nodes are summed into shared memory first (1.9 times the tile's
// nodes, ~30 of the ~270 operations of a node); momentum, force and collision
// follow, one node per thread (two per thread share the row sums of the force
// stencils, 27 operations less per node, but leave half the warps: 128^2 34.2 us per
// step against 25.6, 362^2 142 against 132, 1024^2 964 against 969).  fin holds f*, fout
// receives f^{n+1}.
constexpr int C64_TX = 16, C64_TY = 8, C64_NT = C64_TX * C64_TY;
constexpr int C64_PX = C64_TX + 4, C64_PY = C64_TY + 4;

template <bool DIAG, bool REGU>
__global__ void __launch_bounds__(C64_NT)
    collide64_kernel(const __grid_constant__ StepArgs<double> P) {
  __shared__ double sdr[C64_PY][C64_PX], sph[C64_PY][C64_PX];
  const int Lx = P.Lx, Ly = P.Ly, tid = threadIdx.x;
  const unsigned tx = (unsigned)(Lx + C64_TX - 1) / C64_TX;
  const int by = (int)(blockIdx.x / tx), bx = (int)(blockIdx.x - by * tx);
  const int x0 = bx * C64_TX, y0 = by * C64_TY;
  const double* const fin = static_cast<const double*>(P.fin);
  const long long pl = P.plane;
  previous_step_done();
  for (int e = tid; e < C64_PX * C64_PY; e += C64_NT) {
    const int iy = e / C64_PX, ix = e - iy * C64_PX;
    const int row = y0 - 2 + iy, x = wrapi(x0 - 2 + ix, Lx);
    double f[16];
    if (P.walls && (unsigned)row >= (unsigned)Ly) {  // wall ghost rows keep f^eq(rho_ext, u_wall)
#pragma unroll
      for (int k = 0; k < 16; ++k) f[k] = row < 0 ? P.v[k].gbot : P.v[k].gtop;
    } else {
      const double* src = fin + (long long)wrap_row(row, Ly) * Lx + x;
#pragma unroll
      for (int k = 0; k < 16; ++k) f[k] = src[k * pl];
    }
    double d[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) d[g] = (f[4 * g] + f[4 * g + 2]) + (f[4 * g + 1] + f[4 * g + 3]);
    const double dr = d[0] + (d[1] + (d[2] + d[3])), rho = P.rho_ref + dr, rT = rho * P.Tt;
    sdr[iy][ix] = dr;
    sph[iy][ix] = fma(P.a * rho, rho, fma(rT, rcp(fma(P.b, rho, -1.0)), rT));
  }
  __syncthreads();
  const int ty = tid / C64_TX, ix = tid - ty * C64_TX, x = x0 + ix, y = y0 + ty;
  double mass = 0.0;
  unsigned long long a[6] = {0, 0, 0, 0, 0, 0};
  if (x < Lx && y < Ly) {
    const double* src = fin + (long long)y * Lx + x;
    double f[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) f[k] = src[k * pl];
    const auto load = [&](int k) { return f[k]; };
    const double *ph[5], *dq[5];
#pragma unroll
    for (int b = 0; b < 5; ++b) {
      ph[b] = &sph[ty + b][ix + 2];
      dq[b] = &sdr[ty + b][ix + 2];
    }
    const double rho = P.rho_ref + *dq[2], ir = rcp(rho);
    const NodeConst<One64> C(P);
    double gx, gy, drho, u, v;
    pair_force<One64>(C, ph, dq, ir, gx, gy, drho);
    pair_velocity<One64>(C, load, ir, u, v);
    if (!(rho > 0.0 && rho < 1e30)) atomicOr(P.err, 1u);
    double s1 = P.one_m_omega, rw = rho, cr = 0.0;
    if (P.reservoir) {  // outside R_BC the node is rescaled to rho_ext, s = rho_ext / rho
      const double dx = (double)x - P.cxc, dy = (double)y - P.cyc;
      if (dx * dx + dy * dy > P.rbc2) {
        const double s = P.rho_ext * ir;
        s1 *= s;
        rw *= s;
        cr = P.rho_ref * (s - 1.0) * (REGU ? 1.0 : P.irho_ext);
      }
    }
    double* dst = static_cast<double*>(P.fout) + (long long)y * Lx + x;
    pair_collide<One64, REGU>(P, C, load, [&](int k, double o) { dst[k * pl] = o; }, drho, rho, ir, u,
                              v, gx, gy, s1, rw, cr);
    if (DIAG) {
      mass = rw;
      if (rw < P.diag_thr) {
        const unsigned long long i = (unsigned long long)x, j = (unsigned long long)y;
        a[0] = 1;
        a[1] = i;
        a[2] = j;
        a[3] = i * i;
        a[4] = i * j;
        a[5] = j * j;
      }
    }
  }
  if (DIAG) {  // one add per warp for the mass, per warp with bubble sites for their sums
    const bool any = __ballot_sync(0xffffffffu, a[0] != 0) != 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      mass += __shfl_down_sync(0xffffffffu, mass, o);
      if (any)
#pragma unroll
        for (int q = 0; q < 6; ++q) a[q] += __shfl_down_sync(0xffffffffu, a[q], o);
    }
    if ((tid & 31) == 0) {
      atomicAdd(P.diag_mass, mass);
      if (any)
#pragma unroll
        for (int q = 0; q < 6; ++q) atomicAdd(&P.diag_sums[q], a[q]);
    }
  }
}
