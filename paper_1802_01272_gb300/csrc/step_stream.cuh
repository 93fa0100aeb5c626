// step_stream.cuh -- the fused CTU step for FP32 arithmetic (FP32 and FP16
// storage): included by lbm_kernels.cuh inside namespace ctulbm.
//
// A CTA owns a strip of TW = 56 output columns [56 s, 56 s + 56) and streams
// down a range of rows, four rows (a batch) at a time, over the 64-column
// region [56 s - 4, 56 s + 60): the strip, the two columns of rho* halo the
// force stencil needs on each side, and two more that complete the groups of
// four.  Its eight warps have two roles that run concurrently, one batch
// apart:
//
//  warps 0-3 ADVECT.  Warp q holds the four velocities of sign quadrant q
//   (sgn xi_x, sgn xi_y); the sign of xi_x is a compile-time constant of its code,
//   that of xi_y data.  A lane advects four columns of two velocities (the two
//   with its |xi_x|), row after row, with the row history in registers; a column
//   of the neighbouring group comes from the adjacent lane.  The warp stages its
//   own four planes, half a batch per slot, by tensor copies that its elected
//   lane issues as soon as the slot has been read: no other warp touches its
//   slots, so staging needs no barrier between warps.  The warps with xi_y > 0 stage
//   one row behind the others (see StreamState).  A strip at the periodic x
//   seam is staged by two copies, one per side of the seam.  The advected rows
//   f* go to a ring of ten rows.
//  warps 4-7 COLLIDE.  Warp 4 + r takes row r of the batch, a lane two
//   neighbouring nodes (every operation one packed FP32x2 instruction for the
//   pair): rho*, u*, p^i - p^w of the batch's rows into the moment rings, then,
//   two rows further back, the 5x5 force stencils, the collision of all 16
//   planes, and f^{n+1} by 8-byte stores (28 lanes x 8 bytes = one run of whole
//   sectors per plane).
//
// The roles hand the f* ring over by hardware barriers on which one side only
// arrives; the collide warps have one more per batch among themselves.
//
// What bounds it: instruction issue, then the FMA pipe and shared memory, before
// HBM.  Why two roles: one role per warp keeps the advection's row history out
// of the collision's registers (96 and 64 per thread, three CTAs per SM), lets a
// lane hold twice the work (two velocities, two nodes), which halves the loop,
// barrier and address instructions per node, and replaces three barriers of all
// warps per batch.  Against one kernel body in which all warps advect, then
// collide, with the same operations on every node (30 warp instructions per node;
// now 25.8): 6144^2 FP32 1.25 -> 1.11 ms/step, 2048^2 187 -> 132 us, 1024^2 70 -> 39
// us, 1001 x 777 80 -> 38 us, 4096^2 FP16 660 -> 530 us.  Measured on the way, with
// other sums in the collision (1.08 ms at 6144^2, see group_collide): two CTAs per SM
// with 128 registers, as fast at 1024^2 and 7 % slower at 6144^2; the hand-over by polled mbarriers -3 %;
// the row loop unrolled by four instead of two -9 % and one copy of the advection
// per sign quadrant instead of per sign of xi_x -30 % (instruction fetch); seam
// strips staged by the lanes' 16-byte copies -17 % at 3584 x 2048 (their CTAs were
// the launch's tail).

constexpr int SR = 2;                  // rows per staging slot: half a batch
constexpr int SNS = 2;                 // staging slots per advect warp: the halves of a batch
constexpr int SFR = 10;                // f* ring (and u*): rows B - 4 .. B + 5
constexpr int SMR = 12;                // rho* and p^i - p^w rings: rows B - 6 .. B + 5
constexpr int MC0 = 2, MPP = 60;       // region columns 2 .. 61 of the moments are kept
// Resident CTAs per SM, registers per thread at launch, and after the roles have
// traded them: the advect warps take what the collide warps give up or the other way
// round, no more (a larger sum would wait for registers forever; the host refuses a
// kernel that was not compiled to LAUNCH).  The regularised collision holds the
// polynomial and the group sums at once: at 64 registers it spills 240 bytes.
template <bool REGU>
struct StreamRegs {
  static constexpr int CTAS = REGU ? 2 : 3, LAUNCH = REGU ? 128 : 80;
  static constexpr int ADVECT = REGU ? 104 : 96, COLLIDE = REGU ? 152 : 64;
  static_assert(ADVECT + COLLIDE == 2 * LAUNCH, "");
};
constexpr unsigned WAIT_NS = 1000000000u;

template <typename ST>
struct StreamLayout {
  // Half rows must be whole 16-byte chunks from a 16-byte boundary: they start
  // four columns before the region and end four after it.
  static constexpr int SOFF = sizeof(ST) == 2 ? 4 : 0;
  static constexpr int SCOL = REG + 2 * SOFF;
  static constexpr int SLOT = SR * 4 * SCOL;  // a slot: [row][group][column] of one quadrant
  static constexpr int STAGE = 4 * SNS * SLOT;
};

template <typename ST>
struct StreamSmem {
  using L = StreamLayout<ST>;
  ST* stage;                // [warp][SNS][SR][4][SCOL]
  float* fs;                // [SFR][16][REG]
  float *drho, *phi;        // [SMR][MPP]
  float *ux, *uy;           // [SFR][MPP]
  unsigned long long* dsums;    // [6] fused diagnostics: per-CTA bubble-site sums
  double* mass;                 // [128] and each collide thread's sum of rho - rho_ref
  unsigned long long *full;     // [4][SNS] a staged batch has landed
  int* abort;                   // [4] a bounded wait of this advect warp timed out
  static constexpr size_t bytes() {
    return 128 + sizeof(ST) * L::STAGE + 4 * (SFR * 16 * REG + 2 * (SMR + SFR) * MPP) +
           8 * (6 + 128 + 4 * SNS) + 16;
  }
  __device__ explicit StreamSmem(unsigned char* raw) {
    raw += (128u - (smem_u32(raw) & 127u)) & 127u;  // tensor copies want 128-byte aligned tiles
    stage = reinterpret_cast<ST*>(raw);
    fs = reinterpret_cast<float*>(stage + L::STAGE);
    drho = fs + SFR * 16 * REG;
    phi = drho + SMR * MPP;
    ux = phi + SMR * MPP;
    uy = ux + SFR * MPP;
    dsums = reinterpret_cast<unsigned long long*>(uy + SFR * MPP);
    mass = reinterpret_cast<double*>(dsums + 6);
    full = dsums + 6 + 128;
    abort = reinterpret_cast<int*>(full + 4 * SNS);
  }
  __device__ __forceinline__ void init(bool diag) const {
    if (diag && threadIdx.x < 128) mass[threadIdx.x] = 0.0;
    if (threadIdx.x == 0) {
      for (int t = 0; t < 6; ++t) dsums[t] = 0ULL;
      for (int b = 0; b < 4; ++b) abort[b] = 0;
      for (int b = 0; b < 4 * SNS; ++b) mbar_init(full + b, 1);
      asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    __syncthreads();
  }
};

// Barriers and copies below take shared-memory addresses (smem_u32 once, not at
// each use).
__device__ __forceinline__ bool bar_try_wait(unsigned bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Waits for a phase of `bar`, at most WAIT_NS; false if it was not seen to
// complete.  A timeout sets error bit 1 and the warp's abort flag, after which
// none of its waits waits (the results are void): every role runs to its end.
// Warp-collective, and the whole warp gets one answer: a lane's clock may pass the
// limit while its neighbours see the phase complete, and warp-wide instructions
// follow under the answer.
__device__ __forceinline__ bool stream_wait(unsigned bar, unsigned parity, int* abort,
                                            unsigned* err) {
  bool ok = bar_try_wait(bar, parity);
  if (!ok) {
    const unsigned long long t0 = global_ns();
#pragma unroll 1
    for (;;) {
      ok = bar_try_wait(bar, parity);
      if (ok || *reinterpret_cast<volatile int*>(abort)) break;
      if (global_ns() - t0 > WAIT_NS) {
        *reinterpret_cast<volatile int*>(abort) = 1;
        atomicOr(err, 2u);
        break;
      }
    }
  }
  return __all_sync(0xffffffffu, ok);
}
// One lane of the (converged) warp: a predicate the compiler knows to hold for
// a single thread, so that a tensor copy under it needs no loop over lanes.
__device__ __forceinline__ bool elect_one() {
  unsigned p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ void bar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void bar_arrive_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes)
               : "memory");
}
// Hardware barriers between the roles: one role arrives and goes on, the other
// waits.  F* + p: f* rows of a batch of parity p written; FREE + p: read by the
// batch's collision; COLLIDE: among the collide warps.  (Polling mbarriers for
// these hand-overs took a seventh of the issue slots.)
enum { BAR_FULL = 1, BAR_FREE = 3, BAR_COLLIDE = 5 };
__device__ __forceinline__ void role_wait(int id) {
  asm volatile("barrier.sync %0, 256;\n" ::"r"(id) : "memory");
}
__device__ __forceinline__ void role_arrive(int id) {
  asm volatile("barrier.arrive %0, 256;\n" ::"r"(id) : "memory");
}
__device__ __forceinline__ void collide_barrier() {
  asm volatile("barrier.sync %0, 128;\n" ::"r"((int)BAR_COLLIDE) : "memory");
}
__device__ __forceinline__ void tma_load_quadrant(unsigned dst, const CUtensorMap* map, int x, int q,
                                                  int y, unsigned bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cta.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5}], [%6];\n" ::"r"(dst),
      "l"(map), "r"(x), "r"(q), "r"(0), "r"(y), "r"(bar)
      : "memory");
}

// A segment: rows [ys, ye) of one strip of one lattice.  The feeds list a
// CTA's segments in order; every role walks its own copy.
struct Segment {
  int lattice, strip, ys, ye;
  __device__ int batches() const { return WARM + (ye - ys + RPI - 1) / RPI; }
};

// Work items (row block, strip), row-block-major: CTAs that run at the same
// time work on the same rows of neighbouring strips, so the halo columns they
// share and the output lines they both write meet in L2.  CTA c takes items
// c, c + grid, ...: the host sizes the row blocks so that the items fill whole
// rounds, and a fixed assignment needs no exchange between the roles.
struct SingleFeed {
  const StepArgs<float>& P;
  const RowMaps& M;
  int rb, strip, drb, dstrip;  // the next item, and the step of gridDim.x items
  int blocks;
  __device__ SingleFeed(const StepArgs<float>& p, const RowMaps& m) : P(p), M(m) {
    const unsigned n = (unsigned)P.nstrip;
    rb = (int)(blockIdx.x / n);
    strip = (int)(blockIdx.x - rb * n);
    drb = (int)(gridDim.x / n);
    dstrip = (int)(gridDim.x - drb * n);
    blocks = (int)((unsigned)(P.Ly + P.row_block - 1) / (unsigned)P.row_block);
  }
  __device__ const StepArgs<float>& args(const Segment&) const { return P; }
  __device__ const CUtensorMap* maps(const Segment&) const { return M.m; }
  __device__ bool next(Segment& s) {
    s.lattice = 0;
    s.strip = strip;
    s.ys = rb * P.row_block;
    s.ye = s.ys + min(P.row_block, P.Ly - s.ys);
    const bool more = rb < blocks;
    rb += drb;
    strip += dstrip;
    if (strip >= P.nstrip) {
      strip -= P.nstrip;
      ++rb;
    }
    return more;
  }
};
struct BatchFeed {
  const BatchArgs<float>& B;
  long long item;
  int i = 0;
  __device__ explicit BatchFeed(const BatchArgs<float>& b) : B(b), item(blockIdx.x) {}
  __device__ const StepArgs<float>& args(const Segment& s) const { return B.L[s.lattice]; }
  __device__ const CUtensorMap* maps(const Segment& s) const { return B.maps[s.lattice].m; }
  __device__ bool next(Segment& s) {
    if (item >= B.item_start[B.count]) return false;
    while (B.item_start[i + 1] <= item) ++i;
    const StepArgs<float>& P = B.L[i];
    const unsigned local = (unsigned)(item - B.item_start[i]);
    const unsigned rb = local / (unsigned)P.nstrip;
    // known to be warp-uniform: what is read by them then comes by uniform loads
    // (lattices of 256^2 to 2048^2 together 296 -> 271 us per step)
    const auto uniform = [](int v) { return __shfl_sync(0xffffffffu, v, 0); };
    s.lattice = uniform(i);
    s.strip = uniform((int)(local - rb * (unsigned)P.nstrip));
    s.ys = uniform((int)rb * P.row_block);
    s.ye = uniform(min(P.Ly, s.ys + P.row_block));
    item += gridDim.x;
    return true;
  }
};

// ------------------------------------------------------------- advection
// Row history of four columns (two pairs) of one velocity.  Z is the x part of
// the update, Z = f - c_x (f - f(i - s_x)) - ax dS^x; the update of row j is
//   Z(j) + c_y (Z(j - s_y) - Z(j)) + by0 dS^y(i) + by1 dS^y(i - s_x),
// dS^y = S^y(j + 1) - S^y(j) (Sec. II C 2 collected per node); a uniform state is
// kept exactly.  When row n arrives, S^y is known up to row n for s_y > 0 and row
// n - 1 for s_y < 0, which makes row n - 1 or n - 2 complete: a warp with s_y > 0
// stages one row behind, so that all emit the same rows.  The sign of xi_y is data
// (cy carries it), and the four quadrants run two copies of the code instead of
// four (the instruction cache holds the roles' loops; four copies cost a third of
// the speed).
struct StreamState {
  float2 F[2], Ry[2], Sy[2];  // f, R^y and S^y of the row before
  float2 Z1[2], Z2[2];        // Z of the two rows before
};
struct StreamConst {
  float2 cy, b0;  // s_y c_y; weights of dS^y(i) and (b1) dS^y(i - s_x)
  float b1;
};
struct StreamConstX {
  float2 ncx, nax, q;  // -s_x c_x, -ax, 1/4
};

// One staged row n of a velocity with s_x = SX, own columns (0, 1) in
// B0 and (2, 3) in B1; out receives the advected row n - 1 (sy) or n - 2.  All lanes of a
// warp call it together.  The two edge lanes of a velocity's 16 get no useful
// neighbours: region columns 0, 1, 62, 63 come out void and feed no output.
template <int SX, int ORDER, int LIM>
__device__ __forceinline__ void stream_row(StreamState& s, float2 B0, float2 B1,
                                           const StreamConstX& c, const StreamConst& k, bool sy,
                                           float2 (&out)[2]) {
  float2 Z[2];
  float S0, S1, S2, S3, S4;
  if constexpr (SX > 0) {
    // columns -2, -1; R^x(i) = f(i) - f(i-1), S^x(i) from R(i) and R(i-1), whose
    // quarter sum is (f(i) - f(i-2))/4
    const float Ay = shfl_up1(B1.y);
    const float R0 = B0.x - Ay, R1 = B0.y - B0.x, R2 = B1.x - B0.y, R3 = B1.y - B1.x;
    Z[0] = fma2(c.ncx, make_float2(R0, R1), B0);
    Z[1] = fma2(c.ncx, make_float2(R2, R3), B1);
    if constexpr (ORDER == 2) {
      const float Ax = shfl_up1(B1.x);
      const float Rm = Ay - Ax;
      const float2 h01 = mul2(c.q, sub2(B0, make_float2(Ax, Ay))), h23 = mul2(c.q, sub2(B1, B0));
      S0 = mc_half<LIM>(R0, Rm, h01.x);
      S1 = mc_half<LIM>(R1, R0, h01.y);
      S2 = mc_half<LIM>(R2, R1, h23.x);
      S3 = mc_half<LIM>(R3, R2, h23.y);
      S4 = shfl_dn1(S0);
    }
  } else {
    // columns 4, 5; S^x(i) from R(i) and R(i+1), taken at columns 1 .. 4
    const float Ex = shfl_dn1(B0.x);
    const float R1 = B0.y - B0.x, R2 = B1.x - B0.y, R3 = B1.y - B1.x, R4 = Ex - B1.y;
    Z[0] = fma2(c.ncx, make_float2(R1, R2), B0);
    Z[1] = fma2(c.ncx, make_float2(R3, R4), B1);
    if constexpr (ORDER == 2) {
      const float Ey = shfl_dn1(B0.y);
      const float R5 = Ey - Ex;
      const float2 h12 = mul2(c.q, make_float2(R1 + R2, R2 + R3));
      const float2 h34 = mul2(c.q, make_float2(R3 + R4, R4 + R5));
      S1 = mc_half<LIM>(R1, R2, h12.x);
      S2 = mc_half<LIM>(R2, R3, h12.y);
      S3 = mc_half<LIM>(R3, R4, h34.x);
      S4 = mc_half<LIM>(R4, R5, h34.y);
      S0 = shfl_up1(S4);
    }
  }
  if constexpr (ORDER == 2) {
    Z[0] = fma2(c.nax, make_float2(S1 - S0, S2 - S1), Z[0]);
    Z[1] = fma2(c.nax, make_float2(S3 - S2, S4 - S3), Z[1]);
  }

  const float2 B[2] = {B0, B1};
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    // cy carries the sign of s_y: Z(j) + c_y (Z(j - s_y) - Z(j)) for either
    const float2 D = sub2(s.Z2[m], s.Z1[m]);
    out[m] = fma2(k.cy, D, sy ? s.Z1[m] : s.Z2[m]);
  }
  if constexpr (ORDER == 2) {
    float2 dS[2];
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const float2 Ry = sub2(B[m], s.F[m]);
      const float2 h = mul2(c.q, add2(Ry, s.Ry[m]));
      // s_y > 0: S^y(n), from R^y(n) with the upwind jump R^y(n - 1); s_y < 0:
      // S^y(n - 1), from R^y(n - 1) with R^y(n) (the MC form is symmetric in the two)
      const float2 a = LIM == 0 || sy ? Ry : s.Ry[m], b = LIM == 0 || sy ? s.Ry[m] : Ry;
      const float2 Sy = make_float2(mc_half<LIM>(a.x, b.x, h.x), mc_half<LIM>(a.y, b.y, h.y));
      dS[m] = sub2(Sy, s.Sy[m]);
      s.Ry[m] = Ry;
      s.Sy[m] = Sy;
    }
    // dS^y one column upwind in x
    const float e = SX > 0 ? shfl_up1(dS[1].y) : shfl_dn1(dS[0].x);
    const float u[4] = {SX > 0 ? e : dS[0].y, SX > 0 ? dS[0].x : dS[1].x,
                        SX > 0 ? dS[0].y : dS[1].y, SX > 0 ? dS[1].x : e};
#pragma unroll
    for (int m = 0; m < 2; ++m) {
      const float2 t = fma2(k.b0, dS[m], out[m]);
      out[m] = make_float2(fmaf(k.b1, u[2 * m], t.x), fmaf(k.b1, u[2 * m + 1], t.y));
    }
  }
#pragma unroll
  for (int m = 0; m < 2; ++m) {
    s.F[m] = B[m];
    s.Z2[m] = s.Z1[m];
    s.Z1[m] = Z[m];
  }
}

__device__ __forceinline__ StreamConst stream_const(const VelConst<float>& v, bool sy) {
  StreamConst c;
  c.cy = dup2(sy ? v.cy : -v.cy);
  c.b0 = dup2(v.by0);
  c.b1 = v.by1;
  return c;
}

// How a strip's staged columns lie in a slot.  Away from the periodic x seam:
// [row][group][SCOL].  The first and the last strip cross the seam: their
// columns are two runs of the lattice row, [0, na) and [na, SCOL), each staged by
// its own tensor copy and so each with its own pitch:
// [row][group][na], then [row][group][SCOL - na].
template <typename ST>
struct Split {
  static constexpr int SCOL = StreamLayout<ST>::SCOL;
  int na;  // SCOL: one run
  __device__ __forceinline__ int pitch(int j) const { return j < na ? na : SCOL - na; }
  __device__ __forceinline__ int at(int row_group, int j) const {
    return j < na ? row_group * na + j : SR * 4 * na + row_group * (SCOL - na) + j - na;
  }
};
// Columns before the seam of the strip whose staging starts at x0.
template <typename ST, bool VEC>
__device__ __forceinline__ Split<ST> split_of(int x0, int Lx) {
  constexpr int SCOL = StreamLayout<ST>::SCOL;
  if (!VEC) return {SCOL};
  return {x0 < 0 ? -x0 : min(SCOL, Lx - x0)};
}

// The slot's phase: completed by this arrival and, when the lanes have copies in
// flight, by their landing.
__device__ __forceinline__ void lanes_arrive(unsigned bar) {
  asm volatile("cp.async.mbarrier.arrive.shared.b64 [%0];\n" ::"r"(bar) : "memory");
  __syncwarp();
  if (elect_one()) bar_arrive(bar);
}
// Staging by the lanes' own asynchronous copies of 16-byte chunks (Lx and x0 are
// multiples of a chunk), for slots whose rows wrap in y or are wall ghosts (which
// the advect warp fills in): tensor copies do neither.  fin: plane q.
template <typename ST>
static __device__ __forceinline__ void stage_chunks(ST* dst, unsigned bar, Split<ST> split,
                                                    const ST* fin, long long plane, int x0, int r0,
                                                    int Lx, int Ly, int walls) {
  constexpr int E = 16 / (int)sizeof(ST), N = StreamLayout<ST>::SCOL / E;
  const int lane = threadIdx.x & 31;
  const auto copy = [&](int rg, int x, int j, const ST* row) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(dst + split.at(rg, j))),
                 "l"(row + 4 * (rg & 3) * plane + x)
                 : "memory");
  };
#pragma unroll
  for (int r = 0; r < SR; ++r) {
    if (walls && (unsigned)(r0 + r) >= (unsigned)Ly) continue;
    const ST* row = fin + (long long)wrap_row(r0 + r, Ly) * Lx;
#pragma unroll
    for (int e = lane; e < 4 * N; e += 32) {
      const int grp = e / N, j = (e - grp * N) * E, x = x0 + j;
      copy(4 * r + grp, x < 0 ? x + Lx : (x >= Lx ? x - Lx : x), j, row);
    }
  }
  lanes_arrive(bar);
}
// Staging of a lattice without tensor maps, value by value (half values, for
// which there is no asynchronous copy, by loads): a lane takes columns lane and
// lane + 32 of the region, at lattice columns xa and xb.
template <typename ST>
static __device__ __forceinline__ void stage_values(ST* dst, unsigned bar, const ST* fin,
                                                    long long plane, int xa, int xb, int r0, int Lx,
                                                    int Ly, int walls) {
  using L = StreamLayout<ST>;
  dst += L::SOFF + (threadIdx.x & 31);
#pragma unroll 1
  for (int r = 0; r < SR; ++r) {
    const int row = r0 + r;
    if (walls && (unsigned)row >= (unsigned)Ly) continue;
    const ST* pa = fin + (long long)wrap_row(row, Ly) * Lx + xa;
    const ST* pb = pa + (xb - xa);
    ST* d = dst + r * 4 * L::SCOL;
    if constexpr (sizeof(ST) == 4) {
      const unsigned du = smem_u32(d);
#pragma unroll
      for (int grp = 0; grp < 4; ++grp, pa += 4 * plane, pb += 4 * plane) {
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(du + 4 * grp * L::SCOL), "l"(pa)
                     : "memory");
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(du + 4 * grp * L::SCOL + 128),
                     "l"(pb)
                     : "memory");
      }
    } else {
      ST v[8];
#pragma unroll
      for (int grp = 0; grp < 4; ++grp) {
        v[2 * grp] = pa[4 * grp * plane];
        v[2 * grp + 1] = pb[4 * grp * plane];
      }
#pragma unroll
      for (int grp = 0; grp < 4; ++grp) {
        d[grp * L::SCOL] = v[2 * grp];
        d[grp * L::SCOL + 32] = v[2 * grp + 1];
      }
    }
  }
  lanes_arrive(bar);
}

// The staging of one advect warp: its four planes' batches in the order of the
// CTA's segments.  Slot h holds rows 2h, 2h + 1 of a batch and takes those of the
// next batch as soon as the warp has read it.  Warp-collective.
template <typename ST, bool VEC, typename Feed>
struct Stager {
  using L = StreamLayout<ST>;
  static constexpr unsigned BYTES = L::SLOT * (unsigned)sizeof(ST);
  Feed feed;
  Segment seg;
  int left;          // batches of seg still to stage (0: none left at all)
  int r0, x0;        // the next one's first row; the segment's first staged column
  Split<ST> split;   // of the segment
  int mixed = 0;     // the lanes' copies may still be in the slots
  int xa = 0, xb = 0;  // without tensor maps: the lane's two lattice columns
  const int q;       // quadrants 0 and 1 (s_y > 0) stage one row behind the others
  ST* const base;    // the warp's slots
  const unsigned base_u, full;  // their address and their mbarriers'

  __device__ Stager(const Feed& f, const StreamSmem<ST>& S, int warp)
      : feed(f), q(warp), base(S.stage + warp * (SNS * L::SLOT)), base_u(smem_u32(base)),
        full(smem_u32(S.full + warp * SNS)) {
    open();
  }
  __device__ __forceinline__ void open() {
    left = feed.next(seg) ? seg.batches() : 0;
    r0 = seg.ys - RPI - (q < 2);
    x0 = seg.strip * TW - XOFF - L::SOFF;
    split = split_of<ST, VEC>(x0, feed.args(seg).Lx);
    if (!VEC && left > 0) {
      xa = wrapi(x0 + L::SOFF + (int)(threadIdx.x & 31), feed.args(seg).Lx);
      xb = wrapi(x0 + L::SOFF + 32 + (int)(threadIdx.x & 31), feed.args(seg).Lx);
    }
  }
  // Stage half h of the next batch into slot h, which the warp has read.
  __device__ __forceinline__ void arm(int h) {
    if (left == 0) return;
    const StepArgs<float>& P = feed.args(seg);
    const unsigned bar = full + 8 * h;
    const int row = r0 + SR * h;
    if (VEC && row >= 0 && row + SR <= P.Ly) {
      if (elect_one()) {
        const unsigned dst = base_u + h * BYTES;
        const CUtensorMap* tm = feed.maps(seg);
        if (mixed > 0) fence_proxy_async();  // the lanes' copies before this one
        bar_arrive_expect(bar, BYTES);
        if (split.na == L::SCOL) {
          tma_load_quadrant(dst, tm, x0, q, row, bar);
        } else {
          tm += x0 < 0 ? 1 : 3;
          const unsigned dst2 = dst + SR * 4 * (unsigned)sizeof(ST) * split.na;
          tma_load_quadrant(dst, tm, x0 < 0 ? P.Lx + x0 : x0, q, row, bar);
          tma_load_quadrant(dst2, tm + 1, 0, q, row, bar);
        }
      }
    } else {
      const ST* fin = static_cast<const ST*>(P.fin) + (long long)q * P.plane;
      if constexpr (VEC)
        stage_chunks<ST>(base + h * L::SLOT, bar, split, fin, P.plane, x0, row, P.Lx, P.Ly, P.walls);
      else
        stage_values<ST>(base + h * L::SLOT, bar, fin, P.plane, xa, xb, row, P.Lx, P.Ly, P.walls);
      mixed = 2;
    }
  }
  __device__ __forceinline__ void next() {  // both halves of the batch are staged
    if (left == 0) return;
    r0 += RPI;
    --mixed;
    if (--left == 0) open();
  }
};

// After a timed-out wait copies may still be in flight into this CTA's shared
// memory: wait, bounded, for either phase of each of the warp's slots.
static __device__ __forceinline__ void drain_slots(unsigned full, int* abort) {
  if (!*reinterpret_cast<volatile int*>(abort)) return;
#pragma unroll 1
  for (int b = 0; b < 2 * SNS; ++b) {
    const unsigned long long t0 = global_ns();
    while (!bar_try_wait(full + 8 * (b >> 1), b & 1) && global_ns() - t0 < WAIT_NS) {
    }
  }
}

template <int SX, int ORDER, int LIM, typename ST, bool VEC, typename Feed>
__device__ __forceinline__ void advect_role(Feed feed, const StreamSmem<ST>& S, int q) {
  const bool sy = q < 2;  // quadrants (+,+), (-,+), (-,-), (+,-)
  using L = StreamLayout<ST>;
  const int lane = threadIdx.x & 31, h = lane >> 4, col = 4 * (lane & 15);
  Stager<ST, VEC, Feed> stager(feed, S, q);
#pragma unroll 1
  for (int i = 0; i < SNS; ++i) stager.arm(i);
  stager.next();
  // this lane's velocities: groups h and h + 2 (equal |xi_x|) of the quadrant
  float* const dst0 = S.fs + (4 * h + q) * REG + col;
  constexpr int D2 = 8 * REG;  // f* ring: group h + 2
  unsigned g = 0;  // batches so far
  int ring = 0;
  Segment seg;
  while (feed.next(seg)) {
    const StepArgs<float>& P = feed.args(seg);
    const VelConst<float>&va = P.v[4 * h + q], &vb = P.v[4 * h + 8 + q];
    const StreamConstX cx = {dup2(SX > 0 ? -va.cx : va.cx), dup2(-va.ax), dup2(0.25f)};
    const StreamConst ca = stream_const(va, sy), cb = stream_const(vb, sy);
    StreamState sa, sb;
    memset(&sa, 0, sizeof(sa));
    memset(&sb, 0, sizeof(sb));
    const int Ly = P.Ly, walls = P.walls;
    const Split<ST> split = split_of<ST, VEC>(seg.strip * TW - XOFF - L::SOFF, P.Lx);
    const ST* const src0 = stager.base + split.at(h, L::SOFF + col);
    const int pitch = split.pitch(L::SOFF + col);
    int n = seg.ys - RPI - sy;  // first staged row of the half batch
#pragma unroll 1
    for (int it = seg.batches(); it > 0; --it, ++g) {
      // the ring rows this batch writes were last read by the collision of g - 2
      if (g >= 2) role_wait(BAR_FREE + (g & 1));
#pragma unroll 1
      for (int i = 0; i < SNS; ++i, n += SR) {
        if (!stream_wait(stager.full + 8 * i, g & 1, S.abort + q, P.err))
          stager.left = 0;  // void: nothing more is staged
        const ST* src = src0 + i * L::SLOT;
        float* dst = dst0 + ring * (16 * REG);
        const bool edge = walls && (n < 2 || n + SR > Ly);
        if (edge) {  // wall ghost rows hold f^eq(rho_ext, u_wall)
#pragma unroll 1
          for (int r = 0; r < SR; ++r) {
            if (n + r >= 0 && n + r < Ly) continue;
            ST* d = const_cast<ST*>(src) + r * 4 * pitch;
            const float ga = n < 0 ? va.gbot : va.gtop, gb = n < 0 ? vb.gbot : vb.gtop;
            for (int m = 0; m < 4; ++m) d[m] = to_store<ST, float>(ga);
            for (int m = 0; m < 4; ++m) d[2 * pitch + m] = to_store<ST, float>(gb);
          }
          fence_proxy_async();  // before later tensor copies into the slot
        }
#pragma unroll
        for (int r = 0; r < SR; ++r) {
          float2 a0, a1, b0, b1;
          sload4p<ST>(src + r * 4 * pitch, a0, a1);
          sload4p<ST>(src + (r * 4 + 2) * pitch, b0, b1);
          float2 oa[2], ob[2];
          stream_row<SX, ORDER, LIM>(sa, a0, a1, cx, ca, sy, oa);
          stream_row<SX, ORDER, LIM>(sb, b0, b1, cx, cb, sy, ob);
          float* d = dst + r * (16 * REG);
          *reinterpret_cast<float4*>(d) = make_float4(oa[0].x, oa[0].y, oa[1].x, oa[1].y);
          *reinterpret_cast<float4*>(d + D2) = make_float4(ob[0].x, ob[0].y, ob[1].x, ob[1].y);
        }
        if (edge) {  // ... also after the advection
#pragma unroll 1
          for (int r = 0; r < SR; ++r) {
            const int a = n - 2 + sy + r;
            if (a >= 0 && a < Ly) continue;
            float* d = dst + r * (16 * REG);
            const float ga = a < 0 ? va.gbot : va.gtop, gb = a < 0 ? vb.gbot : vb.gtop;
            for (int m = 0; m < 4; ++m) d[m] = ga;
            for (int m = 0; m < 4; ++m) d[D2 + m] = gb;
          }
        }
        __syncwarp();
        stager.arm(i);
        ring = ring == SFR - SR ? 0 : ring + SR;
      }
      role_arrive(BAR_FULL + (g & 1));
      stager.next();
    }
  }
  for (int i = 0; g > 0 && i < 2; ++i, ++g) role_wait(BAR_FREE + (g & 1));  // the last two batches' arrivals
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  if (VEC) drain_slots(stager.full, S.abort + q);
}

// ------------------------------------------------- moments and collision
template <typename ST, bool VEC, bool DIAG, bool REGU, typename Feed>
__device__ __forceinline__ void collide_role(Feed feed, const StreamSmem<ST>& S, int w,
                                             double& dmass) {
  const int lane = threadIdx.x & 31;
  const int cm = 2 * lane;         // moments: region columns cm, cm + 1
  const int cc = XOFF + 2 * lane;  // collision: lanes 0 .. 27
  unsigned g = 0;
  int ring = 0, mring = 0;  // ring rows of row B - 2
  Segment seg;
  while (feed.next(seg)) {
    const StepArgs<float>& P = feed.args(seg);
    const int nit = seg.batches(), x4 = seg.strip * TW + 2 * lane;
    const NodeConst<Pair32> C(P);
#pragma unroll 1
    for (int it = 0; it < nit; ++it, ++g) {
      role_wait(BAR_FULL + (g & 1));
      const int c0 = seg.ys + RPI * (it - WARM);  // first output row of this batch
      // moments of row B - 2 + w (those of a segment's first batch are void: a branch
      // around them would give the loop a second copy to fetch)
      int row = ring + w;
      row = row >= SFR ? row - SFR : row;
      const float* src = S.fs + row * (16 * REG) + cm;
      float2 dr, ux, uy, phi;
      pair_moments<Pair32>(
          P, [&](int k) { return *reinterpret_cast<const float2*>(src + k * REG); }, dr, ux, uy,
          phi);
      if (cm >= MC0 && cm < MC0 + MPP) {
        const int m = (mring + w) * MPP + cm - MC0, mu = row * MPP + cm - MC0;
        *reinterpret_cast<float2*>(S.drho + m) = dr;
        *reinterpret_cast<float2*>(S.phi + m) = phi;
        *reinterpret_cast<float2*>(S.ux + mu) = ux;
        *reinterpret_cast<float2*>(S.uy + mu) = uy;
      }
      if (it >= WARM) {
        collide_barrier();
        const int c = c0 + w;  // this warp's row
        int bubble = 0;          // fused diagnostics: which of the two nodes are bubble sites
        if (lane < TW / 2) {
          const float *ph[5], *dq[5];
#pragma unroll
          for (int b = 0; b < 5; ++b) {  // rows c - 2 .. c + 2 = (B - 2 + w) - 4 .. + 0
            const unsigned o = (unsigned)(mring + w + b + SMR - 4) * MPP;
            const unsigned r = min(o, o - SMR * MPP) + cc - MC0;  // mod SMR rows
            ph[b] = S.phi + r;
            dq[b] = S.drho + r;
          }
          int frow = ring + SFR - 2 + w;
          frow = frow >= SFR ? frow - SFR : frow;
          const int oc = frow * MPP + cc - MC0;
          const float2 rho = add2(dup2(P.rho_ref), *reinterpret_cast<const float2*>(dq[2]));
          const float2 ir = make_float2(rcp(rho.x), rcp(rho.y));
          float2 gx, gy, drho;
          pair_force<Pair32>(C, ph, dq, ir, gx, gy, drho);
          const float2 u = *reinterpret_cast<const float2*>(S.ux + oc);
          const float2 v = *reinterpret_cast<const float2*>(S.uy + oc);
          const bool in0 = c < seg.ye && x4 < P.Lx, in1 = c < seg.ye && x4 + 1 < P.Lx;
          if ((in0 && !(rho.x > 0.0f && rho.x < 1e30f)) ||
              (in1 && !(rho.y > 0.0f && rho.y < 1e30f)))
            atomicOr(P.err, 1u);
          // outside R_BC the density reservoir rescales the node to rho_ext, s = rho_ext / rho
          const float dx0 = (float)x4 - P.cxc, dx1 = (float)(x4 + 1) - P.cxc, dy = (float)c - P.cyc;
          float2 s = dup2(1.0f);
          if (P.reservoir && dx0 * dx0 + dy * dy > P.rbc2) s.x = P.rho_ext * ir.x;
          if (P.reservoir && dx1 * dx1 + dy * dy > P.rbc2) s.y = P.rho_ext * ir.y;
          const float2 rw = mul2(s, rho);  // the density after the step
          if (DIAG) {
            // The mass goes to FP64 row by row, in shared memory: a sum of many rows would
            // round too much in FP32, and held in registers it costs the loop spills (6144^2
            // with fused diagnostics 1359 -> 1260 us).  A density that is not one (flagged
            // above) counts as none.
            const bool ok0 = in0 && rw.x >= 0.0f, ok1 = in1 && rw.y >= 0.0f;
            S.mass[threadIdx.x & 127] += (double)((in0 ? (ok0 ? rw.x : 0.0f) - P.rho_ref : 0.0f) +
                                                  (in1 ? (ok1 ? rw.y : 0.0f) - P.rho_ref : 0.0f));
            bubble = (ok0 && rw.x < P.diag_thr ? 1 : 0) | (ok1 && rw.y < P.diag_thr ? 2 : 0);
          }
          const float* fsrc = S.fs + frow * (16 * REG) + cc;
          auto load = [&](int k) { return *reinterpret_cast<const float2*>(fsrc + k * REG); };
          // plane k of the pair: one widening multiply-add per store
          char* const dst0 = static_cast<char*>(P.fout) +
                             (unsigned long long)((unsigned)c * (unsigned)P.Lx + (unsigned)x4) * sizeof(ST);
          const auto at = [&](int k) {
            return reinterpret_cast<ST*>(
                dst0 + (unsigned long long)(unsigned)P.plane * (unsigned)(k * sizeof(ST)));
          };
          const auto put = [&](int k, float2 o) {
            if constexpr (VEC) {  // Lx is even: a pair is inside or outside
              if (in0) store_pair(at(k), o);
            } else {
              if (in0) at(k)[0] = to_store<ST, float>(o.x);
              if (in1) at(k)[1] = to_store<ST, float>(o.y);
            }
          };
          if constexpr (REGU) {
            pair_collide<Pair32, REGU>(P, C, load, put, drho, rho, ir, u, v, gx, gy,
                                       mul2(dup2(P.one_m_omega), s), rw,
                                       mul2(dup2(P.rho_ref), sub2(s, dup2(1.0f))));
          } else if (P.reservoir) {
            // the stored deviation becomes s f + w_k rho_ref (s - 1)
            const float2 s_1 = sub2(s, dup2(1.0f));
            group_collide(P, C, load, [&](int k, float2 o) {
              const int grp = k >> 2, cl = grp == 0 ? 0 : (grp == 3 ? 2 : 1);
              put(k, fma2(s, o, mul2(dup2(P.w[cl] * P.rho_ref), s_1)));
            }, drho, rho, ir, u, v, gx, gy);
          } else {
            group_collide(P, C, load, put, drho, rho, ir, u, v, gx, gy);
          }
        }
        if (DIAG && __ballot_sync(0xffffffffu, bubble != 0)) {  // bubble sites are rare
          unsigned long long a[6] = {0, 0, 0, 0, 0, 0};
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            if (bubble >> e & 1) {
              const unsigned long long i = (unsigned long long)(x4 + e), j = (unsigned long long)c;
              a[0] += 1;
              a[1] += i;
              a[2] += j;
              a[3] += i * i;
              a[4] += i * j;
              a[5] += j * j;
            }
          }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
            for (int t = 0; t < 6; ++t) a[t] += __shfl_down_sync(0xffffffffu, a[t], o);
          }
          if (lane == 0) {
#pragma unroll
            for (int t = 0; t < 6; ++t) atomicAdd(&S.dsums[t], a[t]);
          }
        }
      }
      role_arrive(BAR_FREE + (g & 1));
      ring = ring >= SFR - RPI ? ring - (SFR - RPI) : ring + RPI;
      mring = mring == SMR - RPI ? 0 : mring + RPI;
    }
  }
  if (DIAG) dmass = S.mass[threadIdx.x & 127];
}

template <int FROM, int TO>
__device__ __forceinline__ void role_registers() {
  if constexpr (TO < FROM)
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(TO));
  else
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(TO));
}

template <int ORDER, int LIM, typename ST, bool VEC, bool DIAG, bool REGU, typename Feed>
__device__ __forceinline__ void stream_roles(const Feed& feed, const StreamSmem<ST>& S,
                                             double& dmass) {
  using Regs = StreamRegs<REGU>;
  const int warp = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0);  // known to be warp-uniform
  // setmaxnreg must be one and the same instruction for the four warps of a
  // warpgroup (warps 0-3, warps 4-7): it comes before any branch inside a group.
  if (warp >= 4) {
    role_registers<Regs::LAUNCH, Regs::COLLIDE>();
    collide_role<ST, VEC, DIAG, REGU>(feed, S, warp - 4, dmass);
  } else {
    role_registers<Regs::LAUNCH, Regs::ADVECT>();
    if (warp == 0 || warp == 3)
      advect_role<+1, ORDER, LIM, ST, VEC>(feed, S, warp);
    else
      advect_role<-1, ORDER, LIM, ST, VEC>(feed, S, warp);
  }
}

// DIAG: fuse the diagnostics of the state after the step (P.diag_mass and
// P.diag_sums receive them); REGU: the regularised collision (Eq. ereg).  Both
// are separate instantiations, so that the plain step carries none of their
// instructions (cold code in the loop body costs instruction fetch).
template <typename ST, int ORDER, int LIM, bool VEC, bool DIAG, bool REGU>
__global__ void __launch_bounds__(NT, StreamRegs<REGU>::CTAS)
    stream_kernel(const __grid_constant__ StepArgs<float> P, const __grid_constant__ RowMaps maps) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const StreamSmem<ST> S(smem_raw);
  if (VEC && threadIdx.x == 0) prefetch_map(maps.m);
  S.init(DIAG);
  previous_step_done();
  // fused diagnostics: rho - rho_ref of this thread's nodes, and rho_ref of every node once
  double dmass = 0.0;
  stream_roles<ORDER, LIM, ST, VEC, DIAG, REGU>(SingleFeed(P, maps), S, dmass);
  if (DIAG) {
    // one warp sum and one global add per warp for the mass
    if (blockIdx.x == 0 && threadIdx.x == 0) dmass = (double)P.rho_ref * (double)P.plane;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmass += __shfl_down_sync(0xffffffffu, dmass, o);
    if ((threadIdx.x & 31) == 0 && dmass != 0.0) atomicAdd(P.diag_mass, dmass);
    __syncthreads();  // every warp's shared site sums
    if (threadIdx.x < 6) atomicAdd(&P.diag_sums[threadIdx.x], S.dsums[threadIdx.x]);
  }
}

// Several lattices advanced by one launch: their work items are concatenated;
// each lattice brings its own tensor maps.
template <int ORDER, int LIM, bool REGU>
__global__ void __launch_bounds__(NT, StreamRegs<REGU>::CTAS)
    stream_batch_kernel(const __grid_constant__ BatchArgs<float> B) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const StreamSmem<float> S(smem_raw);
  S.init(false);
  previous_step_done();
  double dmass = 0.0;  // unused: batched launches carry no fused diagnostics
  stream_roles<ORDER, LIM, float, true, false, REGU>(BatchFeed(B), S, dmass);
}
