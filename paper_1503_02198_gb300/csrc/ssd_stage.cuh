// ssd_stage.cuh -- one launch per Runge-Kutta stage of the FP32 Euler path
// (double-float or float state): common fluxes of the conforming and periodic
// faces, the sliding interfaces' mortar fluxes, the boundary faces, and the
// element work of k_volume, for every element tile.  Included by
// ssd_engine.cuh.
//
// Why one kernel.  A face pass of its own reads both sides' traces, writes
// both sides' common fluxes and makes the volume kernel read them back: 16 N
// words per element each way, and a launch whose threads wait for two
// dependent memory round trips.  Here the thread that owns an SP line forms
// the Rusanov fluxes of the line's two end points itself: its own traces from
// the line's SP values it holds anyway, the neighbours' traces loaded one tile
// ahead.  Both sides of a face evaluate the same expression (its Rusanov flux
// is symmetric under an exchange of the sides with the sign of the jump term),
// so they get the same bits and the scheme stays conservative.  The arithmetic
// is twice a face pass's, packed two end points per instruction.  Because
// neighbours read a tile's traces while it writes its new ones, a stage reads
// one trace buffer (TR) and writes another (TRo).
//
// What bounds it (N = 6, 246,900 cells, double-float state): shared-memory
// bandwidth 69 %, issue 50 %, DRAM 1.03 GB in the 207 us of a later stage (5.0
// TB/s); barrier, wait and shared-load stalls 1.2 to 1.3 each per issue with 15
// warps per SM.  A step took 703 us with the face pass (48 us) and the volume
// kernel (180 us) apart and takes 606 us here (float state, 123,450 cells: 322 ->
// 286 us; 31,509 cells at N = 3: 72 -> 53 us; 6,016 cells at N = 4: 39 -> 29 us).
// Results are the bits of the separate kernels.
#pragma once

namespace ssd {

// ---- packed pairs of floats: each lane is the scalar operation ----
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 f2_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 f2_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 f2_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 f2_sub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
// -1 / x of both lanes, minus recip() of each (the approximate reciprocal of
// -x is that of x with the other sign, and Newton's step keeps it so)
__device__ __forceinline__ float2 f2_neg_recip(float2 x) {
  float2 r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(-x.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(-x.y));
  return f2_fma(r, f2_fma(x, r, f2(1.0f)), r);
}
__device__ __forceinline__ void cp_async8(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// ---- paired layout ----
// The state planes, the traces and the boundary fluxes of this path hold the
// variables in pairs, (rho, rho u) and (rho v, E): [E][2][N][N][2] and
// [E][4 faces][2][N][2], so that a pair is one 8-byte access and one packed
// operand everywhere (half the load and store instructions of one word per
// variable).  The state crosses the ABI as [E][4][N][N] and is converted with
// the double-float split.

// FP64 state -> hi (and lo) planes in pairs; thread = one pair of one SP
template <int NN>
__global__ void k_split_pairs(const double *__restrict__ Q, float2 *hi, float2 *lo, int n) {
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int t = (blockIdx.x * 4 + u) * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const size_t g = (size_t)(t / NN) * 2 * NN + t % NN;
    const double a = Q[g], b = Q[g + NN];
    const float2 h = make_float2(__double2float_rn(a), __double2float_rn(b));
    hi[t] = h;
    if (lo) lo[t] = make_float2(__double2float_rn(a - (double)h.x), __double2float_rn(b - (double)h.y));
  }
}

template <int NN>
__global__ void k_join_pairs(const float2 *__restrict__ hi, const float2 *__restrict__ lo, double *Q, int n) {
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int t = (blockIdx.x * 4 + u) * blockDim.x + threadIdx.x;
    if (t >= n) return;
    const size_t g = (size_t)(t / NN) * 2 * NN + t % NN;
    const float2 h = hi[t], l = lo ? lo[t] : make_float2(0.0f, 0.0f);
    Q[g] = lo ? (double)h.x + (double)l.x : (double)h.x;
    Q[g + NN] = lo ? (double)h.y + (double)l.y : (double)h.y;
  }
}

// face traces of a state in pairs; thread = one pair at one face point
template <int N>
__global__ void k_trace_pairs(MeshDev md, const float2 *__restrict__ Q) {
  pdl_enter();
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= md.E * 8 * N) return;
  const int e = t / (8 * N), r = t - e * 8 * N;
  const int f = r / (2 * N), p = (r / N) & 1, j = r % N;
  const VolBasis<float, N> &B = cVB<float, N>;
  const float2 *q = Q + ((size_t)e * 2 + p) * N * N;
  float2 acc = make_float2(0.0f, 0.0f);
#pragma unroll
  for (int k = 0; k < N; ++k)
    acc = f2_fma((f == 0 || f == 2) ? q[k * N + j] : q[j * N + k], (f == 1 || f == 2) ? B.H12[k] : B.H02[k], acc);
  ((float2 *)md.TR)[t] = acc;
}

// ---- element-face records ----
// One 16-byte record per element face: the face's unit normal at t = 0 (out
// of its side A, as the face table has it), the signed length s with
// F~_end = s F.n, and the word offset of the neighbour's traces in TR (4 N
// times its element face: a multiple of 4) with bit 1 for a reversed point
// order and bit 0 for side B.  On a straight face between straight stationary
// cells the normal and length are the same at every point and V_g.n is 0.
// x marks the others: kRecTable, the row of the face's per-point table in y
// ([row][N] of nx, ny, s, V_g.n); kRecIface and kRecBoundary, faces that are
// not conforming ones (their offset is the face's own, so that loads need no
// branch).
constexpr float kRecTable = 2.0f, kRecIface = 3.0f, kRecBoundary = 4.0f;

// The records from the face table: one thread per conforming or periodic face
// (its two element faces), then per interface and boundary face.  With rec
// null only the faces that need per-point rows are counted; else each of them
// takes its next two rows of pts from the counter.
template <int N>
__global__ void k_face_records(MeshDev md, float4 *rec, float4 *pts, int *count) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < md.nF) {
    const int4 fc = md.faces[t];
    // the normal or V_g.n varies along the face on rotating zones (low bits of
    // the cell flag) and next to cells with a metric table
    const bool varies = ((md.eflag[fc.x >> 2] | md.eflag[fc.y >> 2]) & ~kIfaceBit) != 0;
    const int row = varies ? 2 * atomicAdd(count, 1) : 0;
    if (!rec) return;
    const float *g = (const float *)md.fgeo + (size_t)t * 5 * N;
    for (int side = 0; side < 2; ++side) {
      float4 r;
      r.w = __int_as_float((side ? fc.x : fc.y) * 4 * N | (fc.z ? 2 : 0) | side);
      if (!varies) {
        r.x = g[0];
        r.y = g[N];
        r.z = side ? -g[3 * N] : g[2 * N];
      } else {
        r.x = kRecTable;
        r.y = __int_as_float(row + side);
        r.z = 0.0f;
        for (int p = 0; p < N; ++p) {
          const int j = (side && fc.z) ? N - 1 - p : p;  // the table is in side A's point order
          pts[(size_t)(row + side) * N + p] = make_float4(g[j], g[N + j], side ? -g[3 * N + j] : g[2 * N + j], g[4 * N + j]);
        }
      }
      rec[side ? fc.y : fc.x] = r;
    }
    return;
  }
  t -= md.nF;
  if (!rec || t >= md.nL + md.nR + md.nB) return;
  const bool iface = t < md.nL + md.nR;
  const int ef = t < md.nL ? md.Lface[t].x : iface ? md.Rface[t - md.nL].x : md.bfaces[t - md.nL - md.nR].x;
  rec[ef] = make_float4(iface ? kRecIface : kRecBoundary, 0.0f, 0.0f, __int_as_float(ef * 4 * N));
}

// Rusanov common fluxes (Sec. 3.1) of a line's two end points, one per lane:
// own state q, neighbour state n, unit normal (nx, ny) out of side A, V_g.n
// (MOVING; zero otherwise); jump is -1/2 where the own side is A, +1/2 where
// it is B (the jump is q_B - q_A).  Each lane gives the bits of rusanov() with
// sides A and B: the sides are symmetric but for the jump's sign, and the
// pressures and fluxes are carried with the sign that 1 / rho comes with.
template <bool MOVING>
__device__ __forceinline__ void rusanov2(const float2 *q, const float2 *n, float2 nx, float2 ny, float2 vg, float2 jump,
                                         float gamma, float2 *F) {
  const float2 ngm1 = f2(-(gamma - 1.0f)), g2 = f2(gamma);
  float2 lam[2], f[2][4];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const float2 *a = s ? n : q;
    const float2 ir = f2_neg_recip(a[0]);  // -1 / rho
    // (products summed elsewhere are formed by an FMA with 0: the compiler
    // fuses a plain multiply with a later sum, which rounds otherwise)
    const float2 e = f2_fma(f2_mul(f2(0.5f), f2_fma(a[1], a[1], f2_mul(a[2], a[2]))), ir, a[3]);
    const float2 p = f2_fma(ngm1, e, f2(0.0f));  // -p
    const float2 mn = f2_fma(a[1], nx, f2_mul(a[2], ny));
    const float2 un = f2_fma(mn, ir, f2(0.0f));  // -V.n
    const float2 h = f2_sub(a[3], p);
    if (MOVING) {
      f[s][0] = f2_fma(a[0], un, f2_mul(vg, a[0]));
      f[s][1] = f2_fma(a[1], un, f2_fma(p, nx, f2_mul(vg, a[1])));
      f[s][2] = f2_fma(a[2], un, f2_fma(p, ny, f2_mul(vg, a[2])));
      f[s][3] = f2_fma(h, un, f2_mul(vg, a[3]));
    } else {
      f[s][0] = f2_fma(a[0], un, f2(0.0f));
      f[s][1] = f2_fma(a[1], un, f2_mul(p, nx));
      f[s][2] = f2_fma(a[2], un, f2_mul(p, ny));
      f[s][3] = f2_fma(h, un, f2(0.0f));
    }
    // (sqrtf: a packed Newton step from the approximate reciprocal root is within
    // an ulp and 1.2 % of a step faster, 2590 instead of 2623 us for four steps of
    // 246,900 cells at N = 6, but gives -2.5e34 where c^2 is subnormal)
    const float2 cc = f2_mul(f2_mul(g2, p), ir);
    const float2 w = MOVING ? f2_add(un, vg) : un;
    lam[s] = make_float2(fabsf(w.x) + sqrtf(cc.x), fabsf(w.y) + sqrtf(cc.y));
  }
  const float2 l = make_float2(lam[0].x > lam[1].x ? lam[0].x : lam[1].x, lam[0].y > lam[1].y ? lam[0].y : lam[1].y);
  const float2 hl = f2_mul(jump, l);
#pragma unroll
  for (int v = 0; v < 4; ++v)
    F[v] = f2_fma(f2(-0.5f), f2_add(f[0][v], f[1][v]), f2_mul(hl, f2_sub(n[v], q[v])));
}

// Shared-memory layout: two stages of a tile's state hi (padded element
// stride, as k_volume's), cell records and flags; three slots of face records
// (a tile's arrive one tile ahead of its state, since they name the traces to
// load); the Runge-Kutta inputs; the two directions' divergences; barriers;
// the zone table; each thread's prefetched end points.  44 KB at N = 6.
template <int N, bool AUX, bool LO>
struct StageCfg {
  using V = VolCfg<float, N, true, AUX, LO>;
  static constexpr int NN = N * N, EPB = V::EPB, THREADS = V::THREADS;
  // element stride (words) of the padded tiles: the padding with the fewest
  // bank conflicts of the 8-byte line accesses (counted over a tile's warps:
  // N = 3: 36 wavefronts per line pass against 18 conflict free, 4: 48 / 24,
  // 5: 77 / 40, 6: 72 / 36)
  static constexpr int SE = 4 * NN + (N == 3 ? 8 : N == 4 ? 4 : N == 5 ? 12 : 24);
  static constexpr int QE = V::QE, QHI = EPB * SE * 4, QB = V::QB, QBL = V::QBL, AUXB = V::AUXB;
  static constexpr int EGB = EPB * 32, EFB = EPB * 4, RECB = EPB * 64;
  static constexpr int O_QHI = 0, O_EG = QHI, O_EF = O_EG + EGB;
  static constexpr int STAGE = (O_EF + EFB + 127) / 128 * 128;
  static constexpr int O_REC = 2 * STAGE;
  static constexpr int O_QLO = O_REC + 3 * RECB, O_NHI = O_QLO + QBL, O_NLO = O_NHI + QB, O_AUX = O_NLO + QBL;
  static constexpr int O_RF = (O_AUX + AUXB + 127) / 128 * 128, O_RG = O_RF + QHI;
  // the mortar flux's work arrays lie over the single-buffered part and the
  // divergence arrays, before the first tile uses them
  using Mort = MortShared<float, N, MORTAR_RUSANOV, EPB>;
  static constexpr int WORK_END = O_RG + QHI > O_QLO + (int)sizeof(Mort) ? O_RG + QHI : O_QLO + (int)sizeof(Mort);
  // each thread's prefetched end points: neighbour traces [end][pair][thread], face table points [end][thread]
  static constexpr int O_NB = (WORK_END + 15) / 16 * 16, O_GEO = O_NB + 4 * THREADS * 8;
  static constexpr int O_BAR = O_GEO + 2 * THREADS * 16;
  static constexpr int O_ZT = O_BAR + 32;
  static constexpr int SMEM = O_ZT + ((3 * kZT + N) * 4 + 15) / 16 * 16;  // zone table, solution points
  static constexpr int TXA = EPB * QE + EGB + EFB;
  static_assert((SE * 4) % 16 == 0 && QE % 16 == 0 && QB % 16 == 0 && RECB % 16 == 0 && O_QLO % 16 == 0, "bulk copies");
  static constexpr int BY_SMEM = 228 * 1024 / (SMEM + 1024);
  // five CTAs of three warps (N = 3, 4 and 6) have 128 registers a thread.  A sixth
  // needs a cap of 96, and the words that spill then come back from L2 (the tiles
  // take the L1): 836 us a step instead of 656 on 246,900 cells at N = 6.  At N = 5
  // a CTA has four warps: shared memory admits four with a double-float state (128
  // registers); with a float state five fit at 96 registers, and there five are
  // better although the residual's form spills two words (three steps of 96,256
  // cells 616 us, 665 with four; 24,064 cells 208 and 218; 6,016 cells 112 and 106)
  static constexpr int MINB = BY_SMEM < 5 ? BY_SMEM : 5;
};

// Waits (bounded) until all nblk coupling blocks of this launch are done.  The
// blocks are claimed by counter, so a CTA that waits first takes what is left
// unclaimed: it only ever waits for blocks that running CTAs have claimed.
__device__ __forceinline__ bool wait_coupling(const int *done, int nblk) {
  for (int i = 0; i < kWaitPolls; ++i) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(done) : "memory");
    if (v >= nblk) return true;
    __nanosleep(64);
  }
  return false;
}

// tiles in the order they are worked: those without an interface or boundary
// face first ([0, nearly)), so that the coupling blocks (nmort mortar blocks,
// then the boundary points) are done long before the first tile that needs them
template <int N, int MODE, bool AUX, bool LO>
__global__ void __launch_bounds__(StageCfg<N, AUX, LO>::THREADS, StageCfg<N, AUX, LO>::MINB)
    k_stage(const __grid_constant__ MeshDev md, const __grid_constant__ VolArgs<float> va, int nitems, int nearly,
            int nmort, int nblk, int ahead, int rev) {
  pdl_begin(ahead);
  using C = StageCfg<N, AUX, LO>;
  constexpr int EPB = C::EPB, NT = C::THREADS, NN = N * N;
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t *bar = (uint64_t *)(smem + C::O_BAR);  // [0], [1]: the two stages; [2]: Runge-Kutta inputs
  float(*sRF)[C::SE] = (float(*)[C::SE])(smem + C::O_RF);
  float(*sRG)[C::SE] = (float(*)[C::SE])(smem + C::O_RG);
  float *sZT = (float *)(smem + C::O_ZT), *sXs = sZT + 3 * kZT;
  __shared__ int s_claim;
  const VolBasis<float, N> &B = cVB<float, N>;
  const int G = gridDim.x;
  const bool use_base = MODE == MODE_RK && va.has_base;
  const uint32_t txB = MODE == MODE_RK ? C::QBL + (va.has_base ? C::QB + C::QBL : 0) + C::AUXB : 0;

  auto issue_rec = [&](int tile, int slot, uint64_t *b) {
    bulk_g2s(smem + C::O_REC + slot * C::RECB, md.frec + (size_t)tile * EPB * 4, C::RECB, b);
  };
  // state hi, cell records and flags of a tile into stage st, and the face
  // records of the tile after it (tile2 >= 0) into the given slot; a CTA's
  // first tile brings its own face records too (slot 0).  (The test switch of
  // sd_test_wait_timeout arms the first tile of CTA 0 with more bytes than its
  // copies deliver; it is 0 otherwise.)
  auto issue_tables = [&](int tile, int st, int tile2, int slot2, bool first) {
    unsigned char *sb = smem + st * C::STAGE;
    const size_t e0 = (size_t)tile * EPB;
    mbar_expect_tx(&bar[st], C::TXA + (tile2 >= 0 ? C::RECB : 0) +
                                 (first ? C::RECB + (blockIdx.x == 0 ? md.test_tx_extra : 0) : 0));
    bulk_g2s(sb + C::O_EG, (const float *)md.egeo + e0 * 8, C::EGB, &bar[st]);
    bulk_g2s(sb + C::O_EF, md.eflag + e0, C::EFB, &bar[st]);
    if (first) issue_rec(tile, 0, &bar[st]);
    if (tile2 >= 0) issue_rec(tile2, slot2, &bar[st]);
  };
  // (after issue_tables has armed the barrier)
  auto issue_state = [&](int tile, int st, int lane) {
    if (lane < EPB)
      bulk_g2s(smem + st * C::STAGE + C::O_QHI + lane * C::SE * 4,
               (const float *)va.in.hi + ((size_t)tile * EPB + lane) * 4 * NN, C::QE, &bar[st]);
  };
  auto issueB = [&](int tile) {
    const size_t e0 = (size_t)tile * EPB;
    mbar_expect_tx(&bar[2], txB);
    if (LO) bulk_g2s(smem + C::O_QLO, (const float *)va.in.lo + e0 * 4 * NN, C::QBL, &bar[2]);
    if (va.has_base) {
      bulk_g2s(smem + C::O_NHI, (const float *)va.base.hi + e0 * 4 * NN, C::QB, &bar[2]);
      if (LO) bulk_g2s(smem + C::O_NLO, (const float *)va.base.lo + e0 * 4 * NN, C::QBL, &bar[2]);
    }
    if (AUX) bulk_g2s(smem + C::O_AUX, va.w_in + e0 * 4 * NN, C::AUXB, &bar[2]);
  };
  // one coupling block: EPB mortars, or NT boundary points
  bool entered = ahead == 0;
  auto enter = [&]() {  // what the launch before this one wrote may be read from here on
    if (!entered) pdl_enter();
    entered = true;
  };
  auto couple = [&](int c) {
    if (c < nmort) {
      mortar_flux_body<float, N, MORTAR_RUSANOV, EPB, LAY_PAIRS>(md, c, *(typename C::Mort *)(smem + C::O_QLO), enter);
    } else {
      enter();
      const int t = (c - nmort) * NT + threadIdx.x;
      if (t < md.nB * N) k_bface_point<float, N, true, LAY_PAIRS>(md, t);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      atomicAdd(&md.clk->done, 1);
    }
  };
  auto claim = [&]() {
    if (threadIdx.x == 0) s_claim = atomicAdd(&md.clk->claim, 1);
    __syncthreads();
    const int c = s_claim;
    __syncthreads();
    return c;
  };

  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_init(&bar[2], 1);
    fence_mbar_init();
  }
  if (threadIdx.x < 3 * kZT) sZT[threadIdx.x] = zone_tab<float>(md.clk)[threadIdx.x];
  if (threadIdx.x < N) sXs[threadIdx.x] = B.Xs[threadIdx.x];
  int item = blockIdx.x;
  // item i's tile; rev: the early tiles from the last to the first, so that a
  // stage begins on what the stage before it wrote last, still in L2 (the trace
  // buffers alternate, and with them the direction): 1 % of a step on 246,900
  // cells, 0.7 % on 123,450 with float state
  auto tile_of = [&](int i) { return i < nitems ? md.tord[rev && i < nearly ? nearly - 1 - i : i] : -1; };
  int tile = tile_of(item), tile1 = tile_of(item + G), tile2 = tile_of(item + 2 * G);
  __syncthreads();
  if (threadIdx.x == 0 && tile >= 0) issue_tables(tile, 0, tile1, 1, true);
  // the first CTAs take the coupling blocks before their tiles, and so does a
  // CTA whose first tile needs them, as long as any is unclaimed
  bool claimed = nblk == 0;  // every block has been claimed
  if ((int)blockIdx.x < nblk || (item >= nearly && !claimed)) {
    const int c = claim();
    if (c < nblk) couple(c);
    else claimed = true;
  }
  bool ready = nblk == 0;
  enter();
  __syncwarp();
  if (threadIdx.x < 32 && tile >= 0) issue_state(tile, 0, threadIdx.x);

  // this thread's SP line (direction d: 0 xi, 1 eta) and its two end faces
  const int d = threadIdx.x >= EPB * N ? 1 : 0;
  const int tl = threadIdx.x - d * EPB * N;
  const int le = tl / N, mline = tl - le * N;
  const int fa = d == 0 ? 3 : 0, fb = d == 0 ? 1 : 2;
  const float gm1 = md.gamma_f - 1.0f;
  // Prefetch of the line's two end points (0: face fa, 1: face fb) for a tile
  // whose records are in the slot: the neighbours' traces and, where the face
  // has one, its point of the per-point table, copied into this thread's own
  // slots of shared memory (held in registers across a tile they spilled, and
  // a spill waits for the load).
  float2 *sNb = (float2 *)(smem + C::O_NB) + threadIdx.x;       // [end][pair][NT]
  float4 *sGeo = (float4 *)(smem + C::O_GEO) + threadIdx.x;     // [end][NT]
  auto fetch = [&](int slot) {
    const float4 *rec = (const float4 *)(smem + C::O_REC + slot * C::RECB) + le * 4;
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float4 r = rec[e ? fb : fa];
      int code = __float_as_int(r.w);
      if (!ssd_check(md, code >= 0 && code < md.E * 16 * N)) code = 0;
      const float2 *t = (const float2 *)((const float *)md.TR + (code & ~3)) + ((code & 2) ? N - 1 - mline : mline);
      cp_async8(sNb + (2 * e) * NT, t);
      cp_async8(sNb + (2 * e + 1) * NT, t + N);
      if (r.x == kRecTable) cp_async16(sGeo + e * NT, md.fgp + (size_t)__float_as_int(r.y) * N + mline);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // common flux of an end point that is not a conforming one: the sum of its
  // interface face's mortar contributions, or the boundary point's flux
  auto special = [&](int ef, float kind, float *val) {
    val[0] = val[1] = val[2] = val[3] = 0.0f;
    if (kind == kRecIface) {
      const int fq = md.efi[ef];
      if (!ssd_check(md, fq >= 0 && fq < md.nL + md.nR)) return;
      const int rev = (fq >= md.nL ? md.Rface[fq - md.nL] : md.Lface[fq]).y;
      int e2, j2;
      gather_sum<float, N, GATHER_FLUX>(md, fq, rev ? N - 1 - mline : mline, val, e2, j2);
    } else {
      const float *cf = (const float *)md.CF + (size_t)ef * 4 * N;
#pragma unroll
      for (int v = 0; v < 4; ++v) val[v] = cf[face_word<LAY_PAIRS, N>(v, mline)];
    }
  };

  // gives up on this CTA: reports the timeout and lets the copies in flight
  // land (full limits) before the CTA exits
  auto give_up = [&](int it, bool b_issued) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (threadIdx.x != 0) return;
    atomicOr(&md.clk->flags, 4);
    if (tile1 >= 0) mbar_wait_bounded(&bar[(it + 1) & 1], (uint32_t)(((it + 1) >> 1) & 1));
    if (b_issued) mbar_wait_bounded(&bar[2], (uint32_t)(it & 1));
  };

  bool bad = false;
  int slot0 = 0, slot1 = 1;  // slots of this and the next tile's face records
  for (int it = 0; item < nitems; item += G, ++it) {
    const int st = it & 1;
    const int slot2 = slot1 == 2 ? 0 : slot1 + 1;
    const int tile3 = tile_of(item + 3 * G);  // used one iteration on
    if (threadIdx.x < 32 && tile1 >= 0) {
      // the refilled regions were last read before the previous iteration's
      // closing barrier; order those generic reads before the async writes
      fence_proxy_async_smem();
      if (threadIdx.x == 0) issue_tables(tile1, st ^ 1, tile2, slot2, false);
      __syncwarp();
      issue_state(tile1, st ^ 1, threadIdx.x);
    }
    if (!claimed && item >= nearly) {
      // this tile needs the coupling blocks' results: a block left unclaimed is
      // taken here (before the Runge-Kutta inputs fill the region its work
      // arrays lie over), so that each one is in the hands of a running CTA
      for (int c = claim(); c < nblk; c = claim()) couple(c);
      claimed = true;
    }
    if (txB && threadIdx.x == 0) {
      fence_proxy_async_smem();
      issueB(tile);
    }
    if (!cta_wait(&bar[st], (uint32_t)((it >> 1) & 1),
                  (blockIdx.x == 0 && it == 0 && md.test_poll) ? md.test_poll : kWaitPolls)) {
      if (threadIdx.x == 0 && blockIdx.x == 0 && it == 0) settle_test_wait(md, smem + C::O_EF, tile * EPB, &bar[0]);
      give_up(it, txB != 0);
      return;
    }
    unsigned char *sb = smem + st * C::STAGE;
    float(*sQ)[C::SE] = (float(*)[C::SE])(sb + C::O_QHI);
    const int *sEF = (const int *)(sb + C::O_EF);
    const float *sEG = (const float *)(sb + C::O_EG);
    const int e0 = tile * EPB;
    const int ne = min(EPB, md.E - e0);
    if (it == 0) fetch(0);
    // the weights through an index the compiler cannot see is 0: it would keep
    // as many of them in registers across the tiles as fit and spill others
    int zero;
    asm volatile("mov.u32 %0, 0;" : "=r"(zero));
    const VolBasis<float, N> &Bw = (&cVB<float, N>)[zero];
    // ---- phase 1: one thread per SP line: its end points' common fluxes, the
    // fluxes at its interior points, its part of the divergence ----
    {
      // a cell of the stationary zone: no rotation, no grid velocity (the same
      // bits as with the identity and zero, every sum's rounding being written out)
      const bool moving = (sEF[le] & kZoneMask) != 0;
      ElemGeo<float, N, true> Gm;
      if (moving) Gm.load_rec(md, e0 + le, sEF[le], sEG + le * 8, sZT);
      else Gm.load_still(md, sEF[le], sEG + le * 8);
      float2 f01[N + 1], f23[N + 1];
      float2 kind;  // above kRecTable: not a conforming face
      {
        // own traces (as the trace phase formed them), then the Rusanov fluxes
        // of both ends, one per lane; on rotating zones the normal is turned
        float2 a0 = f2(0.0f), a1 = f2(0.0f), b0 = f2(0.0f), b1 = f2(0.0f);
#pragma unroll
        for (int k = 0; k < N; ++k) {
          const int sp = d == 0 ? mline * N + k : k * N + mline;
          const float2 qa = *(const float2 *)(sQ[le] + 2 * sp), qb = *(const float2 *)(sQ[le] + 2 * (NN + sp));
          a0 = f2_fma(qa, Bw.H02[k], a0);
          a1 = f2_fma(qa, Bw.H12[k], a1);
          b0 = f2_fma(qb, Bw.H02[k], b0);
          b1 = f2_fma(qb, Bw.H12[k], b1);
        }
        const float2 q[4] = {make_float2(a0.x, a1.x), make_float2(a0.y, a1.y), make_float2(b0.x, b1.x),
                             make_float2(b0.y, b1.y)};
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        const float2 na = sNb[0], nb2 = sNb[NT], nc = sNb[2 * NT], nd = sNb[3 * NT];
        const float2 nb[4] = {make_float2(na.x, nc.x), make_float2(na.y, nc.y), make_float2(nb2.x, nd.x),
                              make_float2(nb2.y, nd.y)};
        const float4 *rec = (const float4 *)(smem + C::O_REC + slot0 * C::RECB) + le * 4;
        float4 ga = rec[fa], gb = rec[fb];
        const float2 jump = make_float2((__float_as_int(ga.w) & 1) ? 0.5f : -0.5f,
                                        (__float_as_int(gb.w) & 1) ? 0.5f : -0.5f);
        ga.w = gb.w = 0.0f;  // V_g.n
        if (ga.x == kRecTable) ga = sGeo[0];
        if (gb.x == kRecTable) gb = sGeo[NT];
        const float2 nx = make_float2(ga.x, gb.x), ny = make_float2(ga.y, gb.y);
        const float2 vgn = make_float2(ga.w, gb.w), fs = make_float2(ga.z, gb.z);
        float2 F[4];
        if (moving) {
          const float2 c2 = f2(Gm.c), s2 = f2(Gm.s), ns2 = f2(-Gm.s);
          const float2 rx = f2_fma(c2, nx, f2_mul(ns2, ny)), ry = f2_fma(s2, nx, f2_mul(c2, ny));
          rusanov2<true>(q, nb, rx, ry, vgn, jump, md.gamma_f, F);
        } else {
          rusanov2<false>(q, nb, nx, ny, vgn, jump, md.gamma_f, F);
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) F[v] = f2_mul(fs, F[v]);
        kind = make_float2(nx.x, nx.y);
        f01[0] = make_float2(F[0].x, F[1].x);
        f23[0] = make_float2(F[2].x, F[3].x);
        f01[N] = make_float2(F[0].y, F[1].y);
        f23[N] = make_float2(F[2].y, F[3].y);
      }
      // the line's values again (read twice: kept across the Rusanov fluxes they
      // cost 24 registers, and spilled words come back from L2)
      asm volatile("" ::: "memory");
      // variables packed in pairs (rho, rho u), (rho v, E)
      float2 q2[2][N];
#pragma unroll
      for (int k = 0; k < N; ++k) {
        const int sp = d == 0 ? mline * N + k : k * N + mline;
        q2[0][k] = *(const float2 *)(sQ[le] + 2 * sp);
        q2[1][k] = *(const float2 *)(sQ[le] + 2 * (NN + sp));
      }
      // the next tile's end points, covered by the rest of this tile's work
      if (tile1 >= 0) fetch(slot1);
      float2 s01[N + 1], s23[N + 1];
#pragma unroll
      for (int i = 1; i < N; ++i) {
        s01[i] = f2(0.0f);
        s23[i] = f2(0.0f);
      }
#pragma unroll
      for (int k = 0; k < N; ++k)
#pragma unroll
        for (int i = 1; i < N; ++i) {
          const float2 h = Bw.Hf2[i * N + k];
          s01[i] = f2_fma(q2[0][k], h, s01[i]);
          s23[i] = f2_fma(q2[1][k], h, s23[i]);
        }
      if (moving) {
        float mvx[N + 1], mvy[N + 1], mvg[N + 1];
        Gm.line_metrics(d, mline, mvx, mvy, mvg);
#pragma unroll
        for (int i = 1; i < N; ++i) {
          const float qf[4] = {s01[i].x, s01[i].y, s23[i].x, s23[i].y};
          float f[4];
          point_flux(qf, mvx[i], mvy[i], mvg[i], gm1, f);
          f01[i] = make_float2(f[0], f[1]);
          f23[i] = make_float2(f[2], f[3]);
        }
      } else {
        float mvx[N + 1], mvy[N + 1];
        Gm.line_metrics_still(d, mline, mvx, mvy);
#pragma unroll
        for (int i = 1; i < N; ++i) {
          const float qf[4] = {s01[i].x, s01[i].y, s23[i].x, s23[i].y};
          float f[4];
          point_flux_still(qf, mvx[i], mvy[i], gm1, f);
          f01[i] = make_float2(f[0], f[1]);
          f23[i] = make_float2(f[2], f[3]);
        }
      }
      if (item >= nearly) {
        // the end points that are not conforming ones, once the coupling blocks
        // are done
        if (!ready) {
          bool done = true;
          if (threadIdx.x == 0) done = wait_coupling(&md.clk->done, nblk);
          if (!__syncthreads_and(done)) {
            give_up(it, txB != 0);
            return;
          }
          ready = true;
        }
        if (le < ne) {
          float val[4];
          if (kind.x > kRecTable) {
            special(4 * (e0 + le) + fa, kind.x, val);
            f01[0] = make_float2(val[0], val[1]);
            f23[0] = make_float2(val[2], val[3]);
          }
          if (kind.y > kRecTable) {
            special(4 * (e0 + le) + fb, kind.y, val);
            f01[N] = make_float2(val[0], val[1]);
            f23[N] = make_float2(val[2], val[3]);
          }
        }
      }
      float2 acc0[N], acc1[N];
#pragma unroll
      for (int k = 0; k < N; ++k) acc0[k] = acc1[k] = f2(0.0f);
#pragma unroll
      for (int i = 0; i <= N; ++i)
#pragma unroll
        for (int k = 0; k < N; ++k) {
          const float2 w = Bw.Dm2[k * (N + 1) + i];
          acc0[k] = f2_fma(w, f01[i], acc0[k]);
          acc1[k] = f2_fma(w, f23[i], acc1[k]);
        }
      float2 *o = (float2 *)(d == 0 ? sRF[le] + 2 * mline * N : sRG[le] + 2 * mline);
      const int ks = d == 0 ? 1 : N;
#pragma unroll
      for (int k = 0; k < N; ++k) {
        o[k * ks] = acc0[k];
        o[NN + k * ks] = acc1[k];
      }
    }
    // the Runge-Kutta inputs must have landed too
    if (txB) {
      if (!cta_wait(&bar[2], (uint32_t)(it & 1))) {
        give_up(it, false);
        return;
      }
    } else {
      __syncthreads();
    }
    // ---- phase 2: dQ/dt at the SPs and the Runge-Kutta combination, two
    // variables per instruction: inc = a0 (Q_base - Q_k) + w_in + bdt R in
    // float, added to the double-float state exactly (two-sum) ----
#pragma unroll 1
    for (int idx = threadIdx.x; idx < ne * NN; idx += NT) {
      const int l2 = idx / NN, sp = idx - l2 * NN;
      const float iJ = ElemGeo<float, N, true>::inv_jac_at(md, sEF[l2], sEG + l2 * 8, sp, sXs[sp % N], sXs[sp / N]);
      // pair p (variables 2 p, 2 p + 1) of the SP in a tile array of element stride es
      auto at = [&](const void *base, int es, int p) { return (float2 *)base + (l2 * es / 2 + p * NN + sp); };
      float hv[4];
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        const float2 div = f2_mul(f2_add(*at(sRF, C::SE, p), *at(sRG, C::SE, p)), f2(iJ));
        if constexpr (MODE == MODE_RESIDUAL) {
          double *R = va.R + ((size_t)(e0 + l2) * 4 + 2 * p) * NN + sp;
          R[0] = -(double)div.x;
          R[NN] = -(double)div.y;
        } else {
          const size_t gi = ((size_t)(e0 + l2) * 2 + p) * NN + sp;
          const float2 h = *at(sQ, C::SE, p);
          float2 inc = f2_fma(f2(-va.rk.bdt), div, f2(0.0f));  // R = -div; never fused into the sums below
          float2 l = f2(0.0f);
          if (LO) l = *at(smem + C::O_QLO, 4 * NN, p);
          if (use_base) {
            float2 db = f2_sub(*at(smem + C::O_NHI, 4 * NN, p), h);
            if (LO) db = f2_add(db, f2_sub(*at(smem + C::O_NLO, 4 * NN, p), l));
            inc = f2_fma(f2(va.rk.a0), db, inc);
          }
          if (AUX) inc = f2_add(inc, *at(smem + C::O_AUX, 4 * NN, p));
          float2 H;
          if (LO) {
            const float2 sum = f2_add(h, inc), bb = f2_sub(sum, h);
            const float2 err = f2_add(f2_add(f2_sub(h, f2_sub(sum, bb)), f2_sub(inc, bb)), l);
            H = f2_add(sum, err);
            ((float2 *)va.out.lo)[gi] = f2_sub(err, f2_sub(H, sum));
          } else {
            H = f2_add(h, inc);  // single-float state: rounded to float once
          }
          ((float2 *)va.out.hi)[gi] = H;
          if (va.w_out) ((float2 *)va.w_out)[gi] = f2_fma(f2(-va.rk.g), inc, f2_mul(f2(-va.rk.ddt), div));
          *at(sQ, C::SE, p) = H;
          hv[2 * p] = H.x;
          hv[2 * p + 1] = H.y;
        }
      }
      if constexpr (MODE == MODE_RK) bad |= !physical(hv);
    }
    if (MODE == MODE_RK) {
      __syncthreads();
      // ---- phase 3: face traces of the new state, one thread per SP line ----
      if (le < ne) {
        float2 *tr = (float2 *)md.TRo + (size_t)(e0 + le) * 8 * N + mline;
#pragma unroll
        for (int vp = 0; vp < 2; ++vp) {
          float2 a0 = f2(0.0f), a1 = f2(0.0f);
#pragma unroll
          for (int k = 0; k < N; ++k) {
            const int sp = d == 0 ? mline * N + k : k * N + mline;
            const float2 qk = *(const float2 *)(sQ[le] + 2 * (vp * NN + sp));
            a0 = f2_fma(qk, Bw.H02[k], a0);
            a1 = f2_fma(qk, Bw.H12[k], a1);
          }
          tr[(fa * 2 + vp) * N] = a0;
          tr[(fb * 2 + vp) * N] = a1;
        }
      }
    }
    __syncthreads();  // every read of this tile's buffers is done before they are refilled
    tile = tile1;
    tile1 = tile2;
    tile2 = tile3;
    slot0 = slot1;
    slot1 = slot2;
  }
  if (MODE == MODE_RK && __syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&md.clk->flags, 1);
}

}  // namespace ssd
