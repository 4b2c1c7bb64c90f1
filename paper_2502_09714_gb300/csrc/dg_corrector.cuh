// Corrector with its contractions over the volume nodes on the tensor cores, degrees 2..4
// (included by dg_step_kernels.cuh).
#pragma once

#include <type_traits>

#include "dg_sparse.cuh"
#include "dg_team.h"

namespace dg {

// ===========================================================================
// One CTA per SM holds two teams of eight worker warps, a warp that issues the team's MMAs and a warp
// that issues its copies.  Each team walks over tiles of TE elements on its own (named barriers, its own buffers and tensor-
// memory columns), so that one team's MMAs, waits and barriers are covered by the other's SIMT
// phases; both read the same constant A operands from tensor memory.
//
// Per tile:
//   1. Volume operand: the Taylor coefficients themselves (order 0: six strains, alpha and its
//      rate; orders 1..N-1: six strains, which live on the modes of degree <= N - o, so that K is
//      shorter), split into TF32 parts.  Order N is one constant per element and stays out.
//   2. Volume MMA, D[q][column] = sum_l phi_l(x_q) C[l][column] (3xTF32).  Meanwhile the workers
//      lift the modal face fluxes and take the modal derivative of the strain rows from the sparse
//      lists; each unit accumulates both for 32 (element, field) columns and a block of modes in
//      registers.
//   3. Pointwise law: a thread owns a volume node of one element, sums the Taylor series at the
//      N + 1 time nodes and integrates stress and rate.  The nine terms -rho^-1 Theta^-1 sigma and
//      the rate become the projection's B operand, less their values at node 0 (which return
//      through the row sums of w_q phi_l(x_q)): the fluctuation sets the rounding.
//   4. Projection MMA, D[l][n] = sum_q w_q phi_l(x_q) B[n][q].  There are at most 35 modes for 128
//      lanes, so the TF32 part of A sits in lanes 0..63 and its remainder in lanes 64..127: two
//      MMAs per K step (high and low part of B) give all four products of the split, against three
//      MMAs for three products.
//   5. Read-out (the two lane halves added), modal derivative of the velocity rows, update.
// Nodes: degree 3 has 64 and degree 2 has 27 volume nodes, so A's rows repeat in the other lanes and
// different warps read different elements' columns of the same result.
//
// Bound by instruction issue and latency: a team's tile takes 18.6k cycles at degree 4 (operand 2.3k,
// lift and strain rows 2.9k, law 5.3k, read-out and velocity rows 2.8k, update 1.5k, waits on the MMAs
// 3.2k), with both teams in flight.  Against one team of 15 workers on nodal-time columns, dense modal
// derivatives and three MMAs per K step of the projection: 2.21 -> 1.35 ms on the 196,608-tet cube of
// degree 4, 2.57 -> 1.31 ms on 331,776 element copies of degree 3, 45 -> 23 us on 5,184 tets of degree 2.
// Tiles of eight elements at degree 3, which spread the barriers, the waits and the velocity rows (24 lanes of a
// warp in place of 12) over twice the work: 1.31 -> 1.02 ms.
// With the copies issued by the workers, fewer blocks per phase and rolled operand loops it took 1.62 ms.
// ===========================================================================
// TE: elements per tile and team, 8 at degree 2, 4 or 8 at degree 3, 4 at degree 4 (shared memory).
template <int N, int TILE>
struct CorrTcCfg : Dim<N> {
  using D = Dim<N>;
  static constexpr int TE = TILE;
  static constexpr int TEAMS = 2, WORK_WARPS = 8, WORKERS = 32 * WORK_WARPS, TEAM_THREADS = WORKERS + 32;
  static constexpr int THREADS = TEAMS * (WORKERS + 64);   // workers of both teams, MMA warps, copy warps
  static constexpr int NQ32 = (D::NQ + 31) / 32 * 32;
  static constexpr int REP = 128 / NQ32;                   // copies of A's rows over the lanes
  static constexpr int WPE = NQ32 / 32;                    // warps per element in the law
  static constexpr int ROUNDS = TE / (2 * REP);            // elements per warp in the law
  static constexpr int KP = tc_kp(N), KH = round8(n_modes(N - 1));   // K of order 0, of the orders >= 1
  static constexpr int KQ = tc_kq(N);                      // K of the projection
  static constexpr int GH = 6 * TE / 8;                    // 8-row groups per order >= 1
  static constexpr int N0 = 8 * TE, NH = (6 * TE * (N - 1) + 15) / 16 * 16;   // MMA N
  static constexpr int NB = 10 * TE, NPC = (NB + 15) / 16 * 16;
  static constexpr int LI = n_modes(N - 1);                // input modes of the modal derivatives
  // tensor memory: each team's volume values (then its projection), the projection's A, the
  // volume A (TF32 part, remainder)
  static constexpr int DC = N0 + NH > NPC ? N0 + NH : NPC;
  static constexpr int COL_A = TEAMS * DC, COL_PH = COL_A + KQ, COL_PL = COL_PH + KP;
  static constexpr int TMEM_NEED = COL_PL + KP;
  static constexpr int TMEM_COLS = TMEM_NEED <= 256 ? 256 : 512;
  // shared memory of a team (floats).  Operand region: the volume operand (high parts: order 0
  // [N0 x KP], orders >= 1 [NH x KH]; then the remainders), later the projection's [NB x KQ],
  // whose core matrices are 36 floats apart along K, so that a warp's 32 nodes hit 32 banks.
  static constexpr int BV = N0 * KP + NH * KH;
  static constexpr int PLBO = 36, PGS = KQ / 4 * PLBO, BP = NB / 8 * PGS;
  static constexpr int OPERAND = 2 * BV > 2 * BP ? 2 * BV : 2 * BP;
  static constexpr int VS = (3 * TE) | 1;                  // row stride of the modal inputs
  static constexpr int oOp = 0;
  static constexpr int oV = oOp + OPERAND;                 // [LI][VS] time-integrated velocity
  static constexpr int oT = oV + LI * VS;                  // [3][LI][VS] projected terms
  static constexpr int oA = round4(oT + 3 * LI * VS);      // [TE][QS] update, rows as the state's
  static constexpr int oGeo = oA + TE * D::QS;             // [TE][40]
  static constexpr int oC = oGeo + TE * 40;                // [TE][12] nodal terms at node 0
  // two tile buffers: state, predictor output, face records, GeomF, MatF, face ids, the next
  // tile's face ids (whose records the next copy fetches)
  static constexpr int FES = 4 * D::FFS + (40 - 4 * D::FFS % 32) % 32;   // face records of an element, off the bank period
  static constexpr int bQ = 0, bD = TE * D::QS, bF = bD + TE * D::DS, bG = bF + TE * FES;
  static constexpr int bM = bG + TE * 32, bE = bM + TE * 8, bI = bE + TE * 4;
  static constexpr int BUF = bI + TE * 4;
  static constexpr int oBuf = oC + TE * 12;
  static constexpr int TEAM_SMEM = oBuf + 2 * BUF;
  static constexpr int SMEM = TEAMS * TEAM_SMEM;
  // output-mode blocks of the lift with the strain derivative, and of the velocity derivative
  // (similar numbers of products each, so that the warps of a phase end together)
  static constexpr int NBLK = TE == 8 ? 2 : 4;
  __host__ __device__ static constexpr int blk(int b) {
    return b >= NBLK ? D::L : (b == 0 ? 0 : (N == 4 ? (b == 1 ? 15 : 11 + 6 * b) : (N == 3 ? (TE == 8 ? 14 : 6 + 4 * b) : 5)));
  }
  static constexpr int VBLK = N == 4 ? 8 : (N == 3 ? 6 : 3);
  __host__ __device__ static constexpr int vblk(int b) {
    return b >= VBLK ? D::L
                     : (b == 0 ? 1 : (N == 4 ? (b < 4 ? 5 + 5 * b : 11 + 3 * b) : (N == 3 ? 8 + 2 * b : 1 + 3 * b)));
  }
  __host__ __device__ static constexpr int prj_canon(int n, int q) {
    return (n >> 3) * PGS + (q >> 2) * PLBO + (n & 7) * 4 + (q & 3);
  }
  // the projection's column of term c, element e
  __host__ __device__ static constexpr int prj_col(int c, int e) { return c * TE + e; }
  static_assert(D::QS % 4 == 0 && D::DS % 4 == 0 && D::FFS % 4 == 0 && sizeof(GeomF) == 128 && sizeof(MatF) == 32,
                "16-byte copies");
  static_assert(REP * NQ32 == 128 && ROUNDS * 2 * REP == TE && KQ == NQ32, "law items");
  static_assert(N0 % 16 == 0 && NH % 16 == 0 && N0 <= 256 && NH <= 256 && NPC <= 256 && KP <= 40, "MMA shapes");
  static_assert(D::L <= 64 && LI <= 32 && 6 * TE % 8 == 0, "read-out: input modes in the first lane quarter");
  static_assert(TMEM_NEED <= 512 && oOp % 4 == 0 && BV % 4 == 0 && TEAM_SMEM % 4 == 0, "operands");
  static_assert(WORK_WARPS % TE == 0 && 8 % TE == 0, "a warp builds one element's rows; columns (term, element)");
  static_assert(KH / 4 <= WORK_WARPS, "a shared group's K");
  static_assert(SMEM * 4 <= 227 * 1024, "tensor-core corrector shared memory");
};

// Velocity rows of block B for one (element, component) column: adds the derivative of the projected
// terms T_e'[l] (rows LI VS apart per direction).
template <class C, int N, int B>
__device__ __forceinline__ void velocity_derivative(int blk, const float* T, float* out) {
  if constexpr (B < C::VBLK) {
    if (blk == B) {
      constexpr int K0 = C::vblk(B), K1 = C::vblk(B + 1), LI = n_modes(N - 1);
      float x[3][LI], acc[K1 - K0];
#pragma unroll
      for (int e = 0; e < 3; ++e)
#pragma unroll
        for (int l = 0; l < LI; ++l) x[e][l] = T[(e * LI + l) * C::VS];
#pragma unroll
      for (int k = 0; k < K1 - K0; ++k) acc[k] = 0.f;
      stiffness_columns<K0, K1>(x, acc);
#pragma unroll
      for (int k = K0; k < K1; ++k) out[k * 10] += acc[k - K0];
    } else {
      velocity_derivative<C, N, B + 1>(blk, T, out);
    }
  }
}

template <int N, int LAW, int TILE>
__global__ void __launch_bounds__(CorrTcCfg<N, TILE>::THREADS, 1) k_corrector_tc(StepArgs a) {
  using C = CorrTcCfg<N, TILE>;
  constexpr int L = C::L, NQ = C::NQ, QS = C::QS, DS = C::DS, AOFF = C::AOFF, FFS = C::FFS, TE = C::TE;
  constexpr int KP = C::KP, KH = C::KH, KQ = C::KQ, N0 = C::N0, NH = C::NH, NPC = C::NPC, LI = C::LI, VS = C::VS;
  constexpr TableLayout T = table_layout(N);
  constexpr int kWaitLimit = 1 << 24;
  // the limit of the waits on the MMAs; the drain after a failure keeps the default
  const int wait_limit = a.wait_limit_set ? a.wait_limit : kWaitLimit;
  extern __shared__ float4 smem4[];
  __shared__ __align__(8) uint64_t mbars[C::TEAMS];
  __shared__ uint32_t tmem_base;
  __shared__ TeamStop stops[C::TEAMS];
  const float* tb = a.tables;
  const float dt = a.dt;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  tc::pdl_launch();
  // sums of w_q phi_l(x_q) at this thread's mode of the projection's lanes
  const float row_sum = __ldg(tb + T.PrjS + min(32 * (warp & 1) + lane, C::LP - 1));
  if (warp == 0) tc::alloc(&tmem_base, C::TMEM_COLS);
  if (threadIdx.x < C::TEAMS) {
    tc::mbar_init(&mbars[threadIdx.x], 1);
    stops[threadIdx.x].init();
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tmem_base;
  // constant A operands into tensor memory: w_q phi_l(x_q) (TF32 part in lanes l, remainder in lanes
  // 64 + l; columns q) on warps 0-3, phi_l(x_q) (lanes q, repeated; columns l) on warps 4-7
  if (warp < 4) {
    const uint32_t lane_base = static_cast<uint32_t>(32 * warp) << 16;
    const float* src = tb + (warp < 2 ? T.PrjH : T.PrjL) + (32 * (warp & 1) + lane) * KQ;
#pragma unroll 1
    for (int c0 = 0; c0 < KQ; c0 += 32) {
      float v[32];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(src + c0) + j);
        v[4 * j] = x.x; v[4 * j + 1] = x.y; v[4 * j + 2] = x.z; v[4 * j + 3] = x.w;
      }
      tc::st_x32(tmem + lane_base + C::COL_A + c0, v);
    }
  } else if (warp < 8) {
    const int q = (32 * (warp - 4) + lane) % C::NQ32;
    const uint32_t lane_base = static_cast<uint32_t>(32 * (warp - 4)) << 16;
#pragma unroll 1
    for (int part = 0; part < 2; ++part) {
      const float* src = tb + (part ? T.PhiL : T.PhiH);
      float v[KP];
#pragma unroll
      for (int j = 0; j < KP / 4; ++j) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(src + tc_canon(q, 4 * j, KP)));
        v[4 * j] = x.x; v[4 * j + 1] = x.y; v[4 * j + 2] = x.z; v[4 * j + 3] = x.w;
      }
      tc::st_cols<KP>(tmem + lane_base + (part ? C::COL_PL : C::COL_PH), v);
    }
  }
  if (warp < 8) tc::wait_st();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();

  // roles: workers, MMA warps, copy warps.  Named barriers: workers with the MMA warp, with the copy
  // warp, among themselves (1..6), the law's warps of one element (7..14)
  constexpr int MMA0 = C::TEAMS * C::WORK_WARPS, COPY0 = MMA0 + C::TEAMS;
  const int team = warp >= COPY0 ? warp - COPY0 : (warp >= MMA0 ? warp - MMA0 : warp / C::WORK_WARPS);
  const int bar_mma = 1 + team, bar_copy = 3 + team, bar_work = 5 + team;
  float* sm = reinterpret_cast<float*>(smem4) + team * C::TEAM_SMEM;
  uint64_t* mbar = &mbars[team];
  TeamStop& stop = stops[team];
  const uint32_t dcol = tmem + team * C::DC;
  float* sBvH = sm + C::oOp;
  float* sBvL = sBvH + C::BV;
  float* sBpH = sm + C::oOp;
  float* sBpL = sBpH + C::BP;

  const int64_t ntiles = (a.E + TE - 1) / TE;
  const int64_t first = static_cast<int64_t>(team) * gridDim.x + blockIdx.x;
  const int64_t step = static_cast<int64_t>(C::TEAMS) * gridDim.x;

  if (warp >= COPY0) {
    // 16-byte asynchronous copies of a tile: state, predictor output, face records (at the face ids
    // `ids`), GeomF, MatF, face ids, and the face ids of the team's tile after it
    auto issue = [&](int64_t tl, float* buf, const int* ids) {
      const int64_t e0 = tl * TE;
      const int ne = static_cast<int>(min(static_cast<int64_t>(TE), a.E - e0));
      for (int c = lane; c < ne * QS / 4; c += 32) tc::cp_async16(buf + C::bQ + 4 * c, a.q_in + e0 * QS + 4 * c);
      for (int c = lane; c < ne * DS / 4; c += 32) tc::cp_async16(buf + C::bD + 4 * c, a.d + e0 * DS + 4 * c);
      for (int ef = 0; ef < 4 * ne; ++ef) {
        const float* src = a.ff + static_cast<int64_t>(ids[ef] >> 1) * FFS;
        float* dst = buf + C::bF + (ef >> 2) * C::FES + (ef & 3) * FFS;
        for (int c = lane; c < FFS / 4; c += 32) tc::cp_async16(dst + 4 * c, src + 4 * c);
      }
      for (int c = lane; c < ne * 8; c += 32) tc::cp_async16(buf + C::bG + 4 * c, reinterpret_cast<const float*>(a.geom + e0) + 4 * c);
      if (lane < ne * 2) tc::cp_async16(buf + C::bM + 4 * lane, reinterpret_cast<const float*>(a.mat + e0) + 4 * lane);
      if (lane < ne) tc::cp_async16(buf + C::bE + 4 * lane, a.elem_face + (e0 + lane) * 4);
      const int64_t n0 = e0 + step * TE;
      if (lane < TE && n0 + lane < a.E) tc::cp_async16(buf + C::bI + 4 * lane, a.elem_face + (n0 + lane) * 4);
    };
    // the previous kernels' results reach the other warps through this one
    tc::pdl_wait();
    int64_t tile = first;
    if (tile < ntiles) issue(tile, sm + C::oBuf, a.elem_face + tile * TE * 4);
    for (int it = 0;; tile += step, ++it) {
      tc::cp_async_wait_all();                 // this tile's copies have landed
      tc::named_barrier(bar_copy, C::TEAM_THREADS);   // the workers start on it; the other buffer is free
      if (stop.copy_stops(it)) break;
      if (tile + step < ntiles)
        issue(tile + step, sm + C::oBuf + ((it + 1) & 1) * C::BUF,
              reinterpret_cast<const int*>(sm + C::oBuf + (it & 1) * C::BUF + C::bI));
    }
  } else if (warp >= MMA0) {
    // volume MMAs, then projection MMAs, each batch when the workers' operand is ready
    for (int n = 0;; n += 2) {
      tc::named_barrier(bar_mma, C::TEAM_THREADS);
      if (stop.mma_stops(n)) break;
      if (lane == 0) {
        tc::fence_after();
        constexpr uint32_t id0 = tc::idesc_tf32(128, N0), idh = tc::idesc_tf32(128, NH);
        const uint32_t bH = tc::smem_u32(sBvH), bL = tc::smem_u32(sBvL);
#pragma unroll
        for (int ks = 0; ks < KP / 8; ++ks) {
          const uint32_t off = ks * 256;   // 8 K-elements = 2 core matrices
          const uint32_t aH = tmem + C::COL_PH + 8 * ks, aL = tmem + C::COL_PL + 8 * ks;
          tc::mma_tf32_ta(dcol, aH, tc::desc_kmajor(bH + off, KP), id0, ks > 0 ? 1u : 0u);
          tc::mma_tf32_ta(dcol, aH, tc::desc_kmajor(bL + off, KP), id0, 1u);
          tc::mma_tf32_ta(dcol, aL, tc::desc_kmajor(bH + off, KP), id0, 1u);
        }
#pragma unroll
        for (int ks = 0; ks < KH / 8; ++ks) {
          const uint32_t off = 4 * N0 * KP + ks * 256;
          const uint32_t aH = tmem + C::COL_PH + 8 * ks, aL = tmem + C::COL_PL + 8 * ks;
          tc::mma_tf32_ta(dcol + N0, aH, tc::desc_kmajor(bH + off, KH), idh, ks > 0 ? 1u : 0u);
          tc::mma_tf32_ta(dcol + N0, aH, tc::desc_kmajor(bL + off, KH), idh, 1u);
          tc::mma_tf32_ta(dcol + N0, aL, tc::desc_kmajor(bH + off, KH), idh, 1u);
        }
        tc::commit(mbar);
      }
      __syncwarp();
      tc::named_barrier(bar_mma, C::TEAM_THREADS);
      if (stop.mma_stops(n + 1)) break;
      if (lane == 0) {
        tc::fence_after();
        constexpr uint32_t idp = tc::idesc_tf32(128, NPC);
        const uint32_t bH = tc::smem_u32(sBpH), bL = tc::smem_u32(sBpL);
        constexpr uint32_t lbo = 4u * C::PLBO, sbo = 4u * C::PGS;
#pragma unroll
        for (int ks = 0; ks < KQ / 8; ++ks) {
          const uint32_t off = ks * 2 * lbo;
          const uint32_t aa = tmem + C::COL_A + 8 * ks;
          tc::mma_tf32_ta(dcol, aa, tc::desc_kmajor_strided(bH + off, lbo, sbo), idp, ks > 0 ? 1u : 0u);
          tc::mma_tf32_ta(dcol, aa, tc::desc_kmajor_strided(bL + off, lbo, sbo), idp, 1u);
        }
        tc::commit(mbar);
      }
      __syncwarp();
    }
  } else {
    const int w = warp % C::WORK_WARPS, tid = 32 * w + lane;
    float* sV = sm + C::oV;
    float* sT = sm + C::oT;
    float* sA = sm + C::oA;
    float* sGeo = sm + C::oGeo;
    float* sC = sm + C::oC;
    uint32_t phase = 0;
    bool failed = false;
    float dto[N + 1];                          // dt^o
    dto[0] = 1.f;
#pragma unroll
    for (int o = 1; o <= N; ++o) dto[o] = dto[o - 1] * dt;
    // the update's row padding stays zero
    if (tid < TE * (QS - 10 * L)) sA[tid / (QS - 10 * L > 0 ? QS - 10 * L : 1) * QS + 10 * L + tid % (QS - 10 * L > 0 ? QS - 10 * L : 1)] = 0.f;
    int it = 0;
    for (int64_t tile = first; tile < ntiles; tile += step, ++it) {
      const int64_t e0 = tile * TE;
      const int ne = static_cast<int>(min(static_cast<int64_t>(TE), a.E - e0));
      float* buf = sm + C::oBuf + (it & 1) * C::BUF;
      const float* sQ = buf + C::bQ;
      const float* sD = buf + C::bD;
      tc::named_barrier(bar_copy, C::TEAM_THREADS);   // this tile's data are there; the previous tile is done

      // ---- 1. volume operand (order o scaled by dt^o), time-integrated velocity, element data
      {
        const int c = lane >> 2, l4 = lane & 3;
        // order 0: the 8-row group of an element, rows c = six strains, alpha, its rate
        {
          const int e = w % TE;
          const float* src = c == 7 ? sD + e * DS + AOFF : sQ + e * QS + (c == 6 ? 9 : c);
          const int st = c == 7 ? 1 : 10;
          const float sc = e >= ne ? 0.f : (c == 7 ? dt : 1.f);
          constexpr int LQS = C::WORK_WARPS / TE, CNT = (KP / 4 + LQS - 1) / LQS;
          float x[CNT];
#pragma unroll
          for (int k = 0; k < CNT; ++k) {
            const int l = 4 * (w / TE + k * LQS) + l4;
            x[k] = l < L ? sc * src[l * st] : 0.f;
          }
#pragma unroll
          for (int k = 0; k < CNT; ++k) {
            const int lq = w / TE + k * LQS;
            const float h = tc::tf32_hi(x[k]);
            const int idx = e * 8 * KP + lq * 32 + lane;
            if (lq < KP / 4) {
              sBvH[idx] = h;
              sBvL[idx] = tc::tf32_hi(x[k] - h);
            }
          }
        }
        // orders o >= 1: rows (element, strain) of an order, GH groups each; warps beyond the last
        // whole round share its groups by K
        auto high = [&](int hg, auto shared) {
          const int o = 1 + hg / C::GH, j = (hg - (o - 1) * C::GH) * 8 + c;
          const int e = j / 6, f = j - 6 * e;
          int off = 0, lim = 0;
          float sc = 0.f;
#pragma unroll
          for (int k = 1; k < N; ++k)
            if (o == k) {
              off = d_offset(N, k);
              lim = n_modes(N - k);
              sc = dto[k];
            }
          if (e >= ne) lim = 0;
          const float* src = sD + e * DS + off + f;
          constexpr bool kShared = decltype(shared)::value;   // the group's K over the team's warps
          constexpr int CNT = kShared ? 1 : KH / 4;
          float x[CNT];
#pragma unroll
          for (int k = 0; k < CNT; ++k) {
            const int l = 4 * (kShared ? w : k) + l4;
            x[k] = l < lim ? sc * src[l * 9] : 0.f;
          }
#pragma unroll
          for (int k = 0; k < CNT; ++k) {
            const int lq = kShared ? w : k;
            const float h = tc::tf32_hi(x[k]);
            const int idx = N0 * KP + hg * 8 * KH + lq * 32 + lane;
            if (lq < KH / 4) {
              sBvH[idx] = h;
              sBvL[idx] = tc::tf32_hi(x[k] - h);
            }
          }
        };
        constexpr int HG = (N - 1) * C::GH, FULL = HG / C::WORK_WARPS * C::WORK_WARPS;
#pragma unroll
        for (int hg = 0; hg < FULL; hg += C::WORK_WARPS) high(hg + w, std::false_type{});
        if constexpr (HG - FULL == 1) high(FULL, std::true_type{});
        else if (FULL + w < HG) high(FULL + w, std::false_type{});
      }
      for (int k = tid; k < LI * 3 * TE; k += C::WORKERS) {
        const int l = k / (3 * TE), ec = k - l * 3 * TE, e = ec / 3;
        sV[l * VS + ec] = e < ne ? velocity_integral<N>(sQ + e * QS, sD + e * DS, l, ec - 3 * e, dt) : 0.f;
      }
      // per element: -dt Theta^{-1} / rho [0, 9), Theta^{-1} [9, 18), material [20, 28), -(signed |S_f| / |J|)
      // [28, 32), strains of order N at every node [32, 38) (mode 0 only, phi_0 = sqrt(6); scaled by dt^N)
      for (int k = tid; k < TE * 40; k += C::WORKERS) {
        const int e = k / 40, c = k - 40 * e;
        float v = 0.f;
        if (e < ne) {
          const float* g = buf + C::bG + e * 32;
          const float* m = buf + C::bM + e * 8;
          if (c < 9) v = -dt * m[6] * g[c];
          else if (c < 18) v = g[c - 9];
          else if (c >= 32) v = c < 38 ? 2.449489742783178f * dto[N] * sD[e * DS + d_offset(N, N) + c - 32] : 0.f;
          else if (c >= 28) v = g[12 + 4 * (c - 28) + 3] * ((__float_as_int(buf[C::bE + e * 4 + c - 28]) & 1) ? 1.f : -1.f);
          else if (c >= 20) v = m[c - 20];
        }
        sGeo[k] = v;
      }
      tc::fence_smem_to_async();
      tc::fence_before();
      tc::named_barrier(bar_mma, C::TEAM_THREADS);   // the issuing warp starts the volume MMAs

      // ---- 2. face lift and strain rows
      {
        constexpr int COLS = 8 * TE, GROUPS = COLS / 32;   // fields 0..7, then field 8 of every element
        for (int u = w; u < (GROUPS + 1) * C::NBLK; u += C::WORK_WARPS) {
          const int g = u / C::NBLK, b = u - g * C::NBLK;
          const int col = 32 * g + lane;
          const int e = g < GROUPS ? col >> 3 : lane, p = g < GROUPS ? col & 7 : 8;
          if (e < ne) {
            const float* f0 = buf + C::bF + e * C::FES + p;
            const float* const F[4] = {f0, f0 + FFS, f0 + 2 * FFS, f0 + 3 * FFS};
            lift_and_strain<C, N, 0>(b, p, sGeo + e * 40, F, sV + 3 * e, sA + e * QS + p);
          }
        }
      }
      {
        const bool ok = tc::wait_parity(mbar, phase, wait_limit);
        phase ^= 1u;
        if (tc::named_barrier_or(bar_work, C::WORKERS, !ok)) {
          if (tid == 0) stop.set(it, 1);
          failed = true;
          break;
        }
      }
      tc::fence_after();

      // ---- 3. pointwise law
      {
        const int wq = w & 3, q = 32 * (wq % C::WPE) + lane;
        const int grp = (w >> 2) * C::REP + wq / C::WPE;
        const uint32_t tcol = dcol + (static_cast<uint32_t>(32 * wq) << 16);
#pragma unroll 1
        for (int r = 0; r < C::ROUNDS; ++r) {
          const int e = grp * C::ROUNDS + r;
          float v0[8], vh[N][8];
          tc::ld_x8(tcol + 8 * e, v0);
#pragma unroll
          for (int o = 1; o < N; ++o) tc::ld_x8(tcol + N0 + 6 * TE * (o - 1) + 6 * e, vh[o - 1]);
          tc::wait_ld();
          float out[10];
#pragma unroll
          for (int c = 0; c < 10; ++c) out[c] = 0.f;
          if (q < NQ && e < ne) {
            const float* gm = sGeo + e * 40;
            const float4 m0 = *reinterpret_cast<const float4*>(gm + 20), m1 = *reinterpret_cast<const float4*>(gm + 24);
            const MatF m{m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, 0.f};
#pragma unroll
            for (int p = 0; p < 6; ++p) vh[N - 1][p] = gm[32 + p];
            float sb[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f}, ib = 0.f, rb = 0.f;
            auto node = [&](float gz, float c1, float c2, float c3, float c4) {
              const float cz[4] = {c1, c2, c3, c4};
              float eps[6];
#pragma unroll
              for (int p = 0; p < 6; ++p) {
                eps[p] = v0[p];
#pragma unroll
                for (int o = 1; o <= N; ++o) eps[p] = fmaf(cz[o - 1], vh[o - 1][p], eps[p]);
              }
              float iso, sh, rate;
              law_moduli<LAW>(a.law, eps, fmaf(c1, v0[7], v0[6]), m, &iso, &sh, &rate);
              ib = fmaf(gz, iso, ib);
              rb = fmaf(gz, rate, rb);
              sh *= gz;
#pragma unroll
              for (int p = 0; p < 6; ++p) sb[p] = fmaf(sh, eps[p], sb[p]);
            };
#define DG_Z(z, gz, c1, c2, c3, c4, c5) node(gz, c1, c2, c3, c4);
            if constexpr (N == 2) { DG_TIME_2(DG_Z) }
            else if constexpr (N == 3) { DG_TIME_3(DG_Z) }
            else { DG_TIME_4(DG_Z) }
#undef DG_Z
            const float S[3][3] = {{sb[0] + ib, sb[3], sb[5]}, {sb[3], sb[1] + ib, sb[4]}, {sb[5], sb[4], sb[2] + ib}};
#pragma unroll
            for (int ep = 0; ep < 3; ++ep) {
              const float t0 = gm[3 * ep], t1 = gm[3 * ep + 1], t2 = gm[3 * ep + 2];
#pragma unroll
              for (int mc = 0; mc < 3; ++mc) out[ep * 3 + mc] = fmaf(t0, S[mc][0], fmaf(t1, S[mc][1], t2 * S[mc][2]));
            }
            out[9] = dt * rb;
          }
          if (q == 0) {
#pragma unroll
            for (int c = 0; c < 10; ++c) sC[e * 12 + c] = out[c];
          }
          if constexpr (C::WPE == 1) __syncwarp();
          else tc::named_barrier(7 + 2 * C::REP * team + grp, 32 * C::WPE);
#pragma unroll
          for (int c = 0; c < 10; ++c) {
            const float x = q < NQ ? out[c] - sC[e * 12 + c] : 0.f;
            // prj_canon(prj_col(c, e), q): the columns of one element differ by constants
            const int idx = C::prj_canon(C::prj_col(c, 0), 0) + 4 * e + (q >> 2) * C::PLBO + (q & 3);
            const float h = tc::tf32_hi(x);
            sBpH[idx] = h;
            sBpL[idx] = tc::tf32_hi(x - h);
          }
        }
      }
      tc::fence_smem_to_async();
      tc::fence_before();
      tc::named_barrier(bar_mma, C::TEAM_THREADS);   // the issuing warp starts the projection MMAs

      // ---- 4. the projection
      {
        const bool ok = tc::wait_parity(mbar, phase, wait_limit);
        phase ^= 1u;
        if (tc::named_barrier_or(bar_work, C::WORKERS, !ok)) {
          if (tid == 0) stop.set(it, 2);
          failed = true;
          break;
        }
      }
      tc::fence_after();

      // ---- 5. read-out: lane quarters 0, 1 hold the products of A's TF32 part (with the node-0 values
      // back through the row sums), 2, 3 those of its remainder; half the terms c each per four warps
      {
        const int wq = w & 3, l = 32 * (wq & 1) + lane, c0 = w >> 2 ? 5 : 0;
        constexpr int CH = 5 * TE;
        float v[CH];
        const uint32_t src = dcol + (static_cast<uint32_t>(32 * wq) << 16) + c0 * TE;
        if constexpr (CH == 20) {
          tc::ld_x16(src, v);
          tc::ld_x4(src + 16, v + 16);
        } else {
          tc::ld_cols<CH>(src, v);
        }
        tc::wait_ld();
        // the term's row: T_e'm at (c = 3 e' + m), the rate (c = 9) into the update
        auto dst = [&](int c, int e) {
          return c < 9 ? sT + ((c / 3) * LI + l) * VS + e * 3 + c % 3 : sA + e * QS + l * 10 + 9;
        };
        if (wq < 2 && l < L) {
#pragma unroll
          for (int j = 0; j < 5; ++j)
            if (l < LI || c0 + j == 9) {
#pragma unroll
              for (int e = 0; e < TE; ++e) *dst(c0 + j, e) = fmaf(sC[e * 12 + c0 + j], row_sum, v[j * TE + e]);
            }
        }
        tc::fence_before();
        tc::named_barrier(bar_work, C::WORKERS);
        if (wq >= 2 && l < L) {
#pragma unroll
          for (int j = 0; j < 5; ++j)
            if (l < LI || c0 + j == 9) {
#pragma unroll
              for (int e = 0; e < TE; ++e) *dst(c0 + j, e) += v[j * TE + e];
            }
        }
      }
      tc::named_barrier(bar_work, C::WORKERS);
      if (w < C::VBLK && lane < 3 * ne)
        velocity_derivative<C, N, 0>(w, sT + lane, sA + (lane / 3) * QS + 6 + lane % 3);
      tc::named_barrier(bar_work, C::WORKERS);
      // update
      bool bad = false;
#pragma unroll
      for (int k0 = 0; k0 < TE * QS / 4; k0 += C::WORKERS) {
        const int k = k0 + tid;
        if (k < ne * QS / 4) {
          const float4 q = reinterpret_cast<const float4*>(sQ)[k], d = reinterpret_cast<const float4*>(sA)[k];
          const float4 v = make_float4(q.x + d.x, q.y + d.y, q.z + d.z, q.w + d.w);
          bad |= !(fmaf(v.x, 0.f, fmaf(v.y, 0.f, fmaf(v.z, 0.f, v.w * 0.f))) == 0.f);   // NaN for any non-finite value
          reinterpret_cast<float4*>(a.q_out + e0 * QS)[k] = v;
        }
      }
      if (bad) atomicOr(a.status, kStatusNonFinite);
    }
    if (failed) {
      if (tid == 0) atomicOr(a.status, kStatusTimeout);
      tc::wait_parity(mbar, phase ^ 1u, kWaitLimit);   // let the MMAs in flight finish before freeing TMEM
    }
    if (tid == 0 && !failed) stop.set(it, 0);
    __threadfence_block();
    tc::named_barrier(bar_mma, C::TEAM_THREADS);       // releases the MMA warp
    tc::named_barrier(bar_copy, C::TEAM_THREADS);      // and the copy warp
  }
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::dealloc(tmem, C::TMEM_COLS);
}

}  // namespace dg
