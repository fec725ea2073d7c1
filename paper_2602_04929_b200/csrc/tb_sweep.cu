// Column sweep (Algorithm 2; Eq. 2): rows against the upper factor U (and P of the propagated-error term).
//
// Rows never interact inside the sweep; a CTA keeps R = 8, 16 or 32 of them.  Left-looking over blocks of 128 columns:
//   w[:, b] = W0[:, b] - Err[:, < b] U[< b, b]  (- Arr[:, < b] P[< b, b]),
// Err the normalised errors and Arr the arrival values of the columns already quantized.
//
// A row is a chain of dependent roundings, column after column; the chain bounds a launch of few rows, the FP64 pipe
// one of many.  One warp walks it, ONE THREAD PER ROW, 16 columns in registers, in units of the row's scale:
//   x = v + z;  q = clamp(round(x));  v' = v_next - x U' + q U',   U' = U[j][j+1] / U[j][j],
// so that only add (rounds), integer clamp, add (back to double) and multiply-add lie between two columns: 33 clocks
// measured, 58 with the other multiply-adds of a 16-column piece (56 to 60 over 8 to 4096 rows; 93 with P; a warp per row with the column's error broadcast
// by shuffles, as it was, takes 88 and 150).  Whether a value lies outside the 31 bits that the integer clamp
// sees is only looked at after a piece; such a piece is walked again with the test in the chain.
// That warp has its scheduler for itself: beside FP64 tensor steps of the same scheduler a dependent multiply-add
// takes 137 clocks instead of 9.  The other three schedulers run, at the same time,
//   spread   (4 warps) after each piece: its errors onto the block's later columns, the next piece first; codes,
//            histories and counters
//   history  (8 warps) the next block's contraction over the earlier columns: chunks of U (and P) and of the histories
//            arrive by TMA in a ring guarded by full / empty mbarriers and feed mma.sync m8n8k4 f64 (the cluster form,
//            whose share of a chunk is small, reads them straight into registers); the block being walked
//            comes last, piece by piece; before that the next block's grids and 16 x 16 triangles of U'
// and a warp beside the chain issues the TMA loads.
// The groups meet at hardware barriers with fixed counts; every trip count depends on the block index alone.  mbarrier
// waits are bounded: when a bound runs out the kernel raises a device error word and stops computing, but still
// passes every barrier, so it terminates.
//
// Cluster form (CLUSTER), for few rows: cs CTAs share a group of 8 rows.  Each contracts the history for 128 / cs
// columns of the next block and writes them into the buffers of all (distributed shared memory, two buffers in
// turn); after one cluster barrier the chain of the block runs in every CTA on identical values, so no result has
// to travel back and all of them write the same outputs.
#include <cooperative_groups.h>

#include "tb_gemm.cuh"
#include "tb_rows.cuh"
#include "tb_tma.cuh"

namespace cg = cooperative_groups;

namespace tb {

enum { SW_THREADS = 512, SW_LDB = 136, SW_LDW = 132, SW_HIST = 8, SW_SPREAD = 4 };

struct SweepP {
  SweepArgs a;
  int rows_per_unit, ctas_per_unit;
  int cs;  // CTAs per cluster (CLUSTER)
};

template <bool WITH_P, int R>
struct SweepSmem {
  static constexpr int CHUNK = (R == 32 || (R == 16 && WITH_P)) ? 32 : 64;
  static constexpr int STAGES = (R == 8) ? (WITH_P ? 2 : 4) : 3;
  struct Stage {
    float Ub[CHUNK][SW_LDB];       // rows of U or P: 128 columns of the target block + 8 spare
    double Eb[R][CHUNK + 4];       // the same contraction columns of a history (+ 4 spare)
  };
  alignas(128) Stage ring[STAGES];  // TMA destinations (not in the cluster form)
  alignas(16) double w[2][R][SW_LDW];   // values of a block; walked columns hold arrival value / scale
  alignas(16) double Es[R][SW_LDW];     // normalised errors of the block
  alignas(16) double As[WITH_P ? R : 1][SW_LDW];  // arrival values of the block
  alignas(16) double cU[2][8][16][16];  // U[j][c] / U[j][j] of the 16-column pieces, zero for c <= j
  alignas(16) double cP[WITH_P ? 2 : 1][WITH_P ? 8 : 1][16][16];
  alignas(16) double part[R == 8 ? 512 : 2];  // partial sums of the contraction's split (cluster form)
  alignas(16) double rd[2][128];        // 1 / U[j][j]
  double gs[2][R][4][3];                // scale, its reciprocal and zero-point per row and 32 columns
  long long row[R];                     // first element of a row in the matrix of codes
  unsigned long long full_bar[8], empty_bar[8];
  int abort_flag;
};

__device__ int g_sweep_error = 0;

template <int N>
__device__ __forceinline__ void sw_sync(int id) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(N) : "memory");
}
template <int N>
__device__ __forceinline__ void sw_arrive(int id) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(N) : "memory");
}
enum { SW_PUB = 1, SW_READY = 3, SW_JOIN = 5, SW_PIECE = 8 };  // two, two, one, eight hardware barriers

// Quantized integer (sw_quant: as a double) of xm = v + z + 1.5 * 2^52: that sum was rounded to nearest-even and holds the
// integer in its low word, where the clamp is one integer instruction.  The low word alone is the integer only below
// 2^31 in magnitude; the high word tells (it is the constant's, or one less for a negative integer, exactly when the
// low word's sign says the same).  CHECKED: beyond that range, infinities included, the code saturates like the clamp
// of the full value, and is 0 for what is no number (a NaN's high word is above infinity's); otherwise `off` becomes
// nonzero there.
template <bool CHECKED>
__device__ __forceinline__ int sw_code(double xm, int maxq, int& off) {
  const int lo = __double2loint(xm), hi = __double2hiint(xm);
  const int hw = (int)((unsigned)hi - 0x43380000u);  // modulo 2^32: a negative xm has a high word far below
  int n = __vimin_s32_relu(lo, maxq);
  if (CHECKED)
    n = (hw == (lo >> 31)) ? n : (((unsigned)hw <= 0x7ff00000u - 0x43380000u) ? maxq : 0);  // up to infinity
  else
    off |= hw ^ (lo >> 31);
  return n;
}
template <bool CHECKED>
__device__ __forceinline__ double sw_quant(double xm, int maxq, int& off) {
  return __hiloint2double(0x43380000, sw_code<CHECKED>(xm, maxq, off)) - 6755399441055744.0;
}

// Code of arrival value v (in units of the scale) as the chain took it, and the two counters.  Near a tie: rounding moved the
// value by almost half a code, and the clamp leaves both neighbours apart.  Clamped: the rounded value is not the code.
__device__ __forceinline__ int sw_output(double v, double z, int maxq, unsigned int& n_near, unsigned int& n_clamp) {
  const double x = v + z, xm = v + (z + 6755399441055744.0);  // the chain's own operations
  int unused = 0;
  const int n = sw_code<true>(xm, maxq, unused);
  const int lo = __double2loint(xm), hw = (int)((unsigned)__double2hiint(xm) - 0x43380000u);
  if (fabs(x - (xm - 6755399441055744.0)) > 0.5 - 1e-6 && x > 0.0 && x < (double)maxq) ++n_near;
  if (lo != n || hw != (lo >> 31)) ++n_clamp;
  return n;
}

// Shared-memory accesses that the compiler leaves in their order: by itself it moves all of a piece's factor loads to
// its beginning and spills them (78 clocks a column instead of 58).
__device__ __forceinline__ double2 sw_ld2(const double* p) {
  double2 v;
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ double sw_ld1(const double* p) {
  double v;
  asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(smem_u32(p)) : "memory");
  return v;
}
__device__ __forceinline__ void sw_st2(double* p, double x, double y) {
  asm volatile("st.shared.v2.f64 [%0], {%1, %2};" ::"r"(smem_u32(p)), "d"(x), "d"(y) : "memory");
}

// 16 columns of one row in registers, in units of its scale s.  v: values, on return on arrival.  The normalised errors
// e s / U_jj go to er two at a time (kept for the end they would cost the registers that the walk needs).
template <bool WITH_P, bool CHECKED>
__device__ __forceinline__ int sw_walk(double (&v)[16], double* er, double s, double z, int maxq, const double* rd,
                                       const double (*cu)[16], const double (*cp)[16]) {
  const double zm = z + 6755399441055744.0;
  int off = 0;
  double x = v[0] + z, xm = v[0] + zm, e_even = 0.0;
  double2 cur[8], nxt[8];  // factors of the column and of the next one, loaded a column ahead
#pragma unroll
  for (int c = 0; c < 8; ++c) cur[c] = sw_ld2(&cu[0][2 * c]);
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    auto u = [&](int c) { return (c & 1) ? cur[c >> 1].y : cur[c >> 1].x; };
    double q, xn = 0.0, xmn = 0.0;
    if (j < 15) {
#pragma unroll
      for (int c = (j + 2) >> 1; c < 8; ++c) nxt[c] = sw_ld2(&cu[j + 1][2 * c]);
      double t = fma(-x, u(j + 1), v[j + 1]);
      if (WITH_P) t = fma(-v[j], sw_ld1(&cp[j][j + 1]), t);
      q = sw_quant<CHECKED>(xm, maxq, off);
      v[j + 1] = fma(q, u(j + 1), t);
      xn = v[j + 1] + z;
      xmn = v[j + 1] + zm;
    } else {
      q = sw_quant<CHECKED>(xm, maxq, off);
    }
    const double e = x - q;
#pragma unroll
    for (int c = j + 2; c < 16; ++c) v[c] = fma(-e, u(c), v[c]);
    if (WITH_P) {
      if ((j & 1) && j + 2 < 16) v[j + 2] = fma(-v[j], sw_ld1(&cp[j][j + 2]), v[j + 2]);
#pragma unroll
      for (int c = (j + 3) & ~1; c < 16; c += 2) {
        const double2 pc = sw_ld2(&cp[j][c]);
        v[c] = fma(-v[j], pc.x, v[c]);
        v[c + 1] = fma(-v[j], pc.y, v[c + 1]);
      }
    }
    if (j & 1) {
      const double2 r = sw_ld2(rd + j - 1);
      sw_st2(er + j - 1, e_even * (s * r.x), e * (s * r.y));
    }
    e_even = e;
    x = xn;
    xm = xmn;
#pragma unroll
    for (int c = 0; c < 8; ++c) cur[c] = nxt[c];
  }
  return off;
}

template <bool WITH_P, int R, bool CLUSTER>
__global__ void __launch_bounds__(SW_THREADS, 1)
    k_sweep_rows(SweepP p, const __grid_constant__ CUtensorMap map_u, const __grid_constant__ CUtensorMap map_e,
                 const __grid_constant__ CUtensorMap map_p, const __grid_constant__ CUtensorMap map_a) {
  static_assert(!CLUSTER || R == 8, "a cluster shares 8 rows");
  extern __shared__ __align__(128) unsigned char sw_raw[];
  using Smem = SweepSmem<WITH_P, R>;
  constexpr int NOP = WITH_P ? 2 : 1;  // operand pairs per chunk: (Err, U) and (Arr, P)
  constexpr int MF = R / 8;
  Smem& sm = *reinterpret_cast<Smem*>(sw_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int fr = lane >> 2, fk = lane & 3;  // fragment row (or column) and k index of this lane
  const SweepArgs& a = p.a;
  const int d = a.d;
  const int cs = CLUSTER ? p.cs : 1;
  const int crank = CLUSTER ? (int)cg::this_cluster().block_rank() : 0;
  const int grp = blockIdx.x / cs;
  const int unit = grp / p.ctas_per_unit, r_first = (grp % p.ctas_per_unit) * R;
  const int rows_here = min(R, p.rows_per_unit - r_first);
  const int m_base = unit * p.rows_per_unit + r_first;
  const long long uoff = (a.units > 1) ? (long long)unit * d * d : 0;
  const float* U = a.U + uoff;
  const float* Pm = WITH_P ? a.P + uoff : nullptr;
  auto src_row = [&](int r) { return (a.src_mapped ? a.rm.row(m_base + r) : (long long)(m_base + r)) * d; };

  // ring of history chunks
  constexpr int ch = Smem::CHUNK, ldb = SW_LDB, lde = ch + 4;  // the cluster form has none
  constexpr int ub_bytes = ch * ldb * (int)sizeof(float), eb_bytes = R * lde * (int)sizeof(double);
  constexpr int stage_bytes = ub_bytes + eb_bytes, stages = Smem::STAGES;
  constexpr int per_blk = (128 / ch) * NOP;  // chunks per 128 contraction rows
  unsigned char* ring = reinterpret_cast<unsigned char*>(&sm.ring[0]);
  volatile int* abort_flag = &sm.abort_flag;

  // What a block needs besides its values, by threads t of nt, in two parts with a barrier between: grids and 1 / U_jj,
  // then the scaled triangles (consecutive threads on consecutive columns: a thread per row would meet 32-way bank
  // conflicts, and the chain's own loads with them)
  auto prepare_pivots = [&](int b, int t, int nt) {
    for (int j = t; j < 128; j += nt) sm.rd[b & 1][j] = 1.0 / (double)U[(long long)(b * 128 + j) * (d + 1)];
  };
  auto prepare_scales = [&](int b, int t, int nt) {
    const int pb = b & 1, c0 = b * 128;
    for (int i = t; i < R * 4; i += nt) {
      const int r = i >> 2, sb = i & 3;
      double s = 1.0, z = 0.0;
      if (r < rows_here) {  // 32 columns lie in one group: groups are multiples of 32 columns
        const long long so = a.rm.row(m_base + r) * a.ng + (c0 + 32 * sb) / a.seg;
        s = a.sD[so];
        z = (double)a.z[so];
      }
      sm.gs[pb][r][sb][0] = s;
      sm.gs[pb][r][sb][1] = 1.0 / s;
      sm.gs[pb][r][sb][2] = z;
    }
  };
  auto prepare_triangles = [&](int b, int t, int nt) {
    const int pb = b & 1, c0 = b * 128;
#pragma unroll 4
    for (int i = t; i < 128 * 16; i += nt) {
      const int j = i >> 4, c = i & 15, jl = j & 15;
      const long long o = (long long)(c0 + j) * d + c0 + (j & ~15) + c;
      sm.cU[pb][j >> 4][jl][c] = (c > jl) ? (double)U[o] * sm.rd[pb][j] : 0.0;
      if (WITH_P) sm.cP[pb][j >> 4][WITH_P ? jl : 0][c] = (c > jl) ? (double)Pm[o] : 0.0;
    }
  };

  if (tid == 0) {
    for (int s = 0; s < 8; ++s) {
      mbar_init(smem_u32(&sm.full_bar[s]), 1);
      mbar_init(smem_u32(&sm.empty_bar[s]), SW_HIST);
    }
    sm.abort_flag = 0;
    mbar_fence_init();
  }
  if (tid < R) sm.row[tid] = a.rm.row(m_base + min(tid, rows_here - 1)) * d;
  // the first block: what depends on the factors alone, then, behind the kernel before, its values and grids
  prepare_pivots(a.blk0, tid, SW_THREADS);
  __syncthreads();
  prepare_triangles(a.blk0, tid, SW_THREADS);
  pdl_wait();
  for (int i = tid; i < R * 128; i += SW_THREADS) {  // the first block arrives unchanged
    const int r = i >> 7, c = i & 127;
    sm.w[a.blk0 & 1][r][c] = (r < rows_here) ? a.src[src_row(r) + a.blk0 * 128 + c] : 0.0;
  }
  prepare_scales(a.blk0, tid, SW_THREADS);
  __syncthreads();
  if (CLUSTER) cg::this_cluster().sync();  // every CTA of the cluster runs before anybody writes into it
  auto next_block = [&]() {  // block b + 1 has been handed over (by all CTAs of the cluster)
    if (CLUSTER)
      cg::this_cluster().sync();
    else
      __syncthreads();
  };

  if (warp == 0) {
    // =========================== the chain: lane = row ===========================
    const int r = lane & (R - 1);  // with fewer than 32 rows several lanes do the same
#pragma unroll 1
    for (int b = a.blk0; b < a.blk1; ++b) {
      const int pb = b & 1;
      const bool more = b + 1 < a.blk1;
      if (!more) pdl_trigger();
#pragma unroll 1
      for (int sb = 0; sb < 8; ++sb) {
        const double* g = sm.gs[pb][r][sb >> 1];
        const double s = g[0], rs = g[1], z = g[2];
        double* wr = &sm.w[pb][r][16 * sb];
        double* er = &sm.Es[r][16 * sb];
        double v[16];
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
          const double2 t = *reinterpret_cast<const double2*>(wr + j);
          v[j] = t.x * rs;
          v[j + 1] = t.y * rs;
        }
        const int off = sw_walk<WITH_P, false>(v, er, s, z, a.maxq, &sm.rd[pb][16 * sb], sm.cU[pb][sb],
                                               sm.cP[WITH_P ? pb : 0][WITH_P ? sb : 0]);
        if (__any_sync(0xffffffffu, off != 0)) {  // again, with the range test in the chain
#pragma unroll
          for (int j = 0; j < 16; j += 2) {
            const double2 t = *reinterpret_cast<const double2*>(wr + j);
            v[j] = t.x * rs;
            v[j + 1] = t.y * rs;
          }
          sw_walk<WITH_P, true>(v, er, s, z, a.maxq, &sm.rd[pb][16 * sb], sm.cU[pb][sb],
                                sm.cP[WITH_P ? pb : 0][WITH_P ? sb : 0]);
        }
        __syncwarp();  // (lanes of one row read its values before one of them overwrites them)
        if (WITH_P) {
#pragma unroll
          for (int j = 0; j < 16; j += 2) sw_st2(&sm.As[r][16 * sb + j], v[j] * s, v[j + 1] * s);
        }
        if (sb >= 6) {
#pragma unroll
          for (int j = 0; j < 16; j += 2) sw_st2(wr + j, v[j], v[j + 1]);
        }
        sw_arrive<32 + 32 * SW_SPREAD>(SW_PUB + (sb & 1));
        if (more) sw_arrive<32 + 32 * SW_HIST>(SW_PIECE + sb);
        if (sb < 6) {  // the arrival values are looked at a piece later, but at the block's end
#pragma unroll
          for (int j = 0; j < 16; j += 2) sw_st2(wr + j, v[j], v[j + 1]);
        }
        if (sb < 7) sw_sync<32 + 32 * SW_SPREAD>(SW_READY + (sb & 1));
      }
      next_block();
    }
    return;
  }

  if (warp == 11 || warp >= 13) {
    // =========================== spread ===========================
    const int sw = (warp == 11) ? 0 : warp - 12, st_tid = sw * 32 + lane;
    unsigned int n_near = 0, n_clamp = 0;
    // fragment (m, n) of the block belongs to warp (n + 2 (m & 1)) & 3: the next piece's fragments to all of them.
    // This warp's columns are n = NS i + n_lo; of each it has all row fragments (8 rows), or those of one parity.
    constexpr int NS = (MF == 1) ? 4 : 2, NI = 16 / NS, MS = (MF == 1) ? 1 : 2;
    const int n_lo = (MF == 1) ? sw : (sw & 1);
    // factor rows of a piece, right of it: fetched a piece ahead
    float u[NI][4], pp[WITH_P ? NI : 1][4], uf[NI][4], pf[WITH_P ? NI : 1][4];
    auto fetch = [&](int b, int sb) {
      const long long o0 = (long long)(b * 128 + 16 * sb + fk) * d + b * 128 + fr;
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const int n = NS * i + n_lo;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (n >= 2 * (sb + 1)) {
            uf[i][q] = U[o0 + (long long)(4 * q) * d + 8 * n];
            if (WITH_P) pf[i][q] = Pm[o0 + (long long)(4 * q) * d + 8 * n];
          }
      }
    };
    // codes, histories and counters of a piece.  With many rows the chain waits for these warps: row offsets are kept (a
    // division each), the counters need no floor, and only the last piece's outputs are left at a block's end (1024 rows of
    // 4096 columns, 8 rows a step, 42.4 -> 40.5 ms; 4096 rows at once 3.65 -> 3.53).
    auto outputs = [&](int b, int sb) {
#pragma unroll
      for (int i = 0; i < R * 16 / 128; ++i) {
        const int idx = st_tid + 128 * i, r = idx >> 4, cl = 16 * sb + (idx & 15), col = b * 128 + cl;
        if (r < rows_here) {
          const double v = sm.w[b & 1][r][cl], z = sm.gs[b & 1][r][sb >> 1][2];
          a.codes[sm.row[r] + col] = (unsigned char)sw_output(v, z, a.maxq, n_near, n_clamp);
          const long long ho = (long long)(m_base + r) * a.err_ld + col - a.err_col0;
          a.Err[ho] = sm.Es[r][cl];
          if (WITH_P) a.Arr[ho] = sm.As[WITH_P ? r : 0][cl];
        }
      }
    };
    fetch(a.blk0, 0);
#pragma unroll 1
    for (int b = a.blk0; b < a.blk1; ++b) {
      const int pb = b & 1;
#pragma unroll 1
      for (int sb = 0; sb < 8; ++sb) {
        const int n1 = 2 * (sb + 1);  // first fragment right of the piece
#pragma unroll
        for (int i = 0; i < NI; ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            u[i][q] = uf[i][q];
            if (WITH_P) pp[WITH_P ? i : 0][q] = pf[WITH_P ? i : 0][q];
          }
        if (sb < 6)
          fetch(b, sb + 1);
        else if (sb == 7 && b + 1 < a.blk1)
          fetch(b + 1, 0);
        // while the piece is being walked: the factor rows that the next piece waits for, negated and as double, and the
        // next piece's values so far
        // this warp's fragment column of the next piece, if any
        const int nn = (MF == 1) ? n1 + ((sw - n1) & 3) : n1 + ((sw ^ n1) & 1);
        const bool first = sb < 7 && (MF > 1 || nn < n1 + 2);
        const int fm0 = (MF == 1) ? 0 : ((sw - nn) & 3) >> 1;
        double nu[4], np[WITH_P ? 4 : 1];
        double2 old[MF / MS];
        if (first) {
#pragma unroll
          for (int i = 0; i < NI; ++i)
            if (NS * i + n_lo == nn)
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                nu[q] = -(double)u[i][q];
                if (WITH_P) np[q] = -(double)pp[WITH_P ? i : 0][q];
              }
#pragma unroll
          for (int mm = 0; mm < MF / MS; ++mm)
            old[mm] = *reinterpret_cast<const double2*>(&sm.w[pb][8 * (fm0 + MS * mm) + fr][8 * nn + 2 * fk]);
        }
        sw_sync<32 + 32 * SW_SPREAD>(SW_PUB + (sb & 1));
        if (sb < 7) {
          if (first) {
#pragma unroll
            for (int mm = 0; mm < MF / MS; ++mm) {
              const int m = fm0 + MS * mm;
              double acc[2][2] = {{old[mm].x, old[mm].y}, {0.0, 0.0}};
#pragma unroll
              for (int q = 0; q < 4; ++q) dmma(acc[q & 1], sm.Es[8 * m + fr][16 * sb + 4 * q + fk], nu[q]);
              if (WITH_P)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                  dmma(acc[q & 1], sm.As[WITH_P ? 8 * m + fr : 0][16 * sb + 4 * q + fk], np[WITH_P ? q : 0]);
              *reinterpret_cast<double2*>(&sm.w[pb][8 * m + fr][8 * nn + 2 * fk]) =
                  make_double2(acc[0][0] + acc[1][0], acc[0][1] + acc[1][1]);
            }
          }
          sw_arrive<32 + 32 * SW_SPREAD>(SW_READY + (sb & 1));
#pragma unroll
          for (int i = 0; i < NI; ++i) {
            const int n = NS * i + n_lo;
            if ((n >> 1) > sb + 1) {
              const int m0 = (MF == 1) ? 0 : ((sw - n) & 3) >> 1;
#pragma unroll
              for (int mm = 0; mm < MF / MS; ++mm) {
                const int m = m0 + MS * mm;
                double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
                for (int q = 0; q < 4; ++q)
                  dmma(acc[q & 1], sm.Es[8 * m + fr][16 * sb + 4 * q + fk], (double)u[i][q]);
                if (WITH_P)
#pragma unroll
                  for (int q = 0; q < 4; ++q)
                    dmma(acc[q & 1], sm.As[WITH_P ? 8 * m + fr : 0][16 * sb + 4 * q + fk], (double)pp[WITH_P ? i : 0][q]);
                double2* wp = reinterpret_cast<double2*>(&sm.w[pb][8 * m + fr][8 * n + 2 * fk]);
                const double2 v = *wp;
                *wp = make_double2(v.x - (acc[0][0] + acc[1][0]), v.y - (acc[0][1] + acc[1][1]));
              }
            }
          }
        }
        if (sb > 0 && sb < 7) outputs(b, sb - 1);
        if (sb >= 6) outputs(b, sb);
      }
      // the histories are read back by TMA (async proxy): order these stores before it
      asm volatile("fence.proxy.async;" ::: "memory");
      next_block();
    }
    if (a.stats && crank == 0) {
      n_near = __reduce_add_sync(0xffffffffu, n_near);
      n_clamp = __reduce_add_sync(0xffffffffu, n_clamp);
      if (lane == 0) {
        if (n_near) atomicAdd(&a.stats->near_tie_codes, (unsigned long long)n_near);
        if (n_clamp) atomicAdd(&a.stats->clamped_codes, (unsigned long long)n_clamp);
        if (grp == 0 && sw == 0) atomicAdd(&a.stats->column_steps, (unsigned long long)(a.blk1 - a.blk0) * 128);
      }
    }
    return;
  }

  if (warp == 4) {
    // =========================== TMA loads ===========================
    const int u_row0 = (a.units > 1) ? unit * d : 0;
    int slot = 0;
    uint32_t phase = 0;
#pragma unroll 1
    for (int b = a.blk0; b < a.blk1; ++b) {
      if (!CLUSTER && lane == 0 && b + 1 < a.blk1) {
        const int n_hist = (b - a.blk0) * per_blk, n_all = n_hist + per_blk;
        for (int c = 0; c < n_all; ++c) {
          unsigned char* stg = ring + (size_t)slot * stage_bytes;
          const uint32_t fb = smem_u32(&sm.full_bar[slot]);
          if (mbar_wait(smem_u32(&sm.empty_bar[slot]), phase ^ 1u, abort_flag, &g_sweep_error)) {
            const bool hist = c < n_hist;  // else the block being walked: its errors are in shared memory
            const bool second = WITH_P && (c & 1);
            const int k0 = a.blk0 * 128 + (c / NOP) * ch;
            mbar_expect_tx(fb, (uint32_t)(ub_bytes + (hist ? eb_bytes : 0)));
            tma_load_2d(smem_u32(stg), second ? &map_p : &map_u, (b + 1) * 128, u_row0 + k0, fb);
            if (hist) tma_load_2d(smem_u32(stg + ub_bytes), second ? &map_a : &map_e, k0 - a.err_col0, m_base, fb);
          }
          if (++slot == stages) {
            slot = 0;
            phase ^= 1u;
          }
        }
      }
      __syncwarp();
      next_block();
    }
    return;
  }

  if (warp == 8 || warp == 12) {  // nothing beside the chain
#pragma unroll 1
    for (int b = a.blk0; b < a.blk1; ++b) next_block();
    return;
  }

  // =========================== history ===========================
  const int hw = (warp < 4) ? warp - 1 : (warp < 8) ? warp - 2 : warp - 3;  // warps 1-3, 5-7, 9, 10
  // columns and share of the contraction of this warp
  const int frags = 16 / cs;                                 // 8-column fragments of this CTA
  const int kgroups = CLUSTER ? max(1, SW_HIST / frags) : 1;  // cluster of 2 and more: one fragment per warp
  const int kg = CLUSTER ? hw / frags : 0;
  const int n_loc = CLUSTER ? (hw % frags) * 8 : hw * 16;
  constexpr int FW = CLUSTER ? 1 : 2;  // fragments per warp
  constexpr int NA = (MF == 1) ? 4 : (MF == 2 ? 2 : 1);  // accumulators per fragment, in turn
  // column of accumulator (fragment t, element e): one 8-byte load feeds both fragments of a warp, so
  // fragment 0 takes the even columns and fragment 1 the odd ones
  auto col_of = [&](int t, int e) { return CLUSTER ? 2 * fk + e : 2 * (2 * fk + e) + t; };
  int slot = 0;
  uint32_t phase = 0;
#pragma unroll 1
  for (int b = a.blk0; b < a.blk1; ++b) {
    if (b + 1 >= a.blk1) {
      next_block();
      break;
    }
    prepare_pivots(b + 1, hw * 32 + lane, 32 * SW_HIST);
    prepare_scales(b + 1, hw * 32 + lane, 32 * SW_HIST);
    sw_sync<32 * SW_HIST>(SW_JOIN);
    prepare_triangles(b + 1, hw * 32 + lane, 32 * SW_HIST);
    double(*wn)[SW_LDW] = sm.w[(b + 1) & 1];
    const int cn = (b + 1) * 128 + crank * (128 / cs) + n_loc;  // first column of this warp
    double w0[MF][FW][2];
    if (kg == 0) {
#pragma unroll
      for (int m = 0; m < MF; ++m) {
        const bool ok = 8 * m + fr < rows_here;
        const double* src = a.src + (ok ? src_row(8 * m + fr) : 0) + cn;
#pragma unroll
        for (int t = 0; t < FW; ++t)
#pragma unroll
          for (int e = 0; e < 2; ++e) w0[m][t][e] = ok ? src[col_of(t, e)] : 0.0;
      }
    }
    double acc[MF][FW][NA][2];
#pragma unroll
    for (int i = 0; i < MF * FW * NA * 2; ++i) (&acc[0][0][0][0])[i] = 0.0;
    const int n_hist = (b - a.blk0) * per_blk, n_all = n_hist + per_blk;
    if constexpr (CLUSTER) {
      // straight from global memory: a warp has one fragment and every kgroups-th step of four rows; the next batch of
      // eight steps is fetched while one is multiplied
      const int n_steps = (b - a.blk0) * (32 / kgroups);  // a multiple of eight
      const long long urow = (long long)(a.blk0 * 128 + 4 * kg + fk) * d + cn + fr;
      const double* ep = a.Err + (long long)(m_base + min(fr, rows_here - 1)) * a.err_ld + a.blk0 * 128 - a.err_col0 + 4 * kg + fk;
      const double* rp = WITH_P ? a.Arr + (ep - a.Err) : nullptr;
      const long long us = (long long)4 * kgroups * d;
      double av[8], rv[WITH_P ? 8 : 1];
      float uv[8], pv[WITH_P ? 8 : 1];
      auto fetch = [&](int q0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          av[i] = __ldcg(ep + (long long)(q0 + i) * 4 * kgroups);
          uv[i] = __ldg(U + urow + (q0 + i) * us);
          if (WITH_P) {
            rv[i] = __ldcg(rp + (long long)(q0 + i) * 4 * kgroups);
            pv[i] = __ldg(Pm + urow + (q0 + i) * us);
          }
        }
      };
      if (n_steps > 0) fetch(0);
      for (int q0 = 0; q0 < n_steps; q0 += 8) {
        double an[8], bn[8], rn[WITH_P ? 8 : 1], pn[WITH_P ? 8 : 1];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          an[i] = av[i];
          bn[i] = (double)uv[i];
          if (WITH_P) {
            rn[i] = rv[i];
            pn[i] = (double)pv[i];
          }
        }
        if (q0 + 8 < n_steps) fetch(q0 + 8);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          dmma(acc[0][0][i & 3], an[i], bn[i]);
          if (WITH_P) dmma(acc[0][0][(i + 2) & 3], rn[i], pn[i]);
        }
      }
      // the block being walked, piece by piece: 4 / kgroups steps of this warp each
      const float* uo = U + (long long)(b * 128 + 4 * kg + fk) * d + cn + fr;
      const float* po = WITH_P ? Pm + (long long)(b * 128 + 4 * kg + fk) * d + cn + fr : nullptr;
      const int own = 4 / kgroups;
      float uc[4], pc[4], uf[4], pf[4];
      auto fetch_own = [&](int sb) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (i < own) {
            uf[i] = __ldg(uo + (long long)(16 * sb) * d + i * us);
            if (WITH_P) pf[i] = __ldg(po + (long long)(16 * sb) * d + i * us);
          }
      };
      fetch_own(0);
#pragma unroll 1
      for (int sb = 0; sb < 8; ++sb) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uc[i] = uf[i];
          pc[i] = pf[i];
        }
        if (sb < 7) fetch_own(sb + 1);
        sw_sync<32 + 32 * SW_HIST>(SW_PIECE + sb);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (i < own) {
            const int k = 16 * sb + 4 * (kg + kgroups * i) + fk;
            dmma(acc[0][0][i], sm.Es[fr][k], (double)uc[i]);
            if (WITH_P) dmma(acc[0][0][(i + 2) & 3], sm.As[WITH_P ? fr : 0][k], (double)pc[i]);
          }
      }
    } else {
      int met = 0;  // pieces of the block being walked that are known to be finished
      for (int c = 0; c < n_all; ++c) {
        const unsigned char* stg = ring + (size_t)slot * stage_bytes;
        const bool ok = mbar_wait(smem_u32(&sm.full_bar[slot]), phase, abort_flag, &g_sweep_error);
        __syncwarp();
        const bool second = WITH_P && (c & 1);
        const bool hist = c < n_hist;
        const int own0 = ((c - n_hist) / NOP) * ch;  // first contraction column of an own chunk inside the block
        const double* ap = hist ? reinterpret_cast<const double*>(stg + ub_bytes) + fr * lde
                                : (second ? &sm.As[WITH_P ? fr : 0][0] : &sm.Es[fr][0]) + own0;
        const int a_ld = hist ? lde : (int)SW_LDW;
        ap += fk;
        const float* bp = reinterpret_cast<const float*>(stg) + fk * ldb + n_loc + 2 * fr;
        for (int qq = 0; qq < ch / 4; qq += 4) {
          if (!hist) {
            const int piece = (own0 >> 4) + (qq >> 2);
            while (met <= piece) {
              sw_sync<32 + 32 * SW_HIST>(SW_PIECE + met);
              ++met;
            }
          }
          if (ok) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const int q = qq + i;
              const float2 bb = *reinterpret_cast<const float2*>(bp + 4 * q * SW_LDB);
              const double b0 = (double)bb.x, b1 = (double)bb.y;
#pragma unroll
              for (int m = 0; m < MF; ++m) {
                const double av = ap[8 * m * a_ld + 4 * q];
                dmma(acc[m][0][i % NA], av, b0);
                dmma(acc[m][FW - 1][i % NA], av, b1);
              }
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&sm.empty_bar[slot]));  // this warp is done with the stage
        if (++slot == stages) {
          slot = 0;
          phase ^= 1u;
        }
      }
    }
#pragma unroll
    for (int m = 0; m < MF; ++m)
#pragma unroll
      for (int t = 0; t < FW; ++t)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          double v = acc[m][t][0][e];
          if (NA == 2) v += acc[m][t][NA - 1][e];
          if (NA == 4) v = (v + acc[m][t][1 % NA][e]) + (acc[m][t][2 % NA][e] + acc[m][t][3 % NA][e]);
          acc[m][t][0][e] = v;
        }
    if (CLUSTER) {
      const int wc = 128 / cs;
      double2 v = make_double2(acc[0][0][0][0], acc[0][0][0][1]);
      double* mine = &sm.part[fr * wc + n_loc + 2 * fk];
      if (kg > 0) sw_st2(mine + (kg - 1) * 8 * wc, v.x, v.y);
      sw_sync<32 * SW_HIST>(SW_JOIN);
      if (kg == 0) {
        for (int k = 1; k < kgroups; ++k) {
          const double2 o = sw_ld2(mine + (k - 1) * 8 * wc);
          v.x += o.x;
          v.y += o.y;
        }
        v = make_double2(w0[0][0][0] - v.x, w0[0][0][1] - v.y);
        double* dst = &wn[fr][crank * wc + n_loc + 2 * fk];
        for (int r = 0; r < cs; ++r) *reinterpret_cast<double2*>(cg::this_cluster().map_shared_rank(dst, r)) = v;
      }
    } else {
#pragma unroll
      for (int m = 0; m < MF; ++m)
#pragma unroll
        for (int t = 0; t < FW; ++t)
#pragma unroll
          for (int e = 0; e < 2; ++e) wn[8 * m + fr][n_loc + col_of(t, e)] = w0[m][t][e] - acc[m][t][0][e];
    }
    next_block();
  }
}

int sweep_error_read_clear() {
  int v = 0;
  if (cudaMemcpyFromSymbol(&v, g_sweep_error, sizeof(int)) != cudaSuccess) return -1;
  if (v) {
    int z = 0;
    cudaMemcpyToSymbol(g_sweep_error, &z, sizeof(int));
  }
  return v;
}

template <bool WITH_P, int R, bool CLUSTER>
static tb_status sweep_launch(SweepP p, cudaStream_t st) {
  const SweepArgs& a = p.a;
  p.ctas_per_unit = (p.rows_per_unit + R - 1) / R;
  CUtensorMap map_u, map_e, map_p, map_a;
  constexpr int ch = SweepSmem<WITH_P, R>::CHUNK;
  const unsigned box_u = (unsigned)(a.d >= SW_LDB ? SW_LDB : a.d);
  const unsigned box_e = (unsigned)(a.err_ld >= ch + 4 ? ch + 4 : a.err_ld);
  const unsigned long long cols = (unsigned long long)a.d, mat_rows = cols * a.units;
  TB_TRY(make_map_2d(&map_u, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, sizeof(float), a.U, cols, mat_rows, box_u, ch,
                     CU_TENSOR_MAP_SWIZZLE_NONE));
  TB_TRY(make_map_2d(&map_e, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, sizeof(double), a.Err, (unsigned long long)a.err_ld,
                     (unsigned long long)a.M, box_e, R, CU_TENSOR_MAP_SWIZZLE_NONE));
  map_p = map_u;
  map_a = map_e;
  if (WITH_P) {
    TB_TRY(make_map_2d(&map_p, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, sizeof(float), a.P, cols, mat_rows, box_u, ch,
                       CU_TENSOR_MAP_SWIZZLE_NONE));
    TB_TRY(make_map_2d(&map_a, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, sizeof(double), a.Arr, (unsigned long long)a.err_ld,
                       (unsigned long long)a.M, box_e, R, CU_TENSOR_MAP_SWIZZLE_NONE));
  }
  auto kern = k_sweep_rows<WITH_P, R, CLUSTER>;
  constexpr size_t smem = sizeof(SweepSmem<WITH_P, R>);
  static_assert(smem <= 227 * 1024, "shared memory of an SM");
  static bool configured[64] = {false};
  TB_TRY(allow_smem(kern, smem, configured));
  const unsigned ctas = (unsigned)((long long)p.ctas_per_unit * a.units * (CLUSTER ? p.cs : 1));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(SW_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)(CLUSTER ? p.cs : 1);
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CLUSTER ? 2 : 1;
  TB_CUDA_CHECK(cudaLaunchKernelEx(&cfg, kern, p, map_u, map_e, map_p, map_a));
  TB_LAUNCH_CHECK();
  return TB_OK;
}

// How a launch over nblk blocks of 128 columns is split: rows a CTA, CTAs a cluster, CTAs in all.
struct SweepShape {
  int rows, cs;
  long long ctas;
};
static SweepShape sweep_shape(int rows_per_unit, int units, bool with_p, int nblk) {
  const long long sms = 148;
  const long long groups = (long long)((rows_per_unit + 7) / 8) * units;  // of 8 rows
  // few rows: a cluster per group of 8 rows shares the contraction
  if (nblk > 1 && groups * 2 <= sms) {
    const int cs = (groups * 8 <= sms) ? 8 : (groups * 4 <= sms) ? 4 : 2;
    return {8, cs, groups * cs};
  }
  // more rows per CTA as soon as 8 would take another round of CTAs: the chain's time does not depend on them
  // (with both factors the registers of 16 rows spill)
  if (with_p || groups <= sms) return {8, 1, groups};
  const long long g16 = (long long)((rows_per_unit + 15) / 16) * units;
  if (g16 <= sms) return {16, 1, g16};
  return {32, 1, (long long)((rows_per_unit + 31) / 32) * units};
}

tb_status sweep_columns(const SweepArgs& a, cudaStream_t st) {
  SweepP p;
  p.a = a;
  p.rows_per_unit = a.M / a.units;
  p.ctas_per_unit = 0;
  const SweepShape s = sweep_shape(p.rows_per_unit, a.units, a.P != nullptr, a.blk1 - a.blk0);
  p.cs = s.cs;
  if (s.cs > 1) return a.P ? sweep_launch<true, 8, true>(p, st) : sweep_launch<false, 8, true>(p, st);
  if (a.P) return sweep_launch<true, 8, false>(p, st);
  if (s.rows == 8) return sweep_launch<false, 8, false>(p, st);
  return s.rows == 16 ? sweep_launch<false, 16, false>(p, st) : sweep_launch<false, 32, false>(p, st);
}


// ---------------------------------------------------------------------------
// work[m][c] = src[m][c] - sum_k Err[m][k] U[k0 + k][c] (- Arr P) for the columns c >= c1 of few rows, K = c1 - k0 = 512.
// The eight warps of a CTA take an eighth of the contraction each, for 8 MF rows x 32 columns, straight from global
// memory (every entry of U is read once per row tile, in full sectors), and add up through shared memory in order.
// Bound: reading U (HBM / L2) for 8 rows, the FP64 pipe from about 64 on.  Up to 16 rows the sweep before leaves most SMs
// idle: the factors are copied into shared memory before the sweep has ended.
// 8 rows x 4096 columns: 3.5 us from the sweep's end to this kernel's, 9.5 when the loads came after the wait.
// ahead: the sweep that follows is launched before this kernel's own wait and prepares its first block from the factors
// meanwhile (RANK_AHEAD_CTAS).
// ---------------------------------------------------------------------------
template <bool WITH_P, int MF>
struct RankTile {
  static constexpr int RT = 8 * MF, CT = 32, LDF = 40;
  static constexpr bool EARLY = MF <= 2;  // factors staged in shared memory ahead of the sweep's end
  static constexpr size_t part = (size_t)8 * RT * CT * sizeof(double);
  static constexpr size_t slab = (size_t)SWEEP_OUTER * LDF * sizeof(float);
  static constexpr size_t smem = part + (EARLY ? slab * (WITH_P ? 2 : 1) : 0);
};

template <bool WITH_P, int MF>
__global__ void __launch_bounds__(256) k_rank_rows(SweepArgs a, double* work, int rows_per_unit, int k0, int c1, const double* err,
                                                   const double* arr, int ahead) {
  using T = RankTile<WITH_P, MF>;
  constexpr int NF = 4, RT = T::RT, CT = T::CT, STEPS = SWEEP_OUTER / 32;
  extern __shared__ __align__(16) double rr_part[];  // [8][RT][CT], then the factors
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, fr = lane >> 2, fk = lane & 3;
  const int unit = blockIdx.z, r0 = blockIdx.y * RT, c0 = c1 + blockIdx.x * CT;
  const int d = a.d;
  const long long uoff = (a.units > 1) ? (long long)unit * d * d : 0;
  const int m0 = unit * rows_per_unit + r0, rows = min(RT, rows_per_unit - r0);
  const int kw = warp * (SWEEP_OUTER / 8);  // STEPS steps of four contraction rows per warp
  double acc[MF][NF][2];
#pragma unroll
  for (int i = 0; i < MF * NF * 2; ++i) (&acc[0][0][0])[i] = 0.0;
  // f: the entry of this lane's fragment in the first step, rows ldf apart
  auto product = [&](const float* f, long long ldf, const double* E) {
#pragma unroll(T::EARLY ? 8 : 2)
    for (int q = 0; q < STEPS; ++q) {
      float b[NF];
      double av[MF];
#pragma unroll
      for (int n = 0; n < NF; ++n) b[n] = f[4 * q * ldf + 8 * n];
#pragma unroll
      for (int m = 0; m < MF; ++m) av[m] = E[(long long)(m0 + min(8 * m + fr, rows - 1)) * a.err_ld + kw + fk + 4 * q];
#pragma unroll
      for (int n = 0; n < NF; ++n) {
        const double bd = (double)b[n];
#pragma unroll
        for (int m = 0; m < MF; ++m) dmma(acc[m][n], av[m], bd);
      }
    }
  };
  if (T::EARLY) {
    // asynchronous copies: loads into registers are scheduled behind the wait by the compiler.  Columns come in whole 32s.
    float* slab = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(rr_part) + T::part);
    auto stage = [&](const float* F, float* dst) {
#pragma unroll 4
      for (int i = threadIdx.x; i < SWEEP_OUTER * (CT / 4); i += 256) {
        const int k = i / (CT / 4), c = 4 * (i % (CT / 4));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst + k * T::LDF + c)),
                     "l"(F + uoff + (long long)(k0 + k) * d + c0 + c)
                     : "memory");
      }
    };
    stage(a.U, slab);
    if (WITH_P) stage(a.P, slab + SWEEP_OUTER * T::LDF);
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (ahead) pdl_trigger();
    pdl_wait();
    product(slab + (kw + fk) * T::LDF + fr, T::LDF, err);
    if (WITH_P) product(slab + (SWEEP_OUTER + kw + fk) * T::LDF + fr, T::LDF, arr);
  } else {
    pdl_wait();
    product(a.U + uoff + (long long)(k0 + kw + fk) * d + c0 + fr, d, err);
    if (WITH_P) product(a.P + uoff + (long long)(k0 + kw + fk) * d + c0 + fr, d, arr);
  }
#pragma unroll
  for (int m = 0; m < MF; ++m)
#pragma unroll
    for (int n = 0; n < NF; ++n)
      *reinterpret_cast<double2*>(rr_part + (warp * RT + 8 * m + fr) * CT + 8 * n + 2 * fk) = make_double2(acc[m][n][0], acc[m][n][1]);
  if (!ahead) pdl_trigger();
  __syncthreads();
  for (int i = threadIdx.x; i < RT * CT; i += 256) {
    const int r = i / CT, c = i % CT;
    if (r >= rows || c0 + c >= d) continue;
    double v = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) v += rr_part[w * RT * CT + i];
    const long long src = (a.src_mapped ? a.rm.row(m0 + r) : (long long)(m0 + r)) * d + c0 + c;
    work[(long long)(m0 + r) * d + c0 + c] = a.src[src] - v;
  }
}

// rows along x, the one grid dimension that holds any number of them
__global__ void k_sweep_gather(SweepArgs a, double* __restrict__ work, int c1) {
  const int m = blockIdx.x;
  const double2* src = reinterpret_cast<const double2*>(a.src + a.rm.row(m) * a.d);
  double2* dst = reinterpret_cast<double2*>(work + (long long)m * a.d);
  for (int c = c1 / 2 + blockIdx.y * blockDim.x + threadIdx.x; c < a.d / 2; c += gridDim.y * blockDim.x) dst[c] = src[c];
}

// An update on digits costs three launches whatever its size, k_rank_rows the FP64 pipe's time for rows x width: about
// equal at 300 rows of 4096 columns.  208 rows of 1664 with P: 11.0 ms of sweep with digits, 7.2 ms without.  With one
// U per head the digits of all of them would have to be kept, for rows of one head each: not taken.
bool sweep_wants_i8(int d, int units, int rows_per_unit) {
  return units == 1 && d > SWEEP_OUTER && d <= I8_MAX_K_BLOCKS * I8_KB && (long long)rows_per_unit * d >= SWEEP_I8_WORK;
}

void sweep_scratch(Bump& b, int M, int d, bool with_p, bool use_i8, SweepScratch* s) {
  *s = SweepScratch{};
  s->use_i8 = use_i8;
  if (d <= SWEEP_OUTER) return;
  s->err = b.take<double>((size_t)M * SWEEP_OUTER);
  if (with_p) s->arr = b.take<double>((size_t)M * SWEEP_OUTER);
  if (!use_i8) return;
  auto mat = [&](long long row_blocks, int k_blocks) {
    I8Mat m;
    m.row_blocks = row_blocks;
    m.k_blocks = k_blocks;
    m.data = b.take<unsigned char>(i8_bytes(row_blocks, k_blocks));
    return m;
  };
  const long long row_blocks = (M + I8_RB - 1) / I8_RB;
  s->Udig = mat(d / I8_RB, d / I8_KB);
  s->Edig = mat(row_blocks, SWEEP_OUTER / I8_KB);
  s->u_max = b.take<unsigned long long>((size_t)d);
  s->e_max = b.take<unsigned long long>((size_t)M);
  s->u_exp = b.take<int>((size_t)d);
  if (with_p) {
    s->Pdig = mat(d / I8_RB, d / I8_KB);
    s->Adig = mat(row_blocks, SWEEP_OUTER / I8_KB);
    s->p_max = b.take<unsigned long long>((size_t)d);
    s->a_max = b.take<unsigned long long>((size_t)M);
  }
}

// Rows of U scale as 1 / U_kk scales the errors: the exponents of the diagonal take that out of both operands.
tb_status sweep_prepare(const float* U, const float* P, int d, const SweepScratch& s, cudaStream_t st) {
  if (!s.use_i8) return TB_OK;
  TB_TRY(i8_diag_exp(U, s.u_exp, d, st));
  const I8Src us{U, d, 0, d, d, 1, true, false, 1, s.u_exp, -1};
  TB_TRY(i8_row_max(us, s.u_max, d, st));
  TB_TRY(i8_slice(us, s.u_max, d, 0, s.Udig, 0, 0, 0, st));
  if (P) {
    const I8Src ps{P, d, 0, d, d, 1, true, false, 1, nullptr, 0};
    TB_TRY(i8_row_max(ps, s.p_max, d, st));
    TB_TRY(i8_slice(ps, s.p_max, d, 0, s.Pdig, 0, 0, 0, st));
  }
  return TB_OK;
}

// CTAs, of a whole SM each, of a sweep that the update before it launches ahead of its own wait: at most half of the SMs, so
// that another stream's kernels find room while they wait.  Rows a step in 2048 or 4096 columns, without -> with: a sweep of 8
// CTAs 41.00 -> 40.56 ms, 16 CTAs 2.811 -> 2.788, 32 CTAs 2.931 -> 2.901, 64 CTAs 3.404 -> 3.366, 128 CTAs 3.116 -> 3.108 (the
// runs of one side differ by as much).
constexpr int RANK_AHEAD_CTAS = 74;

template <bool WITH_P, int MF>
static tb_status rank_launch(const SweepArgs& a, double* work, int rows_per_unit, int k0, int c1, const double* err,
                             const double* arr, int next_blocks, cudaStream_t st) {
  constexpr int CT = RankTile<WITH_P, MF>::CT;
  constexpr size_t smem = RankTile<WITH_P, MF>::smem;
  static bool configured[64] = {false};
  auto kern = k_rank_rows<WITH_P, MF>;
  TB_TRY(allow_smem(kern, smem, configured));
  const dim3 grid((a.d - c1 + CT - 1) / CT, (rows_per_unit + 8 * MF - 1) / (8 * MF), a.units);
  const int ahead =
      RankTile<WITH_P, MF>::EARLY && sweep_shape(rows_per_unit, a.units, WITH_P, next_blocks).ctas <= RANK_AHEAD_CTAS;
  TB_CUDA_CHECK(launch_pdl(kern, grid, dim3(256), smem, st, a, work, rows_per_unit, k0, c1, err, arr, ahead));
  TB_LAUNCH_CHECK();
  return TB_OK;
}

tb_status sweep_step(SweepArgs a, const SweepScratch& s, cudaStream_t st) {
  const int d = a.d, rows_per_unit = a.M / a.units, nblk = d / 128;
  constexpr int OB = SWEEP_OUTER / 128;
  if (nblk <= OB) {  // one launch; the histories take the working copies' places
    a.blk0 = 0;
    a.blk1 = nblk;
    a.err_ld = d;
    a.err_col0 = 0;
    return sweep_columns(a, st);
  }
  double* E = s.err;
  double* A = s.arr;
  a.Err = E;
  a.Arr = A;
  a.err_ld = SWEEP_OUTER;
  if (s.use_i8) {
    k_sweep_gather<<<dim3(a.M, (d / 2 + 255) / 256), 256, 0, st>>>(a, s.work, SWEEP_OUTER);
    TB_LAUNCH_CHECK();
  }
  for (int b0 = 0; b0 < nblk; b0 += OB) {
    const int b1 = (b0 + OB < nblk) ? b0 + OB : nblk, k0 = b0 * 128, c1 = b1 * 128;
    a.blk0 = b0;
    a.blk1 = b1;
    a.err_col0 = k0;
    TB_TRY(sweep_columns(a, st));
    if (c1 >= d) break;
    if (s.use_i8) {
      const I8Src es{E, SWEEP_OUTER, 0, a.M, c1 - k0, 1, false, true, 0, s.u_exp + k0, 1};
      TB_TRY(i8_row_max(es, s.e_max, a.M, st));
      TB_TRY(i8_slice(es, s.e_max, a.M, 0, s.Edig, 0, 0, 0, st));
      I8Gemm g = i8_gemm_params();
      g.A = s.Edig;
      g.B = s.Udig;
      g.b_rb = c1 / I8_RB;
      g.b_kb = k0 / I8_KB;
      g.k_blocks = (c1 - k0) / I8_KB;
      g.a_max = s.e_max;
      g.b_max = s.u_max + c1;
      g.C = s.work + c1;
      g.ldc = d;
      g.M = a.M;
      g.N = d - c1;
      g.alpha = -1.0;
      g.beta = 1.0;
      TB_TRY(i8_gemm(g, st));
      if (a.P) {
        const I8Src as{A, SWEEP_OUTER, 0, a.M, c1 - k0, 1, false, true, 0, nullptr, 0};
        TB_TRY(i8_row_max(as, s.a_max, a.M, st));
        TB_TRY(i8_slice(as, s.a_max, a.M, 0, s.Adig, 0, 0, 0, st));
        g.A = s.Adig;
        g.B = s.Pdig;
        g.a_max = s.a_max;
        g.b_max = s.p_max + c1;
        TB_TRY(i8_gemm(g, st));
      }
    } else {
      // rows per tile: 8, 16 or 32, as few tiles as cover the unit's rows
      const int mf = rows_per_unit <= 8 ? 1 : rows_per_unit <= 16 ? 2 : 4, nb = nblk - b1 < OB ? nblk - b1 : OB;
      if (a.P) {
        if (mf == 1) TB_TRY((rank_launch<true, 1>(a, s.work, rows_per_unit, k0, c1, E, A, nb, st)));
        if (mf == 2) TB_TRY((rank_launch<true, 2>(a, s.work, rows_per_unit, k0, c1, E, A, nb, st)));
        if (mf == 4) TB_TRY((rank_launch<true, 4>(a, s.work, rows_per_unit, k0, c1, E, A, nb, st)));
      } else {
        if (mf == 1) TB_TRY((rank_launch<false, 1>(a, s.work, rows_per_unit, k0, c1, E, A, nb, st)));
        if (mf == 2) TB_TRY((rank_launch<false, 2>(a, s.work, rows_per_unit, k0, c1, E, A, nb, st)));
        if (mf == 4) TB_TRY((rank_launch<false, 4>(a, s.work, rows_per_unit, k0, c1, E, A, nb, st)));
      }
    }
    a.src = s.work;
    a.src_mapped = false;
  }
  return TB_OK;
}

// ---------------------------------------------------------------------------
// One column group of the dynamic-grid sweep: 8 rows of a unit per CTA, the group's factor rows in shared memory.  The
// chain is the sweep's (a thread per row, 16 columns at a time); after a piece all warps apply its errors to the group's
// later columns by FP64 tensor steps, and while the next piece is walked they write the piece's outputs (not the warp
// that shares the chain's scheduler).  Bound by the chain's latency.  1152 rows, group of 64: 8.9 us; a warp per row with
// two divisions and a broadcast per column, as it was, 32.6.
// ---------------------------------------------------------------------------
template <bool WITH_P>
struct PanelSmem {
  alignas(16) double w[8][SW_LDW], Es[8][SW_LDW], As[WITH_P ? 8 : 1][SW_LDW];
  alignas(16) double cU[8][16][16], cP[WITH_P ? 8 : 1][16][16];
  alignas(16) double rd[128];
  double gs[8][3];
  float U[128][SW_LDB], P[WITH_P ? 128 : 1][SW_LDB];
};

template <bool WITH_P>
__global__ void __launch_bounds__(256) k_group_panel(GroupPanelP p, int ctas_per_unit) {
  extern __shared__ __align__(16) unsigned char gp_raw[];
  PanelSmem<WITH_P>& sm = *reinterpret_cast<PanelSmem<WITH_P>*>(gp_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, fr = lane >> 2, fk = lane & 3;
  const int seg = p.seg, d = p.d, c0 = p.grp * seg;
  const int unit = blockIdx.x / ctas_per_unit, r_first = (blockIdx.x % ctas_per_unit) * 8;
  const int rows = min(8, p.rows_per_unit - r_first), m0 = unit * p.rows_per_unit + r_first;
  const long long uoff = ((p.units > 1) ? (long long)unit * d * d : 0) + (long long)c0 * (d + 1);
  for (int i = tid; i < seg * seg / 4; i += 256) {
    const int j = i / (seg / 4), c = 4 * (i % (seg / 4));
    if (c + 3 >= j) {  // the strictly lower triangle is not read
      *reinterpret_cast<float4*>(&sm.U[j][c]) = *reinterpret_cast<const float4*>(p.U + uoff + (long long)j * d + c);
      if (WITH_P) *reinterpret_cast<float4*>(&sm.P[j][c]) = *reinterpret_cast<const float4*>(p.P + uoff + (long long)j * d + c);
    }
  }
  for (int i = tid; i < 8 * seg; i += 256) {
    const int r = i / seg, c = i % seg;
    sm.w[r][c] = (r < rows) ? p.Wk[(long long)(m0 + r) * d + c0 + c] : 0.0;
  }
  if (tid < 8) {
    double s = 1.0, z = 0.0;
    if (tid < rows) {
      const long long so = p.rm.row(m0 + tid) * p.ng + p.grp;
      s = p.sD[so];
      z = (double)p.z[so];
    }
    sm.gs[tid][0] = s;
    sm.gs[tid][1] = 1.0 / s;
    sm.gs[tid][2] = z;
  }
  __syncthreads();
  if (tid < seg) sm.rd[tid] = 1.0 / (double)sm.U[tid][tid];
  __syncthreads();
  for (int i = tid; i < seg * 16; i += 256) {
    const int j = i >> 4, c = i & 15, jl = j & 15, cc = (j & ~15) + c;
    sm.cU[j >> 4][jl][c] = (c > jl) ? (double)sm.U[j][cc] * sm.rd[j] : 0.0;
    if (WITH_P) sm.cP[WITH_P ? j >> 4 : 0][jl][c] = (c > jl) ? (double)sm.P[WITH_P ? j : 0][cc] : 0.0;
  }
  unsigned int n_near = 0, n_clamp = 0;
  auto outputs = [&](int sb, int t, int nt) {  // codes, errors and counters of a piece
    for (int i = t; i < 128; i += nt) {
      const int r = i >> 4, cl = 16 * sb + (i & 15);
      if (r < rows) {
        p.codes[p.rm.row(m0 + r) * d + c0 + cl] = (unsigned char)sw_output(sm.w[r][cl], sm.gs[r][2], p.maxq, n_near, n_clamp);
        p.Err[(long long)(m0 + r) * seg + cl] = sm.Es[r][cl];
        if (WITH_P) p.Arr[(long long)(m0 + r) * seg + cl] = sm.As[WITH_P ? r : 0][cl];
      }
    }
  };
  for (int sb = 0; sb < seg / 16; ++sb) {
    __syncthreads();
    if (warp == 0) {
      const int r = lane & 7;
      const double s = sm.gs[r][0], rs = sm.gs[r][1], z = sm.gs[r][2];
      double* wr = &sm.w[r][16 * sb];
      double* er = &sm.Es[r][16 * sb];
      double v[16];
      auto load = [&]() {
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
          const double2 t = sw_ld2(wr + j);
          v[j] = t.x * rs;
          v[j + 1] = t.y * rs;
        }
      };
      load();
      const int off = sw_walk<WITH_P, false>(v, er, s, z, p.maxq, &sm.rd[16 * sb], sm.cU[sb], sm.cP[WITH_P ? sb : 0]);
      if (__any_sync(0xffffffffu, off != 0)) {  // again, with the range test in the chain
        load();
        sw_walk<WITH_P, true>(v, er, s, z, p.maxq, &sm.rd[16 * sb], sm.cU[sb], sm.cP[WITH_P ? sb : 0]);
      }
      __syncwarp();  // (lanes of one row read its values before one of them overwrites them)
#pragma unroll
      for (int j = 0; j < 16; j += 2) {
        sw_st2(wr + j, v[j], v[j + 1]);
        if (WITH_P) sw_st2(&sm.As[WITH_P ? r : 0][16 * sb + j], v[j] * s, v[j + 1] * s);
      }
    } else if (sb > 0 && warp != 4) {
      outputs(sb - 1, (warp - (warp > 4 ? 2 : 1)) * 32 + lane, 192);
    }
    __syncthreads();
    for (int n = 2 * (sb + 1) + warp; n < seg / 8; n += 8) {
      double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
      for (int q = 0; q < 4; ++q)
        dmma(acc[q & 1], sm.Es[fr][16 * sb + 4 * q + fk], (double)sm.U[16 * sb + 4 * q + fk][8 * n + fr]);
      if (WITH_P)
#pragma unroll
        for (int q = 0; q < 4; ++q)
          dmma(acc[q & 1], sm.As[WITH_P ? fr : 0][16 * sb + 4 * q + fk],
                 (double)sm.P[WITH_P ? 16 * sb + 4 * q + fk : 0][8 * n + fr]);
      double2* wp = reinterpret_cast<double2*>(&sm.w[fr][8 * n + 2 * fk]);
      const double2 o = *wp;
      *wp = make_double2(o.x - (acc[0][0] + acc[1][0]), o.y - (acc[0][1] + acc[1][1]));
    }
  }
  outputs(seg / 16 - 1, tid, 256);
  if (p.stats) {
    n_near = __reduce_add_sync(0xffffffffu, n_near);
    n_clamp = __reduce_add_sync(0xffffffffu, n_clamp);
    if (lane == 0) {
      if (n_near) atomicAdd(&p.stats->near_tie_codes, (unsigned long long)n_near);
      if (n_clamp) atomicAdd(&p.stats->clamped_codes, (unsigned long long)n_clamp);
      if (m0 == 0 && warp == 0) atomicAdd(&p.stats->column_steps, (unsigned long long)seg);
    }
  }
}

// Wk[:, c1 ..] -= Err U[c0 .. c1, c1 ..] (- Arr P): 64 rows x 64 columns per CTA, the contraction (one group, or one group twice)
// 32 rows at a time, the next ones fetched meanwhile.  8 warps of 32 x 16.  Bound by latency: 141 MFLOP a launch.
// 1152 x 960 columns, group of 64: 11.5 us (tiles of 128 x 128 19.1).
__global__ void __launch_bounds__(256, 2) k_group_update(GroupPanelP p) {
  __shared__ double As[64][36];
  __shared__ float Bs[32][72];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, fr = lane >> 2, fk = lane & 3;
  const int d = p.d, seg = p.seg, k_first = p.grp * seg, c0 = k_first + seg + blockIdx.x * 64;
  const int tiles = (p.rows_per_unit + 63) / 64, unit = blockIdx.y / tiles, r0 = (blockIdx.y % tiles) * 64;
  const int rows = min(64, p.rows_per_unit - r0), m0 = unit * p.rows_per_unit + r0;
  const long long uoff = (p.units > 1) ? (long long)unit * d * d : 0;
  const int wr = (warp >> 2) * 32, wc = (warp & 3) * 16;
  const int n_k = p.P ? 2 * seg : seg;
  double acc[4][2][2];
#pragma unroll
  for (int i = 0; i < 16; ++i) (&acc[0][0][0])[i] = 0.0;
  double av[8];
  float bv[8];
  auto fetch = [&](int k0) {
    const bool second = k0 >= seg;
    const int kk = second ? k0 - seg : k0;
    const double* E = second ? p.Arr : p.Err;
    const float* F = (second ? p.P : p.U) + uoff;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int rr = warp + 8 * i, n = tid & 63, k = (tid >> 6) + 4 * i;
      av[i] = (rr < rows) ? E[(long long)(m0 + rr) * seg + kk + lane] : 0.0;
      bv[i] = (c0 + n < d) ? F[(long long)(k_first + kk + k) * d + c0 + n] : 0.0f;
    }
  };
  fetch(0);
  double2 old[4][2];  // the values to be updated, on their way while the product is formed
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int rr = wr + 8 * i + fr, n = c0 + wc + 8 * j + 2 * fk;
      old[i][j] = (rr < rows && n < d) ? *reinterpret_cast<const double2*>(p.Wk + (long long)(m0 + rr) * d + n) : make_double2(0.0, 0.0);
    }
  for (int k0 = 0; k0 < n_k; k0 += 32) {
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      As[warp + 8 * i][lane] = av[i];
      Bs[(tid >> 6) + 4 * i][tid & 63] = bv[i];
    }
    __syncthreads();
    if (k0 + 32 < n_k) fetch(k0 + 32);
#pragma unroll
    for (int k4 = 0; k4 < 8; ++k4) {
      double a[4], b[2];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[wr + 8 * i + fr][4 * k4 + fk];
#pragma unroll
      for (int j = 0; j < 2; ++j) b[j] = (double)Bs[4 * k4 + fk][wc + 8 * j + fr];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) dmma(acc[i][j], a[i], b[j]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int rr = wr + 8 * i + fr, n = c0 + wc + 8 * j + 2 * fk;
      if (rr < rows && n < d)
        *reinterpret_cast<double2*>(p.Wk + (long long)(m0 + rr) * d + n) =
            make_double2(old[i][j].x - acc[i][j][0], old[i][j].y - acc[i][j][1]);
    }
}

tb_status group_panel(const GroupPanelP& p, cudaStream_t st) {
  static bool conf[64] = {false}, conf_p[64] = {false};
  const int ctas = (p.rows_per_unit + 7) / 8, tiles = (p.rows_per_unit + 63) / 64;
  if ((long long)tiles * p.units > 65535) return TB_ERR_UNSUPPORTED;
  if (p.P) {
    TB_TRY(allow_smem(k_group_panel<true>, sizeof(PanelSmem<true>), conf_p));
    k_group_panel<true><<<(unsigned)(ctas * p.units), 256, sizeof(PanelSmem<true>), st>>>(p, ctas);
  } else {
    TB_TRY(allow_smem(k_group_panel<false>, sizeof(PanelSmem<false>), conf));
    k_group_panel<false><<<(unsigned)(ctas * p.units), 256, sizeof(PanelSmem<false>), st>>>(p, ctas);
  }
  TB_LAUNCH_CHECK();
  const int right = p.d - (p.grp + 1) * p.seg;
  if (right > 0) {
    k_group_update<<<dim3((right + 63) / 64, tiles * p.units), 256, 0, st>>>(p);
    TB_LAUNCH_CHECK();
  }
  return TB_OK;
}

}  // namespace tb
