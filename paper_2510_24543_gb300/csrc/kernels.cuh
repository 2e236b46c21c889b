// Kernels of the eGPE hot path.  Two kernel shapes carry every 3D transform:
//
// * xpass_kernel<Op>: lines along x (contiguous).  A block owns MX rows; each
//   row is transformed by L/8 threads.  Op supplies the prologue (values at the
//   transform's entry positions, read straight from global memory) and the
//   epilogue (consumes the exit positions: stores, pointwise physics, sums).
// * colpass_kernel<Op>: lines along y or z (strided).  A tile is M adjacent x
//   columns times one line; lanes run along x so every global access is a
//   full 128-byte row of the tile.
//
// Both are persistent (grid-stride over rows / tiles) so that the per-block
// FP64 partial sums stay few; the last block finalises the sums in a fixed
// order and, where a pipeline needs it, runs the controller step.
#pragma once
#include <type_traits>
#include "common.cuh"
#include "ctrl.cuh"
#include "fft.cuh"
#include "lhy.cuh"
#include "reduce.cuh"
#include "tma.cuh"

namespace egpe {

template <class R> struct KArgs {
  using C = C2<R>;
  int nx, ny, nz, N;
  R hx, hy, hz, Lx, Ly, Lz;
  const R* kq;               // k_a^2 / (2 N) per index: [nx] x, [ny] y, [nz] z
  const R* vt;               // lambda_a^2 x_a^2 / 2 per index, same layout
  R vx;                      // lambda_x^2 / 2
  R g11, g12, g21, g22;      // contact couplings
  R d11, d12, d21, d22;      // k-space dipolar coefficients
  R invN;
  int Q, Qm;  // Gauss-Legendre nodes; the first Qm have det eta > 0
  R nskip;    // LHY terms skipped where n1 + n2 <= nskip (their size is below 1e-30)
  const LhyNode<R>* nodes;   // all Q nodes (parameter derivatives)
  const LhyNode<R>* xnodes;  // the Qx nodes evaluated exactly next to the table (det eta > 0 first: Qxm)
  int Qx, Qxm;
  LhyTab<R> tab;             // interpolated sums over the other nodes (tab.ni = 0: none)
  const C* twx;
  const C* twy;
  const C* twz;
  C* psi[2];                 // psi buffers (2 fields each)
  C* hp[2];                  // H psi buffers
  C* ax[2];                  // aux: field 0 = (Phi1, Phi2), field 1 = (B1, B2), B_i = V + sum_j g_ij n_j + mu_LHY,i:
                             // P_V, the line search and the ITE step need mu_LHY only in this sum
  C* rb[2];                  // residual buffers (current / previous by parity of n)
  C* pb[2];                  // direction buffers (current / previous)
  C* z;                      // preconditioned residual
  C* W;                      // transform workspace, 3 fields
  C* tb[2];                  // T psi of the psi buffers (attempts that carry it along)
  C* tp[2];                  // T p of the direction buffers
  C* wz;                     // P_V^{-1} r, where T z = wz - alpha z
  const C* gin;              // generic in/out of the plain passes; standalone evaluations: the caller's psi
  C* gout;                   // (copied to the psi buffer on the way) and gradient
  double* partials;
  unsigned* counter;
  DevState* st;
  TraceDev* trace;
  const R* kin_tab;          // ITE: e^{-dtau k_a^2/4} per index ([nx] x, [ny] y, [nz] z), then dtau
  int MX, M, nf, f0;         // launch shape: rows per block, columns per tile, fields
  int gate;                  // Gate
  int flag;                  // op-specific (trial / r given / p given)
  int ctrl;                  // run the controller step in the last block
  int diag;                  // P_V part of the preconditioner
  int blend;                 // weighted P_V / P_Delta combination (mode 4)
  int att;                   // AttemptKind
  long long wait_polls;      // poll budget of a TMA tile wait before the pass reports a timeout
};

template <class R> __device__ __forceinline__ bool gate_open(const KArgs<R>& a) {
  if (a.gate == GATE_ALWAYS) return true;
  const int ph = __ldcg(&a.st->phase);
  switch (a.gate) {
    case GATE_NEW_ITER: return ph == PH_NEW_ITER;
    case GATE_CARRIED_PC: return ph == PH_NEW_ITER || ph == PH_DIRECT;
    case GATE_VERIFY: return ph == PH_VERIFY;
  }
  return ph == PH_NEW_ITER || ph == PH_TRIAL;
}

// Batched launches: one launch runs the same pass for up to KB_MAX instances
// of one grid shape, blockIdx.y selecting the instance.  The descriptors (and
// the column passes' tensor maps) travel in the kernel's parameter block.
constexpr int KB_MAX = 16;
template <class R> struct KBatch {
  CUtensorMap tm[KB_MAX];
  KArgs<R> k[KB_MAX];
};
static_assert(sizeof(KBatch<double>) <= 32764, "batched kernel parameters exceed the 32 KB limit");

// Points whose global loads are issued together before any store of the chunk
// (the buffers may alias as far as the compiler knows, so loads and stores are
// grouped explicitly to keep several loads in flight per thread).
template <class R> struct ChunkW;
template <> struct ChunkW<float> { static constexpr int v = 4; };
template <> struct ChunkW<double> { static constexpr int v = 2; };

template <class R> __device__ __forceinline__ LhyCoef<R> lhy_coef(const KArgs<R>& a) {
  LhyCoef<R> c;
  c.g11 = a.g11;
  c.g22 = a.g22;
  c.g12 = a.g12;
  c.d11 = a.d11;
  c.d22 = a.d22;
  c.d12 = a.d12;
  c.nskip = a.nskip;
  return c;
}

// One of a pair, by a select: a run-time index would put a pair held in registers in
// local memory.  The FP32 buffers of the kernel arguments are indexed: the address comes
// from the constant bank at its use, where the select kept both halves in registers
// (128^3 x-inverse line pass 56.4 -> 55.1 us, energy pass 50.8 -> 50.2).  The FP64
// kernels spill with the index (x-inverse preconditioner pass 191 -> 212 us).
template <class T> __device__ __forceinline__ T pick(const T (&p)[2], int i) { return i ? p[1] : p[0]; }
__device__ __forceinline__ C2<float>* pick(C2<float>* const (&p)[2], int i) { return p[i]; }

// Terms of the trap and of |k|^2/2 (over N) that depend on one index come from
// tables: forming them per point took an integer conversion and three products in
// each of a dozen places, on the FP64 pipe of the FP64 kernels.  FP32 kernels form
// the trap's x term (the load's latency costs them more: line pass 57 against 54 us).
template <class R> __device__ __forceinline__ R trap_x(const KArgs<R>& a, int x) {
  if constexpr (sizeof(R) == 8) {
    return a.vt[x];
  } else {
    const R X = fma_((R)x, a.hx, -a.Lx);
    return a.vx * X * X;
  }
}
template <class R> __device__ __forceinline__ R trap_yz(const KArgs<R>& a, int row) {
  const int y = row % a.ny, z = row / a.ny;
  return a.vt[a.nx + y] + a.vt[a.nx + a.ny + z];
}
template <class R> __device__ __forceinline__ R kq_xy(const KArgs<R>& a, int x, int y) { return __ldg(a.kq + x) + __ldg(a.kq + a.nx + y); }
// k_z^2/(2N) at a thread's positions of a z line (the same in every tile).
template <class R, int L> struct KzLine {
  R kz[8];
  __device__ __forceinline__ void set(const KArgs<R>& a, int t) {
#pragma unroll
    for (int e = 0; e < 8; ++e) kz[e] = a.kq[a.nx + a.ny + Plan<L>::exit_pos(false, t, e)];
  }
};
// Dipolar kernel (3 k_z^2/|k|^2 - 1)/N from the table's k_z^2/(2N) and |k|^2/(2N); 0 at k = 0.
template <class R> __device__ __forceinline__ R dip_mult(const KArgs<R>& a, R kz, R k2) {
  return k2 > R(0) ? fma_(R(3) * a.invN * kz, rcp_(k2), -a.invN) : R(0);
}

// Row-pass ops whose LHY terms come from the interpolation table plus the
// exactly evaluated nodes (they stage the exact nodes only).
template <class Op, class = void> struct LhyTabOp {
  static constexpr bool v = false;
};
template <class Op> struct LhyTabOp<Op, std::void_t<decltype(Op::LHY_TAB)>> {
  static constexpr bool v = Op::LHY_TAB;
};

// Row-pass ops that transform the caller's own fields over the whole FP64 range.
template <class Op, class = void> struct WideOp {
  static constexpr bool v = false;
};
template <class Op> struct WideOp<Op, std::void_t<decltype(Op::WIDE)>> {
  static constexpr bool v = Op::WIDE;
};

// Every pass runs whole warps: the block reductions and the warp exchanges use
// full-mask shuffles.  A row (x) pass gives each row L/8 threads and a column
// pass each column L/8 threads, so a block holds a multiple of
// whole_warp_rows(L) rows or columns.
__host__ __device__ constexpr int gcd_i(int a, int b) { return b == 0 ? a : gcd_i(b, a % b); }
__host__ __device__ constexpr int whole_warp_rows(int L) { return 32 / gcd_i(L / 8, 32); }

// Threads per block of a row pass: 256 unless the op asks for fewer, rounded
// down to whole warps of whole rows (at least one such group).
template <class Op, class = void> struct MaxThreadsWant {
  static constexpr int v = 256;
};
template <class Op> struct MaxThreadsWant<Op, std::void_t<decltype(Op::MAXT)>> {
  static constexpr int v = Op::MAXT;
};
// Field groups of a row pass: FP64 fields give every field of a row its own L/8
// threads, FP32 fields one group that holds all fields of the row.  The FP64
// passes wait on FP64 and integer chains, which more warps overlap; the FP32
// passes wait on memory, where one thread's loads for all fields of eight points
// are what is in flight (with groups the FP32 x-inverse passes took 62-66 us for
// 48-54 at 128^3).
template <class Op> struct RowGroups {
  static constexpr int v = sizeof(typename Op::R) == 8 ? Op::NF : 1;
};
// FP64 epilogues of one field (power-of-two lengths, whose transforms need no block
// barrier) may be launched with two groups more that only take points (row_groups).
template <class Op> struct ExtraGroups {
  static constexpr int v = sizeof(typename Op::R) == 8 && Op::NF == 1 && Op::POINTS && IsPow2<Op::L>::v ? 3 : 1;
};
template <class Op> struct MaxThreads {
  static constexpr int G = whole_warp_rows(Op::L) * (Op::L / 8) * RowGroups<Op>::v;
  static constexpr int W = MaxThreadsWant<Op>::v;
  static constexpr int v0 = W >= G ? W - W % G : G;
  static constexpr int v = v0 > G * ExtraGroups<Op>::v ? v0 : G * ExtraGroups<Op>::v;
};

// Minimum resident blocks per SM a row-pass op asks the compiler to allow for
// (caps its registers); 1 unless the op says otherwise.
template <class Op, class = void> struct MinBlocks {
  static constexpr int v = 1;
};
template <class Op> struct MinBlocks<Op, std::void_t<decltype(Op::MINB)>> {
  static constexpr int v = Op::MINB;
};

// ----------------------------------------------------------------------------
// Row (x) pass kernel
// ----------------------------------------------------------------------------
// One point of a row pass's epilogue: its index in a field, its x, the trap terms
// of its row, and its transform outputs: out(f), from registers or from where the
// rows are parked in shared memory.
template <class R, int NF, bool STAGED> struct RowPt {
  C2<R> reg[STAGED ? 1 : NF];
  const C2<R>* sm;
  size_t idx;
  int fs, x;
  R vyz;
  __device__ __forceinline__ C2<R> out(int f) const {
    if constexpr (STAGED) return sm[f * fs];
    else return reg[f];
  }
};
// Row-pass ops that park their outputs with FP32 fields too, which frees the
// transform's registers for the epilogue.
template <class Op, class = void> struct StageOut {
  static constexpr bool v = RowGroups<Op>::v > 1 || sizeof(typename Op::R) == 8;
};
template <class Op> struct StageOut<Op, std::void_t<decltype(Op::STAGE_OUT)>> {
  static constexpr bool v = true;
};

// A thread's NV lines (fields f, f + 1, ...) to or from consecutive fields.
template <class Op, int NV>
__device__ __forceinline__ void store_rows(const KArgs<typename Op::R>& a, C2<typename Op::R>* dst, int f, int row, bool valid,
                                           int t, const C2<typename Op::R> (&v)[NV][8]) {
  if (!valid) return;
#pragma unroll
  for (int e = 0; e < 8; ++e)
#pragma unroll
    for (int k = 0; k < NV; ++k)
      dst[(size_t)(f + k) * a.N + (size_t)row * a.nx + Plan<Op::L>::exit_pos(Op::INV, t, e)] = v[k][e];
}
template <class Op, int NV>
__device__ __forceinline__ void load_rows(const KArgs<typename Op::R>& a, const C2<typename Op::R>* src, int f, int row,
                                          bool valid, int t, C2<typename Op::R> (&v)[NV][8]) {
#pragma unroll
  for (int e = 0; e < 8; ++e)
#pragma unroll
    for (int k = 0; k < NV; ++k)
      v[k][e] = valid ? src[(size_t)(f + k) * a.N + (size_t)row * a.nx + Plan<Op::L>::entry_pos(Op::INV, t, e)]
                      : cmk<C2<typename Op::R>>(0, 0);
}

// A block takes MX rows of the op's NF fields.  With field groups (FP64), field f of
// row m belongs to the L/8 threads of group (f, m): a thread holds eight values of
// one line whatever the op (it used to transform all fields of its row: up to 255
// registers, 8 warps per SM), and the points of the parked rows are then taken in
// order by all threads of the block.  Forward ops, whose fields cost differently,
// rotate the fields among the groups.  Without groups (FP32) a thread keeps to the
// points of its own row.
template <class Op> __device__ __forceinline__ void xpass_body(const KArgs<typename Op::R>& a) {
  using R = typename Op::R;
  using C = C2<R>;
  constexpr int L = Op::L, NF = Op::NF, NS = Op::NS, G = RowGroups<Op>::v, NV = NF / G;
  constexpr int NSR = NS > 0 ? NS : 1;
  constexpr int TPL = L / 8;
  constexpr int LP = row_len_padded<R, L>();
  if (!gate_open(a)) return;
  extern __shared__ __align__(16) unsigned char smraw[];
  C* tw = reinterpret_cast<C*>(smraw);
  LhyNode<R>* nodes = reinterpret_cast<LhyNode<R>*>(tw + L);
  C* buf = reinterpret_cast<C*>(reinterpret_cast<unsigned char*>(nodes) + (Op::USES_LHY ? lhy_stage_bytes<R>(a.Q) : 0));
  double* vrow = reinterpret_cast<double*>(buf + NF * a.MX * LP);  // trap terms of the rows (block-wide epilogues)
  RedSmem<NSR>* red = reinterpret_cast<RedSmem<NSR>*>(vrow + a.MX);
  const int tid = threadIdx.x;
  const int g = G > 1 || ExtraGroups<Op>::v > 1 ? tid / (a.MX * TPL) : 0;
  const int rt = tid - g * a.MX * TPL;
  const int mrow = rt / TPL, t = rt - mrow * TPL;
  const int fs = a.MX * LP;  // a field's rows in buf
  C* line = buf + g * fs + mrow * LP;
  for (int i = tid; i < L; i += blockDim.x) tw[i] = a.twx[i];
  if constexpr (Op::USES_LHY) {
    if constexpr (LhyTabOp<Op>::v) stage_lhy_nodes(nodes, a.xnodes, a.Qx);
    else stage_lhy_nodes(nodes, a.nodes, a.Q);
  }
  __syncthreads();
  typename Op::Uni u;
  Op::uniform(a, u);
  PAcc<R> acc[NSR];
  const int rows = a.ny * a.nz;
  const int ngroups = (rows + a.MX - 1) / a.MX;
  const RowIdx<PadShift<R>::v> si{};
  int f = g;
  for (int grp = blockIdx.x; grp < ngroups; grp += gridDim.x) {
    const int row = grp * a.MX + mrow;
    const bool valid = row < rows;
    C v[NV][8];
    if (ExtraGroups<Op>::v == 1 || g < NF) {
      Op::load(a, u, f, row, valid, t, v);
      fft_line<C, L, Op::INV, NV, WideOp<Op>::v>(v, line, fs, tw, t, si);
    }
    if constexpr (!Op::POINTS) {
      Op::store(a, u, f, row, valid, t, v, acc);
      if constexpr (G > 1 && !Op::INV) f = f + 1 < G ? f + 1 : 0;
    } else {
      constexpr bool ST = StageOut<Op>::v;
      if (ST && (ExtraGroups<Op>::v == 1 || g < NF)) {
#pragma unroll
        for (int k = 0; k < NV; ++k)
#pragma unroll
          for (int e = 0; e < 8; ++e) line[k * fs + si(Plan<L>::exit_pos(Op::INV, t, e))] = v[k][e];
      }
      R s[NSR];
#pragma unroll
      for (int k = 0; k < NSR; ++k) s[k] = 0;
      if constexpr (sizeof(R) == 8) {  // all points of the block's rows, one at a time
        if (tid < a.MX) vrow[tid] = grp * a.MX + tid < rows ? trap_yz(a, grp * a.MX + tid) : 0.0;
        __syncthreads();
        const int P = min(a.MX, rows - grp * a.MX) * L;
        for (int i = tid; i < P; i += blockDim.x) {
          RowPt<R, NF, ST> pt[1];
          const int m = i / L;
          pt[0].x = i - m * L;
          pt[0].idx = (size_t)(grp * a.MX) * L + i;
          pt[0].vyz = vrow[m];
          pt[0].sm = buf + m * LP + si(pt[0].x);
          pt[0].fs = fs;
          Op::points(a, u, pt, s, nodes);
        }
        __syncthreads();  // the next row group reuses the buffers
      } else if (valid) {
        constexpr int NP = Op::PTS;
        const R vyz = trap_yz(a, row);
#pragma unroll
        for (int e0 = 0; e0 < 8; e0 += NP) {
          RowPt<R, NF, ST> pt[NP];
#pragma unroll
          for (int j = 0; j < NP; ++j) {
            pt[j].x = Plan<L>::exit_pos(Op::INV, t, e0 + j);
            pt[j].idx = (size_t)row * L + pt[j].x;
            pt[j].vyz = vyz;
            pt[j].sm = line + si(pt[j].x);
            pt[j].fs = fs;
            if constexpr (!ST) {
#pragma unroll
              for (int k = 0; k < NF; ++k) pt[j].reg[k] = v[k][e0 + j];
            }
          }
          Op::points(a, u, pt, s, nodes);
        }
      }
#pragma unroll
      for (int k = 0; k < NSR; ++k) acc[k].add(s[k]);
      // a thread reads back what it parked; the next exchange overwrites its warp's
      // rows (rows that straddle warps for the mixed-radix lengths)
      if constexpr (ST && sizeof(R) == 4) {
        if constexpr (IsPow2<L>::v) __syncwarp();
        else __syncthreads();
      }
    }
  }
  if constexpr (NS > 0) {
    if (reduce_blocks<NS>(acc, a.partials, a.counter, Op::out(a, u), *red)) {
      if (threadIdx.x == 0) Op::finish(a, u);
    }
  }
}

// Shared memory per row of a block, and the rows per block unless tuned: as many
// as the op's threads and 46 KB allow; FP64 passes (bound by arithmetic) halve them
// while there are fewer row groups than SMs: at 32^3 the line pass ran on 16 SMs,
// 80 us against 51.
template <class Op> __host__ __device__ constexpr size_t row_pass_bytes() {
  return (size_t)Op::NF * row_len_padded<typename Op::R, Op::L>() * sizeof(C2<typename Op::R>) + sizeof(double);
}
template <class Op> inline int default_rows(int rows, int nsm) {
  constexpr int TPL = RowGroups<Op>::v * Op::L / 8;
  int mx = whole_warp_rows(Op::L);
  while (mx * 2 * TPL <= MaxThreads<Op>::v && mx * 2 * row_pass_bytes<Op>() <= 46 * 1024 &&
         (sizeof(typename Op::R) == 4 || rows >= mx * 2 * nsm))
    mx *= 2;
  return mx;
}

// Thread groups of a launch: the extra ones where each SM has at most two row groups
// (at 32^3 the energy epilogue takes 26 us instead of 40, the line epilogue 33 instead
// of 48; at 128^3 they cost 12%).
template <class Op> inline int row_groups(int mx, int rows, int nsm) {
  return ExtraGroups<Op>::v > 1 && mx == whole_warp_rows(Op::L) && rows <= mx * 2 * nsm ? ExtraGroups<Op>::v
                                                                                         : RowGroups<Op>::v;
}

// Row-pass entry points.  A min-blocks bound is given only when the op asks for
// more than one resident block: an explicit 1 lets the compiler take far more
// registers than the default heuristic does.
template <class Op> __global__ void __launch_bounds__(MaxThreads<Op>::v) xpass_kernel(KArgs<typename Op::R> a) {
  xpass_body<Op>(a);
}
template <class Op>
__global__ void __launch_bounds__(MaxThreads<Op>::v, MinBlocks<Op>::v) xpass_kernel_mb(KArgs<typename Op::R> a) {
  xpass_body<Op>(a);
}
template <class Op>
__global__ void __launch_bounds__(MaxThreads<Op>::v) xpass_kernel_b(const __grid_constant__ KBatch<typename Op::R> kb) {
  xpass_body<Op>(kb.k[blockIdx.y]);
}
template <class Op>
__global__ void __launch_bounds__(MaxThreads<Op>::v, MinBlocks<Op>::v)
    xpass_kernel_bmb(const __grid_constant__ KBatch<typename Op::R> kb) {
  xpass_body<Op>(kb.k[blockIdx.y]);
}

#ifndef EGPE_COL_STAGES
#define EGPE_COL_STAGES 2
#endif
// Tiles in flight per block of a TMA-fed column pass (one transformed, the
// rest loading).
constexpr int kColStages = EGPE_COL_STAGES;

// Threads per block of a column pass.  The power-of-two lengths are bound to
// 512 threads (tile rows of 64 to 256 bytes, chosen at run time); the
// mixed-radix lengths keep 128-byte rows, max(128 B / element, whole warps)
// columns times L/8 threads, and give the compiler that exact bound.
template <class Op> struct ColMaxThreads {
  static constexpr int TPL = Op::L / 8;
  static constexpr int MC = (int)(128 / sizeof(C2<typename Op::R>));
  static constexpr int MW = whole_warp_rows(Op::L);
  static constexpr int exact = (MC > MW ? MC : MW) * TPL;
  static constexpr int v = IsPow2<Op::L>::v ? 512 : exact;
  static constexpr int minb = 1;
};

// Columns per tile at the default 128-byte tile rows (what the host picks for
// every grid while the column tile width is untuned): the kernels for this
// width take it as a compile-time constant.
template <class Op> struct ColDefaultM {
  static constexpr int TPL = Op::L / 8;
  static constexpr int MB = (int)(128 / sizeof(C2<typename Op::R>));
  static constexpr int M0 = IsPow2<Op::L>::v ? (MB < 512 / TPL ? MB : 512 / TPL) : MB;
  static constexpr int v = M0 > whole_warp_rows(Op::L) ? M0 : whole_warp_rows(Op::L);
};
// FP64: threads per SM the passes ask for (registers 65536 / this).  The fixed-point
// lines wait on integer chains, which more warps hide.
constexpr int kCol64Threads = 512;
// Launch bounds of a column kernel: the run-time width keeps ColMaxThreads; a
// compile-time width MC has exactly MC L/8 threads, and the FP32 plain y/z
// passes (the ColPlain op, small epilogue) of up to 256 threads ask for three
// resident blocks, as their run-time-width build reached without a bound.  The
// FP32 mixed-radix passes ask for about 576 threads per SM: at 96^3 the energy
// pass takes 24 us with three blocks of 192 and 33 us with two.
template <class Op> struct ColMinB {
  static constexpr int threads = ColDefaultM<Op>::v * (Op::L / 8);
  static constexpr int want = sizeof(typename Op::R) == 8 ? kCol64Threads : !IsPow2<Op::L>::v ? 576 : 0;
  static constexpr int v = want > threads ? want / threads : 1;
};
template <class Op, int MC> struct ColBounds {
  static constexpr int threads = MC > 0 ? MC * (Op::L / 8) : ColMaxThreads<Op>::v;
  static constexpr int minb = MC > 0 && threads <= 256 ? ColMinB<Op>::v : ColMaxThreads<Op>::minb;
};

// ----------------------------------------------------------------------------
// Column (y or z) pass kernel
// ----------------------------------------------------------------------------
template <class Op, int MC> __device__ __forceinline__ void colpass_body(const KArgs<typename Op::R>& a) {
  using R = typename Op::R;
  using C = C2<R>;
  constexpr int L = Op::L, NS = Op::NS;
  constexpr int NSR = NS > 0 ? NS : 1;
  if (!gate_open(a)) return;
  const int M = MC > 0 ? MC : a.M;  // columns per tile
  extern __shared__ __align__(16) unsigned char smraw[];
  C* tw = reinterpret_cast<C*>(smraw);
  C* buf = tw + L;  // two exchange buffers of M lines each
  uint2* slots = reinterpret_cast<uint2*>(buf + 2 * M * L);
  RedSmem<NSR>* red = reinterpret_cast<RedSmem<NSR>*>(reinterpret_cast<unsigned char*>(slots) + line_slots<R>(M * (L / 8)));
  const int tid = threadIdx.x;
  const int m = tid % M, t = tid / M;
  const C* twsrc = (Op::AXIS == 1) ? a.twy : a.twz;
  for (int i = tid; i < L; i += blockDim.x) tw[i] = twsrc[i];
  __syncthreads();
  typename Op::Uni u;
  Op::uniform(a, u, t);
  PAcc<R> acc[NSR];
  const int xb_n = a.nx / M;
  const int other_n = (Op::AXIS == 1) ? a.nz : a.ny;
  const int tiles = xb_n * other_n * a.nf;
  const size_t lstride = (Op::AXIS == 1) ? (size_t)a.nx : (size_t)a.nx * a.ny;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const int xb = tile % xb_n;
    const int rest = tile / xb_n;
    const int o = rest % other_n;
    const int f = a.f0 + rest / other_n;
    const int x = xb * M + m;
    const size_t base = (size_t)f * a.N + (Op::AXIS == 1 ? (size_t)o * a.nx * a.ny : (size_t)o * a.nx) + x;
    const C* src = Op::src(a);
    C v[1][8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[0][e] = src[base + (size_t)Plan<L>::entry_pos(Op::FIRST_INV, t, e) * lstride];
    Op::process(a, u, f, x, o, base, lstride, t, v, buf + m, tw, ColIdxT<MC>{M, M * L, slots + m}, acc);
    // the last exchange's reads end before the next tile's first writes
    if constexpr (IsPow2<L>::v) __syncthreads();
  }
  if constexpr (NS > 0) {
    if (reduce_blocks<NS>(acc, a.partials, a.counter, Op::out(a, u), *red)) {
      if (threadIdx.x == 0) Op::finish(a, u);
    }
  }
}
template <class Op, int MC = 0>
__global__ void __launch_bounds__(ColBounds<Op, MC>::threads, ColBounds<Op, MC>::minb)
    colpass_kernel(KArgs<typename Op::R> a) {
  colpass_body<Op, MC>(a);
}
template <class Op, int MC = 0>
__global__ void __launch_bounds__(ColBounds<Op, MC>::threads, ColBounds<Op, MC>::minb)
    colpass_kernel_b(const __grid_constant__ KBatch<typename Op::R> kb) {
  colpass_body<Op, MC>(kb.k[blockIdx.y]);
}

// ----------------------------------------------------------------------------
// Column (y or z) pass fed by TMA.  The tensor map describes the workspace as
// a 3D array (x in 8-byte elements, y, z x fields); one box is one tile, M
// columns by the whole line, landing in shared memory position-major exactly
// as the FFT's column layout expects.  While tile i is transformed, tile i+1
// is already loading into the other buffer.  Results go straight to global
// memory from registers.
// ----------------------------------------------------------------------------
template <class Op, int MC>
__device__ __forceinline__ void colpass_tma_body(const CUtensorMap* tm, const KArgs<typename Op::R>& a) {
  using R = typename Op::R;
  using C = C2<R>;
  constexpr int L = Op::L, NS = Op::NS;
  constexpr int NSR = NS > 0 ? NS : 1;
  constexpr int NST = kColStages;
  if (!gate_open(a)) return;
  const int M = MC > 0 ? MC : a.M;  // columns per tile
  extern __shared__ __align__(128) unsigned char smraw_tma[];
  const int tileC = M * L;
  C* tiles = reinterpret_cast<C*>(smraw_tma);  // NST tiles, then the second exchange buffer
  C* xbuf = tiles + NST * tileC;
  C* tw = xbuf + tileC;
  uint64_t* bar = reinterpret_cast<uint64_t*>(tw + L);
  uint2* slots = reinterpret_cast<uint2*>(bar + NST);
  RedSmem<NSR>* red = reinterpret_cast<RedSmem<NSR>*>(reinterpret_cast<unsigned char*>(slots) + line_slots<R>(M * (L / 8)));
  const int tid = threadIdx.x;
  const int m = tid % M, t = tid / M;
  const C* twsrc = (Op::AXIS == 1) ? a.twy : a.twz;
  for (int i = tid; i < L; i += blockDim.x) tw[i] = twsrc[i];
  if (tid == 0) {
#pragma unroll
    for (int s = 0; s < NST; ++s) mbar_init(&bar[s], 1);
    fence_barrier_init();
  }
  __syncthreads();
  typename Op::Uni u;
  Op::uniform(a, u, t);
  PAcc<R> acc[NSR];
  const int xb_n = a.nx / M;
  const int other_n = (Op::AXIS == 1) ? a.nz : a.ny;
  const int tiles_n = xb_n * other_n * a.nf;
  const size_t lstride = (Op::AXIS == 1) ? (size_t)a.nx : (size_t)a.nx * a.ny;
  const uint32_t bytes = (uint32_t)(tileC * sizeof(C));
  constexpr int ESZ = (int)(sizeof(C) / 8);  // 8-byte TMA elements per complex value
  auto issue = [&](int tile, int b) {
    const int xb = tile % xb_n;
    const int rest = tile / xb_n;
    const int o = rest % other_n;
    const int f = a.f0 + rest / other_n;
    const int c0 = xb * M * ESZ;
    const int c1 = (Op::AXIS == 1) ? 0 : o;
    const int c2 = (Op::AXIS == 1) ? f * a.nz + o : f * a.nz;
    fence_proxy_async();
    mbar_expect_tx(&bar[b], bytes);
    tma_load_3d(tiles + b * tileC, tm, c0, c1, c2, &bar[b]);
  };
  // iteration q of this block handles tile blockIdx.x + q gridDim.x in buffer q % NST;
  // the copies of the next NST - 1 iterations are in flight while one is transformed
  auto tile_of = [&](int q) { return (int)blockIdx.x + q * (int)gridDim.x; };
  if (tid == 0) {
#pragma unroll
    for (int q = 0; q < NST - 1; ++q)
      if (tile_of(q) < tiles_n) issue(tile_of(q), q);
  }
  bool timed_out = false;
  int it = 0;
  for (int tile = blockIdx.x; tile < tiles_n; tile += gridDim.x, ++it) {
    const int b = it % NST;
    const int ahead = tile_of(it + NST - 1);
    // its buffer was last used by iteration it - 1, which ended with a barrier
    if (tid == 0 && ahead < tiles_n) issue(ahead, (it + NST - 1) % NST);
    const bool ok = mbar_wait(&bar[b], (uint32_t)((it / NST) & 1), a.wait_polls);
    if (__syncthreads_or(!ok)) {
      timed_out = true;
      break;
    }
    C* tb = tiles + b * tileC;
    C v[1][8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[0][e] = tb[Plan<L>::entry_pos(Op::FIRST_INV, t, e) * M + m];
    // power-of-two lengths exchange through the second buffer first, and the
    // barrier of that exchange orders these reads before the tile's reuse;
    // the mixed-radix passes work in place in the tile
    if constexpr (!IsPow2<L>::v) __syncthreads();
    const int xb = tile % xb_n;
    const int rest = tile / xb_n;
    const int o = rest % other_n;
    const int f = a.f0 + rest / other_n;
    const int x = xb * M + m;
    const size_t base = (size_t)f * a.N + (Op::AXIS == 1 ? (size_t)o * a.nx * a.ny : (size_t)o * a.nx) + x;
    Op::process(a, u, f, x, o, base, lstride, t, v, tb + m, tw, ColIdxT<MC>{M, (int)(xbuf - tb), slots + m}, acc);
    __syncthreads();  // buffer b may be refilled, and the second buffer rewritten, from here on
  }
  if (timed_out) {
    // let every copy already issued land before exiting: these waits keep the
    // full budget whatever a.wait_polls says, so no copy can still write into
    // shared memory once the block has left
    for (int q = it; q < it + NST; ++q)
      if (tile_of(q) < tiles_n) mbar_wait(&bar[q % NST], (uint32_t)((q / NST) & 1), kTmaWaitPolls);
    if (tid == 0) {
      a.st->timeout = 1;  // sticky: every later controller step ends the run
      a.st->status = 7;   // EGPE_ERR_TIMEOUT
      a.st->phase = PH_DONE;
    }
  }
  if constexpr (NS > 0) {
    if (reduce_blocks<NS>(acc, a.partials, a.counter, Op::out(a, u), *red)) {
      if (threadIdx.x == 0) Op::finish(a, u);
    }
  }
}
template <class Op, int MC = 0>
__global__ void __launch_bounds__(ColBounds<Op, MC>::threads, ColBounds<Op, MC>::minb)
    colpass_tma_kernel(const __grid_constant__ CUtensorMap tm, KArgs<typename Op::R> a) {
  colpass_tma_body<Op, MC>(&tm, a);
}
template <class Op, int MC = 0>
__global__ void __launch_bounds__(ColBounds<Op, MC>::threads, ColBounds<Op, MC>::minb)
    colpass_tma_kernel_b(const __grid_constant__ KBatch<typename Op::R> kb) {
  colpass_tma_body<Op, MC>(&kb.tm[blockIdx.y], kb.k[blockIdx.y]);
}

struct NoUni {};

// ----------------------------------------------------------------------------
// Plain transforms (diagnostic entry point and the y passes of the pipelines)
// ----------------------------------------------------------------------------
template <class R_, int L_, bool INV_> struct XPlain {
  using R = R_;
  using C = C2<R>;
  static constexpr const char* NAME = "x-plain";
  static double alg_bytes(const KArgs<R>& a) { return 2.0 * a.N * sizeof(C); }
  static constexpr int L = L_, NF = 1, NS = 0;
  static constexpr bool INV = INV_, USES_LHY = false, POINTS = false, WIDE = true;
  using Uni = NoUni;
  static __device__ void uniform(const KArgs<R>&, Uni&) {}
  template <int NV>
  static __device__ void load(const KArgs<R>& a, Uni&, int f, int row, bool valid, int t, C (&v)[NV][8]) {
    load_rows<XPlain>(a, a.gin, f, row, valid, t, v);
  }
  template <int NV>
  static __device__ void store(const KArgs<R>& a, Uni&, int f, int row, bool valid, int t, C (&v)[NV][8], PAcc<R>*) {
    store_rows<XPlain>(a, a.gout, f, row, valid, t, v);
  }
  static __device__ double* out(const KArgs<R>&, Uni&) { return nullptr; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};

template <class R_, int L_, int AXIS_, bool INV_, bool WIDE = false> struct ColPlain {
  using R = R_;
  using C = C2<R>;
  static constexpr const char* NAME = AXIS_ == 1 ? "y-pass" : "z-pass";
  static double alg_bytes(const KArgs<R>& a) { return 2.0 * a.nf * a.N * sizeof(C); }
  static constexpr int L = L_, NS = 0, AXIS = AXIS_;
  static constexpr bool INV = INV_;
  using Uni = NoUni;
  static __device__ void uniform(const KArgs<R>&, Uni&, int) {}
  static constexpr bool FIRST_INV = INV_;
  static __device__ const C* src(const KArgs<R>& a) { return a.gin; }
  template <class SI>
  static __device__ void process(const KArgs<R>& a, Uni&, int, int, int, size_t base, size_t ls, int t,
                                 C (&v)[1][8], C* sm, const C* tw, SI si, PAcc<R>*) {
    fft_line<C, L, INV, 1, WIDE>(v, sm, 0, tw, t, si);
#pragma unroll
    for (int e = 0; e < 8; ++e) a.gout[base + (size_t)Plan<L>::exit_pos(INV, t, e) * ls] = v[0][e];
  }
  static __device__ double* out(const KArgs<R>&, Uni&) { return nullptr; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};
template <int L_, int AXIS_, bool INV_, bool WIDE> struct ColMinB<ColPlain<float, L_, AXIS_, INV_, WIDE>> {
  static constexpr int v = 3;
};

// ----------------------------------------------------------------------------
// Energy / gradient pipeline (Eq. 1, coupled eGPE):
//   x fwd (psi or trial psi; packed dipolar source) -> y fwd -> z fused
//   (kinetic |k|^2/2, dipolar kernel, Parseval kinetic energy) -> y inv ->
//   x inv + H psi, LHY, energy sums.
// Workspace fields: 0, 1 = psi_1, psi_2; 2 = zeta = sum_j gdd_1j n_j + i sum_j gdd_2j n_j
// (both dipolar potentials from one complex transform: the kernel is real and
// even, so Phi_1 = Re and Phi_2 = Im of the inverse).
// ----------------------------------------------------------------------------
template <class R> struct EgUni {
  int cur, slot, nsel;
  R ca[2], cb[2];  // ca: a - 1 in FP32
};

// Controller step after an energy/gradient evaluation (last block, one thread):
// ctrl 1 = NCG (start point or trial), ctrl 2 = end of an imaginary-time step.
template <class R> __device__ __forceinline__ void eg_ctrl(const KArgs<R>& a, int lin) {
  if (a.ctrl == 2) {
    a.st->ffts += 20;  // two kinetic half steps (8) and two evaluations (12)
    Ctrl<R>::after_ite(a.st);
  } else if (a.ctrl) {
    a.st->ffts += lin ? 2 : 6;
    Ctrl<R>::after_eg(a.st, a.flag ? 1 : 0, lin, a.trace);
  }
}

template <class R_, int L_> struct XFwdEG {
  using R = R_;
  using C = C2<R>;
  static constexpr const char* NAME = "x-fwd energy";
  static double alg_bytes(const KArgs<R>& a) { return (a.flag ? 9.0 : a.gin ? 7.0 : 5.0) * a.N * sizeof(C); }
  static constexpr int L = L_, NF = 3, NS = 0;
  static constexpr bool INV = false, USES_LHY = false, POINTS = false;
  using Uni = EgUni<R>;
  static __device__ void uniform(const KArgs<R>& a, Uni& u) {
    u.cur = __ldcg(&a.st->cur);
    u.slot = a.flag ? (u.cur ^ 1) : u.cur;
    u.nsel = __ldcg(&a.st->n) & 1;
    R c[4];
    const double* ca = sizeof(R) == 4 ? a.st->coef_d : a.st->coef_a;
    load_uniforms<R, 4>({&ca[0], &ca[1], &a.st->coef_b[0], &a.st->coef_b[1]}, c);
    u.ca[0] = c[0];
    u.ca[1] = c[1];
    u.cb[0] = c[2];
    u.cb[1] = c[3];
  }
  // fields 0, 1: psi or the trial point on the geodesic (Sec. III), renormalised
  // (Sec. V) and stored; field 2: the dipolar source from both components (a group
  // of its own reads what the other two read at the same time, from L1/L2)
  static __device__ C source(const KArgs<R>& a, C p1, C p2) {
    const R n1 = cabs2(p1), n2 = cabs2(p2);
    return cmk<C>(fma_(a.d12, n2, a.d11 * n1), fma_(a.d22, n2, a.d21 * n1));
  }
  // a p + b q.  FP32: p + ((a - 1) p + b q).  Near convergence a is within a few units
  // of 1: rounded to 24 bits it moves the norm by up to 6e-8, and a p rounded on its
  // own is off in one direction at nearly every point.  FP64: a p is the exact product
  // inside the FMA.
  static __device__ C trial(R ca, C p, R cb, C q) {
    if constexpr (sizeof(R) == 4) return cmk<C>(p.x + fma_(ca, p.x, cb * q.x), p.y + fma_(ca, p.y, cb * q.y));
    else return cmk<C>(fma_(ca, p.x, cb * q.x), fma_(ca, p.y, cb * q.y));
  }
  static __device__ C point(const KArgs<R>& a, const Uni& u, int i, size_t idx) {
    const C p = (a.gin ? a.gin : pick(a.psi, u.cur))[(size_t)i * a.N + idx];
    if (!a.flag) return p;
    const C q = pick(a.pb, u.nsel)[(size_t)i * a.N + idx];
    return trial(pick(u.ca, i), p, pick(u.cb, i), q);
  }
  template <int NV>
  static __device__ void load(const KArgs<R>& a, Uni& u, int f, int row, bool valid, int t, C (&v)[NV][8]) {
    const size_t base = (size_t)row * a.nx, N = a.N;
    if (!valid) {
#pragma unroll
      for (int e = 0; e < 8; ++e)
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k][e] = cmk<C>(0, 0);
      return;
    }
    if constexpr (NV == 1) {
      if (f < 2) {
#pragma unroll
        for (int e = 0; e < 8; ++e) v[0][e] = point(a, u, f, base + Plan<L>::entry_pos(false, t, e));
        if (a.flag || a.gin) {
          C* dst = pick(a.psi, u.slot) + (size_t)f * N + base;
#pragma unroll
          for (int e = 0; e < 8; ++e) dst[Plan<L>::entry_pos(false, t, e)] = v[0][e];
        }
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const size_t idx = base + Plan<L>::entry_pos(false, t, e);
          v[0][e] = source(a, point(a, u, 0, idx), point(a, u, 1, idx));
        }
      }
    } else {
      // both components at once, the loads of a chunk before its arithmetic
      constexpr int CH = ChunkW<R>::v;
      const C* src = a.gin ? a.gin : pick(a.psi, u.cur);
      const C* pd = pick(a.pb, u.nsel);
      C* dst = pick(a.psi, u.slot);
#pragma unroll
      for (int e0 = 0; e0 < 8; e0 += CH) {
        C q1[CH], q2[CH];
#pragma unroll
        for (int j = 0; j < CH; ++j) {
          const size_t idx = base + Plan<L>::entry_pos(false, t, e0 + j);
          v[0][e0 + j] = src[idx];
          v[1][e0 + j] = src[N + idx];
          if (a.flag) {
            q1[j] = pd[idx];
            q2[j] = pd[N + idx];
          }
        }
#pragma unroll
        for (int j = 0; j < CH; ++j) {
          C p1 = v[0][e0 + j], p2 = v[1][e0 + j];
          if (a.flag) {
            p1 = trial(u.ca[0], p1, u.cb[0], q1[j]);
            p2 = trial(u.ca[1], p2, u.cb[1], q2[j]);
            v[0][e0 + j] = p1;
            v[1][e0 + j] = p2;
          }
          if (a.flag || a.gin) {
            const size_t idx = base + Plan<L>::entry_pos(false, t, e0 + j);
            dst[idx] = p1;
            dst[N + idx] = p2;
          }
          v[2][e0 + j] = source(a, p1, p2);
        }
      }
    }
  }
  template <int NV>
  static __device__ void store(const KArgs<R>& a, Uni&, int f, int row, bool valid, int t, C (&v)[NV][8], PAcc<R>*) {
    store_rows<XFwdEG>(a, a.W, f, row, valid, t, v);
  }
  static __device__ double* out(const KArgs<R>&, Uni&) { return nullptr; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};

template <class R_, int L_> struct ZEg {
  using R = R_;
  using C = C2<R>;
  static constexpr const char* NAME = "z fused energy";
  static double alg_bytes(const KArgs<R>& a) { return 6.0 * a.N * sizeof(C); }
  static constexpr int L = L_, NS = 2, AXIS = 2;
  struct Uni : KzLine<R, L_> {
    int slot;
  };
  static __device__ void uniform(const KArgs<R>& a, Uni& u, int t) {
    const int cur = __ldcg(&a.st->cur);
    u.slot = a.flag ? (cur ^ 1) : cur;
    u.set(a, t);
  }
  static constexpr bool FIRST_INV = false;
  static __device__ const C* src(const KArgs<R>& a) { return a.W; }
  template <class SI>
  static __device__ void process(const KArgs<R>& a, Uni& u, int f, int x, int y, size_t base, size_t ls, int t,
                                 C (&v)[1][8], C* sm, const C* tw, SI si, PAcc<R>* acc) {
    fft_line<C, L, false, 1>(v, sm, 0, tw, t, si);
    const R kxy = kq_xy(a, x, y);
    R ekin = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const R kz = u.kz[e];
      R mult = kxy + kz;  // |k|^2/(2N)
      if (f < 2) ekin = fma_(mult, cabs2(v[0][e]), ekin);
      else mult = dip_mult(a, kz, mult);
      v[0][e] = cscale(v[0][e], mult);
    }
    if (f == 0) acc[0].add(ekin);
    else if (f == 1) acc[1].add(ekin);
    col_after<L>(sm, si);
    fft_line<C, L, true, 1>(v, sm, 0, tw, t, si);
#pragma unroll
    for (int e = 0; e < 8; ++e) a.W[base + (size_t)Plan<L>::exit_pos(true, t, e) * ls] = v[0][e];
  }
  static __device__ double* out(const KArgs<R>& a, Uni& u) { return a.st->egz[u.slot]; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};

// mu_LHY,i at NP points: the interpolation table plus the exactly evaluated
// nodes.  (The LHY density is F = (2/5)(n1 mu1 + n2 mu2), Euler's identity for
// degree 5/2; finalize_energy takes it from the sums of n_i mu_i.)
template <class R, int NP>
__device__ __forceinline__ void lhy_terms(const KArgs<R>& a, const LhyNode<R>* nodes, const LhyCoef<R>& cf,
                                          const R (&n1)[NP], const R (&n2)[NP], R (&m1)[NP], R (&m2)[NP]) {
#pragma unroll
  for (int j = 0; j < NP; ++j) m1[j] = m2[j] = R(0);
  if (a.Qx > 0) {
    if constexpr (NP == 1) {
      lhy_points<R, 1>(nodes, a.Qx, a.Qxm, cf, n1, n2, m1, m2);
    } else {
      // exact nodes two points at a time (few registers for a rarely long loop)
#pragma unroll
      for (int j = 0; j < NP; j += 2) {
        const R q1[2] = {n1[j], n1[j + 1]}, q2[2] = {n2[j], n2[j + 1]};
        R x1[2], x2[2];
        lhy_points<R, 2>(nodes, a.Qx, a.Qxm, cf, q1, q2, x1, x2);
        m1[j] = x1[0];
        m1[j + 1] = x1[1];
        m2[j] = x2[0];
        m2[j + 1] = x2[1];
      }
    }
  }
  if (a.tab.ni > 0) {
    R t1[NP], t2[NP];
    lhy_tab_mu<R, NP>(a.tab, n1, n2, t1, t2);
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      m1[j] += t1[j];
      m2[j] += t2[j];
    }
  }
}

// n'^T (d^2 F/dn dn) n' at NP points: table plus exactly evaluated nodes.
template <class R, int NP>
__device__ __forceinline__ void lhy_second(const KArgs<R>& a, const LhyNode<R>* nodes, const LhyCoef<R>& cf,
                                           const R (&n1)[NP], const R (&n2)[NP], const R (&n1p)[NP],
                                           const R (&n2p)[NP], R (&H)[NP]) {
#pragma unroll
  for (int j = 0; j < NP; ++j) H[j] = R(0);
  if (a.Qx > 0) {
    if constexpr (NP == 1) {
      lhy_hess<R, 1>(nodes, a.Qx, a.Qxm, cf, n1, n2, n1p, n2p, H);
    } else {
#pragma unroll
      for (int j = 0; j < NP; j += 2) {
        const R q1[2] = {n1[j], n1[j + 1]}, q2[2] = {n2[j], n2[j + 1]};
        const R p1[2] = {n1p[j], n1p[j + 1]}, p2[2] = {n2p[j], n2p[j + 1]};
        R hx[2];
        lhy_hess<R, 2>(nodes, a.Qx, a.Qxm, cf, q1, q2, p1, p2, hx);
        H[j] = hx[0];
        H[j + 1] = hx[1];
      }
    }
  }
  if (a.tab.ni > 0) {
    R t[NP];
    lhy_tab_hess<R, NP>(a.tab, n1, n2, n1p, n2p, t);
#pragma unroll
    for (int j = 0; j < NP; ++j) H[j] += t[j];
  }
}

template <class R_, int L_, bool LIN> struct XInvEGT {
  using R = R_;
  using C = C2<R>;
  // FP32: 128 threads, 4 blocks per SM (128 registers; the mixed-radix lengths 3, which
  // spill at 4); FP64: three groups of 32 threads
  static constexpr int PTS = 4, MAXT = sizeof(R_) == 4 ? 128 : LIN ? 64 : 96, MINB = sizeof(R_) == 4 ? (IsPow2<L_>::v ? 4 : 3) : 1;
  static constexpr bool STAGE_OUT = true;
  static constexpr const char* NAME = "x-inv energy+LHY";
  static double alg_bytes(const KArgs<R>& a) { return (LIN || a.att == ATT_FULL ? 9.0 : 11.0) * a.N * sizeof(C); }
  static constexpr int L = L_, NF = LIN ? 1 : 3, NS = LIN ? EG_NS : EG_KIN1;
  static constexpr bool INV = true, USES_LHY = true, LHY_TAB = true, POINTS = true;
  using Uni = EgUni<R>;
  static __device__ void uniform(const KArgs<R>& a, Uni& u) { XFwdEG<R, L>::uniform(a, u); }
  template <int NV>
  static __device__ void load(const KArgs<R>& a, Uni&, int f, int row, bool valid, int t, C (&v)[NV][8]) {
    load_rows<XInvEGT>(a, a.W, f, row, valid, t, v);
  }
  template <int NP, bool ST>
  static __device__ void points(const KArgs<R>& a, Uni& u, const RowPt<R, NF, ST> (&pt)[NP], R (&s)[NS],
                                const LhyNode<R>* nodes) {
    const C* ps = pick(a.psi, u.slot);
    C* hp = pick(a.hp, u.slot);
    C* ax = pick(a.ax, u.slot);
    C* tb = pick(a.tb, u.slot);
    const size_t N = a.N;
    C p1[NP], p2[NP], k1[NP], k2[NP];
    R n1[NP], n2[NP], m1[NP], m2[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      p1[j] = ps[pt[j].idx];
      p2[j] = ps[N + pt[j].idx];
      if constexpr (LIN) {
        k1[j] = tb[pt[j].idx];
        k2[j] = tb[N + pt[j].idx];
      }
      n1[j] = cabs2(p1[j]);
      n2[j] = cabs2(p2[j]);
    }
    lhy_terms<R, NP>(a, nodes, lhy_coef(a), n1, n2, m1, m2);
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const size_t idx = pt[j].idx;
      const R V = trap_x(a, pt[j].x) + pt[j].vyz;
      const C T1 = LIN ? k1[j] : pt[j].out(0), T2 = LIN ? k2[j] : pt[j].out(NF > 1 ? 1 : 0);
      const C PH = pt[j].out(NF - 1);
      if constexpr (LIN) {
        cdot_add(s[EG_KIN1], p1[j], T1);
        cdot_add(s[EG_KIN2], p2[j], T2);
      } else if (a.att != ATT_FULL) {
        tb[idx] = T1;
        tb[N + idx] = T2;
      }
      const R phi1 = PH.x, phi2 = PH.y;
      const R c1 = fma_(a.g12, n2[j], a.g11 * n1[j]), c2 = fma_(a.g22, n2[j], a.g21 * n1[j]);
      const R B1 = (V + c1) + m1[j], B2 = (V + c2) + m2[j];
      const R U1 = B1 + phi1, U2 = B2 + phi2;
      const C H1 = cmk<C>(fma_(U1, p1[j].x, T1.x), fma_(U1, p1[j].y, T1.y));
      const C H2 = cmk<C>(fma_(U2, p2[j].x, T2.x), fma_(U2, p2[j].y, T2.y));
      hp[idx] = H1;
      hp[N + idx] = H2;
      if (!LIN && a.gout) {
        a.gout[idx] = H1;
        a.gout[N + idx] = H2;
      }
      ax[idx] = PH;
      ax[N + idx] = cmk<C>(B1, B2);
      // the energies and mu_i are combinations of these (finalize_energy)
      s[EG_TRAP1] = fma_(V, n1[j], s[EG_TRAP1]);
      s[EG_TRAP2] = fma_(V, n2[j], s[EG_TRAP2]);
      s[EG_CON1] = fma_(c1, n1[j], s[EG_CON1]);
      s[EG_CON2] = fma_(c2, n2[j], s[EG_CON2]);
      s[EG_NPHI1] = fma_(n1[j], phi1, s[EG_NPHI1]);
      s[EG_NPHI2] = fma_(n2[j], phi2, s[EG_NPHI2]);
      s[EG_NMUL1] = fma_(n1[j], m1[j], s[EG_NMUL1]);
      s[EG_NMUL2] = fma_(n2[j], m2[j], s[EG_NMUL2]);
      s[EG_NORM1] += n1[j];
      s[EG_NORM2] += n2[j];
    }
  }
  static __device__ double* out(const KArgs<R>& a, Uni& u) { return a.st->eg[u.slot]; }
  static __device__ void finish(const KArgs<R>& a, Uni&) { eg_ctrl(a, LIN); }
};
template <class R, int L> struct XInvEG : XInvEGT<R, L, false> {};
template <class R, int L> struct XInvEL : XInvEGT<R, L, true> {};

// ----------------------------------------------------------------------------
// Preconditioner pipeline (Sec. IV.B): r = H psi - mu psi, z = P^{-1} r with
// P^{-1} = P_Delta^{-1} P_V^{-1}; sums for HS+ beta, projection and descent.
// ----------------------------------------------------------------------------
template <class R> struct PcUni {
  int cur, nsel, rgiven;
  bool direct;  // PH_DIRECT: the passes form w = (alpha + T) r of a residual-fallback step
  R mu[2], shift[2], floor_[2];
  R wv;  // weight of P_V in the blended preconditioner
};
// Only FP64 engines carry T p along (engine.h).
template <class R> __device__ __forceinline__ bool pc_direct(const KArgs<R>& a) {
  return sizeof(R) == 8 && a.att != ATT_FULL && __ldcg(&a.st->phase) == PH_DIRECT;
}
template <class R> __device__ __forceinline__ void pc_uniform(const KArgs<R>& a, PcUni<R>& u) {
  u.direct = pc_direct(a);
  u.cur = __ldcg(&a.st->cur);
  u.nsel = __ldcg(&a.st->n) & 1;
  u.rgiven = a.flag;
  if constexpr (sizeof(R) == sizeof(double)) {
    u.wv = __ldcg(&a.st->opt.pc_blend);
    const double fl = __ldcg(&a.st->opt.pv_floor);
    for (int i = 0; i < 2; ++i) {
      u.mu[i] = __ldcg(&a.st->mu[i]);
      u.shift[i] = __ldcg(&a.st->shift[i]);
      u.floor_[i] = fl * u.shift[i];
      if (u.direct) {  // P_V = 1: r itself is transformed (the z pass has its own shift)
        u.shift[i] = -1e300;
        u.floor_[i] = 1.0;
      }
    }
  } else {
    R c[6];
    load_uniforms<R, 6>(
        {&a.st->opt.pc_blend, &a.st->opt.pv_floor, &a.st->mu[0], &a.st->mu[1], &a.st->shift[0], &a.st->shift[1]}, c);
    u.wv = c[0];
    for (int i = 0; i < 2; ++i) {
      u.mu[i] = c[2 + i];
      u.shift[i] = c[4 + i];
      u.floor_[i] = c[1] * c[4 + i];
    }
  }
}

// P_V,i of component i at a point (Sec. IV.B) from B_i, with the floor.
template <class R> __device__ __forceinline__ R pv_at(const PcUni<R>& u, int i, R B) {
  const R P = pick(u.shift, i) + B, fl = pick(u.floor_, i);
  return P > fl ? P : fl;
}
// r_i = H_i psi_i - mu_i psi_i (stored unless given) and w_i = P_V^{-1} r_i when
// diag, at CH points: both components (NV = 2, i = 0) or component i alone.
template <class R, int CH, int NV>
__device__ __forceinline__ void pc_residual(const KArgs<R>& a, const PcUni<R>& u, int i, const size_t (&idx)[CH],
                                            C2<R> (&w)[NV][CH]) {
  using C = C2<R>;
  const size_t N = a.N;
  C h[NV][CH], p[NV][CH], bb[CH];
#pragma unroll
  for (int j = 0; j < CH; ++j) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const size_t q = (size_t)(i + k) * N + idx[j];
      h[k][j] = u.rgiven ? pick(a.rb, u.nsel)[q] : pick(a.hp, u.cur)[q];
      if (!u.rgiven) p[k][j] = pick(a.psi, u.cur)[q];
    }
    if (a.diag) bb[j] = pick(a.ax, u.cur)[N + idx[j]];
  }
#pragma unroll
  for (int j = 0; j < CH; ++j) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const int c = i + k;
      C r = h[k][j];
      if (!u.rgiven) {
        const R mu = pick(u.mu, c);
        r = cmk<C>(fma_(-mu, p[k][j].x, r.x), fma_(-mu, p[k][j].y, r.y));
        pick(a.rb, u.nsel)[(size_t)c * N + idx[j]] = r;
      }
      if (a.diag) {
        r = cscale(r, rcp_(pv_at(u, c, c ? bb[j].y : bb[j].x)));
        if (a.att != ATT_FULL) a.wz[(size_t)c * N + idx[j]] = r;
      }
      w[k][j] = r;
    }
  }
}

// Inputs of the preconditioner sums at one point.
template <class R> struct PcSumIn {
  C2<R> r1, r2, q1, q2, d1, d2, p1, p2;
};
template <class R>
__device__ __forceinline__ void pc_sum_load(const KArgs<R>& a, const PcUni<R>& u, size_t idx, PcSumIn<R>& in) {
  const size_t N = a.N;
  in.r1 = pick(a.rb, u.nsel)[idx];
  in.r2 = pick(a.rb, u.nsel)[N + idx];
  in.q1 = pick(a.rb, u.nsel ^ 1)[idx];
  in.q2 = pick(a.rb, u.nsel ^ 1)[N + idx];
  in.d1 = pick(a.pb, u.nsel ^ 1)[idx];
  in.d2 = pick(a.pb, u.nsel ^ 1)[N + idx];
  in.p1 = pick(a.psi, u.cur)[idx];
  in.p2 = pick(a.psi, u.cur)[N + idx];
}
template <class R>
__device__ __forceinline__ void pc_sum_add(const PcSumIn<R>& in, C2<R> z1, C2<R> z2, R* s) {
  const C2<R> dr1 = csub(in.r1, in.q1), dr2 = csub(in.r2, in.q2);
  cdot_add(s[PC_SRZ], dr1, z1);
  cdot_add(s[PC_SRZ], dr2, z2);
  cdot_add(s[PC_SRP], dr1, in.d1);
  cdot_add(s[PC_SRP], dr2, in.d2);
  cdot_add(s[PC_ZPSI1], z1, in.p1);
  cdot_add(s[PC_ZPSI2], z2, in.p2);
  cdot_add(s[PC_PPPSI1], in.d1, in.p1);
  cdot_add(s[PC_PPPSI2], in.d2, in.p2);
  cdot_add(s[PC_ZR1], z1, in.r1);
  cdot_add(s[PC_ZR2], z2, in.r2);
  cdot_add(s[PC_PPR1], in.d1, in.r1);
  cdot_add(s[PC_PPR2], in.d2, in.r2);
  cdot_add(s[PC_PSIR1], in.p1, in.r1);
  cdot_add(s[PC_PSIR2], in.p2, in.r2);
  cdot_add(s[PC_RR1], in.r1, in.r1);
  cdot_add(s[PC_RR2], in.r2, in.r2);
}

template <class R_, int L_> struct XFwdPC {
  using R = R_;
  using C = C2<R>;
  static constexpr const char* NAME = "x-fwd precond";
  static double alg_bytes(const KArgs<R>& a) {
    return (a.diag ? a.att != ATT_FULL ? 11.0 : 9.0 : 8.0) * a.N * sizeof(C);
  }
  static constexpr int L = L_, NF = 2, NS = 0;
  static constexpr bool INV = false, USES_LHY = false, POINTS = false;
  using Uni = PcUni<R>;
  static __device__ void uniform(const KArgs<R>& a, Uni& u) { pc_uniform(a, u); }
  template <int NV>
  static __device__ void load(const KArgs<R>& a, Uni& u, int f, int row, bool valid, int t, C (&v)[NV][8]) {
    if (!valid) {
#pragma unroll
      for (int e = 0; e < 8; ++e)
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k][e] = cmk<C>(0, 0);
      return;
    }
    constexpr int CH = ChunkW<R>::v;
#pragma unroll
    for (int e0 = 0; e0 < 8; e0 += CH) {
      size_t idx[CH];
      C w[NV][CH];
#pragma unroll
      for (int j = 0; j < CH; ++j) idx[j] = (size_t)row * a.nx + Plan<L>::entry_pos(false, t, e0 + j);
      pc_residual<R, CH, NV>(a, u, f, idx, w);
#pragma unroll
      for (int j = 0; j < CH; ++j)
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k][e0 + j] = w[k][j];
    }
  }
  template <int NV>
  static __device__ void store(const KArgs<R>& a, Uni&, int f, int row, bool valid, int t, C (&v)[NV][8], PAcc<R>*) {
    store_rows<XFwdPC>(a, a.W, f, row, valid, t, v);
  }
  static __device__ double* out(const KArgs<R>&, Uni&) { return nullptr; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};

template <class R_, int L_> struct ZPc {
  using R = R_;
  using C = C2<R>;
  static constexpr const char* NAME = "z fused precond";
  static double alg_bytes(const KArgs<R>& a) { return 4.0 * a.N * sizeof(C); }
  static constexpr int L = L_, NS = 0, AXIS = 2;
  struct Uni : KzLine<R, L_> {
    R shift[2];
    bool direct;
  };
  static __device__ void uniform(const KArgs<R>& a, Uni& u, int t) {
    u.direct = pc_direct(a);
    load_uniforms<R, 2>({&a.st->shift[0], &a.st->shift[1]}, u.shift);
    u.set(a, t);
  }
  static constexpr bool FIRST_INV = false;
  static __device__ const C* src(const KArgs<R>& a) { return a.W; }
  template <class SI>
  static __device__ void process(const KArgs<R>& a, Uni& u, int f, int x, int y, size_t base, size_t ls, int t,
                                 C (&v)[1][8], C* sm, const C* tw, SI si, PAcc<R>*) {
    fft_line<C, L, false, 1>(v, sm, 0, tw, t, si);
    const R kxy = kq_xy(a, x, y);
    const R sh = a.invN * (f == 0 ? u.shift[0] : u.shift[1]);
    if (u.direct) {  // (shift + |k|^2/2) / N
#pragma unroll
      for (int e = 0; e < 8; ++e) v[0][e] = cscale(v[0][e], sh + (kxy + u.kz[e]));
    } else {
      // invN / (shift + |k|^2/2), numerator and denominator over N
#pragma unroll
      for (int e = 0; e < 8; ++e) v[0][e] = cscale(v[0][e], a.invN * a.invN * rcp_(sh + (kxy + u.kz[e])));
    }
    col_after<L>(sm, si);
    fft_line<C, L, true, 1>(v, sm, 0, tw, t, si);
#pragma unroll
    for (int e = 0; e < 8; ++e) a.W[base + (size_t)Plan<L>::exit_pos(true, t, e) * ls] = v[0][e];
  }
  static __device__ double* out(const KArgs<R>&, Uni&) { return nullptr; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};

template <class R_, int L_> struct XInvPC {
  using R = R_;
  using C = C2<R>;
  static constexpr int PTS = 4, MAXT = sizeof(R_) == 4 ? 128 : 64;  // heavy epilogue: small blocks, more of them per SM
  static constexpr const char* NAME = "x-inv precond sums";
  static double alg_bytes(const KArgs<R>& a) { return 12.0 * a.N * sizeof(C); }
  static constexpr int L = L_, NF = 2, NS = PC_NS;
  static constexpr bool INV = true, USES_LHY = false, POINTS = true;
  using Uni = PcUni<R>;
  static __device__ void uniform(const KArgs<R>& a, Uni& u) { pc_uniform(a, u); }
  template <int NV>
  static __device__ void load(const KArgs<R>& a, Uni&, int f, int row, bool valid, int t, C (&v)[NV][8]) {
    load_rows<XInvPC>(a, a.W, f, row, valid, t, v);
  }
  template <int NP, bool ST>
  static __device__ void points(const KArgs<R>& a, Uni& u, const RowPt<R, NF, ST> (&pt)[NP], R (&s)[PC_NS],
                                const LhyNode<R>*) {
    C* zd = u.direct ? a.wz : a.z;
    PcSumIn<R> in[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) pc_sum_load<R>(a, u, pt[j].idx, in[j]);
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const size_t idx = pt[j].idx;
      C z1 = pt[j].out(0), z2 = pt[j].out(1);
      if (a.blend) {  // z = (1 - w) P_Delta^{-1} r + w P_V^{-1} r
        const C bb = pick(a.ax, u.cur)[(size_t)a.N + idx];
        const R wd = R(1) - u.wv, w1 = u.wv * rcp_(pv_at(u, 0, bb.x)), w2 = u.wv * rcp_(pv_at(u, 1, bb.y));
        z1 = cmk<C>(wd * z1.x + w1 * in[j].r1.x, wd * z1.y + w1 * in[j].r1.y);
        z2 = cmk<C>(wd * z2.x + w2 * in[j].r2.x, wd * z2.y + w2 * in[j].r2.y);
      }
      zd[idx] = z1;
      zd[(size_t)a.N + idx] = z2;
      pc_sum_add<R>(in[j], z1, z2, s);
    }
  }
  static __device__ double* out(const KArgs<R>& a, Uni&) { return a.st->pc; }
  static __device__ void finish(const KArgs<R>& a, Uni&) {
    if (a.ctrl) {
      a.st->ffts += 4;
      Ctrl<R>::after_pc(a.st, a.att);
    }
  }
};

// Pointwise preconditioner (modes none and diagonal): one pass, no transform.
template <class R>
__device__ __forceinline__ void pc_point_body(const KArgs<R>& a) {
  using C = C2<R>;
  if (!gate_open(a)) return;
  __shared__ RedSmem<PC_NS> red;
  PcUni<R> u;
  pc_uniform(a, u);
  PAcc<R> acc[PC_NS];
  const size_t N = a.N;
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += (size_t)gridDim.x * blockDim.x) {
    C w[2][1];
    const size_t id[1] = {idx};
    pc_residual<R, 1, 2>(a, u, 0, id, w);
    const C w1 = w[0][0], w2 = w[1][0];
    a.z[idx] = w1;
    a.z[N + idx] = w2;
    R s[PC_NS];
#pragma unroll
    for (int k = 0; k < PC_NS; ++k) s[k] = 0;
    PcSumIn<R> si;
    pc_sum_load<R>(a, u, idx, si);
    pc_sum_add<R>(si, w1, w2, s);
#pragma unroll
    for (int k = 0; k < PC_NS; ++k) acc[k].add(s[k]);
  }
  if (reduce_blocks<PC_NS>(acc, a.partials, a.counter, a.st->pc, red)) {
    if (threadIdx.x == 0 && a.ctrl) Ctrl<R>::after_pc(a.st, a.att);
  }
}
template <class R> __global__ void __launch_bounds__(256) pc_point_kernel(KArgs<R> a) { pc_point_body(a); }
template <class R> __global__ void __launch_bounds__(256) pc_point_kernel_b(const __grid_constant__ KBatch<R> kb) {
  pc_point_body(kb.k[blockIdx.y]);
}


// ----------------------------------------------------------------------------
// Line-search pipeline (Sec. V): p = -z + beta p_prev - c psi (projected
// direction), forward transforms of p (Parseval <p|T|p>), the packed dipolar
// transform of rho = Re(psi conj p), and the pointwise second-variation sums.
// ----------------------------------------------------------------------------
template <class R> struct LcUni {
  int cur, nsel, pgiven, fallback;
  R beta, c[2];
};
template <class R> __device__ __forceinline__ void lc_uniform(const KArgs<R>& a, LcUni<R>& u) {
  u.cur = __ldcg(&a.st->cur);
  u.nsel = __ldcg(&a.st->n) & 1;
  u.pgiven = a.flag;
  u.fallback = __ldcg(&a.st->fallback);
  R c[3];
  load_uniforms<R, 3>({&a.st->beta, &a.st->c[0], &a.st->c[1]}, c);
  u.beta = c[0];
  u.c[0] = c[1];
  u.c[1] = c[2];
}

template <class R_, int L_> struct XFwdLC {
  using R = R_;
  using C = C2<R>;
  static constexpr const char* NAME = "x-fwd line dir";
  static double alg_bytes(const KArgs<R>& a) { return 11.0 * a.N * sizeof(C); }
  static constexpr int L = L_, NF = 3, NS = 0;
  static constexpr bool INV = false, USES_LHY = false, POINTS = false;
  using Uni = LcUni<R>;
  static __device__ void uniform(const KArgs<R>& a, Uni& u) { lc_uniform(a, u); }
  // direction p_i = -z_i + beta p_prev_i - c_i psi_i (the residual in place of z in
  // a fallback step) at one point; psi_i is returned beside it
  static __device__ C dir(const KArgs<R>& a, const Uni& u, int i, size_t idx, C& p) {
    const size_t k = (size_t)i * a.N + idx;
    p = pick(a.psi, u.cur)[k];
    if (u.pgiven) return pick(a.pb, u.nsel)[k];
    const C w = u.fallback ? pick(a.rb, u.nsel)[k] : a.z[k];
    const R c = pick(u.c, i);
    C q = cmk<C>(fma_(-c, p.x, -w.x), fma_(-c, p.y, -w.y));
    if (u.beta != R(0)) {
      const C d = pick(a.pb, u.nsel ^ 1)[k];
      q = cmk<C>(fma_(u.beta, d.x, q.x), fma_(u.beta, d.y, q.y));
    }
    return q;
  }
  static __device__ C source(const KArgs<R>& a, C p1, C q1, C p2, C q2) {
    const R rho1 = cdot(p1, q1), rho2 = cdot(p2, q2);
    return cmk<C>(fma_(a.d12, rho2, a.d11 * rho1), fma_(a.d22, rho2, a.d21 * rho1));
  }
  // fields 0, 1: p (stored unless given); field 2: the packed source of rho = Re(psi conj p)
  template <int NV>
  static __device__ void load(const KArgs<R>& a, Uni& u, int f, int row, bool valid, int t, C (&v)[NV][8]) {
    const size_t base = (size_t)row * a.nx, N = a.N;
    if (!valid) {
#pragma unroll
      for (int e = 0; e < 8; ++e)
#pragma unroll
        for (int k = 0; k < NV; ++k) v[k][e] = cmk<C>(0, 0);
      return;
    }
    C* dst = pick(a.pb, u.nsel);
    if constexpr (NV == 1) {
      if (f < 2) {
        C p;
#pragma unroll
        for (int e = 0; e < 8; ++e) v[0][e] = dir(a, u, f, base + Plan<L>::entry_pos(false, t, e), p);
        if (!u.pgiven) {
#pragma unroll
          for (int e = 0; e < 8; ++e) dst[(size_t)f * N + base + Plan<L>::entry_pos(false, t, e)] = v[0][e];
        }
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const size_t idx = base + Plan<L>::entry_pos(false, t, e);
          C p1, p2;
          const C q1 = dir(a, u, 0, idx, p1), q2 = dir(a, u, 1, idx, p2);
          v[0][e] = source(a, p1, q1, p2, q2);
        }
      }
    } else {
      // both components at once, the loads of a chunk before its arithmetic
      const C* ps = pick(a.psi, u.cur);
      const C* pp = pick(a.pb, u.nsel ^ 1);
      const C* ws = u.pgiven ? dst : u.fallback ? pick(a.rb, u.nsel) : a.z;
      const bool usepp = !u.pgiven && u.beta != R(0);
      constexpr int CH = ChunkW<R>::v;
#pragma unroll
      for (int e0 = 0; e0 < 8; e0 += CH) {
        C p1[CH], p2[CH], d1[CH], d2[CH];
#pragma unroll
        for (int j = 0; j < CH; ++j) {
          const size_t idx = base + Plan<L>::entry_pos(false, t, e0 + j);
          p1[j] = ps[idx];
          p2[j] = ps[N + idx];
          v[0][e0 + j] = ws[idx];
          v[1][e0 + j] = ws[N + idx];
          if (usepp) {
            d1[j] = pp[idx];
            d2[j] = pp[N + idx];
          }
        }
#pragma unroll
        for (int j = 0; j < CH; ++j) {
          if (u.pgiven) continue;
          C q1 = v[0][e0 + j], q2 = v[1][e0 + j];
          q1 = cmk<C>(fma_(-u.c[0], p1[j].x, -q1.x), fma_(-u.c[0], p1[j].y, -q1.y));
          q2 = cmk<C>(fma_(-u.c[1], p2[j].x, -q2.x), fma_(-u.c[1], p2[j].y, -q2.y));
          if (usepp) {
            q1 = cmk<C>(fma_(u.beta, d1[j].x, q1.x), fma_(u.beta, d1[j].y, q1.y));
            q2 = cmk<C>(fma_(u.beta, d2[j].x, q2.x), fma_(u.beta, d2[j].y, q2.y));
          }
          v[0][e0 + j] = q1;
          v[1][e0 + j] = q2;
        }
#pragma unroll
        for (int j = 0; j < CH; ++j) {
          const int e = e0 + j;
          if (!u.pgiven) {
            const size_t idx = base + Plan<L>::entry_pos(false, t, e);
            dst[idx] = v[0][e];
            dst[N + idx] = v[1][e];
          }
          v[2][e] = source(a, p1[j], v[0][e], p2[j], v[1][e]);
        }
      }
    }
  }
  template <int NV>
  static __device__ void store(const KArgs<R>& a, Uni&, int f, int row, bool valid, int t, C (&v)[NV][8], PAcc<R>*) {
    store_rows<XFwdLC>(a, a.W, f, row, valid, t, v);
  }
  static __device__ double* out(const KArgs<R>&, Uni&) { return nullptr; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};

template <class R_, int L_> struct ZLc {
  using R = R_;
  using C = C2<R>;
  static constexpr const char* NAME = "z line coeffs";
  static double alg_bytes(const KArgs<R>& a) { return 4.0 * a.N * sizeof(C); }
  static constexpr int L = L_, NS = 2, AXIS = 2;
  using Uni = KzLine<R, L_>;
  static __device__ void uniform(const KArgs<R>& a, Uni& u, int t) { u.set(a, t); }
  static constexpr bool FIRST_INV = false;
  static __device__ const C* src(const KArgs<R>& a) { return a.W; }
  template <class SI>
  static __device__ void process(const KArgs<R>& a, Uni& u, int f, int x, int y, size_t base, size_t ls, int t,
                                 C (&v)[1][8], C* sm, const C* tw, SI si, PAcc<R>* acc) {
    fft_line<C, L, false, 1>(v, sm, 0, tw, t, si);
    const R kxy = kq_xy(a, x, y);
    if (f < 2) {  // <p_f | T | p_f> by Parseval: forward transform only
      R tk = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const R kz = u.kz[e];
        tk = fma_(kxy + kz, cabs2(v[0][e]), tk);
      }
      if (f == 0) acc[0].add(tk);
      else acc[1].add(tk);
      return;
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const R kz = u.kz[e];
      v[0][e] = cscale(v[0][e], dip_mult(a, kz, kxy + kz));
    }
    col_after<L>(sm, si);
    fft_line<C, L, true, 1>(v, sm, 0, tw, t, si);
#pragma unroll
    for (int e = 0; e < 8; ++e) a.W[base + (size_t)Plan<L>::exit_pos(true, t, e) * ls] = v[0][e];
  }
  static __device__ double* out(const KArgs<R>& a, Uni&) { return a.st->lcz; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};

template <class R_, int L_, bool LIN> struct XInvLCT {
  using R = R_;
  using C = C2<R>;
  static constexpr int PTS = 4, MAXT = sizeof(R_) == 4 ? 256 : 64, MINB = sizeof(R_) == 4 ? 2 : 1;
  static constexpr const char* NAME = "x-inv line sums+LHY";
  static double alg_bytes(const KArgs<R>& a) { return 9.0 * a.N * sizeof(C); }
  static constexpr int L = L_, NF = 1, NS = LC_NS;
  static constexpr bool INV = true, USES_LHY = true, LHY_TAB = true, POINTS = true;
  using Uni = LcUni<R>;
  static __device__ void uniform(const KArgs<R>& a, Uni& u) { lc_uniform(a, u); }
  template <int NV>
  static __device__ void load(const KArgs<R>& a, Uni&, int, int row, bool valid, int t, C (&v)[NV][8]) {
    load_rows<XInvLCT>(a, a.W, LIN ? 0 : 2, row, valid, t, v);
  }
  template <int NP, bool ST>
  static __device__ void points(const KArgs<R>& a, Uni& u, const RowPt<R, NF, ST> (&pt)[NP], R (&s)[LC_NS],
                                const LhyNode<R>* nodes) {
    const size_t N = a.N;
    const C* ps = pick(a.psi, u.cur);
    const C* pd = pick(a.pb, u.nsel);
    const C* hp = pick(a.hp, u.cur);
    const C* ax = pick(a.ax, u.cur);
    R n1[NP], n2[NP], n1p[NP], n2p[NP], Hh[NP];
    C p1[NP], p2[NP], q1[NP], q2[NP], h1[NP], h2[NP], phi[NP], bb[NP];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const size_t idx = pt[j].idx;
      p1[j] = ps[idx];
      p2[j] = ps[N + idx];
      q1[j] = pd[idx];
      q2[j] = pd[N + idx];
      h1[j] = hp[idx];
      h2[j] = hp[N + idx];
      phi[j] = ax[idx];
      bb[j] = ax[N + idx];
    }
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      n1[j] = cabs2(p1[j]);
      n2[j] = cabs2(p2[j]);
      const R a1 = cabs2(q1[j]), a2 = cabs2(q2[j]);
      const R rho1 = cdot(p1[j], q1[j]), rho2 = cdot(p2[j], q2[j]);
      n1p[j] = rho1 + rho1;
      n2p[j] = rho2 + rho2;
      const C PR = pt[j].out(0);
      const R U1 = phi[j].x + bb[j].x, U2 = phi[j].y + bb[j].y;
      s[LC_P1] += a1;
      s[LC_P2] += a2;
      s[LC_PSIP1] += rho1;
      s[LC_PSIP2] += rho2;
      cdot_add(s[LC_PH1], q1[j], h1[j]);
      cdot_add(s[LC_PH2], q2[j], h2[j]);
      s[LC_UPP1] = fma_(U1, a1, s[LC_UPP1]);
      s[LC_UPP2] = fma_(U2, a2, s[LC_UPP2]);
      s[LC_SRHO] = fma_(rho1, fma_(a.g12, rho2, fma_(a.g11, rho1, PR.x)), s[LC_SRHO]);
      s[LC_SRHO] = fma_(rho2, fma_(a.g22, rho2, fma_(a.g21, rho1, PR.y)), s[LC_SRHO]);
    }
    lhy_second<R, NP>(a, nodes, lhy_coef(a), n1, n2, n1p, n2p, Hh);
#pragma unroll
    for (int j = 0; j < NP; ++j)
      s[LC_HLHY] += Hh[j];
  }
  static __device__ double* out(const KArgs<R>& a, Uni&) { return a.st->lc; }
  static __device__ void finish(const KArgs<R>& a, Uni&) {
    if (a.ctrl) {
      a.st->ffts += LIN ? 2 : 4;
      Ctrl<R>::after_lc(a.st);
    }
  }
};
template <class R, int L> struct XInvLC : XInvLCT<R, L, false> {};
template <class R, int L> struct XInvLL : XInvLCT<R, L, true> {};

// Direction of an attempt that carries T psi and T p along: p and T p from their
// terms (T z = w - alpha z, w = P_V^{-1} r or r; in a fallback step z = r and
// w = (alpha + T) r), and the forward rows of the packed source of rho alone.
template <class R_, int L_> struct XFwdLL {
  using R = R_;
  using C = C2<R>;
  static constexpr int MAXT = 64;
  static constexpr const char* NAME = "x-fwd line dir";
  static double alg_bytes(const KArgs<R>& a) { return 17.0 * a.N * sizeof(C); }
  static constexpr int L = L_, NF = 1, NS = LCZ_NS;
  static constexpr bool INV = false, USES_LHY = false, POINTS = false;
  struct Uni : LcUni<R> {
    R shift[2], tpp[2];  // tpp: <p_i, T p_i> over the thread's points of a row
  };
  static __device__ void uniform(const KArgs<R>& a, Uni& u) {
    lc_uniform(a, u);
    load_uniforms<R, 2>({&a.st->shift[0], &a.st->shift[1]}, u.shift);
  }
  template <int NV>
  static __device__ void load(const KArgs<R>& a, Uni& u, int, int row, bool valid, int t, C (&v)[NV][8]) {
    u.tpp[0] = u.tpp[1] = R(0);
    const size_t N = a.N;
    const C* ps = pick(a.psi, u.cur);
    const C* ts = pick(a.tb, u.cur);
    const C* pp = pick(a.pb, u.nsel ^ 1);
    const C* tpp = pick(a.tp, u.nsel ^ 1);
    const C* zs = u.fallback ? pick(a.rb, u.nsel) : a.z;
    const C* ws = a.diag || u.fallback ? a.wz : pick(a.rb, u.nsel);
    C* pd = pick(a.pb, u.nsel);
    C* td = pick(a.tp, u.nsel);
    const bool usepp = u.beta != R(0);
    constexpr int CH = 2;
#pragma unroll
    for (int e0 = 0; e0 < 8; e0 += CH) {
      C p[2][CH], z[2][CH], w[2][CH], k[2][CH], d[2][CH], td1[2][CH];
#pragma unroll
      for (int j = 0; j < CH; ++j)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const size_t q = valid ? (size_t)i * N + (size_t)row * a.nx + Plan<L>::entry_pos(false, t, e0 + j) : 0;
          p[i][j] = ps[q];
          z[i][j] = zs[q];
          w[i][j] = ws[q];
          k[i][j] = ts[q];
          if (usepp) {
            d[i][j] = pp[q];
            td1[i][j] = tpp[q];
          }
        }
#pragma unroll
      for (int j = 0; j < CH; ++j) {
        R rho[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const R c = u.c[i], al = u.shift[i];
          C q = cmk<C>(fma_(-c, p[i][j].x, -z[i][j].x), fma_(-c, p[i][j].y, -z[i][j].y));
          C tq = cmk<C>(fma_(-c, k[i][j].x, fma_(al, z[i][j].x, -w[i][j].x)),
                        fma_(-c, k[i][j].y, fma_(al, z[i][j].y, -w[i][j].y)));
          if (usepp) {
            q = cmk<C>(fma_(u.beta, d[i][j].x, q.x), fma_(u.beta, d[i][j].y, q.y));
            tq = cmk<C>(fma_(u.beta, td1[i][j].x, tq.x), fma_(u.beta, td1[i][j].y, tq.y));
          }
          if (valid) {
            const size_t o = (size_t)i * N + (size_t)row * a.nx + Plan<L>::entry_pos(false, t, e0 + j);
            pd[o] = q;
            td[o] = tq;
            cdot_add(u.tpp[i], q, tq);
          }
          rho[i] = valid ? cdot(p[i][j], q) : R(0);
        }
        v[0][e0 + j] = cmk<C>(fma_(a.d12, rho[1], a.d11 * rho[0]), fma_(a.d22, rho[1], a.d21 * rho[0]));
      }
    }
  }
  template <int NV>
  static __device__ void store(const KArgs<R>& a, Uni& u, int f, int row, bool valid, int t, C (&v)[NV][8], PAcc<R>* acc) {
    store_rows<XFwdLL>(a, a.W, f, row, valid, t, v);
    acc[0].add(u.tpp[0]);
    acc[1].add(u.tpp[1]);
  }
  static __device__ double* out(const KArgs<R>& a, Uni&) { return a.st->lcz; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};

// Trial point of such an attempt: psi' = a psi + b p and T psi' = a T psi + b T p, and
// the forward rows of the packed dipolar source alone.
template <class R_, int L_> struct XFwdEL {
  using R = R_;
  using C = C2<R>;
  static constexpr const char* NAME = "x-fwd energy";
  static double alg_bytes(const KArgs<R>& a) { return 13.0 * a.N * sizeof(C); }
  static constexpr int L = L_, NF = 1, NS = 0;
  static constexpr bool INV = false, USES_LHY = false, POINTS = false;
  using Uni = EgUni<R>;
  static __device__ void uniform(const KArgs<R>& a, Uni& u) { XFwdEG<R, L>::uniform(a, u); }
  template <int NV>
  static __device__ void load(const KArgs<R>& a, Uni& u, int, int row, bool valid, int t, C (&v)[NV][8]) {
    const size_t N = a.N;
    const C* ps = pick(a.psi, u.cur);
    const C* ts = pick(a.tb, u.cur);
    const C* pd = pick(a.pb, u.nsel);
    const C* td = pick(a.tp, u.nsel);
    C* po = pick(a.psi, u.slot);
    C* to = pick(a.tb, u.slot);
    constexpr int CH = ChunkW<R>::v;
#pragma unroll
    for (int e0 = 0; e0 < 8; e0 += CH) {
      C p[2][CH], k[2][CH], q[2][CH], tq[2][CH];
#pragma unroll
      for (int j = 0; j < CH; ++j)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const size_t o = valid ? (size_t)i * N + (size_t)row * a.nx + Plan<L>::entry_pos(false, t, e0 + j) : 0;
          p[i][j] = ps[o];
          k[i][j] = ts[o];
          q[i][j] = pd[o];
          tq[i][j] = td[o];
        }
#pragma unroll
      for (int j = 0; j < CH; ++j) {
        R n[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const C x = XFwdEG<R, L>::trial(u.ca[i], p[i][j], u.cb[i], q[i][j]);
          if (valid) {
            const size_t o = (size_t)i * N + (size_t)row * a.nx + Plan<L>::entry_pos(false, t, e0 + j);
            po[o] = x;
            to[o] = XFwdEG<R, L>::trial(u.ca[i], k[i][j], u.cb[i], tq[i][j]);
          }
          n[i] = valid ? cabs2(x) : R(0);
        }
        v[0][e0 + j] = cmk<C>(fma_(a.d12, n[1], a.d11 * n[0]), fma_(a.d22, n[1], a.d21 * n[0]));
      }
    }
  }
  template <int NV>
  static __device__ void store(const KArgs<R>& a, Uni&, int f, int row, bool valid, int t, C (&v)[NV][8], PAcc<R>*) {
    store_rows<XFwdEL>(a, a.W, f, row, valid, t, v);
  }
  static __device__ double* out(const KArgs<R>&, Uni&) { return nullptr; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};

// ----------------------------------------------------------------------------
// Imaginary-time evolution, the paper's baseline (Sec. I, Sec. VI.B): Strang
// steps psi <- e^{-dtau T/2} e^{-dtau U[psi_half]} e^{-dtau T/2} psi with per-
// component renormalisation.  A kinetic half step is an FFT pair with the
// separable multiplier e^{-dtau |k|^2/4} = ex(kx) ey(ky) ez(kz); the potential
// step is fused into the prologue of the second half step, with U_i = V +
// sum_j g_ij n_j + Phi_i + mu_LHY^(i) read from the aux fields that the
// energy/gradient pipeline wrote for the half-stepped state.
// ----------------------------------------------------------------------------
template <class R_, int L_> struct XFwdKin {
  using R = R_;
  using C = C2<R>;
  static constexpr const char* NAME = "x-fwd ITE half step";
  static double alg_bytes(const KArgs<R>& a) { return (a.flag ? 6.0 : 4.0) * a.N * sizeof(C); }
  static constexpr int L = L_, NF = 2, NS = 0;
  static constexpr bool INV = false, USES_LHY = false, POINTS = false;
  struct Uni {
    int cur;
    R dtau;
  };
  static __device__ void uniform(const KArgs<R>& a, Uni& u) {
    u.cur = __ldcg(&a.st->cur);
    u.dtau = a.kin_tab[a.nx + a.ny + a.nz];
  }
  template <int NV>
  static __device__ void load(const KArgs<R>& a, Uni& u, int f, int row, bool valid, int t, C (&v)[NV][8]) {
    const size_t N = a.N;
    const C* ps = pick(a.psi, u.cur);
    load_rows<XFwdKin>(a, ps, f, row, valid, t, v);
    if (!a.flag || !valid) return;
    const C* ax = pick(a.ax, u.cur);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const size_t idx = (size_t)row * a.nx + Plan<L>::entry_pos(false, t, e);
      const C phi = ax[idx], bb = ax[N + idx];
#pragma unroll
      for (int k = 0; k < NV; ++k)
        v[k][e] = cscale(v[k][e], exp(-u.dtau * (f + k ? phi.y + bb.y : phi.x + bb.x)));
    }
  }
  template <int NV>
  static __device__ void store(const KArgs<R>& a, Uni&, int f, int row, bool valid, int t, C (&v)[NV][8], PAcc<R>*) {
    store_rows<XFwdKin>(a, a.W, f, row, valid, t, v);
  }
  static __device__ double* out(const KArgs<R>&, Uni&) { return nullptr; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};

template <class R_, int L_> struct ZKin {
  using R = R_;
  using C = C2<R>;
  static constexpr const char* NAME = "z fused ITE half step";
  static double alg_bytes(const KArgs<R>& a) { return 4.0 * a.N * sizeof(C); }
  static constexpr int L = L_, NS = 0, AXIS = 2;
  using Uni = NoUni;
  static __device__ void uniform(const KArgs<R>&, Uni&, int) {}
  static constexpr bool FIRST_INV = false;
  static __device__ const C* src(const KArgs<R>& a) { return a.W; }
  template <class SI>
  static __device__ void process(const KArgs<R>& a, Uni&, int, int x, int y, size_t base, size_t ls, int t,
                                 C (&v)[1][8], C* sm, const C* tw, SI si, PAcc<R>*) {
    fft_line<C, L, false, 1>(v, sm, 0, tw, t, si);
    const R exy = a.kin_tab[x] * a.kin_tab[a.nx + y] * a.invN;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int kz = Plan<L>::exit_pos(false, t, e);
      v[0][e] = cscale(v[0][e], exy * a.kin_tab[a.nx + a.ny + kz]);
    }
    col_after<L>(sm, si);
    fft_line<C, L, true, 1>(v, sm, 0, tw, t, si);
#pragma unroll
    for (int e = 0; e < 8; ++e) a.W[base + (size_t)Plan<L>::exit_pos(true, t, e) * ls] = v[0][e];
  }
  static __device__ double* out(const KArgs<R>&, Uni&) { return nullptr; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};

template <class R_, int L_> struct XInvKin {
  using R = R_;
  using C = C2<R>;
  static constexpr const char* NAME = "x-inv ITE half step";
  static double alg_bytes(const KArgs<R>& a) { return 4.0 * a.N * sizeof(C); }
  static constexpr int L = L_, NF = 2, NS = 2;
  static constexpr bool INV = true, USES_LHY = false, POINTS = false;
  struct Uni {
    int cur;
  };
  static __device__ void uniform(const KArgs<R>& a, Uni& u) { u.cur = __ldcg(&a.st->cur); }
  template <int NV>
  static __device__ void load(const KArgs<R>& a, Uni&, int f, int row, bool valid, int t, C (&v)[NV][8]) {
    load_rows<XInvKin>(a, a.W, f, row, valid, t, v);
  }
  template <int NV>
  static __device__ void store(const KArgs<R>& a, Uni& u, int f, int row, bool valid, int t, C (&v)[NV][8], PAcc<R>* acc) {
    if (!valid) return;
    store_rows<XInvKin>(a, pick(a.psi, u.cur), f, row, valid, t, v);
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      R s = 0;
#pragma unroll
      for (int e = 0; e < 8; ++e) cdot_add(s, v[k][e], v[k][e]);
      if (f + k == 0) acc[0].add(s);
      else acc[1].add(s);
    }
  }
  static __device__ double* out(const KArgs<R>& a, Uni&) { return a.st->rt; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};

// psi_i <- psi_i / ||psi_i|| with the norms the last half step reduced.
template <class R> __device__ __forceinline__ void ite_scale_body(const KArgs<R>& a) {
  if (!gate_open(a)) return;
  const int cur = __ldcg(&a.st->cur);
  const double dV = __ldcg(&a.st->dV);
  R s1, s2;
  if constexpr (sizeof(R) == sizeof(double)) {
    s1 = 1.0 / sqrt(__ldcg(&a.st->rt[0]) * dV);
    s2 = 1.0 / sqrt(__ldcg(&a.st->rt[1]) * dV);
  } else {  // FP32 fields: lane i forms ||psi_i||^2 in FP64, one conversion per warp
    const float q = (float)(__ldcg(&a.st->rt[threadIdx.x & 1]) * dV);
    const float sc = rsqrtf(q);
    s1 = __shfl_sync(0xffffffffu, sc, 0);
    s2 = __shfl_sync(0xffffffffu, sc, 1);
  }
  C2<R>* ps = pick(a.psi, cur);
  const size_t N = a.N;
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += (size_t)gridDim.x * blockDim.x) {
    ps[idx] = cscale(ps[idx], s1);
    ps[N + idx] = cscale(ps[N + idx], s2);
  }
}
template <class R> __global__ void __launch_bounds__(256) ite_scale_kernel(KArgs<R> a) { ite_scale_body(a); }
template <class R> __global__ void __launch_bounds__(256) ite_scale_kernel_b(const __grid_constant__ KBatch<R> kb) {
  ite_scale_body(kb.k[blockIdx.y]);
}


// ----------------------------------------------------------------------------
// Parameter derivatives at fixed psi (the adjoint pass of the energy with
// respect to its couplings, Eq. 1): x fwd of zeta = n1 + i n2 -> y -> z with the
// dipolar kernel K(k) -> y inv -> x inv: K*n1 = Re, K*n2 = Im (the kernel is real
// and even), then the contact, dipolar, trap and LHY (through eta) sums.
// ----------------------------------------------------------------------------
template <class R_, int L_> struct XFwdPG {
  using R = R_;
  using C = C2<R>;
  static constexpr const char* NAME = "x-fwd densities (param grad)";
  static double alg_bytes(const KArgs<R>& a) { return 3.0 * a.N * sizeof(C); }
  static constexpr int L = L_, NF = 1, NS = 0;
  static constexpr bool INV = false, USES_LHY = false, POINTS = false;
  struct Uni {
    int cur;
  };
  static __device__ void uniform(const KArgs<R>& a, Uni& u) { u.cur = __ldcg(&a.st->cur); }
  template <int NV>
  static __device__ void load(const KArgs<R>& a, Uni& u, int, int row, bool valid, int t, C (&v)[NV][8]) {
    const C* ps = a.gin ? a.gin : pick(a.psi, u.cur);
    C* dst = pick(a.psi, u.cur);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const size_t idx = valid ? (size_t)row * a.nx + Plan<L>::entry_pos(false, t, e) : 0;
      const C p1 = ps[idx], p2 = ps[(size_t)a.N + idx];
      v[0][e] = valid ? cmk<C>(cabs2(p1), cabs2(p2)) : cmk<C>(0, 0);
      if (a.gin && valid) {
        dst[idx] = p1;
        dst[(size_t)a.N + idx] = p2;
      }
    }
  }
  template <int NV>
  static __device__ void store(const KArgs<R>& a, Uni&, int f, int row, bool valid, int t, C (&v)[NV][8], PAcc<R>*) {
    store_rows<XFwdPG>(a, a.W, f, row, valid, t, v);
  }
  static __device__ double* out(const KArgs<R>&, Uni&) { return nullptr; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};

template <class R_, int L_> struct ZPg {
  using R = R_;
  using C = C2<R>;
  static constexpr const char* NAME = "z dipolar kernel (param grad)";
  static double alg_bytes(const KArgs<R>& a) { return 2.0 * a.N * sizeof(C); }
  static constexpr int L = L_, NS = 0, AXIS = 2;
  using Uni = KzLine<R, L_>;
  static __device__ void uniform(const KArgs<R>& a, Uni& u, int t) { u.set(a, t); }
  static constexpr bool FIRST_INV = false;
  static __device__ const C* src(const KArgs<R>& a) { return a.W; }
  template <class SI>
  static __device__ void process(const KArgs<R>& a, Uni& u, int, int x, int y, size_t base, size_t ls, int t,
                                 C (&v)[1][8], C* sm, const C* tw, SI si, PAcc<R>*) {
    fft_line<C, L, false, 1>(v, sm, 0, tw, t, si);
    const R kxy = kq_xy(a, x, y);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const R kz = u.kz[e];
      v[0][e] = cscale(v[0][e], dip_mult(a, kz, kxy + kz));
    }
    col_after<L>(sm, si);
    fft_line<C, L, true, 1>(v, sm, 0, tw, t, si);
#pragma unroll
    for (int e = 0; e < 8; ++e) a.W[base + (size_t)Plan<L>::exit_pos(true, t, e) * ls] = v[0][e];
  }
  static __device__ double* out(const KArgs<R>&, Uni&) { return nullptr; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};

template <class R_, int L_> struct XInvPG {
  using R = R_;
  using C = C2<R>;
  static constexpr int PTS = 2, MAXT = 128;
  static constexpr const char* NAME = "x-inv parameter sums";
  static double alg_bytes(const KArgs<R>& a) { return 3.0 * a.N * sizeof(C); }
  static constexpr int L = L_, NF = 1, NS = PG_NS;
  static constexpr bool INV = true, USES_LHY = true, POINTS = true;
  struct Uni {
    int cur;
  };
  static __device__ void uniform(const KArgs<R>& a, Uni& u) { u.cur = __ldcg(&a.st->cur); }
  template <int NV>
  static __device__ void load(const KArgs<R>& a, Uni&, int f, int row, bool valid, int t, C (&v)[NV][8]) {
    load_rows<XInvPG>(a, a.W, f, row, valid, t, v);
  }
  template <int NP, bool ST>
  static __device__ void points(const KArgs<R>& a, Uni& u, const RowPt<R, NF, ST> (&pt)[NP], R (&s)[PG_NS],
                                const LhyNode<R>* nodes) {
    const C* ps = pick(a.psi, u.cur);
    const LhyCoef<R> cf = lhy_coef(a);
    R n1[NP], n2[NP], lh[NP][6];
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      n1[j] = cabs2(ps[pt[j].idx]);
      n2[j] = cabs2(ps[(size_t)a.N + pt[j].idx]);
    }
    lhy_eta_sums<R, NP>(nodes, a.Q, a.Qm, cf, n1, n2, lh);
#pragma unroll
    for (int j = 0; j < NP; ++j) {
      const int row = (int)(pt[j].idx / L), y = row % a.ny, z = row / a.ny;
      const R X = fma_((R)pt[j].x, a.hx, -a.Lx), Y = fma_((R)y, a.hy, -a.Ly), Z = fma_((R)z, a.hz, -a.Lz);
      const C K = pt[j].out(0);
      const R nt = n1[j] + n2[j];
      s[PG_N11] = fma_(n1[j], n1[j], s[PG_N11]);
      s[PG_N12] = fma_(n1[j], n2[j], s[PG_N12]);
      s[PG_N22] = fma_(n2[j], n2[j], s[PG_N22]);
      s[PG_K11] = fma_(n1[j], K.x, s[PG_K11]);
      s[PG_K12] = fma_(n1[j], K.y, s[PG_K12]);
      s[PG_K22] = fma_(n2[j], K.y, s[PG_K22]);
      s[PG_X2] = fma_(X * X, nt, s[PG_X2]);
      s[PG_Y2] = fma_(Y * Y, nt, s[PG_Y2]);
      s[PG_Z2] = fma_(Z * Z, nt, s[PG_Z2]);
#pragma unroll
      for (int k = 0; k < 6; ++k) s[PG_L11 + k] += lh[j][k];
    }
  }
  static __device__ double* out(const KArgs<R>& a, Uni&) { return a.st->pg; }
  static __device__ void finish(const KArgs<R>&, Uni&) {}
};

// ----------------------------------------------------------------------------
// Small pointwise kernels: retraction sums and apply, residual norm, casts.
// ----------------------------------------------------------------------------
// sums over (psi = gin, p = gout-as-input) for the standalone retraction
template <class R> __global__ void __launch_bounds__(256) rt_sums_kernel(KArgs<R> a, const C2<R>* psi, const C2<R>* p) {
  __shared__ RedSmem<RT_NS> red;
  PAcc<R> acc[RT_NS];
  const size_t N = a.N;
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += (size_t)gridDim.x * blockDim.x) {
    for (int i = 0; i < 2; ++i) {
      const C2<R> u = psi[i * N + idx], q = p[i * N + idx];
      acc[RT_P1 + i].add(cabs2(q));
      acc[RT_PSIP1 + i].add(cdot(u, q));
      acc[RT_PSI1 + i].add(cabs2(u));
    }
  }
  reduce_blocks<RT_NS>(acc, a.partials, a.counter, a.st->rt, red);
}

template <class R>
__global__ void __launch_bounds__(256) rt_apply_kernel(size_t N, const C2<R>* psi, const C2<R>* p, C2<R>* out, R a1,
                                                        R b1, R a2, R b2) {
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += (size_t)gridDim.x * blockDim.x) {
    const C2<R> u1 = psi[idx], q1 = p[idx], u2 = psi[N + idx], q2 = p[N + idx];
    out[idx] = cmk<C2<R>>(a1 * u1.x + b1 * q1.x, a1 * u1.y + b1 * q1.y);
    out[N + idx] = cmk<C2<R>>(a2 * u2.x + b2 * q2.x, a2 * u2.y + b2 * q2.y);
  }
}

// ||r_i||^2 of the current point (final report of a solve).
template <class R> __global__ void __launch_bounds__(256) resnorm_kernel(KArgs<R> a) {
  __shared__ RedSmem<2> red;
  PAcc<R> acc[2];
  const int cur = __ldcg(&a.st->cur);
  R mu[2];
  load_uniforms<R, 2>({&a.st->mu[0], &a.st->mu[1]}, mu);
  const size_t N = a.N;
  const C2<R>* ps = pick(a.psi, cur);
  const C2<R>* hp = pick(a.hp, cur);
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < N; idx += (size_t)gridDim.x * blockDim.x) {
    for (int i = 0; i < 2; ++i) {
      const C2<R> u = ps[i * N + idx], h = hp[i * N + idx];
      const C2<R> r = cmk<C2<R>>(h.x - mu[i] * u.x, h.y - mu[i] * u.y);
      acc[i].add(cabs2(r));
    }
  }
  reduce_blocks<2>(acc, a.partials, a.counter, a.st->pca, red);
}

template <class A, class B> __global__ void cast_kernel(size_t n, const A* in, B* out) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const A v = in[i];
    B w;
    w.x = (decltype(w.x))v.x;
    w.y = (decltype(w.y))v.y;
    out[i] = w;
  }
}

}  // namespace egpe
