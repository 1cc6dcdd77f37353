// Sweeps: four time steps of a large lattice in one pass over memory.
//
// A lattice beyond the L2 cache streams its populations from DRAM and back
// at every time step.  Here a block carries a tile of kCols columns down the
// rows of the lattice and keeps, for each of the kSteps steps, the last four
// rows of that step in shared memory: a row of step s is computed as soon as
// the three rows of step s - 1 it pulls from exist, two rows behind them.
// Populations are read once (rows of the state before the sweep, bulk copies
// five rows ahead of their use) and written once (rows of the last step), so
// DRAM traffic per step falls to a quarter plus the halo columns.
//
// Two population buffers: a sweep reads one and writes the other, in the
// canonical layout (F[i][cell] = post-collision g_i), because the tiles
// beside it still read what it would overwrite; solid cells are never
// written.  Two sweeps bring the state back.  The per-cell update is that of
// the other step kernels (d2q9_cell.cuh), every step's values rounded to the
// storage type, so every cell gets the same bits.
//
// Tile.  Columns xs .. xs + 127, of which the first and last four are halo:
// values at the tile's edge miss a neighbour, and the garbage moves one column
// inwards per step, so after four steps all but those are right.  A step-row
// of the tile is two windows of 64 cells, one warp each, lane l cells l and
// l + 32, collided as one in packed FP32 (bgk2): eight warps update four
// step-rows at once, a barrier after each; a ninth issues the copies and waits
// for them.  A window whose cells and all their neighbours are fluid loads and
// stores with compile-time offsets; others select bounce-back per direction
// and apply the port rules.
//
// Work.  The rows of a tile that hold fluid form one list over all tiles; each
// block takes a share of it of about equal cost (a turn on a row with walls or
// a port takes longer), cut into runs of consecutive rows of one tile.  A run
// of n rows costs n + 9 turns (three more rows of the first step on either
// side, and the pipeline of four steps two rows apart).
//
// What bounds it: a turn takes about 1,550 cycles, of which the FMA pipe is
// busy for 560 (18 % of instructions counted once; a packed one holds it for
// two cycles) and issue for 700 (two blocks a SM, so that one computes while
// the other waits at its barrier); DRAM is idle half the time.  8192 x 4096
// cells, 16.8 M of them fluid, FP32: 112 us a step, per-phase kernel 193.  Three
// blocks a SM (80 registers) gave no more; a row copied as nine bulk copies by
// nine lanes took 1,740 cycles to issue, the tensor copy one instruction.
#include <cuda.h>  // CUtensorMap (types only: the encoder is looked up at run time)

#include "d2q9_cell.cuh"

namespace lbm {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kSteps = kSweepSteps;
constexpr int kCols = 128;
constexpr int kWindows = kCols / 64;
constexpr int kWarps = kSteps * kWindows;  // and one that issues the copies
constexpr int kRing0 = 8, kRing = 4;       // rows kept of the input and of each step but the last
constexpr int kRow = 9 * kCols;            // values of a row
constexpr int kPad = 32;                   // words before the first ring (a window's lane 0 reads one to the left)
constexpr unsigned kSpinLimit = 1u << 22;
// relative time of a turn on a row: all windows open, one with a wall, one with a port
constexpr int kCostOpen = 8, kCostClosed = 12, kCostPort = kSweepMaxCost;

constexpr int kHalo = kSteps, kOut = kCols - 2 * kHalo;
constexpr int kSmem = 4 * (kPad + kRing0 * kRow + (kSteps - 1) * kRing * kRow + kPad);
static_assert(kHalo % 4 == 0, "the copies start on 16-byte boundaries");

__device__ __forceinline__ unsigned shared_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void bar_init(unsigned bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");  // seen by the copies
}
__device__ __forceinline__ void bar_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool bar_wait(unsigned bar, unsigned phase) {
  for (unsigned spins = 0; spins < kSpinLimit; ++spins) {
    unsigned done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(phase)
        : "memory");
    if (done) return true;
  }
  return false;
}
// One row of the tile, all nine planes (a box of kCols x 1 x 9): one
// instruction; columns and rows outside the lattice arrive as zeros.
__device__ __forceinline__ void copy_row(unsigned dst, const CUtensorMap* map, int x, int y, unsigned bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
      "[%5];" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(0), "r"(bar)
      : "memory");
}

// What the windows of a tile row hold: bit w of `open` set when the cells of
// window w and all their neighbours are fluid, of `some` when it holds a
// fluid cell.
struct RowState {
  uint8_t open, some;
};

// Solid bits of row y around half a window: for each lane the cell to the west
// (bit 0), its own (1) and the one to the east (2).  `first`: the cell west
// of the half.  Words past the row's padding read as wall.
__device__ __forceinline__ unsigned row_bits(const LatticeView& L, int y, int first, int lane) {
  const uint32_t* row = L.mask + (long long)y * mask_stride(L.wpr);
  const int w0 = first >> 5, s = first & 31;  // w0 >= -1: the padding word
  uint32_t w[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) w[k] = w0 + k <= L.wpr ? row[w0 + k] : 0xffffffffu;
  const uint32_t m0 = __funnelshift_r(w[0], w[1], s), m1 = __funnelshift_r(w[1], w[2], s);
  return __funnelshift_r(m0, m1, lane) & 7u;
}

// solid flag of the cell direction i comes from (rm, r0, rp: bits of rows
// y - 1, y, y + 1)
__device__ __forceinline__ bool source_solid(int i, unsigned rm, unsigned r0, unsigned rp) {
  const unsigned row = cy_of(i) > 0 ? rm : cy_of(i) < 0 ? rp : r0;
  return (row >> (1 - cx_of(i))) & 1u;
}

// The nine incoming populations of one of the lane's cells of a window that
// is not open, with the port rules; false: a solid cell.
__device__ __forceinline__ bool closed_cell(const LatticeView& L, const float* in, int im, int i0, int ip, int x, int y,
                                            int lane, float (&g)[9]) {
  const int first = x - lane - 1;
  const unsigned rm = row_bits(L, y - 1, first, lane), r0 = row_bits(L, y, first, lane),
                 rp = row_bits(L, y + 1, first, lane);
  const bool fluid = !(r0 & 2u);
  g[0] = in[i0];
#pragma unroll
  for (int i = 1; i < 9; ++i) {
    const int at = (cy_of(i) > 0 ? im : cy_of(i) < 0 ? ip : i0) + i * kCols - cx_of(i);
    g[i] = in[source_solid(i, rm, r0, rp) ? i0 + opp_of(i) * kCols : at];
  }
  // the columns beyond the ports read as wall, so port cells are never in open windows
  if (x == 0 && fluid)
    inlet_rule(g, L.u_in[y], L.rho0, L.port_scheme);
  else if (x == L.nx - 1 && fluid)
    outlet_rule(g, L.rho0, L.port_scheme);
  return fluid;
}

// One step-row of a warp's window.  in: the ring of the step before (one
// word a value), im / i0 / ip: this lane's first cell in its rows y - 1, y, y + 1 (the
// second is 32 further).  out: the ring row to write (last step: nullptr, and
// the row goes to G).
__device__ __forceinline__ void window_step(const LatticeView& L, const float* in, int im, int i0, int ip, float* out,
                                            float* G, int x, int y, int x_lo, int x_hi, bool open, int lane, F2 rho0,
                                            F2 omega) {
  F2 g[9];
  bool fa = true, fb = true;
  if (open) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const float* at = in + ((cy_of(i) > 0 ? im : cy_of(i) < 0 ? ip : i0) + i * kCols - cx_of(i));
      g[i] = f2(at[0], at[32]);
    }
  } else {
    float a[9], b[9];
    fa = closed_cell(L, in, im, i0, ip, x, y, lane, a);
    fb = closed_cell(L, in, im + 32, i0 + 32, ip + 32, x + 32, y, lane, b);
#pragma unroll
    for (int i = 0; i < 9; ++i) g[i] = f2(a[i], b[i]);
  }
  F2 drho, ux, uy;
  bgk2(g, rho0, omega, drho, ux, uy);
  if (out) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      float a, b;
      f2_split(g[i], a, b);
      out[i * kCols] = a;
      out[i * kCols + 32] = b;
    }
  } else {
    const long long c = (long long)y * L.pitch + x;
    float* f = G + c;
    const bool wa = fa && x >= x_lo && x < x_hi && LBM_OK_IDX(c, L.plane),
               wb = fb && x + 32 >= x_lo && x + 32 < x_hi && LBM_OK_IDX(c + 32, L.plane);
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      float a, b;
      f2_split(g[i], a, b);
      if (wa) f[0] = a;
      if (wb) f[32] = b;
      f += L.plane;
    }
  }
}

// Entry k of the row list, tile << kSweepRowBits | y; rows of a tile ascend.
// The run that starts at entry i and ends before entry `end`: its rows are
// consecutive exactly while list[j] - list[i] == j - i.
__device__ __forceinline__ int run_length(const int* __restrict__ list, int i, int end, int lane) {
  const int e = list[i];
  int lo = 1, hi = end - i;  // the first lo entries are consecutive; at most hi
  while (lo < hi) {
    const int step = (hi - lo + 31) / 32;
    const int j = min(lo + (lane + 1) * step, hi);  // is entry i + j - 1 still part of the run?
    const unsigned in = __ballot_sync(kFull, list[i + j - 1] - e == j - 1);
    const int n = __popc(in);  // a prefix of the lanes
    const int new_lo = n ? min(lo + n * step, hi) : lo;
    const int new_hi = n < 32 ? min(lo + (n + 1) * step, hi) - 1 : hi;
    lo = new_lo;
    hi = max(new_hi, lo);
  }
  return lo;
}

// First entry of block b's share of the list: the number of entries whose
// costs sum to at most b / G of the whole (cost: exclusive prefix sums, the
// total at [total]).  Every warp calls.
__device__ __forceinline__ int share_begin(const int* __restrict__ cost, int total, int b, int G, int lane) {
  const long long want = (long long)cost[total] * b / G;
  int lo = 0, hi = total;  // the first lo entries lie before the share; at most hi
  while (lo < hi) {
    const int step = (hi - lo + 31) / 32;
    const int j = min(lo + (lane + 1) * step, hi);
    const int n = __popc(__ballot_sync(kFull, cost[j] <= want));
    const int new_hi = n < 32 ? min(lo + (n + 1) * step, hi) - 1 : hi;
    lo = n ? min(lo + n * step, hi) : lo;
    hi = max(new_hi, lo);
  }
  return lo;
}

// One run of a tile's rows, as a warp sees it.
struct Run {
  int x_lo, x_hi;    // output columns
  int k_lo, k_hi;    // turns, both included
  int lo, hi, lag;   // this warp's step: rows lo .. hi - 1, row k - lag in turn k
  int in_slot;       // input ring slot of row lo - 1
  const RowState* st;  // of row lo
};

// The turns of a warp of the first step (FIRST: it reads the input ring), of
// the last (it writes to G) or of one between.  x: the column of the lane's
// first cell, col: its word in a ring row, in / out: the rings read and written.
template <bool FIRST, bool LAST>
__device__ __forceinline__ void run_step(const LatticeView& L, const Run& r, const float* in, float* out, float* G,
                                         int x, int col, int window, int lane, F2 rho0, F2 omega) {
  constexpr int kIn = FIRST ? kRing0 : kRing;
  int k = r.k_lo;
  for (; k < r.lo + r.lag; ++k) __syncthreads();
  const RowState* st = r.st;
  RowState cur = *st;
  // this lane's cell in rows y - 1, y and y + 1 of the step before, and in row y of this one
  const int s0 = FIRST ? r.in_slot : (r.lo - 1) & (kRing - 1);
  int im = s0 * kRow + col, i0 = (s0 + 1) % kIn * kRow + col, ip = (s0 + 2) % kIn * kRow + col;
  int io = (r.lo & (kRing - 1)) * kRow + col;
  for (int y = r.lo; y < r.hi; ++y, ++k) {
    const RowState now = cur;
    cur = *++st;  // for the next turn
    if ((now.some >> window) & 1u)
      window_step(L, in, im, i0, ip, LAST ? nullptr : out + io, G, x, y, r.x_lo, r.x_hi, (now.open >> window) & 1u,
                  lane, rho0, omega);
    im = i0;
    i0 = ip;
    ip = ip == (kIn - 1) * kRow + col ? col : ip + kRow;
    io = io == (kRing - 1) * kRow + col ? col : io + kRow;
    __syncthreads();
  }
  for (; k <= r.k_hi; ++k) __syncthreads();
}

// One sweep: kSteps time steps of the lattice L (its populations read through
// the map `from`, the result written to G).  list: the rows of all tiles
// holding fluid, n_rows their number, cost: see share_begin, states: of every
// row of every tile.  give_up: a block's wait for its input row of that number
// or a later one counts as run out (the test hook; else larger than any).
__global__ void __launch_bounds__((kWarps + 1) * 32, kSweepBlocks)
    k_sweep(const __grid_constant__ LatticeView L, const __grid_constant__ CUtensorMap from, float* __restrict__ G,
            const int* __restrict__ list, const int* __restrict__ cost, const int* __restrict__ n_rows,
            const RowState* __restrict__ states, int* __restrict__ error, unsigned give_up) {
  extern __shared__ __align__(128) unsigned char sweep_smem[];
  __shared__ __align__(8) unsigned long long s_full[kRing0];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  float* ring0 = reinterpret_cast<float*>(sweep_smem) + kPad;
  float* rings = ring0 + kRing0 * kRow;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int level = warp / kWindows + 1;  // the step this warp computes, 1 .. kSteps; one more: it issues the copies
  const int window = warp % kWindows, col = window * 64 + lane;
  const F2 rho0 = f2_c(L.rho0), omega = f2_c(L.omega);
  if (threadIdx.x < kRing0) bar_init(shared_addr(&s_full[threadIdx.x]));
  __syncthreads();
  asm volatile("griddepcontrol.wait;" ::: "memory");  // populations of the previous step are final from here on
  const int total = *n_rows;
  const int begin = share_begin(cost, total, blockIdx.x, gridDim.x, lane);
  const int end = share_begin(cost, total, blockIdx.x + 1, gridDim.x, lane);
  const int ny = L.ny;
  unsigned seq = 0;  // rows copied into the input ring before this run
  for (int at = begin; at < end;) {
    const int e = list[at], n = run_length(list, at, end, lane);
    at += n;
    const int y_lo = e & ((1 << kSweepRowBits) - 1), y_hi = y_lo + n;
    const int r_lo = max(0, y_lo - kSteps), r_hi = min(ny - 1, y_hi + kSteps - 1);  // input rows, both included
    Run r;
    r.x_lo = (e >> kSweepRowBits) * kOut;
    r.x_hi = min(r.x_lo + kOut, L.nx);
    r.k_lo = max(1, y_lo - (kSteps - 1));
    r.k_hi = y_hi - 1 + 2 * (kSteps - 1);
    const int xs = r.x_lo - kHalo;  // the tile's first column
    int failed = 0;
    if (level > kSteps) {  // the warp that issues the copies and waits for them
      int copied = r_lo, arrived = r_lo;  // next input rows to copy and to wait for
      int last = r_hi;                    // (after a failure none)
      auto wait_row = [&](int y) {
        const unsigned i = seq + (unsigned)(y - r_lo);
        return bar_wait(shared_addr(&s_full[i % kRing0]), (i / kRing0) & 1u) && i < give_up;
      };
      for (int k = r.k_lo - 1; k <= r.k_hi; ++k) {
        // row i takes the place of row i - 8, last read in turn i - 7
        for (; copied <= min(k + kRing0 - 2, last); ++copied) {
          const unsigned slot = (seq + (unsigned)(copied - r_lo)) % kRing0;
          const unsigned bar = shared_addr(&s_full[slot]);
          if (lane == 0) {
            bar_expect(bar, (unsigned)(kRow * sizeof(float)));
            copy_row(shared_addr(ring0 + slot * kRow), &from, xs, copied, bar);
          }
        }
        // what the next turn reads has arrived before this one ends
        for (; arrived <= min(k + 2, last); ++arrived)
          if (!wait_row(arrived)) {
            failed = 1;
            last = -1;
          }
        __syncthreads();
      }
      if (failed)  // no copy is issued after the one that failed; those in flight land (or give up) before the block leaves
        for (int y = arrived - 1; y < copied; ++y) (void)wait_row(y);
    } else {
      r.lag = 2 * (level - 1);
      r.lo = max(1, y_lo - (kSteps - level));
      r.hi = max(r.lo, min(ny - 1, y_hi + (kSteps - level)));
      r.in_slot = (int)((seq + (unsigned)(r.lo - 1 - r_lo)) % kRing0);
      r.st = states + (long long)(e >> kSweepRowBits) * ny + r.lo;
      __syncthreads();  // the first rows have arrived
      float* out = rings + (level - 1) * kRing * kRow;
      const float* in = out - kRing * kRow;
      if (level == 1)
        run_step<true, false>(L, r, ring0, out, G, xs + col, col, window, lane, rho0, omega);
      else if (level < kSteps)
        run_step<false, false>(L, r, in, out, G, xs + col, col, window, lane, rho0, omega);
      else
        run_step<false, true>(L, r, in, nullptr, G, xs + col, col, window, lane, rho0, omega);
    }
    seq += (unsigned)(r_hi - r_lo + 1);
    if (__syncthreads_or(failed)) {  // the sweep is void
      if (threadIdx.x == 0) atomicExch(error, 1);
      return;
    }
  }
}

// Tile row i = t ny + y (tile t: output columns t kOut .. t kOut + kOut - 1):
// flags[i] = 1 when its output columns hold a fluid cell, work[i] its cost
// then, and the state of its windows.  One warp per tile row.
__global__ void k_sweep_flags(const __grid_constant__ LatticeView L, int total, int* __restrict__ flags, int* __restrict__ work, RowState* __restrict__ states) {
  const int lane = threadIdx.x & 31;
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (i >= total) return;
  const int t = i / L.ny, y = i - t * L.ny;
  const int x_lo = t * kOut, x_hi = min(x_lo + kOut, L.nx);
  unsigned open = 0, some = 0;
  bool fluid = false, port = false;
  if (y >= 1 && y <= L.ny - 2)
    for (int h = 0; h < 2 * kWindows; ++h) {
      const int x0 = x_lo - kHalo + 32 * h;
      const unsigned r0 = row_bits(L, y, x0 - 1, lane);
      const unsigned near = r0 | row_bits(L, y - 1, x0 - 1, lane) | row_bits(L, y + 1, x0 - 1, lane);
      const bool own = !(r0 & 2u);
      if (!__any_sync(kFull, near != 0u)) open |= 1u << h;
      if (__any_sync(kFull, own)) some |= 1u << (h >> 1);
      fluid |= own && x0 + lane >= x_lo && x0 + lane < x_hi;
      port |= own && (x0 + lane == 0 || x0 + lane == L.nx - 1);
    }
  unsigned both = 0;
  for (int w = 0; w < kWindows; ++w) both |= (((open >> (2 * w)) & 3u) == 3u ? 1u : 0u) << w;
  fluid = __any_sync(kFull, fluid);
  port = __any_sync(kFull, port);
  if (lane == 0) {
    flags[i] = fluid ? 1 : 0;
    work[i] = !fluid ? 0 : port ? kCostPort : some & ~both ? kCostClosed : kCostOpen;
    states[i] = RowState{(uint8_t)both, (uint8_t)some};
  }
}

// list[k] and cost[k] of the k-th row; the total cost after the last.
__global__ void k_sweep_scatter(int ny, int total, const int* __restrict__ flags, const int* __restrict__ offs,
                                const int* __restrict__ work_before, int* __restrict__ list, int* __restrict__ cost) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) cost[offs[total]] = work_before[total];
  if (i >= total || !flags[i]) return;
  const int t = i / ny, y = i - t * ny;
  list[offs[i]] = t << kSweepRowBits | y;
  cost[offs[i]] = work_before[i];
}

// The tensor map of a population buffer: planes x rows x columns, read in
// boxes of one row of a tile over all planes.
bool population_map(CUtensorMap* map, const LatticeView& L, const void* F) {
  using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static const Encode encode = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult r{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &r) != cudaSuccess ||
        r != cudaDriverEntryPointSuccess)
      p = nullptr;
    return reinterpret_cast<Encode>(p);
  }();
  if (!encode) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)L.pitch, (cuuint64_t)L.ny, 9};
  const cuuint64_t strides[2] = {(cuuint64_t)L.pitch * sizeof(float), (cuuint64_t)L.plane * sizeof(float)};
  const cuuint32_t box[3] = {kCols, 1, 9}, unit[3] = {1, 1, 1};
  return encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(F), dims, strides, box, unit, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

long long sweep_rows(int nx, int ny) { return (nx + kOut - 1LL) / kOut * ny; }

SweepList sweep_list(int nx, int ny, void* buffer) {
  const size_t n = (size_t)sweep_rows(nx, ny), tmp = scan_tmp_ints((long long)n);
  int* p = static_cast<int*>(buffer);
  SweepList s;
  auto take = [&p](size_t ints) {
    int* q = p;
    p += ints;
    return q;
  };
  s.flags = take(n);
  s.offs = take(n + 1);
  s.work = take(n);
  s.work_before = take(n + 1);
  s.list = take(n);
  s.cost = take(n + 1);
  s.states = take(n);
  s.tmp = take(tmp);
  s.n_rows = s.offs + n;
  s.total_cost = s.work_before + n;
  s.ints = (size_t)(p - static_cast<int*>(buffer));
  return s;
}

cudaError_t launch_build_sweep(const LatticeView& L, const SweepList& s, cudaStream_t stream) {
  const int total = (int)sweep_rows(L.nx, L.ny);
  k_sweep_flags<<<(total + 7) / 8, 256, 0, stream>>>(L, total, s.flags, s.work,
                                                     static_cast<RowState*>(s.states));
  count_launches(1);
  cudaError_t e = launch_scan(s.flags, s.offs, total, s.tmp, stream);
  if (e == cudaSuccess) e = launch_scan(s.work, s.work_before, total, s.tmp, stream);
  if (e != cudaSuccess) return e;
  k_sweep_scatter<<<(total + 255) / 256, 256, 0, stream>>>(L.ny, total, s.flags, s.offs, s.work_before, s.list,
                                                           s.cost);
  count_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_sweep(const LatticeView& L, const void* F, void* G, const SweepList& sl, int grid, int* error,
                         cudaStream_t stream) {
  if (grid < 1) return cudaErrorInvalidValue;
  void* k = (void*)k_sweep;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
  if (e != cudaSuccess) return e;
  CUtensorMap from;
  if (!population_map(&from, L, F)) return cudaErrorInvalidValue;
  float* g = static_cast<float*>(G);
  unsigned give_up = barrier_timeout_test() ? kRing0 : 0xffffffffu;  // (the first row of a barrier's second phase)
  void* args[] = {(void*)&L, (void*)&from, (void*)&g, (void*)&sl.list, (void*)&sl.cost,
                  (void*)&sl.n_rows, (void*)&sl.states, (void*)&error, (void*)&give_up};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3((kWarps + 1) * 32);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelExC(&cfg, k, args);
  if (e == cudaSuccess) count_launches(1);
  return e;
}

}  // namespace lbm
