// On-chip resident time steps: a whole solve in one launch, the populations
// held in shared memory from its first step to its last.
//
// Method: the same per-cell update as the step kernels (Eq. 1 with the
// equilibrium of Sec. 2.1, the moments of Eq. 2, halfway bounce-back, the
// port rules and the symmetry plane of Sec. 3.3; d2q9_cell.cuh), so every
// cell gets the same bits.
//
// Layout.  A lattice set whose row segments fit in the shared memory of the
// SMs (the 2048 x 1024 distributor: 6976 segments, 5.75 MB of FP32
// populations, against 152 x 227 KB) is split into contiguous ranges of its
// segment list, one range per block (at most kResidentMaxOwn segments, one
// block per SM, all blocks resident: a cooperative launch; longer lists, up to
// kResidentManyOwn a block, in a kernel of their own below).  A block keeps
// its segments' nine population rows as FP32 in two step buffers in shared
// memory (read one, write the other, a plain pull scheme; 16-bit storage
// rounds every value to its type before it is stored, so the values are
// those of 16-bit buffers without their conversions on every load).
//
// Thread mapping.  A warp owns one segment, lane l its cell l; lists of more
// than 32 segments per SM (the register budget of 1024 threads) take two per
// warp, collided as one in the packed FP32 instructions (bgk2).  One is the
// better mapping where it fits: a step is a chain of dependent stages (words
// arrive, pull, ports, collision, publish), and with two segments each stage
// is twice as long (20 segments a block, 1024 x 512 tree: 1.26 us per step
// against 1.56).  Each lane knows, for its cell and eight directions, the
// shared-memory word its incoming value comes from, computed once per launch:
// an own row, another slot's row, a ghost word, its own opposite slot
// (bounce-back), or a word that stays zero (the unknown populations of port
// cells; every direction of a solid cell).  No step branches on the geometry.
//
// Exchange.  After each step a warp publishes, for each of its segments
// that another block reads, 16-byte words {value, value, value, step tag}:
// what streams up (directions 2, 5, 6), what streams down (4, 7, 8) and, for
// the segments beside it, what streams sideways (1, 3).  One word per lane
// carries all that the segment above or below needs of that lane, and value
// and tag travel in one single-copy-atomic 128-bit access, so there is no
// fence and no flag.  Before the next step the warp that owns a reading
// segment polls the words it needs -- a row per vertical neighbour, single
// words at the corners and sides -- into ghost words of its own.  Nothing
// but the block's own barrier orders the warps of a block: a warp whose
// segments touch no other block computes while the others wait for their
// words.  Two parities suffice: a warp overwrites a word of step t only
// after it has read its neighbour's word of step t + 1 (reading is mutual),
// which that neighbour publishes after reading the word of step t.  Every
// wait is bounded: a warp that gives up makes its block set the error word
// and leave, and the others leave when they see it.
//
// What bounds it.  The exchange costs 500 to 720 cycles through L2 between
// SMs of one die and about 1050 between dies; the rest of a lone warp's step
// about 700, and 300 to 400 more where it holds a port cell.  Small lists run
// at that chain: 0.93 us per step (128 x 64 T, 88 segments; 1.31 us before, one
// launch per phase).  The 2048 x 1024 tree (46-48 segments a block) adds the
// issue of 24 packed pairs, 330 warp instructions each: 2.02 us per step, 2.27
// before (ghost rows fetched by the whole block before a barrier, one cell a
// lane, one 64-bit word per value); with BF16 storage 2.14, 2.64 before.
// Barriers between the warps that share segments instead of the block's (one
// mbarrier per warp and parity) ran 2.20; two segments per warp one after the
// other 2.39; a spilled register costs an L2 round trip here, because shared
// memory leaves the L1 cache next to nothing.
#include "d2q9_cell.cuh"

namespace lbm {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr unsigned kResidentSpinLimit = 1u << 22;
constexpr int kFeatModels = 1, kFeatMirror = 2;  // kernel builds, as in step.cu

// A step buffer in shared memory, in 4-byte words: the own rows of every
// slot ([9][32] each), then the ghost words of every slot, then a zero word.
// Ghost words of a slot: six rows of 34 (the word of lane l at 1 + l, the
// corner segments' at 0 and 33), rows 0-2 directions 4, 7, 8 from above,
// rows 3-5 directions 2, 5, 6 from below, then the side segments' words
// (direction 1 from the west, 3 from the east).
constexpr int kSegWords = 9 * 32;
constexpr int kGhostRow = 34;
constexpr int kGhostWest = 6 * kGhostRow, kGhostEast = kGhostWest + 1;
constexpr int kGhostWords = kGhostEast + 1;
template <int S>  // segments per warp
struct Layout {
  static constexpr int kWarps = S == 1 ? kResidentMaxWarps : kResidentMaxOwn / 2;
  static constexpr int kSlots = S * kWarps;
  static constexpr int kGhost0 = kSlots * kSegWords;
  static constexpr int kZero = kGhost0 + kSlots * kGhostWords;
  static constexpr int kWords = (kZero + 4) & ~3;
  static_assert(kWords <= 65536, "two slots' source words share a register");
};

// Published words of a segment, 16 bytes each: [unit][lane]
constexpr int kUnitUp = 0, kUnitDown = 1, kUnitSide = 2;
constexpr int kUnitWords = 32;

// Neighbouring segments of (y, w), position p = 0..7: E N W S NE NW SW SE,
// (dy, dw) = (0,1) (1,0) (0,-1) (-1,0) (1,1) (1,-1) (-1,-1) (-1,1).
__device__ __forceinline__ int pos_dy(int p) { return (int)((0x00220121u >> (4 * p)) & 15u) - 1; }
__device__ __forceinline__ int pos_dw(int p) { return (int)((0x20021012u >> (4 * p)) & 15u) - 1; }
// position of (dy, dw) != (0, 0)
__device__ __forceinline__ int pos_of(int dy, int dw) {
  if (dy == 0) return dw > 0 ? 0 : 2;
  if (dw == 0) return dy > 0 ? 1 : 3;
  if (dy > 0) return dw > 0 ? 4 : 5;
  return dw < 0 ? 6 : 7;
}

// ghost row of direction i arriving from above (4, 7, 8) or below (2, 5, 6)
__host__ __device__ constexpr int ghost_row(int i) {
  return i == 4 ? 0 : i == 7 ? 1 : i == 8 ? 2 : i == 2 ? 3 : i == 5 ? 4 : 5;
}

// Both values to the storage type and back (round to nearest even).
template <class T>
__device__ __forceinline__ void round2(float& a, float& b);
template <>
__device__ __forceinline__ void round2<float>(float&, float&) {}  // (the two may be one and the same)
template <>
__device__ __forceinline__ void round2<__nv_bfloat16>(float& a, float& b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  a = __low2float(h);
  b = __high2float(h);
}
template <>
__device__ __forceinline__ void round2<__half>(float& a, float& b) {
  const float2 v = __half22float2(__floats2half2_rn(a, b));
  a = v.x;
  b = v.y;
}

// A published word: three values and the step tag, one 128-bit access
// (relaxed, GPU scope: coherent in L2).  No memory clobber: each poll's use
// of its value orders it.
struct HaloWord {
  unsigned long long lo, hi;  // lo: values 0 and 1; hi: value 2 and the tag
};
__device__ __forceinline__ HaloWord halo_ld(const HaloWord* p) {
  HaloWord v;
  asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
               : "=l"(v.lo), "=l"(v.hi)
               : "l"(p));
  return v;
}
__device__ __forceinline__ void halo_st(HaloWord* p, float v0, float v1, float v2, unsigned tag) {
  const unsigned long long lo = (unsigned long long)__float_as_uint(v1) << 32 | __float_as_uint(v0);
  const unsigned long long hi = (unsigned long long)tag << 32 | __float_as_uint(v2);
  asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
               "l"(lo), "l"(hi));
}
__device__ __forceinline__ float halo_value(const HaloWord& w, int k) {
  return __uint_as_float(k == 0 ? (unsigned)w.lo : k == 1 ? (unsigned)(w.lo >> 32) : (unsigned)w.hi);
}
__device__ __forceinline__ unsigned halo_tag(const HaloWord& w) { return (unsigned)(w.hi >> 32); }

__device__ __forceinline__ int ld_relaxed_s32(const int* p) {
  int v;
  asm volatile("ld.relaxed.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

// List index of segment (y, w) of lattice `lat`, or -1 (outside the step
// rows, or no fluid cell: such a segment's cells are all solid).
__device__ __forceinline__ int list_index(const LatticeView* __restrict__ views, const int* __restrict__ seg_word_off,
                                          const int* __restrict__ seg_flags, const int* __restrict__ seg_offs, int lat,
                                          int y, int w) {
  const LatticeView& L = views[lat];
  const int y0 = first_step_row(L);
  if (w < 0 || w >= L.wpr || y < y0 || y > L.ny - 2) return -1;
  const int i = seg_word_off[lat] + (y - y0) * L.wpr + w;
  return seg_flags[i] ? seg_offs[i] : -1;
}

__device__ __forceinline__ void block_range(int nseg, int G, int b, int& s0, int& s1) {
  s0 = (int)((long long)b * nseg / G);
  s1 = (int)((long long)(b + 1) * nseg / G);
}

// slot flags
constexpr unsigned kPubUp = 1u, kPubDown = 2u, kPubSide = 4u, kHasPort = 8u, kNeumann = 16u, kSlotModel = 32u;
constexpr unsigned kPublishes = kPubUp | kPubDown | kPubSide;

// What a step seldom needs of a slot, in shared memory.
struct alignas(16) SlotInfo {
  int in_lane, out_lane; // lanes of its inlet and outlet cell, -1: none
  float u_in;            // inlet speed of its row
  int zou_he;            // port scheme
  long long row;         // element offset of the segment's first cell in its lattice
  const LatticeView* L;
  unsigned fluid;        // its fluid lanes
};
struct alignas(16) PairInfo {  // of a warp's two slots
  float rho0[2], omega[2];
  unsigned flags;  // slot flags: slot 2w in the low half, 2w + 1 in the high
  int unit0[2];    // first published word of each slot, (list index * 3) * 32
  int pad;
  int vert[4];    // words of the segments above and below slot 0, then slot 1; -1: none remote
  int edge[16];   // lanes 0-5 (slot 0) and 8-13 (slot 1): (word << 2 | value) of W E NW NE SW SE; -1: none
};

// Wait for the words that a warp's S slots read of other blocks at the step
// tagged `want`: v[2 r] what the lane's upper neighbour of slot r sent down,
// v[2 r + 1] what the lower one sent up, e the lane's edge word (words that
// come from no other block are left unset); false: gave up.
template <int S>
__device__ __forceinline__ bool poll_words(const HaloWord* hb, const int (&src)[4], int es, unsigned want, int lane,
                                           int* error, HaloWord (&v)[2 * S], HaloWord& e) {
  const unsigned long long ready = (unsigned long long)want << 32;
#pragma unroll
  for (int u = 0; u < 2 * S; ++u) {
    v[u].hi = ready;
    if (src[u] >= 0) v[u] = halo_ld(hb + src[u] + lane);  // warp-uniform
  }
  e.hi = ready;
  if (es >= 0) e = halo_ld(hb + (es >> 2));
  unsigned spins = 0;
  for (;;) {
    bool ok = halo_tag(e) == want;
#pragma unroll
    for (int u = 0; u < 2 * S; ++u) ok &= halo_tag(v[u]) == want;
    if (__all_sync(kFull, ok)) break;
#pragma unroll
    for (int u = 0; u < 2 * S; ++u)
      if (halo_tag(v[u]) != want) v[u] = halo_ld(hb + src[u] + lane);
    if (halo_tag(e) != want) e = halo_ld(hb + (es >> 2));
    ++spins;
    if (spins > kResidentSpinLimit || ((spins & 255u) == 0 && __any_sync(kFull, ld_relaxed_s32(error) != 0))) {
      if (lane == 0) atomicExch(error, 1);
      return false;
    }
  }
  return true;
}

// Fetch this warp's ghost words of step k into buffer `buf`; false: gave up.
template <int S>
__device__ __forceinline__ bool fetch_ghosts(float* buf, const PairInfo& pi, const HaloWord* halo, int parity,
                                             unsigned want, int lane, int* error) {
  const int4 vt = *reinterpret_cast<const int4*>(pi.vert);
  const int es = lane < 8 * S ? pi.edge[lane] : -1;
  const int src[4] = {vt.x, vt.y, vt.z, vt.w};
  HaloWord v[2 * S], e;
  if (!poll_words<S>(halo + parity, src, es, want, lane, error, v, e)) return false;
  float* ga = buf + Layout<S>::kGhost0 + S * (threadIdx.x >> 5) * kGhostWords;
#pragma unroll
  for (int u = 0; u < 2 * S; ++u)
    if (src[u] >= 0) {
      float* g = ga + (u >> 1) * kGhostWords + (u & 1) * 3 * kGhostRow + 1 + lane;
#pragma unroll
      for (int d = 0; d < 3; ++d) g[d * kGhostRow] = halo_value(v[u], d);
    }
  if (es >= 0) {
    const int item = lane & 7;
    const int at = item == 0 ? kGhostWest : item == 1 ? kGhostEast : item == 2 ? 2 * kGhostRow
                 : item == 3 ? 1 * kGhostRow + 33 : item == 4 ? 4 * kGhostRow : 5 * kGhostRow + 33;
    ga[(lane >> 3) * kGhostWords + at] = halo_value(e, es & 3);
  }
  __syncwarp();
  return true;
}

// Port rules of the slot's port cells (all lanes call).
__device__ __forceinline__ void ports_of(float (&g)[9], unsigned slot_flags, const SlotInfo& si, float rho0, int lane) {
  const int4 pw = *reinterpret_cast<const int4*>(&si);  // in_lane, out_lane, u_in, zou_he
  const bool out = lane == pw.y;
  if (slot_flags & kNeumann) {  // zero-gradient outlet: cell nx-2 is the lane to the left
    const float n3 = __shfl_up_sync(kFull, g[3], 1);
    const float n6 = __shfl_up_sync(kFull, g[6], 1);
    const float n7 = __shfl_up_sync(kFull, g[7], 1);
    if (out) {
      g[3] = n3;
      g[6] = n6;
      g[7] = n7;
    }
  }
  const int scheme = pw.w ? LBM_PORTS_ZOU_HE : LBM_PORTS_REGULARIZED;
  if (lane == pw.x)
    inlet_rule(g, __int_as_float(pw.z), rho0, scheme);
  else if (out && !(slot_flags & kNeumann))
    outlet_rule(g, rho0, scheme);
}

__device__ __forceinline__ void write_moments(const SlotInfo& si, int lane, bool last, float drho, float ux, float uy) {
  const LatticeView& L = *si.L;
  const long long c = si.row + lane;
  if (!LBM_OK_IDX(c, L.plane)) return;
  L.drho[c] = drho;
  (last ? L.ux : L.ux_prev)[c] = ux;
  (last ? L.uy : L.uy_prev)[c] = uy;
}

// hb: this lane's word of the segment's first unit
__device__ __forceinline__ void publish(HaloWord* hb, unsigned flags, int lane, const float (&g)[9], unsigned tag) {
  if (flags & kPubUp) halo_st(hb + kUnitUp * kUnitWords, g[2], g[5], g[6], tag);
  if (flags & kPubDown) halo_st(hb + kUnitDown * kUnitWords, g[4], g[7], g[8], tag);
  if ((flags & kPubSide) && (lane == 0 || lane == 31)) halo_st(hb + kUnitSide * kUnitWords, g[1], g[3], 0.0f, tag);
}

// One time step of the warp's S segments: buffer PAR read, the other written.
template <class T, int FEAT, int S, int PAR>
__device__ __forceinline__ void warp_step(float* sm, const unsigned (&off)[8], unsigned own, int k, int k_last,
                                          int mom_prev, unsigned epoch0, const PairInfo& pi, const SlotInfo* si,
                                          HaloWord* halo, int parity, int lane) {
  constexpr int kCur = PAR * Layout<S>::kWords, kNxt = (PAR ^ 1) * Layout<S>::kWords;
  float g[S][9];
#pragma unroll
  for (int r = 0; r < S; ++r) g[r][0] = sm[own + r * kSegWords + kCur];
#pragma unroll
  for (int i = 1; i <= 8; ++i) {
    unsigned o = off[i - 1];
    if (S == 2) asm volatile("" : "+r"(o));  // unpacked here, at every step: hoisted, the sixteen words spill
    g[0][i] = sm[(S == 2 ? o & 0xffffu : o) + kCur];
    if (S == 2) g[S - 1][i] = sm[(o >> 16) + kCur];
  }
  const float4 par = *reinterpret_cast<const float4*>(pi.rho0);  // rho0 and omega of the slots
  const int4 units = *reinterpret_cast<const int4*>(&pi.flags);
  const unsigned flags = (unsigned)units.x;
  if (flags & (kHasPort << 16 | kHasPort)) {  // warp-uniform
    if (flags & kHasPort) ports_of(g[0], flags, si[0], par.x, lane);
    if (S == 2 && (flags & kHasPort << 16)) ports_of(g[S - 1], flags >> 16, si[S - 1], par.y, lane);
  }
  float dr[S], ux[S], uy[S];
  const bool models = (FEAT & kFeatModels) && (flags & (kSlotModel << 16 | kSlotModel));
  if (models || S == 1) {
#pragma unroll
    for (int r = 0; r < S; ++r) {
      const float rho0 = r ? par.y : par.x, omega = r ? par.w : par.z;
      if (models && (flags & kSlotModel << (16 * r)))
        collide_other(g[r], rho0, omega, si[r].L->collision, si[r].L->c_smag, dr[r], ux[r], uy[r]);
      else
        bgk(g[r], rho0, omega, dr[r], ux[r], uy[r]);
    }
  } else {
    bgk2(g[0], g[S - 1], f2(par.x, par.y), f2(par.z, par.w), dr[0], ux[0], uy[0], dr[S - 1], ux[S - 1], uy[S - 1]);
  }
#pragma unroll
  for (int i = 0; i < 9; ++i) round2<T>(g[0][i], g[S - 1][i]);
  if ((flags & (kPublishes << 16 | kPublishes)) && k != k_last) {
    const unsigned tag = epoch0 + (unsigned)k + 1u;
    HaloWord* hb = halo + (parity + lane);
    if (flags & kPublishes) publish(hb + units.y, flags, lane, g[0], tag);
    if (S == 2 && (flags & kPublishes << 16)) publish(hb + units.z, flags >> 16, lane, g[S - 1], tag);
  }
#pragma unroll
  for (int r = 0; r < S; ++r)
#pragma unroll
    for (int i = 0; i < 9; ++i) sm[own + r * kSegWords + kNxt + i * 32] = g[r][i];
  if (k == k_last || k == mom_prev) {
#pragma unroll
    for (int r = 0; r < S; ++r)
      if ((si[r].fluid >> lane) & 1u) write_moments(si[r], lane, k == k_last, dr[r], ux[r], uy[r]);
  }
}

// The resident solve: n_steps (even) time steps of the whole set.  halo:
// [2][halo_cap][3][32] published words; tags epoch0 + 1 .. epoch0 + n_steps - 1
// are published by this launch.  Moments go to drho/ux/uy at the last step
// and to drho/ux_prev/uy_prev at step mom_prev (-1: none).  tag_skew is 0, or
// 1 under the bounded-wait test hook (every wait then runs out).
// S: segments per warp, 1 or 2.
template <class T, int FEAT, int S>
__global__ void __launch_bounds__(Layout<S>::kWarps * 32, 1)
    k_stream_collide_resident(const LatticeView* __restrict__ views, const SegRef* __restrict__ segs,
                              const int* __restrict__ n_segs, const int* __restrict__ seg_word_off,
                              const int* __restrict__ seg_flags, const int* __restrict__ seg_offs,
                              HaloWord* __restrict__ halo, int halo_cap, unsigned epoch0, int n_steps, int mom_prev,
                              int* __restrict__ error, unsigned tag_skew) {
  extern __shared__ __align__(16) float sm[];
  __shared__ int s_nbq[Layout<S>::kSlots][8];  // list index of each neighbouring segment, or -1
  __shared__ int s_order[Layout<S>::kSlots], s_slot[Layout<S>::kSlots];
  __shared__ SlotInfo s_slots[Layout<S>::kSlots];
  __shared__ PairInfo s_pairs[Layout<S>::kWarps];
  using P = Pop<T>;
  constexpr int kBufWords = Layout<S>::kWords, kZeroWord = Layout<S>::kZero, kGhost0 = Layout<S>::kGhost0;
  const int nseg = n_segs[0];
  int s0, s1;
  block_range(nseg, gridDim.x, blockIdx.x, s0, s1);
  const int n_own = s1 - s0;  // at most S per warp: the host sizes the grid by a bound on nseg
  if (n_own > S * (int)(blockDim.x >> 5)) {
    if (threadIdx.x == 0) atomicExch(error, 1);
    return;
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* buf0 = sm;

  // ---- once per launch: neighbours, slots, source addresses ----
  for (int i = threadIdx.x; i < 8 * n_own; i += blockDim.x) {
    const SegRef sr = segs[s0 + (i >> 3)];
    const int p = i & 7;
    s_nbq[i >> 3][p] = list_index(views, seg_word_off, seg_flags, seg_offs, sr.lattice,
                                  (sr.yw >> kSegWordBits) + pos_dy(p),
                                  (sr.yw & ((1 << kSegWordBits) - 1)) + pos_dw(p));
  }
  __syncthreads();
  if (warp == 0) {
    // Slots.  A port cell's rules take as long as a collision, so segments with
    // port cells go to slots of different warps, each beside one without.  The
    // others follow with those that read other blocks first, so that they share
    // warps and the remaining warps compute while these wait for their words.
    unsigned port[2], touch[2], plain[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int t = lane + 32 * h;
      bool remote = false, has_port = false;
      if (t < n_own) {
        for (int p = 0; p < 8; ++p) remote |= s_nbq[t][p] >= 0 && (s_nbq[t][p] < s0 || s_nbq[t][p] >= s1);
        const SegRef sr = segs[s0 + t];
        const LatticeView& L = views[sr.lattice];
        const int y = sr.yw >> kSegWordBits, w = sr.yw & ((1 << kSegWordBits) - 1);
        const uint32_t fl = ~L.mask[(long long)y * mask_stride(L.wpr) + w];
        has_port = (w == 0 && (fl & 1u)) || (w == (L.nx - 1) >> 5 && ((fl >> ((L.nx - 1) & 31)) & 1u));
      }
      port[h] = __ballot_sync(kFull, has_port);
      touch[h] = __ballot_sync(kFull, t < n_own && remote && !has_port);
      plain[h] = __ballot_sync(kFull, t < n_own && !remote && !has_port);
    }
    const int n_port = __popc(port[0]) + __popc(port[1]), n_touch = __popc(touch[0]) + __popc(touch[1]);
    const int m = min(n_port, n_own - n_port);  // pairs of a port and another segment
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int t = lane + 32 * h;
      if (t >= n_own) continue;
      auto rank = [&](const unsigned (&b)[2]) {
        const unsigned below = (1u << lane) - 1u;
        return h ? __popc(b[0]) + __popc(b[1] & below) : __popc(b[0] & below);
      };
      const bool is_port = (port[h] >> lane) & 1u;
      const int i = is_port ? rank(port) : ((touch[h] >> lane) & 1u) ? rank(touch) : n_touch + rank(plain);
      const int j = S == 1 ? (is_port ? i : n_port + i) : i < m ? 2 * i + (is_port ? 0 : 1) : m + i;
      s_order[j] = t;
      s_slot[t] = j;
    }
  }
  if (threadIdx.x < 2) sm[threadIdx.x * kBufWords + kZeroWord] = 0.0f;
  __syncthreads();

  const uint16_t* __restrict__ nbs = segment_flags(segs, n_segs);
  unsigned off[8];  // source words of directions 1..8 (two slots: 2w in the low half, 2w + 1 in the high)
  const unsigned own = (unsigned)(S * warp * kSegWords + lane);
  PairInfo& pi = s_pairs[warp];
  unsigned flags = 0;
  if (lane < 4) pi.vert[lane] = -1;
  if (lane < 16) pi.edge[lane] = -1;
  __syncwarp();
#pragma unroll
  for (int r = 0; r < S; ++r) {
    const int j = S * warp + r;
    unsigned sf = 0;
    if (j >= n_own) {  // an empty slot relaxes a resting cell into rows nobody reads
      if (lane == 0) {
        pi.rho0[r] = 1.0f;
        pi.omega[r] = 1.0f;
        pi.unit0[r] = 0;
        s_slots[j] = SlotInfo{-1, -1, 0.0f, 0, 0, views, 0u};
      }
#pragma unroll
      for (int i = 0; i < 9; ++i) buf0[j * kSegWords + i * 32 + lane] = 0.0f;
#pragma unroll
      for (int i = 0; i < 8; ++i) off[i] = r ? off[i] | (unsigned)kZeroWord << 16 : (unsigned)kZeroWord;
      continue;
    }
    const int t = s_order[j], q = s0 + t;
    const SegRef sr = segs[q];
    const LatticeView& L = views[sr.lattice];
    const int y = sr.yw >> kSegWordBits, w = sr.yw & ((1 << kSegWordBits) - 1);
    const int x = (w << 5) + lane;
    const uint32_t mc = L.mask[(long long)y * mask_stride(L.wpr) + w];
    const bool fluid = !((mc >> lane) & 1u);
    const bool inlet = x == 0, outlet = x == L.nx - 1;
    const unsigned nb = nbs[(long long)q * 32 + lane];
    const bool plane = (FEAT & kFeatMirror) && L.mirror && y == 0;  // the row next to the symmetry plane
    const int base = j * kSegWords, gbase = kGhost0 + j * kGhostWords;
#pragma unroll
    for (int i = 1; i <= 8; ++i) {
      int o = kZeroWord;
      const int cx = cx_of(i);
      const bool unknown = (inlet && cx > 0) || (outlet && cx < 0);
      if (fluid && !unknown) {
        if ((nb >> (opp_of(i) - 1)) & 1u) {  // the source cell is solid: bounce-back
          o = base + opp_of(i) * 32 + lane;
        } else {
          // next to the plane a diagonal from below is what the row-0 neighbour sent
          // across it: NE from the west neighbour's SE, NW from the east one's SW
          const bool image = plane && (i == 5 || i == 6);
          const int si = image ? (i == 5 ? 8 : 7) : i;
          const int sl = lane - cx, dy = image ? 0 : -cy_of(i);
          const int dw = sl < 0 ? -1 : sl > 31 ? 1 : 0;
          if (dy == 0 && dw == 0) {
            o = base + si * 32 + sl;
          } else {
            const int nq = s_nbq[t][pos_of(dy, dw)];
            if (nq >= s0 && nq < s1)
              o = s_slot[nq - s0] * kSegWords + si * 32 + (sl & 31);
            else if (nq >= 0)
              o = gbase + ((cy_of(i) == 0) ? (i == 1 ? kGhostWest : kGhostEast) : ghost_row(i) * kGhostRow + 1 + sl);
            // nq < 0 cannot happen for a fluid source; the zero word keeps it harmless
          }
        }
      }
      if (!LBM_OK_IDX(o, kZeroWord + 1)) o = kZeroWord;
      off[i - 1] = r ? off[i - 1] | (unsigned)o << 16 : (unsigned)o;
    }
    // what other blocks read of this segment, and what it reads of theirs
    bool rem[8];
#pragma unroll
    for (int p = 0; p < 8; ++p)
      rem[p] = s_nbq[t][p] >= 0 && (s_nbq[t][p] < s0 || s_nbq[t][p] >= s1) && LBM_OK_IDX(s_nbq[t][p], halo_cap);
    const bool side = rem[0] || rem[2];
    if (rem[1] || rem[4] || rem[5]) sf |= kPubUp;
    if (rem[3] || rem[6] || rem[7] || (plane && side)) sf |= kPubDown;
    if (side) sf |= kPubSide;
    auto word = [&](int p, int unit, int l, int value) {
      return ((s_nbq[t][p] * 3 + unit) * kUnitWords + l) << 2 | value;
    };
    if (lane == 0) {
      if (rem[1]) pi.vert[2 * r] = (s_nbq[t][1] * 3 + kUnitDown) * kUnitWords;
      if (rem[3]) pi.vert[2 * r + 1] = (s_nbq[t][3] * 3 + kUnitUp) * kUnitWords;
      if (rem[2]) pi.edge[8 * r + 0] = word(2, kUnitSide, 31, 0);
      if (rem[0]) pi.edge[8 * r + 1] = word(0, kUnitSide, 0, 1);
      if (rem[5]) pi.edge[8 * r + 2] = word(5, kUnitDown, 31, 2);
      if (rem[4]) pi.edge[8 * r + 3] = word(4, kUnitDown, 0, 1);
      if (rem[6]) pi.edge[8 * r + 4] = word(6, kUnitUp, 31, 1);
      if (rem[7]) pi.edge[8 * r + 5] = word(7, kUnitUp, 0, 2);
      if (plane && rem[2]) pi.edge[8 * r + 4] = word(2, kUnitDown, 31, 2);
      if (plane && rem[0]) pi.edge[8 * r + 5] = word(0, kUnitDown, 0, 1);
      pi.rho0[r] = L.rho0;
      pi.omega[r] = L.omega;
      pi.unit0[r] = LBM_OK_IDX(q, halo_cap) ? q * 3 * kUnitWords : 0;
      const int ol = L.nx - 1 - (w << 5);
      s_slots[j] = SlotInfo{w == 0 && !(mc & 1u) ? 0 : -1, ol < 32 && !((mc >> (ol & 31)) & 1u) ? ol : -1,
                            w == 0 ? L.u_in[y] : 0.0f, L.port_scheme == LBM_PORTS_ZOU_HE,
                            (long long)y * L.pitch + (w << 5), &L, ~mc};
    }
    if (__any_sync(kFull, fluid && (inlet || outlet))) sf |= kHasPort;
    if (L.outlet_rule == LBM_OUT_NEUMANN) sf |= kNeumann;
    if ((FEAT & kFeatModels) && L.collision != LBM_COLLIDE_BGK) sf |= kSlotModel;
    flags |= sf << (16 * r);
    // own populations and the ghost words of step 0 from the canonical layout
    const T* F = static_cast<const T*>(L.f);
    const int pl = (int)L.plane, cell = y * L.pitch + x;
#define FROM(at) (LBM_OK_IDX((at), L.f_elems) ? P::ld(F + at) : 0.0f)
#pragma unroll
    for (int i = 0; i < 9; ++i) buf0[base + i * 32 + lane] = FROM(i * pl + cell);
    float* gw = buf0 + gbase;
    if (rem[1]) {
      gw[1 + lane] = FROM(4 * pl + cell + L.pitch);
      gw[kGhostRow + 1 + lane] = FROM(7 * pl + cell + L.pitch);
      gw[2 * kGhostRow + 1 + lane] = FROM(8 * pl + cell + L.pitch);
    }
    if (rem[3]) {
      gw[3 * kGhostRow + 1 + lane] = FROM(2 * pl + cell - L.pitch);
      gw[4 * kGhostRow + 1 + lane] = FROM(5 * pl + cell - L.pitch);
      gw[5 * kGhostRow + 1 + lane] = FROM(6 * pl + cell - L.pitch);
    }
    if (lane == 0) {
      if (rem[2]) gw[kGhostWest] = FROM(1 * pl + cell - 1);
      if (rem[5]) gw[2 * kGhostRow] = FROM(8 * pl + cell + L.pitch - 1);
      if (rem[6]) gw[4 * kGhostRow] = FROM(5 * pl + cell - L.pitch - 1);
      if (plane && rem[2]) gw[4 * kGhostRow] = FROM(8 * pl + cell - 1);
    }
    if (lane == 31) {
      if (rem[0]) gw[kGhostEast] = FROM(3 * pl + cell + 1);
      if (rem[4]) gw[kGhostRow + 33] = FROM(7 * pl + cell + L.pitch + 1);
      if (rem[7]) gw[5 * kGhostRow + 33] = FROM(6 * pl + cell - L.pitch + 1);
      if (plane && rem[0]) gw[5 * kGhostRow + 33] = FROM(7 * pl + cell + 1);
    }
#undef FROM
  }
  const SlotInfo* si = s_slots + S * warp;
  if (lane == 0) pi.flags = flags;
  // ghost words are read exactly by the segments that publish
  const bool ghosts = (flags & (kPublishes << 16 | kPublishes)) != 0;

  // ---- the time steps, two per turn: step k reads buffer k & 1 ----
  // A warp whose words do not come sets the error word, which ends every other
  // wait, and idles to the next common check; the block leaves there.
  const int parity = halo_cap * 3 * kUnitWords;
  int failed = 0;
  auto turn = [&](int k) {
    if ((k & 127) == 0) return __syncthreads_or(failed) == 0;
    __syncthreads();
    return true;
  };
  for (int k = 0; k < n_steps; k += 2) {
    if (!turn(k)) break;
    if (k > 0 && ghosts && !failed)
      failed = !fetch_ghosts<S>(sm, pi, halo, parity, epoch0 + (unsigned)k + tag_skew, lane, error);
    if (!failed) warp_step<T, FEAT, S, 0>(sm, off, own, k, n_steps - 1, mom_prev, epoch0, pi, si, halo, 0, lane);
    __syncthreads();
    if (ghosts && !failed)
      failed = !fetch_ghosts<S>(sm + kBufWords, pi, halo, 0, epoch0 + (unsigned)k + 1u + tag_skew, lane, error);
    if (!failed) warp_step<T, FEAT, S, 1>(sm, off, own, k + 1, n_steps - 1, mom_prev, epoch0, pi, si, halo, parity, lane);
  }
  if (__syncthreads_or(failed)) return;  // this block stores nothing; others may have ended: the state is void
  // ---- the final state (buffer 0: an even number of steps) to the canonical layout ----
#pragma unroll
  for (int r = 0; r < S; ++r) {
    if (!((si[r].fluid >> lane) & 1u)) continue;
    const LatticeView& L = *si[r].L;
    T* F = static_cast<T*>(L.f) + si[r].row + lane;
    const int pl = (int)L.plane;
#pragma unroll
    for (int i = 0; i < 9; ++i)
      if (LBM_OK_IDX(si[r].row + lane + i * pl, L.f_elems)) P::st(F + i * pl, sm[own + r * kSegWords + i * 32]);
  }
}

// ---- lists of more than kResidentMaxOwn segments per SM ----------------------
//
// One copy of the populations (AA pattern) and several pairs of segments per
// warp.  Step k even reads every population where it lies after the last
// collision -- slot i of the source cell, its own opposite slot beyond a wall
// -- and writes the opposite population to the place just read; step k odd
// finds what streamed to a cell in the cell's own slots (direction i in slot
// opp(i)) and leaves its result there in place.  Every place is read and
// written by one lane within a step, so one copy and the block's barrier
// between steps do.  Source words come from a table in shared memory (two
// slots' words to a register); odd steps need none.  What crosses to another
// block is published and polled exactly as above, but goes from the polled
// words to registers by shuffles; the lane's `remote` bits say where it
// replaces the shared-memory value.  1.8 KB of shared memory per segment
// against 4 KB, so up to kResidentManyOwn of them.
//
// Pairs that exchange come first in the slot order; half of the warps take
// their pairs in reverse, so that words travel while other warps compute.
//
// What bounds it.  15 candidates (111 segments a block, three pairs a warp):
// 3.45 us a step, per phase 5.6; without the exchange 3.3, without the
// collisions as well 2.1 (the FMA pipe needs 1.2 for them).  Twenty warps of
// 96 registers: 24 of 80 spill or, with one code for both kinds of step, run
// 3.8; 16 of 128 take a fourth round, 4.3.  Always all twenty, though the last
// round may be part empty: 52 segments a block 2.4 against 3.0 with thirteen
// warps of two pairs.
constexpr int kManyPairs = kResidentManyOwn / 2;
struct ManyShared {
  float rows[2 * kManyPairs][kSegWords];
  float outside[32];                  // takes what leaves the block
  uint4 src[kManyPairs][2][32];       // source words of directions 1-4 and 5-8: slot 2p low, 2p + 1 high half
  SlotInfo slots[2 * kManyPairs];
  PairInfo pairs[kManyPairs];
  uint16_t remote[kManyPairs][32];    // directions that come from another block, slot 2p in the low byte
};
static_assert(sizeof(ManyShared) <= 227 * 1024, "shared memory of a block");
static_assert((2 * kManyPairs * kSegWords + 32) <= 65536, "two slots' source words share a register");

// What other blocks sent to slot r of the pair replaces what was read of it.
__device__ __forceinline__ void take_words(float (&g)[9], const HaloWord& from_above, const HaloWord& from_below,
                                           float edge, int r, unsigned remote, int lane) {
  const int far = lane == 31 ? 1 : 0;
  const float side = __shfl_sync(kFull, edge, 8 * r + far), above = __shfl_sync(kFull, edge, 8 * r + 2 + far),
              below = __shfl_sync(kFull, edge, 8 * r + 4 + far);
  const float a7 = __shfl_down_sync(kFull, halo_value(from_above, 1), 1);
  const float a8 = __shfl_up_sync(kFull, halo_value(from_above, 2), 1);
  const float b5 = __shfl_up_sync(kFull, halo_value(from_below, 1), 1);
  const float b6 = __shfl_down_sync(kFull, halo_value(from_below, 2), 1);
  if (remote & 1u) g[1] = side;
  if (remote & 2u) g[2] = halo_value(from_below, 0);
  if (remote & 4u) g[3] = side;
  if (remote & 8u) g[4] = halo_value(from_above, 0);
  if (remote & 16u) g[5] = lane == 0 ? below : b5;
  if (remote & 32u) g[6] = lane == 31 ? below : b6;
  if (remote & 64u) g[7] = lane == 31 ? above : a7;
  if (remote & 128u) g[8] = lane == 0 ? above : a8;
}

__device__ __forceinline__ void source_words(const ManyShared& m, int p, int lane, unsigned (&src)[9]) {
  asm volatile("" : "+r"(p));
  const uint4 a = m.src[p][0][lane], b = m.src[p][1][lane];
  src[1] = a.x, src[2] = a.y, src[3] = a.z, src[4] = a.w;
  src[5] = b.x, src[6] = b.y, src[7] = b.z, src[8] = b.w;
}

// Step k of pair p, even or odd; false: a word did not come.
template <class T, int FEAT, bool even>
__device__ __forceinline__ bool many_step(ManyShared& m, int p, int k, int k_last, int mom_prev, unsigned epoch0,
                                          unsigned tag_skew, HaloWord* halo, int parity, int lane, int* error) {
  asm volatile("" : "+r"(lane));  // what follows from it is computed here, not kept over the loop: that spills
  float* sm = m.rows[0];
  const int own = 2 * p * kSegWords + lane;
  const PairInfo& pi = m.pairs[p];
  const SlotInfo* si = m.slots + 2 * p;
  float g[2][9];
#pragma unroll
  for (int r = 0; r < 2; ++r) g[r][0] = sm[own + r * kSegWords];
  if (even) {
    unsigned src[9];
    source_words(m, p, lane, src);
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      g[0][i] = sm[src[i] & 0xffffu];
      g[1][i] = sm[src[i] >> 16];
    }
  } else {
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      g[0][i] = sm[own + opp_of(i) * 32];
      g[1][i] = sm[own + kSegWords + opp_of(i) * 32];
    }
  }
  const float4 par = *reinterpret_cast<const float4*>(pi.rho0);  // rho0 and omega of the slots
  const int4 units = *reinterpret_cast<const int4*>(&pi.flags);
  const unsigned flags = (unsigned)units.x;
  if (flags & (kPublishes << 16 | kPublishes)) {  // warp-uniform
    const int4 vt = *reinterpret_cast<const int4*>(pi.vert);
    const int from[4] = {vt.x, vt.y, vt.z, vt.w};
    const int es = lane < 16 ? pi.edge[lane] : -1;
    const unsigned remote = m.remote[p][lane];
    HaloWord v[4], e;
    if (!poll_words<2>(halo + (even ? parity : 0), from, es, epoch0 + (unsigned)k + tag_skew, lane, error, v, e)) return false;
    const float edge = halo_value(e, es & 3);
    if (flags & kPublishes) take_words(g[0], v[0], v[1], edge, 0, remote, lane);
    if (flags & kPublishes << 16) take_words(g[1], v[2], v[3], edge, 1, remote >> 8, lane);
  }
  if (flags & (kHasPort << 16 | kHasPort)) {
    if (flags & kHasPort) ports_of(g[0], flags, si[0], par.x, lane);
    if (flags & kHasPort << 16) ports_of(g[1], flags >> 16, si[1], par.y, lane);
  }
  float dr[2], ux[2], uy[2];
  if ((FEAT & kFeatModels) && (flags & (kSlotModel << 16 | kSlotModel))) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const float rho0 = r ? par.y : par.x, omega = r ? par.w : par.z;
      if (flags & kSlotModel << (16 * r))
        collide_other(g[r], rho0, omega, si[r].L->collision, si[r].L->c_smag, dr[r], ux[r], uy[r]);
      else
        bgk(g[r], rho0, omega, dr[r], ux[r], uy[r]);
    }
  } else {
    bgk2(g[0], g[1], f2(par.x, par.y), f2(par.z, par.w), dr[0], ux[0], uy[0], dr[1], ux[1], uy[1]);
  }
#pragma unroll
  for (int i = 0; i < 9; ++i) round2<T>(g[0][i], g[1][i]);
  if ((flags & (kPublishes << 16 | kPublishes)) && k != k_last) {
    const unsigned tag = epoch0 + (unsigned)k + 1u;
    HaloWord* out = halo + ((even ? 0 : parity) + lane);
    if (flags & kPublishes) publish(out + units.y, flags, lane, g[0], tag);
    if (flags & kPublishes << 16) publish(out + units.z, flags >> 16, lane, g[1], tag);
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) sm[own + r * kSegWords] = g[r][0];
  if (even) {  // the place direction i came from takes the opposite one
    unsigned src[9];
    source_words(m, p, lane, src);  // read again: kept, they would spill
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      sm[src[i] & 0xffffu] = g[0][opp_of(i)];
      sm[src[i] >> 16] = g[1][opp_of(i)];
    }
  } else {
#pragma unroll
    for (int i = 1; i < 9; ++i) {
      sm[own + i * 32] = g[0][i];
      sm[own + kSegWords + i * 32] = g[1][i];
    }
  }
  if (k == k_last || k == mom_prev) {
#pragma unroll
    for (int r = 0; r < 2; ++r)
      if ((si[r].fluid >> lane) & 1u) write_moments(si[r], lane, k == k_last, dr[r], ux[r], uy[r]);
  }
  return true;
}

// As k_stream_collide_resident.  Tags epoch0 .. epoch0 + n_steps - 1 are
// published (the state before the first step goes the same way).
template <class T, int FEAT>
__global__ void __launch_bounds__(kResidentManyWarps * 32, 1)
    k_stream_collide_resident_many(const LatticeView* __restrict__ views, const SegRef* __restrict__ segs,
                                   const int* __restrict__ n_segs, const int* __restrict__ seg_word_off,
                                   const int* __restrict__ seg_flags, const int* __restrict__ seg_offs,
                                   HaloWord* __restrict__ halo, int halo_cap, unsigned epoch0, int n_steps,
                                   int mom_prev, int* __restrict__ error, unsigned tag_skew) {
  extern __shared__ __align__(16) unsigned char many_smem[];
  using P = Pop<T>;
  ManyShared& m = *reinterpret_cast<ManyShared*>(many_smem);
  const int nseg = n_segs[0];
  int s0, s1;
  block_range(nseg, gridDim.x, blockIdx.x, s0, s1);
  const int n_own = s1 - s0;  // the host sizes the grid by a bound on nseg
  if (n_own > 2 * kManyPairs) {
    if (threadIdx.x == 0) atomicExch(error, 1);
    return;
  }
  const int n_pairs = (n_own + 1) / 2;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;

  // ---- once per launch: neighbours, slots, source words ----
  // (scratch of this part lies where the rows go afterwards)
  int(*s_nbq)[8] = reinterpret_cast<int(*)[8]>(m.rows);  // list index of each neighbouring segment, or -1
  uint8_t* s_order = reinterpret_cast<uint8_t*>(s_nbq + 2 * kManyPairs);
  uint8_t* s_slot = s_order + 2 * kManyPairs;
  for (int i = threadIdx.x; i < 8 * n_own; i += blockDim.x) {
    const SegRef sr = segs[s0 + (i >> 3)];
    const int q = i & 7;
    s_nbq[i >> 3][q] = list_index(views, seg_word_off, seg_flags, seg_offs, sr.lattice,
                                  (sr.yw >> kSegWordBits) + pos_dy(q),
                                  (sr.yw & ((1 << kSegWordBits) - 1)) + pos_dw(q));
  }
  __syncthreads();
  auto is_remote = [&](int q) { return q >= 0 && (q < s0 || q >= s1); };
  constexpr int kParts = (kResidentManyOwn + 31) / 32;
  if (warp == 0) {  // slots: ports beside others, then those that exchange, then the rest (as above)
    unsigned port[kParts], touch[kParts];
#pragma unroll
    for (int h = 0; h < kParts; ++h) {
      const int t = lane + 32 * h;
      bool remote = false, has_port = false;
      if (t < n_own) {
        for (int q = 0; q < 8; ++q) remote |= is_remote(s_nbq[t][q]);
        const SegRef sr = segs[s0 + t];
        const LatticeView& L = views[sr.lattice];
        const int y = sr.yw >> kSegWordBits, w = sr.yw & ((1 << kSegWordBits) - 1);
        const uint32_t fl = ~L.mask[(long long)y * mask_stride(L.wpr) + w];
        has_port = (w == 0 && (fl & 1u)) || (w == (L.nx - 1) >> 5 && ((fl >> ((L.nx - 1) & 31)) & 1u));
      }
      port[h] = __ballot_sync(kFull, has_port);
      touch[h] = __ballot_sync(kFull, remote && !has_port);
    }
    int n_port = 0, n_touch = 0;
#pragma unroll
    for (int h = 0; h < kParts; ++h) n_port += __popc(port[h]), n_touch += __popc(touch[h]);
    const int mixed = min(n_port, n_own - n_port);  // pairs of a port and another segment
    const unsigned below = (1u << lane) - 1u;
    int ports = 0, touching = 0, plain = 0;  // of the parts before
#pragma unroll
    for (int h = 0; h < kParts; ++h) {
      const int t = lane + 32 * h;
      const unsigned own = t < n_own ? 1u << lane : 0u;
      const unsigned all = n_own >= 32 * h + 32 ? kFull : n_own > 32 * h ? (1u << (n_own - 32 * h)) - 1u : 0u;
      const unsigned rest = all & ~port[h] & ~touch[h];
      const bool is_port = port[h] & own;
      const int i = is_port ? ports + __popc(port[h] & below)
                  : (touch[h] & own) ? touching + __popc(touch[h] & below) : n_touch + plain + __popc(rest & below);
      if (own) {
        const int j = i < mixed ? 2 * i + (is_port ? 0 : 1) : mixed + i;
        s_order[j] = (uint8_t)t;
        s_slot[t] = (uint8_t)j;
      }
      ports += __popc(port[h]);
      touching += __popc(touch[h]);
      plain += __popc(rest);
    }
  }
  __syncthreads();
  const uint16_t* __restrict__ nbs = segment_flags(segs, n_segs);
  const int outside = 2 * kManyPairs * kSegWords + lane;  // takes what other blocks' cells get
  for (int p = warp; p < n_pairs; p += n_warps) {
    PairInfo& pi = m.pairs[p];
    if (lane < 4) pi.vert[lane] = -1;
    if (lane < 16) pi.edge[lane] = -1;
    __syncwarp();
    unsigned flags = 0, remote = 0;
    unsigned off[8] = {};
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int j = 2 * p + r, base = j * kSegWords;
      if (j >= n_own) {  // an empty slot relaxes a resting cell
        if (lane == 0) {
          pi.rho0[r] = 1.0f;
          pi.omega[r] = 1.0f;
          pi.unit0[r] = 0;
          m.slots[j] = SlotInfo{-1, -1, 0.0f, 0, 0, views, 0u};
        }
#pragma unroll
        for (int i = 1; i <= 8; ++i) off[i - 1] |= (unsigned)(base + i * 32 + lane) << (16 * r);
        continue;
      }
      const int t = s_order[j], q = s0 + t;
      const SegRef sr = segs[q];
      const LatticeView& L = views[sr.lattice];
      const int y = sr.yw >> kSegWordBits, w = sr.yw & ((1 << kSegWordBits) - 1);
      const int x = (w << 5) + lane;
      const uint32_t mc = L.mask[(long long)y * mask_stride(L.wpr) + w];
      const bool fluid = !((mc >> lane) & 1u);
      const bool inlet = x == 0, outlet = x == L.nx - 1;
      const unsigned nb = nbs[(long long)q * 32 + lane];
      const bool plane = (FEAT & kFeatMirror) && L.mirror && y == 0;  // the row next to the symmetry plane
#pragma unroll
      for (int i = 1; i <= 8; ++i) {
        const int cx = cx_of(i);
        int o = base + opp_of(i) * 32 + lane;  // bounce-back; nobody else's word beyond a port or in a solid cell
        if (fluid && !(inlet && cx > 0) && !(outlet && cx < 0) && !((nb >> (opp_of(i) - 1)) & 1u)) {
          const bool image = plane && (i == 5 || i == 6);  // see k_stream_collide_resident
          const int si = image ? (i == 5 ? 8 : 7) : i;
          const int sl = lane - cx, dy = image ? 0 : -cy_of(i);
          const int dw = sl < 0 ? -1 : sl > 31 ? 1 : 0;
          if (dy == 0 && dw == 0) {
            o = base + si * 32 + sl;
          } else {
            const int nq = s_nbq[t][pos_of(dy, dw)];
            if (is_remote(nq)) {
              o = outside;
              remote |= 1u << (i - 1 + 8 * r);
            } else if (nq >= 0) {  // (a fluid source lies in a listed segment)
              o = s_slot[nq - s0] * kSegWords + si * 32 + (sl & 31);
            }
          }
        }
        if (!LBM_OK_IDX(o, 2 * kManyPairs * kSegWords + 32)) o = outside;
        off[i - 1] |= (unsigned)o << (16 * r);
      }
      // what other blocks read of this segment, and what it reads of theirs
      bool rem[8];
#pragma unroll
      for (int d = 0; d < 8; ++d) rem[d] = is_remote(s_nbq[t][d]) && LBM_OK_IDX(s_nbq[t][d], halo_cap);
      const bool side = rem[0] || rem[2];
      unsigned sf = 0;
      if (rem[1] || rem[4] || rem[5]) sf |= kPubUp;
      if (rem[3] || rem[6] || rem[7] || (plane && side)) sf |= kPubDown;
      if (side) sf |= kPubSide;
      auto word = [&](int d, int unit, int l, int value) {
        return ((s_nbq[t][d] * 3 + unit) * kUnitWords + l) << 2 | value;
      };
      if (lane == 0) {
        if (rem[1]) pi.vert[2 * r] = (s_nbq[t][1] * 3 + kUnitDown) * kUnitWords;
        if (rem[3]) pi.vert[2 * r + 1] = (s_nbq[t][3] * 3 + kUnitUp) * kUnitWords;
        if (rem[2]) pi.edge[8 * r + 0] = word(2, kUnitSide, 31, 0);
        if (rem[0]) pi.edge[8 * r + 1] = word(0, kUnitSide, 0, 1);
        if (rem[5]) pi.edge[8 * r + 2] = word(5, kUnitDown, 31, 2);
        if (rem[4]) pi.edge[8 * r + 3] = word(4, kUnitDown, 0, 1);
        if (rem[6]) pi.edge[8 * r + 4] = word(6, kUnitUp, 31, 1);
        if (rem[7]) pi.edge[8 * r + 5] = word(7, kUnitUp, 0, 2);
        if (plane && rem[2]) pi.edge[8 * r + 4] = word(2, kUnitDown, 31, 2);
        if (plane && rem[0]) pi.edge[8 * r + 5] = word(0, kUnitDown, 0, 1);
        pi.rho0[r] = L.rho0;
        pi.omega[r] = L.omega;
        pi.unit0[r] = LBM_OK_IDX(q, halo_cap) ? q * 3 * kUnitWords : 0;
        const int ol = L.nx - 1 - (w << 5);
        m.slots[j] = SlotInfo{w == 0 && !(mc & 1u) ? 0 : -1, ol < 32 && !((mc >> (ol & 31)) & 1u) ? ol : -1,
                              w == 0 ? L.u_in[y] : 0.0f, L.port_scheme == LBM_PORTS_ZOU_HE,
                              (long long)y * L.pitch + (w << 5), &L, ~mc};
      }
      if (__any_sync(kFull, fluid && (inlet || outlet))) sf |= kHasPort;
      if (L.outlet_rule == LBM_OUT_NEUMANN) sf |= kNeumann;
      if ((FEAT & kFeatModels) && L.collision != LBM_COLLIDE_BGK) sf |= kSlotModel;
      flags |= sf << (16 * r);
    }
    m.src[p][0][lane] = make_uint4(off[0], off[1], off[2], off[3]);
    m.src[p][1][lane] = make_uint4(off[4], off[5], off[6], off[7]);
    m.remote[p][lane] = (uint16_t)remote;
    if (lane == 0) pi.flags = flags;
  }
  __syncthreads();
  // the canonical layout into the rows; what other blocks read of it goes out tagged epoch0
  const int parity = halo_cap * 3 * kUnitWords;
  for (int p = warp; p < n_pairs; p += n_warps) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const SlotInfo& si = m.slots[2 * p + r];
      const unsigned sf = m.pairs[p].flags >> (16 * r);
      const T* F = static_cast<const T*>(si.L->f) + si.row + lane;
      const int pl = (int)si.L->plane;
      float g[9];
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        g[i] = (si.fluid >> lane) & 1u && LBM_OK_IDX(si.row + lane + (long long)i * pl, si.L->f_elems)
                   ? P::ld(F + (long long)i * pl)
                   : 0.0f;
        m.rows[2 * p + r][i * 32 + lane] = g[i];
      }
      if (sf & kPublishes) publish(halo + parity + m.pairs[p].unit0[r] + lane, sf, lane, g, epoch0);
    }
  }
  // ---- the time steps ----
  // this warp's pairs: n_mine of them (negative: a wait gave up) from `first` on, `stride` apart
  int n_mine = n_pairs > warp ? (n_pairs - warp - 1) / n_warps + 1 : 0;
  const bool reverse = (warp >> 2) & 1;
  const int first = reverse ? warp + n_warps * (n_mine - 1) : warp, stride = reverse ? -n_warps : n_warps;
  for (int k = 0; k < n_steps; k += 2) {
    if ((k & 127) == 0) {
      if (__syncthreads_or(n_mine < 0)) break;
    } else {
      __syncthreads();
    }
#pragma unroll 1
    for (int j = 0, p = first; j < n_mine; ++j, p += stride)
      if (!many_step<T, FEAT, true>(m, p, k, n_steps - 1, mom_prev, epoch0, tag_skew, halo, parity, lane, error))
        n_mine = -1;
    __syncthreads();
#pragma unroll 1
    for (int j = 0, p = first; j < n_mine; ++j, p += stride)
      if (!many_step<T, FEAT, false>(m, p, k + 1, n_steps - 1, mom_prev, epoch0, tag_skew, halo, parity, lane, error))
        n_mine = -1;
  }
  if (__syncthreads_or(n_mine < 0)) return;  // this block stores nothing; others may have ended: the state is void
  // ---- the final state (an even number of steps) to the canonical layout ----
  for (int j = warp; j < n_own; j += n_warps) {
    const SlotInfo& si = m.slots[j];
    if (!((si.fluid >> lane) & 1u)) continue;
    T* F = static_cast<T*>(si.L->f) + si.row + lane;
    const int pl = (int)si.L->plane;
#pragma unroll
    for (int i = 0; i < 9; ++i)
      if (LBM_OK_IDX(si.row + lane + (long long)i * pl, si.L->f_elems))
        P::st(F + (long long)i * pl, m.rows[j][i * 32 + lane]);
  }
}

template <class T, int FEAT>
void* resident_kernel(int per_warp) {
  switch (per_warp) {
    case 1: return (void*)k_stream_collide_resident<T, FEAT, 1>;
    case 2: return (void*)k_stream_collide_resident<T, FEAT, 2>;
    default: return (void*)k_stream_collide_resident_many<T, FEAT>;
  }
}

template <class T>
void* resident_kernel(int features, int per_warp) {
  switch (features) {
    case 0: return resident_kernel<T, 0>(per_warp);
    case kFeatModels: return resident_kernel<T, kFeatModels>(per_warp);
    case kFeatMirror: return resident_kernel<T, kFeatMirror>(per_warp);
    case kFeatModels | kFeatMirror: return resident_kernel<T, kFeatModels | kFeatMirror>(per_warp);
    default: return nullptr;
  }
}

void* resident_kernel_for(int precision, int features, int per_warp) {
  switch (precision) {
    case LBM_F32: return resident_kernel<float>(features, per_warp);
    case LBM_BF16_SHIFTED: return resident_kernel<__nv_bfloat16>(features, per_warp);
    case LBM_F16_SHIFTED: return resident_kernel<__half>(features, per_warp);
    default: return nullptr;
  }
}

}  // namespace

size_t resident_halo_bytes(int segments) { return (size_t)2 * segments * 3 * kUnitWords * sizeof(HaloWord); }

cudaError_t launch_stream_collide_resident(int precision, int features, const LatticeView* views, const SegRef* segs,
                                           const int* n_segs, const int* seg_word_off, const int* seg_flags,
                                           const int* seg_offs, const ResidentShape& rs, void* halo, int halo_cap,
                                           unsigned epoch0, int n_steps, int mom_prev, int* error,
                                           cudaStream_t stream) {
  void* k = resident_kernel_for(precision, features, rs.per_warp);
  // under the test hook every wait expects a tag that nobody writes
  unsigned tag_skew = barrier_timeout_test() ? 1u : 0u;
  if (!k || rs.grid < 1 || rs.warps < 1 ||
      rs.warps > (rs.per_warp == 1   ? kResidentMaxWarps
                  : rs.per_warp == 2 ? kResidentMaxOwn / 2
                                     : kResidentManyWarps) ||
      rs.own > kResidentManyOwn || n_steps < 2 || (n_steps & 1) ||
      !halo || halo_cap < 1)
    return cudaErrorInvalidValue;
  const int smem = rs.per_warp == 1   ? 2 * (int)sizeof(float) * Layout<1>::kWords
                   : rs.per_warp == 2 ? 2 * (int)sizeof(float) * Layout<2>::kWords
                                      : (int)sizeof(ManyShared);
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  void* args[] = {(void*)&views, (void*)&segs, (void*)&n_segs, (void*)&seg_word_off, (void*)&seg_flags,
                  (void*)&seg_offs, (void*)&halo, (void*)&halo_cap, (void*)&epoch0, (void*)&n_steps,
                  (void*)&mom_prev, (void*)&error, (void*)&tag_skew};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // every block resident: neighbours' words always come
  attr[0].val.cooperative = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(rs.grid);
  cfg.blockDim = dim3(32 * rs.warps);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelExC(&cfg, k, args);
  if (e == cudaSuccess) count_launches(1);
  return e;
}

}  // namespace lbm
