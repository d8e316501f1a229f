// CSR-part SpMM (the AXPY row kernel of Sec. 3.3 on CUDA cores) and the deterministic sum of
// split-row partials.
//
// A group of G lanes (G divides 32) owns one work item (a CSR row or a segment of a long
// row). Each lane owns VPL 16-byte column vectors of the output row, laid out so that the G
// lanes read consecutive 16-byte pieces of a B row (coalesced 128-bit loads). The group
// reads a chunk of (col, val) pairs at once, one chunk ahead, and broadcasts them with
// shuffles; U B-row loads are kept in flight before their FMAs. Accumulation is in f64 for F64
// and in f32 otherwise. Every output row has one writer; rows split in segments write partials
// that a second kernel sums in segment order, so the result does not depend on scheduling.
#include <cstring>
#include <type_traits>

#include "device_common.cuh"
#include "loops_internal.h"

namespace loops {

namespace {

constexpr int kCsrThreads = 128;
constexpr int32_t kPastEnd = 1 << 30;  // an entry past every item's end

// The long rows of a team launch, in three classes (longest first) of one team size each. They are the
// first items (a set with teams has no cut rows), and the classes have the first blocks, in order.
constexpr int kTeamMax = 8;     // groups
constexpr int kTeamChunk = 32;  // entries
struct Teams {
  int32_t n[3], log_size[3], block_end[3];
};

// Threads of a block: a team of any size fits.
template <int G, bool TEAM>
struct CsrBlock {
  static constexpr int kThreads = TEAM && G * kTeamMax > kCsrThreads ? G * kTeamMax : kCsrThreads;
};

struct CsrKArgs {
  const int32_t* item_row;
  const int64_t* item_ptr;
  const int32_t* col;
  const void* val;
  int64_t n_items;
  const void* B;
  int64_t ldb;
  uint32_t ldb_bytes;    // vector paths only, whose launches check that it fits
  void* C;
  int64_t ldc;
  void* scratch;         // n_slots x N accumulators
  const float* col_scale;
  float inv_scale_f;
  double inv_scale_d;
  int64_t N;
  int accumulate;        // add to C (rows a BCSR part wrote first) instead of overwriting it
};

// Launches without teams do not take these: as part of CsrKArgs they changed the compiled loops of some kernels
// (200,003-node graph, N = 97, FP32: 8 % slower; small graphs 15 %).
struct CsrTeamKArgs : CsrKArgs {
  Teams team;
};
template <bool TEAMS>
using LaunchArgs = std::conditional_t<TEAMS, CsrTeamKArgs, CsrKArgs>;

template <class Tr>
__device__ __forceinline__ typename Tr::TAcc out_scale(const CsrKArgs& a, int64_t n);
template <>
__device__ __forceinline__ double out_scale<TrF64>(const CsrKArgs& a, int64_t) { return a.inv_scale_d; }
template <>
__device__ __forceinline__ float out_scale<TrF32>(const CsrKArgs& a, int64_t) { return a.inv_scale_f; }
template <>
__device__ __forceinline__ float out_scale<TrF16>(const CsrKArgs& a, int64_t n) {
  return a.col_scale ? a.col_scale[n] * a.inv_scale_f : a.inv_scale_f;
}
template <>
__device__ __forceinline__ float out_scale<TrBF16>(const CsrKArgs& a, int64_t n) {
  return a.col_scale ? a.col_scale[n] * a.inv_scale_f : a.inv_scale_f;
}

// Accumulator value of an A value in its register form (Tr::TV).
template <class Tr>
__device__ __forceinline__ typename Tr::TAcc acc_value(typename Tr::TV v) {
  if constexpr (sizeof(typename Tr::TB) == 2) {
    const unsigned short u = (unsigned short)v;
    typename Tr::TB x;
    memcpy(&x, &u, 2);
    return Tr::to_acc(x);
  } else {
    return v;
  }
}

// A chunk of an item's entries, R per lane (entry r * G + sub): columns and values, zeros past the
// item's end.
template <class Tr, int G, int R>
__device__ __forceinline__ void fetch_entries(const CsrKArgs& a, int64_t beg, int32_t len, int32_t k0, int sub,
                                              int32_t (&c)[R], typename Tr::TV (&v)[R]) {
  using TB = typename Tr::TB;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int32_t k = k0 + r * G + sub;
    c[r] = 0;
    v[r] = 0;
    if (k < len) {
      c[r] = __ldg(a.col + beg + k);
      v[r] = Tr::load_v(reinterpret_cast<const TB*>(a.val) + beg + k);
    }
  }
}

// The item of a lane group and its part of the item's entries. One group has a whole item, or in a team
// launch a long row has a team of groups that take kTeamChunk entries each in turn, whatever G, and
// whose sums meet in team_sum in one order: a row's bits do not depend on the kernel or its shape.
struct Share {
  int64_t item;
  int32_t first;     // entry
  int32_t skip;      // entries that the other groups take between two of its pieces
  int32_t log_size;  // of the team
  bool live;
};
// In a block of teams.
template <int G>
__device__ __forceinline__ Share team_share(const CsrTeamKArgs& a) {
  constexpr int kThreads = CsrBlock<G, true>::kThreads;
  const Teams& t = a.team;
  const int b = (int)blockIdx.x, group = (int)threadIdx.x / G;
  const int r = b < t.block_end[0] ? 0 : b < t.block_end[1] ? 1 : 2;
  const int ls = t.log_size[r];
  const int at = ((b - (r ? t.block_end[r - 1] : 0)) * (kThreads / G) + group) >> ls;
  const bool live = at < t.n[r];  // the last block of a class may have teams without a row
  const int before = (r > 0 ? t.n[0] : 0) + (r > 1 ? t.n[1] : 0);
  return {(int64_t)before + (live ? at : 0), live ? (group & ((1 << ls) - 1)) * kTeamChunk : kPastEnd,
          ((1 << ls) - 1) * kTeamChunk, ls, live};
}
// Elsewhere; TEAMS: in a launch that has team blocks.
template <int G, bool TEAMS>
__device__ __forceinline__ Share whole_item(const LaunchArgs<TEAMS>& a) {
  constexpr int kThreads = CsrBlock<G, TEAMS>::kThreads;
  if constexpr (TEAMS) {
    const Teams& t = a.team;
    const int64_t g = (int64_t)((int)blockIdx.x - t.block_end[2]) * (kThreads / G) + (int)threadIdx.x / G;
    return {g + t.n[0] + t.n[1] + t.n[2], 0, 0, 0, true};
  } else {
    return {((int64_t)blockIdx.x * kThreads + threadIdx.x) / G, 0, 0, 0, true};
  }
}

// First entry of the chunk after the one at k0.
template <int CH, bool TEAM>
__device__ __forceinline__ int32_t next_chunk(const Share& sh, int32_t k0) {
  static_assert(kTeamChunk % CH == 0, "chunks tile a group's piece");
  k0 += CH;
  return TEAM && k0 % kTeamChunk == 0 ? k0 + sh.skip : k0;
}

// Sum of the accumulators over a team's groups, pairs first; true in the group that holds it. All
// threads of the block are here (its teams have one size).
template <int G, class TAcc, int P, int E>
__device__ __forceinline__ bool team_sum(const Share& sh, TAcc (&acc)[P][E]) {
  __shared__ TAcc part[CsrBlock<G, true>::kThreads / 32][P * E][G];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int lanes = G << sh.log_size;
  __syncwarp();  // the groups' loops end apart
#pragma unroll
  for (int off = G; off < 32; off <<= 1) {
    if (off >= lanes) break;
#pragma unroll
    for (int i = 0; i < P * E; ++i) acc[i / E][i % E] += __shfl_xor_sync(0xffffffffu, acc[i / E][i % E], off);
  }
  for (int h = 1; h < lanes / 32; h <<= 1) {  // a warp's sums are written once and read once
    if (lane < G && (warp & (2 * h - 1)) == h) {
#pragma unroll
      for (int i = 0; i < P * E; ++i) part[warp][i][lane] = acc[i / E][i % E];
    }
    __syncthreads();
    if (lane < G && (warp & (2 * h - 1)) == 0) {
#pragma unroll
      for (int i = 0; i < P * E; ++i) acc[i / E][i % E] += part[warp + h][i][lane];
    }
  }
  return sh.live && ((int)threadIdx.x & (lanes - 1)) < G;
}

// Output of an item: its C row (scaled), or its slot of partial sums.
template <class Tr, int G, int VPL>
__device__ __forceinline__ void store_item(const CsrKArgs& a, int32_t row, int32_t n0, const bool (&ok)[VPL],
                                           const typename Tr::TAcc (&acc)[VPL][Tr::kVE]) {
  using TAcc = typename Tr::TAcc;
  using TC = typename Tr::TC;
  constexpr int VE = Tr::kVE;
  if (row >= 0) {
    TC* crow = reinterpret_cast<TC*>(a.C) + (int64_t)row * a.ldc + n0;
#pragma unroll
    for (int p = 0; p < VPL; ++p) {
      if (!ok[p]) continue;
      TC* cp = crow + p * G * VE;
      TC o[VE];
#pragma unroll
      for (int e = 0; e < VE; ++e)
        o[e] = Tr::kScaled ? (TC)(acc[p][e] * out_scale<Tr>(a, n0 + p * G * VE + e)) : (TC)acc[p][e];
      if (a.accumulate) {
#pragma unroll
        for (int e = 0; e < VE; ++e) o[e] += cp[e];
      }
      // VE outputs are 16 (F64/F32) or 32 (16-bit inputs, f32 outputs) bytes
#pragma unroll
      for (int q = 0; q < (int)(VE * sizeof(TC) / 16); ++q)
        *reinterpret_cast<uint4*>(cp + q * (16 / sizeof(TC))) =
            *reinterpret_cast<const uint4*>(&o[q * (16 / sizeof(TC))]);
    }
  } else {
    TAcc* srow = reinterpret_cast<TAcc*>(a.scratch) + (int64_t)(-1 - row) * a.N + n0;
#pragma unroll
    for (int p = 0; p < VPL; ++p) {
      if (!ok[p]) continue;
#pragma unroll
      for (int e = 0; e < VE; ++e) srow[p * G * VE + e] = acc[p][e];
    }
  }
}

// Vector path: N % VE == 0, B/C/ld aligned for 16-byte B loads and vector C stores.
//
// The formats other than FP64 are bound by the latency of the gathers of B rows (from L2, from
// DRAM where B exceeds it), so the shape is chosen for bytes in flight and few instructions per
// gathered byte. Measured on GB300 (CSR kernel alone, before -> now):
//   R-MAT 2^20, 14.3 M entries, N = 128, FP16   427 -> 328 us
//   GCN 2^18, 7.4 M entries, N = 256, FP32      503 -> 397 us
//   2^19 rows of 16 entries, N = 64, BF16       186 -> 146 us (63 % of the DRAM rate: B is
//                                               134 MB, and L2 keeps a third of its rows)
// * Blocks of 128 threads: a block holds its registers until its longest row ends, and smaller
//   ones are replaced sooner (256 threads: R-MAT 16-bit 8 % slower, the 16-entry rows 5 %; 64:
//   within 1 %). A persistent grid that strides over the items was 9 % slower.
// * Two vectors per lane with two entries in flight from 16 vectors per row on, one vector
//   with four entries below: the same bytes in flight, half the shuffles per byte. With one
//   vector R-MAT 16-bit is 14 % slower and the GCN row 4 %; with four entries and two vectors the
//   64 registers of 32 warps per SM spill.
// * FULL (the group's vectors cover the columns exactly): loads carry no predicate and no zero
//   fill; the second vector is an immediate offset from the first; a row's address is one
//   32 x 32 -> 64 bit multiply-add.
// * Columns in slices that fit L2 (64 to 512 bytes of each row at a time) were 2 to 40 % slower:
//   the entries are read once per slice, and shorter pieces cost more instructions per byte.
// FP64 is bound by the FP64 pipe: one entry at a time, so that no FMA is spent on a padded slot,
// and no entries ahead; 48 warps per SM with one vector per lane (40 registers; instances of 1 and 32 lanes
// spill 4 to 36 bytes). At 64 warps its 32 registers spill 8, and the time is the same within 2 %.
template <class Tr, int VPL>
struct CsrShape {
  static constexpr bool kF64 = std::is_same<Tr, TrF64>::value;
  static constexpr int kInFlight = kF64 ? 1 : (VPL == 1 ? 4 : 2);  // entries
  static constexpr bool kAhead = !kF64;  // load the next chunk's entries before this chunk's B rows
  static constexpr int kWarps = kF64 && VPL == 1 ? 48 : 32;  // per SM
};

template <class Tr, int G, int VPL, bool FULL, bool TEAM>
__device__ __forceinline__ void spmm_vec_item(const CsrKArgs& a, const Share& sh) {
  using TB = typename Tr::TB;
  using TAcc = typename Tr::TAcc;
  using TV = typename Tr::TV;
  constexpr int VE = Tr::kVE;
  constexpr int U = CsrShape<Tr, VPL>::kInFlight;
  constexpr bool AHEAD = CsrShape<Tr, VPL>::kAhead;
  constexpr int R = G >= 8 ? 1 : 8 / G;  // entries per lane and chunk
  constexpr int CH = G * R;
  static_assert(CH % U == 0, "load batches tile the chunk");
  const int lane = threadIdx.x & 31;
  const int sub = lane & (G - 1);
  const int64_t item = sh.item;
  if (item >= a.n_items) return;  // a group leaves as a whole
  const unsigned gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << (lane & ~(G - 1)));
  const int64_t beg = a.item_ptr[item];
  const int32_t len = (int32_t)(a.item_ptr[item + 1] - beg);  // a row that is not cut, or a segment
  const int32_t row = a.item_row[item];
  const int32_t n0 = (int32_t)blockIdx.y * (G * VPL * VE) + sub * VE;  // vector p starts at column n0 + p * G * VE
  bool ok[VPL];
#pragma unroll
  for (int p = 0; p < VPL; ++p) ok[p] = FULL || n0 + p * G * VE < (int32_t)a.N;
  TAcc acc[VPL][VE];
#pragma unroll
  for (int p = 0; p < VPL; ++p)
#pragma unroll
    for (int e = 0; e < VE; ++e) acc[p][e] = TAcc(0);

  const char* __restrict__ bl = reinterpret_cast<const char*>(a.B) + (int64_t)n0 * sizeof(TB);
  int32_t c[R], c_next[R];
  TV v[R], v_next[R];
  if (AHEAD) fetch_entries<Tr, G>(a, beg, len, sh.first, sub, c_next, v_next);
  for (int32_t k0 = sh.first, k1; k0 < len; k0 = k1) {
    k1 = next_chunk<CH, TEAM>(sh, k0);
    if (AHEAD) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        c[r] = c_next[r];
        v[r] = v_next[r];
      }
      fetch_entries<Tr, G>(a, beg, len, k1, sub, c_next, v_next);
    } else {
      fetch_entries<Tr, G>(a, beg, len, k0, sub, c, v);
    }
    const int cnt = min(len - k0, CH);  // uniform in the group
    // entries e0 .. e0 + U - 1 of the chunk; TAIL: those past its end load nothing and carry
    // zero values, so they add exact zeros
    auto batch = [&](int e0, auto tail_tag) {
      constexpr bool TAIL = decltype(tail_tag)::value;
      uint4 bv[U][VPL];
      TV av[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = e0 + u;
        const uint32_t cj = (uint32_t)__shfl_sync(gmask, R == 1 ? c[0] : c[(e / G) % R], e % G, G);
        av[u] = __shfl_sync(gmask, R == 1 ? v[0] : v[(e / G) % R], e % G, G);
        const char* brow = bl + (uint64_t)cj * a.ldb_bytes;
#pragma unroll
        for (int p = 0; p < VPL; ++p) {
          if constexpr (FULL && !TAIL) bv[u][p] = ldg16(brow + p * G * 16);
          else bv[u][p] = ldg16_if(ok[p] && (!TAIL || e < cnt), brow + p * G * 16);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int p = 0; p < VPL; ++p) fma_vec<Tr>(acc[p], bv[u][p], av[u]);
    };
    if constexpr (R == 1) {
      int e0 = 0;
      for (; e0 + U <= cnt; e0 += U) batch(e0, std::false_type());
      if (U > 1 && e0 < cnt) batch(e0, std::true_type());
    } else {  // unrolled: the entry's register index is a constant
#pragma unroll
      for (int e0 = 0; e0 < CH; e0 += U) {
        if (e0 + U <= cnt) batch(e0, std::false_type());
        else if (e0 < cnt) batch(e0, std::true_type());
      }
    }
  }
  if constexpr (TEAM) {
    if (!team_sum<G>(sh, acc)) return;
  }
  store_item<Tr, G, VPL>(a, row, n0, ok, acc);
}

template <class Tr, int G, int VPL, bool FULL, bool TEAMS>
__global__ void __launch_bounds__((CsrBlock<G, TEAMS>::kThreads), (CsrShape<Tr, VPL>::kWarps * 32 / CsrBlock<G, TEAMS>::kThreads))
    csr_spmm_vec(LaunchArgs<TEAMS> a) {
  if constexpr (TEAMS) {
    if ((int)blockIdx.x < a.team.block_end[2]) {
      spmm_vec_item<Tr, G, VPL, FULL, true>(a, team_share<G>(a));
      return;
    }
  }
  spmm_vec_item<Tr, G, VPL, FULL, false>(a, whole_item<G, TEAMS>(a));
}

// Path for any N and alignment: a group of G lanes per item, each lane with CP pieces of VW adjacent
// columns (one load of VW elements where N and B's rows allow it), G pieces apart, so that a group
// reads consecutive memory and a row of B in one pass. With loads of 2 to 8 bytes instructions
// count first: few lanes with many pieces each (G = 8 up to 64 pieces per row) share an entry's
// column, value and address over CP loads, waste few lanes on a ragged N, and let a warp take
// several items. U entries with 8 to 32 elements in flight per lane, entries one chunk ahead.
// 200,003-node graph, 4.1 M entries, N = 47, FP32: 100 us, against 280 us with one column per lane
// and the entries read per 32 columns, and 165 us with 32 lanes and two pieces.
template <int CP, int VW>
struct OddShape {
  static constexpr int kInFlight = CP * VW <= 2 ? 8 : (CP * VW <= 6 ? 4 : 2);  // entries
  // Warps per SM that team launches must allow (0: as the compiler has it): the other instances reach
  // them by themselves. FP32, N = 97 at 64 registers instead of 56: 14 % slower.
  static constexpr int kTeamWarps = CP == 8 && VW == 1 ? 36 : CP == 6 && VW == 2 ? 32 : 0;
};

// VW adjacent elements of a row of B, zeros when off
template <class TB, int VW>
__device__ __forceinline__ void load_piece(bool on, const TB* p, TB (&x)[VW]) {
#pragma unroll
  for (int w = 0; w < VW; ++w) x[w] = TB(0);
  if (!on) return;
  if constexpr (VW == 1) {
    x[0] = p[0];
  } else if constexpr (VW * sizeof(TB) == 8) {
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
    memcpy(x, &v, 8);
  } else {
    const unsigned v = __ldg(reinterpret_cast<const unsigned*>(p));
    memcpy(x, &v, 4);
  }
}

template <class Tr, int G, int CP, int VW, bool TEAM>
__device__ __forceinline__ void spmm_odd_item(const CsrKArgs& a, const Share& sh) {
  using TB = typename Tr::TB;
  using TAcc = typename Tr::TAcc;
  using TC = typename Tr::TC;
  using TV = typename Tr::TV;
  constexpr int U = OddShape<CP, VW>::kInFlight;
  static_assert(G % U == 0, "load batches tile the chunk of G entries");
  const int lane = threadIdx.x & 31;
  const int sub = lane & (G - 1);
  const int64_t item = sh.item;
  if (item >= a.n_items) return;  // a group leaves as a whole
  const unsigned gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << (lane & ~(G - 1)));
  const int64_t beg = a.item_ptr[item];
  const int32_t len = (int32_t)(a.item_ptr[item + 1] - beg);
  const int32_t row = a.item_row[item];
  const int32_t n0 = (int32_t)blockIdx.y * (G * CP * VW) + sub * VW;  // piece i starts at column n0 + i * G * VW
  bool ok[CP];
#pragma unroll
  for (int i = 0; i < CP; ++i) ok[i] = n0 + i * G * VW < (int32_t)a.N;
  const TB* __restrict__ bl = reinterpret_cast<const TB*>(a.B) + n0;
  TAcc acc[CP][VW];
#pragma unroll
  for (int i = 0; i < CP; ++i)
#pragma unroll
    for (int w = 0; w < VW; ++w) acc[i][w] = TAcc(0);
  int32_t c[1], c_next[1];
  TV v[1], v_next[1];
  fetch_entries<Tr, G>(a, beg, len, sh.first, sub, c_next, v_next);
  for (int32_t k0 = sh.first, k1; k0 < len; k0 = k1) {
    k1 = next_chunk<G, TEAM>(sh, k0);
    c[0] = c_next[0];
    v[0] = v_next[0];
    fetch_entries<Tr, G>(a, beg, len, k1, sub, c_next, v_next);
    const int cnt = min(len - k0, G);  // uniform in the group
    // entries past the chunk's end load nothing and carry zero values
    auto batch = [&](int e0, auto tail_tag) {
      constexpr bool TAIL = decltype(tail_tag)::value;
      TB bv[U][CP][VW];
      TAcc av[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int32_t cj = __shfl_sync(gmask, c[0], e0 + u, G);
        av[u] = acc_value<Tr>(__shfl_sync(gmask, v[0], e0 + u, G));
        const TB* brow = bl + (int64_t)cj * a.ldb;
#pragma unroll
        for (int i = 0; i < CP; ++i) load_piece<TB, VW>(ok[i] && (!TAIL || e0 + u < cnt), brow + i * G * VW, bv[u][i]);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int i = 0; i < CP; ++i)
#pragma unroll
          for (int w = 0; w < VW; ++w) acc[i][w] = fma(av[u], Tr::to_acc(bv[u][i][w]), acc[i][w]);
    };
    int e0 = 0;
    for (; e0 + U <= cnt; e0 += U) batch(e0, std::false_type());
    if (e0 < cnt) batch(e0, std::true_type());
  }
  if constexpr (TEAM) {
    if (!team_sum<G>(sh, acc)) return;
  }
#pragma unroll
  for (int i = 0; i < CP; ++i) {
    if (!ok[i]) continue;
#pragma unroll
    for (int w = 0; w < VW; ++w) {
      const int32_t n = n0 + i * G * VW + w;
      if (row >= 0) {
        TC* cp = reinterpret_cast<TC*>(a.C) + (int64_t)row * a.ldc + n;
        const TC o = Tr::kScaled ? (TC)(acc[i][w] * out_scale<Tr>(a, n)) : (TC)acc[i][w];
        *cp = a.accumulate ? *cp + o : o;
      } else {
        reinterpret_cast<TAcc*>(a.scratch)[(int64_t)(-1 - row) * a.N + n] = acc[i][w];
      }
    }
  }
}

template <class Tr, int G, int CP, int VW>
__global__ void __launch_bounds__(kCsrThreads) csr_spmm_odd(CsrKArgs a) {
  spmm_odd_item<Tr, G, CP, VW, false>(a, whole_item<G, false>(a));
}

template <class Tr, int G, int CP, int VW>
__global__ void __launch_bounds__((CsrBlock<G, true>::kThreads),
                                  (sizeof(typename Tr::TB) <= 4
                                       ? OddShape<CP, VW>::kTeamWarps * 32 / CsrBlock<G, true>::kThreads : 0))
    csr_spmm_odd_teams(CsrTeamKArgs a) {
  if ((int)blockIdx.x < a.team.block_end[2]) spmm_odd_item<Tr, G, CP, VW, true>(a, team_share<G>(a));
  else spmm_odd_item<Tr, G, CP, VW, false>(a, whole_item<G, true>(a));
}

// C[row, n] = scale_n * sum over the row's segments, in segment order, eight partials in flight.
// Threads of a block cover columns x split rows, so that narrow rows fill the block.
constexpr int kReduceThreads = 128;
template <class Tr>
__global__ void __launch_bounds__(kReduceThreads) split_reduce(const int32_t* __restrict__ split_row,
                                                               const int32_t* __restrict__ slot_ptr,
                                                               int64_t n_split, int log_tx, CsrKArgs a) {
  using TAcc = typename Tr::TAcc;
  using TC = typename Tr::TC;
  const int64_t s = (int64_t)blockIdx.x * (kReduceThreads >> log_tx) + (threadIdx.x >> log_tx);
  const int64_t n = ((int64_t)blockIdx.y << log_tx) + (threadIdx.x & ((1 << log_tx) - 1));
  if (s >= n_split || n >= a.N) return;
  const int32_t row = split_row[s];
  const int32_t s0 = slot_ptr[s], s1 = slot_ptr[s + 1];
  const TAcc* sc = reinterpret_cast<const TAcc*>(a.scratch) + n;
  TAcc acc = TAcc(0);
  int32_t q = s0;
  for (; q + 8 <= s1; q += 8) {
    TAcc x[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = sc[(int64_t)(q + i) * a.N];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc += x[i];
  }
  for (; q < s1; ++q) acc += sc[(int64_t)q * a.N];
  TC* cp = reinterpret_cast<TC*>(a.C) + (int64_t)row * a.ldc + n;
  const TC v = Tr::kScaled ? (TC)(acc * out_scale<Tr>(a, n)) : (TC)acc;
  *cp = a.accumulate ? *cp + v : v;
}

// Backward of C = A . B in one pass over A^T: dB[j, :] = sum_i a_ij dC[i, :] and
// dvals[a_ij] = <dC[i, :], B[j, :]> read the same rows of dC, so the group that owns row j of A^T
// keeps B[j, :] (times the column weights) beside its accumulators and takes both from each row
// it gathers. The gathers of dC rows bound it as they bound the SpMM and the SDDMM that it
// replaces, and are made once instead of twice. Measured on GB300 (dB and dvals together):
//   GCN 2^18, 7.4 M entries, N = 256, FP32      930 -> 566 us
//   the same graph, N = 128, BF16               369 -> 265 us (about 4 us more with the check of the weights)
// The shape is the SpMM's: 128 threads, entries one chunk ahead, no predicates where the group
// covers the columns. Bytes in flight and warps decide: FP32 takes four entries in flight at 32
// warps per SM (two: 10 % slower step; 24 warps: 5 %), the 16-bit formats two vectors per lane
// from 16 on with two entries at 28 warps (one vector: 4 % slower step; 32 warps spill: 11 %). Other instances
// spill: partly covered FP32 with two vectors 72 to 92 bytes, one lane per row (N of one vector) 130 to 230. Against
// the two kernels they are still ahead: 100,000 nodes, 1.7 M entries, FP32 N = 4 726 -> 53 us, 36 179 -> 57, 136
// 340 -> 176; BF16 N = 8 758 -> 74; FP64 N = 2 333 -> 69, 72 935 -> 923.
// The input entry of a dot product (`src`) is loaded with its column and value: loaded where
// dvals is stored, it stalled every batch (20 % slower).
template <class Tr, int VPL>
struct BwdShape {
  static constexpr bool kF64 = std::is_same<Tr, TrF64>::value, k16 = Tr::kVE == 8;
  static constexpr int kInFlight = VPL == 2 && (k16 || kF64) ? 2 : 4;  // entries
  static constexpr int kWarps = kF64 ? (VPL == 2 ? 16 : 24) : (k16 && VPL == 2 ? 28 : 32);
};

struct BwdKArgs {
  const void* B;             // rows of B, one per row of A^T
  int64_t ldb;
  void* dvals;               // input order
  const int32_t* src;        // input entry of every stored entry
  const int32_t* split_row;  // rows cut into segments, and their slots
  const int32_t* split_slot_ptr;
  int64_t n_split;
  const float* dc_scale;     // optional column scales of dC and B (16-bit dtypes)
  const float* b_scale;
};

// The dot products of an item's entries with the column weights on dC's side, for the rows j where a
// non-zero element of B[j, :] times its weight leaves binary32's normal range: the loop of
// csr_backward_vec would multiply a zero of dC by infinity there, or lose the element. Plain loops,
// out of line: such weights are far from what a per-column scaling gives.
template <class Tr, int G, bool TEAM>
__device__ __noinline__ void weighted_dots(const int32_t* col, const int32_t* src, int32_t len, const Share sh, int sub,
                                           unsigned gmask, const typename Tr::TB* dC, int64_t lddc,
                                           const typename Tr::TB* Brow, const float* dc_scale, const float* b_scale,
                                           int64_t N, typename Tr::TC* dvals) {
  __syncwarp(gmask);  // the caller's stores to dvals come before those that replace them
  for (int32_t k = sh.first; k < len; k = next_chunk<1, TEAM>(sh, k)) {
    const typename Tr::TB* drow = dC + (int64_t)col[k] * lddc;
    float s = 0.f;
    for (int64_t n = sub; n < N; n += G) {
      const float weight = (dc_scale ? dc_scale[n] : 1.f) * (b_scale ? b_scale[n] : 1.f);
      s = fma(Tr::to_acc(drow[n]) * weight, Tr::to_acc(Brow[n]), s);
    }
    for (int off = G / 2; off > 0; off >>= 1) s += __shfl_xor_sync(gmask, s, off, G);
    if (sub == 0) dvals[src[k]] = s;
  }
}

template <class Tr, int G, int VPL, bool FULL, bool TEAM>
__device__ __forceinline__ void backward_item(const CsrKArgs& a, const BwdKArgs& w, const Share& sh) {
  using TB = typename Tr::TB;
  using TAcc = typename Tr::TAcc;
  using TC = typename Tr::TC;
  using TV = typename Tr::TV;
  constexpr int VE = Tr::kVE;
  constexpr int U = BwdShape<Tr, VPL>::kInFlight;
  constexpr int R = G >= 8 ? 1 : 8 / G;  // entries per lane and chunk
  constexpr int CH = G * R;
  static_assert(CH % U == 0, "load batches tile the chunk");
  const int lane = threadIdx.x & 31;
  const int sub = lane & (G - 1);
  const int64_t item = sh.item;
  if (item >= a.n_items) return;  // a group leaves as a whole
  const unsigned gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << (lane & ~(G - 1)));
  const int64_t beg = a.item_ptr[item];
  const int32_t len = (int32_t)(a.item_ptr[item + 1] - beg);
  const int32_t row = a.item_row[item];
  auto fetch = [&](int32_t k0, int32_t (&c)[R], TV (&v)[R], int32_t (&x)[R]) {
    fetch_entries<Tr, G>(a, beg, len, k0, sub, c, v);
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = k0 + r * G + sub < len ? __ldg(w.src + beg + k0 + r * G + sub) : 0;
  };
  int32_t c_next[R], x_next[R];
  TV v_next[R];
  fetch(sh.first, c_next, v_next, x_next);
  int32_t j = row;
  if (row < 0) {  // a segment: the split row that holds its slot
    const int32_t slot = -1 - row;
    int64_t lo = 0, hi = w.n_split;  // split_slot_ptr[lo] <= slot < split_slot_ptr[hi]
    while (hi - lo > 1) {
      const int64_t mid = (lo + hi) >> 1;
      if (w.split_slot_ptr[mid] <= slot) lo = mid; else hi = mid;
    }
    j = w.split_row[lo];
  }
  const int32_t n0 = sub * VE;
  bool ok[VPL];
  TAcc acc[VPL][VE], bj[VPL][VE];
  bool lossy = false;  // a non-zero element of B[j, :] leaves binary32's normal range with its weight
#pragma unroll
  for (int p = 0; p < VPL; ++p) {
    const int32_t n = n0 + p * G * VE;
    ok[p] = FULL || n < (int32_t)a.N;
    unpack16<Tr>(ldg16_if(ok[p], reinterpret_cast<const TB*>(w.B) + (int64_t)j * w.ldb + n), bj[p]);
    if constexpr (Tr::kScaled) {
      if (ok[p]) {
        float b[VE], lo = 1.f, hi = 0.f;
#pragma unroll
        for (int e = 0; e < VE; ++e) {
          b[e] = bj[p][e];
          bj[p][e] *= (w.dc_scale ? w.dc_scale[n + e] : 1.f) * (w.b_scale ? w.b_scale[n + e] : 1.f);
          lo = fminf(lo, fabsf(bj[p][e]));
          hi = fmaxf(hi, fabsf(bj[p][e]));
        }
        lossy = lossy || hi > 0x1.fffffep127f;
        if (lo < 0x1p-126f) {  // a zero of B, or an element that the product took there
#pragma unroll
          for (int e = 0; e < VE; ++e) lossy |= (b[e] != 0.f) & (fabsf(bj[p][e]) < 0x1p-126f);
        }
      }
    }
#pragma unroll
    for (int e = 0; e < VE; ++e) acc[p][e] = TAcc(0);
  }
  const char* __restrict__ dl = reinterpret_cast<const char*>(a.B) + (int64_t)n0 * sizeof(TB);
  TC* __restrict__ dvals = reinterpret_cast<TC*>(w.dvals);
  for (int32_t k0 = sh.first, k1; k0 < len; k0 = k1) {
    k1 = next_chunk<CH, TEAM>(sh, k0);
    int32_t c[R], x[R];
    TV v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      c[r] = c_next[r];
      v[r] = v_next[r];
      x[r] = x_next[r];
    }
    fetch(k1, c_next, v_next, x_next);
    const int cnt = min(len - k0, CH);  // uniform in the group
    // entries e0 .. e0 + U - 1 of the chunk; TAIL: those past its end load nothing, carry zero
    // values and are not stored
    auto batch = [&](int e0, auto tail_tag) {
      constexpr bool TAIL = decltype(tail_tag)::value;
      uint4 dv[U][VPL];
      TV av[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int e = e0 + u;
        const uint32_t i = (uint32_t)__shfl_sync(gmask, R == 1 ? c[0] : c[(e / G) % R], e % G, G);
        av[u] = __shfl_sync(gmask, R == 1 ? v[0] : v[(e / G) % R], e % G, G);
        const char* drow = dl + (uint64_t)i * a.ldb_bytes;
#pragma unroll
        for (int p = 0; p < VPL; ++p) {
          if constexpr (FULL && !TAIL) dv[u][p] = ldg16(drow + p * G * 16);
          else dv[u][p] = ldg16_if(ok[p] && (!TAIL || e < cnt), drow + p * G * 16);
        }
      }
      TAcc s[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        s[u] = TAcc(0);
#pragma unroll
        for (int p = 0; p < VPL; ++p) {
          TAcc d[VE];
          unpack16<Tr>(dv[u][p], d);
#pragma unroll
          for (int e = 0; e < VE; ++e) s[u] = fma(bj[p][e], d[e], s[u]);
          fma_vec<Tr>(acc[p], dv[u][p], av[u]);
        }
      }
      // sums over the group in a fixed order. With at least U lanes a lane keeps half of the
      // entries at each of the first steps, so that 1 / U of the group ends with one entry's sum
      if constexpr (G >= U) {
        TAcc t;
        int mine;
        if constexpr (U == 4) {
          const bool h1 = (sub & (G / 2)) != 0, h2 = (sub & (G / 4)) != 0;
          TAcc t0 = h1 ? s[2] : s[0], t1 = h1 ? s[3] : s[1];
          t0 += __shfl_xor_sync(gmask, h1 ? s[0] : s[2], G / 2, G);
          t1 += __shfl_xor_sync(gmask, h1 ? s[1] : s[3], G / 2, G);
          t = h2 ? t1 : t0;
          t += __shfl_xor_sync(gmask, h2 ? t0 : t1, G / 4, G);
          mine = e0 + (h1 ? 2 : 0) + (h2 ? 1 : 0);
        } else {
          const bool h1 = (sub & (G / 2)) != 0;
          t = h1 ? s[1] : s[0];
          t += __shfl_xor_sync(gmask, h1 ? s[0] : s[1], G / 2, G);
          mine = e0 + (h1 ? 1 : 0);
        }
#pragma unroll
        for (int off = G / U / 2; off > 0; off >>= 1) t += __shfl_xor_sync(gmask, t, off, G);
        const int32_t at = __shfl_sync(gmask, R == 1 ? x[0] : x[(e0 / G) % R], mine % G, G);
        if ((sub & (G / U - 1)) == 0 && (!TAIL || mine < cnt)) dvals[at] = (TC)t;
      } else {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          TAcc t = s[u];
#pragma unroll
          for (int off = G / 2; off > 0; off >>= 1) t += __shfl_xor_sync(gmask, t, off, G);
          const int32_t at = __shfl_sync(gmask, x[((e0 + u) / G) % R], (e0 + u) % G, G);
          if (sub == 0 && (!TAIL || e0 + u < cnt)) dvals[at] = (TC)t;
        }
      }
    };
    if constexpr (R == 1) {
      int e0 = 0;
      for (; e0 + U <= cnt; e0 += U) batch(e0, std::false_type());
      if (e0 < cnt) batch(e0, std::true_type());
    } else {  // unrolled: the entry's register index is a constant
#pragma unroll
      for (int e0 = 0; e0 < CH; e0 += U) {
        if (e0 + U <= cnt) batch(e0, std::false_type());
        else if (e0 < cnt) batch(e0, std::true_type());
      }
    }
  }
  bool holds = true;
  if constexpr (TEAM) holds = team_sum<G>(sh, acc);
  if (holds) store_item<Tr, G, VPL>(a, row, n0, ok, acc);
  // after the accumulators' last use, so that none is live across the call
  if constexpr (Tr::kScaled) {
    if (__any_sync(gmask, lossy))
      weighted_dots<Tr, G, TEAM>(a.col + beg, w.src + beg, len, sh, sub, gmask, reinterpret_cast<const TB*>(a.B), a.ldb,
                                 reinterpret_cast<const TB*>(w.B) + (int64_t)j * w.ldb, w.dc_scale, w.b_scale, a.N,
                                 dvals);
  }
}

template <class Tr, int G, int VPL, bool FULL, bool TEAMS>
__global__ void __launch_bounds__((CsrBlock<G, TEAMS>::kThreads), (BwdShape<Tr, VPL>::kWarps * 32 / CsrBlock<G, TEAMS>::kThreads))
    csr_backward_vec(LaunchArgs<TEAMS> a, BwdKArgs w) {
  if constexpr (TEAMS) {
    if ((int)blockIdx.x < a.team.block_end[2]) {
      backward_item<Tr, G, VPL, FULL, true>(a, w, team_share<G>(a));
      return;
    }
  }
  backward_item<Tr, G, VPL, FULL, false>(a, w, whole_item<G, TEAMS>(a));
}

inline int next_pow2(int64_t x) {
  int p = 1;
  while (p < x && p < 32) p <<= 1;
  return p;
}

// Launches one of the three item kernels (`kernel` takes whether there are teams) over its items and
// `chunks` column chunks.
template <int G, class K>
cudaError_t launch_items(const CsrKArgs& args, const CsrDev& d, int64_t chunks, K kernel) {
  const int64_t team_rows = d.n_long[0] + d.n_long[1] + d.n_long[2];
  auto blocks_of = [](int64_t groups, int threads) { return (groups * G + threads - 1) / threads; };
  if (team_rows == 0) {
    constexpr int T = CsrBlock<G, false>::kThreads;
    kernel(args, dim3((unsigned)blocks_of(args.n_items, T), (unsigned)chunks), T, std::false_type());
    return cudaGetLastError();
  }
  constexpr int T = CsrBlock<G, true>::kThreads;
  CsrTeamKArgs a;
  static_cast<CsrKArgs&>(a) = args;
  Teams& t = a.team;
  int64_t blocks = 0;
  for (int r = 0; r < 3; ++r) {
    t.n[r] = (int32_t)d.n_long[r];
    t.log_size[r] = long_class_log_team(r, d.team_len);
    blocks += blocks_of(d.n_long[r] << t.log_size[r], T);
    t.block_end[r] = (int32_t)blocks;
  }
  blocks += blocks_of(a.n_items - team_rows, T);
  kernel(a, dim3((unsigned)blocks, (unsigned)chunks), T, std::true_type());
  return cudaGetLastError();
}

template <class Tr, int G, int VPL>
cudaError_t launch_vec_g(const CsrKArgs& a, const CsrDev& d, cudaStream_t s) {
  constexpr int64_t per_chunk = (int64_t)G * VPL * Tr::kVE;
  return launch_items<G>(a, d, (a.N + per_chunk - 1) / per_chunk, [&](const auto& k, dim3 grid, int threads, auto team) {
    constexpr bool T = decltype(team)::value;
    if (k.N % per_chunk == 0) csr_spmm_vec<Tr, G, VPL, true, T><<<grid, threads, 0, s>>>(k);
    else csr_spmm_vec<Tr, G, VPL, false, T><<<grid, threads, 0, s>>>(k);
  });
}

template <class Tr, int VW>
cudaError_t launch_odd_vw(const CsrKArgs& a, const CsrDev& d, cudaStream_t s) {
  const int64_t pieces = a.N / VW;
  auto go = [&](auto g_tag, auto cp_tag) {
    constexpr int G = decltype(g_tag)::value, CP = decltype(cp_tag)::value;
    return launch_items<G>(a, d, (pieces + G * CP - 1) / (G * CP), [&](const auto& k, dim3 grid, int threads, auto team) {
      if constexpr (decltype(team)::value) csr_spmm_odd_teams<Tr, G, CP, VW><<<grid, threads, 0, s>>>(k);
      else csr_spmm_odd<Tr, G, CP, VW><<<grid, threads, 0, s>>>(k);
    });
  };
  using std::integral_constant;
  using G8 = integral_constant<int, 8>;
  if (pieces <= 8) return go(G8(), integral_constant<int, 1>());
  if (pieces <= 16) return go(G8(), integral_constant<int, 2>());
  if (pieces <= 24) return go(G8(), integral_constant<int, 3>());
  if (pieces <= 32) return go(G8(), integral_constant<int, 4>());
  if (pieces <= 48) return go(G8(), integral_constant<int, 6>());
  if (pieces <= 64) return go(G8(), integral_constant<int, 8>());
  if (pieces <= 96) return go(integral_constant<int, 16>(), integral_constant<int, 6>());
  if (pieces <= 128) return go(integral_constant<int, 16>(), integral_constant<int, 8>());
  return go(integral_constant<int, 32>(), integral_constant<int, 6>());
}

// Two columns per load where they divide N and every row of B keeps the load aligned.
template <class Tr>
cudaError_t launch_odd(const CsrKArgs& a, const CsrDev& d, cudaStream_t s) {
  constexpr int64_t eb = sizeof(typename Tr::TB);
  if constexpr (eb <= 4) {
    if (a.N % 2 == 0 && a.ldb % 2 == 0 && (uintptr_t)a.B % (2 * eb) == 0) return launch_odd_vw<Tr, 2>(a, d, s);
  }
  return launch_odd_vw<Tr, 1>(a, d, s);
}

CsrKArgs csr_args(const loops_plan_s* p, const CsrDev& d, const DenseArgs& da, bool accumulate) {
  CsrKArgs a;
  a.accumulate = accumulate ? 1 : 0;
  a.item_row = d.item_row;
  a.item_ptr = d.item_ptr;
  a.col = d.col;
  a.val = d.val;
  a.n_items = d.n_items;
  a.B = da.B;
  a.ldb = da.ldb;
  a.ldb_bytes = (uint32_t)(da.ldb * dense_elem_bytes(p->dtype));
  a.C = da.C;
  a.ldc = da.ldc;
  a.scratch = d.scratch;
  a.col_scale = da.col_scale;
  a.inv_scale_f = da.inv_scale_f;
  a.inv_scale_d = da.inv_scale_d;
  a.N = da.N;
  return a;
}

template <class Tr>
cudaError_t launch_split_reduce(const CsrDev& d, const CsrKArgs& a, cudaStream_t s) {
  if (d.n_split == 0) return cudaSuccess;
  int log_tx = 0;  // threads along the columns: a power of two that covers them, up to the block
  while ((1 << log_tx) < kReduceThreads && (1 << log_tx) < a.N) ++log_tx;
  const int rows = kReduceThreads >> log_tx;
  const dim3 grid((unsigned)((d.n_split + rows - 1) / rows), (unsigned)((a.N + (1 << log_tx) - 1) >> log_tx));
  split_reduce<Tr><<<grid, kReduceThreads, 0, s>>>(d.split_row, d.split_slot_ptr, d.n_split, log_tx, a);
  return cudaGetLastError();
}

template <class Tr>
cudaError_t launch_csr_t(const loops_plan_s* p, const CsrDev& d, const DenseArgs& da, bool accumulate,
                         cudaStream_t s) {
  const CsrKArgs a = csr_args(p, d, da, accumulate);
  using TB = typename Tr::TB;
  using TC = typename Tr::TC;
  constexpr int VE = Tr::kVE;
  const bool vec = (a.N % VE == 0) && ((uintptr_t)a.B % 16 == 0) && ((uintptr_t)a.C % 16 == 0) &&
                   ((a.ldb * (int64_t)sizeof(TB)) % 16 == 0) && ((a.ldc * (int64_t)sizeof(TC)) % 16 == 0) &&
                   a.ldb * (int64_t)sizeof(TB) <= (int64_t)UINT32_MAX;  // row strides of B in 32 bits
  cudaError_t e = cudaSuccess;
  if (a.n_items > 0) {
    if (vec) {
      const int64_t nvec = a.N / VE;
      // lanes per item: the 16-byte vectors of a row, two per lane from 16 vectors on (the
      // reasons stand at the kernel); the plan's csr_vpl, when the autotuner set it, overrides this
      const bool lv = p->csr_vpl == 2 ? nvec >= 2 : p->csr_vpl == 1 ? false : (!std::is_same<Tr, TrF64>::value && nvec >= 16);
      const int64_t nv = lv ? (nvec + 1) / 2 : nvec;
      const int G = next_pow2(nv);
      const bool two = lv || nvec > 32;
      switch (G) {
        case 1: e = two ? launch_vec_g<Tr, 1, 2>(a, d, s) : launch_vec_g<Tr, 1, 1>(a, d, s); break;
        case 2: e = two ? launch_vec_g<Tr, 2, 2>(a, d, s) : launch_vec_g<Tr, 2, 1>(a, d, s); break;
        case 4: e = two ? launch_vec_g<Tr, 4, 2>(a, d, s) : launch_vec_g<Tr, 4, 1>(a, d, s); break;
        case 8: e = two ? launch_vec_g<Tr, 8, 2>(a, d, s) : launch_vec_g<Tr, 8, 1>(a, d, s); break;
        case 16: e = two ? launch_vec_g<Tr, 16, 2>(a, d, s) : launch_vec_g<Tr, 16, 1>(a, d, s); break;
        default: e = two ? launch_vec_g<Tr, 32, 2>(a, d, s) : launch_vec_g<Tr, 32, 1>(a, d, s); break;
      }
    } else {
      e = launch_odd<Tr>(a, d, s);
    }
  }
  if (e == cudaSuccess) e = launch_split_reduce<Tr>(d, a, s);
  return e;
}

template <class Tr>
cudaError_t launch_csr_backward_t(const CsrDev& d, const CsrKArgs& a, const BwdKArgs& w, cudaStream_t s) {
  const int64_t nvec = a.N / Tr::kVE;
  auto go = [&](auto g_tag, auto p_tag) {
    constexpr int G = decltype(g_tag)::value;
    constexpr int VPL = decltype(p_tag)::value;
    return launch_items<G>(a, d, 1, [&](const auto& k, dim3 grid, int threads, auto team) {
      constexpr bool T = decltype(team)::value;
      if (k.N % (G * VPL * Tr::kVE) == 0) csr_backward_vec<Tr, G, VPL, true, T><<<grid, threads, 0, s>>>(k, w);
      else csr_backward_vec<Tr, G, VPL, false, T><<<grid, threads, 0, s>>>(k, w);
    });
  };
  using One = std::integral_constant<int, 1>;
  using Two = std::integral_constant<int, 2>;
  cudaError_t e;
  // two vectors per lane: 16-bit from 16 vectors on, the others where 32 lanes need them
  if (nvec >= (Tr::kVE == 8 ? 16 : 33)) {
    switch (next_pow2((nvec + 1) / 2)) {
      case 8: e = go(std::integral_constant<int, 8>(), Two()); break;
      case 16: e = go(std::integral_constant<int, 16>(), Two()); break;
      default: e = go(std::integral_constant<int, 32>(), Two()); break;
    }
  } else {
    switch (next_pow2(nvec)) {
      case 1: e = go(std::integral_constant<int, 1>(), One()); break;
      case 2: e = go(std::integral_constant<int, 2>(), One()); break;
      case 4: e = go(std::integral_constant<int, 4>(), One()); break;
      case 8: e = go(std::integral_constant<int, 8>(), One()); break;
      case 16: e = go(std::integral_constant<int, 16>(), One()); break;
      default: e = go(std::integral_constant<int, 32>(), One()); break;
    }
  }
  return e == cudaSuccess ? launch_split_reduce<Tr>(d, a, s) : e;
}

}  // namespace

bool csr_backward_applies(const loops_plan_s* p, const void* dC, int64_t lddc, const void* B, int64_t ldb,
                          const void* dB, int64_t lddb) {
  const loops_plan_s* t = p->transposed;
  const int64_t eb = dense_elem_bytes(p->dtype), ec = out_elem_bytes(p->dtype), ve = 16 / eb;
  if (t->dev.bcsr.n_rb > 0 || t->dev.csr_acc.n_items > 0 || !t->has_vmap || t->vmap.wide ||
      t->vmap.n_csr != p->nnz)
    return false;
  return p->N > 0 && p->N % ve == 0 && p->N / ve <= 64 && (uintptr_t)dC % 16 == 0 && (uintptr_t)B % 16 == 0 &&
         (uintptr_t)dB % 16 == 0 && (lddc * eb) % 16 == 0 && (ldb * eb) % 16 == 0 && (lddb * ec) % 16 == 0 &&
         lddc * eb <= (int64_t)UINT32_MAX;
}

cudaError_t launch_csr_backward(const loops_plan_s* p, const DenseArgs& da, const void* B, int64_t ldb, void* dvals,
                                const float* b_scale, cudaStream_t s) {
  const loops_plan_s* t = p->transposed;
  const CsrDev& d = t->dev.csr;
  if (d.n_items == 0) return cudaSuccess;
  const CsrKArgs a = csr_args(p, d, da, false);
  const BwdKArgs w{B, ldb, dvals, (const int32_t*)t->vmap.csr_src, d.split_row, d.split_slot_ptr, d.n_split,
                   da.col_scale, b_scale};
  switch (p->dtype) {
    case LOOPS_F64: return launch_csr_backward_t<TrF64>(d, a, w, s);
    case LOOPS_F32: return launch_csr_backward_t<TrF32>(d, a, w, s);
    case LOOPS_F16: return launch_csr_backward_t<TrF16>(d, a, w, s);
    case LOOPS_BF16: return launch_csr_backward_t<TrBF16>(d, a, w, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_csr(const loops_plan_s* p, const CsrDev& d, const DenseArgs& a, bool accumulate,
                       cudaStream_t s) {
  switch (p->dtype) {
    case LOOPS_F64: return launch_csr_t<TrF64>(p, d, a, accumulate, s);
    case LOOPS_F32: return launch_csr_t<TrF32>(p, d, a, accumulate, s);
    case LOOPS_F16: return launch_csr_t<TrF16>(p, d, a, accumulate, s);
    case LOOPS_BF16: return launch_csr_t<TrBF16>(p, d, a, accumulate, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace loops
