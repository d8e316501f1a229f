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
#include <type_traits>

#include "device_common.cuh"
#include "loops_internal.h"

namespace loops {

namespace {

struct CsrKArgs {
  const int32_t* item_row;
  const int64_t* item_ptr;
  const int32_t* col;
  const void* val;
  int64_t n_items;
  const void* B;
  int64_t ldb;
  void* C;
  int64_t ldc;
  void* scratch;         // n_slots x N accumulators
  const float* col_scale;
  float inv_scale_f;
  double inv_scale_d;
  int64_t N;
  int accumulate;        // add to C (rows a BCSR part wrote first) instead of overwriting it
};

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
// and no entries ahead; 48 warps per SM with one vector per lane (at 64 its 32 registers spill).
constexpr int kCsrThreads = 128;

template <class Tr, int VPL>
struct CsrShape {
  static constexpr bool kF64 = std::is_same<Tr, TrF64>::value;
  static constexpr int kInFlight = kF64 ? 1 : (VPL == 1 ? 4 : 2);  // entries
  static constexpr bool kAhead = !kF64;  // load the next chunk's entries before this chunk's B rows
  static constexpr int kMinBlocks = (kF64 && VPL == 1 ? 48 : 32) * 32 / kCsrThreads;
};

template <class Tr, int G, int VPL, bool FULL>
__global__ void __launch_bounds__(kCsrThreads, (CsrShape<Tr, VPL>::kMinBlocks)) csr_spmm_vec(CsrKArgs a) {
  using TB = typename Tr::TB;
  using TAcc = typename Tr::TAcc;
  using TC = typename Tr::TC;
  using TV = typename Tr::TV;
  constexpr int VE = Tr::kVE;
  constexpr int U = CsrShape<Tr, VPL>::kInFlight;
  constexpr bool AHEAD = CsrShape<Tr, VPL>::kAhead;
  constexpr int R = G >= 8 ? 1 : 8 / G;  // entries per lane and chunk
  constexpr int CH = G * R;
  static_assert(CH % U == 0, "load batches tile the chunk");
  const int lane = threadIdx.x & 31;
  const int sub = lane & (G - 1);
  const int64_t item = ((int64_t)blockIdx.x * kCsrThreads + threadIdx.x) / G;
  if (item >= a.n_items) return;  // a group leaves as a whole
  const unsigned gmask = (G == 32) ? 0xffffffffu : (((1u << G) - 1u) << (lane & ~(G - 1)));
  const int64_t beg = a.item_ptr[item];
  const int32_t len = (int32_t)(a.item_ptr[item + 1] - beg);  // at most split_len
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
  const uint32_t ldb_bytes = (uint32_t)(a.ldb * (int64_t)sizeof(TB));  // the launch checks that it fits
  auto fetch = [&](int32_t k0, int32_t (&c)[R], TV (&v)[R]) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int32_t k = k0 + r * G + sub;
      c[r] = 0;
      v[r] = TV(0);
      if (k < len) {
        c[r] = __ldg(a.col + beg + k);
        v[r] = Tr::load_v(reinterpret_cast<const TB*>(a.val) + beg + k);
      }
    }
  };
  int32_t c[R], c_next[R];
  TV v[R], v_next[R];
  if (AHEAD) fetch(0, c_next, v_next);
  for (int32_t k0 = 0; k0 < len; k0 += CH) {
    if (AHEAD) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        c[r] = c_next[r];
        v[r] = v_next[r];
      }
      fetch(k0 + CH, c_next, v_next);
    } else {
      fetch(k0, c, v);
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
        const char* brow = bl + (uint64_t)cj * ldb_bytes;
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

// Scalar path for any N and alignment: 32 lanes per item, one column per lane per pass.
template <class Tr, int U>
__global__ void __launch_bounds__(256) csr_spmm_scalar(CsrKArgs a) {
  using TB = typename Tr::TB;
  using TAcc = typename Tr::TAcc;
  using TC = typename Tr::TC;
  const int lane = threadIdx.x & 31;
  const int64_t item = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / 32;
  if (item >= a.n_items) return;
  const int64_t beg = a.item_ptr[item];
  const int64_t end = a.item_ptr[item + 1];
  const int32_t row = a.item_row[item];
  const int64_t n = (int64_t)blockIdx.y * 32 + lane;
  const bool colok = n < a.N;
  const TB* __restrict__ Bp = reinterpret_cast<const TB*>(a.B);
  const TB* __restrict__ vals = reinterpret_cast<const TB*>(a.val);
  TAcc acc = TAcc(0);
  for (int64_t k0 = beg; k0 < end; k0 += 32) {
    const int64_t k = k0 + lane;
    int32_t c = 0;
    TAcc v = TAcc(0);
    if (k < end) {
      c = __ldg(a.col + k);
      v = Tr::to_acc(vals[k]);
    }
    const int cnt = (int)(end - k0 < 32 ? end - k0 : 32);
    for (int j0 = 0; j0 < cnt; j0 += U) {
      TAcc bv[U], av[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int j = j0 + u;
        const int cj = __shfl_sync(0xffffffffu, c, j & 31);
        av[u] = __shfl_sync(0xffffffffu, v, j & 31);
        const bool ok = j < cnt && colok;
        bv[u] = ok ? Tr::to_acc(Bp[(int64_t)cj * a.ldb + n]) : TAcc(0);
        if (j >= cnt) av[u] = TAcc(0);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) acc = fma(av[u], bv[u], acc);
    }
  }
  if (!colok) return;
  if (row >= 0) {
    TC* cp = reinterpret_cast<TC*>(a.C) + (int64_t)row * a.ldc + n;
    const TC v = Tr::kScaled ? (TC)(acc * out_scale<Tr>(a, n)) : (TC)acc;
    *cp = a.accumulate ? *cp + v : v;
  } else {
    reinterpret_cast<TAcc*>(a.scratch)[(int64_t)(-1 - row) * a.N + n] = acc;
  }
}

// C[row, n] = scale_n * sum over the row's segments, in segment order.
template <class Tr>
__global__ void __launch_bounds__(256) split_reduce(const int32_t* __restrict__ split_row,
                                                    const int32_t* __restrict__ slot_ptr,
                                                    int64_t n_split, CsrKArgs a) {
  using TAcc = typename Tr::TAcc;
  using TC = typename Tr::TC;
  const int64_t s = blockIdx.x;
  if (s >= n_split) return;
  const int32_t row = split_row[s];
  const int32_t s0 = slot_ptr[s], s1 = slot_ptr[s + 1];
  const TAcc* sc = reinterpret_cast<const TAcc*>(a.scratch);
  for (int64_t n = (int64_t)blockIdx.y * blockDim.x + threadIdx.x; n < a.N; n += (int64_t)gridDim.y * blockDim.x) {
    TAcc acc = TAcc(0);
    for (int32_t q = s0; q < s1; ++q) acc += sc[(int64_t)q * a.N + n];
    TC* cp = reinterpret_cast<TC*>(a.C) + (int64_t)row * a.ldc + n;
    const TC v = Tr::kScaled ? (TC)(acc * out_scale<Tr>(a, n)) : (TC)acc;
    *cp = a.accumulate ? *cp + v : v;
  }
}

inline int next_pow2(int64_t x) {
  int p = 1;
  while (p < x && p < 32) p <<= 1;
  return p;
}

template <class Tr, int G, int VPL>
cudaError_t launch_vec_g(const CsrKArgs& a, cudaStream_t s) {
  constexpr int64_t per_chunk = (int64_t)G * VPL * Tr::kVE;
  const dim3 grid((unsigned)((a.n_items * G + kCsrThreads - 1) / kCsrThreads),
                  (unsigned)((a.N + per_chunk - 1) / per_chunk));
  if (a.N % per_chunk == 0) csr_spmm_vec<Tr, G, VPL, true><<<grid, kCsrThreads, 0, s>>>(a);
  else csr_spmm_vec<Tr, G, VPL, false><<<grid, kCsrThreads, 0, s>>>(a);
  return cudaGetLastError();
}

template <class Tr>
cudaError_t launch_csr_t(const loops_plan_s* p, const CsrDev& d, const DenseArgs& da, bool accumulate,
                         cudaStream_t s) {
  CsrKArgs a;
  a.accumulate = accumulate ? 1 : 0;
  a.item_row = d.item_row;
  a.item_ptr = d.item_ptr;
  a.col = d.col;
  a.val = d.val;
  a.n_items = d.n_items;
  a.B = da.B;
  a.ldb = da.ldb;
  a.C = da.C;
  a.ldc = da.ldc;
  a.scratch = d.scratch;
  a.col_scale = da.col_scale;
  a.inv_scale_f = da.inv_scale_f;
  a.inv_scale_d = da.inv_scale_d;
  a.N = da.N;
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
        case 1: e = two ? launch_vec_g<Tr, 1, 2>(a, s) : launch_vec_g<Tr, 1, 1>(a, s); break;
        case 2: e = two ? launch_vec_g<Tr, 2, 2>(a, s) : launch_vec_g<Tr, 2, 1>(a, s); break;
        case 4: e = two ? launch_vec_g<Tr, 4, 2>(a, s) : launch_vec_g<Tr, 4, 1>(a, s); break;
        case 8: e = two ? launch_vec_g<Tr, 8, 2>(a, s) : launch_vec_g<Tr, 8, 1>(a, s); break;
        case 16: e = two ? launch_vec_g<Tr, 16, 2>(a, s) : launch_vec_g<Tr, 16, 1>(a, s); break;
        default: e = two ? launch_vec_g<Tr, 32, 2>(a, s) : launch_vec_g<Tr, 32, 1>(a, s); break;
      }
    } else {
      dim3 grid((unsigned)((a.n_items * 32 + 255) / 256), (unsigned)((a.N + 31) / 32));
      csr_spmm_scalar<Tr, 8><<<grid, 256, 0, s>>>(a);
      e = cudaGetLastError();
    }
  }
  if (e == cudaSuccess && d.n_split > 0) {
    dim3 grid((unsigned)d.n_split, (unsigned)std::min<int64_t>((a.N + 255) / 256, 64));
    split_reduce<Tr><<<grid, 256, 0, s>>>(d.split_row, d.split_slot_ptr, d.n_split, a);
    e = cudaGetLastError();
  }
  return e;
}

}  // namespace

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
