// Allocation-free CSR SpMM: C = A . B straight from caller-owned device CSR arrays, with no
// plan and no device allocation of any kind.
//
// Who needs it: code that must not call cudaMalloc (or any allocating routine) at the point
// where it multiplies -- for example a kernel sequence being recorded into a CUDA graph under
// the global capture mode, a host callback or real-time path where allocation latency or
// failure is not acceptable, or a service that reserves all device memory up front and runs
// under a fixed memory budget. Building a plan allocates device memory, so those callers
// cannot use loops_plan / loops_spmm; they hand their CSR arrays and dense operands here.
//
// How it works: the stored entries are cut into fixed chunks of kChunk entries; one warp takes
// one chunk (and one slice of N). Rows that start and end inside a chunk are summed and written
// directly. A row that crosses a chunk boundary leaves partial sums: the chunk that owns the
// row's first entry writes a "tail" partial, every later chunk the row runs into writes a "head"
// partial, and a second kernel adds them in chunk order and writes the row. The partial sums live
// in g_noalloc_scratch, a fixed file-scope device array: the library's only scratch memory that
// it never allocates. The order of every sum is fixed, so results do not depend on scheduling.
#include <cstring>
#include <mutex>
#include <type_traits>

#include "device_common.cuh"
#include "loops_internal.h"

namespace loops {

namespace {

constexpr int64_t kChunk = 128;  // stored entries per chunk

// Partial sums of chunk-crossing rows: [2][n_chunks][N] accumulators (head, tail). Every GPU
// that loads the library holds this array until the process exits.
static __device__ __align__(256) unsigned char g_noalloc_scratch[LOOPS_NOALLOC_SCRATCH_BYTES];

// Device address of g_noalloc_scratch per device, looked up once per device.
std::mutex g_mu;
void* g_scratch_ptr[128] = {};

struct NoAllocArgs {
  const int64_t* row_ptr;
  const int32_t* col;
  const void* val;
  int64_t n_rows, n_cols, nnz, n_chunks;
  const void* B;
  int64_t ldb;
  void* C;
  int64_t ldc;
  int64_t N;
  void* scratch;
};

__device__ __forceinline__ int64_t clamp_ptr(const NoAllocArgs& a, int64_t r) {
  const int64_t v = a.row_ptr[r];
  return v < 0 ? 0 : (v > a.nnz ? a.nnz : v);
}

// First r in [0, n_rows) with row_ptr[r] >= x (n_rows if none), by the whole warp: 32 probes per
// step, so 65,536 rows take 4 dependent loads instead of 17.
__device__ __forceinline__ int64_t lower_row(const NoAllocArgs& a, int64_t x) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, hi = a.n_rows;  // the answer lies in [lo, hi]
  while (hi > lo) {
    const int64_t step = (hi - lo + 31) / 32;  // 1 from 32 candidates on down
    const int64_t r = lo + lane * step;
    const unsigned at_or_past = __ballot_sync(0xffffffffu, r >= hi || clamp_ptr(a, r) >= x);
    const int f = at_or_past ? __ffs(at_or_past) - 1 : 32;  // probe f - 1 is before x, probe f is not
    const int64_t top = lo + f * step;
    if (f == 0) return lo;
    lo += (f - 1) * step + 1;
    hi = top < hi ? top : hi;
  }
  return lo;
}

// Accumulator value of an A value in its register form (Tr::TV).
template <class Tr>
__device__ __forceinline__ typename Tr::TAcc value_of(typename Tr::TV v) {
  if constexpr (sizeof(typename Tr::TB) == 2) {
    const unsigned short u = (unsigned short)v;
    typename Tr::TB x;
    memcpy(&x, &u, 2);
    return Tr::to_acc(x);
  } else {
    return v;
  }
}

// Columns of a lane. VEC: one 16-byte vector (VE columns) per lane of a group of G; else CP single
// columns, G apart. A slice has G * VE or G * CP columns, and 32 / G groups take every
// (32 / G)-th entry of a row, summed over the groups at the row's end.
template <class Tr, int G, int CP, bool VEC>
struct Slice {
  static constexpr int kCols = VEC ? Tr::kVE : CP;
  static constexpr int kWidth = G * kCols;
  __device__ __forceinline__ static int64_t column(int64_t n0, int sub, int i) {
    return VEC ? n0 + sub * kCols + i : n0 + i * G + sub;
  }
};

// warps per block; four of FP64 spread a small call's FP64 work over more SMs
template <class Tr>
constexpr int kNoAllocWarps = std::is_same<Tr, TrF64>::value ? 4 : 8;
constexpr int kNoAllocU = 4;  // entries in flight per group

// Bound by the gathers of B rows. The chunk's columns and values are staged in shared memory
// first, so that the gathers depend on no global load, and kNoAllocU of them are in flight per
// group. 65,536 rows of 32 entries, N = 64, FP32: 65 us a call (both kernels), against 196 us with
// one gather in flight, the entries read per 32 columns, and four binary searches per chunk.
// FP64 is bound by the FP64 pipe, where an instruction costs the same for one live lane as for 32: no
// FMA past a row's end, sums over only the groups that had an entry, and up to N = 32 one column per lane,
// since vectors of two mean twice the instructions and more groups to sum. 200,000 rows of 4 entries, N =
// 16, 93 -> 61 us (vectors 158); 30,000 of 33, N = 8, 102 -> 35 us (vectors 55).
template <class Tr, int G, int CP, bool VEC>
__global__ void __launch_bounds__(kNoAllocWarps<Tr> * 32) noalloc_chunks(NoAllocArgs a) {
  using TB = typename Tr::TB;
  using TAcc = typename Tr::TAcc;
  using TC = typename Tr::TC;
  using TV = typename Tr::TV;
  using S = Slice<Tr, G, CP, VEC>;
  constexpr int NC = S::kCols;
  constexpr int NG = 32 / G;
  constexpr int U = kNoAllocU;
  constexpr bool F64 = std::is_same<Tr, TrF64>::value;
  __shared__ int32_t s_col[kNoAllocWarps<Tr>][kChunk];
  __shared__ TV s_val[kNoAllocWarps<Tr>][kChunk];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t c = (int64_t)blockIdx.x * kNoAllocWarps<Tr> + warp;
  if (c >= a.n_chunks) return;
  const int sub = lane & (G - 1), grp = lane / G;
  const int64_t e0 = c * kChunk;
  const int64_t e1 = (e0 + kChunk < a.nnz) ? e0 + kChunk : a.nnz;
  const bool last = c == a.n_chunks - 1;
  int32_t* col = s_col[warp];
  TV* val = s_val[warp];
#pragma unroll
  for (int i = 0; i < (int)kChunk / 32; ++i) {
    const int64_t k = e0 + i * 32 + lane;
    int32_t cj = -1;
    TV v = 0;
    if (k < e1) {
      cj = __ldg(a.col + k);
      v = Tr::load_v(reinterpret_cast<const TB*>(a.val) + k);
      if ((int64_t)cj >= a.n_cols) cj = -1;  // skipped, so no load leaves B
    }
    col[i * 32 + lane] = cj;
    val[i * 32 + lane] = v;
  }
  __syncwarp();
  const int64_t n0 = (int64_t)blockIdx.y * S::kWidth;
  bool ok[NC];
#pragma unroll
  for (int i = 0; i < NC; ++i) ok[i] = S::column(n0, sub, i) < a.N;
  const TB* bl = reinterpret_cast<const TB*>(a.B) + S::column(n0, sub, 0);
  TAcc* head = reinterpret_cast<TAcc*>(a.scratch);
  TAcc* tail = head + a.n_chunks * a.N;

  // sum over the chunk's entries [k0, k1), in the lanes of group 0
  auto dot = [&](int k0, int k1, TAcc (&acc)[NC]) {
#pragma unroll
    for (int i = 0; i < NC; ++i) acc[i] = TAcc(0);
    for (int kb = k0; kb < k1; kb += NG * U) {
      TV av[U];
      if constexpr (VEC) {
        uint4 bv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int k = kb + u * NG + grp;
          const int32_t cj = k < k1 ? col[k] : -1;
          av[u] = cj >= 0 ? val[k] : TV(0);
          bv[u] = ldg16_if(ok[0] && cj >= 0, bl + (int64_t)cj * a.ldb);
        }
        if (!F64 || kb + NG * U <= k1) {
#pragma unroll
          for (int u = 0; u < U; ++u) fma_vec<Tr>(acc, bv[u], av[u]);
        } else {
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (u == 0 || kb + u * NG < k1) fma_vec<Tr>(acc, bv[u], av[u]);
        }
      } else {
        TB bv[U][NC];
        bool live[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int k = kb + u * NG + grp;
          const int32_t cj = k < k1 ? col[k] : -1;
          live[u] = cj >= 0;
          av[u] = live[u] ? val[k] : TV(0);
          const TB* brow = bl + (int64_t)cj * a.ldb;
#pragma unroll
          for (int i = 0; i < NC; ++i)
            if (live[u] && ok[i]) bv[u][i] = brow[i * G];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (F64 && u > 0 && kb + u * NG >= k1) break;
          const TAcc w = value_of<Tr>(av[u]);
#pragma unroll
          for (int i = 0; i < NC; ++i)
            if (live[u] && ok[i]) acc[i] = fma(w, Tr::to_acc(bv[u][i]), acc[i]);
        }
      }
    }
#pragma unroll
    for (int off = G; off < 32; off <<= 1) {
      if (F64 && off >= (k1 - k0) * G) break;  // the groups from off / G on had no entry
#pragma unroll
      for (int i = 0; i < NC; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], off);
    }
  };

  // rows owned by this chunk: first entry in [e0, e1) (the last chunk also owns trailing
  // empty rows); positions below are relative to e0
  const int64_t r0 = lower_row(a, e0);
  const int n_e = (int)(e1 - e0);
  auto rel = [&](int64_t p) { return (int)(p <= e0 ? 0 : (p - e0 > kChunk ? kChunk + 1 : p - e0)); };
  // continuation of a row that started in an earlier chunk
  if (n_e > 0 && r0 > 0) {
    const int end_in = rel(clamp_ptr(a, r0));
    if (end_in > 0) {
      TAcc acc[NC];
      dot(0, min(end_in, n_e), acc);
      if (grp == 0) {
#pragma unroll
        for (int i = 0; i < NC; ++i)
          if (ok[i]) head[c * a.N + S::column(n0, sub, i)] = acc[i];
      }
    }
  }
  // 31 rows per load of row pointers
  bool more = true;
  for (int64_t r = r0; more && r < a.n_rows; r += 31) {
    const int p = rel(r + lane <= a.n_rows ? clamp_ptr(a, r + lane) : a.nnz);
    for (int i = 0; i < 31; ++i) {
      const int b = __shfl_sync(0xffffffffu, p, i), e = __shfl_sync(0xffffffffu, p, i + 1);
      if (r + i >= a.n_rows || (!last && b >= n_e)) {
        more = false;
        break;
      }
      TAcc acc[NC];
      dot(b, min(e, n_e), acc);
      if (grp != 0) continue;
      if (e <= n_e) {  // complete row
        TC* crow = reinterpret_cast<TC*>(a.C) + (r + i) * a.ldc;
        if constexpr (VEC) {
          if (ok[0]) {
            TC o[NC];
#pragma unroll
            for (int x = 0; x < NC; ++x) o[x] = (TC)acc[x];
#pragma unroll
            for (int x = 0; x < (int)(NC * sizeof(TC) / 16); ++x)
              reinterpret_cast<uint4*>(crow + S::column(n0, sub, 0))[x] = reinterpret_cast<const uint4*>(o)[x];
          }
        } else {
#pragma unroll
          for (int x = 0; x < NC; ++x)
            if (ok[x]) crow[S::column(n0, sub, x)] = (TC)acc[x];
        }
      } else {         // continues: partial
#pragma unroll
        for (int x = 0; x < NC; ++x)
          if (ok[x]) tail[c * a.N + S::column(n0, sub, x)] = acc[x];
      }
    }
  }
}

// Rows that cross chunk boundaries: tail partial of the owning chunk plus the head partials of
// the chunks the row runs into, in chunk order (eight loads at a time). A warp per chunk and 128
// columns.
template <class Tr>
__global__ void __launch_bounds__(256) noalloc_fixup(NoAllocArgs a) {
  using TAcc = typename Tr::TAcc;
  using TC = typename Tr::TC;
  const int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (c >= a.n_chunks - 1) return;  // the last chunk's rows end inside it
  const int lane = threadIdx.x & 31;
  const int64_t e0 = c * kChunk, e1 = e0 + kChunk;
  const int64_t r = lower_row(a, e1) - 1;  // the chunk's last row, if it starts in the chunk
  if (r < 0 || clamp_ptr(a, r) < e0) return;
  const int64_t e = clamp_ptr(a, r + 1);
  if (e <= e1) return;
  const TAcc* head = reinterpret_cast<const TAcc*>(a.scratch);
  const TAcc* tail = head + a.n_chunks * a.N;
  const int64_t q1 = min((e + kChunk - 1) / kChunk, a.n_chunks);  // chunks c + 1 .. q1 - 1 hold the rest
  const int64_t n1 = min(a.N, ((int64_t)blockIdx.y + 1) * 128);
  for (int64_t n = (int64_t)blockIdx.y * 128 + lane; n < n1; n += 32) {
    TAcc s = tail[c * a.N + n];
    int64_t q = c + 1;
    for (; q + 8 <= q1; q += 8) {
      TAcc h[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) h[i] = head[(q + i) * a.N + n];
#pragma unroll
      for (int i = 0; i < 8; ++i) s += h[i];
    }
    for (; q < q1; ++q) s += head[q * a.N + n];
    reinterpret_cast<TC*>(a.C)[r * a.ldc + n] = (TC)s;
  }
}

template <class Tr>
cudaError_t launch_noalloc_t(const NoAllocArgs& a, cudaStream_t s) {
  constexpr int kWarps = kNoAllocWarps<Tr>;
  const unsigned gx = (unsigned)((a.n_chunks + kWarps - 1) / kWarps);
  auto go = [&](auto g_tag, auto cp_tag, auto vec_tag) {
    constexpr int G = decltype(g_tag)::value, CP = decltype(cp_tag)::value;
    constexpr bool VEC = decltype(vec_tag)::value;
    constexpr int width = Slice<Tr, G, CP, VEC>::kWidth;
    noalloc_chunks<Tr, G, CP, VEC><<<dim3(gx, (unsigned)((a.N + width - 1) / width)), kWarps * 32, 0, s>>>(a);
  };
  using std::integral_constant;
  using C1 = integral_constant<int, 1>;
  using C32 = integral_constant<int, 32>;
  // whole 16-byte vectors where B's and C's rows allow them; else single columns, more per lane
  // for wider rows (the entries are staged once per slice)
  const int64_t eb = sizeof(typename Tr::TB), ec = sizeof(typename Tr::TC);
  const bool vec = a.N % Tr::kVE == 0 && (uintptr_t)a.B % 16 == 0 && (uintptr_t)a.C % 16 == 0 &&
                   (a.ldb * eb) % 16 == 0 && (a.ldc * ec) % 16 == 0;
  const bool single = std::is_same<Tr, TrF64>::value && a.N <= 32;  // the reasons stand at the kernel
  if (vec && !single) {
    const int64_t nvec = a.N / Tr::kVE;
    if (nvec <= 1) go(C1(), C1(), std::true_type());
    else if (nvec <= 2) go(integral_constant<int, 2>(), C1(), std::true_type());
    else if (nvec <= 4) go(integral_constant<int, 4>(), C1(), std::true_type());
    else if (nvec <= 8) go(integral_constant<int, 8>(), C1(), std::true_type());
    else if (nvec <= 16) go(integral_constant<int, 16>(), C1(), std::true_type());
    else go(C32(), C1(), std::true_type());
  } else if (a.N <= 8) {
    go(integral_constant<int, 8>(), C1(), std::false_type());
  } else if (a.N <= 16) {
    go(integral_constant<int, 16>(), C1(), std::false_type());
  } else if (a.N <= 32) {
    go(C32(), C1(), std::false_type());
  } else if (a.N <= 64 || a.n_chunks <= 2048) {  // few chunks: more slices, so that more warps run
    go(C32(), integral_constant<int, 2>(), std::false_type());
  } else {
    go(C32(), integral_constant<int, 4>(), std::false_type());
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || a.n_chunks < 2) return e;
  noalloc_fixup<Tr><<<dim3((unsigned)((a.n_chunks * 32 + 255) / 256), (unsigned)((a.N + 127) / 128)), 256, 0, s>>>(a);
  return cudaGetLastError();
}

}  // namespace

}  // namespace loops

using namespace loops;

extern "C" loops_status loops_csr_spmm_noalloc(int64_t n_rows, int64_t n_cols, int64_t nnz, const int64_t* row_ptr,
                                               const int32_t* col_idx, const void* vals, loops_dtype dtype,
                                               const void* B, int64_t ldb, int64_t N, void* C, int64_t ldc,
                                               loops_stream_t stream) {
  clear_error();
  if (dtype != LOOPS_F64 && dtype != LOOPS_F32 && dtype != LOOPS_F16 && dtype != LOOPS_BF16) {
    set_error("bad dtype");
    return LOOPS_ERR_INVALID_ARG;
  }
  if (n_rows < 0 || n_cols < 0 || nnz < 0 || N < 0 || ldb < N || ldc < N) {
    set_error("negative size or leading dimension smaller than N");
    return LOOPS_ERR_INVALID_ARG;
  }
  if (n_rows == 0 || N == 0) return LOOPS_OK;
  if (!row_ptr || !C || (nnz > 0 && (!col_idx || !vals || !B))) {
    set_error("NULL pointer");
    return LOOPS_ERR_INVALID_ARG;
  }
  const int64_t n_chunks = nnz > 0 ? (nnz + kChunk - 1) / kChunk : 1;
  const int64_t acc_bytes = dtype == LOOPS_F64 ? 8 : 4;
  // the scratch test divides instead of multiplying, so no product of caller sizes can wrap
  const int64_t per_chunk = 2 * acc_bytes;  // head and tail accumulators per chunk and column
  if (N > (int64_t)LOOPS_NOALLOC_SCRATCH_BYTES / per_chunk ||
      n_chunks > (int64_t)LOOPS_NOALLOC_SCRATCH_BYTES / (per_chunk * N)) {
    set_error("problem too large for the allocation-free path: its scratch needs 2 * ceil(nnz / 128) * N * " +
              std::to_string((long long)acc_bytes) + " bytes (nnz " + std::to_string((long long)nnz) + ", N " +
              std::to_string((long long)N) + "), the static array holds " +
              std::to_string((long long)LOOPS_NOALLOC_SCRATCH_BYTES));
    return LOOPS_ERR_UNSUPPORTED;
  }
  if ((N + 31) / 32 > 65535 || (n_chunks * 32 + 255) / 256 > 0x7fffffffLL) {
    set_error("N too large for the allocation-free path's launch shape (at most 65535 * 32 columns)");
    return LOOPS_ERR_UNSUPPORTED;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= 128) {
    set_error(std::string("cudaGetDevice failed: ") + cudaGetErrorString(e));
    return LOOPS_ERR_CUDA;
  }
  void* scratch = nullptr;
  {
    // set-up, once per device with that device current: the host-side name of a __device__
    // array is not a device address, so look the address up and keep it
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_scratch_ptr[dev]) {
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
      if (e != cudaSuccess) {
        set_error(std::string("cudaGetSymbolAddress failed: ") + cudaGetErrorString(e));
        return LOOPS_ERR_CUDA;
      }
      g_scratch_ptr[dev] = p;
    }
    scratch = g_scratch_ptr[dev];
  }
  NoAllocArgs a;
  a.row_ptr = row_ptr;
  a.col = col_idx;
  a.val = vals;
  a.n_rows = n_rows;
  a.n_cols = n_cols;
  a.nnz = nnz;
  a.n_chunks = n_chunks;
  a.B = B;
  a.ldb = ldb;
  a.C = C;
  a.ldc = ldc;
  a.N = N;
  a.scratch = scratch;
  cudaStream_t s = (cudaStream_t)stream;
  switch (dtype) {
    case LOOPS_F64: e = launch_noalloc_t<TrF64>(a, s); break;
    case LOOPS_F32: e = launch_noalloc_t<TrF32>(a, s); break;
    case LOOPS_F16: e = launch_noalloc_t<TrF16>(a, s); break;
    case LOOPS_BF16: e = launch_noalloc_t<TrBF16>(a, s); break;
  }
  if (e != cudaSuccess) {
    set_error(std::string("launch failed: ") + cudaGetErrorString(e));
    return LOOPS_ERR_CUDA;
  }
  return LOOPS_OK;
}
