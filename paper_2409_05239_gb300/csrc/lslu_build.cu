// Construction of the stored matrices of a handle: the padded CSR of A and of
// A^T (see DevCsr) from the caller's CSR, on the device.
//
//   columns counted (one atomic per entry) and scanned on the host;
//   A filled row by row, in the stored order of its 64-entry blocks; a
//     renumbered row is sorted by its new columns in shared memory first;
//   A^T: every entry takes a slot of its column by an atomic cursor as the
//     key (row, entry), in any order; one block per column sorts its keys in
//     shared memory, so a column lists its rows in increasing order (entries
//     of one row in input order) whatever the atomics did, and writes the row
//     of A^T;
//   16-bit column offsets from the smallest column of every block (or unit).
//
// A 2.5 M-entry matrix (128x128 image, 120 angles) took 28.6 ms to set up
// with host loops (a counting sort with one random write per entry, copies
// into vectors and their page faults) against about 0.5 ms of kernels and
// copies.  The construction needs 8 bytes of device memory per entry beside
// the stored matrices, 20 where the CSR comes from the host (the caller's
// entries are there too).  The host sorts instead, and its rows pass through a
// small buffer, where rows or columns have more than kSortMax entries, where
// that memory is not to be had, and for matrices of at most kHostEntries.
#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <type_traits>
#include <vector>

#include "lslu_internal.cuh"

namespace lslu {

namespace {

constexpr int kSortMax = 8192;  // keys of 8 bytes one block sorts (64 KB of shared memory)
constexpr int kSortThreads = 256;
constexpr int kRowThreads = 256;  // one warp per row
constexpr int64_t kUploadEntries = 4 << 20;   // of the host's rows on their way, 12 bytes each
constexpr int64_t kUploadMinimum = 256 << 10;  // the same where memory is short
constexpr size_t kStageBytes = 512 << 10;       // rows put together for one copy

// Entry of a row that its stored position q holds: full kPermBlock-entry
// blocks are stored transposed (position 4 l + i holds entry 16 i + l).
__device__ __forceinline__ int stored_entry(int q, int plen) {
  const int b = q / kPermBlock, w = q % kPermBlock;
  return b < plen / kPermBlock ? b * kPermBlock + 16 * (w & 3) + (w >> 2) : q;
}

// Where entry e of a row is stored (the inverse).
__device__ __forceinline__ int stored_position(int e, int plen) {
  const int b = e / kPermBlock, w = e % kPermBlock;
  return b < plen / kPermBlock ? b * kPermBlock + 4 * (w & 15) + (w >> 4) : e;
}

__device__ __forceinline__ void put(double* p, double v) { *p = v; }
__device__ __forceinline__ void put(float* p, double v) { *p = __double2float_rn(v); }
// FP64 -> FP32 -> BF16, each to nearest even, on the bits
__device__ __forceinline__ void put(__nv_bfloat16* p, double v) {
  const uint32_t u = __float_as_uint(__double2float_rn(v));
  *reinterpret_cast<uint16_t*>(p) = (uint16_t)((u + 0x7fffu + ((u >> 16) & 1u)) >> 16);
}

// First entry with a column out of range and first non-finite value.
__global__ void k_check(int64_t nnz, int64_t n, const int32_t* __restrict__ ci,
                        const double* __restrict__ vv, unsigned long long* bad) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nnz;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (ci[i] < 0 || ci[i] >= n) atomicMin(bad, (unsigned long long)i);
    if (!isfinite(vv[i])) atomicMin(bad + 1, (unsigned long long)i);
  }
}

__global__ void k_count(int64_t nnz, const int32_t* __restrict__ ci,
                        const int32_t* __restrict__ col_new, int32_t* cnt) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nnz;
       i += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(cnt + (col_new ? col_new[ci[i]] : ci[i]), 1);
}

// Every entry of stored row r takes a slot of its column (cur: next free slot).
__global__ void __launch_bounds__(kRowThreads)
    k_scatter_keys(int64_t rows, const int64_t* __restrict__ rp, const int32_t* __restrict__ ci,
                   const int32_t* __restrict__ inv_row, const int32_t* __restrict__ col_new,
                   int32_t* cur, unsigned long long* __restrict__ keys) {
  const int lane = threadIdx.x & 31;
  const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (r >= rows) return;
  const int64_t src = inv_row ? inv_row[r] : r;
  for (int64_t e = rp[src] + lane; e < rp[src + 1]; e += 32) {
    const int32_t c = col_new ? col_new[ci[e]] : ci[e];
    keys[atomicAdd(cur + c, 1)] = ((unsigned long long)r << 32) | (unsigned long long)e;
  }
}

// Row r of the stored matrix from entry rp[r] - rp[0] on, in the input's order.
template <typename VT>
__global__ void __launch_bounds__(kRowThreads)
    k_fill_rows(int64_t rows, const int64_t* __restrict__ rp, const int32_t* __restrict__ prp,
                const int32_t* __restrict__ prl, const int32_t* __restrict__ ci,
                const double* __restrict__ vv, int32_t* __restrict__ col, VT* __restrict__ val) {
  const int lane = threadIdx.x & 31;
  const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (r >= rows) return;
  const int64_t a = rp[r] - rp[0];
  const int len = (int)(rp[r + 1] - rp[r]), plen = prl[r];
  for (int q = lane; q < plen; q += 32) {
    const int e = stored_entry(q, plen);
    const int64_t s = a + (e < len ? e : len - 1);  // padding repeats the last column
    col[(int64_t)prp[r] + q] = ci[s];
    put(val + prp[r] + q, e < len ? vv[s] : 0.0);
  }
}

// Row r of the stored matrix from its sorted keys, one block per row.  keys
// null: the row is caller row inv_row[r] with its columns renumbered, keys
// (new column, entry of the row).  Else keys (row of A, entry) of column r at
// first[r].
template <typename VT>
__global__ void __launch_bounds__(kSortThreads)
    k_sort_fill(const unsigned long long* __restrict__ keys, const int32_t* __restrict__ first,
                const int64_t* __restrict__ rp, const int32_t* __restrict__ inv_row,
                const int32_t* __restrict__ col_new, const int32_t* __restrict__ prp,
                const int32_t* __restrict__ prl, const int32_t* __restrict__ ci,
                const double* __restrict__ vv, int32_t* __restrict__ col, VT* __restrict__ val) {
  extern __shared__ unsigned long long sk[];
  const int64_t r = blockIdx.x;
  int64_t a;
  int len;
  if (keys) {
    a = first[r];
    len = first[r + 1] - first[r];
  } else {
    a = rp[inv_row[r]];
    len = (int)(rp[inv_row[r] + 1] - a);
  }
  if (len == 0) return;
  int np = 1;
  while (np < len) np <<= 1;
  for (int i = threadIdx.x; i < np; i += blockDim.x)
    sk[i] = i >= len ? ~0ull
            : keys   ? keys[a + i]
                     : ((unsigned long long)(unsigned)col_new[ci[a + i]] << 32) | (unsigned)i;
  __syncthreads();
  for (int size = 2; size <= np; size <<= 1)  // bitonic sort
    for (int s = size >> 1; s > 0; s >>= 1) {
      for (int t = threadIdx.x; t < np / 2; t += blockDim.x) {
        const int i = 2 * t - (t & (s - 1)), j = i + s;
        const unsigned long long x = sk[i], y = sk[j];
        if ((x > y) == ((i & size) == 0)) {
          sk[i] = y;
          sk[j] = x;
        }
      }
      __syncthreads();
    }
  const int plen = prl[r];
  for (int q = threadIdx.x; q < plen; q += blockDim.x) {
    const int e = stored_entry(q, plen);
    const unsigned long long k = sk[e < len ? e : len - 1];
    const int64_t s = (keys ? 0 : a) + (int64_t)(k & 0xffffffffull);
    col[(int64_t)prp[r] + q] = (int32_t)(k >> 32);
    put(val + prp[r] + q, e < len ? vv[s] : 0.0);
  }
}

// Smallest column of every block and unit of a row, one warp per row, two
// entries per lane.  With bbase: the blocks' smallest columns, and (with wide)
// wide[0] / wide[1] set where a block / unit spans 2^16 columns or more.  With
// off: the offsets from the blocks' (by_block) or units' smallest column, and
// that column for every unit.
__global__ void __launch_bounds__(kRowThreads)
    k_offsets(int64_t rows, const int32_t* __restrict__ prp, const int32_t* __restrict__ prl,
              const int32_t* __restrict__ rblk, const int32_t* __restrict__ col,
              int32_t* __restrict__ bbase, int* wide, bool by_block, uint16_t* __restrict__ off,
              int32_t* __restrict__ ubase) {
  const int lane = threadIdx.x & 31;
  const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (r >= rows) return;
  const int64_t p0 = prp[r];
  const int plen = prl[r];
  for (int b = 0; b * kPermBlock < plen; ++b) {
    int32_t c[2], lo[2], hi[2];
    bool in[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int q = b * kPermBlock + 32 * h + lane;
      in[h] = q < plen;
      c[h] = in[h] ? col[p0 + q] : 0;
      lo[h] = in[h] ? c[h] : 0x7fffffff;
      hi[h] = in[h] ? c[h] : -1;
    }
    const int32_t blo = __reduce_min_sync(0xffffffffu, min(lo[0], lo[1]));
    const int32_t bhi = __reduce_max_sync(0xffffffffu, max(hi[0], hi[1]));
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int o = 1; o < kRowAlign; o <<= 1) {
        lo[h] = min(lo[h], __shfl_xor_sync(0xffffffffu, lo[h], o));
        hi[h] = max(hi[h], __shfl_xor_sync(0xffffffffu, hi[h], o));
      }
    if (bbase && lane == 0) bbase[rblk[r] + b] = blo;
    if (wide) {
      if (lane == 0 && bhi - blo > 65535) wide[0] = 1;
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (in[h] && hi[h] - lo[h] > 65535) wide[1] = 1;
    }
    if (!off) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (!in[h]) continue;
      const int64_t p = p0 + b * kPermBlock + 32 * h + lane;
      const int32_t base = by_block ? blo : lo[h];
      off[p] = (uint16_t)(c[h] - base);
      if (lane % kRowAlign == 0) ubase[p / kRowAlign] = base;
    }
  }
}

// Padded layout of rows of the given lengths: where each starts, its padded
// length and its first block, as they are uploaded.
struct Layout {
  std::vector<int32_t> words;      // row pointers, lengths, first blocks
  int64_t len_at = 0, blk_at = 0;  // the latter two in words
  int64_t tot = 0, blocks = 0;
  int32_t max_len = 0;
};
int64_t words64(int64_t count) { return (count + 63) / 64 * 64; }  // whole 256-byte pieces
template <typename Len>
bool make_layout(int64_t rows, Len len, Layout& l) {
  const int64_t nrp = (rows + 1 + 3) / 4 * 4;  // row pointers padded to a multiple of 4 entries
  l.len_at = words64(nrp);
  l.blk_at = l.len_at + words64(rows);
  l.words.resize(l.blk_at + words64(rows));
  int32_t *ptr = l.words.data(), *plens = ptr + l.len_at, *blk = ptr + l.blk_at;
  for (int64_t r = 0; r < rows; ++r) {
    const int64_t plen = (len(r) + kRowAlign - 1) / kRowAlign * kRowAlign;
    ptr[r] = (int32_t)l.tot;
    plens[r] = (int32_t)plen;
    blk[r] = (int32_t)l.blocks;
    l.tot += plen;
    l.max_len = std::max(l.max_len, (int32_t)plen);
    l.blocks += (plen + kPermBlock - 1) / kPermBlock;
    if (l.tot >= (int64_t)INT32_MAX) return false;
  }
  for (int64_t i = rows; i < nrp; ++i) ptr[i] = (int32_t)l.tot;
  return true;
}

#define CE(call)                             \
  do {                                       \
    const cudaError_t e_ = (call);           \
    if (e_ != cudaSuccess) return e_;        \
  } while (0)

size_t align_up(size_t bytes) { return (bytes + 255) / 256 * 256; }

// Arrays carved out of one allocation.
struct Arena {
  char* base = nullptr;
  size_t used = 0;
  template <typename T>
  T* take(size_t count) {
    T* p = reinterpret_cast<T*>(base + used);
    used += align_up(count * sizeof(T));
    return p;
  }
};

template <typename T>
cudaError_t upload(T* dst, const T* src, size_t count, cudaStream_t s) {
  return count ? cudaMemcpyAsync(dst, src, count * sizeof(T), cudaMemcpyHostToDevice, s)
               : cudaSuccess;
}

// The arrays of a stored matrix, columns and values still to be filled.  (Few
// allocations and one upload of the rows: with eight allocations and three
// uploads a handle of 17532 entries took 497 us to set up, now 440.)
cudaError_t allocate(const Layout& l, int64_t rows, int64_t cols, int64_t nnz, int vt, DevCsr* out,
                     cudaStream_t s) {
  out->rows = rows;
  out->cols = cols;
  out->nnz = nnz;
  out->nnz_padded = l.tot;
  out->max_len = l.max_len;
  const size_t vbytes = vt == LSLU_F64 ? 8 : vt == LSLU_F32 ? 4 : 2;
  const int64_t cap = std::max<int64_t>(l.tot, kRowAlign);
  Arena mem;
  CE(cudaMalloc(&out->mem_rows, align_up(l.words.size() * 4) + align_up(l.blocks * 4) + 256));
  mem.base = (char*)out->mem_rows;
  out->row_ptr = mem.take<int32_t>(l.words.size());
  out->row_len = out->row_ptr + l.len_at;
  out->rblk = out->row_ptr + l.blk_at;
  out->bbase = mem.take<int32_t>(l.blocks);
  out->flags = mem.take<int32_t>(4);
  CE(cudaMalloc((void**)&out->col, cap * sizeof(int32_t)));
  CE(cudaMalloc(&out->val, cap * vbytes));
  return upload(out->row_ptr, l.words.data(), l.words.size(), s);
}

template <typename Fn>
void with_value_type(int vt, void* val, Fn f) {
  if (vt == LSLU_F64)
    f((double*)val);
  else if (vt == LSLU_F32)
    f((float*)val);
  else
    f((__nv_bfloat16*)val);
}

unsigned warps_grid(int64_t rows) { return (unsigned)((rows * 32 + kRowThreads - 1) / kRowThreads); }

// Stored rows r0 .. r0 + rows - 1 from a CSR of them alone (rp: the caller's
// row pointers of these rows).
void fill_rows(const DevCsr& A, int vt, int64_t r0, int64_t rows, const int64_t* rp,
               const int32_t* ci, const double* vv, cudaStream_t s) {
  if (A.nnz_padded == 0 || rows == 0) return;
  with_value_type(vt, A.val, [&](auto* v) {
    k_fill_rows<<<warps_grid(rows), kRowThreads, 0, s>>>(rows, rp, A.row_ptr + r0, A.row_len + r0,
                                                         ci, vv, A.col, v);
  });
}

cudaError_t sort_fill(const DevCsr& A, int vt, int max_len, const unsigned long long* keys,
                      const int32_t* first, const int64_t* rp, const int32_t* inv_row,
                      const int32_t* col_new, const int32_t* ci, const double* vv, cudaStream_t s) {
  if (A.nnz_padded == 0) return cudaSuccess;
  int np = 1;
  while (np < max_len) np <<= 1;
  const size_t smem = (size_t)np * 8;
  cudaError_t e = cudaSuccess;
  with_value_type(vt, A.val, [&](auto* v) {
    using VT = typename std::remove_pointer<decltype(v)>::type;
    if (smem > 48 * 1024)
      e = cudaFuncSetAttribute(k_sort_fill<VT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               kSortMax * 8);
    if (e == cudaSuccess)
      k_sort_fill<VT><<<(unsigned)A.rows, kSortThreads, smem, s>>>(
          keys, first, rp, inv_row, col_new, A.row_ptr, A.row_len, ci, vv, A.col, v);
  });
  return e;
}

void launch_offsets(const DevCsr& A, int32_t* bbase, int* wide, uint16_t* off, int32_t* ubase,
                    cudaStream_t s) {
  k_offsets<<<warps_grid(A.rows), kRowThreads, 0, s>>>(A.rows, A.row_ptr, A.row_len, A.rblk, A.col,
                                                       bbase, wide, A.block_compressed != 0, off,
                                                       ubase);
}

// 16-bit column offsets, from the smallest column of every block where all
// blocks span fewer than 2^16 columns, else of every unit where those do.  With
// at most 2^16 columns that holds without a look.
cudaError_t add_offsets(DevCsr* A, DevCsr* AT, cudaStream_t s) {
  DevCsr* both[2] = {A, AT};
  auto narrow = [](const DevCsr& M) { return M.cols <= 65536; };
  int wide[4] = {0, 0, 0, 0};
  if (!narrow(*A) || !narrow(*AT)) {
    CE(cudaMemsetAsync(A->flags, 0, sizeof(wide), s));
    for (int w = 0; w < 2; ++w)
      if (both[w]->nnz_padded && !narrow(*both[w]))
        launch_offsets(*both[w], both[w]->bbase, A->flags + 2 * w, nullptr, nullptr, s);
    CE(cudaGetLastError());
    CE(cudaMemcpyAsync(wide, A->flags, sizeof(wide), cudaMemcpyDeviceToHost, s));
    CE(cudaStreamSynchronize(s));
  }
  for (int w = 0; w < 2; ++w) {
    DevCsr& M = *both[w];
    M.block_compressed = M.nnz_padded > 0 && !wide[2 * w];
    M.compressed = M.nnz_padded > 0 && (M.block_compressed || !wide[2 * w + 1]);
    if (!M.compressed) continue;
    // unit bases readable up to a multiple of 4 units
    const int64_t nub = (M.nnz_padded / kRowAlign + 3) / 4 * 4;
    Arena mem;
    CE(cudaMalloc(&M.mem_off, align_up(M.nnz_padded * sizeof(uint16_t)) + align_up(nub * 4)));
    mem.base = (char*)M.mem_off;
    M.off = mem.take<uint16_t>(M.nnz_padded);
    M.ubase = mem.take<int32_t>(nub);
    launch_offsets(M, narrow(M) ? M.bbase : nullptr, nullptr, M.off, M.ubase, s);
  }
  return cudaGetLastError();
}

// Neighbouring entries of every 16th row: count[0] pairs of different columns,
// count[1] those whose FP32 vector entries share a 32-byte sector.
__global__ void __launch_bounds__(kRowThreads)
    k_near(int64_t rows, const int32_t* __restrict__ prp, const int32_t* __restrict__ prl,
           const int32_t* __restrict__ col, int* count) {
  const int lane = threadIdx.x & 31;
  const int64_t r = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 16;
  if (r >= rows) return;
  const int32_t* c = col + prp[r];
  const int plen = prl[r];
  int pairs = 0, near = 0;
  for (int e = lane; e + 1 < plen; e += 32) {
    const int32_t a = c[stored_position(e, plen)], b = c[stored_position(e + 1, plen)];
    pairs += a != b;  // (the padding repeats a row's last column)
    near += a != b && (a >> 3) == (b >> 3);
  }
  pairs = __reduce_add_sync(0xffffffffu, pairs);
  near = __reduce_add_sync(0xffffffffu, near);
  if (lane == 0) {
    atomicAdd(count, pairs);
    atomicAdd(count + 1, near);
  }
}

// The form of the default FP32 / BF16 products.  A row under 64 entries gives a
// lane one chunk at most: there is nothing for more of them in flight, and the
// plain form's six blocks per SM beat the stream form's four.  Up to 96 entries,
// and where a row's columns are scattered (fewer than one neighbour in ten in
// the same sector, as in a random matrix), the products wait for their gathers,
// and the offsets form does best.  Whole solves of 20 to 300 iterations, FP32 /
// BF16, time against the plain form's (products A and A^T alone behave alike):
//   entries per row (A / A^T)               offsets        stream
//   8 / 12, random columns                  1.00 / 1.00    1.10 / 1.12
//   30 / 30, banded                         1.11 / 0.99    1.11 / 1.21
//   461 / 76, 512x512 CT, 60 angles         0.96 / 0.95    0.97 / 1.05
//   200 / 333, random columns               0.96 / 0.95    1.07 / 1.08
//   144 / 153, 160x160 CT, 120 angles       0.99 / 0.96    0.91 / 0.91
//   461 / 458, 512x512 CT, 360 angles       0.88           0.85
// Two kinds of matrix take the stream form whatever their mean length.  A few
// waves of row groups: resident blocks have no last wave, 40000 random rows of
// 60 entries 0.96 / 0.97, 30000 banded ones of 80 0.87 / 0.87 (the table's first
// rows have 300000 rows).  And a row far longer than a row group's share of the
// matrix, a chain of its own that the product waits for: a banded matrix with 24
// entries per row and a column of some 35000 takes 4.54 ms in place of 5.37.
cudaError_t choose_form(DevCsr* A, int vt, cudaStream_t s) {
  A->form = kFormPlain;
  if (vt == LSLU_F64 || A->nnz_padded < kStreamMinEntries || !A->compressed) return cudaSuccess;
  const int64_t groups = (A->rows + 15) / 16;                      // of 16 rows, one block's
  const int64_t slots = std::max<int64_t>(A->num_sms * 6, 1);      // blocks of the plain form
  const int64_t share = A->nnz_padded / (slots * 16);              // entries of a row group
  const int64_t mean = A->nnz_padded / A->rows;
  A->form = kFormStream;
  if (groups <= 3 * slots || (A->max_len >= 1024 && A->max_len > 4 * share)) return cudaSuccess;
  A->form = mean < 64 ? kFormPlain : kFormOffsets;
  if (mean < 96) return cudaSuccess;
  int count[2];
  CE(cudaMemsetAsync(A->flags, 0, sizeof(count), s));
  k_near<<<warps_grid((A->rows + 15) / 16), kRowThreads, 0, s>>>(A->rows, A->row_ptr, A->row_len,
                                                                 A->col, A->flags);
  CE(cudaGetLastError());
  CE(cudaMemcpyAsync(count, A->flags, sizeof(count), cudaMemcpyDeviceToHost, s));
  CE(cudaStreamSynchronize(s));
  if ((int64_t)count[1] * 10 >= count[0]) A->form = kFormStream;
  return cudaSuccess;
}

// The transpose of a host CSR, by a stable counting sort.
void transpose_host(int64_t m, int64_t n, const int64_t* rp, const int32_t* ci, const double* vv,
                    std::vector<int64_t>& rpt, std::vector<int32_t>& cit, std::vector<double>& vt) {
  const int64_t nnz = rp[m];
  rpt.assign(n + 1, 0);
  for (int64_t i = 0; i < nnz; ++i) rpt[ci[i] + 1]++;
  for (int64_t c = 0; c < n; ++c) rpt[c + 1] += rpt[c];
  std::vector<int64_t> cur(rpt.begin(), rpt.end() - 1);
  cit.resize(nnz);
  vt.resize(nnz);
  for (int64_t r = 0; r < m; ++r)
    for (int64_t i = rp[r]; i < rp[r + 1]; ++i) {
      const int64_t pos = cur[ci[i]]++;
      cit[pos] = (int32_t)r;
      vt[pos] = vv[i];
    }
}

struct Scratch : Arena {  // device memory that the construction gives back
  ~Scratch() { cudaFree(base); }
  cudaError_t reserve(size_t bytes) { return cudaMalloc((void**)&base, bytes); }
};

}  // namespace

// A host CSR renumbered: stored row r holds caller row inv_row[r], with its
// columns mapped through col_new and sorted ascending (stable for repeats).
void renumber_csr(int64_t rows, const int64_t* rp, const int32_t* ci, const double* vv,
                  const std::vector<int32_t>& inv_row, const std::vector<int32_t>& col_new,
                  std::vector<int64_t>& rp_o, std::vector<int32_t>& ci_o,
                  std::vector<double>& vv_o) {
  rp_o.assign(rows + 1, 0);
  for (int64_t r = 0; r < rows; ++r)
    rp_o[r + 1] = rp_o[r] + (rp[inv_row[r] + 1] - rp[inv_row[r]]);
  ci_o.resize(rp_o[rows]);
  vv_o.resize(rp_o[rows]);
  std::vector<uint64_t> key;
  for (int64_t r = 0; r < rows; ++r) {
    const int64_t a = rp[inv_row[r]], len = rp[inv_row[r] + 1] - a, o = rp_o[r];
    key.resize(len);
    for (int64_t i = 0; i < len; ++i)
      key[i] = ((uint64_t)(uint32_t)col_new[ci[a + i]] << 32) | (uint64_t)i;
    std::sort(key.begin(), key.end());
    for (int64_t i = 0; i < len; ++i) {
      ci_o[o + i] = (int32_t)(key[i] >> 32);
      vv_o[o + i] = vv[a + (int64_t)(key[i] & 0xffffffffull)];
    }
  }
}

cudaError_t check_csr_device(int64_t nnz, int64_t n, const int32_t* ci, const double* vv,
                             cudaStream_t s, int64_t* bad_col, int64_t* bad_val) {
  *bad_col = *bad_val = -1;
  if (nnz == 0) return cudaSuccess;
  Scratch mem;
  CE(mem.reserve(256));
  unsigned long long* bad = mem.take<unsigned long long>(2);
  CE(cudaMemsetAsync(bad, 0xff, 16, s));
  k_check<<<(unsigned)std::min<int64_t>((nnz + 255) / 256, 8192), 256, 0, s>>>(nnz, n, ci, vv, bad);
  unsigned long long h[2];
  CE(cudaMemcpyAsync(h, bad, 16, cudaMemcpyDeviceToHost, s));
  CE(cudaStreamSynchronize(s));
  *bad_col = (int64_t)h[0];
  *bad_val = (int64_t)h[1];
  return cudaSuccess;
}

namespace {

// A CSR as the construction takes it: row pointers on the host, columns and
// values on the host or (on_device) the device, an optional renumbering.
struct Source {
  int64_t m, n, nnz;
  const int64_t* rp;
  const int32_t* ci;
  const double* vv;
  bool on_device;
  const std::vector<int32_t>*inv_row, *col_new;
  int64_t max_row;  // longest row
};

// Both matrices on the device.  *fits = false, with nothing left to undo but
// what A holds: a column has more than kSortMax entries.
cudaError_t build_on_device(const Source& in, const Layout& la, int vt, DevCsr* A, DevCsr* AT,
                            cudaStream_t s, bool* fits) {
  const int64_t m = in.m, n = in.n, nnz = in.nnz;
  *fits = true;
  // every host array that an asynchronous copy reads lives until the final
  // synchronisation
  std::vector<int32_t> cnt(n), first(n + 1, 0);
  Layout lt;
  Scratch mem;
  const size_t e = in.on_device ? 0 : (size_t)nnz;  // entries brought from the host
  const size_t bytes = align_up((m + 1) * 8) + align_up(n * 4) + align_up((n + 1) * 4) +
                       (in.inv_row ? align_up(m * 4) + align_up(n * 4) : 0) +
                       align_up((size_t)nnz * 8) + align_up(e * 4) + align_up(e * 8);
  CE(mem.reserve(std::max<size_t>(bytes, 1)));
  int64_t* d_rp = mem.take<int64_t>(m + 1);
  int32_t* d_cnt = mem.take<int32_t>(n);
  int32_t* d_first = mem.take<int32_t>(n + 1);
  int32_t* d_inv = in.inv_row ? mem.take<int32_t>(m) : nullptr;
  int32_t* d_new = in.inv_row ? mem.take<int32_t>(n) : nullptr;
  unsigned long long* d_keys = mem.take<unsigned long long>(nnz);
  const int32_t* ci = in.ci;
  const double* vv = in.vv;
  if (!in.on_device) {
    int32_t* d_ci = mem.take<int32_t>(e);
    double* d_vv = mem.take<double>(e);
    CE(upload(d_ci, in.ci, e, s));
    CE(upload(d_vv, in.vv, e, s));
    ci = d_ci;
    vv = d_vv;
  }
  if (mem.used != bytes) return cudaErrorInvalidValue;  // the sum above and the arrays disagree
  CE(upload(d_rp, in.rp, m + 1, s));
  if (in.inv_row) {
    CE(upload(d_inv, in.inv_row->data(), m, s));
    CE(upload(d_new, in.col_new->data(), n, s));
  }
  CE(cudaMemsetAsync(d_cnt, 0, n * sizeof(int32_t), s));
  if (nnz)
    k_count<<<(unsigned)std::min<int64_t>((nnz + 255) / 256, 8192), 256, 0, s>>>(nnz, ci, d_new,
                                                                                 d_cnt);
  CE(cudaMemcpyAsync(cnt.data(), d_cnt, n * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  CE(allocate(la, m, n, nnz, vt, A, s));
  CE(cudaStreamSynchronize(s));
  int64_t max_col = 0;
  for (int64_t c = 0; c < n; ++c) {
    first[c + 1] = first[c] + cnt[c];
    max_col = std::max<int64_t>(max_col, cnt[c]);
  }
  if (max_col > kSortMax) {
    *fits = false;
    return cudaSuccess;
  }
  if (!make_layout(n, [&](int64_t c) { return (int64_t)cnt[c]; }, lt)) return cudaErrorInvalidValue;
  CE(allocate(lt, n, m, nnz, vt, AT, s));
  CE(upload(d_first, first.data(), n + 1, s));
  CE(cudaMemcpyAsync(d_cnt, d_first, n * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
  if (nnz)
    k_scatter_keys<<<warps_grid(m), kRowThreads, 0, s>>>(m, d_rp, ci, d_inv, d_new, d_cnt, d_keys);
  if (in.inv_row)
    CE(sort_fill(*A, vt, (int)in.max_row, nullptr, nullptr, d_rp, d_inv, d_new, ci, vv, s));
  else
    fill_rows(*A, vt, 0, m, d_rp, ci, vv, s);
  CE(sort_fill(*AT, vt, (int)max_col, d_keys, d_first, nullptr, nullptr, nullptr, ci, vv, s));
  CE(cudaGetLastError());
  return cudaStreamSynchronize(s);
}

// A stored matrix from a host CSR in its final order: whole rows at a time go
// through a device buffer; of small matrices in one copy, put together in stage.
cudaError_t fill_from_host(const DevCsr& A, int vt, const int64_t* rp, const int32_t* ci,
                           const double* vv, char* buffer, int64_t chunk, std::vector<char>& stage,
                           cudaStream_t s) {
  for (int64_t r0 = 0; r0 < A.rows;) {
    int64_t r1 = r0 + 1;  // (a row is no longer than the buffer)
    while (r1 < A.rows && r1 - r0 < chunk && rp[r1 + 1] - rp[r0] <= chunk) ++r1;
    const size_t rows = r1 - r0, e0 = rp[r0], n = rp[r1] - rp[r0];
    const size_t vv_at = (rows + 1) * 8, ci_at = vv_at + n * 8, bytes = ci_at + n * 4;
    if (bytes <= kStageBytes) {
      CE(cudaStreamSynchronize(s));  // the stage's last rows are on the device
      stage.resize(bytes);
      std::memcpy(stage.data(), rp + r0, vv_at);
      if (n) std::memcpy(stage.data() + vv_at, vv + e0, n * 8);
      if (n) std::memcpy(stage.data() + ci_at, ci + e0, n * 4);
      CE(upload(buffer, stage.data(), bytes, s));
    } else {
      CE(upload((int64_t*)buffer, rp + r0, rows + 1, s));
      CE(upload((double*)(buffer + vv_at), vv + e0, n, s));
      CE(upload((int32_t*)(buffer + ci_at), ci + e0, n, s));
    }
    fill_rows(A, vt, r0, rows, (const int64_t*)buffer, (const int32_t*)(buffer + ci_at),
              (const double*)(buffer + vv_at), s);
    r0 = r1;
  }
  return cudaGetLastError();
}

// Both matrices sorted by the host.
cudaError_t build_on_host(Source in, const Layout& la, int vt, DevCsr* A, DevCsr* AT,
                          cudaStream_t s) {
  const int64_t m = in.m, n = in.n, nnz = in.nnz;
  std::vector<int64_t> rp_a, rp_t;
  std::vector<int32_t> ci_h, ci_a, ci_t;
  std::vector<double> vv_h, vv_a, vv_t;
  if (in.on_device) {
    ci_h.resize(nnz);
    vv_h.resize(nnz);
    CE(cudaMemcpyAsync(ci_h.data(), in.ci, nnz * 4, cudaMemcpyDeviceToHost, s));
    CE(cudaMemcpyAsync(vv_h.data(), in.vv, nnz * 8, cudaMemcpyDeviceToHost, s));
    CE(cudaStreamSynchronize(s));
    in.ci = ci_h.data();
    in.vv = vv_h.data();
  }
  if (in.inv_row) {
    renumber_csr(m, in.rp, in.ci, in.vv, *in.inv_row, *in.col_new, rp_a, ci_a, vv_a);
    in.rp = rp_a.data();
    in.ci = ci_a.data();
    in.vv = vv_a.data();
  }
  transpose_host(m, n, in.rp, in.ci, in.vv, rp_t, ci_t, vv_t);
  Layout lt;
  int64_t longest = in.max_row;
  if (!make_layout(n, [&](int64_t c) { return rp_t[c + 1] - rp_t[c]; }, lt))
    return cudaErrorInvalidValue;
  for (int64_t c = 0; c < n; ++c) longest = std::max(longest, rp_t[c + 1] - rp_t[c]);
  CE(allocate(la, m, n, nnz, vt, A, s));
  CE(allocate(lt, n, m, nnz, vt, AT, s));
  // the buffer: at most the whole matrix, at least a row of it
  std::vector<char> stage;
  Scratch mem;
  const int64_t whole = std::max(nnz, std::max(m, n));
  auto reserve = [&](int64_t* chunk, int64_t want) {
    *chunk = std::max(std::min(want, whole), longest);
    return mem.reserve((size_t)(*chunk + 1) * 8 + (size_t)*chunk * 12);
  };
  int64_t chunk = 0;
  cudaError_t e = reserve(&chunk, kUploadEntries);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    e = reserve(&chunk, kUploadMinimum);
  }
  CE(e);
  CE(fill_from_host(*A, vt, in.rp, in.ci, in.vv, mem.base, chunk, stage, s));
  CE(fill_from_host(*AT, vt, rp_t.data(), ci_t.data(), vv_t.data(), mem.base, chunk, stage, s));
  return cudaStreamSynchronize(s);
}

}  // namespace

cudaError_t build_csr_pair(int64_t m, int64_t n, const int64_t* rp, const int32_t* ci,
                           const double* vv, bool on_device, const std::vector<int32_t>* inv_row,
                           const std::vector<int32_t>* col_new, int vt, DevCsr* A, DevCsr* AT,
                           cudaStream_t s) {
  Source in{m, n, rp[m], rp, ci, vv, on_device, inv_row, col_new, 0};
  auto row_len = [&](int64_t r) {
    const int64_t src = inv_row ? (*inv_row)[r] : r;
    return rp[src + 1] - rp[src];
  };
  Layout la;
  if (!make_layout(m, row_len, la)) return cudaErrorInvalidValue;
  for (int64_t r = 0; r < m; ++r) in.max_row = std::max(in.max_row, rp[r + 1] - rp[r]);
  bool done = false;
  if (in.nnz > kHostEntries && !(inv_row && in.max_row > kSortMax)) {
    const cudaError_t e = build_on_device(in, la, vt, A, AT, s, &done);
    if (e == cudaErrorMemoryAllocation) done = false;
    if (e != cudaSuccess && e != cudaErrorMemoryAllocation) return e;
  }
  if (!done) {
    cudaGetLastError();
    CE(cudaStreamSynchronize(s));  // copies into what is given back
    free_csr(A);
    free_csr(AT);
    CE(build_on_host(in, la, vt, A, AT, s));
  }
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess)
    cudaDeviceGetAttribute(&A->num_sms, cudaDevAttrMultiProcessorCount, dev);
  AT->num_sms = A->num_sms;
  A->shape = AT->shape = default_shape(vt);
  CE(add_offsets(A, AT, s));
  CE(choose_form(A, vt, s));
  CE(choose_form(AT, vt, s));
  return cudaStreamSynchronize(s);
}

void free_csr(DevCsr* c) {
  cudaFree(c->mem_rows);
  cudaFree(c->col);
  cudaFree(c->val);
  cudaFree(c->mem_off);
  *c = DevCsr();
}

}  // namespace lslu
