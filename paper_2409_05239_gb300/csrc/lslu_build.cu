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
// copies.  Rows or columns longer than kSortMax entries are sorted on the
// host instead.
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

// Entry of a row that its stored position q holds: full kPermBlock-entry
// blocks are stored transposed (position 4 l + i holds entry 16 i + l).
__device__ __forceinline__ int stored_entry(int q, int plen) {
  const int b = q / kPermBlock, w = q % kPermBlock;
  return b < plen / kPermBlock ? b * kPermBlock + 16 * (w & 3) + (w >> 2) : q;
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

// Row r of the stored matrix from entry rp[r] on, in the input's order.
template <typename VT>
__global__ void __launch_bounds__(kRowThreads)
    k_fill_rows(int64_t rows, const int64_t* __restrict__ rp, const int32_t* __restrict__ prp,
                const int32_t* __restrict__ prl, const int32_t* __restrict__ ci,
                const double* __restrict__ vv, int32_t* __restrict__ col, VT* __restrict__ val) {
  const int lane = threadIdx.x & 31;
  const int64_t r = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (r >= rows) return;
  const int64_t a = rp[r];
  const int len = (int)(rp[r + 1] - a), plen = prl[r];
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
// entries per lane; wide[0] / wide[1] set where a block / unit spans 2^16
// columns or more.  With off: the offsets from the blocks' (by_block) or units'
// smallest column, and that column for every unit.
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
    if (!off) {
      if (lane == 0) {
        bbase[rblk[r] + b] = blo;
        if (bhi - blo > 65535) wide[0] = 1;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (in[h] && hi[h] - lo[h] > 65535) wide[1] = 1;
      continue;
    }
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

// Padded layout of rows of the given lengths.
struct Layout {
  std::vector<int32_t> ptr, len, blk;
  int64_t tot = 0, blocks = 0;
};
template <typename Len>
bool make_layout(int64_t rows, Len len, Layout& l) {
  const int64_t nrp = (rows + 1 + 3) / 4 * 4;  // row pointers padded to a multiple of 4 entries
  l.ptr.resize(nrp);
  l.len.resize(rows);
  l.blk.resize(rows);
  for (int64_t r = 0; r < rows; ++r) {
    const int64_t plen = (len(r) + kRowAlign - 1) / kRowAlign * kRowAlign;
    l.ptr[r] = (int32_t)l.tot;
    l.len[r] = (int32_t)plen;
    l.blk[r] = (int32_t)l.blocks;
    l.tot += plen;
    l.blocks += (plen + kPermBlock - 1) / kPermBlock;
    if (l.tot >= (int64_t)INT32_MAX) return false;
  }
  for (int64_t i = rows; i < nrp; ++i) l.ptr[i] = (int32_t)l.tot;
  return true;
}

#define CE(call)                             \
  do {                                       \
    const cudaError_t e_ = (call);           \
    if (e_ != cudaSuccess) return e_;        \
  } while (0)

template <typename T>
cudaError_t upload(T** dst, const T* src, size_t count, size_t at_least, cudaStream_t s) {
  CE(cudaMalloc((void**)dst, std::max(count, at_least) * sizeof(T)));
  return count ? cudaMemcpyAsync(*dst, src, count * sizeof(T), cudaMemcpyHostToDevice, s)
               : cudaSuccess;
}

// The arrays of a stored matrix, columns and values still to be filled.
cudaError_t allocate(const Layout& l, int64_t rows, int64_t cols, int64_t nnz, int vt, DevCsr* out,
                     cudaStream_t s) {
  out->rows = rows;
  out->cols = cols;
  out->nnz = nnz;
  out->nnz_padded = l.tot;
  const size_t vbytes = vt == LSLU_F64 ? 8 : vt == LSLU_F32 ? 4 : 2;
  const int64_t cap = std::max<int64_t>(l.tot, kRowAlign);
  CE(upload(&out->row_ptr, l.ptr.data(), l.ptr.size(), 1, s));
  CE(upload(&out->row_len, l.len.data(), l.len.size(), 1, s));
  CE(upload(&out->rblk, l.blk.data(), l.blk.size(), 1, s));
  CE(cudaMalloc((void**)&out->bbase, std::max<int64_t>(l.blocks, 1) * sizeof(int32_t)));
  CE(cudaMalloc((void**)&out->col, cap * sizeof(int32_t)));
  return cudaMalloc(&out->val, cap * vbytes);
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

void fill_rows(const DevCsr& A, int vt, const int64_t* rp, const int32_t* ci, const double* vv,
               cudaStream_t s) {
  if (A.nnz_padded == 0) return;
  with_value_type(vt, A.val, [&](auto* v) {
    k_fill_rows<<<warps_grid(A.rows), kRowThreads, 0, s>>>(A.rows, rp, A.row_ptr, A.row_len, ci,
                                                           vv, A.col, v);
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

// 16-bit column offsets, from the smallest column of every block where all
// blocks span fewer than 2^16 columns, else of every unit where those do.
cudaError_t add_offsets(DevCsr* A, const int (&wide)[2], cudaStream_t s) {
  A->block_compressed = A->nnz_padded > 0 && !wide[0];
  A->compressed = A->nnz_padded > 0 && !wide[1];
  if (A->block_compressed) A->compressed = 1;  // a unit lies inside one block
  if (!A->block_compressed) {
    cudaFree(A->bbase);
    cudaFree(A->rblk);
    A->bbase = A->rblk = nullptr;
  }
  if (!A->compressed) return cudaSuccess;
  // unit bases readable up to a multiple of 4 units
  const int64_t nub = (A->nnz_padded / kRowAlign + 3) / 4 * 4;
  CE(cudaMalloc((void**)&A->off, A->nnz_padded * sizeof(uint16_t)));
  CE(cudaMalloc((void**)&A->ubase, nub * sizeof(int32_t)));
  CE(cudaMemsetAsync(A->ubase, 0, nub * sizeof(int32_t), s));
  k_offsets<<<warps_grid(A->rows), kRowThreads, 0, s>>>(A->rows, A->row_ptr, A->row_len, A->rblk,
                                                        A->col, A->bbase, nullptr,
                                                        A->block_compressed != 0, A->off, A->ubase);
  return cudaGetLastError();
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

struct Scratch {  // one allocation for everything the construction needs for itself
  char* base = nullptr;
  size_t used = 0;
  ~Scratch() { cudaFree(base); }
  template <typename T>
  T* take(size_t count) {
    T* p = reinterpret_cast<T*>(base + used);
    used += (count * sizeof(T) + 255) / 256 * 256;
    return p;
  }
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
  CE(cudaMalloc((void**)&mem.base, 256));
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

cudaError_t build_csr_pair(int64_t m, int64_t n, const int64_t* rp, const int32_t* ci,
                           const double* vv, bool on_device, const std::vector<int32_t>* inv_row,
                           const std::vector<int32_t>* col_new, int vt, DevCsr* A, DevCsr* AT,
                           cudaStream_t s) {
  A->shape = AT->shape = default_shape(vt);
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess)
    cudaDeviceGetAttribute(&A->num_sms, cudaDevAttrMultiProcessorCount, dev);
  AT->num_sms = A->num_sms;
  const int64_t nnz = rp[m];
  auto row_len = [&](int64_t r) {
    const int64_t src = inv_row ? (*inv_row)[r] : r;
    return rp[src + 1] - rp[src];
  };
  Layout la, lt;
  if (!make_layout(m, row_len, la)) return cudaErrorInvalidValue;
  int64_t max_row = 0;
  for (int64_t r = 0; r < m; ++r) max_row = std::max(max_row, rp[r + 1] - rp[r]);
  // every host array that an asynchronous copy reads lives until the final
  // synchronisation
  std::vector<int32_t> cnt(n), first(n + 1, 0);
  std::vector<int64_t> rp_a, rp_t;
  std::vector<int32_t> ci_h, ci_a, ci_t;
  std::vector<double> vv_h, vv_a, vv_t;
  Scratch mem;
  const size_t e1 = (size_t)std::max<int64_t>(nnz, 1);
  const size_t bytes = (size_t)(m + 1) * 8 + (size_t)(n + 1) * 8 + (n + 1) * 16 + m * 4 +
                       e1 * (8 + 2 * (4 + 8)) + 16 * 256;
  CE(cudaMalloc((void**)&mem.base, bytes));
  int64_t* d_rp = mem.take<int64_t>(m + 1);
  int64_t* d_rpt = mem.take<int64_t>(n + 1);
  int32_t* d_cnt = mem.take<int32_t>(n);
  int32_t* d_first = mem.take<int32_t>(n + 1);
  int32_t* d_inv = mem.take<int32_t>(m);
  int32_t* d_new = mem.take<int32_t>(n);
  int* d_wide = mem.take<int>(4);
  unsigned long long* d_keys = mem.take<unsigned long long>(e1);
  int32_t* d_ci = mem.take<int32_t>(e1);
  double* d_vv = mem.take<double>(e1);
  auto to_device = [&](auto* dst, const auto* src, size_t count) {
    return count ? cudaMemcpyAsync(dst, src, count * sizeof(*dst), cudaMemcpyHostToDevice, s)
                 : cudaSuccess;
  };
  const int32_t* c_in = ci;
  const double* v_in = vv;
  if (!on_device) {
    CE(to_device(d_ci, ci, nnz));
    CE(to_device(d_vv, vv, nnz));
    c_in = d_ci;
    v_in = d_vv;
  }
  CE(to_device(d_rp, rp, m + 1));
  if (inv_row) CE(to_device(d_inv, inv_row->data(), m));
  if (col_new) CE(to_device(d_new, col_new->data(), n));
  CE(cudaMemsetAsync(d_wide, 0, 4 * sizeof(int), s));
  CE(cudaMemsetAsync(d_cnt, 0, n * sizeof(int32_t), s));
  if (nnz)
    k_count<<<(unsigned)std::min<int64_t>((nnz + 255) / 256, 8192), 256, 0, s>>>(
        nnz, c_in, col_new ? d_new : nullptr, d_cnt);
  CE(cudaMemcpyAsync(cnt.data(), d_cnt, n * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  CE(allocate(la, m, n, nnz, vt, A, s));
  CE(cudaStreamSynchronize(s));
  int64_t max_col = 0;
  for (int64_t c = 0; c < n; ++c) {
    first[c + 1] = first[c] + cnt[c];
    max_col = std::max<int64_t>(max_col, cnt[c]);
  }
  if (!make_layout(n, [&](int64_t c) { return (int64_t)cnt[c]; }, lt)) return cudaErrorInvalidValue;
  CE(allocate(lt, n, m, nnz, vt, AT, s));
  if (max_col > kSortMax || (inv_row && max_row > kSortMax)) {
    // a row or column too long for one block's shared memory: host sorts
    if (on_device) {
      ci_h.resize(nnz);
      vv_h.resize(nnz);
      CE(cudaMemcpy(ci_h.data(), ci, nnz * 4, cudaMemcpyDeviceToHost));
      CE(cudaMemcpy(vv_h.data(), vv, nnz * 8, cudaMemcpyDeviceToHost));
      ci = ci_h.data();
      vv = vv_h.data();
    }
    if (inv_row) {
      renumber_csr(m, rp, ci, vv, *inv_row, *col_new, rp_a, ci_a, vv_a);
      rp = rp_a.data();
      ci = ci_a.data();
      vv = vv_a.data();
    }
    transpose_host(m, n, rp, ci, vv, rp_t, ci_t, vv_t);
    CE(to_device(d_rp, rp, m + 1));
    CE(to_device(d_ci, ci, nnz));
    CE(to_device(d_vv, vv, nnz));
    fill_rows(*A, vt, d_rp, d_ci, d_vv, s);
    CE(to_device(d_rpt, rp_t.data(), n + 1));
    CE(to_device(d_ci, ci_t.data(), nnz));
    CE(to_device(d_vv, vv_t.data(), nnz));
    fill_rows(*AT, vt, d_rpt, d_ci, d_vv, s);
  } else {
    CE(to_device(d_first, first.data(), n + 1));
    CE(cudaMemcpyAsync(d_cnt, d_first, n * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
    if (nnz)
      k_scatter_keys<<<warps_grid(m), kRowThreads, 0, s>>>(m, d_rp, c_in, inv_row ? d_inv : nullptr,
                                                           col_new ? d_new : nullptr, d_cnt, d_keys);
    if (inv_row)
      CE(sort_fill(*A, vt, (int)max_row, nullptr, nullptr, d_rp, d_inv, d_new, c_in, v_in, s));
    else
      fill_rows(*A, vt, d_rp, c_in, v_in, s);
    CE(sort_fill(*AT, vt, (int)max_col, d_keys, d_first, nullptr, nullptr, nullptr, c_in, v_in, s));
  }
  int wide[2][2] = {{0, 0}, {0, 0}};
  DevCsr* both[2] = {A, AT};
  for (int w = 0; w < 2; ++w)
    if (both[w]->nnz_padded)
      k_offsets<<<warps_grid(both[w]->rows), kRowThreads, 0, s>>>(
          both[w]->rows, both[w]->row_ptr, both[w]->row_len, both[w]->rblk, both[w]->col,
          both[w]->bbase, d_wide + 2 * w, false, nullptr, nullptr);
  CE(cudaGetLastError());
  CE(cudaMemcpyAsync(wide, d_wide, sizeof(wide), cudaMemcpyDeviceToHost, s));
  CE(cudaStreamSynchronize(s));
  CE(add_offsets(A, wide[0], s));
  CE(add_offsets(AT, wide[1], s));
  return cudaStreamSynchronize(s);
}

void free_csr(DevCsr* c) {
  cudaFree(c->row_ptr);
  cudaFree(c->row_len);
  cudaFree(c->col);
  cudaFree(c->val);
  cudaFree(c->off);
  cudaFree(c->ubase);
  cudaFree(c->bbase);
  cudaFree(c->rblk);
  *c = DevCsr();
}

}  // namespace lslu
