// Sparse products of Algorithm 4: u = A l_k and q = A^T d_k (host side,
// default row shapes, and the products of right-hand sides sharing one
// matrix).  The device code of the single-vector products is in
// lslu_spmv_impl.cuh; the default shape is 16 lanes per row with two chunks
// in flight (one for FP64 values); other shapes, chosen per matrix by
// lslu_tune_spmv, are instantiated in lslu_spmv_shapes.cu.
#include <cuda_runtime.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>
#include <type_traits>
#include <vector>

#include "lslu_spmv_impl.cuh"

namespace lslu {

namespace {

constexpr int kGroup = 16;  // lanes per row of the shared-matrix product

// ---- several right-hand sides sharing one matrix ---------------------------
// The R input vectors are first interleaved, xi[j * RS + r] (RS = R rounded
// up to 4, zero-padded), so each non-zero fetches all R values with RS/4
// 16-byte loads and the matrix is read once for all R products.  Lane gl of a
// row's 16-lane group takes the same chunks in the same order as row_dot_len,
// and each right-hand side keeps its own accumulator, so every output equals
// the single-vector product of the default 16-lane shapes bit for bit (16x2 on
// 32-bit columns, 16x1 on 16-bit offsets).

template <int F>
constexpr int kFmtChunk = F == kFmtUnit8 ? 8 : 4;

// Columns of the lane's next chunk (entry e of the row, at position p of the
// storage): 8 entries in kFmtUnit8, else 4.
template <int F>
__device__ __forceinline__ void chunk_cols(const ColIdx& ci, int32_t p, int32_t e, int32_t blk,
                                           int32_t (&c)[kFmtChunk<F>]) {
  if constexpr (F == kFmtUnit4 || F == kFmtBlock4) {
    const uint2 o = ld_stream_off4(ci.off + p);
    const int32_t b =
        F == kFmtBlock4 ? __ldg(ci.bbase + blk + e / kPermBlock) : __ldg(ci.ubase + (p >> 3));
    c[0] = b + (int32_t)(o.x & 0xffffu);
    c[1] = b + (int32_t)(o.x >> 16);
    c[2] = b + (int32_t)(o.y & 0xffffu);
    c[3] = b + (int32_t)(o.y >> 16);
  } else if constexpr (F == kFmtUnit8) {
    const uint4 o = ld_stream_off(ci.off + p);
    const int32_t b = __ldg(ci.ubase + (p >> 3));
    const uint32_t w[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      c[2 * q] = b + (int32_t)(w[q] & 0xffffu);
      c[2 * q + 1] = b + (int32_t)(w[q] >> 16);
    }
  } else {
    const int4 c4 = ld_stream(ci.col + p);
    c[0] = c4.x; c[1] = c4.y; c[2] = c4.z; c[3] = c4.w;
  }
}

template <typename VT, int F>
__device__ __forceinline__ void chunk_vals(const VT* val, int32_t p, float (&v)[kFmtChunk<F>]) {
  if constexpr (F == kFmtUnit8)
    load_vals8<float>(val + p, v);
  else
    load_vals_cs<float>(val + p, v);
}

// Product of CSR row `row` with right-hand side r of the interleaved xi, in
// the chunk order of the single-vector default shape (16 lanes).
template <typename VT, int RS, int F>
__device__ __forceinline__ float row_dot_rhs(int64_t row, const int32_t* __restrict__ rp,
                                             const int32_t* __restrict__ rl, const ColIdx ci,
                                             const VT* __restrict__ val,
                                             const float* __restrict__ xi, int r, int gl) {
  constexpr int C = kFmtChunk<F>;
  constexpr int S = kGroup * C;
  const int32_t start = __ldg(rp + row), len = __ldg(rl + row);
  const int32_t blk = F == kFmtBlock4 ? __ldg(ci.rblk + row) : 0;
  float acc = 0.f;
  for (int32_t e = gl * C; e < len; e += S) {
    int32_t c[C];
    float v[C];
    chunk_cols<F>(ci, start + e, e, blk, c);
    chunk_vals<VT, F>(val, start + e, v);
#pragma unroll
    for (int i = 0; i < C; ++i) acc = fmaf(v[i], __ldg(xi + (int64_t)c[i] * RS + r), acc);
  }
  return group_sum<kGroup>(acc);
}

// y[r * ystride + row] = (A xi_r)(row) for r < R, rows of the shared CSR;
// pivot blocks as in k_spmv_pivots, with output rows of problem p at
// p * ystride + row.
// RS / 4 threads stand for one lane of the single-vector group, each with four
// right-hand sides, so a gather request reads whole 4 RS-byte rows of xi (one
// thread gathering all of them took RS / 4 requests of 32 scattered 16-byte
// pieces, and the L1's tag lookups bounded the product).  A warp takes one row
// with RS = 16 (two of the 16 lanes per thread group, kept as separate
// accumulators) or RS = 8, and two rows with RS = 4; the sums and the butterfly
// are those of the 16 lanes, so every output keeps its bits.
// 256x256 CT, 16 right-hand sides, K = 50: 163 -> 77 us per product, the solve
// 21.0 -> 12.4 ms (all gathers of a step ahead of its sums: 12.8 to 13.8 ms).
template <typename VT, int RS, int F>
__global__ void __launch_bounds__(256)
    k_spmm_pivots(int64_t rows, const int32_t* __restrict__ rp, const int32_t* __restrict__ rl,
                  const ColIdx ci, const VT* __restrict__ val, const float* __restrict__ xi,
                  float* __restrict__ y, int64_t ystride, int R, PivotCoef pc) {
  constexpr int C = kFmtChunk<F>;
  constexpr int S = kGroup * C;
  constexpr int T = RS / 4;                     // threads of one lane
  constexpr int V = T == 4 ? 2 : 1;             // lanes per thread
  constexpr int TEAM = kGroup / V * T;          // threads of one row
  constexpr int RPB = 256 / TEAM;               // rows of a block
  const int npiv_all = pc.npiv_blocks * pc.nprob;
  if ((int)blockIdx.x < npiv_all) {
    pivot_blocks<float, kGroup>(pc, [=](int p, int32_t row, int gl) {
      return row_dot_rhs<VT, RS, F>((int64_t)row - (int64_t)p * ystride, rp, rl, ci, val, xi,
                                      p, gl);
    });
    return;
  }
  const int64_t row = (int64_t)(blockIdx.x - npiv_all) * RPB + threadIdx.x / TEAM;
  if (row - (threadIdx.x & 31) / TEAM >= rows) return;  // whole warp past the end
  const bool valid = row < rows;
  const int t = threadIdx.x % T;                     // right-hand sides 4 t .. 4 t + 3
  const int l0 = (threadIdx.x % TEAM) / T * V;       // first lane
  const RowAt at = row_at<F>(row, valid, rp, rl, ci);
  const float4* x4 = reinterpret_cast<const float4*>(xi) + t;
  float acc[V][4];
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[v][q] = 0.f;
  for (int32_t e = l0 * C; e < at.len; e += S) {
    int32_t cs[V][C];
    float a[V][C];
#pragma unroll
    for (int v = 0; v < V; ++v) {
      if (v == 0 || e + v * C < at.len) {
        chunk_cols<F>(ci, at.start + e + v * C, e, at.blk, cs[v]);
        chunk_vals<VT, F>(val, at.start + e + v * C, a[v]);
      } else {
#pragma unroll
        for (int i = 0; i < C; ++i) {
          cs[v][i] = 0;
          a[v][i] = 0.f;
        }
      }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) {
      if (v > 0 && e + v * C >= at.len) break;  // lane v has no chunk left
#pragma unroll
      for (int i = 0; i < C; ++i) {
        const float4 xv = __ldg(x4 + (int64_t)cs[v][i] * T);
        acc[v][0] = fmaf(a[v][i], xv.x, acc[v][0]);
        acc[v][1] = fmaf(a[v][i], xv.y, acc[v][1]);
        acc[v][2] = fmaf(a[v][i], xv.z, acc[v][2]);
        acc[v][3] = fmaf(a[v][i], xv.w, acc[v][3]);
      }
    }
  }
  // the 16-lane butterfly: lanes 8, 4, 2, 1 apart
#pragma unroll
  for (int v = 0; v < V; ++v)
#pragma unroll
    for (int o = TEAM / 2; o >= T; o >>= 1)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[v][q] += __shfl_xor_sync(0xffffffffu, acc[v][q], o);
  if (!valid || l0 != 0) return;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float sum = V == 2 ? acc[0][q] + acc[V - 1][q] : acc[0][q];
    if (4 * t + q < R) y[(int64_t)(4 * t + q) * ystride + row] = sum;
  }
}

// xi[j * RS + r] = x[r * xstride + j] (r < R), 0 for R <= r < RS.
template <int RS>
__global__ void k_interleave(const float* __restrict__ x, int64_t xstride, int64_t count, int R,
                             float* __restrict__ xi) {
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < count;
       j += (int64_t)gridDim.x * blockDim.x) {
    float4* o = reinterpret_cast<float4*>(xi + j * RS);
#pragma unroll
    for (int q = 0; q < RS / 4; ++q) {
      float t[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int r = 4 * q + e;
        t[e] = r < R ? x[(int64_t)r * xstride + j] : 0.f;
      }
      o[q] = make_float4(t[0], t[1], t[2], t[3]);
    }
  }
}

}  // namespace

// 16 lanes per row with 8 entries in flight per lane (two 4-entry chunks of
// 32-bit columns); FP64 values keep 4 in flight (registers).
int default_shape(int vt) { return vt == LSLU_F64 ? kShapeG16U1 : kShapeG16U2; }

namespace {

// The value type's native vector type: FP64 basis for FP64 values, FP32 basis
// otherwise.  Only native products use the tuned shapes.
template <typename XT, typename YT>
bool native(int vt) {
  if (!std::is_same<XT, YT>::value) return false;
  return (vt == LSLU_F64) == std::is_same<XT, double>::value;
}

// Calls f with a value of the FP32 / BF16 storage type and the chunks in
// flight of the form (an integral_constant).
template <typename Fn>
void with_form(int form, int vt, Fn f) {
  auto chunks = [&](auto v) {
    if (form == kFormStream)
      f(v, std::integral_constant<int, 4>{});
    else
      f(v, std::integral_constant<int, 2>{});
  };
  if (vt == LSLU_F32)
    chunks(float{});
  else
    chunks(__nv_bfloat16{});
}

}  // namespace

// Native products (FP64 vectors for FP64 values, FP32 otherwise) run in the
// matrix's shape and column format; the others (FP64 vectors on FP32 / BF16
// values: r0 with x0, the adjoint's x0 term) in the default shape.
template <typename XT, typename YT>
void launch_spmv(const DevCsr& A, int vt, const XT* x, YT* y, cudaStream_t s, int) {
  if (native<XT, YT>(vt) && A.shape != default_shape(vt)) {
    launch_spmv_shape(A.shape, A, vt, x, y, s);
    return;
  }
  if constexpr (std::is_same<XT, float>::value) {
    if (A.form != kFormPlain) {
      with_form(A.form, vt, [&](auto v, auto u) {
        spmv_run<decltype(v), XT, YT, 16, decltype(u)::value, true>(A, x, y, s);
      });
      return;
    }
  }
  if (vt == LSLU_F64)
    spmv_run<double, XT, YT, 16, 1>(A, x, y, s);
  else if (vt == LSLU_F32)
    spmv_run<float, XT, YT, 16, 2>(A, x, y, s);
  else
    spmv_run<__nv_bfloat16, XT, YT, 16, 2>(A, x, y, s);
}

template <typename XT, typename YT>
void launch_spmv_pivots(const DevCsr& A, int vt, const XT* x, YT* y, PivotCoef pc,
                        cudaStream_t s) {
  pc.npiv_blocks = (pc.cnt + 7) / 8;
  if (native<XT, YT>(vt) && A.shape != default_shape(vt)) {
    launch_spmv_pivots_shape(A.shape, A, vt, x, y, pc, s);
    return;
  }
  if constexpr (std::is_same<XT, float>::value) {
    if (A.form != kFormPlain) {
      with_form(A.form, vt, [&](auto v, auto u) {
        spmv_pivots_run<decltype(v), XT, YT, 16, decltype(u)::value, true>(A, x, y, pc, s);
      });
      return;
    }
  }
  if (vt == LSLU_F64)
    spmv_pivots_run<double, XT, YT, 16, 1>(A, x, y, pc, s);
  else if (vt == LSLU_F32)
    spmv_pivots_run<float, XT, YT, 16, 2>(A, x, y, pc, s);
  else
    spmv_pivots_run<__nv_bfloat16, XT, YT, 16, 2>(A, x, y, pc, s);
}

template <typename VT, int RS>
void spmm_typed(const DevCsr& A, const float* xi, float* y, int64_t ystride, int R,
                const PivotCoef& pc, cudaStream_t s) {
  constexpr int kRows = RS == 4 ? 16 : 8;  // rows per block (k_spmm_pivots)
  const int64_t blocks = (int64_t)pc.npiv_blocks * pc.nprob + (A.rows + kRows - 1) / kRows;
  const VT* v = reinterpret_cast<const VT*>(A.val);
  auto run = [&](auto F) {
    k_spmm_pivots<VT, RS, F.value><<<(unsigned)blocks, 256, 0, s>>>(
        A.rows, A.row_ptr, A.row_len, col_idx(A), v, xi, y, ystride, R, pc);
  };
  if (A.nnz_padded >= kStreamMinEntries && !A.use_cmp)
    with_format<true>(A, run);
  else
    with_format<false>(A, run);
}

template <typename VT>
void spmm_rs(const DevCsr& A, const float* xi, float* y, int64_t ystride, int R, int RS,
             const PivotCoef& pc, cudaStream_t s) {
  if (RS == 4)
    spmm_typed<VT, 4>(A, xi, y, ystride, R, pc, s);
  else if (RS == 8)
    spmm_typed<VT, 8>(A, xi, y, ystride, R, pc, s);
  else
    spmm_typed<VT, 16>(A, xi, y, ystride, R, pc, s);
}

int rhs_stride(int R) { return R <= 4 ? 4 : (R <= 8 ? 8 : 16); }

namespace {
// Reads n 16-byte words through L2 (clean lines, as the elimination leaves
// them before a product) and stores one word so the reads are not dropped.
__global__ void k_l2_flush(const int4* __restrict__ p, int64_t n, int* sink) {
  int acc = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int4 v = __ldcg(p + i);
    acc ^= v.x ^ v.y ^ v.z ^ v.w;
  }
  if (acc == 0x7fffffff) *sink = acc;  // practically never; keeps the loads
}
}  // namespace

void launch_l2_flush(const void* buf, size_t bytes, int* sink, cudaStream_t s, int num_sms) {
  const int64_t n = (int64_t)(bytes / 16);
  k_l2_flush<<<num_sms * 8, 256, 0, s>>>(reinterpret_cast<const int4*>(buf), n, sink);
}

void launch_interleave(const float* x, int64_t xstride, int64_t count, int R, float* xi,
                       cudaStream_t s, int num_sms) {
  const int RS = rhs_stride(R);
  const int g = (int)std::min<int64_t>((count + 255) / 256, (int64_t)num_sms * 8);
  if (RS == 4)
    k_interleave<4><<<g, 256, 0, s>>>(x, xstride, count, R, xi);
  else if (RS == 8)
    k_interleave<8><<<g, 256, 0, s>>>(x, xstride, count, R, xi);
  else
    k_interleave<16><<<g, 256, 0, s>>>(x, xstride, count, R, xi);
}

void launch_spmm_pivots(const DevCsr& A, int vt, const float* xi, float* y, int64_t ystride,
                        int R, PivotCoef pc, cudaStream_t s) {
  pc.npiv_blocks = (pc.cnt + 7) / 8;
  const int RS = rhs_stride(R);
  if (vt == LSLU_BF16)
    spmm_rs<__nv_bfloat16>(A, xi, y, ystride, R, RS, pc, s);
  else
    spmm_rs<float>(A, xi, y, ystride, R, RS, pc, s);
}

template void launch_spmv<double, double>(const DevCsr&, int, const double*, double*,
                                          cudaStream_t, int);
template void launch_spmv<float, float>(const DevCsr&, int, const float*, float*, cudaStream_t,
                                        int);
template void launch_spmv_pivots<double, double>(const DevCsr&, int, const double*, double*,
                                                 PivotCoef, cudaStream_t);
template void launch_spmv_pivots<float, float>(const DevCsr&, int, const float*, float*,
                                               PivotCoef, cudaStream_t);

}  // namespace lslu
