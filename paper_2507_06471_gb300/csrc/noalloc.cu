// cd_modularity_noalloc: modularity of a partition computed without any
// device allocation, for callers that cannot call cudaMalloc (for example a
// host process whose device memory is entirely owned and budgeted by another
// allocator, where an extra driver allocation may fail or is not permitted).
//
// The per-community volume accumulators and the few control words live in one
// file-scope static __device__ array, g_noalloc_scratch, sized for at most
// kNoallocMaxN vertices: 16 MiB that every GPU which loads the library keeps
// until the process exits. Host code cannot use the array's name as a device
// address; on the first call on each device (with that device current) the
// entry point looks the address up once with cudaGetSymbolAddress and keeps
// it, and loads the entry point's kernels. That first call should therefore
// come before any stream capture on the device. The kept address belongs to
// the device's primary context: after cudaDeviceReset the library must not be
// used again in the process.
//
// All calls share the one array and it keeps the previous call's contents, so
// each call first clears the part it uses. Calls whose work overlaps on the
// GPU (different streams, or different host threads, without ordering between
// them) race on the array and must not be issued.
#include <mutex>

#include "common.cuh"
#include "rowwalk.cuh"

namespace {

constexpr int64_t kNoallocMaxN = 1 << 21;  // vertices (and community ids) at most
// S low, S high, I, vol(V), status of the offsets and labels, status of the arcs
constexpr int kCtlWords = 8;
constexpr int NT = 256;

static __device__ __align__(256) unsigned long long g_noalloc_scratch[kCtlWords + kNoallocMaxN];  // control words first: one clear covers a call

constexpr int kMaxDevices = 64;
unsigned long long* g_scratch_dev[kMaxDevices] = {};
std::mutex g_scratch_mu;

cudaError_t load_kernels();

int scratch_on_current_device(unsigned long long** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cd::set_cuda_error(e);
  if (dev < 0 || dev >= kMaxDevices) return CD_EINVAL;
  std::lock_guard<std::mutex> lock(g_scratch_mu);
  if (!g_scratch_dev[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return cd::set_cuda_error(e);
    // With lazy module loading a kernel's code is loaded, which can take
    // device memory, at its first launch; load all of this entry point's
    // kernels now so that no later call (weighted or not) loads anything.
    if ((e = load_kernels()) != cudaSuccess) return cd::set_cuda_error(e);
    g_scratch_dev[dev] = (unsigned long long*)p;
  }
  *out = g_scratch_dev[dev];
  return CD_OK;
}

__device__ __forceinline__ void na_fail(unsigned long long* word, int code) {
  atomicCAS(word, 0ull, (unsigned long long)(unsigned)(-code));
}

// deg_w(v) (a loop counted twice) into the volume of v's community, the weight
// of arcs inside communities (a loop arc counts 2L) and vol(V). The arcs are
// split evenly over the warps (rowwalk.cuh), so a long row is no serial chain;
// columns and weights are read 4 bytes at a time, since the caller's arrays may
// start anywhere. Every index is checked before use; a bad one sets a status
// word: offsets and labels are checked by vertex, and their word is reported
// before that of the arcs, whose rows mean nothing if the offsets are bad.
template <bool UNIT>
__global__ void __launch_bounds__(NT) k_noalloc_pass(const int64_t* __restrict__ off,
                                                     const int32_t* __restrict__ cols,
                                                     const int32_t* __restrict__ w,
                                                     const int32_t* __restrict__ labels, int64_t n,
                                                     int64_t nnz, unsigned long long* scratch) {
  __shared__ __align__(16) int32_t mark[NT / 32][cd::WALK_TILE];
  __shared__ cd::CtaSums vol;
  vol.clear();
  __syncthreads();
  unsigned long long* ctl = scratch;
  unsigned long long* volc = scratch + kCtlWords;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t tid = (int64_t)blockIdx.x * NT + threadIdx.x;
  const int64_t threads = (int64_t)gridDim.x * NT;
  for (int64_t v = tid; v < n; v += threads) {
    const int32_t a = labels[v];
    const int64_t beg = off[v], end = off[v + 1];
    if (a < 0 || a >= n) na_fail(&ctl[4], CD_EINVAL);
    else if (beg < 0 || end < beg || end > nnz) na_fail(&ctl[4], CD_ENOTSYM);
  }
  int64_t m0 = off[0], m1 = off[n];  // the rows' arcs
  if (m0 < 0) m0 = 0;
  if (m1 > nnz) m1 = nnz;
  const int64_t piece = cd::walk_piece(m1 - m0, threads >> 5);
  unsigned long long my_in = 0, my_vol = 0;
  for (int64_t e0 = m0 + (tid >> 5) * piece; e0 < m1; e0 += (threads >> 5) * piece) {  // uniform in the warp
    const int64_t e1 = e0 + piece < m1 ? e0 + piece : m1;
    int32_t un[4], xn[4];  // the next tile's columns and weights, in flight during this one's
    auto load = [&](int64_t e) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        un[j] = e + j < e1 ? cols[e + j] : -1;
        xn[j] = UNIT || e + j >= e1 ? 1 : w[e + j];
      }
    };
    load(e0 + 4 * lane);
    int64_t cur = cd::warp_row_of(off, n, e0);
    for (int64_t ts = e0; ts < e1; ts += cd::WALK_TILE) {
      const int64_t e = ts + 4 * lane;
      int32_t u[4];
      long long x[4];
      int64_t row[4];
      unsigned long long val[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        u[j] = un[j];
        x[j] = xn[j];
      }
      if (ts + cd::WALK_TILE < e1) load(e + cd::WALK_TILE);
      cd::warp_tile_rows(off, n, ts, cur, mark[wid], row);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        val[j] = 0;
        if (e + j >= e1) {
          row[j] = -1;
          continue;
        }
        if (u[j] < 0 || u[j] >= n) {  // reported before the arc's weight
          na_fail(&ctl[5], CD_EBOUNDS);
          continue;
        }
        if (x[j] < 1) na_fail(&ctl[5], CD_EINVAL);
        val[j] = (unsigned long long)(u[j] == row[j] ? 2 * x[j] : x[j]);
        my_vol += val[j];
        if (labels[u[j]] == labels[row[j]]) my_in += val[j];
      }
      cd::warp_rows_sum(row, val, [&](int64_t r, unsigned long long sum) {
        const int32_t a = labels[r];
        if (a >= 0 && a < n) vol.add(volc, a, sum);
      });
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    my_in += __shfl_xor_sync(cd::FULL, my_in, o);
    my_vol += __shfl_xor_sync(cd::FULL, my_vol, o);
  }
  if (lane == 0) {
    if (my_in) atomicAdd(&ctl[2], my_in);
    if (my_vol) atomicAdd(&ctl[3], my_vol);
  }
  __syncthreads();
  vol.flush(volc);
}

// Sum of squared community volumes, exact in 128 bits (ctl[0] low, ctl[1] high).
__global__ void __launch_bounds__(NT) k_noalloc_square(int64_t n, unsigned long long* scratch) {
  __shared__ unsigned __int128 part[NT];
  const unsigned long long* volc = scratch + kCtlWords;
  unsigned long long* ctl = scratch;
  unsigned __int128 s = 0;
  const int64_t stride = (int64_t)gridDim.x * NT;
  for (int64_t c = (int64_t)blockIdx.x * NT + threadIdx.x; c < n; c += stride)
    s += (unsigned __int128)volc[c] * volc[c];
  part[threadIdx.x] = s;
  __syncthreads();
  for (int o = NT / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) part[threadIdx.x] += part[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0 && part[0]) {
    const unsigned long long lo = (unsigned long long)part[0], hi = (unsigned long long)(part[0] >> 64);
    const unsigned long long old = atomicAdd(&ctl[0], lo);
    const unsigned long long carry = old + lo < old ? 1ull : 0ull;
    if (hi + carry) atomicAdd(&ctl[1], hi + carry);
  }
}

cudaError_t load_kernels() {
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, k_noalloc_pass<true>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_noalloc_pass<false>);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&a, k_noalloc_square);
  return e;
}

}  // namespace

extern "C" int cd_modularity_noalloc(const int64_t* off, const int32_t* cols, const int32_t* w,
                                     const int32_t* labels, int64_t n, int64_t nnz, void* stream,
                                     double* q_out) {
  if (!q_out || n < 0 || nnz < 0 || (n > 0 && (!off || !labels)) || (nnz > 0 && !cols))
    return CD_EINVAL;
  if (n > kNoallocMaxN) return CD_EINVAL;  // larger than the static scratch
  cudaStream_t s = (cudaStream_t)stream;
  unsigned long long* scratch = nullptr;
  int rc = scratch_on_current_device(&scratch);
  if (rc) return rc;
  CD_CHECK(cudaMemsetAsync(scratch, 0, (size_t)(kCtlWords + n) * sizeof(unsigned long long), s));
  if (n > 0) {
    // from 1,024 arcs or vertices a CTA up to two CTAs per SM (latency), then 4,096 (each popular community
    // costs a CTA one atomic), 8 CTAs per SM at most
    const int64_t work = nnz > n ? nnz : n;
    int64_t blocks = (work + 1023) / 1024;
    if (blocks > 304) blocks = work / 4096 < 304 ? 304 : work / 4096 < 152 * 8 ? work / 4096 : 152 * 8;
    const unsigned grid = (unsigned)blocks;
    if (w)
      CD_LAUNCH(k_noalloc_pass<false><<<grid, NT, 0, s>>>(off, cols, w, labels, n, nnz, scratch));
    else
      CD_LAUNCH(k_noalloc_pass<true><<<grid, NT, 0, s>>>(off, cols, w, labels, n, nnz, scratch));
    int64_t sb = (n + NT - 1) / NT;
    CD_LAUNCH(k_noalloc_square<<<(unsigned)(sb < 152 * 4 ? sb : 152 * 4), NT, 0, s>>>(n, scratch));
    CD_CHECK(cudaGetLastError());
  }
  unsigned long long h[kCtlWords] = {};
  CD_CHECK(cudaMemcpyAsync(h, scratch, sizeof(h), cudaMemcpyDeviceToHost, s));
  CD_CHECK(cudaStreamSynchronize(s));
  if (h[4]) return -(int)h[4];
  if (h[5]) return -(int)h[5];
  const int64_t vol = (int64_t)h[3];
  if (vol == 0) {
    *q_out = 0.0;
    return CD_OK;
  }
  const unsigned __int128 S = ((unsigned __int128)h[1] << 64) | h[0];
  const cd::i128 num = (cd::i128)(int64_t)h[2] * vol - (cd::i128)S;
  const cd::i128 den = (cd::i128)vol * vol;
  *q_out = (double)num / (double)den;
  return CD_OK;
}
