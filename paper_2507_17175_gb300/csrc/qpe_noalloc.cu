// qpe_readout_static: the histogram + readout reduction for callers that
// cannot allocate device memory.
//
// The regular path needs a workspace from the caller (qpe_plan / qpe_bind).
// Some callers cannot provide one: code that runs where device allocation is
// forbidden or unsafe (inside a region that must not synchronise or grow the
// memory pool, under a fixed memory budget, or in a host library that never
// owns device memory). For them this entry point keeps its only scratch, the
// per-block partial results of the reduction, in a fixed array compiled into
// the library. The caller passes the final statevector and receives the
// histogram and the readout in its own buffers; nothing is allocated.
#include <cuda_runtime.h>

#include <mutex>

#include "qpe_internal.cuh"

namespace {

constexpr int kMaxNmeas = 21;       // the largest histogram the entry point takes
constexpr int kBlocksPerSM = 5;      // 48 registers a thread
constexpr int kMaxBlocks = kBlocksPerSM * 152;  // CTAs of a call (resident at once), one partial each

// Scratch shared by every call on a device: one partial per CTA. Every slot a
// call reads is written earlier in the same call, so nothing needs clearing;
// calls whose kernels overlap on the GPU overwrite each other's partials.
static __device__ __align__(256) qpe::Partial g_readout_scratch[kMaxBlocks];

constexpr int kMaxDevices = 64;
std::mutex g_setup_mutex;
qpe::Partial* g_scratch_addr[kMaxDevices] = {};

// Device address of the scratch on the current device, looked up once per
// device (the host-side symbol is only a stand-in for it).
cudaError_t scratch_address(qpe::Partial** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  if (!g_scratch_addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_readout_scratch);
    if (e != cudaSuccess) return e;
    g_scratch_addr[dev] = static_cast<qpe::Partial*>(p);
  }
  *out = g_scratch_addr[dev];
  return cudaSuccess;
}

// ------------------------------------------------------------- row sums
// sum of |X[y][t]|^2 over a row, as accurate as an FP64 sum.
//
// What bounds it: HBM, once the FP64 units are out of the way. GB300 issues
// FP64 at 1/64 of its FP32 rate (2 lanes a clock and SM), so a conversion and
// an FP64 FMA for every float take 10x the time of the loads. complex64 rows
// are therefore summed exactly in FP32:
//   * a row (or 256 columns of it) is scaled by the power of two that brings
//     its largest |float| into [1, 2);
//   * a square is p + e, p = fl(x^2), e = fma(x, x, -p), both exact;
//   * p goes into T1, which starts at the anchor 64 (16 squares < 64 keep it in
//     [64, 128]): T1' = fl(T1 + p) and the rest p - (T1' - T1) are exact; rest and
//     e go into T2 in the same way (anchor 1.5 2^-12, |sum| < 2^-13), and what
//     T2 leaves, below 2^-36 each, into T3. Dropped: T3's roundings, 2^-56 of the
//     largest square.
// 15 FP32 / integer operations a float. The lanes of a row meet in error-free
// sums, and the one FP64 value per row is formed by a whole warp for 32 rows.
// A row with an infinity, a NaN, or no normal number in it is summed in FP64.
// 2^21 rows of 32 columns (complex64, 537 MB): 2180 us a call with converted
// FP64 sums, 134 us so (80 us are the bytes at the copy rate).

// a + b = s + err, exactly
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& err) {
  s = a + b;
  const float bb = s - a;
  err = (a - (s - bb)) + (b - bb);
}

struct RowSum {  // value (a + (b + c)) 2^(2 (ex - 127)); ex < 0: the double (hi, lo) = (bits of a, bits of b)
  float a, b, c;
  int ex;
};
__device__ __forceinline__ RowSum pack_double(double v) {
  return RowSum{__int_as_float(__double2hiint(v)), __int_as_float(__double2loint(v)), 0.f, -1};
}
__device__ __forceinline__ double unpack(const RowSum& r) {
  if (r.ex < 0) return __hiloint2double(__float_as_int(r.a), __float_as_int(r.b));
  const double v = (double)r.a + ((double)r.b + (double)r.c);
  return v * __hiloint2double((1023 + 2 * (r.ex - 127)) << 20, 0);
}

// VPL 16-byte vectors a lane, LANES lanes a row (of at most 256 columns)
template <int VPL, int LANES>
__device__ __forceinline__ RowSum row_sum(const float2* __restrict__ row, int sub, int bytes) {
  float4 v[VPL];
  if (bytes == 16) {
#pragma unroll
    for (int k = 0; k < VPL; ++k) v[k] = __ldcs(reinterpret_cast<const float4*>(row) + sub + k * LANES);
  } else if (bytes == 4) {  // a state on a boundary of 4 bytes
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      const float* f = reinterpret_cast<const float*>(row) + 4 * (sub + k * LANES);
      v[k] = make_float4(__ldcs(f), __ldcs(f + 1), __ldcs(f + 2), __ldcs(f + 3));
    }
  } else {  // of 8
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      const float2 a = __ldcs(row + 2 * (sub + k * LANES)), b = __ldcs(row + 2 * (sub + k * LANES) + 1);
      v[k] = make_float4(a.x, a.y, b.x, b.y);
    }
  }
  uint32_t m = 0;
#pragma unroll
  for (int k = 0; k < VPL; ++k) {
    m = max(m, max(__float_as_uint(v[k].x) & 0x7fffffffu, __float_as_uint(v[k].y) & 0x7fffffffu));
    m = max(m, max(__float_as_uint(v[k].z) & 0x7fffffffu, __float_as_uint(v[k].w) & 0x7fffffffu));
  }
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  const int ex = m ? (int)(m >> 23) : 127;
  const bool plain = ex >= 1 && ex <= 253;  // a row of zeros too
  const float sc = __uint_as_float((uint32_t)(plain ? 254 - ex : 127) << 23);
  constexpr float A1 = 64.f, A2 = 1.5f / 4096.f;
  float t1 = A1, t2 = A2, t3 = 0.f;
  auto add = [&](float xr) {
    const float x = xr * sc;
    const float p = x * x;
    const float e = fmaf(x, x, -p);
    const float n1 = t1 + p;
    const float r1 = p - (n1 - t1);
    t1 = n1;
    const float n2 = t2 + r1;
    const float r2 = r1 - (n2 - t2);
    const float n3 = n2 + e;
    const float r3 = e - (n3 - n2);
    t2 = n3;
    t3 += r2 + r3;
  };
#pragma unroll
  for (int k = 0; k < VPL; ++k) {
    add(v[k].x);
    add(v[k].y);
    add(v[k].z);
    add(v[k].w);
  }
  RowSum r{t1 - A1, t2 - A2, t3, ex};
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) {
    const float oa = __shfl_xor_sync(0xffffffffu, r.a, o);
    const float ob = __shfl_xor_sync(0xffffffffu, r.b, o);
    const float oc = __shfl_xor_sync(0xffffffffu, r.c, o);
    float ea, eb, ec;
    two_sum(r.a, oa, r.a, ea);
    two_sum(r.b, ob, r.b, eb);
    two_sum(r.b, ea, r.b, ec);
    r.c += oc + (eb + ec);
  }
  if (__any_sync(0xffffffffu, !plain)) {
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < VPL; ++k)
      acc += ((double)v[k].x * (double)v[k].x + (double)v[k].y * (double)v[k].y) +
             ((double)v[k].z * (double)v[k].z + (double)v[k].w * (double)v[k].w);
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (!plain) r = pack_double(acc);
  }
  return r;
}
// complex128: two FP64 FMAs an element, nothing else on the FP64 units but the lanes' sums
template <int VPL, int LANES>
__device__ __forceinline__ double row_sum(const double2* __restrict__ row, int sub, int bytes) {
  double2 v[VPL];
  if (bytes == 16) {
#pragma unroll
    for (int k = 0; k < VPL; ++k) v[k] = __ldcs(row + sub + k * LANES);
  } else {  // a state on a boundary of 8 bytes
#pragma unroll
    for (int k = 0; k < VPL; ++k) {
      const double* f = reinterpret_cast<const double*>(row + sub + k * LANES);
      v[k] = make_double2(__ldcs(f), __ldcs(f + 1));
    }
  }
  double acc = 0.0;
#pragma unroll
  for (int k = 0; k < VPL; ++k) acc = fma(v[k].x, v[k].x, fma(v[k].y, v[k].y, acc));
#pragma unroll
  for (int o = LANES / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}
__device__ __forceinline__ double unpack(double v) { return v; }

// P[y] for the tiles of this CTA (grid-stride); partial readout into parts[blockIdx.x].
// LOGC: log2 of the columns summed by one group of lanes (the whole row up to
// 256 columns). A tile is 256 such pieces, 32 per warp; thread t then forms
// the FP64 value of piece t, and the threads at the start of a row finish it.
template <typename C, int LOGC>
__global__ void __launch_bounds__(256, kBlocksPerSM) static_partials_kernel(const C* __restrict__ X, double* __restrict__ probs,
                                                              qpe::Partial* __restrict__ parts, int64_t pieces,
                                                              int logd, int bytes) {
  constexpr int EPV = 16 / (int)sizeof(C);          // elements per 16-byte load
  constexpr int VECS = (1 << LOGC) / EPV;           // loads per piece
  // 64 bytes and more a lane where the row has them, and rows of 16 columns and
  // more read by lanes side by side in whole 32-byte sectors
  constexpr int VPL = LOGC >= 5 ? 8 / EPV : VECS <= 2 ? VECS : VECS / 2 < 4 ? VECS / 2 : 4;
  constexpr int LANES = VECS / VPL;
  static_assert(LANES >= 1 && LANES <= 32 && VPL * LANES == VECS, "a piece is one warp's loads at most");
  static_assert(sizeof(C) == 16 || VPL <= 4, "the FP32 anchors hold 16 squares a lane");
  constexpr int RPS = 32 / LANES;                   // pieces per warp step
  using V = decltype(row_sum<VPL, LANES>(static_cast<const C*>(nullptr), 0, 16));
  __shared__ V vals[256];
  __shared__ double dv[256];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int plog = logd - LOGC;                     // log2 of the pieces per row
  double best = -1.0, wsum = 0.0, psum = 0.0;
  int64_t by = INT64_MAX;
  const int64_t tiles = (pieces + 255) >> 8;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int64_t base = t << 8;
#pragma unroll 2
    for (int s = 0; s < 32; s += RPS) {
      const int q = warp * 32 + s + lane / LANES;
      const int64_t piece = base + q < pieces ? base + q : pieces - 1;  // past the end: the last piece again, unused
      const C* p = X + (piece << LOGC);
      const V v = row_sum<VPL, LANES>(p, lane % LANES, bytes);
      if (lane % LANES == 0) vals[q] = v;
    }
    __syncwarp();  // a warp reads back only its own pieces
    double v = unpack(vals[threadIdx.x]);
    bool whole = base + threadIdx.x < pieces;
    if (plog > 0) {  // uniform: rows of more than 256 columns
      dv[threadIdx.x] = v;
      __syncwarp();  // a row is at most 16 consecutive pieces of one warp
      whole = whole && (threadIdx.x & ((1 << plog) - 1)) == 0;
      if (whole)
        for (int k = 1; k < (1 << plog); ++k) v += dv[threadIdx.x + k];
      __syncwarp();
    }
    if (whole) {
      const int64_t y = (base + threadIdx.x) >> plog;
      probs[y] = v;
      qpe::better(best, by, v, y);
      wsum = fma(v, (double)y, wsum);
      psum += v;
    }
    __syncwarp();  // the values are read before the next tile overwrites them
  }
  for (int off = 16; off > 0; off >>= 1) {
    const double ob = __shfl_xor_sync(0xffffffffu, best, off);
    const int64_t oy = __shfl_xor_sync(0xffffffffu, by, off);
    qpe::better(best, by, ob, oy);
    wsum += __shfl_xor_sync(0xffffffffu, wsum, off);
    psum += __shfl_xor_sync(0xffffffffu, psum, off);
  }
  __shared__ qpe::Partial sp[8];
  if (lane == 0) sp[warp] = qpe::Partial{best, by, wsum, psum};
  __syncthreads();
  if (threadIdx.x == 0) {
    qpe::Partial r = sp[0];
    for (int w = 1; w < 8; ++w) {
      qpe::better(r.best, r.besty, sp[w].best, sp[w].besty);
      r.wsum += sp[w].wsum;
      r.psum += sp[w].psum;
    }
    parts[blockIdx.x] = r;
  }
}

// The same merge and readout as the plan path's finalize; a non-finite sum or
// a histogram without any comparable bin reports argmax = -1 and a NaN
// phase_argmax.
__global__ void __launch_bounds__(256) static_finish_kernel(const qpe::Partial* __restrict__ parts, int count,
                                                            qpe_readout_t* __restrict__ out, int n) {
  const qpe::Partial m = qpe::reduce_partials_256(parts, count);
  if (threadIdx.x == 0) {
    const double N = ldexp(1.0, n);
    const bool ok = qpe::readout_finite(m);
    qpe_readout_t o;
    o.argmax = ok ? m.besty : -1;
    o.phase_argmax = ok ? (double)m.besty / N : __longlong_as_double(0x7ff8000000000000LL);
    o.phase_mean = m.wsum / N;
    o.total = m.psum;
    *out = o;
  }
}

// CTAs of the partials kernel: one wave at most, each taking tiles of 256 pieces
// in turn; one CTA then merges their partials (20 us when there were 8192).
template <typename C>
int launch_partials(const C* X, double* probs, qpe::Partial* parts, int nmat, int nmeas, cudaStream_t s) {
  const int logc = nmat < 8 ? nmat : 8;
  const uintptr_t at = reinterpret_cast<uintptr_t>(X);
  const int bytes = at % 16 == 0 ? 16 : at % 8 == 0 ? 8 : 4;  // the widest loads X allows
  const int64_t pieces = int64_t(1) << (nmeas + nmat - logc);
  const int64_t tiles = (pieces + 255) / 256;
  const int blocks = (int)(tiles < kMaxBlocks ? tiles : kMaxBlocks);
#define QPE_PARTIALS(LC) \
  case LC: static_partials_kernel<C, LC><<<blocks, 256, 0, s>>>(X, probs, parts, pieces, nmat, bytes); break;
  switch (logc) {
    QPE_PARTIALS(1)
    QPE_PARTIALS(2)
    QPE_PARTIALS(3)
    QPE_PARTIALS(4)
    QPE_PARTIALS(5)
    QPE_PARTIALS(6)
    QPE_PARTIALS(7)
    default: static_partials_kernel<C, 8><<<blocks, 256, 0, s>>>(X, probs, parts, pieces, nmat, bytes); break;
  }
#undef QPE_PARTIALS
  return blocks;
}

}  // namespace

extern "C" qpe_status qpe_readout_static(const void* final_state, int32_t nmat, int32_t nmeas, int32_t prec,
                                         double* probs, qpe_readout_t* readout, void* cuda_stream) {
  if (!final_state || !probs || !readout) return QPE_ERR_ARG;
  if (nmat < 1 || nmat > 12 || nmeas < 1 || nmeas > 30) return QPE_ERR_ARG;
  if (prec < QPE_FP64 || prec > QPE_C64_TF32X3) return QPE_ERR_ARG;
  const uintptr_t at = reinterpret_cast<uintptr_t>(final_state);
  if (at % (prec == QPE_FP64 ? 8 : 4) || reinterpret_cast<uintptr_t>(probs) % 8 ||
      reinterpret_cast<uintptr_t>(readout) % 8)
    return QPE_ERR_ARG;
  if (nmeas > kMaxNmeas) return QPE_ERR_WORKSPACE;
  qpe::Partial* scratch = nullptr;
  cudaError_t e = scratch_address(&scratch);
  if (e != cudaSuccess) return QPE_ERR_CUDA;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  const int blocks = prec == QPE_FP64
                         ? launch_partials(static_cast<const double2*>(final_state), probs, scratch, nmat, nmeas, s)
                         : launch_partials(static_cast<const float2*>(final_state), probs, scratch, nmat, nmeas, s);
  if (cudaGetLastError() != cudaSuccess) return QPE_ERR_CUDA;
  static_finish_kernel<<<1, 256, 0, s>>>(scratch, blocks, readout, nmeas);
  if (cudaGetLastError() != cudaSuccess) return QPE_ERR_CUDA;
  return QPE_OK;
}
