// Target estimation on synthesised cubes: range-Doppler maps and the velocity of
// maximum power per CPI (Section III: an FFT of each CPI's cube gives the
// range-Doppler map; the velocity of the strongest response, CPI after CPI, makes
// the Doppler-time plot).
//
//   X_v[k][d]   = sum_n sum_l cube[v][n][l] e^{-j 2 pi (k n / N_s + d l / L)}
//   power[k][d] = sum_v |X_v[k][d]|^2                 (channels added non-coherently)
//   v_est       = velocity of the Doppler bin d of the largest power[k][d]
//
// The slow-time phase of a pixel turns by -f_D T_slow per block, so its Doppler bin
// is (-f_D T_slow L) mod L and bin d (signed d_s in [-L/2, L/2)) maps to
// v = -d_s lambda / (2 T_slow L).  With the static-clutter option the d = 0 column is
// left out of the search (a zero-Doppler notch).
//
// Three kernels, all deterministic, each instantiated for its FFT length:
//   fft_rows   - FFT over l of the (channel, n) rows;
//   fft_cols   - one CTA per (frame, 8 Doppler columns): FFT over n, channel by channel,
//                |X|^2 summed over the channels in registers;
//   rd_argmax  - one CTA per frame: the largest power (first index on ties) -> velocity.
// FFT lengths are powers of two up to 1024 (N_s) and 1024 (L).
//
// The work is bound by memory (the cube is read once, its row transform written and read
// once), so a transform touches shared memory only between passes: every thread holds 16
// values and takes radix-16 (or shorter, last) butterflies in registers, Stockham order,
// two passes up to 256 points.  On 64 cubes of V = 12, N_s = 256, L = 128 (201 MB):
// radix-2 stages in shared memory with a sine and cosine per butterfly took 638 us (rows),
// 521 us (columns) and 70 us (maximum), 1.20 ms a call; these kernels take 0.124 ms a call.
#include <algorithm>

#include "fft_regs.h"
#include "rsim_ctx.h"
#include "rsim_internal.h"

namespace rsim {
namespace {

constexpr int kRdCols = 8;          // Doppler columns per CTA: a 64-byte run of every row
constexpr int kRdThreads = 256;     // row kernel, and the column kernel of many frames
constexpr int kRdThreadsMax = 512;  // column kernel when few frames leave SMs idle
static_assert(kRdThreadsMax == 2 * kRdThreads, "a helper for every group of the smaller block");
constexpr int kRdByValue = 64;      // cube pointers passed in the kernel's arguments

// FFT of N = 2^k points, 2 <= N <= 1024: a thread holds PER values and T threads share a
// sequence.  Pass 1 has radix PER; the second radix R2 and the third R3 (1: no such pass).
template <int N>
struct FftShape {
  static constexpr int PER = N < 16 ? N : 16;
  static constexpr int T = N / PER;
  static constexpr int R2 = N <= 16 ? 1 : (N <= 256 ? N / 16 : 16);
  static constexpr int R3 = N <= 256 ? 1 : N / 256;
  static constexpr int RL = R3 > 1 ? R3 : (R2 > 1 ? R2 : PER);  // radix of the last pass
  static constexpr int kTw2 = R2 > 1 ? 16 * R2 : 0, kTw3 = R3 > 1 ? 256 * R3 : 0;  // twiddles
  // Shared-memory pitch of a sequence (element i sits at i + i / 16, so that the stride-16
  // stores of pass 1 fall on distinct banks).  A half-warp's 16 accesses of 8 bytes reach
  // 16 / T sequences of T threads in the row kernel and two neighbouring threads of 8
  // sequences in the column kernel: the pitch is T, or 2, modulo 16.
  static constexpr int pitch(int want) { return N + N / 16 + ((want - (N + N / 16)) % 16 + 16) % 16; }
  static constexpr int kRowPitch = pitch(T < 16 ? T : 0);
  static constexpr int kColPitch = pitch(2);
  // Floats of a column group: its transforms' buffers, or its sums if it has none.
  static constexpr int kGroupFloats = R2 > 1 ? 16 * kColPitch : 8 * N;
  static_assert(kGroupFloats >= 8 * N, "the sums fit over the buffers");
  // Index in the transform of the i-th value a thread holds after the last pass.
  __device__ static __forceinline__ int pos(int i, int t) { return t + (i / RL) * T + (i % RL) * (N / RL); }
};

// Twiddles exp(+j 2 pi j k / (R ns)) of passes 2 (ns = 16) and 3 (ns = 256) at tw[j ns + k],
// computed by the block.
template <int N>
__device__ void make_twiddles(float2* tw) {
  using S = FftShape<N>;
  for (int e = threadIdx.x; e < S::kTw2 + S::kTw3; e += blockDim.x) {
    const bool third = e >= S::kTw2;
    const int r = third ? e - S::kTw2 : e, ns = third ? 256 : 16, size = third ? S::kTw3 : S::kTw2;
    float sn, cs;
    sincospif((float)(2 * (r / ns) * (r % ns)) / (float)size, &sn, &cs);  // size is a power of two: exact
    tw[e] = make_float2(cs, sn);
  }
}

// One pass of radix R after `ns` points have been combined, from and to the sequence's
// shared-memory buffer x; the results stay in `a` (sub-butterfly by sub-butterfly) when
// `last`.  Sync orders the sequence's threads.
template <int N, int R, class Sync>
__device__ __forceinline__ void rd_pass(float2 (&a)[FftShape<N>::PER], float2* x, int t, int ns, const float2* tw,
                                        bool last, Sync sync) {
  using S = FftShape<N>;
  constexpr int G = S::PER / R;
#pragma unroll
  for (int gi = 0; gi < G; ++gi) {
    const int b = t + gi * S::T, k = b & (ns - 1);
    float2 v[R];
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const int i = b + j * (N / R);
      v[j] = x[i + (i >> 4)];
      if (j > 0) v[j] = cmul(v[j], tw[j * ns + k]);
    }
    dft_inv<R>(v);
#pragma unroll
    for (int j = 0; j < R; ++j) a[gi * R + j] = v[j];
  }
  if (last) return;
  sync();  // every read of x is done
#pragma unroll
  for (int gi = 0; gi < G; ++gi) {
    const int b = t + gi * S::T, k = b & (ns - 1), o = (b - k) * R + k;
#pragma unroll
    for (int m = 0; m < R; ++m) {
      const int i = o + m * ns;
      x[i + (i >> 4)] = a[gi * R + m];
    }
  }
  sync();
}

// Inverse-sign DFT of the sequence whose elements t + j T (j < PER) are in `a`; value i of
// the result is element pos(i, t).  (With the components of every input swapped, the
// result is the forward DFT with its components swapped.)
template <int N, class Sync>
__device__ __forceinline__ void rd_fft(float2 (&a)[FftShape<N>::PER], float2* x, int t, const float2* tw, Sync sync) {
  using S = FftShape<N>;
  dft_inv<S::PER>(a);
  if constexpr (S::R2 > 1) {
    sync();  // the buffer's previous readers are done
#pragma unroll
    for (int m = 0; m < S::PER; ++m) x[17 * t + m] = a[m];  // element 16 t + m
    sync();
    rd_pass<N, S::R2>(a, x, t, 16, tw, S::R3 == 1, sync);
    if constexpr (S::R3 > 1) rd_pass<N, S::R3>(a, x, t, 256, tw + S::kTw2, true, sync);
  }
}

struct CubePtrs {
  const float2* p[kRdByValue];
};

// Rows: FFT over l of every (channel, n) row of frame blockIdx.y, components swapped (the
// column pass only needs |X|).  The cube is read once, so its lines are marked streaming
// and leave L2 to the row transforms.
template <int L>
__global__ void __launch_bounds__(kRdThreads, 3)
fft_rows(const __grid_constant__ CubePtrs byval, const float2* const* __restrict__ cubes, float2* __restrict__ tmp,
         int F, int rows) {
  using S = FftShape<L>;
  constexpr int kSeq = kRdThreads / S::T;  // rows per pass of the block
  extern __shared__ float2 rd_smem[];
  float2* tw = rd_smem;
  make_twiddles<L>(tw);
  __syncthreads();
  const int t = threadIdx.x % S::T, s = threadIdx.x / S::T;
  float2* x = rd_smem + S::kTw2 + S::kTw3 + s * S::kRowPitch;
  auto sync = [] {
    if (S::T <= 32)
      __syncwarp();
    else
      __syncthreads();
  };
  for (int f = blockIdx.y; f < F; f += gridDim.y) {
    const float2* cube = cubes ? cubes[f] : byval.p[f];
    float2* out = tmp + (int64_t)f * rows * L;
    for (int64_t r0 = (int64_t)blockIdx.x * kSeq; r0 < rows; r0 += (int64_t)gridDim.x * kSeq) {
      const int64_t row = r0 + s;
      const bool live = row < rows;
      float2 a[S::PER];
#pragma unroll
      for (int j = 0; j < S::PER; ++j) {
        const float2 c = live ? __ldcs(cube + row * L + t + j * S::T) : make_float2(0.f, 0.f);
        a[j] = make_float2(c.y, c.x);
      }
      rd_fft<L>(a, x, t, tw, sync);
      if (live) {
#pragma unroll
        for (int i = 0; i < S::PER; ++i) out[row * L + S::pos(i, t)] = a[i];
      }
    }
  }
}

// Columns: the threads of a CTA form groups of T x 8, each taking every (number of
// groups)-th channel's 8 columns; a group sums |X|^2 over its channels in registers and the
// groups' sums are added in group order.  In the larger block (kPaired) the second half of the
// groups helps the first: it hands its |X|^2 over in shared memory, and the sums are those of the
// smaller block, so that a map's bits do not depend on the number of frames (with a run-time
// switch in one kernel the smaller block lost 1 to 3%).  Frames run from the last to
// the first: the rows written last are the ones still in L2.
template <int Ns, bool kPaired>
__global__ void __launch_bounds__(kRdThreadsMax)
fft_cols(const float2* __restrict__ tmp, float* __restrict__ power, int F, int V, int L) {
  using S = FftShape<Ns>;
  constexpr int kGroup = S::T * kRdCols;
  extern __shared__ float2 rd_smem[];
  float2* tw = rd_smem;
  make_twiddles<Ns>(tw);
  wait_prior_grid();
  __syncthreads();
  const int c = threadIdx.x % kRdCols, t = (threadIdx.x / kRdCols) % S::T;
  const int g = threadIdx.x / kGroup, groups = blockDim.x / kGroup;
  const int mains = kPaired ? groups / 2 : groups;
  float2* bufs = rd_smem + S::kTw2 + S::kTw3;
  float2* x = bufs + (g * kRdCols + c) * S::kColPitch;
  float* red = reinterpret_cast<float*>(bufs);  // [group][PER][T x 8], over the transform buffers
  // the helpers' values of this round and of the next, [2][group][PER][T x 8], behind the buffers
  [[maybe_unused]] float* handed = red + groups * S::kGroupFloats + (g % mains) * S::PER * kGroup + threadIdx.x % kGroup;
  auto sync = [g] {
    if (kGroup <= 32)
      __syncwarp();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(kGroup) : "memory");
  };
  const int d = blockIdx.x * kRdCols + c;
  for (int f = F - 1 - (int)blockIdx.y; f >= 0; f -= gridDim.y) {
    float pw[S::PER];
#pragma unroll
    for (int i = 0; i < S::PER; ++i) pw[i] = 0.f;
    [[maybe_unused]] int at = 0;  // the round's half of the values handed over
    // every group runs the same number of rounds: for short transforms groups share a warp
    for (int v0 = 0; v0 < V; v0 += groups) {
      const int v = v0 + g;
      const bool live = v < V && d < L;
      const float2* src = tmp + ((int64_t)f * V + v) * Ns * L + d;
      float2 a[S::PER];
#pragma unroll
      for (int j = 0; j < S::PER; ++j)
        a[j] = live ? src[(int64_t)(t + j * S::T) * L] : make_float2(0.f, 0.f);
      rd_fft<Ns>(a, x, t, tw, sync);
#pragma unroll
      for (int i = 0; i < S::PER; ++i) pw[i] += fmaf(a[i].x, a[i].x, a[i].y * a[i].y);
      if constexpr (kPaired) {
        if (g >= mains) {
#pragma unroll
          for (int i = 0; i < S::PER; ++i) handed[at + i * kGroup] = pw[i], pw[i] = 0.f;
        }
        __syncthreads();  // also between a round's reads and the stores of the next but one
        if (g < mains) {
#pragma unroll
          for (int i = 0; i < S::PER; ++i) pw[i] += handed[at + i * kGroup];
        }
        at = mains * S::PER * kGroup - at;
      }
    }
    __syncthreads();
    if (!kPaired || g < mains) {
#pragma unroll
      for (int i = 0; i < S::PER; ++i) red[(g * S::PER + i) * kGroup + threadIdx.x % kGroup] = pw[i];
    }
    __syncthreads();
    // the block size is a multiple of 8, so an output's column is this thread's own
    for (int o = threadIdx.x; o < S::PER * kGroup; o += blockDim.x) {
      float sum = red[o];
      for (int h = 1; h < mains; ++h) sum += red[h * S::PER * kGroup + o];
      const int i = o / kGroup, to = (o % kGroup) / kRdCols;
      if (d < L) power[((int64_t)f * Ns + S::pos(i, to)) * L + d] = sum;
    }
    __syncthreads();  // the next frame's transforms overwrite the sums
  }
}

// Largest power of one frame (first flat index on ties), optionally without d = 0.  Four
// 16-byte loads in flight per thread where the map is 16-byte aligned.
constexpr int kArgThreads = 1024;
__global__ void __launch_bounds__(kArgThreads)
rd_argmax(const float* __restrict__ power, int Ns, int L, int skip_static, double v_per_bin,
          float* __restrict__ v_est, int32_t* __restrict__ peak) {
  wait_prior_grid();
  const int f = blockIdx.x, n = Ns * L;
  const float* p = power + (int64_t)f * n;
  float best = -1.f;
  int bi = 0x7fffffff;
  // within a thread the indices rise, so a strict comparison keeps the first of equals
  auto take = [&](float x, int i) {
    if (x > best && !(skip_static && (i & (L - 1)) == 0)) {
      best = x;
      bi = i;
    }
  };
  if (n % 4 == 0 && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
    const float4* p4 = reinterpret_cast<const float4*>(p);
    for (int i0 = threadIdx.x; i0 < n / 4; i0 += 4 * kArgThreads) {
      float4 q[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * kArgThreads;
        q[u] = i < n / 4 ? p4[i] : make_float4(-1.f, -1.f, -1.f, -1.f);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = 4 * (i0 + u * kArgThreads);
        take(q[u].x, i);
        take(q[u].y, i + 1);
        take(q[u].z, i + 2);
        take(q[u].w, i + 3);
      }
    }
  } else {
    for (int i = threadIdx.x; i < n; i += kArgThreads) take(p[i], i);
  }
  __shared__ float sb[32];
  __shared__ int si[32];
  for (int o = 16; o > 0; o >>= 1) {
    const float ob = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ob > best || (ob == best && oi < bi)) {
      best = ob;
      bi = oi;
    }
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    sb[w] = best;
    si[w] = bi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < kArgThreads / 32; ++k)
      if (sb[k] > best || (sb[k] == best && si[k] < bi)) {
        best = sb[k];
        bi = si[k];
      }
    const int d = bi % L;
    const int ds = (d < L / 2) ? d : d - L;
    v_est[f] = (float)(-(double)ds * v_per_bin);
    if (peak) {
      peak[2 * f] = bi / L;
      peak[2 * f + 1] = d;
    }
  }
}

using RowFn = void (*)(CubePtrs, const float2* const*, float2*, int, int);
using ColFn = void (*)(const float2*, float*, int, int, int);
struct RowKernel {
  RowFn fn;
  int rows, smem;  // rows per pass of a block
};
struct ColKernel {
  ColFn fn, paired;
  int group, fixed, per_group, handed;  // threads of a group; shared memory: twiddles, then per
};                                      // group, and what a helper hands over in a round

template <int N>
RowKernel row_kernel() {
  using S = FftShape<N>;
  const int seq = kRdThreads / S::T;
  return {fft_rows<N>, seq, 8 * (S::kTw2 + S::kTw3 + (S::R2 > 1 ? seq * S::kRowPitch : 0))};
}
template <int N>
ColKernel col_kernel() {
  using S = FftShape<N>;
  static_assert(kRdCols == 8, "kGroupFloats");
  return {fft_cols<N, false>, fft_cols<N, (S::T * kRdCols < kRdThreadsMax)>, S::T * kRdCols, 8 * (S::kTw2 + S::kTw3), 4 * S::kGroupFloats, 4 * kRdCols * N};
}

template <class R, template <int> class Pick>
R by_length(int n) {
  switch (n) {
    case 2: return Pick<2>::get();
    case 4: return Pick<4>::get();
    case 8: return Pick<8>::get();
    case 16: return Pick<16>::get();
    case 32: return Pick<32>::get();
    case 64: return Pick<64>::get();
    case 128: return Pick<128>::get();
    case 256: return Pick<256>::get();
    case 512: return Pick<512>::get();
    default: return Pick<1024>::get();
  }
}
template <int N>
struct PickRow {
  static RowKernel get() { return row_kernel<N>(); }
};
template <int N>
struct PickCol {
  static ColKernel get() { return col_kernel<N>(); }
};

}  // namespace

cudaError_t launch_range_doppler(const float2* const* cubes, const float2* const* cubes_dev, float2* tmp, float* power,
                                 int F, int V, int Ns, int L, int skip_static, double v_per_bin, float* v_est,
                                 int32_t* peak, int num_sms, cudaStream_t st) {
  const RowKernel rk = by_length<RowKernel, PickRow>(L);
  const ColKernel ck = by_length<ColKernel, PickCol>(Ns);
  CubePtrs byval = {};
  if (!cubes_dev)
    for (int f = 0; f < F; ++f) byval.p[f] = cubes[f];
  const int fy = std::min(F, 65535);
  // rows: about four waves of blocks at three per SM, so that a block makes its twiddles
  // once for several passes; at least one block per frame
  const int64_t rows = (int64_t)V * Ns;
  const int64_t passes = (rows + rk.rows - 1) / rk.rows;
  const int64_t bx = std::min<int64_t>(passes, std::max<int64_t>(1, (12ll * num_sms + fy - 1) / fy));
  cudaError_t e = cudaFuncSetAttribute(rk.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, rk.smem);
  if (e != cudaSuccess) return e;
  rk.fn<<<dim3((unsigned)bx, fy), kRdThreads, rk.smem, st>>>(byval, cubes_dev, tmp, F, (int)rows);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // columns: 256 threads where the frames fill the SMs twice over, else 512 (more channels
  // of a frame at a time)
  const int cx = (L + kRdCols - 1) / kRdCols;
  const int threads = std::max(ck.group, (int64_t)cx * F >= 2ll * num_sms ? kRdThreads : kRdThreadsMax);
  // a helper for every second group, two rounds of values each
  const bool paired = threads > kRdThreads && ck.group < kRdThreadsMax;
  const int smem = ck.fixed + (threads / ck.group) * (ck.per_group + (paired ? ck.handed : 0));
  const ColFn cols = paired ? ck.paired : ck.fn;
  e = cudaFuncSetAttribute(cols, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  e = launch_dependent(cols, dim3(cx, fy), dim3(threads), (size_t)smem, st, (const float2*)tmp, power, F, V, L);
  if (e != cudaSuccess) return e;
  return launch_dependent(rd_argmax, dim3(F), dim3(kArgThreads), 0, st, (const float*)power, Ns, L, skip_static,
                          v_per_bin, v_est, peak);
}

}  // namespace rsim

using namespace rsim;

extern "C" rsim_status rsim_range_doppler(rsim_ctx* ctx, const rsim_radar_params* params,
                                          void* const* cubes, int32_t F, float* power, float* v_est,
                                          int32_t* peak, int32_t options, rsim_stream stream) {
  if (!ctx || !cubes || !power || !v_est) return fail(RSIM_ERR_INVALID_ARG, "NULL argument");
  if (F < 1) return fail(RSIM_ERR_INVALID_ARG, "F must be >= 1");
  if (options & ~RSIM_RD_SKIP_STATIC) return fail(RSIM_ERR_INVALID_ARG, "unknown option bits");
  Consts k;
  rsim_status s = check_params(params, &k);
  if (s != RSIM_OK) return s;
  auto pow2 = [](int x) { return x >= 2 && x <= 1024 && (x & (x - 1)) == 0; };
  if (!pow2(k.Ns) || !pow2(k.L))
    return fail(RSIM_ERR_UNSUPPORTED, "range-Doppler processing needs N_s and L powers of two in 2..1024");
  for (int f = 0; f < F; ++f)
    if (!cubes[f]) return fail(RSIM_ERR_INVALID_ARG, "a cube pointer is NULL");
  cudaSetDevice(ctx->device);
  cudaStream_t st = (cudaStream_t)stream;
  const size_t ptr_bytes = ((sizeof(void*) * (size_t)F + 255) / 256) * 256;
  const size_t tmp_bytes = sizeof(float2) * (size_t)F * k.V * k.Ns * k.L;
  s = ensure_workspace(ctx, ptr_bytes + tmp_bytes, st);
  if (s != RSIM_OK) return s;
  char* ws = (char*)ctx->ws;
  cudaError_t e = cudaSuccess;
  const bool table = F > kRdByValue;  // few pointers go in the kernel's arguments
  if (table) {
    e = cudaMemcpyAsync(ws, cubes, sizeof(void*) * (size_t)F, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return cuda_fail(e, "upload of the cube table");
  }
  const double t_slow = params->t_slow > 0 ? params->t_slow : params->M * params->t_b;
  const double v_per_bin = params->lambda / (2.0 * t_slow * k.L);
  e = launch_range_doppler((const float2* const*)cubes, table ? (const float2* const*)ws : nullptr,
                           (float2*)(ws + ptr_bytes), power, F, k.V, k.Ns, k.L,
                           (options & RSIM_RD_SKIP_STATIC) ? 1 : 0, v_per_bin, v_est, peak, ctx->num_sms, st);
  if (e != cudaSuccess) return cuda_fail(e, "range-Doppler kernels");
  return RSIM_OK;
}
