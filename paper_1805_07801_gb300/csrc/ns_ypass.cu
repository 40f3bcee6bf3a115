// The y passes of the solvers (padded rows, 2/3 rule; see k_ns_ypass for the
// general kernel): from 384 points on pipelined (fft_pipe.cuh).  The inverse
// pass stages only the kept rows, the forward pass stores only those.
// Per launch, one tile after the other with one or two CTAs per SM, and so:
// 768^3, six fields inverse 2.43 -> 1.95 ms, three forward 1.16 -> 0.91 ms
// (radix 48, then 16; 2.27 and 1.04 ms with radices 8, 8, 12); 512^3,
// 641 -> 586 us, 310 -> 277 us (0.95 of the copy rate).  At 256 points the
// general kernel, with more CTAs per SM, is as fast (79 / 101 against 82 / 102
// us for six and seven fields).
#include <mutex>

#include "fft_pipe.cuh"
#include "ns_passes.cuh"

namespace fftk {

template <int N, int SIGN>  // N >= 384
struct YPipeCfg {
  static constexpr bool ENGINE = N % 3 == 0 && N != 768;  // else two long-radix stages
  static constexpr int G = ENGINE ? elems_per_thread(N) : (N == 768 ? 48 : 32);
  static constexpr int S = N / G, T = 16, THREADS = S * T;
  static constexpr int MINB = N >= 768 ? 1 : 2;
  static constexpr int KD = (N - 1) / 3;
  // boxes: the inverse pass takes rows 0 .. KD and N - KD - 1 .. N - 1 (the first
  // of these is not used) in halves of at most 256 rows
  static constexpr int PART = SIGN > 0 ? KD + 1 : N;                // rows of one part
  static constexpr int SPLIT = (PART + 255) / 256;                  // boxes per part
  static constexpr int BOXR = (PART + SPLIT - 1) / SPLIT;
  static constexpr int ROWS = (SIGN > 0 ? 2 : 1) * SPLIT * BOXR;    // staged rows
  static constexpr size_t STAGE = sizeof(float2) * ROWS * T;
  static constexpr size_t EX = (ENGINE ? sizeof(float2) : sizeof(float)) * N * T;
  static constexpr size_t SMEM = STAGE + EX + (ENGINE ? 0 : sizeof(float2) * N) + 16;
};

// planes: fields x N; tile t = (plane, k_z tile)
template <int N, int SIGN>
__global__ void __launch_bounds__(YPipeCfg<N, SIGN>::THREADS, YPipeCfg<N, SIGN>::MINB)
    k_ns_ypipe(const __grid_constant__ CUtensorMap map, float2* out, int ntiles, const float2* __restrict__ tw,
               const float2* __restrict__ t3, int* err) {
  pdl_wait();
  using C = YPipeCfg<N, SIGN>;
  constexpr long long HW = ns_row(N);
  constexpr int G = C::G, S = C::S, T = C::T, KD = C::KD, KT = (KD + T) / T;
  extern __shared__ __align__(128) unsigned char smy[];
  __shared__ int ok_flag, next_tile;
  float2* stage = reinterpret_cast<float2*>(smy);
  float* ex = reinterpret_cast<float*>(smy + C::STAGE);
  float2* stw = reinterpret_cast<float2*>(smy + C::STAGE + C::EX);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smy + C::SMEM - 16);
  const int tid = threadIdx.x, c = tid % T, j = tid / T;
  if constexpr (!C::ENGINE)
    for (int i = tid; i < N; i += C::THREADS) stw[i] = N % 3 == 0 ? t3[N + i] : tw[i];
  constexpr int HIGH0 = N - C::SPLIT * C::BOXR;  // first row of the upper part (inverse)
  auto fetch = [&](int t) {  // thread 0
    const int plane = t / KT, x0 = 2 * T * (t - plane * KT);
    tcg::mbar_expect(bar, (uint32_t)C::STAGE);
#pragma unroll 1
    for (int b = 0; b < C::SPLIT; ++b) {
      tcg::tma_load3(stage + (size_t)b * C::BOXR * T, &map, x0, b * C::BOXR, plane, bar);
      if constexpr (SIGN > 0)
        tcg::tma_load3(stage + (size_t)(C::SPLIT + b) * C::BOXR * T, &map, x0, HIGH0 + b * C::BOXR, plane, bar);
    }
  };
  if (tid == 0) tcg::mbar_init(bar);
  __syncthreads();
  int* queue = err + 1;
  uint32_t phase = 0;
  int t = blockIdx.x, drawn = 0;
  if (tid == 0) {
    fetch(t);
    drawn = (int)gridDim.x + atomicAdd(queue, 1);
  }
  while (t < ntiles) {
    if (tid == 0) {
      ok_flag = tcg::mbar_wait(bar, phase) ? 1 : 0;
      next_tile = drawn;
    }
    __syncthreads();
    if (!ok_flag) {  // see k_cpass_pipe
      if (tid == 0) {
        atomicOr(err, 1);
        tcg::mbar_wait(bar, phase);
      }
      break;
    }
    const int tn = next_tile;
    phase ^= 1;
    float2 v[G];
#pragma unroll
    for (int m = 0; m < G; ++m) {
      const int pos = j + m * S;
      if constexpr (SIGN < 0) {
        v[m] = stage[pos * T + c];
      } else {
        v[m] = make_float2(0.f, 0.f);
        if (pos <= KD)
          v[m] = stage[pos * T + c];
        else if (pos >= N - KD)
          v[m] = stage[(C::SPLIT * C::BOXR + pos - HIGH0) * T + c];
      }
    }
    __syncthreads();  // the staging buffer is free, and so is the exchange buffer
    if (tid == 0 && tn < ntiles) {
      tcg::fence_smem_async();
      fetch(tn);
      drawn = (int)gridDim.x + atomicAdd(queue, 1);
    }
    if constexpr (C::ENGINE)
      fft_line<N, G, SIGN>(v, j, ColX<T>{reinterpret_cast<float2*>(ex), c}, tw, t3);
    else
      pipe_transform<N, G, SIGN, T>(v, j, c, ex, stw);
    const int plane = t / KT, kz = T * (t - plane * KT) + c;
    if (kz <= KD) {
      float2* dst = out + (long long)plane * N * HW + kz;
#pragma unroll
      for (int m = 0; m < G; ++m) {
        const int pos = j + m * S;
        if (SIGN > 0 || kept_xy(pos, N, KD)) dst[(long long)pos * HW] = v[m];
      }
    }
    t = tn;
  }
  if (tid == 0) pipe_leave(queue);
}

template <int N, int SIGN>
static cudaError_t ypass_n(fftk_plan p, const float2* in, float2* out, int fields, int kind, cudaStream_t st) {
  constexpr int KD = (N - 1) / 3;
  const float2* tw = twiddles(p, 1 << Log2<N>::value);
  if constexpr (N >= 384) {
    using C = YPipeCfg<N, SIGN>;
    static PerDevice once;
    static int nsm[kMaxDevices];
    int dev = 0;
    const cudaError_t e = once.run(
        [](int d) {
          cudaError_t err = cudaFuncSetAttribute(k_ns_ypipe<N, SIGN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)C::SMEM);
          if (err == cudaSuccess) err = cudaDeviceGetAttribute(&nsm[d], cudaDevAttrMultiProcessorCount, d);
          return err;
        },
        &dev);
    if (e != cudaSuccess) return e;
    constexpr long long HW = ns_row(N);
    const uint64_t dims[3] = {(uint64_t)(2 * HW), (uint64_t)N, (uint64_t)fields * N};
    const uint64_t strides[2] = {(uint64_t)(8 * HW), (uint64_t)(8 * HW * N)};
    const uint32_t box[3] = {2 * C::T, (uint32_t)C::BOXR, 1};
    CUtensorMap m;
    if (encode_f32_map(&m, in, 3, dims, strides, box)) {
      const int ntiles = fields * N * ((KD + C::T) / C::T), cap = nsm[dev] * C::MINB;
      LaunchScope ls(p, kind, st);
      launch_pdl(k_ns_ypipe<N, SIGN>, ntiles < cap ? ntiles : cap, C::THREADS, C::SMEM, st, m, out, ntiles, tw,
                 p->d_tw3,
                                                                                  p->d_err);
      return cudaGetLastError();
    }
  }
  using X = NXCfg<N>;
  static PerDevice once;
  const cudaError_t e = once.run([](int) {
    return cudaFuncSetAttribute(k_ns_ypass<N, SIGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)X::SMEM);
  });
  if (e != cudaSuccess) return e;
  constexpr int KT = (KD + X::T) / X::T;
  LaunchScope ls(p, kind, st);
  launch_pdl(k_ns_ypass<N, SIGN>, fields * N * KT, X::THREADS, X::SMEM, st, in, out, KT, tw, p->d_tw3);
  return cudaGetLastError();
}

cudaError_t ns_ypass(fftk_plan p, const float2* in, float2* out, int fields, int sign, int kind, cudaStream_t st) {
  switch (p->nx) {
#define CASE(n) \
  case n:       \
    return sign > 0 ? ypass_n<n, 1>(p, in, out, fields, kind, st) : ypass_n<n, -1>(p, in, out, fields, kind, st);
    CASE(8) CASE(16) CASE(32) CASE(64) CASE(128) CASE(256) CASE(512) CASE(1024)
    CASE(12) CASE(24) CASE(48) CASE(96) CASE(192) CASE(384) CASE(768)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

}  // namespace fftk
