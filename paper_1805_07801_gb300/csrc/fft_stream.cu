// Pipelined strided pass for lines of 256 to 1024 points and of 3 * 2^m from
// 384 to 1536.
//
// The strided pass of the 3D transform (the y and x line transforms of
// Sec. 3) works on tiles of 16 adjacent columns x L rows.  Persistent CTAs
// stream their next tile into a staging buffer (TMA) while this one, held in
// registers, takes two long-radix stages (32 x 32, 32 x 16, 16 x 16) with one
// exchange through a buffer of half the tile's size: real parts first, then
// imaginary parts.  So the copies overlap the transforms and the stores, and
// the pass is bound by HBM (k_cpass, which loads, transforms and stores in
// turn with one to four CTAs per SM, by its latencies).  Per pass, x / y, with
// k_cpass (512^3 x: with a tile streamed into the exchange buffer) and so:
//   1024^3      2.01 / 2.07 -> 1.35 / 1.37 ms   (0.94 of the copy rate)
//   512^3       187 / 225 -> 168 / 206 us       (0.95 / 0.77)
//   16 x 256^3  423 / 439 -> 322 / 418 us       (0.99 / 0.76)
//   768^3       797 / 858 -> 587 / 626 us       (0.92 / 0.86)
//   2 x 1536 x 1536 x 96   1180 / 1357 -> 823 / 1011 us
// The y passes' rows of n/2 + 1 values leave one column for a last tile and
// store across line boundaries, which the shorter lines' transforms feel.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <cstdint>
#include <cstring>
#include <mutex>

#include "fft_pipe.cuh"
#include "internal.h"
#include "sc_algebra.cuh"
#include "tcgen05.cuh"

namespace fftk {

using tcg::mbar_expect;
using tcg::tma_load3;

// Q even: rows start on 16-byte boundaries and a tile arrives as boxes of 16
// columns x 256 rows.  Q odd (PAIR; the y pass, whose rows of n/2 + 1 values
// start on and 8 bytes past such boundaries in turn): even and odd rows are
// two tensors whose row stride, 16 Q bytes, is a multiple of 16, the second
// one starting 8 bytes early, in boxes of 18 columns.  (One bulk copy of 144
// bytes per row instead: 2.43 against 2.14 ms at 1024^3.)
template <int L_, bool PAIR_>
struct PipeCfg {
  static constexpr int L = L_;
  static constexpr bool PAIR = PAIR_;
  // powers of two and 768: two stages (radix G, then R2) with the half-size
  // exchange; 384 and 1536: the line engine (24 values) with an exchange buffer
  // of the tile's size.  (768 with the engine, radices 8, 8, 12 on 512 threads:
  // 622 / 698 us per 768^3 x / y pass against 587 / 626 us with 48 x 16 on 256.)
  static constexpr bool ENGINE = L % 3 == 0 && L != 768;
  static constexpr int G = ENGINE ? elems_per_thread(L) : (L == 768 ? 48 : (L >= 512 ? 32 : 16));  // values per thread
  static constexpr int R2 = L / G;                  // radix of the second stage
  static constexpr bool PAIRED = L == 512;          // two butterflies per thread in the second stage
  static constexpr int S = L / G;                   // threads per line
  static constexpr int T = L > 1024 ? 8 : 16;       // columns per tile (128-byte rows)
  static constexpr int THREADS = S * T;
  static constexpr int MINB = L >= 768 ? 1 : (L >= 384 ? 2 : 4);
  static constexpr int ODD = PAIR ? T + 2 : T;      // float2 per staged odd row
  static constexpr int ROWS = PAIR ? L / 2 : L;     // rows of a tensor
  static constexpr int NBOX = (ROWS + 255) / 256;
  static constexpr int BOXR = ROWS / NBOX;          // rows per box
  static constexpr size_t STAGE = sizeof(float2) * (L / 2) * (T + ODD);
  static constexpr size_t EX = (ENGINE ? sizeof(float2) : sizeof(float)) * L * T;
  static constexpr size_t SMEM = STAGE + EX + (ENGINE ? 0 : sizeof(float2) * L) + 16;  // + the twiddles, the mbarrier
};

// Array [P][L][Q] of complex values, transform along L (element stride Q);
// tile t = (p, q-tile).
// BASIS: 0 Fourier, 1 cosine, 2 sine (fft_sc.cu states the reduction to one
// complex transform): forward (SIGN -1), the samples are read from the staged
// tile in permuted order and the result is combined with its mirror through
// the exchange buffer; inverse, the mirror coefficient comes from the staged
// tile and the rows are stored in permuted order.
template <int L, int SIGN, bool PAIR, int BASIS>
__global__ void __launch_bounds__(PipeCfg<L, PAIR>::THREADS, PipeCfg<L, PAIR>::MINB)
    k_cpass_pipe(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap map_odd, float2* out,
                 long long Q, int qtiles, int ntiles, const float2* __restrict__ tw, const float2* __restrict__ t3,
                 const float2* __restrict__ tq, float scale, int* err) {
  pdl_wait();
  using C = PipeCfg<L, PAIR>;
  constexpr int G = C::G, S = C::S, T = C::T;
  extern __shared__ __align__(128) unsigned char smp[];
  __shared__ int ok_flag, next_tile;
  float2* stage = reinterpret_cast<float2*>(smp);
  float2* odd = stage + (size_t)(L / 2) * T;  // PAIR: the odd rows
  float* ex = reinterpret_cast<float*>(smp + C::STAGE);
  float2* stw = reinterpret_cast<float2*>(smp + C::STAGE + C::EX);  // (from global memory the gathers cost 3 %)
  uint64_t* bar = reinterpret_cast<uint64_t*>(smp + C::SMEM - 16);
  const int tid = threadIdx.x, c = tid % T, j = tid / T;
  if constexpr (!C::ENGINE)
    for (int i = tid; i < L; i += C::THREADS) stw[i] = L % 3 == 0 ? t3[L + i] : tw[i];

  auto fetch = [&](int t) {  // thread 0
    const int p = t / qtiles, q0 = (t - p * qtiles) * T;
    mbar_expect(bar, (uint32_t)C::STAGE);
#pragma unroll 1
    for (int b = 0; b < C::NBOX; ++b) {
      tma_load3(stage + (size_t)b * C::BOXR * T, &map, 2 * q0, b * C::BOXR, p, bar);
      if constexpr (PAIR) tma_load3(odd + (size_t)b * C::BOXR * C::ODD, &map_odd, 2 * q0, b * C::BOXR, p, bar);
    }
  };
  auto slot = [&](int pos) { return pipe_slot<G, T>(pos, c); };
  if (tid == 0) tcg::mbar_init(bar);
  __syncthreads();
  int* queue = err + 1;  // next tile, CTAs that are done (fft_pipe.cuh)
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
    if (!ok_flag) {
      // The tile never arrived: its copy may still be pending, writing into
      // this CTA's shared memory and completing on the mbarrier there.  Thread
      // 0 reports, then waits once more (bounded) for that copy before the
      // CTA's shared memory is released; the other threads may leave.  The
      // error word is the only signal: the host treats it as fatal for the plan.
      if (tid == 0) {
        atomicOr(err, 1);
        tcg::mbar_wait(bar, phase);
      }
      break;
    }
    const int tn = next_tile;
    phase ^= 1;
    float2 v[G];
    auto staged = [&](int row) -> float2 {
      return !PAIR ? stage[row * T + c] : (row & 1 ? odd[(row >> 1) * C::ODD + 1 + c] : stage[(row >> 1) * T + c]);
    };
    if constexpr (BASIS == 0) {
      const float2* src =
          !PAIR ? stage + j * T + c : (j & 1 ? odd + (j >> 1) * C::ODD + 1 + c : stage + (j >> 1) * T + c);
      const int step = !PAIR ? S * T : (S / 2) * (j & 1 ? C::ODD : T);
#pragma unroll
      for (int m = 0; m < G; ++m) v[m] = src[m * step];
    } else if constexpr (SIGN < 0) {
#pragma unroll
      for (int m = 0; m < G; ++m) {
        const int r = j + m * S;
        const float2 x = staged(sc_perm(r, L));
        v[m] = BASIS == 2 && r >= L / 2 ? make_float2(-x.x, -x.y) : x;  // (-1)^j at odd j
      }
    } else {
#pragma unroll
      for (int m = 0; m < G; ++m) {
        const int k = j + m * S;
        float2 x = staged(BASIS == 2 ? L - 1 - k : k), n = make_float2(0.f, 0.f);
        if (k == 0)
          x = cscale(x, 2.f);
        else
          n = staged(BASIS == 2 ? k - 1 : L - k);
        v[m] = sc_pre(x, n, __ldg(&tq[k]));
      }
    }
    __syncthreads();  // the staging buffer is free, and so is the exchange buffer
    if (tid == 0 && tn < ntiles) {
      tcg::fence_smem_async();
      fetch(tn);
      drawn = (int)gridDim.x + atomicAdd(queue, 1);
    }
    if constexpr (C::ENGINE)
      fft_line<L, G, SIGN>(v, j, ColX<T>{reinterpret_cast<float2*>(ex), c}, tw, t3);
    else
      pipe_transform<L, G, SIGN, T, (C::PAIRED && BASIS != 0 && SIGN < 0)>(v, j, c, ex, stw);
    const int p = t / qtiles;
    const long long q = (long long)(t - p * qtiles) * T + c;
    float2* dst = out + (long long)p * L * Q + q;
    if constexpr (BASIS == 0) {
      if (q < Q) {
#pragma unroll
        for (int m = 0; m < G; ++m) dst[(long long)(j + m * S) * Q] = cscale(v[m], scale);
      }
    } else if constexpr (SIGN > 0) {
      if (q < Q) {
#pragma unroll
        for (int m = 0; m < G; ++m) {
          const int r = j + m * S;
          const float2 x = BASIS == 2 && r >= L / 2 ? make_float2(-v[m].x, -v[m].y) : v[m];
          dst[(long long)sc_perm(r, L) * Q] = cscale(x, scale);
        }
      }
    } else if constexpr (C::PAIRED) {
      constexpr int R2 = C::R2;
      if (q < Q) {
#pragma unroll
        for (int m = 0; m < G; ++m) {
          const int i = m & 1, r = m >> 1;
          const int k = (i == 0 ? j : (j == 0 ? G / 2 : G - j)) + r * G;
          const float2 own = v[i == 0 ? 2 * ((R2 - r) % R2) : 1 + 2 * (R2 - 1 - r)];  // j = 0
          const float2 other = v[(1 - i) + 2 * (R2 - 1 - r)];
          const float2 n = j == 0 ? own : other;
          const float2 ck = sc_post(v[m], n, __ldg(&tq[k]));
          dst[(long long)(BASIS == 2 ? L - 1 - k : k) * Q] = cscale(ck, (k == 0 ? 0.5f : 1.f) * scale);
        }
      }
    } else {
      // the mirrors V[L - k], real parts and then imaginary ones
      float2 n[G];
      __syncthreads();
#pragma unroll
      for (int m = 0; m < G; ++m) ex[slot(j + m * S)] = v[m].x;
      __syncthreads();
#pragma unroll
      for (int m = 0; m < G; ++m) n[m].x = ex[slot((L - (j + m * S)) & (L - 1))];
      __syncthreads();
#pragma unroll
      for (int m = 0; m < G; ++m) ex[slot(j + m * S)] = v[m].y;
      __syncthreads();
#pragma unroll
      for (int m = 0; m < G; ++m) n[m].y = ex[slot((L - (j + m * S)) & (L - 1))];
      if (q < Q) {
#pragma unroll
        for (int m = 0; m < G; ++m) {
          const int k = j + m * S;
          const float2 ck = sc_post(v[m], n[m], __ldg(&tq[k]));
          dst[(long long)(BASIS == 2 ? L - 1 - k : k) * Q] = cscale(ck, (k == 0 ? 0.5f : 1.f) * scale);
        }
      }
    }
    t = tn;
  }
  if (tid == 0) pipe_leave(queue);
}

static PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
    else
      cudaGetLastError();
  });
  return fn;
}

bool encode_f32_map(CUtensorMap* m, const void* base, int rank, const uint64_t* dims, const uint64_t* strides,
                    const uint32_t* box) {
  if (rank < 1 || rank > 5 || reinterpret_cast<uintptr_t>(base) % 16 != 0) return false;
  for (int i = 0; i + 1 < rank; ++i)
    if (strides[i] % 16 != 0 || strides[i] >= (1ULL << 40)) return false;
  if ((box[0] * 4u) % 16 != 0) return false;
  auto enc = tensor_map_encoder();
  if (!enc) return false;
  std::memset(m, 0, sizeof(*m));
  cuuint64_t d[5], s[4];
  cuuint32_t b[5], e[5];
  for (int i = 0; i < rank; ++i) {
    d[i] = (cuuint64_t)dims[i];
    b[i] = (cuuint32_t)box[i];
    e[i] = 1;
    if (i + 1 < rank) s[i] = (cuuint64_t)strides[i];
  }
  const CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, (cuuint32_t)rank, const_cast<void*>(base), d, s, b, e,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

// SMs of the current device
static cudaError_t sm_count(int* n) {
  static PerDevice once;
  static int nsm[kMaxDevices];
  int dev = 0;
  const cudaError_t e =
      once.run([](int d) { return cudaDeviceGetAttribute(&nsm[d], cudaDevAttrMultiProcessorCount, d); }, &dev);
  if (e == cudaSuccess) *n = nsm[dev];
  return e;
}

template <int L, int SIGN, bool PAIR, int BASIS>
static cudaError_t cpass_pipe(fftk_plan p, const CUtensorMap& m, const CUtensorMap& mo, float2* out, long long P,
                              long long Q, float scale, int kind, cudaStream_t st) {
  using C = PipeCfg<L, PAIR>;
  static PerDevice once;
  cudaError_t e = once.run([](int) {
    return cudaFuncSetAttribute(k_cpass_pipe<L, SIGN, PAIR, BASIS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)C::SMEM);
  });
  int nsm = 0;
  if (e == cudaSuccess) e = sm_count(&nsm);
  if (e != cudaSuccess) return e;
  const long long qtiles = (Q + C::T - 1) / C::T, ntiles = P * qtiles, cap = (long long)nsm * C::MINB;
  const unsigned grid = (unsigned)(ntiles < cap ? ntiles : cap);
  LaunchScope ls(p, kind, st);
  launch_pdl(k_cpass_pipe<L, SIGN, PAIR, BASIS>, grid, C::THREADS, C::SMEM, st, m, mo, out, Q, (int)qtiles,
             (int)ntiles, twiddles(p, 1 << Log2<L>::value), p->d_tw3, BASIS ? twiddles(p, 4 * L) : nullptr, scale,
             p->d_err);
  return cudaGetLastError();
}

// The maps of a pass: [P][L][2 Q] floats for even Q; for odd Q those of the
// even rows, [P][L / 2][2 Q], and, from 8 bytes before row 1, of the odd rows,
// [P][L / 2][2 (Q + 1)], with a row stride of 16 Q bytes (the last element of
// the second is the last of the array).
template <int L>
static bool pipe_maps(CUtensorMap* m, CUtensorMap* mo, const float2* in, long long P, long long Q) {
  using E = PipeCfg<L, false>;
  using O = PipeCfg<L, true>;
  if (8LL * Q * L >= (1LL << 40) || 2 * (Q + 1) >= (1LL << 31) || P >= (1LL << 31)) return false;
  const uint64_t rows = Q % 2 == 0 ? L : L / 2;
  const uint64_t strides[2] = {(uint64_t)(8 * Q * (L / (long long)rows)), (uint64_t)(8 * Q * L)};
  const uint64_t dims[3] = {(uint64_t)(2 * Q), rows, (uint64_t)P};
  const uint32_t box[3] = {2 * E::T, (uint32_t)(Q % 2 == 0 ? E::BOXR : O::BOXR), 1};
  if (!encode_f32_map(m, in, 3, dims, strides, box)) return false;
  if (Q % 2 == 0) return true;
  const uint64_t dims_odd[3] = {(uint64_t)(2 * (Q + 1)), rows, (uint64_t)P};
  const uint32_t box_odd[3] = {2 * O::ODD, O::BOXR, 1};
  return encode_f32_map(mo, in + Q - 1, 3, dims_odd, strides, box_odd);
}

// Arrays narrower than 16 columns, bases off 16 bytes and small passes keep the
// general pass (false, nothing launched).  Staging the next tile pays from a CTA's
// second tile on where one CTA fills an SM, and the later the more CTAs share it
// and cover each other's loads: more than one tile per resident CTA for lines of
// 768 points and more, two for 384 and 512, three for 256.  Transforms of batches
// of planes, the y and z or x and z passes, general pass -> here:
//   1024 points   152 tiles 15.6 -> 16.7 us   228 tiles 26.2 -> 25.5   912 tiles 87.1 -> 77.7
//    768          152       12.3 -> 13.3      228       20.7 -> 19.9   912       67.1 -> 59.5
//    512          400       19.8 -> 22.3      608       27.1 -> 26.5   912       39.4 -> 36.1
//    384          400       15.9 -> 15.6      608       20.9 -> 21.1   912       30.1 -> 30.0
//    256          912       18.2 -> 20.3     1824 (x)   90.3 -> 89.2  2432 (x)  117.5 -> 115.6
template <int L>
static bool pipe_applies(const float2* in, long long P, long long Q) {
  if (P <= 0 || Q < 16 || reinterpret_cast<uintptr_t>(in) % 16 != 0) return false;
  using C = PipeCfg<L, false>;
  constexpr int TURNS = C::MINB == 4 ? 3 : C::MINB;
  const long long tiles = P * ((Q + C::T - 1) / C::T);
  int nsm = 0;
  return tiles < (1LL << 31) && sm_count(&nsm) == cudaSuccess && tiles > (long long)TURNS * C::MINB * nsm;
}

// 256-point lines in a sine or cosine basis take the pipelined pass only in the
// inverse with even rows: forward, the mirror exchange spills 120 bytes at the 64
// registers of four CTAs per SM, and odd rows gain nothing (against k_scpass, with
// which these run now: 256^3 cosine-cosine-sine forward 92.7 -> 70.7 us, two such
// axes and Fourier 92.5 -> 68.9 us, its inverse 81.5 -> 73.1 us; the inverse x
// pass of four fields of 256^3, even rows, takes 263.5 us there and 256.7 us here).
constexpr bool pipe_built(int L, int sign, bool pair, int basis) {
  return basis == 0 || L != 256 || (sign > 0 && !pair);
}

template <int L, int SIGN, bool PAIR, int BASIS>
static bool pipe_run(fftk_plan p, const float2* in, float2* out, long long P, long long Q, float scale, int kind,
                     cudaStream_t st, cudaError_t* e) {
  if constexpr (!pipe_built(L, SIGN, PAIR, BASIS)) {
    return false;
  } else {
    CUtensorMap m{}, mo{};
    if (!pipe_applies<L>(in, P, Q) || !pipe_maps<L>(&m, &mo, in, P, Q)) return false;
    *e = cpass_pipe<L, SIGN, PAIR, BASIS>(p, m, PAIR ? mo : m, out, P, Q, scale, kind, st);
    return true;
  }
}

template <int L, int BASIS>
static bool pipe_l(fftk_plan p, int sign, const float2* in, float2* out, long long P, long long Q, float scale,
                   int kind, cudaStream_t st, cudaError_t* e) {
  if (Q % 2 == 0)
    return sign < 0 ? pipe_run<L, -1, false, BASIS>(p, in, out, P, Q, scale, kind, st, e)
                    : pipe_run<L, +1, false, BASIS>(p, in, out, P, Q, scale, kind, st, e);
  return sign < 0 ? pipe_run<L, -1, true, BASIS>(p, in, out, P, Q, scale, kind, st, e)
                  : pipe_run<L, +1, true, BASIS>(p, in, out, P, Q, scale, kind, st, e);
}

bool launch_cpass_tma(fftk_plan p, int L, int sign, const float2* in, float2* out, long long P, long long Q,
                      float scale, int kind, cudaStream_t st, cudaError_t* e) {
  switch (L) {
#define CASE(n) \
  case n:       \
    return pipe_l<n, 0>(p, sign, in, out, P, Q, scale, kind, st, e);
    CASE(256) CASE(384) CASE(512) CASE(768) CASE(1024) CASE(1536)
#undef CASE
  }
  return false;
}

bool launch_scpass_tma(fftk_plan p, int L, bool sine, int dir, const float2* in, float2* out, long long P, long long Q,
                       float scale, int kind, cudaStream_t st, cudaError_t* e) {
  switch (L) {
#define CASE(n) \
  case n:       \
    return sine ? pipe_l<n, 2>(p, dir, in, out, P, Q, scale, kind, st, e) \
                : pipe_l<n, 1>(p, dir, in, out, P, Q, scale, kind, st, e);
    CASE(256) CASE(512) CASE(1024)
#undef CASE
  }
  return false;
}

}  // namespace fftk
