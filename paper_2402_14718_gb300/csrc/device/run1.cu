// k_run_r1: all steps of a one-replica run in one launch.
//
// One replica is one FP32 position per row: an event's whole state is a few KB
// and its couplings fit in the SMs' shared memory, so nothing but latency
// bounds a step. Launched step by step (k_step_r1, k_step_r1g) a step took 2.9 us
// for 1,721 rows (one launch after another) and 20.6 us for 39,165 rows (rowptr,
// then columns, then positions, each an L2 round trip, then the heaviest row's
// chain). Here a cooperative grid of at most one CTA per SM runs all steps: a CTA
// keeps its rows' couplings in shared memory and its positions and momenta in
// registers, one thread per row, and only the new positions travel. A thread
// stores its row's position together with the step number in one 8-byte word;
// the next step gathers the union of a CTA's columns into shared memory by
// reading those words until they carry the step it needs (bounded). Data and flag
// in one word make a step one store and one read through L2: no fence, no grid
// barrier, no second read (a published step number per CTA, then the positions,
// took 9.1 us a step for 39,165 rows with a four-entry chain). Two buffers of
// words suffice: the pattern is symmetric, so a CTA that writes x_{k+1} over x_{k-1}
// has read an x_k from every CTA that reads its rows, and those had all of their
// x_{k-1} before they wrote that.
// A row's entries lie in slices of 32 rows of similar length, four entries of a
// lane together (a warp's reads of weights and indices have no bank conflicts),
// in CSR order: the sum is the one FMA chain of the other one-replica kernels, bit
// for bit, with eight positions in flight and the next indices on their way.
// Measured in runs of 256 to 512 steps, us per step, step kernels in a graph / now:
// 1,879 rows 5.0 / 1.55; 10,152 rows (37,322 nonzeros) 5.3 / 1.5; 10,999 rows 7.5 / 1.9;
// 39,445 rows 22.5 / 3.7; 67,374 rows 8.2 / 2.3. A cluster of 16 CTAs that wrote its
// positions into each other's shared memory took 1.45 us for 1,721 rows with the
// cluster's barrier, where this form then took 1.7, but 2.9 us for 10,214 rows, and 5
// to 9 us when its threads polled shared memory instead.
#include <cuda_bf16.h>

#include <algorithm>

#include "kernels.cuh"
#include "signs.cuh"

namespace sbd {
namespace {

// one 8-byte word {position, step}, read and written whole
__device__ __forceinline__ unsigned long long ld_word(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_word(unsigned long long* p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ unsigned long long pack_word(float x, uint32_t step) {
  return (unsigned long long)step << 32 | __float_as_uint(x);
}
// symplectic Euler and wall, as in the other one-replica kernels
template <int VARIANT>
__device__ __forceinline__ void update_row(const Run1Args& a, float pa, float c0, float h, float acc,
                                           float& x, float& y) {
  float force = -pa * x + c0 * (acc + h);
  if (VARIANT == 0) force -= x * x * x;
  y = y + a.dt * force;
  x = x + a.dta0 * y;
  if (VARIANT != 0 && fabsf(x) > 1.f) {
    x = copysignf(1.f, x);
    y = 0.f;
  }
}

// this thread's row and this CTA's entries
struct Row1 {
  int row = 0, deg = 0, base = 0;
  float x = 0.f, y = 0.f, h = 0.f, c0 = 0.f;
  __device__ __forceinline__ void load(const Run1Args& a, const Run1Cta& c, int t) {
    row = __ldg(a.perm + c.row0 + t);
    deg = __ldg(a.deg + c.row0 + t);
    base = __ldg(a.slice + c.slice0 + (t >> 5)) / 4 + (t & 31);
    x = a.x[a.cur][row];
    y = a.y[row];
    h = __ldg(a.h + row);
    c0 = __ldg(a.c0_ev + (a.row_event ? __ldg(a.row_event + row) : 0));
  }
};
__device__ __forceinline__ void load_entries(const Run1Args& a, const Run1Cta& c, float* wj, uint16_t* wi) {
  for (int i = threadIdx.x; i < c.nent / 4; i += kRun1Threads) {
    reinterpret_cast<float4*>(wj)[i] = __ldg(reinterpret_cast<const float4*>(a.ej + c.ent0) + i);
    reinterpret_cast<uint2*>(wi)[i] = __ldg(reinterpret_cast<const uint2*>(a.ei + c.ent0) + i);
  }
}

// SKIP: the test hook's form (a.skip_step); its test in every step would cost 1.4 % of one.
template <int VARIANT, bool SKIP>
__global__ void __launch_bounds__(kRun1Threads, 1) k_run_r1(const Run1Args a) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int t = threadIdx.x;
  const Run1Cta c = a.cta[blockIdx.x];
  // [positions: nx][weights: max_ent floats][indices: max_ent u16]
  float* const xs = reinterpret_cast<float*>(smem);
  float* const wj = xs + a.nx;
  uint16_t* const wi = reinterpret_cast<uint16_t*>(wj + a.max_ent);
  load_entries(a, c, wj, wi);
  auto g = [](float x) { return VARIANT == 2 ? sgnf(x) : x; };
  const bool own = t < c.nrows;
  Row1 r;
  if (own) r.load(a, c, t);
  const float4* const w4 = reinterpret_cast<const float4*>(wj) + r.base;
  const ushort4* const i4 = reinterpret_cast<const ushort4*>(wi) + r.base;
  const int mute = SKIP && blockIdx.x == 0 && t == 0 ? a.skip_step : -1;
  for (int k = 0; k < a.steps; ++k) {
    const float pa = a.a0 - __ldg(a.sched + k);
    bool late = false;
    if (k == 0) {
      for (int u = t; u < c.nu; u += kRun1Threads)
        xs[u] = g(a.x[a.cur][__ldg(a.ucol + c.u0 + u)]);
    } else {
      const unsigned long long* const in = a.word + (size_t)(k & 1) * a.n;
      for (int u0 = t; u0 < c.nu && !late; u0 += 4 * kRun1Threads) {
        unsigned long long w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int u = u0 + j * kRun1Threads;
          if (u < c.nu) w[j] = ld_word(in + __ldg(a.ucol + c.u0 + u));
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int u = u0 + j * kRun1Threads;
          if (u >= c.nu || late) break;
          unsigned long long since = 0;
          for (uint32_t it = 1; (uint32_t)(w[j] >> 32) != (uint32_t)k; ++it) {
            w[j] = ld_word(in + __ldg(a.ucol + c.u0 + u));
            if (it & 255u) continue;
            const unsigned long long now = now_ns();
            if (!since) since = now;
            if (now - since > a.wait_ns) {
              late = true;
              break;
            }
          }
          xs[u] = g(__uint_as_float((uint32_t)w[j]));
        }
      }
    }
    if (__syncthreads_or(late)) {
      if (t == 0) *a.err = kRun1Late;
      return;
    }
    if (own) {
      float acc = 0.f;
      if (r.deg > 0) {
        ushort4 ia = i4[0], ib = i4[32];
        int q = 0;
        for (; q + 8 <= r.deg; q += 8) {
          const float xv[8] = {xs[ia.x], xs[ia.y], xs[ia.z], xs[ia.w],
                               xs[ib.x], xs[ib.y], xs[ib.z], xs[ib.w]};
          const float4 wa = w4[8 * q], wb = w4[8 * q + 32];
          if (q + 8 < r.deg) {
            ia = i4[8 * q + 64];
            ib = i4[8 * q + 96];
          }
          acc = fmaf(wa.x, xv[0], acc);
          acc = fmaf(wa.y, xv[1], acc);
          acc = fmaf(wa.z, xv[2], acc);
          acc = fmaf(wa.w, xv[3], acc);
          acc = fmaf(wb.x, xv[4], acc);
          acc = fmaf(wb.y, xv[5], acc);
          acc = fmaf(wb.z, xv[6], acc);
          acc = fmaf(wb.w, xv[7], acc);
        }
        if (q < r.deg) {
          const float xv[8] = {xs[ia.x], xs[ia.y], xs[ia.z], xs[ia.w],
                               xs[ib.x], xs[ib.y], xs[ib.z], xs[ib.w]};
          const float4 wa = w4[8 * q], wb = w4[8 * q + 32];
          const float wv[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
          for (int u = 0; u < 7; ++u)
            if (q + u < r.deg) acc = fmaf(wv[u], xv[u], acc);
        }
      }
      update_row<VARIANT>(a, pa, r.c0, r.h, acc, r.x, r.y);
      if (!SKIP || k != mute)
        st_word(a.word + (size_t)((k + 1) & 1) * a.n + r.row, pack_word(r.x, (uint32_t)(k + 1)));
    }
    // every row of this CTA has read xs. (Two copies of xs without this barrier
    // let the threads without a row poll while the others still compute: 4.2
    // against 3.0 us a step for 39,165 rows.)
    __syncthreads();
  }
  if (own) {
    a.x[(a.cur + a.steps) & 1][r.row] = r.x;
    a.y[r.row] = r.y;
  }
}

// A warp fills one slot's entries, padding included (weight 0, index 0).
template <typename JT>
__global__ void __launch_bounds__(256) k_fill_run1(const Run1Cta* cta, const int32_t* perm, const int32_t* deg,
                                                   const int32_t* slice, const int32_t* ucol,
                                                   const int32_t* rowptr, const int32_t* col, const JT* J,
                                                   float* ej, uint16_t* ei) {
  const Run1Cta c = cta[blockIdx.x];
  const int lane = threadIdx.x & 31;
  for (int t = blockIdx.y * 8 + (threadIdx.x >> 5); t < c.nrows; t += 8 * gridDim.y) {
    const int row = perm[c.row0 + t], d = deg[c.row0 + t];
    const int len = (deg[c.row0 + t - t % 32] + 7) / 8 * 8;  // of the slice's longest row, its first
    const size_t e0 = (size_t)c.ent0 + slice[c.slice0 + t / 32] + 4 * (t % 32);
    for (int k = lane; k < len; k += 32) {
      float w = 0.f;
      int u = 0;
      if (k < d) {
        const int p = rowptr[row] + k;
        w = (float)J[p];
        if (ei) {  // binary search: every column of the row is there
          const int j = col[p];
          int hi = c.nu - 1;
          while (u < hi) {
            const int m = (u + hi) / 2;
            if (ucol[c.u0 + m] < j)
              u = m + 1;
            else
              hi = m;
          }
        }
      }
      const size_t e = e0 + (size_t)(k / 4) * 128 + k % 4;
      ej[e] = w;
      if (ei) ei[e] = (uint16_t)u;
    }
  }
}

template <int VARIANT>
cudaError_t launch_t(const Run1Args& a, size_t smem, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(a.nct);
  cfg.blockDim = dim3(kRun1Threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return a.skip_step >= 0 ? cudaLaunchKernelEx(&cfg, k_run_r1<VARIANT, true>, a)
                          : cudaLaunchKernelEx(&cfg, k_run_r1<VARIANT, false>, a);
}

}  // namespace

cudaError_t run1_prepare() {
  cudaError_t e = cudaSuccess;
  for (auto* k : {k_run_r1<0, false>, k_run_r1<1, false>, k_run_r1<2, false>, k_run_r1<0, true>,
                  k_run_r1<1, true>, k_run_r1<2, true>})
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kRun1Smem);
  return e;
}

int run1_blocks_per_sm(size_t smem) {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_run_r1<1, false>, kRun1Threads, smem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

cudaError_t launch_fill_run1(const Run1Cta* cta, int nct, const int32_t* perm, const int32_t* deg,
                             const int32_t* slice, const int32_t* ucol, const int32_t* rowptr,
                             const int32_t* col, const void* J, int jbf16, float* ej, uint16_t* ei,
                             cudaStream_t s) {
  const dim3 grid(nct, 16);
  if (jbf16)
    k_fill_run1<<<grid, 256, 0, s>>>(cta, perm, deg, slice, ucol, rowptr, col,
                                     static_cast<const __nv_bfloat16*>(J), ej, ei);
  else
    k_fill_run1<<<grid, 256, 0, s>>>(cta, perm, deg, slice, ucol, rowptr, col, static_cast<const float*>(J),
                                     ej, ei);
  return cudaGetLastError();
}

cudaError_t launch_run_r1(int variant, const Run1Args& a, size_t smem, cudaStream_t s) {
  // no word carries a step number yet (steps count from 1)
  cudaError_t e = cudaMemsetAsync(a.word, 0, (size_t)2 * a.n * sizeof(unsigned long long), s);
  if (e != cudaSuccess) return e;
  switch (variant) {
    case 0: return launch_t<0>(a, smem, s);
    case 1: return launch_t<1>(a, smem, s);
    default: return launch_t<2>(a, smem, s);
  }
}

}  // namespace sbd
