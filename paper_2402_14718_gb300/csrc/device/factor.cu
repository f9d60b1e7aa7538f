// Factored coupling product of the SB step (Eq. 2 / 6 / 10) for QUBOs whose
// couplings are mostly one weight shared by whole groups of rows.
//
// In the triplet QUBO of Eq. 13 every pair of triplets that share a hit and
// start on the same or adjacent layers is a conflict with the one weight w_c.
// Triplets holding hit h at position p form a group (h, p); triplets of groups
// (h, p) and (h, p') conflict exactly when |p - p'| <= 1. So the conflict part
// of J x is w (M^T W M) x with M the group incidence (three groups per
// triplet) and W the small position-coupling pattern, and the rest -- double
// counts of pairs sharing two hits, the consistent pairs (-1 instead of w_c)
// and the diagonal -- is an exact sparse residual formed on the host.
//
// One step is two launches:
//   k_fac_sum (dSB: k_fac_sum_sgn): for each group block g (one hit), T_s = sum
//               of x (dSB: of sgn x) over the block's members in slot s, then
//               U_s = sum_{s'} W[s][s'] T_{s'} for every slot whose U row a
//               factored row reads;
//   k_step_fac (dSB: k_step_fac_sgn): for each row, f = jf * sum of its U rows
//               + residual row . x, then the fused symplectic-Euler update and wall.
// A row that the host found cheaper in its plain CSR form has no U rows and
// its whole CSR row as residual, so one kernel serves both kinds of rows.
//
// Layout: lane l of a G-lane row group covers, for FP32 state, the replicas
// tile0 + 4 l + 4 G j + v (j < NCH, v < 4), i.e. 16-byte chunks strided by the
// group; for dSB sign bytes the 8 replicas tile0 + 8 l + v (one 8-byte load
// per neighbour). U rows use the same replica layout: FP32 for aSB / bSB; for
// dSB BF16 sums of 2^-7 sgn (exact while no U element sums more than 256
// members), else FP32 sums (the dSB kernels' NCH = 2 instances; NCH has no
// other meaning there).
//
// Every sum is formed in a fixed order (members by slot and row, residual in
// column order), so results are reproducible. For dSB with weights that are
// multiples of 1/4 every partial sum is exact and the step equals the
// CSR-order kernels bit for bit; for aSB / bSB the rounding order differs from
// the CSR order (per-step agreement to ~1e-6 relative).
#include <cuda_bf16.h>

#include "kernels.cuh"
#include "pdl.cuh"
#include "signs.cuh"

namespace sbd {
namespace {

constexpr int kFacBlock = kFacThreads;
// dSB: replicas per lane (measured on the 512-event batch against 16 per lane,
// and against requesting the U rows and own x, y before the residual walk:
// both cost occupancy and were slower)
constexpr int kSgnPer = 8;

// N 32-bit words loaded or stored as one vector (N = 2 or 4)
template <int N>
struct Words;
template <>
struct Words<2> {
  uint32_t w[2];
  __device__ __forceinline__ void ld(const void* p) {
    const uint2 t = *static_cast<const uint2*>(p);
    w[0] = t.x;
    w[1] = t.y;
  }
  __device__ __forceinline__ void st(void* p) const {
    *static_cast<uint2*>(p) = make_uint2(w[0], w[1]);
  }
};
template <>
struct Words<4> {
  uint32_t w[4];
  __device__ __forceinline__ void ld(const void* p) {
    const uint4 t = *static_cast<const uint4*>(p);
    w[0] = t.x;
    w[1] = t.y;
    w[2] = t.z;
    w[3] = t.w;
  }
  __device__ __forceinline__ void st(void* p) const {
    *static_cast<uint4*>(p) = make_uint4(w[0], w[1], w[2], w[3]);
  }
};

__device__ __forceinline__ unsigned lane_group_mask(int G) {
  const int lane = threadIdx.x & 31;
  return G == 32 ? 0xffffffffu : (((1u << G) - 1u) << (lane & ~(G - 1)));
}

// One member's values at this lane's replicas
template <int NCH>
struct Chunk {
  static constexpr int P = 4 * NCH;
  float4 t[NCH];
  __device__ __forceinline__ void load(const FacSumArgs& a, size_t off, int G, int row) {
#pragma unroll
    for (int j = 0; j < NCH; ++j)
      t[j] = reinterpret_cast<const float4*>(a.xin + (size_t)row * a.R + off)[G * j];
  }
  __device__ __forceinline__ void add_to(float (&u)[P]) const {
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
      u[4 * j] += t[j].x;
      u[4 * j + 1] += t[j].y;
      u[4 * j + 2] += t[j].z;
      u[4 * j + 3] += t[j].w;
    }
  }
};
// Adds a member in slot s2 to every U_s it couples to (s2 is the same for the
// whole lane group, so the branches do not diverge inside it).
template <int K, typename CH>
__device__ __forceinline__ void add_member(float (&U)[K][CH::P], const CH& v, int s2,
                                           uint32_t couple) {
#pragma unroll
  for (int s = 0; s < K; ++s)
    if ((couple >> (4 * s + s2)) & 1u) v.add_to(U[s]);
}

// Write the K U rows of block g from the sums U (for every slot in use).
template <int MODE, int NCH, int K, int P>
__device__ __forceinline__ void store_u(const FacSumArgs& a, int g, size_t off, int G,
                                        const float (&U)[K][P]) {
#pragma unroll
  for (int s = 0; s < K; ++s) {
    int u = __ldg(a.gout + (size_t)g * K + s);
    if (u < 0) continue;
    u = chk_idx(u, a.urows, kChkURow);
    if (MODE == 0) {
      float4* p = reinterpret_cast<float4*>(static_cast<float*>(a.U) + (size_t)u * a.R + off);
#pragma unroll
      for (int j = 0; j < NCH; ++j)
        p[G * j] = make_float4(U[s][4 * j], U[s][4 * j + 1], U[s][4 * j + 2], U[s][4 * j + 3]);
    } else if (NCH == 2) {
      // dSB, blocks of more than 256 members: FP32 sums of 2^-7 sgn (exact)
      float4* p = reinterpret_cast<float4*>(static_cast<float*>(a.U) + (size_t)u * a.R + off);
#pragma unroll
      for (int h = 0; h < P / 4; ++h)
        p[h] = make_float4(U[s][4 * h], U[s][4 * h + 1], U[s][4 * h + 2], U[s][4 * h + 3]);
    } else {
      // sums of 2^-7 sgn of at most 256 members: exact in BF16 (the top half of the FP32 word)
      uint16_t* p = static_cast<uint16_t*>(a.U) + (size_t)u * a.R + off;
#pragma unroll
      for (int h = 0; h < P / 8; ++h) {
        Words<4> w;
#pragma unroll
        for (int k = 0; k < 4; ++k)
          w.w[k] = (__float_as_uint(U[s][8 * h + 2 * k]) >> 16) |
                   (__float_as_uint(U[s][8 * h + 2 * k + 1]) & 0xffff0000u);
        w.st(p + 8 * h);
      }
    }
  }
}

// Lane l's P values of slot s of scratch slot c (the lane's own replicas).
__device__ __forceinline__ size_t scr_index(const FacSumArgs& a, int c, int s, size_t off, int G,
                                            int v) {
  return ((size_t)c * a.K + s) * a.R + off + 4 * G * (v >> 2) + (v & 3);
}

// Residency bounds of the FP32 forms (CTAs of 128 threads per SM). Two chunks per
// lane: seven and eight. One chunk: eight or nine, by fac_blocks().
template <int NCH, int B>
struct FacMinBlocks {
  static constexpr int sum = NCH == 2 ? 7 : B, step = NCH == 2 ? 8 : B;
};
// Nine CTAs leave 56 registers and spill up to 52 bytes since x and U come by plain
// loads (pdl.cuh); eight spill nothing, or at most 16. Nine stay the better choice where there are lanes
// enough to use the warps. bSB, us per step with nine / eight, and with __ldg and
// nine, launch by launch, that came before:
//   R = 16: 39,445 rows (158 k lanes) 21.2 / 17.4, 18.3; 98,134 rows (393 k) 28.6 /
//   27.2, 28.1; 156,688 rows (627 k) 31.1 / 31.3, 31.0; 242,044 rows (968 k) 48.3 / 50.4,
//   48.7. R = 32: 39,445 rows 21.2 / 19.6, 21.3; 98,134 rows (785 k) 36.1 / 35.6, 35.8;
//   114,665 rows (917 k) 42.2 / 43.0, 41.7. R = 64: 39,445 rows 25.4 / 24.6, 25.4;
//   108,750 rows (1.7 M) 58.2 / 61.0, 59.4.
//   R = 8 (two lanes a row): 39,445 rows (79 k) 26.4 / 25.5, 26.4; 67,374 rows (135 k)
//   19.2 / 20.8, 19.6; 98,134 rows (196 k) 31.9 / 31.1, 31.0; 242,044 rows 40.8 / 41.4, 40.9.
//   R = 4: 39,445 rows 33.0 / 32.2, 32.7; 472,676 rows 77.4 / 73.0, 71.8.
inline int fac_blocks(int64_t n, int R, int G) {
  const int64_t lanes = n * R / 4;
  return G >= 2 && lanes >= (G == 2 ? 100000 : 800000) ? 9 : 8;
}

// ---------------------------------------------------------------- dSB group sums
// Lane l of a G-lane group holds the replicas tile0 + 8 l .. + 7 (one 8-byte
// load per member). Members come four to a 16-byte word, so a lane reads its
// words itself and has eight members' signs in flight with the next words on
// their way, whatever G is; padding reads row 0 and couples to nothing, so no load has
// a predicate. All sums are whole numbers of 2^-7 below 2^24, exact in FP32 in
// any order: a block of more than kFacBig members is spread over a CTA's lane
// groups and added up by shuffles and through shared memory, so that the
// largest block (178 members on the 512-event batch) does not set the time.
// Per-block chains of four members at two latencies each took 14.3 of the 21 us
// of a step of 10,878 rows at R = 64; whole steps before / now with the row
// step below: 10,878 rows R = 16 35 / 8.7, R = 64 21.4 / 9.4; 39,165 rows R = 16 53
// / 11, R = 64 35 / 16.4, R = 256 63 / 46; 64 events (616,640 rows) R = 64 260 / 219
// early and 240 / 197 late in the run; 472,812 rows R = 128 341 / 303 and 317 / 280.
// Seven CTAs per SM (72 registers); eight spill.
template <bool UF32, int K>
__global__ void __launch_bounds__(kFacBlock, 7) k_fac_sum_sgn(const FacSumArgs a) {
  constexpr int P = kSgnPer;
  __shared__ float part[kFacBlock / 32][K * P][33];
  const int G = a.G;
  const int gq = threadIdx.x / G;
  const int l = threadIdx.x - gq * G;
  const int per = kFacBlock / G;
  const int2 cta = __ldg(a.cta + blockIdx.x);
  const bool big = cta.y == 0;
  if (!big && gq >= cta.y) return;  // the whole lane group leaves together
  const size_t off = (size_t)blockIdx.y * (kSgnPer * G) + kSgnPer * l;
  const uint8_t* const sg = a.sgn_in + off;
  const int R = a.R;
  const int4 item = __ldg(a.item + cta.x + (big ? 0 : gq));
  const int step = big ? per : 1;
  float U[K][P];
#pragma unroll
  for (int s = 0; s < K; ++s)
#pragma unroll
    for (int v = 0; v < P; ++v) U[s][v] = 0.f;
  const uint4 pad = make_uint4(kFacPad, kFacPad, kFacPad, kFacPad);
  int w = item.y + (big ? gq : 0);
  uint4 m0 = w < item.z ? __ldg(a.gword + w) : pad;
  uint4 m1 = w + step < item.z ? __ldg(a.gword + w + step) : pad;
  pdl_wait();  // from here on: what earlier launches write
  while (w < item.z) {
    const uint32_t m[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
    const bool two = w + step < item.z;
    uint2 v[8];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      v[u] = *reinterpret_cast<const uint2*>(
          sg + (size_t)chk_idx((int)(m[u] & 0x0fffffffu), a.n, kChkMember) * R);
    if (two) {
#pragma unroll
      for (int u = 4; u < 8; ++u)
        v[u] = *reinterpret_cast<const uint2*>(
            sg + (size_t)chk_idx((int)(m[u] & 0x0fffffffu), a.n, kChkMember) * R);
    }
    w += 2 * step;
    m0 = w < item.z ? __ldg(a.gword + w) : pad;
    m1 = w + step < item.z ? __ldg(a.gword + w + step) : pad;
    auto add = [&](uint32_t mw, const uint2& sv) {
      const uint32_t cs = a.couple >> (4 * (mw >> 28));  // W is symmetric: bit s of slot s2's nibble
      const uint32_t ww[2] = {sv.x, sv.y};
      float f[P];
#pragma unroll
      for (int k = 0; k < P; ++k) f[k] = scaled_sign_of_byte(ww[k >> 2], k & 3);
#pragma unroll
      for (int s = 0; s < K; ++s)
        if ((cs >> s) & 1u) {
#pragma unroll
          for (int k = 0; k < P; ++k) U[s][k] += f[k];
        }
    };
#pragma unroll
    for (int u = 0; u < 4; ++u) add(m[u], v[u]);
    if (two) {
#pragma unroll
      for (int u = 4; u < 8; ++u) add(m[u], v[u]);
    }
  }
  if (big) {
    for (int o = G; o < 32; o <<= 1)
#pragma unroll
      for (int s = 0; s < K; ++s)
#pragma unroll
        for (int k = 0; k < P; ++k) U[s][k] += __shfl_xor_sync(0xffffffffu, U[s][k], o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane < G)
#pragma unroll
      for (int s = 0; s < K; ++s)
#pragma unroll
        for (int k = 0; k < P; ++k) part[wid][s * P + k][lane] = U[s][k];
    __syncthreads();
    if (gq != 0) return;
#pragma unroll
    for (int s = 0; s < K; ++s)
#pragma unroll
      for (int k = 0; k < P; ++k) {
        float t = 0.f;
#pragma unroll
        for (int q = 0; q < kFacBlock / 32; ++q) t += part[q][s * P + k][l];
        U[s][k] = t;
      }
  }
  store_u<1, UF32 ? 2 : 1, K, P>(a, item.x, off, G, U);
}

template <int NCH, int K, int B>
__global__ void __launch_bounds__(kFacBlock, (FacMinBlocks<NCH, B>::sum)) k_fac_sum(const FacSumArgs a) {
  using C = Chunk<NCH>;
  constexpr int P = C::P;
  const int G = a.G;
  const int gq = threadIdx.x / G;
  const int l = threadIdx.x - gq * G;
  const int it = blockIdx.x * (kFacBlock / G) + gq;
  if (it >= a.nitems) return;  // the whole lane group leaves together
  const unsigned mask = lane_group_mask(G);
  const size_t off = (size_t)blockIdx.y * (4 * G * NCH) + 4 * l;
  const int4 item = __ldg(a.item + it);
  const int g = item.x;
  // slot boundaries of the block's members (members grouped by slot)
  int bnd[K + 1];
#pragma unroll
  for (int s = 0; s <= K; ++s) bnd[s] = __ldg(a.gseg + (size_t)g * K + s);
  float U[K][P];
#pragma unroll
  for (int s = 0; s < K; ++s)
#pragma unroll
    for (int v = 0; v < P; ++v) U[s][v] = 0.f;
  // this item's members in one pass, G entries per load, four rows in flight;
  // each lane's entry carries its row and slot, broadcast by shuffles
  if (item.y >= item.z) pdl_wait();
  for (int mb = item.y; mb < item.z; mb += G) {
    const int cnt = min(G, item.z - mb);
    int mr = 0, ms = 0;
    if (l < cnt) {
      const int t = mb + l;
      mr = chk_idx(__ldg(a.gmem + t), a.n, kChkMember);
#pragma unroll
      for (int s = 1; s < K; ++s) ms += t >= bnd[s] ? 1 : 0;
    }
    if (mb == item.y) pdl_wait();  // from here on: what earlier launches write
    int q = 0;
    for (; q + 4 <= cnt; q += 4) {
      int r[4], sl[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        r[u] = __shfl_sync(mask, mr, q + u, G);
        sl[u] = __shfl_sync(mask, ms, q + u, G);
      }
      C v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u].load(a, off, G, r[u]);
#pragma unroll
      for (int u = 0; u < 4; ++u) add_member<K, C>(U, v[u], sl[u], a.couple);
    }
    for (; q < cnt; ++q) {
      const int r0 = __shfl_sync(mask, mr, q, G), s0 = __shfl_sync(mask, ms, q, G);
      C v0;
      v0.load(a, off, G, r0);
      add_member<K, C>(U, v0, s0, a.couple);
    }
  }
  if (item.w < 0) {  // the whole block in one item
    store_u<0, NCH, K, P>(a, g, off, G, U);
    return;
  }
  // one chunk of a split block: its sums to the scratch slot; the chunk that
  // finishes last adds every chunk's slot in chunk order (a fixed order, so
  // the result does not depend on which chunk finishes last)
#pragma unroll
  for (int s = 0; s < K; ++s)
#pragma unroll
    for (int v = 0; v < P; ++v) a.scratch[scr_index(a, item.w, s, off, G, v)] = U[s][v];
  __threadfence();
  __syncwarp(mask);
  int last = 0;
  const int nc = __ldg(a.gnc + g);
  int* const cnt = a.cnt + (size_t)g * a.tiles + blockIdx.y;  // one counter per replica tile
  if (l == 0) last = atomicAdd(cnt, 1) == nc - 1;
  last = __shfl_sync(mask, last, 0, G);
  if (!last) return;
  __threadfence();
  const int c0 = __ldg(a.gscr0 + g);
#pragma unroll
  for (int s = 0; s < K; ++s)
#pragma unroll
    for (int v = 0; v < P; ++v) U[s][v] = 0.f;
  for (int c = 0; c < nc; ++c)
#pragma unroll
    for (int s = 0; s < K; ++s)
#pragma unroll
      for (int v = 0; v < P; ++v) U[s][v] += __ldcg(a.scratch + scr_index(a, c0 + c, s, off, G, v));
  store_u<0, NCH, K, P>(a, g, off, G, U);
  if (l == 0) *cnt = 0;  // ready for the next launch
}

__device__ __forceinline__ float jv(const float* J, int p) { return __ldg(J + p); }
__device__ __forceinline__ float jv(const __nv_bfloat16* J, int p) {
  return __uint_as_float((uint32_t)__ldg(reinterpret_cast<const unsigned short*>(J) + p) << 16);
}
// value t of a row head's J part (words from kFacHead + kFacHeadU on)
template <typename JT>
__device__ __forceinline__ float head_j(const uint32_t* hd, int t) {
  const uint32_t* p = hd + kFacHead + kFacHeadU;
  if (sizeof(JT) == 4) return __uint_as_float(__ldg(p + t));
  return __uint_as_float((uint32_t)__ldg(reinterpret_cast<const unsigned short*>(p) + t) << 16);
}

__global__ void k_fac_head(const FacHeadArgs a) {
  const int HW = fac_head_words(a.jbytes);
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)a.n * HW) return;
  const int64_t row = t / HW;
  const int w = (int)(t - row * HW);
  const int p0 = a.rrowptr[row], L = a.rrowptr[row + 1] - p0;
  uint32_t v = 0;
  if (w < kFacHead) {
    v = w < L ? (uint32_t)a.rcol[p0 + w] : 0u;
  } else if (w < kFacHead + kFacHeadU) {
    const int s = w - kFacHead;
    v = s < a.K ? (uint32_t)a.uidx[row * a.K + s] : 0xffffffffu;
  } else if (a.jbytes == 4) {
    const int e = w - kFacHead - kFacHeadU;
    v = e < L ? static_cast<const uint32_t*>(a.rJ)[p0 + e] : 0u;
  } else {
    const int e = 2 * (w - kFacHead - kFacHeadU);
    const uint16_t* J = static_cast<const uint16_t*>(a.rJ);
    v = (e < L ? J[p0 + e] : 0u) | (e + 1 < L ? (uint32_t)J[p0 + e + 1] << 16 : 0u);
  }
  a.head[t] = v;
}

// Adds cnt residual entries (lane q of the lane group holds column mc and
// weight mw of entry q) to this lane's replicas, four neighbour rows in flight.
template <int NCH>
__device__ __forceinline__ void walk_entries(float (&acc)[4 * NCH], int cnt, int mc, float mw,
                                             unsigned mask, int G, const float* xin, size_t off,
                                             int R) {
  int q = 0;
  for (; q + 4 <= cnt; q += 4) {
    int c[4];
    float w[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      c[u] = __shfl_sync(mask, mc, q + u, G);
      w[u] = __shfl_sync(mask, mw, q + u, G);
    }
    float4 t[4][NCH];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int j = 0; j < NCH; ++j)
        t[u][j] = reinterpret_cast<const float4*>(xin + (size_t)c[u] * R + off)[G * j];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int j = 0; j < NCH; ++j) {
        acc[4 * j] = fmaf(w[u], t[u][j].x, acc[4 * j]);
        acc[4 * j + 1] = fmaf(w[u], t[u][j].y, acc[4 * j + 1]);
        acc[4 * j + 2] = fmaf(w[u], t[u][j].z, acc[4 * j + 2]);
        acc[4 * j + 3] = fmaf(w[u], t[u][j].w, acc[4 * j + 3]);
      }
  }
  for (; q < cnt; ++q) {
    const int c = __shfl_sync(mask, mc, q, G);
    const float w = __shfl_sync(mask, mw, q, G);
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
      const float4 t = reinterpret_cast<const float4*>(xin + (size_t)c * R + off)[G * j];
      acc[4 * j] = fmaf(w, t.x, acc[4 * j]);
      acc[4 * j + 1] = fmaf(w, t.y, acc[4 * j + 1]);
      acc[4 * j + 2] = fmaf(w, t.z, acc[4 * j + 2]);
      acc[4 * j + 3] = fmaf(w, t.w, acc[4 * j + 3]);
    }
  }
}

// One U row of this lane: FP32 (NCH float4) or BF16 sums of 2^-7 sgn (two uint4)
template <int MODE, int NCH>
struct URow;
template <int NCH>
struct URow<0, NCH> {
  float4 t[NCH];
  __device__ __forceinline__ void load(const void* U, size_t base, int G) {
#pragma unroll
    for (int j = 0; j < NCH; ++j)
      t[j] = reinterpret_cast<const float4*>(static_cast<const float*>(U) + base)[G * j];
  }
  __device__ __forceinline__ void add_to(float (&fu)[4 * NCH]) const {
#pragma unroll
    for (int j = 0; j < NCH; ++j) {
      fu[4 * j] += t[j].x;
      fu[4 * j + 1] += t[j].y;
      fu[4 * j + 2] += t[j].z;
      fu[4 * j + 3] += t[j].w;
    }
  }
};
template <>
struct URow<1, 2> {  // dSB with FP32 U rows
  float4 t[kSgnPer / 4];
  __device__ __forceinline__ void load(const void* U, size_t base, int) {
#pragma unroll
    for (int h = 0; h < kSgnPer / 4; ++h)
      t[h] = reinterpret_cast<const float4*>(static_cast<const float*>(U) + base)[h];
  }
  __device__ __forceinline__ void add_to(float (&fu)[kSgnPer]) const {
#pragma unroll
    for (int h = 0; h < kSgnPer / 4; ++h) {
      fu[4 * h] += t[h].x;
      fu[4 * h + 1] += t[h].y;
      fu[4 * h + 2] += t[h].z;
      fu[4 * h + 3] += t[h].w;
    }
  }
};
template <int NCH>
struct URow<1, NCH> {
  Words<4> t[kSgnPer / 8];  // kSgnPer BF16 sums
  __device__ __forceinline__ void load(const void* U, size_t base, int) {
    const uint16_t* p = static_cast<const uint16_t*>(U) + base;
#pragma unroll
    for (int h = 0; h < kSgnPer / 8; ++h) t[h].ld(p + 8 * h);
  }
  __device__ __forceinline__ void add_to(float (&fu)[kSgnPer]) const {
#pragma unroll
    for (int h = 0; h < kSgnPer / 8; ++h)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        fu[8 * h + 2 * k] += __uint_as_float(t[h].w[k] << 16);
        fu[8 * h + 2 * k + 1] += __uint_as_float(t[h].w[k] & 0xffff0000u);
      }
  }
};

// VARIANT 0 aSB, 1 bSB
template <int VARIANT, int NCH, int K, int B, typename JT>
__global__ void __launch_bounds__(kFacBlock, (FacMinBlocks<NCH, B>::step)) k_step_fac(const FacStepArgs a) {
  constexpr int P = 4 * NCH;
  const int G = a.G;
  const int gq = threadIdx.x / G;
  const int l = threadIdx.x - gq * G;
  const int row = blockIdx.x * (kFacBlock / G) + gq;
  if (row >= a.n) return;
  const unsigned mask = lane_group_mask(G);
  const int R = a.R;
  const size_t off = (size_t)blockIdx.y * (4 * G * NCH) + 4 * l;
  const size_t idx = (size_t)row * R + off;
  const JT* J = static_cast<const JT*>(a.rJ);
  pdl_wait();
  // the row's own x and y and its U rows are read after the residual walk:
  // ask for them in L2 now, so that those loads do not wait on HBM
#pragma unroll
  for (int j = 0; j < NCH; ++j) {
    prefetch_l2(a.xin + idx + 4 * G * j);
    prefetch_l2(a.y + idx + 4 * G * j);
  }
  constexpr int HW = fac_head_words(sizeof(JT));
  const uint32_t* hd = a.head + (size_t)row * HW;
  int us[K];
#pragma unroll
  for (int s = 0; s < K; ++s) {
    us[s] = (int)__ldg(hd + kFacHead + s);
    if (us[s] >= 0) us[s] = chk_idx(us[s], a.urows, kChkURow);
    if (us[s] >= 0) prefetch_l2(static_cast<const char*>(a.U) + ((size_t)us[s] * R + off) * 4);
  }
  int p0 = __ldg(a.rrowptr + row), p1 = __ldg(a.rrowptr + row + 1);
  chk_rows(p0, p1, a.rnnz);

  // residual row, in column order: its first kFacHead entries from the head,
  // the rest from the residual CSR
  float acc[P];
#pragma unroll
  for (int v = 0; v < P; ++v) acc[v] = 0.f;
  const int nh = min(p1 - p0, kFacHead);
  for (int hb = 0; hb < nh; hb += G) {
    const int cnt = min(G, nh - hb);
    int mc = 0;
    float mw = 0.f;
    if (l < cnt) {
      mc = chk_idx((int)__ldg(hd + hb + l), a.n, kChkCol);
      mw = head_j<JT>(hd, hb + l);
    }
    walk_entries<NCH>(acc, cnt, mc, mw, mask, G, a.xin, off, R);
  }
  for (int pb = p0 + kFacHead; pb < p1; pb += G) {
    const int cnt = min(G, p1 - pb);
    int mc = 0;
    float mw = 0.f;
    if (l < cnt) {
      mc = chk_idx(__ldg(a.rcol + pb + l), a.n, kChkCol);
      mw = jv(J, pb + l);
    }
    walk_entries<NCH>(acc, cnt, mc, mw, mask, G, a.xin, off, R);
  }
  // the factored part: sum of this row's U rows (none for a plain row)
  bool any = false;
  float fu[P];
#pragma unroll
  for (int v = 0; v < P; ++v) fu[v] = 0.f;
#pragma unroll
  for (int s = 0; s < K; ++s) {
    if (us[s] < 0) continue;
    any = true;
    URow<0, NCH> ur;
    ur.load(a.U, (size_t)us[s] * R + off, G);
    ur.add_to(fu);
  }
  if (any) {
#pragma unroll
    for (int v = 0; v < P; ++v) acc[v] = fmaf(a.jf, fu[v], acc[v]);
  }

  // symplectic Euler: momentum with the old position, then position, then wall
  const float pa = a.a0 - __ldg(a.sched + a.k);
  const int ev = a.row_event ? __ldg(a.row_event + row) : 0;
  const float c0 = a.c0_ev[ev];
  const float hi = __ldg(a.h + row);
#pragma unroll
  for (int j = 0; j < NCH; ++j) {
    const size_t o = idx + 4 * G * j;
    const float4 xo = *reinterpret_cast<const float4*>(a.xin + o);
    const float4 yo = *reinterpret_cast<const float4*>(a.y + o);
    float xs[4] = {xo.x, xo.y, xo.z, xo.w}, ys[4] = {yo.x, yo.y, yo.z, yo.w};
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      float x = xs[v], y = ys[v];
      float force = -pa * x + c0 * (acc[4 * j + v] + hi);
      if (VARIANT == 0) force -= x * x * x;
      y = y + a.dt * force;
      x = x + a.dta0 * y;
      if (VARIANT != 0 && fabsf(x) > 1.f) {
        x = copysignf(1.f, x);
        y = 0.f;
      }
      xs[v] = x;
      ys[v] = y;
    }
    // a spin that stays on the wall keeps y = 0: nothing to write back there
    const float4 xn = make_float4(xs[0], xs[1], xs[2], xs[3]);
    const float4 yn = make_float4(ys[0], ys[1], ys[2], ys[3]);
    *reinterpret_cast<float4*>(a.xout + o) = xn;
    if (bits_differ(yo, yn)) *reinterpret_cast<float4*>(a.y + o) = yn;
  }
}

// ---------------------------------------------------------------- dSB row step
// One row per G-lane group, 8 replicas per lane. The row head holds the first
// eight residual entries and the U rows in one line: each lane reads it with
// four 16-byte loads (no shuffles), then has all of the head's neighbours (zero
// weights pad them, so no load has a predicate) and the U rows in flight at once;
// longer residual rows follow four neighbours at a time, the U rows after the
// head's neighbours (together with them the registers spill at this residency).
// Bound by latency and issue. Ten CTAs per SM (48 registers); with eight (64,
// U rows first) the 64-event batch takes 216 us a step late in the run, with
// twelve (spills) 218, with ten 197; requesting the own x and y first took 216.
// FP32 U rows (UF32) hold 24 registers in flight and lie in HBM: they are asked for
// in L2 with the head's neighbours and read one after the other at the end.
// 1,031,640 rows, us per step, in flight as the BF16 ones (52 bytes spilled) / so, and
// with the shuffled walk that came before: R = 128 851 / 737, 786; R = 64 501 / 438,
// 454; R = 16 233 / 216, 293. Eight CTAs, in flight 830, one by one 812; nine 794.
template <bool UF32, int K, typename JT>
__global__ void __launch_bounds__(kFacBlock, 10) k_step_fac_sgn(const FacStepArgs a) {
  constexpr int P = kSgnPer;
  constexpr int NCH = UF32 ? 2 : 1;
  const int G = a.G;
  const int gq = threadIdx.x / G;
  const int l = threadIdx.x - gq * G;
  const int row = blockIdx.x * (kFacBlock / G) + gq;
  if (row >= a.n) return;
  const int R = a.R;
  const size_t off = (size_t)blockIdx.y * (kSgnPer * G) + kSgnPer * l;
  const size_t idx = (size_t)row * R + off;
  constexpr int HW = fac_head_words(sizeof(JT));
  const uint4* const hd = reinterpret_cast<const uint4*>(a.head + (size_t)row * HW);
  const uint4 hc0 = __ldg(hd), hc1 = __ldg(hd + 1), hu = __ldg(hd + 2), hj0 = __ldg(hd + 3);
  uint4 hj1 = make_uint4(0u, 0u, 0u, 0u);
  if (sizeof(JT) == 4) hj1 = __ldg(hd + 4);
  int p0 = __ldg(a.rrowptr + row), p1 = __ldg(a.rrowptr + row + 1);
  const int ev = a.row_event ? __ldg(a.row_event + row) : 0;
  const float hi = __ldg(a.h + row);
  chk_rows(p0, p1, a.rnnz);
  pdl_wait();  // from here on: what earlier launches write
  prefetch_l2(a.xin + idx);
  prefetch_l2(a.y + idx);
  const uint8_t* const sg = a.sgn_in + off;
  const int L = p1 - p0;
  auto gather = [&](uint32_t c) {
    return *reinterpret_cast<const uint2*>(sg + (size_t)chk_idx((int)c, a.n, kChkCol) * R);
  };
  uint2 s0[4], s1[4];
  const uint32_t ca[4] = {hc0.x, hc0.y, hc0.z, hc0.w}, cb[4] = {hc1.x, hc1.y, hc1.z, hc1.w};
#pragma unroll
  for (int u = 0; u < 4; ++u) s0[u] = gather(ca[u]);
  if (L > 4) {
#pragma unroll
    for (int u = 0; u < 4; ++u) s1[u] = gather(cb[u]);
  }
  const uint32_t uw[4] = {hu.x, hu.y, hu.z, hu.w};
  if (UF32) {
#pragma unroll
    for (int s = 0; s < K; ++s)
      if ((int)uw[s] >= 0)
        prefetch_l2(static_cast<const float*>(a.U) + (size_t)chk_idx((int)uw[s], a.urows, kChkURow) * R + off);
  }
  const float c0 = a.c0_ev[ev];
  const float pa = a.a0 - __ldg(a.sched + a.k);

  // residual row in column order: weights scaled by 2^7, sign bytes read as 2^-7 sgn
  float acc[P];
#pragma unroll
  for (int v = 0; v < P; ++v) acc[v] = 0.f;
  auto take = [&](float w, const uint2& sv) {
    const uint32_t ww[2] = {sv.x, sv.y};
#pragma unroll
    for (int v = 0; v < P; ++v) acc[v] = fmaf(w, scaled_sign_of_byte(ww[v >> 2], v & 3), acc[v]);
  };
  auto weight = [&](const uint4& lo, const uint4& hi4, int t) {  // head weight t, times 2^7
    if (sizeof(JT) == 4) {
      const uint32_t q[8] = {lo.x, lo.y, lo.z, lo.w, hi4.x, hi4.y, hi4.z, hi4.w};
      return __uint_as_float(q[t]) * kSignScale;
    }
    const uint32_t q[4] = {lo.x, lo.y, lo.z, lo.w};
    const uint32_t wd = q[t >> 1];
    return __uint_as_float(t & 1 ? wd & 0xffff0000u : wd << 16) * kSignScale;
  };
#pragma unroll
  for (int u = 0; u < 4; ++u) take(weight(hj0, hj1, u), s0[u]);
  if (L > 4) {
#pragma unroll
    for (int u = 0; u < 4; ++u) take(weight(hj0, hj1, 4 + u), s1[u]);
  }
  URow<1, NCH> ur[K];
#pragma unroll
  for (int s = 0; s < K; ++s)
    if (!UF32 && (int)uw[s] >= 0)
      ur[s].load(a.U, (size_t)chk_idx((int)uw[s], a.urows, kChkURow) * R + off, G);
  if (L > kFacHead) {
    const JT* J = static_cast<const JT*>(a.rJ);
    int p = p0 + kFacHead;
    for (; p + 4 <= p1; p += 4) {
      uint2 sv[4];
      float w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) sv[u] = gather((uint32_t)__ldg(a.rcol + p + u));
#pragma unroll
      for (int u = 0; u < 4; ++u) w[u] = jv(J, p + u) * kSignScale;
#pragma unroll
      for (int u = 0; u < 4; ++u) take(w[u], sv[u]);
    }
    if (p < p1) {
      uint2 sv[3];
#pragma unroll
      for (int u = 0; u < 3; ++u)
        if (p + u < p1) sv[u] = gather((uint32_t)__ldg(a.rcol + p + u));
#pragma unroll
      for (int u = 0; u < 3; ++u)
        if (p + u < p1) take(jv(J, p + u) * kSignScale, sv[u]);
    }
  }
  // the factored part: U holds sums of 2^-7 sgn, so the scale is 2^7 jf (exact)
  bool any = false;
  float fu[P];
#pragma unroll
  for (int v = 0; v < P; ++v) fu[v] = 0.f;
#pragma unroll
  for (int s = 0; s < K; ++s)
    if ((int)uw[s] >= 0) {
      any = true;
      if (UF32) ur[s].load(a.U, (size_t)chk_idx((int)uw[s], a.urows, kChkURow) * R + off, G);
      ur[s].add_to(fu);
    }
  if (any) {
    const float jf = a.jf * kSignScale;
#pragma unroll
    for (int v = 0; v < P; ++v) acc[v] = fmaf(jf, fu[v], acc[v]);
  }

  // symplectic Euler: momentum with the old position, then position, then wall
  Words<2> sw;  // the new sign bytes
  sw.w[0] = sw.w[1] = 0u;
  const bool inplace = a.xout == a.xin;
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const size_t o = idx + 4 * j;
    const float4 xq = *reinterpret_cast<const float4*>(a.xin + o);
    const float4 yq = *reinterpret_cast<const float4*>(a.y + o);
    float xs[4] = {xq.x, xq.y, xq.z, xq.w}, ys[4] = {yq.x, yq.y, yq.z, yq.w};
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      float x = xs[v], y = ys[v];
      const float force = -pa * x + c0 * (acc[4 * j + v] + hi);
      y = y + a.dt * force;
      x = x + a.dta0 * y;
      if (fabsf(x) > 1.f) {
        x = copysignf(1.f, x);
        y = 0.f;
      }
      xs[v] = x;
      ys[v] = y;
      sw.w[j] |= sign_byte(x) << (8 * v);
    }
    // a spin that stays on the wall keeps x = +-1, y = 0: nothing to write back
    const float4 xn = make_float4(xs[0], xs[1], xs[2], xs[3]);
    const float4 yn = make_float4(ys[0], ys[1], ys[2], ys[3]);
    if (!inplace || bits_differ(xq, xn)) *reinterpret_cast<float4*>(a.xout + o) = xn;
    if (bits_differ(yq, yn)) *reinterpret_cast<float4*>(a.y + o) = yn;
  }
  sw.st(a.sgn_out + idx);
}

template <int NCH, int K>
cudaError_t launch_sum_k(const FacSumArgs& a, cudaStream_t s) {
  if (a.nitems <= 0) return cudaSuccess;
  const int per = kFacBlock / a.G;
  dim3 grid((a.nitems + per - 1) / per, a.tiles);
  if (NCH == 1 && fac_blocks(a.n, a.R, a.G) == 9)
    return launch_pdl(k_fac_sum<NCH, K, NCH == 1 ? 9 : 8>, grid, kFacBlock, a, s);
  return launch_pdl(k_fac_sum<NCH, K, 8>, grid, kFacBlock, a, s);
}

template <int NCH>
cudaError_t launch_sum_n(const FacSumArgs& a, cudaStream_t s) {
  switch (a.K) {
    case 1: return launch_sum_k<NCH, 1>(a, s);
    case 2: return launch_sum_k<NCH, 2>(a, s);
    case 3: return launch_sum_k<NCH, 3>(a, s);
    case 4: return launch_sum_k<NCH, 4>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

template <int VARIANT, int NCH, int K, typename JT>
cudaError_t launch_step_k(const FacStepArgs& a, cudaStream_t s) {
  const int per = kFacBlock / a.G;
  dim3 grid((a.n + per - 1) / per, a.tiles);
  if (NCH == 1 && fac_blocks(a.n, a.R, a.G) == 9)
    return launch_pdl(k_step_fac<VARIANT, NCH, K, NCH == 1 ? 9 : 8, JT>, grid, kFacBlock, a, s);
  return launch_pdl(k_step_fac<VARIANT, NCH, K, 8, JT>, grid, kFacBlock, a, s);
}

template <int VARIANT, int NCH, typename JT>
cudaError_t launch_step_n(const FacStepArgs& a, cudaStream_t s) {
  switch (a.K) {
    case 1: return launch_step_k<VARIANT, NCH, 1, JT>(a, s);
    case 2: return launch_step_k<VARIANT, NCH, 2, JT>(a, s);
    case 3: return launch_step_k<VARIANT, NCH, 3, JT>(a, s);
    case 4: return launch_step_k<VARIANT, NCH, 4, JT>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

template <bool UF32>
cudaError_t launch_sum_sgn(const FacSumArgs& a, cudaStream_t s) {
  if (a.nctas <= 0) return cudaSuccess;
  dim3 grid(a.nctas, a.tiles);
  switch (a.K) {
    case 1: return launch_pdl(k_fac_sum_sgn<UF32, 1>, grid, kFacBlock, a, s);
    case 2: return launch_pdl(k_fac_sum_sgn<UF32, 2>, grid, kFacBlock, a, s);
    case 3: return launch_pdl(k_fac_sum_sgn<UF32, 3>, grid, kFacBlock, a, s);
    case 4: return launch_pdl(k_fac_sum_sgn<UF32, 4>, grid, kFacBlock, a, s);
    default: return cudaErrorInvalidValue;
  }
}

template <bool UF32, typename JT>
cudaError_t launch_step_sgn(const FacStepArgs& a, cudaStream_t s) {
  const int per = kFacBlock / a.G;
  dim3 grid((a.n + per - 1) / per, a.tiles);
  switch (a.K) {
    case 1: return launch_pdl(k_step_fac_sgn<UF32, 1, JT>, grid, kFacBlock, a, s);
    case 2: return launch_pdl(k_step_fac_sgn<UF32, 2, JT>, grid, kFacBlock, a, s);
    case 3: return launch_pdl(k_step_fac_sgn<UF32, 3, JT>, grid, kFacBlock, a, s);
    case 4: return launch_pdl(k_step_fac_sgn<UF32, 4, JT>, grid, kFacBlock, a, s);
    default: return cudaErrorInvalidValue;
  }
}

template <typename JT>
cudaError_t launch_step_j(int variant, const FacStepArgs& a, cudaStream_t s) {
  if (variant == 2) return a.NCH == 2 ? launch_step_sgn<true, JT>(a, s) : launch_step_sgn<false, JT>(a, s);
  if (a.NCH == 2)
    return variant == 0 ? launch_step_n<0, 2, JT>(a, s) : launch_step_n<1, 2, JT>(a, s);
  return variant == 0 ? launch_step_n<0, 1, JT>(a, s) : launch_step_n<1, 1, JT>(a, s);
}

}  // namespace

bool fac_tiling(int variant, int R, int* G, int* NCH, int* tiles) {
  if (R < 1) return false;
  if (variant == 2) {
    if (R % kSgnPer) return false;
    const int C = R / kSgnPer;
    if (C <= 32 && (C & (C - 1)) == 0) {
      *G = C;
      *NCH = 1;
      *tiles = 1;
      return true;
    }
    if (C % 32 == 0) {
      *G = 32;
      *NCH = 1;
      *tiles = C / 32;
      return true;
    }
    return false;
  }
  if (R % 4) return false;
  const int C = R / 4;
  if (C <= 32 && (C & (C - 1)) == 0) {
    *G = C;
    *NCH = 1;
    *tiles = 1;
    return true;
  }
  if (C % 64 == 0) {
    *G = 32;
    *NCH = 2;
    *tiles = C / 64;
    return true;
  }
  if (C % 32 == 0) {
    *G = 32;
    *NCH = 1;
    *tiles = C / 32;
    return true;
  }
  return false;
}

cudaError_t launch_fac_head(const FacHeadArgs& a, cudaStream_t s) {
  const int64_t total = (int64_t)a.n * fac_head_words(a.jbytes);
  if (total <= 0) return cudaSuccess;
  k_fac_head<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_fac_sum(int variant, const FacSumArgs& a, cudaStream_t s) {
  if (variant == 2) return a.NCH == 2 ? launch_sum_sgn<true>(a, s) : launch_sum_sgn<false>(a, s);
  return a.NCH == 2 ? launch_sum_n<2>(a, s) : launch_sum_n<1>(a, s);
}

cudaError_t launch_step_fac(int variant, int jbf16, const FacStepArgs& a, cudaStream_t s) {
  if (a.n <= 0) return cudaSuccess;
  return jbf16 ? launch_step_j<__nv_bfloat16>(variant, a, s) : launch_step_j<float>(variant, a, s);
}

SB_CHECK_READER(chk_read_factor)

}  // namespace sbd
