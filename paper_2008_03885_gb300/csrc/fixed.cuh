// The FP64 refinement residual r = f - L u of second-order levels in fixed point.
//
// GB300 has one FP64 unit of half a lane per clock to each SM quarter, so the residual of a
// 5-point level (about ten FP64 operations a node) is bound by it, where its 20 bytes a node
// need 200 us of HBM at 8193^2. Its 64-bit integer adds run 30 times as fast. The 5-point
// operator is s = 1 / h^2 times the integers (-1; 4), so a tile's u values are written as
// integers in units of 2^(E - 1081) (E: the largest biased exponent in the tile and its halo:
// six bits below the last bit of the largest value), the stencil sum T is formed exactly,
// and r = f - s T is one fused multiply-add; FP64 keeps two operations a node (that one and
// the square for the norm).
//
// Precision. A node takes the integer sum only if each of its five values has no bit below
// the unit (all values within 6 binades of the largest do): T is then exact, r has the
// rounding of T to 53 bits and of the fused multiply-add, and is nowhere further off than the
// FP64 row, which rounds its partial sums too. A value that loses bits is made odd (the
// format's last bit is kept for that), and the nodes that read one take their FP64 row: beside
// zeros of u, in the corners of the grid, in tiles of wide range.
//
// The fourth-order operator (1, -16; 60) / (12 h^2) takes no fixed point: there FP64 rounds
// every product with 1 / 12 h^2 from the first step on, and an exact residual moves the
// residual history of a solve by up to 3e-9 of its start (measured at 4097^2), through the
// FP32 roundings of the inner cycle.
//
// With homogeneous data boundary values are 0 (not read); with data g they are read. A tile
// with an infinity, a NaN, or only tiny values (E < 128) goes through the FP64 rows instead.
#pragma once

#include <type_traits>

#include "device.cuh"

namespace nsmg {
namespace {

constexpr int kFxW = 64, kFxH = 32;  // tile; kernels use 32 x 8 threads
constexpr int kFxRW = kFxW + 2, kFxRH = kFxH + 2;  // with its halo
constexpr int kFxRegion = kFxRW * kFxRH, kFxPer = (kFxRegion + 255) / 256;
constexpr int kFxS0 = 6;  // fraction bits below the largest value's last one

// x in units of 2^(E - 1075 - kFxS0 - 1): even if exact in units twice that (values of exponent
// E - kFxS0 and above, and 0), odd if not (MARK; else not told); E >= exponent of x, E >= 128.
template <bool MARK>
__device__ __forceinline__ int64_t to_fixed(double x, int E) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const int k = min(E - (int)((hi >> 20) & 0x7ffu), 63);
  const uint64_t m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << (kFxS0 + 1);
  uint64_t q = m >> k;  // 0 for zeros and subnormals: k = 63
  if (MARK && k > kFxS0 + 1 && (hi << 1 | lo) != 0) q |= (m << (64 - k)) != 0 ? 1u : 0u;
  const int64_t neg = (int64_t)((int32_t)hi >> 31);
  return ((int64_t)q ^ neg) - neg;
}

// (double)T for |T| <= 2^53, without the FP64 unit.
__device__ __forceinline__ double narrow_to_double(int64_t T) {
  const uint64_t neg = (uint64_t)(T >> 63), a = ((uint64_t)T ^ neg) - neg;
  const int z = __clzll((long long)a);  // 10 .. 64
  const uint64_t m = z < 11 ? a >> 1 : a << (z - 11);  // leading bit at 52 (2^53 itself is even)
  const uint32_t hi = (uint32_t)(m >> 32) + ((uint32_t)(1085 - z) << 20);  // exponent 1086 - z, less the leading bit
  return __hiloint2double((int)(a == 0 ? 0u : hi | ((uint32_t)neg & 0x80000000u)), (int)(uint32_t)m);
}

__device__ __forceinline__ void copy_async8(void* dst, const void* src, bool ok) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src),
               "r"(ok ? 8 : 0)
               : "memory");
}

// Conversions off the common path. Calls, because the compiler would otherwise run them
// under a predicate for every node, and a predicated FP64 instruction occupies the unit too
// (8193^2, order 2: 796 us with them inlined, 709 without, before the copies ran ahead).
__device__ __noinline__ double wide_to_double(int64_t T) { return (double)T; }
__device__ __noinline__ float edge_to_float(double r, double scale) { return (float)(r * scale); }

// fl32(r * 2^k).
__device__ __forceinline__ float scaled_float(double r, int k, double scale) {
  const uint32_t hi = (uint32_t)__double2hiint(r), lo = (uint32_t)__double2loint(r);
  const int e = (int)((hi >> 20) & 0x7ff) - 896 + k;  // biased exponent of the float
  if (e < 1 || e > 253) return edge_to_float(r, scale);  // 0, underflow, overflow, NaN
  const uint32_t m = (hi & 0xfffffu) << 3 | lo >> 29, rem = lo & 0x1fffffffu;
  const uint32_t up = rem > 0x10000000u - (m & 1u) ? 1u : 0u;  // half to even
  return __uint_as_float((hi & 0x80000000u) | (((uint32_t)e << 23 | m) + up));
}

struct FxSmem {
  int64_t q[2][kFxRegion];  // u, then its fixed-point values, of this tile and the next
  uint32_t red[2][8];
};

// Copies u of the region of tile (i0, j0) to `dst` asynchronously, boundary values (unless
// data) and what lies beyond as 0; the grid's corners too, which no row reads: whatever a
// caller's array holds there must not set the tile's scale. Thread tid takes elements
// tid + 256 k.
__device__ __forceinline__ void fx_fetch(const LevelGeo<double>& L, const double* __restrict__ u, int i0, int j0,
                                         int64_t* dst) {
  const int tid = threadIdx.y * kBX + threadIdx.x, n = L.n;
  int x = tid % kFxRW, y = tid / kFxRW;
#pragma unroll
  for (int k = 0; k < kFxPer; ++k) {
    if (tid + 256 * k >= kFxRegion) break;
    const int i = i0 - 1 + x, j = j0 - 1 + y;
    const bool in_i = i >= 1 && i < n, in_j = j >= 1 && j < n;
    const bool ok = (in_i && in_j) || (L.bdata && ((in_i && (j == 0 || j == n)) || (in_j && (i == 0 || i == n))));
    copy_async8(dst + tid + 256 * k, ok ? u + (int64_t)j * L.pitch + i : u, ok);
    x += 256 % kFxRW;
    y += 256 / kFxRW;
    if (x >= kFxRW) {
      x -= kFxRW;
      ++y;
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// One tile whose region fx_fetch has put into `buf` (its copies waited for by each thread):
// store(i, j, r) for every unknown of columns i0 .. i0 + 63, rows j0 .. j0 + 31, in each
// thread for its own nodes. 256 threads as (32, 8), all of them; the caller puts a barrier
// before `buf` or sm.red is written again.
template <bool EXACT, class Store>
__device__ __forceinline__ void fx_tile(const LevelGeo<double>& L, const LevelDev<double>& LD, const double* __restrict__ u,
                                        const double* __restrict__ f, int i0, int j0, int64_t* buf, FxSmem& sm,
                                        Store store) {
  constexpr int W = kFxRW, kRows = kFxH / 4;
  const int tid = threadIdx.y * kBX + threadIdx.x, n = L.n;
  const int cx = tid & 63, r0 = (tid >> 6) * kRows, i = i0 + cx;
  double fv[kRows];
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    const int j = j0 + r0 + r;
    fv[r] = i >= 1 && i < n && j < n ? f[(int64_t)j * L.pitch + i] : 0.0;
  }
  // largest high word, and the smallest one less 1 (zeros wrap to the largest); values below
  // 2^-1042 count as 0: they reach neither the FP32 residual nor the norm
  uint32_t mx = 0, mn = ~0u;
#pragma unroll
  for (int k = 0; k < kFxPer; ++k) {
    if (tid + 256 * k >= kFxRegion) break;
    const uint32_t h = (uint32_t)((uint64_t)buf[tid + 256 * k] >> 32) & 0x7fffffffu;
    mx = max(mx, h);
    mn = min(mn, h - 1);
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  mn = __reduce_min_sync(0xffffffffu, mn);
  if (threadIdx.x == 0) {
    sm.red[0][threadIdx.y] = mx;
    sm.red[1][threadIdx.y] = mn;
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    mx = max(mx, sm.red[0][k]);
    mn = min(mn, sm.red[1][k]);
  }
  const int E = (int)(mx >> 20);
  uint32_t rest = 0;  // bit r: the node of row r takes its FP64 row
  if (mx != 0 && (E == 0x7ff || E < 128)) {  // uniform over the block
    rest = (1u << kRows) - 1;
  } else {
    // whether some value may lose bits (uniform over the block)
    const bool marks = mx != 0 && E - (int)((mn + 1) >> 20) > kFxS0;
    auto convert = [&](auto mark) {
#pragma unroll
      for (int k = 0; k < kFxPer; ++k) {
        if (tid + 256 * k >= kFxRegion) break;
        buf[tid + 256 * k] = to_fixed<decltype(mark)::value>(__longlong_as_double(buf[tid + 256 * k]), E);
      }
    };
    if (mx != 0) {
      if (marks) convert(std::true_type());
      else convert(std::false_type());
    }
    __syncthreads();
    // L u = c0 T, T in units of 2^(E - 1075 - kFxS0 - 1) (mx != 0: E >= 128, so the factor is
    // normal; mx == 0: the region holds zeros)
    const double unit = mx != 0 ? -L.c0 * __hiloint2double((E - 53 - kFxS0) << 20, 0) : 0.0;
    // Most tiles need no marks and run without the tests: 8193^2, order 2, solved u: 545 us
    // (595 with marks in every tile, 515 with none at all, bits lost; white noise, where most
    // warps hold a marked row, 995; FP64 rows 1208)
    auto walk = [&](auto marked) {
      const int64_t* q = buf + (r0 + 1) * W + cx + 1;
      int64_t below = q[-W], here = q[0];
#pragma unroll
      for (int r = 0; r < kRows; ++r, q += W) {
        const int64_t above = q[W], left = q[-1], right = q[1], T = (below + left + right + above) - (here << 2);
        const int j = j0 + r0 + r;
        if (decltype(marked)::value &&
            (((uint32_t)below | (uint32_t)left | (uint32_t)right | (uint32_t)above | (uint32_t)here) & 1u)) {
          rest |= 1u << r;
        } else if (j >= 1 && j < n) {  // |T| < 2^63
          double t;
          if ((uint64_t)(T + (1ll << 53)) <= (1ull << 54)) t = narrow_to_double(T);
          else t = wide_to_double(T);
          store(i, j, fma(unit, t, fv[r]));
        }
        below = here;
        here = above;
      }
    };
    if (i >= 1 && i < n) {
      if (marks) walk(std::true_type());
      else walk(std::false_type());
    }
  }
  // one pass for the marked rows of all lanes, whichever rows they are
  for (; rest; rest &= rest - 1) {
    const int j = j0 + r0 + __ffs((int)rest) - 1;
    if (i < 1 || i >= n || j < 1 || j >= n) continue;
    const int64_t at = (int64_t)j * L.pitch + i;
    store(i, j, Arith<double>::sub(f[at], apply_at<double, EXACT, 1>(LD, u, i, j, at, nullptr)));
  }
}

}  // namespace
}  // namespace nsmg
