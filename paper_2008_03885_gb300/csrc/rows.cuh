// Rows of boundary-class nodes by octets of lanes.
//
// A class row is a list of up to maxcnt (coefficient, offset) records, different for
// neighbouring nodes. One thread per node walks it as a serial chain: record, value,
// record, value, each waiting out an L2 latency, and in FP64 every divergent branch of a
// warp pays the FP64 unit again (one warp instruction occupies it for 64 clocks on GB300,
// however few lanes are active: measured 64.0 clocks with 1 as with 32 active lanes). Small
// levels consist of such nodes alone, and the strips along the boundary of a large level
// end up as the last warps of its grid.
//
// Here eight lanes share a node: the row's records are fetched in one batch (six a lane
// at 45 terms), then its values in a second, and staged in shared memory. In the exact
// order each lane then sums whole groups of equal coefficient (groups g, g + 8, ... in
// lane g: their sums are independent), and the group products are added in group order;
// with FMA the terms are one ordered chain from shared memory. The operations and their
// order are those of RowSum, so the results are the same bits; a 45-point FP64 row takes
// about 20 warp instructions of FP64 instead of 60.
//
// Measured on GB300 (ncu, warm caches), FP64 half-sweeps of 45-point levels: 33^2 rotated
// 18.7 us before; see kernels.cu for the figures after.
#pragma once

#include "device.cuh"

namespace nsmg {
namespace {

constexpr int kOct = 8;  // lanes per node

// Staging of one octet's row in shared memory: K values, K coefficients, K group starts.
template <typename T>
__host__ __device__ constexpr size_t oct_bytes(int K) {
  return (size_t)K * (2 * sizeof(T) + 1);
}
__host__ __device__ constexpr int oct_slots(int maxcnt) { return (maxcnt + kOct - 1) / kOct * kOct; }

// The nodes of one colour (or of all colours) that the octets of a launch take: rows of
// the lattice in three runs (below, above and beside the fast rectangle), each row cut
// into slots of one node. `all`: every unknown, no fast rectangle.
struct StripGeo {
  int32_t all;
  int32_t rstep, cstep;         // step between rows / nodes of a row
  int32_t fA0, cA0, fA1, cA1;   // first row and row count of the runs below and above
  int32_t fB, cB;               // rows beside the fast rectangle
  int32_t wA, wL, wR;           // slots of a full row, left and right of the rectangle
  int32_t total;                // slots
};

enum RowColour : int { kBlackNodes = 0, kRedNodes = 1, kAllNodes = 2 };

template <typename T>
inline StripGeo make_strips(const LevelGeo<T>& L, int colour, bool all) {
  StripGeo S;
  const int lo = L.lo, hi = L.n - 1;
  const bool none = (all && !L.bdata) || L.fxe < L.rx || L.fye < L.ry;
  S.all = none ? 1 : 0;
  S.rstep = (L.kind == kRot && colour != kAllNodes) ? 2 : 1;
  S.cstep = (L.kind == kAxis && colour == kAllNodes) ? 1 : 2;
  auto run = [&](int a, int b, int32_t& first, int32_t& count) {
    first = S.rstep == 2 ? a + ((a ^ colour) & 1) : a;
    count = first > b ? 0 : (b - first) / S.rstep + 1;
  };
  auto slots = [&](int a, int b) { return b < a ? 0 : (b - a) / S.cstep + 1; };
  run(lo, none ? hi : L.ry - 1, S.fA0, S.cA0);
  run(L.fye + 1, none ? L.fye : hi, S.fA1, S.cA1);
  run(L.ry, none ? L.ry - 1 : L.fye, S.fB, S.cB);
  S.wA = slots(lo, hi);
  S.wL = slots(lo, L.rx - 1);
  S.wR = slots(L.fxe + 1, hi);
  S.total = (S.cA0 + S.cA1) * S.wA + S.cB * (S.wL + S.wR);
  return S;
}

// Slot -> node; false for padding slots. colour as in make_strips.
template <typename T>
__device__ __forceinline__ bool strip_node(const LevelGeo<T>& L, const StripGeo& S, int colour, int slot, int& i,
                                           int& j) {
  if (slot >= S.total) return false;
  const int nA = (S.cA0 + S.cA1) * S.wA;
  int a, b, s;
  if (slot < nA) {
    const int r = slot / S.wA;
    s = slot - r * S.wA;
    j = r < S.cA0 ? S.fA0 + r * S.rstep : S.fA1 + (r - S.cA0) * S.rstep;
    a = L.lo;
    b = L.n - 1;
  } else {
    const int w = S.wL + S.wR;
    slot -= nA;
    const int r = slot / w;
    s = slot - r * w;
    j = S.fB + r * S.rstep;
    if (s < S.wL) {
      a = L.lo;
      b = L.rx - 1;
    } else {
      s -= S.wL;
      a = L.fxe + 1;
      b = L.n - 1;
    }
  }
  if (S.cstep == 1) {
    i = a + s;
  } else {
    const int par = L.kind == kRot ? (j & 1) : ((j ^ colour) & 1);  // parity of i
    i = a + ((a ^ par) & 1) + 2 * s;
  }
  return i <= b;
}

// (L u)(i, j) by the octet this lane belongs to, in every lane of it. All 32 lanes of the
// warp call it together; `on` is uniform over an octet (off: cnt = 0, result 0). `at(i, j)`
// gives the position of a node in u; `stage` is the octet's shared memory (oct_bytes(K),
// K >= the row's term count). PB: records a lane fetches per batch.
template <typename T, bool EXACT, int PB, class At>
__device__ __forceinline__ T octet_row(const LevelGeo<T>& L, const T* __restrict__ u, bool on, int i, int j, int cl,
                                       unsigned char* stage, int K, At at) {
  const int lane = threadIdx.x & 31, l8 = lane & 7, sh = lane & 24;
  T* xs = reinterpret_cast<T*>(stage);
  T* cs = xs + K;
  uint8_t* gs = reinterpret_cast<uint8_t*>(cs + K);
  int2 e = make_int2(0, 0);
  if (on) e = __ldg(&L.cls[cl]);
  const ClassTerm<T>* tt = L.terms + e.x;
  const int cnt = e.y;
  const int wmax = __reduce_max_sync(0xffffffffu, cnt);
  int ng = 0;
  for (int k0 = 0; k0 < wmax; k0 += kOct * PB) {
    Term<T> t[PB];
    T x[PB];
#pragma unroll
    for (int p = 0; p < PB; ++p) {
      const int k = k0 + kOct * p + l8;
      t[p].start = false;
      if (k < cnt) t[p] = load_term(tt + k);
    }
#pragma unroll
    for (int p = 0; p < PB; ++p) {
      const int k = k0 + kOct * p + l8;
      if (k < cnt) x[p] = u[at(i + t[p].dx, j + t[p].dy)];
    }
#pragma unroll
    for (int p = 0; p < PB; ++p) {
      const int k = k0 + kOct * p + l8;
      if (k < cnt) {
        xs[k] = x[p];
        cs[k] = t[p].c;
      }
      if (EXACT) {
        const unsigned m = (__ballot_sync(0xffffffffu, t[p].start) >> sh) & 0xffu;
        if (t[p].start) gs[ng + __popc(m & ((1u << l8) - 1u))] = (uint8_t)k;
        ng += __popc(m);
      }
    }
  }
  __syncwarp();
  T s = T(0);
  if (EXACT) {
    for (int g = l8; g < ng; g += kOct) {
      const int k0 = gs[g], k1 = g + 1 < ng ? gs[g + 1] : cnt;
      T v = xs[k0];
#pragma unroll 4
      for (int k = k0 + 1; k < k1; ++k) v = Arith<T>::add(v, xs[k]);
      xs[k0] = Arith<T>::mul(cs[k0], v);
    }
    __syncwarp();
    if (ng > 0) s = xs[0];
#pragma unroll 4
    for (int g = 1; g < ng; ++g) s = Arith<T>::add(s, xs[gs[g]]);
  } else {
    if (cnt > 0) s = Arith<T>::mul(cs[0], xs[0]);
#pragma unroll 8
    for (int k = 1; k < cnt; ++k) s = Arith<T>::fma(cs[k], xs[k], s);
  }
  __syncwarp();  // the stage may be reused
  return s;
}

struct LevelAt {  // positions in a level's global storage
  int kind, pitch;
  __device__ __forceinline__ int64_t operator()(int i, int j) const {
    return (int64_t)j * pitch + (kind == kRot ? (i >> 1) : i);
  }
};

enum RowMode : int { kRowRelax = 0, kRowResidual = 1 };

// One slot per octet of block `bid`: half-sweep (out = relaxed value) or residual
// (out = f - L u) of the strip nodes. blockDim = (32, warps).
template <typename T, bool EXACT, int PB, int MODE>
__device__ __forceinline__ void strip_rows(const LevelGeo<T>& L, const StripGeo& S, int colour, int bid,
                                           const T* __restrict__ u, const T* __restrict__ f, T* __restrict__ out,
                                           unsigned char* smem, int K) {
  const int lane = threadIdx.x & 31, oct = threadIdx.y * 4 + (lane >> 3);
  const int slot = bid * (blockDim.y * 4) + oct;
  int i = 0, j = 0;
  const bool on = strip_node(L, S, colour, slot, i, j);
  const LevelAt pos{L.kind, L.pitch};
  const int64_t at = pos(i, j);
  const int cl = on ? class_of(L, i, j) : 0;
  T fv = T(0), uv = T(0), wd = T(0);
  if (on) {
    fv = f[at];
    if (MODE == kRowRelax) {
      uv = u[at];
      wd = L.cls_wd[cl];
    }
  }
  const T s = octet_row<T, EXACT, PB>(L, u, on, i, j, cl, smem + oct * oct_bytes<T>(K), K, pos);
  if (!on || (lane & 7) != 0) return;
  const T r = Arith<T>::sub(fv, s);
  if (MODE == kRowRelax) out[at] = rnd(L, EXACT ? Arith<T>::add(uv, Arith<T>::mul(r, wd)) : Arith<T>::fma(r, wd, uv));
  else out[at] = rnd(L, r);
}

}  // namespace
}  // namespace nsmg
