// Rows of boundary-class nodes by octets of lanes.
//
// A class row is a list of up to 45 (121 with cubic transfers) coefficients and offsets,
// different for neighbouring nodes. One thread per node walks it as a serial chain:
// record, value, record, value, each waiting out an L2 latency, and in FP64 every divergent
// branch of a warp pays the FP64 unit again (one warp instruction occupies it for 64 clocks
// on GB300, however few lanes are active: measured 64.0 clocks with 1 as with 32 active
// lanes). Small levels consist of such nodes alone, and the strips along the boundary of a
// large level end up as the last warps of its grid.
//
// Here eight lanes share a node and each takes whole groups of equal coefficient (GroupRec:
// coefficient and up to eight offsets in 48 bytes; groups g and g + 8 of the row in lane
// g): one batch of record loads, one batch of value loads, then the group sums of all
// lanes at once, and the group products added in group order by shuffles. With FMA the
// row is one ordered chain, handed from lane to lane; in FP64 each lane's turn takes as many
// operations as the longest of the warp's groups in that place, no more: with turns padded to
// four or eight, rows of many one-term groups (cubic transfers on an 8 x 8 lattice, 49
// groups) took 13.6 us a residual and 26.6 a sweep, 8.4 and 17.0 by one thread a node; now 6.0
// and 11.5 (steps of levels with 45 terms: 0.69 of the padded form). The operations and their order are
// those of RowSum, so the results are the same bits; a 45-point FP64 row takes about 20
// warp instructions of FP64 instead of 60, and about 250 instructions in all (a lone warp
// spends 8-16 clocks on each). A first form that staged records and values in shared
// memory and summed from there took 600 instructions.
#pragma once

#include "device.cuh"

namespace nsmg {
namespace {

constexpr int kOct = 8;  // lanes per node

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
  uint32_t mA, mB;              // ceil(2^32 / wA), ceil(2^32 / (wL + wR)): slot / w = slot m >> 32
                                // (exact for slot w < 2^32; w = 1 is handled apart)
};

enum RowColour : int { kBlackNodes = 0, kRedNodes = 1, kAllNodes = 2 };

template <typename T>
__host__ __device__ inline StripGeo make_strips(const LevelGeo<T>& L, int colour, bool all) {
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
  auto magic = [](uint32_t w) { return w > 1 ? 0xffffffffu / w + 1 : 0u; };
  S.mA = magic(S.wA);
  S.mB = magic(S.wL + S.wR);
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
    const int r = S.mA ? (int)__umulhi((uint32_t)slot, S.mA) : slot;
    s = slot - r * S.wA;
    j = r < S.cA0 ? S.fA0 + r * S.rstep : S.fA1 + (r - S.cA0) * S.rstep;
    a = L.lo;
    b = L.n - 1;
  } else {
    const int w = S.wL + S.wR;
    slot -= nA;
    const int r = S.mB ? (int)__umulhi((uint32_t)slot, S.mB) : slot;
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

// Row of class cl at (i, j), term by term in one thread: rows without group records, and
// FP32 levels in shared memory.
template <typename T, bool EXACT>
__device__ __forceinline__ T serial_row(const LevelGeo<T>& L, const T* own, const T* opp, int i, int j, int cl) {
  RowSum<T, EXACT> acc;
  const int2 e = __ldg(&L.cls[cl]);
  const ClassTerm<T>* tt = L.terms + e.x;
  const int at = (int)sidx(L, i, j);
  const int other_at = (int)(opp - own), rot = L.kind == kRot;
#pragma unroll 4
  for (int k = 0; k < e.y; ++k) {
    const Term<T> t = load_term(tt + k);
    const int other = (rot ? t.dy : t.dx + t.dy) & 1;
    acc.add(t.c, own[(int)sidx(L, i + t.dx, j + t.dy) - at + (other ? other_at : 0)], t.start);
  }
  return acc.value();
}

template <typename T>
__device__ __forceinline__ GroupRec<T> load_group(const GroupRec<T>* p) {
  union {
    int4 w[3];
    GroupRec<T> r;
  } v;
#pragma unroll
  for (int k = 0; k < 3; ++k) v.w[k] = __ldg(reinterpret_cast<const int4*>(p) + k);
  return v.r;
}

// (L u)(i, j) by the octet this lane belongs to, in every lane of it. All 32 lanes of the
// warp call it together; `on` is uniform over an octet (off: some value). `own` and `opp`
// point at the node's position in the arrays that hold the values of its own and of the
// other colour (usually the same array). NREC: records a lane fetches at once. pre() runs
// after the first records' loads and before any value is read.
template <typename T, bool EXACT, int NREC, class Pre>
__device__ __forceinline__ T octet_row(const LevelGeo<T>& L, const T* own, const T* opp, bool on, int i, int j, int cl,
                                       Pre pre) {
  // no records (a group of more than eight terms: true high-order Galerkin, level 1): all eight
  // lanes walk the row; small levels leave the lanes idle anyway, and such solves take 0.3-0.75
  // of their time with one thread a node
  if (L.maxg == 0) {
    pre();
    return on ? serial_row<T, EXACT>(L, own, opp, i, j, cl) : T(0);
  }
  const int l8 = threadIdx.x & 7, par2 = L.kind == kRot ? 2 * (i & 1) : 0;
  const GroupRec<T>* R = L.groups + (int64_t)cl * L.maxg;
  const bool split = own != opp;
  T s = T(-0.0);  // the identity of both sums: x + (-0) = x, fma(c, x, -0) = fl(c x)
  for (int g0 = 0; g0 < L.maxg; g0 += kOct * NREC) {
    GroupRec<T> r[NREC];
    T x[NREC][kGroupMax];
#pragma unroll
    for (int k = 0; k < NREC; ++k) {
      const int g = g0 + kOct * k + l8;
      r[k].cnt = 0;
      r[k].c = T(1);
      if (on && g < L.maxg) r[k] = load_group(R + g);
    }
    if (g0 == 0) pre();
#pragma unroll
    for (int k = 0; k < NREC; ++k) {
      // a missing term adds -0 to either sum
      const T pad = EXACT || r[k].c > T(0) ? T(-0.0) : T(0);
#pragma unroll
      for (int m = 0; m < kGroupMax; ++m) {
        x[k][m] = pad;
        if (m < r[k].cnt) x[k][m] = (split && (r[k].d[m] & 1) ? opp : own)[(r[k].d[m] + par2) >> 2];
      }
    }
#pragma unroll
    for (int k = 0; k < NREC; ++k) {
      // most terms of a group and most groups of a row among the warp's octets
      const int mx = __reduce_max_sync(0xffffffffu, r[k].cnt);
      if (mx == 0) break;
      const unsigned have = __ballot_sync(0xffffffffu, r[k].cnt > 0);
      const int ng = 32 - __clz((have | have >> 8 | have >> 16 | have >> 24) & 0xffu);
      if (EXACT) {
        T p = x[k][0];
#pragma unroll
        for (int m = 1; m < kGroupMax; ++m)
          if (m < mx) p = Arith<T>::add(p, x[k][m]);
        p = r[k].cnt > 0 ? Arith<T>::mul(r[k].c, p) : T(-0.0);
#pragma unroll
        for (int t = 0; t < kOct; ++t)
          if (t < ng) s = Arith<T>::add(s, __shfl_sync(0xffffffffu, p, t, kOct));
      } else {
        // terms of the turns in FP64, four bits each: the most among the warp's octets
        uint32_t turns = 0;
        if constexpr (sizeof(T) == 8) {
          int c = max(r[k].cnt, __shfl_xor_sync(0xffffffffu, r[k].cnt, 8));
          c = max(c, __shfl_xor_sync(0xffffffffu, c, 16));
          turns = __reduce_or_sync(0xffffffffu, (uint32_t)c << (4 * l8));
        }
#pragma unroll
        for (int t = 0; t < kOct; ++t) {
          if (t >= ng) break;
          T v = s;
          if constexpr (sizeof(T) == 8) {
            const int c = (int)(turns >> (4 * t)) & 15;
#pragma unroll
            for (int m = 0; m < kGroupMax; ++m) {
              if (m >= c) break;
              v = Arith<T>::fma(r[k].c, x[k][m], v);
            }
          } else {
#pragma unroll
            for (int m = 0; m < 4; ++m) v = Arith<T>::fma(r[k].c, x[k][m], v);
            if (mx > 4) {
#pragma unroll
              for (int m = 4; m < kGroupMax; ++m) v = Arith<T>::fma(r[k].c, x[k][m], v);
            }
          }
          s = __shfl_sync(0xffffffffu, v, t, kOct);
        }
      }
    }
  }
  return s;
}

enum RowMode : int { kRowRelax = 0, kRowResidual = 1 };

// One slot per octet of block `bid`: half-sweep (out = relaxed value) or residual
// (out = f - L u) of the strip nodes. blockDim = (32, warps).
template <typename T, bool EXACT, int NREC, int MODE>
__device__ __forceinline__ void strip_rows(const LevelGeo<T>& L, const StripGeo& S, int colour, int bid,
                                           const T* u, const T* f, T* out) {
  const int lane = threadIdx.x & 31, oct = threadIdx.y * 4 + (lane >> 3);
  const int slot = bid * (blockDim.y * 4) + oct;
  int i = 0, j = 0;
  const bool on = strip_node(L, S, colour, slot, i, j);
  const int64_t at = sidx(L, i, j);
  const int cl = on ? class_of(L, i, j) : 0;
  T fv = T(0), uv = T(0);
  const T wd = MODE == kRowRelax && on ? L.cls_wd[cl] : T(0);
  const T s = octet_row<T, EXACT, NREC>(L, u + at, u + at, on, i, j, cl, [&]() {
    pdl_wait();
    if (on) {
      fv = f[at];
      if (MODE == kRowRelax) uv = u[at];
    }
  });
  if (!on || (lane & 7) != 0) return;
  const T r = Arith<T>::sub(fv, s);
  if (MODE == kRowRelax) out[at] = rnd(L, EXACT ? Arith<T>::add(uv, Arith<T>::mul(r, wd)) : Arith<T>::fma(r, wd, uv));
  else out[at] = rnd(L, r);
}

}  // namespace
}  // namespace nsmg
