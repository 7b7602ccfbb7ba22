// k right-hand sides at once (Y = alpha * A * X + beta * Y, k <= 8) over
// the same CSR tiles as the SpMV: the served form's sweep of up to eight x
// vectors per request.  X is read interleaved, row c of X holding the KP
// values x_0[c] .. x_{KP-1}[c] (KP = k rounded up to 2, 4 or 8), so a
// nonzero gathers one contiguous 8..64-byte segment, and the matrix is
// streamed once for all k vectors.
//
// One warp works on a tile alone, lane l walking exactly the nonzeros that
// lane l of the SpMV's warp walks, with the same FMAs in the same order for
// each vector and the same warp scan, so Y[:, v] equals msrep_spmv of x_v bit
// for bit.  A lane holds VW vectors: up to 32 bytes of an x row, fetched by one
// 256-bit load (FP64 with eight vectors takes two passes over the tile).  One
// vector takes the SpMV kernels themselves.
//
// What bounds it: one L1 line lookup per nonzero for the gather (16.8M of
// them take about 55 us on 152 SMs) and, above that, the instructions around
// it at 16 warps an SM (87M warp instructions on the R-MAT matrix, k = 8;
// issue slots 46% used, L1 65%).  Measured on R-MAT 2^20 / 2^24 nonzeros,
// FP32, the whole call: k = 2 / 4 / 8 110 / 132 / 208 us, against 186 / 345 /
// 539 us with row ends walked inside the nonzero loop and y written from
// there (197M warp instructions at k = 8); 2048^2 Laplacian k = 8 293 against
// 508 us.  Three things keep the instructions few:
//  * where the rows of the tile end is worked out once per tile, a lane per
//    row, into a bit string in shared memory; the nonzero loop tests one bit
//    instead of walking row pointers on a divergent path;
//  * a finished row is stored into a row buffer in shared memory, and y is
//    written a lane per row afterwards (consecutive rows of one vector in one
//    store), instead of KP scattered stores per row end;
//  * FP32 arithmetic runs on pairs of vectors (the packed f32x2
//    instructions, each half rounded as the scalar instruction).
#pragma once

#include "spmv_core.cuh"

namespace msrep {

template <class Pol>
struct SpmmArgs {
  const int32_t *row_ptr;
  const int32_t *col_idx;
  const typename Pol::V *val;
  const typename Pol::X *xt;  // [n][KP] interleaved, 32-byte aligned
  typename Pol::X *y;         // y[v * ldy + row], v < k
  int64_t ldy;
  int k;
  double alpha, beta;
  int finish;
  const int32_t *tile_row, *tile_k;
  double *head, *tail;  // [T][hs]: tile b's partial of vector v at b * hs + v
  int hs;               // head / tail stride (>= KP)
  int32_t m;
  int32_t nnz;
  unsigned comp_mode;
};

// width of the interleaved x of k vectors: k rounded up to 1, 2, 4 or 8
__host__ __device__ constexpr int spmm_width(int k) {
  return k <= 1 ? 1 : k <= 2 ? 2 : k <= 4 ? 4 : 8;
}

// vectors a lane holds at once: as many as fit a 32-byte load
template <class X, int KP>
struct KvShape {
  static constexpr int VW = KP * int(sizeof(X)) <= 32 ? KP : 32 / int(sizeof(X));
  // Resident blocks (of 4 warps) per SM asked of the register allocator: 32
  // bytes of x a lane need 128 registers, and five blocks (96, with spills) took
  // 215 us where four take 207 (R-MAT, FP32, k = 8); the narrower ones fit more.
  static constexpr int kBlocks = VW * int(sizeof(X)) == 32 ? 4 : VW * int(sizeof(X)) == 16 ? 6 : 7;
};

constexpr int kKvWarps = 4;
constexpr int kKvThreads = 32 * kKvWarps;
constexpr int kKvBitWords = 34;   // a tile of <= 1024 nonzeros in aligned groups of 8
constexpr int kKvRows = 88;       // rows of the row buffer

// Is kShort the better form of kv_tile (see there)?  Where the mean tile has
// clearly more row ends than the row buffer holds.  Rows without nonzeros end
// at none, and how many there are the call does not know: with fewer nonzeros
// than rows most are taken to be such.
inline bool kv_short_rows(int64_t m, int64_t nnz, int32_t tile) {
  return nnz >= m && m * tile > (m + nnz) * (kKvRows + 12);
}

// Shared memory of one warp.  A stored accumulator is VW sums, then (FP32)
// their VW compensations; 16 bytes of padding from 32 bytes on let a warp
// read one per lane without bank conflicts.
template <class X, int VW, bool kShort = false>
struct KvWarpSmem {
  static constexpr int kAcc = (sizeof(X) == 4 ? 2 : 1) * VW;
  static constexpr int kSlot = kAcc * int(sizeof(X)) >= 32 ? kAcc + 16 / int(sizeof(X)) : kAcc;
  // finished rows' accumulators in the order of the rows' ends
  static constexpr int kRows = !kShort                   ? kKvRows
                               : kSlot * sizeof(X) == 16 ? 256
                               : sizeof(X) == 8          ? 192
                                                         : 144;
  alignas(16) X rows[kRows][kSlot];
  alignas(16) X last[kAcc];          // the row that continues past the tile
  uint32_t end[kKvBitWords];         // bit e: a row ends with element e of the tile
  // A tile written directly (kv_tile): the rows that hold a nonzero and end in
  // it, at most 512 of a tile of 1024 items, behind a slot or two a lane.
  static constexpr bool kSpare = sizeof(X) == 4 && VW > 2;
  static constexpr int kList = kSpare ? 64 : 32;
  static_assert(!kShort || (kRows - kList) * kSlot * sizeof(X) >= 512 * sizeof(uint16_t),
                "room for the list");
  __device__ __forceinline__ uint16_t *row_of() { return reinterpret_cast<uint16_t *>(rows[kList]); }
};

// Vector j of a stored accumulator: the total that y takes, and the FP64
// partial of a split row.
template <int VW>
__device__ __forceinline__ double kv_total(const double *p, int j) { return p[j]; }
template <int VW>
__device__ __forceinline__ float kv_total(const float *p, int j) {
  return pair_total(p[j], p[VW + j]);
}
template <int VW>
__device__ __forceinline__ double kv_partial(const double *p, int j) { return p[j]; }
template <int VW>
__device__ __forceinline__ double kv_partial(const float *p, int j) {
  return pair_total_f64(p[j], p[VW + j]);
}

// ---------------------------------------------------------------------------
// VW vectors' accumulators and x values of one lane
// ---------------------------------------------------------------------------

using f32x2 = unsigned long long;  // two binary32 values, the lower lane first

__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float &a, float &b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

template <class Pol, int VW>
struct KvAcc;

// FP64: VW sums.
template <int VW>
struct KvAcc<PolF64, VW> {
  using X = double;
  double a[VW];
  struct XV {
    double d[VW];
    __device__ __forceinline__ void load(const double *p) {
      if constexpr (VW == 2) {
        const double2 t = __ldg(reinterpret_cast<const double2 *>(p));
        d[0] = t.x;
        d[1] = t.y;
      } else {
        static_assert(VW == 4, "32-byte loads");
        asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];"
            : "=d"(d[0]), "=d"(d[1]), "=d"(d[2]), "=d"(d[3])
            : "l"(p));
      }
    }
  };
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int j = 0; j < VW; ++j) a[j] = 0.0;
  }
  template <bool kComp>
  __device__ __forceinline__ void fma(double v, const XV &x) {
#pragma unroll
    for (int j = 0; j < VW; ++j) a[j] = __fma_rn(v, x.d[j], a[j]);
  }
  __device__ __forceinline__ void store(double *p) const {
#pragma unroll
    for (int j = 0; j < VW; j += 2)
      *reinterpret_cast<double2 *>(p + j) = make_double2(a[j], a[j + 1]);
  }
  __device__ __forceinline__ void load(const double *p) {
#pragma unroll
    for (int j = 0; j < VW; j += 2) {
      const double2 t = *reinterpret_cast<const double2 *>(p + j);
      a[j] = t.x;
      a[j + 1] = t.y;
    }
  }
  __device__ __forceinline__ void totals(double (&t)[VW]) const {
#pragma unroll
    for (int j = 0; j < VW; ++j) t[j] = a[j];
  }
  // *this = u + *this
  __device__ __forceinline__ void carry_in(const KvAcc &u) {
#pragma unroll
    for (int j = 0; j < VW; ++j) a[j] = __dadd_rn(u.a[j], a[j]);
  }
  __device__ __forceinline__ KvAcc shfl_up(int o) const {
    KvAcc r;
#pragma unroll
    for (int j = 0; j < VW; ++j) r.a[j] = __shfl_up_sync(0xffffffffu, a[j], o);
    return r;
  }
};

// FP32 sums and their compensation, two vectors to a register pair.  The
// compensated update is PolF32::fma's on each half; the product is formed
// negated (n = -v x, exactly the negative of v x rounded), which turns its
// uses into subtractions and leaves every rounding as it was.
template <class VT, int VW>
struct KvAcc<PolF32<VT>, VW> {
  using X = float;
  static constexpr int N2 = VW / 2;
  f32x2 s[N2], c[N2];
  struct XV {
    f32x2 d[N2];
    __device__ __forceinline__ void load(const float *p) {
      if constexpr (VW == 2) {
        asm("ld.global.nc.b64 %0, [%1];" : "=l"(d[0]) : "l"(p));
      } else if constexpr (VW == 4) {
        asm("ld.global.nc.v2.b64 {%0, %1}, [%2];" : "=l"(d[0]), "=l"(d[1]) : "l"(p));
      } else {
        static_assert(VW == 8, "32-byte loads");
        asm("ld.global.nc.v4.b64 {%0, %1, %2, %3}, [%4];"
            : "=l"(d[0]), "=l"(d[1]), "=l"(d[2]), "=l"(d[3])
            : "l"(p));
      }
    }
  };
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int j = 0; j < N2; ++j) s[j] = c[j] = 0;
  }
  template <bool kComp>
  __device__ __forceinline__ void fma(float v, const XV &x) {
    const f32x2 vv = pack2(v, v);
    if (kComp) {
      const f32x2 nv = pack2(-v, -v);
#pragma unroll
      for (int j = 0; j < N2; ++j) {
        const f32x2 n = mul2(nv, x.d[j]);            // -p
        const f32x2 ep = fma2(vv, x.d[j], n);        // v x - p
        const f32x2 t = sub2(s[j], n);               // s + p
        const f32x2 bb = sub2(t, s[j]), aa = sub2(t, bb);
        const f32x2 es = sub2(sub2(s[j], aa), add2(n, bb));
        s[j] = t;
        c[j] = add2(c[j], add2(ep, es));
      }
    } else {
#pragma unroll
      for (int j = 0; j < N2; ++j) s[j] = fma2(vv, x.d[j], s[j]);
    }
  }
  __device__ __forceinline__ void store(float *p) const {
    ulonglong2 *q = reinterpret_cast<ulonglong2 *>(p);  // 16-byte accesses
    if constexpr (N2 == 1) {
      q[0] = make_ulonglong2(s[0], c[0]);
    } else {
#pragma unroll
      for (int j = 0; j < N2 / 2; ++j) {
        q[j] = make_ulonglong2(s[2 * j], s[2 * j + 1]);
        q[N2 / 2 + j] = make_ulonglong2(c[2 * j], c[2 * j + 1]);
      }
    }
  }
  __device__ __forceinline__ void load(const float *p) {
    const ulonglong2 *q = reinterpret_cast<const ulonglong2 *>(p);
    if constexpr (N2 == 1) {
      const ulonglong2 t = q[0];
      s[0] = t.x;
      c[0] = t.y;
    } else {
#pragma unroll
      for (int j = 0; j < N2 / 2; ++j) {
        const ulonglong2 t = q[j], w = q[N2 / 2 + j];
        s[2 * j] = t.x;
        s[2 * j + 1] = t.y;
        c[2 * j] = w.x;
        c[2 * j + 1] = w.y;
      }
    }
  }
  __device__ __forceinline__ void totals(float (&t)[VW]) const {
#pragma unroll
    for (int j = 0; j < N2; ++j) {
      float s0, s1, c0, c1;
      unpack2(s[j], s0, s1);
      unpack2(c[j], c0, c1);
      t[2 * j] = pair_total(s0, c0);
      t[2 * j + 1] = pair_total(s1, c1);
    }
  }
  __device__ __forceinline__ void carry_in(const KvAcc &u) {
#pragma unroll
    for (int j = 0; j < N2; ++j) {
      const f32x2 t = add2(u.s[j], s[j]);
      const f32x2 bb = sub2(t, u.s[j]), aa = sub2(t, bb);
      const f32x2 e = add2(sub2(u.s[j], aa), sub2(s[j], bb));
      s[j] = t;
      c[j] = add2(add2(u.c[j], c[j]), e);
    }
  }
  __device__ __forceinline__ KvAcc shfl_up(int o) const {
    KvAcc r;
#pragma unroll
    for (int j = 0; j < N2; ++j) {
      r.s[j] = __shfl_up_sync(0xffffffffu, s[j], o);
      r.c[j] = __shfl_up_sync(0xffffffffu, c[j], o);
    }
    return r;
  }
};

// Four consecutive elements at h4 (a multiple of 4): one vector load, or
// element-wise at the array's end.  Loads of 16 bytes and less go through L1,
// which serves the other half of their 32-byte sector to the next load
// (bypassing it read the halves from L2 and DRAM again: Laplacian FP32 k = 8
// 301 us against 290).
__device__ __forceinline__ void ld4(const int32_t *p, int32_t (&r)[4]) {
  asm("ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
      : "l"(p));
}
__device__ __forceinline__ void ld4(const float *p, float (&r)[4]) {
  asm("ld.global.nc.v4.f32 {%0, %1, %2, %3}, [%4];"
      : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3])
      : "l"(p));
}
__device__ __forceinline__ void ld4(const double *p, double (&r)[4]) {
  asm("ld.global.nc.L1::no_allocate.v4.f64 {%0, %1, %2, %3}, [%4];"
      : "=d"(r[0]), "=d"(r[1]), "=d"(r[2]), "=d"(r[3])
      : "l"(p));
}
__device__ __forceinline__ void ld4(const bf16_t *p, float (&r)[4]) {
  uint32_t w[2];
  asm("ld.global.nc.v2.b32 {%0, %1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "l"(p));
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    r[2 * i] = __uint_as_float(w[i] << 16);
    r[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
}
template <class T, class U>
__device__ __forceinline__ void load4(const T *arr, int32_t h4, int32_t nnz, U (&out)[4]) {
  if (h4 < (nnz & ~3)) {
    ld4(arr + h4, out);
  } else {
#pragma unroll
    for (int u = 0; u < 4; ++u) out[u] = (u < nnz - h4) ? U(ld_stream(arr + h4 + u)) : U(0);
  }
}

// Vectors [vb, ve) (a multiple of VW) of tile b by one warp.  kCopy: alpha = 1,
// beta = 0 known at compile time; kComp: compensated sums (low-precision
// form).
//
// A tile with more row ends than the row buffer holds is walked once for each
// kKvRows of them.  kShort: the buffer is larger (the loop then has less L1 for
// x), and a tile beyond it is walked once too, its rows written from the nonzero
// loop, all but each lane's first, which waits for its carry in the lane's slot
// (the wider FP32 layouts through another slot of the lane: from registers the
// stores spilled).  The loop pays a few percent for that choice at each row
// end, so kShort is taken where the mean tile needs it (kv_short_rows).
// Measured without -> with, tile 512: rows of three nonzeros FP64 k = 4 67 -> 47
// us, FP32 k = 2 34 -> 24; of two 80 -> 59 and 37 -> 27; of one 146 -> 116 and 58
// -> 40; Laplacian 2048^2 with tile 1024, FP64 k = 4, 437 -> 283.
template <class Pol, int KP, bool kCopy, bool kComp, bool kShort = false>
__device__ __forceinline__ void kv_tile(
    const SpmmArgs<Pol> &a, int b, int32_t nnz,
    KvWarpSmem<typename Pol::X, KvShape<typename Pol::X, KP>::VW, kShort> &sm, int vb = 0,
    int ve = KP) {
  using X = typename Pol::X;
  using LV = typename LoadT<typename Pol::V>::type;
  constexpr int VW = KvShape<X, KP>::VW;
  using Acc = KvAcc<Pol, VW>;
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int fin = kCopy ? int(kFinishCopy) : a.finish;
  const int32_t r0 = __ldg(a.tile_row + b), k0 = __ldg(a.tile_k + b);
  const int32_t r1 = __ldg(a.tile_row + b + 1), k1 = __ldg(a.tile_k + b + 1);
  const int nrows = r1 - r0;
  const int32_t base = k0 & ~7;  // element e of the tile is nonzero base + e
  const LaneRange lr = lane_range(k0, k1, lane);
  const int h_lo = static_cast<int>(lr.glo) * 2, h_hi = static_cast<int>(lr.ghi) * 2;

  // the lane's first nonzeros, in flight while the rows are worked out
  int32_t cn[4];
  LV vn[4];
  if (h_lo < h_hi) {
    load4(a.col_idx, h_lo * 4, nnz, cn);
    load4(a.val, h_lo * 4, nnz, vn);
  }

  // --- the tile's rows: row i (a lane each) ends in the tile for i < nrows;
  // row nrows, if the matrix has it, continues past it
  for (int i = lane; i < kKvBitWords; i += 32) sm.end[i] = 0;
  __syncwarp();
  bool flag = false, has0 = false;  // row 0: started earlier; holds a nonzero of the tile
  int32_t last_end = 0;             // row_ptr[r1]
  int ends = 0;                     // rows that hold a nonzero of the tile and end in it
  for (int i0 = 0; i0 <= nrows; i0 += 32) {
    const int i = i0 + lane;
    const bool valid = i <= nrows;
    const int32_t st = valid ? __ldg(a.row_ptr + r0 + i) : 0;
    const int32_t en = valid && r0 + i < a.m ? __ldg(a.row_ptr + r0 + i + 1) : k1;
    const int32_t from = max(st, k0), to = min(en, k1);
    const bool holds = valid && to > from;
    const bool done = holds && i < nrows;
    const unsigned dm = __ballot_sync(full, done);
    if (i0 == 0) {
      flag = __shfl_sync(full, st, 0) < k0;
      has0 = (dm & 1u) != 0;
    }
    if (done) atomicOr(sm.end + ((to - 1 - base) >> 5), 1u << ((to - 1 - base) & 31));
    if (nrows - i0 < 32) last_end = __shfl_sync(full, st, nrows - i0);
    ends += __popc(dm);
  }
  __syncwarp();

  // rank of the lane's first row end among the tile's
  const int gA = k0 >> 3;
  int rank0;
  {
    int cnt = 0;
    for (int g = static_cast<int>(lr.glo) - gA; g < static_cast<int>(lr.ghi) - gA; ++g)
      cnt += __popc((sm.end[g >> 2] >> ((g & 3) * 8)) & 0xffu);
    int inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(full, inc, o);
      if (lane >= o) inc += t;
    }
    rank0 = inc - cnt;
  }

  using Smem = KvWarpSmem<X, VW, kShort>;
  constexpr int kRows = Smem::kRows;
  const bool direct = kShort && ends > kRows;
  uint16_t *row_of = sm.row_of();
  if (direct) {
    int before = 0;
    for (int i0 = 0; i0 < nrows; i0 += 32) {
      const int i = i0 + lane;
      const int32_t st = i < nrows ? __ldg(a.row_ptr + r0 + i) : 0;
      const int32_t en = i < nrows ? __ldg(a.row_ptr + r0 + i + 1) : 0;
      const bool holds = i < nrows && en > max(st, k0);
      const unsigned dm = __ballot_sync(full, holds);
      if (holds) row_of[before + __popc(dm & ((1u << lane) - 1u))] = static_cast<uint16_t>(i);
      before += __popc(dm);
    }
    __syncwarp();
  }
  auto write_row = [&](int v0, int32_t i, const Acc &tot, X *p) {
    X *yp = a.y + v0 * a.ldy + r0 + i;
    if constexpr (Smem::kSpare) {
      tot.store(p);
#pragma unroll 1
      for (int j = 0; j < VW && v0 + j < a.k; ++j, yp += a.ldy)
        *yp = finish_total(kv_total<VW>(p, j), fin, a.alpha, a.beta, yp);
    } else {
      X t[VW];
      tot.totals(t);
#pragma unroll
      for (int j = 0; j < VW; ++j)
        if (v0 + j < a.k)
          yp[j * a.ldy] = finish_total(t[j], fin, a.alpha, a.beta, yp + j * a.ldy);
    }
  };

  // rows [w0, w0 + kRows) of the row ends (all of them if direct), vectors
  // [v0, v0 + VW)
  for (int w0 = 0, v0 = vb; v0 < ve;) {
    // --- the lane's nonzeros
    const X *xb = a.xt + v0;
    Acc acc;
    acc.zero();
    // slot of the lane's next row end: its rank in the window, or, written
    // directly, `lane` and then none (its ends counted in steps of kPast)
    constexpr int kPast = 1 << 20;
    const int slot0 = direct ? lane : rank0 - w0, step = direct ? kPast : 1;
    int slot = slot0;
    if ((v0 > vb || w0 > 0) && h_lo < h_hi) {
      load4(a.col_idx, h_lo * 4, nnz, cn);
      load4(a.val, h_lo * 4, nnz, vn);
    }
    for (int h = h_lo; h < h_hi; ++h) {
      const int32_t h4 = h * 4;
      const int e = h4 - base;
      // which of the four are the tile's, and end a row
      const int lo = max(k0 - h4, 0), hi = min(k1 - h4, 4);
      const uint32_t in = hi > lo ? (0xfu >> (4 - (hi - lo))) << lo : 0u;
      const uint32_t eb = sm.end[e >> 5] >> (e & 31);
      LV v[4];
      typename Acc::XV x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        v[u] = vn[u];
        if ((in >> u) & 1u) x[u].load(xb + int64_t(cn[u]) * KP);
      }
      if (h + 1 < h_hi) {
        load4(a.col_idx, h4 + 4, nnz, cn);
        load4(a.val, h4 + 4, nnz, vn);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if ((in >> u) & 1u) acc.template fma<kComp>(v[u], x[u]);
        if ((eb >> u) & 1u) {  // a row ends here
          if constexpr (kShort) {
            if (slot < kRows)
              acc.store(sm.rows[slot]);
            else
              write_row(v0, row_of[rank0 + slot / kPast], acc, sm.rows[32 + lane]);
          } else {
            if (static_cast<unsigned>(slot) < unsigned(kRows)) acc.store(sm.rows[slot]);
          }
          slot += step;
          acc.zero();
        }
      }
    }

    // --- rows split between lanes: warp_seg_scan's doubling, for all VW
    const bool emitted = slot != slot0;
    bool f = emitted;
#pragma unroll 1
    for (int o = 1; o < 32; o <<= 1) {
      if (__all_sync(full, f || lane < o)) break;
      const Acc u = acc.shfl_up(o);
      const int fu = __shfl_up_sync(full, int(f), o);
      if (lane >= o) {
        if (!f) acc.carry_in(u);
        f = f || fu;
      }
    }
    Acc ex = acc.shfl_up(1);
    if (lane == 0) ex.zero();
    if (emitted && static_cast<unsigned>(slot0) < unsigned(kRows)) {
      Acc tot;
      tot.load(sm.rows[slot0]);
      tot.carry_in(ex);
      if (direct && !(rank0 == 0 && has0 && flag))
        write_row(v0, row_of[rank0], tot, sm.rows[lane]);
      else
        tot.store(sm.rows[slot0]);
    }
    const unsigned em = kShort && direct ? __ballot_sync(full, emitted) : 1u;
    if (lane == 31) acc.store(sm.last);
    __syncwarp();

    // --- partials of the rows split between tiles, widened to FP64 a lane
    // per vector (an FP64 warp instruction costs its full slot of the FP64
    // pipe however few lanes it has): lanes 0.. the first row's, lanes 16..
    // the last row's.  A first row that ended where the tile starts adds 0.
    if (w0 == 0) {
      const int j = lane & 15;
      const X *src = lane < 16 ? sm.rows[__ffs(em) - 1] : sm.last;
      double *dst = nullptr;
      if (lane < 16) {
        if (flag && nrows > 0) dst = a.head;
      } else if (nrows == 0) {
        if (flag)
          dst = a.head;
        else if (k1 > k0)
          dst = a.tail;
      } else if (k1 > last_end) {
        dst = a.tail;
      }
      if (j < VW && dst)
        dst[int64_t(b) * a.hs + v0 + j] = lane < 16 && !has0 ? 0.0 : kv_partial<VW>(src, j);
    }

    // --- y, a lane per row (a split first row is the fix-up's)
    int done = -w0;
    for (int i0 = 0; i0 < nrows; i0 += 32) {
      const int i = i0 + lane;
      const bool valid = i < nrows;
      const int32_t st = valid ? __ldg(a.row_ptr + r0 + i) : 0;
      const int32_t en = valid ? __ldg(a.row_ptr + r0 + i + 1) : 0;
      const bool holds = valid && en > max(st, k0);
      const unsigned dm = __ballot_sync(full, holds);
      const int rk = done + __popc(dm & ((1u << lane) - 1u));
      done += __popc(dm);
      if (valid && !(i == 0 && flag) &&
          (holds ? !direct && static_cast<unsigned>(rk) < unsigned(kRows) : w0 == 0)) {
        X t[VW];
        if (holds) {
          Acc tot;
          tot.load(sm.rows[rk]);
          tot.totals(t);
        } else {
#pragma unroll
          for (int j = 0; j < VW; ++j) t[j] = X(0);
        }
        X *yp = a.y + v0 * a.ldy + r0 + i;
#pragma unroll
        for (int j = 0; j < VW; ++j)
          if (v0 + j < a.k)
            yp[j * a.ldy] = finish_total(t[j], fin, a.alpha, a.beta, yp + j * a.ldy);
      }
    }
    __syncwarp();
    w0 += kRows;
    if (direct || w0 >= ends) {
      w0 = 0;
      v0 += VW;
    }
  }
}

// fixup_tile for vector j of tile b: partials at head/tail[tile * hs + j];
// the sums are formed in the same order as fixup_tile's.
template <class X, class View>
__device__ __forceinline__ void fixup_tile_k(const View &v, int T, int b, int j, int hs,
                                             const double *head, const double *tail, X *y,
                                             int64_t ldy, double alpha, double beta) {
  int32_t r;
  if (!fixup_run_start(v, T, b, r)) return;
  double s = tail[int64_t(b - 1) * hs + j];
  for (int j0 = b; fixup_chunk(v, T, j0, r, head + j, s, hs) == 8; j0 += 8) {
  }
  fixup_write(y + j * ldy, r, s, alpha, beta);
}

}  // namespace msrep
