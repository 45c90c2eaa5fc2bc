// P2 velocity stencil kernels (see p2stencil.h).
#include <math_constants.h>

#include <cmath>

#include "p2slots.h"

namespace chnss {
namespace {

constexpr int TPB = 256;

constexpr SlotTable kSlots = slot_table();

__constant__ SlotTable c_slots = kSlots;

template <typename T> struct V2;
template <> struct V2<float> { using type = float2; };
template <> struct V2<double> { using type = double2; };
template <typename T>
__device__ __forceinline__ typename V2<T>::type mk(T x, T y) {
  typename V2<T>::type v;
  v.x = x;
  v.y = y;
  return v;
}
__device__ __forceinline__ float2 load_pair(const float *p) { return __ldg(reinterpret_cast<const float2 *>(p)); }
__device__ __forceinline__ float2 load_pair(const __nv_bfloat16 *p) {
  return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p));
}
template <typename T> __device__ __forceinline__ T from_double(double x) { return (T)x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_double<__nv_bfloat16>(double x) { return __double2bfloat16(x); }

template <typename T>
struct Coef {
  T c[2 * (kP2Slots + kP2TopSlots)];
};
struct Args {
  const void *b, *w, *dinv;
  const double *coef, *scale;
};

// what the sweep's result for one node needs beside its row sums
template <typename T>
struct NodeIn {
  using P = typename V2<T>::type;
  P b, d, w;
  T c0 = 0, c1 = 0, c2 = 0;
  bool has_w = false;
  __device__ __forceinline__ void load(int mode, int start, long r, T sc, const Args &a, const T *out) {
    if (mode == SPMV_PLAIN) return;
    if (mode == SPMV_ADD) {
      b = reinterpret_cast<const P *>(out)[r];
      return;
    }
    b = static_cast<const P *>(a.b)[r];
    if (mode == SPMV_RES) return;
    d = static_cast<const P *>(a.dinv)[r];
    c0 = (T)a.coef[0];
    c1 = (T)a.coef[1];
    c2 = (T)a.coef[2];
    has_w = start == P2_SECOND || a.w != nullptr;
    if (start == P2_SECOND) w = mk<T>(sc * d.x * b.x, sc * d.y * b.y);
    else if (a.w) w = static_cast<const P *>(a.w)[r];
  }
  __device__ __forceinline__ P result(int mode, T s0, T s1, P ui) const {
    if (mode == SPMV_PLAIN) return mk<T>(s0, s1);
    if (mode == SPMV_RES) return mk<T>(b.x - s0, b.y - s1);
    if (mode == SPMV_ADD) return mk<T>(b.x + s0, b.y + s1);
    return mk<T>(cheb_step<T>(c0, c1, c2, ui.x, d.x, b.x, s0, has_w, w.x),
                 cheb_step<T>(c0, c1, c2, ui.y, d.y, b.y, s1, has_w, w.y));
  }
};

// Fine levels: one cell (its four nodes) a thread.  The 19 neighbours of the
// vertex are all the cell reads, every value load is one coalesced access of
// two values, and all loads are independent.
template <typename T, typename VT, bool OPEN>
__global__ void __launch_bounds__(kSellMaxBlock, 2) k_p2_spmv(int n, long ld, const VT *__restrict__ val,
                                                           const T *__restrict__ u, T *out, int mode, int start,
                                                           Args a, const __grid_constant__ Coef<T> cf) {
  using P = typename V2<T>::type;
  const int cell = blockIdx.x * blockDim.x + threadIdx.x;
  const int w1 = n + 1, m = 2 * n + 1;
  if (cell >= w1 * w1) return;
  const int j = cell / w1, i = cell - j * w1;
  P *o2 = reinterpret_cast<P *>(out);
  const T sc = start != P2_PLAIN ? (T)*a.scale : (T)0;
  auto iterate = [&](long r) {
    if (start == P2_FIRST) {
      const P d = static_cast<const P *>(a.dinv)[r], b = static_cast<const P *>(a.b)[r];
      return mk<T>(sc * d.x * b.x, sc * d.y * b.y);
    }
    return reinterpret_cast<const P *>(u)[r];
  };
  const long r0 = (long)(2 * j) * m + 2 * i;
  constexpr SlotTable st = slot_table();
  P x[19];
#pragma unroll
  for (int k = 0; k < 19; ++k) {
    const int I = 2 * i + st.di[k], J = 2 * j + st.dj[k];
    x[k] = prescribed(I, J, m, OPEN) ? mk<T>(0, 0) : iterate(r0 + st.dj[k] * m + st.di[k]);
  }
  auto row = [&](auto tyc) {
    constexpr int TY = decltype(tyc)::value;
    constexpr int oi = TY & 1, oj = TY >> 1, base = slot_base(TY), cnt = slot_count(TY);
    const int I = 2 * i + oi, J = 2 * j + oj;
    if (I >= m || J >= m) return;
    const long r = r0 + oj * m + oi;
    T s0 = 0, s1 = 0;
    P ui;
    if (prescribed(I, J, m, OPEN)) {   // identity row
      ui = iterate(r);
      s0 = ui.x;
      s1 = ui.y;
    } else {
      const int top = OPEN && TY < 2 && j == n ? kP2Slots : 0;
#pragma unroll
      for (int k = 0; k < cnt; ++k) {
        const int di = oi + st.di[base + k], dj = oj + st.dj[base + k];
        int xi = 0;
#pragma unroll
        for (int q = 0; q < 19; ++q)
          if (st.di[q] == di && st.dj[q] == dj) xi = q;
        const P v = load_pair(val + 2 * ((base + k) * ld + cell));
        const P xk = x[xi];
        if (di == oi && dj == oj) ui = xk;
        s0 = fma_of(cf.c[2 * (top + base + k)], xk.y, fma_of((T)v.x, xk.x, s0));
        s1 = fma_of((T)v.y, xk.y, fma_of(cf.c[2 * (top + base + k) + 1], xk.x, s1));
      }
    }
    NodeIn<T> in;
    in.load(mode, start, r, sc, a, out);
    o2[r] = in.result(mode, s0, s1, ui);
  };
  row(std::integral_constant<int, 0>());
  row(std::integral_constant<int, 1>());
  row(std::integral_constant<int, 2>());
  row(std::integral_constant<int, 3>());
}

// Coarse levels (fewer rows than one wave of threads), FP32: 32 cells of one
// node type (blockIdx.y) a block and KS warps a row, warp q summing entries q,
// q + KS, ..., the partial sums added in warp order, so that a thread has at
// most three (KS = 8) dependent blocks.  Latency bound.
template <typename VT, int KS, bool OPEN>
__global__ void __launch_bounds__(32 * KS) k_p2_split(int n, long ld, const VT *__restrict__ val,
                                                      const float *__restrict__ u, float *out, int mode, int start,
                                                      Args a, const float *__restrict__ tab) {
  using T = float;
  using P = float2;
  __shared__ P part[KS][32];
  const int lane = threadIdx.x & 31, q = threadIdx.x >> 5, ty = blockIdx.y;
  const int cell = blockIdx.x * 32 + lane, w1 = n + 1, m = 2 * n + 1;
  const int j = cell / w1, i = cell - j * w1;
  const int I = 2 * i + (ty & 1), J = 2 * j + (ty >> 1);
  const bool live = cell < w1 * w1 && I < m && J < m;
  const P *u2 = reinterpret_cast<const P *>(u);
  const T sc = start != P2_PLAIN ? (T)*a.scale : (T)0;
  auto iterate = [&](long r) {
    if (start == P2_FIRST) {
      const P d = static_cast<const P *>(a.dinv)[r], b = static_cast<const P *>(a.b)[r];
      return mk<T>(sc * d.x * b.x, sc * d.y * b.y);
    }
    return u2[r];
  };
  const long r = (long)J * m + I;
  NodeIn<T> in;
  P ui = mk<T>(0, 0);
  if (q == 0 && live) {   // the result's operands, requested with the matrix
    ui = iterate(r);
    in.load(mode, start, r, sc, a, out);
  }
  const bool fixed = live && prescribed(I, J, m, OPEN);
  T s0 = 0, s1 = 0;
  if (live && !fixed) {
    const int base = slot_base(ty), cnt = slot_count(ty), top = OPEN && J == m - 1 ? kP2Slots : 0;
    constexpr int most = (19 + KS - 1) / KS;
#pragma unroll
    for (int t = 0; t < most; ++t) {
      const int k = base + q + KS * t;
      if (k < base + cnt) {
        const int di = c_slots.di[k], dj = c_slots.dj[k];
        const float2 v = load_pair(val + 2 * (k * ld + cell)), c = load_pair(tab + 2 * (top + k));
        const float2 x = prescribed(I + di, J + dj, m, OPEN) ? make_float2(0.f, 0.f) : iterate(r + dj * m + di);
        s0 = fmaf(c.x, x.y, fmaf(v.x, x.x, s0));
        s1 = fmaf(v.y, x.y, fmaf(c.y, x.x, s1));
      }
    }
  }
  part[q][lane] = mk<T>(s0, s1);
  __syncthreads();
  if (q != 0 || !live) return;
  if (fixed) {   // identity row
    s0 = ui.x;
    s1 = ui.y;
  } else {
#pragma unroll
    for (int p = 1; p < KS; ++p) {
      s0 += part[p][lane].x;
      s1 += part[p][lane].y;
    }
  }
  reinterpret_cast<P *>(out)[r] = in.result(mode, s0, s1, ui);
}

// diagonal values of every block, slot by slot; entry k of a row is its k-th
// CSR entry (rows with prescribed velocity have none, an open top's rows lack
// the last ones)
template <typename VT>
__global__ void k_p2_values(int n, int open, long ld, const int *__restrict__ rowptr, const double *__restrict__ A,
                            VT *__restrict__ out) {
  const int cell = blockIdx.x * TPB + threadIdx.x, k = blockIdx.y;
  if (cell >= ld) return;
  const int w1 = n + 1, m = 2 * n + 1, j = cell / w1, i = cell - j * w1;
  const int ty = k < 19 ? 0 : (k - 10) / 9;
  const int I = 2 * i + (ty & 1), J = 2 * j + (ty >> 1);
  const int CI = I + c_slots.di[k], CJ = J + c_slots.dj[k];
  double2 v = make_double2(0.0, 0.0);
  if (cell < w1 * w1 && !prescribed(I, J, m, open) && !prescribed(CI, CJ, m, open)) {
    const int q = rowptr[J * m + I] + k - slot_base(ty);
    v = make_double2(A[4L * q], A[4L * q + 3]);
  }
  const long e = 2 * (k * ld + cell);
  out[e] = from_double<VT>(v.x);
  out[e + 1] = from_double<VT>(v.y);
}

// the off-diagonal entries of the rows nearest the centre, then a check of
// every row against them (bad[0] counts the blocks that differ)
__global__ void k_p2_table(int n, int open, const int *__restrict__ rowptr, const double *__restrict__ A,
                           double *__restrict__ c) {
  const int k = threadIdx.x;
  if (k >= kP2Slots + kP2TopSlots) return;
  const int m = 2 * n + 1, s = k < kP2Slots ? k : k - kP2Slots;
  const int ty = s < 19 ? 0 : (s - 10) / 9;
  c[2 * k] = c[2 * k + 1] = CUDART_NAN;   // no such coupling
  const int I = 2 * (n / 2) + (ty & 1), J = k < kP2Slots ? 2 * (n / 2) + (ty >> 1) : 2 * n;
  if (prescribed(I, J, m, open) || J + c_slots.dj[s] >= m) return;
  // a coupling to a prescribed node holds zeros: take it from another row of the type
  int ci = I, cj = J;
  for (int t = 0; t < n && prescribed(ci + c_slots.di[s], cj + c_slots.dj[s], m, open); ++t) {
    ci = 2 * t + (ty & 1);
    for (int v = 0; v < n; ++v) {
      cj = k < kP2Slots ? 2 * v + (ty >> 1) : 2 * n;
      if (!prescribed(ci, cj, m, open) && !prescribed(ci + c_slots.di[s], cj + c_slots.dj[s], m, open)) break;
    }
  }
  if (prescribed(ci, cj, m, open) || prescribed(ci + c_slots.di[s], cj + c_slots.dj[s], m, open)) return;
  const int q = rowptr[cj * m + ci] + s - slot_base(ty);
  c[2 * k] = A[4L * q + 1];
  c[2 * k + 1] = A[4L * q + 2];
}
__global__ void k_p2_check(int n, int open, const int *__restrict__ rowptr, const int *__restrict__ col,
                           const double *__restrict__ A, const double *__restrict__ c, int *bad) {
  const int r = blockIdx.x * TPB + threadIdx.x, m = 2 * n + 1;
  if (r >= m * m) return;
  const int I = r % m, J = r / m, ty = type_of(I, J);
  bool same = true;
  if (prescribed(I, J, m, open)) {
    for (int q = rowptr[r]; q < rowptr[r + 1]; ++q) {
      const double d = col[q] == r ? 1.0 : 0.0;
      same = same && A[4L * q] == d && A[4L * q + 3] == d && A[4L * q + 1] == 0.0 && A[4L * q + 2] == 0.0;
    }
  } else {
    const int top = J == m - 1 ? kP2Slots : 0;
    const int len = rowptr[r + 1] - rowptr[r];
    same = len == (top ? (ty == 0 ? 12 : 6) : slot_count(ty));
    for (int k = 0; same && k < len; ++k) {
      const int s = slot_base(ty) + k, q = rowptr[r] + k;
      const int CI = I + c_slots.di[s], CJ = J + c_slots.dj[s];
      same = col[q] == CJ * m + CI;
      const bool off = prescribed(CI, CJ, m, open);
      same = same && A[4L * q + 1] == (off ? 0.0 : c[2 * (top + s)]) && A[4L * q + 2] == (off ? 0.0 : c[2 * (top + s) + 1]);
      if (off) same = same && A[4L * q] == 0.0 && A[4L * q + 3] == 0.0;
    }
  }
  if (!same) atomicAdd(bad, 1);
}

}  // namespace

constexpr int kCount = 2 * (kP2Slots + kP2TopSlots);

bool p2_applies(const P2Table &t, size_t value_size) {
  return t.ok && value_size < 8;
}

P2Table p2_table(Arena &keep, const Level &L, int open_top, const double *A, cudaStream_t s) {
  P2Table t;
  Arena ar;
  double *c = ar.alloc<double>(2 * (kP2Slots + kP2TopSlots));
  int *bad = ar.alloc<int>(1);
  CHNSS_CK(cudaMemsetAsync(bad, 0, sizeof(int), s));
  k_p2_table<<<1, 128, 0, s>>>(L.n, open_top, L.p2.rowptr, A, c);
  CHNSS_LAUNCH_CK();
  k_p2_check<<<(L.N2 + TPB - 1) / TPB, TPB, 0, s>>>(L.n, open_top, L.p2.rowptr, L.p2.col, A, c, bad);
  CHNSS_LAUNCH_CK();
  int hbad = 0;
  CHNSS_CK(cudaMemcpyAsync(t.c, c, sizeof(t.c), cudaMemcpyDeviceToHost, s));
  CHNSS_CK(cudaMemcpyAsync(&hbad, bad, sizeof(int), cudaMemcpyDeviceToHost, s));
  CHNSS_CK(cudaStreamSynchronize(s));
  t.ok = hbad == 0;
  for (int k = 0; k < kP2Slots + kP2TopSlots; ++k) {
    t.seen[k] = !std::isnan(t.c[2 * k]);
    if (!t.seen[k]) t.c[2 * k] = t.c[2 * k + 1] = 0.0;
  }
  std::vector<float> f(t.c, t.c + kCount), h(kCount);
  for (int k = 0; k < kCount; ++k) h[k] = __bfloat162float(__double2bfloat16(t.c[k]));
  t.d32 = keep.upload(f);
  t.d16 = keep.upload(h);
  return t;
}

template <typename VT>
void p2_values(const Level &L, int open_top, const double *A, VT *out, cudaStream_t s) {
  const long ld = p2_ld(L.n);
  const dim3 g((unsigned)((ld + TPB - 1) / TPB), kP2Slots);
  k_p2_values<VT><<<g, TPB, 0, s>>>(L.n, open_top, ld, L.p2.rowptr, A, out);
  CHNSS_LAUNCH_CK();
}
template void p2_values<float>(const Level &, int, const double *, float *, cudaStream_t);
template void p2_values<__nv_bfloat16>(const Level &, int, const double *, __nv_bfloat16 *, cudaStream_t);

namespace {
inline bool aligned(const void *p, size_t bytes) { return (reinterpret_cast<uintptr_t>(p) % bytes) == 0; }

template <typename T, typename VT, bool OPEN>
void launch(const Level &L, int ks, const VT *val, const T *u, T *out, SpmvMode mode, P2Start start, const Args &a,
            const Coef<T> &cf, const T *tab, cudaStream_t s) {
  const int cells = (L.n + 1) * (L.n + 1), tpb = L.p2.sell.block, nb = (cells + tpb - 1) / tpb;
  const long ld = p2_ld(L.n);
  const dim3 gs((unsigned)((cells + 31) / 32), 4);
  switch (ks) {
    case 2: k_p2_split<VT, 2, OPEN><<<gs, 64, 0, s>>>(L.n, ld, val, u, out, mode, start, a, tab); return;
    case 4: k_p2_split<VT, 4, OPEN><<<gs, 128, 0, s>>>(L.n, ld, val, u, out, mode, start, a, tab); return;
    case 8: k_p2_split<VT, 8, OPEN><<<gs, 256, 0, s>>>(L.n, ld, val, u, out, mode, start, a, tab); return;
  }
  k_p2_spmv<T, VT, OPEN><<<nb, tpb, 0, s>>>(L.n, ld, val, u, out, mode, start, a, cf);
}
// the table in the precision of the values, on the device and (rounded the
// same way) as kernel arguments
const float *device_table(const P2Table &t, const float *) { return t.d32; }
const float *device_table(const P2Table &t, const __nv_bfloat16 *) { return t.d16; }
float rounded(double x, const float *) { return (float)x; }
float rounded(double x, const __nv_bfloat16 *) { return __bfloat162float(__double2bfloat16(x)); }
}  // namespace

namespace {
__device__ const P2Transfers g_transfers = p2_transfers();

// Grid transfers of the velocity with their columns and weights computed:
// the SELL form streamed 8 bytes an entry (10.7 entries a fine node, both
// ways) beside the vectors.  Entries in CSR order, so results are the same
// bit for bit.  One thread a coarse node of the type (blockIdx.z the parity
// of I, so that a warp's nodes share a type).
template <typename T, bool OPEN>
__global__ void k_p2_restrict(int nc, const T *__restrict__ r, T *__restrict__ b) {
  using P = typename V2<T>::type;
  constexpr int open = OPEN ? 1 : 0;
  const int mc = 2 * nc + 1, m = 4 * nc + 1;
  const int I = 2 * (blockIdx.x * blockDim.x + threadIdx.x) + blockIdx.z, J = blockIdx.y;
  if (I >= mc) return;
  T a0 = 0, a1 = 0;
  if (!prescribed(I, J, mc, open)) {
    const P *r2 = reinterpret_cast<const P *>(r) + (long)(2 * J) * m + 2 * I;
    auto sum = [&](auto tyc) {
      constexpr P2Transfers t = p2_transfers();
      constexpr int ty = decltype(tyc)::value, cnt = t.rn[ty];
#pragma unroll
      for (int k = 0; k < cnt; ++k) {
        P x = mk<T>(0, 0);
        if (!OPEN || 2 * J + t.rj[ty][k] < m) x = r2[t.rj[ty][k] * m + t.ri[ty][k]];   // else above the top
        a0 = fma_of((T)t.rw[ty][k], x.x, a0);
        a1 = fma_of((T)t.rw[ty][k], x.y, a1);
      }
    };
    switch (type_of(I, J)) {
      case 0: sum(std::integral_constant<int, 0>()); break;
      case 1: sum(std::integral_constant<int, 1>()); break;
      case 2: sum(std::integral_constant<int, 2>()); break;
      default: sum(std::integral_constant<int, 3>());
    }
  }
  reinterpret_cast<P *>(b)[(long)J * mc + I] = mk<T>(a0, a1);
}

// x += P xc, one thread a fine node.  Coarse nodes with prescribed velocity
// are left out by zero weights: a block's line knows its own, and a thread
// takes the weights of an inner cell, the first or the last one of the line.
// Latency bound: the tables come from global memory (divergent loads of
// constant memory take turns) and the old value is requested with them.  384^2
// Oseen solve, against the form that left no node out: 34.36 and 34.38, 34.86
// and 34.87, 36.35 and 36.18 ms; with a check at the coarse nodes 0.2 to 0.6 %
// more in every run.
template <typename T>
__global__ void k_p2_prolong(int nc, int open, const T *__restrict__ xc, T *__restrict__ x) {
  using P = typename V2<T>::type;
  __shared__ float w[4][4][6];
  __shared__ int off[4][6], cnt[4];
  const int mc = 2 * nc + 1, m = 4 * nc + 1, J = blockIdx.y;
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  const bool fixed = prescribed(I, J, m, open);
  P *xi = reinterpret_cast<P *>(x) + (long)J * m + I;
  P old = mk<T>(0, 0);
  if (!fixed) old = *xi;   // requested with the tables
  if (threadIdx.x < 96) {   // the line's four classes, by (first cell) + 2 (last cell)
    const int t = threadIdx.x % 24, at = threadIdx.x / 24, c = 4 * (J & 3) + t / 6, k = t % 6;
    const int ti = g_transfers.pi[c][k], tj = g_transfers.pj[c][k], line = 2 * (J >> 2) + tj;
    const bool out = ((at & 1) && ti == 0) || ((at & 2) && ti == 2) || line == 0 || (!open && line == mc - 1);
    w[at][t / 6][k] = out ? 0.f : g_transfers.pw[c][k];
    if (at == 0) {
      off[t / 6][k] = tj * mc + ti;
      if (k == 0) cnt[t / 6] = g_transfers.pn[c];
    }
  }
  __syncthreads();
  if (fixed) return;
  const P *c = reinterpret_cast<const P *>(xc) + (long)(2 * (J >> 2)) * mc + 2 * (I >> 2);
  const int q = I & 3, n = cnt[q], at = ((I >> 2) == 0 ? 1 : 0) + ((I >> 2) == nc - 1 ? 2 : 0);
  T a0 = 0, a1 = 0;
#pragma unroll
  for (int k = 0; k < 6; ++k)
    if (k < n) {
      const P v = c[off[q][k]];
      a0 = fma_of((T)w[at][q][k], v.x, a0);
      a1 = fma_of((T)w[at][q][k], v.y, a1);
    }
  *xi = mk<T>(old.x + a0, old.y + a1);
}
}  // namespace

template <typename T>
void p2_restrict(int nc, int open_top, const T *r, T *b, cudaStream_t s) {
  const dim3 g((unsigned)((nc + 1 + 127) / 128), (unsigned)(2 * nc + 1), 2);
  if (open_top) k_p2_restrict<T, true><<<g, 128, 0, s>>>(nc, r, b);
  else k_p2_restrict<T, false><<<g, 128, 0, s>>>(nc, r, b);
  CHNSS_LAUNCH_CK();
}
template <typename T>
void p2_prolong_add(int nc, int open_top, const T *xc, T *x, cudaStream_t s) {
  const dim3 g((unsigned)((4 * nc + 1 + 255) / 256), (unsigned)(4 * nc + 1));
  k_p2_prolong<T><<<g, 256, 0, s>>>(nc, open_top, xc, x);
  CHNSS_LAUNCH_CK();
}
template void p2_restrict<float>(int, int, const float *, float *, cudaStream_t);
template void p2_restrict<double>(int, int, const double *, double *, cudaStream_t);
template void p2_prolong_add<float>(int, int, const float *, float *, cudaStream_t);
template void p2_prolong_add<double>(int, int, const double *, double *, cudaStream_t);

template <typename VT>
void p2_spmv(const Level &L, int open_top, const P2Table &tab, const VT *val, const float *u, float *out, SpmvMode mode,
             const SpmvArgs &a, P2Start start, const double *scale, cudaStream_t s) {
  using T = float;
  for (const void *q : {(const void *)u, (const void *)out, a.b, a.w, a.dinv})
    if (!aligned(q, 2 * sizeof(T))) throw Error{CHNSS_ERR_ARG, "velocity vectors must be aligned to one node"};
  Coef<T> cf;
  for (int k = 0; k < kCount; ++k) cf.c[k] = rounded(tab.c[k], val);
  const T *dt = device_table(tab, val);
  const Args ka = {a.b, a.w, a.dinv, a.coef, scale};
  const int ks = sell_warps_bsr2(L.p2.sell);
  if (open_top) launch<T, VT, true>(L, ks, val, u, out, mode, start, ka, cf, dt, s);
  else launch<T, VT, false>(L, ks, val, u, out, mode, start, ka, cf, dt, s);
  CHNSS_LAUNCH_CK();
}
template void p2_spmv<float>(const Level &, int, const P2Table &, const float *, const float *, float *,
                                    SpmvMode, const SpmvArgs &, P2Start, const double *, cudaStream_t);
template void p2_spmv<__nv_bfloat16>(const Level &, int, const P2Table &, const __nv_bfloat16 *, const float *,
                                            float *, SpmvMode, const SpmvArgs &, P2Start, const double *, cudaStream_t);

}  // namespace chnss
