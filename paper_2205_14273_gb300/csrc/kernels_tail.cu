// Coarse-level transition (the hybrid idea of Section 3.5): below a chosen
// level the V-cycle leaves the stencil kernels.  At setup every level from
// the transition level T down to the coarsest is assembled: A_l = S_l + U_l
// as CSR rows (stencil entries inside the box in entry order, then the
// couplings), the smoother diagonal omega M^-1 (Section 3.4), P's row of
// every fine cell (Section 3.2) and the restriction row P^T of every coarse
// cell, and the coarsest operator's explicit inverse.  The rows of each level
// are split into NC contiguous slices, one per CTA of a thread-block cluster;
// each CTA's share is laid out as one contiguous image in global memory.
//
// In the solve one cluster runs the whole tail of the V(1,1) cycle: every
// CTA copies its image into shared memory, the level vectors (x, b, r) live
// in the CTAs' shared memory (distributed shared memory: a column index packs
// the owning CTA and the position in its slice), and cluster barriers
// separate the steps that other launches separate elsewhere: pre-relaxation
// from zero, residual, restriction, coarsest solve, prolongation, post-
// relaxation (Eq. relax0).  Every row is summed in a fixed order (its
// entries strided over a group of lanes, then a fixed shuffle tree), so a tail
// result is the same bit for bit from run to run.
//
// The smallest levels (at most SSAMG_CTAIL_LOCAL_CELLS cells) cost the same
// four barriers and remote round trips as the others, ~3.8 us (FP32) and
// ~4.7 us (FP64) each, with nothing to spread.  In FP32 every CTA holds them
// whole and runs them for itself: block barriers and its own shared memory,
// each row summed as a cluster of 16 would.  In FP64 an SM's two multiply-adds per
// clock forbid that (256 rows x 30 entries are 2 us an apply); there the rest
// of the cycle from the first such level down, a linear map of its right-hand
// side, is formed at setup as a dense matrix (one block per column runs that
// sub-cycle on a unit vector) and applied like the coarsest inverse, one
// barrier and 65,536 multiply-adds over the cluster.
// Measured (tail of one cycle, replayed alone): 13 levels of one part, FP64 61.6 ->
// 25.4 us, FP32 39.4 -> 25.2; 10 levels of 8 parts, FP64 55.4 -> 32.4, FP32 34.6 -> 26.0;
// 13 levels of two parts, FP64 64.4 -> 31.3, FP32 43.6 -> 29.9 us.  A row's arithmetic is a small part of a step: four
// barriers of ~0.3-0.5 us and a remote round trip remain per cluster level.
#include <cooperative_groups.h>

#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "kernels_common.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int CT = SSAMG_CTAIL_THREADS;

// Packed column: owning CTA (high bits) and position in its slice.
__device__ __forceinline__ unsigned short ctail_pack(int g, int S) {
  const int o = g / S;
  return (unsigned short)((o << SSAMG_CTAIL_LOCAL_BITS) | (g - o * S));
}

// Row lengths of the tail levels: entries of S inside the box plus the row's
// couplings.
// Row lengths of one level, a warp per row: lane e tests entry e.
__device__ __forceinline__ void ctail_rowlen_row(const LevelView<double>& L, int* __restrict__ len,
                                                 int g) {
  const int lane = threadIdx.x & 31;
  if (g >= L.N) return;
  const int p = find_part_cell(L.cellstart, L.np, g);
  const DPart& dp = L.parts[p];
  int i, j, k;
  cell_coords(dp, g - dp.off, i, j, k);
  const bool ok = lane < dp.nent && inside(dp, i + dp.o[lane][0], j + dp.o[lane][1], k + dp.o[lane][2]);
  int n = __popc(__ballot_sync(0xffffffffu, ok));
  if (lane == 0) {
    if (dp.has_u && L.u_map) {
      const int r = L.u_map[g];
      if (r >= 0) n += L.u_ptr[r + 1] - L.u_ptr[r];
    }
    len[g] = n;
  }
}

// Every candidate level in one launch: block b works on the level whose
// block range holds it (8 rows per block).
struct CTailRowlenArgs {
  int nl;
  int b0[SSAMG_CTAIL_MAX_LEVELS + 1];
  int* len[SSAMG_CTAIL_MAX_LEVELS];
  LevelView<double> lv[SSAMG_CTAIL_MAX_LEVELS];
};
__global__ void __launch_bounds__(256) k_ctail_rowlen(const __grid_constant__ CTailRowlenArgs A) {
  int l = 0;
  while (l + 1 < A.nl && (int)blockIdx.x >= A.b0[l + 1]) ++l;
  const int g = ((int)blockIdx.x - A.b0[l]) * 8 + (int)(threadIdx.x >> 5);
  ctail_rowlen_row(A.lv[l], A.len[l], g);
}

// Fills the images of one tail level l: for every row g, in the slice of its
// owning CTA: its CSR entries (columns packed in this level's slices), the
// smoother diagonal, P's row (columns packed in level l+1's slices) when
// has_p, the restriction row from level l-1 (columns packed in l-1's
// slices) when Fm is given, and the coarsest inverse's row when inv is
// given.  The row pointers were written by the host.
// One tail level's share of a fill launch.
struct CTailFillLevel {
  LevelView<double> L, fm, ln;
  const double* dinv;
  const double* inv;
  CTailLevel lv;
  int has_fm, has_p, Sm, Sn;
};
struct CTailFillArgs {
  int nl, nL;
  long long ro_bytes;
  char* image;
  char* common;
  int b0[SSAMG_CTAIL_MAX_LEVELS + 1];
  CTailFillLevel lev[SSAMG_CTAIL_MAX_LEVELS];
};

template <class T>
__device__ __forceinline__ void ctail_fill_row(const LevelView<double>& L,
                                               const double* __restrict__ dinv64,
                                               const LevelView<double>& Fm, int has_fm,
                                               const LevelView<double>& Ln, int has_p,
                                               const double* __restrict__ inv, int nL,
                                               const CTailLevel& lv, int Sm, int Sn,
                                               char* __restrict__ image, long long ro_bytes,
                                               char* __restrict__ common, int g) {
  // a warp per row: the stencil entries one per lane (slots by ballot, in
  // entry order), the coupling entries strided over the lanes, the rest by
  // lane 0
  const int lane = threadIdx.x & 31;
  if (g >= L.N) return;
  const int owner = g / lv.S, li = g - owner * lv.S;
  char* img = lv.local ? common : image + owner * ro_bytes;
  const int* rowptr = reinterpret_cast<const int*>(img + lv.o_rowptr);
  unsigned short* col = reinterpret_cast<unsigned short*>(img + lv.o_col);
  T* val = reinterpret_cast<T*>(img + lv.o_val);
  T* dv = reinterpret_cast<T*>(img + lv.o_dinv);
  const int p = find_part_cell(L.cellstart, L.np, g);
  const DPart& dp = L.parts[p];
  const int c = g - dp.off;
  int i, j, k;
  cell_coords(dp, c, i, j, k);
  const int q0 = rowptr[li];
  const bool ok = lane < dp.nent && inside(dp, i + dp.o[lane][0], j + dp.o[lane][1], k + dp.o[lane][2]);
  const unsigned m = __ballot_sync(0xffffffffu, ok);
  if (ok) {
    const int q = q0 + __popc(m & ((1u << lane) - 1u));
    col[q] = ctail_pack(g + dp.disp[lane], lv.S);
    val[q] = (T)coef_at(dp, L.coef, lane, c);
  }
  if (dp.has_u && L.u_map) {
    const int r = L.u_map[g];
    if (r >= 0) {
      const int t0 = L.u_ptr[r], t1 = L.u_ptr[r + 1], q1 = q0 + __popc(m) - t0;
      for (int t = t0 + lane; t < t1; t += 32) {
        col[q1 + t] = ctail_pack(L.u_col[t], lv.S);
        val[q1 + t] = (T)L.u_val[t];
      }
    }
  }
  if (inv) {
    double* iv = reinterpret_cast<double*>(img + lv.o_inv);
    for (int t = lane; t < nL; t += 32) iv[(long long)li * nL + t] = inv[(long long)g * nL + t];
  }
  if (lane != 0) return;
  dv[li] = (T)dinv64[g];
  if (has_p) {
    // P's row of fine cell g (Section 3.2), coarse columns on level l+1
    const PRow<double> pr = p_row(dp, L.Pw, L.Pe, i, j, k);
    unsigned short* pc = reinterpret_cast<unsigned short*>(img + lv.o_pcol);
    T* pv = reinterpret_cast<T*>(img + lv.o_pval);
    pc[li] = pr.j0 >= 0 ? ctail_pack(pr.j0, Sn) : 0;
    pv[li] = pr.j0 >= 0 ? (T)pr.w0 : (T)0;
    pc[lv.S + li] = pr.j1 >= 0 ? ctail_pack(pr.j1, Sn) : 0;
    pv[lv.S + li] = pr.j1 >= 0 ? (T)pr.w1 : (T)0;
  }
  if (has_fm) {
    // restriction row of coarse cell g from level l-1: the anchor (weight 1)
    // and the fine points beside it along d* (PE of the west one, PW of the
    // east one), as the stencil restriction applies them
    const DPart& fp = Fm.parts[p];
    unsigned short* rc = reinterpret_cast<unsigned short*>(img + lv.o_rcol);
    T* rv = reinterpret_cast<T*>(img + lv.o_rval);
    int f0, f1 = -1, f2 = -1;
    double w1 = 0.0, w2 = 0.0;
    const int d = fp.dstar;
    if (d < 0) {
      f0 = fp.off + (k * fp.n[1] + j) * fp.n[0] + i;
    } else {
      int f[3] = {i, j, k};
      const int anchor = 2 * f[d] + fp.par;
      f[d] = anchor;
      const int sd = (d == 0) ? 1 : (d == 1 ? fp.n[0] : fp.n[0] * fp.n[1]);
      f0 = fp.off + (f[2] * fp.n[1] + f[1]) * fp.n[0] + f[0];
      if (anchor - 1 >= 0) {
        f[d] = anchor - 1;
        f1 = f0 - sd;
        w1 = Fm.Pe[fp.poff + fine_point_index(fp, f[0], f[1], f[2])];
      }
      if (anchor + 1 < fp.n[d]) {
        f[d] = anchor + 1;
        f2 = f0 + sd;
        w2 = Fm.Pw[fp.poff + fine_point_index(fp, f[0], f[1], f[2])];
      }
    }
    rc[li] = ctail_pack(f0, Sm);
    rv[li] = (T)1;
    rc[lv.S + li] = f1 >= 0 ? ctail_pack(f1, Sm) : 0;
    rv[lv.S + li] = f1 >= 0 ? (T)w1 : (T)0;
    rc[2 * lv.S + li] = f2 >= 0 ? ctail_pack(f2, Sm) : 0;
    rv[2 * lv.S + li] = f2 >= 0 ? (T)w2 : (T)0;
  }
}

// Every tail level's images in one launch (8 rows per block).
template <class T>
__global__ void __launch_bounds__(256) k_ctail_fill(const __grid_constant__ CTailFillArgs A) {
  int l = 0;
  while (l + 1 < A.nl && (int)blockIdx.x >= A.b0[l + 1]) ++l;
  const CTailFillLevel& v = A.lev[l];
  const int g = ((int)blockIdx.x - A.b0[l]) * 8 + (int)(threadIdx.x >> 5);
  ctail_fill_row<T>(v.L, v.dinv, v.fm, v.has_fm, v.ln, v.has_p, v.inv, A.nL, v.lv, v.Sm, v.Sn,
                    A.image, A.ro_bytes, A.common, g);
}

// Cluster-wide barrier between the tail's steps.  The non-aligned forms of
// barrier.cluster (release on arrival, acquire on the wait) do not need the
// warp's lanes to arrive together, so a warp whose lanes left a row loop at
// different times still counts as arrived only once every lane has; the
// release/acquire pair makes each CTA's shared-memory writes before the
// barrier visible to every CTA's reads after it.
__device__ __forceinline__ void ctail_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// Value of a packed column of vector `off` (byte offset of that level's
// vector in every CTA's shared memory); of a local level, from this CTA's own.
template <class T>
__device__ __forceinline__ T ctail_get(cg::cluster_group& cl, char* sm, int off,
                                       unsigned short pk, int local = 0) {
  if (local) return reinterpret_cast<const T*>(sm + off)[pk];
  const unsigned o = pk >> SSAMG_CTAIL_LOCAL_BITS;
  const unsigned l = pk & ((1u << SSAMG_CTAIL_LOCAL_BITS) - 1u);
  const T* base = cl.map_shared_rank(reinterpret_cast<T*>(sm + off), o);
  return base[l];
}

// The same over all rows of a level by NTH threads (tid among them), x in this
// CTA's shared memory.  For FP64: four entries at a time and then one by one, as
// an add that is predicated off takes the pipe as long as one that is not.
template <int NTH, class T, class Epi>
__device__ __forceinline__ void ctail_apply_local(int tid, const T* x, const CTailLevel& L,
                                                  const int* rp, const unsigned short* col,
                                                  const T* val, Epi&& epi) {
  const int tpr = L.tpr;
  const int lane = tid & 31, warp = tid >> 5;
  const int rpw = 32 / tpr;
  const int sub = lane / tpr, k = lane & (tpr - 1);
  for (int r0 = warp * rpw; r0 < L.S; r0 += (NTH / 32) * rpw) {
    const int li = r0 + sub;
    T acc = (T)0;
    if (li < L.S) {
      int q = rp[li] + k;
      const int q1 = rp[li + 1];
      for (; q + 3 * tpr < q1; q += 4 * tpr) {
        T v[4], a[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          a[u] = val[q + u * tpr];
          v[u] = x[col[q + u * tpr]];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) acc = fma(a[u], v[u], acc);
      }
      for (; q < q1; q += tpr) acc = fma(val[q], x[col[q]], acc);
    }
    __syncwarp();
    for (int o = tpr >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (li < L.S && k == 0) epi(li, acc);
  }
}

// Operator apply over the CSR rows of one level's slice: L.tpr lanes take a
// row (its entries strided over the lanes, each lane fetching up to eight of
// its entries before summing them, so that a row's remote loads are in
// flight together), their partial sums are added by a fixed shuffle tree,
// and the row's first lane hands the result to epi(li, (A x)(li)).  The loop
// bound is uniform over each warp, so every lane takes part in the shuffles.
template <class T, class Epi>
__device__ __forceinline__ void ctail_apply(cg::cluster_group& cl, char* sm, int xoff,
                                            const CTailLevel& L, const int* rp,
                                            const unsigned short* col, const T* val, Epi&& epi) {
  const int tpr = L.tpr;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rpw = 32 / tpr;  // rows per warp and pass
  const int sub = lane / tpr, k = lane & (tpr - 1);
  for (int r0 = warp * rpw; r0 < L.S; r0 += (CT / 32) * rpw) {
    const int li = r0 + sub;
    T acc = (T)0;
    if (li < L.S) {
      // this lane's entries q0 + k, q0 + k + tpr, ... eight loads at a time
      const int q1 = rp[li + 1];
      for (int q = rp[li] + k; q < q1; q += 8 * tpr) {
        T v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u)
          v[u] = q + u * tpr < q1 ? ctail_get<T>(cl, sm, xoff, col[q + u * tpr]) : (T)0;
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (q + u * tpr < q1) acc = fma(val[q + u * tpr], v[u], acc);
      }
    }
    for (int o = tpr >> 1; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (li < L.S && k == 0) epi(li, acc);
  }
}

// Sum of entries [q, q1) of a local level's row by G neighbouring lanes, lane
// h of them holding the partial sums of ctail_apply's lanes h, h + G, ... in
// registers: its tree, within a lane as far as it goes, with log2 G shuffles.
// With 16 CTAs a level of at most SSAMG_CTAIL_LOCAL_CELLS cells has 32 lanes a row
// there and the result is the same bit for bit (with 8 CTAs and more than 128
// cells it has 16, another order).  All lanes of the warp call.
template <int G, class T>
__device__ __forceinline__ T ctail_row_sum(const T* x, const unsigned short* col, const T* val,
                                           int q, int q1) {
  constexpr int K = 32 / G;
  T a[K];
#pragma unroll
  for (int j = 0; j < K; ++j) a[j] = q + G * j < q1 ? val[q + G * j] * x[col[q + G * j]] : (T)0;
  for (q += 32; q < q1; q += 32) {
#pragma unroll
    for (int j = 0; j < K; ++j)
      if (q + G * j < q1) a[j] = fma(val[q + G * j], x[col[q + G * j]], a[j]);
  }
#pragma unroll
  for (int o = K / 2; o > 0; o >>= 1) {
#pragma unroll
    for (int j = 0; j < o; ++j) a[j] += a[j + o];
  }
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
  return a[0];
}

// Operator apply over the rows of a local level by all threads of the CTA:
// as many lanes per row as give every row a group at once, the row's result to
// epi on its first lane.
template <class T, class Epi>
__device__ __forceinline__ void ctail_apply_rows(const CTailLevel& L, const T* x, const char* ro,
                                                 Epi&& epi) {
  const int* rp = reinterpret_cast<const int*>(ro + L.o_rowptr);
  const unsigned short* col = reinterpret_cast<const unsigned short*>(ro + L.o_col);
  const T* val = reinterpret_cast<const T*>(ro + L.o_val);
  auto rows = [&](auto g) {
    constexpr int G = decltype(g)::value;
    const int li = threadIdx.x / G, h = threadIdx.x % G;
    if ((int)(threadIdx.x & ~31u) / G >= L.n) return;  // (whole warps)
    const bool in = li < L.n;
    const T v = ctail_row_sum<G, T>(x, col, val, in ? rp[li] + h : 0, in ? rp[li + 1] : 0);
    if (in && h == 0) epi(li, v);
  };
  static_assert(SSAMG_CTAIL_LOCAL_CELLS * 2 <= CT, "two lanes for every row");
  if (L.n > CT / 4)
    rows(std::integral_constant<int, 2>{});
  else if (L.n > CT / 8)
    rows(std::integral_constant<int, 4>{});
  else
    rows(std::integral_constant<int, 8>{});
}

// The local levels jl .. nt - 1 in this CTA (b and x of level jl are in its
// shared memory): down, the last level and up, ending with the corrected x
// of level jl.
template <class T>
__device__ __forceinline__ void ctail_local_cycle(const CTailArgs& a, int jl, char* sm,
                                                  const char* ro) {
  const int li = threadIdx.x, nt = a.nt;
  auto vec = [&](int off) { return reinterpret_cast<T*>(sm + off); };
  for (int l = jl; l + 1 < nt; ++l) {
    const CTailLevel& L = a.lev[l];
    const CTailLevel& C = a.lev[l + 1];
    const T* b = vec(L.o_b);
    T* r = vec(L.o_r);
    __syncthreads();  // x of level l
    ctail_apply_rows<T>(L, vec(L.o_x), ro, [&](int i, T ax) { r[i] = b[i] - ax; });
    __syncthreads();  // r of level l
    if (li < C.n) {
      const unsigned short* rc = reinterpret_cast<const unsigned short*>(ro + C.o_rcol);
      const T* rv = reinterpret_cast<const T*>(ro + C.o_rval);
      T v = rv[li] * r[rc[li]];
      v = fma(rv[C.S + li], r[rc[C.S + li]], v);
      v = fma(rv[2 * C.S + li], r[rc[2 * C.S + li]], v);
      vec(C.o_b)[li] = v;
      vec(C.o_x)[li] = reinterpret_cast<const T*>(ro + C.o_dinv)[li] * v;
    }
  }
  if (a.direct) {
    const CTailLevel& L = a.lev[nt - 1];
    __syncthreads();  // b of the last level
    if (li < L.n) {
      const double* iv = reinterpret_cast<const double*>(ro + L.o_inv) + (long long)li * a.nL;
      const T* b = vec(L.o_b);
      double s = 0.0;
#pragma unroll 8
      for (int t = 0; t < a.nL; ++t) s = fma(iv[t], (double)b[t], s);
      vec(L.o_x)[li] = (T)s;
    }
  }
  for (int l = nt - 2; l >= jl; --l) {
    const CTailLevel& L = a.lev[l];
    const CTailLevel& C = a.lev[l + 1];
    const T* e = vec((l + 1 == nt - 1) ? C.o_x : C.o_r);
    const T* b = vec(L.o_b);
    T* x = vec(L.o_x);
    T* out = vec(L.o_r);
    __syncthreads();  // x of level l+1
    if (li < L.n) {
      const unsigned short* pc = reinterpret_cast<const unsigned short*>(ro + L.o_pcol);
      const T* pv = reinterpret_cast<const T*>(ro + L.o_pval);
      T v = x[li];
      v = fma(pv[li], e[pc[li]], v);
      v = fma(pv[L.S + li], e[pc[L.S + li]], v);
      x[li] = v;
    }
    __syncthreads();  // x + P e of level l
    const T* dv = reinterpret_cast<const T*>(ro + L.o_dinv);
    ctail_apply_rows<T>(L, x, ro, [&](int i, T ax) { out[i] = fma(dv[i], b[i] - ax, x[i]); });
  }
}

// The tail of one V(1,1) cycle: from the right-hand side of level T (global,
// b_top) to the corrected x of level T (global, x_top).
template <class T>
__global__ void __launch_bounds__(CT, 1) k_ctail(const CTailArgs a, const T* b_top, T* x_top) {
  pdl_trigger();
  extern __shared__ __align__(16) char sm[];
  cg::cluster_group cl = cg::this_cluster();
  const int c = (int)cl.block_rank();
  const int tid = threadIdx.x;
  // the read-only images (setup data) first, then the wait for the
  // predecessor that wrote b_top
  {
    const int4* src = reinterpret_cast<const int4*>(a.image + (long long)c * a.ro_bytes);
    int4* dst = reinterpret_cast<int4*>(sm + a.vec_bytes);
    const int n16 = (int)(a.ro_bytes / 16);
#pragma unroll 4
    for (int t = tid; t < n16; t += CT) dst[t] = src[t];
    src = reinterpret_cast<const int4*>(a.common);
    dst += n16;
    const int l16 = (int)(a.lo_bytes / 16);
#pragma unroll 4
    for (int t = tid; t < l16; t += CT) dst[t] = src[t];
  }
  pdl_wait();
  __syncthreads();  // the image (read below: level T's diagonal) is staged
  const int nt = a.nt;
  const char* const ro_s = sm + a.vec_bytes;
  const char* const ro_l = ro_s + a.ro_bytes;
  auto ro_of = [&](const CTailLevel& L) { return L.local ? ro_l : ro_s; };
  auto apply = [&](const CTailLevel& L, auto&& epi) {
    ctail_apply<T>(cl, sm, L.o_x, L, reinterpret_cast<const int*>(ro_s + L.o_rowptr),
                   reinterpret_cast<const unsigned short*>(ro_s + L.o_col),
                   reinterpret_cast<const T*>(ro_s + L.o_val), epi);
  };
  {
    const CTailLevel& L = a.lev[0];
    T* b = reinterpret_cast<T*>(sm + L.o_b);
    T* x = reinterpret_cast<T*>(sm + L.o_x);
    const T* dv = reinterpret_cast<const T*>(ro_of(L) + L.o_dinv);
    for (int li = tid; li < L.S; li += CT) {
      const int g = (L.local ? 0 : c * L.S) + li;
      const T v = g < L.n ? b_top[g] : (T)0;
      b[li] = v;
      x[li] = dv[li] * v;  // pre-relaxation from zero
    }
  }
  // down: residual, then restriction with the coarse level's pre-relaxation
  // (onto the first local level every CTA restricts all of it)
  for (int l = 0; l + 1 < nt && !a.lev[l].local; ++l) {
    const CTailLevel& L = a.lev[l];
    const CTailLevel& C = a.lev[l + 1];
    const T* b = reinterpret_cast<const T*>(sm + L.o_b);
    T* r = reinterpret_cast<T*>(sm + L.o_r);
    ctail_sync();  // x of level l complete in every CTA
    apply(L, [&](int li, T ax) { r[li] = b[li] - ax; });
    ctail_sync();  // r of level l complete
    const char* ro = ro_of(C);
    const unsigned short* rc = reinterpret_cast<const unsigned short*>(ro + C.o_rcol);
    const T* rv = reinterpret_cast<const T*>(ro + C.o_rval);
    const T* dvc = reinterpret_cast<const T*>(ro + C.o_dinv);
    T* bc = reinterpret_cast<T*>(sm + C.o_b);
    T* xc = reinterpret_cast<T*>(sm + C.o_x);
    for (int li = tid; li < C.S; li += CT) {
      T v = rv[li] * ctail_get<T>(cl, sm, L.o_r, rc[li]);
      v = fma(rv[C.S + li], ctail_get<T>(cl, sm, L.o_r, rc[C.S + li]), v);
      v = fma(rv[2 * C.S + li], ctail_get<T>(cl, sm, L.o_r, rc[2 * C.S + li]), v);
      bc[li] = v;
      xc[li] = dvc[li] * v;
    }
  }
  if (a.jl < nt) {
    if constexpr (sizeof(T) == 4)  // (FP64 has no local levels)
      ctail_local_cycle<T>(a, a.jl, sm, ro_l);
    __syncthreads();  // the corrected x of the first local level
  } else if (a.direct) {
    // last level: its explicit matrix (FP64)
    const CTailLevel& L = a.lev[nt - 1];
    T* x = reinterpret_cast<T*>(sm + L.o_x);
    const double* iv = reinterpret_cast<const double*>(ro_s + L.o_inv);
    ctail_sync();  // b of the last level
    if (a.dense) {
      // every CTA gathers b, then eight lanes per row of its slice
      double* sb = reinterpret_cast<double*>(sm + a.o_sb);
      for (int t = tid; t < a.nL; t += CT) {
        const int o = t / L.S;
        sb[t] = (double)cl.map_shared_rank(reinterpret_cast<T*>(sm + L.o_b), o)[t - o * L.S];
      }
      __syncthreads();
      constexpr int DL = 8;  // lanes per row (each add of a lane tree takes the FP64 pipe 16 cycles)
      for (int l0 = 0; l0 < L.S; l0 += CT / DL) {
        const int li = l0 + tid / DL;
        double s = 0.0;
        if (li < L.S) {
          const double* row = iv + (long long)li * a.nL;
#pragma unroll 8
          for (int t = tid % DL; t < a.nL; t += DL) s = fma(row[t], sb[t], s);
        }
        if (l0 + (tid & ~31) / DL < L.S)  // (warps with a row)
          for (int o = DL / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (li < L.S && tid % DL == 0) x[li] = (T)s;
      }
    } else {
      for (int li = tid; li < L.S; li += CT) {
        double s = 0.0;
        if (c * L.S + li < L.n) {
          int t = 0;
          for (; t + 8 <= a.nL; t += 8) {
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const int o = (t + u) / L.S;
              v[u] = (double)cl.map_shared_rank(reinterpret_cast<T*>(sm + L.o_b), o)[t + u - o * L.S];
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) s = fma(iv[(long long)li * a.nL + t + u], v[u], s);
          }
          for (; t < a.nL; ++t) {
            const int o = t / L.S;
            const T* bb = cl.map_shared_rank(reinterpret_cast<T*>(sm + L.o_b), o);
            s = fma(iv[(long long)li * a.nL + t], (double)bb[t - o * L.S], s);
          }
        }
        x[li] = (T)s;
      }
    }
  }
  // (without the direct solve x = omega M^-1 b is already there)
  // up: prolongation x_l += P x_{l+1}, then post-relaxation into r_l
  for (int l = min(nt - 2, a.jl - 1); l >= 0; --l) {
    const CTailLevel& L = a.lev[l];
    const CTailLevel& C = a.lev[l + 1];
    const char* ro = ro_s;
    const int xcoff = (l + 1 == nt - 1) ? C.o_x : C.o_r;  // the corrected x of level l+1
    const unsigned short* pc = reinterpret_cast<const unsigned short*>(ro + L.o_pcol);
    const T* pv = reinterpret_cast<const T*>(ro + L.o_pval);
    T* x = reinterpret_cast<T*>(sm + L.o_x);
    if (!C.local) ctail_sync();  // x of level l+1
    for (int li = tid; li < L.S; li += CT) {
      T v = x[li];
      v = fma(pv[li], ctail_get<T>(cl, sm, xcoff, pc[li], C.local), v);
      v = fma(pv[L.S + li], ctail_get<T>(cl, sm, xcoff, pc[L.S + li], C.local), v);
      x[li] = v;
    }
    ctail_sync();  // x + P e of level l complete
    const T* dv = reinterpret_cast<const T*>(ro + L.o_dinv);
    const T* b = reinterpret_cast<const T*>(sm + L.o_b);
    T* out = reinterpret_cast<T*>(sm + L.o_r);
    apply(L, [&](int li, T ax) { out[li] = fma(dv[li], b[li] - ax, x[li]); });
  }
  // the corrected x of level T (own slice) to global memory; its rows were
  // written by the first lanes of the row groups
  __syncthreads();
  {
    const CTailLevel& L = a.lev[0];
    const T* res = reinterpret_cast<const T*>(sm + (nt > 1 ? L.o_r : L.o_x));
    if (!L.local || c == 0)
      for (int li = tid; li < L.S; li += CT) {
        const int g = (L.local ? 0 : c * L.S) + li;
        if (g < L.n) x_top[g] = res[li];
      }
  }
  ctail_sync();  // no CTA leaves while another may still read its shared memory
}

// CTAIL_COLS columns of the dense matrix of the levels of `a` (all local, FP64):
// their cycle applied to unit vectors, a group of CT / CTAIL_COLS threads each,
// vectors in shared memory, and the image too where it fits (`staged`: read
// where it lies, every step is two dependent L2 round trips; 256 cells of one
// part: 94 -> 36 us).
constexpr int CTAIL_COLS = 2;
__global__ void __launch_bounds__(CT) k_ctail_columns(const CTailArgs a, int staged, double* dense) {
  constexpr int NTH = CT / CTAIL_COLS;
  extern __shared__ __align__(16) char smem[];
  const int grp = threadIdx.x / NTH, tid = threadIdx.x % NTH;
  char* const sm = smem + grp * a.vec_bytes;
  const char* img = a.common;
  if (staged) {
    char* to = smem + CTAIL_COLS * a.vec_bytes;
    const int4* src = reinterpret_cast<const int4*>(a.common);
    const int n16 = (int)(a.lo_bytes / 16);
#pragma unroll 8
    for (int t = threadIdx.x; t < n16; t += CT) reinterpret_cast<int4*>(to)[t] = src[t];
    img = to;
    __syncthreads();
  }
  const int column = blockIdx.x * CTAIL_COLS + grp;  // (beyond the last: a zero vector, not stored)
  const int nt = a.nt;
  auto vec = [&](int off) { return reinterpret_cast<double*>(sm + off); };
  auto ro = [&](int off) { return img + off; };
  auto apply = [&](const CTailLevel& L, auto&& epi) {
    ctail_apply_local<NTH, double>(tid, vec(L.o_x), L, reinterpret_cast<const int*>(ro(L.o_rowptr)),
                              reinterpret_cast<const unsigned short*>(ro(L.o_col)),
                              reinterpret_cast<const double*>(ro(L.o_val)), epi);
  };
  {
    const CTailLevel& L = a.lev[0];
    const double* dv = reinterpret_cast<const double*>(ro(L.o_dinv));
    for (int li = tid; li < L.S; li += NTH) {
      const double v = li == column ? 1.0 : 0.0;
      vec(L.o_b)[li] = v;
      vec(L.o_x)[li] = dv[li] * v;
    }
  }
  for (int l = 0; l + 1 < nt; ++l) {
    const CTailLevel& L = a.lev[l];
    const CTailLevel& C = a.lev[l + 1];
    const double* b = vec(L.o_b);
    double* r = vec(L.o_r);
    __syncthreads();
    apply(L, [&](int li, double ax) { r[li] = b[li] - ax; });
    __syncthreads();
    const unsigned short* rc = reinterpret_cast<const unsigned short*>(ro(C.o_rcol));
    const double* rv = reinterpret_cast<const double*>(ro(C.o_rval));
    const double* dvc = reinterpret_cast<const double*>(ro(C.o_dinv));
    for (int li = tid; li < C.S; li += NTH) {
      double v = rv[li] * r[rc[li]];
      v = fma(rv[C.S + li], r[rc[C.S + li]], v);
      v = fma(rv[2 * C.S + li], r[rc[2 * C.S + li]], v);
      vec(C.o_b)[li] = v;
      vec(C.o_x)[li] = dvc[li] * v;
    }
  }
  __syncthreads();
  if (a.direct) {
    const CTailLevel& L = a.lev[nt - 1];
    const double* iv = reinterpret_cast<const double*>(ro(L.o_inv));
    for (int li = tid; li < L.S; li += NTH) {
      double s = 0.0;
      for (int t = 0; t < a.nL; ++t) s = fma(iv[li * a.nL + t], vec(L.o_b)[t], s);
      vec(L.o_x)[li] = s;
    }
  }
  for (int l = nt - 2; l >= 0; --l) {
    const CTailLevel& L = a.lev[l];
    const CTailLevel& C = a.lev[l + 1];
    const double* e = vec((l + 1 == nt - 1) ? C.o_x : C.o_r);
    const unsigned short* pc = reinterpret_cast<const unsigned short*>(ro(L.o_pcol));
    const double* pv = reinterpret_cast<const double*>(ro(L.o_pval));
    double* x = vec(L.o_x);
    __syncthreads();
    for (int li = tid; li < L.S; li += NTH) {
      double v = x[li];
      v = fma(pv[li], e[pc[li]], v);
      v = fma(pv[L.S + li], e[pc[L.S + li]], v);
      x[li] = v;
    }
    __syncthreads();
    const double* dv = reinterpret_cast<const double*>(ro(L.o_dinv));
    const double* b = vec(L.o_b);
    double* out = vec(L.o_r);
    apply(L, [&](int li, double ax) { out[li] = fma(dv[li], b[li] - ax, x[li]); });
  }
  __syncthreads();
  const CTailLevel& L = a.lev[0];
  const double* res = vec(nt > 1 ? L.o_r : L.o_x);
  if (column < L.n)
    for (int li = tid; li < L.S; li += NTH) dense[(long long)li * L.n + column] = res[li];
}

inline int cdiv(long long a, long long b) { return (int)((a + b - 1) / b); }

}  // namespace

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
template <class T>
bool ctail_query(int nc, long long smem);
void launch_ctail_rowlen(const std::vector<Level>& lev, int first, int last, int* const* len,
                         cudaStream_t st) {
  for (int l0 = first; l0 <= last; l0 += SSAMG_CTAIL_MAX_LEVELS) {
    CTailRowlenArgs a{};
    int nb = 0;
    for (int l = l0; l <= last && a.nl < SSAMG_CTAIL_MAX_LEVELS; ++l) {
      a.b0[a.nl] = nb;
      a.len[a.nl] = len[l - first];
      a.lv[a.nl] = lev[l].view<double>();
      ++a.nl;
      nb += cdiv(lev[l].N, 8);
    }
    a.b0[a.nl] = nb;
    if (nb == 0) continue;
    k_ctail_rowlen<<<nb, 256, 0, st>>>(a);
    SSAMG_LAUNCH_CHECK();
  }
}

void launch_ctail_fill(bool fp32, const std::vector<Level>& lev, int t0, const CTailArgs& ta,
                       const double* inv, char* image, char* common, cudaStream_t st) {
  const int nt = ta.nt;
  CTailFillArgs a{};
  a.nl = nt;
  a.nL = ta.nL;
  a.ro_bytes = ta.ro_bytes;
  a.image = image;
  a.common = common;
  int nb = 0;
  for (int j = 0; j < nt; ++j) {
    const Level& L = lev[t0 + j];
    CTailFillLevel& v = a.lev[j];
    v.L = L.view<double>();
    v.fm = j > 0 ? lev[t0 + j - 1].view<double>() : v.L;
    v.ln = j + 1 < nt ? lev[t0 + j + 1].view<double>() : v.L;
    v.has_fm = j > 0;
    v.has_p = j + 1 < nt;
    v.dinv = L.dinv;
    v.inv = (j + 1 == nt) ? inv : nullptr;
    v.lv = ta.lev[j];
    v.Sm = j > 0 ? ta.lev[j - 1].S : 1;
    v.Sn = j + 1 < nt ? ta.lev[j + 1].S : 1;
    a.b0[j] = nb;
    nb += cdiv(L.N, 8);
  }
  a.b0[nt] = nb;
  if (fp32)
    k_ctail_fill<float><<<nb, 256, 0, st>>>(a);
  else
    k_ctail_fill<double><<<nb, 256, 0, st>>>(a);
  SSAMG_LAUNCH_CHECK();
}

// Dynamic shared memory kernel `k` is allowed on device dev: at least smem.  The
// attribute belongs to the function, not to a launch, so it is never lowered: a
// solver set up later with a smaller tail must not cut off the launches of one
// set up before.
static cudaError_t allow_smem(const void* k, int dev, long long smem) {
  static std::mutex mu;
  static std::map<std::pair<const void*, int>, long long> allowed;
  std::lock_guard<std::mutex> lock(mu);
  long long& a = allowed[{k, dev}];
  if (smem <= a) return cudaSuccess;
  const cudaError_t e =
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) a = smem;
  return e;
}

// Shared memory of k_ctail_columns: the vectors of its columns, and the image
// where both fit SSAMG_CTAIL_STAGE_BYTES.  Without the image it can still be
// beyond the 48 KB a kernel has by default (levels of more than 1024 cells
// together, as many small parts leave: 149 parts of 2^3 beside one of 16^3,
// 1170 cells, 56 KB).
static long long ctail_columns_smem(const CTailArgs& a, bool& staged) {
  const long long vec = (long long)CTAIL_COLS * a.vec_bytes, all = vec + a.lo_bytes;
  staged = all <= SSAMG_CTAIL_STAGE_BYTES;
  return staged ? all : vec;
}

bool ctail_columns_prepare(const CTailArgs& a, long long optin) {
  int dev = 0;
  bool staged;
  const long long smem = ctail_columns_smem(a, staged);
  if (smem > optin) return false;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      allow_smem((const void*)k_ctail_columns, dev, smem) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return true;
}

void launch_ctail_columns(const CTailArgs& a, double* dense, cudaStream_t st) {
  bool staged;
  const long long smem = ctail_columns_smem(a, staged);
  k_ctail_columns<<<cdiv(a.lev[0].n, CTAIL_COLS), CT, (size_t)smem, st>>>(a, staged, dense);
  SSAMG_LAUNCH_CHECK();
}

template <class T>
bool ctail_prepare(int nc, long long smem) {
  // the answer per device and (nc, smem) is kept: the occupancy query costs
  // more than the rest of a small setup
  static std::mutex mu;
  static std::map<std::tuple<int, int, long long>, bool> known;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const auto key = std::make_tuple(dev, nc, smem);
  std::lock_guard<std::mutex> lock(mu);
  auto it = known.find(key);
  if (it != known.end()) return it->second;
  if (allow_smem((const void*)k_ctail<T>, dev, smem) != cudaSuccess) {
    cudaGetLastError();
    return known[key] = false;
  }
  return known[key] = ctail_query<T>(nc, smem);
}

template <class T>
bool ctail_query(int nc, long long smem) {
  if (cudaFuncSetAttribute(k_ctail<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
          cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nc);
  cfg.blockDim = dim3(CT);
  cfg.dynamicSmemBytes = (size_t)smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = nc;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int nclusters = 0;
  if (cudaOccupancyMaxActiveClusters(&nclusters, k_ctail<T>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return nclusters >= 1;
}

template <class T>
void launch_ctail(const CTailArgs& a, int nc, long long smem, const T* b_top, T* x_top,
                  cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nc);
  cfg.blockDim = dim3(CT);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = nc;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = g_ssamg_pdl ? 2 : 1;
  SSAMG_CUDA(cudaLaunchKernelEx(&cfg, k_ctail<T>, a, b_top, x_top));
  SSAMG_LAUNCH_CHECK();
}

template bool ctail_prepare<float>(int, long long);
template bool ctail_prepare<double>(int, long long);
template void launch_ctail<float>(const CTailArgs&, int, long long, const float*, float*,
                                  cudaStream_t);
template void launch_ctail<double>(const CTailArgs&, int, long long, const double*, double*,
                                   cudaStream_t);
