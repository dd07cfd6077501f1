// rtm_resident.cu — propagation with the whole grid on chip (sm_103a).
//
// k_resident runs a whole phase (every time step of a forward, backward,
// modelling or Born range) of one item in one launch: a cluster of C blocks
// owns the grid, H rows each.  v^n lives in two shared-memory buffers with a
// 4-row halo; d^n, the update's coefficients and (backward) num and den in the
// registers of the threads that own the points (R rows x 4 columns each).  A
// step reads one buffer and writes v^{n+1} into the other and its first and
// last 4 rows into the neighbour blocks' halos (st.async, counted by their
// mbarriers).  A block waits for its neighbours' rows and for its own threads,
// nothing else, so a step costs its arithmetic and a barrier of one block: no
// launch, no tile halo recomputed, and no field traffic to L2 or HBM (only
// snapshots, traces and data cross it).  The tile kernels' launch of two steps
// takes 6 us or more however small the grid is.
//
// Bound by one step's chain: stencil, store to the neighbours, wait for theirs.
// One shot of 201 x 101, forward: 1.08 us a step, 3.2 with two-step launches (1.6-1.8
// with a cluster barrier a step and plain remote stores, 1.3 with st.async before
// the sponge's products were kept); the shot modelled over 1000 steps 3.24 -> 0.98 ms,
// its migration 7.33 -> 2.35 ms, a 32-item ensemble of it 12.4 -> 4.9 ms.  7 rows a
// thread would take 851 x 176 on chip but spill in the backward phase (5.6-6.6 us
// a step, 2.6-4.8 with tiles).
//
// A neighbour writes a block's halo again only after it has received all 4 rows
// that border it, and those rows are computed from the halo: it is read by then.
//
// Per-point arithmetic, injection order and rounding are those of the other
// propagation kernels (rtm_step2_dev.cuh), so fields, snapshots and images
// agree with theirs bit for bit.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <array>
#include <cmath>
#include <map>
#include <mutex>
#include <type_traits>
#include <vector>

#include "rtm_common.h"
#include "rtm_launch.h"
#include "rtm_step2_dev.cuh"

namespace rtm {

namespace {

using namespace s2;

constexpr int kResThreads[2] = {384, 512};  // of a block at most: two builds
constexpr int kResCluster = 16;   // blocks of a cluster at most

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// release / acquire at cluster scope: orders this block's shared-memory and
// distributed shared-memory writes before the other blocks' next reads
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::
                   : "memory");
}
// shared::cluster address of this block's shared-memory address in block `rank`
__device__ __forceinline__ unsigned remote_smem(unsigned addr, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// 4 points into another block's shared memory, counted by its mbarrier
__device__ __forceinline__ void st_async4(unsigned addr, unsigned bar, const float4 &v) {
  asm volatile(
      "st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, "
      "[%5];" ::"r"(addr),
      "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned long long *bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void st_remote1(unsigned addr, unsigned v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// A stored snapshot of 4 points, as it lies in memory, and its dequantisation.
__device__ __forceinline__ uint4 snap_raw4(const void *base, long long off, int dtype) {
  if (dtype == 0) return __ldg(reinterpret_cast<const uint4 *>(reinterpret_cast<const float *>(base) + off));
  const uint2 u = __ldg(reinterpret_cast<const uint2 *>(reinterpret_cast<const __half *>(base) + off));
  return make_uint4(u.x, u.y, 0u, 0u);
}
__device__ __forceinline__ float4 snap_value4(uint4 u, int dtype, float s) {
  if (dtype == 0)
    return make_float4(__uint_as_float(u.x), __uint_as_float(u.y), __uint_as_float(u.z),
                       __uint_as_float(u.w));
  float2 a, b;
  if (dtype == 2) {
    a = __half22float2(*reinterpret_cast<__half2 *>(&u.x));
    b = __half22float2(*reinterpret_cast<__half2 *>(&u.y));
  } else {
    a = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162 *>(&u.x));
    b = __bfloat1622float2(*reinterpret_cast<__nv_bfloat162 *>(&u.y));
  }
  return make_float4(a.x * s, a.y * s, b.x * s, b.y * s);
}

__device__ __forceinline__ float &el4(float4 &v, int l) {
  return l == 0 ? v.x : (l == 1 ? v.y : (l == 2 ? v.z : v.w));
}

// num += S w, den += S^2
__device__ __forceinline__ void image_add(const float4 &S, const float4 &w, float4 &nu, float4 &de) {
  nu.x = fmaf(S.x, w.x, nu.x);
  nu.y = fmaf(S.y, w.y, nu.y);
  nu.z = fmaf(S.z, w.z, nu.z);
  nu.w = fmaf(S.w, w.w, nu.w);
  de.x = fmaf(S.x, S.x, de.x);
  de.y = fmaf(S.y, S.y, de.y);
  de.z = fmaf(S.z, S.z, de.z);
  de.w = fmaf(S.w, S.w, de.w);
}
// component l (known at run time) by selection: the vector stays in registers
__device__ __forceinline__ void set4(float4 &v, int l, float x) {
  v.x = l == 0 ? x : v.x;
  v.y = l == 1 ? x : v.y;
  v.z = l == 2 ? x : v.z;
  v.w = l == 3 ? x : v.w;
}

}  // namespace

// One update of 4 consecutive points with the sponge's products of the point's
// factor g and c precomputed (constants in time): gc = g c; in the sponge g2 =
// g g, q = (1 - g)(g - 1), m = 0; where g == 1, g2 = q = 0 and m = 1.  Then
//   d' = g2 p + (gc L v + (q v + m p))
// is the sponge form g^2 p + (g c L v + q v) or the interior form c L v + p with
// the roundings of update4 (a product with 0 or 1 and a sum with 0 are exact),
// without computing and selecting between both.
template <bool SPONGE, bool ISO>
__device__ __forceinline__ float4 update4_pre(const float4 *zc, const float4 &xl, const float4 &xr,
                                              const float4 &dv, const float4 &gc, const float4 &g2,
                                              const float4 &q, const float4 &m, const Coef &k) {
  float2 lap[2];
  laplacian4<ISO>(zc, xl, xr, k, lap);
  const float4 ce = zc[4];
  float2 out[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float2 c = h ? make_float2(gc.z, gc.w) : make_float2(gc.x, gc.y);
    const float2 p = h ? make_float2(dv.z, dv.w) : make_float2(dv.x, dv.y);
    if (!SPONGE) {
      out[h] = __ffma2_rn(c, lap[h], p);
    } else {
      const float2 gg = h ? make_float2(g2.z, g2.w) : make_float2(g2.x, g2.y);
      const float2 qq = h ? make_float2(q.z, q.w) : make_float2(q.x, q.y);
      const float2 mm = h ? make_float2(m.z, m.w) : make_float2(m.x, m.y);
      const float2 e = h ? make_float2(ce.z, ce.w) : make_float2(ce.x, ce.y);
      out[h] = __ffma2_rn(gg, p, __ffma2_rn(c, lap[h], __ffma2_rn(qq, e, __fmul2_rn(mm, p))));
    }
  }
  return make_float4(out[0].x, out[0].y, out[1].x, out[1].y);
}

// What stays in registers depends on R: up to 3 rows a thread keep the sponge's
// products (PRE), up to 4 keep num, den and the next snapshot (HOLD); beyond,
// the sponge is evaluated from its factors and num and den go through L2 at
// imaging steps.  T: threads at most, 384 (168 registers each; backward phases of 3,
// 4 and 6 rows spill 120, 96 and 8 bytes) or, for grids that do not fit them, 512
// (128 registers; every phase spills, backward 232 bytes with 5 rows and 500 with 6:
// a 32-item phase of 201 x 101 in 4 blocks takes 2.9-3.7 us a step with 512 threads,
// 2.6-3.2 with 384).
template <int MODE, int R, int T>
__global__ void __launch_bounds__(T, 1) k_resident(const __grid_constant__ ResArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr bool PRE = R <= 3, HOLD = R <= 4;
  constexpr bool SRC = MODE == MODE_FWD || MODE == MODE_MODEL, BWD = MODE == MODE_BWD;
  constexpr bool BORN = MODE == MODE_BORN, IMG = BWD || BORN, REC = MODE == MODE_MODEL || BORN;
  constexpr bool KEEP = HOLD && IMG;  // imaging operands in registers
  const Geo &g = A.g;
  const int H = A.H, NS = A.NS, PV = 4 * (NS + 2);  // rows of a block, strips and floats of a row
  const int G = (H + R - 1) / R, HA = G * R;
  unsigned long long *s_bar = reinterpret_cast<unsigned long long *>(smem_raw);  // [2] by buffer
  unsigned *s_max = reinterpret_cast<unsigned *>(s_bar + 2);  // [2] block max by parity (and 2 of padding)
  unsigned *s_all = s_max + 4;                                // [2][kResCluster] every block's max
  float *vbuf = reinterpret_cast<float *>(s_all + 2 * kResCluster);  // [2][HA + 8][PV]
  const int plane_v = (HA + 8) * PV;
  float *s_gx = vbuf + 2 * plane_v, *s_gz = s_gx + 4 * NS;    // [4 NS], [HA] sponge factors
  float *s_dat = s_gz + ((HA + 3) & ~3);                      // [2][max_ent] data of this block's receivers
  int2 *s_ent = reinterpret_cast<int2 *>(s_dat + 2 * A.max_ent);  // [max_ent]
  const unsigned rank = cluster_rank(), C = A.C;
  const int b = blockIdx.x / C;
  const int tid = threadIdx.x, nth = blockDim.x;
  const int row0 = rank * H, nrow = max(0, min(H, g.NZ - row0));
  const bool has_prev = rank > 0 && nrow > 0, has_next = rank + 1 < C && row0 + H < g.NZ;
  const int smp = RTM_IN(b, A.len.items, A.err) ? A.item_sample[b] : 0;
  const int shot = RTM_IN(b, A.len.items, A.err) ? A.item_shot[b] : 0;
  const float *cc = A.c_all + (long long)smp * g.plane;
  float *gv = A.v + (long long)b * g.plane, *gd = A.d + (long long)b * g.plane;
  // bytes of the neighbours' rows per step: 4 rows of the block before (full),
  // up to 4 of the block after
  const unsigned halo_tx =
      16u * NS * ((has_prev ? 4 : 0) + (has_next ? min(4, g.NZ - row0 - H) : 0));

  // ---- set up: zero fields and halos, barriers, tables, state ----------------
  for (int i = tid; i < plane_v / 2; i += nth)
    reinterpret_cast<float4 *>(vbuf)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int i = tid; i < 4 * NS; i += nth) s_gx[i] = A.gx[i];
  for (int i = tid; i < HA; i += nth) s_gz[i] = A.gz[min(row0 + i, g.NZ - 1)];
  if (tid < 4) s_max[tid] = 0;
  if (tid < 2 * kResCluster) s_all[tid] = 0;
  if (tid == 0) {
    for (int i = 0; i < 2; ++i)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&s_bar[i])), "r"(1) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (halo_tx) {
      mbar_expect(&s_bar[0], halo_tx);
      mbar_expect(&s_bar[1], halo_tx);
    }
  }
  // this block's receivers: entries of rows [row0, row0 + nrow) of the table
  // sorted by row and strip
  int ne = 0;
  if (MODE != MODE_FWD) {
    auto lower = [&](int key) {
      int lo = 0, hi = A.nent;
      while (lo < hi) {
        const int m = (lo + hi) / 2;
        if (A.ent[m].x < key) lo = m + 1;
        else hi = m;
      }
      return lo;
    };
    const int e0 = lower(row0 * NS);
    ne = min(lower((row0 + nrow) * NS) - e0, A.max_ent);
    for (int e = tid; e < ne; e += nth) s_ent[e] = A.ent[e0 + e];
  }
  __syncthreads();
  if (A.load_state) {
    for (int i = tid; i < (nrow + 8) * NS; i += nth) {
      const int r = i / NS, s = i - r * NS, row = row0 - 4 + r;
      if (row >= 0 && row < g.NZ)
        *reinterpret_cast<float4 *>(vbuf + r * PV + 4 + 4 * s) =
            *reinterpret_cast<const float4 *>(gv + (long long)row * g.P + 4 * s);
    }
  }
  // this thread's points: rows lr0 .. lr0 + nr - 1 of R, columns col .. col + 3
  const int q_ = tid / NS, s = tid - q_ * NS, lr0 = q_ * R, col = 4 * s, j0 = col - g.CP;
  const int nr = tid < NS * G ? min(R, nrow - lr0) : 0;
  // its physical rows: bit r set, row i0 + r
  const int i0 = row0 + lr0 - g.nb;
  unsigned pmask = 0;
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (r < nr && j0 >= 0 && j0 < g.SX && i0 + r >= 0 && i0 + r < g.nz) pmask |= 1u << r;
  float4 gc[R], d[R], g2[PRE ? R : 1], gq[PRE ? R : 1], gm[PRE ? R : 1];  // gc: c without PRE
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int x = PRE ? r : 0;
    d[r] = g2[x] = gq[x] = gm[x] = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
    if (r < nr) {
      const long long o = (long long)(row0 + lr0 + r) * g.P + col;
      c = __ldg(reinterpret_cast<const float4 *>(cc + o));
      if (A.load_state) d[r] = *reinterpret_cast<const float4 *>(gd + o);
      if (PRE) {
        const float gz = A.gz[row0 + lr0 + r];
#pragma unroll
        for (int l = 0; l < 4; ++l) {
          const float gg = __fmul_rn(gz, A.gx[col + l]);
          el4(c, l) = __fmul_rn(gg, lane4(c, l));
          if (gg == 1.f) {
            el4(gm[x], l) = 1.f;
          } else {
            el4(g2[x], l) = __fmul_rn(gg, gg);
            el4(gq[x], l) = __fmul_rn(__fmaf_rn(gg, -1.f, 1.f), __fmaf_rn(gg, 1.f, -1.f));
          }
        }
      }
    }
    gc[r] = c;
  }
  // a warp clear of the sponge takes the interior formula
  const bool edge = nr > 0 && (row0 + lr0 < g.nb || row0 + lr0 + R > g.NZ - g.nb ||
                               col < g.X0 + g.nb || col + 4 > g.X0 + g.NX - g.nb);
  const bool sponge = __any_sync(0xffffffffu, edge);
  // a warp that owns rows next to a neighbour block waits for its halo
  const bool border = __any_sync(0xffffffffu, nr > 0 && ((has_prev && lr0 < 4) ||
                                                         (has_next && lr0 + R > H - 4))) ||
                      tid < 32;
  // source cell of this thread: its row (-1: none) and column in the strip
  int src_r = -1, src_l = 0;
  if (SRC && RTM_IN(shot, A.len.nshot, A.err)) {
    const int sr = A.src_row[shot] - row0 - lr0, sc = A.src_col[shot] - col;
    if (sr >= 0 && sr < nr && sc >= 0 && sc < 4) {
      src_r = sr;
      src_l = sc;
    }
  }
  // receivers: rows with some, the first of them and its first entry
  auto first_ent = [&](int r) {
    const int key = (row0 + lr0 + r) * NS + s;
    int lo = 0, hi = ne;
    while (lo < hi) {
      const int m = (lo + hi) / 2;
      if (s_ent[m].x < key) lo = m + 1;
      else hi = m;
    }
    return lo < ne && s_ent[lo].x == key ? lo : -1;
  };
  unsigned rmask = 0;
  int rfirst = 0, rstart = 0;
  if (MODE != MODE_FWD && ne > 0) {
    for (int r = nr - 1; r >= 0; --r) {
      const int e = first_ent(r);
      if (e >= 0) {
        rmask |= 1u << r;
        rfirst = r;
        rstart = e;
      }
    }
  }
  // usually a strip's only receivers are one per column, in order: no loop
  bool rfast = rmask != 0 && (rmask & (rmask - 1u)) == 0 && rstart + 4 <= ne;
  if (rfast) {
    const int key = (row0 + lr0 + rfirst) * NS + s, y = s_ent[rstart].y;
    for (int l = 0; l < 4; ++l) rfast &= s_ent[rstart + l].x == key && s_ent[rstart + l].y == y + 5 * l;
    rfast &= (y & 3) == 0 && !(rstart + 4 < ne && s_ent[rstart + 4].x == key);
  }
  const int rfirst_rec = rfast ? s_ent[rstart].y >> 2 : 0;
  // warps with a source or receivers
  const bool special = __any_sync(0xffffffffu, src_r >= 0 || rmask != 0);
  const int isnap = A.isnap;
  // BWD: k = k_first, k_first - 1, ..; otherwise k = n + 1, n = k_first, ..
  constexpr int step = BWD ? -1 : 1;
  int k = BWD ? A.k_first : A.k_first + 1;
  int to_img = 0x7fffffff;  // steps until the next imaging field (0: this step's output)
  int sidx = 0;             // its snapshot slot
  if (isnap > 0) {
    const int m = k % isnap;
    to_img = BWD ? m : (m ? isnap - m : 0);
    sidx = (k + step * to_img) / isnap - 1 - A.kbase;
  }
  const long long pix0 = (long long)i0 * g.SX + j0;  // this thread's first pixel
  auto fetch = [&](int t, int p) {  // this block's data of sample t into s_dat[p]
    const float *src = A.seis + ((long long)shot * A.nt + t) * A.nrec;
    for (int e = tid; e < ne; e += nth) {
      const int r = s_ent[e].y >> 2;
      if (RTM_IN(r, A.nrec, A.err) && RTM_IN(t, A.nt, A.err))
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_u32(s_dat + p * A.max_ent + e)),
                     "l"(src + r)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  // imaging: num and den (backward) or c m (Born) held for the whole phase, and
  // the snapshot of the next imaging step, loaded one imaging step ahead
  constexpr int KB = KEEP && BWD ? R : 1, KM = KEEP && BORN ? R : 1, KS = KEEP ? R : 1;
  float4 num[KB], den[KB], cm[KM];
  uint4 Sp[KS];
  unsigned Smax = 0;
  auto load_snap = [&](int idx) {
    if (!RTM_IN((long long)b * A.nsnap + idx, A.len.smax, A.err)) return;
    Smax = A.snap_dtype == 0 ? 0u : A.smax[(long long)b * A.nsnap + idx];
    const long long o = ((long long)b * A.nsnap + idx) * g.pplane + pix0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      Sp[KEEP ? r : 0] = make_uint4(0u, 0u, 0u, 0u);
      if (((pmask >> r) & 1u) && RTM_IN(o + (long long)r * g.SX + 3, A.len.snap, A.err))
        Sp[KEEP ? r : 0] = snap_raw4(A.snap, o + r * g.SX, A.snap_dtype);
    }
  };
  const long long pbase = (long long)b * g.pplane + pix0;
  auto refl4 = [&](int r) {  // c m of physical row r (g == 1 there; 0 past the row's end)
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (RTM_IN((long long)(i0 + r) * g.nx + min(j0 + 3, g.nx - 1), A.len.refl, A.err)) {
      const float *m = A.refl + (long long)(i0 + r) * g.nx + j0;
      const float4 c = gc[r];
#pragma unroll
      for (int l = 0; l < 4; ++l)
        if (j0 + l < g.nx) el4(x, l) = __fmul_rn(lane4(c, l), __ldg(m + l));
    }
    return x;
  };
  if (KEEP) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const bool in = (pmask >> r) & 1u;
      if (BWD) {
        float4 &nu = num[KB > 1 ? r : 0], &de = den[KB > 1 ? r : 0];
        nu = de = make_float4(0.f, 0.f, 0.f, 0.f);
        if (in && RTM_IN(pbase + (long long)r * g.SX + 3, A.len.items * g.pplane, A.err)) {
          nu = *reinterpret_cast<const float4 *>(A.num + pbase + r * g.SX);
          de = *reinterpret_cast<const float4 *>(A.den + pbase + r * g.SX);
        }
      }
      if (BORN) cm[KM > 1 ? r : 0] = in ? refl4(r) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (to_img < A.count) load_snap(sidx);
  }
  if (BWD) {
    fetch(k - 1, 0);
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  }
  float wav = SRC && src_r >= 0 ? A.wav[k - 1] : 0.f;
  cluster_sync();  // every block's barriers and halos are set up

  const unsigned v_here = smem_u32(vbuf), bar_here = smem_u32(s_bar);
  const unsigned v_next = has_next ? remote_smem(v_here, rank + 1) : 0u;
  const unsigned v_prev = has_prev ? remote_smem(v_here, rank - 1) : 0u;
  const unsigned b_next = has_next ? remote_smem(bar_here, rank + 1) : 0u;
  const unsigned b_prev = has_prev ? remote_smem(bar_here, rank - 1) : 0u;
  int pending = -1;  // half precision: slot of the input field's snapshot, its max known now
  unsigned pmax = 0;
  float dm = 0.f;     // backward: max(den) behind the last imaging step
  auto ok_img = [&](int r, long long so) {
    return RTM_IN(so + (long long)r * g.SX + 3, A.len.snap, A.err) &&
           RTM_IN(pbase + (long long)r * g.SX + 3, A.len.items * g.pplane, A.err);
  };
  bool dead = false;  // a wait gave up: the flag is raised, the phase runs out unsynchronised

  // quantised store of this thread's part of a field in shared memory
  auto store_snap = [&](const float *v, int idx, unsigned mbits) {
    float sdq, inv;
    snap_scale(A.snap_dtype, mbits, sdq, inv);
    const long long o = ((long long)b * A.nsnap + idx) * g.pplane + pix0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (!((pmask >> r) & 1u)) continue;
      float4 x = *reinterpret_cast<const float4 *>(v + (lr0 + r + 4) * PV + 4 + col);
      if (j0 + 1 >= g.nx) x.y = 0.f;
      if (j0 + 2 >= g.nx) x.z = 0.f;
      if (j0 + 3 >= g.nx) x.w = 0.f;
      if (RTM_IN(o + (long long)r * g.SX + 3, A.len.snap, A.err))
        snap_store4(A.snap, o + r * g.SX, A.snap_dtype, x, inv);
    }
  };

#pragma unroll 1
  for (int it = 0; it < A.count; ++it) {
    const int p = it & 1;
    const float *vin = vbuf + p * plane_v;
    float *vout = vbuf + (p ^ 1) * plane_v;
    const bool img = to_img == 0;  // this step's output is an imaging field
    const int t = k - 1;           // sample injected or recorded
    const bool more = it + 1 < A.count;
    if (it > 0 && halo_tx && border) {  // the neighbours' rows of the input field
      if (!dead && !mbar_wait_bounded(&s_bar[p], ((it - 1) >> 1) & 1, kWaitNs)) {
        dead = true;
        atomicExch(A.err, 1);
      }
      if (tid == 0) mbar_expect(&s_bar[p], halo_tx);
    }
    if (BWD && more) fetch(t - 1, p ^ 1);
    float wav_next = 0.f;
    if (SRC && src_r >= 0 && more) wav_next = A.wav[t + 1];
    if (MODE == MODE_FWD && pending >= 0) {
      store_snap(vin, pending, pmax);
      pending = -1;
    }
    float Ss = 0.f, Sinv;
    if (IMG && !KEEP && img && A.snap_dtype != 0 &&
        RTM_IN((long long)b * A.nsnap + sidx, A.len.smax, A.err))
      Smax = A.smax[(long long)b * A.nsnap + sidx];
    if (IMG && img) snap_scale(A.snap_dtype, Smax, Ss, Sinv);
    float mx = 0.f;
    const long long soff = ((long long)b * A.nsnap + sidx) * g.pplane + pix0;
    // The rows in chunks of RC: within a chunk straight-line code, so that its
    // rows' chains overlap; more rows at once would not leave the registers.
    constexpr int RC = R <= 4 ? R : (R + 1) / 2;
    float4 nvr[R <= 4 ? R : 1];  // v^{n+1} (more rows: read back from vout)
    auto chunk = [&](auto sp, auto iso, auto first) {
      constexpr bool SP = decltype(sp)::value, ISO = decltype(iso)::value;
      constexpr int RA = decltype(first)::value, N = R - RA < RC ? R - RA : RC;
      const float *w = vin + (lr0 + RA) * PV + 4 + col;
      float4 zc[N + 8], xl[N], xr[N], nv[N];
#pragma unroll
      for (int z = 0; z < N + 8; ++z) zc[z] = *reinterpret_cast<const float4 *>(w + z * PV);
#pragma unroll
      for (int i = 0; i < N; ++i) {
        xl[i] = *reinterpret_cast<const float4 *>(w + (i + 4) * PV - 4);
        xr[i] = *reinterpret_cast<const float4 *>(w + (i + 4) * PV + 4);
      }
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const int r = RA + i;
        if constexpr (PRE)
          d[r] = update4_pre<SP, ISO>(&zc[i], xl[i], xr[i], d[r], gc[r], g2[r], gq[r], gm[r], A.k);
        else
          d[r] = update4<SP, ISO>(&zc[i], xl[i], xr[i], d[r], gc[r], A.k, SP ? s_gz[lr0 + r] : 1.f,
                                  s_gx + col);
      }
      if (BORN && img) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
          const int r = RA + i;
          if (((pmask >> r) & 1u) &&
              (KEEP || RTM_IN(soff + (long long)r * g.SX + 3, A.len.snap, A.err))) {
            const float4 S = snap_value4(KEEP ? Sp[KEEP ? r : 0] : snap_raw4(A.snap, soff + r * g.SX, A.snap_dtype),
                                         A.snap_dtype, Ss);
            const float4 m = KEEP ? cm[KM > 1 ? r : 0] : refl4(r);
            d[r].x = fmaf(m.x, S.x, d[r].x);
            if (j0 + 1 < g.nx) d[r].y = fmaf(m.y, S.y, d[r].y);
            if (j0 + 2 < g.nx) d[r].z = fmaf(m.z, S.z, d[r].z);
            if (j0 + 3 < g.nx) d[r].w = fmaf(m.w, S.w, d[r].w);
          }
        }
      }
      if ((SRC || BWD) && special) {
#pragma unroll
        for (int i = 0; i < N; ++i) {
          const int r = RA + i;
          if (SRC && r == src_r)
            set4(d[r], src_l, fmaf(lane4(gc[r], src_l), wav * A.src_scale, lane4(d[r], src_l)));
          if (BWD && ((rmask >> r) & 1u)) {
            const float *dat = s_dat + p * A.max_ent;
            const float4 c = gc[r];
            if (rfast) {
              d[r].x = __fadd_rn(d[r].x, __fmul_rn(c.x, dat[rstart]));
              d[r].y = __fadd_rn(d[r].y, __fmul_rn(c.y, dat[rstart + 1]));
              d[r].z = __fadd_rn(d[r].z, __fmul_rn(c.z, dat[rstart + 2]));
              d[r].w = __fadd_rn(d[r].w, __fmul_rn(c.w, dat[rstart + 3]));
            } else {
              const int e = r == rfirst ? rstart : first_ent(r), key = s_ent[e].x;
              for (int x = e; x < ne && s_ent[x].x == key; ++x) {
                const int l = s_ent[x].y & 3;
                set4(d[r], l, __fadd_rn(lane4(d[r], l), __fmul_rn(lane4(c, l), dat[x])));
              }
            }
          }
        }
      }
      // the rows that border a neighbour go out first
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const int r = RA + i;
        const float4 ce = zc[i + 4];
        nv[i] = make_float4(ce.x + d[r].x, ce.y + d[r].y, ce.z + d[r].z, ce.w + d[r].w);
        if (R <= 4) nvr[R <= 4 ? r : 0] = nv[i];
      }
      if (border && more) {
        const unsigned ro = (unsigned)((p ^ 1) * plane_v + (lr0 + 4) * PV + 4 + col);
#pragma unroll
        for (int i = 0; i < N; ++i) {
          const int r = RA + i;
          if (r < nr && has_next && lr0 + r >= H - 4)
            st_async4(v_next + (ro + (r - H) * PV) * 4, b_next + 8 * (p ^ 1), nv[i]);
          if (r < nr && has_prev && lr0 + r < 4)
            st_async4(v_prev + (ro + (r + H) * PV) * 4, b_prev + 8 * (p ^ 1), nv[i]);
        }
      }
      float *wo = vout + (lr0 + RA + 4) * PV + 4 + col;
#pragma unroll
      for (int i = 0; i < N; ++i)
        if (RA + i < nr) *reinterpret_cast<float4 *>(wo + i * PV) = nv[i];
    };
    auto rows = [&](auto sp, auto iso) {
      chunk(sp, iso, std::integral_constant<int, 0>());
      if constexpr (RC < R) chunk(sp, iso, std::integral_constant<int, RC>());
    };
    if (nr > 0) {
      const std::true_type yes;
      const std::false_type no;
      if (A.k.iso) {
        if (sponge) rows(yes, yes);
        else rows(no, yes);
      } else {
        if (sponge) rows(yes, no);
        else rows(no, no);
      }
    }
    auto value = [&](int r) {  // v^{n+1} of this thread's row r
      return R <= 4 ? nvr[R <= 4 ? r : 0]
                    : *reinterpret_cast<const float4 *>(vout + (lr0 + r + 4) * PV + 4 + col);
    };
    if (REC && special) {
      const long long o = ((long long)b * A.nt + t) * A.nrec;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!((rmask >> r) & 1u)) continue;
        if (rfast) {
          if (RTM_IN(o + rfirst_rec + 3, A.len.rec_out, A.err)) {
            float *out = A.rec_out + o + rfirst_rec;
            const float4 x = value(r);
            out[0] = x.x;
            out[1] = x.y;
            out[2] = x.z;
            out[3] = x.w;
          }
        } else {
          const int e = r == rfirst ? rstart : first_ent(r), key = s_ent[e].x;
          for (int x = e; x < ne && s_ent[x].x == key; ++x)
            if (RTM_IN(o + (s_ent[x].y >> 2), A.len.rec_out, A.err))
              A.rec_out[o + (s_ent[x].y >> 2)] = lane4(value(r), s_ent[x].y & 3);
        }
      }
    }
    if (MODE == MODE_FWD && img && A.store) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if (!((pmask >> r) & 1u)) continue;
        float4 x = value(r);
        if (A.snap_dtype == 0) {
          if (j0 + 1 >= g.nx) x.y = 0.f;
          if (j0 + 2 >= g.nx) x.z = 0.f;
          if (j0 + 3 >= g.nx) x.w = 0.f;
          if (RTM_IN(soff + (long long)r * g.SX + 3, A.len.snap, A.err))
            snap_store4(A.snap, soff + r * g.SX, 0, x, 1.f);
        } else {
#pragma unroll
          for (int l = 0; l < 4; ++l)
            if (j0 + l < g.nx) mx = fmaxf(mx, fabsf(lane4(x, l)));
        }
      }
    }
    if (KEEP && BWD && img) {
#pragma unroll
      for (int r = 0; r < R; ++r)
        image_add(snap_value4(Sp[KEEP ? r : 0], A.snap_dtype, Ss), value(r), num[KB > 1 ? r : 0],
                  den[KB > 1 ? r : 0]);
    }
    if (!KEEP && BWD && img) {  // num and den through L2, two rows' loads in flight at once
#pragma unroll
      for (int r2 = 0; r2 < R; r2 += 2) {
        float4 nu[2], de[2];
        uint4 raw[2];
#pragma unroll
        for (int y = 0; y < 2; ++y)
          if (r2 + y < R && ((pmask >> (r2 + y)) & 1u) && ok_img(r2 + y, soff)) {
            raw[y] = snap_raw4(A.snap, soff + (r2 + y) * g.SX, A.snap_dtype);
            nu[y] = *reinterpret_cast<const float4 *>(A.num + pbase + (r2 + y) * g.SX);
            de[y] = *reinterpret_cast<const float4 *>(A.den + pbase + (r2 + y) * g.SX);
          }
#pragma unroll
        for (int y = 0; y < 2; ++y)
          if (r2 + y < R && ((pmask >> (r2 + y)) & 1u) && ok_img(r2 + y, soff)) {
            image_add(snap_value4(raw[y], A.snap_dtype, Ss), value(r2 + y), nu[y], de[y]);
            *reinterpret_cast<float4 *>(A.num + pbase + (r2 + y) * g.SX) = nu[y];
            *reinterpret_cast<float4 *>(A.den + pbase + (r2 + y) * g.SX) = de[y];
            if (k == isnap) dm = fmaxf(dm, fmaxf(fmaxf(de[y].x, de[y].y), fmaxf(de[y].z, de[y].w)));
          }
      }
    }
    if (KEEP && img && it + isnap < A.count) load_snap(sidx + step);
    // half precision: the max of the imaging field over the cluster
    const bool red = MODE == MODE_FWD && img && A.store && A.snap_dtype != 0;
    if (red) {
#pragma unroll
      for (int o = 16; o; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      // two slots in turn: a block writes a slot again only behind the cluster
      // barrier of the reduction between, when every block has read it
      if ((tid & 31) == 0 && mx > 0.f) atomicMax(&s_max[0], __float_as_uint(mx));
      __syncthreads();
      if (tid < (int)C)
        st_remote1(remote_smem(smem_u32(&s_all[(sidx & 1) * kResCluster + rank]), tid), s_max[0]);
      cluster_sync();
      unsigned m = 0;
      for (int x = 0; x < (int)C; ++x) m = max(m, s_all[(sidx & 1) * kResCluster + x]);
      pmax = m;
      pending = sidx;
      if (tid == 0) {  // (read before the cluster barrier)
        s_max[0] = 0;
        if (rank == 0 && RTM_IN((long long)b * A.nsnap + sidx, A.len.smax, A.err))
          A.smax[(long long)b * A.nsnap + sidx] = m;
      }
    }
    if (BWD && more) asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    if (img) {
      to_img = isnap;
      sidx += step;
    }
    --to_img;
    k += step;
    wav = wav_next;
  }
  const float *vend = vbuf + (A.count & 1) * plane_v;
  if (MODE == MODE_FWD && pending >= 0) store_snap(vend, pending, pmax);
  if (BWD) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (!KEEP || !((pmask >> r) & 1u) || !RTM_IN(pbase + (long long)r * g.SX + 3, A.len.items * g.pplane, A.err))
        continue;
      const float4 de = den[KB > 1 ? r : 0];
      *reinterpret_cast<float4 *>(A.num + pbase + r * g.SX) = num[KB > 1 ? r : 0];
      *reinterpret_cast<float4 *>(A.den + pbase + r * g.SX) = de;
      dm = fmaxf(dm, fmaxf(fmaxf(de.x, de.y), fmaxf(de.z, de.w)));
    }
    if (A.dmax_flag) {
#pragma unroll
      for (int o = 16; o; o >>= 1) dm = fmaxf(dm, __shfl_xor_sync(0xffffffffu, dm, o));
      if ((tid & 31) == 0 && dm > 0.f && RTM_IN(b, A.len.items, A.err))
        atomicMax(&A.dmax[b], __float_as_uint(dm));
    }
  }
  if (A.store_state) {
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (r < nr) {
        const long long o = (long long)(row0 + lr0 + r) * g.P + col;
        *reinterpret_cast<float4 *>(gd + o) = d[r];
        *reinterpret_cast<float4 *>(gv + o) =
            *reinterpret_cast<const float4 *>(vend + (lr0 + r + 4) * PV + 4 + col);
      }
  }
  cluster_sync();  // no block leaves while another may still write into it
}

// ---------------------------------------------------------------- launch --

namespace {

// Shared memory of a block (bytes).
size_t res_smem(const ResPlan &p, int max_ent) {
  const size_t HA = (size_t)p.G * p.R, PV = 4 * (size_t)(p.NS + 2);
  return 4 * (8 + 2 * kResCluster + 2 * (HA + 8) * PV + 4 * (size_t)p.NS + ((HA + 3) & ~(size_t)3) +
              4 * (size_t)max_ent);
}

constexpr size_t kResSmem = 226 << 10;

template <class F>
cudaError_t with_kernel(int mode, const ResPlan &p, F f) {
#define RTM_RES_ROWS(M)                                                             \
  switch (p.R) {                                                                     \
    case 1: return f(k_resident<M, 1, 384>);                                         \
    case 2: return f(k_resident<M, 2, 384>);                                         \
    case 3: return f(k_resident<M, 3, 384>);                                         \
    case 4: return f(k_resident<M, 4, 384>);                                         \
    case 5: return p.threads <= 384 ? f(k_resident<M, 5, 384>) : f(k_resident<M, 5, 512>); \
    case 6: return p.threads <= 384 ? f(k_resident<M, 6, 384>) : f(k_resident<M, 6, 512>); \
  }                                                                                  \
  break;
  switch (mode) {
    case MODE_FWD: RTM_RES_ROWS(MODE_FWD)
    case MODE_MODEL: RTM_RES_ROWS(MODE_MODEL)
    case MODE_BWD: RTM_RES_ROWS(MODE_BWD)
    case MODE_BORN: RTM_RES_ROWS(MODE_BORN)
  }
#undef RTM_RES_ROWS
  return cudaErrorInvalidValue;
}

struct Launch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  Launch(const ResPlan &p, int blocks, size_t smem, cudaStream_t st) {
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)p.threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)p.C;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
  }
};

template <class K>
cudaError_t allow(K kernel) {
  cudaError_t e =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kResSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

}  // namespace

bool resident_shape(const Geo &g, int C, int R, ResPlan &p) {
  p.C = C;
  p.NS = (g.X0 + g.NX + 3) / 4;
  p.H = (g.NZ + C - 1) / C;
  if (C > 1 && p.H < HALO) return false;  // a halo spans one neighbour
  // the fewest rows a thread that fit 384 threads, else (5 rows and more) 512
  bool fits = false;
  for (int t : kResThreads) {
    for (p.R = R > 0 ? R : (t > 384 ? 5 : 1); !fits && p.R <= (R > 0 ? R : kResRows); ++p.R) {
      p.G = (p.H + p.R - 1) / p.R;
      fits = p.NS * p.G <= t && (t <= 384 || p.R >= 5);
      if (fits) break;
    }
    if (fits) break;
  }
  if (!fits) return false;
  p.threads = (p.NS * p.G + 31) / 32 * 32;
  return res_smem(p, 0) <= kResSmem;
}

// The block waits for the thread with the most receivers.  One row of them costs
// little beside the step (a strip's 4 columns in order nothing); otherwise a thread
// takes its entries one by one, about 0.1 us each, and looks up each row but its
// first, 0.2 us and 0.02 a halving of the block's table.  Measured against this
// (added us a step; 201 x 101 with 2 and with 6 rows a thread): four receivers a
// cell 1.8 (1.6), a well 0.5 / 2.0 (0.5 / 1.9), ten rows 1.5 / 5.1 (1.2 / 4.5), every
// cell 3.4 / 7.8, its traces' stores included (1.3 / 4.7).
// Stops at `limit`, where the tile kernels are the faster form.
double resident_receivers_us(const ResPlan &p, const std::vector<ResCell> &cells, double limit) {
  const size_t n = cells.size();
  if (n == 0) return 0.0;
  bool plain = cells[0].row == cells[n - 1].row;  // one row, 4 entries a strip at most
  for (size_t i = 0; plain && i < n; ++i) plain = cells[i].n <= 4;
  if (plain) return 0.0;
  std::vector<float> us(p.NS, 0.f);  // of the strips' threads in the present band of R rows
  std::vector<char> rows(p.NS, 0);
  float search = 0.f, most = 0.f;
  int block = -1, block_end = 0, band_end = 0;  // rows behind the present block and band
  for (size_t i = 0; i < n && most < limit; ++i) {
    const ResCell &c = cells[i];
    if (c.row >= block_end) {  // the block's table: the entries up to the next block
      block = c.row / p.H;
      block_end = (block + 1) * p.H;
      band_end = 0;
      const auto e = std::lower_bound(cells.begin() + i, cells.end(), block_end,
                                      [](const ResCell &a, int x) { return a.row < x; });
      const int last = e == cells.end() ? cells[n - 1].first + cells[n - 1].n : e->first;
      search = 0.2f + 0.02f * std::log2((float)(last - c.first));
    }
    if (c.row >= band_end) {
      band_end = block * p.H + ((c.row - block * p.H) / p.R + 1) * p.R;
      std::fill(us.begin(), us.end(), 0.f);
      std::fill(rows.begin(), rows.end(), 0);
    }
    float &t = us[c.strip];
    char &seen = rows[c.strip];
    if (seen == 0) {
      t = c.fast ? 0.f : 0.1f * c.n;
      seen = c.fast ? 1 : 2;
    } else {
      if (seen == 1) t = 0.4f;  // its first row is not its only one
      t += 0.1f * c.n + search;
      seen = 2;
    }
    most = std::max(most, t);
  }
  return most;
}

// The strips of 4 columns with receivers, in the order of ent (sorted by row and strip).
std::vector<ResCell> resident_cells(const std::vector<int2> &ent, int NS) {
  std::vector<ResCell> cells;
  cells.reserve(ent.size() / 2 + 16);
  int row = 0;
  for (size_t i = 0, k; i < ent.size(); i += k) {
    const int key = ent[i].x;
    bool fast = (ent[i].y & 3) == 0;
    for (k = 1; i + k < ent.size() && ent[i + k].x == key; ++k)
      fast &= ent[i + k].y == ent[i].y + 5 * (int)k;
    while (key >= (row + 1) * NS) ++row;
    cells.push_back({row, key - row * NS, (int)i, (int)k, fast && k == 4});
  }
  return cells;
}

// The receivers of one block at most (for the shared-memory tables).
int resident_max_ent(const ResPlan &p, const std::vector<ResCell> &cells) {
  int most = 0, n = 0, end = 0;  // the last block takes what lies behind it, too
  for (const ResCell &c : cells) {
    if (c.row >= end && end < p.C * p.H) {
      n = 0;
      end = std::min(c.row / p.H + 1, p.C) * p.H;
    }
    n += c.n;
    most = std::max(most, n);
  }
  return most;
}

bool resident_fits(const ResPlan &p, int max_ent) { return res_smem(p, max_ent) <= kResSmem; }

// Clusters of this shape the current device runs at once (0: none); asked of
// the runtime once per shape and device.
int resident_clusters(const ResPlan &p, int max_ent) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  const size_t smem = res_smem(p, max_ent);
  static std::mutex mu;
  static std::map<std::array<int, 5>, int> known;
  const std::array<int, 5> key = {dev, p.C, p.R, p.threads, (int)(smem >> 10)};
  {
    std::lock_guard<std::mutex> lk(mu);
    auto it = known.find(key);
    if (it != known.end()) return it->second;
  }
  int n = 0;
  Launch l(p, p.C, (smem + 1023) & ~(size_t)1023, nullptr);
  // (the backward kernel: the one that takes the most registers)
  const cudaError_t e = with_kernel(MODE_BWD, p, [&](auto kernel) {
    cudaError_t r = allow(kernel);
    return r == cudaSuccess ? cudaOccupancyMaxActiveClusters(&n, kernel, &l.cfg) : r;
  });
  if (e != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  std::lock_guard<std::mutex> lk(mu);
  if (known.size() > 4096) known.clear();
  known[key] = n;
  return n;
}

cudaError_t launch_resident(int mode, const ResPlan &p, ResArgs A, int B, cudaStream_t st) {
  A.C = (unsigned)p.C;
  A.H = p.H;
  A.NS = p.NS;
  if (A.count < 1) return cudaSuccess;
  const size_t smem = res_smem(p, A.max_ent);
  if (smem > kResSmem) return cudaErrorInvalidValue;
  Launch l(p, B * p.C, smem, st);
  return with_kernel(mode, p, [&](auto kernel) {
    const cudaError_t e = allow(kernel);
    return e == cudaSuccess ? cudaLaunchKernelEx(&l.cfg, kernel, A) : e;
  });
}

}  // namespace rtm
