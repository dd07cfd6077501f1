// rtm_eikonal.cu — first-arrival traveltimes on the device: the forward
// operator of the tomography stage (§2.1 Eq. 1: traveltimes from the eikonal
// equation |grad T| = 1/v; §3: one solve per source for every proposed
// velocity model, which dominates that stage's cost).
//
// Discretisation: the first-order upwind scheme on an nz x nx grid (spacings
// dz, dx): with a, b the smaller vertical and horizontal neighbour times,
//     ((T - a)^+ / dz)^2 + ((T - b)^+ / dx)^2 = s^2,  s = 1/v,
// and T = 0 at the source node.  Its discrete solution is unique; fast
// marching reaches it in one ordered pass, and Gauss-Seidel sweeps in the four
// diagonal directions reach it by iterating to a fixed point (Zhao 2005).
//
// Any order of updates in which every node sees each neighbour as the
// sequential row-by-row sweep does (updated in this sweep, or from the
// previous one) gives the sequential sweep's result bit for bit.
//
// k_eik_rows (grids whose tile map fits, about 0.7 M nodes, but not thousands of
// tall ones: row_plan): each lane
// owns R <= 4 consecutive rows, a warp up to 32 R rows, and walks tiles of R x
// 4 nodes along them, one tile behind the lane of the rows before.  A tile's
// neighbours above, below and beside come from the lane's registers and from
// its neighbour lanes by shuffles, so a sweep has no barrier (grids of more
// than 128 rows take several warps, joined every few tiles), and the next tiles'
// fields and slowness load while the current one is updated.  Tiles none of
// whose neighbours changed since their last update are not evaluated again
// (they could not change), and a problem ends once no tile is left to
// evaluate, instead of sweeping once more to find that nothing changes.
//
// k_eik_sweep (the others, and RTM_EIK_TILE): one CTA per problem, tiles on
// one diagonal in parallel, a barrier per diagonal (Detrixhe, Gibou and Min
// 2013).
//
// Either way the field lives in shared memory or in an L2-resident buffer, and
// iterations (four sweeps each) stop at the fixed point, or at a cap.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <type_traits>
#include <vector>

#include "rtm_engine.h"
#include "rtm_launch.h"

namespace {

using u32 = uint32_t;
constexpr float kInf = __builtin_huge_valf();

struct EikArgs {
  const float *slow;     // [nsample][nz][nx] slowness (s/m)
  int nz, nx, nsrc, nrec;
  float dz, dx, wz, wx, wsum, wprod, inv_wsum;  // spacings, 1/dz^2, 1/dx^2, sum, product, 1/sum
  const int *src;        // [nsrc][2] (iz, ix)
  const int *rec;        // [nrec][2]
  float *times;          // [nsample][nsrc][nrec] or null
  float *fields;         // [nsample][nsrc][nz][nx]: output, and the work field off-chip
  int max_iter;
  int *iters;            // [nsample * nsrc] iterations to the fixed point, -1 at the cap
};

// The upwind update from the smaller vertical (a) and horizontal (b)
// neighbour times: one-sided from the smaller one if that does not exceed
// the other, else the larger root of the two-term quadratic.  The root takes
// the hardware reciprocal square root and a multiply by 1/(wz + wx): a few
// ulps per update, far inside the FP32 error of a path of updates.
__device__ __forceinline__ float update(float a, float b, float s, const EikArgs &A) {
  const bool vz = a <= b;
  const float u1 = vz ? a : b, u2 = vz ? b : a;
  const float h1 = vz ? A.dz : A.dx, w1 = vz ? A.wz : A.wx, w2 = vz ? A.wx : A.wz;
  const float t1 = u1 + s * h1;
  if (t1 <= u2) return t1;  // also both neighbours unknown: inf
  const float d = u1 - u2;
  const float disc = fmaxf(A.wsum * (s * s) - A.wprod * (d * d), 1e-30f);
  return (w1 * u1 + w2 * u2 + disc * rsqrtf(disc)) * A.inv_wsum;
}

// One tile of TZ x TX nodes, updated in the sweep's order by one thread: the
// tile and its halo are loaded into registers, the nodes are updated one
// after the other, and the changed values are stored.  Tiles on one tile
// diagonal run in parallel; every node sees each neighbour in the same state
// (updated in this sweep, or from the previous one) as in the sequential
// sweep, so the result is the sequential sweep's, bit for bit.
template <int TZ, int TX, bool FZ, bool FX>
__device__ __forceinline__ bool sweep_tile(float *T, const float *s, int i0, int j0, int nz, int nx,
                                           const EikArgs &A) {
  float t[TZ][TX], sl[TZ][TX], up[TX], dn[TX], lf[TZ], rt[TZ];
#pragma unroll
  for (int r = 0; r < TZ; ++r) {
    const int i = i0 + r;
#pragma unroll
    for (int c = 0; c < TX; ++c) {
      const int j = j0 + c;
      const bool in = i < nz && j < nx;
      const long long k = (long long)i * nx + j;
      t[r][c] = in ? T[k] : kInf;
      sl[r][c] = in ? __ldg(s + k) : 0.f;
    }
    lf[r] = i < nz && j0 > 0 ? T[(long long)i * nx + j0 - 1] : kInf;
    rt[r] = i < nz && j0 + TX < nx ? T[(long long)i * nx + j0 + TX] : kInf;
  }
#pragma unroll
  for (int c = 0; c < TX; ++c) {
    const int j = j0 + c;
    up[c] = j < nx && i0 > 0 ? T[(long long)(i0 - 1) * nx + j] : kInf;
    dn[c] = j < nx && i0 + TZ < nz ? T[(long long)(i0 + TZ) * nx + j] : kInf;
  }
  u32 changed = 0;
#pragma unroll
  for (int rr = 0; rr < TZ; ++rr) {
    const int r = FZ ? rr : TZ - 1 - rr;
#pragma unroll
    for (int cc = 0; cc < TX; ++cc) {
      const int c = FX ? cc : TX - 1 - cc;
      if (i0 + r >= nz || j0 + c >= nx) continue;  // outside the grid: stays infinite
      const float a = fminf(r > 0 ? t[r - 1][c] : up[c], r < TZ - 1 ? t[r + 1][c] : dn[c]);
      const float b = fminf(c > 0 ? t[r][c - 1] : lf[r], c < TX - 1 ? t[r][c + 1] : rt[r]);
      const float v = update(a, b, sl[r][c], A);
      if (v < t[r][c]) {
        t[r][c] = v;
        changed |= 1u << (r * TX + c);
      }
    }
  }
#pragma unroll
  for (int r = 0; r < TZ; ++r)
#pragma unroll
    for (int c = 0; c < TX; ++c)
      if ((changed >> (r * TX + c)) & 1u) T[(long long)(i0 + r) * nx + j0 + c] = t[r][c];
  return changed != 0;
}

template <int TZ, int TX, bool FZ, bool FX>
__device__ __forceinline__ int sweep(float *T, const float *s, const EikArgs &A) {
  const int nz = A.nz, nx = A.nx;
  const int ntz = (nz + TZ - 1) / TZ, ntx = (nx + TX - 1) / TX;
  int changed = 0;
  for (int l = 0; l < ntz + ntx - 1; ++l) {
    const int lo = max(0, l - (ntx - 1)), hi = min(ntz - 1, l);
    for (int ip = lo + (int)threadIdx.x; ip <= hi; ip += blockDim.x) {
      const int jp = l - ip;
      const int ti = FZ ? ip : ntz - 1 - ip, tj = FX ? jp : ntx - 1 - jp;
      changed |= sweep_tile<TZ, TX, FZ, FX>(T, s, ti * TZ, tj * TX, nz, nx, A);
    }
    __syncthreads();
  }
  return changed;
}

template <int TZ, int TX, bool RESIDENT>
__global__ void __launch_bounds__(256, 4) k_eik_sweep(const __grid_constant__ EikArgs A) {
  extern __shared__ float s_T[];
  const int p = blockIdx.x;  // sample * nsrc + source
  const int sample = p / A.nsrc, src = p % A.nsrc;
  const int nz = A.nz, nx = A.nx;
  const long long N = (long long)nz * nx;
  const float *s = A.slow + (long long)sample * N;
  float *T = RESIDENT ? s_T : A.fields + (long long)p * N;
  for (long long k = threadIdx.x; k < N; k += blockDim.x) T[k] = kInf;
  __syncthreads();
  if (threadIdx.x == 0) T[(long long)A.src[2 * src] * nx + A.src[2 * src + 1]] = 0.0f;
  __syncthreads();
  int it = 0;
  bool converged = false;
  for (; it < A.max_iter; ++it) {
    // the four diagonal directions: (+z, +x), (+z, -x), (-z, -x), (-z, +x)
    int changed = sweep<TZ, TX, true, true>(T, s, A);
    changed |= sweep<TZ, TX, true, false>(T, s, A);
    changed |= sweep<TZ, TX, false, false>(T, s, A);
    changed |= sweep<TZ, TX, false, true>(T, s, A);
    if (!__syncthreads_or(changed)) {
      converged = true;
      break;
    }
  }
  if (threadIdx.x == 0) A.iters[p] = converged ? it + 1 : -1;
  if (A.times) {
    float *out = A.times + (long long)p * A.nrec;
    for (int r = threadIdx.x; r < A.nrec; r += blockDim.x)
      out[r] = T[(long long)A.rec[2 * r] * nx + A.rec[2 * r + 1]];
  }
  if (RESIDENT && A.fields) {
    float *out = A.fields + (long long)p * N;
    for (long long k = threadIdx.x; k < N; k += blockDim.x) out[k] = T[k];
  }
}

__global__ void k_eik_slowness(const float *vel, long long n, float *slow) {
  for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < n;
       k += (long long)gridDim.x * blockDim.x)
    slow[k] = __frcp_rn(vel[k]);
}

// ------------------------------------------------- row-owning warps --

// Geometry of k_eik_rows for an nz x nx grid: W warps of lanes that own R rows
// each, NL lanes in all, NC tiles of 4 columns a row.  Every array is padded so
// that a lane ahead of or behind its own tiles reads in bounds (and +inf one
// tile beside the grid), which saves the loop all range checks of its loads.
struct RowGeo {
  int R, W, NL, NC;
  int PB;            // bytes of a lane's row of the tile map: PB - 1 is 4 x odd, so that lanes
                     // one tile apart touch different banks in the sweeps of either family
  int P;             // shared-memory field: floats per row, one tile of +inf on either side (a
                     // multiple of 8: 16-byte accesses of lanes R rows and one tile apart touch
                     // different banks)
  int pad;           // rows of the skewed copies before the first tile
  int rowq;          // float4 of one row of a skewed copy: R x 32 W
  int quads;         // ... and of one copy
  int map_bytes, ring_bytes, field_bytes;  // shared memory: map, warp seams, field
  int map0, field0;  // offsets of tile (0, 0) within the map (bytes) and the field (floats)
};

constexpr int kRowGap = 4;    // tiles between the barriers of a CTA of several warps
constexpr int kRowRing = 16;  // tiles of a seam's ring (> kRowGap + 1 in flight)
constexpr int kRowMap = 64 << 10;  // largest tile map (bytes)
constexpr int kRowMaxWarps = 12;   // of a CTA: 1536 rows
constexpr int kRowWarps = 8;  // resident warps an SM for shared-memory fields to win: row_plan

// False: too large (k_eik_sweep solves it).
bool row_geo(int nz, int nx, RowGeo &g) {
  if ((long long)((nz + 3) / 4) * ((nx + 3) / 4) > kRowMap) return false;
  g.W = (nz + 127) / 128;
  g.R = (nz + 32 * g.W - 1) / (32 * g.W);
  g.NL = (nz + g.R - 1) / g.R;
  g.W = (g.NL + 31) / 32;
  g.NC = (nx + 3) / 4;
  if (g.W > kRowMaxWarps) return false;
  const int lanes = 32 * g.W, slack = lanes + kRowGap * g.W + 4;  // tiles a lane runs past its row
  g.PB = (g.NC + 7) / 8 * 8 + 5;
  g.P = (4 * (g.NC + 2) + 7) / 8 * 8;
  g.pad = kRowGap * (g.W - 1) + 4;
  g.rowq = g.R * lanes;
  const long long quads = (long long)(g.NC + lanes - 1 + 2 * g.pad) * g.rowq;
  const long long map = (long long)lanes * g.PB + 2 * slack;
  const long long field = 4ll * ((long long)lanes * g.R * g.P + 8 * slack + 8);
  if (map > kRowMap || quads > (1 << 28) || field > (1ll << 30)) return false;
  g.quads = (int)quads;
  g.map0 = slack;
  g.map_bytes = (int)((map + 15) / 16 * 16);
  g.ring_bytes = ((g.W - 1) * kRowRing * 20 + 15) / 16 * 16;
  g.field0 = 4 * slack + 4;
  g.field_bytes = (int)((field + 15) / 16 * 16);
  return true;
}

struct RowArgs {
  EikArgs e;
  RowGeo g;
  const float4 *slow_a, *slow_b;  // [nsample][quads] skewed slowness (+inf outside the grid)
  float4 *work;                   // off chip: [problems][2][quads] both skewed copies of T
  int p0, s0;                     // first problem of this launch, first sample of slow_a / slow_b
};

// The two skewed layouts of a grid's tiles: tile (lane g, column c), row r of
// the lane at (pad + c + g) rowq + 32 W r + g (family A) or (pad + c + NL-1-g)
// rowq + 32 W r + g (family B).  The sweeps (+z, +x) and (-z, -x) hold lanes at
// one c + g, the other two at one c - g, so each reads whole lines of its
// family's copy: 4 wavefronts a load instruction instead of 32 from the
// row-major field.  A changed tile is written to both copies.
__global__ void k_eik_skew(const float *vel, int nz, int nx, RowGeo g, float4 *slow_a,
                           float4 *slow_b) {
  const float *v = vel + (long long)blockIdx.y * nz * nx;
  float4 *oa = slow_a + (long long)blockIdx.y * g.quads, *ob = slow_b + (long long)blockIdx.y * g.quads;
  const int lanes = 32 * g.W;
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < g.quads; q += gridDim.x * blockDim.x) {
    const int lane = q % lanes, lr = q / lanes, r = lr % g.R, l = lr / g.R - g.pad;
    const int row = lane * g.R + r;
#pragma unroll
    for (int fam = 0; fam < 2; ++fam) {
      const int c = l - (fam ? g.NL - 1 - lane : lane);
      float s[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const bool in = lane < g.NL && row < nz && c >= 0 && 4 * c + e < nx;
        s[e] = in ? __frcp_rn(v[(long long)row * nx + 4 * c + e]) : kInf;
      }
      (fam ? ob : oa)[q] = make_float4(s[0], s[1], s[2], s[3]);
    }
  }
}

__device__ __forceinline__ float &el(float4 &v, int e) { return reinterpret_cast<float *>(&v)[e]; }

// A problem as its CTA sees it; positions count from tile (0, 0).
struct RowProblem {
  const float4 *sa, *sb;  // slowness
  float4 *ta, *tb;        // off-chip copies of T
  float *st;              // shared-memory T [NL R][P]
  unsigned char *map;     // [NL][PB] 1: the tile has to be evaluated
  float4 *ring;           // [W-1][kRowRing] last rows handed over a seam
  int *ringf;             // [W-1][kRowRing] and whether they changed
};

// update() without branches, for a chain of dependent updates: the expressions
// are the same, so are the bits (the root's argument is at least 1e-30, where
// the flushing reciprocal square root equals the plain one).  ISO: dz == dx and
// wz == wx.
template <bool ISO>
__device__ __forceinline__ float update_flat(float a, float b, float s, const EikArgs &A) {
  const float u1 = fminf(a, b), u2 = fmaxf(a, b);
  float h1 = A.dz, w1 = A.wz, w2 = A.wz;
  if (!ISO) {
    const bool vz = a <= b;
    h1 = vz ? A.dz : A.dx;
    w1 = vz ? A.wz : A.wx;
    w2 = vz ? A.wx : A.wz;
  }
  const float t1 = u1 + s * h1;
  const float d = u1 - u2;
  const float disc = fmaxf(A.wsum * (s * s) - A.wprod * (d * d), 1e-30f);
  float rs;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(rs) : "f"(disc));
  const float two = (w1 * u1 + w2 * u2 + disc * rs) * A.inv_wsum;
  return t1 <= u2 ? t1 : two;
}

// What a sweep leaves for the next ones.
struct RowLeft {
  bool changed = false;  // a node changed
  bool map = true;       // tiles are left to evaluate
  int lo = 0, hi = -1;   // this lane's first and last column with one (one warp only)
};

// One sweep.  FZ / FX: towards +z / +x.  Order and columns below count in the
// sweep's direction.  A problem of one warp (W1) starts at the first tile left
// to evaluate and stops behind the last.
template <int R, bool RES, bool ISO, bool W1, bool FZ, bool FX>
__device__ __forceinline__ void row_sweep(const RowProblem &Q, const RowGeo &g, const EikArgs &A,
                                          RowLeft &B) {
  const int lane = threadIdx.x & 31, warp = W1 ? 0 : threadIdx.x >> 5, gl = threadIdx.x;
  const bool own = gl < g.NL;
  const int NC = own ? g.NC : 0, W = W1 ? 1 : g.W, lanes = 32 * W;
  const int lastlane = min(31, g.NL - 1 - 32 * warp);
  const int seam_in = FZ ? warp - 1 : warp;        // seam to the warp of the rows before
  const int seam_out = FZ ? warp : warp - 1;       // ... and after
  const bool has_in = !W1 && (FZ ? warp > 0 : warp < W - 1);
  const bool has_out = !W1 && (FZ ? warp < W - 1 : warp > 0);
  const bool first = lane == (FZ ? 0 : lastlane), last = lane == (FZ ? lastlane : 0);
  const int ko = FZ ? gl : g.NL - 1 - gl;
  const int start = ko + kRowGap * (FZ ? warp : W - 1 - warp);
  const int lb = FZ ? max(lane - 1, 0) : min(lane + 1, 31);   // lanes before and after
  const int la = FZ ? min(lane + 1, 31) : max(lane - 1, 0);
  constexpr int r0 = FZ ? 0 : R - 1, r1 = FZ ? R - 1 : 0;     // first and last row of a tile
  constexpr bool FA = FZ == FX;                               // family of this sweep
  constexpr int dir = FX ? 1 : -1;
  const int steps = g.NC + g.NL - 1 + kRowGap * (W - 1) + 1;
  // the first step with a tile to evaluate, and the last one known now
  int l0 = 0, l1 = steps;
  if (W1) {
    const bool some = B.hi >= B.lo;
    l0 = __reduce_min_sync(0xffffffffu, some ? start + (FX ? B.lo : NC - 1 - B.hi) : steps);
    l1 = __reduce_max_sync(0xffffffffu, some ? start + (FX ? B.hi : NC - 1 - B.lo) : 0);
  }
  B.lo = g.NC;
  B.hi = -1;
  // this lane's positions at column c0 = l0 - start, advanced tile by tile
  int c = l0 - start;
  const int cp0 = FX ? c : g.NC - 1 - c;
  const int q0 = (cp0 + (FA ? gl : g.NL - 1 - gl)) * g.rowq + gl;
  const int dq = dir * g.rowq;
  const float4 *S = (FA ? Q.sa : Q.sb) + q0;
  const float4 *T = RES ? nullptr : (FA ? Q.ta : Q.tb) + q0;
  float4 *To = RES ? nullptr : (FA ? Q.tb : Q.ta) + (cp0 + (FA ? g.NL - 1 - gl : gl)) * g.rowq + gl;
  float *F = RES ? Q.st + gl * R * g.P + 4 * cp0 : nullptr;
  unsigned char *M = Q.map + gl * g.PB + cp0;
  // (the seam's rows after: the lane after the last one, same column)
  const int g2 = FZ ? gl + 1 : gl - 1;
  const int qb = (cp0 + (FA ? g2 : g.NL - 1 - g2)) * g.rowq + r0 * lanes + g2;
  const float4 *Tb = RES ? nullptr : (FA ? Q.ta : Q.tb) + qb;
  const float *Fb = RES ? Q.st + (g2 * R + r0) * g.P + 4 * cp0 : nullptr;
  auto load_t = [&](int ahead, float4 (&t)[R]) {
#pragma unroll
    for (int r = 0; r < R; ++r)
      t[r] = RES ? *reinterpret_cast<const float4 *>(F + r * g.P + 4 * dir * ahead)
                 : T[ahead * dq + r * lanes];
  };
  auto load_s = [&](int ahead, float4 (&t)[R]) {
#pragma unroll
    for (int r = 0; r < R; ++r) t[r] = __ldg(S + ahead * dq + r * lanes);
  };
  const float4 inf4 = make_float4(kInf, kInf, kInf, kInf);
  auto load_b = [&](int ahead) {
    if (W1 || !has_out || !last) return inf4;
    return RES ? *reinterpret_cast<const float4 *>(Fb + 4 * dir * ahead) : Tb[ahead * dq];
  };

  float4 cur[R], nxt[R], pft[R], sc[R], sn[R], bnx, prev;
  load_t(-1, cur);
  load_t(0, nxt);
  load_t(1, pft);
  load_s(0, sn);
  bnx = load_b(0);
  prev = cur[r1];  // last row of the tile before
  unsigned mnext = M[0];
  bool ch = false, nd = false, any_ch = false, any_map = false;
  unsigned chb = 0;  // lanes that changed in the step before
#pragma unroll 1
  for (int l = l0; l < steps; ++l) {
    const bool in = (unsigned)c < (unsigned)NC;
    float carry[R];  // each row's neighbour behind (updated in this sweep)
#pragma unroll
    for (int r = 0; r < R; ++r) {
      carry[r] = FX ? cur[r].w : cur[r].x;
      cur[r] = nxt[r];
      nxt[r] = pft[r];
      sc[r] = sn[r];
    }
    load_t(2, pft);
    load_s(1, sn);
    const float4 bcur = bnx;
    if (!W1) bnx = load_b(1);
    bool act = in && (mnext || nd);
    mnext = M[dir];
    float4 seam = inf4;
    if (!W1 && has_in && first && in) {
      const int k = seam_in * kRowRing + (c & (kRowRing - 1));
      seam = Q.ring[k];
      act = act || Q.ringf[k];
    }
    const bool pend = ch;
    ch = false;
    if (__any_sync(0xffffffffu, act)) {
      // the tile's neighbours across lanes: the rows before at this column,
      // updated (that lane was here one step ago), and the rows after, old
      float4 bef, aft;
      bef.x = __shfl_sync(0xffffffffu, prev.x, lb);
      bef.y = __shfl_sync(0xffffffffu, prev.y, lb);
      bef.z = __shfl_sync(0xffffffffu, prev.z, lb);
      bef.w = __shfl_sync(0xffffffffu, prev.w, lb);
      aft.x = __shfl_sync(0xffffffffu, nxt[r0].x, la);
      aft.y = __shfl_sync(0xffffffffu, nxt[r0].y, la);
      aft.z = __shfl_sync(0xffffffffu, nxt[r0].z, la);
      aft.w = __shfl_sync(0xffffffffu, nxt[r0].w, la);
      if (first) bef = seam;
      if (last) aft = bcur;
      if (act) {
#pragma unroll
        for (int rr = 0; rr < R; ++rr) {
          const int r = FZ ? rr : R - 1 - rr;
#pragma unroll
          for (int cc = 0; cc < 4; ++cc) {
            const int e = FX ? cc : 3 - cc;
            const float zb = rr > 0 ? el(cur[FZ ? r - 1 : r + 1], e) : el(bef, e);
            const float za = rr < R - 1 ? el(cur[FZ ? r + 1 : r - 1], e) : el(aft, e);
            const float xb = cc > 0 ? el(cur[r], FX ? e - 1 : e + 1) : carry[r];
            const float xa = cc < 3 ? el(cur[r], FX ? e + 1 : e - 1) : (FX ? nxt[r].x : nxt[r].w);
            const float v = update_flat<ISO>(fminf(zb, za), fminf(xb, xa), el(sc[r], e), A);
            ch |= v < el(cur[r], e);
            el(cur[r], e) = fminf(el(cur[r], e), v);
          }
        }
        if (ch) {
#pragma unroll
          for (int r = 0; r < R; ++r) {
            if (RES) {
              *reinterpret_cast<float4 *>(F + r * g.P) = cur[r];
            } else {
              const_cast<float4 *>(T)[r * lanes] = cur[r];
              To[r * lanes] = cur[r];
            }
          }
        }
      }
    }
    prev = cur[r1];
    if (!W1 && has_out && last && in) {  // hand the last row over the seam
      const int k = seam_out * kRowRing + (c & (kRowRing - 1));
      Q.ring[k] = cur[r1];
      Q.ringf[k] = ch;
    }
    // what this step's changes leave to evaluate: the lane before changed its
    // next column (evaluated in this sweep), this lane's next column
    // likewise; the column behind is final for this sweep
    const unsigned chm = __ballot_sync(0xffffffffu, ch);
    const bool ch_b = !first && ((chm >> lb) & 1u), ch_a = !last && ((chm >> la) & 1u);
    nd = ch || ch_b;
    if ((unsigned)(c - 1) < (unsigned)NC) {
      const bool left = pend || ch || ch_a;
      M[-dir] = left;
      any_map |= left;
      if (W1 && left) {
        const int cp = FX ? c - 1 : NC - c;
        B.lo = min(B.lo, cp);
        B.hi = max(B.hi, cp);
      }
    }
    if (!W1 && has_in && first && ch) {  // the rows before passed this column already
      Q.map[(FZ ? gl - 1 : gl + 1) * g.PB + (FX ? c : NC - 1 - c)] = 1;
      any_map = true;
    }
    any_ch |= ch;
    if (!W1) {
      if ((l & (kRowGap - 1)) == kRowGap - 1) __syncthreads();
    } else if (l > l1 && !(chm | chb)) {
      break;
    }
    chb = chm;
    ++c;
    S += dq;
    M += dir;
    if (RES) {
      F += 4 * dir;
      Fb += 4 * dir;
    } else {
      T += dq;
      To += dq;
      Tb += dq;
    }
  }
  if (!W1) {
    B.changed |= __syncthreads_or(any_ch) != 0;
    B.map = __syncthreads_or(any_map) != 0;
  } else {
    __syncwarp();
    B.changed |= __any_sync(0xffffffffu, any_ch) != 0;
    B.map = __any_sync(0xffffffffu, any_map) != 0;
  }
}

// One problem per CTA.  64 models x 34 sources of 426 x 88 (R = 3, one warp,
// fields off chip): 11.2 ms with k_eik_sweep, 2.3 ms here, bound by the fields'
// stream (9.1 GB through L2 and DRAM at 3.6 TB/s) and the latency of its loads,
// 4 to 5 problems a scheduler at 122 registers; ten problems' worth of L2
// prefetch did not help (2.64 -> 2.78 ms), and keeping three tiles in turn
// instead of moving registers costs residency (142 registers, 3.88 ms).  One
// model x 34 sources (fields in shared memory): 4.26 -> 0.85 ms, bound by one
// solve's chain of tile updates.
template <int R, bool RES, bool ISO, bool W1>
__global__ void __launch_bounds__(W1 ? 32 : 32 * kRowMaxWarps) k_eik_rows(const __grid_constant__ RowArgs A) {
  extern __shared__ __align__(16) unsigned char s_raw[];
  const RowGeo &g = A.g;
  const EikArgs &E = A.e;
  const int p = A.p0 + blockIdx.x, sample = p / E.nsrc, src = p % E.nsrc;
  const int tid = threadIdx.x, nth = blockDim.x, lanes = 32 * g.W;
  const float4 inf4 = make_float4(kInf, kInf, kInf, kInf);
  RowProblem Q;
  Q.map = s_raw + g.map0;
  Q.ring = reinterpret_cast<float4 *>(s_raw + g.map_bytes);
  Q.ringf = reinterpret_cast<int *>(Q.ring + (g.W - 1) * kRowRing);
  float *field = reinterpret_cast<float *>(s_raw + g.map_bytes + g.ring_bytes);
  Q.st = field + g.field0;
  const long long s0 = (long long)(sample - A.s0) * g.quads + g.pad * g.rowq;
  Q.sa = A.slow_a + s0;
  Q.sb = A.slow_b + s0;
  float4 *work = RES ? nullptr : A.work + (long long)blockIdx.x * 2 * g.quads;
  Q.ta = RES ? nullptr : work + g.pad * g.rowq;
  Q.tb = RES ? nullptr : Q.ta + g.quads;
  for (int k = tid; k < g.map_bytes / 4; k += nth) reinterpret_cast<unsigned *>(s_raw)[k] = 0;
  if (RES) {
    for (int k = tid; k < g.field_bytes / 16; k += nth) reinterpret_cast<float4 *>(field)[k] = inf4;
  } else {
    for (int k = tid; k < 2 * g.quads; k += nth) work[k] = inf4;
  }
  __syncthreads();
  const int iz = E.src[2 * src], ix = E.src[2 * src + 1];
  const int gs = iz / R, rs = iz - gs * R, cs = ix >> 2;
  if (tid == 0) {
    if (RES) {
      Q.st[iz * g.P + ix] = 0.0f;
    } else {
      reinterpret_cast<float *>(Q.ta + (cs + gs) * g.rowq + rs * lanes + gs)[ix & 3] = 0.0f;
      reinterpret_cast<float *>(Q.tb + (cs + g.NL - 1 - gs) * g.rowq + rs * lanes + gs)[ix & 3] = 0.0f;
    }
    Q.map[gs * g.PB + cs] = 1;
    if (gs > 0) Q.map[(gs - 1) * g.PB + cs] = 1;
    if (gs + 1 < g.NL) Q.map[(gs + 1) * g.PB + cs] = 1;
    if (cs > 0) Q.map[gs * g.PB + cs - 1] = 1;
    if (cs + 1 < g.NC) Q.map[gs * g.PB + cs + 1] = 1;
  }
  __syncthreads();
  // the four diagonal directions: (+z, +x), (+z, -x), (-z, -x), (-z, +x); an
  // iteration that changes nothing ends the solve, and an empty map means
  // that the rest of this iteration and the next one change nothing
  RowLeft B;
  B.lo = tid == gs ? max(cs - 1, 0) : cs;
  B.hi = tid == gs ? min(cs + 1, g.NC - 1) : (abs(tid - gs) == 1 && tid < g.NL ? cs : -1);
  int it = 0;
  bool converged = false;
  for (; it < E.max_iter; ++it) {
    B.changed = false;
    if (B.map) row_sweep<R, RES, ISO, W1, true, true>(Q, g, E, B);
    if (B.map) row_sweep<R, RES, ISO, W1, true, false>(Q, g, E, B);
    if (B.map) row_sweep<R, RES, ISO, W1, false, false>(Q, g, E, B);
    if (B.map) row_sweep<R, RES, ISO, W1, false, true>(Q, g, E, B);
    if (!B.changed) {
      converged = true;
      break;
    }
  }
  if (tid == 0) E.iters[p] = converged ? it + 1 : -1;
  __syncthreads();
  auto value = [&](int i, int j) {
    if (RES) return Q.st[i * g.P + j];
    const int lane = i / R;
    return reinterpret_cast<const float *>(Q.ta + ((j >> 2) + lane) * g.rowq + (i - lane * R) * lanes +
                                           lane)[j & 3];
  };
  if (E.times) {
    float *out = E.times + (long long)p * E.nrec;
    for (int r = tid; r < E.nrec; r += nth) out[r] = value(E.rec[2 * r], E.rec[2 * r + 1]);
  }
  if (E.fields) {
    float *out = E.fields + (long long)p * E.nz * E.nx;
    for (int i = 0; i < E.nz; ++i)
      for (int j = tid; j < E.nx; j += nth) out[(long long)i * E.nx + j] = value(i, j);
  }
}

}  // namespace

namespace rtm {

// Largest field kept in shared memory (bytes).
size_t eik_resident_limit() {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return (size_t)std::max(0, optin - 1024);
}

static EikArgs eik_args(int nz, int nx, double dz, double dx, int nsrc, const int *src, int nrec,
                        const int *rec, int max_iter, float *times, float *fields, int *iters) {
  EikArgs A{};
  A.nz = nz;
  A.nx = nx;
  A.nsrc = nsrc;
  A.nrec = nrec;
  A.dz = (float)dz;
  A.dx = (float)dx;
  A.wz = (float)(1.0 / (dz * dz));
  A.wx = (float)(1.0 / (dx * dx));
  A.wsum = (float)(1.0 / (dz * dz) + 1.0 / (dx * dx));
  A.wprod = (float)(1.0 / (dz * dz * dx * dx));
  A.inv_wsum = (float)(1.0 / (1.0 / (dz * dz) + 1.0 / (dx * dx)));
  A.src = src;
  A.rec = rec;
  A.times = times;
  A.fields = fields;
  A.max_iter = max_iter;
  A.iters = iters;
  return A;
}

// The row-owning solver over all problems.  vel: device.  `work` and `slow`
// hold one group of samples (or, for a sample of many sources, a part of its
// problems) at a time: RowPlan.
struct RowPlan {
  RowGeo g;
  bool resident = false;
  int smem = 0;
  int group = 1;         // samples whose skewed slowness is held at once
  long long chunk = 1;   // problems of one launch
  size_t slow_bytes = 0, work_bytes = 0;
};

// Off-chip fields and slowness stay within about this much scratch, and within
// less where the device has less (rtm_eikonal).
constexpr size_t kRowScratch = size_t(2) << 30;

// Beyond this much of padded off-chip fields in all, tall grids go to k_eik_sweep.
constexpr size_t kRowMost = size_t(4) << 30;

// Where the fields live: in shared memory if every problem is resident at once
// (nothing is gained by more of them an SM), or if 8 warps an SM are, enough to
// hide each other's latencies; else off chip.  Kernel ms, shared / off chip, nodes
// from 1500 to 4500 m/s at random: 152 problems of 88 x 426 3.31 / 3.45, of 176 x
// 176 2.27 / 2.94; 4800 problems of 20 x 40 0.35 / 0.53, of 64 x 64 (about 10 an SM)
// 1.56 / 1.66, of 40 x 100 (fewer than 8) 1.81 / 1.66, of 64 x 200 7.09 / 5.35,
// of 88 x 426 (one an SM) 78.6 / 26.6.
//
// False, too, for many problems of tall grids (unless any_shape): the skewed
// copies pad every tile row by the lanes' offsets (1500 x 40: 50 times its nodes,
// 24 MB a problem), and every sweep streams them, at a cost a quad that grows with
// the warps of a problem, while k_eik_sweep costs about the same a node whatever
// the shape.
// Whole calls, ms, rows / sweeps: while all copies stay within 2 GB the rows win
// everywhere (1500 x 40 x 100: 9.0 / 10.2); beyond 4 GB by pad (quads x 4 / nodes)
// times warps: 600 x 200 x 4800 (27) 45.2 / 60.0, 500 x 100 x 4800 (30) 24.5 / 25.5,
// 400 x 120 x 4800 (32) 21.5 / 22.4, 300 x 60 x 4800 (34) 9.1 / 8.3, 1000 x 300 x
// 1600 (43) 70.8 / 63.3, 400 x 60 x 4800 (59) 18.0 / 11.7, 1000 x 100 x 1600 (113)
// 58.1 / 18.3, 1500 x 40 x 4800 (600) 460 / 33.  Problems of two warps never lose
// (129 x 8 x 4800: 1.37 / 1.75).
static bool row_plan(RowPlan &p, int nz, int nx, int nsample, int nsrc, int flags, int sms,
                     int smem_cta, int smem_sm, size_t scratch, bool any_shape) {
  if (!row_geo(nz, nx, p.g)) return false;
  const RowGeo &g = p.g;
  const int base = g.map_bytes + g.ring_bytes;
  const long long problems = (long long)nsample * nsrc;
  p.resident = false;
  if (!(flags & RTM_EIK_OFFCHIP) && base + g.field_bytes <= smem_cta) {
    const long long per_sm = std::min(32 / g.W, smem_sm / (base + g.field_bytes + 1024));
    p.resident = (flags & RTM_EIK_SHARED) || problems <= per_sm * sms || per_sm * g.W >= kRowWarps;
  }
  // forced into shared memory, but too large with its padding: k_eik_sweep keeps
  // the bare field there
  if ((flags & RTM_EIK_SHARED) && !p.resident && (size_t)nz * nx * 4 <= eik_resident_limit())
    return false;
  p.smem = base + (p.resident ? g.field_bytes : 0);
  const size_t per = 2 * (size_t)g.quads * sizeof(float4);  // both copies
  if (!any_shape && !p.resident && g.W > 2 && (size_t)problems > kRowMost / per &&
      4ll * g.quads * g.W > 33ll * nz * nx)
    return false;
  const size_t per_sample = per + (p.resident ? 0 : per * nsrc);
  p.group = (int)std::max<size_t>(1, std::min<size_t>(nsample, scratch / per_sample));
  p.chunk = (long long)p.group * nsrc;
  if (!p.resident)
    p.chunk = std::max<long long>(1, std::min<long long>(p.chunk, (long long)(scratch / per)));
  p.slow_bytes = per * p.group;
  p.work_bytes = p.resident ? 16 : per * (size_t)p.chunk;
  return true;
}

static cudaError_t launch_eik_rows(const RowPlan &P, const float *vel, int nsample,
                                   const EikArgs &E, float4 *slow, float4 *work, cudaStream_t st) {
  RowArgs A{};
  A.e = E;
  A.g = P.g;
  A.slow_a = slow;
  A.slow_b = slow + (size_t)P.group * P.g.quads;
  A.work = work;
  auto run = [&](auto kernel, unsigned n) -> cudaError_t {
    const cudaError_t e = allow_shared_memory(kernel);
    if (e != cudaSuccess) return e;
    kernel<<<n, 32 * P.g.W, P.smem, st>>>(A);
    return cudaGetLastError();
  };
  // (spacings that only round to the same float differ in their squares)
  const bool iso = E.dz == E.dx && E.wz == E.wx;
  auto go = [&](auto rows, unsigned n) -> cudaError_t {
    constexpr int R = decltype(rows)::value;
    auto one = [&](auto res, auto same) -> cudaError_t {
      constexpr bool RES = decltype(res)::value, ISO = decltype(same)::value;
      return P.g.W == 1 ? run(k_eik_rows<R, RES, ISO, true>, n) : run(k_eik_rows<R, RES, ISO, false>, n);
    };
    const std::true_type yes;
    const std::false_type no;
    if (P.resident) return iso ? one(yes, yes) : one(yes, no);
    return iso ? one(no, yes) : one(no, no);
  };
  for (int s0 = 0; s0 < nsample; s0 += P.group) {
    const int ns = std::min(P.group, nsample - s0);
    const unsigned bx = (unsigned)std::min((P.g.quads + 255) / 256, 1024);
    for (int y0 = 0; y0 < ns; y0 += 65535) {
      const long long at = (long long)y0 * P.g.quads;
      k_eik_skew<<<dim3(bx, std::min(65535, ns - y0)), 256, 0, st>>>(
          vel + (long long)(s0 + y0) * E.nz * E.nx, E.nz, E.nx, P.g, slow + at,
          slow + (long long)P.group * P.g.quads + at);
    }
    A.s0 = s0;
    const long long p1 = (long long)(s0 + ns) * E.nsrc;
    for (long long p0 = (long long)s0 * E.nsrc; p0 < p1; p0 += P.chunk) {
      A.p0 = (int)p0;
      const unsigned n = (unsigned)std::min(P.chunk, p1 - p0);
      cudaError_t e = cudaErrorInvalidValue;
      switch (P.g.R) {
        case 1: e = go(std::integral_constant<int, 1>(), n); break;
        case 2: e = go(std::integral_constant<int, 2>(), n); break;
        case 3: e = go(std::integral_constant<int, 3>(), n); break;
        case 4: e = go(std::integral_constant<int, 4>(), n); break;
      }
      if (e != cudaSuccess) return e;
    }
  }
  return cudaGetLastError();
}

static cudaError_t launch_eikonal(EikArgs A, const float *slow, int nsample, bool resident,
                                  cudaStream_t st) {
  A.slow = slow;
  const int nz = A.nz, nx = A.nx, nsrc = A.nsrc;
  const long long problems = (long long)nsample * nsrc;
  // tile shape: 2 x 2 (a short chain of dependent updates per thread, half
  // the diagonals of single nodes); RTM_EIK_TILE=TZxTX overrides it (one of
  // 1x1 2x2 2x4 4x2), for measurements
  const int shapes[4][2] = {{2, 2}, {1, 1}, {2, 4}, {4, 2}};
  int best = 0;
  if (const char *env = getenv("RTM_EIK_TILE")) {
    for (int q = 0; q < 4; ++q) {
      char name[8];
      snprintf(name, sizeof name, "%dx%d", shapes[q][0], shapes[q][1]);
      if (!strcmp(env, name)) best = q;
    }
  }
  const int tz = shapes[best][0], tx = shapes[best][1];
  const int level = std::min((nz + tz - 1) / tz, (nx + tx - 1) / tx);  // tiles per diagonal
  const int threads = std::min(256, std::max(32, (level + 31) / 32 * 32));
  const size_t smem = resident ? (size_t)nz * nx * 4 : 0;
  auto go = [&](auto kernel) -> cudaError_t {
    if (resident) {
      const cudaError_t e = allow_shared_memory(kernel);
      if (e != cudaSuccess) return e;
    }
    kernel<<<(unsigned)problems, threads, smem, st>>>(A);
    return cudaGetLastError();
  };
  switch (best) {
    case 1: return resident ? go(k_eik_sweep<1, 1, true>) : go(k_eik_sweep<1, 1, false>);
    case 2: return resident ? go(k_eik_sweep<2, 4, true>) : go(k_eik_sweep<2, 4, false>);
    case 3: return resident ? go(k_eik_sweep<4, 2, true>) : go(k_eik_sweep<4, 2, false>);
    default: return resident ? go(k_eik_sweep<2, 2, true>) : go(k_eik_sweep<2, 2, false>);
  }
}

static cudaError_t launch_eik_slowness(const float *vel, long long n, float *slow, cudaStream_t st) {
  const long long blocks = std::min<long long>((n + 255) / 256, 152 * 32);
  k_eik_slowness<<<(unsigned)std::max<long long>(1, blocks), 256, 0, st>>>(vel, n, slow);
  return cudaGetLastError();
}

}  // namespace rtm

// ------------------------------------------------------------------ ABI --

using namespace rtm;

#define EIK_CU(x)                                                                      \
  do {                                                                                 \
    cudaError_t e_ = (x);                                                              \
    if (e_ != cudaSuccess) return fail(ctx, RTM_ERR_CUDA, "%s: %s", #x, cudaGetErrorString(e_)); \
  } while (0)

extern "C" int rtm_eikonal(rtm_ctx *ctx, int nz, int nx, double dz, double dx, int nsample,
                           const float *vel, int nsrc, const int *src_iz, const int *src_ix,
                           int nrec, const int *rec_iz, const int *rec_ix, int max_iter,
                           int flags, float *times, float *fields, int *iters, void *stream) {
  if (!ctx) return RTM_ERR_ARG;
  if (nz < 1 || nx < 1 || !(dz > 0) || !(dx > 0) || !std::isfinite(dz) || !std::isfinite(dx) ||
      nsample < 1 || nsrc < 1 || nrec < 0 || (nrec > 0 && (!rec_iz || !rec_ix)))
    return fail(ctx, RTM_ERR_ARG, "bad eikonal grid or acquisition arguments");
  if (!vel || !src_iz || !src_ix || (!times && !fields))
    return fail(ctx, RTM_ERR_ARG, "vel, sources and one of times / fields are required");
  if (nrec == 0 && times) return fail(ctx, RTM_ERR_ARG, "times needs receivers");
  if ((long long)nz * nx > (1ll << 31) / 4) return fail(ctx, RTM_ERR_ARG, "grid too large");
  for (int k = 0; k < nsrc; ++k)
    if (src_iz[k] < 0 || src_iz[k] >= nz || src_ix[k] < 0 || src_ix[k] >= nx)
      return fail(ctx, RTM_ERR_ARG, "source %d at (%d, %d) is outside the grid", k, src_iz[k],
                  src_ix[k]);
  for (int r = 0; r < nrec; ++r)
    if (rec_iz[r] < 0 || rec_iz[r] >= nz || rec_ix[r] < 0 || rec_ix[r] >= nx)
      return fail(ctx, RTM_ERR_ARG, "receiver %d at (%d, %d) is outside the grid", r, rec_iz[r],
                  rec_ix[r]);
  // the kernels, on either path, count problems in 32 bits
  if ((long long)nsample * nsrc > 0x7fffffffll)
    return fail(ctx, RTM_ERR_ARG, "%d samples x %d sources are more than 2^31 - 1 problems", nsample,
                nsrc);
  if (max_iter <= 0) max_iter = 64;
  if ((flags & ~(RTM_EIK_OFFCHIP | RTM_EIK_SHARED)) || flags == (RTM_EIK_OFFCHIP | RTM_EIK_SHARED))
    return fail(ctx, RTM_ERR_ARG, "bad flags %d", flags);
  if (cudaSetDevice(ctx->device) != cudaSuccess) return fail(ctx, RTM_ERR_CUDA, "cudaSetDevice");
  cudaStream_t st = (cudaStream_t)stream;
  const long long N = (long long)nz * nx, problems = (long long)nsample * nsrc;
  const size_t vbytes = (size_t)nsample * N * 4;
  DevBuf dvel, dslow, dwork, dtab, dtimes, dfields, diters, drng;
  const float *v = vel;
  if (!is_device_ptr(vel)) {
    EIK_CU(dvel.alloc(ctx, vbytes, st));
    EIK_CU(cudaMemcpyAsync(dvel.p, vel, vbytes, cudaMemcpyHostToDevice, st));
    v = dvel.as<float>();
  }
  // velocities must be positive and finite (one synchronisation)
  {
    EIK_CU(drng.alloc(ctx, 16, st));
    const unsigned init[4] = {0u, 0x7f7fffffu, 0u, 0u};
    EIK_CU(cudaMemcpyAsync(drng.p, init, 16, cudaMemcpyHostToDevice, st));
    EIK_CU(launch_vrange(v, (long long)nsample * N, drng.as<unsigned>(), st));
    unsigned out[4];
    EIK_CU(cudaMemcpyAsync(out, drng.p, 16, cudaMemcpyDeviceToHost, st));
    EIK_CU(cudaStreamSynchronize(st));
    if (out[2])
      return fail(ctx, RTM_ERR_ARG, "%u velocity values are non-positive or not finite", out[2]);
  }
  std::vector<int> tab(2 * (size_t)(nsrc + nrec));
  for (int k = 0; k < nsrc; ++k) {
    tab[2 * k] = src_iz[k];
    tab[2 * k + 1] = src_ix[k];
  }
  for (int r = 0; r < nrec; ++r) {
    tab[2 * (nsrc + r)] = rec_iz[r];
    tab[2 * (nsrc + r) + 1] = rec_ix[r];
  }
  EIK_CU(dtab.alloc(ctx, tab.size() * 4, st));
  EIK_CU(cudaMemcpyAsync(dtab.p, tab.data(), tab.size() * 4, cudaMemcpyHostToDevice, st));
  int sms = 0, smem_cta = 0, smem_sm = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device);
  cudaDeviceGetAttribute(&smem_cta, cudaDevAttrMaxSharedMemoryPerBlockOptin, ctx->device);
  cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, ctx->device);
  const bool fits = (size_t)N * 4 <= eik_resident_limit();
  const bool resident = fits && !(flags & RTM_EIK_OFFCHIP) &&
                        ((flags & RTM_EIK_SHARED) || problems <= (long long)sms);
  const size_t tbytes = (size_t)problems * nrec * 4, fbytes = (size_t)problems * N * 4;
  float *dt = times;
  if (times && !is_device_ptr(times)) {
    EIK_CU(dtimes.alloc(ctx, tbytes, st));
    dt = dtimes.as<float>();
  }
  float *df = fields;
  if (fields && !is_device_ptr(fields)) {
    EIK_CU(dfields.alloc(ctx, fbytes, st));
    df = dfields.as<float>();
  }
  EIK_CU(diters.alloc(ctx, (size_t)problems * 4, st));
  // the row-owning solver's scratch; where the device is too full for it, groups of
  // half as many problems, down to one, and then the diagonal sweeps, which need none
  // but the bare fields
  RowPlan plan;
  auto take_rows = [&](bool any_shape) -> bool {
    for (size_t scratch = kRowScratch; !getenv("RTM_EIK_TILE");) {
      if (!row_plan(plan, nz, nx, nsample, nsrc, flags, sms, smem_cta, smem_sm, scratch, any_shape))
        break;
      if (dslow.alloc(ctx, plan.slow_bytes, st) == cudaSuccess &&
          dwork.alloc(ctx, plan.work_bytes, st) == cudaSuccess)
        return true;
      cudaGetLastError();
      dslow.release();
      dwork.release();
      if (plan.group == 1 && (plan.resident || plan.chunk == 1)) break;
      scratch = std::min(scratch, plan.slow_bytes + plan.work_bytes) / 2;
    }
    return false;
  };
  bool rows = take_rows(false);
  if (!rows && !fields && !resident) {  // the off-chip work fields of all problems
    const cudaError_t e = dfields.alloc(ctx, fbytes, st);
    if (e == cudaSuccess) {
      df = dfields.as<float>();
    } else {  // more than the device has: groups of the row-owning solver, whatever the grid
      cudaGetLastError();
      rows = take_rows(true);
      if (!rows) EIK_CU(e);
    }
  }
  if (!rows) {
    EIK_CU(dslow.alloc(ctx, vbytes, st));
    EIK_CU(launch_eik_slowness(v, (long long)nsample * N, dslow.as<float>(), st));
  }
  struct Timer {  // the solver's device time (profiling), released on every path
    cudaEvent_t a = nullptr, b = nullptr;
    ~Timer() {
      if (a) cudaEventDestroy(a);
      if (b) cudaEventDestroy(b);
    }
  } tm;
  if (ctx->prof && cudaEventCreate(&tm.a) == cudaSuccess && cudaEventCreate(&tm.b) == cudaSuccess)
    cudaEventRecord(tm.a, st);
  const cudaEvent_t e0 = tm.b ? tm.a : nullptr, e1 = tm.b;
  const EikArgs E = eik_args(nz, nx, dz, dx, nsrc, dtab.as<int>(), nrec, dtab.as<int>() + 2 * nsrc,
                             max_iter, dt, df, diters.as<int>());
  if (rows)
    EIK_CU(launch_eik_rows(plan, v, nsample, E, dslow.as<float4>(), dwork.as<float4>(), st));
  else
    EIK_CU(launch_eikonal(E, dslow.as<float>(), nsample, resident, st));
  if (e1) cudaEventRecord(e1, st);
  std::vector<int> it((size_t)problems);
  EIK_CU(cudaMemcpyAsync(it.data(), diters.p, (size_t)problems * 4, cudaMemcpyDeviceToHost, st));
  if (times && dt != times) EIK_CU(cudaMemcpyAsync(times, dt, tbytes, cudaMemcpyDeviceToHost, st));
  if (fields && df != fields) EIK_CU(cudaMemcpyAsync(fields, df, fbytes, cudaMemcpyDeviceToHost, st));
  EIK_CU(cudaStreamSynchronize(st));
  long long sweeps = 0, stuck = 0;
  for (int x : it) {
    sweeps += x > 0 ? x : max_iter;
    stuck += x < 0;
  }
  {
    float ms = 0.f;
    if (e0 && cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) ms = 0.f;
    std::lock_guard<std::mutex> lk(ctx->mu);
    ctx->stats.launches += 3;
    if (e0) {
      ctx->stats.eik_launches += 1;
      ctx->stats.eik_ms += ms;
      ctx->stats.eik_updates += 4.0 * (double)sweeps * (double)N;
    }
  }
  if (iters) std::copy(it.begin(), it.end(), iters);
  if (stuck)
    return fail(ctx, RTM_ERR_STATE, "%lld problem(s) did not reach the fixed point in %d iterations",
                stuck, max_iter);
  return RTM_OK;
}
