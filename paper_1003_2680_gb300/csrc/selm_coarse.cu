// Coarse-level engine: the part of the V-cycle (Algorithm 3) below the finest
// level, for one component per thread-block cluster.
//
// Why: on the Galerkin levels the 3x3x5 stencil needs 12 colour classes, so a
// V-cycle runs ~200 dependent colour passes on small grids.  As separate
// launches each pass costs a full launch plus a chain of dependent global
// loads.  Here one cluster per velocity component runs all of them:
//   * "cluster" levels are split into z-slabs, one per CTA; a CTA keeps its
//     slab plus two halo planes on each side in shared memory and, after
//     updating a site that lies in a neighbour's halo, stores the new value
//     into the neighbour's shared memory (DSMEM); cluster barriers separate
//     the colour passes;
//   * "single" levels (small grids) are held entirely by CTA 0, which runs
//     their passes with block barriers while the other CTAs wait at the next
//     cluster barrier;
//   * b, residuals and the hand-off of corrections between levels go through
//     global memory (L2), read with L1-bypassing loads.
// The visiting order (colour classes in increasing id, all sites of a class
// updated together) and the Philox streams are those of the per-pass kernels,
// so both paths produce the same chain.
//
// What bounds it: latency.  A pass is a barrier, a site's 45 shared loads and
// its sum, and about 150 passes follow one another.  So a level's constants
// sit in registers, all of a site's loads are issued before the first sum,
// everything about a site but the values v is loaded off the critical path,
// the normals of a noisy launch are drawn once at its start, and the coarsest
// step is spread over the cluster.  One launch by events, before and after: 48^3
// (levels of 24^3 and below) 152 -> 95 us, noisy 215 -> 112; 64^3 162 -> 127, noisy
// 214 -> 156; 96^3 331 -> 207, noisy 425 -> 273; in FP64 64^2 185 -> 107, noisy
// 403 -> 137, and 48^3 634 -> 408, noisy 1015 -> 493.  Where 64^3's go, noise-free:
// 48 passes of 32^3 at 0.8 us, of 16^3 at 0.7 us, of 8^3 at 0.3 us, the coarsest
// step 5 us, transfers 17 us, staging 5 us.
// The 2-D and 3-D forms are separate kernels: as branches of one kernel their
// code, twice as long, came from L2 anew in every launch (17 us more at 64^3).

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>
#include <type_traits>

#include "../../include/selm_mg.h"
#include "selm_coarse.h"
#include "selm_internal.h"
#include "selm_devmath.h"
#include "selm_pdl.h"
#include "selm_prof.h"

namespace cg = cooperative_groups;

namespace selm {
namespace {

// Threads per CTA.  FP32: 384, so that a thread has 168 registers for the 45
// loads of a row in flight at once (512 threads: 128 registers, spills; a pass
// of an 8^3 level 0.37 instead of 0.31 us).  FP64: 256; a row takes twice the
// registers, and the FP64 pipe (two lanes per clock) is busy with eight warps.
template <typename T>
struct EngThreads {
  static constexpr int value = sizeof(T) == 4 ? 384 : 256;
};

__device__ __forceinline__ uint4 eng_philox10(uint4 c, uint32_t k0, uint32_t k1) { return philox4x32_10(c, k0, k1); }

__device__ __forceinline__ int ewrap(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }

template <typename T>
__device__ __forceinline__ T ld_cg(const T* p) {
  return __ldcg(p);
}

// Position of x in a shared v row: the even x first, then the odd x, so that
// the sites of a colour class (x modulus 2) are consecutive words.
__device__ __forceinline__ int xpos(int i, int half) { return (i & 1) ? half + (i >> 1) : (i >> 1); }

// q = (kr * ny + j) * nx + i  ->  i, j, kr (shifts when nx, ny are powers of two).
template <typename T>
__device__ __forceinline__ void split_xy(const EngLevel<T>& L, int q, int* i, int* j, int* kr) {
  int r;
  if (L.lx >= 0) {
    *i = q & (L.nx - 1);
    r = q >> L.lx;
  } else {
    *i = q % L.nx;
    r = q / L.nx;
  }
  if (L.ly >= 0) {
    *j = r & (L.ny - 1);
    *kr = r >> L.ly;
  } else {
    *j = r % L.ny;
    *kr = r / L.ny;
  }
}

// Per-CTA view of one level.
template <typename T>
struct View {
  const EngLevel<T>* L;
  int z0, z1;          // owned planes [z0, z1)
  T* v;                // local v buffer: planes [z0-2, z1+2), pitches L->rp, L->pp
  int plane;           // nx * ny (sites per plane in the natural field order)
  const T* tab;        // shared: [nz][12] = z bands (10), 1/A_ii, 1/sqrt(A_ii)
  const EngColour* col;  // shared: colour classes of this level for this CTA
  __device__ __forceinline__ int loc(int i, int j, int k) const {
    return (k - z0 + 2) * L->pp + j * L->rp + xpos(i, L->half);
  }
};

template <typename T>
__device__ __forceinline__ View<T> make_view(const EngLevel<T>& L, unsigned char* smem, int rank, bool cluster) {
  View<T> w;
  w.L = &L;
  if (cluster) {
    w.z0 = min(rank * L.P, L.nz);
    w.z1 = min(w.z0 + L.P, L.nz);
  } else {
    w.z0 = 0;
    w.z1 = L.nz;
  }
  w.v = (T*)(smem + L.sv);
  w.plane = L.nx * L.ny;
  w.tab = nullptr;
  w.col = nullptr;
  return w;
}

// q = n / d for 0 <= n < 2^24: float reciprocal estimate, then exact correction.
__device__ __forceinline__ int fdiv(int n, int d, float inv) {
  int q = (int)((float)n * inv);
  if (q * d > n) --q;
  if ((q + 1) * d <= n) ++q;
  return q;
}

// The launch's dynamic shared memory.  What the passes read is addressed by
// element numbers from here (32-bit shared-memory addressing).
template <typename T>
__device__ __forceinline__ T* sm() {
  extern __shared__ __align__(16) unsigned char smem[];
  return reinterpret_cast<T*>(smem);
}
template <typename T>
__device__ __forceinline__ int sm_at(const T* p) {
  return (int)(p - sm<T>());
}

// A level's constants in registers: the passes read them at every site, and
// the compiler cannot keep shared-memory values across the stores of v.
template <typename T>
struct LevReg {
  int nx, ny, mx, my, mz, half, rp, pp, z0, ncol, P;
  int xlast;        // position of x = nx - 1 in a row
  int v;            // plane z0 of the slab (element of sm<T>())
  int tab;          // row tables
  int col;          // colour classes (byte of sm)
  // w1 and w2 at a corner, a y edge, an x edge and the centre of the 3 x 3 window
  T a0, a1, a3, a4, b0, b1, b3, b4;
  __device__ __forceinline__ explicit LevReg(const View<T>& w) {
    const EngLevel<T>& L = *w.L;
    nx = L.nx; ny = L.ny; mx = L.mx; my = L.my; mz = L.mz;
    half = L.half; rp = L.rp; pp = L.pp; z0 = w.z0; ncol = L.ncol; P = L.P;
    xlast = xpos(L.nx - 1, L.half);
    v = sm_at(w.v) + 2 * pp;
    tab = sm_at(w.tab);
    col = (int)(reinterpret_cast<const unsigned char*>(w.col) - sm<unsigned char>());
    a0 = L.w1[0]; a1 = L.w1[1]; a3 = L.w1[3]; a4 = L.w1[4];
    b0 = L.w2[0]; b1 = L.w2[1]; b3 = L.w2[3]; b4 = L.w2[4];
  }
};

// Positions, within a plane of the slab, of the 3 x 3 window around (i, j)
// (D2: the three sites of the one row): index (dy + 1) * 3 + dx + 1.
template <typename T, bool D2>
__device__ __forceinline__ void window_of(const LevReg<T>& R, int i, int j, int c[9]) {
  const int h = i >> 1;
  const int x0 = (i & 1) ? R.half + h : h;
  const int xm = i == 0 ? R.xlast : ((i & 1) ? h : R.half + h - 1);
  const int xp = i == R.nx - 1 ? 0 : ((i & 1) ? h + 1 : R.half + h);
  const int r1 = D2 ? 0 : j * R.rp;
  c[3] = r1 + xm; c[4] = r1 + x0; c[5] = r1 + xp;
  if (!D2) {
    const int r0 = (j == 0 ? R.ny - 1 : j - 1) * R.rp, r2 = (j == R.ny - 1 ? 0 : j + 1) * R.rp;
    c[0] = r0 + xm; c[1] = r0 + x0; c[2] = r0 + xp;
    c[6] = r2 + xm; c[7] = r2 + x0; c[8] = r2 + xp;
  }
}

// The two x-y partial sums w1 . v and w2 . v of one plane (separable form of
// the Galerkin row); CENTRE == false leaves out the site itself.
template <typename T, bool D2, bool CENTRE>
__device__ __forceinline__ void plane_sums(const LevReg<T>& R, int plane, const int c[9], T* s1, T* s2) {
  const T* vp = sm<T>() + plane;
  T p1, p2;
  if (D2) {
    const T a = vp[c[3]], d = vp[c[5]];
    p1 = R.a3 * a + R.a3 * d;
    p2 = R.b3 * a + R.b3 * d;
  } else {
    const T a0 = vp[c[0]], b0 = vp[c[1]], c0 = vp[c[2]];
    const T a1 = vp[c[3]], c1 = vp[c[5]];
    const T a2 = vp[c[6]], b2 = vp[c[7]], c2 = vp[c[8]];
    p1 = R.a0 * a0 + R.a1 * b0 + R.a0 * c0 + R.a3 * a1 + R.a3 * c1 + R.a0 * a2 + R.a1 * b2 +
         R.a0 * c2;
    p2 = R.b0 * a0 + R.b1 * b0 + R.b0 * c0 + R.b3 * a1 + R.b3 * c1 + R.b0 * a2 + R.b1 * b2 +
         R.b0 * c2;
  }
  if (CENTRE) {
    const T b1 = vp[c[4]];
    p1 += R.a4 * b1;
    p2 += R.b4 * b1;
  }
  *s1 = p1;
  *s2 = p2;
}

// Row k of the staged table: 10 z-band entries, 1/A_ii, 1/sqrt(A_ii).
__device__ __forceinline__ void row_table(const float* tab, int k, float t[12]) {
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const float4 a = *reinterpret_cast<const float4*>(tab + 12 * k + 4 * q);
    t[4 * q] = a.x; t[4 * q + 1] = a.y; t[4 * q + 2] = a.z; t[4 * q + 3] = a.w;
  }
}
__device__ __forceinline__ void row_table(const double* tab, int k, double t[12]) {
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const double2 a = *reinterpret_cast<const double2*>(tab + 12 * k + 2 * q);
    t[2 * q] = a.x; t[2 * q + 1] = a.y;
  }
}

// Everything one site's update needs but the values v: its window, its row
// of the table, b and its normal.  None of it depends on the passes before,
// so it is formed between a pass's arrival at the barrier and its release.
template <typename T>
struct Site {
  bool on;
  int kz;          // plane within the slab
  int c[9];
  T row[12], b, n;
};

template <typename T>
struct PassArgs {
  int level, first;            // sweep index of the first pass
  const T* gb;                 // b of the level in global memory, or
  int sb;                      // the owned planes' b (element of sm<T>(), less the first plane's field index)
  bool b_local;
  int noise;                   // normals of every sweep (element of sm<T>()), -1: formed here
  int nstride;                 // normals per sweep
  uint32_t c1;                 // level and component of the noise counter
  Key key;
  unsigned long long cyc;
};

template <typename T, bool NOISE, bool D2>
__device__ __forceinline__ void load_site(const LevReg<T>& R, const PassArgs<T>& A, const EngColour& cc, int q,
                                          int sweep, int s, Site<T>& x) {
  x.on = s < cc.nsite;
  if (!x.on) return;
  const int rk = cc.rank_lo + s;
  int t, ii, kk, jj;
  if (cc.sx >= 0) {
    t = rk >> cc.sx;
    ii = rk & (cc.nxc - 1);
  } else {
    t = fdiv(rk, cc.nxc, cc.inv_nxc);
    ii = rk - t * cc.nxc;
  }
  if (cc.sy >= 0) {
    kk = t >> cc.sy;
    jj = t & (cc.nyc - 1);
  } else {
    kk = fdiv(t, cc.nyc, cc.inv_nyc);
    jj = t - kk * cc.nyc;
  }
  const int i = cc.cx + R.mx * ii, j = cc.cy + R.my * jj, k = cc.cz + R.mz * kk;
  x.kz = k - R.z0;
  const int gidx = (k * R.ny + j) * R.nx + i;
  x.b = A.b_local ? sm<T>()[A.sb + gidx] : ld_cg(A.gb + gidx);
  if (NOISE) {
    if (A.noise >= 0) {
      x.n = sm<T>()[A.noise + sweep * A.nstride + cc.noff + s];
    } else {
      normal_of(eng_philox10(make_uint4((uint32_t)(rk >> 2), A.c1 | ((uint32_t)q << 8) | ((uint32_t)sweep << 12),
                                        (uint32_t)A.cyc, (uint32_t)(A.cyc >> 32)),
                             A.key.k0, A.key.k1),
                rk & 3, &x.n);
    }
  }
  window_of<T, D2>(R, i, j, x.c);
  row_table(sm<T>() + R.tab, k, x.row);
}

// The heat-bath update of a loaded site.  The planes beyond a wall are the
// slab's zeroed halo planes and carry zero band weights.  FP32: the whole
// window is loaded before the first sum, so that its loads share one latency.
template <typename T, bool NOISE, bool D2>
__device__ __forceinline__ T site_value(const LevReg<T>& R, const Site<T>& x) {
  const int vp = R.v + x.kz * R.pp;
  T acc = (T)0;
  if constexpr (sizeof(T) == 4) {
    T f[5][9];
#pragma unroll
    for (int d = 0; d < 5; ++d)
#pragma unroll
      for (int q = D2 ? 3 : 0; q < (D2 ? 6 : 9); ++q) {
        if (d == 2 && q == 4) continue;
        f[d][q] = sm<T>()[vp + (d - 2) * R.pp + x.c[q]];
      }
    asm volatile("" ::: "memory");
#pragma unroll
    for (int d = 0; d < 5; ++d) {
      const T* w = f[d];
      T p1, p2;
      if (D2) {
        p1 = R.a3 * w[3] + R.a3 * w[5];
        p2 = R.b3 * w[3] + R.b3 * w[5];
      } else {
        p1 = R.a0 * w[0] + R.a1 * w[1] + R.a0 * w[2] + R.a3 * w[3] + R.a3 * w[5] + R.a0 * w[6] +
             R.a1 * w[7] + R.a0 * w[8];
        p2 = R.b0 * w[0] + R.b1 * w[1] + R.b0 * w[2] + R.b3 * w[3] + R.b3 * w[5] + R.b0 * w[6] +
             R.b1 * w[7] + R.b0 * w[8];
      }
      if (d != 2) {
        p1 += R.a4 * w[4];
        p2 += R.b4 * w[4];
      }
      acc += x.row[d] * p1 + x.row[5 + d] * p2;
    }
  } else {
#pragma unroll
    for (int dz = -2; dz <= 2; ++dz) {
      T p1, p2;
      if (dz == 0)
        plane_sums<T, D2, false>(R, vp, x.c, &p1, &p2);
      else
        plane_sums<T, D2, true>(R, vp + dz * R.pp, x.c, &p1, &p2);
      acc += x.row[dz + 2] * p1 + x.row[5 + dz + 2] * p2;
    }
  }
  T nv = (x.b - acc) * x.row[10];
  if (NOISE) nv += x.n * x.row[11];
  return nv;
}

// ---- five lanes per site --------------------------------------------------------
// A pass of a small class is latency: one warp alone works through its sites'
// 45 loads and 100 operations.  Five consecutive lanes (six sites per warp)
// each take one plane of the window, exchange the five terms by shuffles and
// add them in the single lane's order.
constexpr int kSplit = 5, kSplitSites = 32 / kSplit;

template <typename T>
struct SplitSite {
  bool on;
  int kz, c[9];
  T z1, z2, rd, rs, b, n;
};

template <typename T, bool NOISE, bool D2>
__device__ __forceinline__ T split_value(const LevReg<T>& R, const SplitSite<T>& x, int d, int lane0) {
  T t = (T)0;
  if (x.on) {
    const int vp = R.v + (x.kz + d - 2) * R.pp;
    T p1, p2;
    plane_sums<T, D2, false>(R, vp, x.c, &p1, &p2);
    if (d != 2) {
      const T b1 = sm<T>()[vp + x.c[4]];
      p1 += R.a4 * b1;
      p2 += R.b4 * b1;
    }
    t = x.z1 * p1 + x.z2 * p2;
  }
  __syncwarp();
  T acc = __shfl_sync(0xffffffffu, t, lane0);
#pragma unroll
  for (int e = 1; e < kSplit; ++e) acc += __shfl_sync(0xffffffffu, t, lane0 + e);
  T nv = (x.b - acc) * x.rd;
  if (NOISE) nv += x.n * x.rs;
  return nv;
}

// Slabs of the CTAs at distance 1 and 2 (null: none, or the slab is empty).
template <typename T>
struct Remote {
  T* v[4];   // rank - 2, - 1, + 1, + 2: their plane z0, expressed from this CTA's plane z0
};

// `count` sweeps of a level: every colour class in turn, a thread (SPLIT: five
// lanes) per site, a barrier after each class.  In the cluster a site within
// two planes of another slab is also stored into that slab's halo.  What does
// not depend on v is loaded off the critical path: when a class fits half of
// the threads, the two halves take alternate passes, and one loads its next
// pass while the other updates; else each thread loads its next site between
// arrival and release of the barrier.  most: sites of the CTA's largest class.
template <typename T, bool NOISE, bool D2, bool SPLIT>
__device__ void sweeps(const View<T>& w, const PassArgs<T>& A, int count, int rank, int csize, bool cluster, int most) {
  const LevReg<T> R(w);
  Remote<T> rem;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int d = q < 2 ? q - 2 : q - 1, r2 = rank + d;
    rem.v[q] = nullptr;
    if (cluster && r2 >= 0 && r2 < csize && min(r2 * R.P, w.L->nz) < min((r2 + 1) * R.P, w.L->nz))
      rem.v[q] = cg::this_cluster().map_shared_rank(sm<T>() + R.v, r2) - (long long)d * R.P * R.pp;
  }
  // whether slab rank + d (q = 0..3: d = -2, -1, 1, 2) holds plane kz in its halo
  auto near = [&](int q, int kz) { return q < 2 ? kz < 2 + (q - 1) * R.P : kz >= (q - 1) * R.P - 2; };
  const int lane = threadIdx.x & 31;
  const int part = SPLIT ? lane % kSplit : 0, lane0 = lane - part;   // SPLIT: this lane's plane
  const bool idle = SPLIT && lane0 + kSplit > 32;                    // (lanes 30 and 31)
  T* push = nullptr;   // SPLIT: lanes 1..4 of a site store into one neighbouring slab each
  if (SPLIT && !idle) push = part == 1 ? rem.v[0] : part == 2 ? rem.v[1] : part == 3 ? rem.v[2] : part == 4 ? rem.v[3] : nullptr;
  using Unit = std::conditional_t<SPLIT, SplitSite<T>, Site<T>>;
  auto load = [&](const EngColour& cc, int q, int sweep, int u, Unit& x) {
    if constexpr (SPLIT) {
      Site<T> y;
      load_site<T, NOISE, D2>(R, A, cc, q, sweep, u, y);
      x.on = y.on;
      if (!y.on) return;
      x.kz = y.kz;
#pragma unroll
      for (int e = 0; e < 9; ++e) x.c[e] = y.c[e];
      const T* tr = sm<T>() + R.tab + 12 * (y.kz + R.z0);
      x.z1 = tr[part];
      x.z2 = tr[5 + part];
      x.rd = tr[10];
      x.rs = tr[11];
      x.b = y.b;
      x.n = y.n;
    } else {
      load_site<T, NOISE, D2>(R, A, cc, q, sweep, u, x);
    }
  };
  auto update = [&](const Unit& x) {
    if constexpr (SPLIT) {   // every lane of the warp comes here
      const T nv = split_value<T, NOISE, D2>(R, x, part, idle ? 0 : lane0);
      if (!x.on) return;
      const int pos = x.kz * R.pp + x.c[4];
      if (part == 0)
        sm<T>()[R.v + pos] = nv;
      else if (push && near(part - 1, x.kz))
        push[pos] = nv;
    } else {
      if (!x.on) return;
      const T nv = site_value<T, NOISE, D2>(R, x);
      const int pos = x.kz * R.pp + x.c[4];
      sm<T>()[R.v + pos] = nv;
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (rem.v[q] && near(q, x.kz)) rem.v[q][pos] = nv;
    }
  };
  // sites that one round of `threads` threads takes
  auto sites_of = [](int threads) { return SPLIT ? (threads >> 5) * kSplitSites : threads; };
  const int half_t = blockDim.x >> 1;
  const bool halves = most <= sites_of(half_t);
  const int tid = halves ? (int)threadIdx.x % half_t : (int)threadIdx.x;
  const int group = halves ? (int)threadIdx.x / half_t : 0;
  const int stride = sites_of(blockDim.x);
  const int me = SPLIT ? (idle ? 1 << 24 : (tid >> 5) * kSplitSites + lane / kSplit) : tid;
  const int npass = count * R.ncol;
  int q = 0, sweep = A.first;   // class and sweep of pass p
  auto colour = [&](int q) { return *reinterpret_cast<const EngColour*>(sm<unsigned char>() + R.col + q * (int)sizeof(EngColour)); };
  EngColour cc = colour(0);
  Unit x;
  x.on = false;
  if (group == 0 && npass > 0) load(cc, 0, sweep, me, x);
  for (int p = 0; p < npass; ++p) {
    const int q1 = q + 1 == R.ncol ? 0 : q + 1, sweep1 = q1 == 0 ? sweep + 1 : sweep;
    if (halves) {
      if ((p & 1) == group) {
        update(x);
      } else if (p + 1 < npass) {
        cc = colour(q1);
        load(cc, q1, sweep1, me, x);
      }
      if (cluster) {
        cg::this_cluster().barrier_arrive();
        cg::this_cluster().barrier_wait();
      } else {
        __syncthreads();
      }
    } else {
      update(x);
      if constexpr (!SPLIT) {   // (a SPLIT class fits one round)
        for (int u = me + stride; u < cc.nsite; u += stride) {
          load(cc, q, sweep, u, x);
          update(x);
        }
      }
      if (cluster) cg::this_cluster().barrier_arrive();
      if (p + 1 < npass) {
        cc = colour(q1);
        load(cc, q1, sweep1, me, x);
      }
      if (cluster)
        cg::this_cluster().barrier_wait();
      else
        __syncthreads();
    }
    q = q1;
    sweep = sweep1;
  }
}

template <typename T, bool NOISE, bool D2>
__device__ __forceinline__ void sweeps_any(const View<T>& w, const PassArgs<T>& A, int count, int rank, int csize,
                                           bool cluster) {
  int most = 0;
  for (int q = 0; q < w.L->ncol; ++q) most = max(most, w.col[q].nsite);
  if constexpr (sizeof(T) == 8) {   // (FP32: a site's row is short work for one lane)
    if (most <= (int)(blockDim.x >> 5) * kSplitSites) {
      sweeps<T, NOISE, D2, true>(w, A, count, rank, csize, cluster, most);
      return;
    }
  }
  sweeps<T, NOISE, D2, false>(w, A, count, rank, csize, cluster, most);
}

template <typename T>
__device__ void zero_local(const View<T>& w) {
  const int n = (w.z1 - w.z0 + 4) * w.L->pp;
  for (int q = threadIdx.x; q < n; q += blockDim.x) w.v[q] = (T)0;
}

// t = b - A v on the owned planes; t written at field index (global or local
// buffer).  A thread takes a column of the slab (one x, y) over a chunk of
// planes: the x-y sums of a plane are formed once and kept for the five rows
// that read them (9 shared loads per site instead of 45).
template <typename T, bool D2>
__device__ void residual(const View<T>& w, const T* b, bool b_local, int boff, T* t) {
  const LevReg<T> R(w);
  const int cols = w.plane, np = w.z1 - w.z0;
  if (np <= 0) return;
  // chunks of planes: as many as give every thread one column
  const int want = max(1, (int)blockDim.x / cols), kc = max((np + want - 1) / want, 1), chunks = (np + kc - 1) / kc;
  for (int q = threadIdx.x; q < cols * chunks; q += blockDim.x) {
    const int chunk = q / cols;
    int i, j, dummy;
    split_xy(*w.L, q - chunk * cols, &i, &j, &dummy);
    const int k0 = chunk * kc, k1 = min(k0 + kc, np);
    int c[9];
    window_of<T, D2>(R, i, j, c);
    T P1[5], P2[5];
#pragma unroll
    for (int d = 0; d < 4; ++d) plane_sums<T, D2, true>(R, R.v + (k0 - 2 + d) * R.pp, c, &P1[d], &P2[d]);
    for (int k = k0; k < k1; ++k) {
      plane_sums<T, D2, true>(R, R.v + (k + 2) * R.pp, c, &P1[4], &P2[4]);
      const int gidx = ((k + R.z0) * R.ny + j) * R.nx + i;
      const T bb = b_local ? b[gidx - boff] : ld_cg(b + gidx);
      T row[12];
      row_table(sm<T>() + R.tab, k + R.z0, row);
      T acc = (T)0;
#pragma unroll
      for (int d = 0; d < 5; ++d) acc += row[d] * P1[d] + row[5 + d] * P2[d];
      t[gidx] = bb - acc;
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        P1[d] = P1[d + 1];
        P2[d] = P2[d + 1];
      }
    }
  }
}

// b_c = P^T t on the coarse planes [Z0, Z1) of level Lc (tables on the fine
// level Lf).  All taps of a site are loaded before they are summed.
template <typename T, bool D2>
__device__ void restrict_to(const EngLevel<T>& Lf, const EngLevel<T>& Lc, const T* t, bool t_local, T* bc, int Z0,
                              int Z1) {
  constexpr int NY = D2 ? 1 : 3;
  const int nx = Lf.nx, ny = Lf.ny, ncx = Lc.nx, ncy = Lc.ny;
  const int n = (Z1 - Z0) * ncx * ncy;
  const int* rz_idx = Lf.rz_idx;
  const T* rz_w = Lf.rz_w;
  for (int q = threadIdx.x; q < n; q += blockDim.x) {
    int I, J, K;
    split_xy(Lc, q, &I, &J, &K);
    K += Z0;
    int col[NY * 3], kr[4];
    T wz[4], x[4][NY * 3];
#pragma unroll
    for (int qy = 0; qy < NY; ++qy) {
      const int row = D2 ? 0 : ewrap(2 * J + qy - 1, ny) * nx;
#pragma unroll
      for (int qx = 0; qx < 3; ++qx) col[qy * 3 + qx] = row + ewrap(2 * I + qx - 1, nx);
    }
#pragma unroll
    for (int qz = 0; qz < 4; ++qz) {
      // an unused tap (index -1) reads row 0 with weight 0: no branch between taps
      kr[qz] = rz_idx[K * 4 + qz];
      wz[qz] = kr[qz] < 0 ? (T)0 : rz_w[K * 4 + qz];
      const T* tp = t + (kr[qz] < 0 ? 0 : kr[qz]) * ny * nx;
#pragma unroll
      for (int c = 0; c < NY * 3; ++c) x[qz][c] = t_local ? tp[col[c]] : ld_cg(tp + col[c]);
    }
    T acc = (T)0;
#pragma unroll
    for (int qz = 0; qz < 4; ++qz)
#pragma unroll
      for (int qy = 0; qy < NY; ++qy) {
        const T wy = D2 || qy == 1 ? (T)1 : (T)0.5;
#pragma unroll
        for (int qx = 0; qx < 3; ++qx) {
          const T wx = qx == 1 ? (T)1 : (T)0.5;
          acc += wz[qz] * wy * wx * x[qz][qy * 3 + qx];
        }
      }
    bc[(K * ncy + J) * ncx + I] = acc;
  }
}

// v_f += P v_c on the local planes [z0-2, z1+2) of the fine view (halo
// included).  A thread takes the pair of fine sites 2 I, 2 I + 1 of a row: the
// even one is the coarse node I in x, the odd one the mean of I and I + 1.
template <typename T, bool D2>
__device__ void prolong_into(const View<T>& w, const EngLevel<T>& Lc, const T* vc, bool vc_local) {
  const EngLevel<T>& L = *w.L;
  const int nx = L.nx, ny = L.ny, rp = L.rp, pp = L.pp, half = L.half, z0 = w.z0;
  const int ncx = Lc.nx, ncy = Lc.ny, crp = Lc.rp, cpp = Lc.pp, chalf = Lc.half;
  const int* pz_idx = L.pz_idx;
  const T* pz_w = L.pz_w;
  const int p0 = max(0, z0 - 2), p1 = min(L.nz, w.z1 + 2);
  const int hx = nx >> 1, n = (p1 - p0) * ny * hx;
  const int lh = L.lx >= 1 ? L.lx - 1 : -1;
  for (int q = threadIdx.x; q < n; q += blockDim.x) {
    const int r = lh >= 0 ? q >> lh : q / hx;
    const int I = lh >= 0 ? q & (hx - 1) : q - r * hx;
    const int kr0 = D2 ? r : (L.ly >= 0 ? r >> L.ly : r / ny);
    const int j = D2 ? 0 : (L.ly >= 0 ? r & (ny - 1) : r - kr0 * ny), k = p0 + kr0;
    const int I1 = I + 1 == ncx ? 0 : I + 1;
    const bool yo = !D2 && (j & 1) != 0;
    const int yi[2] = {D2 ? 0 : j >> 1, yo ? ((j >> 1) + 1 == ncy ? 0 : (j >> 1) + 1) : 0};
    const T yw = yo ? (T)0.5 : (T)1;
    const int xa = vc_local ? xpos(I, chalf) : I, xb = vc_local ? xpos(I1, chalf) : I1;
    T acc0 = (T)0, acc1 = (T)0;
#pragma unroll
    for (int qz = 0; qz < 2; ++qz) {
      // an unused tap reads the row's first tap with weight 0
      const int kr = pz_idx[k * 2 + qz];
      const int kc = kr < 0 ? max(pz_idx[k * 2], 0) : kr;
      const T wz = kr < 0 ? (T)0 : pz_w[k * 2 + qz];
#pragma unroll
      for (int a = 0; a < (D2 ? 1 : 2); ++a) {
        if (a == 1 && !yo) continue;
        const int row = vc_local ? (kc + 2) * cpp + yi[a] * crp : (kc * ncy + yi[a]) * ncx;
        const T u0 = vc_local ? vc[row + xa] : ld_cg(vc + row + xa);
        const T u1 = vc_local ? vc[row + xb] : ld_cg(vc + row + xb);
        acc0 += wz * yw * (T)1 * u0;
        acc1 += wz * yw * (T)0.5 * u0;
        acc1 += wz * yw * (T)0.5 * u1;
      }
    }
    T* out = w.v + (k - z0 + 2) * pp + j * rp + I;
    out[0] += acc0;
    out[half] += acc1;
  }
}

template <typename T>
__device__ void store_owned(const View<T>& w, T* g) {
  const EngLevel<T>& L = *w.L;
  const int n = (w.z1 - w.z0) * w.plane;
  const int base = w.z0 * w.plane;
  for (int q = threadIdx.x; q < n; q += blockDim.x) {
    int i, j, k;
    split_xy(L, q, &i, &j, &k);
    g[base + q] = w.v[w.loc(i, j, w.z0 + k)];
  }
}

// Copies b of the owned planes [z0, z1) (natural order) into shared memory.
template <typename T>
__device__ void load_owned(const View<T>& w, const T* g, T* dst) {
  const int n = (w.z1 - w.z0) * w.plane;
  const T* src = g + w.z0 * w.plane;
  for (int q = threadIdx.x; q < n; q += blockDim.x) dst[q] = ld_cg(src + q);
}

template <typename T>
__device__ void load_all(const View<T>& w, const T* g, T* dst) {
  const int n = (w.z1 - w.z0) * w.plane;
  for (int q = threadIdx.x; q < n; q += blockDim.x) dst[q] = ld_cg(g + q);
}

// Exact coarsest step: v = L^-T (L^-1 b + noise n), FP64.  Each row of L^-1 b
// and each column of L^-T y is a dot product split over eight consecutive
// lanes and reduced with shuffles.  With `spread` the rows (columns) are dealt
// round-robin to the CTAs of the cluster, which take b from CTA 0, exchange y
// and give v to CTA 0 through distributed shared memory (three cluster
// barriers; the last one leaves v complete); else CTA 0 computes them all.
// 216 unknowns (6^3): 27.3 us in CTA 0, 62 us noisy with its normals drawn by
// one lane in eight.  On entry y[r] holds the normals of this CTA's rows.
template <typename T, bool NOISE>
__device__ void coarsest_step(const View<T>& w, T* b, double* y, bool spread, int rank, int csize) {
  const EngLevel<T>& L = *w.L;
  cg::cluster_group cl = cg::this_cluster();
  const int N = L.nx * L.ny * L.nz;
  const int first = spread ? rank : 0, step = spread ? csize : 1;
  constexpr int G = 8;
  const int rows = (N - first + step - 1) / step;
  const int span = (max(rows, 0) * G + 31) / 32 * 32;   // whole warps: every lane reaches the shuffles
  if (spread) {
    cl.sync();   // CTA 0's b is complete
    if (rank != 0) {
      const T* b0 = cl.map_shared_rank(b, 0);
      for (int q = threadIdx.x; q < N; q += blockDim.x) b[q] = b0[q];
      __syncthreads();
    }
  }
  for (int t = threadIdx.x; t < span; t += blockDim.x) {
    const int r = first + t / G * step, g = t % G;
    double acc = 0.0;
    if (r < N)
      for (int q = g; q <= r; q += G) acc += __ldg(L.Linv + (long long)r * N + q) * (double)b[q];
    acc += __shfl_xor_sync(0xffffffffu, acc, 4);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    if (NOISE) {   // the row's lanes take their normal before one of them replaces it
      const double nn = r < N && g == 0 ? y[r] : 0.0;
      acc += __shfl_sync(0xffffffffu, nn, (threadIdx.x & 31) & ~(G - 1));
    }
    if (r < N)
      for (int c = g; c < step; c += G) (spread ? cl.map_shared_rank(y, c) : y)[r] = acc;
  }
  if (spread)
    cl.sync();
  else
    __syncthreads();
  T* v = spread ? cl.map_shared_rank(w.v, 0) : w.v;
  for (int t = threadIdx.x; t < span; t += blockDim.x) {
    const int col = first + t / G * step, g = t % G;
    double acc = 0.0;
    if (col < N)
      for (int r = col + g; r < N; r += G) acc += __ldg(L.Linv + (long long)r * N + col) * y[r];
    acc += __shfl_xor_sync(0xffffffffu, acc, 4);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    if (col < N && g == 0) {
      const int i = col % L.nx, rr = col / L.nx;
      v[w.loc(i, rr % L.ny, rr / L.ny)] = (T)acc;
    }
  }
  if (spread)
    cl.sync();
  else
    __syncthreads();
}

// Fills the colour-class table of the staged level L as seen by the CTA
// owning planes [z0, z1): per class the geometry and the owned rank range.
// (No barrier: the caller syncs.)
template <typename T>
__device__ void stage_colours(const EngLevel<T>& L, int z0, int z1, EngColour* col) {
  for (int q = threadIdx.x; q < L.ncol; q += blockDim.x) {
    EngColour c;
    c.cx = q % L.mx;
    c.cy = (q / L.mx) % L.my;
    c.cz = q / (L.mx * L.my);
    c.nxc = (L.nx - c.cx + L.mx - 1) / L.mx;
    c.nyc = (L.ny - c.cy + L.my - 1) / L.my;
    const int nzc = (L.nz - c.cz + L.mz - 1) / L.mz;
    c.inv_nxc = 1.0f / (float)max(c.nxc, 1);
    c.inv_nyc = 1.0f / (float)max(c.nyc, 1);
    c.sx = (c.nxc > 0 && (c.nxc & (c.nxc - 1)) == 0) ? __ffs(c.nxc) - 1 : -1;
    c.sy = (c.nyc > 0 && (c.nyc & (c.nyc - 1)) == 0) ? __ffs(c.nyc) - 1 : -1;
    int kk_lo = z0 <= c.cz ? 0 : (z0 - c.cz + L.mz - 1) / L.mz;
    int kk_hi = z1 <= c.cz ? 0 : (z1 - c.cz + L.mz - 1) / L.mz;
    kk_hi = min(kk_hi, nzc);
    const int pr = c.nxc * c.nyc;
    c.rank_lo = kk_lo * pr;
    c.nsite = (c.nxc > 0 && c.nyc > 0 && nzc > 0 && kk_hi > kk_lo) ? (kk_hi - kk_lo) * pr : 0;
    c.noff = 0;
    col[q] = c;
  }
}

// The normals of every sweep of the levels that the plan gave a buffer, drawn
// once at the start of the launch by all threads, a whole Philox block at a
// time: a cluster level's by the CTA that owns the planes, CTA 0's levels by
// all CTAs of the cluster (through distributed shared memory; called behind a
// cluster barrier, since a CTA's shared memory may be written only once it
// runs).  The cluster barrier before the first use orders them.  Normal of (sweep, class, rank)
// at [sweep * sites per CTA + the class's offset + rank - its first rank].
template <typename T>
__device__ void stage_noise(const EngParams<T>* P, const EngRun& run, unsigned char* smem, const EngLevel<T>* lev0,
                            const EngColour* col0, int rank, int csize, unsigned long long cyc) {
  const int lt = P->l0, lc = P->L - 1, ns = run.mu1 + run.mu2;
  if (run.coarse_mode == SELM_COARSE_CHOLESKY) {   // the coarsest step's rows of this CTA
    const EngLevel<T>& L = lev0[lc - lt];
    const bool spread = lev0[0].cluster != 0;
    const int N = L.nx * L.ny * L.nz, first = spread ? rank : 0, step = spread ? csize : 1;
    double* y = reinterpret_cast<double*>(smem + P->y_off);
    // from the last thread down: the level normals below start with the first
    for (int t = blockDim.x - 1 - threadIdx.x; first + t * step < N && (spread || rank == 0); t += blockDim.x) {
      const int r = first + t * step;
      normal_of(eng_philox10(make_uint4((uint32_t)(r >> 2), (uint32_t)lc | ((uint32_t)L.comp_id << 4) | (1u << 20),
                                        (uint32_t)cyc, (uint32_t)(cyc >> 32)),
                             run.key.k0, run.key.k1),
                r & 3, y + r);
    }
  }
  for (int l = lt; l <= lc; ++l) {
    if (P->nz_off[l] < 0 || (l == lc && run.coarse_mode == SELM_COARSE_CHOLESKY)) continue;
    const EngLevel<T>& L = lev0[l - lt];
    const EngColour* col = col0 + (size_t)(l - lt) * kEngMaxColours;
    const bool own = L.cluster != 0;
    T* dst = reinterpret_cast<T*>(smem + P->nz_off[l]);
    if (!own && csize > 1) dst = cg::this_cluster().map_shared_rank(dst, 0);
    const int stride = L.P * L.nx * L.ny, ncol = L.ncol;
    int gmax = 0;   // noise groups of the largest class
    for (int q = 0; q < ncol; ++q)
      if (col[q].nsite > 0) gmax = max(gmax, ((col[q].rank_lo + col[q].nsite - 1) >> 2) - (col[q].rank_lo >> 2) + 1);
    const int total = ns * ncol * gmax;
    const int first = own ? threadIdx.x : rank * blockDim.x + threadIdx.x;
    const int step = own ? blockDim.x : csize * blockDim.x;
    for (int t = first; t < total; t += step) {
      const int u = t / gmax, sweep = u / ncol, q = u - sweep * ncol;
      const EngColour& c = col[q];
      const int g = (c.rank_lo >> 2) + t - u * gmax;
      if (c.nsite <= 0 || 4 * g >= c.rank_lo + c.nsite) continue;
      T n4[4];
      Normals<T>::get(eng_philox10(make_uint4((uint32_t)g,
                                              (uint32_t)l | ((uint32_t)L.comp_id << 4) | ((uint32_t)q << 8) |
                                                  ((uint32_t)sweep << 12),
                                              (uint32_t)cyc, (uint32_t)(cyc >> 32)),
                                   run.key.k0, run.key.k1),
                      n4);
      T* out = dst + (size_t)sweep * stride + c.noff;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int s = 4 * g + e - c.rank_lo;
        if (s >= 0 && s < c.nsite) out[s] = n4[e];
      }
    }
  }
}

template <typename T, bool NOISE, bool D2>
__global__ void __launch_bounds__(EngThreads<T>::value, 1) k_coarse_engine(const EngParams<T>* __restrict__ P, EngRun run) {
  extern __shared__ __align__(16) unsigned char smem[];
  cg::cluster_group cl = cg::this_cluster();
  const int csize = (int)cl.num_blocks();
  const int rank = (int)cl.block_rank();
  // stage_noise() stores into CTA 0's shared memory: every CTA of the cluster
  // has to run before the first store (the wait stands in front of it)
  if (NOISE && csize > 1) cl.barrier_arrive();
  const int comp = blockIdx.x / csize;
  const EngComp<T>* E = &P->comp[comp];
  const unsigned long long cyc = *run.cyc;
  const int lt = P->l0, lc = P->L - 1;
  const int mu1 = run.mu1, mu2 = run.mu2;
  const Key key = run.key;
  EngLevel<T>* const lev0 = reinterpret_cast<EngLevel<T>*>(smem + P->lev_off);   // levels lt..lc
  EngColour* const col0 = reinterpret_cast<EngColour*>(smem + P->col_off);
  T* const stab = reinterpret_cast<T*>(smem + P->tab_off);
  auto sl_at = [&](int l) -> EngLevel<T>& { return lev0[l - lt]; };
  auto col_at = [&](int l) { return col0 + (size_t)(l - lt) * kEngMaxColours; };

  // ---- stage every level once: descriptors, then colour classes and row tables ----
  {
    constexpr int n = (int)(sizeof(EngLevel<T>) / sizeof(int));
    const int total = (lc - lt + 1) * n;
    for (int q = threadIdx.x; q < total; q += blockDim.x) {
      const int l = lt + q / n, e = q - (q / n) * n;
      reinterpret_cast<int*>(&sl_at(l))[e] = reinterpret_cast<const int*>(&E->lev[l])[e];
    }
    __syncthreads();
    for (int l = lt; l <= lc; ++l) {
      const EngLevel<T>& L = sl_at(l);
      const View<T> w = make_view(L, smem, rank, L.cluster != 0);
      stage_colours(L, w.z0, w.z1, col_at(l));
    }
    // Row tables (per row k of each level: the z bands, 1/A_ii, 1/sqrt(A_ii))
    // and transfer tables (prolongation and restriction taps along z) of all
    // levels as one list of entries.  Each thread issues the global loads of
    // up to kStageUnroll entries before it stores any of them, so the list
    // costs about one memory latency instead of one per level and table.
    {
      // entries of level l: 12 nz row-table words, then (below the coarsest
      // level) 2 nz prolongation taps and 4 nz_c restriction taps
      auto level_entries = [&](int l) {
        const EngLevel<T>& L = sl_at(l);
        return 12 * L.nz + (l < lc ? 2 * L.nz + 4 * sl_at(l + 1).nz : 0);
      };
      int total = 0;
      for (int l = lt; l <= lc; ++l) total += level_entries(l);
      constexpr int kStageUnroll = 4;
      for (int base = threadIdx.x; base < total; base += kStageUnroll * blockDim.x) {
        T val[kStageUnroll];
        int ival[kStageUnroll], kind[kStageUnroll], lev[kStageUnroll], pos[kStageUnroll];
#pragma unroll
        for (int u = 0; u < kStageUnroll; ++u) {
          int q = base + u * (int)blockDim.x;
          kind[u] = -1;
          if (q >= total) continue;
          int l = lt;
          while (q >= level_entries(l)) {
            q -= level_entries(l);
            ++l;
          }
          const EngLevel<T>& L = sl_at(l);
          lev[u] = l;
          pos[u] = q;
          if (q < 12 * L.nz) {   // row table: band, or the diagonal (inverted below)
            const int k = q / 12, e = q - k * 12;
            kind[u] = e < 10 ? 0 : e == 10 ? 1 : 2;
            val[u] = e < 10 ? L.zb[k * 10 + e] : L.S[(long long)k * kStencil + 22];
          } else {   // transfer tap, at its slot of the level's transfer rows
            const int t = q - 12 * L.nz;
            kind[u] = 3;
            pos[u] = t;
            if (t < 2 * L.nz) {
              ival[u] = L.pz_idx[t];
              val[u] = L.pz_w[t];
            } else {
              ival[u] = L.rz_idx[t - 2 * L.nz];
              val[u] = L.rz_w[t - 2 * L.nz];
            }
          }
        }
#pragma unroll
        for (int u = 0; u < kStageUnroll; ++u) {
          if (kind[u] < 0) continue;
          const int l = lev[u];
          if (kind[u] < 3) {
            const T v = val[u];
            stab[(size_t)P->tab_row[l] * 12 + pos[u]] =
                kind[u] == 0 ? v : kind[u] == 1 ? (T)1 / v : (T)1 / tsqrt(v);
          } else {
            reinterpret_cast<int*>(smem + P->xfi_off)[P->xf_row[l] + pos[u]] = ival[u];
            reinterpret_cast<T*>(smem + P->xfw_off)[P->xf_row[l] + pos[u]] = val[u];
          }
        }
      }
    }
    __syncthreads();
    if (threadIdx.x >= 32 && threadIdx.x <= 32 + lc - lt) {   // offset of each class in the level's normals
      const int l = lt + threadIdx.x - 32;
      int off = 0;
      for (int q = 0; q < sl_at(l).ncol; ++q) {
        col_at(l)[q].noff = off;
        off += col_at(l)[q].nsite;
      }
    }
    if (threadIdx.x == 0)
      for (int l = lt; l < lc; ++l) {
        EngLevel<T>& L = sl_at(l);
        int* xi = reinterpret_cast<int*>(smem + P->xfi_off) + P->xf_row[l];
        T* xw = reinterpret_cast<T*>(smem + P->xfw_off) + P->xf_row[l];
        L.pz_idx = xi;
        L.pz_w = xw;
        L.rz_idx = xi + 2 * L.nz;
        L.rz_w = xw + 2 * L.nz;
      }
    __syncthreads();
  }
  auto view_of = [&](int l, bool cluster) {
    View<T> w = make_view(sl_at(l), smem, rank, cluster);
    w.tab = stab + (size_t)P->tab_row[l] * 12;
    w.col = col_at(l);
    return w;
  };
  if (NOISE) {
    if (csize > 1) cl.barrier_wait();
    stage_noise<T>(P, run, smem, lev0, col0, rank, csize, cyc);
  }
  // the sweeps of level l from sweep index `first`, with b in shared memory
  // (blocal) or read from L2
  auto pass_args = [&](int l, int first, const T* b, bool blocal, int boff) {
    const EngLevel<T>& L = sl_at(l);
    PassArgs<T> A;
    A.level = l;
    A.first = first;
    A.gb = L.gb;
    A.b_local = blocal;
    A.sb = blocal ? sm_at(b) - boff : 0;
    A.noise = NOISE && P->nz_off[l] >= 0 ? P->nz_off[l] / (int)sizeof(T) : -1;
    A.nstride = L.P * L.nx * L.ny;
    A.c1 = (uint32_t)l | ((uint32_t)L.comp_id << 4);
    A.key = key;
    A.cyc = cyc;
    return A;
  };

  for (int l = lt; l <= lc; ++l) zero_local(make_view(sl_at(l), smem, rank, sl_at(l).cluster != 0));
  pdl_wait();   // everything above reads only the plan and the counter
  // ---- down leg over the cluster levels ----
  int l = lt;
  for (; l < lc && sl_at(l).cluster; ++l) {
    const EngLevel<T>& L = sl_at(l);
    const EngLevel<T>& Lc = sl_at(l + 1);
    View<T> w = view_of(l, true);
    // b of the owned planes in shared memory when the plan has room for it
    const bool bl = L.sb >= 0;
    const T* bsrc = bl ? (const T*)(smem + L.sb) : L.gb;
    const int boff = bl ? w.z0 * w.plane : 0;
    if (bl) load_owned(w, L.gb, (T*)(smem + L.sb));
    cl.sync();
    sweeps_any<T, NOISE, D2>(w, pass_args(l, 0, bsrc, bl, boff), mu1, rank, csize, true);
    residual<T, D2>(w, bsrc, bl, boff, L.gt);
    cl.sync();
    // the coarse planes of the restriction are split over the cluster's CTAs
    // (also when the coarse level is held by CTA 0: it reads them back)
    const int Pc = (Lc.nz + csize - 1) / csize;
    const int Z0 = min(rank * Pc, Lc.nz);
    const int Z1 = min(Z0 + Pc, Lc.nz);
    // into the first level held by CTA 0: its shared b, through distributed shared memory
    T* bdst = Lc.cluster ? Lc.gb : cl.map_shared_rank(reinterpret_cast<T*>(smem + Lc.sb), 0);
    restrict_to<T, D2>(L, Lc, L.gt, false, bdst, Z0, Z1);
    cl.sync();
  }
  const int lsingle = l;   // first level held by CTA 0 alone
  if (lsingle == lt && csize > 1) {
    // no cluster level: the other CTAs were here for the normals only
    cl.sync();
    if (rank != 0) return;
  }
  // the coarsest step is spread over the cluster: the other CTAs wait in it
  const bool spread = lsingle > lt && run.coarse_mode == SELM_COARSE_CHOLESKY;
  if (spread && rank != 0)
    coarsest_step<T, NOISE>(view_of(lc, false), (T*)(smem + sl_at(lc).sb), (double*)(smem + P->y_off), true, rank,
                            csize);
  if (rank == 0) {
    // ---- single-CTA part: levels lsingle .. lc and back ----
    if (lsingle == lt) {   // b from global only when no cluster level restricted into it
      View<T> w = view_of(lsingle, false);
      load_all(w, sl_at(lsingle).gb, (T*)(smem + sl_at(lsingle).sb));
    }
    for (int k = lsingle; k <= lc; ++k) {
      const EngLevel<T>& L = sl_at(k);
      View<T> w = view_of(k, false);
      T* b = (T*)(smem + L.sb);
      __syncthreads();
      if (k == lc && run.coarse_mode == SELM_COARSE_CHOLESKY) {
        coarsest_step<T, NOISE>(w, b, (double*)(smem + P->y_off), spread, rank, csize);
        break;
      }
      sweeps_any<T, NOISE, D2>(w, pass_args(k, 0, b, true, 0), mu1, 0, 1, false);
      if (k == lc) {
        sweeps_any<T, NOISE, D2>(w, pass_args(k, mu1, b, true, 0), mu2, 0, 1, false);
        break;
      }
      const EngLevel<T>& Lc = sl_at(k + 1);
      residual<T, D2>(w, b, true, 0, (T*)(smem + L.st));
      __syncthreads();
      restrict_to<T, D2>(L, Lc, (const T*)(smem + L.st), true, (T*)(smem + Lc.sb), 0, Lc.nz);
      __syncthreads();
    }
    for (int k = lc - 1; k >= lsingle; --k) {
      const EngLevel<T>& L = sl_at(k);
      const EngLevel<T>& Lc = sl_at(k + 1);
      View<T> w = view_of(k, false);
      prolong_into<T, D2>(w, Lc, (const T*)(smem + Lc.sv), true);
      __syncthreads();
      sweeps_any<T, NOISE, D2>(w, pass_args(k, mu1, (const T*)(smem + L.sb), true, 0), mu2, 0, 1, false);
    }
    {   // the engine's result, or the hand-off to the cluster's prolongation
      View<T> w = view_of(lsingle, false);
      store_owned(w, sl_at(lsingle).gv);
    }
  }
  if (lsingle == lt) return;
  cl.sync();
  // ---- up leg over the cluster levels ----
  for (int k = lsingle - 1; k >= lt; --k) {
    const EngLevel<T>& L = sl_at(k);
    const EngLevel<T>& Lc = sl_at(k + 1);
    View<T> w = view_of(k, true);
    if (Lc.cluster) {
      prolong_into<T, D2>(w, Lc, Lc.gv, false);
    } else {
      // the coarse level is held by CTA 0, which still has its v in shared
      // memory; the other CTAs first copy the coarse planes that their slab and
      // halo read (independent loads) into their own unused slab of that
      // level, then prolong from shared memory
      View<T> wc = view_of(k + 1, false);
      if (rank != 0) {
        const int p0 = max(0, w.z0 - 2), p1 = min(L.nz, w.z1 + 2);
        int c0 = Lc.nz, c1 = 0;
        for (int z = p0; z < p1; ++z)
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            const int kr = L.pz_idx[2 * z + t], kc = kr < 0 ? max(L.pz_idx[2 * z], 0) : kr;
            c0 = min(c0, kc);
            c1 = max(c1, kc + 1);
          }
        const int base = c0 * wc.plane, nc = max(0, c1 - c0) * wc.plane;
#pragma unroll 4
        for (int q = threadIdx.x; q < nc; q += blockDim.x) {
          int i, j, kk;
          split_xy(Lc, q, &i, &j, &kk);
          wc.v[wc.loc(i, j, c0 + kk)] = ld_cg(Lc.gv + base + q);
        }
        __syncthreads();
      }
      prolong_into<T, D2>(w, Lc, (const T*)wc.v, true);
    }
    cl.sync();
    const bool bl = L.sb >= 0;   // staged on the way down, untouched since
    sweeps_any<T, NOISE, D2>(w, pass_args(k, mu1, bl ? (const T*)(smem + L.sb) : L.gb, bl, bl ? w.z0 * w.plane : 0), mu2,
                         rank, csize, true);
    store_owned(w, L.gv);
    cl.sync();
  }
}

template <typename T>
size_t level_bytes_cluster(const LevelDev& L, int c, int C) {
  const CompDev& d = L.c[c];
  const int P = (d.nz + C - 1) / C;
  return (size_t)(P + 4) * d.nx * d.ny * sizeof(T);
}

inline size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

// Pitches of a level's shared v slab.  A warp of a colour pass holds
// consecutive ranks of the class: x runs fastest (nx/2 sites of one parity,
// consecutive words within a row), then y in steps of 2, then z in steps of
// mz.  The row pitch rp is padded so that the rows one warp spans start on
// distinct banks (2 rp = sites per row, modulo 32 words), and the plane
// pitch pp likewise for the planes one warp spans (mz pp = sites per plane,
// modulo 32), when a warp spans more than one row or plane.
void slab_pitches(int nx, int ny, int mz, int* half, int* rp, int* pp) {
  const int h = (nx + 1) / 2;
  *half = h;
  int r = nx;
  if (ny > 1 && h < 32) {
    const int want = (((h + 1) & ~1) % 32) / 2;   // rp == want (mod 16)
    r = nx + (((want - nx) % 16) + 16) % 16;
  }
  *rp = r;
  int p = r * ny;
  const int per_plane = h * (ny > 1 ? (ny + 1) / 2 : 1);
  if (per_plane < 32 && mz > 0) {
    for (int c = p; c < p + 32; ++c)
      if ((long long)mz * c % 32 == per_plane % 32) {
        p = c;
        break;
      }
  }
  *pp = p;
}

template <typename T>
bool try_plan(const LevelDev* levs, int L, int l0, int C, bool stage_b, int sweeps, size_t smem_cap, EnginePlanT<T>* out) {
  // cluster levels first (largest), then single levels
  const int ncomp = levs[0].ncomp;
  size_t need_max = 0;
  EngParams<T>& p = out->params;
  p.l0 = l0;
  p.L = L;
  p.ncomp = ncomp;
  bool any_cluster = false;
  for (int c = 0; c < ncomp; ++c) {
    size_t off = 0;
    bool single_started = false;
    for (int l = l0; l < L; ++l) {
      const CompDev& d = levs[l].c[c];
      EngLevel<T>& e = p.comp[c].lev[l];
      const long long sites = (long long)d.nx * d.ny * d.nz;
      if (sites >= (1ll << 24)) return false;   // rank decode uses float reciprocals
      for (const double* wt : {d.w1, d.w2})   // the passes keep one weight per kind of neighbour
        if (wt[0] != wt[2] || wt[0] != wt[6] || wt[0] != wt[8] || wt[1] != wt[7] || wt[3] != wt[5]) return false;
      const bool single = single_started || l == L - 1 || sites <= eng_single_sites<T>() || C == 1;
      if (single) single_started = true;
      e.cluster = single ? 0 : 1;
      if (e.cluster) any_cluster = true;
      e.P = single ? d.nz : (d.nz + C - 1) / C;
      slab_pitches(d.nx, d.ny, d.mz, &e.half, &e.rp, &e.pp);
      const size_t vbytes = (size_t)(e.P + 4) * e.pp * sizeof(T);
      e.sv = (int)off;
      off = align16(off + vbytes);
      if (single) {
        e.sb = (int)off;
        off = align16(off + (size_t)sites * sizeof(T));
        e.st = (int)off;
        off = align16(off + (size_t)sites * sizeof(T));
      } else {
        e.sb = e.st = -1;
        if (stage_b) {   // b of the owned planes
          e.sb = (int)off;
          off = align16(off + (size_t)e.P * d.nx * d.ny * sizeof(T));
        }
      }
    }
    const CompDev& dc = levs[L - 1].c[c];
    const size_t Nc = (size_t)dc.nx * dc.ny * dc.nz;
    if (Nc > 1024) return false;
    out->y_off_comp[c] = off;
    off = align16(off + Nc * sizeof(double));
    need_max = need_max > off ? need_max : off;
  }
  // row tables of every level (components share the layout: the largest nz)
  int rows = 0;
  for (int l = l0; l < L; ++l) {
    p.tab_row[l] = rows;
    int nzl = 0;
    for (int c = 0; c < ncomp; ++c) nzl = nzl > levs[l].c[c].nz ? nzl : levs[l].c[c].nz;
    rows += nzl;
  }
  for (int c = 0; c < ncomp; ++c)
    for (int l = l0; l < L; ++l)
      if (levs[l].c[c].ncol > kEngMaxColours) return false;
  // transfer tables of the levels with a coarser level below them
  int xrows = 0;
  for (int l = l0; l < L; ++l) {
    p.xf_row[l] = xrows;
    if (l == L - 1) continue;
    int nzl = 0, nzc = 0;
    for (int c = 0; c < ncomp; ++c) {
      nzl = nzl > levs[l].c[c].nz ? nzl : levs[l].c[c].nz;
      nzc = nzc > levs[l + 1].c[c].nz ? nzc : levs[l + 1].c[c].nz;
    }
    xrows += 2 * nzl + 4 * nzc;
  }
  const size_t staged = (size_t)rows * 12 * sizeof(T) + (size_t)(L - l0) * sizeof(EngLevel<T>) +
                        (size_t)(L - l0) * kEngMaxColours * sizeof(EngColour) +
                        (size_t)xrows * (sizeof(int) + sizeof(T)) + 96;
  if (need_max + staged > smem_cap) return false;
  if (!any_cluster) C = 1;
  // every component gets the same y offset (the maximum) so that the kernel
  // can use one field
  size_t yo = 0;
  for (int c = 0; c < ncomp; ++c) yo = yo > out->y_off_comp[c] ? yo : out->y_off_comp[c];
  p.y_off = (int)yo;
  size_t ymax = 0;
  for (int c = 0; c < ncomp; ++c) {
    const CompDev& dc = levs[L - 1].c[c];
    const size_t Nc = (size_t)dc.nx * dc.ny * dc.nz;
    ymax = ymax > Nc ? ymax : Nc;
  }
  const size_t tab_off = align16(yo + ymax * sizeof(double));
  const size_t lev_off = align16(tab_off + (size_t)rows * 12 * sizeof(T));
  const size_t col_off = align16(lev_off + (size_t)(L - l0) * sizeof(EngLevel<T>));
  const size_t xfi_off = align16(col_off + (size_t)(L - l0) * kEngMaxColours * sizeof(EngColour));
  const size_t xfw_off = align16(xfi_off + (size_t)xrows * sizeof(int));
  p.tab_off = (int)tab_off;
  p.lev_off = (int)lev_off;
  p.col_off = (int)col_off;
  p.xfi_off = (int)xfi_off;
  p.xfw_off = (int)xfw_off;
  out->smem_bytes = align16(xfw_off + (size_t)xrows * sizeof(T));
  if (out->smem_bytes > smem_cap) return false;
  // normals of the noisy launches, in what is left: the coarsest levels first
  // (their passes are the shortest); a level without room draws at its sites
  out->smem_noise = out->smem_bytes;
  for (int l = 0; l < kMaxLevels; ++l) p.nz_off[l] = -1;
  for (int l = L - 1; l >= l0; --l) {
    size_t sites = 0;
    for (int c = 0; c < ncomp; ++c) {
      const CompDev& d = levs[l].c[c];
      const size_t n = (size_t)p.comp[c].lev[l].P * d.nx * d.ny;
      sites = sites > n ? sites : n;
    }
    const size_t bytes = align16(sites * (size_t)sweeps * sizeof(T));
    if (out->smem_noise + bytes > smem_cap) break;
    p.nz_off[l] = (int)out->smem_noise;
    out->smem_noise += bytes;
  }
  out->cluster = C;
  return true;
}

}  // namespace

template <typename T>
void fill_engine_tables(const LevelDev* levs, int L, void* const* gb, void* const* gv, void* const* gt,
                        EnginePlanT<T>* plan) {
  EngParams<T>& p = plan->params;
  for (int c = 0; c < p.ncomp; ++c)
    for (int l = p.l0; l < L; ++l) {
      const CompDev& d = levs[l].c[c];
      EngLevel<T>& e = p.comp[c].lev[l];
      e.nx = d.nx;
      e.ny = d.ny;
      e.nz = d.nz;
      e.mx = d.mx;
      e.my = d.my;
      e.mz = d.mz;
      e.ncol = d.ncol;
      e.comp_id = d.comp_id;
      e.S = sizeof(T) == 4 ? (const T*)d.S32 : (const T*)d.S64;
      e.zb = sizeof(T) == 4 ? (const T*)d.zb32 : (const T*)d.zb64;
      for (int q = 0; q < 9; ++q) {
        e.w1[q] = (T)d.w1[q];
        e.w2[q] = (T)d.w2[q];
      }
      auto log2_or = [](int n) {
        int l = 0;
        while ((1 << l) < n) ++l;
        return (1 << l) == n ? l : -1;
      };
      e.lx = log2_or(d.nx);
      e.ly = log2_or(d.ny);
      e.inv_nxc = 1.0f / (float)((d.nx + d.mx - 1) / d.mx);
      e.inv_nyc = 1.0f / (float)((d.ny + d.my - 1) / d.my);
      e.rz_idx = d.rz_idx;
      e.rz_w = sizeof(T) == 4 ? (const T*)d.rz_w32 : (const T*)d.rz_w64;
      e.pz_idx = d.pz_idx;
      e.pz_w = sizeof(T) == 4 ? (const T*)d.pz_w32 : (const T*)d.pz_w64;
      e.Linv = d.Linv;
      e.gb = (T*)gb[l] + d.off;
      e.gv = (T*)gv[l] + d.off;
      e.gt = (T*)gt[l] + d.off;
    }
}

namespace {
template <typename T>
bool raise_smem_limit() {
  static std::atomic<bool> done{false};
  if (done.load()) return true;
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  for (auto fn : {k_coarse_engine<T, true, false>, k_coarse_engine<T, false, false>, k_coarse_engine<T, true, true>,
                  k_coarse_engine<T, false, true>}) {
    cudaFuncAttributes fa{};
    if (cudaFuncGetAttributes(&fa, fn) != cudaSuccess ||
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes) !=
            cudaSuccess ||
        cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
  }
  done.store(true);
  return true;
}
}  // namespace

template <typename T>
bool plan_coarse_engine(const LevelDev* levs, int L, void* const* gb, void* const* gv, void* const* gt,
                        void* dev_params, cudaStream_t st, EnginePlanT<T>* plan, int sweeps, int want_cluster,
                        int min_level) {
  static_assert(sizeof(EngParams<T>) <= kEngParamBytes, "engine plan exceeds its workspace slot");
  plan->valid = false;
  if (L < 2 || !dev_params) return false;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  int cap = 0, cluster_ok = 0;
  cudaDeviceGetAttribute(&cap, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaDeviceGetAttribute(&cluster_ok, cudaDevAttrClusterLaunch, dev);
  const size_t smem_cap = (size_t)cap > 2048 ? (size_t)cap - 1024 : 0;
  const int sizes[5] = {16, 8, 4, 2, 1};
  for (int l0 = min_level > 1 ? min_level : 1; l0 < L; ++l0) {
    for (int si = 0; si < 5; ++si) {
      const int C = sizes[si];
      if (C > 1 && !cluster_ok) continue;
      if (want_cluster > 0 && C > want_cluster) continue;
      EnginePlanT<T> cand{};
      // with b of the cluster levels staged in shared memory if it fits
      if (!try_plan<T>(levs, L, l0, C, true, sweeps, smem_cap, &cand) &&
          !try_plan<T>(levs, L, l0, C, false, sweeps, smem_cap, &cand))
        continue;
      // The dynamic shared-memory limit is a per-kernel setting shared by every
      // handle of the process: raise it once to the device maximum so that
      // plans of any size stay launchable.
      if (!raise_smem_limit<T>()) continue;
      auto fits = [&](int c, size_t smem) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(c * levs[0].ncomp);
        cfg.blockDim = dim3(EngThreads<T>::value);
        cfg.dynamicSmemBytes = smem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = c;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int nclusters = 0;
        if (cudaOccupancyMaxActiveClusters(
                &nclusters, levs[0].c[0].ny == 1 ? k_coarse_engine<T, true, true> : k_coarse_engine<T, true, false>, &cfg) == cudaSuccess && nclusters >= 1)
          return true;
        cudaGetLastError();
        return false;
      };
      if (cand.cluster > 1 && !fits(cand.cluster, cand.smem_noise)) continue;
      // Without cluster levels CTA 0 holds everything; the noisy launch takes
      // more CTAs to draw its normals (FP64 Box-Muller at two lanes per clock
      // is most of such a cycle on one SM).
      cand.noise_cluster = cand.cluster;
      for (int c = 16; cand.cluster == 1 && c > 1; c /= 2)
        if (cluster_ok && (want_cluster <= 0 || c <= want_cluster) && cand.params.nz_off[l0] >= 0 &&
            fits(c, cand.smem_noise)) {
          cand.noise_cluster = c;
          break;
        }
      *plan = cand;
      fill_engine_tables<T>(levs, L, gb, gv, gt, plan);
      if (cudaMemcpyAsync(dev_params, &plan->params, sizeof(EngParams<T>), cudaMemcpyHostToDevice, st) !=
              cudaSuccess ||
          cudaStreamSynchronize(st) != cudaSuccess) {
        cudaGetLastError();
        return false;
      }
      plan->dev = (const EngParams<T>*)dev_params;
      plan->valid = true;
      return true;
    }
  }
  return false;
}

template <typename T>
cudaError_t launch_coarse_engine(const EnginePlanT<T>& plan, int mu1, int mu2, int coarse_mode, bool noise, Key key,
                                 const unsigned long long* cyc, cudaStream_t st) {
  EngRun run{mu1, mu2, coarse_mode, key, cyc};
  const int cluster = noise ? plan.noise_cluster : plan.cluster;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(cluster * plan.params.ncomp);
  cfg.blockDim = dim3(EngThreads<T>::value);
  cfg.dynamicSmemBytes = noise ? plan.smem_noise : plan.smem_bytes;
  cfg.stream = st;
  // Programmatic launch: the tables and normals are staged while the kernel
  // before it drains.
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  prof::Scope ps(SELM_K_COARSE_SWEEP, st);
  const bool d2 = plan.params.comp[0].lev[plan.params.l0].ny == 1;
  if (noise && d2) return cudaLaunchKernelEx(&cfg, k_coarse_engine<T, true, true>, plan.dev, run);
  if (noise) return cudaLaunchKernelEx(&cfg, k_coarse_engine<T, true, false>, plan.dev, run);
  if (d2) return cudaLaunchKernelEx(&cfg, k_coarse_engine<T, false, true>, plan.dev, run);
  return cudaLaunchKernelEx(&cfg, k_coarse_engine<T, false, false>, plan.dev, run);
}

template bool plan_coarse_engine<float>(const LevelDev*, int, void* const*, void* const*, void* const*, void*,
                                        cudaStream_t, EnginePlanT<float>*, int, int, int);
template bool plan_coarse_engine<double>(const LevelDev*, int, void* const*, void* const*, void* const*, void*,
                                         cudaStream_t, EnginePlanT<double>*, int, int, int);
template cudaError_t launch_coarse_engine<float>(const EnginePlanT<float>&, int, int, int, bool, Key,
                                                 const unsigned long long*, cudaStream_t);
template cudaError_t launch_coarse_engine<double>(const EnginePlanT<double>&, int, int, int, bool, Key,
                                                  const unsigned long long*, cudaStream_t);

}  // namespace selm
