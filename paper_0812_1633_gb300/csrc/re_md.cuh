// re_md.cuh -- device building blocks of the sm_103a replica-exchange LJ MD
// kernels shared by every translation unit of the library: cell binning,
// neighbour-list build, pair forces, thermostat records, the exchange rule
// and the free-running exchange protocol.  Internal header.
#pragma once
#include <cooperative_groups.h>
#include <cuda_fp16.h>

#include <algorithm>

#include "re_device.cuh"
#include "re_internal.h"

namespace re {
namespace cg = cooperative_groups;

namespace {

constexpr int kMaxCluster = 8;
constexpr int kMaxWarps = 32;
constexpr int kPlainRed = 1024;  // per-replica reduction slots of the plain path
constexpr int kNoiseChunk = 64;  // thermostat records prepared at a time (double buffered)
constexpr int kSvrStepBytes = 32;  // sizeof(SvrStep)

// ------------------------------------------------------------------ cells
// Top 32 bits of a position (enough for binning and list radii).
struct Hi3 {
  uint32_t x, y, z;
};

__device__ __forceinline__ int cell_of(Hi3 p, int nc) {
  return ((int)__umulhi(p.x, (uint32_t)nc) * nc + (int)__umulhi(p.y, (uint32_t)nc)) * nc +
         (int)__umulhi(p.z, (uint32_t)nc);
}

// Exclusive scan of cnt[0..n) into start[0..n], start[n] = total.  Whole block.
__device__ void block_exclusive_scan(const int* cnt, int* start, int n, int* scratch) {
  const int T = blockDim.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int nw = (T + 31) >> 5;
  const int per = (n + T - 1) / T;
  const int lo = min(n, tid * per), hi = min(n, lo + per);
  int s = 0;
  for (int c = lo; c < hi; ++c) s += cnt[c];
  int incl = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  __syncthreads();
  if (lane == 31) scratch[warp] = incl;
  __syncthreads();
  int off = 0;
  for (int w = 0; w < warp; ++w) off += scratch[w];
  int run = off + incl - s;
  for (int c = lo; c < hi; ++c) {
    start[c] = run;
    run += cnt[c];
  }
  if (tid == T - 1) {
    int tot = 0;
    for (int w = 0; w < nw; ++w) tot += scratch[w];
    start[n] = tot;
  }
  __syncthreads();
}

// Cell binning and counting sort of all N atoms of a replica (whole block):
// cstart[c]..cstart[c+1] index spos, the atoms of cell c in increasing index
// order (cells x-major, as ((cx * nc) + cy) * nc + cz); spos[k] holds the top
// 32 bits of the position and, in .w, the atom index, so that the list build
// scans contiguous ranges with one load per candidate.
template <class PosFn>
__device__ void cta_build_cells(PosFn pos_hi, int N, int nc, int* cstart, int* ccnt, uint4* spos,
                                uint16_t* acell, int* scratch) {
  const int T = blockDim.x, tid = threadIdx.x;
  const int ncell = nc * nc * nc;
  for (int c = tid; c < ncell; c += T) ccnt[c] = 0;
  __syncthreads();
  for (int i = tid; i < N; i += T) {
    const int c = cell_of(pos_hi(i), nc);
    acell[i] = (uint16_t)c;
    atomicAdd(&ccnt[c], 1);
  }
  __syncthreads();
  block_exclusive_scan(ccnt, cstart, ncell, scratch);
  for (int c = tid; c < ncell; c += T) ccnt[c] = cstart[c];
  __syncthreads();
  for (int i = tid; i < N; i += T) {
    const int k = atomicAdd(&ccnt[acell[i]], 1);
    const Hi3 p = pos_hi(i);
    spos[k] = make_uint4(p.x, p.y, p.z, (uint32_t)i);
  }
  __syncthreads();
  for (int c = tid; c < ncell; c += T) {
    const int b = cstart[c], e = cstart[c + 1];
    for (int k = b + 1; k < e; ++k) {
      const uint4 v = spos[k];
      int j = k - 1;
      while (j >= b && spos[j].w > v.w) {
        spos[j + 1] = spos[j];
        --j;
      }
      spos[j + 1] = v;
    }
  }
  __syncthreads();
}

__device__ __forceinline__ float sep2_hi(Hi3 a, Hi3 b) {
  const float dx = (float)(int)(b.x - a.x), dy = (float)(int)(b.y - a.y),
              dz = (float)(int)(b.z - a.z);
  return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

// ------------------------------------------------------------------ forces
// Mixed precision pair forces.  Separations are exact 32-bit integer minimum
// images (units lam = L / 2^32) converted to FP32 once; the pair force and
// energy are FP32, and so are the sums over one sub-list.  Force on i from j =
// fs * d with fs = s^4 (24 - 48 s^3), s = 1/r^2 (sigma units); pair energy
// 4 s^3 (s^3 - 1).
//
// Two list entries are taken at a time, as packed f32x2 instructions (21
// instead of 28 issued instructions per entry), without a branch per pair:
// with q = -2 s^3 the force is fs = 24 s^4 (1 + q) (the factor 24 is part of
// StepConst::hlf) and the pair energy q (q + 2); outside the cutoff s is 0.
//
// The cutoff test.  The force is truncated at rc (Example section), so it
// jumps there by F(rc) ~ 0.04: a pair put on the wrong side of rc costs its
// atoms a force error of ~1e-3 of the rms force, and the FP32 r^2 (relative
// error below 3e-7) would do that for pairs within ~1e-7 of rc -- about one
// pair per ten evaluations of a 4000-atom replica.  So FP32 decides every
// pair outside a relative band of 2e-6 around rc^2, and pairs inside the band
// are decided in FP64 on 42-bit separations: the top 32 bits and the next 10
// bits of each coordinate (kept in .w of the shared-memory position, 10 bits
// per coordinate).  The loop counts every pair with FP32 r^2 < rc^2 (1 + 2e-6)
// and keeps the smallest distance of any r^2 from that limit; a lane that saw
// one near the band (about one in 1500 sub-lists) goes over its list again and
// takes out the pairs that the 42-bit separations put outside.  The result
// equals the FP64 test on the full positions except for pairs within ~1e-11
// of rc.

// Packed FP32 pairs (one 64-bit register pair; low half first).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(a), "f"(b));
  return v;
}
__device__ __forceinline__ float lo2(f32x2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return a;
}
__device__ __forceinline__ float hi2(f32x2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return b;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 v;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(v) : "l"(a), "l"(b), "l"(c));
  return v;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 v;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
  return v;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 v;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v) : "l"(a), "l"(b));
  return v;
}
__device__ __forceinline__ float min3_abs(float a, float b, float c) {
  float v;
  asm("min.abs.f32 %0, %1, %2, %3;" : "=f"(v) : "f"(a), "f"(b), "f"(c));
  return v;
}

struct PairAcc {
  f32x2 fx, fy, fz;  // force sums over the even and the odd entries
  f32x2 e, n;        // ENERGY: pair energies (times c1^2), pairs counted inside
  float tmin;        // smallest |r^2 - rc^2 (1 + 2e-6)| met
};

// 42-bit minimum-image separation of one coordinate: top 32 bits (hj, hi) and
// the next 10 bits (lj, li) of the two positions.
__device__ __forceinline__ double sep42(uint32_t hj, uint32_t hi, uint32_t lj, uint32_t li) {
  return (double)(((long long)(int)(hj - hi) << 10) + ((long long)lj - (long long)li));
}

__device__ __forceinline__ bool inside_cutoff_42(uint4 pi, uint4 pj, double x42) {
  const double dx = sep42(pj.x, pi.x, (pj.w >> 20) & 1023u, (pi.w >> 20) & 1023u);
  const double dy = sep42(pj.y, pi.y, (pj.w >> 10) & 1023u, (pi.w >> 10) & 1023u);
  const double dz = sep42(pj.z, pi.z, pj.w & 1023u, pi.w & 1023u);
  return fma(dx, dx, fma(dy, dy, dz * dz)) < x42;
}

// Of two pairs from their r^2, with s = cs / r^2 and u = c1 + c3 s^3 = c1 (1 + q):
// the force s^4 u, c1 q and c1 (q + 2).  The scale 2^k in cs (exact) keeps the
// powers in range; c3 / c1, the one constant of the force that cannot be exact, is
// off by some 1e-9 (set_pair_constants).
__device__ __forceinline__ void lj2(f32x2 r2, f32x2 cs, f32x2 c1, f32x2 c3, f32x2& fs, f32x2& q,
                                    f32x2& q2) {
  const f32x2 s = mul2(pack2(rcp_approx(lo2(r2)), rcp_approx(hi2(r2))), cs);
  const f32x2 s2 = mul2(s, s), s3 = mul2(s2, s);
  const f32x2 u = fma2(s3, c3, c1);
  fs = mul2(mul2(s2, s2), u);
  q = mul2(s3, c3);
  q2 = add2(u, c1);
}

__device__ __forceinline__ f32x2 len2(f32x2 dx, f32x2 dy, f32x2 dz) {
  return fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
}

// Atom i against two list entries j, k.  TAIL: only the first `real` of them
// count (list padding, which may be the atom itself).
template <bool ENERGY, bool TAIL>
__device__ __forceinline__ void mixed_pair2(const Hi3& pi, uint4 pj, uint4 pk, f32x2 cs, f32x2 c1, f32x2 c3,
                                            f32x2 nhi, int real, PairAcc& a) {
  const f32x2 dx = pack2((float)(int)(pj.x - pi.x), (float)(int)(pk.x - pi.x));
  const f32x2 dy = pack2((float)(int)(pj.y - pi.y), (float)(int)(pk.y - pi.y));
  const f32x2 dz = pack2((float)(int)(pj.z - pi.z), (float)(int)(pk.z - pi.z));
  const f32x2 r2 = len2(dx, dy, dz);
  const f32x2 t = add2(r2, nhi);  // negative: inside (the sign is exact)
  a.tmin = min3_abs(lo2(t), hi2(t), a.tmin);
  const f32x2 m = pack2(__saturatef(lo2(t) * -1e30f), __saturatef(hi2(t) * -1e30f));
  f32x2 fs, q, q2;
  lj2(r2, mul2(cs, m), c1, c3, fs, q, q2);
  if (TAIL) fs = pack2(real > 0 ? lo2(fs) : 0.0f, real > 1 ? hi2(fs) : 0.0f);
  a.fx = fma2(fs, dx, a.fx);
  a.fy = fma2(fs, dy, a.fy);
  a.fz = fma2(fs, dz, a.fz);
  if (ENERGY) {
    f32x2 n = m;
    if (TAIL) {
      q = pack2(real > 0 ? lo2(q) : 0.0f, real > 1 ? hi2(q) : 0.0f);
      q2 = pack2(real > 0 ? lo2(q2) : 0.0f, real > 1 ? hi2(q2) : 0.0f);
      n = pack2(real > 0 ? lo2(n) : 0.0f, real > 1 ? hi2(n) : 0.0f);
    }
    a.e = fma2(q, q2, a.e);
    a.n = add2(a.n, n);
  }
}

// Takes one pair's contribution out again.
template <bool ENERGY>
__device__ __forceinline__ void mixed_pair_remove(float dx, float dy, float dz, float r2,
                                                  const StepConst& K, PairAcc& a) {
  f32x2 fs, q, q2;
  lj2(pack2(r2, r2), pack2(K.cs, K.cs), pack2(K.c1, K.c1), pack2(K.c3, K.c3), fs, q, q2);
  const f32x2 m = pack2(-1.0f, 0.0f);
  fs = mul2(fs, m);
  a.fx = fma2(fs, pack2(dx, dx), a.fx);
  a.fy = fma2(fs, pack2(dy, dy), a.fy);
  a.fz = fma2(fs, pack2(dz, dz), a.fz);
  if (ENERGY) {
    a.e = fma2(mul2(q, m), q2, a.e);
    a.n = add2(a.n, m);
  }
}

// Positions of the FP64 path: 64-bit fixed-point words (units L / 2^64).
struct Pos64 {
  uint64_t x, y, z, w;
};

// ------------------------------------------------------------------ batched
struct BatchedSmem {
  uint16_t* nb_sm;  // this CTA's neighbour sub-lists when they fit in shared memory
  void* pos;       // uint4[N] (mixed: top 32 bits of x, y, z) or Pos64[N] (fp64)
  uint4* hk;       // f16 screening vectors of the atoms, rows of 32 (list build)
  uint2* box;      // bounding box of each row: centre bytes, half-width bytes
  uint8_t* act;    // per warp: the rows in reach of its atoms
  uint32_t* ref;     // 3 per own atom: top 32 bits of the coordinates at the last list build
  long long* rec_k;  // kNoiseChunk: 2K of each step (fixed point), CTA 0
  float* rec_e;      // kNoiseChunk: alpha - 1 of each step
  double2* noise;  // 2 x kNoiseChunk thermostat records (double buffered)
  float* slot_md;  // [cluster][warps]
  double* slot_uk; // [cluster][warps][2]
  int* slot_st;    // [cluster]
};

__host__ __device__ inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

// A warp's list of rows (of 32 atoms), with room for four more.
__host__ __device__ inline size_t row_list_bytes(int n) { return (size_t)((n + 31) / 32 + 11) / 8 * 8; }

__host__ __device__ inline size_t batched_layout(int max_n, int threads, bool fp64,
                                                 size_t list_elems, unsigned char* base,
                                                 BatchedSmem* out) {
  size_t off = 0;
  auto take = [&](size_t bytes, size_t al) {
    off = align_up(off, al);
    size_t o = off;
    off += bytes;
    return o;
  };
  const size_t o_pos = take((size_t)max_n * (fp64 ? 32 : 16), 32);  // at the base: fixed offset
  const size_t o_nbs = take(list_elems * 2, 16);
  const size_t rows = ((size_t)max_n + 31) / 32;  // of 32 atoms
  // the screening vectors of a list build, or the FP64 pair loop's notes (32 a
  // thread; with P >= 4 threads an atom, at most 2048 atoms in 8 CTAs)
  const size_t hk_bytes = rows * 512, notes = fp64 && max_n <= 2048 ? (size_t)threads * 64 : 0;
  const size_t o_hk = take(hk_bytes > notes ? hk_bytes : notes, 128);
  const size_t o_bx = take(rows * sizeof(uint2), 8);
  const size_t o_ar = take((size_t)kMaxWarps * row_list_bytes(max_n), 8);
  const size_t o_noise = take((size_t)kNoiseChunk * 2 * kSvrStepBytes, 16);
  const size_t o_uk = take((size_t)kMaxCluster * kMaxWarps * 2 * 8, 16);
  const size_t o_md = take((size_t)kMaxCluster * kMaxWarps * 4, 4);
  const size_t o_st = take(kMaxCluster * 4, 4);
  const size_t o_ref = take(fp64 ? 0 : (size_t)threads * 3 * 4, 4);  // own atoms <= threads
  const size_t o_rk = take((size_t)kNoiseChunk * 8, 8);
  const size_t o_re = take((size_t)kNoiseChunk * 4, 4);
  if (out) {
    out->nb_sm = reinterpret_cast<uint16_t*>(base + o_nbs);
    out->pos = base + o_pos;
    out->noise = reinterpret_cast<double2*>(base + o_noise);
    out->slot_uk = reinterpret_cast<double*>(base + o_uk);
    out->slot_md = reinterpret_cast<float*>(base + o_md);
    out->slot_st = reinterpret_cast<int*>(base + o_st);
    out->ref = reinterpret_cast<uint32_t*>(base + o_ref);
    out->rec_k = reinterpret_cast<long long*>(base + o_rk);
    out->rec_e = reinterpret_cast<float*>(base + o_re);
    out->hk = reinterpret_cast<uint4*>(base + o_hk);
    out->box = reinterpret_cast<uint2*>(base + o_bx);
    out->act = reinterpret_cast<uint8_t*>(base + o_ar);
  }
  return align_up(off, 128);
}

struct KernelDims {
  int max_n;
  size_t list_elems;  // shared-memory list entries per CTA (0: lists in global memory)
  int async_nx;       // > 0: free-running mode with this many master steps
};

// free-running mode: step cap of the non-master replicas (a bound, not a budget)
constexpr int kAsyncCapFactor = 16;

__device__ __forceinline__ uint64_t* qcomp(const StateDev& S, int d) {
  return d == 0 ? S.qx : (d == 1 ? S.qy : S.qz);
}
__device__ __forceinline__ double* vcomp(const StateDev& S, int d) {
  return d == 0 ? S.vx : (d == 1 ? S.vy : S.vz);
}
__device__ __forceinline__ double* fcomp(const StateDev& S, int d) {
  return d == 0 ? S.fx : (d == 1 ? S.fy : S.fz);
}
__device__ __forceinline__ uint32_t* rcomp(const StateDev& S, int d) {
  return d == 0 ? S.rx : (d == 1 ? S.ry : S.rz);
}

// The list of atom i on the plain path (one thread an atom), from the cells
// (nc > 0) or all atoms: entry k at element ((k / 4) * N + i) * 4 + k % 4 of nb.
template <class PosFn>
__device__ int build_list_cells(int i, PosFn pos_hi, int N, int nc, int m, const int* cstart,
                                const uint4* spos, float rl2u, uint16_t* nb, int cap,
                                int* overflow) {
  const Hi3 pi = pos_hi(i);
  // a running offset: +1 inside a block of four, + N*4 - 3 across blocks
  uint32_t wofs = (uint32_t)i * 4;
  const uint32_t jump = (uint32_t)N * 4 - 3u;
  int cnt = 0;
  bool coincident = false;
  auto accept = [&](int j, Hi3 pj) {
    const float r2 = sep2_hi(pi, pj);
    if (j != i && r2 < rl2u) {
      // two distinct atoms at one point (closer than L / 2^32): the pair loop
      // treats distance 0 as the sub-list padding, so report it (below)
      coincident |= (r2 == 0.0f);
      if (cnt < cap) {
        nb[wofs] = (uint16_t)j;
        wofs += ((cnt & 3) == 3) ? jump : 1u;
      }
      ++cnt;
    }
  };
  if (nc == 0) {
    for (int j = 0; j < N; ++j) accept(j, pos_hi(j));
  } else {
    const int cx = (int)__umulhi(pi.x, (uint32_t)nc), cy = (int)__umulhi(pi.y, (uint32_t)nc),
              cz = (int)__umulhi(pi.z, (uint32_t)nc);
    // cells z in [cz - m, cz + m] (periodic) are at most two contiguous ranges
    // of the cell order: [lo1, hi1) and [0, hi2) (empty when hi2 == 0).
    // (Pruning columns and z ranges to the sphere with the atom's exact offset
    // scans fewer candidates but was not faster: the per-column work and the
    // lane divergence it adds cost as much as the candidates it saves.)
    const int zlo = cz - m, zhi = cz + m;
    const int lo1 = zlo < 0 ? zlo + nc : zlo;
    const int hi1 = (zlo < 0 || zhi >= nc) ? nc : zhi + 1;
    const int hi2 = zlo < 0 ? zhi + 1 : (zhi >= nc ? zhi - nc + 1 : 0);
    for (int ox = -m; ox <= m; ++ox) {
      int x = cx + ox;
      x += (x < 0) ? nc : 0;
      x -= (x >= nc) ? nc : 0;
      for (int oy = -m; oy <= m; ++oy) {
        int y = cy + oy;
        y += (y < 0) ? nc : 0;
        y -= (y >= nc) ? nc : 0;
        const int base = (x * nc + y) * nc;
        const int b1 = cstart[base + lo1], e1 = cstart[base + hi1];
        const int b2 = cstart[base], e2 = cstart[base + hi2];
        const int n1 = e1 - b1, n = n1 + (e2 - b2);
        // two candidates per iteration: both loads issue before either test
        // (four were measured slower)
        int t = 0;
        for (; t + 1 < n; t += 2) {
          const int t2 = t + 1;
          const uint4 v = spos[t < n1 ? b1 + t : b2 + (t - n1)];
          const uint4 w = spos[t2 < n1 ? b1 + t2 : b2 + (t2 - n1)];
          accept((int)v.w, Hi3{v.x, v.y, v.z});
          accept((int)w.w, Hi3{w.x, w.y, w.z});
        }
        if (t < n) {
          const uint4 v = spos[t < n1 ? b1 + t : b2 + (t - n1)];
          accept((int)v.w, Hi3{v.x, v.y, v.z});
        }
      }
    }
  }
  if (coincident) *overflow |= kStNumeric;
  if (cnt > cap) {
    *overflow |= kStOverflow;
    cnt = cap;
  }
  // pad to a whole block of four with the atom's own index (skipped by r2 > 0)
  for (int k = cnt; k & 3; ++k) nb[wofs++] = (uint16_t)i;
  return cnt;
}

// ------------------------------------------------- list build, batched kernel
// Which atoms lie within the list radius of which is first screened on the
// tensor cores: with a = 2 pi / L,
//   S = sum over d of cos(a dx_d) = sum of cos a x_d cos a x'_d + sin a x_d sin a x'_d
// is a dot product of two six-vectors, periodic by itself, and within a
// distance r it is at least 3 cos(a r / sqrt 3) (cos(a sqrt u) is convex in u,
// so the least sum at a given r^2 is the one of equal components).  One
// mma.m16n8k8 (f16 vectors, f32 sums; the other two of its eight products add
// the limit, and put the last row's missing atoms beyond it) screens 16 atoms
// against 8; one funnel shift per result collects its sign.  Of the candidates that
// pass (7 to 20 % more than the list at L = 17 to 10) the exact test on the 32-bit
// positions keeps the list, so the pair set does not depend on the screening.  No
// cells are built or sorted: a warp goes through the rows (32 consecutive atoms)
// whose bounding box lies within the list radius of its own atoms' box.  Atoms are
// renumbered in space order from time to time, so both boxes are small; the order
// affects the time only.
//
// A lane's hits come unevenly from mask to mask, but in all the lanes of a warp
// have nearly the same number.  So the masks are only noted, and the loop over
// their bits, with the exact test, lets every lane go through its own notes at
// its own pace: as many turns as the fullest lane has hits (emptying mask by
// mask takes three times as many).  Bound by instruction issue.  A build took,
// against the cell scan it replaces, in thousand clocks: 53 against 74 (864
// atoms on two CTAs, skin 0.3), 162 against 175 (2048, skin 0.5), 189 against
// 440 (4000 on four); 14, 55 and 77 of them screen, the rest is the exact test.

__device__ __forceinline__ uint32_t pack8(Hi3 p) {
  return (p.x >> 24) | ((p.y >> 24) << 8) | ((p.z >> 24) << 16);
}

// Bounding box of the bytes of a warp's values w (those with `in`): centre and
// half-width bytes of the interval of every coordinate around one of them.
__device__ __forceinline__ uint2 warp_box(uint32_t w, bool in) {
  const uint32_t ref = __shfl_sync(0xffffffffu, w, __ffs(__ballot_sync(0xffffffffu, in)) - 1);
  uint32_t cen = 0, half = 0;
#pragma unroll
  for (int d = 0; d < 24; d += 8) {
    const int e = in ? (int)(int8_t)((w >> d) - (ref >> d)) : 0;
    const int l = __reduce_min_sync(0xffffffffu, e), h = __reduce_max_sync(0xffffffffu, e);
    const int m = (l + h) >> 1;
    cen |= (((ref >> d) + (uint32_t)m) & 255u) << d;
    half |= (uint32_t)(h - m) << d;
  }
  return make_uint2(cen, half);
}

__device__ __forceinline__ uint32_t half2_bits(float lo, float hi) {
  const __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// Screening vectors and row boxes of all N atoms (whole block): atom j's
// (cx, cy, cz, sx, sy, sz, 0, 1) at hk[j].  Ends with a block barrier.
template <class PosFn>
__device__ __forceinline__ void cta_screen_vectors(PosFn pos_hi, int N, uint4* hk, uint2* box) {
  const int T = blockDim.x, lane = threadIdx.x & 31;
  constexpr float kTurn = 1.4629180792671596e-09f;  // 2 pi / 2^32
  for (int r = threadIdx.x >> 5; r < (N + 31) / 32; r += T >> 5) {
    const int j = r * 32 + lane;
    const Hi3 p = j < N ? pos_hi(j) : Hi3{0u, 0u, 0u};
    // signed: angles in [-pi, pi], where the fast functions are accurate
    const float ax = (float)(int)p.x * kTurn, ay = (float)(int)p.y * kTurn, az = (float)(int)p.z * kTurn;
    hk[j] = make_uint4(half2_bits(__cosf(ax), __cosf(ay)), half2_bits(__cosf(az), __sinf(ax)),
                       half2_bits(__sinf(ay), __sinf(az)), j < N ? 0x3C000000u : 0x3C007800u);
    const uint2 b = warp_box(pack8(p), j < N);
    if (lane == 0) box[r] = b;
  }
  __syncthreads();
}

// The end of a sub-list: coincident atoms (closer than L / 2^32: the pair loop
// cannot give their force a direction) reported, the last block filled up with
// the atom's own index.  cnt, which the caller compares with cap_sub, is
// returned as it is.
__device__ __forceinline__ int finish_sublist(int cnt, uint2 blk, uint2* out, int i,
                                              bool coincident, int cap_sub, int* status) {
  if (coincident) *status |= kStNumeric;
  if (cnt <= cap_sub && (cnt & 3)) {
    for (int k = cnt; k & 3; ++k) {
      blk.x = __funnelshift_r(blk.x, blk.y, 16);
      blk.y = __byte_perm(blk.y, (uint32_t)i, 0x5432);
    }
    *out = blk;
  }
  return cnt;
}

// The sub-lists of atoms whose neighbours the builds below spread too unevenly
// over the lanes: they go by the atoms' numbers, so an order that puts the
// neighbours of an atom into one residue class (the atoms of P spatial domains
// taken in turn) gives one lane all of them.  Here the entries found so far
// decide: the k-th goes to lane k % P, the P counts differ by one at most, and
// an atom overflows only when its whole list does.  `redo` (equal on an atom's
// lanes) says whose lists are made; the order depends on the atom and P alone.
// Whole warps; some 35 instructions per P atoms, run when a sub-list overflowed.
template <int P, class PosFn>
__device__ __forceinline__ int deal_sublist(int i, int q, bool redo, PosFn pos_hi, int N, float rl2u,
                                            uint16_t* nb, uint32_t col, uint32_t ncols, int cap_sub,
                                            int* status) {
  const int group = threadIdx.x & 31 & ~(P - 1);  // the atom's first lane
  const Hi3 pi = redo ? pos_hi(i) : Hi3{0u, 0u, 0u};
  int cnt = 0, total = 0;
  uint2 blk = make_uint2(0u, 0u);  // the last four entries
  uint2* out = reinterpret_cast<uint2*>(nb) + col;
#pragma unroll 1
  for (int j0 = 0; j0 < N; j0 += P) {
    const int j = j0 + q;
    const bool hit = redo && j < N && j != i && sep2_hi(pi, pos_hi(j)) < rl2u;
    uint32_t b = (__ballot_sync(0xffffffffu, hit) >> group) & ((1u << P) - 1u);
    const int k = (q - total) & (P - 1);  // which of these hits is this lane's
    total += __popc(b);
    for (int s = 0; s < k; ++s) b &= b - 1;
    if (b == 0u) continue;
    blk.x = __funnelshift_r(blk.x, blk.y, 16);
    blk.y = __byte_perm(blk.y, (uint32_t)(j0 + __ffs(b) - 1), 0x5432);
    if ((cnt & 3) == 3) {
      if (cnt < cap_sub) *out = blk;
      out += ncols;
    }
    ++cnt;
  }
  return finish_sublist(cnt, blk, out, i, false, cap_sub, status);
}

// The list of a small replica, by testing every atom: lane q takes the atoms j
// with j % P == q, in increasing order: 20 instructions an atom, no divergence.
// Both builds share an atom's work among its P lanes, so the line between them is
// a number of atoms, and their cost grows with N here and with the list there.
// Steps with a rebuild in 2.6 of them (four replicas, skin 0.1), testing every atom
// against screening, us: 256 atoms P = 1, 2, 4 11.9, 9.0, 6.8 against 17.3, 11.5,
// 8.3; 500 atoms P = 1, 2, 4 (eight CTAs) 15.4, 11.7, 8.6 against 21.1, 12.6, 9.5;
// 864 atoms P = 4 on four and eight CTAs 21.9 and 15.0 against 14.2 and 11.3 (no
// FCC box lies between).  With eight lanes screening gains at 864 atoms, 13.1
// against 14.6, but would need room for its notes.
template <int P, class PosFn>
__device__ __forceinline__ int build_sublist_direct(int i, int q, bool own, PosFn pos_hi, int N,
                                                    float rl2u, uint16_t* nb, uint32_t col,
                                                    uint32_t ncols, int cap_sub, int* status) {
  if (!own) return 0;
  const Hi3 pi = pos_hi(i);
  int cnt = 0;
  uint2 blk = make_uint2(0u, 0u);  // the last four entries
  uint2* out = reinterpret_cast<uint2*>(nb) + col;
  bool coincident = false;
#pragma unroll 4
  for (int j = q; j < N; j += P) {
    const float r2 = sep2_hi(pi, pos_hi(j));
    const bool add = r2 < rl2u && j != i;
    coincident |= add && r2 == 0.0f;
    if (add) {
      blk.x = __funnelshift_r(blk.x, blk.y, 16);
      blk.y = __byte_perm(blk.y, (uint32_t)j, 0x5432);
    }
    const bool full = add && (cnt & 3) == 3;
    if (full && cnt < cap_sub) *out = blk;
    if (full) out += ncols;
    cnt += add ? 1 : 0;
  }
  return finish_sublist(cnt, blk, out, i, coincident, cap_sub, status);
}

// Sub-list of lane q (of P) of atom i, by whole warps (every lane of the warp
// calls; `own` says whether it holds an atom; iw: the warp's first atom): entry
// k at element ((k / 4) * ncols + col) * 4 + k % 4 of nb, written four at a
// time, the last four filled up with the atom's own index.  raw, rcol, rncols:
// room for max_notes >= 1 notes, one 8-byte word each, laid out likewise.  act: this
// warp's row list.
//
// Tile v of a row (v = 0..3) holds the atoms t + 8 v + 4 c at columns 2 t + c,
// and lane 4 g + t gets columns 2 t, 2 t + 1 of the tile rows g and g + 8: it
// sees the row's atoms j with j % 4 == t, in increasing order.  Tile rows are
// the warp's atoms so placed that the four lanes 4 g + t own the atoms of the
// rows g, g + 8 (of one tile, or two for P = 1); they swap their masks so that
// each keeps its own atom's.  Neighbouring atoms go to different lanes of an
// atom: its sub-lists are nearly equal.  The order of a sub-list (by row, then
// column, then tile) depends on the atom and P alone, so that the FP32 sums, and
// with them the trajectories, do not change with the cluster size.
template <int P, class PosFn>
__device__ __forceinline__ int build_sublist(int i, bool own, int iw, PosFn pos_hi, int N,
                                             const uint4* hk, const uint2* box, uint8_t* act,
                                             float rl2u, uint16_t* nb, uint32_t col,
                                             uint32_t ncols, uint16_t* raw, uint32_t rcol,
                                             uint32_t rncols, int max_notes, int cap_sub,
                                             int* status) {
  static_assert(P <= 4, "eight threads an atom: build_sublist_direct");
  const int lane = threadIdx.x & 31, t = lane & 3, g = lane >> 2;
  if (!__any_sync(0xffffffffu, own)) return 0;
  const Hi3 pi = own ? pos_hi(i) : Hi3{0u, 0u, 0u};
  // the rows in reach: gap between the boxes, in units of L / 256 (a byte
  // stands for a unit's width)
  const float rl = sqrtf(rl2u);
  int nact = 0;
  {
    const uint2 mine = warp_box(pack8(pi), own);
    const float r8 = rl * 5.9604644775390625e-08f;
    const int gap_max = (int)ceilf(r8 * r8) + 1;
    const int nrow = (N + 31) / 32;
    for (int r0 = 0; r0 < nrow; r0 += 32) {
      bool near = false;
      if (r0 + lane < nrow) {
        const uint2 b = box[r0 + lane];
        int g2 = 0;
#pragma unroll
        for (int d = 0; d < 24; d += 8) {
          const int e = abs((int)(int8_t)((b.x >> d) - (mine.x >> d)));
          const int gap = max(0, e - (int)((b.y >> d) & 255u) - (int)((mine.y >> d) & 255u) - 1);
          g2 += gap * gap;
        }
        near = g2 <= gap_max;
      }
      const uint32_t bal = __ballot_sync(0xffffffffu, near);
      if (near) act[nact + __popc(bal & ((1u << lane) - 1u))] = (uint8_t)(r0 + lane);
      nact += __popc(bal);
    }
    if (lane < 4) act[nact + lane] = 0;  // for the rest of the last four
    __syncwarp();
  }
  // tile rows: minus the atoms' vectors, 1 and the limit.  Below it by 2.2e-3:
  // each of the twelve f16 values is off by at most 2^-12, which moves S by at
  // most 6 sqrt 2 2^-12 = 2.1e-3
  constexpr int NT = P == 1 ? 2 : 1;  // tiles
  uint32_t A[NT][2];
  {
    const float lim = 3.0f * __cosf(rl * (1.4629180792671596e-09f * 0.57735026918962576f)) - 2.2e-3f;
    const uint32_t lim2 = 0x3C00u | ((uint32_t)__half_as_ushort(__float2half_rd(lim)) << 16);
    const uint32_t* h = reinterpret_cast<const uint32_t*>(hk);
#pragma unroll
    for (int k = 0; k < NT; ++k)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int a = P == 1 ? 4 * g + 2 * k + u : (P == 2 ? 2 * g + u : g);
        A[k][u] = t == 3 ? lim2 : h[min(iw + a, N - 1) * 4 + t] ^ 0x80008000u;
      }
  }
  int cnt = 0, nm = 0;             // entries, notes
  uint2 blk = make_uint2(0u, 0u);  // the last four entries
  uint2* out = reinterpret_cast<uint2*>(nb) + col;
  uint2* const rawp = reinterpret_cast<uint2*>(raw) + rcol;
  int zeros = 0;
  // the exact test of the candidates noted so far (whole warps; without
  // branches: a lane that has none left tests something, and keeps nothing).
  // Bit 31 - k of a note's mask .x stands for an atom 4 (k % 8) + column of the
  // row in byte k / 8 of .y.
  auto drain = [&]() {
    uint2 cur = make_uint2(0u, 0u), next = cur;
    if (nm > 0) cur = rawp[0];
    if (nm > 1) next = rawp[rncols];
    int left = nm - 1;  // notes after `cur`
    const uint2* in = rawp + 2 * (size_t)rncols;
    while (__any_sync(0xffffffffu, cur.x != 0u)) {
      const uint32_t k = (uint32_t)__clz(cur.x) & 31u;
      const uint32_t column = P == 1 ? k >> 3 : (P == 2 ? (uint32_t)(t & 1) + ((k >> 2) & 2u) : (uint32_t)t);
      const uint32_t j = ((cur.y >> (k & 24u)) & 255u) * 32u + (k & 7u) * 4u + column;
      const float r2 = sep2_hi(pi, pos_hi((int)j));
      const bool in_list = cur.x != 0u && r2 < rl2u;
      const bool zero = in_list && r2 == 0.0f;  // the atom itself, or another at the same point
      const bool add = in_list && !zero;
      zeros += zero ? 1 : 0;
      cur.x &= ~(0x80000000u >> k);
      if (add) {
        blk.x = __funnelshift_r(blk.x, blk.y, 16);
        blk.y = __byte_perm(blk.y, j, 0x5432);
      }
      const bool full = add && (cnt & 3) == 3;
      if (full && cnt < cap_sub) *out = blk;
      if (full) out += ncols;
      cnt += add ? 1 : 0;
      const bool turn = cur.x == 0u && left > 0;
      if (turn) cur = next;
      left -= turn ? 1 : 0;
      if (turn && left > 0) next = *in;
      if (turn) in += rncols;
    }
    nm = 0;
  };
  const uint32_t hk_lane = (uint32_t)__cvta_generic_to_shared(hk) +
                           (uint32_t)(((lane & 7) >> 1) + (lane & 24) + 4 * (lane & 1)) * 16u;
  constexpr int NM = P == 1 ? 4 : (P == 2 ? 2 : 1);  // masks a lane keeps of four rows
  for (int a0 = 0; a0 < nact; a0 += 4) {
    uint32_t m[2 * NT] = {};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      uint32_t b[4];
      asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                   : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3])
                   : "r"(hk_lane + (uint32_t)act[a0 + u] * 512u)
                   : "memory");
#pragma unroll
      for (int v = 0; v < 4; ++v)
#pragma unroll
        for (int k = 0; k < NT; ++k) {
          float c0, c1, c2, c3;
          asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5}, {%6}, "
              "{%7, %7, %7, %7};"
              : "=f"(c0), "=f"(c1), "=f"(c2), "=f"(c3)
              : "r"(A[k][0]), "r"(A[k][1]), "r"(b[v]), "f"(0.0f));
          m[2 * k] = __funnelshift_l(__float_as_uint(c0), m[2 * k], 1);
          m[2 * k] = __funnelshift_l(__float_as_uint(c1), m[2 * k], 1);
          if (P <= 2) {
            m[2 * k + 1] = __funnelshift_l(__float_as_uint(c2), m[2 * k + 1], 1);
            m[2 * k + 1] = __funnelshift_l(__float_as_uint(c3), m[2 * k + 1], 1);
          }
        }
    }
    // each lane's own atom's masks (a byte a row, the first row on top): of the
    // columns t, and of the columns t ^ 1, t ^ 2, t ^ 3 (P = 1) or t ^ 2 (P = 2).
    // Nothing of rows past the last one, nothing for lanes without an atom
    const uint32_t valid = !own ? 0u : (nact - a0 >= 4 ? 0xffffffffu : ~(0xffffffffu >> (8 * (nact - a0))));
    uint32_t mk[NM];
    if (P == 1) {
      uint32_t w[4];
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int want = t ^ x;  // the lane that this one gives to owns row `want`
        const uint32_t give = want & 2 ? (want & 1 ? m[2 * NT - 1] : m[2 * NT - 2])
                                       : (want & 1 ? m[1] : m[0]);
        w[x] = (x == 0 ? give : __shfl_xor_sync(0xffffffffu, give, x)) & valid;
      }
      // a note a row, the columns 0..3 from the top byte down
      const uint32_t l0 = __byte_perm(w[0], w[1], 0x5140), l1 = __byte_perm(w[2], w[3], 0x5140),
                     h0 = __byte_perm(w[0], w[1], 0x7362), h1 = __byte_perm(w[2], w[3], 0x7362);
      const uint32_t order = 0x3210u ^ ((uint32_t)(t ^ 3) * 0x1111u);
      mk[0] = __byte_perm(__byte_perm(h0, h1, 0x7632), 0, order);
      mk[1 % NM] = __byte_perm(__byte_perm(h0, h1, 0x5410), 0, order);
      mk[2 % NM] = __byte_perm(__byte_perm(l0, l1, 0x7632), 0, order);
      mk[3 % NM] = __byte_perm(__byte_perm(l0, l1, 0x5410), 0, order);
    } else if (P == 2) {
      const uint32_t own_cols = (t & 2 ? m[1] : m[0]) & valid;
      const uint32_t others = __shfl_xor_sync(0xffffffffu, t & 2 ? m[0] : m[1], 2) & valid;
      const uint32_t c0 = t & 2 ? others : own_cols, c1 = t & 2 ? own_cols : others;
      // a note two rows, of each the columns t & 1, then those two further
      mk[0] = __byte_perm(c0, c1, 0x3726);
      mk[NM - 1] = __byte_perm(c0, c1, 0x1504);
    } else {
      mk[0] = m[0] & valid;
    }
    const uint32_t rows4 = *reinterpret_cast<const uint32_t*>(act + a0);
#pragma unroll 1
    for (int x = 0; x < NM; ++x) {
      const uint32_t w = mk[0];
#pragma unroll
      for (int y = 0; y + 1 < NM; ++y) mk[y] = mk[y + 1];
      if (__any_sync(0xffffffffu, nm == max_notes)) drain();
      // the row of each byte from the top, lowest byte first
      const uint32_t sel = P == 1 ? x * 0x1111u : (P == 2 ? 0x1100u + x * 0x2222u : 0x3210u);
      if (w) rawp[(size_t)nm++ * rncols] = make_uint2(w, __byte_perm(rows4, 0, sel));
    }
  }
  drain();
  if (!own) return 0;
  // of the atom's lanes, the one whose columns hold the atom met it once
  const bool self = P == 1 || (P == 2 && (t & 1) == (i & 1)) || (P == 4 && t == (i & 3));
  return finish_sublist(cnt, blk, out, i, zeros > (self ? 1 : 0), cap_sub, status);
}

// Mixed-precision forces of atom i from this lane's sub-list; see mixed_pair2.
// ENERGY: also the pair energies (only when U is reported).
template <bool ENERGY>
__device__ __forceinline__ PairAcc mixed_sublist_forces(Hi3 pi, const uint4* pos,
                                                        const uint16_t* __restrict__ nb,
                                                        uint32_t col, uint32_t ncols, int cnt,
                                                        const StepConst& K) {
  PairAcc a{0ull, 0ull, 0ull, 0ull, 0ull, 3.0e38f};
  const f32x2 cs = pack2(K.cs, K.cs), c1 = pack2(K.c1, K.c1), c3 = pack2(K.c3, K.c3);
  const f32x2 nhi = pack2(-K.rc2u_hi, -K.rc2u_hi);
  const uint2* list = reinterpret_cast<const uint2*>(nb) + col;
  const int nblk = (cnt + 3) >> 2;
  const int nfull = cnt >> 2;
  uint2 w = nblk > 0 ? *list : make_uint2(0u, 0u);
  for (int kb = 0; kb < nfull; ++kb) {
    // the next block of indices is requested before this block is used
    list += ncols;
    const uint2 wn = kb + 1 < nblk ? *list : w;
    const uint4 p0 = pos[w.x & 0xFFFFu], p1 = pos[w.x >> 16];
    const uint4 p2 = pos[w.y & 0xFFFFu], p3 = pos[w.y >> 16];
    mixed_pair2<ENERGY, false>(pi, p0, p1, cs, c1, c3, nhi, 2, a);
    mixed_pair2<ENERGY, false>(pi, p2, p3, cs, c1, c3, nhi, 2, a);
    w = wn;
  }
  if (nblk > nfull) {  // the last block, in part padding
    const int left = cnt & 3;
    const uint4 p0 = pos[w.x & 0xFFFFu], p1 = pos[w.x >> 16];
    mixed_pair2<ENERGY, true>(pi, p0, p1, cs, c1, c3, nhi, left, a);
    const uint4 p2 = pos[w.y & 0xFFFFu];
    mixed_pair2<ENERGY, true>(pi, p2, p2, cs, c1, c3, nhi, left - 2, a);
  }
  return a;
}

// Whole warps: the lanes that met an r^2 near the band (`near`) take out again
// what the 42-bit separations put outside rc.  The warp goes over such a lane's
// list together (one lane alone would hold up its CTA for as long as the whole
// pair loop takes, in most steps of a large replica).
template <bool ENERGY>
__device__ __forceinline__ void mixed_cut_fix(bool near, int i, const uint4* pos,
                                              const uint16_t* __restrict__ nb, uint32_t col,
                                              uint32_t ncols, int cnt, const StepConst& K,
                                              PairAcc& a) {
  const int lane = threadIdx.x & 31;
  for (uint32_t todo = __ballot_sync(0xffffffffu, near); todo; todo &= todo - 1) {
    const int src = __ffs(todo) - 1;
    const int n = __shfl_sync(0xffffffffu, cnt, src);
    const uint32_t c = __shfl_sync(0xffffffffu, col, src);
    const uint4 pi = pos[__shfl_sync(0xffffffffu, i, src)];
    for (int k0 = 0; k0 < n; k0 += 32) {
      const int k = k0 + lane;
      int j = 0;
      bool band = false;
      if (k < n) {
        j = nb[((size_t)(k >> 2) * ncols + c) * 4 + (k & 3)];
        const uint4 pj = pos[j];
        const float dx = (float)(int)(pj.x - pi.x), dy = (float)(int)(pj.y - pi.y),
                    dz = (float)(int)(pj.z - pi.z);
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        band = r2 > K.rc2u_lo && r2 < K.rc2u_hi && !inside_cutoff_42(pi, pj, K.rc2x);
      }
      for (uint32_t hit = __ballot_sync(0xffffffffu, band); hit; hit &= hit - 1) {
        const uint4 pj = pos[__shfl_sync(0xffffffffu, j, __ffs(hit) - 1)];
        if (lane == src) {
          const float dx = (float)(int)(pj.x - pi.x), dy = (float)(int)(pj.y - pi.y),
                      dz = (float)(int)(pj.z - pi.z);
          mixed_pair_remove<ENERGY>(dx, dy, dz, fmaf(dx, dx, fmaf(dy, dy, dz * dz)), K, a);
        }
      }
    }
  }
}

// v 2^-64 as a double, v a positive normal float, by its bits (the conversion
// instruction runs on the FP64 unit).
__device__ __forceinline__ double float_to_double_2m64(float v) {
  const uint32_t u = __float_as_uint(v);
  return __hiloint2double((int)((u >> 3) + 0x34000000u), (int)(u << 29));
}

// FP64 force of one pair, separation d (units of L / 2^64), hi the FP32 r^2 of
// its top words: 17 FP64 operations.  1/r^2 starts from the FP32 value x0 with
// one third-order step x = x0 (1 + e + e^2), e = 1 - r^2 x0 (the partial sum
// of the geometric series of 1 / (1 - e)); |e| < 4e-6 while the top words tell the
// atoms 2^20 units (2.4e-4 L) and more apart.  All stay in units of the separation:
// s = 1/r^2 is about 1e-37 and s^7 about 1e-260, in range.
// edge (fp64_edge of the top words' r^2): near the cutoff, decided on the FP64 r^2,
// or closer than that, x0 from the FP64 r^2 (no liquid has such pairs; a test in
// every pair took 6 % of a step).
__device__ __forceinline__ bool fp64_edge(float r2, const StepConst& K) {
  return r2 > K.rc2u_lo || r2 < 0x1p40f;
}
struct Fp64Acc {
  double fx, fy, fz, e;  // sums of 24 s^4 (1 - 2 s^3) d and of the pair energies
};
struct Fp64Const {
  double m2, rc2, uc;  // -2 s3 factor (2^64 / L)^6, rc^2 in these units, shift
};
template <bool ENERGY>
__device__ __forceinline__ void fp64_pair(const Pos64& pi, const Pos64& pj, const Hi3& hi, bool edge,
                                          const Fp64Const& c, Fp64Acc& a) {
  const double dx = (double)(long long)(pj.x - pi.x), dy = (double)(long long)(pj.y - pi.y),
               dz = (double)(long long)(pj.z - pi.z);
  const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
  double x0 = float_to_double_2m64(
      rcp_approx(sep2_hi(hi, Hi3{(uint32_t)(pj.x >> 32), (uint32_t)(pj.y >> 32), (uint32_t)(pj.z >> 32)})));
  if (edge) {
    if (!(r2 < c.rc2)) return;
    if (r2 < 0x1p105) x0 = (double)rcp_approx((float)r2);
  }
  const double er = fma(-r2, x0, 1.0);
  const double s = fma(x0, fma(er, er, er), x0);
  const double s2 = s * s, s3 = s2 * s;
  const double q = fma(c.m2, s3, 1.0);
  const double fs = (s2 * s2) * q;
  a.fx = fma(fs, dx, a.fx);
  a.fy = fma(fs, dy, a.fy);
  a.fz = fma(fs, dz, a.fz);
  if (ENERGY) {
    const double t = c.m2 * s3;  // -2 s^3 in sigma units: 4 (s^6 - s^3) = t (t + 2)
    a.e += fma(t, t + 2.0, -c.uc);
  }
}

// FP64 pair forces of atom i from its sub-lists, whole warps.  The FP64 unit
// (1.7 operations per clock and SM, whatever the active lanes) bounds this
// loop, so everything else is kept off it, and its turns are kept full: FP32
// distances on the top 32 bits first pick the entries inside the cutoff (55 of
// 95 at the default skin), 32 entries of a lane at a time; only those take an
// FP64 turn.  With P >= 4 lanes of an atom the hits of all of them are then
// dealt out evenly (buf: 32 noted entries a thread in shared memory), since
// one lane's 14 +- 3 hits would make the fullest of 32 lanes need 21 to 24
// turns; with fewer lanes each goes through its own hits (a bit mask), 28 +- 4
// or 55 +- 5 of them.  Entries within 2e-6 of rc^2, and very close ones, are
// marked (fp64_edge).
template <bool ENERGY, int P>
__device__ __forceinline__ Fp64Acc fp64_sublist_forces(const Pos64* pos, int i, bool own,
                                                       const uint16_t* __restrict__ nb, uint32_t col,
                                                       uint32_t ncols, int cnt, uint16_t* buf,
                                                       const StepConst& K, const Fp64Const& c) {
  Fp64Acc a{0.0, 0.0, 0.0, 0.0};
  const Pos64 pi = pos[own ? i : 0];
  const Hi3 hi{(uint32_t)(pi.x >> 32), (uint32_t)(pi.y >> 32), (uint32_t)(pi.z >> 32)};
  if (!own) cnt = 0;
  const int nmax = __reduce_max_sync(0xffffffffu, cnt);
  auto hi_of = [&](int j) {
    return Hi3{(uint32_t)(pos[j].x >> 32), (uint32_t)(pos[j].y >> 32), (uint32_t)(pos[j].z >> 32)};
  };
  for (int k0 = 0; k0 < nmax; k0 += 32) {
    uint32_t m = 0, band = 0;  // P < 4: bit k is entry k0 + k
    int n = 0;                 // P >= 4: noted entries
    uint16_t* mine = P >= 4 ? buf + threadIdx.x * 32 : nullptr;
    const uint2* list = reinterpret_cast<const uint2*>(nb) + (size_t)(k0 >> 2) * ncols + col;
    uint2 wn = make_uint2(0u, 0u);
    if (k0 < cnt) wn = *list;
    for (int b = 0; b < 32 && k0 + b < cnt; b += 4) {
      const uint2 w = wn;
      list += ncols;
      if (k0 + b + 4 < cnt) wn = *list;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t j = ((k < 2 ? w.x : w.y) >> (16 * (k & 1))) & 0xFFFFu;
        const float r2 = sep2_hi(hi, hi_of((int)j));
        const bool hit = k0 + b + k < cnt && r2 < K.rc2u_hi, edge = fp64_edge(r2, K);
        if (P >= 4) {
          if (hit) mine[n++] = (uint16_t)(j | (edge ? 0x8000u : 0u));
        } else if (hit) {
          m |= 1u << (b + k);
          if (edge) band |= 1u << (b + k);
        }
      }
    }
    if (P >= 4) {
      // hit number r of the atom, r = q, q + P, ...: note r - first[l] of lane l
      const int lane = threadIdx.x & 31, g0 = lane & ~(P - 1);
      int first[P + 1];
      first[0] = 0;
#pragma unroll
      for (int l = 0; l < P; ++l) first[l + 1] = first[l] + __shfl_sync(0xffffffffu, n, g0 + l);
      __syncwarp();
      const uint16_t* group = buf + (threadIdx.x & ~(P - 1)) * 32;
      for (int r = lane & (P - 1); __any_sync(0xffffffffu, r < first[P]); r += P) {
        if (r < first[P]) {
          int at = r;
#pragma unroll
          for (int l = 1; l < P; ++l)
            if (r >= first[l]) at = r - first[l] + 32 * l;
          const uint32_t j = group[at];
          fp64_pair<ENERGY>(pi, pos[j & 0x7FFFu], hi, j >> 15, c, a);
        }
      }
      __syncwarp();
    } else {
      auto entry = [&](int k) {
        return (int)nb[((size_t)((k0 + k) >> 2) * ncols + col) * 4 + (k & 3)];
      };
      int k = __ffs(m) - 1;
      int j = k >= 0 ? entry(k) : 0;
      while (__any_sync(0xffffffffu, m != 0u)) {
        if (m != 0u) {
          const int jc = j;
          const bool edge = (band >> k) & 1u;
          m &= m - 1;
          if (m != 0u) {  // the next turn's entry is read one turn ahead
            k = __ffs(m) - 1;
            j = entry(k);
          }
          fp64_pair<ENERGY>(pi, pos[jc], hi, edge, c, a);
        }
      }
    }
  }
  return a;
}

template <int P>
__device__ __forceinline__ float group_sum(float v) {
#pragma unroll
  for (int o = 1; o < P; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
template <int P>
__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
  for (int o = 1; o < P; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
template <int P>
__device__ __forceinline__ int group_sum(int v) {
#pragma unroll
  for (int o = 1; o < P; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Per-step thermostat draws, generated ahead of the step (off the critical
// path).  With K the kinetic energy after the second half kick, the SVR update
// is K'/K = 1 + delta with delta = (c - 1) + (a + b sqrt(K)) / K, where
// a = (1 - c) Kbar (R1^2 + S) / Nf and b = 2 R1 sqrt(c (1 - c) Kbar / Nf); the
// factor alpha = +-sqrt(1 + delta) is negative when R1 + g sqrt(K) < 0,
// g = sqrt(c Nf / ((1 - c) Kbar)).
struct SvrStep {
  double r1, s;  // the draws (FP64 path)
  float r1f, sf; // the draws (mixed path)
  int bad;       // the Gamma sampler hit its trial cap
  int pad;
};
static_assert(sizeof(SvrStep) == kSvrStepBytes, "thermostat record size");

__device__ inline SvrStep svr_step(bool fp64, int nf, uint64_t seed, uint64_t stream,
                                   uint64_t n, int* capped) {
  SvrStep t;
  t.bad = 0;
  t.pad = 0;
  if (fp64) {
    const double2 z = svr_noise(nf, seed, stream, n, capped);
    t.r1 = z.x;
    t.s = z.y;
    t.r1f = (float)z.x;
    t.sf = (float)z.y;
  } else {
    const float2 z = svr_noise_f32(nf, seed, stream, n, capped);
    t.r1 = z.x;
    t.s = z.y;
    t.r1f = z.x;
    t.sf = z.y;
  }
  return t;
}

// alpha - 1 in FP32 without cancellation: sqrt(1 + delta) - 1 = delta / (1 + sqrt(1 + delta)).
// The temperature-dependent constants are read from K at the step (the
// target may change within a launch).
__device__ __forceinline__ float svr_eps(const SvrStep& t, float Kf, const StepConst& K) {
  const float a = K.af * fmaf(t.r1f, t.r1f, t.sf);
  const float b = K.bf * t.r1f;
  const float sk = sqrtf(Kf);
  const float delta = K.cm1f + (a + b * sk) / Kf;
  const float root = sqrtf(1.0f + delta);
  if (t.r1f + K.gf * sk < 0.0f) return -1.0f - root;  // alpha = -sqrt(1 + delta)
  return delta / (1.0f + root);
}

// Fixed-point scales of the mixed path: velocities in units of 2^-48 (64-bit,
// |v| < 2^15), energy partial sums in units of 2^-28 (64-bit, |sum| < 2^35).
constexpr float kVelScale = 281474976710656.0f;        // 2^48
constexpr float kVelUnit = 3.5527136788005009e-15f;   // 2^-48
constexpr float kEnScale = 268435456.0f;              // 2^28
constexpr double kEnUnit = 3.7252902984619140625e-09; // 2^-28

__device__ __forceinline__ long long warp_sum_i64(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Metropolis rule of the Implementation section for the pair (a before b in
// ladder order), generalised to parameter sets (T, lam) whose Hamiltonians
// are K + lam U_LJ: D = (lam_a/T_a - lam_b/T_b)(U_a/lam_a - U_b/lam_b) with U
// the stored (scaled) potential energies; lam = 1 gives
// D = (1/T_a - 1/T_b)(U_a - U_b).  Accept iff D >= 0 or r < exp(D), r the
// uniform of the lower replica id for this attempt.
__device__ __forceinline__ bool metropolis(double Ta, double Tb, double la, double lb, double Ua,
                                           double Ub, uint64_t seed, int id_lo, int64_t attempt) {
  const double d = __dmul_rn(__dsub_rn(__ddiv_rn(la, Ta), __ddiv_rn(lb, Tb)),
                             __dsub_rn(__ddiv_rn(Ua, la), __ddiv_rn(Ub, lb)));
  if (d >= 0.0) return true;
  const Uni4 u = uniforms(seed, (uint64_t)id_lo, (uint64_t)attempt, kTagExch, 0ull);
  return u.u0 < exp(d);
}

// Partner position of ladder position q: pairs (q, q + d) for q - o in
// [0, d) modulo 2d, o = p d (p the parity offset); -1 when unpaired.
__device__ __forceinline__ int ladder_partner(int q, int R, int p, int d) {
  const int o = p * d;
  if (q < o) return -1;
  if ((q - o) % (2 * d) < d) return q + d < R ? q + d : -1;
  return q - d;
}

__device__ __forceinline__ int pair_offset(int mode, uint64_t seed, int64_t attempt) {
  if (mode == 0) return (int)(attempt & 1);
  const Uni4 u = uniforms(seed, ~0ull, (uint64_t)attempt, kTagParity, 0ull);
  return u.u0 < 0.5 ? 0 : 1;
}

// ------------------------------------------------------ free-running exchange
// The asynchronous scheme of the Implementation section inside one persistent
// launch: every replica integrates without stopping; the master of pattern k
// (member (attempt + k) mod R, so the role rotates with every attempt), after
// nx of its own steps since it took part in pattern k - 1, waits until every
// member has taken part in pattern k - 1, sorts the members' temperatures and
// publishes pattern k.  Each replica checks for a new pattern after every
// step; when one is there it publishes (T, U), waits for its partner's pair,
// and both take the same Metropolis decision with the lower id's uniform.
// Every wait is bounded (fr.wait_ns of the global timer, and an iteration
// cap); a replica that gives up or fails raises the ensemble's abort flag.
// The master's collection of temperatures also ends when that flag is up.  A
// replica waiting for its partner's pair message does not: the partner has
// already seen the pattern (it is issued before any abort can follow from
// it), so it either publishes or has stopped answering, and ending the wait
// early on the flag could leave one member of a pair swapped and the other
// not.

// true when *p >= want; false when the wait ran out or abort_flag (if not
// null) was raised
__device__ bool wait_at_least(const int* p, int want, const int* abort_flag, uint64_t wait_ns) {
  const uint64_t t0 = global_ns();
  for (uint32_t it = 0; it < (1u << 26); ++it) {
    if (ld_acquire(p) >= want) return true;
    if (abort_flag && *reinterpret_cast<const volatile int*>(abort_flag)) return false;
    if ((it & 63u) == 63u && global_ns() - t0 > wait_ns) return false;
    __nanosleep(32);
  }
  return false;
}

// The master's part, by one warp: pattern k of ensemble e.  Returns false when
// a wait gave up.
__device__ bool issue_pattern(const FreeDev& fr, const StateDev& S, const EnsHdr& E, int e, int k,
                              int64_t attempt) {
  const int lane = threadIdx.x & 31;
  const int R = E.R, base = E.rep_off;
  bool ok = true;
  if (k > 0)
    for (int m = lane; m < R && ok; m += 32) ok = wait_at_least(fr.done + base + m, k, fr.abort_ + e, fr.wait_ns);
  ok = __all_sync(0xffffffffu, ok);
  if (!ok) return false;
  __threadfence();
  // ladder keys T/lam (positive: their bit patterns order like the values)
  for (int m = lane; m < R; m += 32)
    fr.key[base + m] = __ldcg(S.T + base + m) / __ldcg(S.lam + base + m);
  __syncwarp();
  const long long* key = reinterpret_cast<const long long*>(fr.key + base);
  for (int m = lane; m < R; m += 32) {
    const long long t = key[m];
    int rank = 0;
    for (int b = 0; b < R; ++b) {
      const long long u = key[b];
      rank += (u < t) || (u == t && b < m);
    }
    fr.order[base + rank] = m;
    fr.pos[base + m] = rank;
  }
  __syncwarp();
  const int p = pair_offset(E.parity_mode, E.seed, attempt);
  const int d = max(1, E.xdist);
  for (int m = lane; m < R; m += 32) {
    const int q = ladder_partner(fr.pos[base + m], R, p, d);
    fr.partner[base + m] = q < 0 ? -1 : fr.order[base + q];
  }
  __syncwarp();
  if (lane == 0) {
    __threadfence();
    st_release(fr.issue + e, k + 1);
  }
  return true;
}

// A replica's part of pattern k (one thread), parameters (Tcur, lcur).
// Returns the velocity scale sqrt(T_new / T_old) and sets *us =
// lam_new / lam_old (both 1 when not accepted); *ok = false when the wait
// gave up.
__device__ double pair_exchange(const FreeDev& fr, const StateDev& S, const EnsHdr& E,
                                const RepDev& rd, int r, int k, int64_t attempt, double Tcur,
                                double lcur, double U, double* Tnew, double* lnew, double* us,
                                int* partner_out, int* acc_out, bool* ok) {
  const int p = __ldcg(fr.partner + r);
  *Tnew = Tcur;
  *lnew = lcur;
  *us = 1.0;
  *partner_out = p;
  *acc_out = 0;
  *ok = true;
  if (p < 0) return 1.0;
  fr.slot[3 * r] = Tcur;
  fr.slot[3 * r + 1] = U;
  fr.slot[3 * r + 2] = lcur;
  __threadfence();
  st_release(fr.flag + r, k + 1);
  const int gp = E.rep_off + p;
  if (!wait_at_least(fr.flag + gp, k + 1, nullptr, fr.wait_ns)) {
    *ok = false;
    return 1.0;
  }
  __threadfence();
  const double Tp = __ldcg(fr.slot + 3 * gp), Up = __ldcg(fr.slot + 3 * gp + 1),
               lp = __ldcg(fr.slot + 3 * gp + 2);
  const int q = __ldcg(fr.pos + r), qp = __ldcg(fr.pos + gp);
  const bool lower = q < qp;  // this replica comes first in ladder order
  const int id_lo = min(rd.id, p);
  const bool accept = lower ? metropolis(Tcur, Tp, lcur, lp, U, Up, E.seed, id_lo, attempt)
                            : metropolis(Tp, Tcur, lp, lcur, Up, U, E.seed, id_lo, attempt);
  if (lower) {
    atomicAdd(reinterpret_cast<unsigned long long*>(S.pair_att + E.pair_off + q), 1ull);
    if (accept) atomicAdd(reinterpret_cast<unsigned long long*>(S.pair_acc + E.pair_off + q), 1ull);
  }
  if (!accept) return 1.0;
  *acc_out = 1;
  *Tnew = Tp;
  *lnew = lp;
  *us = lp / lcur;
  return sqrt(Tp / Tcur);
}

}  // namespace
}  // namespace re
