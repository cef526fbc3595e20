// re_forces.cu -- LJ forces and energy of one configuration given on the device
// (re_lj_forces_device, re_lj_forces_device_noalloc), without lists.
#include "re_md.cuh"

namespace re {
namespace {

// Fixed-point words of the caller's positions; clears the words of the call and
// keeps what f holds (which may be x): a call that fails gives it back.
__global__ void __launch_bounds__(256) direct_fix_kernel(const double* x, const double* f, DirectScratch s,
                                                         int N, double inv_l) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) {
    uint64_t q[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) q[d] = fix_from_double(x[3 * (size_t)i + d], inv_l);
    s.hi[i] = make_uint4((uint32_t)(q[0] >> 32), (uint32_t)(q[1] >> 32), (uint32_t)(q[2] >> 32), 0u);
    s.lo[i] = make_uint4((uint32_t)q[0], (uint32_t)q[1], (uint32_t)q[2], 0u);
  }
  for (int k = i; k < 3 * N; k += gridDim.x * blockDim.x) s.old[k] = f[k];
  if (i < 2) s.words[i] = 0;
}

// One warp per atom, W warps a CTA.  Every CTA holds the top 32 bits of all
// positions in shared memory; a warp tests 32 atoms at a time in FP32, notes
// those inside the cutoff (in increasing index) and computes 32 noted pairs at
// a time, in FP64 on the full words or in FP32 (MIXED), so that nearly all
// lanes work (the FP64 unit bounds the FP64 form).  All atoms are tested
// directly: at 4000 atoms 125 tests a lane, less than building cells and a list
// for one use and spread over all SMs (the former way, the context's prologue,
// ran on the 8 CTAs of one cluster: 38 us for 987 atoms in mixed precision, the
// plain path's list and force kernels 447 us for 2048 in FP64, against 17 us
// here, and 29 for 4000).  Energies: FP64 sums in a fixed order, by warp, CTA
// and, in the last CTA to finish, over the CTAs.
template <bool MIXED>
__global__ void __launch_bounds__(512) direct_force_kernel(DirectScratch s, int N, StepConst K,
                                                           Fp64Const c, double unit, double eunit,
                                                           int cap, double* __restrict__ f,
                                                           double* __restrict__ U) {
  extern __shared__ __align__(16) uint4 hi[];
  __shared__ double esum[16];
  __shared__ uint16_t noted[16][64];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = blockDim.x >> 5;
  for (int k = threadIdx.x; k < N; k += blockDim.x) hi[k] = s.hi[k];
  __syncthreads();
  const int i = blockIdx.x * W + warp;
  double e = 0.0;
  if (i < N) {
    auto hi_of = [&](int j) {
      const uint4 w = hi[j];
      return Hi3{w.x, w.y, w.z};
    };
    auto full = [&](int j) {
      const uint4 h = hi[j], l = s.lo[j];
      return Pos64{((uint64_t)h.x << 32) | l.x, ((uint64_t)h.y << 32) | l.y, ((uint64_t)h.z << 32) | l.z, 0ull};
    };
    const Hi3 ph = hi_of(i);
    const Pos64 pi = full(i);
    Fp64Acc a{0.0, 0.0, 0.0, 0.0};
    float gx = 0.0f, gy = 0.0f, gz = 0.0f, ge = 0.0f, gn = 0.0f;
    int near = 0, n = 0, st = 0;  // atoms within the list radius (this lane's), noted pairs
    auto pair = [&](int j, bool edge) {
      if (MIXED) {
        const Hi3 pj = hi_of(j);
        const float dx = (float)(int)(pj.x - ph.x), dy = (float)(int)(pj.y - ph.y),
                    dz = (float)(int)(pj.z - ph.z);
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        if (edge) {
          const Pos64 q = full(j);
          const double ex = (double)(long long)(q.x - pi.x), ey = (double)(long long)(q.y - pi.y),
                       ez = (double)(long long)(q.z - pi.z);
          if (!(fma(ex, ex, fma(ey, ey, ez * ez)) < c.rc2)) return;
        }
        // rounded to nearest: the approximate one is off by 4e-9 in the mean, s^7 by 3e-8
        const float v = __frcp_rn(r2) * K.cs, v2 = v * v, v3 = v2 * v, v4 = v2 * v2;
        const float u = fmaf(v3, K.c3, K.c1), fs = v4 * u;
        gx = fmaf(fs, dx, gx);
        gy = fmaf(fs, dy, gy);
        gz = fmaf(fs, dz, gz);
        ge = fmaf(v3 * K.c3, u + K.c1, ge);
        gn += 1.0f;
      } else {
        fp64_pair<true>(pi, full(j), ph, edge, c, a);
      }
    };
    uint16_t* note = noted[warp];
    // 32 atoms against atom i; nearly all tests end at the first branch
    auto test = [&](int j) {
      const float r2 = j < N ? sep2_hi(ph, hi_of(j)) : 3.0e38f;
      const bool close = r2 < K.rl2u;
      if (!__any_sync(0xffffffffu, close)) return;
      near += close && j != i ? 1 : 0;
      if (close && r2 == 0.0f && j != i) st = kStNumeric;  // at one point: no direction
      const bool hit = r2 < K.rc2u_hi && j != i;
      const uint32_t b = __ballot_sync(0xffffffffu, hit);
      if (hit) note[n + __popc(b & ((1u << lane) - 1u))] = (uint16_t)(j | (fp64_edge(r2, K) ? 0x8000 : 0));
      n += __popc(b);
      if (n >= 32) {
        __syncwarp();
        const uint32_t w = note[lane];
        const uint16_t rest = note[32 + lane];
        __syncwarp();
        note[lane] = rest;
        __syncwarp();
        n -= 32;
        pair((int)(w & 0x7FFFu), w >> 15);
      }
    };
    for (int j0 = 0; j0 < N; j0 += 32) test(j0 + lane);
    __syncwarp();
    if (lane < n) pair((int)(note[lane] & 0x7FFFu), note[lane] >> 15);
    // the four sums, halving what a lane holds with the distance: lanes 0-7 end
    // with F_x, 8-15 with F_y, 16-23 with F_z, 24-31 with the energy
    double v[4] = {MIXED ? (double)gx : a.fx, MIXED ? (double)gy : a.fy, MIXED ? (double)gz : a.fz,
                   MIXED ? (double)ge * eunit - K.uc * (double)gn : a.e};
    const bool h16 = lane & 16, h8 = lane & 8;
    double p = (h16 ? v[2] : v[0]) + __shfl_xor_sync(0xffffffffu, h16 ? v[0] : v[2], 16);
    double q = (h16 ? v[3] : v[1]) + __shfl_xor_sync(0xffffffffu, h16 ? v[1] : v[3], 16);
    p = (h8 ? q : p) + __shfl_xor_sync(0xffffffffu, h8 ? p : q, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
    if (!isfinite(p)) st |= kStNumeric;
    if ((lane & 7) == 0 && lane < 24) f[3 * (size_t)i + (lane >> 3)] = p * unit;
    e = __shfl_sync(0xffffffffu, p, 24);
    near = __reduce_add_sync(0xffffffffu, near);
    if (near > cap) st |= kStOverflow;
    st = __reduce_or_sync(0xffffffffu, (unsigned)st);
    if (lane == 0 && st) atomicOr(s.words + 1, st);
  }
  if (lane == 0) esum[warp] = e;
  __syncthreads();
  if (warp == 0) {
    const double t = warp_sum(lane < W ? esum[lane] : 0.0);
    if (lane == 0) {
      s.part[blockIdx.x] = t;
      __threadfence();
      last = atomicAdd(s.words, 1) == (int)gridDim.x - 1;
    }
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (__ldcg(s.words + 1) != 0) {  // failed: f and U stay as they were
    for (int k = threadIdx.x; k < 3 * N; k += blockDim.x) f[k] = s.old[k];
  } else if (warp == 0) {
    double u = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) u += __ldcg(s.part + b);
    u = warp_sum(u);
    if (lane == 0) *U = 0.5 * u;
  }
}

// Warps per CTA: two CTAs an SM hold all atoms up to 16 warps, four at least
// (each CTA reads all positions once).
int direct_warps(int N, int sms) { return std::min(16, std::max(4, (N + 2 * sms - 1) / (2 * sms))); }

}  // namespace

size_t direct_scratch_bytes(int N) {
  return (size_t)N * (32 + 3 * sizeof(double)) + (((size_t)N + 3) / 4 + 2) * sizeof(double);
}

cudaError_t launch_lj_direct(void* scratch, int N, const StepConst& K, bool mixed, int cap, int sms,
                             const double* x, double* f, double* U, int32_t** status,
                             cudaStream_t st) {
  if (N > kMaxNotedAtoms) return cudaErrorInvalidValue;
  DirectScratch s;
  s.hi = static_cast<uint4*>(scratch);
  s.lo = s.hi + N;
  s.old = reinterpret_cast<double*>(s.lo + N);
  s.part = s.old + 3 * (size_t)N;
  s.words = reinterpret_cast<int32_t*>(s.part + (N + 3) / 4);
  *status = s.words + 1;
  direct_fix_kernel<<<(N + 255) / 256, 256, 0, st>>>(x, f, s, N, K.inv_l);
  const int W = direct_warps(N, sms);
  const size_t smem = (size_t)N * 16;
  auto fn = mixed ? direct_force_kernel<true> : direct_force_kernel<false>;
  if (smem > 40 * 1024) {
    // the largest any call may ask for (beside the kernel's own 2.2 KB): a limit
    // of this call's size could undercut another thread's launch
    const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               std::max((int)smem, 232448 - 4096));
    if (e != cudaSuccess) return e;
  }
  const double i2 = 1.0 / (K.lam64 * K.lam64);  // (2^64 / L)^2
  const Fp64Const c{-2.0 * i2 * i2 * i2, K.rc2 * i2, K.uc};
  // of the pair sums: see lj2 and fp64_pair
  const double unit = mixed ? K.f24 * K.lam32 : 24.0 * i2 * i2 * i2 * (i2 * K.lam64);
  const double eunit = 1.0 / ((double)K.c1 * K.c1);
  fn<<<(N + W - 1) / W, 32 * W, smem, st>>>(s, N, K, c, unit, eunit, cap, f, U);
  return cudaGetLastError();
}

}  // namespace re
