// mx_detect_body.cuh -- the per-tile body of close-encounter detection
// (k_detect.cu), shared by its kernel and the persistent step kernel.
#pragma once
#include "mx_common.cuh"
#include "mx_encounter.cuh"

namespace mx {

// Big bodies staged per pass, in the block's dynamic shared memory: `chunk`
// = min(threads per block, most big bodies of a system) entries of each
// array (a disk with a few big bodies leaves the SM its shared memory).
__host__ __device__ __forceinline__ int det_chunk(int tile, int big_max) {
  const int c = big_max < tile ? big_max : tile;
  return c < 1 ? 1 : c;
}

// A staged big body: the FP32 copies the two screens read, in rows of 16 bytes
// (80 bytes a body, so that lanes reading different bodies spread over the
// banks).  The FP64 endpoints of the few pairs that pass are read from memory.
struct DetBig {
  float4 p0;   // x0, y0, z0, reach (encounter_reach)
  float4 v0;   // u0, v0, w0, rc
  float4 p1;   // x1, y1, z1, 1 if removed from the integration (Sec. 3.5)
  float4 v1;   // u1, v1, w1
  float4 pad;
};

// With fewer big bodies than this the kernel (FEW) has no first screen: every
// lane takes the big bodies in turn, and the FP64 endpoints stay at hand (the
// target's in registers, the big bodies' staged), since a small system's time
// is the latency of one warp (two giants + 1,000 planetesimals, and four cores
// + 100,000: 2 us of 14 a launch against the first screen).
constexpr int kDetMinScreen = 8;
__host__ __device__ __forceinline__ bool det_few(int big_max) { return big_max < kDetMinScreen; }

__host__ __device__ __forceinline__ size_t det_smem_bytes(int chunk, bool few) {
  return (size_t)chunk * (sizeof(DetBig) + (few ? 12 * sizeof(double) : 0));
}

// The FP64 test of a pair, from the endpoint states in memory.
static __device__ __noinline__ bool encounter_pair(const double* xv0, const double* xv1, size_t N,
                                                   int j, int g, double h, double rc2) {
  double a0[6], a1[6], b0[6], b1[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    a0[q] = xv0[q * N + j];
    a1[q] = xv1[q * N + j];
    b0[q] = xv0[q * N + g];
    b1[q] = xv1[q * N + g];
  }
  return encounter_fp64(a0, b0, a1, b1, h, rc2);
}

// xv0, xv1: 6 x N endpoint states; keys/count/cap: pair output.
// runs = 1 (the step): a target with more than kMaxGroup flagged big bodies
// would make a group larger than kMaxGroup, reported as ST_GROUP.
// Tile `bid`, one target per thread; dsm_det: the block's dynamic shared
// memory (det_smem_bytes).
template <bool FEW>
__device__ __forceinline__ void detect_tile(const Dev& d, const double* xv0, const double* xv1,
                                            unsigned char* flags, unsigned long long* keys,
                                            int* count, int cap, int runs, int bid,
                                            unsigned char* dsm_det) {
  const int chunk = det_chunk(blockDim.x, d.big_max);
  DetBig* sm = reinterpret_cast<DetBig*>(dsm_det);
  double* sd = reinterpret_cast<double*>(sm + chunk);   // FEW: 12 a body
  const Tile t = d.tiles[bid];
  const SysDev& S = d.sys[t.sys];
  const int N = d.N;
  const int j = t.start + threadIdx.x;
  // a deferred planetesimal is tested by the window's catch-up instead; a
  // removed body meets nothing
  const bool act = threadIdx.x < t.count && !(d.defer && d.lag[j]) && !removed(d, j);
  const int jl = j - S.off;
  const bool jbig = jl < S.nbig;
  const int lane = threadIdx.x & 31;
  const double h = S.h;
  const float hf = to_float_bits(h);
  float af[12];
  double rcj = 0.0;
  double ad[FEW ? 12 : 1];
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const double e0 = act ? xv0[(size_t)k * N + j] : 0.0, e1 = act ? xv1[(size_t)k * N + j] : 0.0;
    af[k] = to_float_bits(e0);
    af[6 + k] = to_float_bits(e1);
    if constexpr (FEW) {
      ad[k] = e0;
      ad[6 + k] = e1;
    }
  }
  if (act && jbig) rcj = d.brc[S.boff + jl];
  const float rcjf = to_float_bits(rcj);
  const float reach = FEW ? 0.0f : encounter_reach(af, rcjf, hf);
  int hits[kMaxGroup];
  int nh = 0;
  const unsigned long long tag = ((unsigned long long)(jbig ? 0u : 1u) << 63) |
                                 ((unsigned long long)(unsigned)j << 32);
  // writes the buffered hits of the lanes with `mine` set, each lane's as one
  // run (the warp takes its space with one atomic); every lane calls it
  auto flush = [&](bool mine) {
    const int own = mine ? nh : 0;
    int inc = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    const int total = __shfl_sync(0xffffffffu, inc, 31);
    if (total == 0) return;
    int base = 0;
    if (lane == 31) base = atomicAdd(count, total);
    base = __shfl_sync(0xffffffffu, base, 31);
    const int start = base + inc - own;
    for (int e = 0; e < own; ++e)
      if (start + e < cap) keys[start + e] = tag | (unsigned)(S.off + hits[e]);
    if (mine) nh = 0;
  };
  // the second screen and the FP64 test of staged big body k of the chunk at
  // c0, for the lanes with ok set; every lane calls it
  auto test = [&](int c0, int k, bool ok) {
    const int il = c0 + k;
    bool hit = false;
    // big-big pairs are tested once, with the lower index as the big one
    if (ok && (!jbig || il < jl)) {
      const DetBig& q = sm[k];
      const float4 p0 = q.p0, v0 = q.v0, p1 = q.p1, v1 = q.v1;
      const float bf[12] = {p0.x, p0.y, p0.z, v0.x, v0.y, v0.z,
                            p1.x, p1.y, p1.z, v1.x, v1.y, v1.z};
      const float rcf = fmaxf(v0.w, rcjf);
      if (p1.w == 0.0f && encounter_screen(af, bf, rcf * rcf, hf)) {
        const double rc = fmax(d.brc[S.boff + il], rcj);
        if constexpr (FEW) hit = encounter_fp64(ad, sd + 12 * k, ad + 6, sd + 12 * k + 6, h, rc * rc);
        else hit = encounter_pair(xv0, xv1, N, j, S.off + il, h, rc * rc);
      }
    }
    if (hit) {
      const int gi = S.off + il;
      flags[gi] = 1;
      flags[j] = 1;
      if (d.ever) {
        d.ever[gi] = 1;
        d.ever[j] = 1;
      }
      if (nh == kMaxGroup) {   // a run split in two: only past the group limit
        if (runs) report(d.status, ST_GROUP);
        nh = -1;               // marks the flush below as due
      } else {
        hits[nh++] = il;
      }
    }
    // a full buffer is written out (every lane of the warp takes part)
    if (__any_sync(0xffffffffu, nh < 0)) {
      const bool redo = nh < 0;
      if (redo) nh = kMaxGroup;
      flush(redo);
      if (redo) hits[nh++] = il;
    }
  };
  for (int c0 = 0; c0 < S.nbig; c0 += chunk) {
    const int cn = min(chunk, S.nbig - c0);
    __syncthreads();
    if (threadIdx.x < cn) {
      const int g = S.off + c0 + threadIdx.x;
      float bf[12];
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const double e0 = xv0[(size_t)k * N + g], e1 = xv1[(size_t)k * N + g];
        bf[k] = to_float_bits(e0);
        bf[6 + k] = to_float_bits(e1);
        if constexpr (FEW) {
          sd[12 * threadIdx.x + k] = e0;
          sd[12 * threadIdx.x + 6 + k] = e1;
        }
      }
      const float rcf = to_float_bits(d.brc[S.boff + c0 + threadIdx.x]);
      DetBig& q = sm[threadIdx.x];
      q.p0 = make_float4(bf[0], bf[1], bf[2], FEW ? 0.0f : encounter_reach(bf, rcf, hf));
      q.v0 = make_float4(bf[3], bf[4], bf[5], rcf);
      q.p1 = make_float4(bf[6], bf[7], bf[8], removed(d, g) ? 1.0f : 0.0f);
      q.v1 = make_float4(bf[9], bf[10], bf[11], 0.0f);
    }
    __syncthreads();
    if constexpr (FEW) {
      for (int k = 0; k < cn; ++k) test(c0, k, act);
    } else {
      for (int k0 = 0; k0 < cn; k0 += 32) {
        // first screen: 32 big bodies, one bit each
        const int kn = min(32, cn - k0);
        unsigned mask = 0;
#pragma unroll 8
        for (int k = 0; k < kn; ++k) {
          const float4 b = sm[k0 + k].p0;
          const float dx = af[0] - b.x, dy = af[1] - b.y, dz = af[2] - b.z;
          const float r = reach + b.w;
          if (fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < r * r) mask |= 1u << k;
        }
        if (!act) mask = 0;
        // the pairs it left, each lane its own next one
        while (__any_sync(0xffffffffu, mask != 0)) {
          const int k = k0 + max(__ffs(mask) - 1, 0);
          const bool ok = mask != 0;
          mask &= mask - 1;
          test(c0, k, ok);
        }
      }
    }
  }
  flush(true);
}

}  // namespace mx
