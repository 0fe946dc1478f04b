// Float32 near field with up to 8 right-hand sides, each unordered pair of
// near leaves evaluated once (the near relation and phi are symmetric).
//
// A CTA takes target leaf T and 512 sources of its upper entries (T, S >= T),
// which are laid end to end.  A lane holds 4 sources; at step s lane l meets
// T's site l + s (modulo T's size, at least 32), so a warp's targets differ
// and each lane adds to its target's sum in shared memory (one array per
// warp, no atomics) while the sources' sums stay in registers.  The turn takes
// exactly T's size and the sources are a stream, so ragged leaves leave no
// lane idle.  Sums of at most 512 terms leave the kernel: forward sums per
// chunk, transposed sums per entry; the scatter adds them in list order, with
// compensation.
//
// Bound by the float32 pipe (a subtraction and a multiply-add per pair and
// dimension, packed in twos) with the special function unit close behind.
// Against one CTA per target leaf over all its neighbours (k_sum_f32), which
// evaluates each pair twice and had 512 CTAs of 64 threads for 152 SMs in the
// first case: d = 16 exponential, N = 50021, 1 right-hand side 1.87 -> 0.44 ms;
// d = 8 Matern, N = 100003, 4: 2.25 -> 0.94 ms; N = 3001, 1: 174 -> 20 us.
#pragma once

#include "dwfmm_internal.cuh"
#include "sum_f32.cuh"

namespace dw {
namespace rot {

using namespace sk;

constexpr int kRotThreads = 128;
constexpr int kRotWarps = kRotThreads / 32;
constexpr int kRotPer = kRotWarps * 128;   // sources of a chunk
constexpr int kRotMaxLeaf = 256;
constexpr int kRotMinLeaf = 32;
constexpr int kRotMaxRc = 8;

// floats between targets: 4 mod 8, so that 16-byte loads of consecutive
// targets fall into different banks
template <int D>
constexpr int rot_stride() { return D % 8 == 4 ? D : (D + 4) % 8 == 4 ? D + 4 : 12; }

template <int D, int RC>
constexpr size_t rot_smem(int ld) {
  return static_cast<size_t>(ld) * (rot_stride<D>() + 1 + RC + kRotWarps * RC) * sizeof(float);
}

// One chunk by a CTA of kRotThreads threads; rsm: rot_smem bytes, free for
// other use once every thread is past the next barrier.
template <int D, int RC, int KER>
__device__ __forceinline__ void rot_chunk(const RotArgs& a, int chunk, float* rsm) {
  constexpr int TS = rot_stride<D>();
  const int ld = a.ld;
  float* trec = rsm;                       // [ld][TS]
  float* facc = trec + ld * TS;            // [kRotWarps][ld][RC]
  float* tq = facc + kRotWarps * ld * RC;  // [ld][RC]
  float* tn = tq + ld * RC;                // [ld] squared norms (Gaussian)
  const int gchunk = chunk + a.chunk0;
  const int T = a.chunk_t[gchunk];
  const int cmax = a.cmax_of ? a.cmax_of[T] : a.cmax;
  const int c = a.count[T];
  const int e0 = a.uprow[T], ne = a.uprow[T + 1] - e0;
  const int warp = static_cast<int>(threadIdx.x) >> 5, lane = static_cast<int>(threadIdx.x) & 31;
  const int base = (gchunk - a.chunk_ptr[T]) * kRotPer + warp * 128;

  const float* tb = a.pts + static_cast<int64_t>(T) * (D + 1) * ld;
  for (int i = threadIdx.x; i < c; i += kRotThreads) {
#pragma unroll
    for (int k = 0; k < D; ++k) trec[i * TS + k] = KER == DWFMM_K_GAUSS ? 2.0f * tb[k * ld + i] : tb[k * ld + i];
    if (KER == DWFMM_K_GAUSS) tn[i] = tb[D * ld + i];
  }
  for (int i = threadIdx.x; i < c * RC; i += kRotThreads) tq[i] = a.q[static_cast<int64_t>(T) * ld * RC + i];
  for (int i = threadIdx.x; i < kRotWarps * ld * RC; i += kRotThreads) facc[i] = 0.0f;

  // the lane's sources, packed in pairs: sources (0, 1) and (2, 3)
  u64 s2[2][D], q2[2][RC], n2[2];
  int ent[4], slot[4];   // entry, -1: nothing to write
  {
    float v[4], w[4];
    int64_t at[4];
    bool ok[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int j = base + u * 32 + lane;
      const int en = j / cmax;
      slot[u] = j - en * cmax;
      int S = T;
      ok[u] = en < ne;
      if (ok[u]) {
        S = a.up_s[e0 + en];
        ok[u] = slot[u] < a.count[S];
      }
      ent[u] = ok[u] && S != T ? e0 + en - a.e_base : -1;
      at[u] = static_cast<int64_t>(S);
      if (!ok[u]) slot[u] = 0;
    }
#pragma unroll
    for (int k = 0; k < D; ++k) {
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = a.pts[(at[u] * (D + 1) + k) * ld + slot[u]];
      s2[0][k] = pk2(v[0], v[1]);
      s2[1][k] = pk2(v[2], v[3]);
    }
    if (KER == DWFMM_K_GAUSS) {
#pragma unroll
      for (int u = 0; u < 4; ++u) w[u] = -a.pts[(at[u] * (D + 1) + D) * ld + slot[u]];
      n2[0] = pk2(w[0], w[1]);
      n2[1] = pk2(w[2], w[3]);
    }
#pragma unroll
    for (int r = 0; r < RC; ++r) {
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = ok[u] ? a.q[(at[u] * ld + slot[u]) * RC + r] : 0.0f;
      q2[0][r] = pk2(v[0], v[1]);
      q2[1][r] = pk2(v[2], v[3]);
    }
  }
  __syncthreads();

  u64 t2[2][RC];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int r = 0; r < RC; ++r) t2[h][r] = 0ull;
  float* fw = facc + warp * ld * RC;
  if (base < ne * cmax) {
    int t = lane;
    for (int s = 0; s < c; ++s) {
      const float* rec = trec + t * TS;
      u64 e[2];
      if (KER == DWFMM_K_GAUSS) {
        const float nt = tn[t];
        const u64 nt2 = pk2(nt, nt);
        e[0] = fsub2(n2[0], nt2);
        e[1] = fsub2(n2[1], nt2);
      } else {
        e[0] = e[1] = 0ull;
      }
#pragma unroll
      for (int k = 0; k < D; k += 2) {
        float x[4];
        if (k % 4 == 0 && k + 4 <= D) {
          const float4 v = *reinterpret_cast<const float4*>(rec + k);
          x[0] = v.x;
          x[1] = v.y;
          x[2] = v.z;
          x[3] = v.w;
        } else if (k % 4 == 0) {
          const float2 v = *reinterpret_cast<const float2*>(rec + k);
          x[0] = v.x;
          x[1] = v.y;
        } else {
          continue;   // taken with the dimensions before
        }
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          if (k + z >= D) break;
          const u64 x2 = pk2(x[z], x[z]);
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (KER == DWFMM_K_GAUSS) {
              e[h] = ffma2(x2, s2[h][k + z], e[h]);
            } else {
              const u64 df = fsub2(x2, s2[h][k + z]);
              e[h] = ffma2(df, df, e[h]);
            }
          }
        }
      }
      u64 p2[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float p0, p1;
        up2(e[h], p0, p1);
        p2[h] = pk2(phi_scaled<KER>(p0), phi_scaled<KER>(p1));
      }
      auto add = [&](int r, float xq) -> float {   // the target's share of the four pairs
        const u64 xq2 = pk2(xq, xq);
        u64 f2 = 0ull;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          t2[h][r] = ffma2(p2[h], xq2, t2[h][r]);
          f2 = ffma2(p2[h], q2[h][r], f2);
        }
        float f0, f1;
        up2(f2, f0, f1);
        return f0 + f1;
      };
      if constexpr (RC == 1) {
        fw[t] += add(0, tq[t]);
      } else {
#pragma unroll
        for (int r = 0; r < RC; r += 4) {
          float4* fp = reinterpret_cast<float4*>(fw + t * RC + r);
          const float4 xq = *reinterpret_cast<const float4*>(tq + t * RC + r);
          float4 f = *fp;
          f.x += add(r, xq.x);
          f.y += add(r + 1, xq.y);
          f.z += add(r + 2, xq.z);
          f.w += add(r + 3, xq.w);
          *fp = f;
        }
      }
      if (++t >= c) t -= c;
      __syncwarp();
    }
  }
#pragma unroll
  for (int r = 0; r < RC; ++r) {
    if (r >= a.Rc) break;
    float v[4];
    up2(t2[0][r], v[0], v[1]);
    up2(t2[1][r], v[2], v[3]);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (ent[u] >= 0) a.pt[(static_cast<int64_t>(ent[u]) * a.Rc + r) * a.ldp + slot[u]] = v[u];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < a.Rc * c; i += kRotThreads) {
    const int r = i / c, t = i - r * c;
    // the four warps' sums, rounded once (the float64 unit is too narrow here)
    float v = facc[t * RC + r], lost = 0.0f;
#pragma unroll
    for (int w = 1; w < kRotWarps; ++w) {
      const float f = facc[(w * ld + t) * RC + r], sum = v + f, back = sum - v;
      lost += (v - (sum - back)) + (f - back);
      v = sum;
    }
    a.pf[(static_cast<int64_t>(chunk) * a.Rc + r) * a.ldp + t] = v + lost;
  }
}

}  // namespace rot
}  // namespace dw
