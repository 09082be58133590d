// Screening of the rigid alignment's poses on a trilinear grid.
//
// The alignment keeps one of N*N poses, so most of its FP32 lookups only show that a pose is not the
// best.  Screening finds that out from an estimate with a proved error bound E: every pose is
// estimated, one pose is scored in full (score s0), and only the poses whose estimate reaches s0 - E
// are scored in full.  A pose below that line scores less than s0, so the best score, its ties and the
// pose index kept are those of scoring every pose; no estimate enters a result.
//
// What it saves: an FP32 lookup gathers a 32-byte cell and is bound by the L1 data pipe (about 23
// wavefronts per warp-wide load, 13-18 for the 16-byte FP16 cells).  A screening cell is 8 bytes (about 12
// wavefronts, and twice to four times the cells per byte of L1), and the coordinates are fixed point, so
// the index and the fractions are bit fields and the interpolation is exact integer arithmetic.  The same
// idea with 16-byte cells of FP16 polynomial coefficients was 1.2 times slower: bound by the data pipe.
//
// Error bound, in steps of the voxels' quantisation (per atom, summed over the n atoms):
//  - the voxels, rounded to integers: ScreenDev::quant (the integers are one field shared by all cells,
//    so the estimate is continuous and its error at any position is at most the corners');
//  - the position: the fixed-point coordinate starts from t + 2064 and is rounded to 2^-12 by each of the
//    sum and three multiply-adds (4 times 2^-13), the exact lookup's by its own FP32 steps; times the
//    field's slope (ScreenDev::slope, summed over the axes).  Where the field jumps, at the faces of a grid
//    with nonzero boundary voxels, screen_usable asks that no pose reaches a face;
//  - the FP32 rounding of the exact lookups and their n-term sums, (n + 32) 2^-23 of ScreenDev::vabs.
#pragma once

namespace dockgpu {

// Kernels that hold the screening code.  Not with 8 warps per item: that is for small batches, where an item's
// latency counts; a warp has two or three passes then, and the dependent steps of screening cost more than its
// lookups save (12 ligands in the service 400 us screened, 330 not; 15 large molecules 777 and 673).  On FP16 cells a
// lookup costs half an FP32 one and screening gains less: nothing with 4 warps per item (screened / not, N = 30:
// 1.03 at 10-80 atoms, 1.07 at 80-150).
__host__ __device__ constexpr bool screen_compiled(int gt, int g) {
  return gt == 0 ? g < 8 : gt == 1 && g <= 2;
}

// Whether a launch screens its alignments of N*N poses, `items` ligand-restarts filling the GPU of `sms` SMs
// together.  With few poses per warp the estimates and the dealt scoring of the survivors cost more than they save.
// Measured, screened / not, 10-80 atoms, at N = 12, 16, 20, 24:
//   FP32, 1, 2, 4 warps: 1.10 0.92 0.80 0.75;  1.25 1.06 0.87 0.79;  1.23 1.12 0.98 0.88
//   FP16, 1, 2 warps:    1.15 1.08 0.97 0.94;  1.44 1.25 1.08 0.99
// A large molecule's screening is a long chain, which a GPU with few warps resident cannot hide.  80-150 atoms: 60 ligands
// with 2 warps per item (24 warps per SM) 1.27, 80 ligands (32) 0.89; one warp, 100 ligands (20) 1.13, 150 (30) 0.86; 4
// warps, 41 ligands (32) 1.09, 60 (47) 0.91.  10-80 atoms, where the 65-96-atom bucket decides: less than 8 warps per SM
// one warp per item 1.16 (FP16 1.18), 4 warps 1.10, but 2 warps 0.82-0.98.  (FP16, 2 warps, full GPU: 501 large molecules
// 0.96 on a 96^3 grid, 1.05 on 64^3, whose cells stay closer; both ways below the time before the screening.)
inline bool screening_pays(int maxn, int gt, int g, int N, int items, int sms) {
  if (!screen_compiled(gt, g)) return false;
  const int least = gt == 0 ? (g == 1 ? 16 : g == 2 ? 18 : 22) : (g == 1 ? 20 : 24);
  const int warps = maxn <= 64 ? 0 : maxn <= 96 ? (g == 2 ? 0 : 8) : g == 4 ? 40 : 28;  // per SM
  return N >= least && (int64_t)items * g >= (int64_t)warps * sms;
}

// Whether a warp that gave up screening an item's first alignment tries again in its post-alignment.  On a field that
// screening does not suit it gives up there too; on one that it suits the few items that gave up would run longest, and
// with one warp per item and less than 100 items per SM the launch waits for them (without a second try: 41-150 ligands
// 1.15-1.25, 400 small ones 1.04); with more warps an item's share is shorter and that shows below 30 only (100 ligands
// 1.05).
inline int screening_retries(int g, int items, int sms) { return (int64_t)items < (int64_t)(g == 1 ? 100 : 30) * sms; }

// Lanes with two candidates after which a warp gives up screening (about 55 candidates in 32 lanes).  On a field whose
// range is large against the differences between good poses (a large constant, deep repulsion in few places) the
// bound excludes little: the estimates cost about half of the poses' lookups (FP32 cells; three quarters on FP16) and
// most poses are then looked up as well.  In the workloads' fields 3-5 of 900 poses are within the bound of the best
// (98th percentile 22; 50 with large molecules), with repulsion of depth 1000 around 5% of a pocket of depth 1 100
// (270), in a flat field all.  Time against not screening, 10-80 atoms, without and with giving up (and not trying again,
// screening_retries): that repulsion, 1,500 ligands, FP32 1.39 -> 1.06, FP16 1.76 -> 1.19, 400 ligands 1.35 -> 1.17 and
// 1.68 -> 1.44; voxels of -5000 strewn over the workload's field, FP16 1.28 -> 1.03.
constexpr int kScreenCrowd = 16;
constexpr int kScreenKeep = 4;     // best estimates a lane keeps; a lane with more candidates than that falls
                                   // back to scoring all its poses
constexpr float kScreenMag = 2048.f + kScreenPad;  // 2^11: 12 fraction bits below it in FP32; cell -kScreenPad at 0

// Whether the poses of a ligand whose centred atoms are `rel` and whose centroid is at grid position t
// may be screened: inside the padded grid, or inside the grid itself where the field jumps at its
// faces.  False on coordinates that are not finite.  `mag` receives a bound on the coordinates.
__device__ __forceinline__ bool screen_usable(const PocketDev& pk, const float4* rel, int n, float3 t, float ih, int lane,
                                              float& mag) {
  if (pk.screen.base == nullptr) return false;
  float r2 = 0.f;
  bool finite = true;
  for (int a = lane; a < n; a += 32) {
    const float4 d = rel[a];
    const float q = fmaf(d.x, d.x, fmaf(d.y, d.y, d.z * d.z));
    finite &= q < 1e12f;
    r2 = fmaxf(r2, q);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) r2 = fmaxf(r2, __shfl_xor_sync(kFull, r2, o));
  const float r = sqrtf(r2) * ih * 1.001f + 0.01f;  // a rotation keeps the distance to the centroid
  const float lo = fminf(t.x, fminf(t.y, t.z)) - r;
  const float pad = pk.screen.inside ? 0.f : (float)kScreenPad;
  const bool ok = finite && lo > -pad && t.x + r < (float)(pk.nx - 1) + pad && t.y + r < (float)(pk.ny - 1) + pad &&
                  t.z + r < (float)(pk.nz - 1) + pad;
  mag = fmaxf(t.x, fmaxf(t.y, t.z)) + r + 2.f * kScreenPad;
  return __all_sync(kFull, ok);
}

// q / d by the reciprocal: (q + 1/2) / d stays 1/(2 d) clear of an integer, far past the rounding at q < 2^14,
// d <= 160.
__device__ __forceinline__ int quotient(int q, float inv_d) { return __float2int_rd(((float)q + 0.5f) * inv_d); }

// The rotation of pose f = i * N + j with the grid scale folded in (align_pass's factors).  inv_N: 1 / N, or 0 for
// an integer division.
struct PoseRot {
  float r00, r01, r02, r11, r12, r20, r21, r22;
};
__device__ __forceinline__ PoseRot pose_rot(int f, const float2* tab, int N, float inv_N, float ih) {
  const int i = inv_N > 0.f ? quotient(f, inv_N) : f / N, j = f - i * N;
  const float2 ca = tab[i], cb = tab[j];  // (cos, sin)
  PoseRot r;
  r.r00 = cb.x * ih, r.r01 = cb.y * ca.y * ih, r.r02 = cb.y * ca.x * ih;
  r.r11 = ca.x * ih, r.r12 = -ca.y * ih;
  r.r20 = -cb.y * ih, r.r21 = cb.x * ca.y * ih, r.r22 = cb.x * ca.x * ih;
  return r;
}
__device__ __forceinline__ float3 pose_at(const PoseRot& r, const float4& d, const float3& t) {
  return make_float3(fmaf(r.r00, d.x, fmaf(r.r01, d.y, fmaf(r.r02, d.z, t.x))), fmaf(r.r11, d.y, fmaf(r.r12, d.z, t.y)),
                     fmaf(r.r20, d.x, fmaf(r.r21, d.y, fmaf(r.r22, d.z, t.z))));
}

// Estimates the poses f0 + lane + 32 t, t < T, in units of step / kScreenUnits, and puts them into the
// lane's kScreenKeep best (top[0] the highest) and the best one left out (top[kScreenKeep]).  The low 9
// bits of an entry hold the pass f / 32 (at most 511); 0 is no entry.
template <int T, int U, bool kRecip>
__device__ __forceinline__ void screen_pass(const PocketDev& pk, const float4* rel, int n, const float2* tab, int N,
                                            float ih, const float3& t3, int f0, int lane, unsigned (&top)[kScreenKeep + 1]) {
  const int NN = N * N;
  PoseRot r[T];
  unsigned long long acc[T];  // sum of corners * weights, 3 x 12 fraction bits
  unsigned bases[T];          // 128 * sum of the cells' bases
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const int f = f0 + lane + 32 * t;
    r[t] = pose_rot(f < NN ? f : 0, tab, N, kRecip ? 1.0f / (float)N : 0.f, ih);
    acc[t] = 0;
    bases[t] = 0;
  }
  const uint2* cells = reinterpret_cast<const uint2*>(pk.screen.base);
  const unsigned cx = pk.screen.cx, cy = pk.screen.cy;
  constexpr unsigned one = 1u << kScreenFrac;
#pragma unroll(U)
  for (int a = 0; a < n; ++a) {
    const float4 d = rel[a];
#pragma unroll
    for (int t = 0; t < T; ++t) {
      const float3 x = pose_at(r[t], d, t3);
      const unsigned ub = __float_as_uint(x.x), vb = __float_as_uint(x.y), wb = __float_as_uint(x.z);
      const uint2* p = cells + (((wb >> kScreenFrac) * cy + (vb >> kScreenFrac)) * cx + (ub >> kScreenFrac));
      DOCK_CNT(cnt_lookup(true, (unsigned long long)p, false);)
      const uint2 q = __ldg(p);
      const unsigned fx = ub & (one - 1), fy = vb & (one - 1), fz = wb & (one - 1);
      const unsigned wx = fx * 0xffffu + one;  // {1 - x, x} as 16-bit halves
      bases[t] = __dp4a(q.x & 0x80808080u, 0x08040201u, bases[t]);
      const unsigned lo = q.x & 0x7f7f7f7fu;
      const unsigned v0 = __dp2a_lo(wx, lo, 0u) * (one - fy) + __dp2a_hi(wx, lo, 0u) * fy;
      const unsigned v1 = __dp2a_lo(wx, q.y, 0u) * (one - fy) + __dp2a_hi(wx, q.y, 0u) * fy;
      acc[t] += (unsigned long long)v0 * (one - fz);
      acc[t] += (unsigned long long)v1 * fz;
    }
  }
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const int f = f0 + lane + 32 * t;
    // 36 fraction bits to 12 (kScreenUnits); at most 160 * (127 + 15 * 100) steps, below 2^31
    const unsigned est = (unsigned)(acc[t] >> 24) + ((bases[t] >> 7) * pk.screen.mult << 12) + 1024u;
    unsigned v = f < NN ? (est & ~511u) | ((f0 >> 5) + t) : 0u;
#pragma unroll
    for (int k = 0; k < kScreenKeep; ++k) {
      const unsigned hi = max(top[k], v);
      v = min(top[k], v);
      top[k] = hi;
    }
    top[kScreenKeep] = max(top[kScreenKeep], v);
  }
}

// Scores in full the pose f of every lane set in `mask` and folds them into (best, bidx), which end up
// spread over the warp's lanes.  The (pose, atom) pairs are dealt to the lanes and each pose's values
// are then summed in atom order by one lane: the additions of align_pass in their order.
template <int GT, int CAP, bool kRecip>
__device__ __forceinline__ void screen_score(const GridK& g, const float4* rel, int n, const float2* tab, int N,
                                             const float3& t3, unsigned mask, int f, float* buf, int lane, float& best,
                                             int& bidx) {
  unsigned short* list = reinterpret_cast<unsigned short*>(buf);  // up to 32 poses (f < 2^14)
  float* val = buf + 16;
  const int cnt = __popc(mask);
  if ((mask >> lane) & 1u) list[__popc(mask & lanemask_lt())] = (unsigned short)f;
  __syncwarp();
  const int stride = n | 1;
  const int per = min((CAP - 16) / stride, 32);
  const float inv_n = 1.0f / (float)n, inv_N = kRecip ? 1.0f / (float)N : 0.f;
  for (int c0 = 0; c0 < cnt; c0 += per) {
    const int m = min(per, cnt - c0);
    for (int q = lane; q < m * n; q += 32) {
      const int c = kRecip ? quotient(q, inv_n) : q / n, a = q - c * n;
      const float3 x = pose_at(pose_rot(list[c0 + c], tab, N, inv_N, g.inv_h), rel[a], t3);
      val[c * stride + a] = lookup<GT>(g, x.x, x.y, x.z);
    }
    __syncwarp();
    if (lane < m) {
      float s = 0.f;
      for (int a = 0; a < n; ++a) s += val[lane * stride + a];
      const int fl = list[c0 + lane];
      if (s > best || (s == best && fl < bidx)) {
        best = s;
        bidx = fl;
      }
    }
    __syncwarp();
  }
}

// The best of the warp's poses (blocks wig, wig + G, ... of 64), as align_pass over them finds it,
// left spread over the warp's lanes.  Returns false, with (best, bidx) to be ignored, where screening does
// not pay: after the first, third, ... block of poses more than kScreenCrowd lanes hold two poses within the bound of
// the best estimate, or in the end a lane holds more than kScreenKeep candidates.
template <int GT, int CAP, int G>
__device__ bool screen_align(const PocketDev& pk, const GridK& g, const float4* rel, int n, const float2* tab, int N,
                             const float3& t3, float mag, int wig, float* buf, int lane, float& best, int& bidx) {
  // Poses per lane and atoms per loop step, four lookups in flight either way: with one warp per item
  // 2 x 2 (at 96 registers, 2,000 ligands of the uneven mix: 9.25 ms, against 9.9 for 2 x 1, 9.8 for 1 x 4
  // and 11.9 for 2 x 4, whose loop outgrows the instruction cache); with more warps 1 x 4 (at 80
  // registers: 9.5, against 11.4 for 2 x 2 at 96).  Prefetching the next atom's cells instead was
  // no faster (9.3 against 8.7 on the FP16 grid).
  constexpr int T = G == 1 ? 2 : 1, U = G == 1 ? 2 : 4;
  // Reciprocals for the pose and pair indices with one warp per item (4,003 uneven ligands 17.3 -> 16.6 ms);
  // at the 80 registers of 2 warps per item they spill (18.2 -> 18.8) and the divisions stay.
  constexpr bool kRecip = G == 1;
  const int NN = N * N;
  if (wig * kDeal >= NN) return true;  // no pose of this warp
  const float fn = (float)n;
  // error bound of a pose's estimate in steps, the dropped low bits included
  const float bound = fn * (pk.screen.quant + pk.screen.slope * (4.f / 8192.f + 2.4e-7f * mag) +
                            (fn + 32.f) * 1.1920929e-7f * pk.screen.vabs) + 0.5f;
  const unsigned slack = __float2uint_ru(bound * kScreenUnits);
  const float3 start = make_float3(t3.x + kScreenMag, t3.y + kScreenMag, t3.z + kScreenMag);
  unsigned top[kScreenKeep + 1];
#pragma unroll
  for (int k = 0; k <= kScreenKeep; ++k) top[k] = 0u;
  int tail = NN;  // the last few poses: scored in full without an estimate
  for (int f0 = wig * kDeal; f0 < NN; f0 += G * kDeal) {
    int f = f0;
    for (; f < f0 + kDeal && NN - f > 32 * (T - 1) + 8; f += 32 * T)
      screen_pass<T, U, kRecip>(pk, rel, n, tab, N, g.inv_h, start, f, lane, top);
    if (T > 1 && f < f0 + kDeal && NN - f > 8) {  // half a pass
      screen_pass<1, U, kRecip>(pk, rel, n, tab, N, g.inv_h, start, f, lane, top);
      f += 32;
    }
    if (f < min(f0 + kDeal, NN)) tail = f;
    if ((f0 / kDeal - wig) / G % 2 == 0) {  // every second block
      // poses within the bound of the best estimate so far are candidates, as it stands
      const unsigned hi = __reduce_max_sync(kFull, top[0]);
      if (__popc(__ballot_sync(kFull, top[1] >= (hi > slack ? hi - slack : 1u))) > kScreenCrowd) return false;
    }
  }
  // the highest estimate's pose, in full
  const unsigned m = __reduce_max_sync(kFull, top[0]);  // 0: every pose of the warp is in the tail
  const int who = __ffs(__ballot_sync(kFull, top[0] == m)) - 1;
  float b = -CUDART_INF_F;
  int bi = 0;
  unsigned line = 0;
  bool ok = true;
#pragma unroll 1
  for (int k = tail < NN ? -2 : -1; k < kScreenKeep; ++k) {
    unsigned e = top[0];
#pragma unroll
    for (int i = 1; i < kScreenKeep; ++i) e = k == i ? top[i] : e;
    const unsigned mask = k == -2 ? (1u << (NN - tail)) - 1u
                          : k < 0 ? (m ? 1u << who : 0u)
                                  : __ballot_sync(kFull, e >= line && !(k == 0 && lane == who));
    if (mask == 0) {
      if (k != 0) break;
      continue;
    }
    screen_score<GT, CAP, kRecip>(g, rel, n, tab, N, t3, mask, k == -2 ? tail + lane : (int)(e & 511u) * 32 + lane, buf, lane, b, bi);
    if (k == -1) {
      // the line: the score just found in units of the estimates, less the bound
      float s0 = b;
#pragma unroll
      for (int o = 16; o; o >>= 1) s0 = fmaxf(s0, __shfl_xor_sync(kFull, s0, o));
      const float l = ((s0 - fn * pk.screen.vmin) * pk.screen.units - bound * kScreenUnits) + 1024.f;
      line = l > 1.f ? (unsigned)l : 1u;
      ok = !__any_sync(kFull, top[kScreenKeep] >= line);
      if (!ok) break;
    }
  }
  best = b;
  bidx = bi;
  return ok;
}

}  // namespace dockgpu
