// Backward pass of the enhanced min-sum iterations (the subgradient stated in k_train.cu),
// row by row like rc_device.cuh with 32 frames per block, compiled at run time for one code.
//
// Per frame, iteration (from its checkpoint y^(t-1)) and copy: a warp task is one check row of
// 32 frames -- its two smallest magnitudes, the sums over the other edges' gradients, and
// the two contributions alpha acc (at the minimum and at the second minimum), which go to the
// row's state with the two variables.  The contributions are then added to per-copy sums by
// RCB_ACC warps, each running through its own rows in order into sums of its own, so that
// no two threads touch one address and the result does not depend on timing; the merge adds
// those sums to the gradient position by position.  A per-edge column pass (as the forward
// has) would read 12 bytes for each of a row's ~23 edges, of which two matter.
//
// Bound: the ALU pipe.  Per edge: an address, 2.5 minima, half a sign xor and two equality
// tests on it (3 SM cycles per 32 lanes), beside two shared-memory reads and
// three additions.  BCH(127,64), 65 536 frames x 12 iterations x P = 3: 4.14 ms, against 45.0 ms
// of the one-thread-per-frame kernel (rows from shared-memory tables, 64 threads and 98 KB
// per block); per group of 32 frames and iteration the rows take ~39 k cycles (4.4 per
// warp-edge), the additions of the row states 6.5 k, positions and checkpoints 7 k.  Tried:
// moving the two edges' addresses and values under the tests instead of counting (6.2 ms),
// one row at a time in the additions (+0.5 ms).
#pragma once

namespace bchlib {

// Shared memory in words (rcb_words gives the total): two buffers of y[n][33] and g[n][33]
// by position, one copy's z and gs = sgn(z) g / P by variable, the row states (c1, c2) and
// variable pairs, RCB_ACC sums by variable, and small arrays.
constexpr int kRcbN33 = RC_N * 33, kRcbHead = (3 * kRcbN33 + 3) & ~3, kRcbZ = RC_N * 32;

struct RcbPtr {
  const unsigned char *z, *gs;  // this lane's columns
  float2 *c;                    // [R][32]
  uint32_t *u;                  // [R][32]: byte offset of a1 | of a2 << 16
  const uint16_t *cols;         // [R][4 RC_W4]: the rows' variables
  int warp, nwarps;
  float alpha, dal;
  bool bad;  // this lane's frame holds an infinity or NaN
  bool live;
};

__device__ __forceinline__ float rcb_ld(const unsigned char *p) { return *reinterpret_cast<const float *>(p); }

// One row in edge order, exactly as the precompiled backward kernel takes it: for ties at
// the minimum, infinities and NaN.
struct RcbRow {
  float c1, c2, dal;
  uint32_t u;
};
__device__ __noinline__ RcbRow rcb_row_ordered(const unsigned char *z, const unsigned char *gs, const int *tab, int W,
                                               float alpha) {
  float m1 = FLT_MAX, m2 = FLT_MAX;
  int a1 = 0, a2 = 0;
  uint32_t sg = 0;
#pragma unroll 1
  for (int e = 0; e < W; e++) {
    const float v = rcb_ld(z + tab[e]), av = fabsf(v);
    if (av < m1) {
      m2 = m1;
      a2 = a1;
      m1 = av;
      a1 = e;
    } else if (av < m2) {
      m2 = av;
      a2 = e;
    }
    sg ^= __float_as_uint(v);
  }
  RcbRow r;
  r.dal = 0.0f;
  float acc1 = 0.0f, acc2 = 0.0f;
#pragma unroll 1
  for (int e = 0; e < W; e++) {
    const float g = flip_sign(rcb_ld(gs + tab[e]), sg);
    r.dal += g * (e == a1 ? m2 : m1);
    if (e == a1) acc2 = g;
    else acc1 += g;
  }
  r.c1 = flip_sign(alpha * acc1, __float_as_uint(rcb_ld(z + tab[a1])));
  r.c2 = flip_sign(alpha * acc2, __float_as_uint(rcb_ld(z + tab[a2])));
  r.u = uint32_t(tab[a1]) | uint32_t(tab[a2]) << 16;
  return r;
}

// The rows of weight W (as rc_rows in rc_device.cuh).
template <int W>
__device__ __forceinline__ void rcb_rows(RcbPtr &c, int nr, int r0, int t0) {
  int t = c.warp - r0 % c.nwarps;
  if (t < 0) t += c.nwarps;
  for (; t < nr; t += c.nwarps) {
    float v[W], av[W], m1, m2;
    int off[W];
    uint32_t sg = 0;
#pragma unroll
    for (int q = 0; q < (W + 3) / 4; q++) {
      const int4 o = rc_rowtab[t0 + t * ((W + 3) / 4) + q];
      off[4 * q] = o.x;
      if (4 * q + 1 < W) off[4 * q + 1 < W ? 4 * q + 1 : 0] = o.y;
      if (4 * q + 2 < W) off[4 * q + 2 < W ? 4 * q + 2 : 0] = o.z;
      if (4 * q + 3 < W) off[4 * q + 3 < W ? 4 * q + 3 : 0] = o.w;
    }
#pragma unroll
    for (int e = 0; e < W; e++) v[e] = rcb_ld(c.z + off[e]);
#pragma unroll
    for (int e = 0; e < W; e++) {
      sg ^= __float_as_uint(v[e]);
      av[e] = fabsf(v[e]);
    }
    min12<float, W>(av, m1, m2);
    // Sums without the row's sign, which all terms share.  The edges of the two minima are
    // counted up on the FMA pipe (the ALU pipe bounds this loop): e1 = the one edge at min1,
    // e2 = 256 + the edge at min2, 512 or more when several are.
    float sum[2] = {0.0f, 0.0f}, e1 = 0.0f, e2 = 0.0f;
#pragma unroll
    for (int e = 0; e < W; e++) {
      const float gs = rcb_ld(c.gs + off[e]);
      if (av[e] == m1) e1 += float(e);
      else sum[e & 1] += gs;
      if (av[e] == m2) e2 += float(256 + e);
    }
    const bool odd = c.live && (c.bad || !(m1 < m2) || e2 >= 512.0f);
    const uint16_t *cols = c.cols + (r0 + t) * (4 * RC_W4);
    const int u1 = cols[min(int(e1), W - 1)] * 128, u2 = cols[min(int(e2) & 255, W - 1)] * 128;
    const uint32_t s1 = __float_as_uint(rcb_ld(c.z + u1)), s2 = __float_as_uint(rcb_ld(c.z + u2));
    const float acc1 = flip_sign(sum[0] + sum[1], sg), acc2 = flip_sign(rcb_ld(c.gs + u1), sg);
    float c1 = flip_sign(c.alpha * acc1, s1), c2 = flip_sign(c.alpha * acc2, s2);
    float d = __fmaf_rn(acc1, m1, acc2 * m2);
    uint32_t u = uint32_t(u1) | uint32_t(u2) << 16;
    if (__any_sync(kFull, odd)) {
      const RcbRow r = rcb_row_ordered(c.z, c.gs, reinterpret_cast<const int *>(rc_rowtab) + 4 * (t0 + t * ((W + 3) / 4)),
                                       W, c.alpha);
      if (odd) {
        c1 = r.c1;
        c2 = r.c2;
        d = r.dal;
        u = r.u;
      }
    }
    c.dal += d;
    c.c[(r0 + t) * 32] = make_float2(c1, c2);
    c.u[(r0 + t) * 32] = u;
  }
}

__device__ __forceinline__ void rcb_row_pass(RcbPtr &c);

__device__ __forceinline__ uint32_t rcb_pos(uint32_t i, uint32_t cx) {  // as rc_pos
  return addmod(bfe32(i | (i << RC_M), cx & 0xffu, RC_M), cx >> 8, RC_N);
}

// 4-byte copy from global to shared memory, not waited for (rcb_copies_done).
__device__ __forceinline__ void rcb_copy4(float *dst, const float *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(uint32_t(__cvta_generic_to_shared(dst))), "l"(src)
               : "memory");
}
__device__ __forceinline__ void rcb_copies_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ void rcb_persistent(const BwdArgs &a, float *sm) {
  constexpr int kWarps = RCB_WARPS, kAcc = RCB_ACC, kChunk = (RC_N + kWarps - 1) / kWarps, NW = (RC_N + 31) / 32;
  const int lane = int(lane_id()), warp = __shfl_sync(kFull, int(threadIdx.x) >> 5, 0);
  float *y_s = sm, *g_s = y_s + 2 * kRcbN33, *z_s = sm + kRcbHead, *gs_s = z_s + kRcbZ, *c_s = gs_s + kRcbZ;
  uint32_t *u_s = reinterpret_cast<uint32_t *>(c_s + RC_R * 64);
  float *acc_s = reinterpret_cast<float *>(u_s + RC_R * 32);
  float *dsum_s = acc_s + kAcc * kRcbZ;
  float *red_s = dsum_s + 32;
  uint32_t *bad_s = reinterpret_cast<uint32_t *>(red_s + kWarps);
  uint32_t *ctx_s = bad_s + 32, *cols_s = ctx_s + a.P * 32;
  RcbPtr c;
  c.z = reinterpret_cast<const unsigned char *>(z_s + lane);
  c.gs = reinterpret_cast<const unsigned char *>(gs_s + lane);
  c.c = reinterpret_cast<float2 *>(c_s) + lane;
  c.u = u_s + lane;
  c.cols = reinterpret_cast<const uint16_t *>(cols_s);
  c.warp = warp;
  c.nwarps = kWarps;
  const int i0 = min(warp * kChunk, RC_N), P = a.P;
  const float invP = 1.0f / float(P);
  if (threadIdx.x < 32) dsum_s[threadIdx.x] = 0.0f;
  for (int i = int(threadIdx.x); i < RC_R * RC_W4 * 2; i += kWarps * 32)
    cols_s[i] = reinterpret_cast<const uint32_t *>(rcb_cols)[i];
  const int groups = (a.F + 31) / 32;
  for (int grp = int(blockIdx.x); grp < groups; grp += int(gridDim.x)) {
    const int f0 = grp * 32;
    c.live = f0 + lane < a.F;
    // checkpoint t of the group's frames to buffer t & 1: a warp per frame, lanes over
    // positions (coalesced)
    auto fetch = [&](int t) {
      for (int s = warp; s < 32; s += kWarps) {
        const float *src = a.ckpt + (size_t(t) * a.F + min(f0 + s, a.F - 1)) * a.ld;
#pragma unroll
        for (int w = 0; w < NW; w++)
          if (lane + 32 * w < RC_N) rcb_copy4(y_s + (t & 1) * kRcbN33 + (lane + 32 * w) * 33 + s, src + lane + 32 * w);
      }
    };
    fetch(a.I - 1);
    for (int s = warp; s < 32; s += kWarps) {
      const int f = f0 + s;
#pragma unroll
      for (int w = 0; w < NW; w++) {
        const int i = lane + 32 * w;
        if (i < RC_N) g_s[i * 33 + s] = f < a.F ? a.grad_out[size_t(f) * a.ld + i] : 0.0f;
      }
      if (lane < P) {
        uint32_t v = 0;
        if (f < a.F) v = checked_auto(a.autos[size_t(f) * P + lane], RC_N, RC_M, a.check, f);
        ctx_s[lane * 32 + s] = (RC_M - (v >> 8) % RC_M) | ((v & 0xffu) % RC_N) << 8;
      }
    }
    for (int t = a.I; t >= 1; t--) {
      const float *y = y_s + ((t - 1) & 1) * kRcbN33;
      rcb_copies_done();
      __syncthreads();  // y^(t-1) is there; the last iteration has written g and left the other buffer
      if (t > 1) fetch(t - 2);
      c.alpha = a.alpha[t - 1];
      c.dal = 0.0f;
      float gn[kChunk];
      bool odd = false;
#pragma unroll
      for (int k = 0; k < kChunk; k++) {
        const int at = min(i0 + k, RC_N - 1) * 33 + lane;
        gn[k] = g_s[at];
        odd |= !(fabsf(y[at]) <= FLT_MAX);
      }
      if (lane == 0) bad_s[warp] = 0u;
      __syncwarp();
      if (odd) atomicOr(&bad_s[warp], 1u << lane);
      for (int p = 0; p < P; p++) {
        const uint32_t cx = ctx_s[p * 32 + lane];
        uint32_t u[kChunk];
#pragma unroll
        for (int k = 0; k < kChunk; k++) {
          const int i = min(i0 + k, RC_N - 1);
          u[k] = rcb_pos(uint32_t(i), cx) * 32 + lane;
          const float yv = y[i * 33 + lane];
          z_s[u[k]] = yv;
          gs_s[u[k]] = flip_sign(g_s[i * 33 + lane] * invP, __float_as_uint(yv));
        }
#pragma unroll 4
        for (int i = int(threadIdx.x); i < kAcc * kRcbZ; i += kWarps * 32) acc_s[i] = 0.0f;
        __syncthreads();
        if (p == 0) {
          uint32_t bad = 0;
#pragma unroll
          for (int w = 0; w < kWarps; w++) bad |= bad_s[w];
          c.bad = (bad >> lane) & 1u;
        }
        rcb_row_pass(c);
        __syncthreads();
        if (warp < kAcc) {
          // this warp's rows, in order, into its own sums (a row's two variables are the same
          // one only where nothing in it is finite)
          unsigned char *acc = reinterpret_cast<unsigned char *>(acc_s + warp * kRcbZ + lane);
          constexpr int per = (RC_R + kAcc - 1) / kAcc;
          const int r1 = min(RC_R, (warp + 1) * per);
          auto at = [&](uint32_t o) { return reinterpret_cast<float *>(acc + o); };
          // two rows at a time: the second row's values are read ahead of the first's stores
          // and replaced where the variables meet
          int r = warp * per;
#pragma unroll 2
          for (; r + 1 < r1; r += 2) {
            const float2 v = c.c[r * 32], w = c.c[r * 32 + 32];
            const uint32_t i = c.u[r * 32], j = c.u[r * 32 + 32];
            const uint32_t i1 = i & 0xffffu, i2 = i >> 16, j1 = j & 0xffffu, j2 = j >> 16;
            float a1 = *at(i1), a2 = *at(i2), b1 = *at(j1), b2 = *at(j2);
            a1 += v.x;
            a2 = (i1 == i2 ? a1 : a2) + v.y;
            b1 = (j1 == i2 ? a2 : j1 == i1 ? a1 : b1) + w.x;
            b2 = (j2 == j1 ? b1 : j2 == i2 ? a2 : j2 == i1 ? a1 : b2) + w.y;
            *at(i1) = a1;
            *at(i2) = a2;
            *at(j1) = b1;
            *at(j2) = b2;
          }
          if (r < r1) {
            const float2 v = c.c[r * 32];
            const uint32_t i1 = c.u[r * 32] & 0xffffu, i2 = c.u[r * 32] >> 16;
            const float a1 = *at(i1) + v.x, a2 = (i1 == i2 ? a1 : *at(i2)) + v.y;
            *at(i1) = a1;
            *at(i2) = a2;
          }
        }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < kAcc; w++)
#pragma unroll
          for (int k = 0; k < kChunk; k++) gn[k] += acc_s[w * kRcbZ + u[k]];
        if (p + 1 < P) __syncthreads();  // the sums are read before they are cleared
      }
#pragma unroll
      for (int k = 0; k < kChunk; k++)
        if (i0 + k < RC_N) g_s[(i0 + k) * 33 + lane] = gn[k];
      // dL/dalpha_t of this group: lanes, then warps in order
      float d = c.live ? c.dal : 0.0f;
      for (int off = 16; off > 0; off >>= 1) d += __shfl_xor_sync(kFull, d, off);
      if (lane == 0) red_s[warp] = d;
      __syncthreads();
      if (threadIdx.x == 0) {
        float s = 0.0f;
#pragma unroll
        for (int w = 0; w < kWarps; w++) s += red_s[w];
        dsum_s[t - 1] += s;
      }
    }
    if (a.grad_llr)
      for (int s = warp; s < 32; s += kWarps)
        if (f0 + s < a.F)
          for (int i = lane; i < RC_N; i += 32) a.grad_llr[size_t(f0 + s) * a.ld + i] = g_s[i * 33 + s];
    __syncthreads();
  }
  if (int(threadIdx.x) < a.I) a.partial[size_t(blockIdx.x) * a.I + threadIdx.x] = dsum_s[threadIdx.x];
}

}  // namespace bchlib
