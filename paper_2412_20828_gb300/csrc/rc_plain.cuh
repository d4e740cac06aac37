// Plain (single-decoder) normalized min-sum, Eqs. (2)-(5), row by row and column by column
// like rc_device.cuh, compiled at run time for one code: a block decodes RC_FB frames with
// every edge's check-to-variable message in shared memory.
//   row pass     a task is one check row: v2c = total - own message, min1 / min2 / first
//                minimum / signs in edge order, then the row's new messages
//   column pass  a task is one variable: the channel value plus its messages in row order,
//                the new total and hard decision, and its column of the standard matrix into
//                the frame's syndrome
// The operations and their order are those of nms_plain_kernel: the same bits.  That kernel
// ran a frame's 8 iterations x 486 edges as one thread's chain, 64 frames per SM: 10 000
// frames of BCH(63,36) took 372 us.
//
// Needs before this text: RC_FB, RC_N, RC_R, RC_KW, RC_W4 (largest row weight / 4), RC_D4
// (largest column degree / 4) and the 16-bit tables rcp_rows (groups of four variables,
// [group][row], padded with RC_N) and rcp_cols (a head {variable, groups} per column, then
// groups of four message indices, [group][column], padded with the neutral message RC_R 4 RC_W4)
// with their lengths RCP_ROWS, RCP_COLS, and rc_cmask.
#pragma once

namespace bchlib {

constexpr int kRcpM = RC_R * 4 * RC_W4;  // messages per frame; one more stays 0

__device__ __forceinline__ void rcp_persistent(const NmsArgs &a, uint32_t *sm) {
  constexpr int FB = RC_FB, YS = FB == 32 ? 33 : FB, NW = (RC_N + 31) / 32, KW = RC_KW;
  const int tid = int(threadIdx.x), nthr = int(blockDim.x), lane = int(lane_id());
  const int warp = __shfl_sync(kFull, tid >> 5, 0), nwarps = nthr >> 5;
  const RcpLayout L = rcp_layout(RC_N, RC_R, RC_W4, FB, KW, RCP_ROWS, RCP_COLS);
  float *L_s = reinterpret_cast<float *>(sm + L.ch), *x_s = reinterpret_cast<float *>(sm + L.x);
  float *m_s = reinterpret_cast<float *>(sm + L.msg);
  uint32_t *synd_s = sm + L.synd;
  int *f_s = reinterpret_cast<int *>(sm + L.f);
  const uint32_t *cmask = sm + L.cmask;
  const uint2 *rows = reinterpret_cast<const uint2 *>(sm + L.rows);
  const uint32_t *head = sm + L.cols;
  const uint2 *cols = reinterpret_cast<const uint2 *>(head) + (RC_N + 1) / 2;
  float *alpha_s = reinterpret_cast<float *>(sm + L.alpha);
  const int slot = FB == 32 ? lane : tid % FB, task = FB == 32 ? warp : tid / FB;
  const int stride = FB == 32 ? nwarps : nthr / FB;
  float *x = x_s + slot, *msg = m_s + slot;
  const float *ch = L_s + slot;

  if (tid < 32) alpha_s[tid] = a.alpha[tid];
  for (int i = tid; i < KW * RC_N; i += nthr) (sm + L.cmask)[i] = rc_cmask[i];
  for (int i = tid; i < (RCP_ROWS + 1) / 2; i += nthr) (sm + L.rows)[i] = reinterpret_cast<const uint32_t *>(rcp_rows)[i];
  for (int i = tid; i < (RCP_COLS + 1) / 2; i += nthr) (sm + L.cols)[i] = reinterpret_cast<const uint32_t *>(rcp_cols)[i];
  for (int i = tid; i < FB; i += nthr) {
    x_s[RC_N * FB + i] = FLT_MAX;  // the value of padded edges
    m_s[kRcpM * FB + i] = 0.0f;    // the neutral message
  }
  __syncthreads();
  // Lane s of every warp follows slot s (as in rc_persistent).
  const int start = int(gridDim.x) * FB;
  int my_f = lane < FB ? int(blockIdx.x) * FB + lane : -1, my_t = 0;
  if (my_f >= a.F) my_f = -1;
  uint32_t nw = __ballot_sync(kFull, my_f >= 0);
  for (;;) {
    if (nw) {
      for (int s = warp; s < FB; s += nwarps) {
        const int f = __shfl_sync(kFull, my_f, s);
        if (!((nw >> s) & 1u)) continue;
        const float *src = a.llr + size_t(f) * a.ld;
        for (int i = lane; i < RC_N; i += 32) {
          const float v = src[i] + 0.0f;
          L_s[i * YS + s] = v;
          x_s[i * FB + s] = v;
        }
      }
      if ((nw >> slot) & 1u)
        for (int i = task; i < kRcpM; i += stride) msg[i * FB] = 0.0f;
      if ((nw >> lane) & 1u) my_t = 0;
      __syncthreads();
    }
    if (!__any_sync(kFull, my_f >= 0)) break;
    const float alpha = alpha_s[__shfl_sync(kFull, my_t, slot) & 31];
    for (int r = task; r < RC_R; r += stride) {
      float *mr = msg + r * (4 * RC_W4 * FB);
      float m1 = FLT_MAX, m2 = FLT_MAX;
      uint32_t am = 0, sg = 0, lo = 0, hi = 0;
#if RC_FB == 32
#pragma unroll
#else
#pragma unroll 2
#endif
      for (int q = 0; q < RC_W4; q++) {
        const uint2 o = rows[q * RC_R + r];
        const uint32_t u[4] = {o.x & 0xffffu, o.x >> 16, o.y & 0xffffu, o.y >> 16};
#pragma unroll
        for (int h = 0; h < 4; h++) {
          const int e = 4 * q + h;
          const float v = x[u[h] * FB] - mr[e * FB];  // Eq. (2); a padded edge's message stays 0
          const float ax = fabsf(v);
          if (ax < m1) am = uint32_t(e);
          m2 = fminf(m2, fmaxf(m1, ax));
          m1 = fminf(m1, ax);
          const uint32_t xs = __float_as_uint(v) >> 31;
          sg ^= xs;
          if (e < 32) lo |= xs << (e & 31);
          else hi |= xs << (e & 31);
        }
      }
      const float v1 = flip_sign(alpha * m1, sg << 31), v2 = flip_sign(alpha * m2, sg << 31);
#if RC_FB == 32
#pragma unroll
#else
#pragma unroll 2
#endif
      for (int q = 0; q < RC_W4; q++) {
        const uint2 o = rows[q * RC_R + r];
        const uint32_t u[4] = {o.x & 0xffffu, o.x >> 16, o.y & 0xffffu, o.y >> 16};
#pragma unroll
        for (int h = 0; h < 4; h++) {
          const int e = 4 * q + h;
          const uint32_t xs = e < 32 ? lo << (31 - (e & 31)) : hi << (31 - (e & 31));
          if (u[h] != RC_N) mr[e * FB] = flip_sign(am == uint32_t(e) ? v2 : v1, xs);
        }
      }
    }
    if (warp == nwarps - 1 && lane < FB) {  // every warp has read it (barriers below)
#pragma unroll
      for (int w = 0; w < KW; w++) synd_s[w * FB + lane] = 0u;
    }
    __syncthreads();
    uint32_t synd[KW];
#pragma unroll
    for (int w = 0; w < KW; w++) synd[w] = 0u;
    for (int i = task; i < RC_N; i += stride) {
      const uint32_t hd = head[i], u = hd & 0xffffu;
      float S = ch[u * YS];
#pragma unroll 2
      for (int q = 0; q < int(hd >> 16); q++) {
        const uint2 o = cols[q * RC_N + i];
        const float c0 = msg[(o.x & 0xffffu) * FB], c1 = msg[(o.x >> 16) * FB];
        const float c2 = msg[(o.y & 0xffffu) * FB], c3 = msg[(o.y >> 16) * FB];
        S += c0;
        S += c1;
        S += c2;
        S += c3;
      }
      x[u * FB] = S;
      const uint32_t neg = uint32_t(int(__float_as_uint(S)) >> 31);
#pragma unroll
      for (int w = 0; w < KW; w++) synd[w] ^= neg & cmask[u * KW + w];
    }
#pragma unroll
    for (int w = 0; w < KW; w++) {
#pragma unroll
      for (int off = FB; off < 32; off <<= 1) synd[w] ^= __shfl_xor_sync(kFull, synd[w], off);
      if (lane < FB && synd[w]) atomicXor(&synd_s[w * FB + slot], synd[w]);
    }
    __syncthreads();
    uint32_t nz = 0;
    if (my_f >= 0) {
#pragma unroll
      for (int w = 0; w < KW; w++) nz |= synd_s[w * FB + lane];
      my_t++;
    }
    const bool fin = my_f >= 0 && (my_t >= a.I || (a.early_stop && nz == 0));
    const uint32_t finm = __ballot_sync(kFull, fin);
    nw = 0;
    if (!finm) {
      __syncthreads();  // every warp has read the syndrome before it is cleared
      continue;
    }
    for (int s = warp; s < FB; s += nwarps) {
      const int f = __shfl_sync(kFull, my_f, s), t = __shfl_sync(kFull, my_t, s);
      const bool ok = __shfl_sync(kFull, nz, s) == 0u;
      if (!((finm >> s) & 1u)) continue;
      uint32_t cb[NW];
#pragma unroll
      for (int w = 0; w < NW; w++) {
        const int i = lane + 32 * w;
        const float v = x_s[min(i, RC_N - 1) * FB + s];
        cb[w] = __ballot_sync(kFull, i < RC_N && (__float_as_uint(v) >> 31));
        if (a.llr_out && i < RC_N) a.llr_out[size_t(f) * a.ld + i] = v;
      }
      if (lane == 0) {
        if (a.hard) write_hard<NW>(a.hard, f, cb);
        if (a.iters) a.iters[f] = uint8_t(t);
        if (a.flags) a.flags[f] = ok ? uint8_t(kFlagConverged) : 0;
      }
    }
    if (a.F > start) {
      if (warp == 0) {
        const int got = pull_frame(a.queue, fin, a.F - start);
        if (fin) f_s[lane] = got >= 0 ? got + start : -1;
      }
      __syncthreads();
      if (fin) my_f = f_s[lane];
    } else {
      __syncthreads();
      if (fin) my_f = -1;
    }
    nw = __ballot_sync(kFull, fin && my_f >= 0);
  }
}

}  // namespace bchlib
