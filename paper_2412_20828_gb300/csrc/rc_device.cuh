// Row/column mapping of the enhanced min-sum decoder, compiled at run time for one code.
//
// The one-thread-per-frame kernel (nms_device.cuh) streams the whole Tanner graph as
// straight-line code through every thread: a single frame takes 12 iterations x P copies
// x ~6 k dependent instructions (280 us), and a code of more than ~1000 edges no longer
// fits the instruction cache.  Here a block decodes RC_FB frames together and every
// iteration runs in passes whose tasks are independent:
//   row pass     a task is one check row (of one copy, or of all copies with 32 slots):
//                min1, min2 and the sign product of its z values; the row state
//                (sign min1, sign min2) goes to shared memory
//   column pass  a task is one variable: it adds the row states of its rows in row order
//                -- the additions and their order are those of the straight-line kernel,
//                so both give the same bits
//   merge        a task is one position: the copies' sums in copy order, the new y, its
//                scatter to the copies' permuted words, and its column of the standard
//                matrix into the frame's syndrome (H_o has rank n - k, so both matrices
//                vanish on the same words)
// Every warp follows the slots' frames and iteration counts in its lanes, so an iteration
// has three block barriers (four in the reduced formats, which store y after its scale is
// known) and more only when frames finish.  Shared arrays are
// [index][slot], so with RC_FB = 32 a warp is 32 frames of one task and every access is
// free of bank conflicts.  With RC_FB = 1 a block is one frame: a warp spans 32 tasks, the
// copies of one row or variable next to each other (some bank conflicts, but no frame waits
// for another's time; many such blocks share an SM).  4 and 16 slots lay between the two at
// every batch size.
//
// Needs before this text: RC_FB, RC_PC (number of copies when fixed, else 0), RC_N, RC_M,
// RC_R, RC_KW (words of a syndrome), the column masks rc_cmask, and
//   RC_FB = 32: the tables rc_rowtab, rc_coltab (int4, constant memory: byte offsets into
//     the [index][slot] arrays), and after this text rc_row_pass and rc_column_pass (the
//     classes of rows by weight and of columns by degree);
//   else: RC_W4 (largest row weight / 4), RC_ROWTAB16 / RC_COLTAB16 (lengths) and the tables
//     rc_rowtab16, rc_coltab16 (groups of four 16-bit indices, [group][row or column];
//     the latter after a head {variable, groups} per column).
#pragma once

namespace bchlib {

template <int MSG>
struct RcV {
  using T = float;
};
template <>
struct RcV<kINT8> {
  using T = int;
};
constexpr int kRcZP = (RC_N + 1) | 1, kRcRP = (RC_R + 1) | 1;  // pitches, as in rc_layout

// One thread's view of the block: its slot's columns of the shared arrays and its tasks.
struct RcPtr {
  unsigned char *z;    // + (p kRcZP + u) RC_FB 4
  unsigned char *rs;   // + (p kRcRP + r) RC_FB 8
  unsigned char *rsm;  // 8-bit form: min1 plane, + (p kRcRP + r) RC_FB 4
  const uint2 *rows, *cols;
  int P, task, stride;
  float alpha;
  bool slow;  // the warp holds a frame with a NaN
};

template <int MSG>
__device__ __forceinline__ typename RcV<MSG>::T rc_ld(const unsigned char *p) {
  return *reinterpret_cast<const typename RcV<MSG>::T *>(p);
}

// ---------------------------------------------------------------- rows
// min1 / min2 of a row with a NaN among its values, in the order of the
// one-thread-per-frame kernels (fminf / fmaxf pass over a NaN, and a NaN edge lowers min2
// to the running min1; n = 127: two halves of the variables, then joined).  off(e): byte
// offset of edge e's value.
template <class Off>
__device__ __forceinline__ float2 rc_min12_ordered(const unsigned char *z, int W, const Off &off) {
  float a1 = FLT_MAX, a2 = FLT_MAX, b1 = FLT_MAX, b2 = FLT_MAX;
#pragma unroll 1
  for (int e = 0; e < W; e++) {
    const int o = off(e);
    const float x = fabsf(rc_ld<kFP32>(z + o));
    if (o < 64 * RC_FB * 4) {
      a2 = fminf(a2, fmaxf(a1, x));
      a1 = fminf(a1, x);
    } else {
      b2 = fminf(b2, fmaxf(b1, x));
      b1 = fminf(b1, x);
    }
  }
  return make_float2(fminf(a1, b1), fminf(fmaxf(a1, b1), fminf(a2, b2)));
}

// Row state at byte offset at * 8 (min1 plane: at * 4) from the row's min1, min2 and sign.
template <int MSG>
__device__ __forceinline__ void rc_store_row(const RcPtr &c, int at, typename RcV<MSG>::T m1,
                                             typename RcV<MSG>::T m2, uint32_t sg) {
  if constexpr (MSG == kINT8) {
    const float as = flip_sign(c.alpha, sg);
    const int v1 = rne_product(as, m1);
    *reinterpret_cast<int2 *>(c.rs + at * 8) = make_int2(v1, rne_product(as, m2) - v1);
    *reinterpret_cast<int *>(c.rsm + at * 4) = m1;
  } else if constexpr (MSG == kFP16) {
    // the two messages are binary16 values (the rounded products): one word holds both
    const float as = flip_sign(c.alpha, sg);
    const __half2 h = __floats2half2_rn(half_product(as, m1), half_product(as, m2));
    *reinterpret_cast<float2 *>(c.rs + at * 8) = make_float2(*reinterpret_cast<const float *>(&h), m1);
  } else {
    *reinterpret_cast<float2 *>(c.rs + at * 8) = make_float2(flip_sign(m1, sg), flip_sign(m2, sg));
  }
}

template <class V>
__device__ __forceinline__ uint32_t rc_take(V &v) {  // v to |v|, its sign bits returned
  if constexpr (sizeof(V) == 4 && V(0.5f) == V(0)) {
    const uint32_t s = uint32_t(v);
    v = abs(v);
    return s;
  } else {
    const uint32_t s = __float_as_uint(v);
    v = fabsf(v);
    return s;
  }
}

// One row state into a variable's sum: S + v1, and + (v2 - v1) where |z| is the row's
// minimum -- the rounding of the straight-line rows (v1 = alpha min1 with the row's sign,
// v2 - v1 by one fused multiply-add).  az = |z|.
template <int MSG>
__device__ __forceinline__ void rc_add(const RcPtr &c, typename RcV<MSG>::T &S, typename RcV<MSG>::T az, int at) {
  if constexpr (MSG == kINT8) {
    const int2 st = *reinterpret_cast<const int2 *>(c.rs + at * 8);
    const int m1 = *reinterpret_cast<const int *>(c.rsm + at * 4);
    S += st.x;
    if (az == m1) S += st.y;
  } else if constexpr (MSG == kFP16) {
    const float2 st = *reinterpret_cast<const float2 *>(c.rs + at * 8);
    const __half2 h = *reinterpret_cast<const __half2 *>(&st.x);
    const float v1 = __low2float(h);
    const float dv = __high2float(h) - v1;
    S += v1;
    if (az == st.y) S += dv;
  } else {
    const float2 st = *reinterpret_cast<const float2 *>(c.rs + at * 8);
    const float v1 = c.alpha * st.x;
    const float dv = __fmaf_rn(c.alpha, st.y, -v1);
    S += v1;
    if (az == fabsf(st.x)) S += dv;
  }
}
template <int MSG>
__device__ __forceinline__ typename RcV<MSG>::T rc_sign(typename RcV<MSG>::T S, typename RcV<MSG>::T z) {
  if constexpr (MSG == kINT8) return z < 0 ? -S : S;
  else return flip_sign(S, __float_as_uint(z));
}

#if RC_FB == 32
// ---------------------------------------------------------------- 32 slots: a warp per task
// A task is a row or variable of all copies: the table entries and the address additions
// serve RC_PC copies (the copies' arrays lie at constant offsets).
#define RC_COPIES(p) (RC_PC ? RC_PC : (p))

// The check rows of weight W: nr rows, states r0 ..., table offset t0.
template <int MSG, int W>
__device__ __forceinline__ void rc_rows(const RcPtr &c, int nr, int r0, int t0) {
  using V = typename RcV<MSG>::T;
  int t = c.task - r0 % c.stride;  // the round-robin goes on where the classes before left it
  if (t < 0) t += c.stride;
  for (; t < nr; t += c.stride) {
    const unsigned char *zr[W];
#pragma unroll
    for (int q = 0; q < (W + 3) / 4; q++) {
      const int4 o = rc_rowtab[t0 + t * ((W + 3) / 4) + q];
      zr[4 * q] = c.z + o.x;
      if (4 * q + 1 < W) zr[4 * q + 1 < W ? 4 * q + 1 : 0] = c.z + o.y;
      if (4 * q + 2 < W) zr[4 * q + 2 < W ? 4 * q + 2 : 0] = c.z + o.z;
      if (4 * q + 3 < W) zr[4 * q + 3 < W ? 4 * q + 3 : 0] = c.z + o.w;
    }
#pragma unroll
    for (int p = 0; p < RC_COPIES(c.P); p++) {
      V v[W], m1, m2;
      uint32_t sg = 0;
#pragma unroll
      for (int e = 0; e < W; e++) v[e] = rc_ld<MSG>(zr[e] + p * (kRcZP * 128));
#pragma unroll
      for (int e = 0; e < W; e++) sg ^= rc_take(v[e]);
      min12<V, W>(v, m1, m2);
      if constexpr (MSG == kFP32) {
        m1 = fminf(m1, FLT_MAX);  // the running pair's start value, which rows of infinities show
        m2 = fminf(m2, FLT_MAX);
        if (c.slow) {
          const float2 o = rc_min12_ordered(c.z + p * (kRcZP * 128), W, [&](int e) {
            return reinterpret_cast<const int *>(rc_rowtab)[4 * t0 + t * ((W + 3) & ~3) + e];
          });
          m1 = o.x;
          m2 = o.y;
        }
      }
      rc_store_row<MSG>(c, (p * kRcRP + r0 + t) * 32, m1, m2, sg);
    }
  }
}

// The variables of degree 4 Q - 3 .. 4 Q (padded with the neutral row state): nc of them,
// c0 variables before them in degree order, table offset t0 (per variable a head {byte
// offset of its z, -, -, -} and Q entries of row state indices x 32).
template <int MSG, int Q>
__device__ __forceinline__ void rc_cols(const RcPtr &c, int nc, int c0, int t0) {
  using V = typename RcV<MSG>::T;
  int t = c.task - c0 % c.stride;
  if (t < 0) t += c.stride;
  for (; t < nc; t += c.stride) {
    unsigned char *zu = c.z + rc_coltab[t0 + t * (Q + 1)].x;
#if RC_PC > 0
    V z[RC_PC], S[RC_PC];
#pragma unroll
    for (int p = 0; p < RC_PC; p++) {
      z[p] = rc_ld<MSG>(zu + p * (kRcZP * 128));
      S[p] = 0;
    }
#pragma unroll
    for (int q = 0; q < Q; q++) {
      const int4 o = rc_coltab[t0 + t * (Q + 1) + q + 1];
      const int at[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
      for (int h = 0; h < 4; h++)
#pragma unroll
        for (int p = 0; p < RC_PC; p++) {
          V a = z[p];
          rc_take(a);
          rc_add<MSG>(c, S[p], a, at[h] + p * (kRcRP * 32));
        }
    }
#pragma unroll
    for (int p = 0; p < RC_PC; p++) *reinterpret_cast<V *>(zu + p * (kRcZP * 128)) = rc_sign<MSG>(S[p], z[p]);
#else
    for (int p = 0; p < c.P; p++) {
      const V z = rc_ld<MSG>(zu + p * (kRcZP * 128));
      V S = 0, a = z;
      rc_take(a);
#pragma unroll
      for (int q = 0; q < Q; q++) {
        const int4 o = rc_coltab[t0 + t * (Q + 1) + q + 1];
        rc_add<MSG>(c, S, a, o.x + p * (kRcRP * 32));
        rc_add<MSG>(c, S, a, o.y + p * (kRcRP * 32));
        rc_add<MSG>(c, S, a, o.z + p * (kRcRP * 32));
        rc_add<MSG>(c, S, a, o.w + p * (kRcRP * 32));
      }
      *reinterpret_cast<V *>(zu + p * (kRcZP * 128)) = rc_sign<MSG>(S, z);
    }
#endif
  }
}

template <int MSG>
__device__ __forceinline__ void rc_row_pass(const RcPtr &c);
template <int MSG>
__device__ __forceinline__ void rc_column_pass(const RcPtr &c);

#else
// ---------------------------------------------------------------- one slot: a thread per task
// A task is a row or variable of one copy; the copies of one row are neighbouring lanes.
// Short loops: a block of few warps runs each line of code once or twice an iteration, so
// it pays for fetching instructions as much as for issuing them.
template <int MSG>
__device__ __forceinline__ void rc_row_pass(const RcPtr &c) {
  using V = typename RcV<MSG>::T;
  const int P = RC_PC ? RC_PC : c.P;
  for (int t = c.task; t < P * RC_R; t += c.stride) {
    const int r = t / P, p = t - r * P;
    const unsigned char *z = c.z + p * (kRcZP * RC_FB * 4);
    V m1 = MSG == kINT8 ? V(1 << 20) : V(FLT_MAX), m2 = m1;
    uint32_t sg = 0;
    const uint2 *tab = c.rows + r;
#pragma unroll 2
    for (int q = 0; q < RC_W4; q++) {
      const uint2 o = tab[q * RC_R];
      V x0 = rc_ld<MSG>(z + (o.x & 0xffffu) * (RC_FB * 4)), x1 = rc_ld<MSG>(z + (o.x >> 16) * (RC_FB * 4));
      V x2 = rc_ld<MSG>(z + (o.y & 0xffffu) * (RC_FB * 4)), x3 = rc_ld<MSG>(z + (o.y >> 16) * (RC_FB * 4));
      sg ^= rc_take(x0) ^ rc_take(x1) ^ rc_take(x2) ^ rc_take(x3);
      const V l0 = mn2(x0, x1), h0 = mx2(x0, x1), l1 = mn2(x2, x3), h1 = mx2(x2, x3);
      const V lo = mn2(l0, l1), hi = mn3(mx2(l0, l1), h0, h1);
      m2 = mn3(m2, mx2(m1, lo), hi);
      m1 = mn2(m1, lo);
    }
    if constexpr (MSG == kFP32)
      if (c.slow) {
        const float2 o = rc_min12_ordered(z, 4 * RC_W4, [&](int e) {
          const uint32_t w = reinterpret_cast<const uint32_t *>(tab + (e >> 2) * RC_R)[(e >> 1) & 1];
          return int((w >> (16 * (e & 1))) & 0xffffu) * (RC_FB * 4);
        });
        m1 = o.x;
        m2 = o.y;
      }
    rc_store_row<MSG>(c, (p * kRcRP + r) * RC_FB, m1, m2, sg);
  }
}

template <int MSG>
__device__ __forceinline__ void rc_column_pass(const RcPtr &c) {
  using V = typename RcV<MSG>::T;
  const int P = RC_PC ? RC_PC : c.P;
  const uint32_t *head = reinterpret_cast<const uint32_t *>(c.cols);
  const uint2 *groups = c.cols + (RC_N + 1) / 2;
  for (int t = c.task; t < P * RC_N; t += c.stride) {
    const int i = t / P, p = t - i * P;
    const uint32_t hd = head[i];
    V *zu = reinterpret_cast<V *>(c.z + (p * kRcZP + (hd & 0xffffu)) * (RC_FB * 4));
    const V z = *zu;
    V S = 0, a = z;
    rc_take(a);
    const int base = p * (kRcRP * RC_FB);
#pragma unroll 1
    for (int q = 0; q < int(hd >> 16); q++) {
      const uint2 o = groups[q * RC_N + i];
      rc_add<MSG>(c, S, a, base + int(o.x & 0xffffu) * RC_FB);
      rc_add<MSG>(c, S, a, base + int(o.x >> 16) * RC_FB);
      rc_add<MSG>(c, S, a, base + int(o.y & 0xffffu) * RC_FB);
      rc_add<MSG>(c, S, a, base + int(o.y >> 16) * RC_FB);
    }
    *zu = rc_sign<MSG>(S, z);
  }
}
#endif

// Position pi(i) = 2^j i + s mod n of the packed map cx = (m - j) | s << 8 (j < m, s < n).
__device__ __forceinline__ uint32_t rc_pos(uint32_t i, uint32_t cx) {
  return addmod(bfe32(i | (i << RC_M), cx & 0xffu, RC_M), cx >> 8, RC_N);
}

// ---------------------------------------------------------------- merge
// The merged value of the thread's positions [i0, i1) (numerators for the reduced formats),
// its sign's column mask into the syndrome; FP32 also scatters the new y.
struct RcMerged {
  uint32_t synd[RC_KW];
  float mx;    // reduced formats: largest magnitude
  bool large;  // FP32: a value beyond 2^100, infinite or NaN
};

template <int MSG>
__device__ __forceinline__ RcMerged rc_merge(const NmsArgs &a, const RcPtr &c, const uint32_t *ctx,
                                             typename RcV<MSG>::T *y, int ys, int i0, int i1,
                                             const uint32_t *cmask, uint32_t *cb) {
  using V = typename RcV<MSG>::T;
  const int P = RC_PC ? RC_PC : c.P;
  const float invP = 1.0f / float(P), fP = float(P);
  RcMerged m;
#pragma unroll
  for (int w = 0; w < RC_KW; w++) m.synd[w] = 0u;
  m.mx = 0.0f;
  m.large = false;
#if RC_PC > 0
  // byte offsets pi_p(i) RC_FB 4 of the copies' entries, stepping by 2^j mod n
  constexpr uint32_t kEnd = RC_N * RC_FB * 4;
  uint32_t at[RC_PC], step[RC_PC];
#pragma unroll
  for (int p = 0; p < RC_PC; p++) {
    const uint32_t cx = ctx[p * RC_FB];
    at[p] = rc_pos(uint32_t(i0), cx) * (RC_FB * 4);
    step[p] = (1u << (RC_M - (cx & 0xffu))) * (RC_FB * 4);
  }
#endif
#if RC_FB == 32
#pragma unroll 4
#else
#pragma unroll 1
#endif
  for (int i = i0; i < i1; i++) {
    V acc = 0;
#if RC_PC > 0
#pragma unroll
    for (int p = 0; p < RC_PC; p++) acc += rc_ld<MSG>(c.z + at[p] + p * (kRcZP * RC_FB * 4));
#else
    for (int p = 0; p < P; p++) acc += rc_ld<MSG>(c.z + (p * kRcZP + rc_pos(i, ctx[p * RC_FB])) * (RC_FB * 4));
#endif
    float yn;
    if constexpr (MSG == kFP32) {
      yn = __fmaf_rn(acc, invP, y[i * ys]);
      y[i * ys] = yn;
#if RC_PC > 0
#pragma unroll
      for (int p = 0; p < RC_PC; p++) *reinterpret_cast<V *>(c.z + at[p] + p * (kRcZP * RC_FB * 4)) = yn;
#else
      for (int p = 0; p < P; p++)
        *reinterpret_cast<V *>(c.z + (p * kRcZP + rc_pos(i, ctx[p * RC_FB])) * (RC_FB * 4)) = yn;
#endif
      m.large |= !(fabsf(yn) <= 0x1p100f);
    } else {
      if constexpr (MSG == kINT8)
        yn = BCH_QFRAC(a) ? int8_numerator(y[i * ys], acc, P << BCH_QFRAC(a))
                          : float(y[i * ys]) + __fdiv_rn(float(acc), fP);
      else
        yn = __fmaf_rn(y[i * ys], fP, acc);
      reinterpret_cast<float *>(y)[i * ys] = yn;
      m.mx = fmaxf(m.mx, fabsf(yn));
      // the stored value may round to zero: the hard decision is the numerator's sign
      if (__float_as_uint(yn) >> 31) atomicOr(&cb[(i >> 5) * RC_FB], 1u << (i & 31));
    }
    const uint32_t neg = uint32_t(int(__float_as_uint(yn)) >> 31);
#pragma unroll
    for (int w = 0; w < RC_KW; w++) m.synd[w] ^= neg & cmask[i * RC_KW + w];
#if RC_PC > 0
#pragma unroll
    for (int p = 0; p < RC_PC; p++) at[p] = addmod(at[p], step[p], kEnd);
#endif
  }
  return m;
}

// y of the positions [i0, i1) to the copies' permuted words.
template <int MSG>
__device__ __forceinline__ void rc_scatter(const RcPtr &c, const uint32_t *ctx, const typename RcV<MSG>::T *y,
                                           int ys, int i0, int i1) {
  using V = typename RcV<MSG>::T;
  const int P = RC_PC ? RC_PC : c.P;
#pragma unroll 1
  for (int p = 0; p < P; p++) {
    const uint32_t cx = ctx[p * RC_FB];
    for (int i = i0; i < i1; i++) *reinterpret_cast<V *>(c.z + (p * kRcZP + rc_pos(i, cx)) * (RC_FB * 4)) = y[i * ys];
  }
}

// Halvings that bring max |numerator| mx to the format's limit (rescale on).
template <int MSG>
__device__ __forceinline__ int rc_halvings(const NmsArgs &a, float mx, int P) {
  const float lim = MSG == kINT8 ? (BCH_QFRAC(a) ? 31.0f * float(P << BCH_QFRAC(a)) : 31.0f) : 16384.0f * float(P);
  float sc = 1.0f;
  int kr = 0;
  while (mx * sc > lim && kr < 126) {
    sc *= 0.5f;
    kr++;
  }
  return kr;
}

template <int MSG>
__device__ __forceinline__ void rc_persistent(const NmsArgs &a, uint32_t *sm) {
  using V = typename RcV<MSG>::T;
  constexpr int FB = RC_FB, YS = FB == 32 ? 33 : FB, NW = (RC_N + 31) / 32, KW = RC_KW;
  // the frames of this launch: 0 .. F - 1, or those of a list another kernel wrote
  const int n_frames = a.list ? int(min(*a.list_count, unsigned(a.F))) : a.F;
  if (int(blockIdx.x) * FB >= n_frames) return;
  auto frame = [&](int i) { return i < 0 || i >= n_frames ? -1 : a.list ? int(a.list[i]) : i; };
  const int P = RC_PC ? RC_PC : a.P, tid = int(threadIdx.x), nthr = int(blockDim.x);
  // the shuffle tells the compiler that the warp index, and with it every table index
  // computed from it, is uniform
  const int lane = int(lane_id()), warp = __shfl_sync(kFull, tid >> 5, 0), nwarps = nthr >> 5;
#if RC_FB == 32
  const RcLayout L = rc_layout(RC_N, P, RC_R, FB, MSG == kINT8 ? 3 : 2, KW, 0, 0);
#else
  const RcLayout L = rc_layout(RC_N, P, RC_R, FB, MSG == kINT8 ? 3 : 2, KW, RC_ROWTAB16, RC_COLTAB16);
#endif
  V *y_s = reinterpret_cast<V *>(sm + L.y);
  int *k0_s = reinterpret_cast<int *>(sm + L.k0), *f_s = reinterpret_cast<int *>(sm + L.f);
  uint32_t *cb_s = sm + L.cb, *mx_s = sm + L.mx, *bad_s = sm + L.bad, *synd_s = sm + L.synd, *ctx_s = sm + L.ctx;
  float *alpha_s = reinterpret_cast<float *>(sm + L.alpha);
  const int slot = FB == 32 ? lane : tid % FB;
  RcPtr c;
  c.z = reinterpret_cast<unsigned char *>(sm + L.z) + slot * 4;
  c.rs = reinterpret_cast<unsigned char *>(sm + L.rs) + slot * 8;
  c.rsm = reinterpret_cast<unsigned char *>(sm + L.rsm) + slot * 4;
  c.rows = reinterpret_cast<const uint2 *>(sm + L.tab_rows);
  c.cols = reinterpret_cast<const uint2 *>(sm + L.tab_cols);
  c.P = P;
  c.task = FB == 32 ? warp : tid / FB;
  c.stride = FB == 32 ? nwarps : nthr / FB;
  c.slow = false;
  V *y = y_s + slot;
  const uint32_t *ctx = ctx_s + slot;
  // positions of this thread in the merge
  const int chunk = (RC_N + c.stride - 1) / c.stride;
  const int i0 = min(c.task * chunk, RC_N), i1 = min(i0 + chunk, RC_N);

  if (tid < 32) alpha_s[tid] = a.alpha[tid];
  for (int i = tid; i < P * FB; i += nthr) {
    const int p = i / FB, s = i - p * FB;
    ctx_s[i] = uint32_t(RC_M);  // idle slots run on a valid map
    // the neutral value and the neutral row of every copy
    reinterpret_cast<V *>(sm + L.z)[(p * kRcZP + RC_N) * FB + s] = MSG == kINT8 ? V(1 << 20) : V(FLT_MAX);
    const int at = (p * kRcRP + RC_R) * FB + s;
    reinterpret_cast<uint2 *>(sm + L.rs)[at] = make_uint2(0u, 0u);
    if constexpr (MSG == kINT8) (sm + L.rsm)[at] = 0xffffffffu;
  }
  for (int i = tid; i < FB; i += nthr) bad_s[i] = 0u;
  for (int i = tid; i < KW * RC_N; i += nthr) (sm + L.cmask)[i] = rc_cmask[i];
#if RC_FB < 32
  for (int i = tid; i < (RC_ROWTAB16 + 1) / 2; i += nthr)
    (sm + L.tab_rows)[i] = reinterpret_cast<const uint32_t *>(rc_rowtab16)[i];
  for (int i = tid; i < (RC_COLTAB16 + 1) / 2; i += nthr)
    (sm + L.tab_cols)[i] = reinterpret_cast<const uint32_t *>(rc_coltab16)[i];
#endif
  __syncthreads();
  // Lane s of every warp holds slot s's frame, iteration count and exponent.  The block's
  // first frames are fixed; later ones come from the queue.
  const int start = int(gridDim.x) * FB;
  int my_f = lane < FB ? frame(int(blockIdx.x) * FB + lane) : -1, my_t = 0, my_e = 0;
  uint32_t nw = __ballot_sync(kFull, my_f >= 0);
  for (;;) {
    if (nw) {
      // a warp per new slot, lanes over positions (copies): the frame's input and maps
      for (int s = warp; s < FB; s += nwarps) {
        const int f = __shfl_sync(kFull, my_f, s);
        if (!((nw >> s) & 1u)) continue;
        const float *src = a.llr + size_t(f) * a.ld;
        float x[NW];
#pragma unroll
        for (int w = 0; w < NW; w++) x[w] = lane + 32 * w < RC_N ? src[lane + 32 * w] + 0.0f : 0.0f;  // -0 -> +0
        if (lane < P) {
          const uint32_t v = checked_auto(a.autos[size_t(f) * P + lane], RC_N, RC_M, a.check, f);
          ctx_s[lane * FB + s] = (RC_M - (v >> 8) % RC_M) | ((v & 0xffu) % RC_N) << 8;
        }
        if constexpr (MSG == kFP32) {
          bool odd = false;
#pragma unroll
          for (int w = 0; w < NW; w++) odd |= x[w] != x[w];
          const bool any = __any_sync(kFull, odd);
          if (lane == 0) bad_s[s] = any ? 1u : 0u;
        }
        float s4 = 4.0f;
        if constexpr (MSG == kINT8) {
          int k = 0;
          if (BCH_QFRAC(a) && a.rescale) {  // as int8_input_shift, by the whole warp
            float mx = 0.0f;
#pragma unroll
            for (int w = 0; w < NW; w++) mx = fmaxf(mx, fabsf(4.0f * x[w]));
            for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, off));
            float lim = 31.0f;
            while (mx > lim && k < 60) {
              lim *= 2.0f;
              k++;
            }
            s4 = ldexpf(4.0f, -k);
          }
          if (lane == 0) k0_s[s] = k;
        }
#pragma unroll
        for (int w = 0; w < NW; w++) {
          const int i = lane + 32 * w;
          if (i < RC_N) {
            if constexpr (MSG == kFP32) y_s[i * YS + s] = x[w];
            if constexpr (MSG == kFP16) y_s[i * YS + s] = __half2float(to_half_sat(x[w]));
            if constexpr (MSG == kINT8) y_s[i * YS + s] = int(to_q(s4 * x[w]));
            if (a.ckpt) a.ckpt[size_t(f) * a.ld + i] = x[w];
          }
        }
      }
      __syncthreads();
      if ((nw >> slot) & 1u) rc_scatter<MSG>(c, ctx, y, YS, i0, i1);
      if ((nw >> lane) & 1u) {
        my_t = 0;
        my_e = MSG == kINT8 ? k0_s[lane] : 0;
      }
      __syncthreads();
    }
    const uint32_t act = __ballot_sync(kFull, my_f >= 0);
    if (!act) break;
    const bool live = (act >> slot) & 1u;  // idle slots run on whatever their columns hold
    c.alpha = alpha_s[__shfl_sync(kFull, my_t, slot) & 31];
    if constexpr (MSG == kFP32) c.slow = __any_sync(kFull, live && bad_s[slot] != 0u);
    rc_row_pass<MSG>(c);
    __syncthreads();
    if (warp == nwarps - 1 && lane < FB) {  // the merge's accumulators (last read before the row pass)
#pragma unroll
      for (int w = 0; w < KW; w++) synd_s[w * FB + lane] = 0u;
      mx_s[lane] = 0u;
      if constexpr (MSG != kFP32) {
#pragma unroll
        for (int w = 0; w < NW; w++) cb_s[w * FB + lane] = 0u;
      }
    }
    rc_column_pass<MSG>(c);
    __syncthreads();
    {
      RcMerged m = rc_merge<MSG>(a, c, ctx, y, YS, i0, i1, sm + L.cmask, cb_s + slot);
      // lanes of one slot first join their parts
#pragma unroll
      for (int w = 0; w < KW; w++) {
#pragma unroll
        for (int off = FB; off < 32; off <<= 1) m.synd[w] ^= __shfl_xor_sync(kFull, m.synd[w], off);
        if (lane < FB && m.synd[w]) atomicXor(&synd_s[w * FB + slot], m.synd[w]);
      }
      if constexpr (MSG == kFP32) {
        if (__any_sync(kFull, live && m.large)) {
          // rare: mark the slots with a finite or infinite value past 2^100, and those with a NaN
          for (int i = i0; i < i1; i++) {
            const float v = fabsf(y[i * YS]);
            if (v > 0x1p100f) mx_s[slot] = 1u;
            if (v != v) bad_s[slot] = 1u;
          }
        }
      } else if (a.rescale) {
#pragma unroll
        for (int off = FB; off < 32; off <<= 1) m.mx = fmaxf(m.mx, __shfl_xor_sync(kFull, m.mx, off));
        if (lane < FB) atomicMax(&mx_s[slot], __float_as_uint(m.mx));
      }
    }
    __syncthreads();
    uint32_t nz = 0;
    if (my_f >= 0) {
#pragma unroll
      for (int w = 0; w < KW; w++) nz |= synd_s[w * FB + lane];
      my_t++;
    }
    if constexpr (MSG == kFP32) {
      const bool big = my_f >= 0 && !a.ckpt && mx_s[my_f >= 0 ? lane : 0] != 0u;
      const uint32_t bigm = __ballot_sync(kFull, big);
      if (bigm) {  // exact power-of-two renormalisation past 2^100 (as in the one-thread kernel)
        if (big) my_e += 64;
        if ((bigm >> slot) & 1u) {
          for (int i = i0; i < i1; i++) y[i * YS] *= 0x1p-64f;
          rc_scatter<MSG>(c, ctx, y, YS, i0, i1);
        }
        __syncthreads();
      }
    } else {
      int kr = 0;
      if (a.rescale) {
        kr = rc_halvings<MSG>(a, __uint_as_float(mx_s[slot]), P);
        if (my_f >= 0) my_e += rc_halvings<MSG>(a, __uint_as_float(mx_s[lane]), P);
      }
      const float sc = ldexpf(1.0f, -kr);
      for (int i = i0; i < i1; i++) {
        const float num = reinterpret_cast<float *>(y)[i * YS];
        if constexpr (MSG == kINT8)
          y[i * YS] = BCH_QFRAC(a) ? int8_store_quotient(num, kr, P << BCH_QFRAC(a)) : to_q(num * sc);
        else
          y[i * YS] = __half2float(half_of_quotient(num * sc, float(P)));
      }
      rc_scatter<MSG>(c, ctx, y, YS, i0, i1);
      __syncthreads();
    }
    if (a.ckpt)
      for (int s = warp; s < FB; s += nwarps) {
        const int f = __shfl_sync(kFull, my_f, s), t = __shfl_sync(kFull, my_t, s);
        if (f < 0) continue;
        float *dst = a.ckpt + (size_t(t) * a.F + f) * a.ld;
        for (int i = lane; i < RC_N; i += 32) dst[i] = float(y_s[i * YS + s]);
      }
    const bool fin = my_f >= 0 && (my_t >= a.I || (a.early_stop && nz == 0));
    const uint32_t finm = __ballot_sync(kFull, fin);
    nw = 0;
    if (!finm) continue;
    // ---- outputs of the finished slots, a warp per slot
    for (int s = warp; s < FB; s += nwarps) {
      const int f = __shfl_sync(kFull, my_f, s), t = __shfl_sync(kFull, my_t, s), e = __shfl_sync(kFull, my_e, s);
      const bool ok = __shfl_sync(kFull, nz, s) == 0u;
      if (!((finm >> s) & 1u)) continue;
      uint32_t cb[NW];
#pragma unroll
      for (int w = 0; w < NW; w++) {
        if constexpr (MSG == kFP32) {
          const int i = lane + 32 * w;
          cb[w] = __ballot_sync(kFull, i < RC_N && (__float_as_uint(y_s[min(i, RC_N - 1) * YS + s]) >> 31));
        } else {
          cb[w] = cb_s[w * FB + s];
        }
      }
      if (lane == 0) {
        if (a.hard) write_hard<NW>(a.hard, f, cb);
        if (a.iters) a.iters[f] = uint8_t(t);
        if (a.flags) a.flags[f] = ok ? uint8_t(kFlagConverged) : 0;
      }
      if (a.llr_out) {
        float *dst = a.llr_out + size_t(f) * a.ld;
        const float unit = MSG == kINT8 ? 0.25f : 1.0f;
        for (int i = lane; i < RC_N; i += 32) dst[i] = ldexpf(float(y_s[i * YS + s]) * unit, e);
      }
    }
    if (n_frames > start) {
      if (warp == 0) {
        const int got = pull_frame(a.queue, fin, n_frames - start);
        if (fin) f_s[lane] = got >= 0 ? frame(got + start) : -1;
      }
      __syncthreads();
      if (fin) my_f = f_s[lane];
    } else if (fin) {
      my_f = -1;
    }
    nw = __ballot_sync(kFull, fin && my_f >= 0);
  }
}

}  // namespace bchlib
