// Shared-memory layout of the row/column kernels (32-bit words), used by the host to size
// a launch and by the kernels compiled at run time to carve it up.  No includes under
// NVRTC.
#pragma once

namespace bchlib {

struct RcLayout {
  int zp, rp;  // pitches of a copy: entries of z (n, a neutral one, made odd), row states
  int y, z, rs, rsm, cb, mx, bad, synd, k0, f, ctx, alpha, cmask, tab_rows, tab_cols, words;
};

// n columns, P copies, R rows (plus one neutral row state), FB frame slots; rs_words
// words per row state (2, or 3 for the 8-bit form); kw words per syndrome; tab_*: lengths
// of the 16-bit index tables (kept in shared memory when a warp spans several tasks).
// Odd pitches put the copies of one variable or row in different banks.
#ifdef __CUDACC__
__host__ __device__
#endif
inline RcLayout rc_layout(int n, int P, int R, int FB, int rs_words, int kw, int tab_rows, int tab_cols) {
  RcLayout L;
  L.zp = (n + 1) | 1;
  L.rp = (R + 1) | 1;
  int o = 0;
  L.y = o;  // y[n], row stride 33 for 32 slots: a warp reads a frame's column without conflicts
  o += (n * (FB == 32 ? 33 : FB) + 3) & ~3;
  L.z = o;
  o += (P * L.zp * FB + 3) & ~3;
  L.rs = o;
  o += (P * L.rp * FB * 2 + 3) & ~3;
  L.rsm = o;
  if (rs_words > 2) o += (P * L.rp * FB + 3) & ~3;
  L.cb = o;
  o += 4 * FB;
  L.mx = o;
  o += FB;
  L.bad = o;
  o += FB;
  L.synd = o;
  o += kw * FB;
  L.k0 = o;
  o += FB;
  L.f = o;
  o += FB;
  L.ctx = o;
  o += P * FB;
  L.alpha = o;
  o += 32;
  L.cmask = o;
  o += kw * n;
  o = (o + 3) & ~3;  // the tables are read 64 bits at a time
  L.tab_rows = o;
  if (FB < 32) o += (tab_rows + 1) / 2;
  o = (o + 3) & ~3;
  L.tab_cols = o;
  if (FB < 32) o += (tab_cols + 1) / 2;
  L.words = o;
  return L;
}

// The plain decoder's kernel (rc_plain.cuh): channel values and totals (with a padded edge's
// value), messages (with a neutral one), the tables.
struct RcpLayout {
  int ch, x, msg, synd, f, alpha, cmask, rows, cols, words;
};
#ifdef __CUDACC__
__host__ __device__
#endif
inline RcpLayout rcp_layout(int n, int R, int w4, int FB, int kw, int tab_rows, int tab_cols) {
  RcpLayout L;
  int o = 0;
  L.ch = o;
  o += n * (FB == 32 ? 33 : FB);
  L.x = o;
  o += (n + 1) * FB;
  L.msg = o;
  o += (R * 4 * w4 + 1) * FB;
  L.synd = o;
  o += kw * FB;
  L.f = o;
  o += FB;
  L.alpha = o;
  o += 32;
  L.cmask = o;
  o += kw * n;
  o = (o + 1) & ~1;
  L.rows = o;
  o += (tab_rows + 1) / 2;
  o = (o + 1) & ~1;
  L.cols = o;
  o += (tab_cols + 1) / 2;
  L.words = o;
  return L;
}

// Words of the backward kernel (rc_backward.cuh) with n_acc sums.
#ifdef __CUDACC__
__host__ __device__
#endif
inline int rcb_words(int n, int P, int R, int w4, int warps, int n_acc) {
  return ((3 * n * 33 + 3) & ~3) + 2 * n * 32 + R * 96 + n_acc * n * 32 + 32 + warps + 32 + P * 32 +
         R * w4 * 2;
}

}  // namespace bchlib
