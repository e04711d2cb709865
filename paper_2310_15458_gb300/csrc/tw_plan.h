// Shared memory of the tensor-core sweeps' products (sweep_tc.cuh), and which colour
// classes fit it.  Host code only.
#pragma once
#include <algorithm>

constexpr int TW_MAXN = 1024;                 // rows of the products that write what they read: a cluster of 8 tiles
constexpr int TW_MAXC = 6000;                 // (the plan's own limit lies below)
constexpr int TW_SMEM = 222 * 1024;

// NST stages of the rows' digits (rows8 rows of 8 slices x 32 entries) and of 2 gw real
// columns, then the places in x of the K rows and the exponents of rows and columns in up
// to nstr stretches of K.
struct TwPlan {
  int rows8, nst, nstr, smem;
};
// ks: entries of K of a stage, sx: stages of a stretch
inline TwPlan tw_plan(int max_rows, int max_k, int gw, int ks, int sx) {
  TwPlan p;
  p.rows8 = std::min(128, (max_rows + 7) & ~7);
  const int st = p.rows8 * 512 + 1024 * gw, ns = (max_k + ks - 1) / ks;
  // the products of a short tile read (and ignore) up to 128 rows past each slice
  p.nstr = (ns + sx - 1) / sx + 1;   // (a share of K may start inside a stretch)
  const int tail = (int)sizeof(int) * (max_k + p.nstr * (128 + 2 * gw)) + (128 - p.rows8) * 64;
  p.nst = std::max(2, std::min({4, std::max(ns, 2), (TW_SMEM - tail) / st}));
  p.smem = p.nst * st + tail;
  return p;
}

// entries of K of a stage, and stages that share scales and sums, for a class whose boxes
// have at most n points (the reasons: sweep_tc.cuh)
constexpr int TW_SX = 12, TW_SX_LONG = 2, TW_SXZ = 3;
inline int tw_stage(bool real) { return real ? 32 : 16; }
inline int tw_stages(bool real, int n) { return real ? (n > 128 ? TW_SX_LONG : TW_SX) : TW_SXZ; }
enum { TW_UPW = 0, TW_UPE = 1, TW_DNF = 2, TW_DNW = 3 };
// the launch of product op for a class whose boxes have at most n points, r of them
// redundant, and c neighbours
inline TwPlan tw_plan_op(int op, int n, int r, int c, int gw, bool real) {
  const int rows = op == TW_UPE ? std::max(1, c) : op == TW_DNW ? n : r, k = op == TW_UPW ? n : op == TW_DNF ? c : r;
  return tw_plan(rows, k, gw, tw_stage(real), tw_stages(real, n));
}
// columns of a group: 32, or 16 where 32 do not fit
inline int tw_group(int op, int n, int r, int c, bool real) {
  return tw_plan_op(op, n, r, c, 32, real).smem > TW_SMEM ? 16 : 32;
}
// Whether all four products of such a class fit.  (With 128 rows and two stages, groups of
// 32 columns do up to c of about 5,000 (n <= 128) and 1,800 for real factors and 1,500 for
// complex ones; groups of 16 up to the limit, 4,400 and 3,600.)
inline bool tw_shape_fits(int n, int r, int c, bool real) {
  if (n > TW_MAXN || c > TW_MAXC) return false;
  for (int op = 0; op < 4; ++op)
    if (tw_plan_op(op, n, r, c, 16, real).smem > TW_SMEM) return false;
  return true;
}
