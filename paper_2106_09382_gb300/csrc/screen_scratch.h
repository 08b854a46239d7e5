// The screened kernel's scratch block: candidate lists and per-candidate,
// per-row arrays, carved from one allocation of the FP64 widths (both
// precisions fit).  Internal: not part of the C ABI.
#pragma once
#include "kernels.h"

namespace concord {

struct ScreenLayout {
  size_t ctr, cand0, cand1, cnt_r0, cnt_r1, fail, off_r, cur_r, nd_pi, nd_pj, row_ent, term_ptr, term_pred, term_s, nd_rec, nd_delta, nd_new, jac,
      diag_old, omdiag_old, diag_new, dpart, dfill, diag_dd, pend_u, pend_d, pend_n, pend_new,
      rowacc, rowa_new, apart, loud, loudf, total;
};

inline ScreenLayout screen_layout(int p, int P, int nc, int tc) {
  ScreenLayout L;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off += (bytes + 255) / 256 * 256;
    return at;
  };
  L.ctr = take(sizeof(int) * kCtrs);
  L.cand0 = take(sizeof(int2) * (size_t)nc);
  L.cand1 = take(sizeof(int2) * (size_t)nc);
  L.cnt_r0 = take(sizeof(int) * (size_t)(p + 1));
  L.cnt_r1 = take(sizeof(int) * (size_t)(p + 1));
  L.fail = take(sizeof(int2) * (size_t)nc);
  L.off_r = take(sizeof(int) * (size_t)(p + 1));
  L.cur_r = take(sizeof(int) * (size_t)(p + 1));
  L.nd_pi = take(sizeof(int) * (size_t)nc);
  L.nd_pj = take(sizeof(int) * (size_t)nc);
  L.row_ent = take(sizeof(int) * 2 * (size_t)nc);
  L.term_ptr = take(sizeof(int) * ((size_t)nc + 1));
  L.term_pred = take(sizeof(int) * (size_t)tc);
  L.term_s = take(sizeof(double) * (size_t)tc);
  L.nd_rec = take(sizeof(double) * 4 * (size_t)nc);
  L.nd_delta = take(sizeof(double) * (size_t)nc);
  L.nd_new = take(sizeof(double) * (size_t)nc);
  L.jac = take(sizeof(unsigned long long) * kJacMax);
  L.diag_old = take(sizeof(double) * (size_t)p);

  L.omdiag_old = take(sizeof(double) * (size_t)p);
  L.diag_new = take(sizeof(double) * (size_t)p);
  L.dpart = take(sizeof(double) * 1024);
  L.dfill = take(sizeof(int) * 1024);
  L.diag_dd = take(sizeof(double) * (size_t)p);
  L.pend_u = take(sizeof(int) * (size_t)p * kPendRow);
  L.pend_d = take(sizeof(double) * (size_t)p * kPendRow);
  L.pend_n = take(sizeof(int) * (size_t)p);
  L.pend_new = take(sizeof(int) * (size_t)p);
  L.rowacc = take(sizeof(double) * (size_t)p);
  L.rowa_new = take(sizeof(double) * (size_t)p);
  L.apart = take(sizeof(double) * 1024);
  L.loud = take(sizeof(int) * kLoudMax);
  L.loudf = take(sizeof(int) * (size_t)p);
  L.total = off;
  return L;
}

template <typename T>
ScreenWork<T> screen_work_at(void* scr, int p, int P, int nc, int tc) {
  const ScreenLayout L = screen_layout(p, P, nc, tc);
  char* b = (char*)scr;
  ScreenWork<T> w;
  w.ctr = (int*)(b + L.ctr);
  w.cand[0] = (int2*)(b + L.cand0);
  w.cand[1] = (int2*)(b + L.cand1);
  w.cnt_r[0] = (int*)(b + L.cnt_r0);
  w.cnt_r[1] = (int*)(b + L.cnt_r1);
  w.fail = (int2*)(b + L.fail);
  w.off_r = (int*)(b + L.off_r);
  w.cur_r = (int*)(b + L.cur_r);
  w.nd_pi = (int*)(b + L.nd_pi);
  w.nd_pj = (int*)(b + L.nd_pj);
  w.row_ent = (int*)(b + L.row_ent);
  w.term_ptr = (int*)(b + L.term_ptr);
  w.term_pred = (int*)(b + L.term_pred);
  w.term_s = (T*)(b + L.term_s);
  w.nd_rec = (T*)(b + L.nd_rec);
  w.nd_delta = (T*)(b + L.nd_delta);
  w.nd_new = (T*)(b + L.nd_new);
  w.jac = (unsigned long long*)(b + L.jac);
  w.diag_old = (T*)(b + L.diag_old);

  w.omdiag_old = (double*)(b + L.omdiag_old);
  w.diag_new = (double*)(b + L.diag_new);
  w.dpart = (double*)(b + L.dpart);
  w.dfill = (int*)(b + L.dfill);
  w.diag_dd = (T*)(b + L.diag_dd);
  w.pend_u = (int*)(b + L.pend_u);
  w.pend_d = (T*)(b + L.pend_d);
  w.pend_n = (int*)(b + L.pend_n);
  w.pend_new = (int*)(b + L.pend_new);
  w.rowacc = (double*)(b + L.rowacc);
  w.rowa_new = (double*)(b + L.rowa_new);
  w.apart = (double*)(b + L.apart);
  w.loud = (int*)(b + L.loud);
  w.loudf = (int*)(b + L.loudf);
  w.nc_cap = nc;
  w.term_cap = tc;
  w.fail_cap = nc;
  return w;
}

}  // namespace concord
