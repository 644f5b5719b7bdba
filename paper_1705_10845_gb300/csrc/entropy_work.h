// Work area of the entropy's log-determinants: cap matrices np x np, and per matrix the rows below a panel,
// the panel's inverse factor and the panels' parts.
//
// One area serves all systems of a context, since their energies run one after another on its stream, and it
// grows to the largest system's need.  It takes the matrices of all levels at once up to 2 GB (the
// batch of panels is what fills the GPU); where that does not fit the free memory the batch is halved, down to none
// at all: the caller then runs matrix by matrix on work matrices of its own (on).
#pragma once
#include <algorithm>
#include <cstddef>

namespace xl {

struct EntropyWork {
  static constexpr int kPanel = 64;
  double *mats = nullptr, *rows = nullptr, *li = nullptr, *part = nullptr;
  int cap = 0;

  static size_t per(int np) { return (size_t)np * np + side(np); }   // doubles of one matrix and what goes with it
  static size_t side(int np) { return (size_t)np * kPanel + kPanel * kPanel + np / kPanel; }

  // The area for up to nmat matrices of size np: alloc(bytes) returns a pointer or null, release(p) gives one
  // back.  cap = 0 when nothing fits.
  template <class Alloc, class Release>
  void reserve(int np, int nmat, Alloc alloc, Release release) {
    const size_t one = per(np) * sizeof(double);
    int want = (int)std::max<size_t>(1, std::min<size_t>((size_t)nmat, kMost / one));
    if (one * want > bytes_) {
      if (buf_) release(buf_);
      buf_ = nullptr;
      bytes_ = 0;
      for (; want > 0 && !buf_; want = buf_ ? want : want / 2) buf_ = static_cast<double*>(alloc(one * want));
      if (buf_) bytes_ = one * want;
    }
    cap = want;
    if (!buf_) return;
    mats = buf_;
    rows = mats + (size_t)np * np * cap;
    li = rows + (size_t)np * kPanel * cap;
    part = li + (size_t)kPanel * kPanel * cap;
  }
  // One matrix at a time in a, the rest in b (np x np each, np a multiple of 128).
  static EntropyWork on(double* a, double* b, int np) {
    EntropyWork w;
    w.mats = a;
    w.rows = b;
    w.li = w.rows + (size_t)np * kPanel;
    w.part = w.li + (size_t)kPanel * kPanel;
    w.cap = 1;
    return w;
  }
  template <class Release>
  void free_all(Release release) {
    if (buf_) release(buf_);
    *this = EntropyWork();
  }

 private:
  static constexpr size_t kMost = (size_t)2 << 30;
  double* buf_ = nullptr;
  size_t bytes_ = 0;
};

}  // namespace xl
