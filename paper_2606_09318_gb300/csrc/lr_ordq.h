// lr_ordq.h -- the ordered queue that hands the positions of a ruler sequence
// to the threads of many CTAs (k_chase, levels in element order).
//
// CTAs draw positions from one global counter, kOrdChunk at a time, and hand
// them to their threads through a shared-memory window, (end << 32) | next.
// The lanes of a warp that ask together take theirs with one atomic.  The
// group that brings the window down to kOrdLow positions draws the next chunk,
// which waits in `next`; the first group that runs past the window's end and
// finds it there makes it the window.  A group that does not find it draws
// just what it lacks from the global counter.  Nobody waits.
//
// A group that was slow to look may find a chunk while a window is open.  It
// takes its share of that and puts the rest back, which may so shrink to fewer
// positions than the next such group lacks: its other threads ask again.
//
// The counter is one address, which serves an atomic in 0.65 ns at best, so
// how often it is asked can bound the chase.  With 32 positions a draw, fetched
// only when the window had run out, and single draws until they came, a batch
// of 7.5e7 unweighted elements took 1.51 ms, however many threads chased; now
// 1.37 ms, and 1.06 with half as many threads again.  A CTA that starts with
// one draw for all its threads saves 0.23 ms at any size, and once the
// sequence has run out, nobody asks.  What a group gets beyond the window goes
// round the warp in one word, and only where a group lacks something (1024
// weighted lists, 4.6e8 elements: 11.80 ms with a second shuffle for every
// request, 11.64 now).
//
// The memory operations come from the template argument, so that the host can
// run the queue under any interleaving of them.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define LR_ORDQ_FN __device__ __forceinline__
#else
#define LR_ORDQ_FN inline
#endif

namespace lr {

constexpr uint32_t kOrdChunk = 128, kOrdLow = kOrdChunk / 2;
static_assert(kOrdLow >= 32, "a chunk serves a warp and stays above the low mark");

LR_ORDQ_FN unsigned long long ord_window(uint32_t from, uint32_t to) {
  return ((unsigned long long)to << 32) | from;
}

// What a group of threads gets beyond the window's end, (limit << 32) | first:
// the positions from `first` on that are below `limit`.  A thread whose
// position would lie beyond a limit below the sequence's length asks again;
// the sequence's length or more: none left.  (A sequence has fewer than 2^31.)
constexpr uint32_t kOrdAgain = 0xFFFFFFFFu;

LR_ORDQ_FN uint32_t ord_window_has(unsigned long long w, uint32_t cnt) {
  const uint32_t next = (uint32_t)w, end = (uint32_t)(w >> 32);
  return next >= end ? 0u : end - next < cnt ? end - next : cnt;
}

// The position of the group's thread i: w is what the window was, `more` what
// the group got beyond it.
LR_ORDQ_FN uint32_t ord_position(unsigned long long w, uint32_t have, unsigned long long more, uint32_t total, uint32_t i) {
  if (i < have) return (uint32_t)w + i;
  const uint32_t p = (uint32_t)more + (i - have), limit = (uint32_t)(more >> 32);
  return p < limit || limit >= total ? p : kOrdAgain;
}

// The rest of a group's request, after it has added its cnt threads to the
// window, which was w.  M: exchange_window(w) on the CTA's window, window()
// reads it; exchange_next(w) on the chunk after it (0: not there); draw(c)
// adds to the global counter; out() and set_out(): the sequence has run out.
// *fresh: the first position of a chunk it drew.
template <class M>
LR_ORDQ_FN unsigned long long ord_ask(const M &q, unsigned long long w, uint32_t cnt, uint32_t total, uint32_t *fresh) {
  const uint32_t next = (uint32_t)w, end = (uint32_t)(w >> 32), lack = cnt - ord_window_has(w, cnt);
  unsigned long long more = ord_window(total, total);
  bool draw = next + kOrdLow < end && next + cnt + kOrdLow >= end;     // brings the window down to the mark
  if (lack) {
    const unsigned long long c = q.exchange_next(0ull);
    if (c) {
      const uint32_t from = (uint32_t)c, to = (uint32_t)(c >> 32), left = to - from;
      more = c;
      draw = left <= lack + kOrdLow;         // a short chunk starts below the mark
      if (left > lack) {
        // the window, unless another group has opened one since this one
        // asked: then it goes back (whoever holds the chunk is the only one
        // who could open a window)
        const unsigned long long now = q.window();
        const bool spent = (uint32_t)now >= (uint32_t)(now >> 32);
        if (spent) q.exchange_window(ord_window(from + lack, to));
        else q.exchange_next(ord_window(from + lack, to));
        draw = draw && spent;
      } else if (left < lack && to >= total) {        // the sequence's last chunk: the rest is past its end
        q.set_out();
        draw = false;
      }
    } else if (!q.out()) {
      const uint32_t j = q.draw(lack);
      more = ord_window(j, total);
      if (j >= total) q.set_out();
    }
  }
  if (draw && !q.out()) {
    const uint32_t j = q.draw(kOrdChunk);
    if (j >= total) {
      q.set_out();
    } else {
      *fresh = j;
      // the chunk is this CTA's whatever its length: every position of it must
      // be handed out, up to the end of the sequence
      q.exchange_next(ord_window(j, (uint64_t)j + kOrdChunk < total ? j + kOrdChunk : total));
    }
  }
  return more;
}

}  // namespace lr
