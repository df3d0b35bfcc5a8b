// Rules by which a call's work is laid out that need no device: plain C++, so
// that the CPU tests compile and check them as they are.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <vector>

namespace gpss {

// What the choice between parallel and serial gradient segments looks at.
struct SegmentCase {
  bool product;   // product kernel: forward-mode tangents, no segments
  int comb_prec;  // arithmetic of the cross-chunk combination: 32 or 64
  int D, NP;      // state dimension and its packed covariance
  int max_chunk;  // events of the longest chunk
  int ck;         // events per segment
  int n_vch;      // chunks of the call (all parameter sets)
  int64_t steps;  // lane-steps of their warps: 32 x each warp's longest chunk
  int n_sm;       // multiprocessors
};

// Bytes of the replay buffers of n_seg segments per chunk.
inline size_t replay_bytes(int ck, int D, int NP, int n_vch, int n_seg) {
  return (size_t)n_seg * ck * (4 * ((D + NP + 3) / 4)) * n_vch * sizeof(float);
}

// Segments of ck events per chunk that the gradient walks in parallel, one
// thread each (1: one thread per chunk walks them in turn).  A thread takes
// the serial time of its events, so too few chunks leave the GPU idle;
// parallel segments cost each segment's own element beside the chunk's and a
// boundary adjoint per segment.  The line lies where both take the same time,
// which for chunks of one length is 1000 to 1100 warps of them on 152 SMs: two
// SHO terms 912 warps 1132 us against 1233, 1064 warps 1311 against 1253; SHO +
// Matern-3/2 on instants 912 warps 942 against 1094, 1216 warps 1263 against
// 1153, 1824 warps 1787 against 1361; SHO alone 912 warps 541 against 597, 1216
// warps 683 against 637.  Where lengths differ the work counts, not the warps:
// with as many steps as 836 (1043) warps of the longest chunk have, 1306 (1616)
// warps of instants took 995 us against 1145 (1195 against 1214), SHO alone 561
// against 617 (639 against 659).  So: up to 6 warps of chunks per SM, or for
// states of at most 4 up to 12 that have no more steps than 7 of the longest.
// The adjoint at a segment's end differs from the walked one in rounding, which
// shows in differences of nearly equal terms: with parallel segments, 1600
// exposures of one SHO term, the exposure gradient's error against FP64 is 5.7e-6
// of its largest instead of 3.9e-6 and a predicted variance's 1.0e-4 instead of
// 6.1e-5.  Exposure gradients and predictions keep the walk in turn.  The
// segments' elements and the information carried back through them are FP32: a
// model whose combination runs in FP64 starts the walk in turn from the FP64
// adjoint at the chunk's end and keeps it.
inline int grad_segments(const SegmentCase &c) {
  constexpr int kMaxSegments = 1024;  // k_seg_info carries the adjoints back through them in turn
  constexpr size_t kMaxReplay = (size_t)2 << 30;  // bytes of the replay buffers
  // shorter segments would put a boundary adjoint's rounding every few events
  if (c.product || c.comb_prec != 32 || c.ck < 32) return 1;
  // and a second segment of less than half the events gives too little: 608 warps
  // of chunks of 34 events 282 us against 256 in turn, of 40 290 against 275, of
  // 48 302 against 301, of 64 323 against 353 (two SHO terms)
  if (2 * c.max_chunk < 3 * c.ck) return 1;
  const int n_seg = (c.max_chunk + c.ck - 1) / c.ck;
  const int per_sm = c.D <= 4 ? 12 : 6;
  if (c.n_vch / 32 > per_sm * c.n_sm || n_seg < 2 || n_seg > kMaxSegments) return 1;
  if (c.steps > (int64_t)32 * c.max_chunk * 7 * c.n_sm) return 1;
  return replay_bytes(c.ck, c.D, c.NP, c.n_vch, n_seg) <= kMaxReplay ? n_seg : 1;
}

// Whether a product model's step scalars are formed for all steps at once
// rather than by the chunks' threads.  For a gradient always: every
// parameter's thread reads them (150 series of 500 to 5000 instants 1633 ->
// 601 us; one of 100: 92 -> 86 us).  The log-likelihood alone reads each once:
// they shorten a chunk's serial chain but cost a pass over memory and two
// launches, so they are formed where chunks are long and warps of chunks too
// few to hide the chain.  Product alone (two oscillators), at once against
// step by step, 152 SMs: 30 warps, chunks of 32 events 72 us against 77, of 64
// 91 against 116; 304 warps, 64 events 108 against 116; 608 warps, 64 events
// 128 against 120, 250 events 435 against 397.  With a plain term (three): 30
// warps, 8 events 74 against 75, 32 events 95 against 140; 608 warps, 32 events
// 130 against 159; 912 warps 32 events 153 against 163, 128 events 464 against
// 454.  Rows with an overdamped factor, whose elements form their own, pay 7 to
// 10 us for the launches that skip them, which is why the shorter chunks
// with a small gain are left out (64 and 32 events: 2 to 7 % of such a call).
inline bool prod_scalars_at_once(bool grad, bool plain_term, int max_chunk, int n_vch, int n_sm) {
  if (grad) return true;
  return max_chunk >= (plain_term ? 32 : 64) && n_vch / 32 <= (plain_term ? 4 : 2) * n_sm;
}

// First series of each group in which a re-sent event stream goes up, and the
// number of series at the end.  A group's element pass takes at least its
// longest chunk's serial time however few chunks it has, so groups hold
// block_chunks chunks (one block of them per multiprocessor) on average, there
// are at most four, and a cut is made only where the group it closes and the
// rest each hold half of that.  Groups are cut at series by events, the
// copies' share: few long series among many short ones hold most of the events
// and few of the chunks.  90112 chunks of two terms: element phase with the
// upload 1.84 ms with four groups, 1.90 ms with two; 11424 chunks: the whole
// call 1.75 ms with four, 1.17 ms with one.  Parameter sets do not count as
// chunks: with 2 to 70 sets, calls of 1152 to 24000 chunks took 2 to 24 % longer
// in the groups that chunks times sets would give (3200 chunks, 16 sets: 0.90
// ms with one group, 1.03 with two; 2560 chunks, 64 sets: 5.0 ms, 5.5 with four).
inline std::vector<int> upload_groups(const int64_t *ev_off, const int32_t *ch_first,
                                      int n_series, int64_t block_chunks) {
  const int64_t n_chunks = ch_first[n_series], least = block_chunks / 2;
  const int64_t n_groups =
      std::max<int64_t>(1, std::min<int64_t>(4, n_chunks / std::max<int64_t>(1, block_chunks)));
  std::vector<int> cut{0};
  for (int64_t g = 1; g < n_groups; ++g) {
    const int64_t target = ev_off[n_series] * g / n_groups;
    const int sp = (int)(std::lower_bound(ev_off, ev_off + n_series + 1, target) - ev_off);
    if (sp > cut.back() && sp < n_series && ch_first[sp] - ch_first[cut.back()] >= least &&
        n_chunks - ch_first[sp] >= least)
      cut.push_back(sp);
  }
  cut.push_back(n_series);
  return cut;
}

// Scratch buffers of one call: *p receives the address.
struct Buffer {
  void **p;
  size_t bytes;
};

inline size_t total_bytes(const std::vector<Buffer> &list) {
  size_t n = 0;
  for (const Buffer &b : list) n += b.bytes;
  return n;
}

// Takes every buffer of the list; when one cannot be had, gives back those
// before it and leaves all null.  take(p, bytes) says whether it succeeded,
// give() returns the buffer taken last.
template <class Take, class Give>
bool take_all(const std::vector<Buffer> &list, Take take, Give give) {
  for (size_t i = 0; i < list.size(); ++i) {
    if (take(list[i].p, std::max<size_t>(list[i].bytes, 16))) continue;
    for (; i > 0; --i) give();
    for (const Buffer &b : list) *b.p = nullptr;
    return false;
  }
  return true;
}

enum class Scratch { none, plain, fast };

// A call's scratch in two steps, so that the second step's allocations run
// behind the first kernels.  First what these need, then what they need for
// the fast way, all or none.
template <class Take, class Give>
Scratch take_first(const std::vector<Buffer> &first, const std::vector<Buffer> &fast, Take take,
                   Give give) {
  if (!take_all(first, take, give)) return Scratch::none;
  return !fast.empty() && take_all(fast, take, give) ? Scratch::fast : Scratch::plain;
}

// Then the rest of either way.  Where the fast way's cannot be had, its buffers
// of the first step are given back for the plain one's: a call is refused only
// where the plain way does not fit.
template <class Take, class Give>
Scratch take_rest(Scratch way, const std::vector<Buffer> &fast,
                  const std::vector<Buffer> &rest_fast, const std::vector<Buffer> &rest_plain,
                  Take take, Give give) {
  if (way == Scratch::fast) {
    if (take_all(rest_fast, take, give)) return Scratch::fast;
    for (const Buffer &b : fast) {
      give();
      *b.p = nullptr;
    }
  }
  return take_all(rest_plain, take, give) ? Scratch::plain : Scratch::none;
}

}  // namespace gpss
