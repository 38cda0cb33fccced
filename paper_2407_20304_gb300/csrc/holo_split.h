// Pass B's split last round: the integer rules shared by the host, the column pass and the kernel
// that combines its partial sums.  Plain C++, so that they can be compiled and checked without CUDA.
//
// The column groups of pass B go to `nblk` persistent blocks in whole rounds.  The groups left over
// form a list of titems = (groups left) x per (group, plane) items, `per` planes to a group, and block
// b takes the items [split_begin(b), split_begin(b + 1)): even shares, in order, so a group belongs to
// a run of consecutive blocks.

#pragma once

#if defined(__CUDACC__)
#define HOLO_SPLIT_FN __host__ __device__ __forceinline__
#else
#define HOLO_SPLIT_FN inline
#endif

namespace holo {

// Blocks of a split of `items` (group, plane) items, full: the resident blocks of the chip.  Never
// more blocks than items; one item to a block up to two blocks per SM, where a second plane is pure
// latency (258^2 on 512^2, 2 x 4 planes, 264 items, pass B and combine kernel: 264 blocks 25.6 us,
// 152 blocks 39.5 us); at least two items from there on, which halves the prologues and the sums to
// combine (128^2, 8 x 4 planes, 512 items: 256 blocks 22.2 us, 512 blocks 23.7 us).
HOLO_SPLIT_FN int split_blocks(int full, int sms, long long items) {
  long long b = items / 2 > 2 * sms ? items / 2 : 2 * sms;
  if (b > items) b = items;
  if (b > full) b = full;
  return (int)(b < 1 ? 1 : b);
}

// The form of pass B's last round: 0 whole groups, 1 split without the Y stage, 2 split with it.
// sched: what the user asked for (-1 automatic).  With full rounds only there is nothing to split,
// whatever was asked for, and the stage stays.
HOLO_SPLIT_FN int split_form(int sched, int groups, int full) {
  if (groups % full == 0) return 0;
  if (sched >= 0) return sched;
  return groups / full < 3 ? 2 : 0;
}

// First item of block b.
HOLO_SPLIT_FN long long split_begin(long long titems, int nblk, int b) { return titems * b / nblk; }

// The block that item i belongs to.
HOLO_SPLIT_FN int split_owner(long long titems, int nblk, long long i) {
  return (int)(((i + 1) * nblk - 1) / titems);
}

// The blocks first .. last that hold items of group tg (counted among the groups left over).  A block
// writes the partial sum of the s-th group that its share meets to its slot s: `slot` for the first
// block, whose share may begin in an earlier group, 0 for the others.  With fewer items than blocks
// some blocks in the run hold none.
struct SplitRun {
  int first, last, slot;
};
HOLO_SPLIT_FN SplitRun split_run(long long titems, int nblk, long long per, int tg) {
  SplitRun r;
  r.first = split_owner(titems, nblk, tg * per);
  r.last = split_owner(titems, nblk, (tg + 1) * per - 1);
  r.slot = tg - (int)(split_begin(titems, nblk, r.first) / per);
  return r;
}

// Slots per block: the most groups that one share can meet.
HOLO_SPLIT_FN int split_slots(long long titems, int nblk, long long per) {
  const long long range = (titems + nblk - 1) / nblk;
  return titems > 0 ? (int)((range + per - 1) / per + 1) : 0;
}

}  // namespace holo
