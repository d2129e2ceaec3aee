// Row bins side by side: three streams beside the caller's, forked from it and
// joined to it, and who owns them.  The runtime calls come through R (Stream,
// Event, Capture and static functions that return whether the call succeeded),
// so that the ordering can be checked on the host without a GPU.
#pragma once
#include <cstdint>
#include <new>

namespace hs {

constexpr int FAN_SIDES = 3;

// Side streams of one device at one priority, with the events that order them.
template <class R> struct SideSet {
  typename R::Stream s[FAN_SIDES]{};
  typename R::Event fork{}, join[FAN_SIDES]{};
  int device = -1, priority = 0;
  bool ok = false;
  SideSet() = default;
  SideSet(const SideSet &) = delete;
  SideSet &operator=(const SideSet &) = delete;
  ~SideSet() {
    for (int i = 0; i < FAN_SIDES; ++i) {
      if (s[i]) R::destroy(s[i]);
      if (join[i]) R::destroy(join[i]);
    }
    if (fork) R::destroy(fork);
  }
  // on the current device, at the priority of `like`
  bool make(typename R::Stream like) {
    ok = R::device(&device) && R::priority(like, &priority) && R::create(&fork);
    for (int i = 0; i < FAN_SIDES; ++i) ok = ok && R::create(&s[i], priority) && R::create(&join[i]);
    return ok;
  }
  // Streams of another device, at another priority than the caller's, or that
  // belong to a capture in which the caller's does not take part (a stream
  // stays in a capture from its first fork until the capture ends) would
  // change what the caller's stream means: its work then stays on it.
  bool serves(typename R::Stream main) const {
    int d = -1, p = 0;
    typename R::Capture mine{}, side{};
    if (!ok || !R::device(&d) || d != device || !R::priority(main, &p) || p != priority || !R::capture(main, &mine))
      return false;
    for (int i = 0; i < FAN_SIDES; ++i)
      if (!R::capture(s[i], &side) || (side.active && !(mine.active && side.id == mine.id))) return false;
    return true;
  }
};

// Sets for calls that own none (single products), a few per host thread: one
// for each of the caller's streams, so that work of two streams is not queued
// behind each other; with more streams than sets the one used longest ago is
// taken over, which costs its two streams their independence and nothing else.
// A set from here serves the stream it was asked for: device and priority are
// looked at, and a call that waits for the GPU takes part in no capture.
template <class R> struct SidePool {
  static constexpr int MOST = 8;
  struct Entry {
    SideSet<R> set;
    typename R::Stream owner{};
    uint64_t used = 0;
  };
  Entry *e[MOST] = {nullptr};
  uint64_t clock = 0;
  ~SidePool() {
    for (Entry *x : e) delete x;
  }
  SideSet<R> *of(typename R::Stream main) {
    int d = -1, p = 0;
    if (!R::device(&d) || !R::priority(main, &p)) return nullptr;
    int at = -1;  // main's entry, else an empty place, else the oldest entry of this device and priority
    for (int i = 0; i < MOST; ++i) {
      if (!e[i]) {
        if (at < 0 || e[at]) at = i;
        continue;
      }
      if (e[i]->set.device != d || e[i]->set.priority != p) continue;
      if (e[i]->owner == main) {
        at = i;
        break;
      }
      if (at < 0 || (e[at] && e[i]->used < e[at]->used)) at = i;
    }
    if (at < 0) return nullptr;  // all of other devices or priorities
    if (!e[at]) {
      e[at] = new (std::nothrow) Entry();
      if (!e[at]) return nullptr;
      if (!e[at]->set.make(main)) {  // (the caller's stream serves alone; asked again next time)
        delete e[at];
        e[at] = nullptr;
        return nullptr;
      }
    }
    e[at]->owner = main;
    e[at]->used = ++clock;
    return &e[at]->set;
  }
};

// One pass: stream(g) is where group g's kernels go (group 0: the caller's
// stream).  All of it starts after what the caller's stream holds, and after
// join() the caller's stream goes on after all of it.
template <class R> struct FanOf {
  using Stream = typename R::Stream;
  Stream main;
  SideSet<R> *d = nullptr;
  bool used[FAN_SIDES] = {false};
  // groups: bit g set when group g has work; with one group nothing is forked.
  // serves: known to hold for the set.
  FanOf(Stream st, unsigned groups, SideSet<R> *set, bool serves = false) : main(st) {
    if ((groups & (groups - 1)) == 0 || !set || !(serves || set->serves(main))) return;
    if (R::record(set->fork, main)) d = set;
  }
  FanOf(const FanOf &) = delete;
  FanOf &operator=(const FanOf &) = delete;
  Stream stream(int group) {
    if (!d || group == 0) return main;
    const int i = group - 1;
    if (!used[i]) {
      if (!R::wait(d->s[i], d->fork)) return main;  // not ordered behind the caller's stream: not used
      used[i] = true;
    }
    return d->s[i];
  }
  bool join() {
    bool done = true;
    for (int i = 0; i < FAN_SIDES; ++i) {
      if (!used[i]) continue;
      used[i] = false;
      if (R::record(d->join[i], d->s[i]) && R::wait(main, d->join[i])) continue;
      done = false;
      // the side stream's work must end before the caller's buffers are touched again
      typename R::Capture side{};
      if (R::capture(d->s[i], &side) && !side.active) R::synchronize(d->s[i]);
    }
    return done;
  }
  ~FanOf() { join(); }
};

}  // namespace hs
