// Which cooperative grids of the process may run side by side (host code, no
// CUDA calls; CoopOrder in internal.h drives it).
//
// A grid with grid-wide barriers must become fully resident.  Grids that start
// together and need more SMs than there are could each hold some and wait for
// the rest forever, so a grid takes as many units of a budget of one unit per SM
// as it has blocks (all of them when it has more), and a unit passes from one
// grid to the next only behind the end of the first: the later grid's stream
// waits for the event recorded after the earlier one.  At any time the running
// grids hold different units, so while a block of theirs is not placed, some SM
// has none of their blocks; every other kernel runs to completion without
// waiting on blocks, so the block gets that SM.  (Every cooperative kernel's
// block fits an SM by itself.)  Waits point to grids launched before, so they
// form no cycle.
#pragma once
#include <algorithm>
#include <cstdint>
#include <vector>

namespace mslice {

class CoopBudget {
 public:
  static constexpr int FREE = -1;  // "event" of units that no grid holds

  explicit CoopBudget(int units) : units_(units > 0 ? units : 1) { segs_.push_back({FREE, units_, 0}); }

  int units() const { return units_; }

  // Takes min(blocks, units()) units for a grid launched on stream `owner`.
  // `wait` receives the events its stream has to wait for; returns the event to
  // record behind it.  Units come from grids of the same stream first (behind
  // them anyway), then from those that `done` (event) says have finished, then
  // from the oldest.
  template <class Done>
  int take(int blocks, uintptr_t owner, Done&& done, std::vector<int>& wait) {
    int need = std::max(1, std::min(blocks, units_));
    const int taken = need;
    wait.clear();
    for (size_t i = segs_.size(); i-- > 0 && need > 0;)
      if (segs_[i].event != FREE && segs_[i].owner == owner) need -= draw(segs_[i], need, wait);
    for (size_t i = 0; i < segs_.size() && need > 0; ++i) {
      Seg& s = segs_[i];
      if (s.units > 0 && s.event != FREE && done(s.event)) s.event = FREE;
      if (s.event == FREE) need -= draw(s, need, wait);
    }
    for (size_t i = 0; i < segs_.size() && need > 0; ++i) need -= draw(segs_[i], need, wait);
    segs_.erase(std::remove_if(segs_.begin(), segs_.end(), [](const Seg& s) { return s.units == 0; }), segs_.end());
    int event = 0;
    while (std::any_of(segs_.begin(), segs_.end(), [&](const Seg& s) { return s.event == event; })) ++event;
    segs_.push_back({event, taken, owner});
    return event;
  }

 private:
  struct Seg {
    int event;  // of the grid that held the units last
    int units;
    uintptr_t owner;
  };

  static int draw(Seg& s, int need, std::vector<int>& wait) {
    const int n = std::min(s.units, need);
    if (n > 0 && s.event != FREE && std::find(wait.begin(), wait.end(), s.event) == wait.end())
      wait.push_back(s.event);
    s.units -= n;
    return n;
  }

  int units_;
  std::vector<Seg> segs_;  // in launch order; their units sum to units_
};

}  // namespace mslice
