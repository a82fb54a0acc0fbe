// step_records.h -- which forces steps of a context are recorded (host bookkeeping only, no CUDA).
//
// A step is known by a 64-bit key of everything its recording bakes in.  Its first run under a key is
// eager (buffers may grow, which changes the key), the second records, later ones replay.  Recording
// costs 14 to 42 us on top of an eager call and a replay saves about 150 us (GB300, 192 to 98,000 atoms),
// so it pays from the first replay on, and a loop that runs every system twice loses 2 % of its second
// calls.  The recordings of the kSlots keys used last are kept, so that a caller that alternates between
// a few systems or outputs replays each of them.  A key whose recording did not complete is not tried
// again while it is among them.
#pragma once
#include <cstdint>

namespace ctd {

// Exec: a pointer type; Drop: a functor that releases one.
template <class Exec, class Drop>
class StepRecords {
 public:
  static constexpr int kSlots = 4;
  enum class Act { kEager, kRecord, kReplay };

  StepRecords() = default;
  StepRecords(const StepRecords&) = delete;
  StepRecords& operator=(const StepRecords&) = delete;
  ~StepRecords() { clear(); }

  // What to do with a step of this key (never 0).
  Act next(uint64_t key) const {
    const Slot* s = find(key);
    return !s || s->refused ? Act::kEager : s->exec ? Act::kReplay : Act::kRecord;
  }
  // The recording to replay; it becomes the one used last.
  Exec replay(uint64_t key) {
    Slot* s = take(key);
    return s->exec;
  }
  // A step of this key has run eagerly and grew nothing under it.
  void ran(uint64_t key) { take(key); }
  void recorded(uint64_t key, Exec exec) {
    Slot* s = take(key);
    if (s->exec) Drop()(s->exec);
    s->exec = exec;
  }
  void refused(uint64_t key) { take(key)->refused = true; }
  void clear() {
    for (Slot& s : slots_) release(s);
  }

 private:
  struct Slot {
    uint64_t key = 0, used = 0;
    bool refused = false;
    Exec exec = nullptr;
  };
  const Slot* find(uint64_t key) const {
    for (const Slot& s : slots_)
      if (s.key == key) return &s;
    return nullptr;
  }
  // The slot of this key, the one used longest ago made over to it if there is none.
  Slot* take(uint64_t key) {
    Slot* s = const_cast<Slot*>(find(key));
    if (!s) {
      s = &slots_[0];
      for (Slot& o : slots_)
        if (o.used < s->used) s = &o;
      release(*s);
      s->key = key;
    }
    s->used = ++clock_;
    return s;
  }
  static void release(Slot& s) {
    if (s.exec) Drop()(s.exec);
    s = Slot();
  }
  Slot slots_[kSlots];
  uint64_t clock_ = 0;
};

}  // namespace ctd
