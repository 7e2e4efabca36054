// The captured runs that are kept for the last few configurations, in plain C++
// so that the bookkeeping can be checked on the host.  An executable graph
// belongs to the context it was made in: after cudaDeviceReset the device has a
// new context and the handles of the old one are dropped, not destroyed (they
// died with their context).
#pragma once

namespace wmc {

template <class Key, class Exec, int N>
struct GraphSlots {
  struct Slot {
    bool valid = false;
    unsigned long long last_use = 0, ctx = 0;
    int device = 0;
    Key key{};
    Exec exec{};
  };
  Slot slot[N];
  unsigned long long uses = 0;

  // The slot made on this device and in its present context whose key matches,
  // or null.
  template <class Match>
  Slot* find(int device, unsigned long long ctx, Match match) {
    Slot* hit = nullptr;
    for (Slot& s : slot) {
      if (!s.valid || s.device != device) continue;
      if (s.ctx != ctx) s = Slot();
      else if (!hit && match(s.key)) hit = &s;
    }
    if (hit) hit->last_use = ++uses;
    return hit;
  }

  // An empty slot, the least recently used one emptied if there is none.
  template <class Destroy>
  Slot& take(Destroy destroy) {
    Slot* best = &slot[0];
    for (Slot& s : slot)
      if (!s.valid ? best->valid : best->valid && s.last_use < best->last_use) best = &s;
    if (best->valid) destroy(best->exec);
    *best = Slot();
    return *best;
  }

  Slot* fill(Slot& s, const Key& key, Exec exec, int device, unsigned long long ctx) {
    s.valid = true;
    s.last_use = ++uses;
    s.ctx = ctx;
    s.device = device;
    s.key = key;
    s.exec = exec;
    return &s;
  }
};

}  // namespace wmc
