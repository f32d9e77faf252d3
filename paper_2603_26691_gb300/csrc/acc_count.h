// Word-capacity bookkeeping of the carry-save accumulator: how many digits launches can have added to any word since
// the carries were last propagated, and whether the next launch needs a propagation first.
//
// Each int64 word takes digits of magnitude < 2^32: 2^31 of them cannot overflow it; beside the sorted-step kernel's far
// commits (which stay within 2^60 and what is in flight, see there) 2^30 of them.
//
// The host keeps the count while it sees every launch.  A replay of a captured graph adds to the words without it, so
// from a handle's first captured launch on the count lives on the device, where a kernel before each launch decides.
// What the host had counted until then stays with it as the base and goes along with every later decision, until one
// of them has propagated the carries (or a reset has cleared the words): a captured launch may run late, several
// times or never, so it cannot be the one that hands the count over.
//
// Plain C++, so that the rule can be run without a GPU.
#pragma once

#ifdef __CUDACC__
#define ST_ACC_HD __host__ __device__
#else
#define ST_ACC_HD
#endif

namespace st {

constexpr double kAddLimit = 2147483648.0 - 1048576.0, kAddLimitFar = 1073741824.0;

// the device's side, in the handle's flags buffer (zero at first)
struct AccDeviceCount {
  unsigned long long adds;  // digits since the last propagation or reset there
  int propagate;            // the last decision
  int base_gone;            // nonzero once the host's base is no longer in the words
};

// before a launch that adds at most `add` digits to a word: whether to propagate first
ST_ACC_HD inline bool acc_decide(AccDeviceCount& d, double base, double add) {
  d.propagate = (double)d.adds + (d.base_gone ? 0.0 : base) + add > kAddLimitFar;
  if (d.propagate) {
    d.adds = 1;  // every word holds one digit
    d.base_gone = 1;
  }
  d.adds += (unsigned long long)add;
  return d.propagate != 0;
}
ST_ACC_HD inline void acc_cleared(AccDeviceCount& d) {
  d.adds = 0;
  d.base_gone = 1;
}

// the host's side
struct AccCount {
  double adds = 0.0;       // until on_device: digits since the last propagation; then the base of acc_decide
  bool far = false;        // the sorted-step kernel ran since then
  bool on_device = false;  // steps were captured in a graph

  enum Action { kNothing, kPropagate, kAskDevice };
  Action launch(double add, bool far_commits, bool capturing) {
    on_device = on_device || capturing;
    if (on_device) return kAskDevice;
    Action act = kNothing;
    if (adds + add > (far_commits || far ? kAddLimitFar : kAddLimit)) {
      act = kPropagate;
      adds = 1.0;
      far = false;
    }
    adds += add;
    far = far || far_commits;
    return act;
  }
  // the words are cleared or their carries propagated by what is queued (or captured) now: whether the device's side
  // has to hear of it (acc_cleared)
  bool cleared(bool capturing) {
    on_device = on_device || capturing;
    if (on_device) return true;
    adds = 0.0;
    far = false;
    return false;
  }
};

}  // namespace st
