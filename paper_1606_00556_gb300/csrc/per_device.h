// A whole number found out once per device of the process (launch limits and
// the like: another device of the same process has its own, and function
// attributes set while one device is current do not hold on another).
#pragma once
#include <atomic>

namespace bo {

class PerDevice {
 public:
  static constexpr int kMax = 64;  // devices beyond it are asked every time
  // find() >= 0 runs with `device` current
  template <typename F>
  int get(int device, F find) {
    if (device < 0 || device >= kMax) return find();
    int v = v_[device].load();
    if (v == 0) v_[device].store(v = find() + 1);
    return v - 1;
  }

 private:
  std::atomic<int> v_[kMax] = {};  // the number plus one, 0: not known yet
};

}  // namespace bo
