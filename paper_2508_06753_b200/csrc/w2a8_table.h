// Numbers that are looked up once per device.  Host code, no CUDA.
#pragma once

#include <mutex>

namespace w2a8 {

constexpr int kMaxDevices = 64;

// One row of N numbers per device ordinal.  The first caller for a device fills its row, callers beside it wait, and
// nobody reads a row that is still being written: launch plans follow from these numbers, and equal calls have to get
// equal plans from every thread.
template <int N>
class PerDeviceTable {
  public:
    // fill(row): writes the N numbers of device `dev`
    template <typename Fill>
    const int *get(int dev, Fill fill) {
        std::call_once(once_[dev], [&] { fill(rows_[dev]); });
        return rows_[dev];
    }

  private:
    std::once_flag once_[kMaxDevices];
    int rows_[kMaxDevices][N] = {};
};

}  // namespace w2a8
