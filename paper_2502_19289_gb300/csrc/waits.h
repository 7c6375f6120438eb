// waits.h -- which bounded wait ran out: the kernels' codes and their names.
#pragma once

namespace ctebd {

enum { kWaitNone = 0, kWaitTensor = 1, kWaitSplit = 2, kWaitAmplitude = 3 };

inline const char* wait_name(int code) {
  switch (code) {
    case kWaitNone: return "no wait";
    case kWaitTensor: return "a tensor-core completion wait";
    case kWaitSplit: return "an exchange of the direct split";
    case kWaitAmplitude: return "an exchange of the amplitude";
  }
  return "a wait of unknown kind";
}

}  // namespace ctebd
