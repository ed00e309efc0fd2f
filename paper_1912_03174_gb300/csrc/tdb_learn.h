// What the shift network's API and its kernels share.
#pragma once

#include <cuda_runtime.h>

namespace tdb {
namespace learn {

// Adam's bias corrections (1 - beta1^t, 1 - beta2^t) of the steps of one epoch launch.
constexpr int kEpochSteps = 256;
struct Corrections {
    float2 c[kEpochSteps];
};

}  // namespace learn
}  // namespace tdb
