// batchcost.cuh -- estimated time of one detector's forward path, for the order of a batch's branches
// (batch.cu).  Plain C++, so that a host test can hold it to the measured steps.
#pragma once

#include "../../include/sidelobe.h"

namespace sl {

// Milliseconds from the plan's recurrence steps and (kmax + 1) x samples: per step the contraction, per
// order and sample the sort and the interpolation, both as measured at LFI size (6.63e9 steps, 17 x 1e8;
// contraction 1.97, 8.2, 28.1 and 22.1 ms, the rest with the ring FFT 6.0, 6.2, 22.9 and 22.6).
inline double batch_cost_ms(int precision, double lsteps, double order_samples) {
    double step = 0.30e-9, sample = 3.5e-9;                         // SL_FP32
    if (precision == SL_TF32X3) step = 1.24e-9;
    if (precision == SL_FP64) step = 4.24e-9, sample = 13.4e-9;
    if (precision == SL_DF64) step = 3.33e-9, sample = 13.2e-9;
    return lsteps * step + order_samples * sample;
}

}  // namespace sl
