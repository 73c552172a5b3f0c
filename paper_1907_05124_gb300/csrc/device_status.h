// Status words that kernels leave for the host, and what callers are told.
#pragma once

#include "../../include/mars.h"

#include <cstdint>

namespace mars {

// Device-side status words (status[0]); MARS_OK when clean.
enum DeviceStatus : int32_t { kDevOk = 0, kDevBadIndex = 1, kDevTimeout = 2 };

// The status of an energy pass: only a spin that is not +-1 is the caller's fault.
inline int energy_status_rc(int32_t status)
{
    switch (status) {
    case kDevOk: return MARS_OK;
    case kDevBadIndex: return MARS_EINVAL;
    case kDevTimeout: return MARS_ETIMEOUT;
    default: return MARS_EDEVICE;
    }
}

}  // namespace mars
