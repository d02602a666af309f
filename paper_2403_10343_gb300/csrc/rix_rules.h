// Rules of the launches that need no CUDA (plain C++; not part of the ABI).
#pragma once

namespace rix {

// SMs of a GB300.  The rules that split work by it take this number and not the device's: some of
// them decide the order of a sum, and the same system gives the same bits wherever it runs.
constexpr int SMS = 152;

}  // namespace rix
