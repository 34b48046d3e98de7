// Timeout flags of several kernel families fetched together.
#pragma once
#include <string>

namespace sg {

// The names of the families whose flag is set, joined; empty when none is.
// Every set flag is cleared (clear(k)), whichever is reported: once fetched,
// a flag is not fetched again before its family has run again, and one left
// set would then be taken for that run's.
template <typename Clear>
std::string collect_timeouts(const int* flags, const char* const* names, int count, Clear clear) {
  std::string who;
  for (int k = 0; k < count; ++k) {
    if (!flags[k]) continue;
    clear(k);
    who += (who.empty() ? "" : ", ") + std::string(names[k]);
  }
  return who;
}

}  // namespace sg
