// Whether a launch comes straight behind another one of the same context: what a kernel may assume of its predecessor's
// shared memory and length.  A hint -- work that the caller puts between the two is not seen -- so no result may hang on it.
// (Plain C++.)
#pragma once
#include <stdint.h>

namespace kvd {

struct LaunchMark {
  uint64_t at = ~0ull;           // launches of the context, the marked one included
  const void *stream = nullptr;
  void set(uint64_t launches, const void *s) {
    at = launches;
    stream = s;
  }
  bool directly_before(uint64_t launches, const void *s) const { return at == launches && stream == s; }
};

}  // namespace kvd
