// The rule by which the fused preparation reads an archive list, for every entry below its total.
#include "ebic_internal.h"

extern "C" void list_entries(const uint32_t* offsets, uint32_t n, uint32_t total, uint32_t* member) {
  for (uint32_t t = 0; t < total; ++t) member[t] = ebic::entry_member(offsets, n, t);
}
