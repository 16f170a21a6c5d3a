// Host side of the resident solver's plan (cg_resident.cu): what the context knows about
// the plan in its buffer.  Plain C++, so that it can be checked without a GPU.
#pragma once

#include <cstddef>

namespace qp {

struct ResidentPlan {
  int chunk = 0;  // contacts a block of the plan in the buffer (0: none)

  // Room for a plan of `bytes` for blocks of `want` contacts.  A buffer that grows loses
  // its contents, and one that cannot grow is gone when ensure() throws, so the plan is
  // disowned before either can happen.
  template <class B>
  void* room(B& buf, size_t bytes, int want) {
    if (chunk != want || bytes > buf.cap) chunk = 0;
    return buf.ensure(bytes);
  }
};

}  // namespace qp
