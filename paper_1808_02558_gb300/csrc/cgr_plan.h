// Host side of the resident solver's plan (cg_resident.cu): the room of a block's lists,
// and what the context knows about the plan in its buffer.  Plain C++, so that it can be
// checked without a GPU.
#pragma once

#include <algorithm>
#include <cstddef>

namespace qp {

constexpr int CR_WR = 9;        // stride of a contact's wrench in shared memory
constexpr int CR_WL = 7;        // stride of a body's intermediate (odd: no bank conflicts)
constexpr int CR_CHUNK1 = 512;  // contacts a block with one a thread
constexpr int CR_CHUNK2 = 1280; // with two (FP32)

// What a block of `chunk` contacts has room for.
struct ResidentShape {
  int chunk;
  int own_rb;  // remote partials have shared memory of their own
  int nbcap;   // bodies
  int rcap;    // remote partials, and shared runs
  bool full;   // no more bodies than that, with all the room

  // Dynamic shared memory; two: with two contacts a thread p lies behind the lists.
  size_t smem() const {
    return (size_t)chunk * (CR_WR * 8 + 8 + (chunk > CR_CHUNK1 ? 3 * 4 : 0)) + (size_t)nbcap * ((CR_WL + 2) * 8 + 12) +
           (size_t)rcap * (8 + (own_rb ? CR_WL * 8 : 0)) + 16;
  }
};

// The shape for a block with `room` bytes of dynamic shared memory.  A contact touches two
// bodies at most, so 2 chunk bodies always suffice.  Above 512 contacts a block shared
// memory is short and what it leaves is L1: piles, with about half a body a contact (654
// at 1262 on the 40^3 pile), get 800 bodies, and contact sets that do not fit these, such
// as a walled box of falling spheres with about one body a contact, `all` the room (1175
// at 1262).  Given all of it, piles of 35^3 to 39^3 take 4 % longer (550 -> 575 us a solve
// at 35^3); the box of 55^3 takes 635 us resident and 1270 in the global kernel.
// rcap is even: 32-bit data follows two 16-bit lists of that length in shared memory.
inline ResidentShape resident_shape(int chunk, size_t room, bool all) {
  ResidentShape s{chunk, chunk <= CR_CHUNK1 ? 1 : 0, 0, 0, true};
  s.rcap = s.own_rb ? std::min(std::max(256, 2 * chunk), 1024) : (chunk * CR_WR / CR_WL) & ~1;
  const size_t rest = s.smem();
  s.nbcap = room > rest ? (int)std::min<size_t>(2 * (size_t)chunk, (room - rest) / ((CR_WL + 2) * 8 + 12)) : 0;
  if (!all && chunk > CR_CHUNK1 && s.nbcap > 800) {
    s.nbcap = 800;
    s.full = false;
  }
  return s;
}

struct ResidentPlan {
  enum Room { USUAL, ALL, NONE };  // resident_shape with the usual room, with all of it, not resident
  int chunk = 0;                   // contacts a block of the plan in the buffer (0: none)
  Room tried[2] = {USUAL, USUAL};  // what FP64 and mixed solves are left with

  // A new contact set: no plan, and the room that the last one took (the next is much
  // like it), so that a step that reassembles pays for a refusal once at most.
  void assembled() {
    chunk = 0;
    for (Room& t : tried) t = std::min(t, ALL);
  }
  // The plan found no room in that shape: the next solves of the contact set do not ask again.
  void refused(bool mixed, bool full) {
    chunk = 0;
    tried[mixed] = full ? NONE : ALL;
  }

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
