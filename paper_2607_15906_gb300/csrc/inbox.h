// What a block of a list chain (k_chain_list) may see of the others at a step.
//
// One barrier lies between two steps.  A block that passes it early works on
// step i while a slower one still reads what step i - 1 sent it, so a word that
// step i writes must not be one that step i reads.  Each inbox therefore has
// three words: the next free place, which only senders touch, and the numbers of
// entries sent in even and in odd steps.  Step i counts in the word of its own
// parity and its receivers read the other one: nobody writes that word before
// the next barrier, which the receiver joins after reading.  Places are handed
// out in order, so the entries of steps before i, all stored before the barrier,
// occupy the places below the sum of the two numbers as of step i - 1.
//
// The flag that gives the lists up holds the step that set it (the first one
// wins), and a step heeds a flag of an earlier step only, so that every block
// changes over at the same step.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define GOCP_HD __host__ __device__ __forceinline__
#else
#define GOCP_HD inline
#endif

namespace gocp {

// Words of a block's inbox record.
constexpr int kInboxNext = 0, kInboxSent = 1;   // kInboxSent + 0, 1: sent in even, odd steps

GOCP_HD int inbox_send_word(int step) { return kInboxSent + (step & 1); }
GOCP_HD int inbox_read_word(int step) { return kInboxSent + ((step + 1) & 1); }

// Entries in the inbox at a step: the word read there, the other word as read
// the step before, and the inbox's room.
GOCP_HD uint32_t inbox_length(uint32_t read, uint32_t before, uint32_t room) {
  const uint32_t n = read + before;
  return n < room ? n : room;
}

GOCP_HD uint32_t full_mark(int step) { return (uint32_t)step + 1u; }   // 0: not given up
GOCP_HD bool full_heeded(uint32_t mark, int step) { return mark != 0u && mark <= (uint32_t)step; }

}  // namespace gocp
