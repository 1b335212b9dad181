// The step protocol of a list chain's inboxes (csrc/inbox.h), run with the
// blocks interleaved in every order that the barrier allows: seeded schedules
// that favour one block for a while, so that fast senders meet slow receivers.
//
//   inbox_model <rule> <runs>     rule 0: csrc/inbox.h; 1: one length word and a
//                                 flag without its step (what goes wrong then)
//
// A block at step i reads its inbox, then sends; each send takes a place, raises
// the count, stores the entry (or gives up where there is no room), with other
// blocks in between.  Entries carry their step.  Prints the number of faults:
// an entry of the same step seen, one missing, a place read before it was
// written, or blocks that disagree on the step from which the lists are given
// up.
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "inbox.h"

using namespace gocp;

int main(int argc, char** argv) {
  const int rule = std::atoi(argv[1]), runs = std::atoi(argv[2]);
  long faults = 0;
  for (int run = 0; run < runs; ++run) {
    std::mt19937 rng(run);
    const int G = 2 + (int)(rng() % 4), steps = 3 + (int)(rng() % 6);
    const uint32_t room = run % 2 ? 4u : 64u;
    struct Box {
      uint32_t w[3] = {0, 0, 0};
      std::vector<int> entry;
    };
    std::vector<Box> box(G);
    for (Box& b : box) b.entry.assign(room, -1);
    uint32_t flag = 0, arrived = 0;
    std::vector<std::vector<int>> sent(G, std::vector<int>(steps + 1, 0));   // [block][step]: sends to it before the step
    struct Block {
      int step = 0, op = 0, left = 0, to = 0;
      uint32_t seen[2] = {0, 0}, pos = 0;
      int full_from = -1;
    };
    std::vector<Block> blk(G);
    auto advance = [&](int r) -> bool {   // one operation of block r; false: it waits, or is done
      Block& b = blk[r];
      if (b.step == steps) return false;
      const int i = b.step;
      switch (b.op) {
        case 0: {   // the barrier, then the inbox
          if (arrived < (uint32_t)(i * G)) return false;
          if (i > 0) {
            uint32_t got;
            bool over;
            if (rule == 0) {
              const uint32_t v = box[r].w[inbox_read_word(i)];
              got = inbox_length(v, b.seen[i & 1], room);
              b.seen[(i + 1) & 1] = v;
              over = full_heeded(flag, i);
            } else {
              got = box[r].w[0] < room ? box[r].w[0] : room;
              over = flag != 0;
            }
            if (over && b.full_from < 0) b.full_from = i;
            const int want = sent[r][i] < (int)room ? sent[r][i] : (int)room;
            if ((int)got != want) ++faults;
            for (uint32_t q = 0; q < got; ++q) faults += box[r].entry[q] < 0 || box[r].entry[q] >= i;
          }
          b.left = (int)(rng() % 4);
          b.op = b.left ? 1 : 5;
          return true;
        }
        case 1:   // a place
          b.to = (int)(rng() % G);
          b.pos = box[b.to].w[kInboxNext]++;
          for (int s = i + 1; s <= steps; ++s) ++sent[b.to][s];
          b.op = 2;
          return true;
        case 2:   // the count
          if (rule == 0) ++box[b.to].w[inbox_send_word(i)];
          b.op = 3;
          return true;
        case 3:   // the entry, or no room
          if (b.pos < room) box[b.to].entry[b.pos] = i;
          else if (rule == 0) { if (!flag) flag = full_mark(i); }
          else flag = 1;
          b.op = --b.left ? 1 : 5;
          return true;
        default:   // arrive
          ++arrived;
          ++b.step;
          b.op = 0;
          return true;
      }
    };
    int fav = 0;
    for (;;) {
      if (rng() % 7 == 0) fav = (int)(rng() % G);
      bool moved = advance(fav);
      for (int k = 1; k < G && !moved; ++k) moved = advance((fav + k) % G);
      if (!moved) break;
    }
    for (const Block& b : blk) faults += b.step != steps;
    int from = -1;   // blocks that reached a step at or after the change must agree on it
    for (const Block& b : blk) if (b.full_from >= 0) from = from < 0 ? b.full_from : (b.full_from < from ? b.full_from : from);
    for (const Block& b : blk) faults += from >= 0 && b.full_from != from;
  }
  std::printf("%ld\n", faults);
  return 0;
}
