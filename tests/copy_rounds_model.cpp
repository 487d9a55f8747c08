// Every interleaving of a copy CTA's two producer warps over a few rounds, with
// stage waits that give up anywhere: do both always leave at the same round,
// and does each read the chunks published for its round?  Exits 1 (and says
// why) where they do not.  Built with -DPRIVATE_BASE the producers keep the
// round's chunk to themselves and a wait that gives up does not advance it.
#include <cstdio>
#include <cstring>
#include <set>
#include <string>

#include "copy_rounds.h"

static const unsigned MAX_ROUNDS = 8;
enum Pc : unsigned char { PUBLISH, AT_BARRIER, AFTER, STAGE_WAIT, LEFT };

struct Producer {
  Pc pc;
  unsigned r, base;
};
struct State {
  ro::CopyRounds rounds;
  Producer p[2];
  unsigned next, gave_up;
  unsigned published[MAX_ROUNDS + 2];   // each round's first chunk, as it was published
};

static unsigned n_chunks;
static std::set<std::string> seen;
static const char* wrong;

static void visit(const State& s) {
  if (wrong) return;
  if (!seen.insert(std::string((const char*)&s, sizeof s)).second) return;
  for (int i = 0; i < 2; ++i)
    if (s.p[i].pc == LEFT && s.p[1 - i].pc == AT_BARRIER) wrong = "one producer left, the other waits at the barrier";
  if (s.p[0].pc == LEFT && s.p[1].pc == LEFT && s.p[0].r != s.p[1].r) wrong = "left at different rounds";
  if (wrong) return;
  if (!s.gave_up) {   // a consumer's wait
    State t = s;
    t.gave_up = 1;
    visit(t);
  }
  if (s.p[0].pc == AT_BARRIER && s.p[1].pc == AT_BARRIER) {
    State t = s;
    t.p[0].pc = t.p[1].pc = AFTER;
    visit(t);
    return;
  }
  for (int i = 0; i < 2; ++i) {
    State t = s;
    Producer& p = t.p[i];
    switch (s.p[i].pc) {
      case PUBLISH:
        if (i == 0) {
          t.rounds.publish(p.r, t.next, t.gave_up);
          t.published[p.r + 1] = t.next;
        }
        p.pc = AT_BARRIER;
        if (i == 0 && t.next < n_chunks) {   // the next claim: right behind this one, or past what other CTAs took
          const unsigned step[3] = {2, 4, n_chunks};
          for (unsigned k : step) {
            State v = t;
            v.next += k;
            visit(v);
          }
        } else {
          visit(t);
        }
        break;
      case AFTER: {
#ifdef PRIVATE_BASE
        const bool leave = p.base >= n_chunks || t.rounds.stop[p.r & 1u];
#else
        const bool leave = t.rounds.leave(p.r, n_chunks);
        if (t.rounds.chunk(p.r) != t.published[p.r]) wrong = "read another round's chunks";
#endif
        if (!leave && t.rounds.chunk(p.r + 1) != t.published[p.r + 1]) wrong = "read another round's chunks";
        p.pc = leave ? LEFT : STAGE_WAIT;
        visit(t);
        break;
      }
      case STAGE_WAIT:
        for (int ok = 0; ok < 2; ++ok) {
          State v = t;
          if (!ok) v.gave_up = 1;
#ifdef PRIVATE_BASE
          if (ok) v.p[i].base = v.rounds.chunk(p.r + 1);
#endif
          v.p[i].r += 1;
          v.p[i].pc = PUBLISH;
          if (v.p[i].r > MAX_ROUNDS) wrong = "more rounds than chunks";
          visit(v);
        }
        break;
      default:
        break;
    }
  }
}

int main() {
  for (n_chunks = 1; n_chunks <= 9; ++n_chunks) {
    seen.clear();
    State s;
    std::memset(&s, 0, sizeof s);   // (states are compared as bytes)
    s.rounds.start(0);
    s.next = 2;
    visit(s);
    if (wrong) {
      std::printf("%u chunks: %s\n", n_chunks, wrong);
      return 1;
    }
    std::printf("%u chunks: %zu states\n", n_chunks, seen.size());
  }
  return 0;
}
