// Host-side checks of csrc/pinned_words.h with plain memory in place of pinned memory: no
// GPU, no CUDA.  Built and run by tests/test_pinned_words.py; prints "<name> ok" a scenario.
#include <cstdio>
#include <cstdlib>
#include <set>

#include "pinned_words.h"

#define CHECK(c)                                                                 \
  do {                                                                           \
    if (!(c)) {                                                                  \
      std::fprintf(stderr, "%s:%d: check failed: %s\n", __FILE__, __LINE__, #c); \
      std::exit(1);                                                              \
    }                                                                            \
  } while (0)

namespace {
std::set<void *> live;
bool out_of_memory = false;
void *get(size_t n) {
  if (out_of_memory) return nullptr;
  void *p = std::malloc(n);
  live.insert(p);
  return p;
}
void put(void *p) {
  live.erase(p);
  std::free(p);
}
const auto yes = [] { return true; };
const auto no = [] { return false; };
}  // namespace

int main() {
  using dem::PinnedLease;
  using dem::PinnedWords;
  PinnedWords pool(get, put);
  double *first;
  {
    PinnedLease a(pool);
    first = a.words();
    CHECK(a.fetch(yes, yes) && a.fetch(yes, yes));
    PinnedLease b(pool);
    CHECK(b.words() && b.words() != first);   // words in use are not handed out
  }
  {
    PinnedLease a(pool), b(pool);
    CHECK(live.size() == 2 && (a.words() == first || b.words() == first));
  }
  std::puts("reused ok");
  // a copy that was issued and not seen done keeps its words: the wait failed or timed out, in
  // the first fetch or a later one, or the copy itself reported an error
  for (int k = 0; k < 3; ++k) {
    PinnedWords q(get, put);
    double *lost;
    {
      PinnedLease a(q);
      lost = a.words();
      if (k == 2) CHECK(a.fetch(yes, yes));
      CHECK(!(k == 1 ? a.fetch(no, yes) : a.fetch(yes, no)));
    }
    for (int n = 0; n < 4; ++n) {
      PinnedLease a(q), b(q);
      CHECK(a.words() != lost && b.words() != lost && live.count(lost));
      CHECK(a.fetch(yes, yes));
    }
  }
  std::puts("withheld ok");
  out_of_memory = true;
  {
    PinnedWords q(get, put);
    PinnedLease a(q);
    CHECK(!a.words());
  }
  out_of_memory = false;
  {
    PinnedWords q(get, put);
    const size_t before = live.size();
    {
      PinnedLease *l[40];
      for (auto &x : l) x = new PinnedLease(q);
      CHECK(live.size() == before + 40);
      for (auto &x : l) delete x;
    }
    CHECK(live.size() == before + PinnedWords::kKept);   // bounded
  }
  std::puts("bounded ok");
  return 0;
}
