// Host check of csrc/hw_workpool.h: pools that share a memory of fixed size. Prints the number of failed expectations.
#include <cstdio>
#include <cstdlib>
#include <map>

#include "hw_workpool.h"

static std::map<void*, std::size_t> g_live;
static std::size_t g_used = 0;
constexpr std::size_t kMemory = 100;

struct Mem {
  static void* get(std::size_t bytes) {
    if (g_used + bytes > kMemory) return nullptr;
    void* p = malloc(1);
    g_live[p] = bytes;
    g_used += bytes;
    return p;
  }
  static void put(void* p) {
    if (!g_live.count(p)) abort();  // freed twice
    g_used -= g_live[p];
    g_live.erase(p);
    free(p);
  }
};

static int failed = 0;
#define EXPECT(x) do { if (!(x)) { ++failed; fprintf(stderr, "line %d: %s\n", __LINE__, #x); } } while (0)

using Pool = hw::WorkPool<Mem>;
enum { SAVE, VALUES, TAPE, SLOT };

int main() {
  auto none = [] { return false; };
  {
    // a tape is kept; a call with snapshots that need its room gets them
    Pool a;
    a.begin();
    EXPECT(a.get(VALUES, 1, none) && a.get(TAPE, 60, none));
    a.end(80);
    EXPECT(a.held() == 61 && g_used == 61);
    a.begin();
    void* const v = a.get(VALUES, 1, none);
    EXPECT(v);
    bool all = true;
    for (int k = 0; k < 9; ++k) all &= a.get(SLOT + k, 10, none) != nullptr;
    EXPECT(all && g_used == 91);
    EXPECT(a.get(VALUES, 1, none) == v);  // the call's own memory is never given back
    EXPECT(!a.get(TAPE, 60, none));       // more than there is
    EXPECT(a.get(VALUES, 1, none) == v && a.held() == 91);
    a.end(80);
    EXPECT(a.held() <= 80 && a.held() == g_used);
    // slots are kept; a call with a tape gets it, the copy of another kind of call goes too
    a.begin();
    EXPECT(a.get(SAVE, 9, none));
    a.end(80);
    a.begin();
    EXPECT(a.get(VALUES, 1, none) && a.get(TAPE, 95, none));
    EXPECT(g_used == 96);
    a.end(80);
    EXPECT(a.held() == 1);
    // enough bytes: the same memory again, without a new allocation
    a.begin();
    void* const t = a.get(TAPE, 50, none);
    a.end(80);
    a.begin();
    EXPECT(a.get(TAPE, 40, none) == t && a.held() == 51);
    a.end(0);
    EXPECT(a.held() == 0 && g_used == 0);
  }
  {
    // what others keep is asked for after the pool's own, and only then
    Pool a, b;
    a.begin();
    EXPECT(a.get(TAPE, 50, none));
    a.end(80);
    b.begin();
    EXPECT(b.get(SAVE, 30, none));
    b.end(80);
    int asked = 0;
    auto others = [&] {
      ++asked;
      return a.release_unclaimed();
    };
    b.begin();
    EXPECT(b.get(TAPE, 45, others) && asked == 0 && a.held() == 50);  // its own SAVE was enough
    EXPECT(b.get(SLOT, 20, others) && asked == 1 && a.held() == 0);
    EXPECT(!b.get(SLOT + 1, 60, others) && asked == 2 && g_used == 65);
    b.end(0);
    EXPECT(g_used == 0);
  }
  printf("%d\n", failed);
}
