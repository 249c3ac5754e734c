// The device-block cache (csrc/devcache.cuh) over a host allocator of two fake
// devices that records its calls.  Reads commands from stdin:
//   use d | alloc id bytes | release id.. -1 | trim | limit bytes
// and prints, per command, what the allocator was asked for ("malloc d bytes",
// "free d", "sync d"), the block an alloc returned ("block n": n-th malloc) and the
// device current afterwards ("cur d").
#include <cstdio>
#include <cstring>
#include <map>
#include "../../paper_1810_07067_gb300/csrc/devcache.cuh"

static int g_cur = 0, g_count = 0;
static std::map<void*, std::pair<int, int>> g_owner;  // block -> (number, device)

struct Fake {
  using Error = int;
  static constexpr Error ok = 0;
  struct Guard {};
  static int device() { return g_cur; }
  static void use(int d) { g_cur = d; }
  static Error alloc(void** p, size_t bytes) {
    *p = (void*)(size_t)(++g_count);
    g_owner[*p] = {g_count, g_cur};
    printf("malloc %d %zu;", g_cur, bytes);
    return 0;
  }
  static void free(void* p) { printf(g_owner[p].second == g_cur ? "free %d;" : "BAD free %d;", g_cur); }
  static void sync() { printf("sync %d;", g_cur); }
  static void clear_error() {}
};

int main() {
  DeviceCache<Fake> cache;
  std::map<int, DevBlock> have;
  char op[16];
  while (scanf("%15s", op) == 1) {
    if (!strcmp(op, "use")) scanf("%d", &g_cur);
    else if (!strcmp(op, "trim")) cache.trim();
    else if (!strcmp(op, "limit")) {
      size_t b;
      scanf("%zu", &b);
      cache.limit(b);
    } else if (!strcmp(op, "alloc")) {
      int id;
      size_t b;
      scanf("%d %zu", &id, &b);
      DevBlock v;
      if (cache.alloc(&v, b) != 0) return 1;
      have[id] = v;
      printf("block %d;", g_owner[v.p].first);
      if (g_owner[v.p].second != g_cur) printf("BAD device;");
    } else if (!strcmp(op, "release")) {
      std::vector<DevBlock> v;
      for (int id; scanf("%d", &id) == 1 && id >= 0;) v.push_back(have[id]);
      cache.release(v.data(), v.size());
    }
    printf("cur %d held %zu\n", g_cur, cache.bytes_held());
  }
  return 0;
}
