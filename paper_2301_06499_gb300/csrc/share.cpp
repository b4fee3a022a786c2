// Division of a device's SMs between the propagations that are on it.
//
// A resident round loop (resident.cu) holds its SMs for its whole length: a
// block of 512 threads takes all registers of one, and what does not fit waits
// for the loop to end. So propagations of different graphs from different host
// threads, which a caller may run side by side, are told to each other here:
// with one on the device it gets all SMs it may use; with several each gets its
// part, in equal parts up to what it can use (the caller's limit, else a block
// per 256 rows, 8 at least, so that a small graph beside a large one takes
// little from it). A loop reads its part once a round and, when that has
// changed, ends its launch after the round and goes on with a launch of the new
// size. Propagations in kernels of their own cannot be told, but count.
#include <algorithm>
#include <mutex>
#include <vector>

#include "host.cuh"

namespace pg {

namespace {

std::mutex g_mu;
std::vector<Share *> g_live;  // on all devices

}  // namespace

// Parts of total for n propagations that may use cap[i] SMs and, beside
// others, need[i] of them: equal parts, what one does not need going to the
// others. The parts add up to at most total (unless there are more
// propagations than SMs: one each then).
void share_parts(int n, const int *cap, const int *need, int total, int *part) {
  if (n == 1) {
    part[0] = std::max(1, std::min(cap[0], total));
    return;
  }
  std::vector<int> order(n);
  for (int i = 0; i < n; ++i) order[i] = i;
  auto use = [&](int i) { return std::max(1, std::min(cap[i], need[i])); };
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return use(a) < use(b); });
  int left = total;
  for (int k = 0; k < n; ++k) {  // the least needy first
    const int i = order[k];
    part[i] = std::max(1, std::min(use(i), left / (n - k)));
    left = std::max(0, left - part[i]);
  }
}

static void divide(int device) {  // under g_mu
  if (g_live.size() == 1 && g_live[0]->device == device) {  // alone
    Share *x = g_live[0];
    x->part = x->cap;
    if (x->want) *x->want = x->cap;
    return;
  }
  std::vector<Share *> s;
  std::vector<int> cap, need;
  for (Share *x : g_live)
    if (x->device == device) {
      s.push_back(x);
      cap.push_back(x->cap);
      need.push_back(x->need);
    }
  if (s.empty()) return;
  std::vector<int> part(s.size());
  share_parts((int)s.size(), cap.data(), need.data(), s[0]->total, part.data());
  for (size_t i = 0; i < s.size(); ++i) {
    s[i]->part = part[i];
    if (s[i]->want) *s[i]->want = part[i];
  }
}

Share::Share(int device_, int total_, int cap_, int64_t rows, volatile int32_t *want_)
    : device(device_), total(total_), cap(cap_ > 0 ? std::min(cap_, total_) : total_),
      want(want_) {
  need = cap_ > 0 ? cap : (int)std::min<int64_t>(cap, std::max<int64_t>(8, rows / 256));
  std::lock_guard<std::mutex> lk(g_mu);
  g_live.push_back(this);
  divide(device);
}

Share::~Share() {
  std::lock_guard<std::mutex> lk(g_mu);
  g_live.erase(std::find(g_live.begin(), g_live.end(), this));
  divide(device);
}

void Share::limit(int sms) {
  std::lock_guard<std::mutex> lk(g_mu);
  cap = std::min(cap, sms);
  divide(device);
}

}  // namespace pg

#ifdef PG_DEBUG_BOUNDS
// For tests: share_parts.
extern "C" void pg_debug_share_parts(int n, const int *cap, const int *need, int total, int *part) {
  pg::share_parts(n, cap, need, total, part);
}
#endif
