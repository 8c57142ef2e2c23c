// The operator dispatch of the orders without kernels of their own: the form that is chosen for an order
// launches it, and a form asked for an order that it has no kernel for says so (run by
// test_operator_dispatch.py).
#include "fake_cudart.h"

using namespace chebmg;

template <typename T>
static bool run(const char* type) {
  bool good = true;
  char msg[96];
  const T* G = nullptr;
  for (int Q = 2; Q <= 11; ++Q) {
    for (int64_t E : {(int64_t)1, (int64_t)100, (int64_t)700, (int64_t)100000}) {
      if (Q == 8 || Q > 10) continue;   // order 7: sem_ax8
      const int before = g_seen;
      const bool ok = sem_axl_chosen<T>(Q, E) ? sem_axl<T>(Q, E, nullptr, nullptr, G, nullptr, nullptr, nullptr)
                                              : sem_ax<T>(Q, E, nullptr, G, nullptr, nullptr, nullptr, nullptr);
      std::snprintf(msg, sizeof msg, "%s Q = %d on %lld elements launches", type, Q, (long long)E);
      good &= check(msg, ok && g_seen == before + 1);
    }
    // either form launches, or says that it did not
    int before = g_seen;
    bool ok = sem_axl<T>(Q, 10, nullptr, nullptr, G, nullptr, nullptr, nullptr);
    std::snprintf(msg, sizeof msg, "%s Q = %d: line passes report a launch truly", type, Q);
    good &= check(msg, ok == (g_seen == before + 1) && ok == sem_axl_supported(Q));
    before = g_seen;
    ok = sem_ax<T>(Q, 10, nullptr, G, nullptr, nullptr, nullptr, nullptr);
    std::snprintf(msg, sizeof msg, "%s Q = %d: a thread per point reports a launch truly", type, Q);
    good &= check(msg, ok == (g_seen == before + 1));
  }
  return good;
}

int main() {
  const bool f = run<float>("FP32"), d = run<double>("FP64");
  return f && d ? 0 : 1;
}
