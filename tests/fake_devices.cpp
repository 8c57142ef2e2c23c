// Host code of the operator files on two devices: what a launch needs on a device must have been set on
// that device (run by test_per_device.py).
#include <thread>
#include <vector>

#include "fake_cudart.h"

using namespace chebmg;

template <typename T>
static void operators(int64_t E, const Lattice& lat) {
  for (int Q : {3, 5, 6, 7, 9, 10})
    for (const Lattice* l : {&lat, static_cast<const Lattice*>(nullptr)})
      sem_axl<T>(Q, E, nullptr, l, static_cast<const T*>(nullptr), nullptr, nullptr, nullptr);
  for (int v : {1, 2, 4, 12, 14, 21, 22, 31, 32, 101, 102, 104, 112, 114, 121, 122, 131, 132})
    if (sem_ax8_variant_fits<T>(v)) sem_ax8<T>(E, nullptr, lat, static_cast<const T*>(nullptr), nullptr, nullptr, nullptr, v, nullptr);
  for (int v : {1, 2, 4, 11, 12, 21, 22, 101, 102, 104, 111, 112, 121, 122})
    if (sem_ax8_batched_fits<T>(2000 + v))
      sem_ax8_batched<T>(E, nullptr, lat, static_cast<const T*>(nullptr), nullptr, nullptr, nullptr, 2000 + v, 4, 512, nullptr);
}

static void all() {
  Lattice lat{};
  lat.nex = lat.ney = lat.nez = 16;
  for (int64_t E : {(int64_t)30, (int64_t)4096}) {
    operators<float>(E, lat);
    operators<double>(E, lat);
  }
  for (int v : {1, 2, 4, 101, 102, 104})
    sem_ax8_x2(4096, nullptr, lat, nullptr, nullptr, nullptr, nullptr, v, nullptr);
}

int main() {
  bool bad = false;
  // one device after the other, in one process
  for (int d : {0, 1}) {
    t_dev = d;
    const int before = g_bad, large = g_large;
    all();
    char msg[64];
    std::snprintf(msg, sizeof msg, "shared-memory limits on device %d", d);
    bad |= !check(msg, g_bad == before && g_large > large);
  }
  // sizes that follow the device's SM count
  for (int d : {0, 1, 0}) {
    t_dev = d;
    int grid = 0, rows = 0;
    coarse_pcg_shape(30000, 1, &grid, &rows);
    char msg[64];
    std::snprintf(msg, sizeof msg, "rows per coarse block on device %d: %d", d, rows);
    bad |= !check(msg, rows == (d == 0 ? 256 : 1024));
    std::snprintf(msg, sizeof msg, "FP64 order-5 kernel of 300 elements on device %d", d);
    bad |= !check(msg, sem_axl_chosen<double>(6, 300) == (d == 1));
    std::snprintf(msg, sizeof msg, "lattice coarse blocks of 256 rows on device %d", d);
    bad |= !check(msg, coarse_lat_fits(30000, 31, 256) == (d == 0));
  }
  // both at once: several threads start together on fresh limits of both devices
  {
    std::vector<std::thread> th;
    const int before = g_bad;
    for (int q = 0; q < 8; ++q)
      th.emplace_back([q] {
        t_dev = q & 1;
        all();
      });
    for (auto& t : th) t.join();
    bad |= !check("eight threads on two devices", g_bad == before);
  }
  std::printf("launches %d, with large blocks %d\n", g_seen, g_large);
  return bad ? 1 : 0;
}
