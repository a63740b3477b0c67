// Values that hold on one device (function attributes that were set there, what
// an occupancy query answered there), made on first use and kept for the process.
#pragma once

#include <map>
#include <mutex>
#include <utility>

namespace gw {

template <class K, class V> class DeviceCache {
 public:
  // The value of key on device dev; make(&v) returns whether it made it.  A
  // failure is not kept: the next call tries again.
  template <class Make> bool get(int dev, const K& key, V* out, Make make) {
    std::lock_guard<std::mutex> lock(mu_);
    auto it = map_.find({dev, key});
    if (it == map_.end()) {
      V v{};
      if (!make(&v)) return false;
      it = map_.emplace(std::make_pair(dev, key), v).first;
    }
    *out = it->second;
    return true;
  }

  // A limit that is only ever raised: set(v) runs on device dev where v is
  // above what was set there; its status (0: success) is returned.
  template <class Set> int raise(int dev, const K& key, const V& v, Set set) {
    std::lock_guard<std::mutex> lock(mu_);
    auto it = map_.find({dev, key});
    if (it != map_.end() && !(it->second < v)) return 0;
    const int e = set(v);
    if (e == 0) map_[{dev, key}] = v;
    return e;
  }

 private:
  std::mutex mu_;
  std::map<std::pair<int, K>, V> map_;
};

}  // namespace gw
