// Where a network's forward writes its output.
#pragma once

namespace fh {

// The last kernel writes `y` itself if that is device memory of the network's own device;
// anything else (host, managed, another device's memory, which a kernel may not be able
// to reach) goes through a copy.
inline bool writes_directly(bool device_memory, int memory_device, int network_device) {
  return device_memory && memory_device == network_device;
}

}  // namespace fh
