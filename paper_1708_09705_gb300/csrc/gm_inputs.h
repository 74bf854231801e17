// Which of a caller's arrays a kernel may read where they are (host code).
#pragma once
#include <cstddef>
#include <cstdint>

namespace gm {

// device: the device whose memory p points to, negative for any other memory.
// Memory of another device is out: without peer access a kernel could not read it.
// So is an address that the kernel's loads could not use.
inline bool read_in_place(int device, int ctx_device, const void* p, size_t align) {
  return device >= 0 && device == ctx_device && reinterpret_cast<uintptr_t>(p) % align == 0;
}

}  // namespace gm
