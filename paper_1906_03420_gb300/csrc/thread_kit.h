// What a host thread keeps between its calls.  Host code only.
#pragma once

#include <cstddef>

#include <cuda_runtime.h>

namespace gsi {

// PINNED_READ + PINNED_STAGE bytes of pinned memory of the calling thread:
// small readbacks first, then an upload area.  Null without memory.
constexpr size_t PINNED_READ = 4096, PINNED_STAGE = 60 * 1024;
unsigned char *thread_pinned();
// The calling thread's event on a device, for waits within one entry point.
// Null: none.
cudaEvent_t thread_event(int dev);
// Every use is complete before the entry point that makes it returns, so a
// thread that ends hands both on to the next new one (cudaFreeHost would
// synchronise the whole device): there are as many as there were threads in the
// library at the same time.

}  // namespace gsi
