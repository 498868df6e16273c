// The buffers of the multi-context launches that a context or a batcher leads: the flags the host reads and the words the
// CTAs poll. Compiled by test_gpu_multi_launcher.py against the library's internal header.
#include "aim_internal.h"

extern "C" {

int* probe_err_host(aim_ctx* ctx) { return ctx->multi ? ctx->multi->err_host : nullptr; }
void* probe_scratch(aim_ctx* ctx) { return ctx->multi ? ctx->multi->scratch : nullptr; }
int* probe_batcher_err_host(aim_batcher* b) { return aim::batcher_launcher(b).err_host; }

// Whether a launcher whose device allocation had failed takes up the pinned flags that it already held.
int probe_init_keeps_flags() {
  aim::MultiLauncher first, rest;
  if (first.init(nullptr) != AIM_OK) return -1;
  int* flags = first.err_host;
  rest.scratch = first.scratch;   // freed with `rest`
  first.scratch = nullptr;        // as after a refused cudaMalloc
  if (first.init(nullptr) != AIM_OK) return -1;
  return first.err_host == flags && first.scratch != nullptr;
}

}  // extern "C"
