// The buffers of the multi-context launches that a context leads: the flags the host reads and the words the
// CTAs poll. Compiled by test_gpu_multi_launcher.py against the library's internal header.
#include "aim_internal.h"

extern "C" {

int* probe_err_host(aim_ctx* ctx) { return ctx->multi ? ctx->multi->err_host : nullptr; }
void* probe_scratch(aim_ctx* ctx) { return ctx->multi ? ctx->multi->scratch : nullptr; }

}  // extern "C"
