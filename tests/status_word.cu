// Test-only: writes the status word that a kernel's expired wait would leave in a context.
#include "tbpm_internal.cuh"

extern "C" void set_status_word(tbpm_ctx* ctx, int code) {
  *reinterpret_cast<volatile int*>(ctx->pinned + tbpm::kSweepStatusSlot) = code;
}
