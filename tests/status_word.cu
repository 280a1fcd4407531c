// Test-only: writes into a context what cannot be had on demand: the status word that a kernel's expired wait
// leaves, and a number of SMs other than the device's.
#include "tbpm_internal.cuh"

extern "C" void set_status_word(tbpm_ctx* ctx, int code) {
  *reinterpret_cast<volatile int*>(ctx->pinned + tbpm::kSweepStatusSlot) = code;
}

extern "C" void set_num_sms(tbpm_ctx* ctx, int n) { ctx->num_sms = n; }
