// Declarations of the fused LM head + row statistics (lm_head.cu), used by the ABI.
#pragma once

#include "common.cuh"

namespace specv {

constexpr int kLmMaxSms = 160;     // multiprocessors the tile plan uses at most
constexpr int kLmMaxVocab = 65535 * 224;
struct LmLayout {
  size_t parts;  // 16 B [rows][vocab tiles]: (max, sum, argmax, token logit) per tile
  size_t end;    // sized for the widest plan of any device with up to kLmMaxSms SMs
};
LmLayout lm_layout(const spec_lm_head_args_t& a, size_t base);
// starve (test hook only): the producer issues no copies, so the kernel's bounded waits
// run out and it returns with SPEC_FLAG_TIMEOUT set (outputs undefined).
cudaError_t launch_lm_head(const spec_lm_head_args_t& a, const LmLayout& L, char* ws, int sms,
                           cudaStream_t stream, bool starve = false);

}  // namespace specv
