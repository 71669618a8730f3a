// Between the library and the Python marshalling module (not part of the public interface): a segment plan's words on their way to
// the device as the arguments of a kernel.
#pragma once
#include <stdint.h>

namespace mpipe {
constexpr int32_t kPlanWordsMax = 8128;   // a kernel's arguments end at 32 764 bytes
}

// n <= kPlanWordsMax words to device memory, in stream order; an mpipe status.
extern "C" int32_t mpipe_plan_words_to_device(const void* words, int32_t n, void* dst, void* stream);
