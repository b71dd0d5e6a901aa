// Sizes and index walks that hold for every row count a call accepts (up to
// INT32_MAX), in plain C++ so that they are also compiled and checked on the host.
#pragma once
#include <cstddef>
#include <cstdint>

// Bytes of shared memory that n staged 32-bit keys take: they are written and read
// four at a time, so the last group is whole.
constexpr size_t key_stage_bytes(int n) { return ((size_t)n + 3) / 4 * 16; }
