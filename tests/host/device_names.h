// Names that the device code of common.cuh uses, declared so that the host
// translation units (which call none of it) compile as plain C++.
#pragma once
#include <cstddef>
#include <cstdint>
#include <math.h>
unsigned __umulhi(unsigned, unsigned);
size_t __cvta_generic_to_shared(const void*);
unsigned atomicOr(unsigned*, unsigned);
float __shfl_xor_sync(unsigned, float, int);
