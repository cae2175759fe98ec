// The stand-in runtime's state (fake_cudart.cpp).
#pragma once
#include <cstddef>
extern int g_device;               // the current device
extern int g_fail_attributes;      // attribute calls to fail
extern void (*g_meanwhile)();      // another thread's call, right after an attribute is set
extern int g_launched;             // launches that were not refused
extern size_t g_last_smem;         // the last one's dynamic shared memory
extern unsigned g_last_blocks;     // and blocks
extern int g_splits;               // kernels that were given a split of L1 and shared memory
