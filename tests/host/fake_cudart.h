// The stand-in runtime's state (fake_cudart.cpp).
#pragma once
extern int g_device;               // the current device
extern int g_fail_attributes;      // attribute calls to fail
extern void (*g_meanwhile)();      // another thread's call, right after an attribute is set
extern int g_launched;             // launches that were not refused
