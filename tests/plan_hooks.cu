// Handles for the tests on state that no public call changes: a device of another size.
#include "kx_internal.h"

// The number of SMs the plan's launches count on; returns the number before.
extern "C" int hook_num_sms(kx_plan *p, int n) {
    const int old = p->num_sms;
    p->num_sms = n;
    return old;
}
