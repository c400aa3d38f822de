// The choice between storing results straight into a caller's device array and copying them there
// (csrc/mhd_internal.h), on the host.
#include "mhd_internal.h"

extern "C" int direct_output_choice(int type, int owner, int device, unsigned long long address) {
  return mhd::direct_output(type, owner, device, reinterpret_cast<const void *>(address));
}
