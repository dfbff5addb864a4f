// device_drain.h -- waiting for one device's work whatever device is current.
// Plain C++: tests/test_device_drain.py runs it on a fake runtime.
#pragma once

namespace spm {

// Waits for all queued work of `device` and leaves the current device as it
// was.  Rt: get(int*), set(int) and sync() of the runtime, true on success.
// False: the wait did not take place or reported an error.
template <class Rt>
bool drain_device(Rt& rt, int device) {
  int current = -1;
  if (!rt.get(&current)) return false;
  if (current == device) return rt.sync();
  if (!rt.set(device)) return false;
  const bool ok = rt.sync();
  rt.set(current);
  return ok;
}

}  // namespace spm
