// A plan's calls run on the device that was current when it was created.  The CUDA device is
// a property of the host thread, so a thread that only reads a plan back may have another one
// current: what the call creates or launches there (the read-back's stream, the sort's buffers
// and kernels) would land on that device and address the plan's memory from it.
#pragma once

namespace fstat {

// Makes `device` current while it lives and the caller's device again after.  Api: bool
// get(int *) and bool set(int) of the current device.
template <class Api>
class DeviceGuard {
public:
    explicit DeviceGuard(int device) {
        if (device < 0) return;   // a plan that has no device yet
        ok_ = Api::get(&before_);
        if (!ok_ || before_ == device) return;
        ok_ = changed_ = Api::set(device);
    }
    ~DeviceGuard() {
        if (changed_) Api::set(before_);
    }
    DeviceGuard(const DeviceGuard &) = delete;
    DeviceGuard &operator=(const DeviceGuard &) = delete;
    bool ok() const { return ok_; }

private:
    int before_ = -1;
    bool ok_ = true, changed_ = false;
};

}  // namespace fstat
