// o2pic_device.h -- the device a handle lives on, current for the length of a
// call.
#ifndef O2PIC_DEVICE_H
#define O2PIC_DEVICE_H

namespace o2 {

// Api: int get(int *device), int set(int device), 0 = success (the CUDA runtime's
// in the library).  Kernels launch on the current device: a call made with
// another one current switches to the handle's and back again.
template <typename Api>
class OnDevice {
public:
    explicit OnDevice(int device)
    {
        int now = -1;
        err_ = Api::get(&now);
        if (err_ == 0 && now != device) {
            err_ = Api::set(device);
            if (err_ == 0) back_ = now;
        }
    }
    ~OnDevice()
    {
        if (back_ >= 0) Api::set(back_);
    }
    OnDevice(const OnDevice &) = delete;
    OnDevice &operator=(const OnDevice &) = delete;
    int error() const { return err_; }  // not 0: the device could not be made current

private:
    int err_ = 0, back_ = -1;
};

} // namespace o2

#endif
