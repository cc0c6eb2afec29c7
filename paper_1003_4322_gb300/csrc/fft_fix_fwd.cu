// fft_fix_fwd.cu -- the forward x and y passes of the FP64 transforms (kernel:
// fft_fix_strided.cuh).
#include "fft_fix_strided.cuh"

namespace nsk {

const void *fix_fwd_kernel(int E, int in, int out) {
    if (in == kIoFixed)
        return out == kIoFixed ? fix_kernel_of<-1, kIoFixed, kIoFixed>(E) : fix_kernel_of<-1, kIoFixed, kIoDouble>(E);
    return in == kIoDouble && out == kIoDouble ? fix_kernel_of<-1, kIoDouble, kIoDouble>(E) : nullptr;
}

}  // namespace nsk
