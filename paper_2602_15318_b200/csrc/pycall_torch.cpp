// What pycall.c takes from torch's own objects without going through their Python methods: a tensor's address
// (75 ns as a method call, 5 like this) and the current stream (100 ns as two calls).
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/autograd/python_variable.h>

// 1: *out is the tensor's address; 0: not a plain tensor, or one without memory (its method says why)
extern "C" int sparrow_tensor_address(PyObject* o, int64_t* out)
{
    if (!THPVariable_CheckExact(o)) return 0;
    try {
        *out = (int64_t)(intptr_t)THPVariable_Unpack(o).data_ptr();
        return 1;
    } catch (...) {
        return 0;
    }
}

// torch's current stream on the current device; 0 when there is none to be had
extern "C" int sparrow_current_stream(int64_t* out)
{
    try {
        *out = (int64_t)(intptr_t)c10::cuda::getCurrentCUDAStream().stream();
        return 1;
    } catch (...) {
        return 0;
    }
}
