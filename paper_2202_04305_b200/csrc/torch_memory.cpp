// torch's caching allocator and torch views of device memory for the Python binding, as plain C calls.
//
// The library asks for scratch inside its calls: reached through a Python callback each request took
// 4 to 5 microseconds of host time, more than the launch it served; this one takes about 0.3.
#include <Python.h>

#include <ATen/ops/from_blob.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <torch/csrc/autograd/python_variable.h>

extern "C" {

// The two hooks of sp_set_allocator.  No exception leaves them: NULL means that there is no memory.
void* sp_torch_alloc(size_t bytes, void* stream, void*) {
    try {
        return c10::cuda::CUDACachingAllocator::raw_alloc_with_stream(bytes ? bytes : 1, static_cast<cudaStream_t>(stream));
    } catch (...) {
        return nullptr;
    }
}

void sp_torch_free(void* ptr, void*, void*) {
    try {
        if (ptr) c10::cuda::CUDACachingAllocator::raw_delete(ptr);
    } catch (...) {
    }
}

// A one-dimensional tensor over n elements of device memory (code: 1, 2 = uint8, uint16; 4, 8 = int32,
// int64; 0 = float64) that keeps `owner` alive.  Called with the GIL held.
PyObject* sp_torch_view(void* ptr, int64_t n, int code, PyObject* owner) {
    try {
        const at::ScalarType type = code == 1   ? at::kByte
                                    : code == 2 ? at::kUInt16
                                    : code == 4 ? at::kInt
                                    : code == 8 ? at::kLong
                                                : at::kDouble;
        Py_INCREF(owner);
        at::Tensor t = at::from_blob(
            ptr, {n},
            [owner](void*) {
                if (!Py_IsInitialized()) return;         // the interpreter is gone, and the owner with it
                const PyGILState_STATE s = PyGILState_Ensure();
                Py_DECREF(owner);
                PyGILState_Release(s);
            },
            at::TensorOptions().dtype(type).device(at::kCUDA));
        return THPVariable_Wrap(std::move(t));
    } catch (const std::exception& e) {
        PyErr_SetString(PyExc_RuntimeError, e.what());
        return nullptr;
    }
}

}  // extern "C"
