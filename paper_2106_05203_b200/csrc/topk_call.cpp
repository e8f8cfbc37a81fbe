// The Python call of the standalone Top-k for the usual arguments (an ordinary contiguous float32 CUDA tensor on the current device, the
// current stream), in native code: on short vectors the call was bound by its host side, 8.9 us against a kernel of 3 to 4 -- two
// allocations through the interpreter, a foreign call with nine arguments, a dozen attribute look-ups.  Everything else -- another stream
// or device, wrong arguments -- is left to binding.py: topk(v, k) then returns None.
//
// The entry points of libef21 come as addresses (set_entry), so that this module does not link against the library.
#include <ATen/ATen.h>
#include <c10/cuda/CUDAFunctions.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>

#include <cstdint>

namespace {

typedef size_t (*WorkspaceBytes)(int32_t, int64_t, int32_t);
typedef int (*Topk)(const float*, int32_t, int64_t, int32_t, int32_t*, float*, void*, size_t, void*);
WorkspaceBytes workspace_bytes = nullptr;
Topk topk_entry = nullptr;
constexpr size_t ALIGN = 256;

// Allocation and launch can wait for the device (a full launch queue, memory given back to the driver): not with the interpreter held.
struct Released {
    PyThreadState* state = PyEval_SaveThread();
    ~Released() { PyEval_RestoreThread(state); }
};

// topk(v, k) -> (idx, val), the library's status where it refuses, or None where the call is not one of the usual ones.
PyObject* topk(PyObject*, PyObject* const* args, Py_ssize_t nargs) {
    HANDLE_TH_ERRORS
    if (nargs != 2 || !topk_entry || !THPVariable_CheckExact(args[0]) || !PyLong_CheckExact(args[1])) Py_RETURN_NONE;
    const at::Tensor& v = THPVariable_Unpack(args[0]);
    if (!v.has_storage() || !v.is_cuda() || v.scalar_type() != at::kFloat || v.layout() != at::kStrided) Py_RETURN_NONE;
    const int64_t dim = v.dim();
    if ((dim != 1 && dim != 2) || !v.is_contiguous() || v.get_device() != c10::cuda::current_device()) Py_RETURN_NONE;
    const int64_t batch = dim == 2 ? v.size(0) : 1, d = v.size(dim - 1);
    int overflow = 0;
    const long long k = PyLong_AsLongLongAndOverflow(args[1], &overflow);
    if (overflow || k < 1 || k > d || k > INT32_MAX || batch < 1 || batch > 65535) Py_RETURN_NONE;
    at::Tensor idx, val;
    int status = 0;
    {
        const Released released;
        const size_t bytes = workspace_bytes((int32_t)batch, d, (int32_t)k);
        if (bytes != 0) {
            const at::TensorOptions here = at::TensorOptions().device(v.device());
            idx = at::empty({batch, k}, here.dtype(at::kInt)); val = at::empty({batch, k}, here.dtype(at::kFloat));
            at::Tensor ws;
            void* scratch = idx.data_ptr();                 // up to ALIGN bytes: checked, not used
            if (bytes > ALIGN || reinterpret_cast<uintptr_t>(scratch) % ALIGN != 0) {
                ws = at::empty({(int64_t)(bytes + ALIGN)}, here.dtype(at::kByte));
                scratch = reinterpret_cast<void*>((reinterpret_cast<uintptr_t>(ws.data_ptr()) + ALIGN - 1) / ALIGN * ALIGN);
            }
            status = topk_entry(static_cast<const float*>(v.data_ptr()), (int32_t)batch, d, (int32_t)k, static_cast<int32_t*>(idx.data_ptr()),
                                static_cast<float*>(val.data_ptr()), scratch, bytes, c10::cuda::getCurrentCUDAStream(v.get_device()).stream());
        }
    }
    if (!idx.defined()) Py_RETURN_NONE;
    if (status != 0) return PyLong_FromLong(status);
    PyObject* out = PyTuple_New(2);
    if (!out) return nullptr;
    PyTuple_SET_ITEM(out, 0, THPVariable_Wrap(std::move(idx)));
    PyTuple_SET_ITEM(out, 1, THPVariable_Wrap(std::move(val)));
    return out;
    END_HANDLE_TH_ERRORS
}

PyObject* set_entry(PyObject*, PyObject* args) {
    unsigned long long bytes = 0, entry = 0;
    if (!PyArg_ParseTuple(args, "KK", &bytes, &entry)) return nullptr;
    workspace_bytes = reinterpret_cast<WorkspaceBytes>(bytes);
    topk_entry = reinterpret_cast<Topk>(entry);
    Py_RETURN_NONE;
}

PyMethodDef methods[] = {{"topk", reinterpret_cast<PyCFunction>(reinterpret_cast<void*>(topk)), METH_FASTCALL, nullptr},
                         {"set_entry", set_entry, METH_VARARGS, nullptr},
                         {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_topk_call", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

// EF21_BUILT_FOR: the torch and the interpreter that this was compiled against (build.py), which are looked at before the module is used
extern "C" __attribute__((visibility("default"))) PyObject* PyInit__topk_call() {
    PyObject* m = PyModule_Create(&module);
    if (m && PyModule_AddStringConstant(m, "built_for", EF21_BUILT_FOR) != 0) { Py_DECREF(m); return nullptr; }
    return m;
}
