// The views of an export as torch tensors: sizes, one allocation, the queued copy and the five tensors in one call from Python.  Bound by the
// host: 32 mini-batches' views are asked for while the export runs, and in Python one took 13 us, half of it for cutting the allocation up.
// The library itself stays free of torch types: its entry point comes in as an address.
#define PY_SSIZE_T_CLEAN
#include <ATen/ops/empty.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/utils/pybind.h>

#include "mgdense.h"

namespace {

constexpr int64_t kAlign = 128;   // int32 values: the arrays of a view start 512 bytes apart, as allocations of their own would

typedef int (*ExportCopy)(mg_ctx*, mg_dense*, int32_t, mg_dense_arrays*, int32_t*, int32_t, void*);

// export_view(address of mg_dense_export_copy_aligned, context, sample, mini-batch, device, stream): the five tensors, or the call's error code
PyObject* export_view(PyObject*, PyObject* const* args, Py_ssize_t n_args) {
    HANDLE_TH_ERRORS
    TORCH_CHECK(n_args == 6, "export_view takes six arguments");
    void* address[3];
    for (int i = 0; i < 3; ++i) address[i] = PyLong_AsVoidPtr(args[i]);
    const int32_t batch = (int32_t)PyLong_AsUnsignedLongLongMask(args[3]);   // (the low 32 bits, as ctypes takes an int32)
    if (PyErr_Occurred()) return nullptr;
    const int64_t device = PyLong_AsLongLong(args[4]);
    void* stream = PyLong_AsVoidPtr(args[5]);
    if (PyErr_Occurred()) return nullptr;
    const ExportCopy copy = reinterpret_cast<ExportCopy>(address[0]);
    mg_ctx* ctx = static_cast<mg_ctx*>(address[1]);
    mg_dense* dense = static_cast<mg_dense*>(address[2]);
    mg_dense_arrays arrays;
    at::Tensor block;
    int64_t length[5];
    int rc;
    {
        pybind11::gil_scoped_release released;
        rc = copy(ctx, dense, batch, &arrays, nullptr, (int32_t)kAlign, nullptr);
        if (rc == 0) {
            const int64_t lengths[5] = {arrays.n_nodes, arrays.k + 2, arrays.n_entries, arrays.n_sampled + 1, arrays.n_entries};
            int64_t total = 0;
            for (int i = 0; i < 5; ++i) { length[i] = lengths[i]; total += (lengths[i] + kAlign - 1) / kAlign * kAlign; }
            block = at::empty({total}, at::TensorOptions().dtype(at::kInt).device(at::kCUDA, (c10::DeviceIndex)device));
            rc = copy(ctx, dense, batch, &arrays, block.data_ptr<int32_t>(), (int32_t)kAlign, stream);
        }
    }
    if (rc != 0) return PyLong_FromLong(rc);
    PyObject* views = PyTuple_New(5);
    if (!views) return nullptr;
    int64_t at = 0;
    for (int i = 0; i < 5; ++i) {
        // a tensor of its own on the block's memory, no view of it: what is done to one in place is no change of the others
        at::Tensor piece = at::detail::make_tensor<c10::TensorImpl>(c10::Storage(block.storage()), block.key_set(), block.dtype());
        c10::TensorImpl* impl = piece.unsafeGetTensorImpl();
        impl->set_storage_offset(at);
        impl->set_sizes_contiguous(c10::IntArrayRef(&length[i], 1));
        at += (length[i] + kAlign - 1) / kAlign * kAlign;
        PyObject* wrapped = THPVariable_Wrap(std::move(piece));
        if (!wrapped) { Py_DECREF(views); return nullptr; }
        PyTuple_SET_ITEM(views, i, wrapped);
    }
    return views;
    END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {{"export_view", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(export_view)), METH_FASTCALL, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_mgviews", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__mgviews() { return PyModule_Create(&module); }
