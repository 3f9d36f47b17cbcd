// The parts of the autograd integration that run once per layer and direction, as a CPython extension on torch's C++ API:
// the node of the ReLU that stashes its activation, the restore of a stash, and the wait for a stash's count.  No
// arithmetic here: every function allocates its outputs and calls the library's C ABI, through the address it is given
// (a caller may have more than one build of the library open).
//
// What bounds a training step of small layers is the host.  Eight layers of 512 x 512 in float32 with an arena: 1115 us with
// the node and the restore in Python, 960 with them here (641 without any stash); six of 8192 x 1024 in bfloat16 with
// exact-size values 1093 and 990.  What is left above the bare step: the saved-tensor hooks, which torch calls in Python,
// 12 us per stashing ReLU against 6.5 for torch.relu, 4.7 per restore, and the one read of the status words.
#define PY_SSIZE_T_CLEAN
#include <Python.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Dtype.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/custom_function.h>
#include <torch/csrc/autograd/python_variable.h>

#include "bittrain.h"

namespace {

using at::Tensor;

// A stash's record: the bitmap, from the next multiple of 16 bytes on the chunk prefix array, behind it two words (the
// count and, in an arena, the byte offset of the values).  The same layout as _Record in autograd.py.
constexpr int64_t kChunk = BT_CHUNK_ELEMS;
int64_t prefix_at(const int64_t n) { return ((n + 31) / 32 * 4 + 15) & ~int64_t(15); }
int64_t words_at(const int64_t n) { return prefix_at(n) + (n + kChunk - 1) / kChunk * 8; }

bool usable(const Tensor &t) { return t.is_contiguous() && reinterpret_cast<uintptr_t>(t.data_ptr()) % 16 == 0; }
Tensor flat(const Tensor &t) { return usable(t) ? t : t.clone(at::MemoryFormat::Contiguous); }
void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

int code_of(const at::ScalarType t)
{
    switch (t) {
    case at::kFloat: return BT_F32;
    case at::kHalf: return BT_F16;
    case at::kBFloat16: return BT_BF16;
    case at::kDouble: return BT_F64;
    default: TORCH_CHECK(false, "no stash of this dtype: ", t);
    }
}

// Which of the ABI's fused compressors `call` is.
enum Form { kPlain = 0, kNarrow = 1, kArena = 2 };

struct Request {
    uintptr_t call, bwd;     // compressor (0: an empty tensor, nothing to call) and backward
    int       form, code;    // code: type of the stored values
    bool      inplace;
    void     *store;         // values or arena, of `room` elements or bytes
    uint64_t  room;
    void     *cursor, *nnz;  // arena cursor; where the count goes (NULL: the record's first word)
    void     *ws;
    size_t    ws_bytes;
    void     *status;
    Tensor    record;        // out
    int       result = 0;    // out: the ABI's status code
    bool      called = false;   // out: the compressor is on its stream (or has refused)
};

struct ReLUStash : torch::autograd::Function<ReLUStash> {
    static Tensor forward(torch::autograd::AutogradContext *ctx, const Tensor &x, Request *r)
    {
        Tensor in, y;
        if (r->inplace && usable(x)) {
            in = y = x;      // the kernel may write the activation over its input
            ctx->mark_dirty({x});
        } else {
            in = flat(x);
            y  = at::empty_like(in);
        }
        const int64_t n = in.numel();
        r->record       = at::empty({words_at(n) + 16}, in.options().dtype(at::kByte));
        auto *const rec = static_cast<unsigned char *>(r->record.data_ptr());
        auto *const bitmap = reinterpret_cast<uint32_t *>(rec);
        auto *const prefix = reinterpret_cast<uint64_t *>(rec + prefix_at(n));
        auto *const words  = reinterpret_cast<uint64_t *>(rec + words_at(n));
        auto *const nnz    = r->nnz ? static_cast<uint64_t *>(r->nnz) : words;
        auto *const status = static_cast<int32_t *>(r->status);
        r->called              = r->call != 0;
        if (!r->called) r->result = BT_OK;
        else if (r->form == kArena)
            r->result = reinterpret_cast<decltype(&bt_prune_fwd_compress_arena)>(r->call)(
                in.data_ptr(), n, r->code, 0.0f, y.data_ptr(), bitmap, r->store, r->room, static_cast<uint64_t *>(r->cursor), words + 1, prefix, nnz,
                r->ws, r->ws_bytes, status, stream());
        else if (r->form == kNarrow)
            r->result = reinterpret_cast<decltype(&bt_prune_fwd_compress_narrow)>(r->call)(in.data_ptr(), n, r->code, 0.0f, y.data_ptr(), bitmap, r->store,
                                                                                           r->room, prefix, nnz, r->ws, r->ws_bytes, status, stream());
        else
            r->result = reinterpret_cast<decltype(&bt_relu_fwd_compress)>(r->call)(in.data_ptr(), n, r->code, y.data_ptr(), bitmap, r->store, r->room, prefix,
                                                                                   nnz, r->ws, r->ws_bytes, status, stream());
        ctx->save_for_backward({r->record});      // released with the graph, like any saved tensor
        ctx->saved_data["bwd"] = static_cast<int64_t>(r->bwd);
        return y;
    }

    // reads only the bitmap, with which the record begins
    static torch::autograd::variable_list backward(torch::autograd::AutogradContext *ctx, const torch::autograd::variable_list &grads)
    {
        const Tensor record = ctx->get_saved_variables()[0];
        const Tensor g      = flat(grads[0]);
        Tensor       gin    = at::empty_like(g);
        const auto   call   = reinterpret_cast<decltype(&bt_relu_bwd_from_bitmap)>(ctx->saved_data["bwd"].toInt());
        const int    st     = call(static_cast<const uint32_t *>(record.data_ptr()), g.data_ptr(), g.numel(), code_of(g.scalar_type()), gin.data_ptr(), stream());
        TORCH_CHECK(st == BT_OK, "bt_relu_bwd_from_bitmap: status ", st);
        return {gin, Tensor()};
    }
};

// An argument that is an address, a tensor (its data) or None.  (The test for a tensor is slow on anything else, and may not
// be made with an error set.)
void *address(PyObject *o)
{
    if (o == Py_None || PyErr_Occurred()) return nullptr;
    if (PyLong_CheckExact(o) || !THPVariable_Check(o)) return PyLong_AsVoidPtr(o);
    return THPVariable_Unpack(o).data_ptr();
}
bool arguments(const Py_ssize_t have, const Py_ssize_t want)
{
    if (have == want) return true;
    PyErr_Format(PyExc_TypeError, "%zd arguments, not %zd", want, have);
    return false;
}
bool is_tensor(PyObject *o)
{
    if (THPVariable_Check(o)) return true;
    PyErr_SetString(PyExc_TypeError, "a tensor is wanted");
    return false;
}

// relu_stash(x, call, bwd, form, code, inplace, store, room, cursor, nnz, ws, ws_bytes, status) -> (status, y, record)
PyObject *relu_stash(PyObject *, PyObject *const *a, const Py_ssize_t count)
{
    HANDLE_TH_ERRORS
    if (!arguments(count, 13) || !is_tensor(a[0])) return nullptr;
    const Tensor &x = THPVariable_Unpack(a[0]);
    Request r;
    r.call = reinterpret_cast<uintptr_t>(address(a[1])), r.bwd = reinterpret_cast<uintptr_t>(address(a[2]));
    r.form = static_cast<int>(PyLong_AsLong(a[3])), r.code = static_cast<int>(PyLong_AsLong(a[4])), r.inplace = a[5] == Py_True;
    r.store = address(a[6]), r.room = PyLong_AsUnsignedLongLong(a[7]), r.cursor = address(a[8]), r.nnz = address(a[9]);
    r.ws = address(a[10]), r.ws_bytes = PyLong_AsSize_t(a[11]), r.status = address(a[12]);
    if (PyErr_Occurred()) return nullptr;
    TORCH_CHECK(x.is_cuda(), "a CUDA tensor is wanted");
    Tensor y;
    {
        pybind11::gil_scoped_release no_gil;
        try {
            y = ReLUStash::apply(x, &r);
        } catch (...) {
            // A saved-tensor hook raised behind the launch (a recomputation under a checkpoint ends that way).  With a count
            // word of the caller's the kernel still has to store into memory that the caller's next call waits on: not later
            // than here.
            if (r.called && r.nnz) c10::cuda::getCurrentCUDAStream().synchronize();
            throw;
        }
    }
    return Py_BuildValue("(iNN)", r.result, THPVariable_Wrap(y), THPVariable_Wrap(r.record));
    END_HANDLE_TH_ERRORS
}

// restore(call, record, store, in_arena, code, shape, dtype) -> (status, tensor); code: type of the stored values
PyObject *restore(PyObject *, PyObject *const *a, const Py_ssize_t count)
{
    HANDLE_TH_ERRORS
    if (!arguments(count, 7) || !is_tensor(a[1])) return nullptr;
    const uintptr_t call   = reinterpret_cast<uintptr_t>(address(a[0]));
    const Tensor    record = THPVariable_Unpack(a[1]);
    void *const     store  = address(a[2]);
    const int       code   = static_cast<int>(PyLong_AsLong(a[4]));
    if (PyErr_Occurred()) return nullptr;
    if (!PyTuple_Check(a[5]) || !THPDtype_Check(a[6])) {
        PyErr_SetString(PyExc_TypeError, "a shape and a dtype are wanted");
        return nullptr;
    }
    c10::SmallVector<int64_t, 6> shape;
    for (Py_ssize_t k = 0; k < PyTuple_GET_SIZE(a[5]); ++k) shape.push_back(PyLong_AsLongLong(PyTuple_GET_ITEM(a[5], k)));
    if (PyErr_Occurred()) return nullptr;
    const at::ScalarType type = reinterpret_cast<THPDtype *>(a[6])->scalar_type;
    const bool in_arena       = a[3] == Py_True;
    Tensor out;
    int    st = 0;
    {
        pybind11::gil_scoped_release no_gil;
        out             = at::empty(shape, record.options().dtype(type));
        const int64_t n = out.numel();
        TORCH_CHECK(record.nbytes() >= static_cast<size_t>(words_at(n) + (in_arena ? 16 : 0)), "not the record of such a tensor");
        auto *const rec    = static_cast<unsigned char *>(record.data_ptr());
        auto *const bitmap = reinterpret_cast<uint32_t *>(rec);
        auto *const prefix = reinterpret_cast<uint64_t *>(rec + prefix_at(n));
        auto *const words  = reinterpret_cast<uint64_t *>(rec + words_at(n));
        // the widening forms have the same arguments
        if (in_arena) st = reinterpret_cast<decltype(&bt_decompress_arena)>(call)(bitmap, store, words + 1, prefix, n, code, out.data_ptr(), stream());
        else st = reinterpret_cast<decltype(&bt_decompress)>(call)(bitmap, store, prefix, n, code, out.data_ptr(), stream());
    }
    return Py_BuildValue("(iN)", st, THPVariable_Wrap(out));
    END_HANDLE_TH_ERRORS
}

// synchronize(): waits for the current stream
PyObject *synchronize(PyObject *, PyObject *)
{
    HANDLE_TH_ERRORS
    {
        pybind11::gil_scoped_release no_gil;
        c10::cuda::getCurrentCUDAStream().synchronize();
    }
    Py_RETURN_NONE;
    END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {
    {"relu_stash", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(relu_stash)), METH_FASTCALL, nullptr},
    {"restore", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(restore)), METH_FASTCALL, nullptr},
    {"synchronize", synchronize, METH_NOARGS, nullptr},
    {nullptr, nullptr, 0, nullptr},
};
PyModuleDef module = {PyModuleDef_HEAD_INIT, "_autograd", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__autograd() { return PyModule_Create(&module); }
