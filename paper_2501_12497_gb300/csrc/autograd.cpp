// The autograd nodes of autograd.py in C++: H u with H^T db, and Mhat(s, s') u with
// Mhat(s, s')^T dr and its velocity gradient. Each pass is one or two calls into the C ABI.
//
// Why native: at the sizes of a training step (181 x 149 x 9: 60 us of kernels) the host bounds the
// step. Forward and backward of both operators with a loss gradient: 441 us with Python functions,
// whose five calls through the interpreter and ctypes cost 15 to 40 us each, 268 us so (of which the
// engine, the leaves and the gradient sum take about 230).
#include <torch/csrc/autograd/custom_function.h>
#include <torch/csrc/utils/pybind.h>
#include <torch/csrc/Exceptions.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>

#include "mof.h"

namespace py = pybind11;
using at::Tensor;
using torch::autograd::AutogradContext;
using torch::autograd::variable_list;

namespace {

// A reference to the Python problem, which owns the handle: read at every use, so that a problem
// closed between forward and backward is refused and not used. Given back under the GIL.
struct ProblemRef : torch::CustomClassHolder {
    PyObject *o;
    explicit ProblemRef(py::object p) : o(p.release().ptr()) {}
    ~ProblemRef() override {
        if (!Py_IsInitialized()) return;
        py::gil_scoped_acquire gil;
        Py_DECREF(o);
    }
    // the handle and the sizes
    struct View {
        mof_problem *handle;
        int64_t n, m, nv, flow;
        at::ScalarType type;
    };
    View view() const {
        py::gil_scoped_acquire gil;
        const py::handle p(o);
        View v{};
        const py::object h = p.attr("handle").attr("value");
        v.handle = h.is_none() ? nullptr : reinterpret_cast<mof_problem *>(h.cast<uintptr_t>());
        v.n = p.attr("n").cast<int64_t>();
        v.m = p.attr("m").cast<int64_t>();
        v.nv = p.attr("nv").cast<int64_t>();
        v.flow = v.nv;  // 2 (nt - 1) values per pixel, as the velocities
        v.type = p.attr("precision").cast<int>() == MOF_FP64 ? at::kDouble : at::kFloat;
        return v;
    }
};
using Ref = c10::intrusive_ptr<ProblemRef>;

// A Python exception as one that keeps its type on its way through autograd's threads.
[[noreturn]] void raise(const py::object &type, const py::tuple &args) {
    PyErr_SetObject(type.ptr(), type(*args).ptr());
    python_error e;
    e.persist();
    throw e;
}

void check(mof_status st) {
    if (st == MOF_OK) return;
    const std::string msg = mof_last_error();
    py::gil_scoped_acquire gil;
    raise(py::module_::import("paper_2501_12497_gb300.api").attr("MofError"), py::make_tuple((int)st, msg));
}

void *ptr(const ProblemRef::View &v, const Tensor &t, int64_t numel, const char *name) {
    const char *what = nullptr;
    std::string detail;
    if (!t.is_cuda()) {
        what = " must be a CUDA tensor";
    } else if (t.scalar_type() != v.type) {
        what = v.type == at::kDouble ? " must be torch.float64" : " must be torch.float32";
    } else if (t.numel() != numel) {
        what = " has ";
        detail = std::to_string(t.numel()) + " elements, expected " + std::to_string(numel);
    }
    if (what) {
        py::gil_scoped_acquire gil;
        raise(py::reinterpret_borrow<py::object>(PyExc_ValueError), py::make_tuple(name + std::string(what) + detail));
    }
    return t.data_ptr();
}

void *stream() { return c10::cuda::getCurrentCUDAStream().stream(); }
Tensor flat(const Tensor &t) { return t.contiguous().reshape({-1}); }
Ref problem_of(AutogradContext *ctx) {
    return c10::static_intrusive_pointer_cast<ProblemRef>(ctx->saved_data["p"].toCapsule());
}
void keep(AutogradContext *ctx, const Ref &p) {
    ctx->saved_data["p"] = c10::IValue::make_capsule(c10::static_intrusive_pointer_cast<torch::CustomClassHolder>(p));
}

struct Project : torch::autograd::Function<Project> {
    static Tensor forward(AutogradContext *ctx, const Tensor &u, const Ref &p) {
        keep(ctx, p);
        const auto v = p->view();
        Tensor b = at::empty({v.m}, u.options());
        const Tensor uf = flat(u);
        void *const pu = ptr(v, uf, v.n, "u"), *const pb = ptr(v, b, v.m, "b");
        check(mof_apply_A(v.handle, pu, pb, stream()));
        return b;
    }
    static variable_list backward(AutogradContext *ctx, variable_list g) {
        const auto v = problem_of(ctx)->view();
        const Tensor db = flat(g[0]);
        Tensor du = at::empty({v.n}, db.options());
        void *const pb = ptr(v, db, v.m, "b"), *const pu = ptr(v, du, v.n, "u");
        check(mof_apply_AT(v.handle, pb, pu, stream()));
        return {du, Tensor()};
    }
};

struct FlowResidual : torch::autograd::Function<FlowResidual> {
    static Tensor forward(AutogradContext *ctx, const Tensor &u0, const Tensor &s0, const Tensor &sr0, const Ref &p) {
        keep(ctx, p);
        const auto v = p->view();
        const Tensor u = flat(u0), s = flat(s0), sr = flat(sr0);
        ctx->save_for_backward({u, s, sr});
        Tensor r = at::empty({v.flow}, u.options());
        void *const pu = ptr(v, u, v.n, "u"), *const ps = ptr(v, s, v.nv, "s"), *const psr = ptr(v, sr, v.nv, "sr"),
                   *const pr = ptr(v, r, v.flow, "r");
        check(mof_apply_flow(v.handle, pu, ps, psr, pr, stream()));
        return r;
    }
    static variable_list backward(AutogradContext *ctx, variable_list g) {
        const auto v = problem_of(ctx)->view();
        const auto saved = ctx->get_saved_variables();
        const Tensor &u = saved[0], &s = saved[1], &sr = saved[2], dr = flat(g[0]);
        Tensor du, gs, gsr;
        void *const pu = ptr(v, u, v.n, "u"), *const ps = ptr(v, s, v.nv, "s"), *const psr = ptr(v, sr, v.nv, "sr"),
                   *const pr = ptr(v, dr, v.flow, "r");
        if (ctx->needs_input_grad(0)) {
            du = at::empty_like(u);
            check(mof_apply_flowT(v.handle, pr, ps, psr, du.data_ptr(), stream()));
        }
        if (ctx->needs_input_grad(1) || ctx->needs_input_grad(2)) {
            gs = at::empty_like(s);
            gsr = at::empty_like(sr);
            check(mof_apply_flow_ds(v.handle, pu, ps, psr, pr, gs.data_ptr(), gsr.data_ptr(), stream()));
        }
        return {du, gs, gsr, Tensor()};
    }
};

Tensor project(py::object p, const Tensor &u) {
    const Ref ref = c10::make_intrusive<ProblemRef>(std::move(p));
    py::gil_scoped_release no_gil;
    return Project::apply(u, ref);
}
Tensor flow_residual(py::object p, const Tensor &u, const Tensor &s, const Tensor &sr) {
    const Ref ref = c10::make_intrusive<ProblemRef>(std::move(p));
    py::gil_scoped_release no_gil;
    return FlowResidual::apply(u, s, sr, ref);
}

}  // namespace

PYBIND11_MODULE(_autograd, m) {
    m.def("project", torch::wrap_pybind_function(project));
    m.def("flow_residual", torch::wrap_pybind_function(flow_residual));
}
