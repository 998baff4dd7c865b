// The differentiable operator as a native autograd function over the C ABI (include/sna.h).  Nothing is computed here.
//
// Why native: a small training step is bound by the host.  32x64, N = 1, C = 16 takes 30 us on the GPU; written in Python, its
// forward and backward calls (argument checks, allocations, foreign-function calls, and the interpreter's lock in the autograd
// engine's thread) took 123 us.
#include <torch/extension.h>

#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>

#include <atomic>

#include "../../include/sna.h"

namespace {

using torch::autograd::AutogradContext;
using torch::autograd::Variable;
using torch::autograd::variable_list;

// Owner of an sna_plan_t: the Python plan and every graph recorded with it hold references.
struct Plan : torch::CustomClassHolder {
    std::atomic<sna_plan_t*> handle;
    const int64_t nlat_in, nlon_in, nlat_out, nlon_out;
    Plan(uintptr_t h, int64_t nlat_in, int64_t nlon_in, int64_t nlat_out, int64_t nlon_out)
        : handle(reinterpret_cast<sna_plan_t*>(h)), nlat_in(nlat_in), nlon_in(nlon_in), nlat_out(nlat_out), nlon_out(nlon_out) {}
    ~Plan() override { close(); }
    int close() {
        sna_plan_t* h = handle.exchange(nullptr);
        return h == nullptr ? SNA_OK : sna_plan_destroy(h);
    }
};

// Raises sna.SnaError: as Python's own exception, the only kind that the autograd engine hands on as it is.
void check(int status) {
    if (status == SNA_OK) return;
    py::gil_scoped_acquire gil;
    const py::object type = py::module_::import("paper_2505_11157_b200.sna").attr("SnaError");
    PyErr_SetObject(type.ptr(), type(status).ptr());
    python_error e;
    e.persist();
    throw e;
}

float* data(const at::Tensor& t) { return t.data_ptr<float>(); }
void* current_stream() { return c10::cuda::getCurrentCUDAStream().stream(); }

// Saved tensors come back through hooks (offloading, compression): the kernels read raw pointers, so anything but the tensor that was
// saved, or its equal, is refused here.
void check_saved(const at::Tensor& t, const char* name, at::IntArrayRef shape, const at::Tensor& dout) {
    TORCH_CHECK_VALUE(t.defined() && t.scalar_type() == at::kFloat, name, " must be float32");
    TORCH_CHECK_VALUE(t.sizes() == shape, name, " has shape ", t.sizes(), ", expected ", shape);
    TORCH_CHECK_VALUE(t.is_contiguous(), name, " must be contiguous");
    TORCH_CHECK_VALUE(t.is_cuda() && t.device() == dout.device(), name, " must be a CUDA tensor on the device of dout (", dout.device(), "), got ", t.device());
}

class Attention : public torch::autograd::Function<Attention> {
public:
    static at::Tensor forward(AutogradContext* ctx, const c10::intrusive_ptr<Plan>& plan, at::Tensor q, at::Tensor k, at::Tensor v) {
        q = q.contiguous(); k = k.contiguous(); v = v.contiguous();
        at::Tensor out = at::empty_like(q), lse = at::empty(q.sizes().slice(0, 4), q.options());
        check(sna_forward_ex(plan->handle, data(q), data(k), data(v), data(out), data(lse), (int)q.size(0), (int)q.size(1), (int)q.size(4), current_stream()));
        ctx->saved_data["plan"] = c10::IValue::make_capsule(plan);
        ctx->save_for_backward({q, k, v, out, lse});
        return out;
    }
    static variable_list backward(AutogradContext* ctx, variable_list grads) {
        const auto saved = ctx->get_saved_variables();
        const at::Tensor &q = saved[0], &k = saved[1], &v = saved[2], &out = saved[3], &lse = saved[4];
        const auto plan = c10::static_intrusive_pointer_cast<Plan>(ctx->saved_data["plan"].toCapsule());
        const at::Tensor dout = grads[0].contiguous().to(at::kFloat);
        const at::IntArrayRef on = dout.sizes();
        const int64_t in[5] = {on[0], on[1], plan->nlat_in, plan->nlon_in, on[4]};
        check_saved(q, "q", on, dout); check_saved(k, "k", in, dout); check_saved(v, "v", in, dout);
        check_saved(out, "out", on, dout); check_saved(lse, "lse", on.slice(0, 4), dout);
        const int B = (int)on[0], H = (int)on[1], C = (int)on[4];
        at::Tensor dq = at::empty_like(q), dk = at::empty_like(k), dv = at::empty_like(k);
        sna_plan_t* handle = plan->handle;
        const size_t bytes = sna_workspace_bytes(handle, B, H, C);
        at::Tensor workspace = at::empty({(int64_t)bytes}, q.options().dtype(at::kByte));
        check(sna_backward_ex(handle, data(q), data(k), data(v), data(dout), data(out), data(lse), data(dq), data(dk), data(dv),
                              workspace.data_ptr(), bytes, B, H, C, current_stream()));
        return {Variable(), dq, dk, dv};
    }
};

bool usable(const at::Tensor& t, at::IntArrayRef shape, const at::Tensor& q) {
    return t.is_cuda() && t.device() == q.device() && t.scalar_type() == at::kFloat && t.sizes() == shape;
}

// The output, or nothing if the arguments are not tensors that the plan takes (the caller finds out what is wrong).
std::optional<at::Tensor> attention(const c10::intrusive_ptr<Plan>& plan, const at::Tensor& q, const at::Tensor& k, const at::Tensor& v) {
    if (q.dim() != 5) return std::nullopt;
    const int64_t B = q.size(0), H = q.size(1), C = q.size(4);
    const int64_t in[5] = {B, H, plan->nlat_in, plan->nlon_in, C}, on[5] = {B, H, plan->nlat_out, plan->nlon_out, C};
    if (!usable(q, on, q) || !usable(k, in, q) || !usable(v, in, q)) return std::nullopt;
    return Attention::apply(plan, q, k, v);
}

}  // namespace

PYBIND11_MODULE(_sna_torch, m) {
    py::class_<Plan, c10::intrusive_ptr<Plan>>(m, "Plan")
        .def(py::init([](uintptr_t h, int64_t a, int64_t b, int64_t c, int64_t d) { return c10::make_intrusive<Plan>(h, a, b, c, d); }))
        .def("close", &Plan::close);
    m.def("attention", &attention, py::call_guard<py::gil_scoped_release>());
}
