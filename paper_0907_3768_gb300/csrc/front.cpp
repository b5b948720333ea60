// Native half of the Python front end: the argument checks, the output tensors
// and the call of dust_solve / dust_solve_mass in one step.
//
// A solve of a few cells takes the GPU 15 to 25 us.  In Python its host side
// took 31 us: 6 us are the C call with its two launches, the rest four tensor
// allocations, a slice and a stream look-up, each of them short alone (1 to 2
// us) but two to three times that between launches, when its code has left the
// caches.  Here the whole call takes 20 us (1024 cells x 64 x 16, one call after another).
//
// The calls return None where an argument is not what they take (wrong shape,
// type or device): api.py then goes its own way and reports what is wrong.
#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/utils/pybind.h>

#include "../../include/dust.h"

namespace py = pybind11;

namespace {

using SolveFn = int (*)(dust_ctx *, int64_t, const float *, int64_t, const float *, float *, float *, double *,
                        uint8_t *, void *);

struct Outputs {
    at::Tensor T, L_buf, L, resid, flags;
};

Outputs alloc(int64_t C, int64_t G, int64_t K, int64_t ld, int device, bool want_L, bool want_resid, bool want_flags) {
    const auto opt = at::TensorOptions().device(at::kCUDA, device);
    Outputs o;
    o.T = at::empty({C, G}, opt.dtype(at::kFloat));
    if (want_L) {
        o.L_buf = at::empty({C, ld}, opt.dtype(at::kFloat));
        o.L = o.L_buf.slice(1, 0, K);
    }
    if (want_resid) o.resid = at::empty({C}, opt.dtype(at::kDouble));
    if (want_flags) o.flags = at::empty({C, G}, opt.dtype(at::kByte));
    return o;
}

py::dict as_dict(const Outputs &o) {
    auto or_none = [](const at::Tensor &t) -> py::object { return t.defined() ? py::cast(t) : py::none(); };
    py::dict d;
    d["T"] = o.T;
    d["L_buf"] = or_none(o.L_buf);
    d["L"] = or_none(o.L);
    d["resid"] = or_none(o.resid);
    d["flags"] = or_none(o.flags);
    return d;
}

py::dict alloc_outputs(int64_t C, int64_t G, int64_t K, int64_t ld, int device, bool want_L, bool want_resid,
                       bool want_flags) {
    return as_dict(alloc(C, G, K, ld, device, want_L, want_resid, want_flags));
}

// fn: address of dust_solve (n [C, G]) or dust_solve_mass (n [C], mass = true); ctx: the
// context's handle.  New outputs on the current stream of `device`; returns (outputs, status).
py::object solve(uintptr_t fn, uintptr_t ctx, int64_t G, int64_t K, int device, const at::Tensor &J, const at::Tensor &n,
                 bool mass, bool want_L, bool want_resid, bool want_flags) {
    if (!J.is_cuda() || !n.is_cuda() || J.scalar_type() != at::kFloat || n.scalar_type() != at::kFloat || J.dim() != 2 ||
        J.size(1) != K || J.stride(1) != 1 || (!mass && J.stride(0) < K) || !n.is_contiguous())
        return py::none();
    const int64_t C = J.size(0), ld = J.stride(0);
    if (mass ? (n.dim() != 1 || n.size(0) != C) : (n.dim() != 2 || n.size(0) != C || n.size(1) != G)) return py::none();
    const Outputs o = alloc(C, G, K, ld, device, want_L, want_resid, want_flags);
    const float *Jp = J.const_data_ptr<float>(), *np = n.const_data_ptr<float>();
    float *Tp = o.T.mutable_data_ptr<float>(), *Lp = want_L ? o.L_buf.mutable_data_ptr<float>() : nullptr;
    double *rp = want_resid ? o.resid.mutable_data_ptr<double>() : nullptr;
    uint8_t *fp = want_flags ? o.flags.mutable_data_ptr<uint8_t>() : nullptr;
    void *st = c10::cuda::getCurrentCUDAStream((c10::DeviceIndex)device).stream();
    int rc = 0;
    {
        py::gil_scoped_release free_;
        rc = reinterpret_cast<SolveFn>(fn)(reinterpret_cast<dust_ctx *>(ctx), C, Jp, ld, np, Tp, Lp, rp, fp, st);
    }
    return py::make_tuple(as_dict(o), rc);
}

}  // namespace

PYBIND11_MODULE(_front, m) {
    m.def("alloc_outputs", &alloc_outputs);
    m.def("solve", &solve);
}
