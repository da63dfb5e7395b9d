// PyTorch side of the hot calls: the autograd functions of the DPSR layer, the
// grid lookup, the Chamfer distance and the mesh points as C++ nodes over the
// C ABI of dpsr.h. They do what the Python classes of the same purpose do
// (dpsr.py, loop.py, optimize.py, mesh.py) for the inputs that a program
// passes: plain dense FP32 CUDA tensors. For anything else (another type,
// layout or device, a tensor subclass, tracing, functorch, forward-mode AD, a
// torch function or dispatch mode) an entry returns None, and the Python class
// answers, with its checks and its errors.
//
// Why: with 20 to 130 us of kernels a call, the Python forward and backward
// and their argument handling took longer than the GPU.
//
// The interpreter lock is held to look at the arguments and at the plan's
// attributes, and let go for the calls themselves: a first solve is tuned, a
// plan grows its workspace and an extraction reads its count back, and each of
// these waits for everything queued on the stream.
#include <ATen/cuda/CUDAContext.h>
#include <c10/core/impl/LocalDispatchKeySet.h>
#include <c10/core/impl/TorchDispatchModeTLS.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/custom_function.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/jit/frontend/tracer.h>
#include <torch/csrc/utils/pybind.h>

#include "dpsr.h"

namespace py = pybind11;
using at::Tensor;
using torch::autograd::AutogradContext;
using torch::autograd::variable_list;

namespace {

py::object* g_error = nullptr;  // libdpsr.DPSRError(code, what); never freed: the module lives as long as the process

// Raise DPSRError from a thread that may not hold the interpreter lock.
void check(int rc, const char* what) {
  if (rc == DPSR_OK) return;
  py::gil_scoped_acquire gil;
  py::object e = (*g_error)(rc, what);
  PyErr_SetObject(g_error->ptr(), e.ptr());
  python_error err;
  err.persist();
  throw err;
}

// What a layer's node keeps: the plan, held (the node may die on any thread),
// and the forward that it belongs to.
struct LayerState : torch::CustomClassHolder {
  PyObject* plan;
  int64_t generation = 0, n, r;
  LayerState(PyObject* p, int64_t n_, int64_t r_) : plan(p), n(n_), r(r_) { Py_INCREF(plan); }
  ~LayerState() override {
    if (!Py_IsInitialized()) return;
    py::gil_scoped_acquire gil;
    Py_DECREF(plan);
  }
};

// Nothing that looks at operators from outside is active on this thread.
bool quiet() {
  return !torch::jit::tracer::isTracing() && !at::impl::torch_function_mode_enabled() &&
         !c10::impl::dispatch_mode_enabled() &&
         !c10::impl::tls_is_dispatch_key_included(c10::DispatchKey::FuncTorchDynamicLayerFrontMode);
}

// The tensor behind `o` if it is a plain dense contiguous FP32 CUDA tensor.
const Tensor* plain(const py::handle& o) {
  if (!THPVariable_CheckExact(o.ptr())) return nullptr;
  const Tensor& t = THPVariable_Unpack(o.ptr());
  if (!t.defined()) return nullptr;
  const auto ks = t.key_set();  // first: wrappers answer little else
  if (ks.has(c10::DispatchKey::Python) || ks.has(c10::DispatchKey::FuncTorchBatched) ||
      ks.has(c10::DispatchKey::FuncTorchGradWrapper))
    return nullptr;
  if (!t.is_cuda() || t.scalar_type() != at::kFloat || t.layout() != at::kStrided || !t.has_storage() ||
      !t.is_contiguous() || t.is_neg() || t._fw_grad(0).defined())
    return nullptr;
  return &t;
}

bool points3(const Tensor& t) { return t.dim() == 2 && t.size(1) == 3; }
bool cube(const Tensor& t) { return t.dim() == 3 && t.size(0) == t.size(1) && t.size(1) == t.size(2); }
bool here(const Tensor& t) { return t.get_device() == c10::cuda::current_device(); }
void* stream(const Tensor& t) { return (void*)at::cuda::getCurrentCUDAStream(t.get_device()).stream(); }
const float* ro(const Tensor& t) { return t.const_data_ptr<float>(); }
float* rw(const Tensor& t) { return t.mutable_data_ptr<float>(); }

// Gradients arrive as autograd hands them over: dense ones are made contiguous FP32 here.
Tensor dense(const Tensor& g) {
  TORCH_CHECK_TYPE(g.is_cuda() && g.scalar_type() == at::kFloat, "the incoming gradient must be a float32 CUDA tensor");
  return g.contiguous();
}

// The result of `fn` for Python; fn runs without the interpreter lock.
template <class F>
py::object unlocked(const F& fn) {
  auto v = [&] {
    py::gil_scoped_release free;
    return fn();
  }();
  return py::cast(v);
}

// ---------------------------------------------------------------------------
// chi = DPSR(points, normals)
// ---------------------------------------------------------------------------
dpsr_plan handle_of(PyObject* plan) {  // with the interpreter lock; NULL after close()
  py::object h = py::reinterpret_borrow<py::object>(plan).attr("handle");
  return h.is_none() ? nullptr : (dpsr_plan)h.cast<uintptr_t>();
}

// The tensor without its graph (a leaf has none).
py::object bare(const Tensor& t) { return py::cast(t.is_leaf() ? t : t.variable_data()); }

// chi of a forward pass; without the interpreter lock.
Tensor solve(dpsr_plan h, const Tensor& points, const Tensor& normals, int64_t r) {
  Tensor chi = at::empty({r, r, r}, points.options());
  check(dpsr_plan_set_stream(h, stream(points)), "dpsr_plan_set_stream");
  check(dpsr_forward(h, ro(points), ro(normals), points.size(0), rw(chi)), "dpsr_forward");
  return chi;
}

// A forward pass has run: the backward reads its buffers, so the plan keeps
// them alive, and the count of forwards tells a backward whether they are still
// its own.
int64_t keep(py::handle plan, py::object points, py::object normals, py::object chi) {
  plan.attr("_saved") = py::make_tuple(std::move(points), std::move(normals), std::move(chi));
  const int64_t gen = plan.attr("generation").cast<int64_t>() + 1;
  plan.attr("generation") = gen;
  return gen;
}

struct Layer : torch::autograd::Function<Layer> {
  static Tensor forward(AutogradContext* ctx, const Tensor& points, const Tensor& normals,
                        const c10::intrusive_ptr<LayerState>& st, dpsr_plan h) {
    ctx->saved_data["state"] = c10::IValue::make_capsule(st);
    return solve(h, points, normals, st->r);
  }
  static variable_list backward(AutogradContext* ctx, variable_list grads) {
    const auto held = ctx->saved_data["state"].toCapsule();
    const LayerState& st = *static_cast<const LayerState*>(held.get());
    Tensor g = dense(grads[0]);
    TORCH_CHECK_VALUE(cube(g) && g.size(0) == st.r, "dchi has another shape than chi");
    dpsr_plan h = nullptr;
    {
      py::gil_scoped_acquire gil;
      TORCH_CHECK(py::handle(st.plan).attr("generation").cast<int64_t>() == st.generation,
                  "the plan ran another forward pass since this one: one pending backward per plan (use one Plan "
                  "per graph node)");
      h = handle_of(st.plan);
    }
    Tensor dp = at::empty({st.n, 3}, g.options()), dn = at::empty({st.n, 3}, g.options());
    check(dpsr_plan_set_stream(h, stream(g)), "dpsr_plan_set_stream");
    check(dpsr_backward(h, ro(g), rw(dp), rw(dn)), "dpsr_backward");
    return {dp, dn, Tensor(), Tensor()};
  }
};

py::object layer(py::handle points, py::handle normals, py::handle plan) {
  const Tensor *p = plain(points), *n = plain(normals);
  if (!p || !n || !points3(*p) || p->sizes() != n->sizes() || p->device() != n->device() || p->size(0) < 1 || !quiet())
    return py::none();
  if (plan.attr("handle").is_none() || plan.attr("_index").cast<int64_t>() != p->get_device() || !here(*p))
    return py::none();
  const Tensor a = *p, b = *n;
  const dpsr_plan h = handle_of(plan.ptr());
  auto st = c10::make_intrusive<LayerState>(plan.ptr(), a.size(0), plan.attr("r").cast<int64_t>());
  Tensor chi;
  {
    py::gil_scoped_release free;
    chi = Layer::apply(a, b, st, h);
  }
  st->generation = keep(plan, bare(a), bare(b), py::cast(chi.variable_data()));
  return py::cast(chi);
}

// Plan.forward into a new grid.
py::object plan_forward(py::handle plan, py::handle points, py::handle normals) {
  const Tensor *p = plain(points), *n = plain(normals);
  if (!p || !n || !points3(*p) || p->sizes() != n->sizes() || p->device() != n->device() || p->size(0) < 1 ||
      !quiet())
    return py::none();
  if (plan.attr("handle").is_none() || plan.attr("_index").cast<int64_t>() != p->get_device() || !here(*p))
    return py::none();
  const Tensor a = *p, b = *n;
  const dpsr_plan h = handle_of(plan.ptr());
  const int64_t r = plan.attr("r").cast<int64_t>();
  Tensor chi;
  {
    py::gil_scoped_release free;
    chi = solve(h, a, b, r);
  }
  py::object out = py::cast(chi);
  keep(plan, py::reinterpret_borrow<py::object>(points), py::reinterpret_borrow<py::object>(normals), out);
  return out;
}

// ---------------------------------------------------------------------------
// chi(q): trilinear lookup, and its adjoint
// ---------------------------------------------------------------------------
struct Lookup : torch::autograd::Function<Lookup> {
  static Tensor forward(AutogradContext* ctx, const Tensor& chi, const Tensor& q) {
    Tensor out = at::empty({q.size(0)}, chi.options());
    check(dpsr_grid_sample(ro(chi), (int)chi.size(0), ro(q), q.size(0), rw(out), stream(chi)), "dpsr_grid_sample");
    ctx->save_for_backward({q});
    ctx->saved_data["r"] = chi.size(0);
    return out;
  }
  static variable_list backward(AutogradContext* ctx, variable_list grads) {
    const Tensor q = ctx->get_saved_variables()[0];
    const int64_t r = ctx->saved_data["r"].toInt();
    Tensor g = dense(grads[0]);
    Tensor d = at::empty({r, r, r}, g.options());
    check(dpsr_grid_splat(rw(d), (int)r, ro(q), ro(g), q.size(0), 0, stream(g)), "dpsr_grid_splat");
    return {d, Tensor()};
  }
};

py::object grid_sample(py::handle chi, py::handle q) {
  const Tensor *c = plain(chi), *p = plain(q);
  if (!c || !p || !cube(*c) || !points3(*p) || c->device() != p->device() || p->size(0) < 1 || !here(*c) || !quiet())
    return py::none();
  return unlocked([a = *c, b = *p] { return Lookup::apply(a, b); });
}

// ---------------------------------------------------------------------------
// Chamfer distance
// ---------------------------------------------------------------------------
struct Chamfer : torch::autograd::Function<Chamfer> {
  static Tensor forward(AutogradContext* ctx, const Tensor& a, const Tensor& b) {
    const int64_t na = a.size(0), nb = b.size(0);
    const size_t bytes = dpsr_chamfer_ws_bytes(na, nb);
    // one scratch block: the FP64 loss, then the trees
    Tensor ws = at::empty({(int64_t)bytes + 256}, a.options().dtype(at::kByte));
    Tensor grad = at::empty({na, 3}, a.options()), loss = at::empty({}, a.options());
    char* w = (char*)ws.mutable_data_ptr();
    check(dpsr_chamfer_tree(ro(a), na, ro(b), nb, w + 256, bytes, rw(grad), (double*)w, rw(loss), stream(a)),
          "dpsr_chamfer_tree");
    ctx->save_for_backward({grad});
    return loss;
  }
  static variable_list backward(AutogradContext* ctx, variable_list grads) {
    return {ctx->get_saved_variables()[0].mul(grads[0]), Tensor()};
  }
};

py::object chamfer(py::handle a, py::handle b) {
  const Tensor *p = plain(a), *q = plain(b);
  if (!p || !q || !points3(*p) || !points3(*q) || p->device() != q->device() || p->size(0) < 1 || q->size(0) < 1 ||
      !here(*p) || !quiet())
    return py::none();
  return unlocked([a = *p, b = *q] { return Chamfer::apply(a, b); });
}

// ---------------------------------------------------------------------------
// Mesh: triangles, points drawn on them, and Eq. 6 back to the grid
// ---------------------------------------------------------------------------
std::pair<Tensor, Tensor> extract_raw(const Tensor& chi, double level) {
  const int64_t r = chi.size(0);
  Tensor count = at::empty({1}, chi.options().dtype(at::kLong));
  int64_t cap = std::max<int64_t>(1024, 24 * r * r);
  for (int it = 0; it < 2; ++it) {
    Tensor tris = at::empty({cap, 3, 3}, chi.options()), nrm = at::empty({cap, 3}, chi.options());
    check(dpsr_mesh_extract(ro(chi), (int)r, (float)level, rw(tris), rw(nrm), cap,
                            (unsigned long long*)count.mutable_data_ptr<int64_t>(), stream(chi)),
          "dpsr_mesh_extract");
    const int64_t n = count.item<int64_t>();
    if (n <= cap) return {tris.narrow(0, 0, n), nrm.narrow(0, 0, n)};
    cap = n;
  }
  TORCH_CHECK(false, "mesh extraction did not converge");
}

std::pair<Tensor, Tensor> sample_raw(const Tensor& tris, const Tensor& nrm, int64_t m, uint64_t seed) {
  const int64_t t = tris.size(0);
  Tensor ws = at::empty({t + (t + 1023) / 1024 + 1}, tris.options().dtype(at::kDouble));
  Tensor p = at::empty({m, 3}, tris.options()), n = at::empty({m, 3}, tris.options());
  check(dpsr_mesh_sample(ro(tris), ro(nrm), t, m, seed, ws.mutable_data_ptr<double>(), rw(p), rw(n), stream(tris)),
        "dpsr_mesh_sample");
  return {p, n};
}

struct MeshPoints : torch::autograd::Function<MeshPoints> {
  static variable_list forward(AutogradContext* ctx, const Tensor& chi, double level, int64_t samples, uint64_t seed) {
    auto [tris, nrm] = extract_raw(chi, level);
    Tensor p, n;
    if (samples) std::tie(p, n) = sample_raw(tris, nrm, samples, seed);
    else p = tris.mean(1), n = nrm;
    ctx->save_for_backward({p, n});
    ctx->saved_data["r"] = chi.size(0);
    ctx->mark_non_differentiable({n});
    return {p, n};
  }
  static variable_list backward(AutogradContext* ctx, variable_list grads) {
    const auto saved = ctx->get_saved_variables();
    const Tensor p = saved[0].contiguous(), n = saved[1].contiguous(), g = dense(grads[0]);
    const int64_t r = ctx->saved_data["r"].toInt();
    Tensor d = at::empty({r, r, r}, g.options());
    check(dpsr_mesh_surrogate_splat(rw(d), (int)r, ro(p), ro(n), ro(g), p.size(0), 0, stream(g)),
          "dpsr_mesh_surrogate_splat");
    return {d, Tensor(), Tensor(), Tensor()};
  }
};

py::object mesh_points(py::handle chi, double level, int64_t samples, uint64_t seed) {
  const Tensor* c = plain(chi);
  if (!c || !cube(*c) || !here(*c) || samples < 0 || !quiet()) return py::none();
  return unlocked([a = *c, level, samples, seed] {
    const variable_list v = MeshPoints::apply(a, level, samples, seed);
    return std::make_pair(v[0], v[1]);
  });
}

py::object extract(py::handle chi, double level) {
  const Tensor* c = plain(chi);
  if (!c || !cube(*c) || !here(*c) || !quiet()) return py::none();
  return unlocked([a = *c, level] { return extract_raw(a, level); });
}

py::object sample(py::handle tris, py::handle nrm, int64_t m, uint64_t seed) {
  const Tensor *t = plain(tris), *n = plain(nrm);
  if (!t || !n || t->dim() != 3 || t->size(1) != 3 || t->size(2) != 3 || !points3(*n) || n->size(0) != t->size(0) ||
      t->size(0) < 1 || m < 1 || t->device() != n->device() || !here(*t) ||
      !quiet())
    return py::none();
  return unlocked([a = *t, b = *n, m, seed] { return sample_raw(a, b, m, seed); });
}

}  // namespace

PYBIND11_MODULE(_dpsr_torch, m) {
  m.def("init", [](py::object error) { if (!g_error) g_error = new py::object(std::move(error)); });
  m.def("layer", &layer);
  m.def("plan_forward", &plan_forward);
  m.def("grid_sample", &grid_sample);
  m.def("chamfer", &chamfer);
  m.def("mesh_points", &mesh_points);
  m.def("extract", &extract);
  m.def("sample", &sample);
}
