// The autograd nodes of the torch front end in C++: the backward halves of rasterize() and of
// l1_dssim_loss().  The autograd engine runs them on its device thread, where nodes written in Python cost
// a hand-over of the interpreter lock each way besides their own marshalling: 430 of the 615 us
// of host time of a 10k-Gaussian training step, which the GPU's 340 us waited for.
//
// The forward halves stay in Python (workspace growth, counters, checks); what they computed is handed
// to a node here with copies of the call's camera and options.  The C ABI is reached through the addresses
// that the Python binding loaded, so that one copy of the library serves both.
#include <ATen/ATen.h>
#include <c10/cuda/CUDAStream.h>
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/custom_function.h>
#include <torch/csrc/utils/pybind.h>

#include <cstring>
#include <memory>
#include <stdexcept>
#include <string>

#include "vgrast.h"

// What this file was compiled against: the build compares it with what is installed.
__attribute__((used)) extern const char vg_front_key[] = VG_FRONT_KEY;

namespace {

using torch::autograd::AutogradContext;
using torch::autograd::Function;
using torch::autograd::variable_list;

decltype(&vg_rasterize_forward) g_rasterize_forward = nullptr;
decltype(&vg_rasterize_backward) g_rasterize_backward = nullptr;
decltype(&vg_loss_l1_dssim_grad) g_loss_grad = nullptr;

// Raises the binding's VGError, as a call from Python would.
[[noreturn]] void raise_status(vg_status status, const char* where) {
  pybind11::gil_scoped_acquire gil;
  pybind11::object type = pybind11::module_::import("paper_2402_17427_gb300.binding").attr("VGError");
  pybind11::object value = type(static_cast<int>(status), where);
  PyErr_SetObject(type.ptr(), value.ptr());
  python_error e;
  e.persist();
  throw e;
}

vg_stream current_stream(const at::Tensor& t) {
  return reinterpret_cast<vg_stream>(c10::cuda::getCurrentCUDAStream(t.get_device()).stream());
}

template <typename T>
T from_bytes(const std::string& s) {
  if (s.size() != sizeof(T)) throw std::invalid_argument("structure of another size");
  T v;
  std::memcpy(&v, s.data(), sizeof(T));
  return v;
}

// Forward calls made on one workspace, shared by its owner and the nodes that read the workspace later.
struct Uses {
  std::shared_ptr<int64_t> n = std::make_shared<int64_t>(0);
};

// What a render's backward needs besides the saved tensors.
struct RenderCall : torch::CustomClassHolder {
  vg_camera cam;
  vg_raster_opts opts;
  int32_t degree = 0;
  int64_t capacity = 0;
  at::Tensor rgb, T, last, workspace;
  std::shared_ptr<int64_t> uses;      // null: the workspace is this render's alone
  int64_t use = 0;
};

struct RenderNode : Function<RenderNode> {
  static at::Tensor forward(AutogradContext* ctx, const at::Tensor& means, const at::Tensor& log_scales,
                            const at::Tensor& quats, const at::Tensor& logits, const at::Tensor& sh,
                            c10::intrusive_ptr<RenderCall> call) {
    ctx->save_for_backward({means, log_scales, quats, logits, sh, call->T, call->last});
    at::Tensor rgb = std::move(call->rgb);
    call->T.reset();
    call->last.reset();
    ctx->saved_data["call"] = c10::IValue::make_capsule(std::move(call));
    return rgb;
  }

  static variable_list backward(AutogradContext* ctx, variable_list grad_outputs) {
    const variable_list s = ctx->get_saved_variables();
    const auto call = c10::static_intrusive_pointer_cast<RenderCall>(ctx->saved_data["call"].toCapsule());
    const at::Tensor dL = grad_outputs[0].contiguous();
    // what saved-tensor hooks hand back may be anything
    for (int k = 0; k < 5; ++k)
      TORCH_CHECK_VALUE(s[k].is_cuda() && s[k].scalar_type() == at::kFloat && s[k].is_contiguous(),
                        "Gaussian parameters must be contiguous float32 CUDA tensors");
    for (int k = 5; k < 7; ++k)
      TORCH_CHECK_VALUE(s[k].is_cuda() && s[k].is_contiguous() && s[k].element_size() == 4,
                        "the saved transmittance and last indices must be contiguous CUDA tensors of 4-byte entries");
    variable_list g(6);                                    // the call itself has no gradient
    for (int k = 0; k < 5; ++k) g[k] = at::empty_like(s[k]);
    auto ptr = [](const at::Tensor& t) { return static_cast<float*>(t.data_ptr()); };
    vg_gaussians p{};
    p.means = ptr(s[0]);
    p.log_scales = ptr(s[1]);
    p.quats = ptr(s[2]);
    p.opacity_logits = ptr(s[3]);
    p.sh = ptr(s[4]);
    p.n = s[0].size(0);
    p.sh_degree = call->degree;
    at::Tensor workspace = call->workspace;
    if (call->uses && *call->uses != call->use) {
      // Another forward has overwritten the workspace (two renders of one Rasterizer before the first one's
      // backward): its lists are another render's, perhaps in another layout.  This one's are made again, in a
      // workspace of their own, since the later render's backward still needs the shared one.
      workspace = at::empty_like(call->workspace);
      const at::Tensor T = at::empty_like(s[5]), last = at::empty_like(s[6]);
      const at::Tensor rgb = at::empty_like(dL), counters = at::empty({VG_CNT_LEN}, dL.options().dtype(at::kLong));
      const vg_status again = g_rasterize_forward(
          &p, &call->cam, &call->opts, workspace.data_ptr(), static_cast<size_t>(workspace.numel()), call->capacity,
          ptr(rgb), ptr(T), static_cast<uint32_t*>(last.data_ptr()), static_cast<int64_t*>(counters.data_ptr()),
          current_stream(dL));
      if (again != VG_OK) raise_status(again, "vg_rasterize_forward");
    }
    const vg_status status = g_rasterize_backward(
        &p, &call->cam, &call->opts, workspace.data_ptr(), static_cast<size_t>(workspace.numel()),
        call->capacity, ptr(s[5]), static_cast<const uint32_t*>(s[6].data_ptr()), ptr(dL), ptr(g[0]), ptr(g[1]),
        ptr(g[2]), ptr(g[3]), ptr(g[4]), nullptr, current_stream(dL));
    if (status != VG_OK) raise_status(status, "vg_rasterize_backward");
    return g;
  }
};

at::Tensor attach_render(const at::Tensor& means, const at::Tensor& log_scales, const at::Tensor& quats,
                         const at::Tensor& logits, const at::Tensor& sh, const at::Tensor& rgb, const at::Tensor& T,
                         const at::Tensor& last, const at::Tensor& workspace, int64_t capacity, int32_t degree,
                         const pybind11::bytes& cam, const pybind11::bytes& opts, const Uses* uses) {
  auto call = c10::make_intrusive<RenderCall>();
  call->cam = from_bytes<vg_camera>(cam);
  call->opts = from_bytes<vg_raster_opts>(opts);
  call->degree = degree;
  call->capacity = capacity;
  call->rgb = rgb;
  call->T = T;
  call->last = last;
  call->workspace = workspace;
  if (uses) {
    call->uses = uses->n;
    call->use = *uses->n;
  }
  return RenderNode::apply(means, log_scales, quats, logits, sh, std::move(call));
}

struct LossCall : torch::CustomClassHolder {
  int32_t width = 0, height = 0;
  float lambda = 0.f;
  at::Tensor loss, img, target, workspace;
  std::shared_ptr<int64_t> uses;
  int64_t use = 0;
};

struct LossNode : Function<LossNode> {
  // img and target are the graph's inputs; the call holds what the pass read (contiguous copies where
  // they were not).  The target gets no gradient, as with a node that returns None for it.
  static at::Tensor forward(AutogradContext* ctx, const at::Tensor& /*img*/, const at::Tensor& /*target*/,
                            c10::intrusive_ptr<LossCall> call) {
    ctx->save_for_backward({call->img, call->target});
    at::Tensor loss = std::move(call->loss);
    call->img.reset();
    call->target.reset();
    ctx->saved_data["call"] = c10::IValue::make_capsule(std::move(call));
    return loss;
  }

  static variable_list backward(AutogradContext* ctx, variable_list grad_outputs) {
    const variable_list s = ctx->get_saved_variables();
    const auto call = c10::static_intrusive_pointer_cast<LossCall>(ctx->saved_data["call"].toCapsule());
    if (*call->uses != call->use)
      throw std::runtime_error("the loss workspace was used by another forward before this backward");
    for (const at::Tensor& t : s)
      TORCH_CHECK_VALUE(t.is_cuda() && t.scalar_type() == at::kFloat && t.is_contiguous(),
                        "the saved images must be contiguous float32 CUDA tensors");
    const at::Tensor scale = grad_outputs[0].detach().to(at::kFloat).contiguous();
    at::Tensor grad = at::empty_like(s[0]);
    const vg_status status = g_loss_grad(
        static_cast<const float*>(s[0].data_ptr()), static_cast<const float*>(s[1].data_ptr()), call->width,
        call->height, call->lambda, call->workspace.data_ptr(), static_cast<size_t>(call->workspace.numel()),
        static_cast<const float*>(scale.data_ptr()), static_cast<float*>(grad.data_ptr()), current_stream(s[0]));
    if (status != VG_OK) raise_status(status, "vg_loss_l1_dssim_grad");
    return {grad, at::Tensor(), at::Tensor()};
  }
};

at::Tensor attach_loss(const at::Tensor& img, const at::Tensor& target, const at::Tensor& img_c, const at::Tensor& target_c,
                       const at::Tensor& loss, const at::Tensor& workspace, const Uses& uses, int32_t width,
                       int32_t height, double lambda) {
  auto call = c10::make_intrusive<LossCall>();
  call->width = width;
  call->height = height;
  call->lambda = static_cast<float>(lambda);
  call->loss = loss;
  call->img = img_c;
  call->target = target_c;
  call->workspace = workspace;
  call->uses = uses.n;
  call->use = *uses.n;
  return LossNode::apply(img, target, std::move(call));
}

}  // namespace

PYBIND11_MODULE(_vgfront, m) {
  m.def("init", [](uintptr_t rasterize_forward, uintptr_t rasterize_backward, uintptr_t loss_grad) {
    g_rasterize_forward = reinterpret_cast<decltype(g_rasterize_forward)>(rasterize_forward);
    g_rasterize_backward = reinterpret_cast<decltype(g_rasterize_backward)>(rasterize_backward);
    g_loss_grad = reinterpret_cast<decltype(g_loss_grad)>(loss_grad);
  });
  pybind11::class_<Uses>(m, "Uses")
      .def(pybind11::init<>())
      .def(pybind11::pickle([](const Uses& u) { return *u.n; },        // a copy of a workspace counts by itself
                            [](int64_t n) {
                              Uses u;
                              *u.n = n;
                              return u;
                            }))
      .def("bump", [](Uses& u) { ++*u.n; })
      .def_property_readonly("value", [](const Uses& u) { return *u.n; });
  using pybind11::arg;
  m.def("attach_render", &attach_render, arg("means"), arg("log_scales"), arg("quats"), arg("logits"), arg("sh"),
        arg("rgb"), arg("T"), arg("last"), arg("workspace"), arg("capacity"), arg("degree"), arg("cam"), arg("opts"),
        arg("uses") = nullptr);
  m.def("attach_loss", &attach_loss);
}
