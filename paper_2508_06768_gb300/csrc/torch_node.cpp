// The differentiable render of one pose as a native autograd node.
//
// A frame's device work is a few tens of microseconds, less than a Python
// autograd function, its argument conversions and the engine's hand-over of
// the interpreter lock to its backward thread take on the host.  This node
// makes the same C-ABI calls with the same buffers from C++: one pass of a 64 x
// 256 frame took 89 us forward and 357 us with the pose gradient through the
// Python function, 36 and 170 us through this one.
#include <torch/extension.h>

#include <c10/cuda/CUDAStream.h>

#include <cstring>
#include <string>
#include <vector>

#include "diffus.h"

namespace {

using torch::Tensor;
using torch::autograd::AutogradContext;
using torch::autograd::variable_list;

// What render() packs per call: spacing, origin, fan and parameters.
struct Call {
    double spacing[3], origin[3];
    diffus_fan fan;
    diffus_params prm;
};
static_assert(sizeof(Call) == 176 && sizeof(Call) % sizeof(int64_t) == 0, "binding.py packs this layout");

PyObject *g_error = nullptr;   // binding.DiffusError

void check(int rc, const char *what)
{
    if (rc == DIFFUS_OK) return;
    const std::string msg = std::string(what) + " failed: " + diffus_strerror(rc) + " (" + std::to_string(rc) + ")";
    pybind11::gil_scoped_acquire gil;
    PyErr_SetString(g_error ? g_error : PyExc_RuntimeError, msg.c_str());
    python_error e;
    e.persist();
    throw e;
}

diffus_volume_desc desc(const Tensor &vol, const Call &c)
{
    const auto s = vol.sizes();
    return {(int32_t)s[2], (int32_t)s[1], (int32_t)s[0], vol.scalar_type() == at::kFloat ? DIFFUS_F32 : DIFFUS_BF16,
            c.spacing[0], c.spacing[1], c.spacing[2], c.origin[0], c.origin[1], c.origin[2]};
}

Tensor workspace(const diffus_volume_desc &vd, const Call &c, int with_bwd, const Tensor &like)
{
    const size_t n = diffus_workspace_bytes(&vd, &c.fan, &c.prm, with_bwd);
    if (n == 0) {
        pybind11::gil_scoped_acquire gil;
        PyErr_SetString(g_error ? g_error : PyExc_RuntimeError, "invalid volume/fan/params for workspace sizing");
        python_error e;
        e.persist();
        throw e;
    }
    return at::empty({(int64_t)n}, like.options().dtype(at::kByte));
}

diffus_stream_t stream() { return (diffus_stream_t)c10::cuda::getCurrentCUDAStream().stream(); }

struct RenderNode : public torch::autograd::Function<RenderNode> {
    static variable_list forward(AutogradContext *ctx, const Tensor &volume, const Tensor &pose, const std::string &blob)
    {
        Call c;
        std::memcpy(&c, blob.data(), sizeof c);
        const Tensor vol = volume.detach().contiguous();
        const Tensor p = pose.detach().contiguous().to(at::kFloat);
        const diffus_volume_desc vd = desc(vol, c);
        const Tensor ws = workspace(vd, c, 0, vol);
        const Tensor img = at::empty({c.fan.n_rays, c.fan.n_samples}, vol.options().dtype(at::kFloat));
        const Tensor valid = at::empty({c.fan.n_rays}, vol.options().dtype(at::kInt));
        check(diffus_render_fwd(vol.data_ptr(), &vd, p.data_ptr<float>(), &c.fan, &c.prm, img.data_ptr<float>(),
                                valid.data_ptr<int>(), nullptr, ws.data_ptr(), (size_t)ws.numel(), stream()),
              "diffus_render_fwd");
        const int64_t want = (int64_t)volume.requires_grad() + 2 * (int64_t)pose.requires_grad();
        if (want == 0) return {img, valid};
        ctx->set_materialize_grads(false);   // valid has none: no zeros are made for it
        ctx->save_for_backward({vol, p});
        // as integers: compiled autograd reads what a node keeps and takes a
        // string only as UTF-8
        std::vector<int64_t> words(sizeof c / sizeof(int64_t));
        std::memcpy(words.data(), &c, sizeof c);
        ctx->saved_data["call"] = std::move(words);
        ctx->saved_data["want"] = want;
        return {img, valid};   // an integer output is not differentiable, and compiled autograd takes no such marks
    }

    static variable_list backward(AutogradContext *ctx, variable_list grads)
    {
        const int64_t want = ctx->saved_data["want"].toInt();
        const auto saved = ctx->get_saved_variables();
        const Tensor &vol = saved[0], &p = saved[1];
        Call c;
        const std::vector<int64_t> words = ctx->saved_data["call"].toIntVector();
        std::memcpy(&c, words.data(), sizeof c);
        const diffus_volume_desc vd = desc(vol, c);
        const Tensor g = grads[0].defined() ? grads[0].detach().contiguous().to(at::kFloat)
                                            : at::zeros({c.fan.n_rays, c.fan.n_samples}, vol.options().dtype(at::kFloat));
        Tensor gv, gp;
        if (want & 1) gv = at::empty(vol.sizes(), vol.options().dtype(at::kFloat));
        if (want & 2) gp = at::empty({6}, vol.options().dtype(at::kFloat));
        const Tensor ws = workspace(vd, c, 1, vol);
        check(diffus_render_bwd(vol.data_ptr(), &vd, p.data_ptr<float>(), &c.fan, &c.prm, g.data_ptr<float>(),
                                gv.defined() ? gv.data_ptr<float>() : nullptr,
                                gp.defined() ? gp.data_ptr<float>() : nullptr, nullptr, ws.data_ptr(),
                                (size_t)ws.numel(), stream()),
              "diffus_render_bwd");
        if (gv.defined() && vol.scalar_type() != at::kFloat) gv = gv.to(vol.scalar_type());
        return {gv, gp, Tensor()};
    }
};

pybind11::tuple render(const Tensor &volume, const Tensor &pose, const std::string &blob)
{
    if (blob.size() != sizeof(Call)) throw std::invalid_argument("packed call has the wrong size");
    variable_list out;
    try {
        pybind11::gil_scoped_release nogil;
        out = RenderNode::apply(volume, pose, blob);
    } catch (python_error &e) {
        e.restore();
        throw pybind11::error_already_set();
    }
    return pybind11::make_tuple(out[0], out[1]);
}

}  // namespace

PYBIND11_MODULE(TORCH_EXTENSION_NAME, m)
{
    m.def("render", &render);
    m.def("set_error", [](pybind11::object cls) { g_error = cls.release().ptr(); });
}
