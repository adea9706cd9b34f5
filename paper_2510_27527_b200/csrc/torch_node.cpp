// The autograd node of NVFP4Linear (Python module `_node`): one forward call of the layer and, later, its backward, without Python in
// between. It allocates from torch's caching allocator, fills the C structures and calls nvfp4_linear_fwd / nvfp4_linear_bwd; the
// arithmetic is the library's.
//
// What it replaces is host time, which bounds layers up to a few thousand tokens: a torch.autograd.Function whose two methods go
// through ctypes spends two thirds of a step of a 512-wide layer on 256 tokens in the interpreter, half of it on the engine's own
// thread, which has to wait for the interpreter lock first. us a step, that function / this: 256 x 512 -> 512 134 / 86 (its kernels
// 30), 77 x 1024 -> 3072 forward only 32 / 18, 1999 x 1000 -> 1416 with per-row scales 168 / 117, 4095 x 1024 -> 2816 with outlier
// channels 183 / 130, 8192 x 1024 -> 3072 145 / 136.
#include <torch/csrc/Exceptions.h>
#include <torch/csrc/autograd/function.h>
#include <torch/csrc/autograd/python_variable.h>
#include <torch/csrc/dynamo/compiled_autograd.h>

#include <ATen/ATen.h>
#include <c10/cuda/CUDACachingAllocator.h>
#include <c10/cuda/CUDAGuard.h>
#include <c10/cuda/CUDAStream.h>

#include <array>
#include <cstring>
#include <list>

#include "../../include/nvfp4.h"

namespace {

using torch::autograd::variable_list;

constexpr int64_t up(int64_t n, int64_t to) { return (n + to - 1) / to * to; }

// The calling thread's second stream and events for calls on `stream`, made on first use. A thread enqueues its calls on one stream one
// after another, so they share a set: a call's waits refer to the records before them in host order, and recording an event again does
// not change what was already waited for. A thread holds the sets of the eight streams it used last and gives them back when it ends.
struct Side {
  cudaStream_t of;
  c10::DeviceIndex device;
  c10::cuda::CUDAStream stream;
  std::array<cudaEvent_t, 3> events{};
  Side(c10::cuda::CUDAStream main) : of(main.stream()), device(main.device_index()), stream(c10::cuda::getStreamFromPool(false, main.device_index())) {
    for (cudaEvent_t& e : events) C10_CUDA_CHECK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
  }
  Side(const Side&) = delete;
  ~Side() {
    for (cudaEvent_t e : events)
      if (e) (void)cudaEventDestroy(e);  // (fails at the end of the process, when the driver has gone before)
  }
};
void set_side(nvfp4_layer_cfg& c, c10::cuda::CUDAStream main) {
  thread_local std::list<Side> sides;
  auto it = sides.begin();
  while (it != sides.end() && !(it->of == main.stream() && it->device == main.device_index())) ++it;
  if (it == sides.end()) {
    sides.emplace_front(main);
    if (sides.size() > 8) sides.pop_back();  // the one used longest ago
  } else {
    sides.splice(sides.begin(), sides, it);
  }
  const Side& s = sides.front();
  c.side_stream = s.stream.stream();
  c.ev_fork = s.events[0];
  c.ev_join = s.events[1];
  c.ev_aux = s.events[2];
}

// Row-major BF16 matrix whose rows start on 16-byte boundaries. (Not a tracked view of its buffer: a result of its own.)
at::Tensor matrix(int64_t rows, int64_t cols, const at::TensorOptions& opt) {
  const int64_t ld = up(cols, 8);
  at::Tensor t = at::empty({rows, ld}, opt);
  if (ld == cols) return t;
  at::AutoDispatchBelowADInplaceOrView below;
  return t.narrow(1, 0, cols);
}

// Status of a library call, as the exception that the binding raises for it.
[[noreturn]] void raise_status(nvfp4_status status, const char* where) {
  pybind11::gil_scoped_acquire gil;
  try {
    pybind11::object type = pybind11::module_::import("paper_2510_27527_b200.binding").attr("Nvfp4Error");
    PyErr_SetObject(type.ptr(), type((int)status, where).ptr());
  } catch (pybind11::error_already_set& e) {
    e.restore();
  }
  python_error e;
  e.persist();
  throw e;
}

// What a call is beside its tensors.
struct Fixed {
  nvfp4_saved saved{};                     // (into Call::buf)
  nvfp4_layer_cfg cfg{};
  cudaStream_t stream = nullptr;           // of forward
  bool concurrent = false;
};
static_assert(std::is_trivially_copyable_v<Fixed>);

struct Call : Fixed {
  at::Tensor buf;                          // what forward leaves for backward, in one piece, and forward's workspace
  std::array<at::Tensor, 3> index;         // outlier channels, kept channels, channel map
  at::Tensor dev_status;

  at::Tensor forward(const at::Tensor& x, const at::Tensor& w) {
    TORCH_CHECK(x.is_cuda() && w.device() == x.device(), "NVFP4Linear: input on ", x.device(), ", weight on ", w.device());
    const c10::cuda::CUDAGuard guard(x.device());
    const c10::cuda::CUDAStream main = c10::cuda::getCurrentCUDAStream();
    const int64_t N = x.size(0), D = x.size(1), C = w.size(0), Dk = D - cfg.n_out, Kh = nvfp4_outlier_pad(cfg.n_out);
    // the pieces of the buffer: codes, scales and global scales of both operands, the compact outlier matrices, the workspace
    int64_t at = 0;
    auto piece = [&](int64_t bytes) {
      const int64_t here = at;
      at = up(at + bytes, 256);
      return here;
    };
    int64_t offs[6], hp[2] = {-1, -1};
    const int64_t rows[2] = {N, C};
    for (int i = 0; i < 2; ++i) {
      offs[3 * i] = piece((int64_t)nvfp4_operand_codes_bytes(rows[i], Dk));
      offs[3 * i + 1] = piece((int64_t)nvfp4_operand_sf_bytes(rows[i], Dk, NVFP4_SF_TILED128x4));
      offs[3 * i + 2] = piece(4 * (int64_t)nvfp4_operand_gscale_count(rows[i], Dk, cfg.gs_mode));
    }
    for (int i = 0; i < 2; ++i)
      if (Kh) hp[i] = piece(rows[i] * Kh * 2);
    const size_t ws_bytes = nvfp4_linear_workspace_bytes(NVFP4_OP_FWD, N, D, C, cfg.n_out, cfg.gs_mode);
    const int64_t ws = at;
    buf = at::empty({ws + (int64_t)ws_bytes}, x.options().dtype(at::kByte));
    at::Tensor y = matrix(N, C, x.options());
    uint8_t* const p = static_cast<uint8_t*>(buf.data_ptr());
    for (int i = 0; i < 2; ++i) {
      nvfp4_operand& q = i ? saved.qw : saved.qx;
      q.codes = p + offs[3 * i];
      q.sf = p + offs[3 * i + 1];
      q.gscale = reinterpret_cast<float*>(p + offs[3 * i + 2]);
      q.R = rows[i];
      q.K = Dk;
      q.gs_mode = cfg.gs_mode;
      q.sf_layout = NVFP4_SF_TILED128x4;
    }
    saved.N_tok = N;
    saved.D = D;
    saved.C = C;
    saved.X_out = hp[0] < 0 ? nullptr : p + hp[0];
    saved.W_out = hp[1] < 0 ? nullptr : p + hp[1];
    if (concurrent) set_side(cfg, main);
    stream = main.stream();
    const nvfp4_status st = nvfp4_linear_fwd(x.data_ptr(), x.stride(0), w.data_ptr(), w.stride(0), N, D, C, &cfg, y.data_ptr(), y.stride(0), &saved,
                                             p + ws, ws_bytes, main.stream());
    if (st != NVFP4_OK) raise_status(st, "nvfp4_linear_fwd");
    return y;
  }

  variable_list backward(at::Tensor dy) const {
    // (the engine has seen to that; a node can also be called by hand)
    TORCH_CHECK(dy.dim() == 2 && dy.size(0) == saved.N_tok && dy.size(1) == saved.C && dy.device() == buf.device(), "NVFP4LinearBackward: gradient of shape ",
                dy.sizes(), " on ", dy.device(), " for an output of shape [", saved.N_tok, ", ", saved.C, "] on ", buf.device());
    dy = dy.contiguous();
    if (dy.scalar_type() != at::kBFloat16) dy = dy.to(at::kBFloat16);
    const c10::cuda::CUDAGuard guard(dy.device());
    const c10::cuda::CUDAStream main = c10::cuda::getCurrentCUDAStream();
    const int64_t N = saved.N_tok, D = saved.D, C = saved.C;
    at::Tensor dx = matrix(N, D, dy.options()), dw = matrix(C, D, dy.options());
    const size_t ws_bytes = nvfp4_linear_workspace_bytes(NVFP4_OP_BWD, N, D, C, cfg.n_out, cfg.gs_mode);
    at::Tensor ws = at::empty({(int64_t)ws_bytes}, dy.options().dtype(at::kByte));
    nvfp4_layer_cfg c = cfg;
    if (concurrent) set_side(c, main);  // (the engine's thread has its own)
    if (main.stream() != stream)  // (by hand, or compiled autograd: the engine keeps to forward's) given back, their memory waits for this stream too
      for (const at::Tensor* t : {&buf, &index[0], &dev_status})  // (the three index arrays are pieces of one allocation)
        if (t->defined()) c10::cuda::CUDACachingAllocator::recordStream(t->storage().data_ptr(), main);
    const nvfp4_status st = nvfp4_linear_bwd(dy.data_ptr(), dy.stride(0), &saved, &c, dx.data_ptr(), dx.stride(0), dw.data_ptr(), dw.stride(0),
                                             ws.data_ptr(), ws_bytes, main.stream());
    if (st != NVFP4_OK) raise_status(st, "nvfp4_linear_bwd");
    return {std::move(dx), std::move(dw)};
  }
};

struct NVFP4LinearBackward : torch::autograd::Node {
  Call call;
  std::string name() const override { return "NVFP4LinearBackward"; }
  variable_list apply(variable_list&& grads) override {
    return call.backward(grads[0].defined() ? std::move(grads[0]) : input_metadata(0).zeros_like());
  }

  // Compiled autograd records a graph of the whole backward and runs it again on other calls of the same form: the node becomes one call of
  // a function that is not looked into, and all that belongs to this call goes in as tensors.
  mutable at::Tensor fixed;  // the bytes of call's Fixed
  void compiled_args(torch::dynamo::autograd::CompiledNodeArgs& args) const override {
    if (!fixed.defined()) {
      fixed = at::empty({(int64_t)sizeof(Fixed)}, at::kByte);
      std::memcpy(fixed.data_ptr(), static_cast<const Fixed*>(&call), sizeof(Fixed));
    }
    for (const at::Tensor* t : {&std::as_const(fixed), &call.buf, &call.index[0], &call.dev_status}) args.collect(*t);
  }
  variable_list apply_with_saved(const variable_list& grads, torch::dynamo::autograd::SwapSavedVariables& saved) override {
    namespace dynamo = torch::dynamo::autograd;
    const std::array<at::Tensor*, 4> all{&fixed, &call.buf, &call.index[0], &call.dev_status};
    for (at::Tensor* t : all) saved.before(*t);
    std::vector<c10::IValue> args;
    std::vector<at::TypePtr> schema;
    for (const at::Tensor* t : all)
      if (t->defined()) {
        args.emplace_back(*t);
        schema.emplace_back(at::TensorType::get());
      }
    const auto& py = dynamo::getPyCompilerInterface();
    const std::string function = py->bind_function(saved.get_py_compiler(), name(), replay, schema, /*is_custom_function=*/true, /*is_traceable=*/false);
    variable_list out = py->call_function(saved.get_py_compiler(), "apply_functional", function, grads, args,
                                          dynamo::IValuePacker<std::vector<std::optional<torch::autograd::InputMetadata>>>::pack(
                                              dynamo::get_input_metadata(next_edges())));
    for (at::Tensor* t : all) saved.after(*t);
    return out;
  }
  static variable_list replay(const variable_list& grads, const std::vector<c10::IValue>& args) {
    Call c;
    std::memcpy(static_cast<Fixed*>(&c), args.at(0).toTensor().data_ptr(), sizeof(Fixed));
    c.buf = args.at(1).toTensor();
    if (c.cfg.n_out > 0) c.index[0] = args.at(2).toTensor();
    if (c.cfg.dev_status) c.dev_status = args.back().toTensor();
    return c.backward(grads[0].defined() ? grads[0] : at::zeros({c.saved.N_tok, c.saved.C}, c.buf.options().dtype(at::kBFloat16)));
  }
};

// An attribute of the configuration.
pybind11::object attribute(PyObject* cfg, PyObject* name) {
  pybind11::object v = pybind11::reinterpret_steal<pybind11::object>(PyObject_GetAttr(cfg, name));
  if (!v) throw python_error();
  return v;
}
// A 32-bit field from it, as ctypes fills one: whole numbers only (a float or a text is a TypeError), the low bits of larger ones.
int32_t field(pybind11::handle v) {
  const pybind11::object i = pybind11::reinterpret_steal<pybind11::object>(PyNumber_Index(v.ptr()));
  const unsigned long long n = i ? PyLong_AsUnsignedLongLongMask(i.ptr()) : ~0ull;
  if (n == ~0ull && PyErr_Occurred()) throw python_error();
  return (int32_t)(uint32_t)n;
}
// The same of int(v), for the switches.
int32_t switch_field(pybind11::handle v) {
  const pybind11::object i = pybind11::reinterpret_steal<pybind11::object>(PyNumber_Long(v.ptr()));
  if (!i) throw python_error();
  return field(i);
}

struct Names {
  PyObject *gs_mode, *rounding, *rht, *outlier_fp8, *w_block16, *concurrent, *dev_status;
} names;

// linear(x, weight, cfg, index, seed, graph): index = (outlier channels, kept channels, channel map) or None; with `graph` the result
// carries the node. x is contiguous BF16 [tokens, D].
PyObject* linear(PyObject*, PyObject* const* args, Py_ssize_t n) {
  HANDLE_TH_ERRORS
  TORCH_CHECK_TYPE(n == 6 && THPVariable_Check(args[0]) && THPVariable_Check(args[1]), "linear(x, weight, cfg, index, seed, graph)");
  const at::Tensor x = THPVariable_Unpack(args[0]), w = THPVariable_Unpack(args[1]);
  const bool graph = args[5] == Py_True;
  std::shared_ptr<NVFP4LinearBackward> node;
  Call local;
  if (graph) {
    node = std::shared_ptr<NVFP4LinearBackward>(new NVFP4LinearBackward(), torch::autograd::deleteNode);
    node->set_next_edges(torch::autograd::collect_next_edges(x, w));
  }
  Call& call = graph ? node->call : local;
  // the configuration as it is now: what the caller changes later belongs to later calls
  nvfp4_layer_cfg& c = call.cfg;
  PyObject* cfg = args[2];
  c.gs_mode = field(attribute(cfg, names.gs_mode));
  c.rht = switch_field(attribute(cfg, names.rht));
  c.outlier_format = switch_field(attribute(cfg, names.outlier_fp8));
  c.weight_block = switch_field(attribute(cfg, names.w_block16));
  call.concurrent = PyObject_IsTrue(attribute(cfg, names.concurrent).ptr()) == 1;
  c.seed = PyLong_AsUnsignedLongLong(args[4]);
  if (PyErr_Occurred()) throw python_error();
  const pybind11::tuple rounding(attribute(cfg, names.rounding));
  TORCH_CHECK_INDEX(rounding.size() <= 6, "LayerConfig.rounding has ", rounding.size(), " entries instead of 6");
  for (size_t i = 0; i < rounding.size(); ++i) c.rounding[i] = field(rounding[i]);  // what is not given is to nearest
  const pybind11::object status = attribute(cfg, names.dev_status);
  if (!status.is_none()) {
    TORCH_CHECK_TYPE(THPVariable_Check(status.ptr()), "LayerConfig.dev_status is not a tensor");
    call.dev_status = THPVariable_Unpack(status.ptr());
    c.dev_status = static_cast<int32_t*>(call.dev_status.data_ptr());
  }
  c.y_dtype = c.dx_dtype = c.dw_dtype = NVFP4_DT_BF16;
  if (args[3] != Py_None) {
    for (int i = 0; i < 3; ++i) {
      PyObject* t = PyTuple_GetItem(args[3], i);
      if (!t) throw python_error();
      TORCH_CHECK_TYPE(THPVariable_Check(t), "linear: index arrays are tensors");
      call.index[i] = THPVariable_Unpack(t);
    }
    c.n_out = call.index[0].numel();
    c.outlier_cols = static_cast<const int32_t*>(call.index[0].data_ptr());
    c.keep_cols = static_cast<const int32_t*>(call.index[1].data_ptr());
    c.col_map = static_cast<const int32_t*>(call.index[2].data_ptr());
  }
  at::Tensor y;
  {
    pybind11::gil_scoped_release no_gil;
    const at::NoGradGuard no_grad;
    y = call.forward(x, w);
    if (graph) torch::autograd::create_gradient_edge(y, node);
  }
  return THPVariable_Wrap(std::move(y));
  END_HANDLE_TH_ERRORS
}

PyMethodDef methods[] = {{"linear", reinterpret_cast<PyCFunction>(reinterpret_cast<void (*)()>(linear)), METH_FASTCALL, nullptr}, {nullptr, nullptr, 0, nullptr}};
PyModuleDef module_def = {PyModuleDef_HEAD_INIT, "_node", nullptr, -1, methods, nullptr, nullptr, nullptr, nullptr};

}  // namespace

PyMODINIT_FUNC PyInit__node() {
  names = {PyUnicode_InternFromString("gs_mode"),    PyUnicode_InternFromString("rounding"),   PyUnicode_InternFromString("rht"),
           PyUnicode_InternFromString("outlier_fp8"), PyUnicode_InternFromString("w_block16"), PyUnicode_InternFromString("concurrent"),
           PyUnicode_InternFromString("dev_status")};
  PyObject* module = PyModule_Create(&module_def);
  if (module && PyModule_AddStringConstant(module, "built_for", NODE_TAG) < 0) {
    Py_DECREF(module);
    return nullptr;
  }
  return module;
}
