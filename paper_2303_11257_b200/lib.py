"""ctypes binding of libunitscale: same names as the C ABI, argument marshalling only.

Tensors are torch CUDA tensors (device memory and streams come from torch); every
computation happens inside the library's kernels.  Importing this module needs the
compiled library: there is no fallback of any kind.
"""
from __future__ import annotations

import ctypes as C
import os

import torch

US_OK, US_ERR_INVALID_ARG, US_ERR_UNSUPPORTED, US_ERR_ALIGNMENT, US_ERR_WORKSPACE, US_ERR_CUDA, US_ERR_TIMEOUT = range(7)
STATUS_NAMES = {
    0: "US_OK", 1: "US_ERR_INVALID_ARG", 2: "US_ERR_UNSUPPORTED", 3: "US_ERR_ALIGNMENT",
    4: "US_ERR_WORKSPACE", 5: "US_ERR_CUDA", 6: "US_ERR_TIMEOUT",
}
US_F32, US_BF16, US_F16, US_E4M3, US_E5M2 = range(5)
US_ACT_NONE, US_ACT_GELU, US_ACT_GELU_GRAD, US_ACT_RELU, US_ACT_RELU_GRAD, US_ACT_TANH, US_ACT_TANH_GRAD, US_ACT_SIGMOID, US_ACT_SIGMOID_GRAD = range(9)
US_FN_GELU, US_FN_RELU, US_FN_TANH, US_FN_SIGMOID = range(4)
FN_BY_NAME = {"gelu": US_FN_GELU, "relu": US_FN_RELU, "tanh": US_FN_TANH, "sigmoid": US_FN_SIGMOID}

_TORCH_DTYPES = {
    torch.float32: US_F32, torch.bfloat16: US_BF16, torch.float16: US_F16,
    torch.float8_e4m3fn: US_E4M3, torch.float8_e5m2: US_E5M2,
}


class us_mat(C.Structure):
    _fields_ = [("ptr", C.c_void_p), ("dtype", C.c_int32), ("rows", C.c_int64), ("cols", C.c_int64), ("ld", C.c_int64)]


class us_epilogue(C.Structure):
    _fields_ = [
        ("act", C.c_int32), ("act_in_scale", C.c_float), ("act_out_scale", C.c_float),
        ("aux", us_mat), ("skip", us_mat), ("skip_coef", C.c_float), ("out_coef", C.c_float),
    ]


class us_batch(C.Structure):
    _fields_ = [("count", C.c_int64 * 2), ("a_stride", C.c_int64 * 2), ("b_stride", C.c_int64 * 2), ("out_stride", C.c_int64 * 2)]


class us_attention_batch(C.Structure):
    _fields_ = [("count", C.c_int64 * 2), ("q_stride", C.c_int64 * 2), ("k_stride", C.c_int64 * 2),
                ("v_stride", C.c_int64 * 2), ("c_stride", C.c_int64 * 2), ("p_stride", C.c_int64 * 2)]


class us_attention_bwd_batch(C.Structure):
    _fields_ = [("count", C.c_int64 * 2), ("dc_stride", C.c_int64 * 2), ("p_stride", C.c_int64 * 2), ("k_stride", C.c_int64 * 2),
                ("v_stride", C.c_int64 * 2), ("ds_stride", C.c_int64 * 2), ("dq_stride", C.c_int64 * 2)]


class us_attention_bwd_all_batch(C.Structure):
    _fields_ = [(n, C.c_int64 * 2) for n in ("count", "dc_stride", "p_stride", "q_stride", "k_stride", "v_stride", "ds_stride",
                                             "dq_stride", "dk_stride", "dv_stride")]


class us_linear_call(C.Structure):
    _fields_ = [("op", C.c_int32), ("a", us_mat), ("b", us_mat), ("scale", C.c_float), ("ep", us_epilogue), ("out", us_mat)]


US_OP_FWD, US_OP_BWD_X, US_OP_BWD_W = 0, 1, 2


class UnitScaleError(RuntimeError):
    def __init__(self, fn: str, status: int):
        self.status = status
        super().__init__(f"{fn}: {STATUS_NAMES.get(status, status)}")


def library_path() -> str:
    return os.path.join(os.path.dirname(os.path.abspath(__file__)), "libunitscale.so")


def _load() -> C.CDLL:
    path = library_path()
    if not os.path.exists(path):
        raise ImportError(
            f"{path} is missing: build it with `python -m paper_2303_11257_b200.build` "
            "(there is no fallback implementation)")
    lib = C.CDLL(path)
    P, MP, EP, F, V, SZ = C.c_void_p, C.POINTER(us_mat), C.POINTER(us_epilogue), C.c_float, C.c_void_p, C.c_size_t
    for name in ("us_linear_fwd", "us_linear_bwd_x", "us_linear_bwd_w"):
        fn = getattr(lib, name)
        fn.argtypes = [MP, MP, F, EP, MP, V, SZ, V]
        fn.restype = C.c_int
    for name in ("us_linear_fwd_batched", "us_linear_bwd_x_batched", "us_linear_bwd_w_batched"):
        fn = getattr(lib, name)
        fn.argtypes = [MP, MP, F, MP, C.POINTER(us_batch), V, SZ, V]
        fn.restype = C.c_int
    lib.us_attention_fwd.argtypes = [MP, MP, MP, F, F, F, MP, MP, C.POINTER(us_attention_batch), V, SZ, V]
    lib.us_attention_fwd.restype = C.c_int
    lib.us_attention_bwd.argtypes = [MP, MP, MP, MP, F, F, F, F, MP, MP, C.POINTER(us_attention_bwd_batch), V, SZ, V]
    lib.us_attention_bwd.restype = C.c_int
    lib.us_attention_bwd_all.argtypes = [MP] * 5 + [F] * 6 + [MP] * 4 + [C.POINTER(us_attention_bwd_all_batch), V, SZ, V]
    lib.us_test_attention_bwd_all_starved.argtypes = [MP] * 5 + [F] + [MP] * 4 + [C.POINTER(us_attention_bwd_all_batch), V, SZ, C.c_uint, C.c_int, C.c_int, V]
    lib.us_attention_bwd_all.restype = lib.us_test_attention_bwd_all_starved.restype = C.c_int
    lib.us_linear_fwd_static_ws.argtypes = [MP, MP, F, EP, MP, C.POINTER(C.c_void_p), V]
    lib.us_linear_fwd_static_ws.restype = C.c_int
    lib.us_linear_fwd_check.argtypes = [MP, MP, EP, MP, V, SZ]
    lib.us_linear_fwd_check.restype = C.c_int
    lib.us_test_linear_fwd_starved.argtypes = [MP, MP, F, MP, V, SZ, C.c_uint, V]
    lib.us_test_linear_fwd_starved.restype = C.c_int
    lib.us_linear_group.argtypes = [C.c_int, C.POINTER(us_linear_call), V, SZ, V]
    lib.us_linear_group_any.argtypes = lib.us_linear_group.argtypes
    lib.us_linear_group.restype = lib.us_linear_group_any.restype = C.c_int
    lib.us_test_linear_tiling.argtypes = [C.c_int, MP, MP, EP, MP, V, SZ] + [C.POINTER(C.c_int)] * 3
    lib.us_test_linear_tiling.restype = C.c_int
    lib.us_linear_group_launches.argtypes = [C.c_int, C.POINTER(us_linear_call), C.POINTER(C.c_int)]
    lib.us_linear_group_launches.restype = C.c_int
    lib.us_linear_fwd_cast.argtypes = [MP, MP, F, EP, MP, MP, V, SZ, V]
    lib.us_linear_group_cast.argtypes = [C.c_int, C.POINTER(us_linear_call), MP, V, SZ, V]
    lib.us_layer_norm_fwd_cast.argtypes = [MP, MP, MP, F, MP, MP, V]
    lib.us_layer_norm_bwd_cast.argtypes = [MP, MP, MP, F, F, F, MP, MP, MP, MP, V, SZ, V]
    for name in ("us_linear_fwd_cast", "us_linear_group_cast", "us_layer_norm_fwd_cast", "us_layer_norm_bwd_cast"):
        getattr(lib, name).restype = C.c_int
    lib.us_ffn_hidden.argtypes = [MP, MP, F, MP, MP, F, F, F, F, C.c_int32, MP, MP, MP, V, SZ, V]
    lib.us_ffn_hidden_any.argtypes = lib.us_ffn_hidden.argtypes
    lib.us_ffn_hidden.restype = lib.us_ffn_hidden_any.restype = C.c_int
    lib.us_test_ffn_hidden_starved.argtypes = [MP, MP, MP, MP, MP, MP, V, SZ, C.c_uint, V]
    lib.us_test_ffn_hidden_starved.restype = C.c_int
    lib.us_test_linear_fwd_starved_cta.argtypes = [MP, MP, F, MP, V, SZ, C.c_uint, C.c_int, C.c_int, V]
    lib.us_test_ffn_hidden_starved_cta.argtypes = [MP] * 6 + [V, SZ, C.c_uint, C.c_int, C.c_int, V]
    lib.us_test_linear_group_starved.argtypes = [C.c_int, C.POINTER(us_linear_call), V, SZ, C.c_uint, C.c_int, C.c_int, V]
    for name in ("us_test_linear_fwd_starved_cta", "us_test_ffn_hidden_starved_cta", "us_test_linear_group_starved"):
        getattr(lib, name).restype = C.c_int
    lib.us_workspace_bytes.argtypes = []
    lib.us_workspace_bytes.restype = SZ
    lib.us_workspace_status.argtypes = [V, V]
    lib.us_workspace_status.restype = C.c_int
    lib.us_gelu_fwd.argtypes = [MP, F, F, MP, V]
    lib.us_gelu_bwd.argtypes = [MP, MP, F, F, MP, V]
    lib.us_residual_add.argtypes = [MP, MP, F, MP, V]
    lib.us_cast_fp8.argtypes = [MP, F, MP, V]
    lib.us_activation_fwd.argtypes = [C.c_int, MP, F, F, MP, V]
    lib.us_activation_bwd.argtypes = [C.c_int, MP, MP, F, F, MP, V]
    lib.us_activation_fwd.restype = lib.us_activation_bwd.restype = C.c_int
    lib.us_cast_fp8_multi.argtypes = lib.us_cast_multi.argtypes = lib.us_cast_multi_pitched.argtypes = [C.c_int, MP, C.POINTER(C.c_float), MP, V]
    lib.us_weighted_add.argtypes = [C.c_int, MP, C.POINTER(C.c_float), F, MP, V]
    lib.us_weighted_add.restype = C.c_int
    lib.us_softmax_fwd.argtypes = [MP, F, MP, V]
    lib.us_softmax_bwd.argtypes = [MP, MP, F, F, MP, V]
    lib.us_softmax_xent_fwd.argtypes = [MP, V, V, V]
    lib.us_softmax_xent_bwd.argtypes = [MP, V, V, F, MP, V]
    lib.us_softmax_xent_fwd.restype = lib.us_softmax_xent_bwd.restype = C.c_int
    lib.us_layer_norm_fwd.argtypes = [MP, MP, MP, F, MP, V]
    lib.us_layer_norm_bwd.argtypes = [MP, MP, MP, F, F, F, MP, MP, MP, V, SZ, V]
    lib.us_layer_norm_fwd.restype = lib.us_layer_norm_bwd.restype = C.c_int
    lib.us_layer_norm_bwd_workspace_bytes.argtypes = [C.c_int64, C.c_int64]
    lib.us_layer_norm_bwd_workspace_bytes.restype = SZ
    lib.us_quant_stats_workspace_bytes.argtypes = []
    lib.us_quant_stats_workspace_bytes.restype = SZ
    lib.us_quant_stats.argtypes = [MP, F, C.c_int, C.c_int, C.c_int, V, V, V, SZ, V]
    lib.us_quant_stats.restype = C.c_int
    for name in ("us_gelu_fwd", "us_gelu_bwd", "us_residual_add", "us_cast_fp8", "us_cast_fp8_multi", "us_cast_multi", "us_cast_multi_pitched", "us_softmax_fwd", "us_softmax_bwd"):
        getattr(lib, name).restype = C.c_int
    FP = C.POINTER(C.c_float)
    lib.us_scales_linear.argtypes = [C.c_int64, C.c_int64, C.c_int64, C.c_int, FP, FP, FP]
    lib.us_scales_linear.restype = C.c_int
    lib.us_scales_gelu.argtypes = [C.c_int, FP, FP]
    lib.us_scales_activation.argtypes = [C.c_int, C.c_int, FP, FP]
    lib.us_scales_activation.restype = C.c_int
    lib.us_scales_gelu.restype = C.c_int
    lib.us_scales_residual.argtypes = [C.c_float, FP, FP]
    lib.us_scales_residual.restype = C.c_int
    lib.us_scales_attention.argtypes = [C.c_int64, C.c_int64, C.c_int, FP, FP, FP, FP, FP, FP]
    lib.us_scales_attention.restype = C.c_int
    lib.us_status_string.argtypes = [C.c_int]
    lib.us_status_string.restype = C.c_char_p
    lib.us_version.argtypes = []
    lib.us_version.restype = C.c_int
    return lib


_lib = _library = _load()
from .build import built_for                                  # noqa: E402
try:
    from . import _binding                                    # links the library that has just been loaded
    if _binding.built_for != built_for():                     # torch's C++ interface is another one from version to version
        raise ImportError(f"{_binding.built_for} {built_for()}")
except ImportError as e:
    raise ImportError(f"the Python binding is missing or was built for another Python or torch ({e}): build it with "
                      "`python -m paper_2303_11257_b200.build`") from e

_binding.register_types((us_mat, us_epilogue, us_batch, us_attention_batch, us_attention_bwd_batch, us_attention_bwd_all_batch, us_linear_call, C.c_float))


def _entry(name: str):
    """The function of that name: through the binding, which takes tensors as they are."""
    return _binding.calls[name] if _lib is _library else getattr(_lib, name)


def raw() -> C.CDLL:
    """The loaded CDLL, for callers that want to build us_mat structures themselves."""
    return _lib


def describe(t: torch.Tensor) -> tuple:
    """The fields of a us_mat for a 2-D row-major torch tensor (last stride 1)."""
    shape, stride = t.shape, t.stride()
    if len(shape) != 2 or (shape[1] > 1 and stride[1] != 1):
        raise ValueError("expected a 2-D tensor with unit column stride")
    rows, cols = shape
    return t.data_ptr(), _TORCH_DTYPES[t.dtype], rows, cols, stride[0] if rows > 1 else max(cols, stride[0])


def mat(t: torch.Tensor) -> us_mat:
    """Describe a 2-D row-major torch tensor (last stride 1) without copying it."""
    return us_mat(*describe(t))


def current_stream() -> int:
    """Handle of the current device's current stream.  Asks torch's C layer for the handle itself (0.4 us, against 3.4 us
    for making a Stream object of it); every launch asks."""
    if torch.cuda.is_initialized():
        return torch._C._cuda_getCurrentRawStream(torch._C._cuda_getDevice())
    return torch.cuda.current_stream().cuda_stream


def _stream(stream) -> int:
    if stream is None:
        return current_stream()
    return stream.cuda_stream if hasattr(stream, "cuda_stream") else int(stream)


class Call:
    """A library call whose arguments are laid out once.  It points into tensors that the caller keeps (a block's own
    buffers); descriptions that change from call to call -- the tensors a user passes to a step -- are written into its us_mat
    slots before each call.  instead: (statuses, fn); a call that the library refuses with one of those statuses, having
    launched nothing, issues fn(stream) in its place."""
    __slots__ = ("name", "fn", "args", "keep", "instead", "refused")

    def __init__(self, name, *args, instead=((), None)):
        self.name, self.fn, self.keep, self.instead, self.refused = name, _entry(name), args, instead, False
        self.args = args if _lib is _library else tuple(C.byref(a) if isinstance(a, C.Structure) else a for a in args)

    def __call__(self, stream: int) -> None:
        self.finish(self.fn(*self.args, stream), stream)

    def finish(self, status: int, stream: int) -> None:
        if status != US_OK:
            if status not in self.instead[0]:
                raise UnitScaleError(self.name, status)
            self.refused = True
            self.instead[1](stream)


class Plan:
    """The calls of one pass over an object's own buffers, and the slots its inputs go to.  `owned` are those buffers,
    `state` every other value the calls were laid out for: same() says whether both are still what they were.  issue() makes
    a pass: lay_out(plan) yields the calls in order, or (where, call) pairs (see MAIN); the first pass issues each as soon as
    it is laid out, later ones go out as one call of the binding."""

    # where a call goes: the main stream; the side stream, once all that was issued before has finished; or, without a call,
    # the main stream waits for the side stream
    MAIN, SIDE, JOIN = range(3)

    def __init__(self, owned, state):
        self.owned, self.state, self.ptrs = owned, state, tuple(t.data_ptr() for t in owned)
        self.slots, self.inputs, self.done, self.mats, self.program = {}, {}, None, {}, None

    def same(self, owned, state) -> bool:
        return self.state == state and _binding.unchanged(owned, self.owned, self.ptrs)

    def mat(self, t: torch.Tensor) -> us_mat:
        """mat(t), made once for all calls of the pass that is being laid out."""
        known = self.mats.get(id(t))
        if known is None:
            known = self.mats[id(t)] = (t, mat(t))              # t is held: its id stays its own
        return known[1]

    def slot(self, name: str, m: us_mat = None) -> us_mat:
        """A us_mat (m, or a new one) that put() fills for the input `name`."""
        m = us_mat() if m is None else m
        self.slots.setdefault(name, []).append(m)
        m.ptr, m.dtype, m.rows, m.cols, m.ld = self.inputs[name]
        return m

    def put(self, name: str, t: torch.Tensor) -> None:
        d = self.inputs[name] = describe(t)
        for m in self.slots.get(name, ()):
            m.ptr, m.dtype, m.rows, m.cols, m.ld = d

    def calls(self, lay_out):
        """The calls of a pass whose inputs have been put."""
        return self.done if self.done is not None else self._first(lay_out)

    def _first(self, lay_out):
        self.slots, self.mats, made = {}, {}, []
        for c in lay_out(self):
            made.append(c)
            yield c
        self.done, self.mats = made, {}                         # a pass that ended early is laid out again

    def issue(self, lay_out, inputs: dict, main: int, side=None) -> Call:
        """One pass with these inputs (tensors by name) on the stream `main`; side: (stream, fork event, join event) for the
        calls that go to the side stream, which otherwise go to the main one.  Returns the pass's last call."""
        if self.done is not None and _lib is _library:
            if self.program is None:
                self._compile(tuple(inputs))
            names, program = self.program
            values = tuple(inputs.values()) if tuple(inputs) == names else tuple(inputs[n] for n in names)
            handles = (main, side[0].cuda_stream, side[1].cuda_event, side[2].cuda_event) if side else (main, 0, 0, 0)
            r = _binding.run(program, 0, values, *handles)
            while r >= 0:                                       # a call that was refused: what it has instead, then the rest
                where, call = self._steps[r >> 8]
                if call is None:
                    raise UnitScaleError("join", r & 255)
                call.finish(r & 255, handles[1] if where == self.SIDE and side else main)
                r = _binding.run(program, (r >> 8) + 1, values, *handles)
            return self._steps[-1][1]
        for name, t in inputs.items():
            self.put(name, t)
        call = None
        for entry in self.calls(lay_out):
            where, this = entry if isinstance(entry, tuple) else (self.MAIN, entry)
            if where == self.JOIN:
                if side:
                    side[2].record(side[0])
                    torch.cuda.current_stream().wait_event(side[2])
                continue
            call = this
            if where == self.SIDE and side:
                side[1].record(torch.cuda.current_stream())
                side[0].wait_event(side[1])
                call(side[0].cuda_stream)
            else:
                call(main)
        return call

    def _compile(self, names):
        self._steps = [e if isinstance(e, tuple) else (self.MAIN, e) for e in self.done]
        steps = [(w, c if c is None else _binding.prepare(c.name, c.keep)) for w, c in self._steps]
        slots = [(i, m) for i, n in enumerate(names) for m in self.slots.get(n, ())]
        self.program = names, _binding.program(steps, slots)

    def cast_multi(self, srcs, dsts, padded=False):
        """us_cast_multi (us_cast_multi_pitched where a destination has padded rows) at scale 1; an entry of srcs is a tensor or
        the name of an input.  padded: rows that it does not take (padded or unaligned ones) go out as one us_residual_add per
        tensor, for 16-bit destinations."""
        n = len(srcs)
        sm = (us_mat * n)()
        for i, s in enumerate(srcs):
            if isinstance(s, str):
                self.slot(s, sm[i])
            else:
                sm[i] = self.mat(s)
        dm = (us_mat * n)(*[self.mat(t) for t in dsts])

        def each(stream):
            for s, d in zip(sm, dm):
                _check("us_residual_add", _entry("us_residual_add")(s, s, 0.0, d, stream))

        return Call("us_cast_multi_pitched" if _padded(dsts) else "us_cast_multi", n, sm, (C.c_float * n)(*[1.0] * n), dm,
                    instead=((US_ERR_UNSUPPORTED, US_ERR_ALIGNMENT) if padded else (), each))

    def residual(self, skip, coef):
        """The fixed(tau) residual epilogue; skip is a tensor or the name of an input."""
        ep = us_epilogue()
        ep.act, ep.act_in_scale, ep.act_out_scale, ep.skip_coef, ep.out_coef = US_ACT_NONE, 1.0, 1.0, *coef
        if isinstance(skip, str):
            self.slot(skip, ep.skip)
        else:
            ep.skip = self.mat(skip)
        return ep

    def group(self, entries, ws, copies=None):
        """us_linear_group_any over (op, a, b, scale, out, skip or None, (skip_coef, out_coef)); as single launches where
        there are more tiles than its work list holds.  copies: FP8 copies of the outputs (us_linear_group_cast), by entry."""
        arr = (us_linear_call * len(entries))()
        for c, (op, a, b, scale, out, skip, coef) in zip(arr, entries):
            c.op, c.a, c.b, c.scale, c.out, c.ep.out_coef = op, self.mat(a), self.mat(b), scale, self.mat(out), 1.0
            if skip is not None:
                c.ep.act_in_scale = c.ep.act_out_scale = 1.0
                c.ep.skip_coef, c.ep.out_coef = coef
                if isinstance(skip, str):
                    self.slot(skip, c.ep.skip)
                else:
                    c.ep.skip = self.mat(skip)
        if not copies:
            return Call("us_linear_group_any", len(entries), arr, ws.data_ptr(), ws.numel(),
                        instead=((US_ERR_UNSUPPORTED,), lambda stream: linear_each(arr, ws, stream)))
        cp = (us_mat * len(entries))()
        for i, t in copies.items():
            cp[i] = self.mat(t)

        def each(stream):
            linear_each(arr, ws, stream)
            for i in copies:
                _check("us_cast_fp8", _entry("us_cast_fp8")(arr[i].out, 1.0, cp[i], stream))

        return Call("us_linear_group_cast", len(entries), arr, cp, ws.data_ptr(), ws.numel(), instead=((US_ERR_UNSUPPORTED,), each))

    def linear(self, name, a, b, scale, out, ws, ep=None):
        return Call(name, self.mat(a), self.mat(b), scale, ep, self.mat(out), ws.data_ptr(), ws.numel())

    def batched(self, name, a, b, scale, out, bt, ws):
        return Call(name, self.mat(a), self.mat(b), scale, self.mat(out), bt, ws.data_ptr(), ws.numel())


def _check(fn: str, status: int) -> None:
    if status != US_OK:
        raise UnitScaleError(fn, status)


def epilogue(act: int = US_ACT_NONE, act_in_scale: float = 1.0, act_out_scale: float = 1.0,
             aux: torch.Tensor | None = None, skip: torch.Tensor | None = None,
             skip_coef: float = 0.0, out_coef: float = 1.0) -> us_epilogue:
    ep = us_epilogue()
    ep.act, ep.act_in_scale, ep.act_out_scale = act, act_in_scale, act_out_scale
    if aux is not None:
        ep.aux = mat(aux)
    if skip is not None:
        ep.skip = mat(skip)
    ep.skip_coef, ep.out_coef = skip_coef, out_coef
    ep._keep_alive = (aux, skip)      # the struct holds raw pointers only
    return ep


def us_workspace_bytes() -> int:
    return int(_lib.us_workspace_bytes())


def new_workspace(device="cuda") -> torch.Tensor:
    """A zeroed workspace of the size the linear ops ask for."""
    return torch.zeros(us_workspace_bytes(), dtype=torch.uint8, device=device)


def us_workspace_status(ws: torch.Tensor, stream=None) -> int:
    return int(_lib.us_workspace_status(ws.data_ptr(), _stream(stream)))


def _linear(name, a, b, scale, ep, out, ws, stream):
    fn = _entry(name)
    _check(name, fn(a, b, scale, ep, out, ws, ws, _stream(stream)))
    return out


def us_linear_fwd(X, W, alpha, Y, ws, ep=None, stream=None):
    return _linear("us_linear_fwd", X, W, alpha, ep, Y, ws, stream)


def us_linear_bwd_x(G, W, beta_x, dX, ws, ep=None, stream=None):
    return _linear("us_linear_bwd_x", G, W, beta_x, ep, dX, ws, stream)


def us_linear_bwd_w(X, G, beta_w, dW, ws, ep=None, stream=None):
    return _linear("us_linear_bwd_w", X, G, beta_w, ep, dW, ws, stream)


def linear_call(op: int, a, b, scale: float, out, ep=None) -> us_linear_call:
    """One entry of a us_linear_group launch: op in (US_OP_FWD, US_OP_BWD_X, US_OP_BWD_W), operands in that op's order."""
    c = us_linear_call()
    c.op, c.a, c.b, c.scale, c.out = op, mat(a), mat(b), scale, mat(out)
    if ep is not None:
        c.ep = ep
    else:
        c.ep.out_coef = 1.0
    c._keep_alive = (a, b, out, ep)
    return c


def us_linear_group(calls, ws, stream=None, name="us_linear_group"):
    """Several independent linear ops in one launch (see the header for what this form covers)."""
    arr = (us_linear_call * len(calls))(*calls)
    _check(name, _entry(name)(len(calls), arr, ws, ws, _stream(stream)))


def us_linear_group_any(calls, ws, stream=None):
    """us_linear_group for 16-bit operands and outputs of any size, too."""
    us_linear_group(calls, ws, stream, "us_linear_group_any")


def us_linear_group_launches(calls) -> int:
    """Number of kernels us_linear_group_any launches for these calls; one each where it refuses them (linear_together)."""
    n = C.c_int()
    status = _lib.us_linear_group_launches(len(calls), (us_linear_call * len(calls))(*calls), C.byref(n))
    if status == US_ERR_UNSUPPORTED:
        return len(calls)
    _check("us_linear_group_launches", status)
    return n.value


def linear_each(calls, ws, stream=None):
    """The same ops as single launches, in order (for a group with more tiles than the grouped form's work list holds)."""
    for c in calls:
        name = ("us_linear_fwd", "us_linear_bwd_x", "us_linear_bwd_w")[c.op]
        _check(name, _entry(name)(c.a, c.b, c.scale, c.ep, c.out, ws, ws, _stream(stream)))


def linear_together(calls, ws, stream=None):
    """The ops as one launch, or one by one where the grouped form does not cover them."""
    try:
        us_linear_group_any(calls, ws, stream)
    except UnitScaleError as e:
        if e.status != US_ERR_UNSUPPORTED:
            raise
        linear_each(calls, ws, stream)


def batch(count, a_stride, b_stride, out_stride) -> us_batch:
    """us_batch from (outer, inner) pairs of counts and element strides."""
    b = us_batch()
    for i in range(2):
        b.count[i], b.a_stride[i], b.b_stride[i], b.out_stride[i] = count[i], a_stride[i], b_stride[i], out_stride[i]
    return b


def _linear_batched(name, a, b, scale, out, bt, ws, stream):
    fn = _entry(name)
    _check(name, fn(a, b, scale, out, bt,
                    ws, ws, _stream(stream)))
    return out


def us_linear_fwd_batched(X, W, alpha, Y, bt, ws, stream=None):
    return _linear_batched("us_linear_fwd_batched", X, W, alpha, Y, bt, ws, stream)


def us_linear_bwd_x_batched(G, W, beta_x, dX, bt, ws, stream=None):
    return _linear_batched("us_linear_bwd_x_batched", G, W, beta_x, dX, bt, ws, stream)


def us_linear_bwd_w_batched(X, G, beta_w, dW, bt, ws, stream=None):
    return _linear_batched("us_linear_bwd_w_batched", X, G, beta_w, dW, bt, ws, stream)


def attention_batch(count, q_stride, k_stride, v_stride, c_stride, p_stride=(0, 0)) -> us_attention_batch:
    """us_attention_batch from (outer, inner) pairs of counts and element strides."""
    b = us_attention_batch()
    for i in range(2):
        b.count[i] = count[i]
        b.q_stride[i], b.k_stride[i], b.v_stride[i] = q_stride[i], k_stride[i], v_stride[i]
        b.c_stride[i], b.p_stride[i] = c_stride[i], p_stride[i]
    return b


def us_attention_fwd(Q, K, V, alpha_scores, softmax_scale, alpha_context, Cx, P, bt, ws, stream=None):
    """Fused scaled dot-product attention forward; P may be None (weights not stored)."""
    _check("us_attention_fwd", _entry("us_attention_fwd")(Q, K, V, alpha_scores, softmax_scale, alpha_context, Cx, P, bt, ws, ws, _stream(stream)))
    return Cx


def attention_bwd_batch(count, dc_stride, p_stride, k_stride, v_stride, ds_stride, dq_stride) -> us_attention_bwd_batch:
    b = us_attention_bwd_batch()
    for i in range(2):
        b.count[i] = count[i]
        b.dc_stride[i], b.p_stride[i], b.k_stride[i] = dc_stride[i], p_stride[i], k_stride[i]
        b.v_stride[i], b.ds_stride[i], b.dq_stride[i] = v_stride[i], ds_stride[i], dq_stride[i]
    return b


def us_attention_bwd(dC, P, K, V, beta_p, softmax_alpha, softmax_beta, beta_q, dS, dQ, bt, ws, stream=None):
    """Attention backward down to the queries: dS (for the dK matmul) and dQ from dC, the stored P, K and V."""
    _check("us_attention_bwd", _entry("us_attention_bwd")(dC, P, K, V, beta_p, softmax_alpha, softmax_beta, beta_q, dS, dQ, bt, ws, ws, _stream(stream)))
    return dQ


def attention_bwd_all_batch(count, dc_stride, p_stride, q_stride, k_stride, v_stride, ds_stride, dq_stride, dk_stride, dv_stride) -> us_attention_bwd_all_batch:
    b = us_attention_bwd_all_batch()
    for (name, _), v in zip(b._fields_, (count, dc_stride, p_stride, q_stride, k_stride, v_stride, ds_stride, dq_stride, dk_stride, dv_stride)):
        getattr(b, name)[:] = v
    return b


def us_attention_bwd_all(dC, P, Q, K, V, beta_p, softmax_alpha, softmax_beta, beta_q, beta_k, beta_v, dS, dQ, dK, dV, bt, ws, stream=None):
    """The whole backward pass of attention in one launch; dS may be None (not stored)."""
    _check("us_attention_bwd_all", _entry("us_attention_bwd_all")(dC, P, Q, K, V, beta_p, softmax_alpha, softmax_beta, beta_q, beta_k, beta_v, dS, dQ, dK, dV, bt, ws, ws, _stream(stream)))
    return dQ, dK, dV


def us_test_attention_bwd_all_starved(dC, P, Q, K, V, softmax_alpha, dS, dQ, dK, dV, bt, ws, wait_limit: int, rank: int, tile: int, stream=None):
    """us_test_linear_fwd_starved for the kernel of us_attention_bwd_all: CTA `rank` of a cluster gets dC for `tile` tiles only."""
    _check("us_test_attention_bwd_all_starved",
           _lib.us_test_attention_bwd_all_starved(*(C.byref(mat(t)) for t in (dC, P, Q, K, V)), softmax_alpha, *(C.byref(mat(t)) for t in (dS, dQ, dK, dV)),
                                                  C.byref(bt), ws.data_ptr(), ws.numel() * ws.element_size(), wait_limit, rank, tile, _stream(stream)))


def us_linear_fwd_static_ws(X, W, alpha, Y, ep=None, stream=None) -> int:
    """us_linear_fwd without a caller workspace: the library's built-in scratch array is used and
    nothing is allocated.  For callers that cannot allocate device memory (see the header).
    Returns the device address of the built-in scratch, which us_workspace_status_ptr accepts."""
    ws = C.c_void_p()
    epp = C.byref(ep) if ep is not None else None
    _check("us_linear_fwd_static_ws",
           _lib.us_linear_fwd_static_ws(C.byref(mat(X)), C.byref(mat(W)), alpha, epp, C.byref(mat(Y)),
                                        C.byref(ws), _stream(stream)))
    return ws.value


def us_linear_fwd_check(X, W, Y, ws, ep=None) -> int:
    """Status us_linear_fwd would return from its host-side checks (0 = it would launch); launches nothing."""
    epp = C.byref(ep) if ep is not None else None
    return int(_lib.us_linear_fwd_check(C.byref(mat(X)), C.byref(mat(W)), epp, C.byref(mat(Y)),
                                        ws.data_ptr(), ws.numel() * ws.element_size()))


def us_test_linear_fwd_starved(X, W, alpha, Y, ws, wait_limit: int, stream=None):
    """The failure-path exercise of the header: a forward linear launch whose loads are withheld and
    whose waits give up after wait_limit polls; the status word in ws is raised and the kernel returns."""
    _check("us_test_linear_fwd_starved",
           _lib.us_test_linear_fwd_starved(C.byref(mat(X)), C.byref(mat(W)), alpha, C.byref(mat(Y)), ws.data_ptr(),
                                           ws.numel() * ws.element_size(), wait_limit, _stream(stream)))


def us_ffn_hidden(X, W1, alpha, G, W2, beta_x, act_in_scale, act_out_scale, grad_out_scale, A, dH, ws,
                  H=None, h_dtype=torch.bfloat16, stream=None, name="us_ffn_hidden"):
    """Hidden layer of the FFN block, forward and backward, in one launch (see the header): A and dH are written,
    H (optional) receives the pre-activation rounded to h_dtype."""
    _check(name, _entry(name)(X, W1, alpha, G, W2, beta_x, act_in_scale, act_out_scale, grad_out_scale, _TORCH_DTYPES[h_dtype], H, A, dH,
                              ws, ws, _stream(stream)))
    return A, dH


def us_ffn_hidden_any(*args, **kwargs):
    """us_ffn_hidden for 16-bit operands and any number of rows and hidden units, too."""
    return us_ffn_hidden(*args, **kwargs, name="us_ffn_hidden_any")


def us_test_ffn_hidden_starved(X, W1, G, W2, A, dH, ws, wait_limit: int, stream=None):
    """us_test_linear_fwd_starved for the kernel of us_ffn_hidden."""
    _check("us_test_ffn_hidden_starved",
           _lib.us_test_ffn_hidden_starved(C.byref(mat(X)), C.byref(mat(W1)), C.byref(mat(G)), C.byref(mat(W2)),
                                           C.byref(mat(A)), C.byref(mat(dH)), ws.data_ptr(),
                                           ws.numel() * ws.element_size(), wait_limit, _stream(stream)))


def us_test_linear_fwd_starved_cta(X, W, alpha, Y, ws, wait_limit: int, cta: int, tiles: int, stream=None):
    """us_test_linear_fwd_starved with loads withheld from one CTA of each cluster (-1: every CTA) after its first `tiles` tiles."""
    _check("us_test_linear_fwd_starved_cta",
           _lib.us_test_linear_fwd_starved_cta(C.byref(mat(X)), C.byref(mat(W)), alpha, C.byref(mat(Y)), ws.data_ptr(), ws.numel(), wait_limit, cta, tiles,
                                               _stream(stream)))


def us_test_linear_tiling(op: int, a, b, out, ws, ep=None) -> tuple[int, int, int]:
    """Columns of a tile, CTAs that work on it as a pair, CTAs or pairs that share its contraction."""
    r = [C.c_int() for _ in range(3)]
    _check("us_test_linear_tiling", _lib.us_test_linear_tiling(op, C.byref(mat(a)), C.byref(mat(b)), C.byref(ep) if ep is not None else None, C.byref(mat(out)),
                                                               ws.data_ptr(), ws.numel(), *(C.byref(x) for x in r)))
    return tuple(x.value for x in r)


def us_test_ffn_hidden_starved_cta(X, W1, G, W2, A, dH, ws, wait_limit: int, cta: int, tiles: int, stream=None):
    """us_test_linear_fwd_starved_cta for the kernel of us_ffn_hidden."""
    _check("us_test_ffn_hidden_starved_cta",
           _lib.us_test_ffn_hidden_starved_cta(*(C.byref(mat(t)) for t in (X, W1, G, W2, A, dH)), ws.data_ptr(), ws.numel(), wait_limit, cta, tiles, _stream(stream)))


def us_test_linear_group_starved(calls, ws, wait_limit: int, cta: int, tiles: int, stream=None):
    """us_test_linear_fwd_starved_cta for the kernels of us_linear_group_any."""
    _check("us_test_linear_group_starved",
           _lib.us_test_linear_group_starved(len(calls), (us_linear_call * len(calls))(*calls), ws.data_ptr(), ws.numel(), wait_limit, cta, tiles, _stream(stream)))


def us_workspace_status_ptr(ws_ptr: int, stream=None) -> int:
    """us_workspace_status for a raw device address."""
    return int(_lib.us_workspace_status(ws_ptr, _stream(stream)))


def us_gelu_fwd(H, s_in, alpha, A, stream=None):
    _check("us_gelu_fwd", _entry("us_gelu_fwd")(H, s_in, alpha, A, _stream(stream)))
    return A


def us_gelu_bwd(H, dA, s_in, beta, dH, stream=None):
    _check("us_gelu_bwd", _entry("us_gelu_bwd")(H, dA, s_in, beta, dH, _stream(stream)))
    return dH


def us_activation_fwd(fn, H, s_in, alpha, A, stream=None):
    _check("us_activation_fwd", _entry("us_activation_fwd")(FN_BY_NAME.get(fn, fn), H, s_in, alpha, A, _stream(stream)))
    return A


def us_activation_bwd(fn, H, dA, s_in, beta, dH, stream=None):
    _check("us_activation_bwd", _entry("us_activation_bwd")(FN_BY_NAME.get(fn, fn), H, dA, s_in, beta, dH, _stream(stream)))
    return dH


def us_scales_activation(fn, constrained: bool = False):
    a, b = C.c_float(), C.c_float()
    _check("us_scales_activation", _lib.us_scales_activation(FN_BY_NAME.get(fn, fn), int(constrained), C.byref(a), C.byref(b)))
    return a.value, b.value


def us_residual_add(skip, branch, tau, out, stream=None):
    _check("us_residual_add", _entry("us_residual_add")(skip, branch, tau, out, _stream(stream)))
    return out


def us_cast_fp8(src, scale, dst, stream=None):
    _check("us_cast_fp8", _entry("us_cast_fp8")(src, scale, dst, _stream(stream)))
    return dst


def us_weighted_add(srcs, gammas, alpha, out, stream=None):
    n = len(srcs)
    sm = (us_mat * n)(*[mat(t) for t in srcs])
    gm = (C.c_float * n)(*[float(g) for g in gammas])
    _check("us_weighted_add", _entry("us_weighted_add")(n, sm, gm, alpha, out, _stream(stream)))
    return out


def us_cast_fp8_multi(srcs, scales, dsts, stream=None, name="us_cast_fp8_multi"):
    """One launch for len(srcs) casts; scales: one float per tensor."""
    n = len(srcs)
    sm = (us_mat * n)(*[mat(t) for t in srcs])
    dm = (us_mat * n)(*[mat(t) for t in dsts])
    sc = (C.c_float * n)(*[float(x) for x in scales])
    _check(name, _entry(name)(n, sm, sc, dm, _stream(stream)))
    return dsts


def us_cast_multi(srcs, scales, dsts, stream=None):
    """us_cast_fp8_multi with BF16 / F16 destinations allowed."""
    return us_cast_fp8_multi(srcs, scales, dsts, stream, "us_cast_multi")


def us_cast_multi_pitched(srcs, scales, dsts, stream=None):
    """us_cast_multi with destinations whose rows may be padded."""
    return us_cast_fp8_multi(srcs, scales, dsts, stream, "us_cast_multi_pitched")


def operand(rows: int, cols: int, dtype, device="cuda") -> torch.Tensor:
    """An uninitialised matmul operand [rows x cols] with rows on 128-byte boundaries, the width of the boxes in which a GEMM fetches
    it: a box of rows on 16-byte boundaries touches two lines a row and takes twice as long (1000 x 2096 x 2096, FP8, input gradient, rows
    of 2096 / 2112 / 2176 bytes: 10.0 / 7.5 / 6.6 us; BF16 12.5 / 9.5 / 9.5).  Rows of less than 128 bytes, and columns that are no multiple
    of 16, are not padded."""
    per = 128 // dtype.itemsize
    pitch = -(-cols // per) * per if cols % 16 == 0 and cols >= per else cols
    return torch.empty_strided((rows, cols), (pitch, 1), dtype=dtype, device=device)   # (a slice of torch.empty: 5 us instead of 1.4)


def _padded(dsts) -> bool:
    return any(t.stride(0) != t.shape[1] for t in dsts)


def us_softmax_fwd(S, alpha, P, stream=None):
    _check("us_softmax_fwd", _entry("us_softmax_fwd")(S, alpha, P, _stream(stream)))
    return P


def us_softmax_bwd(P, dP, alpha, beta, dS, stream=None):
    _check("us_softmax_bwd", _entry("us_softmax_bwd")(P, dP, alpha, beta, dS, _stream(stream)))
    return dS


def us_softmax_xent_fwd(X, targets, out, stream=None):
    """targets: int32 CUDA tensor [rows]; out: float32 CUDA tensor [rows]."""
    assert targets.dtype == torch.int32 and out.dtype == torch.float32 and targets.is_contiguous() and out.is_contiguous()
    _check("us_softmax_xent_fwd", _entry("us_softmax_xent_fwd")(X, targets.data_ptr(), out.data_ptr(), _stream(stream)))
    return out


def us_softmax_xent_bwd(X, targets, g, beta, dX, stream=None):
    """g: float32 CUDA tensor [rows] or None (ones)."""
    assert targets.dtype == torch.int32 and targets.is_contiguous() and (g is None or (g.dtype == torch.float32 and g.is_contiguous()))
    _check("us_softmax_xent_bwd", _entry("us_softmax_xent_bwd")(X, targets.data_ptr(), g.data_ptr() if g is not None else None, beta, dX, _stream(stream)))
    return dX


def us_quant_stats(src, scale, fmt, exp_lo, nbins, stream=None):
    """Returns (snr, sum v^2, sum err^2, hist) with hist a list of nbins + 2 counts; fmt: a torch dtype.
    Allocates its small outputs and the workspace with torch and synchronises to read them back."""
    sums = torch.empty(2, dtype=torch.float64, device=src.device)
    hist = torch.empty(nbins + 2, dtype=torch.int64, device=src.device)
    ws = torch.empty(int(_lib.us_quant_stats_workspace_bytes()), dtype=torch.uint8, device=src.device)
    _check("us_quant_stats", _lib.us_quant_stats(C.byref(mat(src)), scale, _TORCH_DTYPES[fmt], exp_lo, nbins, sums.data_ptr(),
                                                 hist.data_ptr(), ws.data_ptr(), ws.numel(), _stream(stream)))
    s = sums.cpu().tolist()
    return (s[0] / s[1] if s[1] > 0 else float("inf")), s[0], s[1], hist.cpu().tolist()


def _vec(t: torch.Tensor) -> us_mat:
    """A 1-D parameter tensor as a 1 x n us_mat."""
    return mat(t.view(1, -1))


def us_layer_norm_fwd(X, w, c, eps, Y, stream=None):
    _check("us_layer_norm_fwd", _entry("us_layer_norm_fwd")(X, w.view(1, -1), c.view(1, -1), eps, Y, _stream(stream)))
    return Y


def us_layer_norm_bwd_workspace_bytes(rows: int, cols: int) -> int:
    return int(_lib.us_layer_norm_bwd_workspace_bytes(rows, cols))


def us_layer_norm_bwd(X, w, G, eps, beta_x, beta_wc, dX, dw, dc, ws, stream=None):
    """ws: a uint8 CUDA tensor of at least us_layer_norm_bwd_workspace_bytes(rows, cols) bytes."""
    _check("us_layer_norm_bwd", _entry("us_layer_norm_bwd")(
        X, w.view(1, -1), G, eps, beta_x, beta_wc, dX, dw.view(1, -1),
        dc.view(1, -1), ws, ws, _stream(stream)))
    return dX, dw, dc


def us_scales_linear(b: int, m: int, n: int, constrained: bool = False):
    a, bx, bw = C.c_float(), C.c_float(), C.c_float()
    _check("us_scales_linear", _lib.us_scales_linear(b, m, n, int(constrained), C.byref(a), C.byref(bx), C.byref(bw)))
    return a.value, bx.value, bw.value


def us_scales_gelu(constrained: bool = False):
    a, b = C.c_float(), C.c_float()
    _check("us_scales_gelu", _lib.us_scales_gelu(int(constrained), C.byref(a), C.byref(b)))
    return a.value, b.value


def us_scales_residual(tau: float):
    """(sqrt(1 - tau), sqrt(tau)) as the float32 values the library uses."""
    a, b = C.c_float(), C.c_float()
    _check("us_scales_residual", _lib.us_scales_residual(tau, C.byref(a), C.byref(b)))
    return a.value, b.value


def us_scales_attention(s: int, d_head: int, constrained: bool = False) -> dict:
    """Factors of scaled dot-product attention (see the header), keyed as the encoder driver uses them."""
    v = [C.c_float() for _ in range(6)]
    _check("us_scales_attention", _lib.us_scales_attention(s, d_head, int(constrained), *[C.byref(x) for x in v]))
    a_s, b_s, sm, a_c, b_p, b_v = (x.value for x in v)
    return dict(alpha_s=a_s, beta_Q=b_s, beta_K=b_s, sm=sm, alpha_c=a_c, beta_P=b_p, beta_V=b_v)


def us_status_string(status: int) -> str:
    return _lib.us_status_string(status).decode()


def us_version() -> int:
    return int(_lib.us_version())
