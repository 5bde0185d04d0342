"""Bounded waits of the digit products (csrc/slice_gemm.cu) and of the
eigenvector estimate (csrc/eigvec.cu) running out, through the library's test
hook: CSS_ERR_TIMEOUT after the caller's budget, and the next call on the same
workspace gives what it gave before.  With sync = 0 css_read_status reports it."""
import ctypes as C

import pytest
import torch

import css_inputs as ci
from tests.gpu_helpers import dev_matrix

pytestmark = pytest.mark.gpu

BUDGET_NS = 20_000_000   # 20 ms: far longer than any wait of these problems


def _p(t):
    return C.c_void_p(t.data_ptr())


class _Call:
    """One of the calls on a workspace of its own: (opts) -> (code, outputs)."""

    def __init__(self, kind):
        from paper_1312_6838_gb300 import _lib as L, css
        self.L, self.lib = L, L.load()
        self.kind = kind
        m, n, k = 700, 21000, 150   # split and unsplit products, more tiles than SMs
        o = L.default_opts()
        if kind == "lowrank":
            g = torch.Generator(device="cuda").manual_seed(5)
            self.W = torch.randn(130, n, generator=g, device="cuda", dtype=torch.float64)
            size = self.lib.css_workspace_size(L.CSS_OP_LOWRANK, L.CSS_F64, 0, n, 130, k := 60, 0, C.byref(o))
            self.out = [torch.empty(k, dtype=torch.float64, device="cuda"),
                        torch.empty(k, n, dtype=torch.float64, device="cuda")]
        else:
            self.A, _ = dev_matrix(ci.lowrank_uv(m, n, 200, 0.05, 813), torch.float64)
            self.S = torch.arange(k, dtype=torch.int32, device="cuda")
            op = {"select": L.CSS_OP_SELECT, "embed": L.CSS_OP_EMBED, "residual": L.CSS_OP_BACKWARD}[kind]
            size = self.lib.css_workspace_size(op, L.CSS_F64, m, n, 0, 16 if kind == "select" else k, 0, C.byref(o))
            f64 = dict(dtype=torch.float64, device="cuda")
            self.out = {"select": lambda: [torch.empty(16, dtype=torch.int32, device="cuda"), torch.empty(17, **f64),
                                           torch.zeros(1, dtype=torch.int32, device="cuda")],
                        "embed": lambda: [torch.empty(k, m, **f64), torch.empty(k, n, **f64)],
                        "residual": lambda: [css.empty_colmajor(m, n, torch.float64), torch.empty(1, **f64)]}[kind]()
        self.m, self.n, self.k, self.size = m, n, k, size
        buf = torch.empty(size + 256, dtype=torch.uint8, device="cuda")
        self.keep, self.ws = buf, C.c_void_p((buf.data_ptr() + 255) // 256 * 256)

    def __call__(self, hook=0, sync=1):
        o = self.L.default_opts()
        o.spin_budget_ns, o.test_unmet_wait, o.sync = BUDGET_NS, hook, sync
        st = C.c_void_p(torch.cuda.current_stream().cuda_stream)
        null, f64, out, m, n, k = C.c_void_p(0), self.L.CSS_F64, self.out, self.m, self.n, self.k
        if self.kind == "lowrank":
            return self.lib.css_lowrank(_p(self.W), n, null, 1, 0, n, 130, k, _p(out[0]), null, 1, _p(out[1]), n, null,
                                        null, self.ws, self.size, C.byref(o), st)
        if self.kind == "select":
            return self.lib.css_select(_p(self.A), f64, m, n, m, 16, _p(out[0]), _p(out[1]), _p(out[2]), null, self.ws,
                                       self.size, C.byref(o), st)
        if self.kind == "embed":
            return self.lib.css_embed(_p(self.A), f64, m, n, m, _p(self.S), k, _p(out[0]), m, _p(out[1]), n, self.ws,
                                      self.size, C.byref(o), st)
        return self.lib.css_residual_backward(_p(self.A), f64, m, n, m, _p(self.S), k, 1.0, _p(out[0]), m, _p(out[1]),
                                              self.ws, self.size, C.byref(o), st)

    def status(self):
        return self.lib.css_read_status(self.ws, C.c_void_p(torch.cuda.current_stream().cuda_stream))


@pytest.mark.parametrize("kind,hook", [("select", 2), ("embed", 2), ("residual", 2), ("lowrank", 2), ("lowrank", 1)])
def test_wait_runs_out_then_the_next_call_is_right(kind, hook):
    call = _Call(kind)
    assert call() == 0
    ref = [t.clone() for t in call.out]
    assert call(hook) == call.L.CSS_ERR_TIMEOUT
    assert call() == 0
    assert all(torch.equal(a, b) for a, b in zip(call.out, ref))
    assert call(hook, sync=0) == 0
    assert call.status() == call.L.CSS_ERR_TIMEOUT
    assert call(sync=0) == 0
    assert call.status() == 0
    assert all(torch.equal(a, b) for a, b in zip(call.out, ref))
