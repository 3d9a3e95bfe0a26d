"""Entry points of the C ABI called one by one through ctypes, as a host that drives the steps itself does."""
import ctypes as C

import numpy as np
import pytest
import torch

from oracle import ref
from paper_2608_04962_b200 import binding as S
from paper_2608_04962_b200 import inputs as I
from tests.test_gpu_verify_fused import _case
from tests.util import dev, dev_bf16, host

pytestmark = pytest.mark.gpu


def call(name, *args):
    """Tensors and host arrays as pointers, Python numbers as 32-bit integers or floats; on the current stream."""
    keep = []

    def conv(a):
        if a is None:
            return C.c_void_p(0)
        if isinstance(a, torch.Tensor):
            return C.c_void_p(a.data_ptr())
        if isinstance(a, np.ndarray):
            keep.append(np.ascontiguousarray(a, np.int32))
            return keep[-1].ctypes.data_as(C.c_void_p)
        if isinstance(a, C.Structure):
            return C.byref(a)
        return a if not isinstance(a, (int, float)) else (C.c_int32(a) if isinstance(a, int) else C.c_float(a))

    rc = getattr(S.lib(), name)(*[conv(a) for a in args], C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert rc == 0, (name, rc)


def empty(*shape, dtype=torch.int32):
    return S.alloc(shape, dtype=dtype, device="cuda")


def verify_outputs(w):
    return {"n_acc": empty(w.B), "path_node": empty(w.B, w.K + 1), "out_tok": empty(w.B, w.K + 1), "term_node": empty(w.B),
            "term_kind": empty(w.B), "min_margin": empty(w.B, dtype=torch.float32)}


class Hidden:
    """A verification from hidden states, step by step."""

    def __init__(self, name, B, V, d, T, seed):
        w, parent, H, W, o, cid, cl, dr, u_acc, u_fin = _case(name, B, V, d, T, seed)
        self.w, self.parent, self.T, self.V, self.d = w, parent, T, V, d
        self.H, self.W, self.cid, self.cl = dev_bf16(H), dev_bf16(W), dev(cid), dev(cl)
        self.tok, self.tcand, self.u_acc, self.u_fin = dev(dr["tree_tok"]), dev(dr["tree_cand"]), dev(u_acc), dev(u_fin)
        self.desc = S.VerifyDesc(B, w.N, w.K, w.k, V, T, 0)
        self.want, self.want_logit = empty(B * w.N, w.k), empty(B * w.N, w.k, dtype=torch.bfloat16)
        self.rmax, self.rsum = empty(B, w.N, dtype=torch.float32), empty(B, w.N, dtype=torch.float32)

    def project(self, tiles=True):
        R, L = self.w.B * self.w.N, S.lib()
        for n in ("specroll_target_head_stats_workspace_bytes", "specroll_target_head_tile_mass_bytes"):
            getattr(L, n).restype = C.c_size_t
        self.ws = empty(L.specroll_target_head_stats_workspace_bytes(R, self.d, self.V), dtype=torch.uint8)
        self.mass = empty(L.specroll_target_head_tile_mass_bytes(R, self.V), dtype=torch.uint8)
        call("specroll_verify_want_ids", self.desc, self.parent, self.cid, self.want)
        call("specroll_target_head_stats_tiles", R, self.d, self.V, self.T, self.H, self.W, self.want, self.w.k, self.rmax, self.rsum,
             self.want_logit, self.mass if tiles else None, self.ws, C.c_size_t(self.ws.numel()))

    def hidden(self):
        o = verify_outputs(self.w)
        call("specroll_verify_hidden", self.desc, self.d, self.H, self.W, self.want_logit, self.mass, self.rmax, self.rsum, self.parent,
             self.tok, self.tcand, self.cid, self.cl, self.u_acc, self.u_fin, *o.values())
        return o


def test_inputs_written_by_the_kernel_in_front_of_the_walk():
    """The uniforms come from a library kernel that lets the next one start early, between the projection and the walk."""
    x = Hidden("tiny", 256, 4096, 256, 1.0, 7)
    x.project()
    g = I.rng(5)
    d = 12288
    X, Pi = dev(g.random((x.w.B, d), dtype=np.float32)), dev(g.random((x.w.N, d), dtype=np.float32))
    want_u = S.reflex_sketch(X, Pi)      # (positive, about 8 ** -0.5 each)
    torch.cuda.synchronize()
    x.u_acc = want_u
    want = {k: v.clone() for k, v in x.hidden().items()}
    x.u_acc = empty(x.w.B, x.w.N, dtype=torch.float32)
    for i in range(20):
        x.u_acc.zero_()
        call("specroll_reflex_sketch", x.w.B, d, x.w.N, X, None, Pi, x.u_acc)
        got = x.hidden()
        for k in want:
            assert torch.equal(got[k], want[k]), (i, k)
    x.u_acc.zero_()
    assert not torch.equal(x.hidden()["n_acc"], want["n_acc"])


@pytest.mark.parametrize("name,B,V,d,T", [("tiny", 41, 1032, 128, 1.0), ("qwen7b", 6, 8200, 256, 0.7), ("qwen1.5b", 3, 151936, 64, 1.3)])
def test_the_steps_of_a_verification_from_hidden_states_one_by_one(name, B, V, d, T):
    """Walk on the wanted logits, the last nodes' rows by the storing projection, the draw from them; against the oracle on
    the stored logits of the same projection.  Bounds: those of the verification on stored logits."""
    x = Hidden(name, B, V, d, T, 60 + B)
    x.project(tiles=False)
    w, o = x.w, verify_outputs(x.w)
    S.lib().specroll_verify_workspace_bytes.restype = C.c_size_t
    ws = empty(S.lib().specroll_verify_workspace_bytes(C.byref(x.desc)), dtype=torch.uint8)
    call("specroll_verify_walk_sparse", x.desc, x.want_logit, x.rmax, x.rsum, x.parent, x.tok, x.tcand, x.cid, x.cl, x.u_acc,
         *o.values(), ws, C.c_size_t(ws.numel()))
    last = S.target_head_rows(S.gather_hidden(x.H, o["term_node"]), x.W)
    call("specroll_verify_terminal_rows", x.desc, last, x.rmax, o["n_acc"], o["term_node"], x.u_fin, o["out_tok"], ws,
         C.c_size_t(ws.numel()))
    logits = S.bf16_bits(S.target_head_rows(x.H.view(B * w.N, d), x.W)).reshape(B, w.N, V)
    want = ref.verify(logits, x.parent, host(x.tok), host(x.tcand), host(x.cid), host(x.cl), host(x.u_acc), host(x.u_fin),
                      temperature=T)
    sure = want["min_margin"] >= 1e-4
    assert sure.mean() >= 0.8
    for key in ("n_acc", "path_node", "term_node", "term_kind"):
        assert np.array_equal(host(o[key])[sure], want[key][sure]), key
    sure &= want["fin_margin"] >= 1e-6
    assert np.array_equal(host(o["out_tok"])[sure], want["out_tok"][sure])
