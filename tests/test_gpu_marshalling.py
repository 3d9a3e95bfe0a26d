"""What the binding accepts and refuses: argument types and forms that reach the C entry points."""
from collections import UserDict

import numpy as np
import pytest
import torch

from oracle import ref
from paper_2608_04962_b200 import binding as S
from paper_2608_04962_b200 import inputs as I
from tests.util import dev, dev_bf16, host

pytestmark = pytest.mark.gpu


def _verify_case(B=5):
    w = I.scaled(I.WORKLOADS["tiny"], B=B)
    parent = I.topology(w)
    cid, cl = I.synthetic_candidates(w)
    u = I.uniforms24(3, (B, w.N))
    d = ref.tree_draw(parent, np.zeros(B, np.int32), cid, cl, u)
    lg = I.target_logits(w, parent, d["tree_tok"], boost=4.0)
    u_acc, u_fin = I.verify_uniforms(w)
    args = (dev_bf16(lg), parent, dev(d["tree_tok"]), dev(d["tree_cand"]), dev(cid), dev(cl), dev(u_acc), dev(u_fin))
    return w, parent, dev(cid), dev(cl), dev(u), args


@pytest.mark.parametrize("one", [1, np.float32(1), np.int64(1), torch.tensor(1.0)])
def test_numbers_of_any_type(one):
    w, parent, cid, cl, u, args = _verify_case()
    anchor = torch.zeros(w.B, dtype=torch.int32, device="cuda")
    a, b = S.tree_draw(parent, anchor, cid, cl, u, temperature=one), S.tree_draw(parent, anchor, cid, cl, u)
    assert all(torch.equal(a[n], b[n]) for n in b)
    a, b = S.verify_nucleus(*args, one, temperature=one), S.verify_nucleus(*args, 1.0)
    assert all(torch.equal(a[n], b[n]) for n in ("n_acc", "path_node", "out_tok", "row_max", "row_sum"))


def test_what_is_not_a_number_raises_and_leaves_the_binding_usable():
    w, parent, cid, cl, u, args = _verify_case()
    anchor = torch.zeros(w.B, dtype=torch.int32, device="cuda")
    for bad in ("1.0", None, object()):
        with pytest.raises(TypeError):
            S.tree_draw(parent, anchor, cid, cl, u, temperature=bad)
        with pytest.raises(TypeError):
            S.verify_nucleus(*args, bad)
    S.tree_draw(parent, anchor, cid, cl, u)
    S.verify_nucleus(*args, 0.95)


def test_outputs_in_any_mapping():
    *_, args = _verify_case()
    a = S.verify_nucleus(*args, 0.9)
    for drop in ((), ("min_margin", "nucleus_thr", "nucleus_sum")):
        given = UserDict({k: torch.empty_like(v) for k, v in a.items() if k not in drop})
        b = S.verify_nucleus(*args, 0.9, out=given)
        assert b is given and all(torch.equal(a[k], b[k]) for k in ("n_acc", "path_node", "out_tok"))
    del given["n_acc"]
    with pytest.raises(KeyError):
        S.verify_nucleus(*args, 0.9, out=given)


def test_a_lazily_cloned_output_leaves_its_source_alone():
    g = I.rng(4)
    R, rank, d = 40, 8, 64
    f = lambda *s: dev(g.standard_normal(s).astype(np.float32))  # noqa: E731
    zeros = lambda: torch.zeros(R, dtype=torch.int32, device="cuda")  # noqa: E731
    state = (zeros(), torch.zeros(R, device="cuda"), torch.zeros(R, device="cuda"), zeros())
    clones = [torch._lazy_clone(t) for t in state]
    one = torch.ones(1, dtype=torch.int32, device="cuda")
    S.reflex_gate(f(R, rank), f(R, rank), torch.arange(R, dtype=torch.int32, device="cuda"), None, *clones, f(R, d), zeros(), one,
                  one.view(1, 1), torch.zeros(1, device="cuda"), torch.ones(1, device="cuda"))
    assert all(int((t != 0).sum()) == 0 for t in state) and int(clones[0].sum()) == R


def test_shapes_that_attention_takes():
    w = I.scaled(I.WORKLOADS["tiny"], B=3, N=8)
    x = I.attn_inputs(w)
    ip, parent = x["kv_indptr"], np.asarray(x["parent"], np.int32)
    q, kc, vc, kt, vt = (dev_bf16(x[n]) for n in ("Q", "Kc", "Vc", "Kt", "Vt"))
    want = S.tree_attn(q, kc, vc, dev(ip), ip, kt, vt, parent)
    longer = np.concatenate([parent, np.full(5, 77, np.int32)])
    assert torch.equal(S.tree_attn(q, kc, vc, dev(ip), ip, kt, vt, longer), want)
    assert torch.equal(S.tree_attn(q, kc, vc, dev(ip), list(ip), kt, vt, [int(p) for p in parent]), want)
    Kp, Vp, pt, pi, kl = I.paged_cache(x["Kc"], x["Vc"], ip, spare_tokens=0, seed=3)
    got = S.tree_attn_paged(q, dev_bf16(Kp), dev_bf16(Vp), dev(pt), dev(pi).view(-1, 1), dev(kl).view(1, -1), kl, kt, vt, longer)
    assert torch.equal(got, want)
    with pytest.raises(S.SpecrollError):
        S.tree_attn(q, kc, vc, dev(ip), ip, kt, vt, parent[:-1])


def test_layers_as_one_tensor_and_pools_of_any_shape():
    w = I.scaled(I.WORKLOADS["qwen1.5b"], B=3, N=16, K=4)
    x = I.attn_inputs(I.scaled(w, kv_kind="uniform", kv_a=100, kv_b=300))
    Kp, Vp, pt, pi, kl = I.paged_cache(x["Kc"], x["Vc"], x["kv_indptr"], spare_tokens=w.K + 1, seed=14)
    path = dev(np.tile(np.arange(w.K + 1, dtype=np.int32), (w.B, 1)))
    n_acc = dev(np.array([4, 0, 2], np.int32))
    kt, vt, tail = dev_bf16(x["Kt"]), dev_bf16(x["Vt"]), (dev(pt), dev(pi), dev(kl))
    want = [dev_bf16(Kp), dev_bf16(Vp)]
    S.commit_path_layers([kt], (vt,), path, n_acc, [want[0]], [want[1]], *tail)
    assert not torch.equal(want[0], dev_bf16(Kp))
    two = [torch.stack([dev_bf16(p)] * 2) for p in (Kp, Vp)]
    S.commit_path_layers(torch.stack([kt, kt]), torch.stack([vt, vt]), path, n_acc, two[0], two[1], *tail)
    flat = [dev_bf16(p).flatten(2) for p in (Kp, Vp)]
    S.commit_path(kt, vt.flatten(2), path, n_acc, *flat, *tail)
    listed = [dev_bf16(p).flatten(1) for p in (Kp, Vp)]
    S.commit_path_layers([kt], [vt], path, n_acc, [listed[0]], [listed[1]], *tail)
    for i in range(2):
        assert torch.equal(two[i][0], want[i]) and torch.equal(two[i][1], want[i])
        assert torch.equal(flat[i].view_as(want[i]), want[i]) and torch.equal(listed[i].view_as(want[i]), want[i])
    with pytest.raises(S.SpecrollError):
        S.commit_path_layers([kt], [vt.flatten(2)], path, n_acc, [want[0]], [want[1]], *tail)
    with pytest.raises(TypeError):
        S.commit_path_layers((t for t in [kt]), [vt], path, n_acc, [want[0]], [want[1]], *tail)


def test_flat_arrays_of_a_verification_from_hidden_states():
    w, parent, cid, cl, u, args = _verify_case()
    g = torch.Generator(device="cuda").manual_seed(1)
    W = torch.randn((w.V, 64), generator=g, device="cuda").to(torch.bfloat16)
    h = torch.randn((w.B, w.N, 64), generator=g, device="cuda").to(torch.bfloat16)
    a = S.verify_fused(h, W, *args[1:])
    longer = np.concatenate([parent, [3]])
    b = S.verify_fused(h, W, longer, args[2].view(-1), args[3].view(-1), args[4], args[5], args[6].view(-1), args[7])
    assert all(np.array_equal(host(a[k]), host(b[k])) for k in a)
    with pytest.raises(S.SpecrollError):
        S.verify_fused(h, W, parent, args[2][:-1], *args[3:])
