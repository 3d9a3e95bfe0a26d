"""GPU: verification from hidden states (projection with fused statistics and tile masses, then the walk and the last token from
one vocabulary tile) against the verification on stored logits and against the CPU oracle."""
import numpy as np
import pytest
import torch

from oracle import ref
from paper_2608_04962_b200 import binding as S
from paper_2608_04962_b200 import inputs as I
from tests.util import dev, dev_bf16, host

pytestmark = pytest.mark.gpu


def _case(name, B, V, d, T, seed):
    w = I.scaled(I.WORKLOADS[name], B=B, V=V, d=d, temperature=T, k=min(I.WORKLOADS[name].k, 8))
    parent = I.topology(w)
    depth = I.node_depths(parent)
    g = I.rng(seed)
    H = I.f32_to_bf16_bits((2.0 * g.standard_normal((B, w.N, d))).astype(np.float32))
    W = I.f32_to_bf16_bits((g.standard_normal((V, d)) / np.sqrt(d)).astype(np.float32))
    o = ref.target_head(H.reshape(B * w.N, d), W, temperature=T)
    lg = I.bf16_bits_to_f32(o["logits"]).reshape(B, w.N, V)
    # proposals close to the target: head h proposes the target's top tokens at the first node of depth h, with noise
    cid = np.zeros((B, w.K, w.k), np.int32)
    cl = np.zeros((B, w.K, w.k), np.float32)
    for h in range(w.K):
        u = int(np.flatnonzero(depth == min(h, depth.max()))[0])
        noisy = lg[:, u, :] + 0.7 * g.standard_normal((B, V))
        order = np.argsort(-noisy, axis=-1)[:, : w.k]
        cid[:, h] = order
        cl[:, h] = np.take_along_axis(noisy, order, -1)
    u_draw = I.uniforms24(seed + 1, (B, w.N))
    dr = ref.tree_draw(parent, np.zeros(B, np.int32), cid, cl, u_draw, temperature=T)
    u_acc, u_fin = I.verify_uniforms(w)
    return w, parent, H, W, o, cid, cl, dr, u_acc, u_fin


@pytest.mark.parametrize("name,B,V,d,T", [("qwen1.5b", 40, 8192, 256, 1.0), ("qwen7b", 12, 20008, 512, 0.7),
                                          ("tiny", 4, 1024, 256, 1.0)])
def test_fused_path_equals_the_path_through_stored_logits(name, B, V, d, T):
    w, parent, H, W, o, cid, cl, dr, u_acc, u_fin = _case(name, B, V, d, T, 90 + B)
    dH, dW = dev_bf16(H), dev_bf16(W)
    args = (parent, dev(dr["tree_tok"]), dev(dr["tree_cand"]), dev(cid), dev(cl), dev(u_acc), dev(u_fin))
    f = {k: host(v) for k, v in S.verify_fused(dH, dW, *args, temperature=T).items()}
    # the storing form of the same projection gives bit-identical logits, and specroll_verify is oracle-checked
    logits = S.target_head_rows(dH.reshape(B * w.N, d), dW).reshape(B, w.N, V)
    u = {k: host(v) for k, v in S.verify(logits, *args, temperature=T).items()}
    torch.cuda.synchronize()
    assert np.array_equal(f["row_max"], u["row_max"])
    np.testing.assert_allclose(f["row_sum"], u["row_sum"], rtol=2e-5)
    same = (f["n_acc"] == u["n_acc"]) & (f["path_node"] == u["path_node"]).all(1) & (f["out_tok"] == u["out_tok"]).all(1) & \
           (f["term_node"] == u["term_node"]) & (f["term_kind"] == u["term_kind"])
    # the two normalisers differ in the last bits: only a decision within 1e-4 of its uniform may flip
    for b in np.flatnonzero(~same):
        assert u["min_margin"][b] < 1e-4 or (f["n_acc"][b] == u["n_acc"][b] and (f["path_node"][b] == u["path_node"][b]).all())
    assert (~same).sum() <= max(1, B // 100)
    if B >= 12:
        assert u["n_acc"].max() >= 1      # the case does accept something
    # and against the oracle on the oracle's own logits (a few logits differ by one bf16 unit between fp32 and fp64
    # accumulation, which can move a decision): most sequences agree token for token
    oo = ref.verify(o["logits"].reshape(B, w.N, V), parent, dr["tree_tok"], dr["tree_cand"], cid, cl, u_acc, u_fin,
                    temperature=T)
    agree = (f["n_acc"] == oo["n_acc"]) & (f["out_tok"] == oo["out_tok"]).all(1)
    assert agree.mean() >= 0.9


@pytest.mark.parametrize("name,B,V,d,T", [("tiny", 300, 264, 64, 1.0), ("tiny", 100, 4360, 192, 1.3), ("qwen1.5b", 60, 256, 128, 0.7),
                                          ("qwen7b", 3, 40, 4096, 1.0)])
def test_last_token_from_one_tile(name, B, V, d, T):
    """One to eight CTAs per sequence; vocabularies below, at and above one tile, with a ragged last one."""
    test_fused_path_equals_the_path_through_stored_logits(name, B, V, d, T)


@pytest.mark.parametrize("name,B,V,d,T", [("tiny", 300, 4104, 512, 1.0), ("qwen7b", 20, 40008, 64, 0.7), ("tiny", 150, 264, 4096, 1.3),
                                          ("tiny", 2, 8, 128, 1.0)])
def test_last_token_follows_the_projections_own_logits(name, B, V, d, T):
    """Two large products that cancel, one at either end of the contraction: a logit then follows the order of its sum by many
    bf16 steps, and a last token drawn from logits of another order is often another token.  Compared with the oracle on the
    stored logits of the same projection; excluded are draws within 3e-6 of a bound (the tiles' masses are fp32 sums of
    exponentials with a relative error of 1e-6) and walks within 1e-4 of a uniform."""
    w, parent, H, W, _, cid, cl, dr, u_acc, u_fin = _case(name, B, V, d, T, 190 + B)
    big, a = I.f32_to_bf16_bits(np.float32([8192.0, -1.0])), I.f32_to_bf16_bits(I.rng(3).standard_normal(V).astype(np.float32))
    H[:, :, 0] = H[:, :, -1] = big[0]
    W[:, 0], W[:, -1] = a, a ^ np.uint16(0x8000)
    dH, dW = dev_bf16(H), dev_bf16(W)
    args = (parent, dev(dr["tree_tok"]), dev(dr["tree_cand"]), dev(cid), dev(cl), dev(u_acc), dev(u_fin))
    f = {k: host(v) for k, v in S.verify_fused(dH, dW, *args, temperature=T).items()}
    logits = S.bf16_bits(S.target_head_rows(dH.reshape(B * w.N, d), dW)).reshape(B, w.N, V)
    o = ref.verify(logits, parent, dr["tree_tok"], dr["tree_cand"], cid, cl, u_acc, u_fin, temperature=T)
    sure = (o["min_margin"] >= 1e-4) & (o["fin_margin"] >= 3e-6)
    assert sure.mean() >= 0.8
    for key in ("n_acc", "path_node", "out_tok", "term_node", "term_kind"):
        assert np.array_equal(f[key][sure], o[key][sure]), key
