"""What the binding accepts and refuses: argument types and forms that reach the C entry points."""
import numpy as np
import pytest
import torch

from oracle import ref
from paper_2608_04962_b200 import binding as S
from paper_2608_04962_b200 import inputs as I
from tests.util import dev, dev_bf16

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
