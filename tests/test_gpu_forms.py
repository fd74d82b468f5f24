"""The forms that a dispatch rule chooses between by size, at the edges of their ranges."""
import numpy as np
import pytest

from oracle import core as O
from paper_2609_13804_gb300 import synth as S
import _parity as PT

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda"


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2609_13804_gb300 import binding
    binding.lib()
    return binding


def np_(t):
    return t.float().cpu().numpy() if t.dtype == torch.bfloat16 else t.cpu().numpy()


@pytest.mark.parametrize("D", [384, 2176, 4096, 4224])
def test_encoder_row_forms(B, D):
    """The encoder's input assembly and LayerNorms: rows of a warp (with and without a remainder) and rows
    wider than the register form, within the encoder's stated tolerance."""
    w = S.tiny_workload(91, [21, 9], [0, 3], D=D, D_text=128, h=128, enc_head_dim=64)
    w.selector.enc_ffn_mult = 1
    w.selector.n_enc_layers = 1
    s = w.selector
    sel, inp = S.make_selector_weights(w, ln_affine=True), S.make_inputs(w)
    selector = B.Selector(s, sel, DEV)
    out = B.sp_select(selector, w.n_vis, w.n_txt, X=B.dev_bf16(inp["X"], DEV), E_text=B.dev_bf16(inp["E_text"], DEV),
                      stop_bias=B.dev_f32(np.zeros(2), DEV), k_max=4, memory=True)
    torch.cuda.synchronize()
    assert int(out["err"].item()) == 0
    got, v0, t0 = np_(out["memory"]), 0, 0
    for n, t in zip(w.n_vis, w.n_txt):
        Et = O.text_projection(inp["E_text"][t0:t0 + t], sel, s.ln_eps, s.g_text)
        ref = O.encoder(inp["X"][v0:v0 + n], Et, sel, s.enc_heads, s.ln_eps, store="bf16")
        assert np.abs(got[v0:v0 + n] - ref).max() <= PT.HID_MAX_ABS * np.sqrt((ref ** 2).mean())
        v0, t0 = v0 + n, t0 + t
    selector.close()
