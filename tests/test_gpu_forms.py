"""The forms that a dispatch rule chooses between by size, at the edges of their ranges."""
import threading

import numpy as np
import pytest

from oracle import core as O
from paper_2609_13804_gb300 import synth as S
import _parity as PT
import test_gpu_parity as GP

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


def general_workspace(n_vis, D, h):
    """What the general kernel carves from a given memory (one layer, D >= h), in 256-byte slices."""
    rows = sum(n_vis) + 2
    return 4 * rows * (D + h + 2 * h + 3 * h) + 2 * rows * 3 * D + 4 * len(n_vis) * 1024 + 16 * 256


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


@pytest.mark.parametrize("n_vis,h,g,k_max,group", [
    ([1, 126, 2, 127], 128, 1, 8, 0),          # one row tile, its last row and one more
    ([1, 9, 17, 33, 49], 128, 1, 49, 0),       # CTAs without candidates
    ([254, 255, 31], 256, 1, 40, 0),           # the edges of one column tile
    ([509, 33], 512, 1, 96, 0),                # history registers at their smaller capacity
    ([330], 1024, 1, 223, 0),                  # and at the larger one
    ([1016, 700], 128, 5, 120, 0),             # the widest slices, grouped rounds
    ([64, 300], 128, 16, 100, 100),            # candidate groups, the longest lists
])
def test_selection_tables(B, n_vis, h, g, k_max, group):
    """The table-driven selection at the edges of its tiles, slices and lists, with LN2's gain and bias."""
    w = S.tiny_workload(93, n_vis, [1] * len(n_vis), D=128, D_text=128, h=h, enc_head_dim=64, k_max=k_max,
                        group_size=group, g=g)
    GP._run_select_case(B, w, scale=4.0 if h <= 256 else 2.0)


def test_selection_tables_and_keys_agree(B):
    """A workspace without room for the tables takes the general kernel: the same selection."""
    w = S.tiny_workload(95, [700, 650], [1, 1], D=128, D_text=128, h=128, k_max=48)
    s = S.SelectorShape(D=128, D_text=128, h=128, n_enc_layers=0)
    selector = B.Selector(s, PT.scale_decoder(S.make_selector_weights(w, ln_affine=True), 4.0), DEV)
    H, bias = B.dev_f32(S.make_memory(w), DEV), B.dev_f32(np.full(2, -1e30, np.float32), DEV)
    full = B.sp_select(selector, w.n_vis, w.n_txt, H=H, stop_bias=bias, k_max=48)
    need = general_workspace(w.n_vis, 128, 128)
    assert need < full["_ws"].numel()
    small = B.sp_select(selector, w.n_vis, w.n_txt, H=H, stop_bias=bias, k_max=48, ws=full["_ws"][:need].clone())
    torch.cuda.synchronize()
    assert int(full["err"].item()) == 0 and int(small["err"].item()) == 0
    assert (full["margin"][:, :48] > 1e-4).all()
    np.testing.assert_array_equal(np_(full["order"]), np_(small["order"]))
    g0, g1 = np_(full["gap"])[:, :48], np_(small["gap"])[:, :48]
    assert np.abs(g0 - g1).max() <= 2e-4 * max(1.0, np.abs(g1).max())
    selector.close()


def test_selections_of_different_sizes_from_two_threads(B):
    """Every selection gets the shared memory that its own size needs, whatever another thread launches meanwhile.
    (STOP wins at once, so that the threads spend their time launching.)"""
    shapes = [([24, 24], 8), ([1016, 900], 223)]
    w = [S.tiny_workload(96 + i, n, [1, 1], D=128, D_text=128, h=128, k_max=k) for i, (n, k) in enumerate(shapes)]
    s = S.SelectorShape(D=128, D_text=128, h=128, n_enc_layers=0)
    selector = B.Selector(s, S.make_selector_weights(w[0]), DEV)
    bias = B.dev_f32(np.full(2, 1e30, np.float32), DEV)
    H = [B.dev_f32(S.make_memory(x), DEV) for x in w]
    failed = []

    def work(i):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                ws = None
                for _ in range(3000):
                    out = B.sp_select(selector, w[i].n_vis, w[i].n_txt, H=H[i], stop_bias=bias, k_max=w[i].k_max,
                                      traces=False, ws=ws)
                    ws = out["_ws"]
                torch.cuda.current_stream().synchronize()
            assert int(out["err"].item()) == 0 and out["count"].tolist() == [0, 0]
        except Exception as e:
            failed.append((shapes[i], e))

    torch.cuda.synchronize()
    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
    selector.close()
