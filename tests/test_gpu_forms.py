"""The forms that a dispatch rule chooses between by size, at the edges of their ranges."""
import threading

import numpy as np
import pytest

from oracle import core as O
from paper_2609_13804_gb300 import synth as S
import _parity as PT
import test_gpu_parity as GP
import test_gpu_train as GT

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


def attention_can_cancel(H, sel):
    """Whether the tables' kernel asks in its rounds for a cancelling attention output (none of these decoders'
    START rows cancels by itself): a value longer than half of a residual."""
    z = O.decoder_tokens(np.concatenate([H, sel["s_start"][None]]).astype(np.float64), sel)
    x = O.layer_norm(z, 1e-5, sel.get("ln1_g"), sel.get("ln1_b"))
    v = x @ sel["Wv_s"].T.astype(np.float64) @ sel["Wo_s"].T.astype(np.float64)
    z, v = z - z.mean(-1, keepdims=True), v - v.mean(-1, keepdims=True)
    return 4 * (v ** 2).sum(-1).max() > (z[:-1] ** 2).sum(-1).min()


def run_with_tables(B, run):
    """run(), which makes one selection: by tables, whose two kernels are launched together."""
    B.sp_profile_begin()
    try:
        return run()
    finally:
        assert B.sp_profile_end()["select"]["launches"] == 2


@pytest.mark.parametrize("D", [128, 1024])     # attention outputs that may cancel the residual, and that cannot
@pytest.mark.parametrize("n_vis,h,g,k_max,group", [
    ([1, 126, 2, 127], 128, 1, 8, 0),          # one row tile, its last row and one more
    ([1, 9, 17, 33, 49], 128, 1, 49, 0),       # CTAs without candidates
    ([254, 255, 31], 256, 1, 40, 0),           # the edges of one column tile
    ([509, 33], 512, 1, 96, 0),                # history registers at their smaller capacity
    ([330], 1024, 1, 223, 0),                  # and at the larger one
    ([1016, 700], 128, 5, 120, 0),             # the widest slices, grouped rounds
    ([64, 300], 128, 16, 100, 100),            # candidate groups, the longest lists
])
def test_selection_tables(B, n_vis, h, g, k_max, group, D):
    """The table-driven selection at the edges of its tiles, slices and lists, with LN2's gain and bias."""
    w = S.tiny_workload(93, n_vis, [1] * len(n_vis), D=D, D_text=128, h=h, enc_head_dim=64, k_max=k_max,
                        group_size=group, g=g)
    scale = (4.0 if h <= 256 else 2.0) if D == 128 else min(3.0, 512.0 / h)
    sel = PT.scale_decoder(S.make_selector_weights(w, ln_affine=True), scale)
    assert attention_can_cancel(S.make_memory(w), sel) == (D == 128)
    run_with_tables(B, lambda: GP._run_select_case(B, w, scale=scale))


@pytest.mark.parametrize("D", [128, 1024])
def test_training_tables(B, D):
    """The aggregates from the tables over a long history, in both forms of the rounds."""
    w = S.tiny_workload(94, [260, 210], [1, 1], D=D, D_text=128, h=128, k_max=200)
    scale = 4.0 if D == 128 else 3.0
    sel = PT.scale_decoder(S.make_selector_weights(w, ln_affine=True), scale)
    assert attention_can_cancel(S.make_memory(w), sel) == (D == 128)
    GT._train_case(B, w, tau=1.0, beta=0.99, scale=scale, targets=[200, 150])


def test_selection_tables_and_keys_agree(B):
    """A workspace without room for the tables takes the general kernel: the same selection."""
    w = S.tiny_workload(95, [700, 650], [1, 1], D=128, D_text=128, h=128, k_max=48)
    s = S.SelectorShape(D=128, D_text=128, h=128, n_enc_layers=0)
    selector = B.Selector(s, PT.scale_decoder(S.make_selector_weights(w, ln_affine=True), 4.0), DEV)
    H, bias = B.dev_f32(S.make_memory(w), DEV), B.dev_f32(np.full(2, -1e30, np.float32), DEV)
    full = run_with_tables(B, lambda: B.sp_select(selector, w.n_vis, w.n_txt, H=H, stop_bias=bias, k_max=48))
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


def test_selection_tables_where_attention_cancels_the_residual(B):
    """A decoder whose attention output is nearly the negative of its residual (|u| about 0.03 |z|): the tables'
    logits are as close to the 64-bit ones as the general kernel's, which forms u.  Both start from the same
    precomputed rows, whose rounding that cancellation magnifies alike."""
    n, h, k = [300], 128, 24
    w = S.tiny_workload(97, n, [1], D=128, D_text=128, h=h, k_max=k)
    sel = PT.scale_decoder(S.make_selector_weights(w, ln_affine=False), 4.0)
    eye = np.eye(h, dtype=np.float32)
    sel["Wq_s"], sel["Wk_s"] = 1.5 * eye, 1.5 * eye  # every position attends to itself
    sel["Wv_s"], sel["Wo_s"] = eye, (-0.98 * eye + 0.02 / np.sqrt(h) * S.normal(97, "R", (h, h))).astype(np.float32)

    def unit(m):  # decoder tokens with a standard deviation of one
        return (m / (m.astype(np.float64) @ sel["W_in"].T.astype(np.float64)).std(-1, keepdims=True)).astype(np.float32)

    H, sel["s_start"] = unit(S.make_memory(w)), unit(sel["s_start"][None])[0]
    bias = np.full(1, -1e30, np.float32)
    selector = B.Selector(S.SelectorShape(D=128, D_text=128, h=h, n_enc_layers=0), sel, DEV)
    args = dict(H=B.dev_f32(H, DEV), stop_bias=B.dev_f32(bias, DEV), k_max=k)
    full = run_with_tables(B, lambda: B.sp_select(selector, n, [1], **args))
    need = general_workspace(n, 128, h)
    assert need < full["_ws"].numel()
    small = B.sp_select(selector, n, [1], ws=full["_ws"][:need].clone(), **args)
    torch.cuda.synchronize()
    replay, _ = PT.replayer(H, n, sel, k_max=k, g=1, group_size=0, biases=bias)
    err = []
    for out in (full, small):
        assert int(out["err"].item()) == 0
        ref = np.asarray(replay(0, [int(x) for x in np_(out["order"])[0]])["gap"][:k])
        err.append(np.linalg.norm(np_(out["gap"])[0, :k] - ref) / np.linalg.norm(ref))
    print("relative errors of the gaps, tables and general kernel:", err)
    # (two roundings of the operands in place of one)
    assert err[0] <= 2 * err[1], err
    selector.close()


@pytest.mark.parametrize("n,h,g,k_max", [(2100, 128, 1, 12), (2100, 128, 5, 12), (300, 1024, 1, 40), (300, 1024, 5, 60)])
def test_a_nan_candidate_is_passed_over_where_keys_are_streamed(B, n, h, g, k_max):
    """Episodes whose keys do not fit shared memory select as if a candidate with a NaN row were not there, also
    where the tables take their place (h = 1,024 here). (All logits negative: the keys rank a NaN next to zero.)"""
    w = S.tiny_workload(98, [n], [1], D=128, D_text=128, h=h, k_max=k_max)
    sel = PT.scale_decoder(S.make_selector_weights(w, ln_affine=True), 4.0 if h == 128 else 1.0)
    sel["ln2_b"] = 3 * S.normal(98, "b", (h,))
    away = sel["Wk_p"].T @ sel["Wq_p"] @ sel["ln2_b"]
    H, bias = S.make_memory(w) - 8 * away / np.linalg.norm(away), B.dev_f32(np.full(1, -1e30, np.float32), DEV)
    selector = B.Selector(S.SelectorShape(D=128, D_text=128, h=h, n_enc_layers=0), sel, DEV)
    j = n // 3
    args = dict(stop_bias=bias, k_max=w.k_max, g=g)
    want = B.sp_select(selector, [n - 1], [1], H=B.dev_f32(np.delete(H, j, 0), DEV), **args)
    H[j] = np.nan
    got = B.sp_select(selector, [n], [1], H=B.dev_f32(H, DEV), **args)
    torch.cuda.synchronize()
    assert int(got["err"].item()) == 0 and int(want["err"].item()) == 0
    order = np_(want["order"])
    np.testing.assert_array_equal(np_(got["order"]), order + (order >= j))
    np.testing.assert_array_equal(np_(got["gap"]), np_(want["gap"]))
    selector.close()
