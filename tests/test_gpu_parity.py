"""CUDA path vs float64 oracle, through the C-ABI binding (needs a B200)."""
import numpy as np
import pytest
import torch

import paper_2504_02692_b200 as g
import workloads as wl
from oracle import gptaq_oracle as orc
from tests import helpers as hp

pytestmark = pytest.mark.gpu


def batches_of(cfg, device="cpu", n_batches=None, tokens=None):
    nb = cfg.n_batches if n_batches is None else n_batches
    return [wl.make_batch(cfg, b, device, tokens) for b in range(nb)]


def test_library_is_the_cuda_one():
    lib = g.load_library()
    assert lib._name.endswith("libgptaq.so")


def test_cfg1_full_parity():
    cfg = wl.CONFIGS["cfg1"]
    out = hp.check_layer(cfg, wl.make_weight(cfg), batches_of(cfg))
    hp.assert_parity(out)
    # tensor-core statistics (split H, single-term fp16 dXX^T): the sums carry the operand rounding, 2^-11 per factor
    assert out["H_rel"] < 1e-5 and out["D_rel"] < 2.0 ** -10 and out["P_rel"] < 5e-3


@pytest.mark.parametrize("alpha", [0.0, 1.0])
def test_cfg1_alpha_limits(alpha):
    cfg = wl.scaled(wl.CONFIGS["cfg1"], alpha=alpha)
    out = hp.check_layer(cfg, wl.make_weight(cfg), batches_of(cfg))
    hp.assert_parity(out)
    if alpha == 0.0:
        assert out["P_rel"] == 0.0   # P == 0 exactly: the solve is GPTQ


@pytest.mark.parametrize("n,m,tokens,nb,bits,group,sym,B", [
    (200, 37, 333, 2, 4, 0, False, 32),      # ragged everything, per-channel
    (200, 37, 333, 2, 3, 8, False, 32),      # small groups, ragged last group/block
    (328, 70, 1000, 1, 4, 32, True, 64),     # symmetric groups, B = 64
    (520, 150, 2048, 2, 2, 128, False, 128), # 2-bit, several 128-blocks plus a ragged tail
    (1, 5, 16, 1, 4, 0, False, 32),          # a single input neuron
    (129, 3, 700, 1, 8, 0, True, 128),       # one column beyond a tile
])
def test_ragged_shapes(n, m, tokens, nb, bits, group, sym, B):
    cfg = wl.scaled(wl.CONFIGS["cfg1"], name="ragged", n=n, m=m, batch_tokens=tokens, n_batches=nb,
                    bits=bits, group=group, sym=sym, blocksize=B, outlier_channels=min(2, n),
                    act="student")
    out = hp.check_layer(cfg, wl.make_weight(cfg), batches_of(cfg))
    hp.assert_parity(out)


@pytest.mark.parametrize("n,m,B,group,sym,bits", [(576, 70, 64, 64, True, 4), (640, 33, 32, 32, False, 3),
                                                   (516, 129, 128, 0, False, 4), (576, 120, 64, 16, False, 4),
                                                   (648, 50, 128, 8, True, 4)])
def test_tensor_path_block_sizes_and_tails(n, m, B, group, sym, bits):
    """Widths >= 512 (float32-grade tensor-core products) with the smaller lazy-batch blocks, a width that is
    a multiple of 4 only, row counts that do not fill the last CTA, and grids per group of fewer than 32 columns
    (the general column kernel feeding the fp16-split tensor-core update)."""
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="tails", n=n, m=m, batch_tokens=1500, n_batches=2, bits=bits, group=group,
                    sym=sym, blocksize=B, outlier_channels=5)
    out = hp.check_layer(cfg, wl.make_weight(cfg), batches_of(cfg))
    hp.assert_parity(out)


@pytest.mark.parametrize("n,m,B,group,bits", [(1416, 100, 128, 128, 4), (1160, 40, 64, 64, 3)])
def test_super_panels_and_super_blocks(n, m, B, group, bits):
    """Widths beyond one super-panel of the factorisation (1024 columns) and beyond one super-block of the
    lazy-batch update (8 blocks), with ragged last panels: the rank-1024 update, the updates inside a
    super-panel at a column offset and the wide update with one scale per row all run."""
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="super", n=n, m=m, batch_tokens=3000, n_batches=2, bits=bits, group=group,
                    blocksize=B, outlier_channels=12)
    out = hp.check_layer(cfg, wl.make_weight(cfg), batches_of(cfg), rows=np.arange(0, m, 3))
    hp.assert_parity(out)


def test_no_damping_keeps_the_unbounded_operand_form():
    """damp = 0: nothing bounds the entries of the factor and of its inverse in advance, so rank updates and block inverse are
    plain float32 products, while P and the lazy-batch updates keep their fp16-split form."""
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="nodamp", n=768, m=40, batch_tokens=4096, n_batches=2, damp=0.0,
                    outlier_channels=6)
    out = hp.check_layer(cfg, wl.make_weight(cfg), batches_of(cfg))
    hp.assert_parity(out)


@pytest.mark.parametrize("scale", [1e-3, 250.0])
def test_activation_units_do_not_matter(scale):
    """The fp16-split operands of the solve carry power-of-two scales taken from their own ranges: the
    same layer with its activations in other units (U scales with 1 / unit, P not at all) keeps parity."""
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="units", n=640, m=48, batch_tokens=2048, n_batches=2, outlier_channels=6)
    bt = [(X * scale, Xfp * scale) for X, Xfp in batches_of(cfg)]
    out = hp.check_layer(cfg, wl.make_weight(cfg), bt)
    hp.assert_parity(out)


def test_strided_inputs():
    """Activations and weights given as views with a leading dimension larger than n."""
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="strided", n=512, m=64, batch_tokens=1024, n_batches=2, outlier_channels=5)
    W = wl.make_weight(cfg)
    bt = batches_of(cfg)
    ref = hp.gpu_layer(cfg, W, bt)
    st = g.LayerState(cfg.n, cfg.m, cfg.batch_tokens, cfg.blocksize, total_tokens=cfg.tokens)
    for X, Xfp in bt:
        big = torch.zeros((2, X.shape[0], cfg.n + 12), device="cuda")
        big[0, :, :cfg.n] = X.cuda(); big[1, :, :cfg.n] = Xfp.cuda()
        g.gptaq_accumulate(st.handle, big[0, :, :cfg.n], big[1, :, :cfg.n])
    g.gptaq_factor(st.handle, cfg.damp)
    g.gptaq_build_P(st.handle, cfg.alpha)
    Wbig = torch.zeros((cfg.m, cfg.n + 20), device="cuda")
    Wbig[:, :cfg.n] = W.cuda()
    G = hp.n_groups(cfg.n, cfg.group)
    codes = torch.empty((cfg.m, cfg.n), dtype=torch.uint8, device="cuda")
    sc = torch.empty((cfg.m, G), dtype=torch.float32, device="cuda")
    zp = torch.empty((cfg.m, G), dtype=torch.float32, device="cuda")
    g.gptaq_quantize(st.handle, Wbig[:, :cfg.n], cfg.bits, cfg.group, cfg.sym, cfg.blocksize, codes, sc, zp, None)
    assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
    assert np.array_equal(codes.cpu().numpy(), ref.codes)
    assert np.array_equal(Wbig[:, :cfg.n].cpu().numpy().astype(np.float64), ref.Wq)      # in place, strided
    assert float(Wbig[:, cfg.n:].abs().max()) == 0.0                                    # nothing written beyond n
    st.close()


def test_cfg4_shape_row_subset():
    """ViT-shaped layer at full n and tokens; the oracle loop replays a seeded row subset
    (rows are independent)."""
    cfg = wl.CONFIGS["cfg4"]
    W = wl.make_weight(cfg)
    rows = np.sort(np.random.default_rng(0).choice(cfg.m, 192, replace=False))
    out = hp.check_layer(cfg, W, batches_of(cfg), rows=rows)
    hp.assert_parity(out)


def test_mid_llama_like_groups():
    """LLaMA-like recipe (Student-t, outlier channels, W4 g128) at n = 1024."""
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="cfg2_small", n=1024, m=512, batch_tokens=4096, n_batches=4,
                    outlier_channels=10)
    out = hp.check_layer(cfg, wl.make_weight(cfg), batches_of(cfg), rows=np.arange(0, 512, 4))
    hp.assert_parity(out)


def test_gated_3bit_bf16_weights():
    cfg = wl.scaled(wl.CONFIGS["cfg5"], name="cfg5_small", n=768, m=256, batch_tokens=2048, n_batches=3)
    out = hp.check_layer(cfg, wl.make_weight(cfg), batches_of(cfg), rows=np.arange(0, 256, 2))
    hp.assert_parity(out)


def test_deterministic_and_host_entry_points_agree():
    cfg = wl.scaled(wl.CONFIGS["cfg1"], n=256, m=96, batch_tokens=700, n_batches=2, group=32, blocksize=64)
    W = wl.make_weight(cfg)
    bt = batches_of(cfg)
    a = hp.gpu_layer(cfg, W, bt)
    b = hp.gpu_layer(cfg, W, bt)
    assert np.array_equal(a.codes, b.codes) and np.array_equal(a.U, b.U) and np.array_equal(a.P, b.P)
    # host entry points: pinned host buffers in, host results out
    st = g.LayerState(cfg.n, cfg.m, cfg.batch_tokens, cfg.blocksize)
    stage = torch.empty(max(2 * cfg.batch_tokens * cfg.n * 4, g.gptaq_quantize_stage_bytes(cfg.m, cfg.n, cfg.group)),
                        dtype=torch.uint8, device="cuda")
    for X, Xfp in bt:
        g.gptaq_accumulate_host(st.handle, X.pin_memory(), Xfp.pin_memory(), stage)
        torch.cuda.synchronize()
    g.gptaq_factor(st.handle, cfg.damp)
    g.gptaq_build_P(st.handle, cfg.alpha)
    G = hp.n_groups(cfg.n, cfg.group)
    codes = torch.empty((cfg.m, cfg.n), dtype=torch.uint8).pin_memory()
    scales = torch.empty((cfg.m, G), dtype=torch.float32).pin_memory()
    zeros = torch.empty((cfg.m, G), dtype=torch.float32).pin_memory()
    Wq = torch.empty((cfg.m, cfg.n), dtype=torch.float32).pin_memory()
    g.gptaq_quantize_host(st.handle, W.pin_memory(), cfg.bits, cfg.group, cfg.sym, cfg.blocksize,
                          codes, scales, zeros, stage, Wq)
    assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
    assert np.array_equal(codes.numpy(), a.codes)
    assert np.array_equal(Wq.numpy().astype(np.float64), a.Wq)
    assert g.gptaq_launch_count(st.handle) > 0
    st.close()


def test_shared_state_quantizes_several_matrices_and_in_place():
    cfg = wl.scaled(wl.CONFIGS["cfg1"], n=192, m=64, batch_tokens=600, group=0, blocksize=64)
    bt = batches_of(cfg)
    W = wl.make_weight(cfg)
    ref = hp.gpu_layer(cfg, W, bt)
    st = g.LayerState(cfg.n, cfg.m, cfg.batch_tokens, cfg.blocksize)
    for X, Xfp in bt:
        g.gptaq_accumulate(st.handle, X.cuda(), Xfp.cuda())
    g.gptaq_factor(st.handle, cfg.damp)
    g.gptaq_build_P(st.handle, cfg.alpha)
    for rep in range(2):      # q/k/v-style: same statistics, several weights
        Wd = W.cuda().clone()
        codes = torch.empty((cfg.m, cfg.n), dtype=torch.uint8, device="cuda")
        sc = torch.empty((cfg.m, 1), dtype=torch.float32, device="cuda")
        zp = torch.empty((cfg.m, 1), dtype=torch.float32, device="cuda")
        g.gptaq_quantize(st.handle, Wd, cfg.bits, cfg.group, cfg.sym, cfg.blocksize, codes, sc, zp, None)
        assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
        assert np.array_equal(codes.cpu().numpy(), ref.codes)
        assert np.array_equal(Wd.cpu().numpy().astype(np.float64), ref.Wq)   # in place when d_Wq is NULL
    st.close()


@pytest.mark.parametrize("terms", [0, g.GPTAQ_TERM_ERR, g.GPTAQ_TERM_ASYM])
@pytest.mark.parametrize("n,group,B", [(160, 0, 32), (640, 128, 128)])
def test_update_term_switches(terms, n, group, B):
    """Ablation switches (GPTQ, GPTAQ', RTN) against the oracle with the same terms."""
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="terms", n=n, m=48, batch_tokens=1536, n_batches=1, group=group,
                    blocksize=B, outlier_channels=3, alpha=1.0)
    bt = batches_of(cfg)
    W = wl.make_weight(cfg)
    st = g.LayerState(cfg.n, cfg.m, cfg.batch_tokens, cfg.blocksize, total_tokens=cfg.tokens)
    for X, Xfp in bt:
        g.gptaq_accumulate(st.handle, X.cuda(), Xfp.cuda())
    g.gptaq_factor(st.handle, cfg.damp)
    g.gptaq_build_P(st.handle, cfg.alpha)
    with pytest.raises(g.GptaqError):
        g.gptaq_set_update_terms(st.handle, 4)
    g.gptaq_set_update_terms(st.handle, terms)
    G = hp.n_groups(cfg.n, cfg.group)
    codes = torch.empty((cfg.m, cfg.n), dtype=torch.uint8, device="cuda")
    sc = torch.empty((cfg.m, G), dtype=torch.float32, device="cuda")
    zp = torch.empty((cfg.m, G), dtype=torch.float32, device="cuda")
    g.gptaq_quantize(st.handle, W.cuda(), cfg.bits, cfg.group, cfg.sym, cfg.blocksize, codes, sc, zp, None)
    assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
    so = hp.oracle_stats(cfg, bt)
    U, dead = orc.factor(so.H, so.tokens, cfg.damp)
    P = orc.build_P(so.D, so.tokens, U, cfg.alpha) if terms & g.GPTAQ_TERM_ASYM else None
    Wn = W.numpy().astype(np.float64)
    rep = orc.follow(Wn, U, P, dead, cfg.bits, cfg.group, cfg.sym, codes.cpu().numpy(),
                     sc.cpu().numpy().astype(np.float64), zp.cpu().numpy().astype(np.float64),
                     band=hp.TOL_FLIP_BAND, error_term=bool(terms & g.GPTAQ_TERM_ERR))
    assert rep.disallowed == 0 and rep.allowed <= hp.TOL_FLIP_RATE * rep.total, rep
    if terms == 0:
        rtn = orc.quantize(Wn, U, None, dead, cfg.bits, cfg.group, cfg.sym, update=False)
        assert np.mean(codes.cpu().numpy() != rtn.codes) < 1e-3
    st.close()


@pytest.mark.parametrize("n,m,group,B", [(160, 24, 0, 32), (640, 40, 128, 128), (516, 16, 0, 64)])
def test_rowwise_P_matches_the_row_by_row_form(n, m, group, B):
    """gptaq_build_P_rowwise (Eq. "unparallel") against the oracle's row-by-row form: stage-wise from the device's
    own dXX^T and U widened to float64, end to end through the codes that the loop then produces (which shows
    that the operand copies of the lazy-batch update were made from this P)."""
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="rowwise", n=n, m=m, batch_tokens=2048, n_batches=2, group=group,
                    blocksize=B, outlier_channels=5)
    batches = batches_of(cfg)
    st = g.LayerState(cfg.n, m, cfg.batch_tokens, cfg.blocksize, total_tokens=cfg.tokens)
    h = st.handle
    for X, Xfp in batches:
        g.gptaq_accumulate(h, X.cuda(), Xfp.cuda())
    D_dev = st.D().cpu().numpy().astype(np.float64)
    g.gptaq_factor(h, cfg.damp)
    U_dev = np.triu(st.H().cpu().numpy().astype(np.float64))
    g.gptaq_build_P_rowwise(h, cfg.alpha)
    assert g.gptaq_sync_status(h)[0] == g.GPTAQ_OK
    P_dev = st.D().cpu().numpy().astype(np.float64)
    assert np.abs(np.tril(P_dev)).max() == 0.0
    want = orc.build_P_rowwise(D_dev, cfg.tokens, U_dev, cfg.alpha)
    assert hp.rel_fro(P_dev, want) <= 1e-5
    # the loop on this P against the oracle's end-to-end U and P
    ost = hp.oracle_stats(cfg, batches)
    U, dead = orc.factor(ost.H, ost.tokens, cfg.damp)
    P = orc.build_P_rowwise(ost.D, ost.tokens, U, cfg.alpha)
    W = wl.make_weight(cfg)
    G = hp.n_groups(n, group)
    codes = torch.empty((m, n), dtype=torch.uint8, device="cuda")
    scales = torch.empty((m, G), device="cuda"); zeros = torch.empty((m, G), device="cuda")
    Wq = torch.empty((m, n), device="cuda")
    g.gptaq_quantize(h, W.cuda(), cfg.bits, group, cfg.sym, B, codes, scales, zeros, Wq)
    assert g.gptaq_sync_status(h)[0] == g.GPTAQ_OK
    rep = orc.follow(W.numpy().astype(np.float64), U, P, dead, cfg.bits, group, cfg.sym, codes.cpu().numpy(),
                     scales.cpu().numpy().astype(np.float64), zeros.cpu().numpy().astype(np.float64), band=hp.TOL_FLIP_BAND)
    assert rep.disallowed == 0 and rep.allowed <= hp.TOL_FLIP_RATE * rep.total, rep
    assert rep.grid_rel_err <= hp.TOL_GRID and rep.zero_mismatch == 0, rep
    # wrong call order and the width limit are refused on the host
    with pytest.raises(g.GptaqError):
        g.gptaq_build_P_rowwise(h, cfg.alpha)
    st.close()


@pytest.mark.parametrize("n,m,group,B,bf16", [(160, 40, 0, 32, False), (200, 24, 32, 64, False),
                                                (640, 96, 128, 128, False), (768, 64, 0, 128, True)])
def test_act_order(n, m, group, B, bf16):
    """Columns sorted by diag(H).  Several orders are valid where two diagonal entries agree to within the
    rounding of the statistics, so the device's permutation is checked for validity (it sorts the device's own
    diagonal; against the float64 diagonal only near-ties may be swapped) and then handed to the oracle."""
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="act", n=n, m=m, batch_tokens=2048, n_batches=2, group=group,
                    blocksize=B, outlier_channels=4, w_bf16=bf16)
    bt = batches_of(cfg)
    W = wl.make_weight(cfg)
    st = g.LayerState(cfg.n, cfg.m, cfg.batch_tokens, cfg.blocksize, total_tokens=cfg.tokens)
    g.gptaq_set_act_order(st.handle, True)
    assert st.perm() is None
    for X, Xfp in bt:
        g.gptaq_accumulate(st.handle, X.cuda(), Xfp.cuda())
    diag_dev = torch.diagonal(st.H()).cpu().numpy().astype(np.float64)
    g.gptaq_factor(st.handle, cfg.damp)
    g.gptaq_build_P(st.handle, cfg.alpha)
    perm = st.perm().cpu().numpy().astype(np.int64)
    assert sorted(perm.tolist()) == list(range(n))
    assert np.all(np.diff(diag_dev[perm]) <= 0)                       # sorts the device's own diagonal
    so = hp.oracle_stats(cfg, bt)
    d64 = np.diag(so.H)[perm]
    assert np.all(np.diff(d64) <= 2.0 ** -9 * d64[:-1])               # only near-ties out of float64 order
    Ug = st.H().cpu().numpy().astype(np.float64)
    Pg = st.D().cpu().numpy().astype(np.float64)
    G = hp.n_groups(cfg.n, cfg.group)
    codes = torch.empty((m, n), dtype=torch.uint8, device="cuda")
    sc = torch.empty((m, G), dtype=torch.float32, device="cuda")
    zp = torch.empty((m, G), dtype=torch.float32, device="cuda")
    Wq = torch.empty((m, n), dtype=torch.float32, device="cuda")
    Wd = W.cuda().to(torch.bfloat16) if bf16 else W.cuda()
    with pytest.raises(g.GptaqError):                                  # needs a second buffer
        g.gptaq_quantize(st.handle, W.cuda(), cfg.bits, cfg.group, cfg.sym, cfg.blocksize, codes, sc, zp, None)
    g.gptaq_quantize(st.handle, Wd, cfg.bits, cfg.group, cfg.sym, cfg.blocksize, codes, sc, zp, Wq)
    assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
    Wn = W.numpy().astype(np.float64)
    U, P, dead, res, _ = orc.solve_act_order(Wn, so.H, so.D, so.tokens, cfg.damp, cfg.alpha, cfg.bits, cfg.group,
                                             cfg.sym, perm=perm)
    assert hp.rel_fro(np.triu(Ug), U) <= hp.TOL_FACTOR
    assert hp.rel_fro(np.triu(Pg, 1), P) <= 5e-3
    cg = codes.cpu().numpy()
    rep = orc.follow(Wn[:, perm], U, P, dead, cfg.bits, cfg.group, cfg.sym, cg[:, perm],
                     sc.cpu().numpy().astype(np.float64), zp.cpu().numpy().astype(np.float64), band=hp.TOL_FLIP_BAND)
    assert rep.disallowed == 0 and rep.allowed <= hp.TOL_FLIP_RATE * rep.total, rep
    assert rep.grid_rel_err <= hp.TOL_GRID and rep.zero_mismatch == 0, rep
    # dequantized weights come back in the caller's column order and match codes and grids
    gsz = cfg.group if cfg.group > 0 else n
    scp = np.repeat(sc.cpu().numpy(), gsz, axis=1)[:, :n]
    zpp = np.repeat(zp.cpu().numpy(), gsz, axis=1)[:, :n]
    deq_sorted = scp * (cg[:, perm].astype(np.float32) - zpp)
    assert np.array_equal(Wq.cpu().numpy()[:, perm], deq_sorted.astype(np.float32))
    J_gpu, J_orc = orc.objective(Wn, Wq.cpu().numpy().astype(np.float64), so), orc.objective(Wn, res.Wq, so)
    assert abs(J_gpu - J_orc) <= hp.TOL_OBJECTIVE * J_orc
    st.close()


@pytest.mark.parametrize("n,m,group,B,act,bf16,ndead", [(192, 24, 32, 64, True, False, 0), (640, 40, 128, 128, True, False, 0),
                                                        (768, 33, 64, 128, True, True, 0), (640, 20, 128, 128, False, False, 0),
                                                        (320, 30, 64, 64, True, False, 3), (512, 33, 64, 64, False, True, 3),
                                                        (768, 24, 128, 128, True, True, 0), (1024, 24, 32, 64, True, True, 3),
                                                        (320, 64, 32, 128, True, True, 3),
                                                        # more rows than a round of CTAs, without the tensor cores
                                                        (96, 4737, 32, 64, False, False, 3), (129, 4800, 16, 32, True, False, 0)])
def test_static_groups(n, m, group, B, act, bf16, ndead):
    """Static groups, with and without act_order: grids per group of the caller's columns from the original
    weights (inputs that never fired count as zero weights); the loop replayed by the oracle in the device's
    processing order with those grids."""
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="static_groups", n=n, m=m, batch_tokens=2048, n_batches=2, group=group,
                    blocksize=B, outlier_channels=4, w_bf16=bf16)
    bt = batches_of(cfg)
    W = wl.make_weight(cfg)
    if ndead:
        for X, Xfp in bt:
            X[:, 7:7 + ndead] = 0.0
            Xfp[:, 7:7 + ndead] = 0.0
        W[:, 7] = 30.0 * W.abs().max()          # a dead input's weight must not stretch its group's grid
    st = g.LayerState(cfg.n, cfg.m, cfg.batch_tokens, cfg.blocksize, total_tokens=cfg.tokens)
    g.gptaq_set_act_order(st.handle, act)
    g.gptaq_set_static_groups(st.handle, True)
    for X, Xfp in bt:
        g.gptaq_accumulate(st.handle, X.cuda(), Xfp.cuda())
    g.gptaq_factor(st.handle, cfg.damp)
    g.gptaq_build_P(st.handle, cfg.alpha)
    perm = st.perm().cpu().numpy().astype(np.int64) if act else np.arange(n)
    G = hp.n_groups(n, group)
    codes = torch.empty((m, n), dtype=torch.uint8, device="cuda")
    sc = torch.empty((m, G), dtype=torch.float32, device="cuda")
    zp = torch.empty((m, G), dtype=torch.float32, device="cuda")
    Wq = torch.empty((m, n), dtype=torch.float32, device="cuda")
    Wd = W.cuda().to(torch.bfloat16) if bf16 else W.cuda()
    g.gptaq_quantize(st.handle, Wd, cfg.bits, group, cfg.sym, B, codes, sc, zp, Wq)
    assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
    so = hp.oracle_stats(cfg, bt)
    Wn = W.numpy().astype(np.float64)
    U, P, dead, res, _ = orc.solve_act_order(Wn, so.H, so.D, so.tokens, cfg.damp, cfg.alpha, cfg.bits, group, cfg.sym,
                                             perm=perm, static_groups=True)
    cg, scn, zpn = codes.cpu().numpy(), sc.cpu().numpy(), zp.cpu().numpy()
    dead0 = np.zeros(n, bool)
    dead0[perm] = dead
    assert dead0.sum() == ndead
    # the grids are those of the original weights, float32 arithmetic on both sides of a min/max.  A zero
    # point whose pre-rounding value -lo / scale is a tie (x.5: bf16 weights have short mantissas, and a group
    # whose extremes are symmetric gives exactly maxq / 2) may round either way, to the floor or to the ceiling
    assert np.abs(scn - res.scales).max() <= 1e-6 * np.abs(res.scales).max()
    W0 = Wn.copy()
    W0[:, dead0] = 0.0
    lo = np.stack([np.minimum(W0[:, k * group:(k + 1) * group].min(axis=1), 0.0) for k in range(G)], axis=1)
    t = -lo / res.scales
    tie = np.abs(t - np.floor(t) - 0.5) <= 1e-6
    differs = zpn != res.zeros
    assert not (differs & ~tie).any(), int((differs & ~tie).sum())
    assert np.isin(zpn[differs] - np.floor(t[differs]), (0.0, 1.0)).all()
    if differs.any():
        # the oracle's free run again, with the device's choice at the ties
        r2 = orc.quantize(Wn[:, perm], U, P, dead, cfg.bits, group, cfg.sym,
                          static=(res.scales, zpn.astype(np.float64), perm // group))
        Wq2 = np.empty_like(r2.Wq)
        Wq2[:, perm] = r2.Wq
        res = orc.QuantResult(None, res.scales, zpn.astype(np.float64), Wq2)
    rep = orc.follow(Wn[:, perm], U, P, dead, cfg.bits, group, cfg.sym, cg[:, perm], scn.astype(np.float64),
                     zpn.astype(np.float64), band=hp.TOL_FLIP_BAND, static=(Wn, perm // group, dead0))
    assert rep.disallowed == 0 and rep.allowed <= hp.TOL_FLIP_RATE * rep.total, rep
    assert rep.grid_rel_err <= 1e-6 and rep.zero_mismatch == 0, rep
    # the outputs dequantize with the grid of group column // group, in the caller's column order
    g_of = np.arange(n) // group
    assert np.array_equal(Wq.cpu().numpy(), (scn[:, g_of] * (cg.astype(np.float32) - zpn[:, g_of])).astype(np.float32))
    J_gpu, J_orc = orc.objective(Wn, Wq.cpu().numpy().astype(np.float64), so), orc.objective(Wn, res.Wq, so)
    assert abs(J_gpu - J_orc) <= hp.TOL_OBJECTIVE * J_orc
    st.close()


@pytest.mark.parametrize("n,m,group,B,sym,bits", [(160, 40, 0, 32, False, 3), (200, 24, 8, 32, False, 2),
                                                   (640, 96, 128, 128, False, 3), (576, 130, 64, 64, True, 3)])
def test_clip_search(n, m, group, B, sym, bits):
    """Grids chosen by the clipping-range search.  Which candidate wins is decided by sums of squares that the
    device takes in float32: where two candidates are within rounding of each other either is valid, so the
    oracle's follow mode checks that the device's grid IS a candidate and that its float64 error equals the
    best one up to 1e-5, then replays the codes with it."""
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="clip", n=n, m=m, batch_tokens=2048, n_batches=1, group=group,
                    blocksize=B, sym=sym, bits=bits, outlier_channels=3)
    bt = batches_of(cfg)
    W = wl.make_weight(cfg)
    clip = (24, 0.4)
    st = g.LayerState(cfg.n, cfg.m, cfg.batch_tokens, cfg.blocksize, total_tokens=cfg.tokens)
    with pytest.raises(g.GptaqError):
        g.gptaq_set_clip_search(st.handle, 8, 1.5)
    g.gptaq_set_clip_search(st.handle, *clip)
    for X, Xfp in bt:
        g.gptaq_accumulate(st.handle, X.cuda(), Xfp.cuda())
    g.gptaq_factor(st.handle, cfg.damp)
    g.gptaq_build_P(st.handle, cfg.alpha)
    G = hp.n_groups(cfg.n, cfg.group)
    codes = torch.empty((m, n), dtype=torch.uint8, device="cuda")
    sc = torch.empty((m, G), dtype=torch.float32, device="cuda")
    zp = torch.empty((m, G), dtype=torch.float32, device="cuda")
    Wq = torch.empty((m, n), dtype=torch.float32, device="cuda")
    g.gptaq_quantize(st.handle, W.cuda(), cfg.bits, cfg.group, cfg.sym, cfg.blocksize, codes, sc, zp, Wq)
    assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
    so = hp.oracle_stats(cfg, bt)
    U, dead = orc.factor(so.H, so.tokens, cfg.damp)
    P = orc.build_P(so.D, so.tokens, U, cfg.alpha)
    Wn = W.numpy().astype(np.float64)
    rep = orc.follow(Wn, U, P, dead, cfg.bits, cfg.group, cfg.sym, codes.cpu().numpy(),
                     sc.cpu().numpy().astype(np.float64), zp.cpu().numpy().astype(np.float64),
                     band=hp.TOL_FLIP_BAND, clip=clip)
    assert rep.disallowed == 0 and rep.allowed <= hp.TOL_FLIP_RATE * rep.total, rep
    assert rep.grid_rel_err <= hp.TOL_GRID and rep.zero_mismatch == 0, rep
    # the search does change grids on this input, and the objective matches the oracle's
    plain = orc.quantize(Wn, U, P, dead, cfg.bits, cfg.group, cfg.sym)
    res = orc.quantize(Wn, U, P, dead, cfg.bits, cfg.group, cfg.sym, clip=clip)
    assert np.mean(res.scales < plain.scales * (1 - 1e-9)) > 0.05
    J_gpu, J_orc = orc.objective(Wn, Wq.cpu().numpy().astype(np.float64), so), orc.objective(Wn, res.Wq, so)
    assert abs(J_gpu - J_orc) <= 5 * hp.TOL_OBJECTIVE * J_orc, (J_gpu, J_orc)
    st.close()


def test_correlated_inputs_stress():
    """Correlated channels (X <- X A, A = identity + low rank): cond(H_d) grows from ~1e3 (independent
    channels of the benchmark layers) to ~2e4.  float32 sums and a float32 factorization then carry
    cond * 1e-8 of relative error into U, which is past the 1e-4 bound of the benchmark layers for any choice of
    statistics arithmetic (the exact-float32 path included); this test records that, and checks what must
    hold regardless: a clean status, the loop's parity given the device's own U and P, and the objective."""
    n = 1024
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="stress", n=n, m=128, batch_tokens=4096, n_batches=4, outlier_channels=10)
    gen = torch.Generator().manual_seed(5)
    A = torch.eye(n) + 10.0 / n ** 0.5 * (torch.randn(n, 64, generator=gen) @ torch.randn(64, n, generator=gen)) / 8.0
    bt = [((X @ A).contiguous(), (Xfp @ A).contiguous()) for X, Xfp in batches_of(cfg)]
    W = wl.make_weight(cfg)
    run = hp.gpu_layer(cfg, W, bt)
    assert run.status[0] == g.GPTAQ_OK
    so = hp.oracle_stats(cfg, bt)
    U, dead = orc.factor(so.H, so.tokens, cfg.damp)
    P = orc.build_P(so.D, so.tokens, U, cfg.alpha)
    Hd, _ = orc.damped_hessian(so.H, so.tokens, cfg.damp)
    cond = np.linalg.cond(Hd)
    U_rel = hp.rel_fro(np.triu(run.U), U)
    assert 5e3 < cond < 1e5 and U_rel < 1e-7 * cond, (cond, U_rel)
    Wn = W.numpy().astype(np.float64)
    rep = orc.follow(Wn, np.triu(run.U), np.triu(run.P, 1), dead, cfg.bits, cfg.group, cfg.sym, run.codes, run.scales,
                     run.zeros, band=hp.TOL_FLIP_BAND)
    assert rep.disallowed == 0 and rep.allowed <= hp.TOL_FLIP_RATE * rep.total, rep
    res = orc.quantize(Wn, U, P, dead, cfg.bits, cfg.group, cfg.sym)
    J_gpu, J_orc = orc.objective(Wn, run.Wq, so), orc.objective(Wn, res.Wq, so)
    assert abs(J_gpu - J_orc) <= hp.TOL_OBJECTIVE * J_orc, (J_gpu, J_orc)
    print(f"correlated stress: cond {cond:.2e}, U rel {U_rel:.2e}, J rel {abs(J_gpu - J_orc) / J_orc:.2e}, "
          f"free-running mismatch {np.mean(run.codes != res.codes):.2e}")


def test_call_order_empty_inputs_and_bad_arguments():
    n, m = 96, 8
    st = g.LayerState(n, m, 64, 32)
    h = st.handle
    X = torch.randn(64, n, device="cuda")
    with pytest.raises(g.GptaqError) as e:
        g.gptaq_factor(h, 0.01)                      # nothing accumulated yet
    assert e.value.status == g.GPTAQ_ERR_BAD_STATE
    with pytest.raises(g.GptaqError) as e:
        g.gptaq_build_P(h, 1.0)
    assert e.value.status == g.GPTAQ_ERR_BAD_STATE
    g.gptaq_accumulate(h, X[:0], X[:0])              # empty batch: no-op
    assert g.gptaq_tokens(h) == 0
    g.gptaq_accumulate(h, X, X)
    assert g.gptaq_tokens(h) == 64
    g.gptaq_factor(h, 0.01)
    with pytest.raises(g.GptaqError) as e:
        g.gptaq_accumulate(h, X, X)                  # sums are gone after factor
    assert e.value.status == g.GPTAQ_ERR_BAD_STATE
    g.gptaq_build_P(h, 0.5)
    W = torch.randn(m, n, device="cuda")
    codes = torch.empty((m, n), dtype=torch.uint8, device="cuda")
    s = torch.empty((m, 1), device="cuda"); z = torch.empty((m, 1), device="cuda")
    for kw in (dict(bits=1), dict(bits=9), dict(blocksize=48), dict(group=24)):
        a = dict(bits=4, group=0, blocksize=32); a.update(kw)
        with pytest.raises(g.GptaqError) as e:
            g.gptaq_quantize(h, W, a["bits"], a["group"], False, a["blocksize"], codes, s, z)
        assert e.value.status == g.GPTAQ_ERR_UNSUPPORTED
    g.gptaq_quantize(h, W[:0], 4, 0, False, 32, codes[:0], s[:0], z[:0])   # m == 0: no-op
    assert g.gptaq_sync_status(h)[0] == g.GPTAQ_OK
    # X~ == X gave dXX^T == 0 exactly, hence P == 0
    assert float(st.D().abs().max()) == 0.0
    g.gptaq_reset(h)
    assert g.gptaq_tokens(h) == 0
    g.gptaq_accumulate(h, X, X)
    st.close()


def test_device_side_conditions_are_reported_not_trapped():
    n = 64
    st = g.LayerState(n, 4, 16, 32)
    h = st.handle
    X = torch.randn(16, n, device="cuda")            # rank 16 < n and no damping
    g.gptaq_accumulate(h, X, X)
    g.gptaq_factor(h, 0.0)
    status, info = g.gptaq_sync_status(h)
    assert status == g.GPTAQ_ERR_NOT_SPD and 0 <= info < n
    # the context is still usable: damped, the same statistics factor fine
    g.gptaq_reset(h)
    g.gptaq_accumulate(h, X, X)
    g.gptaq_factor(h, 0.01)
    assert g.gptaq_sync_status(h)[0] == g.GPTAQ_OK
    # a NaN in the input is reported by factor
    g.gptaq_reset(h)
    Xn = X.clone(); Xn[3, 5] = float("nan")
    g.gptaq_accumulate(h, Xn, Xn)
    g.gptaq_factor(h, 0.01)
    status, info = g.gptaq_sync_status(h)
    assert status == g.GPTAQ_ERR_NONFINITE
    st.close()
    # a NaN / Inf in the LAST column of W propagates nowhere and quantizes to a finite code: it is
    # reported from its value before the rounding, with its row, by both column kernels (groups of 8 take
    # column_loop_kernel, the others quant_block_kernel)
    for group, bad_value, row in ((32, float("nan"), 2), (8, float("inf"), 1), (0, float("nan"), 3)):
        st = g.LayerState(n, 4, 256, 32)
        h = st.handle
        Xb = torch.randn(256, n, device="cuda")
        g.gptaq_accumulate(h, Xb, Xb + 0.01 * torch.randn_like(Xb))
        g.gptaq_factor(h, 0.01)
        g.gptaq_build_P(h, 0.25)
        W = 0.02 * torch.randn(4, n, device="cuda")
        W[row, n - 1] = bad_value
        G = hp.n_groups(n, group)
        codes = torch.empty((4, n), dtype=torch.uint8, device="cuda")
        scales = torch.empty((4, G), device="cuda"); zeros = torch.empty((4, G), device="cuda")
        g.gptaq_quantize(h, W, 4, group, False, 32, codes, scales, zeros)
        status, info = g.gptaq_sync_status(h)
        assert status == g.GPTAQ_ERR_NONFINITE and info == row, (group, status, info)
        st.close()


def test_bounded_wait_runs_out_and_is_reported():
    """A wait that nothing satisfies ends by itself with a status, not a hang or a trap."""
    st = g.LayerState(64, 4, 16, 32)
    h = st.handle
    lib = g.load_library()
    assert not lib.gptaq_U(h) and not lib.gptaq_P(h)
    g.gptaq_selftest_bounded_wait(h, 0.05)
    status, info = g.gptaq_sync_status(h)
    assert status == g.GPTAQ_ERR_TIMEOUT and info == 2000000
    assert g.gptaq_status_string(status) == "bounded device wait ran out"
    g.gptaq_reset(h)                                  # clears the status; the context is still usable
    X = torch.randn(16, 64, device="cuda")
    g.gptaq_accumulate(h, X, X)
    g.gptaq_factor(h, 0.01)
    assert g.gptaq_sync_status(h)[0] == g.GPTAQ_OK
    assert lib.gptaq_U(h) == g.gptaq_H_ptr(h) and not lib.gptaq_P(h)
    g.gptaq_build_P(h, 1.0)
    assert lib.gptaq_P(h) == g.gptaq_D_ptr(h)
    st.close()


def test_dead_inputs():
    cfg = wl.scaled(wl.CONFIGS["cfg1"], n=160, m=24, batch_tokens=500, group=32, blocksize=32)
    W = wl.make_weight(cfg)
    bt = [(X.clone(), Xfp.clone()) for X, Xfp in batches_of(cfg)]
    for X, Xfp in bt:
        X[:, 7] = 0.0
        X[:, 100] = 0.0
    out = hp.check_layer(cfg, W, bt)
    hp.assert_parity(out)


def _stats_only(cfg, bt, precision, scale=1.0):
    st = g.LayerState(cfg.n, 8, cfg.batch_tokens, cfg.blocksize)
    g.gptaq_set_stats_precision(st.handle, precision)
    g.gptaq_set_kernel_timing(st.handle, True)
    for X, Xfp in bt:
        g.gptaq_accumulate(st.handle, (X * scale).cuda(), (Xfp * scale).cuda())
    assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
    H = st.H().cpu().numpy().astype(np.float64)
    D = st.D().cpu().numpy().astype(np.float64)
    # which kernel ran: the tensor-core one, once per batch at least, beyond 2^25 of tokens * n^2
    _, launches = g.gptaq_stats_kernel_time(st.handle)
    tensor = precision != g.GPTAQ_STATS_FP32 and cfg.batch_tokens * cfg.n ** 2 > 2 ** 25
    assert launches >= len(bt) if tensor else launches == 0
    st.close()
    return H, D


# (a small batch that takes float32 products whatever the precision; a single K-block of 64, padded and whole; several)
@pytest.mark.parametrize("n,tokens,nb", [(256, 64, 1), (1024, 33, 2), (1024, 64, 1), (384, 1000, 2), (1024, 4112, 2),
                                         (2052, 777, 1)])
def test_tensor_core_statistics_against_oracle(n, tokens, nb):
    """Tensor-core sums vs float64.  Elementwise error relative to sqrt(H_ii H_jj) is bounded by
    the rounding of the operands: 2^-11 per fp16 factor in the single-term mode; the split mode
    keeps ~22 bits of X for H (dXX^T stays single-term in both), the full split mode keeps them in
    dXX^T too."""
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="stats", n=n, m=8, batch_tokens=tokens, n_batches=nb,
                    outlier_channels=max(1, n // 100))
    bt = batches_of(cfg)
    so = hp.oracle_stats(cfg, bt)
    iu = np.triu_indices(n)
    iu1 = np.triu_indices(n, 1)          # of dXX^T the part above the diagonal is defined (all that P uses)
    d = np.sqrt(np.diag(so.H))
    dd = np.sqrt(np.diag(so.G))
    for prec, tolH, tolD in ((g.GPTAQ_STATS_FP16_TENSOR, 2.0 ** -10, 2.0 ** -10),
                             (g.GPTAQ_STATS_FP16_SPLIT_TENSOR, 1e-5, 2.0 ** -10),
                             (g.GPTAQ_STATS_FP16_SPLIT_FULL_TENSOR, 1e-5, 1e-5),
                             (g.GPTAQ_STATS_FP32, 1e-5, 1e-5)):
        H, D = _stats_only(cfg, bt, prec)
        errH = np.abs(H - so.H)[iu] / np.outer(d, d)[iu]
        assert errH.max() < tolH, (prec, errH.max())
        errD = np.abs(D - so.D)[iu1] / np.outer(dd, d)[iu1]
        assert errD.max() < tolD, (prec, errD.max())
        assert np.linalg.norm((D - so.D)[iu1]) / np.linalg.norm(so.D[iu1]) < tolD
        assert np.linalg.norm((H - so.H)[iu]) / np.linalg.norm(so.H[iu]) < tolH


def test_act_order_accumulates_the_whole_of_dxx_and_must_be_enabled_first():
    """The permutation of act_order mixes the two triangles of dXX^T: a handle with act_order enabled
    accumulates all of it, and enabling it after a batch went in without the lower triangle is refused
    until the sums are reset."""
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="stats", n=768, m=8, batch_tokens=1000, n_batches=2, outlier_channels=7)
    bt = batches_of(cfg)
    so = hp.oracle_stats(cfg, bt)
    d = np.sqrt(np.diag(so.H))
    dd = np.sqrt(np.diag(so.G))
    st = g.LayerState(cfg.n, 8, cfg.batch_tokens, cfg.blocksize)
    try:
        g.gptaq_set_act_order(st.handle, True)
        for X, Xfp in bt:
            g.gptaq_accumulate(st.handle, X.cuda(), Xfp.cuda())
        D = st.D().cpu().numpy().astype(np.float64)
        assert (np.abs(D - so.D) / np.outer(dd, d)).max() < 2.0 ** -10
        g.gptaq_set_act_order(st.handle, False)
        g.gptaq_reset(st.handle)
        g.gptaq_accumulate(st.handle, bt[0][0].cuda(), bt[0][1].cuda())
        with pytest.raises(g.GptaqError) as ei:
            g.gptaq_set_act_order(st.handle, True)
        assert ei.value.status == g.GPTAQ_ERR_BAD_STATE
        g.gptaq_reset(st.handle)
        g.gptaq_set_act_order(st.handle, True)
    finally:
        st.close()


def test_full_split_statistics_carry_a_hard_layer():
    """Eight bits, alpha = 1, damping 0.001, sparse gated activations: the 3e-4 that single fp16 terms leave
    in dXX^T (and in P) flips codes outside the tie band here; with both sums split the layer is exact to
    the tolerances again."""
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="hard", n=512, m=64, batch_tokens=3000, n_batches=1, bits=8, group=32,
                    blocksize=32, damp=0.001, alpha=1.0, act="gated", outlier_channels=3, seed=1002)
    out = hp.check_layer(cfg, wl.make_weight(cfg), batches_of(cfg), stats_precision=g.GPTAQ_STATS_FP16_SPLIT_FULL_TENSOR)
    hp.assert_parity(out)
    assert out["D_rel"] < 1e-5 and out["P_rel"] < 2e-5, out


@pytest.mark.parametrize("prec", [g.GPTAQ_STATS_FP16_TENSOR, g.GPTAQ_STATS_FP16_SPLIT_TENSOR,
                                  g.GPTAQ_STATS_FP16_SPLIT_FULL_TENSOR])
@pytest.mark.parametrize("scale", [3e5, 1e-7])
def test_tensor_core_statistics_rescale_out_of_range_batches(scale, prec):
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="stats", n=512, m=8, batch_tokens=640, n_batches=1, outlier_channels=5)
    bt = batches_of(cfg)
    H, D = _stats_only(cfg, bt, prec, scale)
    so = hp.oracle_stats(cfg, [(X * scale, Xfp * scale) for X, Xfp in bt])
    iu = np.triu_indices(cfg.n)
    assert np.isfinite(H).all() and np.isfinite(D).all()
    assert np.linalg.norm((H - so.H)[iu]) / np.linalg.norm(so.H[iu]) < 2.0 ** -10
    assert hp.rel_fro(np.triu(D, 1), np.triu(so.D, 1)) < 2.0 ** -10


@pytest.mark.parametrize("n,m,tokens,group,B", [
    (31, 5, 40, 0, 32),          # one tile, less than one of its rows and steps
    (33, 33, 127, 32, 32),       # one row beyond a tile, contraction just below the shortest that is shared
    (96, 40, 4097, 0, 32),       # contraction shared by eight CTAs, one step beyond whole ones
    (250, 70, 2050, 32, 64),     # no aligned rows (4-byte copies), ragged in every direction
    # more than a panel, one column beyond it (per-channel grids: the scale of a group of one column is that one updated
    # weight, and relative to a weight that happens to be small any difference is large, so the grid bound does not apply)
    (385, 200, 900, 0, 128),
])
def test_small_float32_products(n, m, tokens, group, B):
    """Products of few tiles (32 x 32 tiles, K shared by a cluster) in every step of a narrow float32 layer.  Sums of
    `tokens` rounded products: each of the at most tokens / 8 additions of a part rounds by 2^-24 of the partial sum,
    which averages to sqrt(tokens) * 2^-24; twice that is allowed."""
    cfg = wl.scaled(wl.CONFIGS["cfg1"], name="small", n=n, m=m, batch_tokens=tokens, n_batches=2, group=group, blocksize=B,
                    outlier_channels=2)
    out = hp.check_layer(cfg, wl.make_weight(cfg), batches_of(cfg), stats_precision=g.GPTAQ_STATS_FP32)
    hp.assert_parity(out)
    bound = 2.0 ** -23 * np.sqrt(2 * tokens)
    assert out["H_rel"] < bound and out["D_rel"] < 8 * bound, out       # (X~ - X cancels: 20 times smaller terms)


@pytest.mark.parametrize("n", [
    100,           # less than one panel
    129, 257,      # one column beyond a panel: no aligned rows
    516, 520,      # one super-panel on split operands, its last panel ragged; row pitch of their copies padded / not
    1024,          # ... its last panel full
    1032, 1160,    # a second super-panel of 8 columns / of one panel and 8 columns
    1153,          # the same in float32 (odd width): no block is factored ahead, the inverse beside the panels all the same
    2504,          # more rows than one warp per 4 of them can take at once
])
def test_factor_panels(n):
    """Diagonal block, rows above it and the update beside the next diagonal block, at the edges of panels and super-panels.
    The device's own H goes through the float64 factorisation, so only this step is compared: the backward error of
    n-term sums of products with 2^-22 relative error each averages to sqrt(n) * 2^-22, and U = R^-1 answers to a relative
    change of H with at most its condition number."""
    torch.manual_seed(n)
    X = torch.randn(3 * n, n, device="cuda") * torch.logspace(-0.5, 0.5, n, device="cuda")
    st = g.LayerState(n, 1, 3 * n, 32, "cuda")
    try:
        g.gptaq_accumulate(st.handle, X, X)
        H = st.H().cpu().numpy().astype(np.float64)
        g.gptaq_factor(st.handle, 0.01)
        U = np.triu(st.H().cpu().numpy().astype(np.float64))
        assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
    finally:
        st.close()
    ref, _ = orc.factor(np.triu(H) + np.triu(H, 1).T, 3 * n, 0.01)
    sv = np.linalg.svd(ref, compute_uv=False)
    bound = (sv[0] / sv[-1]) ** 2 * np.sqrt(n) * 2.0 ** -22
    assert np.linalg.norm(U - ref) <= bound * np.linalg.norm(ref), (hp.rel_fro(U, ref), bound)


@pytest.mark.parametrize("n,m,damp", [
    (1027, 150, 0.01),          # odd rows, 81 tiles of 128 x 128 and more: the 32 x 32 form all the same
    (1156, 130, 0.0),           # aligned rows, plain float32 without damping, 100 tiles
])
def test_float32_products_of_many_tiles(n, m, damp):
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="tiles", n=n, m=m, batch_tokens=5 * n, n_batches=2, damp=damp, outlier_channels=4)
    out = hp.check_layer(cfg, wl.make_weight(cfg), batches_of(cfg), rows=np.arange(0, m, 7))
    hp.assert_parity(out)


# (a diagonal block's pieces of eight columns and sub-blocks of 32, and the block beside which another is inverted)
@pytest.mark.parametrize("n", [7, 33, 64, 97, 128, 136])
def test_factor_inside_a_block(n):
    test_factor_panels(n)


@pytest.mark.parametrize("n", [1, 3, 31, 33, 97, 126, 128, 255, 383, 384, 385])
def test_correction_matrix_of_narrow_layers(n):
    """One launch up to n = 384, two products beyond: P from the device's own U and dXX^T against float64; sums of up to n float32
    products in short pieces, 2^-21 of the sum of their sizes leaves a factor of eight over one rounding each."""
    torch.manual_seed(n)
    tokens, alpha = 4 * n + 40, 0.5
    X = torch.randn(tokens, n, device="cuda")
    st = g.LayerState(n, 8, tokens, 32)
    try:
        g.gptaq_set_stats_precision(st.handle, g.GPTAQ_STATS_FP32)
        g.gptaq_accumulate(st.handle, X, X + 0.3 * torch.randn_like(X))
        D = np.triu(st.D().cpu().numpy().astype(np.float64), 1) / tokens
        g.gptaq_factor(st.handle, 0.05)
        g.gptaq_build_P(st.handle, alpha)
        U = np.triu(st.H().cpu().numpy().astype(np.float64))
        P = st.D().cpu().numpy().astype(np.float64)
        assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
    finally:
        st.close()
    ref = alpha * np.triu(np.triu(D @ U.T, 1) @ U, 1)
    size = alpha * np.triu(np.triu(abs(D) @ abs(U).T, 1) @ abs(U), 1)
    assert np.array_equal(np.tril(P), np.zeros_like(P))
    assert np.linalg.norm(P - ref) <= 2.0 ** -21 * np.linalg.norm(size)


@pytest.mark.parametrize("n", [512, 516, 1036, 1284])
def test_split_operand_row_pitch(n):
    """Tensor-core products whose fp16 operand copies have rows of 8 k and of 8 k + 4 columns (row pitch padded to a multiple
    of 8): P from the device's own U and dXX^T.  Two products after one another, each an n-term sum whose factors and
    roundings are good to 2^-22 of the products of the magnitudes."""
    torch.manual_seed(n)
    tokens, alpha = 2 * n, 0.5
    X = torch.randn(tokens, n, device="cuda")
    Xfp = X + 0.05 * torch.randn(tokens, n, device="cuda")
    st = g.LayerState(n, 1, tokens, 32, "cuda")
    try:
        g.gptaq_accumulate(st.handle, X, Xfp)
        D = np.triu(st.D().cpu().numpy().astype(np.float64), 1) / tokens
        g.gptaq_factor(st.handle, 0.05)
        g.gptaq_build_P(st.handle, alpha)
        U = np.triu(st.H().cpu().numpy().astype(np.float64))
        P = np.triu(st.D().cpu().numpy().astype(np.float64), 1)
        assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
    finally:
        st.close()
    ref = alpha * np.triu(np.triu(D @ U.T, 1) @ U, 1)
    size = alpha * np.triu(np.triu(abs(D) @ abs(U).T, 1) @ abs(U), 1)
    assert np.linalg.norm(P - ref) <= 2.0 ** -21 * np.linalg.norm(size), np.linalg.norm(P - ref) / np.linalg.norm(size)


@pytest.mark.parametrize("n,m,group,B", [
    (96, 4737, 32, 32),         # block by block, one row more than a CTA of 32 on each of 148 SMs: two to an SM
    (321, 31, 0, 128),          # odd width, a row short of a CTA
    (512, 33, 64, 64),          # the narrowest tensor-core form, exactly one launch; a row more than a CTA
    (516, 32, 128, 128),        # a launch of 512 columns and one of 4
    (1060, 40, 32, 64),         # a grid at every step; the last block has two steps, the last of them 4 columns
    (644, 4737, 64, 64),        # more rows than a round of CTAs: two parts of 2432 and 2305 rows on two streams
])
def test_quantize_launch_edges(n, m, group, B):
    """Forms of the column loop at the edges of their rows, blocks and launches (bounds as in the other parity tests)."""
    cfg = wl.scaled(wl.CONFIGS["cfg2"], name="edges", n=n, m=m, batch_tokens=3 * n, n_batches=1, group=group, blocksize=B,
                    outlier_channels=4)
    out = hp.check_layer(cfg, wl.make_weight(cfg), batches_of(cfg), rows=np.unique(np.r_[0:m:max(1, m // 16), m - 1]))
    hp.assert_parity(out)


@pytest.mark.parametrize("n,m,group,B,static,clip", [
    (512, 2385, 64, 64, False, 0),          # tensor-core form: CTAs of 32 rows, of 16 for 37 rows alone
    (644, 2369, 0, 128, False, 0),
    (126, 801, 32, 32, False, 0),           # rows of U and P that are no 16-byte multiples (one launch: the float32 products
                                            # behind it would have other tiles, and other sums, for other numbers of rows)
    (516, 2400, 128, 128, True, 0),
    (520, 2370, 32, 32, False, 20),
    (200, 801, 64, 64, False, 0),           # without tensor cores the line lies lower
    (300, 2400, 128, 128, True, 0),
    (202, 1000, 32, 64, False, 7),
])
def test_a_row_does_not_depend_on_how_many_there_are(n, m, group, B, static, clip):
    """CTAs of 32 and of 16 rows: the same arithmetic per row, hence the same results to the last bit."""
    torch.manual_seed(n)
    X = torch.randn(2 * n, n, device="cuda")
    W = 0.02 * torch.randn(m, n, device="cuda")
    st = g.LayerState(n, m, 2 * n, B)
    try:
        g.gptaq_accumulate(st.handle, X, X + 0.05 * torch.randn_like(X))
        g.gptaq_factor(st.handle, 0.01)
        g.gptaq_build_P(st.handle, 0.25)
        g.gptaq_set_static_groups(st.handle, static)
        g.gptaq_set_clip_search(st.handle, clip, 0.3)

        def quantize(rows):
            G = hp.n_groups(n, group)
            out = [torch.empty((len(rows), w), dtype=d, device="cuda") for w, d in
                   ((n, torch.uint8), (G, torch.float32), (G, torch.float32), (n, torch.float32))]
            g.gptaq_quantize(st.handle, W[rows].contiguous(), 4, group, False, B, *out)
            assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
            return out
        rows = torch.arange(m, device="cuda")
        some = torch.cat([rows[:21], rows[-16:]])
        assert [int((x[some] != y).sum()) for x, y in zip(quantize(rows), quantize(some))] == [0, 0, 0, 0]
    finally:
        st.close()


@pytest.mark.parametrize("n,m,group,B,clip,static", [
    (96, 70, 0, 32, 0, False), (128, 800, 0, 128, 0, False),        # one block: grids per channel inside the launch
    (97, 33, 0, 64, 5, False),                                      # ... before it where ranges are searched
    (100, 45, 32, 64, 0, False), (512, 40, 128, 128, 0, False),     # one launch, groups
    (512, 2400, 0, 128, 0, False), (508, 50, 64, 64, 0, True),      # (508: several launches, a working copy)
])
def test_a_single_launch_reads_the_callers_weights(n, m, group, B, clip, static):
    """From a second buffer, from bfloat16 and from rows at odd addresses: as in place on float32 copies, bit for bit."""
    torch.manual_seed(n)
    X = torch.randn(3 * n, n, device="cuda")
    X[:, n // 3] = 0.0                                              # a dead input
    wide = (0.02 * torch.randn(m, n + 5, device="cuda")).bfloat16()
    st = g.LayerState(n, m, 3 * n, B)
    try:
        g.gptaq_accumulate(st.handle, X, X + 0.05 * torch.randn_like(X))
        g.gptaq_factor(st.handle, 0.01)
        g.gptaq_build_P(st.handle, 0.25)
        g.gptaq_set_static_groups(st.handle, static)
        g.gptaq_set_clip_search(st.handle, clip, 0.3)
        G = hp.n_groups(n, group)

        def quantize(W, in_place):
            out = [torch.empty((m, w), dtype=d, device="cuda") for w, d in ((n, torch.uint8), (G, torch.float32), (G, torch.float32))]
            Wq = None if in_place else torch.empty((m, n), device="cuda")
            g.gptaq_quantize(st.handle, W, 4, group, False, B, *out, Wq)
            assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
            return out + [W if in_place else Wq]
        view = wide[:, 1:n + 1]
        want = quantize(view.float().contiguous(), True)
        floats = wide.float()
        for W in (view, view.contiguous(), floats[:, 1:n + 1], view.float().contiguous()):
            before = W.clone()
            got = quantize(W, False)
            assert [int((x != y).sum()) for x, y in zip(got, want)] == [0, 0, 0, 0]
            assert torch.equal(W, before)
    finally:
        st.close()


@pytest.mark.parametrize("n,tokens,act_order", [
    (128, 2048, False), (128, 2049, False),     # float32 products up to here / one tile of either sum, cut
    (640, 520, False), (640, 520, True),        # a few tiles, of dXX^T the upper ones or all
    (2048, 520, False),                         # as many tiles as pairs allow without a cut
])
def test_statistics_cut_by_length(n, tokens, act_order):
    """Tiles of H three times as long as those of dXX^T, cut into different numbers of items (two batches, so that the
    partial sums are added to).  Bounds as in test_tensor_core_statistics_against_oracle: operands of 22 bits for H, 11 for
    dXX^T, relative to sqrt(H_ii H_jj)."""
    torch.manual_seed(n + tokens)
    st = g.LayerState(n, 8, tokens, 128)
    try:
        g.gptaq_set_stats_precision(st.handle, g.GPTAQ_STATS_FP16_SPLIT_TENSOR)
        g.gptaq_set_act_order(st.handle, act_order)
        H, D = np.zeros((n, n)), np.zeros((n, n))
        d = np.zeros(n)
        for _ in range(2):
            X = torch.randn(tokens, n, device="cuda")
            F = X + 0.05 * torch.randn(tokens, n, device="cuda")
            g.gptaq_accumulate(st.handle, X, F)
            x, dx = X.double().cpu().numpy(), (F - X).double().cpu().numpy()
            H += x.T @ x; D += dx.T @ x; d += (dx ** 2).sum(0)
        assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
        Hg, Dg = st.H().cpu().numpy().astype(np.float64), st.D().cpu().numpy().astype(np.float64)
    finally:
        st.close()
    h = np.sqrt(np.diag(H))
    assert (np.abs(np.triu(Hg - H)) / np.outer(h, h)).max() < 1e-5
    err = Dg - D if act_order else np.triu(Dg - D, 1)
    assert (np.abs(err) / np.outer(np.sqrt(d), h)).max() < 2.0 ** -10


# (boxes of 32 columns x 128 rows: a last box of 4 columns and of 28, of 4 rows and of 124; a width whose rows are no 16-byte
# multiples; 72 tiles for the 74 pairs of 148 SMs, none of them cut; 90 tiles, of which 74 are whole and 16 cut in two, so that a
# CTA's boxes go to the sums first and to the partial sums then)
@pytest.mark.parametrize("n,tokens", [(260, 1111), (380, 1111), (388, 2048), (386, 1111), (1916, 1111), (2052, 2777)])
def test_statistics_at_the_edges_of_the_boxes(n, tokens):
    test_statistics_cut_by_length(n, tokens, False)


@pytest.mark.parametrize("n", [512, 1024, 1416])
def test_correction_matrix_sums_keep_their_precision_in_narrow_tiles(n):
    """P from the device's own U and dXX^T where the products take 64-wide tiles.  A chain of 256 contraction steps is 48
    MMAs, and each of them truncates the running sum.  The largest term of an entry of O is that of the diagonal entry of U;
    what counts are the MMAs behind it in its chain, 24 on average when chains are cut at multiples of 256.  Half a unit in
    the last place each, 2^-24 times the mean of one over a mantissa, 1 / (2 ln 2): 24 * 0.72 * 2^-24.  (Chains that begin
    at a tile's own first column have 42 of them.)"""
    torch.manual_seed(n)
    tokens, alpha = 4 * n, 0.25
    X = torch.randn(tokens, n, device="cuda")
    Xfp = X + 0.05 * torch.randn(tokens, n, device="cuda")
    st = g.LayerState(n, 1, tokens, 32, "cuda")
    try:
        g.gptaq_accumulate(st.handle, X, Xfp)
        D = np.triu(st.D().cpu().numpy().astype(np.float64), 1) / tokens
        g.gptaq_factor(st.handle, 0.01)
        g.gptaq_build_P(st.handle, alpha)
        U = np.triu(st.H().cpu().numpy().astype(np.float64))
        P = np.triu(st.D().cpu().numpy().astype(np.float64), 1)
        assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
    finally:
        st.close()
    err = hp.rel_fro(P, alpha * np.triu(np.triu(D @ U.T, 1) @ U, 1))
    assert err <= 24 * 0.72 * 2.0 ** -24, err


@pytest.mark.parametrize("n,c,group,tokens", [
    (96, 40, 32, 200),       # one block, inside it
    (96, 93, 0, 200),        # the last step of a block
    (512, 100, 128, 700),    # one launch: to later blocks through the tensor cores
    (1032, 1010, 0, 1100),   # the last block of a launch
    (1032, 1026, 0, 1100),   # the last launch
    (64, 40, 8, 200),        # groups of fewer than 32 columns
])
def test_a_non_finite_correction_is_reported(n, c, group, tokens):
    """A NaN in one channel of X~ alone: H and U are finite, row c of P is not, and every column behind c is lost in every
    row, while all codes and dequantized weights come out finite."""
    torch.manual_seed(n + c)
    m = 5
    X = torch.randn(tokens, n, device="cuda")
    F = X + 0.05 * torch.randn_like(X)
    st = g.LayerState(n, m, tokens, 64)
    try:
        for poison in (False, True):
            g.gptaq_reset(st.handle)
            if poison:
                F[3, c] = float("nan")
            g.gptaq_accumulate(st.handle, X, F)
            g.gptaq_factor(st.handle, 0.01)
            g.gptaq_build_P(st.handle, 0.25)
            G = hp.n_groups(n, group)
            codes = torch.empty((m, n), dtype=torch.uint8, device="cuda")
            sc, zp = torch.empty((m, G), device="cuda"), torch.empty((m, G), device="cuda")
            g.gptaq_quantize(st.handle, 0.02 * torch.randn(m, n, device="cuda"), 4, group, False, 128, codes, sc, zp)
            status, info = g.gptaq_sync_status(st.handle)
            assert status == (g.GPTAQ_ERR_NONFINITE if poison else g.GPTAQ_OK) and 0 <= info < m, (poison, status, info)
    finally:
        st.close()


@pytest.mark.parametrize("bad", ["U", "P", "pivot"])
@pytest.mark.parametrize("n,group,B", [(96, 32, 32), (200, 0, 128), (64, 16, 64)])
def test_a_non_finite_factor_of_the_static_entry_point_is_reported(n, group, B, bad):
    torch.manual_seed(n)
    m, row = 37, n - 12
    U = torch.eye(n, device="cuda") + torch.triu(0.1 * torch.randn(n, n, device="cuda"), 1)
    P = torch.triu(0.1 * torch.randn(n, n, device="cuda"), 1)
    G = hp.n_groups(n, group)
    codes = torch.empty((m, n), dtype=torch.uint8, device="cuda")
    sc, zp = torch.empty((m, G), device="cuda"), torch.empty((m, G), device="cuda")
    W = 0.02 * torch.randn(m, n, device="cuda")
    status = torch.zeros(2, dtype=torch.int64, device="cuda")
    g.gptaq_quantize_static(U, P, W.clone(), 4, group, False, B, codes, sc, zp, None, status)
    assert status.tolist()[0] == g.GPTAQ_OK
    if bad == "pivot":
        U[row, row] = 0.0                       # 1 / U_kk
    else:
        (U if bad == "U" else P)[row, row + 3] = float("inf")
    g.gptaq_quantize_static(U, P, W.clone(), 4, group, False, B, codes, sc, zp, None, status)
    assert status.tolist()[0] == g.GPTAQ_ERR_NONFINITE


def _replays_match(n, m, B, group, solve_too):
    """gptaq_quantize, or the whole solve, in a CUDA graph that is replayed twice: the direct calls' results bit for bit."""
    torch.manual_seed(n)
    X = torch.randn(2 * n, n, device="cuda")
    F = X + 0.05 * torch.randn_like(X)
    W = 0.02 * torch.randn(m, n, device="cuda")
    G = hp.n_groups(n, group)
    codes = torch.empty((m, n), dtype=torch.uint8, device="cuda")
    sc, zp, Wq = torch.empty((m, G), device="cuda"), torch.empty((m, G), device="cuda"), torch.empty((m, n), device="cuda")
    out = (codes, sc, zp, Wq)
    st = g.LayerState(n, m, 2 * n, B)
    h = st.handle

    def solve():
        g.gptaq_reset(h)
        g.gptaq_accumulate(h, X, F)
        g.gptaq_factor(h, 0.01)
        g.gptaq_build_P(h, 0.25)

    def quantize():
        g.gptaq_quantize(h, W, 4, group, False, B, *out)

    try:
        solve()
        quantize()
        torch.cuda.synchronize()
        want = [t.clone() for t in out]
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            if solve_too:
                solve()
            quantize()
        for call in (graph.replay, graph.replay, quantize):           # a direct call last
            for t in out:
                t.zero_()
            call()
            assert g.gptaq_sync_status(h)[0] == g.GPTAQ_OK
            assert [int((x != y).sum()) for x, y in zip(out, want)] == [0, 0, 0, 0]
        del graph
    finally:
        st.close()


@pytest.mark.parametrize("n,m,B,group", [(2048, 4096, 32, 32), (1024, 9000, 128, 128)])
def test_captured_quantize_can_be_replayed(n, m, B, group):
    """Products of more tiles than SMs draw their tile numbers from a counter on the device."""
    _replays_match(n, m, B, group, False)


@pytest.mark.parametrize("n,m,B,group", [
    (2048, 300, 128, 128), (520, 9000, 64, 64),
    (384, 300, 128, 128),       # the column loop without tensor cores: three launches, the later ones overlap the products
    (129, 5000, 32, 32),        # ... two CTAs to an SM; the second launch has one column
    (1153, 40, 64, 64),         # factorisation in plain float32
])
def test_captured_solve_can_be_replayed(n, m, B, group):
    """Launches that overlap their predecessors, and three streams, in one graph."""
    _replays_match(n, m, B, group, True)


@pytest.mark.parametrize("n,m,B,group", [(1024, 1024, 128, 128), (200, 70, 32, 0)])
def test_captured_static_entry_point_can_be_replayed(n, m, B, group):
    """The launches after the first read U and P before the product in front of them has ended.  Other U and P before each
    replay, written on the stream just before it: the first launch of a call has to wait for them."""
    torch.manual_seed(n)
    G = hp.n_groups(n, group)
    new = lambda *shape: torch.empty(shape, device="cuda")
    U, P, W = new(n, n), new(n, n), 0.02 * torch.randn(m, n, device="cuda")
    out = (torch.empty((m, n), dtype=torch.uint8, device="cuda"), new(m, G), new(m, G), new(m, n))
    status = torch.zeros(2, dtype=torch.int64, device="cuda")
    factors = [(torch.eye(n, device="cuda") + torch.triu(torch.randn(n, n, device="cuda"), 1) / n,
                torch.triu(torch.randn(n, n, device="cuda"), 1) / n) for _ in range(3)]

    def quantize():
        g.gptaq_quantize_static(U, P, W, 4, group, False, B, *out, status)

    def with_factors(u, p, call):
        U.copy_(u)
        P.copy_(p)
        call()
        assert status.tolist()[0] == g.GPTAQ_OK
        return [t.clone() for t in out]

    want = [with_factors(u, p, quantize) for u, p in factors]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        quantize()
    for (u, p), w in zip(factors, want):
        assert [int((x != y).sum()) for x, y in zip(with_factors(u, p, graph.replay), w)] == [0, 0, 0, 0]


@pytest.mark.parametrize("n", [516, 520, 1036])
def test_correction_matrix_rows_of_inputs_in_small_units(n):
    """Inputs whose units span a factor of 1e4: every row of P is as good as its own size, not only that of the largest.
    From the device's own U and dXX^T: two products after one another, of factors good to 2^-22 each."""
    torch.manual_seed(n)
    tokens, alpha = 2 * n, 0.5
    unit = torch.logspace(-2, 2, n, device="cuda")[torch.randperm(n, device="cuda")]
    X = torch.randn(tokens, n, device="cuda") * unit
    Xfp = X + 0.05 * torch.randn(tokens, n, device="cuda") * unit
    st = g.LayerState(n, 1, tokens, 32, "cuda")
    try:
        g.gptaq_accumulate(st.handle, X, Xfp)
        D = np.triu(st.D().cpu().numpy().astype(np.float64), 1) / tokens
        g.gptaq_factor(st.handle, 0.01)
        g.gptaq_build_P(st.handle, alpha)
        U = np.triu(st.H().cpu().numpy().astype(np.float64))
        P = np.triu(st.D().cpu().numpy().astype(np.float64), 1)
        assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
    finally:
        st.close()
    ref = alpha * np.triu(np.triu(D @ U.T, 1) @ U, 1)
    size = alpha * np.triu(np.triu(abs(D) @ abs(U).T, 1) @ abs(U), 1)
    err = np.linalg.norm(P - ref, axis=1)[:-1] / np.linalg.norm(size, axis=1)[:-1]        # (the last row is empty)
    assert err.max() <= 2.0 ** -20, err.max()


@pytest.mark.parametrize("n", [516, 1024, 2052])
def test_factor_without_damping_of_inputs_in_small_units(n):
    """Inputs whose units span a factor of 2^26 and no damping: rows of R span as much.  Bound and comparison as in
    test_factor_panels, for float32 products (2^-24 each) and with the units taken out of the condition number: a scaling of
    the inputs by powers of two changes no rounding of a float32 factorisation, only the columns of U."""
    torch.manual_seed(n)
    unit = 2.0 ** torch.randint(-13, 14, (n,), device="cuda")
    X = torch.randn(3 * n, n, device="cuda") * unit
    st = g.LayerState(n, 1, 3 * n, 32, "cuda")
    try:
        g.gptaq_set_stats_precision(st.handle, g.GPTAQ_STATS_FP32)
        g.gptaq_accumulate(st.handle, X, X)
        H = st.H().cpu().numpy().astype(np.float64)
        g.gptaq_factor(st.handle, 0.0)
        U = np.triu(st.H().cpu().numpy().astype(np.float64))
        assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
    finally:
        st.close()
    ref, _ = orc.factor(np.triu(H) + np.triu(H, 1).T, 3 * n, 0.0)
    u = unit.cpu().numpy()
    U, ref = U * u, ref * u
    sv = np.linalg.svd(ref, compute_uv=False)
    bound = (sv[0] / sv[-1]) ** 2 * np.sqrt(n) * 2.0 ** -24
    err = np.linalg.norm(U - ref, axis=1) / np.linalg.norm(ref, axis=1)
    assert err.max() <= bound, (err.max(), bound)


def test_solve_without_damping_of_inputs_in_small_units():
    """The same through P and the loop at a width that is a multiple of 4 only: P from the device's own U and dXX^T as in
    test_correction_matrix_rows_of_inputs_in_small_units, the loop replayed from the device's own U and P with the bounds of
    the parity tests."""
    n, m, alpha = 516, 40, 0.25
    torch.manual_seed(n)
    unit = 2.0 ** torch.randint(-10, 11, (n,), device="cuda")
    X = torch.randn(3 * n, n, device="cuda") * unit
    Xfp = X + 0.05 * torch.randn(3 * n, n, device="cuda") * unit
    W = 0.02 * torch.randn(m, n, device="cuda")
    G = hp.n_groups(n, 32)
    codes = torch.empty((m, n), dtype=torch.uint8, device="cuda")
    sc, zp = torch.empty((m, G), device="cuda"), torch.empty((m, G), device="cuda")
    st = g.LayerState(n, m, 3 * n, 128, "cuda")
    try:
        g.gptaq_set_stats_precision(st.handle, g.GPTAQ_STATS_FP32)
        g.gptaq_accumulate(st.handle, X, Xfp)
        D = np.triu(st.D().cpu().numpy().astype(np.float64), 1) / (3 * n)
        g.gptaq_factor(st.handle, 0.0)
        g.gptaq_build_P(st.handle, alpha)
        U = np.triu(st.H().cpu().numpy().astype(np.float64))
        P = np.triu(st.D().cpu().numpy().astype(np.float64), 1)
        g.gptaq_quantize(st.handle, W.clone(), 4, 32, True, 128, codes, sc, zp)
        assert g.gptaq_sync_status(st.handle)[0] == g.GPTAQ_OK
    finally:
        st.close()
    ref = alpha * np.triu(np.triu(D @ U.T, 1) @ U, 1)
    size = alpha * np.triu(np.triu(abs(D) @ abs(U).T, 1) @ abs(U), 1)
    err = np.linalg.norm(P - ref, axis=1)[:-1] / np.linalg.norm(size, axis=1)[:-1]
    assert err.max() <= 2.0 ** -20, err.max()
    rep = orc.follow(W.cpu().numpy().astype(np.float64), U, P, np.zeros(n, bool), 4, 32, True, codes.cpu().numpy(),
                     sc.cpu().numpy().astype(np.float64), zp.cpu().numpy().astype(np.float64), band=hp.TOL_FLIP_BAND)
    assert rep.disallowed == 0 and rep.allowed <= hp.TOL_FLIP_RATE * rep.total and rep.grid_rel_err <= hp.TOL_GRID, rep
