"""The expert GEMMs' row tiles (N of 32 to 256 tokens, tiles of equal size per
expert) at the edges of their sizes, for a hidden size whose last 256-row weight
block is half empty, and the ways the gate and up tensors can lie in memory."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_06690_gb300.inputs import LayerShape
from pmpe_testlib import check_against_oracle, check_audit, check_dispatch, make_layer, run_gpu_layer, to_device

pytestmark = pytest.mark.gpu


def check_gradients(shape, w, h, pol, dout, got):
    """The private gradients and d_hidden of one pass against the oracle, at twice
    the forward's tolerance, as in the backward's tests."""
    L = oracle.Layer(shape, dict(w, hidden=h), pol.numpy())
    d = dout.cpu().double().numpy()
    ref = dict(oracle.backward_private(L, d), d_hidden=oracle.backward_input(L, d))
    for n, v in got.items():
        err = np.abs(v.cpu().double().numpy() - ref[n])
        assert err.max() <= 2e-2 * max(np.abs(ref[n]).max(), 1e-30), n
        assert err.sum() <= 1e-2 * max(np.abs(ref[n]).sum(), 1e-30), n


@pytest.mark.parametrize("T", [1, 32, 33, 97, 224, 225, 256, 257, 289, 513, 800])
@pytest.mark.parametrize("H, E_sh", [(256, 0), (384, 2)])
def test_rows_of_one_expert(T, H, E_sh):
    """k = 1 and one expert a pool: expert 0 gets every DENY token (all but
    three), so its tiles split T - 3 rows, and the shared group's T."""
    shape = LayerShape(T=T, H=H, I=128, E_pub=1, E_priv=1, E_sh=E_sh, k=1, renormalize=True)
    w, h, _ = make_layer(shape, 60 + T)
    pol = torch.zeros(T, dtype=torch.uint8)
    pol[T // 2:T // 2 + 3] = 1
    gpu = run_gpu_layer(shape, *to_device(w, h, pol))
    check_against_oracle(shape, w, h, pol, gpu)
    check_audit(shape, pol, gpu)
    check_dispatch(shape, h, gpu)


@pytest.mark.parametrize("layout", ["up_first", "same"])
@pytest.mark.parametrize("T", [40, 300])
def test_gate_and_up_tensors(layout, T):
    """The gate and up rows come as one box of both tensors: the up tensor
    below the gate tensor in memory, and one tensor as both (two boxes)."""
    shape = LayerShape(T=T, H=256, I=256, E_pub=6, E_priv=4, E_sh=1, k=2, renormalize=True)
    w, h, pol = make_layer(shape, 71)
    for n in ("pub", "priv", "sh"):
        if layout == "same":
            w["up_" + n] = w["gate_" + n]
    wd, hd, pd = to_device(w, h, pol)
    for n in ("pub", "priv", "sh"):
        if layout == "same":
            wd["up_" + n] = wd["gate_" + n]
        else:
            both = torch.stack([wd["up_" + n], wd["gate_" + n]]).contiguous()
            wd["up_" + n], wd["gate_" + n] = both[0], both[1]
            assert wd["up_" + n].data_ptr() < wd["gate_" + n].data_ptr()
    gpu = run_gpu_layer(shape, wd, hd, pd)
    check_against_oracle(shape, w, h, pol, gpu)
    check_audit(shape, pol, gpu)


@pytest.mark.parametrize("T", [33, 130, 257, 300, 520])
def test_backward_rows_of_one_expert(T):
    """The backward's row tiles over one expert's rows per pool and one shared
    expert: both gradients against the oracle, and the same bits from the
    forward's saved accumulators as from the recompute."""
    from paper_2608_06690_gb300 import pmpe
    shape = LayerShape(T=T, H=384, I=256, E_pub=1, E_priv=1, E_sh=1, k=1, renormalize=False)
    w, h, _ = make_layer(shape, 90 + T)
    pol = torch.ones(T, dtype=torch.uint8)
    pol[T // 2:T // 2 + 40] = 0
    dout = torch.randn((T, shape.H), generator=torch.Generator().manual_seed(T)).to(torch.bfloat16)
    wd, hd, pd = to_device(w, h, pol)
    layer = pmpe.MoeLayer(shape, wd)
    got = []
    for saved in (False, True):
        layer.forward(hd, pd, save_for_backward=saved)
        got.append(layer.backward(hd, pd, dout.cuda()))
    torch.cuda.synchronize()
    (g, dh), (g2, dh2) = got
    assert torch.equal(dh, dh2)
    for n in g:
        assert torch.equal(g[n], g2[n]), n
    check_gradients(shape, w, h, pol, dout, dict(g, d_hidden=dh))


@pytest.mark.parametrize("E_pub, E_priv", [(2, 2), (7, 3), (3, 7), (8, 1), (5, 4)])
def test_interleaved_pools(E_pub, E_priv):
    """At 64 rows an expert and more the GEMMs take the two pools' experts
    interleaved: the forward and the combined backward of uneven pools against
    the oracle and the separate passes."""
    from paper_2608_06690_gb300 import pmpe
    shape = LayerShape(T=700, H=256, I=128, E_pub=E_pub, E_priv=E_priv, E_sh=1, k=1, renormalize=False)
    assert shape.T * shape.k >= 64 * shape.E
    w, h, pol = make_layer(shape, 120 + E_pub)
    wd, hd, pd = to_device(w, h, pol)
    gpu = run_gpu_layer(shape, wd, hd, pd)
    check_against_oracle(shape, w, h, pol, gpu)
    check_audit(shape, pol, gpu)
    check_dispatch(shape, h, gpu)
    layer = pmpe.MoeLayer(shape, wd)
    dout = torch.randn((shape.T, shape.H), generator=torch.Generator().manual_seed(5)).to(torch.bfloat16).cuda()
    layer.forward(hd, pd)
    g_sep = {n: v.clone() for n, v in layer.backward_private(hd, pd, dout).items()}
    dh_sep = layer.backward_input(hd, pd, dout).clone()
    g, dh = layer.backward(hd, pd, dout)
    torch.cuda.synchronize()
    for n in g:
        assert torch.equal(g[n], g_sep[n]), n
    assert torch.equal(dh, dh_sep)
    check_gradients(shape, w, h, pol, dout, dict(g, d_hidden=dh))


@pytest.mark.parametrize("T", [40, 129, 600])
def test_short_tiles_round_the_queue(T):
    """Many down tiles of two K steps after gate/up tiles of eight, at 10 stages (no
    expert above 32 rows): the pairs go round the tile queue several times after
    the gather warps leave it, with the loader up to five tiles ahead of the MMAs.
    Same bits as the two GEMMs in separate launches."""
    from paper_2608_06690_gb300 import pmpe
    shape = LayerShape(T=T, H=512, I=128, E_pub=256, E_priv=256, E_sh=0, k=1, renormalize=True)
    w, h, pol = make_layer(shape, 140 + T)
    wd, hd, pd = to_device(w, h, pol)
    layer = pmpe.MoeLayer(shape, wd)
    split = torch.full((T, shape.H), float("nan"), dtype=torch.bfloat16, device="cuda")
    for st in (pmpe.STAGE_ROUTE | pmpe.STAGE_PERMUTE, pmpe.STAGE_GATEUP, pmpe.STAGE_DOWN, pmpe.STAGE_COMBINE):
        layer.forward(hd, pd, out=split, stages=st)
    for _ in range(3):
        out = layer.forward(hd, pd).clone()
        torch.cuda.synchronize()
        assert torch.equal(out.view(torch.int16), split.view(torch.int16))


@pytest.mark.parametrize("T, E_sh", [(100, 0), (128, 2), (700, 0), (1500, 2)])
def test_down_tiles_read_this_launchs_activations(T, E_sh):
    """Forwards of two inputs in turn on one workspace, whose activation rows still
    hold the other input's values when a launch starts: a down tile that read a row
    before this launch's gate/up tiles had stored it would show.  Same bits as the
    two GEMMs in separate launches."""
    from paper_2608_06690_gb300 import pmpe
    shape = LayerShape(T=T, H=256, I=256, E_pub=12, E_priv=4, E_sh=E_sh, k=1, renormalize=True)
    w, h, pol = make_layer(shape, 160 + T)
    wd, hd, pd = to_device(w, h, pol)
    layer = pmpe.MoeLayer(shape, wd)
    ins = [hd, (hd * -0.5).contiguous()]
    ref = []
    for x in ins:
        split = torch.full((T, shape.H), float("nan"), dtype=torch.bfloat16, device="cuda")
        for st in (pmpe.STAGE_ROUTE | pmpe.STAGE_PERMUTE, pmpe.STAGE_GATEUP, pmpe.STAGE_DOWN, pmpe.STAGE_COMBINE):
            layer.forward(x, pd, out=split, stages=st)
        ref.append(split)
    got = [layer.forward(ins[i & 1], pd).clone() for i in range(40)]
    torch.cuda.synchronize()
    for i, out in enumerate(got):
        assert torch.equal(out.view(torch.int16), ref[i & 1].view(torch.int16)), i


@pytest.mark.parametrize("T", [500, 16128])
def test_dispatch_table_in_the_ring(T):
    """The expert launch derives the dispatch order in the ring's memory before the
    first copies land there; at T = 16128 its table of 384 experts x 127 router
    tiles fills the ring.  Same bits as the dispatch and the GEMMs in launches of
    their own."""
    from paper_2608_06690_gb300 import pmpe
    shape = LayerShape(T=T, H=1024, I=1024, E_pub=256, E_priv=128, E_sh=0, k=1, renormalize=True)
    w, h, pol = make_layer(shape, 170, device="cuda")
    wd, hd, pd = to_device(w, h, pol)
    layer = pmpe.MoeLayer(shape, wd)
    split = torch.full((T, shape.H), float("nan"), dtype=torch.bfloat16, device="cuda")
    for st in (pmpe.STAGE_ROUTE, pmpe.STAGE_PERMUTE, pmpe.STAGE_GATEUP, pmpe.STAGE_DOWN, pmpe.STAGE_COMBINE):
        layer.forward(hd, pd, out=split, stages=st)
    for _ in range(3):
        out = layer.forward(hd, pd).clone()
        torch.cuda.synchronize()
        assert torch.equal(out.view(torch.int16), split.view(torch.int16))
