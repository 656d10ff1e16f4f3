"""GPU parity of mala_bwd (through the C ABI) against the fp64 oracle.

Isolated runs give the oracle the SAME forward output o (bf16) and saved lse (fp32) that the GPU backward
receives (those written by mala_fwd), so that only the backward kernels are under test; end-to-end runs
compare GPU fwd -> bwd with oracle fwd -> bwd in fp64."""
import numpy as np
import pytest
import torch

from paper_2609_32712_b200 import workloads as W
from tests import parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mala():
    from paper_2609_32712_b200 import mala as m
    m.lib()
    return m


def _check_bwd_masks(st, ref, B, Hq, T, causal, band_extra=0.0):
    gm = st.mask(T).cpu().numpy()                       # [B,Hq,Tc,Tr]
    flips = 0
    for b in range(B):
        for h in range(Hq):
            for j in range(T):
                om, oc = ref["mask"][b, h, j], ref["crit"][b, h, j]
                for i in range(T):
                    if om[i] == 0:
                        assert not gm[b, h, j, i]
                        continue
                    if bool(gm[b, h, j, i]) != (om[i] == 2):
                        assert abs(oc[i]) <= parity.MASK_BAND + band_extra, (b, h, j, i, oc[i])
                        flips += 1
                assert int(st.retained[b, h, j]) == int(gm[b, h, j].sum())
    return flips


def _run_isolated(mala, oracle, w, tau, causal=True):
    q, k, v, do = (w[x].cuda() for x in ("q", "k", "v", "do"))
    B, N, Hq, d = q.shape
    o, lse, fst = mala.fwd(q, k, v, w["scale"], tau, causal=causal, stats=True)
    dq, dk, dv, st = mala.bwd(q, k, v, o, do, lse, w["scale"], tau, causal=causal, stats=True)
    torch.cuda.synchronize()
    assert mala.device_status() == 0
    Bq, Bk = mala.tile_shape(mala.OP_BWD, d)
    ref = oracle.bwd(w["q"], w["k"], w["v"], o.float().cpu(), w["do"], lse.cpu().numpy(), w["scale"], tau, Bq, Bk,
                     causal=causal)
    T = -(-N // Bq)
    flips = _check_bwd_masks(st, ref, B, Hq, T, causal)
    e = [parity.check_grad(dq.float().cpu().numpy(), ref["dq"], "dq"),
         parity.check_grad(dk.float().cpu().numpy(), ref["dk"], "dk"),
         parity.check_grad(dv.float().cpu().numpy(), ref["dv"], "dv")]
    # nesting: backward support inside forward support, same partition, nothing stored
    fm = fst.mask(T).cpu().numpy()
    bm = st.mask(T).cpu().numpy().transpose(0, 1, 3, 2)
    assert (bm <= fm).all()
    crit = np.abs(ref["crit"][ref["mask"] > 0])
    return dict(flips=flips, err=e, skipped=int((ref["mask"] == 1).sum()), retained=int((ref["mask"] == 2).sum()),
                totals=st.totals.cpu().numpy(), near=int((crit < 1e-2).sum()), band=int((crit <= parity.MASK_BAND).sum()))


@pytest.mark.parametrize("tau", [0.0, 1e-4])
@pytest.mark.parametrize("N,d,Hq,Hkv", [(128, 128, 1, 1), (384, 128, 2, 1), (333, 128, 4, 2), (512, 64, 2, 2),
                                        (200, 64, 2, 1)])
def test_bwd_small_shapes_literal(mala, oracle, N, d, Hq, Hkv, tau):
    w = W.custom_prefill(2, Hq, Hkv, N, d, seed=N + d)
    _run_isolated(mala, oracle, w, tau)


@pytest.mark.parametrize("tau", [1e-4, 1e-2])
@pytest.mark.parametrize("N,d,Hq,Hkv", [(300, 128, 49, 49), (300, 128, 50, 50), (512, 64, 8, 2), (513, 64, 8, 2)])
def test_bwd_one_or_two_passes(mala, oracle, N, d, Hq, Hkv, tau):
    # key blocks for as many SMs as the GPU has and just more of them; sixteen tiles per key block and more
    w = W.custom_prefill(1, Hq, Hkv, N, d, seed=N + Hq, preset="R")
    _run_isolated(mala, oracle, w, tau)


@pytest.mark.parametrize("tau", [0.0, 1e-3])
@pytest.mark.parametrize("B,N,d,Hq,Hkv", [(1, 300, 128, 16, 1), (1, 300, 128, 17, 1), (1, 640, 64, 33, 1), (38, 250, 64, 34, 2)])
def test_bwd_groups_of_more_than_sixteen_heads(mala, oracle, B, N, d, Hq, Hkv, tau):
    # the two-pass path ends at sixteen query heads per KV head; the kernel that walks all heads of a group takes any number
    # (the last case: more key blocks than a GPU of 148 SMs has SMs)
    w = W.custom_prefill(B, Hq, Hkv, N, d, head_types=["diffuse", "peaked"] * (Hq // 2) + ["peaked"] * (Hq % 2), seed=N, preset="R")
    _run_isolated(mala, oracle, w, tau)


@pytest.mark.parametrize("N,d,Hq,Hkv", [(520, 128, 147, 49), (520, 128, 148, 37), (600, 64, 160, 40), (385, 64, 148, 74)])
def test_bwd_first_pass_of_two_or_four_key_blocks(mala, oracle, N, d, Hq, Hkv):
    # on a GPU of 148 SMs the first pass takes four key blocks per CTA from 296 CTAs on; ragged last blocks and pairs
    w = W.custom_prefill(1, Hq, Hkv, N, d, head_types=["diffuse", "peaked"] * (Hq // 2) + ["peaked"] * (Hq % 2), seed=N, preset="R")
    r = _run_isolated(mala, oracle, w, 1e-3)
    assert r["skipped"] > 0


@pytest.mark.parametrize("T,d", [(95, 128), (96, 128), (191, 64), (192, 64)])
def test_bwd_with_and_without_samples(mala, oracle, T, d):
    # just below and at the length from which rows that retain everything are left to the one-pass kernel, which then adds to the
    # dK, dV of the list (a diffuse and a peaked head share them): key blocks with rows of more and of fewer than 32 tiles
    N = T * 128 - 9
    w = W.custom_prefill(1, 2, 1, N, d, head_types=["diffuse", "peaked"], seed=T, preset="R", device="cuda")
    q, k, v, do = (w[x] for x in ("q", "k", "v", "do"))
    o, lse, _ = mala.fwd(q, k, v, w["scale"], 1e-4)
    dq, dk, dv, st = mala.bwd(q, k, v, o, do, lse, w["scale"], 1e-4, stats=True)
    torch.cuda.synchronize()
    assert mala.device_status() == 0
    units, rows_of = [(0, 0, 3), (0, 0, T - 40), (0, 0, T - 20), (0, 0, T - 1)], [(0, 0, T // 2), (0, 1, T - 1)]
    ref = oracle.bwd(*(x.cpu() for x in (q, k, v)), o.float().cpu(), do.cpu(), lse.cpu().numpy(), w["scale"], 1e-4, 128, 128,
                     key_units=units, dq_units=rows_of)
    gm = st.mask(T)[0].cpu().numpy()
    for _, _, j in units:
        for h in range(2):
            om, oc = ref["mask"][0, h, j], ref["crit"][0, h, j]
            differ = gm[h, j] != (om == 2)
            assert (np.abs(oc[differ]) <= parity.MASK_BAND).all()
        rows = slice(j * 128, min(N, (j + 1) * 128))
        parity.check_grad(dk[0, rows, 0].float().cpu().numpy(), ref["dk"][0, rows, 0], f"dk block {j}")
        parity.check_grad(dv[0, rows, 0].float().cpu().numpy(), ref["dv"][0, rows, 0], f"dv block {j}")
    for _, h, i in rows_of:
        rows = slice(i * 128, min(N, (i + 1) * 128))
        parity.check_grad(dq[0, rows, h].float().cpu().numpy(), ref["dq"][0, rows, h], f"dq block {i}")


def test_bwd_first_pass_long_rows(mala, oracle):
    # so many query blocks (2057) that the masks of a CTA leave room for two Q tiles instead of three; sampled key blocks
    N = 263200
    w = W.custom_prefill(1, 1, 1, N, 128, head_types=["peaked"], seed=5, preset="S", device="cuda")
    q, k, v, do = (w[x] for x in ("q", "k", "v", "do"))
    o, lse, _ = mala.fwd(q, k, v, w["scale"], 1e-4)
    dq, dk, dv, st = mala.bwd(q, k, v, o, do, lse, w["scale"], 1e-4, stats=True)
    torch.cuda.synchronize()
    assert mala.device_status() == 0
    units = [(0, 0, 1601), (0, 0, 2056)]
    ref = oracle.bwd(*(x.cpu() for x in (q, k, v)), o.float().cpu(), do.cpu(), lse.cpu().numpy(), w["scale"], 1e-4, 128, 128,
                     key_units=units)
    gm = st.mask(2057)[0, 0].cpu().numpy()
    for _, _, j in units:
        om, oc = ref["mask"][0, 0, j], ref["crit"][0, 0, j]
        differ = gm[j] != (om == 2)
        assert (np.abs(oc[differ]) <= parity.MASK_BAND).all()
        rows = slice(j * 128, min(N, (j + 1) * 128))
        parity.check_grad(dk[0, rows, 0].float().cpu().numpy(), ref["dk"][0, rows, 0], f"dk block {j}")
        parity.check_grad(dv[0, rows, 0].float().cpu().numpy(), ref["dv"][0, rows, 0], f"dv block {j}")


@pytest.mark.parametrize("tau", [1e-5, 1e-4, 1e-3, 1.0])
@pytest.mark.parametrize("N,d", [(1024, 128), (1000, 128), (1024, 64)])
def test_bwd_skipping_regime(mala, oracle, N, d, tau):
    w = W.custom_prefill(1, 4, 2, N, d, head_types=["diffuse", "peaked", "peaked", "sink"], seed=7, preset="R")
    res = _run_isolated(mala, oracle, w, tau)
    assert res["skipped"] > 0
    assert res["totals"][1] == res["retained"] + res["skipped"]


@pytest.mark.parametrize("tau", [0.0, 1e-3])
def test_bwd_cfg1_end_to_end(mala, oracle, tau):
    w = W.make_prefill(W.prefill_config("cfg1"))
    q, k, v, do = (w[x].cuda() for x in ("q", "k", "v", "do"))
    o, lse, _ = mala.fwd(q, k, v, w["scale"], tau)
    dq, dk, dv, st = mala.bwd(q, k, v, o, do, lse, w["scale"], tau, stats=True)
    torch.cuda.synchronize()
    f = oracle.fwd(w["q"], w["k"], w["v"], w["scale"], tau, 128, 128)
    g = oracle.bwd(w["q"], w["k"], w["v"], f["o"], w["do"], f["lse"], w["scale"], tau, 128, 128)
    _check_bwd_masks(st, g, 1, 2, 8, True, band_extra=1e-3)
    parity.check_grad(dq.float().cpu().numpy(), g["dq"], "dq")
    parity.check_grad(dk.float().cpu().numpy(), g["dk"], "dk")
    parity.check_grad(dv.float().cpu().numpy(), g["dv"], "dv")


@pytest.mark.parametrize("tau", [0.0, 1e-2])
def test_bwd_non_causal(mala, oracle, tau):
    w = W.custom_prefill(1, 2, 1, 300, 128, head_types=["peaked", "diffuse"], seed=5, preset="R")
    _run_isolated(mala, oracle, w, tau, causal=False)


def test_bwd_near_threshold_decisions(mala, oracle, capsys):
    """Eq. 4 next to equality: softmax mass decaying smoothly toward earlier keys puts tile criteria within 1e-2 of zero
    and some inside the 1e-3 band; decisions outside the band must be the oracle's, flips inside it are reported."""
    w = W.custom_prefill(2, 6, 6, 4096, 64, head_types=["decay"] * 6, seed=5)
    near = band = flips = 0
    for tau in (1.0,):
        res = _run_isolated(mala, oracle, w, tau)
        assert res["skipped"] > 0
        flips += res["flips"]
        near += res["near"]
        band += res["band"]
    with capsys.disabled():
        print(f"\n[near-threshold backward] tiles with |C| < 1e-2: {near}, inside the 1e-3 band: {band}, "
              f"decisions that differ from the oracle (all inside the band): {flips}")
    assert near >= 3 and band >= 1, "the workload must put tiles next to the threshold"
