"""GPU parity of mala_fwd (through the C ABI) against the fp64 oracle."""
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


def _run_and_check(mala, oracle, w, tau, causal=True, units=None, rounding_bound=False):
    dev = "cuda"
    q, k, v = (w[x].to(dev) for x in ("q", "k", "v"))
    B, N, Hq, d = q.shape
    o, lse, st = mala.fwd(q, k, v, w["scale"], tau, causal=causal, stats=True)
    torch.cuda.synchronize()
    assert mala.device_status() == 0
    Bq, Bk = mala.tile_shape(mala.OP_FWD, d)
    ref = oracle.fwd(w["q"], w["k"], w["v"], w["scale"], tau, Bq, Bk, causal=causal, units=units)
    # (the same call on |V|: a = sum_k p_k |v_k| over the retained keys, for the rounding bound of parity.check_output)
    ref_abs = oracle.fwd(w["q"], w["k"], w["v"].abs(), w["scale"], tau, Bq, Bk, causal=causal, units=units) if rounding_bound else None
    T = -(-N // Bq)
    gm = st.mask(T).cpu().numpy()
    o_c, lse_c = o.float().cpu().numpy(), lse.cpu().numpy()
    if units is None:
        units = [(b, h, i) for b in range(B) for h in range(Hq) for i in range(T)]
    flips = 0
    retained = skipped = 0
    worst = 0.0
    for (b, h, i) in units:
        order = list(range(i, -1, -1)) if causal else list(range(T - 1, -1, -1))
        rows = slice(i * Bq, min(N, (i + 1) * Bq))
        flips += parity.check_mask(gm[b, h, i], ref["mask"][b, h, i], ref["crit"][b, h, i], order, tau,
                                   i * Bq + 1 if causal else N, Bk)
        err = parity.check_output(o_c[b, rows, h], ref["o"][b, rows, h],
                                  a_ref=ref_abs["o"][b, rows, h] if rounding_bound else None)
        worst = max(worst, err[0])
        assert np.abs(lse_c[b, h, rows] - ref["lse"][b, h, rows]).max() <= parity.LSE_ABS
        retained += int((ref["mask"][b, h, i] == 2).sum())
        skipped += int((ref["mask"][b, h, i] == 1).sum())
        assert int(st.retained[b, h, i]) == int(gm[b, h, i].sum())
    crit = np.abs(ref["crit"][ref["mask"] > 0])
    return dict(flips=flips, retained=retained, skipped=skipped, totals=st.totals.cpu().numpy(), max_err=worst,
                near=int((crit < 1e-2).sum()), band=int((crit <= parity.MASK_BAND).sum()),
                o_absmax=float(np.abs(ref["o"][np.isfinite(ref["o"])]).max()))


@pytest.mark.parametrize("tau", [0.0, 1e-4])
@pytest.mark.parametrize("N,d,Hq,Hkv", [(128, 128, 1, 1), (384, 128, 2, 1), (333, 128, 2, 2), (512, 64, 2, 2),
                                        (200, 64, 1, 1)])
def test_fwd_small_shapes_literal(mala, oracle, N, d, Hq, Hkv, tau):
    w = W.custom_prefill(2, Hq, Hkv, N, d, seed=N + d)
    _run_and_check(mala, oracle, w, tau)


@pytest.mark.parametrize("tau", [0.0, 1e-3])
@pytest.mark.parametrize("N,d,H", [(130, 64, 74), (130, 64, 75), (300, 128, 49), (300, 128, 50), (130, 64, 148), (130, 64, 149),
                                   (300, 128, 98), (300, 128, 99), (300, 96, 98), (300, 96, 99)])
def test_fwd_one_or_two_blocks_per_cta(mala, oracle, N, d, H, tau):
    # on a GPU of 148 SMs: one query block per SM and just more of them; two per SM (up to here a CTA has one block) and just more
    w = W.custom_prefill(1, H, H, N, d, seed=N + H, preset="R")
    _run_and_check(mala, oracle, w, tau)


@pytest.mark.parametrize("tau", [0.0, 1e-3])
@pytest.mark.parametrize("N,d,H", [(130, 64, 74), (130, 64, 75), (300, 128, 49), (300, 128, 50)])
def test_fwd_one_or_two_blocks_per_cta_non_causal(mala, oracle, N, d, H, tau):
    # (here a CTA has one block up to one query block per SM)
    w = W.custom_prefill(1, H, H, N, d, seed=N + H, preset="R")
    _run_and_check(mala, oracle, w, tau, causal=False)


@pytest.mark.parametrize("tau", [0.0, 1e-5, 1e-3])
@pytest.mark.parametrize("N,d", [(1000, 128), (1100, 64), (900, 96)])
def test_fwd_rows_are_the_same_whichever_kernel_takes_them(mala, N, d, tau):
    # 8 blocks of 4 heads: one block per CTA; the same heads among 80 of them: two per CTA (on any GPU of up to 300 SMs)
    w = W.custom_prefill(1, 80, 80, N, d, head_types=["diffuse", "sink", "peaked", "planted"] * 20, seed=N, preset="R", device="cuda")
    q, k, v = (w[x] for x in ("q", "k", "v"))
    o, lse, st = mala.fwd(q, k, v, w["scale"], tau, stats=True)
    T = -(-N // 128)
    for h in (0, 40, 76):
        o1, lse1, st1 = mala.fwd(*(x[:, :, h:h + 4].contiguous() for x in (q, k, v)), w["scale"], tau, stats=True)
        assert torch.equal(o1, o[:, :, h:h + 4]) and torch.equal(lse1, lse[:, h:h + 4])
        assert torch.equal(st1.mask(T), st.mask(T)[:, h:h + 4])
    assert mala.device_status() == 0


@pytest.mark.parametrize("tau", [1e-5, 1e-4, 1e-3, 1.0])
@pytest.mark.parametrize("N,d", [(1024, 128), (1000, 128), (1024, 64)])
def test_fwd_skipping_regime(mala, oracle, N, d, tau):
    w = W.custom_prefill(1, 4, 2, N, d, head_types=["diffuse", "peaked", "peaked", "sink"], seed=7, preset="R")
    res = _run_and_check(mala, oracle, w, tau)
    assert res["skipped"] > 0, "workload must exercise skipping"
    assert res["totals"][0] == res["retained"] + 0 or res["flips"] > 0
    assert res["totals"][1] == res["retained"] + res["skipped"]


@pytest.mark.parametrize("tau", [0.0, 1e-4, 1e-3])
def test_fwd_cfg1(mala, oracle, tau):
    w = W.make_prefill(W.prefill_config("cfg1"))
    _run_and_check(mala, oracle, w, tau)


@pytest.mark.parametrize("tau", [0.0, 1e-2])
def test_fwd_non_causal(mala, oracle, tau):
    w = W.custom_prefill(1, 2, 1, 300, 128, head_types=["peaked", "diffuse"], seed=5, preset="R")
    _run_and_check(mala, oracle, w, tau, causal=False)


def test_fwd_tau_zero_equals_dense_kernel_bitwise_mask(mala, oracle):
    w = W.custom_prefill(1, 2, 1, 640, 128, seed=9, preset="R")
    q, k, v = (w[x].cuda() for x in ("q", "k", "v"))
    _, _, st = mala.fwd(q, k, v, w["scale"], 0.0, stats=True)
    T = 5
    m = st.mask(T).cpu().numpy()
    for i in range(T):
        assert m[0, :, i, :i + 1].all() and not m[0, :, i, i + 1:].any()


def test_fwd_near_threshold_decisions(mala, oracle, capsys):
    """Inputs whose tile criteria pass through zero with a small slope per tile (softmax mass decaying smoothly toward
    earlier keys): a visible number of tiles has |C| < 1e-2 and some lie inside the 1e-3 band in which the fp32 / log2
    evaluation of Eq. 3 may decide differently from the fp64 oracle.  Every decision outside the band must be the
    oracle's (parity.check_mask); the number of exempted flips is reported."""
    near = band = flips = 0
    for seed in (5, 6, 7, 8):
        w = W.custom_prefill(2, 6, 6, 4096, 64, head_types=["decay"] * 6, seed=seed)
        for tau in (1.0, 0.3):
            res = _run_and_check(mala, oracle, w, tau)
            assert res["skipped"] > 0
            flips += res["flips"]
            near += res["near"]
            band += res["band"]
    with capsys.disabled():
        print(f"\n[near-threshold forward] tiles with |C| < 1e-2: {near}, inside the 1e-3 band: {band}, "
              f"decisions that differ from the oracle (all inside the band): {flips}")
    assert near >= 10 and band >= 1, "the workload must put tiles next to the threshold"


# One query block per CTA (mala_fwd_one.cuh): score levels of the key blocks, newest first, in nats.  One to seven tiles; every
# order of retained and skipped tiles that the V copies ahead of the vote can meet; maxima that move the reference of the
# exponentials while the product before is still running.
@pytest.mark.parametrize("levels", [[0], [0, 0], [0, -30], [0, -30, 0], [0, 0, -30, 0], [0, -30, -30, 0, 0], [0, -30, 0, -30, 0, -30, 0],
                                    [0, 20, 40, 60], [0, 30, -30, 30, 60, 0, 62], [0, 0, 0, -30, -30, -30, -30]])
@pytest.mark.parametrize("d,tau", [(64, 1e-3), (128, 1e-3), (128, 0.0), (192, 1e-3), (256, 1e-3), (256, 0.0)])
def test_fwd_one_block_orders(mala, oracle, d, tau, levels):
    N = 128 * len(levels) - 5
    g = torch.Generator().manual_seed(d + len(levels))
    q, k, v = (torch.randn((1, N, 2, d), generator=g) * s for s in (0.3, 0.3, 1.0))
    scale = d ** -0.5
    T = len(levels)
    for x, level in enumerate(levels):
        k[:, 128 * (T - 1 - x):128 * (T - x), :, 0] = level / (8 * scale)
    q[..., 0] = 8.0
    w = {"q": q.bfloat16(), "k": k.bfloat16(), "v": v.bfloat16(), "scale": scale}
    r = _run_and_check(mala, oracle, w, tau, rounding_bound=True)
    assert r["retained"] > 0 and (tau == 0.0 or r["skipped"] > 0 or min(levels) == 0)
