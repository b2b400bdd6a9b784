"""Blocks of a factorisation leave the walker's SM, but never all of them.

On the host: the rule's bound, read from the source, in a model of the
placement that is worst for it: every block comes in on the walker's SM,
`slots` at a time, the next when one has left.  The walker waits for tasks
that other blocks run, so one of them has to stay.

On the GPU: a calibration with the factorisation capped to a few blocks, where
two or three can land on one SM, gives the bits of the one without a cap (a
tile is formed by the same operations whichever block forms it).  A cap of
one block counts as two: the walker alone would wait for tiles of others.
"""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1910_13908_gb300", "csrc")


def _max_leavers():
    text = open(os.path.join(CSRC, "chol_tiles.cuh")).read()
    m = re.search(r"constexpr int max_leavers\(int blocks\) \{ return ([^;]*); \}", text)
    assert m, "no bound on the blocks that leave"
    return eval("lambda blocks: " + m.group(1).replace("/", "//"))  # the operands are positive


@pytest.mark.parametrize("slots", [2, 3, 4, 6])
def test_some_block_stays_wherever_they_land(slots):
    bound = _max_leavers()
    for blocks in list(range(2, 40)) + [152, 304, 608]:
        queued, asked, stay = blocks - 1, 0, 0  # the first is the walker and takes a slot
        while queued and stay < slots - 1:
            queued -= 1
            stay += asked >= bound(blocks)  # else it leaves and its slot is free again
            asked += 1
        assert stay >= 1, (blocks, slots)
        assert blocks - 1 - bound(blocks) >= (blocks - 1) / 2  # half of them, when all are placed at once


def test_both_factorisations_ask_before_a_claim():
    for name, asks in (("cholesky.cu", 2), ("chol_f64.cu", 1)):
        text = open(os.path.join(CSRC, name)).read()
        assert len(re.findall(r"leave\.ask\(sv\.sctr, (?:gridDim\.x|per_job)\)", text)) == asks
        assert "%%smid" not in text  # no other rule on the SM


@pytest.mark.gpu
@pytest.mark.parametrize("max_ctas", [1, 2, 3, 5, 17, 40])
@pytest.mark.parametrize("prec,kernel", [("mixed", 0), ("mixed", 1), ("fp64", 0)])
def test_few_blocks_give_the_bits_of_many(prec, kernel, max_ctas):
    torch = pytest.importorskip("torch")
    from paper_1910_13908_gb300 import sagecal as sc
    from paper_1910_13908_gb300 import synth
    prec = sc.SC_MIXED if prec == "mixed" else sc.SC_FP64
    spec = synth.JobSpec(N=70, T=2, F=1, K=1, S=4, f_lo=150e6, f_hi=150e6, seed=5)  # nine tile rows, the last ragged
    shp = sc.Shape(spec.N, spec.T, spec.F, spec.K, spec.S)
    uvw, freqs = torch.as_tensor(synth.station_uvw(spec)).cuda(), torch.as_tensor(synth.freqs(spec)).cuda()
    sky, ws = sc.DeviceSky.from_synth(synth.sky(spec)), sc.workspace(shp, prec)
    C = sc.predict_coherencies(shp, uvw, freqs, sky, prec, ws)[0]
    J = torch.as_tensor(synth.jones_true(spec)[0]).to("cuda", C.dtype)
    p, q = torch.triu_indices(spec.N, spec.N, 1, device="cuda")
    V = (C[..., None, None] * (J[p] @ J[q].mH)[None, :, None]).contiguous()
    start = torch.as_tensor(synth.identity_jones(1, spec.N)).cuda()

    def calibrate(cap):
        out = sc.calibrate_sage(shp, uvw, freqs, sky, V, start.clone(), prec, ws, n_em=1, n_lm=6, max_ctas=cap,
                                chol_kernel=kernel)
        assert sc.device_status(ws) == 0
        return out

    for a, b in zip(calibrate(max_ctas), calibrate(0)):
        assert torch.equal(a, b)
