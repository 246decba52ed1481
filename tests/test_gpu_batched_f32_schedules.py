"""Schedules of a block-diagonal FP32 projection: its products run over 256 x 256 tiles on
SM pairs, and the autotuner orders those."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2507_09165_gb300 import binding as b, synth  # noqa: E402

DEV = torch.device("cuda")
SIZES = [900, 17, 640, 256, 1000, 3, 450, 128, 777, 64, 1024, 257, 513, 302] * 8


def _run(mats):
    outs = [torch.full_like(m, float("nan")) for m in mats]
    infos = [torch.zeros(b.INFO_BYTES, dtype=torch.uint8, device=DEV) for _ in mats]
    descs = b.block_descs([(m.shape[0], m, m.shape[0], o, m.shape[0], i) for m, o, i in zip(mats, outs, infos)])
    b.psd_project_batched(len(mats), descs, "fp32")
    torch.cuda.synchronize()
    return outs, [b.info_from_bytes(i.cpu().numpy()) for i in infos]


def test_schedules_give_the_same_bits_and_only_distinct_ones_are_timed():
    base = {n: torch.from_numpy(synth.wigner(n, 4400 + n)).to(DEV) for n in set(SIZES)}
    mats = [base[n] for n in SIZES]
    ref = None
    try:
        for idx in (0, 3):  # largest first; by cost in rounds of the SM pairs
            b.psd_batched_force_schedule(idx)
            b.psd_release_workspaces()
            outs, infos = _run(mats)
            assert b.psd_batched_last_tuning()[0] == idx
            assert all(i["status"] == 0 and np.isfinite(i["compl_resid"]) for i in infos)
            if ref is None:
                ref = outs, infos
            assert all(torch.equal(o, r) for o, r in zip(outs, ref[0]))
            assert infos == ref[1]
        b.psd_batched_force_schedule(-1)
        b.psd_release_workspaces()
        outs, infos = _run(mats)
        chosen, ms = b.psd_batched_last_tuning()
        assert chosen in (0, 3) and ms[chosen] == min(ms)
        assert ms[0] == ms[1] == ms[2] and ms[3] == ms[4] == ms[5]
        assert all(torch.equal(o, r) for o, r in zip(outs, ref[0])) and infos == ref[1]
    finally:
        b.psd_batched_force_schedule(-1)
