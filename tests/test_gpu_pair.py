"""The contraction on pairs of SMs over many tiles: every cluster's accumulator
buffers and ring slots (of one pipeline or two) go round several times."""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["bf16x3", "tf32"])
@pytest.mark.parametrize("mo_num", [60, 150, 250, 300])
def test_many_tiles_same_values_as_single_sm(cfg, mode, mo_num):
    """1151 tiles (the last pair has one) of the organic chain: N tiles of 64,
    160 (an odd buffer count), 256 and twice 160 columns, 7 to 15 pair-tiles per
    cluster.  Both kernels add the same products in the same k order; the pair's
    extra k-steps add zeros.  Bar: 1e-6 of sum |C||AO|, eight FP32 roundings."""
    from paper_2512_16677_gb300 import qmckl
    m = cfg(2, walk_num=48)
    m = m.with_points(m.points[:1151 * 25 - 7])
    m = dataclasses.replace(m, mo_coef=np.ascontiguousarray(m.mo_coef[:mo_num]))
    outs = []
    for pairs in (True, False):
        c = qmckl.Context(mode)
        c.set_molecule(m)
        c.set_sm_pairs(pairs)
        c.set_points_device(torch.from_numpy(m.coord).cuda())
        for _ in range(2):
            out = c.mo_vgl_device()
        outs.append(out.reshape(-1, mo_num))
        if pairs:
            ao = c.ao_vgl_device().reshape(-1, m.ao_num).abs_()
            size = ao @ torch.from_numpy(np.abs(m.mo_coef).T.copy()).to(ao)
        torch.cuda.synchronize()
        c.synchronize()
        c.close()
    worst = float(((outs[0] - outs[1]).abs_() / (size + 1e-30)).max())
    assert worst <= 1e-6, worst


@pytest.mark.parametrize("mode", ["bf16x3", "tf32"])
@pytest.mark.parametrize("mo_num,n", [(20, 30), (33, 1), (100, 60), (150, 280), (300, 280),
                                      (300, 900), (300, 1900)])
def test_few_tiles_same_values_as_many(cfg, mode, mo_num, n):
    """The single-SM contraction of few tiles takes narrower N tiles (32 to the
    default width, by the tile count); the products of an output and their order
    are the same, so the first n points alone equal those of a call of 12 000 points
    bit for bit."""
    from paper_2512_16677_gb300 import qmckl
    m = cfg(2, walk_num=20)
    m = dataclasses.replace(m, mo_coef=np.ascontiguousarray(m.mo_coef[:mo_num]))
    outs = []
    for k in (12000, n):
        c = qmckl.Context(mode)
        c.set_molecule(m)
        c.set_sm_pairs(False)
        c.set_points_device(torch.from_numpy(np.ascontiguousarray(m.points[:k])).cuda())
        outs.append(c.mo_vgl_device().reshape(-1, 5, mo_num)[:n].clone())
        torch.cuda.synchronize()
        c.synchronize()
        c.close()
    assert torch.equal(outs[0], outs[1])


@pytest.mark.parametrize("mode", ["bf16x3", "tf32"])
@pytest.mark.parametrize("n", [1, 26, 600, 1200])
def test_small_calls_same_values_as_pairs(cfg, mode, n):
    """Calls of few tiles leave the pairs of SMs to the single-SM kernel: the first n
    points alone against the same points of a call that runs on pairs.  Both add
    the same products in the same k order; bar 1e-6 of sum |C||AO|."""
    from paper_2512_16677_gb300 import qmckl
    m = cfg(2, walk_num=20)
    outs = []
    for k in (12000, n):
        c = qmckl.Context(mode)
        c.set_molecule(m)
        c.set_points_device(torch.from_numpy(np.ascontiguousarray(m.points[:k])).cuda())
        outs.append(c.mo_vgl_device().reshape(-1, m.mo_num)[:5 * n].clone())
        if k == n:
            ao = c.ao_vgl_device().reshape(-1, m.ao_num).abs_()
            size = ao @ torch.from_numpy(np.abs(m.mo_coef).T.copy()).to(ao)
        torch.cuda.synchronize()
        c.synchronize()
        c.close()
    worst = float(((outs[0] - outs[1]).abs_() / (size + 1e-30)).max())
    assert worst <= 1e-6, worst
