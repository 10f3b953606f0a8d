"""Work lists of a batch: the reach pre-pass (items of whole blocks of tiles) and
ao_vgl (items handed out to the CTAs that are free)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walkers", [[1], [1, 30, 2], [40, 1, 1, 1, 9, 3]])
def test_uneven_batches_equal_single_contexts(cfg, walkers):
    """One molecule, and very uneven ones (1 to 960 tiles, so that a problem has one
    reach item or many), each run twice with other points in between: every
    output equals the context's own call bit for bit (same products, same order)."""
    from paper_2512_16677_gb300 import qmckl
    mols = [cfg(2 if i % 2 == 0 else 3, walk_num=w) for i, w in enumerate(walkers)]
    ctxs = []
    for m in mols:
        c = qmckl.Context("bf16x3")
        c.set_molecule(m)
        c.set_points_device(torch.from_numpy(m.coord).cuda())
        ctxs.append(c)
    batch = qmckl.Batch(ctxs)
    for shift in (0.0, 0.3, 0.0):
        coords = [torch.from_numpy(m.coord + shift).cuda() for m in mols]
        for c, x in zip(ctxs, coords):
            c.set_points_device(x)
        outs = [o.clone() for o in batch.run()]
        batch.synchronize()
        for m, x, o in zip(mols, coords, outs):
            single = qmckl.Context("bf16x3")
            single.set_molecule(m)
            single.set_points_device(x)
            ref = single.mo_vgl_device()
            torch.cuda.synchronize()
            single.synchronize()
            assert torch.equal(ref, o), float((ref - o).abs().max())
            single.close()
