"""Gas phase, FP64: every sum has a fixed order, whatever the order in which
warps finish, so the same call gives the same bits."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2201_00804_gb300 import build
    build.build()


@pytest.mark.parametrize("virial", [False, True], ids=["forces", "virial"])
@pytest.mark.parametrize("sizes", [[8], [200], [2, 70, 5, 130, 33, 1, 64]], ids=["small", "one", "batch"])
@pytest.mark.parametrize("prec", ["PREC_FP64", "PREC_MIXED"])
def test_same_call_same_bits(sizes, virial, prec):
    import paper_2201_00804_gb300 as pkg
    s, start, _ = synth.make_cluster_sizes(sizes, seed=33)
    pos = np.ascontiguousarray(s.pos.reshape(-1))
    kw = dict(cluster_start=start) if len(sizes) > 1 else {}
    ctx = pkg.sibfa_create(synth.PARAMS, s.mp_local, periodic=False, pcg_tol_D=1e-9, precision=getattr(pkg, prec),
                           warm_start=False, **kw)
    try:
        seen = set()
        for _ in range(30):
            F, W = np.zeros_like(pos), np.zeros((3, 3))
            e = pkg.sibfa_energy_forces(ctx, pos, F, **(dict(virial=W) if virial else {}))
            seen.add((tuple(e.values()), F.tobytes(), W.tobytes()))
        assert len(seen) == 1, len(seen)
    finally:
        pkg.sibfa_destroy(ctx)
