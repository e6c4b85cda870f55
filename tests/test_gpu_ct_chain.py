"""Mixed path: the charge transfer's chain rule through the intramolecular
potentials V_int takes dE/dV_int times ke as an FP64 product, rounded once."""
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


def test_v_int_chain_takes_ke_in_fp64():
    """Parameters under which that chain is the force: no radial decay and no
    p overlap (eta = 0, cp_lp = 0: the transfer depends on V_int alone, but for
    some 1e-3 through the denominator), and a strength far above the other
    terms'.  Against FP64 the forces are off by a part that all molecules share
    (their geometry is the same, and so are its roundings) and a random one.  ke is taken
    once as an FP32 number and once 0.499 of its last place higher, 5e-8 of itself: a product
    with the rounded ke moves the shared part by those 5e-8, an FP64 product by
    nothing but the random roundings, 1.3e-7 a molecule and so 8e-9 of the
    difference over 600 of them.  Held to half of 5e-8."""
    import paper_2201_00804_gb300 as pkg
    s, start, _ = synth.make_cluster_sizes([3] * 200, seed=90)
    pos = np.ascontiguousarray(s.pos.reshape(-1))

    def shift(ke):
        P = dict(synth.PARAMS, ke=ke, ct_eta=0.0, cp_lp=0.0, cs_lp=1.0, ct_t=1024.0, ct_m=0.0, ct_ae=2.0 ** 20,
                 ct_ah=0.0)
        F = []
        for prec in (pkg.PREC_FP64, pkg.PREC_MIXED):
            ctx = pkg.sibfa_create(P, s.mp_local, periodic=False, cluster_start=start, pcg_tol_D=1e-9, precision=prec,
                                   warm_start=False)
            f = np.zeros_like(pos)
            try:
                e = pkg.sibfa_energy_forces(ctx, pos, f)
            finally:
                pkg.sibfa_destroy(ctx)
            assert abs(e["ct"]) > 1e4 * sum(abs(e[t]) for t in ("elec", "pen", "rep", "disp", "xdisp", "pol"))
            F.append(f)
        return float((F[1] - F[0]) @ F[0] / (F[0] @ F[0]))

    ke = np.float32(301.37)
    up = float(ke) + 0.499 * float(np.spacing(ke))
    assert np.float32(up) == ke and up / float(ke) - 1.0 > 5e-8
    d = shift(up) - shift(float(ke))
    assert abs(d) <= 2.5e-8, d
