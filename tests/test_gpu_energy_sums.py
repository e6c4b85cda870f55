"""Mixed path: the short-range energies of a box leave FP32 molecule by
molecule, as compensated sums carried on in FP64."""
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


def _lattice(n, edge, seed):
    """n^3 waters on a lattice, O displaced by up to 0.1 A, random orientations."""
    rng = np.random.default_rng(seed)
    O = (np.stack(np.meshgrid(*[np.arange(n)] * 3, indexing="ij"), -1).reshape(-1, 3) + 0.5) * edge
    O = O + rng.uniform(-0.1, 0.1, O.shape)
    q, _ = np.linalg.qr(rng.normal(size=(n ** 3, 3, 3)))
    half = np.radians(104.52) / 2
    h = 0.9572 * np.array([[np.sin(half), np.cos(half), 0.0], [-np.sin(half), np.cos(half), 0.0]])
    return np.concatenate([O[:, None], O[:, None] + np.einsum("ka,mab->mkb", h, q)], 1)


def test_a_large_pair_energy_costs_the_molecules_after_it_nothing():
    """32,768 waters at rc 9, where a warp takes 27 molecules.  One pair of waters
    0.3 A apart, owned by the second molecule of a warp, has an undamped dispersion energy G
    above 1e3 times all the rest.  Moving molecules that follow in that warp changes the energy by
    as much with as without that pair, up to the rounding of sums that hold G: in
    FP64 some 30 additions of rms error 0.29 x 1.1e-16 G each, 2e-16 G, and twice that in the
    difference of two; an FP32 (hi, lo) pair carried from molecule to molecule rounds each of
    the lane's some 300 later additions to about 2^-49 G, 0.29 x 1.8e-15 x 17 = 9e-15 G in
    all.  Held to 2e-15 G."""
    import torch
    import paper_2201_00804_gb300 as pkg
    n, edge, mpw = 32, 3.1, 27
    x = _lattice(n, edge, 3)
    P = dict(synth.PARAMS, gamma6=0.0, gamma8=0.0, gamma10=0.0, ct_ae=2e5, alpha_o=0.01, alpha_h=0.01,
             alpha_m_damp=0.01)
    mp = np.tile(synth.make_config("water216")[0].mp_local.reshape(-1, 5, 10)[:1], (n ** 3, 1, 1))
    ctx = pkg.sibfa_create(P, mp, periodic=True, box=(n * edge,) * 3, rc=9.0, grid=96, ewald_alpha=0.4, pcg_tol_D=1e-3,
                           precision=pkg.PREC_MIXED, warm_start=False)

    def disp(y):
        return pkg.sibfa_energy_forces(ctx, torch.tensor(y.reshape(-1), dtype=torch.float64, device="cuda"))["disp"]

    worst, G = 0.0, 0.0
    rng = np.random.default_rng(4)
    partner = n ** 3 - 5                         # an odd place: its pair with an even lower one is the lower one's
    try:
        for row in (16, 124, 232, 340):          # lattice rows of 32 molecules
            i = row * n + 2
            assert i % mpw == 1 and i % 2 == 0
            moved = np.arange(i + 4, i + 24)     # the same warp's, 12 A and more from molecule i
            with_g = x.copy()
            with_g[partner] = x[i] + np.array([0.3, 0.0, 0.0])
            base, base_g = disp(x), disp(with_g)
            G = max(G, abs(base_g - base))
            for _ in range(5):
                s = rng.uniform(-0.1, 0.1, (20, 1, 3))
                a, b = x.copy(), with_g.copy()
                a[moved] += s
                b[moved] += s
                worst = max(worst, abs((disp(b) - base_g) - (disp(a) - base)))
    finally:
        pkg.sibfa_destroy(ctx)
    assert G > 1e7 and worst <= 2e-15 * G, (worst / G, G)
