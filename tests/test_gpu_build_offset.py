"""A mesh far from the origin of its coordinates (a site's geographic system, a part in an assembly's
frame) gives the blocks it gives at the origin: the FP32 entries take differences of points, and
those must not lose to the distance more than FP64 coordinates do.

The vertices are multiples of 2^-26, so that moving the mesh by integers below 2^26 is exact; its
quadrature points are FP64 sums at 2^26 then, off by up to 2^-27 a term, 1e-8 of the shortest edges'
1e-3: 1e-5, which the entries (1/R and its differences over an edge) answer with a few times that.
Held to 1e-4 of the block's largest entry; points held to 2^-49 of their distance give 7e-4.
"""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("basis", ["rwg", "swg"])
def test_blocks_of_a_moved_mesh(basis):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from synth import box_tets, icosphere, random_permittivity
    from paper_2307_03968_gb300.hm import HMatrix
    rng = np.random.default_rng(8)
    if basis == "rwg":
        (xyz, cells), eps = icosphere(2, 0.01), None
    else:
        xyz, cells = box_tets((0.0045, 0.003, 0.003), (3, 2, 2))
        eps = random_permittivity(len(cells), 2.0, 6.0, seed=1)
    xyz = np.round((xyz + 1e-4 * rng.uniform(-1, 1, xyz.shape)) * 2.0 ** 26) * 2.0 ** -26
    here, there = [HMatrix.build(x, cells, eps_r=eps, leaf_size=24, arity=2, adm=1.0, aca_tol=1e-4, wavelength=0.1, levels=1)
                   for x in (xyz, xyz + np.array([46976205.0, -59055801.0, 33554435.0]))]
    assert np.array_equal(here.perm(), there.perm())
    k = here.blocks(1)[4]
    assert np.array_equal(k == 0, there.blocks(1)[4] == 0)
    worst = 0.0
    for idx in np.nonzero(k == 0)[0]:
        a, b = here.block(1, idx), there.block(1, idx)
        worst = max(worst, np.abs(a - b).max() / np.abs(a).max())
    here.close()
    there.close()
    assert worst < 1e-4, worst
