"""The two-node kernel with the pairs of a plane in one run over the blocks
(its default where rows fill their warps badly) against blocks of 64 pairs x 2 rows: the same
bits, on rows of one node, of odd lengths, around a warp and a block, and on
longer rows without padding."""

import numpy as np
import pytest
import torch

from paper_1309_1983_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1309_1983_gb300 import build as B
    B.build()


GEOMS = {"periodic": ((0, 0, 0), None, False), "walls_y": ((0, 1, 0), None, False),
         "cavity": ((1, 1, 1), (0.05, 0.01, 0.0), False),
         "onsite": ((1, 1, 1), (0.05, 0.0, 0.0), True)}
SHAPES = [(1, 90, 60), (3, 70, 30), (37, 61, 9), (63, 33, 5), (101, 30, 11), (127, 17, 4),
          (160, 9, 11), (193, 8, 9), (300, 5, 7)]


@pytest.mark.parametrize("storage", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("geom", sorted(GEOMS))
@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
def test_same_bits_as_blocks_of_rows(shape, geom, storage):
    from paper_1309_1983_gb300.lattice import Lattice
    nx, ny, nz = shape
    walls, lid, onsite = GEOMS[geom]
    if onsite and nx < 3:
        pytest.skip("on-site walls need three nodes")
    u = torch.from_numpy(W.noise((3, nz, ny, nx), 2, 0.04)).float().cuda()
    F = torch.from_numpy(W.noise((3, nz, ny, nx), 3, 1e-3)).float().cuda()
    for force in (False, True):
        got = []
        for blocks in (False, True):
            L = Lattice(nx, ny, nz, 0.7, walls=tuple(bool(w) for w in walls), lid=lid,
                        storage=storage, force=force, onsite=onsite)
            L.set_fusion("off")
            if blocks:
                L.set_pair_block(64, 2)
            if force:
                L.force.copy_(F)
            L.init_equilibrium(u=u)
            rho, v = L.step_moments(5)
            got.append((L.get_f(), rho.cpu().numpy(), v.cpu().numpy()))
            L.close()
        for a, b in zip(*got):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("walls", [(0, 0, 0), (1, 1, 1), (1, 0, 1)])
@pytest.mark.parametrize("shape", [(1, 40, 9), (33, 21, 7), (65, 12, 5), (101, 30, 4), (193, 8, 9)],
                         ids=lambda s: "x".join(map(str, s)))
def test_reverse_step_has_the_bits_of_the_regathering_form(shape, walls):
    """The reverse step from moments, a run over the padded rows, against
    lbm_adjoint_step, which keeps blocks of rows."""
    import ctypes

    from paper_1309_1983_gb300 import capi
    from paper_1309_1983_gb300.lattice import Lattice

    def ptr(t):
        return ctypes.c_void_p(t.data_ptr())

    nx, ny, nz = shape
    L = Lattice(nx, ny, nz, 0.7, walls=tuple(bool(w) for w in walls),
                lid=(0.05, 0.0, 0.0) if walls[2] else None, force=True)
    L.force.copy_(torch.from_numpy(W.noise((3, nz, ny, nx), 3, 1e-3)).float())
    L.init_equilibrium(u=torch.from_numpy(W.noise((3, nz, ny, nx), 2, 0.04)).float().cuda())
    cur, other = L.current_buffers()
    rho = torch.empty((nz, ny, nx), device="cuda")
    u = torch.empty((3, nz, ny, nx), device="cuda")
    L.step_to_moments(cur, other, rho, u)
    n = L.layout.lambda_bytes // 4
    lam = torch.from_numpy(W.noise(n, 8, 1.0)).float().cuda()
    got = []
    for name, state in (("lbm_adjoint_step", (ptr(cur),)),
                        ("lbm_adjoint_step_moments", (ptr(rho), ptr(u)))):
        out = torch.zeros(n, device="cuda")
        gF = torch.ones((3, nz, ny, nx), device="cuda")
        capi.call(name, L.handle, *state, ptr(lam), ptr(out), ptr(gF))
        got.append((out.cpu().numpy(), gF.cpu().numpy()))
    np.testing.assert_array_equal(got[0][0], got[1][0])
    np.testing.assert_array_equal(got[0][1], got[1][1])
