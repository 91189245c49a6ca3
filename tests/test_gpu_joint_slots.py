"""The probe block of joint products: teams' accumulators that their first position overwrites
(nothing zeroes them), summed over the teams that had one.  Position counts below, at and
above the teams in flight; a second product on the same context finds the first one's values
in the accumulators; results written over the input vector.  Against the FP64 oracle at the
suite's 1e-5 (Gaussian metric)."""
import numpy as np
import pytest

import oracle
from paper_2103_01767_gb300 import synth
from tests import parity
from tests.test_gpu_joint import c64, f32, host, lib, setup  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,vpt", [((96, 32, 1), 0), ((96, 32, 5), 32), ((96, 32, 2500), 32), ((96, 32, 1300), 16),
                                       ((160, 64, 3), 0), ((160, 64, 700), 32), ((160, 64, 310), 16), ((200, 128, 153), 0)])
def test_joint_product_team_slots(lib, shape, vpt):  # noqa: F811
    n, m, K = shape
    case, ctx, O, P = setup(lib, shape)
    lib.lm_destroy(ctx)
    ctx = lib.lm_init(n, n, m, m, torch.from_numpy(case.pos).cuda(), f32(case.y), 0, case.b, joint=1, values_per_thread=vpt)
    lib.forward_loss(ctx, c64(O), c64(P), cache=1)
    pb = case.problem()
    for seed in (70, 71):
        v = synth.to_c64(synth.random_complex(n * n + m * m, seed=seed))
        ref = oracle.ggn_matvec_z(pb, O, v, lam=0.2, P=P, joint=True)
        vO, vP = c64(v[:n * n].reshape(n, n)), c64(v[n * n:].reshape(m, m))
        outO, outP = torch.empty_like(vO), torch.empty_like(vP)
        lib.ggn_matvec(ctx, vO, outO, 0.2, vP=vP, outP=outP)
        parity.check("joint product, object block (team slots)", host(outO).ravel(), ref[:n * n])
        parity.check("joint product, probe block (team slots)", host(outP).ravel(), ref[n * n:])
        lib.ggn_matvec(ctx, vO, vO, 0.2, vP=vP, outP=vP)      # in place
        parity.check("joint product in place, object block", host(vO).ravel(), ref[:n * n])
        parity.check("joint product in place, probe block", host(vP).ravel(), ref[n * n:])
    D = torch.empty(n * n + m * m, device="cuda")
    for floor in (0.0, 0.05):
        lib.ggn_diag(ctx, D, floor)
        rO, rP = oracle.ggn_diag(pb, O, P, floor_rel=floor)
        parity.check(f"Dg(G) (floor {floor}, position counts)", host(D), np.concatenate([rO.ravel(), rP.ravel()]))
    lib.lm_destroy(ctx)
