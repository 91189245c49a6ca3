"""The CG iteration's one-cluster form at the edges of its range (elements per thread 1 to 12,
then the cooperative form), against the three-launch form: the same bits on tiled scans, as in
test_gpu_cg_forms.py.  And linearisation and product at a point the caller hands over in
buffers that are overwritten right after the calls, with positions fewer than CTAs."""
import numpy as np
import pytest

import oracle
from paper_2103_01767_gb300 import synth
from tests import parity
from tests.problems import make_case
from tests.test_gpu_cg_forms import both_forms, c64, lib  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,scaled,joint", [(64, 0, 0), (64, 1, 1), (128, 0, 0), (160, 1, 0), (192, 0, 1), (224, 1, 0),
                                            (256, 0, 1), (288, 0, 0), (320, 1, 0)])
def test_cluster_cg_is_bit_identical(lib, n, scaled, joint):  # noqa: F811
    m = 32
    case = make_case(n, m, loss=0, seed=6, grid=n // m, step=m, radius=0.3 * m)
    for kw in (dict(max_outer=2, fixed_cg=5), dict(max_outer=3)):
        a, b = both_forms(lib, case, joint, scaled=scaled, **kw)
        assert a["st"] == b["st"] and a["info"]["cg_total"] == b["info"]["cg_total"] > 0
        for key in ("f", "gnorm", "mu", "cg"):
            assert np.array_equal(a["info"][key], b["info"][key]), key
        assert np.array_equal(a["O"], b["O"]) and np.array_equal(a["P"], b["P"])


@pytest.mark.parametrize("n,m,K,joint", [(96, 32, 1, 0), (128, 64, 7, 1), (300, 128, 400, 0), (256, 64, 900, 0)])
def test_point_and_direction_may_be_overwritten_after_the_call(lib, n, m, K, joint):  # noqa: F811
    case = make_case(n, m, K=K, loss=0, seed=8)
    ctx = lib.lm_init(n, n, m, m, torch.from_numpy(case.pos).cuda(),
                      torch.from_numpy(np.ascontiguousarray(case.y, np.float32)).cuda(), 0, case.b, joint=joint)
    O = synth.to_c64(case.O_true + synth.random_complex((n, n), seed=9, scale=0.05))
    P = synth.to_c64(case.P * 1.02)
    pb = oracle.Problem((n, n), P, case.pos, case.y, 0, case.b)
    v = synth.to_c64(synth.random_complex(n * n + (m * m if joint else 0), seed=10))
    ref = oracle.ggn_matvec_z(pb, O, v, lam=0.4, P=P, joint=bool(joint))
    for _ in range(2):
        dO, dP, dv = c64(O), c64(P), c64(v)
        vO, vP = dv[:n * n].view(n, n), dv[n * n:].view(m, m) if joint else None
        out = torch.empty_like(dv)
        lib.forward_loss(ctx, dO, dP, cache=1)
        dO.fill_(7.0)
        dP.fill_(7.0)
        lib.ggn_matvec(ctx, vO, out[:n * n], 0.4, vP=vP, outP=out[n * n:] if joint else None)
        dv.fill_(7.0)
        parity.check("(G + 0.4 I) v, overwritten inputs", out.cpu().numpy(), ref)
        g = torch.empty((n, n), dtype=torch.complex64, device="cuda")
        lib.gradient(ctx, g)
        parity.check("grad f, overwritten inputs", g.cpu().numpy(), oracle.gradient(pb, O))
    lib.lm_destroy(ctx)
