"""What this library is measured on: its public calls at the sizes its users run.

Inputs are synthetic data of the workloads in ``synth.py`` and ``bench.py``: textured objects
(amplitude in [0.8, 1], phase in [-pi/4, pi/4]), a defocused disk probe, a jittered raster scan,
noiseless amplitudes or Poisson counts over a small detector background.  They are drawn here
with torch alone, so that every build of the library sees the same numbers.  A case names its
kind and sizes; ``exact`` evaluates the same call in FP64 with plain torch.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2103_01767_gb300 import ptylm
from paper_2103_01767_gb300.autograd import MagnitudeProblem, far_field_magnitude

DEV = "cuda"
GAUSSIAN, POISSON = 0, 1


# ---------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------
def listed():
    return [
        # one GGN product of the smallest workload (128^2 object, 32^2 probe): launches and latency
        dict(name="matvec_small", kind="matvec", ny=128, nx=128, m=32, K=64, loss=GAUSSIAN, peak=0.0, joint=False,
             scaled=False),
        # a whole reconstruction of that workload's first outer iterations, adaptive CG
        dict(name="lm_small", kind="lm", ny=128, nx=128, m=32, K=64, loss=GAUSSIAN, peak=0.0, joint=False, scaled=False,
             projected=False, outer=3, fixed_cg=0),
        # the blind workload's product over (object, probe) with the diagonal scaling of PLM
        dict(name="matvec_joint", kind="matvec", ny=256, nx=256, m=64, K=400, loss=POISSON, peak=1e4, joint=True,
             scaled=True),
        # the blind workload's solver: PLM-J with the projection of Algorithm 2
        dict(name="lm_joint", kind="lm", ny=256, nx=256, m=64, K=400, loss=POISSON, peak=1e4, joint=True, scaled=True,
             projected=True, outer=3, fixed_cg=8),
        # a linearisation for a caller's own solver: loss, gradient and GGN diagonal, odd sizes
        dict(name="linearise", kind="linearise", ny=611, nx=747, m=64, K=1531, loss=POISSON, peak=1e3, joint=False),
        # the product of the large workload, the inner loop of every LM step
        dict(name="matvec_large", kind="matvec", ny=1024, nx=1024, m=128, K=3600, loss=POISSON, peak=1e3, joint=False,
             scaled=False),
        # one outer iteration of the large workload with 10 CG iterations, as bench.py steps it
        dict(name="lm_large", kind="lm", ny=1024, nx=1024, m=128, K=3600, loss=POISSON, peak=1e3, joint=False,
             scaled=False, projected=False, outer=1, fixed_cg=10),
        # torch training through the forward model: magnitudes and their reverse-mode gradient
        dict(name="autograd_vjp", kind="vjp", ny=900, nx=777, m=128, K=1400, joint=False, stored=True),
        # forward mode, exit waves recomputed (what a memory budget below the phasors' size asks for)
        dict(name="autograd_jvp", kind="jvp", ny=1024, nx=1024, m=128, K=2025, joint=False, stored=False),
        # 64 independent reconstructions of uneven sizes, one LM step of all of them
        dict(name="batch_lm", kind="batch", B=64, sizes=7, outer=1, fixed_cg=10),
        # the learned start of a 1024^2 reconstruction: 225 patterns through the network, stitched
        dict(name="learned_init", kind="learned", ny=1024, nx=1024, K=900, count=225, c1=64, c2=128, c3=256, max_batch=256),
        # the gradient of one training step of that network
        dict(name="train_grad", kind="train", N=64, c1=64, c2=128, c3=256),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["matvec", "matvec", "linearise", "lm", "vjp", "jvp", "batch", "learned", "train"])
    if kind == "batch":
        return dict(kind=kind, B=rng.randint(6, 48), sizes=rng.randint(100, 10**6), outer=1, fixed_cg=rng.randint(3, 10))
    if kind == "learned":
        K = rng.randint(300, 900)
        return dict(kind=kind, ny=rng.randint(700, 1024), nx=rng.randint(700, 1024), K=K, count=rng.randint(20, 225),
                    c1=64, c2=128, c3=256, max_batch=rng.choice([64, 256]))
    if kind == "train":
        return dict(kind=kind, N=rng.randint(7, 64), c1=64, c2=128, c3=256)
    m = rng.choice([32, 64, 128])
    K = _log_int(rng, 50, {32: 12000, 64: 5000, 128: 3500}[m])
    lo = max(2 * m, 128)
    case = dict(kind=kind, ny=_log_int(rng, lo, 1024), nx=_log_int(rng, lo, 1024), m=m, K=K,
                joint=m < 128 and rng.random() < 0.4)
    if kind in ("vjp", "jvp"):
        return dict(case, stored=rng.random() < 0.5)
    loss = rng.choice([GAUSSIAN, POISSON])
    case.update(loss=loss, peak=rng.choice([1e3, 1e4]) if loss == POISSON else 0.0)
    if kind == "matvec":
        case.update(scaled=rng.random() < 0.3)
    if kind == "lm":
        case.update(scaled=case["joint"] or rng.random() < 0.5, projected=False, outer=rng.randint(1, 2),
                    fixed_cg=rng.randint(3, 8))
        case["K"] = min(case["K"], 900)
    return case


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
def _gen(seed, tag):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1000003 + tag) & 0x7FFFFFFF)


def _texture(ny, nx, g, lo, hi):
    """A Gaussian-filtered (sigma 3 px, periodic) noise field, min-max mapped to [lo, hi]."""
    f = torch.randn(ny, nx, generator=g, device=DEV)
    fy = torch.fft.fftfreq(ny, device=DEV)[:, None]
    fx = torch.fft.rfftfreq(nx, device=DEV)[None]
    f = torch.fft.irfft2(torch.fft.rfft2(f) * torch.exp(-2 * (math.pi * 3.0) ** 2 * (fy ** 2 + fx ** 2)), s=(ny, nx))
    f = f - f.min()
    return lo + (hi - lo) * f / f.max()


def _object(ny, nx, seed, tag):
    g = _gen(seed, tag)
    return torch.polar(_texture(ny, nx, g, 0.8, 1.0), _texture(ny, nx, g, -math.pi / 4, math.pi / 4))


def _probe(m):
    """Disk of radius 0.3125 m with a quadratic phase reaching pi at its edge."""
    c, radius = (m - 1) / 2.0, 0.3125 * m
    a = torch.arange(m, device=DEV, dtype=torch.float64) - c
    r = torch.sqrt(a[:, None] ** 2 + a[None] ** 2)
    p = (r <= radius) * torch.exp(1j * math.pi * (r / radius) ** 2)
    return p.to(torch.complex64)


def _positions(ny, nx, m, K, seed):
    """The first K points of a raster spread over the object, +-2 px of jitter (int32, host)."""
    rng = np.random.default_rng([int(seed), 11])
    gy = max(1, int(math.ceil(math.sqrt(K * max(1, ny - m) / max(1, nx - m)))))
    gx = -(-K // gy)
    y = np.linspace(0, ny - m, gy) if gy > 1 else np.array([(ny - m) / 2])
    x = np.linspace(0, nx - m, gx) if gx > 1 else np.array([(nx - m) / 2])
    pos = np.stack(np.meshgrid(y, x, indexing="ij"), -1).reshape(-1, 2)[:K].round().astype(np.int64)
    pos = pos + rng.integers(-2, 3, pos.shape)
    return np.clip(pos, 0, [ny - m, nx - m]).astype(np.int32)


def _index(pos, m, nx):
    a = torch.arange(m, device=DEV)
    return (pos[:, 0, None, None].long() + a[:, None]) * nx + pos[:, 1, None, None].long() + a


def _intensity(O, P, pos):
    """|F(P . patch)|^2, single precision, in chunks of positions."""
    m, out = P.shape[0], []
    for i in range(0, pos.shape[0], 512):
        psi = O.reshape(-1)[_index(pos[i:i + 512], m, O.shape[1])] * P
        out.append(torch.fft.fft2(psi, norm="ortho").abs().square())
    return torch.cat(out)


def _scan(ny, nx, m, K, loss, peak, seed):
    """Object, probe (scaled to `peak` photons in the brightest pixel), positions, counts y and
    the background they carry: a tenth of a count per pixel, or 1e-8 for noiseless amplitudes."""
    O, P = _object(ny, nx, seed, 1), _probe(m)
    pos = torch.from_numpy(_positions(ny, nx, m, K, seed)).to(DEV)
    h = _intensity(O, P, pos)
    b = 1e-8
    if loss == POISSON:
        s = peak / float(h.max())
        P = (P * math.sqrt(s)).to(torch.complex64)
        b = 0.1
        y = torch.poisson(h * s + b, generator=_gen(seed, 2))
    else:
        y = h + b
    return O.contiguous(), P.contiguous(), pos, y.contiguous(), b


def _iterate(O, seed):
    """An iterate part of the way to O: O with a smooth error of some 10 %."""
    return (O + 0.3 * (_object(*O.shape, seed, 3) - 0.9)).contiguous()


def _vector(shape, seed, tag):
    g = _gen(seed, tag)
    return torch.complex(torch.randn(shape, generator=g, device=DEV), torch.randn(shape, generator=g, device=DEV))


def _start(case, O, P):
    """Flat object; blind problems also start from the unphased disk."""
    return torch.ones_like(O), (P.abs().to(torch.complex64) if case["joint"] else P.clone())


def _members(case):
    """Sizes of a batch's problems (probe 32/64/128, object 128..512, 64..1024 positions)."""
    rng = np.random.default_rng(case["sizes"])
    out = []
    for _ in range(case["B"]):
        m = int(rng.choice([32, 64, 128]))
        out.append(dict(m=m, ny=int(rng.integers(max(128, 2 * m), 513)), nx=int(rng.integers(max(128, 2 * m), 513)),
                        K=int(rng.integers(64, 1025)), loss=int(rng.integers(0, 2)), peak=1e3))
    return out


def _net_params(case, seed):
    """He-normal weights and zero biases, W1 b1 ... W6 b6 flat."""
    g, parts = _gen(seed, 5), []
    for ci, co, *_ in _layers(case):
        parts.append((torch.randn(co * ci * 9, generator=g, device=DEV) * math.sqrt(2 / (9 * ci))))
        parts.append(torch.zeros(co, device=DEV))
    return torch.cat(parts)


def _layers(case):
    """(c_in, c_out, stride, upsampled, relu)"""
    a, b, c = case["c1"], case["c2"], case["c3"]
    return [(2, a, 2, 0, 1), (a, b, 2, 0, 1), (b, c, 2, 0, 1), (c, b, 1, 1, 1), (b, a, 1, 1, 1), (a, 2, 1, 1, 0)]


def _physics(y, P):
    """F^-1(sqrt(y) u) conj(P) / (|P|^2 + 1e-3 max|P|^2), u = F(P) / max(|F(P)|, 1e-3 max|F(P)|)."""
    fp = torch.fft.fft2(P, norm="ortho")
    u = fp / fp.abs().clamp_min(1e-3 * float(fp.abs().max()))
    e = torch.fft.ifft2(y.sqrt() * u, norm="ortho")
    p2 = P.abs().square()
    e = e * (P.conj() / (p2 + 1e-3 * p2.max()))
    return torch.stack([e.real, e.imag], 1).contiguous()


def _training_pairs(case, seed):
    """(physics input, object patch) pairs from random places of a 1024^2 object."""
    O, P = _object(1024, 1024, seed, 1), _probe(128)
    rng = np.random.default_rng([int(seed), 13])
    pos = torch.from_numpy(rng.integers(0, 1024 - 128 + 1, (case["N"], 2)).astype(np.int32)).to(DEV)
    T = O.reshape(-1)[_index(pos, 128, 1024)]
    X = _physics(_intensity(O, P, pos), P)
    return X, torch.stack([T.real, T.imag], 1).contiguous(), (P.abs() > 0).float().contiguous()


def _inputs(case, seed):
    k = case["kind"]
    if k == "train":
        X, T, mask = _training_pairs(case, seed)
        return dict(X=X, T=T, mask=mask, params=_net_params(case, seed))
    if k == "learned":
        O, P, pos, y, b = _scan(case["ny"], case["nx"], 128, case["K"], GAUSSIAN, 0.0, seed)
        idx = torch.from_numpy(np.linspace(0, case["K"] - 1, case["count"]).astype(np.int32)).to(DEV)
        return dict(P=P, pos=pos, y=y, b=b, idx=idx, params=_net_params(case, seed))
    if k == "batch":
        out = []
        for i, q in enumerate(_members(case)):
            O, P, pos, y, b = _scan(q["ny"], q["nx"], q["m"], q["K"], q["loss"], q["peak"], seed * 64 + i)
            out.append(dict(ny=q["ny"], nx=q["nx"], m=q["m"], positions=pos, y=y, probe=P, loss=q["loss"], background=b))
        return dict(problems=out)
    if k in ("vjp", "jvp"):
        # magnitudes of some 10^3 photons over a background of 0.1
        O, P, pos, y, b = _scan(case["ny"], case["nx"], case["m"], case["K"], POISSON, 1e3, seed)
        return dict(O=_iterate(O, seed), P=P, pos=pos, b=b, root_y=y.sqrt(), v=_vector(O.shape, seed, 4),
                    vP=_vector(P.shape, seed, 6))
    O, P, pos, y, b = _scan(case["ny"], case["nx"], case["m"], case["K"], case["loss"], case["peak"], seed)
    if k == "lm":
        O0, P0 = _start(case, O, P)
        return dict(O0=O0, P0=P0, pos=pos, y=y, b=b)
    d = dict(O=_iterate(O, seed), P=P, pos=pos, y=y, b=b)
    if k == "matvec":
        d.update(v=_vector(O.shape, seed, 4), vP=_vector(P.shape, seed, 6), lam=0.25)
        # a positive diagonal with a large spread, as the closed-form scaling of PLM has
        n = O.numel() + (P.numel() if case["joint"] else 0)
        d["D"] = (0.01 + torch.rand(n, generator=_gen(seed, 7), device=DEV) ** 2 * 10) if case["scaled"] else None
    return d


# ---------------------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------------------
def _context(case, d):
    return ptylm.lm_init(case["ny"], case["nx"], case["m"], case["m"], d["pos"], d["y"], case["loss"], d["b"],
                         joint=int(case["joint"]))


def prepare(case, seed):
    k, d = case["kind"], _inputs(case, seed)
    s = dict(d, case=case)
    if k == "train":
        s["net"] = ptylm.net_create((case["c1"], case["c2"], case["c3"]), max_batch=case["N"])
        ptylm.net_set_params(s["net"], d["params"].cpu().numpy())
    elif k == "learned":
        s["net"] = ptylm.net_create((case["c1"], case["c2"], case["c3"]), max_batch=case["max_batch"])
        ptylm.net_set_params(s["net"], d["params"].cpu().numpy())
        s["ctx"] = ptylm.lm_init(case["ny"], case["nx"], 128, 128, d["pos"], d["y"], GAUSSIAN, d["b"])
        s["O0"] = torch.empty((case["ny"], case["nx"]), dtype=torch.complex64, device=DEV)
    elif k == "batch":
        s["batch"] = ptylm.batch_init(d["problems"])
        s["flat"] = torch.ones(s["batch"].total, dtype=torch.complex64, device=DEV)
        ptylm.batch_forward_loss(s["batch"], s["flat"], cache=1)
        ptylm.batch_tune(s["batch"])
        del s["problems"]
    elif k in ("vjp", "jvp"):
        s["problem"] = MagnitudeProblem(case["ny"], case["nx"], case["m"], d["pos"], background=d["b"], joint=case["joint"],
                                        phasor_budget=2 ** 40 if case["stored"] else 0)
    else:
        s["ctx"] = _context(case, d)
        del s["y"]
        if k != "lm":
            s["out"] = torch.empty_like(d["O"])
            s["outP"] = torch.empty_like(d["P"]) if case["joint"] else None
        if k == "matvec":
            ptylm.forward_loss(s["ctx"], d["O"], d["P"], cache=1)
        if k == "linearise":
            s["D"] = torch.empty(d["O"].numel() + (d["P"].numel() if case["joint"] else 0), device=DEV)
    return s


def run(s):
    case = s["case"]
    k = case["kind"]
    if k == "matvec":
        joint = case["joint"]
        ptylm.ggn_matvec(s["ctx"], s["v"], s["out"], s["lam"], D=s["D"], vP=s["vP"] if joint else None, outP=s["outP"])
        return [s["out"], s["outP"]]
    if k == "linearise":
        f, dl2 = ptylm.forward_loss(s["ctx"], s["O"], s["P"], cache=1)
        ptylm.gradient(s["ctx"], s["out"], s["outP"])
        ptylm.ggn_diag(s["ctx"], s["D"])
        return [f, dl2, s["out"], s["outP"], s["D"]]
    if k == "lm":
        O, P = s["O0"].clone(), s["P0"].clone()
        _, info = ptylm.lm_solve(s["ctx"], O, P, max_outer=case["outer"], fixed_cg=case["fixed_cg"],
                                 scaled=int(case["scaled"]), projected=int(case["projected"]))
        return [O, P, info["f_final"]]
    if k == "vjp":
        O = s["O"].detach().requires_grad_(True)
        P = s["P"].detach().requires_grad_(case["joint"])
        zeta = far_field_magnitude(O, P, s["problem"])
        zeta.backward(zeta.detach() - s["root_y"])   # the gradient of sum (zeta - sqrt y)^2 / 2
        return [zeta.detach(), O.grad, P.grad]
    if k == "jvp":
        with torch.autograd.forward_ad.dual_level():
            O = torch.autograd.forward_ad.make_dual(s["O"], s["v"])
            P = torch.autograd.forward_ad.make_dual(s["P"], s["vP"]) if case["joint"] else s["P"]
            zeta, jv = torch.autograd.forward_ad.unpack_dual(far_field_magnitude(O, P, s["problem"]))
        return [zeta, jv]
    if k == "batch":
        z = s["flat"].clone()
        _, info = ptylm.batch_lm_solve(s["batch"], z, max_outer=case["outer"], fixed_cg=case["fixed_cg"])
        return [z, np.array([q["f_final"] for q in info], np.float32)]
    if k == "learned":
        ptylm.learned_init(s["ctx"], s["net"], s["P"], s["idx"], s["O0"])
        return [s["O0"]]
    loss = ptylm.net_loss_grad(s["net"], s["X"], s["T"], s["mask"])
    return [loss, ptylm.net_get_params(s["net"])[1]]


# ---------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------
def _fft_flops(K, M):
    return K * 5.0 * M * math.log2(M)


def _lm_work(K, M, N, joint, outer, cg):
    per = 2 * _fft_flops(K, M) + 24.0 * K * M * (2 if joint else 1)
    return dict(bytes=4.0 * K * M + 16.0 * N + 8.0 * M * (2 if joint else 1), flops=outer * (cg + 2.5) * per)


def work(case):
    k = case["kind"]
    if k in ("train", "learned"):
        n = case["N"] if k == "train" else case["count"]
        side, per = 128, 0.0
        for ci, co, stride, up, _ in _layers(case):
            side = side // 2 if stride == 2 else 2 * side
            per += 2.0 * side * side * ci * co * 9
        params = sum(co * ci * 9 + co for ci, co, *_ in _layers(case))
        if k == "train":
            return dict(bytes=n * 4.0 * 128 * 128 * 4 + 8.0 * params, flops=3 * n * per)
        return dict(bytes=n * 128 * 128 * 4.0 + 8.0 * case["ny"] * case["nx"] + 4.0 * params,
                    flops=n * per + _fft_flops(n, 128 * 128))
    if k == "batch":
        ws = [_lm_work(q["K"], q["m"] ** 2, q["ny"] * q["nx"], False, case["outer"], case["fixed_cg"]) for q in _members(case)]
        return dict(bytes=sum(w["bytes"] for w in ws), flops=sum(w["flops"] for w in ws))
    K, M, N = case["K"], case["m"] ** 2, case["ny"] * case["nx"]
    joint = case["joint"]
    if k == "matvec":
        # the cached factor a, v and out, P (and its block), D
        return dict(bytes=8.0 * K * M + 16.0 * N + 8.0 * M * (4 if joint else 1) + (4.0 * N if case["scaled"] else 0),
                    flops=2 * _fft_flops(K, M) + 24.0 * K * M * (2 if joint else 1))
    if k == "linearise":
        # y, O, P in; the cached factor, gradient and diagonal out
        return dict(bytes=12.0 * K * M + 20.0 * N + 8.0 * M, flops=2 * _fft_flops(K, M) + 40.0 * K * M)
    if k == "vjp":
        return dict(bytes=8.0 * K * M + 16.0 * N + 8.0 * M, flops=2 * _fft_flops(K, M) + 30.0 * K * M)
    if k == "jvp":
        return dict(bytes=8.0 * K * M + 16.0 * N + 8.0 * M, flops=2 * _fft_flops(K, M) + 30.0 * K * M)
    return _lm_work(K, M, N, joint, case["outer"], case["fixed_cg"] or 12)


# ---------------------------------------------------------------------------------------
# the same calls in FP64
# ---------------------------------------------------------------------------------------
class _Model:
    """The forward model, its metric and derivatives at (O, P), complex128, chunked over positions."""

    def __init__(self, pos, y, b, loss, m, shape):
        self.pos, self.y, self.b, self.loss, self.m, self.shape = pos, y, float(np.float32(b)), loss, m, shape

    def chunks(self):
        for i in range(0, self.pos.shape[0], 512):
            yield slice(i, i + 512), _index(self.pos[i:i + 512], self.m, self.shape[1])

    @staticmethod
    def gather(O, idx):
        return O.reshape(-1)[idx]

    def adjoint(self, out, idx, val):
        out.index_add_(0, idx.reshape(-1), torch.view_as_real(val.reshape(-1)))

    def terms(self, h, y):
        """l, dl/dzeta, d2l/dzeta2"""
        z = h.sqrt()
        if self.loss == GAUSSIAN:
            d = z - y.sqrt()
            return 0.5 * d * d, d, torch.ones_like(d)
        return h - torch.where(y > 0, y * h.log(), 0.0), 2 * z - 2 * y / z, 2 + 2 * y / h

    def linearise(self, O, P, grad=True):
        f = dl2 = 0.0
        gO = torch.zeros(O.numel(), 2, dtype=torch.float64, device=DEV)
        gP = torch.zeros_like(P)
        tr = torch.zeros(self.pos.shape[0], dtype=torch.float64, device=DEV)
        for sl, idx in self.chunks():
            o = self.gather(O, idx)
            ps = torch.fft.fft2(P * o, norm="ortho")
            h = ps.abs().square() + self.b
            l, d, d2 = self.terms(h, self.y[sl].double())
            f, dl2 = f + float(l.sum()), dl2 + float((d * d).sum())
            if grad:
                tr[sl] = d2.sum((1, 2))
                e = torch.fft.ifft2(ps * d / h.sqrt(), norm="ortho")
                self.adjoint(gO, idx, P.conj() * e)
                gP += (o.conj() * e).sum(0)
        return f, dl2, torch.view_as_complex(gO).reshape(O.shape), gP, tr

    def product(self, O, P, v, vP=None, weights=True):
        out = torch.zeros(O.numel(), 2, dtype=torch.float64, device=DEV)
        outP = torch.zeros_like(P)
        for sl, idx in self.chunks():
            o = self.gather(O, idx)
            ps = torch.fft.fft2(P * o, norm="ortho")
            d = P * self.gather(v, idx)
            d = torch.fft.fft2(d if vP is None else d + vP * o, norm="ortho")
            h = ps.abs().square() + self.b
            _, _, d2 = self.terms(h, self.y[sl].double())
            e = torch.fft.ifft2(ps * (d2 * (ps.conj() * d).real / h), norm="ortho")
            self.adjoint(out, idx, P.conj() * e)
            outP += (o.conj() * e).sum(0)
        return torch.view_as_complex(out).reshape(O.shape), outP

    def diagonal(self, O, P, tr, joint):
        M = self.m ** 2
        D = torch.zeros(O.numel(), dtype=torch.float64, device=DEV)
        DP = torch.zeros(P.shape, dtype=torch.float64, device=DEV)
        for sl, idx in self.chunks():
            t = (tr[sl] / (2 * M))[:, None, None]
            D.index_add_(0, idx.reshape(-1), (P.abs().square() * t).reshape(-1))
            DP += (self.gather(O, idx).abs().square() * t).sum(0)
        return torch.cat([D, DP.reshape(-1)]) if joint else D


def _flat(O, P=None):
    return torch.cat([O.reshape(-1), P.reshape(-1)]) if P is not None else O.reshape(-1).clone()


def _dot(a, b):
    return float((a.conj() * b).real.sum())


def _exact_lm(model, O, P, joint, scaled, projected, outer, fixed_cg, loss):
    """Algorithm 1 (and 2) with the library's default parameters."""
    N, beta = O.numel(), (0.9 if loss == POISSON else 0.1)
    split = lambda z: (z[:N].reshape(O.shape), z[N:].reshape(P.shape) if joint else P)  # noqa: E731
    z = _flat(O, P if joint else None)
    x = torch.zeros_like(z)
    mu, f_out = 1e-5, 0.0
    f_min = 0.0
    if projected and loss == POISSON:
        y = model.y.double()
        f_min = float((y - torch.where(y > 0, y * y.log(), 0.0)).sum())

    def project(z):
        r = torch.full((z.numel(),), 1.0, dtype=torch.float64, device=DEV)
        r[N:] = 1e8
        a = z.abs()
        return torch.where(a > r, z * (r / a.clamp_min(1e-300)), z)

    for _ in range(outer):
        f, dl2, gO, gP, tr = model.linearise(*split(z))
        g = _flat(gO, gP if joint else None)
        gnorm = math.sqrt(_dot(g, g))
        tol = min(beta, math.sqrt(gnorm)) * gnorm
        D = None
        if scaled:
            D = model.diagonal(*split(z), tr, joint)
            D[:N] = D[:N].clamp_min(1e-6 * float(D[:N].max()))
            if joint:
                D[N:] = D[N:].clamp_min(1e-6 * float(D[N:].max()))
        rho = 0.0
        while not rho > 1e-4:
            lam = mu if scaled else mu * math.sqrt(dl2)

            def A(v):
                w, wP = split(v)
                o, oP = model.product(*split(z), w, wP if joint else None)
                return _flat(o, oP if joint else None) + lam * (v if D is None else D * v)

            pre = (lambda r: r) if D is None else (lambda r: r / ((1 + lam) * D))
            r = -g - A(x)
            p = pre(r)
            rz, it = _dot(r, p), 0
            while it < (fixed_cg or 100):
                if not fixed_cg and math.sqrt(_dot(r, r)) <= tol:
                    break
                q = A(p)
                alpha = rz / _dot(p, q)
                x = x + alpha * p
                r = r - alpha * q
                w = pre(r)
                new = _dot(r, w)
                p, rz, it = w + (new / rz) * p, new, it + 1
            trial = z + x
            f_t = model.linearise(*split(trial), grad=False)[0]
            dd = _dot(x, x if D is None else D * x)
            dfp = 0.5 * (lam * dd - _dot(g, x)) + 0.5 * _dot(x, r)
            rho = (f - f_t) / dfp if dfp > 0 else -1.0
            mu = max(mu / 4, 1e-8) if rho > 0.75 else mu if rho > 0.25 else 4 * mu
        f_out = f
        if not projected:
            z, f_out = trial, f_t
            continue
        trial = project(trial)
        f_t = model.linearise(*split(trial), grad=False)[0]
        if f_t - f_min < 1e-6 * (f - f_min):
            z, f_out = trial, f_t
            continue
        s = trial - z
        ss = _dot(s, s)
        if not _dot(g, s) <= -1e-8 * math.sqrt(ss) ** 2.1:
            s, ss = -g, gnorm ** 2
        a = 1.0
        for _ in range(30):
            trial = project(z + a * s)
            f_t = model.linearise(*split(trial), grad=False)[0]
            if f_t <= f - 1e-4 * a * ss:
                z, f_out = trial, f_t
                break
            a *= 0.5
    return (*split(z), f_out)


def _network(case, params, X):
    """The encoder-decoder in FP64 with bfloat16-rounded weights; returns (output, weights, biases)."""
    a, off, ws = X.double(), 0, []
    for ci, co, stride, up, relu in _layers(case):
        w = params[off:off + co * ci * 9].bfloat16().double().reshape(co, ci, 3, 3).requires_grad_(True)
        off += co * ci * 9
        b = params[off:off + co].double().requires_grad_(True)
        off += co
        ws += [w, b]
        if up:
            a = a.repeat_interleave(2, 2).repeat_interleave(2, 3)
        a = F.conv2d(a, w, b, stride=stride, padding=1)
        a = F.relu(a) if relu else a
    return a, ws


def exact(case, seed):
    k, d = case["kind"], _inputs(case, seed)
    c128 = torch.complex128
    if k == "train":
        loss, grads = 0.0, None
        n_terms = 2.0 * case["N"] * float(d["mask"].double().sum())
        for i in range(0, case["N"], 16):
            out, ws = _network(case, d["params"], d["X"][i:i + 16])
            part = (d["mask"].double() * (out - d["T"][i:i + 16].double()).square()).sum() / n_terms
            gs = torch.autograd.grad(part, ws)
            loss += float(part.detach())
            grads = list(gs) if grads is None else [x + y for x, y in zip(grads, gs)]
        return [loss, torch.cat([g.reshape(-1) for g in grads])]
    if k == "learned":
        P = d["P"].to(c128)
        num = torch.zeros(case["ny"] * case["nx"], 2, dtype=torch.float64, device=DEV)
        den = torch.zeros(case["ny"] * case["nx"], dtype=torch.float64, device=DEV)
        w = P.abs().square()
        for i in range(0, case["count"], 32):
            sel = d["idx"][i:i + 32].long()
            with torch.no_grad():
                e = _network(case, d["params"], _physics(d["y"][sel].double(), P))[0]
            at = _index(d["pos"][sel], 128, case["nx"]).reshape(-1)
            num.index_add_(0, at, (e * w[None, None]).permute(0, 2, 3, 1).reshape(-1, 2))
            den.index_add_(0, at, w.expand(len(sel), -1, -1).reshape(-1))
        O = torch.where(den > 0, torch.view_as_complex(num) / den.clamp_min(1e-300), 1.0)
        return [O.reshape(case["ny"], case["nx"])]
    if k == "batch":
        zs, fs = [], []
        for q in d["problems"]:
            model = _Model(q["positions"], q["y"], q["background"], q["loss"], q["m"], (q["ny"], q["nx"]))
            O, _, f = _exact_lm(model, torch.ones(q["ny"], q["nx"], dtype=c128, device=DEV), q["probe"].to(c128), False,
                                False, False, case["outer"], case["fixed_cg"], q["loss"])
            zs.append(O.reshape(-1))
            fs.append(f)
        return [torch.cat(zs), torch.tensor(fs, dtype=torch.float64)]
    if k in ("vjp", "jvp"):
        O, P = d["O"].to(c128), d["P"].to(c128)
        model = _Model(d["pos"], d["root_y"], d["b"], GAUSSIAN, case["m"], O.shape)
        zs, js = [], []
        gO = torch.zeros(O.numel(), 2, dtype=torch.float64, device=DEV)
        gP = torch.zeros_like(P)
        for sl, idx in model.chunks():
            o = model.gather(O, idx)
            ps = torch.fft.fft2(P * o, norm="ortho")
            z = (ps.abs().square() + model.b).sqrt()
            zs.append(z)
            if k == "vjp":
                e = torch.fft.ifft2(ps * (z - d["root_y"][sl].double()) / z, norm="ortho")
                model.adjoint(gO, idx, P.conj() * e)
                gP += (o.conj() * e).sum(0)
            else:
                t = P * model.gather(d["v"].to(c128), idx)
                t = torch.fft.fft2(t + d["vP"].to(c128) * o if case["joint"] else t, norm="ortho")
                js.append((ps.conj() * t).real / z)
        if k == "jvp":
            return [torch.cat(zs), torch.cat(js)]
        return [torch.cat(zs), torch.view_as_complex(gO).reshape(O.shape), gP if case["joint"] else None]
    if k == "lm":
        model = _Model(d["pos"], d["y"], d["b"], case["loss"], case["m"], d["O0"].shape)
        return list(_exact_lm(model, d["O0"].to(c128), d["P0"].to(c128), case["joint"], case["scaled"], case["projected"],
                              case["outer"], case["fixed_cg"], case["loss"]))
    O, P = d["O"].to(c128), d["P"].to(c128)
    model = _Model(d["pos"], d["y"], d["b"], case["loss"], case["m"], O.shape)
    if k == "linearise":
        f, dl2, gO, gP, tr = model.linearise(O, P)
        return [f, dl2, gO, gP if case["joint"] else None, model.diagonal(O, P, tr, case["joint"])]
    joint, D = case["joint"], d["D"]
    v, vP = d["v"].to(c128), d["vP"].to(c128)
    o, oP = model.product(O, P, v, vP if joint else None)
    lam = d["lam"] * (torch.ones((), device=DEV) if D is None else D.double())
    N = O.numel()
    o = o + (lam if D is None else lam[:N].reshape(O.shape)) * v
    return [o, oP + (lam if D is None else lam[N:].reshape(P.shape)) * vP if joint else None]
