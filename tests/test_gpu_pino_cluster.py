"""The PINO's network paths (the cluster kernel to 128 x 128, the staged one beyond): layer counts,
hidden widths at and between their column passes, ragged states, and the two cluster sizes, against the network in 64 bits with the kernel's BF16
rounding points."""
import dataclasses

import numpy as np
import pytest

import workloads as wl
from tests.gpu_util import start_state, to_gpu, to_np

pytestmark = pytest.mark.gpu

def rounded_network(u, xmax, tau, dtau, p, w):
    """The increment w on the network grid and, per node, the sum of magnitudes it cancels from."""
    import torch
    MP = 128 if u.shape[0] <= 128 else 256
    r = lambda a: a.float().bfloat16().double()                                     # noqa: E731
    t = lambda a: torch.tensor(np.asarray(a), device="cuda").double()               # noqa: E731
    C, mx, my = 32, 12, 12
    M = u.shape[0]
    if M != MP:
        pos = torch.arange(MP, device="cuda").double() * ((M - 1) / (MP - 1))
        i0 = pos.floor().clamp(max=M - 2).long()
        f = pos - i0
        uu = t(u)
        rows = uu[i0] * (1 - f)[:, None] + uu[i0 + 1] * f[:, None]
        un = rows[:, i0] * (1 - f) + rows[:, i0 + 1] * f
    else:
        un = t(u)
    x = torch.arange(MP, device="cuda").double() * (xmax / (MP - 1))
    one = torch.ones_like(un)
    a = torch.stack([un, x[None, :] * one, x[:, None] * one] +
                    [float(v) * one for v in (tau, dtau, p.sigma1, p.sigma2, p.rho, p.r)])
    act = r(torch.einsum("cyx,co->yxo", a, t(w["lift_w"])) + t(w["lift_b"]))
    n = torch.arange(MP, device="cuda").double()
    kx = torch.arange(mx, device="cuda").double()
    ky = torch.cat([torch.arange(my), torch.arange(MP - my, MP)]).to("cuda").double()
    ph, th = 2 * np.pi * kx[:, None] * n / MP, 2 * np.pi * ((ky[:, None] * n) % MP) / MP
    cx, sx, cy, sy = r(ph.cos()), r(ph.sin()), r(th.cos()), r(th.sin())
    g = torch.where(kx == 0, 1.0, 2.0)[:, None] / MP ** 2
    gc, gs = r(g * ph.cos()), r(g * ph.sin())
    for l in range(w["pw_w"].shape[0]):
        re, im = r(torch.einsum("yxc,kx->yck", act, cx)), r(torch.einsum("yxc,kx->yck", act, -sx))
        e = lambda m, v: torch.einsum("qy,yck->qkc", m, v)                          # noqa: E731
        re, im = r(e(cy, re) + e(sy, im)), r(e(cy, im) - e(sy, re))
        wr, wi = r(t(w["spec_w"][l].real)), r(t(w["spec_w"][l].imag))
        m = lambda v, k: torch.einsum("qkc,qkco->qko", v, k)                        # noqa: E731
        re, im = r(m(re, wr) - m(im, wi)), r(m(re, wi) + m(im, wr))
        e = lambda k, v: torch.einsum("qy,qko->yko", k, v)                          # noqa: E731
        re, im = r(e(cy, re) - e(sy, im)), r(e(sy, re) + e(cy, im))
        v = torch.einsum("yko,kx->yxo", re, gc) - torch.einsum("yko,kx->yxo", im, gs)
        v = v + act @ r(t(w["pw_w"][l])) + t(w["pw_b"][l])
        act = r(v.clamp(min=0.0))
    h = (act @ r(t(w["proj1_w"])) + t(w["proj1_b"])).clamp(min=0.0)
    w2 = t(w["proj2_w"])
    return h @ w2 + float(w["proj2_b"]), h @ w2.abs()


@pytest.mark.parametrize("layers,hidden,M", [(1, 16, 128), (2, 144, 128), (3, 256, 41), (5, 128, 127), (1, 112, 8),
                                             (1, 16, 256), (2, 144, 200)])
def test_shapes(tmp_path, layers, hidden, M):
    import torch
    import paper_2404_02521_gb300 as bs
    from paper_2404_02521_gb300 import pino_io
    bs.load()
    arch = dataclasses.replace(wl.PinoArch(), layers=layers, proj_hidden=hidden)
    path = str(tmp_path / "w.bin")
    pino_io.write_weights(path, wl.pino_random_weights(arch, seed=layers, spectral_scale=8.0), arch.in_channels,
                          arch.width, arch.modes_x, arch.modes_y, layers, hidden)
    w, _ = pino_io.read_weights(path)
    net, g, p = bs.Pino(path), bs.Grid(M, 4.0), wl.basket_cfg1().params
    # 20 states are more than the clusters of 16 that fit: they run on clusters of 8
    ins = [start_state(M, 4.0, p, "random", seed=k) for k in range(20)]
    taus = [0.05 * k for k in range(20)]
    outs = [torch.empty((M, M), device="cuda") for _ in ins]
    bs.coarse_propagate_batched(g, bs.COARSE_PINO, net, [p] * 20, [to_gpu(u) for u in ins], outs, taus, 1.0 / 64)
    for k in (0, 19):
        one = torch.empty((M, M), device="cuda")
        bs.coarse_propagate(g, bs.COARSE_PINO, net, p, to_gpu(ins[k]), one, taus[k], 1.0 / 64, 1)
        torch.cuda.synchronize()
        assert torch.equal(one, outs[k])
        want, size = (v.cpu().numpy() for v in rounded_network(ins[k], 4.0, taus[k], 1.0 / 64, p, w))
        MP = want.shape[0]
        if M != MP:
            pos = np.arange(M) * ((MP - 1) / (M - 1))
            i0 = np.minimum(np.floor(pos).astype(int), MP - 2)
            f = pos - i0
            rows = want[i0] * (1 - f)[:, None] + want[i0 + 1] * f[:, None]
            want = rows[:, i0] * (1 - f) + rows[:, i0 + 1] * f
        # FP32 sums in another order round a few BF16 values the other way, each by 2^-8 of itself
        tol = 2.0 ** -8 * np.max(size)
        d = (to_np(one) - ins[k])[:-1, :-1] - want[:-1, :-1]
        print(layers, hidden, M, k, "max deviation / tolerance", np.max(np.abs(d)) / tol)
        assert np.max(np.abs(d)) <= tol
