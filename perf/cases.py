"""What is timed: the work that a program built on this library has it do, through its
public classes and calls, each case with its inputs, one pass, the work that pass cannot do
without, and the same result in 64 bits from plain torch.

The kinds of cases (the key "kind"):
  lattice    one periodic D2Q9 lattice: a number of steps, with S(k) where the run samples it
  lattice3   one periodic D3Q19 lattice, with S(k) on its axes or on every wave vector
  ensemble   replicas advanced together, with the radial S(k) of each one read at the end
  train      one training iteration of the surrogate (forward, loss, backward, Adam)
  rollout    strides of the surrogate from one frame
  conv       one convolution layer: forward, input gradient, weight and bias gradients
"""
import ctypes as C
import math

import numpy as np
import torch

from paper_2212_07848_gb300 import abi
from paper_2212_07848_gb300 import surrogate as S
from paper_2212_07848_gb300.ensemble import Ensemble
from paper_2212_07848_gb300.lattice import Lattice
from paper_2212_07848_gb300.lattice3 import Lattice3

LN2 = math.log(2.0)
DEV = "cuda" if torch.cuda.is_available() else "cpu"
NET = [(16, 32), (32, 64), (64, 128), (128, 64), (64, 16)]   # (cin, cout) of the surrogate


# ---- the cases ---------------------------------------------------------------------------
def _lattice(nx, ny, steps, **kw):
    c = dict(kind="lattice", nx=nx, ny=ny, steps=steps, precision="fp32", G=-3.6, tau=1.0,
             tau_bulk=0.0, tau_ghost=0.0, kT=1e-5, rho0=LN2, psi_kind=0, psi_p1=0.0, psi_p2=0.0,
             stencil=4, sk="none", field="uniform")
    c.update(kw)
    return c


def _lattice3(nx, ny, nz, steps, **kw):
    c = dict(kind="lattice3", nx=nx, ny=ny, nz=nz, steps=steps, precision="fp32", G=-3.6, tau=1.0,
             kT=1e-6, rho0=LN2, psi_kind=0, psi_p1=0.0, psi_p2=0.0, sk="axes", init_amp=1e-3)
    c.update(kw)
    return c


def listed():
    return [
        # A small box driven a few steps at a time by a program that looks at the state in
        # between: every step is one small launch.
        dict(_lattice(64, 64, 20), name="small_64_steps20"),
        # The supercritical FP64 run: 128^2 with S(k) sampled after every step.
        dict(_lattice(128, 128, 64, precision="fp64", sk="every_step"), name="fp64_128_sk"),
        # The metastable density sweep towards the spinodal: 1024^2, S(k) every 100 steps.
        dict(_lattice(1024, 1024, 100, G=-4.5, kT=1e-6, rho0=0.33, sk="at_end"),
             name="sweep_1024"),
        # The unstable-branch quench: 4096^2 with domains formed, S(k, t) and L(t) between runs
        # of steps.
        dict(_lattice(4096, 4096, 100, G=-5.0, kT=1e-6, sk="quench", field="domains"),
             name="quench_4096"),
        # A box of no special size with the widest stencil, the pseudopotential of Eq. (5) and
        # separate relaxation times: every option that is not the default.
        dict(_lattice(708, 452, 50, G=-3.0, tau=0.8, tau_bulk=1.3, tau_ghost=1.1, rho0=0.9,
                      psi_kind=1, psi_p1=5.0 / 12.0, psi_p2=1.0, stencil=8), name="ragged_e8_mrt"),
        # The batched ensemble: 256 replicas of 64^2 to 512^2, one persistent launch a window.
        dict(kind="ensemble", nrep=256, sizes="64,128,256,512", steps=100, sk_every=50,
             launch="persistent", name="ensemble_mix256"),
        # Many small replicas (the statistics near the critical point).
        dict(kind="ensemble", nrep=1024, sizes="64", steps=600, sk_every=50, launch="persistent",
             name="ensemble_1024x64"),
        # The 3D lattice at the size that fills the card's memory system, axis S(k).
        dict(_lattice3(256, 256, 256, 50, G=-5.0), name="d3q19_256"),
        # 3D domain growth: Eq. (5) on the T = 0.8 isotherm, the full S(k) and L(t).
        dict(_lattice3(128, 128, 128, 100, G=-3.0, rho0=0.75, psi_kind=1, psi_p1=5.0 / 12.0,
                       psi_p2=1.0, sk="full"), name="growth3_128"),
        # One training iteration of the surrogate at its training size.
        dict(kind="train", n=512, batch=8, name="train_512x8"),
        # The trained operator in use: twenty strides from one frame.
        dict(kind="rollout", n=512, strides=20, name="rollout_512x20"),
        # One layer of it by itself, all three directions.
        dict(kind="conv", nb=8, h=128, w=128, cin=64, cout=128, name="conv_64to128"),
    ]


def _log(rng, lo, hi, mult=1):
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(mult, int(round(v / mult)) * mult)


def draw(rng):
    kind = rng.choice(["lattice", "lattice", "lattice", "lattice3", "lattice3", "ensemble",
                       "train", "rollout", "conv"])
    if kind == "lattice":
        fp64 = rng.random() < 0.25
        nx, ny = _log(rng, 32, 2048 if fp64 else 4096, 4), _log(rng, 32, 2048 if fp64 else 4096, 4)
        sk = "none"
        if rng.random() < 0.5:          # S(k) needs powers of two
            nx, ny = (1 << round(math.log2(v)) for v in (nx, ny))
            sk = rng.choice(["every_step", "at_end", "quench"])
        stencil = rng.choice([4, 4, 6, 8])
        tau = rng.choice([1.0, 1.0, round(rng.uniform(0.6, 1.5), 3)])
        mrt = tau != 1.0 and rng.random() < 0.5
        kw = dict(G=round(rng.uniform(-5.2, -3.6), 3), rho0=round(rng.uniform(0.3, 1.1), 3))
        if rng.random() < 0.3:
            kw = dict(G=-3.0, rho0=round(rng.uniform(0.75, 1.6), 3), psi_kind=1,
                      psi_p1=5.0 / 12.0, psi_p2=1.0)
        most = 4.0e7 if fp64 else 1.2e9   # site updates
        steps = max(2, min(200 if sk != "every_step" else 40, int(most / (nx * ny))))
        return _lattice(nx, ny, rng.randint(max(2, steps // 2), steps),
                        precision="fp64" if fp64 else "fp32", tau=tau, stencil=stencil,
                        tau_bulk=round(rng.uniform(0.7, 1.4), 3) if mrt else 0.0,
                        tau_ghost=round(rng.uniform(0.7, 1.4), 3) if mrt else 0.0,
                        kT=rng.choice([1e-6, 1e-5]), sk=sk,
                        field=rng.choice(["uniform", "domains"]) if "psi_kind" not in kw
                        else "uniform", **kw)
    if kind == "lattice3":
        fp64 = rng.random() < 0.2
        top = 96 if fp64 else 224
        nx = _log(rng, 32, top, 32)
        ny, nz = _log(rng, 16, top, 4), _log(rng, 8, top)
        sk = "axes"
        if rng.random() < 0.4:
            nx, ny, nz = (1 << round(math.log2(v)) for v in (nx, ny, nz))
            sk = "full"
        steps = max(4, min(100, int((2.0e7 if fp64 else 4.0e8) / (nx * ny * nz))))
        kw = dict(G=round(rng.uniform(-5.0, -3.6), 3))
        if rng.random() < 0.5:
            kw = dict(G=-3.0, rho0=round(rng.uniform(0.65, 1.6), 3), psi_kind=1,
                      psi_p1=5.0 / 12.0, psi_p2=1.0)
        return _lattice3(nx, ny, nz, rng.randint(max(2, steps // 2), steps), sk=sk,
                         precision="fp64" if fp64 else "fp32",
                         tau=rng.choice([1.0, round(rng.uniform(0.6, 1.5), 3)]), **kw)
    if kind == "ensemble":
        sizes = rng.choice(["64,128,256,512", "64", "32", "128", "32,64,128", "256"])
        mean = sum(int(s) ** 2 for s in sizes.split(",")) / len(sizes.split(","))
        nrep = max(2, min(1024, _log(rng, 1.0e5 / mean + 2, 2.0e7 / mean)))
        steps = max(20, min(400, int(1.5e9 / (nrep * mean))))
        return dict(kind="ensemble", nrep=nrep, sizes=sizes, steps=steps,
                    sk_every=rng.choice([10, 25, 50]),
                    launch=rng.choice(["persistent", "per_step"]))
    if kind == "train":
        return dict(kind="train", n=rng.choice([64, 128, 192, 256, 384, 512]),
                    batch=rng.randint(2, 8))
    if kind == "rollout":
        return dict(kind="rollout", n=rng.choice([64, 128, 256, 384, 512]),
                    strides=rng.randint(4, 20))
    while True:
        h, w = _log(rng, 16, 512, 8), rng.choice([16, 32, 48, 64, 96, 128, 256, 384, 512])
        nb = rng.randint(1, 8)
        ci, co = rng.choice(NET + [(32, 32), (64, 64), (128, 128), (48, 80)])
        if h * w % 128 == 0 and nb * h * w * ci * co < 8 * 512 * 512 * 64 * 16 * 1.01:
            return dict(kind="conv", nb=nb, h=h, w=w, cin=ci, cout=co)


# ---- inputs ------------------------------------------------------------------------------
def _gen(seed, dev=None):
    return torch.Generator(device=dev or DEV).manual_seed(int(seed))


def _domains(ny, nx, seed, lo=0.12, hi=1.9, nb=1):
    """Densities of a coarsening quench: domains of gas and liquid (the coexisting densities
    at G = -5) about 24 sites across with smooth interfaces, from filtered white noise."""
    z = torch.randn((nb, ny, nx), generator=_gen(seed), device=DEV)
    k2 = (torch.fft.fftfreq(ny, device=DEV)[:, None] ** 2 +
          torch.fft.rfftfreq(nx, device=DEV)[None, :] ** 2)
    f = torch.fft.irfft2(torch.fft.rfft2(z) * torch.exp(-0.5 * k2 * (2 * math.pi * 6.0) ** 2),
                         s=(ny, nx))
    f = f / f.std(dim=(1, 2), keepdim=True)
    return (0.5 * (lo + hi) + 0.5 * (hi - lo) * torch.tanh(1.5 * f)).float()


def _replicas(case, seed):
    rng = np.random.default_rng(seed)
    sizes = [int(s) for s in case["sizes"].split(",")]
    out = []
    for k in rng.permutation(case["nrep"]):     # every size as often, in any order
        n = sizes[k % len(sizes)]
        out.append((n, n, float(rng.uniform(-4.8, -3.6)), 1.0, 1e-6,
                    float(LN2 * rng.uniform(0.9, 1.1))))
    return out


def _weights(seed):
    """Parameters of a network in training: He-scaled kernels, a small output layer."""
    g = _gen(seed)
    w, b = [], []
    for ci, co in NET:
        a = math.sqrt(2.0 / (9 * ci)) * torch.randn((9, co, ci), generator=g, device=DEV)
        w.append(a * 0.01 if co == 16 else a)
        b.append(0.01 * torch.randn(co, generator=g, device=DEV))
    return w, b


LR, ADAM_V, ADAM_STEP = 1e-4, 1e-6, 1000   # a late iteration: second moments are settled


def _net(n, batch, seed):
    net = S.SurrogateNet(n, batch)
    for i, (w, b) in enumerate(zip(*_weights(seed))):
        net.w[i].copy_(w)
        net.b[i].copy_(b)
        net.wb[i].copy_(w.to(torch.bfloat16))
        net.vw[i].fill_(ADAM_V)
        net.vb[i].fill_(ADAM_V)
    net.step_count = ADAM_STEP
    return net


def _frames(n, nb, seed):
    """(the frame before, this frame, the next one) as coarse density deviations, and G."""
    f = _domains(n, n, seed, 0.2 - LN2, 1.8 - LN2, nb)
    d = 0.02 * _domains(n, n, seed + 7919, -1.0, 1.0, 2 * nb)
    G = np.random.default_rng(seed).uniform(-5.2, -4.4, nb)
    return f - d[:nb], f, f + d[nb:], G


def _conv_inputs(case, seed):
    g = _gen(seed)
    nb, h, w, ci, co = (case[k] for k in ("nb", "h", "w", "cin", "cout"))
    bf = torch.bfloat16
    x = torch.randn((nb, h, w, ci), generator=g, device=DEV).relu().to(bf)
    dy = (0.01 * torch.randn((nb, h, w, co), generator=g, device=DEV)).to(bf)
    k = (math.sqrt(2.0 / (9 * ci)) * torch.randn((9, co, ci), generator=g, device=DEV)).to(bf)
    b = 0.1 * torch.randn(co, generator=g, device=DEV)
    return x, dy, k, b


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "lattice":
        lat = Lattice(case["nx"], case["ny"], case["G"], case["tau"], case["kT"],
                      psi_kind=case["psi_kind"], stencil=case["stencil"],
                      precision=case["precision"], psi_p1=case["psi_p1"], psi_p2=case["psi_p2"],
                      tau_bulk=case["tau_bulk"], tau_ghost=case["tau_ghost"])
        lat.init(case["rho0"], seed, 1e-3 if case["field"] == "uniform" else 0.0)
        if case["field"] == "domains":
            lat.sync()
            df = lat.torch_populations()
            d = _domains(case["ny"], case["nx"], seed)[0].double() - case["rho0"]
            for i, w in enumerate(W2):
                df[i].copy_(w * d)
        if case["sk"] != "none":
            every = {"every_step": 1, "at_end": case["steps"], "quench": 0}[case["sk"]]
            lat.sk_config(every, every)
        st["lat"] = lat
    elif kind == "lattice3":
        lat = Lattice3(case["nx"], case["ny"], case["nz"], case["G"], case["tau"], case["kT"],
                       precision=case["precision"], psi_kind=case["psi_kind"],
                       psi_p1=case["psi_p1"], psi_p2=case["psi_p2"])
        lat.init(case["rho0"], seed, case["init_amp"])
        lat.sk_config(case["steps"], case["steps"])
        if case["sk"] == "full":
            lat.sk_full()
        st["lat"] = lat
    elif kind == "ensemble":
        e = Ensemble(_replicas(case, seed), seed=seed)
        if case["launch"] == "persistent":
            e.set_launch(abi.LB_ENS_PERSISTENT)
        e.init(1e-3)
        e.sk_config(case["sk_every"], case["sk_every"])
        e.autotune(10)
        st["ens"] = e
    elif kind == "train":
        n, nb = case["n"], case["batch"]
        net = _net(n, nb, seed)
        before, now, after, G = _frames(n, nb, seed)
        x = torch.empty((nb, n, n, 16), dtype=torch.bfloat16, device=DEV)
        for j in range(nb):
            S.expand_state(net.L, now[j], G[j], x[j], before[j])
        st.update(net=net, x=x, base=now.contiguous(), target=after.contiguous())
    elif kind == "rollout":
        net = _net(case["n"], 1, seed)
        before, now, _, G = _frames(case["n"], 1, seed)
        st.update(net=net, frame=now[0].contiguous(), prev=before[0].contiguous(), G=float(G[0]))
    else:
        L = abi.load()
        x, dy, k, b = _conv_inputs(case, seed)
        ws = L.lb_nn_wgrad_workspace(case["nb"], case["h"], case["w"], case["cin"], case["cout"])
        st.update(L=L, x=x, dy=dy, k=k, b=b, y=torch.empty_like(dy), dx=torch.empty_like(x),
                  dw=torch.empty(k.shape, device=DEV), db=torch.empty_like(b), ws_bytes=ws,
                  ws=torch.empty(ws // 4 + 1, device=DEV))
    torch.cuda.synchronize()
    return st


# ---- one pass ----------------------------------------------------------------------------
def _as_stored(a, case):
    """S(k) read from a lattice, in the precision that the lattice stores its state in."""
    return np.asarray(a, np.float32 if case.get("precision", "fp32") == "fp32" else np.float64)


def _shells(case):
    return max(case["nx"], case["ny"]) // 2


def _shells3(case):
    return int(math.ceil(math.sqrt(3.0) * max(case["nx"], case["ny"], case["nz"]) / 2)) + 1


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "lattice":
        lat = st["lat"]
        lat.step(case["steps"])
        out = [lat.torch_populations()]
        out[0].lattice = lat    # the view does not own its memory: it keeps the lattice instead
        if case["sk"] == "quench":
            lat.sk_reset()
            lat.sk_sample_now()
        if case["sk"] != "none":
            out.append(_as_stored(lat.structure_factor(_shells(case))[0], case))
        if case["sk"] == "quench":
            out.append(_as_stored(lat.domain_size(), case))
        return out
    if kind == "lattice3":
        lat = st["lat"]
        lat.step(case["steps"])
        if case["sk"] == "axes":
            out = [_as_stored(lat.structure_factor_axes()[0], case)]
        else:
            out = [_as_stored(lat.structure_factor(_shells3(case))[0], case),
                   _as_stored(lat.domain_size(), case)]
        lat.sk_reset()
        return out
    if kind == "ensemble":
        e = st["ens"]
        e.step(case["steps"])
        return [_as_stored(np.concatenate([e.structure_factor(r, n[0] // 2)[0]
                                           for r, n in enumerate(e.reps)]), case)]
    if kind == "train":
        net = st["net"]
        net.zero_grad()
        net.forward(st["x"])
        loss = net.loss_and_grad(st["x"], st["target"], st["base"])
        net.backward(st["x"])
        net.adam(LR)
        return [loss, list(net.dw), list(net.db), list(net.w), list(net.b)]
    if kind == "rollout":
        return [S.rollout(st["net"], st["frame"], st["G"], case["strides"], st["prev"])]
    L, p = st["L"], lambda t: C.c_void_p(t.data_ptr())
    a = [case[k] for k in ("nb", "h", "w")]
    ci, co = case["cin"], case["cout"]
    st["dw"].zero_()
    st["db"].zero_()
    for rc in (L.lb_nn_conv3x3(p(st["x"]), p(st["k"]), p(st["b"]), p(st["y"]), *a, ci, co, 1, 0,
                               None),
               L.lb_nn_conv3x3(p(st["dy"]), p(st["k"]), None, p(st["dx"]), *a, co, ci, 0, 1, None),
               L.lb_nn_conv3x3_wgrad(p(st["x"]), p(st["dy"]), p(st["dw"]), p(st["db"]), *a, ci, co,
                                     p(st["ws"]), st["ws_bytes"], None)):
        if rc != 0:
            raise abi.LbError(rc, "conv")
    return [st["y"], st["dx"], st["dw"], st["db"]]


# ---- the work that a pass cannot do without ------------------------------------------------
def work(case):
    kind = case["kind"]
    if kind == "lattice":       # each population once in, once out a step; about 220 operations
        n, e = case["nx"] * case["ny"] * case["steps"], 8 if case["precision"] == "fp64" else 4
        return {"bytes": 18 * e * n, "flops": 220 * n}
    if kind == "lattice3":
        n = case["nx"] * case["ny"] * case["nz"] * case["steps"]
        return {"bytes": 38 * (8 if case["precision"] == "fp64" else 4) * n, "flops": 500 * n}
    if kind == "ensemble":
        sizes = [int(s) for s in case["sizes"].split(",")]
        n = case["nrep"] * sum(s * s for s in sizes) / len(sizes) * case["steps"]
        return {"bytes": 72 * n, "flops": 220 * n}
    if kind == "conv":          # x and dy in, y and dx out (16 bits each); three products
        px = case["nb"] * case["h"] * case["w"]
        ci, co = case["cin"], case["cout"]
        return {"bytes": 4 * px * (ci + co) + 9 * ci * co * 6, "flops": 3 * 18.0 * px * ci * co}
    n = case["n"]
    # pixels of each layer's output, by level
    lay = list(zip([1, 4, 16, 4, 1], NET))
    macs = sum(9 * n * n / d * ci * co for d, (ci, co) in lay)
    params = sum(9 * ci * co + co for ci, co in NET)
    if kind == "rollout":       # the weights and both frames in, every stride's frame out
        s = case["strides"]
        return {"bytes": 2 * params + 4 * n * n * (2 + s), "flops": 2 * macs * s}
    nb = case["batch"]          # input, target and base in; activations out and back for the
    acts = sum(n * n / d * co * 2 for d, (_, co) in lay) * nb   # gradients; parameters updated
    return {"bytes": nb * n * n * 40 + 2 * acts + 32 * params, "flops": 6 * macs * nb}


# ---- the same results in 64 bits, from plain torch -----------------------------------------
C2 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W2 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
      (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
      (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
W3 = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
STENCIL = {4: {1: 1 / 3, 2: 1 / 12}, 6: {1: 4 / 15, 2: 1 / 10, 4: 1 / 120},
           8: {1: 4 / 21, 2: 4 / 45, 4: 1 / 60, 5: 2 / 315, 8: 1 / 5040}}


def _noise_basis(dim):
    """The moments that carry noise, as polynomials of the velocities [modes][q]."""
    if dim == 2:
        x, y = np.array(C2, float).T
        c = x * x + y * y
        rows = [3 * c - 2, x * x - y * y, x * y, (3 * c - 4) * x, (3 * c - 4) * y,
                9 * c * c - 15 * c + 2]
    else:
        x, y, z = np.array(C3, float).T
        c = x * x + y * y + z * z
        rows = [c - 1, 3 * x * x - c, y * y - z * z, x * y, y * z, z * x, (3 * c - 5) * x,
                (3 * c - 5) * y, (3 * c - 5) * z, (y * y - z * z) * x, (z * z - x * x) * y,
                (x * x - y * y) * z, 3 * c * c - 6 * c + 1, (2 * c - 3) * (3 * x * x - c),
                (2 * c - 3) * (y * y - z * z)]
    return np.array(rows)


def _mulhilo(a, m):
    lo, hi = a * (m & 0xFFFF), a * (m >> 16)
    return (hi + (lo >> 16)) >> 16, (lo + ((hi & 0xFFFF) << 16)) & 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    z = torch.zeros_like(c0)
    c = [c0, z + c1, z + c2, z + c3]
    for _ in range(10):
        h0, l0 = _mulhilo(c[0], 0xD2511F53)
        h1, l1 = _mulhilo(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


class _Exact:
    """Lattices [q][R][(nz,) ny, nx] in 64 bits: streaming, pseudopotential force, relaxation
    with the Guo source and noise in moment space.  G, kT, rho0 and the noise's replica word
    are numbers or tensors [R, 1, ...]."""

    def __init__(self, dim, R, shape, G, kT, rho0, seed, replica=0, tau=1.0, tau_bulk=0.0,
                 tau_ghost=0.0, psi=(0, 0.0, 0.0), stencil=4):
        self.dim, self.shape, self.seed, self.t = dim, shape, int(seed), 0
        self.G, self.kT, self.rho0, self.replica, self.psi_kind = G, kT, rho0, replica, psi
        self.c, self.w = (C2, W2) if dim == 2 else (C3, W3)
        self.site = torch.arange(math.prod(shape), device=DEV).view(1, *shape).expand(
            R, *shape).contiguous()
        E = _noise_basis(dim)
        b = (E * E * np.array(self.w)).sum(1)
        tb, tg = tau_bulk or tau, tau_ghost or tau
        lam = [1 / tb, 1 / tau, 1 / tau] + [1 / tg] * 3 if dim == 2 else [1 / tau] * 15
        self.lam, self.one_rate = lam, len(set(lam)) == 1
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=DEV)
        self.E, self.back = t(E), t((E / b[:, None] * np.array(self.w)).T)   # [k][q], [q][k]
        self.amp = [math.sqrt(3.0 * bk * (1.0 - (1.0 - a) ** 2)) for bk, a in zip(b, lam)]
        self.lam_t = t(lam)
        if dim == 3:
            st = {1: 1 / 6, 2: 1 / 12}
            self.half = [(e, st[sum(v * v for v in e)]) for e in C3 if e > (0, 0, 0)]
        else:
            r = 1 if stencil == 4 else 2
            self.half = [((x, y), STENCIL[stencil][x * x + y * y]) for x in range(-r, r + 1)
                         for y in range(-r, r + 1)
                         if (x, y) > (0, 0) and x * x + y * y in STENCIL[stencil]]
        self.f = None

    def roll(self, a, e):
        """a(x + e) (the array's axes run z, y, x)."""
        return torch.roll(a, [-v for v in e], [-1 - i for i in range(self.dim)])

    def uniform(self, r, word=32):
        return (r.double() + 0.5) * 2.0 ** -word

    def kick(self, amp):
        d = 0.0
        if amp:
            r = _philox(self.site, 0, self.replica, 2 if self.dim == 2 else 3, self.seed)
            d = amp * torch.sqrt(-2.0 * torch.log(self.uniform(r[0]))) * torch.cos(
                2 * math.pi * self.uniform(r[1]))
        self.f = torch.stack([w * (self.rho0 + d) + 0.0 * self.site for w in self.w])

    def normals(self):
        pairs = []
        if self.dim == 2:
            r = _philox(self.site, self.t, self.replica, 0, self.seed)
            for k in range(3):
                pairs.append((self.uniform(r[k]), (r[3] >> (10 * k)) & 1023))
        else:
            for blk in (0, 1):
                for r in _philox(self.site, self.t, self.replica, blk, self.seed):
                    pairs.append((self.uniform(r >> 10, 22), r & 1023))
        z = []
        for u, a in pairs:
            rad, th = torch.sqrt(-2.0 * torch.log(u)), (a.double() + 0.5) * (2 * math.pi / 1024)
            z += [rad * torch.cos(th), rad * torch.sin(th)]
        return z[:len(self.amp)]

    def psi(self, rho):
        kind, p1, p2 = self.psi_kind
        if kind == 0:
            return -torch.expm1(-rho)
        return math.sqrt(p1 * p2) * torch.exp(1.0 - p2 / rho) if kind == 1 else (
            p1 * torch.exp(-p2 / rho))

    def step(self, n=1):
        for _ in range(n):
            g = torch.stack([self.roll(self.f[i], [-v for v in c]) for i, c in enumerate(self.c)])
            rho = g.sum(0)
            psi = self.psi(rho)
            F = [torch.zeros_like(rho) for _ in range(self.dim)]
            for e, w in self.half:
                d = w * (self.roll(psi, e) - self.roll(psi, [-v for v in e]))
                for a in range(self.dim):
                    if e[a]:
                        F[a] += e[a] * d
            F = [-self.G / 3.0 * psi * v for v in F]
            u = [(sum(c[a] * g[i] for i, c in enumerate(self.c) if c[a]) + 0.5 * F[a]) / rho
                 for a in range(self.dim)]
            uu, uF = sum(v * v for v in u), sum(v * w for v, w in zip(u, F))
            feq, src = torch.empty_like(g), torch.empty_like(g)
            for i, c in enumerate(self.c):
                cu = sum(c[a] * u[a] for a in range(self.dim))
                cF = sum(c[a] * F[a] for a in range(self.dim))
                feq[i] = self.w[i] * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * uu)
                src[i] = self.w[i] * (3.0 * (cF - uF) + 9.0 * cu * cF)
            g -= feq
            if self.one_rate:
                lam = self.lam[0]
                self.f = feq + (1.0 - lam) * g + (1.0 - 0.5 * lam) * src
            else:   # every mode at its own rate; feq + g + src carries j + F whatever the rates
                m = (self.E @ (g + 0.5 * src).flatten(1)) * -self.lam_t[:, None]
                self.f = feq + g + src + (self.back @ m).view_as(g)
            if not isinstance(self.kT, float) or self.kT > 0.0:
                root = torch.sqrt(self.kT * rho)
                z = torch.stack([a * v * root for a, v in zip(self.amp, self.normals())])
                self.f += (self.back @ z.flatten(1)).view_as(g)
            self.t += 1

    def rho(self):
        return self.f.sum(0)

    def power(self):
        """|delta rho(k)|^2 / N on the full plane or box, k = 0 at zero."""
        ax = list(range(-self.dim, 0))
        r = self.rho()
        p = torch.fft.fftn(r - r.mean(dim=ax, keepdim=True), dim=ax).abs() ** 2
        p[(slice(None),) + (0,) * self.dim] = 0.0
        return p / math.prod(self.shape)


def _folded(n):
    return torch.fft.fftfreq(n, device=DEV, dtype=torch.float64) * n


def _radii(shape):
    """|k| in units of 2 pi / (the longest side), on the full plane or box."""
    q2 = 0.0
    for i, n in enumerate(shape):
        v = _folded(n) * (max(shape) / n)
        q2 = q2 + (v * v).view([-1 if j == i else 1 for j in range(len(shape))])
    return torch.sqrt(q2)


def _radial(P, shape, nbins, empty):
    """Means over the shells round(|k|) of [R] powers, without k = 0."""
    q = _radii(shape)
    b = torch.round(q).long()
    b[(0,) * len(shape)] = 1 << 20
    keep = b < nbins
    cnt = torch.bincount(b[keep], minlength=nbins).double()
    rows = [torch.bincount(b[keep], weights=p[keep], minlength=nbins) for p in P]
    return torch.stack([torch.where(cnt > 0, r / cnt.clamp(min=1), torch.full_like(r, empty))
                        for r in rows])


def _size(P, shape):
    """L = 2 pi sum S / sum |k| S."""
    return float(2 * math.pi * P.sum() / (P * _radii(shape) * (2 * math.pi / max(shape))).sum())


def _exact_lattice(case, seed):
    shape = (case["ny"], case["nx"])
    ex = _Exact(2, 1, shape, case["G"], case["kT"], case["rho0"], seed, tau=case["tau"],
                tau_bulk=case["tau_bulk"], tau_ghost=case["tau_ghost"],
                psi=(case["psi_kind"], case["psi_p1"], case["psi_p2"]), stencil=case["stencil"])
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    ex.kick(1e-3 if case["field"] == "uniform" else 0.0)
    if case["field"] == "domains":
        d = _domains(case["ny"], case["nx"], seed)[0].double() - case["rho0"]
        ex.f = torch.stack([w * case["rho0"] + (w * d).to(dt).double() for w in W2])[:, None]
    P, n = 0.0, 0
    for t in range(1, case["steps"] + 1):
        ex.step()
        if case["sk"] == "every_step" or (case["sk"] != "none" and t == case["steps"]):
            P, n = P + ex.power(), n + 1
    w = torch.tensor(W2, dtype=torch.float64, device=DEV).view(9, 1, 1)
    out = [ex.f[:, 0] - w * case["rho0"]]
    if n:
        out.append(_radial(P / n, shape, _shells(case), float("nan"))[0].cpu().numpy())
    if case["sk"] == "quench":
        out.append(np.asarray(_size(P[0], shape)))
    return out


def _exact_lattice3(case, seed):
    shape = (case["nz"], case["ny"], case["nx"])
    ex = _Exact(3, 1, shape, case["G"], case["kT"], case["rho0"], seed, tau=case["tau"],
                psi=(case["psi_kind"], case["psi_p1"], case["psi_p2"]))
    ex.kick(case["init_amp"])
    ex.step(case["steps"])
    P = ex.power()[0]
    if case["sk"] == "full":
        return [_radial([P], shape, _shells3(case), 0.0)[0].cpu().numpy(),
                np.asarray(_size(P, shape))]
    return [torch.cat([P[0, 0, 1:case["nx"] // 2 + 1], P[0, 1:case["ny"] // 2 + 1, 0],
                       P[1:case["nz"] // 2 + 1, 0, 0]]).cpu().numpy()]


def _exact_ensemble(case, seed):
    reps = _replicas(case, seed)
    rows = [None] * len(reps)
    for n in sorted({r[0] for r in reps}):
        ids = [i for i, r in enumerate(reps) if r[0] == n]
        t = lambda v, d=torch.float64: torch.tensor(v, dtype=d, device=DEV).view(-1, 1, 1)
        ex = _Exact(2, len(ids), (n, n), t([reps[i][2] for i in ids]),
                    t([reps[i][4] for i in ids]), t([reps[i][5] for i in ids]), seed,
                    replica=t(ids, torch.int64))
        ex.kick(1e-3)
        P, k = 0.0, 0
        for _ in range(case["steps"] // case["sk_every"]):
            ex.step(case["sk_every"])
            P, k = P + ex.power(), k + 1
        for i, row in zip(ids, _radial(P / k, (n, n), n // 2, float("nan"))):
            rows[i] = row
    return [torch.cat(rows).cpu().numpy()]


def _conv(x, w, b=None):
    """3x3 periodic convolution of [nb][c][h][w] with taps [9][co][ci], in 64 bits."""
    k = w.view(3, 3, w.shape[1], w.shape[2]).permute(2, 3, 0, 1)
    return torch.nn.functional.conv2d(torch.nn.functional.pad(x, (1, 1, 1, 1), "circular"), k, b)


def _exact_net(x, w, b):
    """The network's output [nb][16][n][n] from input [nb][16][n][n]."""
    F = torch.nn.functional
    up = lambda v: F.interpolate(v, scale_factor=2, mode="nearest")
    a1 = F.relu(_conv(x, w[0], b[0]))
    a2 = F.relu(_conv(F.avg_pool2d(a1, 2), w[1], b[1]))
    a3 = F.relu(_conv(F.avg_pool2d(a2, 2), w[2], b[2]))
    a4 = F.relu(_conv(up(a3), w[3], b[3]))
    return _conv(up(a4 + a2), w[4], b[4])


def _exact_input(now, before, G):
    x = torch.zeros((len(G), 16) + tuple(now.shape[1:]), dtype=torch.float64, device=DEV)
    x[:, 0] = now.double()
    x[:, 1] = torch.tensor((np.asarray(G) + 4.8) / 0.4, device=DEV).view(-1, 1, 1)
    x[:, 2] = now.double() - before.double()
    return x


def _exact_train(case, seed):
    w, b = _weights(seed)
    wd = [a.to(torch.bfloat16).double().requires_grad_() for a in w]
    bd = [a.double().requires_grad_() for a in b]
    before, now, after, G = _frames(case["n"], case["batch"], seed)
    x = _exact_input(now, before, G).to(torch.bfloat16).double()
    y = _exact_net(x, wd, bd)[:, 0]
    loss = ((now.double() + y - after.double()) ** 2).mean()
    loss.backward()
    step = ADAM_STEP + 1

    def adam(p, g):
        m, v = 0.1 * g / (1 - 0.9 ** step), (0.999 * ADAM_V + 0.001 * g * g) / (1 - 0.999 ** step)
        return p.double() - LR * m / (torch.sqrt(v) + 1e-8)

    return [loss.detach().view(1), [a.grad for a in wd], [a.grad for a in bd],
            [adam(p, a.grad) for p, a in zip(w, wd)], [adam(p, a.grad) for p, a in zip(b, bd)]]


def _exact_rollout(case, seed):
    w, b = _weights(seed)
    wd = [a.to(torch.bfloat16).double() for a in w]
    bd = [a.double() for a in b]
    before, now, _, G = _frames(case["n"], 1, seed)
    prev, state, out = before.double(), now.double(), []
    for _ in range(case["strides"]):
        y = _exact_net(_exact_input(state, prev, G), wd, bd)[:, 0]
        prev, state = state, state + y - y.mean()
        out.append(state[0])
    return [torch.stack(out)]


def _exact_conv(case, seed):
    x, dy, k, b = _conv_inputs(case, seed)
    xd = x.double().permute(0, 3, 1, 2).requires_grad_()
    kd, bd = k.double().requires_grad_(), b.double().requires_grad_()
    z = _conv(xd, kd, bd)
    z.backward(dy.double().permute(0, 3, 1, 2))
    nhwc = lambda v: v.permute(0, 2, 3, 1).contiguous()
    return [nhwc(torch.relu(z.detach())), nhwc(xd.grad), kd.grad, bd.grad]


def exact(case, seed):
    return {"lattice": _exact_lattice, "lattice3": _exact_lattice3, "ensemble": _exact_ensemble,
            "train": _exact_train, "rollout": _exact_rollout, "conv": _exact_conv}[case["kind"]](
                case, seed)
