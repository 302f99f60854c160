"""What the performance of this framework is measured on: simulations as a
user's program runs them, through the package's public calls.

A case is a dict of plain values with a "kind":

  net      a whole network: ``steps`` steps, then the rates, the event totals
           and the neuron state are read.
  loop     a closed loop: one step, then that step's spikes are read.
  batch    a sweep of small networks advanced together, then every member read.
  grad     loss and gradient of the differentiable form as a torch function of
           a float32 parameter vector.
  noalloc  one neuron update on torch-owned state buffers.
  shards   a grid split into two column-tile shards stepped on one GPU, spike
           lists exchanged on the host every step.

Networks are the package's workloads (1240 neurons a column unless ``npc``
says otherwise), built from the seed and stepped past the initial synchronous
volley by ``prepare``; every pass goes on from where the last one ended.
"""
import math

import numpy as np
import torch

from paper_1511_09325_gb300 import snn
from paper_1511_09325_gb300 import workloads as W

THETA = (1.0, 1.0, 1.0, 1.0, 0.02, 2.5)  # a_EE, a_EI, a_IE, a_II, g_c, nu_ext


def listed():
    return [
        # the smallest call: a controller around the 2x2 network that reads
        # each millisecond's spikes before it takes the next
        dict(name="loop_2x2_f32w", kind="loop", gw=2, gh=2, precision="f32w", settle=600),
        # the 2x2 parity workload, one model second
        dict(name="net_2x2_f32w", kind="net", gw=2, gh=2, precision="f32w", steps=1000, settle=600),
        # a ragged network: odd column size and sides, 5x5 stencil, short
        # delays from 2 ms
        dict(name="net_13x7_ragged_f16w", kind="net", gw=13, gh=7, precision="f16w", steps=1000,
             settle=600, npc=1001, k_out=997, radius=2, d_min=2, d_max=9),
        # the paper's 24x24 problem size, one model second
        dict(name="net_24x24_f32w", kind="net", gw=24, gh=24, precision="f32w", steps=1000,
             settle=600),
        # the same size under the paper's own connectivity law
        dict(name="paper_24x24_f32w", kind="net", gw=24, gh=24, precision="f32w", steps=1000,
             settle=600, law=1),
        # the paper's 48x48 problem size
        dict(name="net_48x48_f32w", kind="net", gw=48, gh=48, precision="f32w", steps=1000,
             settle=600),
        # the paper's largest problem size, as this package recommends it (FP16 weights)
        dict(name="net_96x96_f16w", kind="net", gw=96, gh=96, precision="f16w", steps=1000,
             settle=600),
        # a seed and drive sweep over 64 networks of 1x1 to 8x8 columns
        dict(name="batch_64_f32w", kind="batch", nets=64, precision="f32w", steps=500),
        # gradient training of the 4x4 network, half a model second, hard spikes
        dict(name="grad_4x4_hard", kind="grad", gw=4, gh=4, T=500, every=50, hard=True),
        # a short relaxed run of the 2x2 network (exact gradient)
        dict(name="grad_2x2_soft", kind="grad", gw=2, gh=2, T=6, every=50, hard=False),
        # another framework's arena: one neuron update at the 24x24 size
        dict(name="noalloc_24x24", kind="noalloc", gw=24, gh=24),
        # two shards of the 24x24 network, spikes exchanged every step
        dict(name="shards_24x24_f16w", kind="shards", gw=24, gh=24, precision="f16w", steps=50,
             settle=100),
    ]


def _side(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["net"] * 5 + ["loop", "batch", "grad", "noalloc", "shards"])
    prec = rng.choice(["f32w", "f16w"])
    if kind == "net":
        c = dict(kind=kind, gw=_side(rng, 1, 60), gh=_side(rng, 1, 60), precision=prec,
                 steps=rng.randint(200, 1000), settle=rng.randint(300, 700))
        form = rng.choice(["fixed", "fixed", "paper", "ragged"])
        if form == "paper":
            c["law"] = 1
        if form == "ragged":
            d0 = rng.randint(1, 4)
            c.update(npc=rng.randint(200, 2048), k_out=rng.randint(300, 1500),
                     radius=rng.randint(1, 3), d_min=d0, d_max=rng.randint(d0 + 2, 32))
        return c
    if kind == "loop":
        return dict(kind=kind, gw=_side(rng, 1, 24), gh=_side(rng, 1, 24), precision=prec,
                    settle=rng.randint(300, 700))
    if kind == "batch":
        return dict(kind=kind, nets=_side(rng, 4, 64), precision=prec, steps=rng.randint(100, 500))
    if kind == "grad":
        return dict(kind=kind, gw=rng.randint(1, 5), gh=rng.randint(1, 5), T=rng.randint(60, 500),
                    every=rng.randint(10, 80), hard=True)
    if kind == "noalloc":
        return dict(kind=kind, gw=_side(rng, 1, 100), gh=_side(rng, 1, 100),
                    npc=rng.choice([1240, 1240, 1001, 512]))
    return dict(kind=kind, gw=rng.randint(2, 30), gh=rng.randint(1, 30), precision=prec,
                steps=rng.randint(10, 50), settle=rng.randint(50, 150))


def _params(case):
    npc = case.get("npc", 1240)
    n = W.neuron_params(n_per_col=npc, n_exc=npc * 4 // 5)
    s = W.synapse_params(k_out=case.get("k_out", 1240), stencil_radius=case.get("radius", 3),
                         d_min=case.get("d_min", 1), d_max=case.get("d_max", 20),
                         connectivity=case.get("law", 0))
    return n, s


def prepare(case, seed):
    n, s = _params(case)
    kind = case["kind"]
    st = dict(case)
    if kind in ("net", "loop"):
        st["net"] = snn.Net(case["gw"], case["gh"], n, s, seed + 1, case["precision"])
        st["net"].step(case["settle"])
        if kind == "loop":
            st["net"].spikes()
            st["t"], st["ids"] = (np.zeros(st["net"].n, np.int32) for _ in range(2))
    elif kind == "batch":
        grids, neurons, synapses, seeds = W.batch_workload(case["nets"], seed0=100 + 1000 * (seed % 1000003))
        st["batch"] = snn.Batch(grids, neurons, synapses, seeds, case["precision"])
        st["batch"].tune(20)
    elif kind == "grad":
        st["stream"] = torch.cuda.Stream()  # the training program's stream
        st["net"] = snn.Net(case["gw"], case["gh"], n, s, seed + 1, "f32w",
                            st["stream"].cuda_stream)
        st["view"] = snn.Grad(st["net"], case["T"], checkpoint_every=case["every"], hard=case["hard"])
    elif kind == "noalloc":
        st.update(_noalloc_buffers(case, seed), neuron=n, seed=seed, step=0)
    else:
        tiles = snn.split_grid(case["gw"], case["gh"], 2, 1)
        st["shards"] = [snn.Shard(case["gw"], case["gh"], t, n, s, seed + 1, case["precision"])
                        for t in tiles]
        st["n"] = case["gw"] * case["gh"] * n["n_per_col"]
        for _ in range(case["settle"]):
            _shard_step(st["shards"])
    return st


def _noalloc_buffers(case, seed):
    """State of a running network: potentials up to threshold, calcium of a
    few spikes, about 2 % of the neurons refractory, synaptic input of a few
    mV for some neurons."""
    n_cols, npc = case["gw"] * case["gh"], case.get("npc", 1240)
    N = n_cols * npc
    P = (N + 3) // 4 * 4
    g = torch.Generator(device="cuda").manual_seed(seed)
    dev = dict(device="cuda", generator=g)
    v = torch.rand(P, **dev) * 20.0
    c = torch.rand(P, **dev) * 6.0
    r = (torch.rand(P, **dev) < 0.02).to(torch.uint8) * 2
    drive = (torch.randn(P, **dev) * 1.5 * 65536.0).to(torch.int32)
    return dict(N=N, v=v, c=c, r=r, drive=drive, input=torch.zeros_like(drive),
                spikes=torch.zeros(N, dtype=torch.int32, device="cuda"),
                fired=torch.zeros(N, dtype=torch.uint8, device="cuda"),
                counts=torch.zeros(2 * n_cols, dtype=torch.int64, device="cuda"))


def _shard_step(shards):
    for sh in shards:
        sh.update()
    ids = np.concatenate([sh.spikes()[1] for sh in shards])
    for sh in shards:
        sh.deliver(ids)
    return ids


def run(state):
    kind = state["kind"]
    if kind == "net":
        net = state["net"]
        net.step(state["steps"])
        hz, pop = net.rates()
        return dict(hz=hz, pop=pop, stats=net.stats(), state=net.state())
    if kind == "loop":
        net = state["net"]
        net.step(1)
        n, _ = net.spikes_into(state["t"], state["ids"])
        fired = np.zeros(net.n, np.uint8)  # the order within a step is unspecified
        fired[state["ids"][:n]] = 1
        return fired
    if kind == "batch":
        state["batch"].step(state["steps"])
        read = [(m.rates(), m.stats(), m.state()) for m in state["batch"].members]
        cat = np.concatenate
        return dict(hz=cat([r[0].ravel() for r, _, _ in read]), pop=cat([r[1] for r, _, _ in read]),
                    stats=np.array([t for _, t, _ in read]),
                    v=cat([x[0] for _, _, x in read]), c=cat([x[1] for _, _, x in read]),
                    r=cat([x[2] for _, _, x in read]))
    if kind == "grad":
        th = torch.tensor(THETA, dtype=torch.float32, requires_grad=True)
        loss = snn.rate_loss(state["view"], th)
        loss.backward()
        return dict(loss=loss.detach(), grad=th.grad)
    if kind == "noalloc":
        s = state
        s["input"].copy_(s["drive"])  # the caller's own delivery
        n, ext = snn.snn_update_noalloc(
            s["gw"], s["gh"], s["neuron"], s["seed"], s["step"], s["v"].data_ptr(),
            s["c"].data_ptr(), s["r"].data_ptr(), s["input"].data_ptr(), s["spikes"].data_ptr(),
            s["counts"].data_ptr())
        s["step"] += 1
        s["fired"].zero_()
        s["fired"][s["spikes"][:n].long()] = 1  # the list's order is unspecified
        N = s["N"]
        return dict(v=s["v"][:N], c=s["c"][:N], r=s["r"][:N], fired=s["fired"], counts=s["counts"],
                    n=n, ext=ext)
    per_neuron = np.zeros(state["n"], np.int64)
    for _ in range(state["steps"]):
        per_neuron[_shard_step(state["shards"])] += 1
    out = dict(spikes=per_neuron)
    for k, sh in enumerate(state["shards"]):
        loc = sh.tile_local_neurons()
        out["shard%d" % k] = [x[loc] for x in sh.state()]
    return out


RATE = 0.0104  # spikes per neuron and step of the settled default network


def _net_bytes(n, s, precision, n_cols, steps):
    """26 B of state and input per neuron and step; per spike its list entry,
    its record, its synapses and two bucket bounds per delay."""
    N = n_cols * n["n_per_col"]
    k = 1307 if s["connectivity"] else s["k_out"]
    rec = 4 if precision == "f16w" else 8
    spikes = RATE * N * steps
    ev = spikes * k
    b = steps * 26.0 * N + spikes * (k * rec + 6.0 * (s["d_max"] - s["d_min"] + 1) + 12.0)
    return b, ev + 20.0 * N * steps


def work(case):
    n, s = _params(case)
    kind = case["kind"]
    if kind == "batch":
        grids, _, _, _ = W.batch_workload(case["nets"])
        b = [_net_bytes(n, s, case["precision"], w * h, case["steps"]) for w, h in grids]
        return dict(bytes=sum(x for x, _ in b), flops=sum(x for _, x in b))
    cols = case["gw"] * case["gh"]
    N = cols * n["n_per_col"]
    if kind == "noalloc":
        return dict(bytes=26.0 * N + 8.0 * 0.02 * N + 16.0 * cols, flops=20.0 * N)
    if kind == "grad":
        # the backward pass reads every synapse once per step, the forward
        # those of the spikes; state and adjoints of every neuron once per step
        b = case["T"] * N * (8.0 * s["k_out"] * (1.0 if not case["hard"] else 1.02) + 52.0)
        return dict(bytes=b, flops=case["T"] * N * 2.0 * s["k_out"])
    steps = 1 if kind == "loop" else case["steps"]
    b, f = _net_bytes(n, s, case["precision"], cols, steps)
    return dict(bytes=b, flops=f)


# --- 64-bit references -----------------------------------------------------


def _philox(seed, a, b, tag):
    """Philox4x32-10 (Salmon et al., SC'11), counter (a, b, tag, 0), key = seed."""
    M = np.uint64(0xFFFFFFFF)
    c = [np.asarray(x, np.uint64) for x in np.broadcast_arrays(a, b, tag, 0)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    s32 = np.uint64(32)
    for _ in range(10):
        p0, p1 = c[0] * np.uint64(0xD2511F53), c[2] * np.uint64(0xCD9E8D57)
        c = [(p1 >> s32) ^ c[1] ^ np.uint64(k0), p1 & M, (p0 >> s32) ^ c[3] ^ np.uint64(k1), p0 & M]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _per_neuron(seed, N, b, tag):
    q = np.arange((N + 3) // 4, dtype=np.uint64)
    return np.stack(_philox(seed, q, np.uint64(b), np.uint64(tag)), 1).reshape(-1)[:N]


def _f32(x):
    return float(np.float32(x))


def _propagators(n):
    tm, tc = _f32(n["tau_m"]), _f32(n["tau_c"])
    pvv, pcc = math.exp(-1.0 / tm), math.exp(-1.0 / tc)
    return pvv, pcc, -tm * tc / (tc - tm) * (pcc - pvv)


def exact(case, seed):
    if case["kind"] == "noalloc":
        return _exact_update(case, seed)
    if case["kind"] == "grad" and not case["hard"] and case["T"] <= 8:
        return _exact_soft(case, seed)
    return None  # spiking runs: a chaotic recursion has no 64-bit counterpart


def _exact_update(case, seed):
    n, _ = _params(case)
    b = _noalloc_buffers(case, seed)
    N, npc = b["N"], n["n_per_col"]
    v, c = (b[k][:N].cpu().numpy().astype(np.float64) for k in ("v", "c"))
    r, drive = (b[k][:N].cpu().numpy().astype(np.int64) for k in ("r", "drive"))
    lam = float(np.float32(n["nu_ext_kHz"]))
    cdf, p, k = [math.exp(-lam)], math.exp(-lam), 0
    while cdf[-1] < 1.0 - 2.0 ** -31:
        k += 1
        p = p * lam / k
        cdf.append(cdf[-1] + p)
    thr = np.floor(np.array(cdf[:-1]) * 2.0 ** 32).astype(np.uint64)
    ext = np.searchsorted(thr, _per_neuron(seed, N, 0, 2), side="right")
    jx = int(round(_f32(n["j_ext_mV"]) * 65536.0))
    u = v + (drive + ext * jx) / 65536.0
    active = r == 0
    fired = active & (u >= _f32(n["theta"]))
    vr = _f32(n["v_reset"])
    v1 = np.where(active & ~fired, u, vr)
    c1 = c + fired * _f32(n["dc"])
    exc = np.arange(N) % npc < n["n_exc"]
    pvv, pcc, kappa = _propagators(n)
    gc = np.where(exc, _f32(n["gc_exc"]), _f32(n["gc_inh"]))
    r1 = np.where(active, fired * int(round(n["t_ref"])), r - 1)
    col = np.arange(N) // npc
    counts = np.bincount(2 * col + ~exc, weights=fired, minlength=2 * (N // npc)).astype(np.int64)
    return dict(v=v1 * pvv + c1 * (gc * kappa), c=c1 * pcc, r=r1.astype(np.uint8),
                fired=fired.astype(np.uint8), counts=counts, n=int(fired.sum()), ext=int(ext.sum()))


def _exact_soft(case, seed):
    """The relaxed recursion and its gradient by torch's own autograd in FP64,
    on the synapses drawn from the seed."""
    n, s = _params(case)
    seed = seed + 1
    npc, gw, gh, K, T = n["n_per_col"], case["gw"], case["gh"], s["k_out"], case["T"]
    N = gw * gh * npc
    # synapses: counter (neuron, k, 1)
    j = np.repeat(np.arange(N, dtype=np.uint64), K)
    kk = np.tile(np.arange(K, dtype=np.uint64), N)
    x0, x1, x2, x3 = _philox(seed, j, kk, np.uint64(1))
    j, local = j.astype(np.int64), kk < round(_f32(s["frac_local"]) * K)
    R = s["stencil_radius"]
    off = [(dx, dy) for dy in range(-R, R + 1) for dx in range(-R, R + 1) if dx or dy]
    w = np.exp(-np.hypot(*np.array(off, float).T) / _f32(s["lambda_cols"]))
    m = np.searchsorted(np.floor(np.cumsum(w)[:-1] / w.sum() * 2.0 ** 32).astype(np.uint64), x1,
                        side="right")
    dx, dy = np.array(off).T
    col, l = j // npc, j % npc
    below = lambda x, k: ((x * np.uint64(k)) >> np.uint64(32)).astype(np.int64)
    own = below(x0, npc - 1)
    own += own >= l
    far = ((col // gw + dy[m]) % gh * gw + (col % gw + dx[m]) % gw) * npc + below(x0, npc)
    target = np.where(local, col * npc + own, far)
    delay = s["d_min"] + below(x2, s["d_max"] - s["d_min"] + 1)
    z = torch.special.ndtri((torch.arange(65536, dtype=torch.float64) + 0.5) / 65536.0).numpy()
    wt = []
    for mu in (_f32(s["w_exc_mV"]), _f32(s["w_inh_mV"])):
        a = mu * (1.0 + _f32(s["w_cv"]) * z)
        a = np.maximum(a, 0.0) if mu > 0 else np.minimum(a, 0.0)
        wt.append(np.rint(a.astype(np.float32).astype(np.float64) * 65536.0) / 65536.0)
    src_exc = l < n["n_exc"]
    weight = np.stack(wt)[(~src_exc).astype(np.int64), (x3 >> np.uint64(16)).astype(np.int64)]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    D = s["d_max"]
    order = np.argsort(target, kind="stable")
    to = lambda a: torch.from_numpy(np.ascontiguousarray(a[order])).to(dev)
    tgt, src, dly, wgt, sexc = to(target), to(j), to(delay), to(weight), to(src_exc)
    exc = torch.from_numpy(np.arange(N) % npc < n["n_exc"]).to(dev)
    v = torch.from_numpy(_per_neuron(seed, N, 0, 3).astype(np.int64) >> 8).to(dev).double()
    v = v * (_f32(n["theta"]) * 2.0 ** -24)
    th = torch.tensor(THETA, dtype=torch.float32).double().to(dev).requires_grad_(True)
    pvv, pcc, kappa = _propagators(n)
    J, vr, theta, beta = _f32(n["j_ext_mV"]), _f32(n["v_reset"]), _f32(n["theta"]), 5.0
    aE, aI = torch.where(exc, th[0], th[1]), torch.where(exc, th[2], th[3])
    pvc = torch.where(exc, th[4] * kappa, torch.tensor(_f32(n["gc_inh"]) * kappa, device=dev).double())
    c = torch.zeros_like(v)
    zero = torch.zeros_like(v)
    hist = [zero] * D  # hist[d - 1] = s(t - d)
    total = zero
    qf = torch.from_numpy(z.astype(np.float32)).to(dev).double()
    for t in range(T):
        part = wgt * torch.cat(hist)[(dly - 1) * N + src]
        XE = torch.zeros_like(v).index_add(0, tgt, torch.where(sexc, part, 0.0))
        XI = torch.zeros_like(v).index_add(0, tgt, torch.where(sexc, 0.0, part))
        xi = qf[torch.from_numpy((_per_neuron(seed, N, t, 4) >> np.uint64(16)).astype(np.int64)).to(dev)]
        inp = aE * XE + aI * XI + J * (th[5] + torch.sqrt(th[5]) * xi)
        g = torch.clamp(1.0 - hist[0] - hist[1], min=0.0)
        U = g * (v + inp) + (1.0 - g) * vr
        sp = torch.sigmoid(beta * (U - theta))
        vp = U - sp * (U - vr)
        cp = c + _f32(n["dc"]) * sp
        v, c = pvv * vp + pvc * cp, pcc * cp
        hist = [sp] + hist[:-1]
        total = total + sp
    rE, rI = (1000.0 * total[p].sum() / (T * int(p.sum())) for p in (exc, ~exc))
    loss = (rE - 3.0) ** 2 + (rI - 8.0) ** 2
    loss.backward()
    return dict(loss=loss.detach().cpu(), grad=th.grad.cpu())
