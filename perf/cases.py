"""What this library is used for, as timed cases: single layers through the public binding (`alif`, `autograd`,
`network`) and one whole neuron fit, over the sizes of the workloads in `synth.py`, the tests and `bench.py`.

Inputs are drawn on the GPU from the seed; currents that a projection would produce are formed with a plain torch
matmul, so that they do not depend on the library.  `exact()` evaluates the step-by-step model (Eqs 1-5 and its
reverse pass) with plain torch in float64."""
import math

import torch

from paper_2311_11390_gb300 import alif, autograd, network

DEV = "cuda"
SLOPE = 25.0
TAU_VR = 5.0
LARGEST = 32 * 1024 * 16000  # neuron-steps of the largest listed layers


def listed():
    return [
        # The single population of the speed-accuracy study: a launch-bound call that records both traces.
        dict(name="population_traces", kind="traces", B=8, N=128, T=1000, dt=0.1, arp=2.0),
        # The last chunk of a served fit request: ragged T, odd N, a carried state, parameter gradients only.
        dict(name="fit_chunk", kind="chunk", B=1, N=777, T=3001, dt=0.1, arp=2.0),
        # The input layer of the feedforward benchmark: 1000 Poisson channels onto 1024 neurons.
        dict(name="project_input", kind="project", B=32, Nin=1000, N=1024, T=16000, dt=0.1),
        # The same layer with exact FP32 weights (the event-driven projection).
        dict(name="project_events", kind="events", B=32, Nin=1000, N=1024, T=4000, dt=0.1),
        # Synapses between the two hidden layers of the classification network, forward and backward.
        dict(name="hidden_synapses", kind="synapses", B=128, Nin=256, N=256, T=1000, dt=1.0),
        # The feedforward benchmark's neurons: spikes, checkpoints and final state.
        dict(name="layer_forward", kind="forward", B=32, N=1024, T=16000, dt=0.1, arp=2.0),
        # Their surrogate-gradient backward: dL/dI and the five parameter gradients.
        dict(name="layer_backward", kind="backward", B=32, N=1024, T=16000, dt=0.1, arp=2.0),
        # One hidden ALIF layer of the classification network under torch.autograd (DT 1 ms, T_R 2).
        dict(name="alif_layer", kind="layer", B=128, N=256, T=1000, dt=1.0, arp=2.0),
        # A whole neuron fit: 1024 candidates, 20 s of one current at 0.05 ms, van Rossum loss and its gradients.
        dict(name="neuron_fit", kind="fit", B=1, N=1024, T=400000, dt=0.05, arp=2.0),
        # Weight and bias gradients of the feedforward benchmark's input layer.
        dict(name="project_gradients", kind="gradients", B=32, Nin=1000, N=1024, T=16000, dt=0.1),
        # The feedforward layer with recurrent synapses (latency = ARP).
        dict(name="recurrent", kind="recurrent", B=32, N=1024, T=4000, dt=0.1, arp=2.0),
        # The classification head: leaky readout, cross-entropy and their gradients.
        dict(name="readout_loss", kind="head", B=128, Nin=256, N=20, T=1000, dt=1.0),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def steps(lo, hi):  # recordings are of round or of any length
        t = log(lo, hi)
        return t if rng.random() < 0.5 else max(lo, t // 100 * 100)

    kind = rng.choice(["traces", "chunk", "project", "events", "synapses", "forward", "backward", "layer", "fit",
                       "gradients", "recurrent", "head"])
    dt, arp = rng.choice([0.05, 0.1, 1.0]), rng.choice([1.0, 2.0, 4.0])
    if kind == "traces":
        return dict(kind=kind, B=rng.randint(1, 16), N=log(32, 512), T=steps(500, 2000), dt=0.1, arp=arp)
    if kind == "chunk":
        return dict(kind=kind, B=1, N=log(64, 8192), T=steps(1000, 16384), dt=dt, arp=2.0)
    if kind in ("project", "events", "gradients"):
        B, N, T = rng.randint(1, 32), log(64, 1024), steps(1000, 16000)
        return dict(kind=kind, B=B, Nin=rng.choice([512, 700, 1000, log(64, 1000)]), N=N, T=T, dt=dt)
    if kind in ("forward", "backward"):
        N, T = log(64, 8192), steps(1000, 16000)
        return dict(kind=kind, B=rng.randint(1, max(1, min(32, LARGEST // (N * T)))), N=N, T=T, dt=0.1, arp=arp)
    if kind == "fit":
        return dict(kind=kind, B=1, N=log(64, 1024), T=steps(20000, 400000), dt=rng.choice([0.05, 0.1]), arp=2.0)
    if kind == "recurrent":
        return dict(kind=kind, B=rng.randint(1, 32), N=log(64, 1024), T=steps(500, 4000), dt=0.1, arp=arp)
    # the classification network's layers: DT 1 ms over 1 s or 0.1 ms over a shorter stretch
    dt = rng.choice([0.1, 1.0])
    c = dict(kind=kind, B=rng.randint(16, 128), N=256, T=steps(250, 2000), dt=dt)
    if kind == "synapses":
        return dict(c, Nin=log(64, 700), N=log(64, 512))
    if kind == "head":
        return dict(c, Nin=log(64, 512), N=rng.choice([10, 20, 35]))
    return dict(c, arp=2.0)


# ------------------------------------------------------------------ inputs
def _rand(g, *shape, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(shape, generator=g, device=DEV)


def _spikes(g, B, C, T, dt, lo=10.0, hi=50.0):
    """Poisson rasters, one batch element at a time as float 0/1 [C, T]: rates U[lo, hi] Hz per channel."""
    p = _rand(g, C, 1, lo=lo, hi=hi) * (dt * 1e-3)
    for _ in range(B):
        yield (torch.rand((C, T), generator=g, device=DEV) < p).float()


def _params(g, c):
    """[5, N] tau_mem, tau_adapt, theta0, d, R in the ranges of the case's workload."""
    N = c["N"]
    if c["kind"] == "fit":
        r = ((5.0, 40.0), (50.0, 1000.0), (0.5, 2.0), (0.0, 0.5), (0.5, 2.0))
    elif c["kind"] == "traces":
        r = ((20.0, 20.0), (200.0, 200.0), (1.0, 1.0), (0.1, 0.1), (1.0, 1.0))
    elif c["kind"] == "layer":
        r = ((20.0, 20.0), (150.0, 150.0), (1.0, 1.0), (1.8, 1.8), (1.0, 1.0))
    else:
        r = ((10.0, 30.0), (100.0, 500.0), (1.0, 1.0), (0.0, 0.2), (1.0, 1.0))
    return torch.stack([_rand(g, N, lo=a, hi=b) for a, b in r])


def _currents(g, c):
    """float32 [B, N, T] input currents: the projection of 512 Poisson channels plus a bias U[0.8, 1.6]; the small
    population's bias plus white noise; one Ornstein-Uhlenbeck current for all candidates of a fit."""
    B, N, T = c["B"], c["N"], c["T"]
    if c["kind"] == "fit":
        return _ou(g, T, c["dt"]).expand(1, N, T).contiguous()
    bias = _rand(g, N, 1, lo=0.8, hi=1.6)
    if c["kind"] == "traces":
        return bias + 0.3 * torch.randn((B, N, T), generator=g, device=DEV)
    W = math.sqrt(2.0 / 512) * torch.randn((N, 512), generator=g, device=DEV)
    out = torch.empty((B, N, T), device=DEV)
    for b, S in enumerate(_spikes(g, B, 512, T, c["dt"])):
        torch.addmm(bias, W, S, out=out[b])
    return out


def _ou(g, T, dt, tau=3.0, mean=0.5, sigma=0.5, K=500):
    """Exact Ornstein-Uhlenbeck update, K steps at a time: x[k] = e^(k+1) x_in + sum_j e^(k-j) s xi[j]."""
    e = math.exp(-dt / tau)
    n = -(-T // K)
    xi = torch.randn((n, K), generator=g, device=DEV).double() * (sigma * math.sqrt(1.0 - e * e))
    k = torch.arange(K, device=DEV, dtype=torch.float64)
    chain = (xi @ torch.tril(e ** (k[:, None] - k[None, :])).T).cpu()
    grow = (e ** (k + 1.0)).cpu()
    x, last = [], sigma * float(torch.randn((1,), generator=g, device=DEV))
    for row in chain:
        x.append(row + grow * last)
        last = float(x[-1][-1])
    return (mean + torch.cat(x)[:T]).float().to(DEV)


def _inputs(c, seed):
    """Everything a case starts from, as plain float tensors (rasters excepted: `spikes()` walks them)."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    k, B, N, T = c["kind"], c["B"], c["N"], c["T"]
    x = {}
    if k in ("project", "events", "synapses", "gradients", "head"):
        Nin = c["Nin"]
        if k in ("project", "events", "gradients"):
            x["W"] = math.sqrt(2.0 / Nin) * torch.randn((N, Nin), generator=g, device=DEV)
        else:
            x["W"] = _rand(g, N, Nin, lo=-1.0, hi=1.0) / math.sqrt(Nin)
        x["bias"] = torch.zeros(N, device=DEV) if k == "head" else _rand(g, N, lo=0.8, hi=1.6)
        if k in ("synapses", "gradients"):
            x["gI"] = torch.randn((B, N, T), generator=g, device=DEV)
        if k == "head":
            x["labels"] = torch.randint(0, N, (B,), generator=g, device=DEV, dtype=torch.int32)
        seeded = int(torch.randint(1 << 30, (1,), generator=g, device=DEV))
        x["spikes"] = lambda: _spikes(torch.Generator(device=DEV).manual_seed(seeded), B, Nin, T, c["dt"])
        return x
    x["par"] = _params(g, c)
    x["I"] = _currents(g, c)
    if k in ("backward", "layer", "chunk"):
        x["gS"] = torch.randn((B, N, T), generator=g, device=DEV)
    if k == "chunk":  # mid-sequence state: sub-threshold membranes, some adaptation, some neurons refractory
        rem = torch.randint(-20, 10, (B, N), generator=g, device=DEV).clamp_(min=0, max=max(1, round(c["arp"] / c["dt"]) - 1))
        x["rem"] = rem
        x["v"] = _rand(g, B, N, hi=0.9) * (rem == 0)
        x["a"] = _rand(g, B, N, hi=3.0)
        x["gfin"] = torch.randn((B, N, 2), generator=g, device=DEV)
    if k == "recurrent":
        x["W"] = 1.5 / math.sqrt(N) * torch.randn((N, N), generator=g, device=DEV)
    return x


HIDDEN = torch.tensor([[20.0], [200.0], [1.0], [0.1], [1.5]])  # the neuron that a fit looks for


def _table(par, c):
    return alif.neuron_table(*(p.cpu().numpy() for p in par), dt_ms=c["dt"], arp_ms=c["arp"], device=DEV)


def _words(x):
    """The raster as bits [B, C, ceil(T/32)]."""
    return torch.stack([alif.pack_spikes(S) for S in x["spikes"]()])


# --------------------------------------------------------------- a user's program
def prepare(case, seed):
    c, x = case, _inputs(case, seed)
    k, T = c["kind"], c["T"]
    s = dict(c=c)
    if k == "project":
        hi, lo = alif.split_bf16(x["W"])
        return dict(s, S=_words(x), hi=hi, lo=lo, bias=x["bias"])
    if k == "events":
        return dict(s, S=_words(x), Wt=alif.transpose_weights(x["W"]), bias=x["bias"])
    if k == "gradients":
        return dict(s, S=_words(x), gI=x["gI"])
    if k in ("synapses", "head"):
        words = _words(x)
        leaf = [t.requires_grad_() for t in (alif.spikes_to_float(words, T), x["W"], x["bias"])]
        if k == "head":
            s["w_t"], s["w_sum"] = alif.readout_weights(T, c["dt"], 20.0, DEV)
            s["labels"] = x["labels"]
        return dict(s, words=words, leaf=leaf, gI=x.get("gI"))
    if k == "layer":
        return dict(s, net=autograd.ALIFLayer(c["N"], dt=c["dt"], arp=c["arp"]).to(DEV), I=x["I"].requires_grad_(), gS=x["gS"])
    s.update(I=x["I"], table=_table(x["par"], c))
    if k == "backward":
        out = alif.forward(s["I"], s["table"], want_final=False)
        s.update(spikes=out["spikes"], ckpt=out["ckpt"], gS=x["gS"])
    if k == "chunk":
        s.update(init=alif.state_tensor(1, c["N"], DEV, x["v"], x["a"], x["rem"]), gS=x["gS"], gfin=x["gfin"])
    if k == "fit":
        target = alif.forward(s["I"][:, :1].contiguous(), _table(HIDDEN, c), want_ckpt=False, want_final=False)["spikes"]
        s["target"] = target[0].expand(c["N"], -1).contiguous()
    if k == "recurrent":
        s["Wt"] = alif.transpose_weights(x["W"])
    return s


def _state(t):
    """(v, a, steps still refractory) as the state holds them: three 32-bit fields, read as floats."""
    return t.view(torch.float32)


def run(s):
    c = s["c"]
    k, T = c["kind"], c["T"]
    if k == "project":
        return alif.syn_project(s["S"], s["hi"], s["lo"], s["bias"], Nin=c["Nin"], T=T)
    if k == "events":
        return alif.syn_project_events(s["S"], s["Wt"], s["bias"], Nin=c["Nin"], T=T)
    if k == "gradients":
        gW, _, gb = alif.syn_project_backward(s["S"], s["gI"], Nin=c["Nin"])
        return dict(gW=gW, gb=gb)
    if k == "synapses":
        I = network.SynProject.apply(*s["leaf"], s["words"], T)
        gS, gW, gb = torch.autograd.grad(I, s["leaf"], s["gI"])
        return dict(I=I, gS=gS, gW=gW, gb=gb)
    if k == "head":
        logits = network.Readout.apply(*s["leaf"], s["words"], T, s["w_t"], s["w_sum"])
        loss = network.CrossEntropy.apply(logits, s["labels"])
        gS, gW, gb = torch.autograd.grad(loss, s["leaf"])
        return dict(logits=logits, loss=loss, gS=gS, gW=gW, gb=gb)
    if k == "layer":
        net = s["net"]
        S = net(s["I"])
        gI, *gp = torch.autograd.grad(S, [s["I"], net.tau_mem, net.tau_adapt, net.theta0, net.d], s["gS"])
        return dict(S=S, gI=gI, gp=gp)
    if k == "traces":
        o = alif.forward(s["I"], s["table"], want_v=True, want_a=True, want_ckpt=False)
        return dict(spikes=o["spikes"], v=o["v"], a=o["a"], final=_state(o["final"]))
    if k == "forward":
        o = alif.forward(s["I"], s["table"])
        return dict(spikes=o["spikes"], ckpt=_state(o["ckpt"]), final=_state(o["final"]))
    if k == "backward":
        gI, _, gp = alif.backward(s["I"], s["table"], s["spikes"], s["gS"], ckpt=s["ckpt"], slope=SLOPE)
        return dict(gI=gI, gp=gp)
    if k == "chunk":
        o = alif.forward(s["I"], s["table"], init=s["init"])
        _, ginit, gp = alif.backward(s["I"], s["table"], o["spikes"], s["gS"], ckpt=o["ckpt"], grad_final=s["gfin"],
                                     init=s["init"], slope=SLOPE, want_gI=False, want_ginit=True)
        return dict(spikes=o["spikes"], final=_state(o["final"]), ginit=ginit, gp=gp)
    if k == "recurrent":
        o = alif.forward_recurrent(s["I"], s["Wt"], s["table"], c["dt"], c["arp"])
        return dict(spikes=o["spikes"], I=o["I_total"], ckpt=_state(o["ckpt"]), final=_state(o["final"]))
    # fit: forward, van Rossum distance to the target train, its gradient, parameter gradients
    N = c["N"]
    o = alif.forward(s["I"], s["table"], want_final=False)
    x, y = o["spikes"][0], s["target"]
    loss = torch.empty(N, device=DEV)
    alif.vanrossum_forward(x, y, T, c["dt"], TAU_VR, -(-T // 256) * 256, loss=loss)
    zero, gS = torch.zeros((2, N), device=DEV), torch.empty((1, N, T), device=DEV)
    alif.vanrossum_backward(x, y, T, c["dt"], TAU_VR, 0, T, zero[0], zero[1], gS[0])
    _, _, gp = alif.backward(s["I"], s["table"], o["spikes"], gS, ckpt=o["ckpt"], slope=SLOPE, want_gI=False)
    return dict(spikes=o["spikes"], loss=loss, gp=gp)


def work(case):
    """Bytes: every input read once, every output written once.  Operations: one addition per input spike and
    target neuron for the projections (at the mean rate), a step's few per neuron elsewhere."""
    c = case
    k, B, N, T = c["kind"], c["B"], c["N"], c["T"]
    words = 4 * -(-T // 32)
    rows, cur, ck = B * N, B * N * T * 4, B * N * -(-T // 256) * 12
    if "Nin" in c:
        Nin = c["Nin"]
        adds = B * Nin * T * 30.0 * c["dt"] * 1e-3 * N
        raster, W = B * Nin * words, N * Nin * 4
        if k == "head":
            return dict(bytes=raster + 2 * W + B * Nin * T * 4, flops=6.0 * B * Nin * N + B * Nin * T * 1.03)
        if k == "synapses":  # I, gW and gb, and the dense gS = W^T gI
            return dict(bytes=2 * raster + 2 * cur + B * Nin * T * 4 + 3 * W, flops=2 * adds + 2.0 * B * Nin * N * T)
        return dict(bytes=raster + cur + W, flops=adds)
    per = dict(traces=12 * rows * T, chunk=8 * rows * T, forward=cur + ck, backward=3 * cur + rows * words + ck,
               layer=6 * cur, fit=2 * cur + 4 * ck, recurrent=2 * cur + ck)[k]
    ops = dict(traces=8, chunk=30, forward=8, backward=22, layer=30, fit=36, recurrent=8)[k] * rows * T
    if k == "recurrent":
        per += N * N * 4
        ops += rows * T * N * 20.0 * c["dt"] * 1e-3
    return dict(bytes=per + rows * words + rows * 12 + N * 64, flops=float(ops))


# ------------------------------------------------------------ the model in 64 bits
def _replayed(step, n, before):
    """step(0) .. step(n - 1) as one captured graph."""
    step(0)  # first use of every operation outside the capture
    torch.cuda.synchronize()
    before()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        for k in range(n):
            step(k)
    return g


def _scan(f, x, init, K=500):
    """y[t] = f[t] y[t-1] + x[t] along the first axis (f one row for all t, or one per t)."""
    T, R = x.shape
    y = torch.empty_like(x)
    fc, xc, yc = (torch.zeros((K + 1, R), dtype=torch.float64, device=DEV) for _ in range(3))
    if f.dim() == 1:
        fc[:] = f
    g = _replayed(lambda k: torch.addcmul(xc[k], fc[k], yc[k], out=yc[k + 1]), K, lambda: None)
    yc[K] = init
    for t in range(0, T, K):
        n = min(K, T - t)
        yc[0] = yc[K]
        xc[:n] = x[t:t + n]
        if f.dim() == 2:
            fc[:n] = f[t:t + n]
        g.replay()
        y[t:t + n] = yc[1:n + 1]
    return y


class _Model:
    """The standard model (Eqs 1-5) and its detached surrogate gradient, time first, one column per row."""

    def __init__(self, c, par, rows_b):
        par = par.double().repeat(1, rows_b)
        tm, ta, self.th0, self.d, self.R = par
        self.dt, self.T_R = c["dt"], int(round(c["arp"] / c["dt"]))
        self.beta, self.p = torch.exp(-self.dt / tm), torch.exp(-self.dt / ta)
        self.dbeta, self.dp = self.beta * self.dt / tm ** 2, self.p * self.dt / ta ** 2
        self.c = (1.0 - self.beta) * self.R
        self.teff = max(self.T_R, 2)

    def forward(self, I, state=None, delayed=None, K=500):
        """I [T, R] -> V, a, S, m (m: input admitted).  delayed(t0, n, S): current added to steps t0 .. t0 + n."""
        T, R = I.shape
        new = lambda *s: torch.zeros(s, dtype=torch.float64, device=DEV)  # noqa: E731
        V, A, M, S = new(T, R), new(T, R), torch.zeros((T, R), dtype=torch.bool, device=DEV), torch.zeros((T, R), dtype=torch.bool, device=DEV)
        v, a, rem = (new(R) for _ in range(3)) if state is None else (t.double().reshape(-1).clone() for t in state)
        xc, Vc, Ac, Mc, Sc = new(K, R), new(K, R), new(K, R), M.new_zeros((K, R)), S.new_zeros((K, R))
        th, start = new(R), (v.clone(), a.clone(), rem.clone())

        def step(k):
            torch.le(rem, 0.0, out=Mc[k])
            v.mul_(self.beta).addcmul_(xc[k], Mc[k].double())
            Vc[k].copy_(v)
            Ac[k].copy_(a)
            torch.addcmul(self.th0, self.d, a, out=th)
            torch.gt(v, th, out=Sc[k])
            v.masked_fill_(Sc[k], 0.0)
            a.mul_(self.p).add_(Sc[k])
            rem.sub_(1.0).clamp_(min=0.0).masked_fill_(Sc[k], self.teff - 1.0)

        g = _replayed(step, K, lambda: [x.copy_(y) for x, y in zip((v, a, rem), start)])
        for t in range(0, T, K):
            n = min(K, T - t)
            xc.zero_()
            xc[:n] = self.c * (I[t:t + n] if delayed is None else delayed(t, n, S))
            g.replay()
            for full, part in ((V, Vc), (A, Ac), (M, Mc), (S, Sc)):
                full[t:t + n] = part[:n]
        self.V, self.A, self.M, self.S, self.start = V, A, M, S, start
        return self

    def states(self, at):
        """[R, len(at), 3] states entering the steps `at` (the refractory count as the bits of an integer)."""
        out = []
        for t in at:
            if t == 0:
                out.append(torch.stack(self.start, -1))
                continue
            s = self.S[t - 1].double()
            look = self.S[max(0, t - self.teff + 1):t].double()  # the spikes that still mask step t
            since = look.shape[0] - (look * torch.arange(1, look.shape[0] + 1, device=DEV)[:, None]).amax(0) if look.shape[0] else None
            rem = torch.zeros_like(s) if since is None else torch.where(look.amax(0) > 0, self.teff - 1 - since, torch.zeros_like(s))
            if t < self.teff:
                rem = torch.maximum(rem, self.start[2] - t)
            out.append(torch.stack([self.V[t - 1] * (1 - s), self.p * self.A[t - 1] + s, rem], -1))
        out = torch.stack(out, 1)
        out[..., 2] *= 2.0 ** -149
        return out

    def backward(self, I, gS, gfin=None):
        """dL/dI [T, R], dL/d(init v, init a) [R, 2] and the parameter gradients [5, R]."""
        s = self.S.double()
        u = self.V - self.th0 - self.d * self.A
        e = gS / (SLOPE * u.abs() + 1.0).square()
        del u
        f = self.beta * (1.0 - s)
        gv = e[-1] if gfin is None else e[-1] + (1.0 - s[-1]) * gfin[:, 0]
        ga = gfin[:, 1] if gfin is not None else torch.zeros_like(gv)
        GV = torch.cat([gv[None], _scan(f[:-1].flip(0), e[:-1].flip(0), gv)]).flip(0)
        GA = _scan(self.p, -self.d * e.flip(0), ga).flip(0)
        GAn = torch.cat([GA[1:], ga[None]])  # dL/da of the next step
        ginit = torch.stack([self.beta * GV[0], GA[0]], -1)
        MI = self.M * I
        vin = torch.cat([self.start[0][None], self.V[:-1] * (1.0 - s[:-1])])
        gp = torch.stack([self.dbeta * ((vin - self.R * MI) * GV).sum(0), self.dp * (self.A * GAn).sum(0), -e.sum(0),
                          -(self.A * e).sum(0), (1.0 - self.beta) * (MI * GV).sum(0)])
        return self.c * self.M * GV, ginit, gp


def exact(case, seed):
    c, x = case, _inputs(case, seed)
    k, B, N, T = c["kind"], c["B"], c["N"], c["T"]
    dbl = {n: v.double() for n, v in x.items() if n in ("W", "bias")}
    if k in ("project", "events"):
        out = torch.empty((B, N, T), dtype=torch.float64, device=DEV)
        for b, S in enumerate(x["spikes"]()):
            torch.addmm(dbl["bias"][:, None], dbl["W"], S.double(), out=out[b])
        return out
    if k in ("gradients", "synapses"):
        o = dict(gW=torch.zeros((N, c["Nin"]), dtype=torch.float64, device=DEV), gb=x["gI"].double().sum((0, 2)))
        I, gS = [], []
        for b, S in enumerate(x["spikes"]()):
            S, g = S.double(), x["gI"][b].double()
            o["gW"] += g @ S.T
            if k == "synapses":
                I.append(torch.addmm(dbl["bias"][:, None], dbl["W"], S))
                gS.append(dbl["W"].T @ g)
        return dict(o, I=torch.stack(I), gS=torch.stack(gS)) if I else o
    if k == "head":
        beta = math.exp(-c["dt"] / 20.0)
        w = 1.0 - beta ** torch.arange(T, 0, -1, device=DEV, dtype=torch.float64)
        n = torch.stack([S.double() @ w for S in x["spikes"]()])
        logits = n @ dbl["W"].T + dbl["bias"] * w.sum()
        lab = x["labels"].long()
        g = (torch.softmax(logits, 1) - torch.nn.functional.one_hot(lab, N)) / B
        return dict(logits=logits, loss=torch.nn.functional.cross_entropy(logits, lab), gS=(g @ dbl["W"])[:, :, None] * w,
                    gW=g.T @ n, gb=g.sum(0) * w.sum())
    R = B * N
    time_first = lambda t: t.reshape(R, T).T  # noqa: E731
    rows = lambda t: t.T.reshape(B, N, T).contiguous()  # noqa: E731
    I = time_first(x["I"]).double().contiguous()
    m = _Model(c, x["par"], B)
    cks = range(0, T, 256)
    if k == "recurrent":
        W, total = dbl["W"], torch.empty_like(I)

        def delayed(t, n, S):
            total[t:t + n] = I[t:t + n]
            a = t - m.T_R
            s = S[max(a, 0):a + n].double().reshape(-1, B, N)
            if s.shape[0]:
                total[t + n - s.shape[0]:t + n] += (s.reshape(-1, N) @ W.T).reshape(-1, R)
            return total[t:t + n]

        m.forward(I, delayed=delayed, K=m.T_R)
        return dict(spikes=None, I=rows(total), ckpt=m.states(cks).reshape(B, N, -1, 3), final=m.states([T]).reshape(B, N, 3))
    if k == "fit":  # the neuron that is looked for runs as one more row
        m = _Model(c, torch.cat([x["par"], HIDDEN.to(DEV)], 1), 1).forward(torch.cat([I, I[:, :1]], 1))
        y = m.S[:, N:].double()
        m = _Rows(m, N)
        decay = torch.full((N,), math.exp(-c["dt"] / TAU_VR), dtype=torch.float64, device=DEV)
        f = _scan(decay, m.S.double() - y, 0.0)
        loss = c["dt"] / TAU_VR * f.square().sum(0)
        gS = 2.0 * c["dt"] / TAU_VR * _scan(decay, f.flip(0), 0.0).flip(0)
        return dict(spikes=None, loss=loss, gp=m.backward(I, gS)[2])
    m.forward(I, (x["v"], x["a"], x["rem"]) if k == "chunk" else None)
    if k == "traces":
        return dict(spikes=None, v=rows(m.V), a=rows(m.A), final=m.states([T]).reshape(B, N, 3))
    if k == "forward":
        return dict(spikes=None, ckpt=m.states(cks).reshape(B, N, -1, 3), final=m.states([T]).reshape(B, N, 3))
    gI, ginit, gp = m.backward(I, time_first(x["gS"]).double(), x["gfin"].double().reshape(R, 2) if k == "chunk" else None)
    gp = gp.reshape(5, B, N).sum(1)
    if k == "chunk":
        return dict(spikes=None, final=m.states([T]).reshape(B, N, 3), ginit=ginit.reshape(B, N, 2), gp=gp)
    if k == "layer":
        return dict(S=rows(m.S.double()), gI=rows(gI), gp=list(gp[:4]))
    return dict(gI=rows(gI), gp=gp)


def _Rows(m, n):
    """The model's first n rows."""
    for name in ("V", "A", "M", "S"):
        setattr(m, name, getattr(m, name)[:, :n].contiguous())
    for name in ("th0", "d", "R", "beta", "p", "dbeta", "dp", "c"):
        setattr(m, name, getattr(m, name)[:n])
    m.start = tuple(t[:n] for t in m.start)
    return m
