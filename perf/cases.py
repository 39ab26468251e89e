"""Performance cases of the library: what its users run, through the public
entry points of ``paper_1909_02549_gb300.snn``.

A case's ``kind`` is the program it stands for:

* ``train``  a minibatch is presented to a plastic network from a checkpoint of
             its weights and thresholds; the spike counts, the updated weights
             and thresholds and the final voltages are taken.  ``net`` is the
             digit network ("digits"), the same with the paper's own learning
             rule ("rule"), or the two-layer scaling network ("scaling");
* ``infer``  the same with the parameters frozen;
* ``rec``    a presentation through the recurrent inference network;
* ``serve``  a queue of requests of mixed lengths through the serving loop.

Every input is made from the seed alone: images of which 70 % of the pixels are
dark (rates intensity/4 or intensity/2 Hz), rates U[0, 120] Hz for the scaling
network and U[0, 50] Hz for the recurrent one.
"""
import math

import numpy as np
import torch

from paper_1909_02549_gb300 import snn

# Adaptive-threshold LIF network with lateral inhibition (mV, ms).
DIGITS = dict(e_rest=-65.0, e_reset=-60.0, e_thresh=-52.0, e_tau=100.0, e_refrac=5.0, theta_plus=0.05,
              theta_tau=1e7, i_rest=-60.0, i_reset=-45.0, i_thresh=-40.0, i_tau=10.0, i_refrac=2.0,
              w_ei=22.5, w_ie=-17.5, trace_tau=20.0, nu_pre=1e-4, nu_post=1e-2, w_min=0.0, w_max=1.0)
SCALING = dict(DIGITS, e_reset=-65.0, theta_plus=0.0, w_ei=0.0, w_ie=0.0)
REC = dict(tau_mem=20.0, tau_syn=5.0, v_thresh=1.0, v_reset=0.0)
WPREC = {"fp32": snn.SNN_W_FP32, "bf16": snn.SNN_W_BF16, "fp8": snn.SNN_W_FP8E4M3}
SERVE_CHUNK = 10


def _net(name, n_in, n_exc, batch, steps, *, kind="train", net="digits", mode="auto", reduce="mean", wprec="fp32"):
    c = dict(kind=kind, net=net, n_in=n_in, n_exc=n_exc, batch=batch, steps=steps, mode=mode, reduce=reduce,
             wprec=wprec)
    return dict(c, name=name) if name else c


def _rec(name, n_in, n_hid, batch, steps, form):
    c = dict(kind="rec", n_in=n_in, n_hid=n_hid, n_out=10, batch=batch, steps=steps, form=form)
    return dict(c, name=name) if name else c


def _serve(name, n_in, n_exc, requests, longest):
    c = dict(kind="serve", net="digits", n_in=n_in, n_exc=n_exc, requests=requests, longest=longest, wprec="fp32")
    return dict(c, name=name) if name else c


def listed():
    return [
        # online learning, one sample at a time: the small network of the digits experiment
        _net("train_784x100_b1", 784, 100, 1, 250),
        # the paper's own rule (post-triggered, normalised, per-parameter maximum), its usual batch
        _net("rule_784x100_b64_max", 784, 100, 64, 250, net="rule", reduce="max"),
        # minibatch training of the medium network: a small batch, and the largest of the batch sweep
        _net("train_784x400_b16", 784, 400, 16, 250),
        _net("train_784x400_b1024_sum", 784, 400, 1024, 250, reduce="sum"),
        # the headline workload: the large network, pair rule, mean over the batch
        _net("train_784x6400_b256", 784, 6400, 256, 250),
        # the tensor-core form: the largest batch, and reduced-precision weights
        _net("tensor_784x6400_b1024", 784, 6400, 1024, 250, mode="tensor"),
        _net("tensor_784x6400_b256_bf16", 784, 6400, 256, 250, mode="tensor", wprec="bf16"),
        # evaluation of a trained network, nothing learns
        _net("infer_784x400_b256", 784, 400, 256, 350, kind="infer"),
        # the scaling experiment's widest layer at its largest batch
        _net("scaling_100x10000_b1024", 100, 10000, 1024, 250, net="scaling"),
        # recurrent inference: the full size on the tensor cores, and a small one in the exact order
        _rec("rec_1024x4096_b4096", 1024, 4096, 4096, 500, "tensor"),
        _rec("rec_1024x512_b64_gather", 1024, 512, 64, 100, "gather"),
        # serving: a burst of requests of 50 to 500 steps on a frozen network
        _serve("serve_784x400", 784, 400, 512, 500),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train", "train", "train", "tensor", "tensor", "infer", "scaling", "rule", "rec", "rec", "serve"])
    steps = _log_int(rng, 60, 350)
    if kind in ("train", "infer"):
        n = _log_int(rng, 50, 6400)
        b = _log_int(rng, 1, min(1024, 6400 * 256 // n))
        wprec = rng.choice(["fp32", "fp32", "fp32", "bf16", "fp8"])
        return _net(None, rng.choice([784, 784, 100, 225, 1023]), n, b, steps, kind=kind, wprec=wprec,
                    reduce=rng.choice(["mean", "mean", "sum", "max"]) if kind == "train" else "mean")
    if kind == "tensor":
        n, b = _log_int(rng, 300, 6400), _log_int(rng, 64, 1024)
        return _net(None, rng.choice([784, 784, 500, 1023]), n, b, min(steps, 250), mode="tensor",
                    wprec=rng.choice(["fp32", "fp32", "bf16"]), reduce=rng.choice(["mean", "mean", "sum"]))
    if kind == "scaling":
        n = _log_int(rng, 100, 10000)
        return _net(None, 100, n, _log_int(rng, 1, min(1024, 10000 * 256 // n)), steps, net="scaling",
                    kind=rng.choice(["train", "train", "infer"]))
    if kind == "rule":
        return _net(None, 784, _log_int(rng, 50, 400), _log_int(rng, 1, 256), steps, net="rule",
                    reduce=rng.choice(["max", "max", "mean", "sum"]))
    if kind == "rec":
        if rng.random() < 0.3:
            return _rec(None, rng.choice([64, 200, 1024]), _log_int(rng, 128, 1024), _log_int(rng, 1, 128), steps,
                        "gather")
        return _rec(None, rng.choice([64, 300, 1024]), _log_int(rng, 256, 4096), _log_int(rng, 16, 4096), steps,
                    rng.choice(["tensor", "tensor", "auto"]))
    return _serve(None, 784, _log_int(rng, 100, 1000), _log_int(rng, 16, 1024), rng.randint(100, 500))


# ------------------------------------------------------------------ inputs ---

def _generator(seed, part):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + part)


def _params(case):
    p = dict(SCALING if case["net"] == "scaling" else DIGITS, n_in=case["n_in"], n_exc=case["n_exc"])
    if case["net"] == "rule":
        p.update(theta_tau=1e6, rule=snn.SNN_RULE_POST_NORM, w_norm=0.1 * case["n_in"])
    return p


def _rates(case, n, seed):
    g = _generator(seed, 1)
    u = torch.rand((n, case["n_in"]), generator=g, device="cuda")
    if case["kind"] == "rec":
        return 50.0 * u
    if case["net"] == "scaling":
        return 120.0 * u
    lit = torch.rand((n, case["n_in"]), generator=g, device="cuda") >= 0.7
    return torch.where(lit, 255.0 * u / (2.0 if case["net"] == "rule" else 4.0), torch.zeros_like(u))


def _seeds(n, seed):
    return torch.randint(0, 1 << 62, (n,), generator=_generator(seed, 2), device="cuda")


def _weights(case, seed):
    shape, g = (case["n_in"], case["n_exc"]), _generator(seed, 3)
    if case["net"] == "scaling":
        return 0.1 + 0.01 * torch.randn(shape, generator=g, device="cuda")
    u = torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)
    return (torch.clamp(torch.floor(u * 0.3 * 4096 + 0.5), max=1228.0) / 4096).float()


def _theta(case, seed):
    """Thresholds of a network that has been training for a while (mV)."""
    t = torch.rand(case["n_exc"], generator=_generator(seed, 4), device="cuda", dtype=torch.float64)
    return torch.zeros_like(t) if case["net"] == "scaling" else t


def _rec_weights(case, seed):
    g, ni, nh, no = _generator(seed, 5), case["n_in"], case["n_hid"], case["n_out"]
    w_ff = 0.05 * torch.randn((ni, nh), generator=g, device="cuda")
    w_rec = 0.02 * torch.randn((nh, nh), generator=g, device="cuda")
    w_rec = torch.where(torch.rand((nh, nh), generator=g, device="cuda") < 0.1, w_rec, torch.zeros_like(w_rec))
    w_out = 0.05 * torch.randn((nh, no), generator=g, device="cuda")
    return [w.bfloat16() for w in (w_ff, w_rec, w_out)]


def _lengths(case, seed):
    return np.random.RandomState(seed % (1 << 31)).randint(50, case["longest"] + 1, case["requests"])


def prepare(case, seed):
    if case["kind"] == "rec":
        w = [x.view(torch.int16).cpu().numpy().view(np.uint16) for x in _rec_weights(case, seed)]
        b, nh, no = case["batch"], case["n_hid"], case["n_out"]
        net = snn.RecNetwork(dict(REC, n_in=case["n_in"], n_hid=nh, n_out=no), *w)
        return dict(case=case, net=net, rates=_rates(case, b, seed), seeds=_seeds(b, seed),
                    out=dict(v_out=torch.empty((b, no), device="cuda"),
                             counts=torch.empty((b, nh), device="cuda", dtype=torch.int32),
                             v=torch.empty((b, nh), device="cuda")))
    w, theta = _weights(case, seed), _theta(case, seed)
    net = snn.Network(_params(case), w_init=w.cpu().numpy(), theta_init=theta.cpu().numpy(),
                      wprec=WPREC[case["wprec"]])
    if case["kind"] == "serve":
        n = case["requests"]
        return dict(case=case, net=net, server=_Server(snn.snn_serve_create(net.handle, 4096, 1 << 30)),
                    rates=_rates(case, n, seed).cpu().numpy(), seeds=_seeds(n, seed).tolist(),
                    lengths=_lengths(case, seed).tolist())
    b, n = case["batch"], case["n_exc"]
    out = dict(counts=torch.empty((b, n), device="cuda", dtype=torch.int32), v=torch.empty((b, n), device="cuda"))
    if case["kind"] == "train":
        out.update(w=torch.empty_like(w), theta=torch.empty_like(theta))
    return dict(case=case, net=net, w=w, theta=theta, rates=_rates(case, b, seed), seeds=_seeds(b, seed), out=out)


class _Server:
    """Destroys the server with its state."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        snn.snn_serve_destroy(self.handle)


# --------------------------------------------------------------------- run ---

def run(state):
    return {"rec": _run_rec, "serve": _run_serve}.get(state["case"]["kind"], _run_net)(state)


def _run_net(s):
    c, net, out = s["case"], s["net"], s["out"]
    train = c["kind"] == "train"
    if train:          # from the checkpoint
        snn.snn_write_weights(net.handle, s["w"])
        snn.snn_write_state(net.handle, snn.SNN_FIELD_THETA, s["theta"])
    net.run(s["rates"], s["seeds"], c["steps"], learn=train, reduce=c["reduce"], mode=c["mode"])
    snn.snn_read_state(net.handle, snn.SNN_FIELD_SPIKE_COUNTS, out["counts"])
    snn.snn_read_state(net.handle, snn.SNN_FIELD_V_EXC, out["v"])
    if train:
        snn.snn_read_weights(net.handle, out["w"])
        snn.snn_read_state(net.handle, snn.SNN_FIELD_THETA, out["theta"])
    return out


def _run_rec(s):
    c, net, out = s["case"], s["net"], s["out"]
    net.run(s["rates"], s["seeds"], c["steps"], form=c["form"])
    for field, t in ((snn.SNN_REC_V_OUT, out["v_out"]), (snn.SNN_REC_COUNTS, out["counts"]), (snn.SNN_REC_V, out["v"])):
        status = snn.lib().snn_rec_read(net.handle, field, t.data_ptr(), t.numel() * t.element_size(), 1)
        if status != snn.SNN_OK:
            raise snn.SNNError(status, "snn_rec_read")
    return out


def _run_serve(s):
    c, srv = s["case"], s["server"].handle
    place = {}
    for q in range(c["requests"]):
        place[snn.snn_serve_submit(srv, s["rates"][q], s["seeds"][q], s["lengths"][q])] = q
    counts = np.empty((c["requests"], c["n_exc"]), np.uint32)
    left = c["requests"]
    while left:
        status = snn.snn_serve_status(srv)
        if status["active"] or status["queued"]:
            snn.snn_serve_step(srv, SERVE_CHUNK)
        else:
            snn.snn_serve_wait(srv)
        ids, got = snn.snn_serve_poll(srv, c["n_exc"])
        for i, x in zip(ids, got):
            counts[place[int(i)]] = x
        left -= len(ids)
    return counts.view(np.int32)


# -------------------------------------------------------------------- work ---

def work(case):
    """Bytes of one pass: each sample's state, rates and spikes read and written every step and the weights
    once a step (twice with learning), as a clock-based simulation defines its steps.  Operations: the additions
    of the active inputs' weights at the mean rates, and a multiply-add per synapse and step of the update."""
    if case["kind"] == "serve":
        s = sum(int(t) for t in _lengths(case, 1))
        n, ni = case["n_exc"], case["n_in"]
        return {"bytes": s * (21 * n + 4 * ni) + 4 * ni * n, "flops": s * n * (0.01 * ni + 20)}
    b, t, ni = case["batch"], case["steps"], case["n_in"]
    if case["kind"] == "rec":
        n, no = case["n_hid"], case["n_out"]
        step = b * (26 * n + 6 * ni + 8 * no) + 2 * n * (ni + n + no)
        return {"bytes": t * step, "flops": t * b * (n * (0.025 * ni + 0.2 * 0.1 * n + 10) + 0.2 * n * no)}
    n, learn = case["n_exc"], case["kind"] == "train"
    step = b * ((29 if learn else 21) * n + (12 if learn else 4) * ni) + (8 if learn else 4) * ni * n
    rate = {"digits": 0.0096, "rule": 0.019, "scaling": 0.06}[case["net"]]
    return {"bytes": t * step, "flops": t * (b * n * (rate * ni + 20) + (2 * ni * n if learn else 0))}


# ------------------------------------------------------------------- exact ---

def _i64(x):
    return x - (1 << 64) if x >= 1 << 63 else x


def _shift(z, k):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _splitmix(x):
    z = x + _i64(0x9E3779B97F4A7C15)
    z = (z ^ _shift(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _shift(z, 27)) * _i64(0x94D049BB133111EB)
    return z ^ _shift(z, 31)


def _draws(rates, seeds, t):
    """The step's Poisson spikes as 0/1 doubles: one hashed trial per input, sample and step."""
    thr = torch.clamp(torch.floor(rates.double() * 1e-3 * 4294967296.0), 0, 4294967295.0).long()
    ctr = torch.arange(rates.shape[1], device=rates.device) + t * rates.shape[1]
    h = _splitmix(seeds[:, None] ^ _splitmix(ctr)[None, :])
    return (_shift(h, 32) < thr).double()


def _f(x):
    return float(np.float32(x))


def exact(case, seed):
    kind = case["kind"]
    if kind == "serve":      # whole numbers only
        return None
    b, steps = case["batch"], case["steps"]
    n = case["n_hid"] if kind == "rec" else case["n_exc"]
    # 64-bit products run at about a teraflop a second
    k = case["n_in"] + n if kind == "rec" else (3 if kind == "train" else 1) * case["n_in"]
    if 2.0 * b * n * k * steps > 1.2e13:
        return None
    with torch.no_grad():
        return _exact_rec(case, seed) if kind == "rec" else _exact_net(case, seed)


def _exact_rec(case, seed):
    wf, wr, wo = (w.double() for w in _rec_weights(case, seed))
    rates, seeds = _rates(case, case["batch"], seed), _seeds(case["batch"], seed)
    am, asyn = math.exp(-1.0 / REC["tau_mem"]), math.exp(-1.0 / REC["tau_syn"])
    v = torch.zeros((case["batch"], case["n_hid"]), device="cuda", dtype=torch.float64)
    cur, s, out = torch.zeros_like(v), torch.zeros_like(v), 0.0
    for t in range(case["steps"]):
        cur = asyn * cur + _draws(rates, seeds, t) @ wf + s @ wr
        v = am * v + cur
        s = (v >= REC["v_thresh"]).double()
        v = torch.where(s > 0, torch.full_like(v, REC["v_reset"]), v)
        out = out + s @ wo
    return {"v_out": out, "counts": None, "v": v}


def _current_weights(w, wprec):
    """The weights as the synaptic current reads them."""
    if wprec == "bf16":
        return w.float().bfloat16().double()
    if wprec == "fp8":       # per-column power-of-two scale, the smallest with 448 * scale >= the largest weight
        m = w.abs().amax(0)
        scale = torch.where(m > 0, torch.exp2(torch.ceil(torch.log2(m / 448.0))), torch.ones_like(m))
        return (w / scale).float().to(torch.float8_e4m3fn).double() * scale
    return w


def _exact_net(case, seed):
    p, b, n, reduce = _params(case), case["batch"], case["n_exc"], case["reduce"]
    learn, rule = case["kind"] == "train", case["net"] == "rule"
    if learn and reduce == "max" and b * case["n_in"] * n > 1 << 27:
        return None          # the per-sample updates of a step do not fit a quick evaluation
    rates, seeds = _rates(case, b, seed), _seeds(b, seed)
    w, theta = _weights(case, seed).double(), _theta(case, seed)
    a_e, a_i, a_x = (math.exp(-1.0 / p[k]) for k in ("e_tau", "i_tau", "trace_tau"))
    a_th = math.exp(-1.0 / p["theta_tau"])
    nu_pre, nu_post, plus = _f(p["nu_pre"]), _f(p["nu_post"]), _f(p["theta_plus"])
    v = torch.full((b, n), p["e_rest"], device="cuda", dtype=torch.float64)
    vi = torch.full_like(v, p["i_rest"])
    ref_e, ref_i = torch.zeros_like(v), torch.zeros_like(v)
    se, si, x_post = torch.zeros_like(v), torch.zeros_like(v), torch.zeros_like(v)
    x_pre = torch.zeros((b, case["n_in"]), device="cuda", dtype=torch.float64)
    wc = _current_weights(w, case["wprec"])
    for t in range(case["steps"]):
        s_in = _draws(rates, seeds, t)
        drive = s_in @ wc + p["w_ie"] * (si.sum(1, keepdim=True) - si)
        drive_i = p["w_ei"] * se
        v = p["e_rest"] + (v - p["e_rest"]) * a_e
        free = ref_e == 0
        v = torch.where(free, v + drive, v)
        se = (free & (v >= p["e_thresh"] + theta)).double()
        ref_e = torch.where(free, se * round(p["e_refrac"]), ref_e - 1)
        v = torch.where(se > 0, torch.full_like(v, p["e_reset"]), v)
        vi = p["i_rest"] + (vi - p["i_rest"]) * a_i
        free = ref_i == 0
        vi = torch.where(free, vi + drive_i, vi)
        si = (free & (vi >= p["i_thresh"])).double()
        ref_i = torch.where(free, si * round(p["i_refrac"]), ref_i - 1)
        vi = torch.where(si > 0, torch.full_like(vi, p["i_reset"]), vi)
        x_pre = x_pre * a_x + s_in
        x_post = x_post * a_x + se
        if not learn:
            continue
        if reduce == "max":
            d = nu_post * x_pre[:, :, None] * se[:, None, :]
            if not rule:
                d = d - nu_pre * s_in[:, :, None] * x_post[:, None, :]
            d = d.amax(0)
        else:
            d = nu_post * (x_pre.T @ se)
            if not rule:
                d = d - nu_pre * (s_in.T @ x_post)
            d = d / b if reduce == "mean" else d
        w = torch.clamp(w + d, _f(p["w_min"]), _f(p["w_max"]))
        fired = se.sum(0)
        if rule:
            total = w.sum(0)
            scale = torch.where((fired > 0) & (total != 0), _f(p["w_norm"]) / total, torch.ones_like(total))
            w = w * scale
        r = fired if reduce == "sum" else fired / b if reduce == "mean" else (fired > 0).double()
        theta = theta * a_th + plus * r
        wc = _current_weights(w, case["wprec"])
    out = {"counts": None, "v": v}
    return dict(out, w=w, theta=theta) if learn else out
