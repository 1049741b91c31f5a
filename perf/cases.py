"""The work that this framework's users have it do, as cases that can be prepared, run and timed.

Six kinds, each through a public entry point:

  fit     Signal2SH of an acquisition (a preprocessing step, no gradients): 2-D [features, voxels]
          or the paper's 5-D tensor [subjects, features, H, W, D]
  eval    SH2Signal inside a training step: the signal and the gradient of the coefficients
  gather  Signal2SH of a volume's masked voxels with the division by b0 in the load
  lsc     one local spherical convolution: forward, or forward and backward (the gradients of the
          weights, the bias and, unless the layer is a network's first, of its input)
  chain   Signal2SH -> LSC -> SH2Signal, forward and backward, on preallocated buffers
  net     one training step of the four-layer network up to the gradients
  volume  inference of one whole masked volume with that network

`listed()` are the sizes of the repository's own benchmark, network, volume runs and tests; `draw()`
gives others of the same ranges, odd sizes among them.
"""
import math

import numpy as np
import torch

from paper_1808_01517_gb300 import _lib as L
from paper_1808_01517_gb300 import layers, net, volume
from paper_1808_01517_gb300.chain import Chain, ChainConfig

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
LAM = 0.006
BVALS = (1000.0, 2000.0, 3000.0)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the smallest call: one shell of 60 directions, a slab of 1,000 voxels; latency counts
        dict(name="fit_small_f32", kind="fit", shells=1, dirs=60, order=8, channels=1, vox=1000, dtype="f32"),
        # the paper's whole scan (about 450,000 voxels) on 3 shells of 90 directions
        dict(name="fit_scan_f32", kind="fit", shells=3, dirs=90, order=8, channels=1, vox=450000, dtype="f32"),
        # a whole volume as the paper's 5-D tensor: an odd voxel count, rows on no 16-byte boundary
        dict(name="fit_volume_5d_f32", kind="fit", shells=1, dirs=30, order=4, channels=1, vox=0, height=145,
             width=174, depth=145, dtype="f32"),
        # the last step of a network under training: coefficients to signals and the gradient back
        dict(name="eval_train_f32", kind="eval", shells=3, dirs=90, order=8, channels=1, vox=262144, dtype="f32"),
        # volume inference's first step: one chunk of masked voxels of a raw 30-direction volume
        dict(name="gather_b0_bf16", kind="gather", dirs=30, order=4, height=145, width=174, depth=145, vox=262144,
             dtype="bf16"),
        # a single-shell layer on few voxels, forward and backward: launches and latency count
        dict(name="lsc_small_f32", kind="lsc", shells=1, shells_in=1, dirs=60, order_in=8, order=8, c_in=1, c_out=8,
             rings=3, sectors=8, radius=30.0, window="same", vox=1000, dtype="f32", train=True, d_input=True,
             ring_tied=False),
        # the network's first layer in a training step: 15 input rows, no gradient of the input
        dict(name="lsc_first_bf16", kind="lsc", shells=3, shells_in=1, dirs=90, order_in=4, order=8, c_in=1, c_out=64,
             rings=4, sectors=12, radius=25.0, window="all", vox=8192, dtype="bf16", train=True, d_input=False,
             ring_tied=False),
        # a hidden layer of the network in a training step at its batch size
        dict(name="lsc_hidden_bf16", kind="lsc", shells=3, shells_in=3, dirs=90, order_in=8, order=8, c_in=64,
             c_out=64, rings=4, sectors=12, radius=25.0, window="adjacent", vox=8192, dtype="bf16", train=True,
             d_input=True, ring_tied=False),
        # the accurate form of a multi-shell layer, a ragged number of voxels
        dict(name="lsc_train_f32", kind="lsc", shells=3, shells_in=3, dirs=90, order_in=8, order=8, c_in=16, c_out=64,
             rings=4, sectors=12, radius=25.0, window="adjacent", vox=16001, dtype="f32", train=True, d_input=True,
             ring_tied=False),
        # the benchmark's step: fit, convolve, evaluate, and back
        dict(name="chain_bf16", kind="chain", dirs=90, order=8, order_in=8, c_in=16, c_out=64, rings=4, sectors=12,
             radius=25.0, window="adjacent", vox=65536, dtype="bf16"),
        # one training step of the whole network at its batch size
        dict(name="net_train_bf16", kind="net", hidden=64, vox=8192, dtype="bf16"),
        # one subject of the whole-volume run
        dict(name="volume_bf16", kind="volume", hidden=64, height=145, width=174, depth=145, vox=900000,
             dtype="bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vox(rng, lo, hi):
    """A voxel count spread over the logarithm: any number, or one that keeps rows aligned."""
    n = _log_int(rng, lo, hi)
    return n if rng.random() < 0.5 else max(8, n // 8 * 8)


def draw(rng):
    kind = rng.choice(["fit", "eval", "gather", "lsc", "lsc", "lsc", "chain", "net", "volume"])
    dtype = rng.choice(["f32", "bf16"])
    if kind in ("fit", "eval"):
        c = dict(kind=kind, shells=rng.choice([1, 2, 3]), dirs=rng.randint(20, 100), order=rng.choice([4, 6, 8]),
                 channels=rng.choice([1, 1, 4, 16]), vox=0, dtype=dtype)
        if kind == "fit" and rng.random() < 0.3:
            c.update(channels=1, height=rng.randint(40, 110), width=rng.randint(40, 110), depth=rng.randint(40, 110))
        else:
            c["vox"] = _vox(rng, 500, 800000 // c["channels"])
        return c
    if kind == "gather":
        h, w, d = rng.randint(60, 145), rng.randint(60, 174), rng.randint(60, 145)
        return dict(kind=kind, dirs=rng.randint(20, 60), order=rng.choice([4, 6]), height=h, width=w, depth=d,
                    vox=min(_vox(rng, 2000, 400000), h * w * d // 2), dtype=dtype)
    if kind == "lsc":
        shells, window = rng.choice([1, 2, 3]), rng.choice(["same", "adjacent", "all"])
        c = dict(kind=kind, shells=shells, shells_in=rng.choice([1, shells]) if window == "all" else shells,
                 dirs=rng.randint(30, 90), order_in=rng.choice([4, 6, 8]), order=rng.choice([4, 6, 8]),
                 c_in=rng.choice([1, 2, 4, 5, 8, 16, 24, 32, 64]), c_out=rng.choice([1, 4, 7, 8, 16, 32, 48, 64]),
                 rings=rng.randint(1, 4), sectors=rng.choice([5, 6, 8, 12]), radius=float(rng.randint(15, 36)),
                 window=window, vox=_vox(rng, 250, 32768), dtype=dtype, train=rng.random() < 0.7, d_input=True,
                 ring_tied=rng.random() < 0.2)
        # as much work as a layer of the benchmark's step, at most
        most = (4e12 if dtype == "bf16" else 6e11) / (work(c)["flops"] / c["vox"])
        c["vox"] = int(max(64, min(c["vox"], most)))
        return c
    if kind == "chain":
        return dict(kind=kind, dirs=rng.randint(45, 96), order=8, order_in=rng.choice([4, 8]),
                    c_in=rng.choice([4, 8, 16]), c_out=rng.choice([8, 16, 32, 64]), rings=rng.randint(2, 4),
                    sectors=rng.choice([6, 8, 12]), radius=25.0, window=rng.choice(["adjacent", "all"]),
                    vox=_vox(rng, 1000, 65000 if dtype == "bf16" else 16000), dtype=dtype)
    if kind == "net":
        return dict(kind=kind, hidden=rng.choice([16, 24, 32, 48, 64]), vox=_vox(rng, 256, 12000), dtype="bf16")
    h, w, d = rng.randint(60, 130), rng.randint(60, 150), rng.randint(60, 130)
    return dict(kind=kind, hidden=rng.choice([16, 32, 64]), height=h, width=w, depth=d,
                vox=_log_int(rng, 20000, h * w * d // 3), dtype="bf16")


# ---------------------------------------------------------------------------
# inputs: gradient tables, signals, coefficients, gradients and weights, from the seed alone
# ---------------------------------------------------------------------------
def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _gen(seed, purpose):
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed) * 1009 + purpose)
    return g


def _table(n_shells, dirs, seed):
    """Directions (one independent set per shell, on the upper hemisphere) and b-values, by shell."""
    r = np.random.default_rng([int(seed), 17])
    g = r.standard_normal((n_shells * dirs, 3))
    g /= np.linalg.norm(g, axis=1, keepdims=True)
    g[g[:, 2] < 0] *= -1.0
    return g, np.repeat(np.asarray(BVALS[:n_shells]), dirs)


def _signals(g, b, channels, vox, seed, dtype):
    """Stick + zeppelin signals of two crossing fibres with Rician noise at SNR 20, rows (shell,
    channel, direction)."""
    gen, dev = _gen(seed, 1), _dev()
    n = channels * vox
    gt = torch.as_tensor(g, dtype=torch.float32, device=dev)
    bt = torch.as_tensor(b, dtype=torch.float32, device=dev)[:, None]
    f = torch.rand((1, n), generator=gen, device=dev)
    s = torch.zeros((g.shape[0], n), device=dev)
    for k in range(2):
        u = torch.randn((3, n), generator=gen, device=dev)
        c2 = (gt @ (u / u.norm(dim=0, keepdim=True))) ** 2
        part = 0.65 * torch.exp(-1.7e-3 * bt * c2) + 0.35 * torch.exp(-bt * (0.3e-3 + 1.4e-3 * c2))
        s += (f if k == 0 else 1.0 - f) * part
    s = torch.sqrt((s + 0.05 * torch.randn(s.shape, generator=gen, device=dev)) ** 2
                   + (0.05 * torch.randn(s.shape, generator=gen, device=dev)) ** 2).to(dtype)
    m = g.shape[0] // len(np.unique(b))
    if channels == 1:
        return s
    s = s.reshape(-1, m, channels, vox).transpose(1, 2)  # (shell, channel, direction, voxel)
    return s.reshape(-1, vox)


def _lsizes(order):
    return np.array([l for l in range(0, order + 1, 2) for _ in range(2 * l + 1)])


def _coeffs(blocks, order, vox, seed, purpose, std, dtype):
    """Coefficient rows (shell, channel, coefficient): Gaussian, falling with the degree as those of
    smooth functions do; `blocks` = shells x channels."""
    fall = torch.as_tensor(1.0 / (1.0 + _lsizes(order)) ** 1.5, dtype=torch.float32, device=_dev())
    x = torch.randn((blocks, fall.numel(), vox), generator=_gen(seed, purpose), device=_dev())
    return _act((x * (std * fall)[None, :, None]).reshape(-1, vox).to(dtype))


def _act(x):
    """Rows at the library's padded stride, as activations are that its layers made."""
    return layers.as_act(x)


def _weights(case, seed, purpose, c_in, c_out, s_in, s_out, K, window):
    """He-scaled kernel weights (zero outside the window) and small biases."""
    fan = c_in * (1 if window == "same" or s_in == 1 else s_in) * K
    w = torch.randn((c_out, s_out, c_in, s_in, K), generator=_gen(seed, purpose), device=_dev())
    w *= math.sqrt(2.0 / fan)
    w *= torch.as_tensor(_window(s_out, s_in, window), dtype=w.dtype, device=w.device)[None, :, None, :, None]
    b = 0.1 * torch.randn((c_out, s_out), generator=_gen(seed, purpose + 1), device=_dev())
    return w, b


def _window(s_out, s_in, mode):
    d = np.abs(np.arange(s_out)[:, None] - np.arange(s_in)[None, :])
    return np.ones((s_out, s_in), bool) if mode == "all" else d <= (0 if mode == "same" else 1)


def _points(case):
    return 1 + (case["rings"] if case.get("ring_tied") else case["rings"] * case["sectors"])


def _voxels(case):
    return case["height"] * case["width"] * case["depth"] if case.get("height") else case["vox"]


GRAD_STD = 1e-4  # upstream gradients of a loss averaged over a batch


def _inputs(case, seed):
    """Everything that a case computes from, as tensors on the device: what run() and exact() share."""
    kind, dt = case["kind"], DTYPES[case["dtype"]]
    d = {}
    if kind == "fit":
        d["g"], d["b"] = _table(case["shells"], case["dirs"], seed)
        x = _signals(d["g"], d["b"], case["channels"], _voxels(case), seed, dt)
        if case.get("height"):  # one subject's volume, contiguous
            x = x.reshape(1, x.shape[0], case["height"], case["width"], case["depth"])
        else:
            x = _act(x)
        d["x"] = x
    elif kind == "eval":
        d["g"], d["b"] = _table(case["shells"], case["dirs"], seed)
        d["x"] = _coeffs(case["shells"] * case["channels"], case["order"], case["vox"], seed, 2, 0.5, dt)
        gy = torch.randn((case["channels"] * d["g"].shape[0], case["vox"]), generator=_gen(seed, 3), device=_dev())
        d["gy"] = _act((GRAD_STD * gy).to(dt))
    elif kind == "gather":
        d["g"], d["b"] = _table(1, case["dirs"], seed)
        n, k = _voxels(case), case["vox"]
        gen = _gen(seed, 4)
        # the mask: a solid body in the middle of the volume, its voxels in C order
        axes = [torch.linspace(-1, 1, s, device=_dev()) for s in (case["height"], case["width"], case["depth"])]
        r = sum(a ** 2 for a in torch.meshgrid(*axes, indexing="ij")).reshape(-1)
        d["index"] = torch.sort(torch.topk(r, k, largest=False).indices).values
        d["b0"] = 1000.0 * (1.2 - 0.3 * r + 0.01 * torch.randn(n, generator=gen, device=_dev()))
        dwi = torch.zeros((case["dirs"], n), dtype=dt, device=_dev())
        dwi[:, d["index"]] = (_signals(d["g"], d["b"], 1, k, seed, torch.float32) * d["b0"][d["index"]]).to(dt)
        d["dwi"] = dwi
    elif kind == "lsc":
        d["g"], d["b"] = _table(case["shells"], case["dirs"], seed)
        K = _points(case)
        d["w"], d["bias"] = _weights(case, seed, 5, case["c_in"], case["c_out"], case["shells_in"], case["shells"], K,
                                     case["window"])
        d["x"] = _coeffs(case["shells_in"] * case["c_in"], case["order_in"], case["vox"], seed, 2, 1.0, dt)
        if case["train"]:
            d["gy"] = _coeffs(case["shells"] * case["c_out"], case["order"], case["vox"], seed, 3, GRAD_STD, dt)
    elif kind == "chain":
        d["g"], d["b"] = _table(3, case["dirs"], seed)
        d["w"], d["bias"] = _weights(case, seed, 5, case["c_in"], case["c_out"], 3, 3, _points(case), case["window"])
        d["x"] = _signals(d["g"], d["b"], case["c_in"], case["vox"], seed, dt)
        gy = torch.randn((case["c_out"] * d["g"].shape[0], case["vox"]), generator=_gen(seed, 3), device=_dev())
        d["gy"] = (GRAD_STD * gy).to(dt)
    elif kind == "net":
        cfg = net.NetConfig(hidden=case["hidden"])
        d["g"], d["b"] = _table(3, cfg.dirs_per_shell[0], seed)
        d["sel"] = np.sort(np.random.default_rng([int(seed), 19]).choice(cfg.dirs_per_shell[0], cfg.n_in_dirs,
                                                                         replace=False))
        clean = _signals(d["g"], d["b"], 1, case["vox"], seed, torch.float32)
        d["x"], d["y"] = clean[torch.as_tensor(d["sel"], device=clean.device)].to(dt), clean.to(dt)
        K = 1 + cfg.rings * cfg.sectors
        ch = [1] + [cfg.hidden] * (cfg.n_lsc - 1) + [1]
        d["params"] = [_weights(case, seed, 10 + 2 * i, ch[i], ch[i + 1], 1 if i == 0 else 3, 3, K,
                                "all" if i == 0 else "adjacent") for i in range(cfg.n_lsc)]
        d["cfg"] = cfg
    return d


def prepare(case, seed):
    kind = case["kind"]
    if kind == "volume":
        cfg = net.NetConfig(hidden=case["hidden"], seed=1808 + int(seed))
        dirs, bvals, sel = net.tables(cfg)
        weights = net.SphericalNet(cfg, dirs[sel], dirs, bvals).state_dict()
        sb = volume.Subject(0, cfg, weights, shape=(case["height"], case["width"], case["depth"]),
                            mask_voxels=case["vox"], seed=1808 + int(seed))
        return dict(kind=kind, subject=sb)
    d = _inputs(case, seed)
    s = dict(kind=kind, case=case)
    if kind == "fit":
        s.update(x=d["x"], layer=layers.Signal2SH(case["order"], d["g"], LAM, bvals=d["b"], channels=case["channels"]))
    elif kind == "eval":
        # the loss's own gradient has run on the backward thread before this layer's does
        torch.ones(1, device=_dev(), requires_grad=True).square().backward()
        s.update(x=d["x"].requires_grad_(), gy=d["gy"],
                 layer=layers.SH2Signal(case["order"], d["g"], bvals=d["b"], channels=case["channels"]))
    elif kind == "gather":
        s.update(dwi=d["dwi"], index=d["index"], b0=d["b0"], basis=L.SHBasis(d["g"], d["b"], case["order"], LAM))
    elif kind == "lsc":
        layer = layers.LocalSphericalConvolution(
            case["shells_in"], case["shells"], d["g"], case["order_in"], case["order"],
            [case["sectors"]] * case["rings"], LAM, math.radians(case["radius"]), d["b"], case["c_in"], case["c_out"],
            case["window"], ring_tied=case["ring_tied"]).cuda()
        with torch.no_grad():
            layer.weight.copy_(d["w"])
            layer.bias.copy_(d["bias"])
        x = d["x"].requires_grad_(case["train"] and case["d_input"])
        s.update(layer=layer, x=x, gy=d.get("gy"))
    elif kind == "chain":
        cfg = ChainConfig(n_vox=case["vox"], dirs_per_shell=(case["dirs"],) * 3, bvals=BVALS, order=case["order"],
                          lam=LAM, c_in=case["c_in"], c_out=case["c_out"], radius_deg=case["radius"],
                          rings=case["rings"], sectors=case["sectors"], window=case["window"],
                          order_in=case["order_in"])
        ch = Chain(cfg, d["g"], d["b"], DTYPES[case["dtype"]])
        ch.set_inputs(d["x"], d["gy"], d["w"], d["bias"])
        s.update(chain=ch)
    else:
        model = net.SphericalNet(d["cfg"], d["g"][d["sel"]], d["g"], d["b"], DTYPES[case["dtype"]]).cuda()
        with torch.no_grad():
            for lsc, (w, b) in zip(model.lscs, d["params"]):
                lsc.weight.copy_(w)
                lsc.bias.copy_(b)
        s.update(model=model, x=d["x"], y=d["y"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "fit":
        with torch.no_grad():
            return {"sh": s["layer"](s["x"])}
    if kind == "eval":
        y = s["layer"](s["x"])
        (dx,) = torch.autograd.grad(y, s["x"], s["gy"])
        return {"signal": y, "d_sh": dx}
    if kind == "gather":
        return {"sh": layers.signal2sh_gather(s["basis"], s["dwi"], s["index"], b0=s["b0"])}
    if kind == "lsc":
        layer, x = s["layer"], s["x"]
        if not s["case"]["train"]:
            with torch.no_grad():
                return {"sh": layer(x)}
        y = layer(x)
        wrt = [layer.weight, layer.bias] + ([x] if x.requires_grad else [])
        grads = torch.autograd.grad(y, wrt, s["gy"])
        return dict(zip(("sh", "d_weight", "d_bias", "d_sh"), (y,) + grads))
    if kind == "chain":
        ch = s["chain"]
        ch.step()
        return {"signal": ch.s_out, "d_signal": ch.ds_in, "d_weight": ch.dw, "d_bias": ch.db}
    if kind == "net":
        model = s["model"]
        pred = model(s["x"])
        loss = torch.mean((pred.float() - s["y"].float()) ** 2)
        grads = torch.autograd.grad(loss, list(model.parameters()))
        return {"signal": pred, "loss": loss, "grads": list(grads)}
    outs, _, _ = volume.run([s["subject"]])
    return {"signal": outs[0]}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _n(order):
    return (order + 1) * (order + 2) // 2


def _lsc_work(vox, e, s_in, s_out, c_in, c_out, n_in, n_out, K, window, train, d_input):
    """(bytes, flops): activations and weights once each; the collapsed operator's build, the
    products over the voxels and the weight gradient's way back to the kernel points."""
    pairs = int(_window(s_out, s_in, window).sum())
    rows_in, rows_out, nw = s_in * c_in * n_in, s_out * c_out * n_out, c_out * s_out * c_in * s_in * K
    gemm = 2.0 * pairs * c_out * n_out * c_in * n_in * vox
    side = 2.0 * pairs * c_out * c_in * n_out * n_in * K
    by, fl = e * vox * (rows_in + rows_out) + 4.0 * nw, gemm + side
    if train:
        by += e * vox * (rows_out + (rows_in if d_input else 0)) + 4.0 * nw
        fl += gemm * (2 if d_input else 1) + side
    return by, fl


def work(case):
    kind, e = case["kind"], DTYPES[case["dtype"]].itemsize
    if kind in ("fit", "eval"):
        N, v = _n(case["order"]), _voxels(case) * case["channels"] * case["shells"]
        passes = 2 if kind == "eval" else 1
        return {"bytes": passes * e * v * (case["dirs"] + N), "flops": passes * 2.0 * v * case["dirs"] * N}
    if kind == "gather":
        v, N = case["vox"], _n(case["order"])
        return {"bytes": v * (e * (case["dirs"] + N) + 12.0), "flops": 2.0 * v * case["dirs"] * N}
    if kind == "lsc":
        by, fl = _lsc_work(case["vox"], e, case["shells_in"], case["shells"], case["c_in"], case["c_out"],
                           _n(case["order_in"]), _n(case["order"]), _points(case), case["window"], case["train"],
                           case["d_input"])
        return {"bytes": by, "flops": fl}
    if kind == "chain":
        v, Ni, No, m = case["vox"], _n(case["order_in"]), _n(case["order"]), 3 * case["dirs"]
        _, fl = _lsc_work(v, e, 3, 3, case["c_in"], case["c_out"], Ni, No, _points(case), case["window"], True, True)
        # s_in, ds_out and the weights in, s_out, ds_in and the gradients out
        by = 2.0 * e * v * m * (case["c_in"] + case["c_out"]) + 8.0 * 9 * case["c_in"] * case["c_out"] * _points(case)
        return {"bytes": by, "flops": fl + 4.0 * v * m * (case["c_in"] * Ni + case["c_out"] * No)}
    cfg = net.NetConfig(hidden=case["hidden"])
    v, train = case["vox"], kind == "net"
    ch = [1] + [cfg.hidden] * (cfg.n_lsc - 1) + [1]
    K, fl, nw = 1 + cfg.rings * cfg.sectors, 0.0, 0
    for i in range(cfg.n_lsc):
        s_in = 1 if i == 0 else 3
        fl += _lsc_work(v, e, s_in, 3, ch[i], ch[i + 1], _n(4) if i == 0 else _n(8), _n(8), K,
                        "all" if i == 0 else "adjacent", train, i > 0)[1]
        nw += 3 * s_in * ch[i] * ch[i + 1] * K
    fl += 2.0 * v * 30 * _n(4) + (4.0 if train else 2.0) * v * 270 * _n(8)
    if train:
        return {"bytes": e * v * (30.0 + 2 * 270) + 8.0 * nw, "flops": fl}
    # the masked signal and b0, the mask, the dense volume (written whole) and the weights
    n = _voxels(case)
    return {"bytes": v * (30.0 * e + 4) + n + 270.0 * e * n + 4.0 * nw, "flops": fl}


# ---------------------------------------------------------------------------
# the same results in 64 bits: the definitions, in numpy and torch
# ---------------------------------------------------------------------------
def _basis(order, dirs):
    """Real symmetric even-order SH at unit vectors: j = l(l+1)/2 + m, sqrt(2) Re Y_l^|m| for m < 0,
    Y_l^0, sqrt(2) Im Y_l^m for m > 0, with the Condon-Shortley phase."""
    x, y, z = np.moveaxis(np.asarray(dirs, np.float64), -1, 0)
    phi, sin = np.arctan2(y, x), np.sqrt(np.clip(1.0 - z * z, 0.0, None))
    out = np.empty(z.shape + (_n(order),))
    pmm = np.full_like(z, math.sqrt(1.0 / (4.0 * math.pi)))  # normalised P_m^m, by recurrence in m
    for m in range(order + 1):
        if m:
            pmm = -math.sqrt((2 * m + 1) / (2.0 * m)) * sin * pmm
        below, cur = np.zeros_like(z), pmm
        for l in range(m, order + 1):
            if l > m:
                a = math.sqrt((4.0 * l * l - 1) / (l * l - m * m))
                c = math.sqrt(((l - 1.0) ** 2 - m * m) / (4 * (l - 1.0) ** 2 - 1)) if l > m + 1 else 0.0
                below, cur = cur, a * (z * cur - c * below)
            if l % 2 == 0:
                j = l * (l + 1) // 2
                out[..., j + m] = cur if m == 0 else math.sqrt(2.0) * np.sin(m * phi) * cur
                if m:
                    out[..., j - m] = math.sqrt(2.0) * np.cos(m * phi) * cur
    return out


def _fit(order, dirs):
    B, l = _basis(order, dirs), _lsizes(order)
    return np.linalg.solve(B.T @ B + LAM * np.diag((l * (l + 1.0)) ** 2), B.T)


def _kernel_points(g, radius, rings, sectors):
    """[directions, points, 3]: the direction, then each ring's points in its tangent frame."""
    a = np.eye(3)[np.argmin(np.abs(g), axis=1)]
    e1 = a - np.sum(a * g, 1, keepdims=True) * g
    e1 /= np.linalg.norm(e1, axis=1, keepdims=True)
    e2 = np.cross(g, e1)
    pts = [g]
    for r in range(1, rings + 1):
        for q in range(sectors):
            t, p = r * radius / rings, 2 * math.pi * q / sectors
            pts.append(math.cos(t) * g + math.sin(t) * (math.cos(p) * e1 + math.sin(p) * e2))
    return np.stack(pts, 1)


def _f64(a):
    return torch.as_tensor(a, device=_dev()).double()


class _Lsc64:
    """The layer in 64 bits through its exact collapse: one matrix per pair of shells."""

    def __init__(self, g, s_out, order_in, order, radius, rings, sectors, window, s_in):
        m = g.shape[0] // s_out
        self.win, self.s_in, self.s_out = _window(s_out, s_in, window), s_in, s_out
        self.M, self.q = [], []
        for s in range(s_out):
            gs = g[s * m:(s + 1) * m]
            P = _fit(order, gs)
            BK = _basis(order_in, _kernel_points(gs, radius, rings, sectors))
            self.M.append(_f64(np.einsum("ai,ikb->kab", P, BK)))
            self.q.append(_f64(P.sum(1)))

    def _op(self, w, s, p):
        co, ci, (_, a, b) = w.shape[0], w.shape[2], self.M[s].shape
        W = w[:, s, :, p].reshape(co * ci, -1) @ self.M[s].reshape(-1, a * b)
        return W.reshape(co, ci, a, b).transpose(1, 2).reshape(co * a, ci * b)

    def forward(self, x, w, bias):
        xs = x.reshape(self.s_in, -1, x.shape[1])
        out = []
        for s in range(self.s_out):
            y = (bias[:, s, None] * self.q[s]).reshape(-1, 1).expand(-1, x.shape[1]).clone()
            for p in np.flatnonzero(self.win[s]):
                y.addmm_(self._op(w, s, p), xs[p])
            out.append(y)
        return torch.cat(out)

    def backward(self, x, w, gy, d_input=True):
        xs, gs = x.reshape(self.s_in, -1, x.shape[1]), gy.reshape(self.s_out, -1, x.shape[1])
        dx, dw = torch.zeros_like(xs) if d_input else None, torch.zeros_like(w)
        db = torch.empty((w.shape[0], self.s_out), dtype=w.dtype, device=w.device)
        for s in range(self.s_out):
            K, a, b = self.M[s].shape
            co, ci = w.shape[0], w.shape[2]
            db[:, s] = gs[s].sum(1).reshape(co, a) @ self.q[s]
            for p in np.flatnonzero(self.win[s]):
                if d_input:
                    dx[p].addmm_(self._op(w, s, p).T, gs[s])
                G = (gs[s] @ xs[p].T).reshape(co, a, ci, b).transpose(1, 2).reshape(co * ci, a * b)
                dw[:, s, :, p] = (G @ self.M[s].reshape(K, -1).T).reshape(co, ci, K)
        return dx.reshape(x.shape) if d_input else None, dw, db


def _per_shell(mats, x, channels, n_in):
    """mats[s] applied to every channel's n_in rows of shell s."""
    xs = x.reshape(len(mats), channels, n_in, x.shape[1])
    return torch.cat([torch.matmul(_f64(T), xs[s]).reshape(-1, x.shape[1]) for s, T in enumerate(mats)])


def _shells(g, n):
    return np.split(g, n)


def _expand(w, rings, sectors):
    return torch.cat([w[..., :1]] + [w[..., r:r + 1].expand(w.shape[:-1] + (sectors,)) for r in range(1, rings + 1)], -1)


def _fold(dw, rings, sectors):
    return torch.cat([dw[..., :1], dw[..., 1:].reshape(dw.shape[:-1] + (rings, sectors)).sum(-1)], -1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "volume":
        return None  # four layers over a whole brain: minutes in 64 bits
    d = _inputs(case, seed)
    if kind == "fit":
        x = d["x"].double()
        mats = [_fit(case["order"], g) for g in _shells(d["g"], case["shells"])]
        if case.get("height"):
            y = _per_shell(mats, x.reshape(x.shape[1], -1), 1, case["dirs"])
            return {"sh": y.reshape((1, y.shape[0]) + tuple(x.shape[2:]))}
        return {"sh": _per_shell(mats, x, case["channels"], case["dirs"])}
    if kind == "eval":
        mats = [_basis(case["order"], g) for g in _shells(d["g"], case["shells"])]
        return {"signal": _per_shell(mats, d["x"].double(), case["channels"], _n(case["order"])),
                "d_sh": _per_shell([T.T for T in mats], d["gy"].double(), case["channels"], case["dirs"])}
    if kind == "gather":
        x = d["dwi"][:, d["index"]].double() / d["b0"][d["index"]].double()
        return {"sh": _per_shell([_fit(case["order"], d["g"])], x, 1, case["dirs"])}
    if kind == "lsc":
        lsc = _Lsc64(d["g"], case["shells"], case["order_in"], case["order"], math.radians(case["radius"]),
                     case["rings"], case["sectors"], case["window"], case["shells_in"])
        x, w, tied = d["x"].double(), d["w"].double(), case["ring_tied"]
        w = _expand(w, case["rings"], case["sectors"]) if tied else w
        out = {"sh": lsc.forward(x, w, d["bias"].double())}
        if case["train"]:
            dx, dw, db = lsc.backward(x, w, d["gy"].double(), case["d_input"])
            out.update(d_weight=_fold(dw, case["rings"], case["sectors"]) if tied else dw, d_bias=db)
            if case["d_input"]:
                out["d_sh"] = dx
        return out
    if kind == "chain":
        gs, ci, co, m = _shells(d["g"], 3), case["c_in"], case["c_out"], case["dirs"]
        P, B = [_fit(case["order_in"], g) for g in gs], [_basis(case["order"], g) for g in gs]
        lsc = _Lsc64(d["g"], 3, case["order_in"], case["order"], math.radians(case["radius"]), case["rings"],
                     case["sectors"], case["window"], 3)
        w = d["w"].double()
        c = _per_shell(P, d["x"].double(), ci, m)
        signal = _per_shell(B, lsc.forward(c, w, d["bias"].double()), co, _n(case["order"]))
        dc, dw, db = lsc.backward(c, w, _per_shell([T.T for T in B], d["gy"].double(), co, m))
        return {"signal": signal, "d_signal": _per_shell([T.T for T in P], dc, ci, _n(case["order_in"])),
                "d_weight": dw, "d_bias": db}
    cfg, gs = d["cfg"], _shells(d["g"], 3)
    args = (cfg.order, math.radians(cfg.radius_deg), cfg.rings, cfg.sectors)
    lscs = [_Lsc64(d["g"], 3, cfg.order_in if i == 0 else cfg.order, *args, "all" if i == 0 else "adjacent",
                   1 if i == 0 else 3) for i in range(cfg.n_lsc)]
    params = [(w.double(), b.double()) for w, b in d["params"]]
    B = [_basis(cfg.order, g) for g in gs]
    hs, h = [], _per_shell([_fit(cfg.order_in, d["g"][d["sel"]])], d["x"].double(), 1, cfg.n_in_dirs)
    for i, (lsc, (w, b)) in enumerate(zip(lscs, params)):
        hs.append(h)
        h = lsc.forward(h, w, b)
        if i < cfg.n_lsc - 1:
            h = torch.where(h > 0, h, cfg.slope * h)
    pred = _per_shell(B, h, 1, _n(cfg.order))
    diff = pred - d["y"].double()
    gh = _per_shell([T.T for T in B], 2.0 * diff / diff.numel(), 1, cfg.dirs_per_shell[0])
    grads = []
    for i in reversed(range(cfg.n_lsc)):
        gx, dw, db = lscs[i].backward(hs[i], params[i][0], gh, i > 0)
        grads = [dw, db] + grads
        if i > 0:
            gh = torch.where(hs[i] > 0, gx, cfg.slope * gx)
    return {"signal": pred, "loss": torch.mean(diff ** 2), "grads": grads}
