"""Timed workloads of the denoiser, through the package's public entry points.

A case names one of the ways a program uses the library:

* ``single``  one image in device memory, ``Denoiser.denoise``;
* ``host``    one image in ordinary host memory, ``Denoiser.denoise``;
* ``batch``   images of mixed sizes in device memory, one ``denoise_batch``;
* ``serve``   a burst of requests (device images) through ``Server``;
* ``predict`` the k estimate of a batch of images, ``Denoiser.predict_k``;
* ``fit``     some epochs of fitting the k estimator (forward, input and
  weight gradients, optimiser), ``Denoiser.train_predictor``.

The images follow the recipe of ``synth.py`` (Gaussian bumps and a gradient,
optionally a texture and bounded noise, then salt-and-pepper impulses), drawn
on the GPU.  Denoising works in place, so a pass first copies the noisy image
over the working copy - the place of a decoder or a camera that fills it - and
then makes the call.
"""
import math
import os

import numpy as np
import torch

from paper_1306_5390_gb300 import hgrms

_PHOTO = (321, 481)  # one of the two shapes of the photographs the method is published with
_MASK64 = (1 << 64) - 1


def listed():
    return [
        # The latency of one small picture (the bench's 256 x 256 workload).
        dict(name="single_256_b1", kind="single", rows=256, cols=256, density=0.10, alpha=10, beta=1, max_k=32,
             texture=False),
        # One photograph from ordinary host memory with the published fixed iteration factor, k = 5.
        dict(name="host_photo_k5", kind="host", rows=321, cols=481, density=0.20, alpha=10, beta=1, max_k=5,
             texture=True),
        # An HD frame with the wider window the sweep uses.
        dict(name="single_hd_b2", kind="single", rows=1080, cols=1920, density=0.20, alpha=10, beta=2, max_k=32,
             texture=True),
        # A 4K-sized crop of odd width, 7 x 7 windows, the sweep's largest tolerance.
        dict(name="single_uhd_odd_b3", kind="single", rows=2161, cols=3839, density=0.30, alpha=20, beta=3, max_k=32,
             texture=False),
        # A window beyond the tuned ones (the interface takes beta up to 7), on the sparse noise that such windows suit:
        # with more, nearly every impulse has its like in the window and nothing is replaced.
        dict(name="single_wide_b5", kind="single", rows=1000, cols=1500, density=0.02, alpha=10, beta=5, max_k=32,
             texture=False),
        # The bench's large image, two of its windows.
        dict(name="single_8192_b1", kind="single", rows=8192, cols=8192, density=0.30, alpha=10, beta=1, max_k=32,
             texture=False),
        dict(name="single_8192_b2", kind="single", rows=8192, cols=8192, density=0.30, alpha=10, beta=2, max_k=32,
             texture=False),
        # The 64 photographs of one setting of the noise sweep (half of them upright).
        dict(name="batch_photos_64", kind="batch", n=64, lo=0, hi=0, dmin=0.50, dmax=0.50, alpha=10, beta=1, max_k=32,
             texture=True),
        # A quarter of the bench's uneven batch: sides 128..2048, impulses 5..70 %.
        dict(name="batch_uneven_128", kind="batch", n=128, lo=128, hi=2048, dmin=0.05, dmax=0.70, alpha=10, beta=1,
             max_k=32, texture=False),
        # A burst of requests of the serving workload (square images 256..4096, beta 1 or 2).
        dict(name="serve_burst_24", kind="serve", n=24, lo=256, hi=4096, dmin=0.05, dmax=0.80, alpha=10, beta=0,
             max_k=32, texture=False),
        # The estimate of k for a part of the uneven batch.
        dict(name="predict_64", kind="predict", n=64, lo=128, hi=2048, dmin=0.05, dmax=0.70, beta=1, texture=False),
        # Two epochs of fitting the estimator with the shipped fit's minibatch.
        dict(name="fit_1024", kind="fit", n=1024, batch=256, epochs=2),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["single"] * 5 + ["host"] + ["batch"] * 2 + ["serve", "predict", "fit"])
    texture = rng.random() < 0.4
    if kind in ("single", "host"):
        beta = rng.choice([1, 1, 1, 2, 2, 3, 3, 4, 5, 7])
        most = 2e6 if kind == "host" else {1: 67e6, 2: 40e6, 3: 16e6}.get(beta, 1.5e6)
        px = math.exp(rng.uniform(math.log(3e4), math.log(most)))
        aspect = math.exp(rng.uniform(-0.9, 0.9))
        rows, cols = max(40, int(math.sqrt(px * aspect))), max(40, int(math.sqrt(px / aspect)))
        if rng.random() < 0.4:
            cols = cols // 16 * 16
        density = rng.uniform(0.05, 0.70) if beta <= 3 else rng.uniform(0.005, 0.10)
        return dict(kind=kind, rows=rows, cols=cols, density=round(density, 3),
                    alpha=rng.choice([5, 10, 10, 20]), beta=beta, max_k=rng.choice([5, 16, 32, 32]), texture=texture)
    dmin = round(rng.uniform(0.05, 0.40), 3)
    many = dict(dmin=dmin, dmax=round(dmin + rng.uniform(0.0, 0.30), 3), texture=texture)
    if kind == "batch":
        photos = rng.random() < 0.5
        return dict(kind=kind, n=_log_uniform(rng, 2, 64 if photos else 100), lo=0 if photos else rng.randint(100, 300),
                    hi=0 if photos else rng.randint(900, 2048), alpha=rng.choice([5, 10, 20]),
                    beta=rng.choice([1, 1, 2]) if photos else 1, max_k=rng.choice([8, 32]), **many)
    if kind == "serve":
        return dict(kind=kind, n=rng.randint(4, 20), lo=256, hi=rng.randint(700, 4000), alpha=10,
                    beta=rng.choice([0, 1, 2]), max_k=32, **many)
    if kind == "predict":
        return dict(kind=kind, n=_log_uniform(rng, 2, 60), lo=rng.randint(100, 300), hi=rng.randint(900, 2048), beta=1,
                    **many)
    batch = rng.choice([64, 128, 200, 256])
    return dict(kind="fit", n=batch * rng.randint(1, 3) + rng.randint(0, 40), batch=batch, epochs=rng.randint(1, 2))


# ---- Inputs ----------------------------------------------------------------

def _fields(n, rows, cols, rng):
    """n smooth fields in [20, 235] (float32, CUDA): 8 Gaussian bumps and a gradient each."""
    m, span = float(min(rows, cols)), float(max(rows, cols, 2) - 1)

    def t(a):
        return torch.tensor(np.asarray(a, dtype=np.float32), device="cuda")
    cy, cx = t(rng.uniform(0, rows, (n, 8, 1))), t(rng.uniform(0, cols, (n, 8, 1)))
    sig, amp = t(rng.uniform(0.05, 0.3, (n, 8, 1)) * m), t(rng.uniform(-1.0, 1.0, (n, 8, 1)))
    theta, gamp = rng.uniform(0.0, 2.0 * np.pi, (n, 1, 1)), rng.uniform(0.0, 1.0, (n, 1, 1))
    y, x = torch.arange(rows, device="cuda").float(), torch.arange(cols, device="cuda").float()
    gy = amp * torch.exp(-(y - cy) ** 2 / (2.0 * sig ** 2))
    gx = torch.exp(-(x - cx) ** 2 / (2.0 * sig ** 2))
    f = torch.bmm(gy.transpose(1, 2), gx)
    f += (t(gamp * np.cos(theta)) * (x / span)) + (t(gamp * np.sin(theta)) * (y / span)[:, None])
    lo, hi = f.amin(dim=(1, 2), keepdim=True), f.amax(dim=(1, 2), keepdim=True)
    return (f - lo) * (215.0 / (hi - lo).clamp_min(1e-6)) + 20.0


def _noisy(rows, cols, density, texture, rng, gen, n=1):
    """[n, rows, cols] uint8 images with impulses (density: a number, or n of them)."""
    f = _fields(n, rows, cols, rng)
    if texture:  # four plane sinusoids and integer noise in [-8, 8]
        y = torch.arange(rows, device="cuda").float()[:, None]
        x = torch.arange(cols, device="cuda").float()
        f = (f - 20.0) * (203.0 / 215.0) + 26.0
        for _ in range(4):
            per, ang, ph = rng.uniform(4.0, 32.0), rng.uniform(0.0, 2.0 * np.pi), rng.uniform(0.0, 2.0 * np.pi)
            f += 1.5 * torch.sin(2.0 * np.pi / per * (math.cos(ang) * x + math.sin(ang) * y) + ph)
        f = f.round_() + torch.randint(-8, 9, f.shape, device="cuda", generator=gen)
    img = f.round_().clamp_(0, 255).to(torch.uint8)
    del f
    u = torch.rand(img.shape, device="cuda", generator=gen)
    d = torch.as_tensor(np.asarray(density, dtype=np.float32), device="cuda").reshape(-1, 1, 1)
    img[u < 0.5 * d] = 0
    img[(u >= 0.5 * d) & (u < d)] = 255
    return img


def _draws(seed):
    return np.random.default_rng(seed), torch.Generator(device="cuda").manual_seed(int(seed))


def _shapes(case):
    """The image sizes of a case of several images (the same for every seed)."""
    n = case["n"]
    if case["lo"] == 0:
        return [_PHOTO if i % 2 == 0 else _PHOTO[::-1] for i in range(n)]
    rng = np.random.default_rng(1000003 * n + 1009 * case["lo"] + case["hi"])
    if case["kind"] == "serve":  # square, log-uniform
        side = np.exp(rng.uniform(np.log(case["lo"]), np.log(case["hi"]), n)).round().astype(int)
        return [(int(s), int(s)) for s in side]
    return [(int(r), int(c)) for r, c in rng.integers(case["lo"], case["hi"] + 1, size=(n, 2))]


def _many(case, seed):
    """A case's images in one device buffer (each from a 256-byte boundary on): the buffer and the images' views."""
    rng, gen = _draws(seed)
    shapes = _shapes(case)
    at = np.concatenate([[0], np.cumsum([(r * c + 255) // 256 * 256 for r, c in shapes])])
    src = torch.zeros(int(at[-1]), dtype=torch.uint8, device="cuda")
    for (r, c), o in zip(shapes, at):
        src[int(o):int(o) + r * c] = _noisy(r, c, rng.uniform(case["dmin"], case["dmax"]), case["texture"], rng,
                                            gen).reshape(-1)

    def views(buf):
        return [buf[int(o):int(o) + r * c].view(r, c) for (r, c), o in zip(shapes, at)]
    return src, views


def _fit_inputs(case, seed):
    """Features of n 256 x 256 images, targets and the initial weights, on the host."""
    rng, gen = _draws(seed)
    n = case["n"]
    density = rng.uniform(0.0, 0.8, n)
    x0, hist = [], []
    for s in range(0, n, 256):
        img = _noisy(256, 256, density[s:s + 256], False, rng, gen, n=len(density[s:s + 256]))
        x0.append((img.view(-1, 64, 4, 64, 4).float().mean(dim=(2, 4)) / 255.0).cpu().numpy())
        bins = (img >> 4).view(len(img), -1)
        hist.append(torch.stack([(bins == b).float().mean(dim=1) for b in range(16)], dim=1).cpu().numpy())
    k = np.clip(np.rint(4.0 + 70.0 * density + rng.normal(0.0, 3.0, n)), 1, 32).astype(np.float32)
    w = np.zeros(hgrms.PREDICTOR_WEIGHTS, dtype=np.float32)
    off = 0
    for cin in (1, 16, 16, 16):  # He-normal convolutions, a head that starts at the mean k
        w[off:off + 144 * cin] = rng.normal(0.0, math.sqrt(2.0 / (9 * cin)), 144 * cin)
        off += 144 * cin
    w[-1] = k.mean()
    return dict(weights=w, x0=np.concatenate(x0), hist=np.concatenate(hist), k=k)


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind in ("single", "host"):
        rng, gen = _draws(seed)
        img = _noisy(case["rows"], case["cols"], case["density"], case["texture"], rng, gen)[0]
        st["src"] = img.cpu().numpy() if kind == "host" else img
        st["work"] = st["src"].copy() if kind == "host" else torch.empty_like(img)
        st["denoiser"] = hgrms.Denoiser(0)
    elif kind in ("batch", "serve"):
        st["src"], views = _many(case, seed)
        st["work"] = torch.empty_like(st["src"])
        st["views"] = views(st["work"])
        if kind == "batch":
            st["denoiser"] = hgrms.Denoiser(0)
        else:
            st["server"] = hgrms.Server(0, hbm_budget_bytes=16 << 30, slots=4)
            st["betas"] = [case["beta"] or 1 + i % 2 for i in range(case["n"])]
    elif kind == "predict":
        src, views = _many(case, seed)
        st["views"] = views(src)
        st["denoiser"] = hgrms.Denoiser(0)
        st["denoiser"].load_predictor(case["beta"])  # the shipped weights
    else:
        st.update(_fit_inputs(case, seed))
        st["denoiser"] = hgrms.Denoiser(0)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "single":
        st["work"].copy_(st["src"])
        k = st["denoiser"].denoise(st["work"], case["alpha"], case["beta"], case["max_k"])
        return dict(image=st["work"], k=k)
    if kind == "host":
        np.copyto(st["work"], st["src"])
        k = st["denoiser"].denoise(st["work"], case["alpha"], case["beta"], case["max_k"])
        return dict(image=st["work"], k=k)
    if kind == "batch":
        st["work"].copy_(st["src"])
        k = st["denoiser"].denoise_batch(st["views"], case["alpha"], case["beta"], case["max_k"])
        return dict(images=st["work"], k=np.array(k, dtype=np.int32))
    if kind == "serve":
        st["work"].copy_(st["src"])
        torch.cuda.current_stream().synchronize()  # the server works on streams of its own
        srv = st["server"]
        ids = [srv.submit(v, case["alpha"], b, case["max_k"]) for v, b in zip(st["views"], st["betas"])]
        k = [srv.wait(i)[0] for i in ids]
        return dict(images=st["work"], k=np.array(k, dtype=np.int32))
    if kind == "predict":
        return dict(k_hat=st["denoiser"].predict_k(case["beta"], st["views"]))
    w, loss = st["denoiser"].train_predictor(st["weights"], st["x0"], st["hist"], st["k"], epochs=case["epochs"],
                                             batch=case["batch"], lr=3e-3, seed=5)
    return dict(weights=w, loss=np.float32(loss))


# ---- Work and exact values -------------------------------------------------

_CONV_FLOPS = 2.0 * 4096 * (9 * 16 + 3 * 9 * 16 * 16)  # one image, forward


def work(case):
    """Each image byte read and written once; one comparison per pixel and
    neighbour (the first pass; what later passes must look at depends on the
    image).  The estimator: its multiply-adds, inputs and results."""
    kind = case["kind"]
    if kind == "fit":
        steps = case["epochs"] * (case["n"] // min(case["batch"], case["n"]))
        return dict(bytes=4.0 * case["n"] * (4096 + 17) + 8.0 * hgrms.PREDICTOR_WEIGHTS,
                    flops=3.0 * _CONV_FLOPS * steps * min(case["batch"], case["n"]))
    if kind == "predict":
        return dict(bytes=float(sum(r * c for r, c in _shapes(case)) + 4 * case["n"]), flops=_CONV_FLOPS * case["n"])
    sizes = [(case["rows"], case["cols"])] if kind in ("single", "host") else _shapes(case)
    betas = [case["beta"] or 1 + i % 2 for i in range(len(sizes))]
    return dict(bytes=float(sum(2 * r * c + 4 for r, c in sizes)),
                flops=float(sum(r * c * ((2 * b + 1) ** 2 - 1) for (r, c), b in zip(sizes, betas))))


def _net(w, x):
    """The estimator's channel means for x [n, 64, 64] (torch, float64): the layers' weights as [tap, in, out]."""
    x, off = x[:, None], 0
    for layer, cin in enumerate((1, 16, 16, 16)):
        wl = w[off:off + 144 * cin].view(3, 3, cin, 16).permute(3, 2, 0, 1)
        off += 144 * cin
        b = w[7056 + 16 * layer:7072 + 16 * layer]
        x = torch.relu(torch.nn.functional.conv2d(x, wl, b, padding=1))
    return x.mean(dim=(2, 3))


def _head(w, gap, hist):
    return gap @ w[7120:7136] + hist @ w[7136:7152] + w[7152]


def _features(img):
    """Area means (64 x 64, / 255) and 16-bin fractions of one image, in float64."""
    r, c = img.shape
    s = torch.zeros(r + 1, c + 1, dtype=torch.float64, device=img.device)
    s[1:, 1:] = img.double().cumsum(0).cumsum(1)

    def edges(m):
        lo = torch.arange(64, device=img.device) * m // 64
        return lo, torch.maximum(lo + 1, (torch.arange(64, device=img.device) + 1) * m // 64)
    (r0, r1), (c0, c1) = edges(r), edges(c)
    cell = s[r1][:, c1] - s[r0][:, c1] - s[r1][:, c0] + s[r0][:, c0]
    x0 = cell / ((r1 - r0)[:, None] * (c1 - c0)[None, :]).double() / 255.0
    return x0, torch.bincount((img >> 4).reshape(-1).long(), minlength=16).double() / (r * c)


def exact(case, seed):
    kind = case["kind"]
    if kind == "predict":
        src, views = _many(case, seed)
        feats = [_features(v) for v in views(src)]
        w = torch.from_numpy(_shipped_weights(case["beta"])).double().cuda()
        k = _head(w, _net(w, torch.stack([f[0] for f in feats])), torch.stack([f[1] for f in feats]))
        return dict(k_hat=k.clamp_min(0.0))
    if kind == "fit":
        return _exact_fit(case, _fit_inputs(case, seed))
    return None  # bytes and counts: whole numbers


def _shipped_weights(beta):
    return np.load(os.path.join(os.path.dirname(hgrms.__file__), f"predictor_b{beta}.npy")).astype(np.float64)


def _exact_fit(case, st):
    """The fit in float64: minibatches of a permutation drawn by a 64-bit
    linear congruential generator, mean squared error, Adam with the step size
    a third for the last quarter of the epochs."""
    n, batch, epochs, lr = case["n"], min(case["batch"], case["n"]), case["epochs"], 3e-3
    w = torch.from_numpy(st["weights"]).double().cuda()
    x0, hist, k = (torch.from_numpy(st[a]).double().cuda() for a in ("x0", "hist", "k"))
    m, v = torch.zeros_like(w), torch.zeros_like(w)
    state = (5 * 6364136223846793005 + 1442695040888963407) & _MASK64
    perm, step, losses = list(range(n)), 0, []
    for ep in range(epochs):
        for i in range(n - 1, 0, -1):
            state = (state * 6364136223846793005 + 1442695040888963407) & _MASK64
            j = ((state >> 33) & 0xFFFFFFFF) % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        losses = []
        rate = lr / 3.0 if ep >= (3 * epochs) // 4 else lr
        for b in range(0, n - batch + 1, batch):
            idx = torch.tensor(perm[b:b + batch], device="cuda")
            p = w.clone().requires_grad_(True)
            total = torch.zeros((), dtype=torch.float64, device="cuda")
            for part in idx.split(64):
                e = _head(p, _net(p, x0[part]), hist[part]) - k[part]
                loss = (e * e).sum() / batch
                loss.backward()
                total += loss.detach()
            step += 1
            m = 0.9 * m + 0.1 * p.grad
            v = 0.999 * v + 0.001 * p.grad * p.grad
            w = w - rate * (m / (1 - 0.9 ** step)) / ((v / (1 - 0.999 ** step)).sqrt() + 1e-8)
            losses.append(float(total))
    return dict(weights=w, loss=sum(losses) / len(losses) if losses else 0.0)
