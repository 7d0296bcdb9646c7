"""The list passes' rules: which pixels a pass evaluates, when the lists
change from C_t (pixels that differ from the previous pass's image) to D_t
(pixels that differ from the image two passes back), and how k and the
converged flag follow from the counts.

CPU: the rules restated in numpy on top of the oracle's single passes, from
every pass on, against the oracle's own iteration - bytes, k and converged
flag are whole numbers, so equality.  GPU: the calls that reach each branch
(one CTA alone, its hand-back to the grid when a list grows, the switch from C
to D, empty D lists with pixels still alternating, capped lists, per-image k)
against the oracle, tolerance zero.
"""
import numpy as np
import pytest

from paper_1306_5390_gb300 import synth


def dilate(m, b):
    rows, cols = m.shape
    out = np.zeros_like(m)
    for dy in range(-b, b + 1):
        for dx in range(-b, b + 1):
            ys, yd = max(0, -dy), max(0, dy)
            xs, xd = max(0, -dx), max(0, dx)
            if rows > abs(dy) and cols > abs(dx):
                out[yd:rows - ys, xd:cols - xs] |= m[ys:rows - yd, xs:cols - xd]
    return out


def makes_c(n, before, alpha, k0, c_first_below, dense, short):
    """Whether a pass that reads a list C of n pixels makes C again (before: the
    length of the list before it, 0 for the first pass)."""
    if n > dense and (before == 0 or n * 16 < before * 15 or (alpha == 0 and n // 4 > dense)):
        return True
    if before == 0:
        return k0 < c_first_below
    return n * 4 < before * 3 if n > short else n * 5 < before * 3


def list_passes(oracle_mod, cur, aux, k, alpha, beta, max_k, c_first_below, sizes=None, dense=1 << 30, short=4096):
    """The loop from I_k = cur and I_(k-1) = aux on: (image, k, converged).
    c_first_below: the first pass makes C when k is below it; longer lists than
    dense and short follow other lines.  sizes, when given, receives the length
    of the list that each pass reads."""
    rows, cols = cur.shape
    inner = np.zeros((rows, cols), dtype=bool)
    if rows > 2 * beta and cols > 2 * beta:
        inner[beta:rows - beta, beta:cols - beta] = True
    listed, c_list, before, k0, N = cur != aux, True, 0, k, 0
    while True:
        n = int(listed.sum())
        if sizes is not None:
            sizes.append(n)
        make_c = c_list and makes_c(n, before, alpha, k0, c_first_below, dense, short)
        ev = dilate(listed, beta) & inner
        new, _ = oracle_mod.one_pass(cur, alpha, beta)
        out = np.where(ev, new, aux)  # a pixel that is not evaluated keeps what the output holds
        now, was = ev & (out != cur), ev & (cur != aux)
        if not make_c:
            N += int(now.sum()) - (0 if c_list else int(was.sum()))
        listed = ev & (out != (cur if make_c else aux))
        cur, aux, before, c_list, k = out, cur, n, make_c, k + 1
        if not listed.any() or k >= max_k:
            break
    empty = not listed.any()
    still = (not empty) if c_list else N != 0
    if still and empty:
        return (aux if (max_k - k) % 2 else cur), max_k, False
    if not still:
        return cur, k - (2 if empty and not c_list else 1), True
    return cur, k, False


@pytest.mark.parametrize("beta", [1, 2, 3])
def test_rules_give_the_oracles_iteration(oracle_mod, beta):
    rng = np.random.default_rng(5390 + beta)
    seen = set()
    for trial in range(60):
        rows, cols = (int(v) for v in rng.integers(2 * beta + 1, 2 * beta + 22, size=2))
        alpha = int(rng.choice([0, 1, 5, 10, 60]))
        kind = trial % 3
        if kind == 0:
            img = synth.noisy_image(rows, cols, float(rng.uniform(0.02, 0.7)), 100 * trial + beta)[1]
        elif kind == 1:
            img = synth.random_image(rows, cols, trial, levels=(0, 90, 100, 255))
        else:
            img = np.full((rows, cols), 100, np.uint8)
            img[rows // 2, cols // 2] = 180
        max_k = int(rng.choice([2, 3, 4, 9, 10, 33]))
        ref, k_ref, c_ref = oracle_mod.denoise(img, alpha, beta, max_k)
        aux, cur = img, img
        for k0 in range(1, min(k_ref, max_k - 1) + 1):
            aux, cur = cur, oracle_mod.one_pass(cur, alpha, beta)[0]
            for below, dense, short in ((0, 1 << 30, 4096), (99, 1 << 30, 4096), (0, 4, 4), (6, 16, 0), (0, 0, 0)):
                out, k, c = list_passes(oracle_mod, cur, aux, k0, alpha, beta, max_k, below, dense=dense, short=short)
                assert (k, c) == (k_ref, c_ref) and np.array_equal(out, ref), (trial, rows, cols, alpha, max_k, k0,
                                                                               below, dense, short, k, k_ref)
            seen.add((bool(c_ref), k_ref == max_k))
    assert {(True, False), (False, True)} <= seen


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return torch


@pytest.fixture(scope="module")
def den(torch_cuda):
    from paper_1306_5390_gb300 import build, hgrms
    build.build()
    d = hgrms.Denoiser(0)
    yield d
    d.close()


def single_dot(rows, cols):
    img = np.full((rows, cols), 100, np.uint8)
    img[rows // 2, cols // 3] = 201
    return img


# (image, alpha, beta, max_k, passes per launch, list capacity)
CASES = [
    ("dot", 0, 1, 60, 1, 0),     # spreads without end: one CTA, then the grid
    ("dot", 0, 2, 41, 1, 0),
    ("dot", 0, 7, 6, 1, 0),
    ("dot", 0, 1, 60, 1, 300),   # ... and past the list's capacity
    ("few", 10, 1, 9, 8, 0),     # one list pass
    ("few", 10, 1, 10, 8, 0),
    ("few", 10, 1, 33, 8, 0),
    ("few", 10, 3, 33, 1, 0),
    ("many", 10, 1, 31, 1, 0),   # both parities of the passes left over
    ("many", 10, 1, 32, 1, 0),
    ("many", 10, 2, 32, 2, 0),
    ("many", 10, 2, 33, 4, 0),
    ("many", 10, 3, 32, 1, 0),
    ("many", 5, 1, 40, 1, 50),
    ("many", 10, 2, 2000, 4, 0),
    ("low", 10, 5, 32, 1, 0),    # dies out: C lists to the end
    ("low", 10, 7, 32, 1, 0),
]


@pytest.mark.gpu
@pytest.mark.parametrize("name,alpha,beta,max_k,passes,cap", CASES)
def test_list_pass_branches(oracle_mod, den, torch_cuda, name, alpha, beta, max_k, passes, cap):
    from paper_1306_5390_gb300 import hgrms
    img = {"dot": lambda: single_dot(151, 263),
           "few": lambda: synth.noisy_image(200, 300, 0.2, 71)[1],
           "many": lambda: synth.noisy_image(403, 517, 0.5, 72)[1],
           "low": lambda: synth.noisy_image(500, 301, 0.02, 73)[1]}[name]()
    den.set_option(hgrms.HGRMS_OPT_PASSES, passes)
    den.set_option(hgrms.HGRMS_OPT_LIST_CAP, cap)
    try:
        t = torch_cuda.from_numpy(img.copy()).cuda()
        k = den.denoise(t, alpha, beta, max_k)
        conv = den.converged()
    finally:
        den.set_option(hgrms.HGRMS_OPT_PASSES, 0)
        den.set_option(hgrms.HGRMS_OPT_LIST_CAP, 0)
    ref, k_ref, c_ref = oracle_mod.denoise(img, alpha, beta, max_k)
    assert (k, conv) == (k_ref, c_ref)
    assert np.array_equal(t.cpu().numpy(), ref)


@pytest.mark.gpu
@pytest.mark.parametrize("beta,max_k,cap", [(1, 9, 0), (1, 12, 0), (1, 33, 0), (2, 6, 0), (2, 32, 0), (3, 17, 0), (1, 33, 200)])
def test_batch_k_of_images_that_stop_at_different_passes(oracle_mod, den, torch_cuda, beta, max_k, cap):
    from paper_1306_5390_gb300 import hgrms
    imgs = [synth.noisy_image(40 + 23 * i, 300 - 17 * i, 0.05 * i, 900 + i)[1] for i in range(12)]
    imgs.append(single_dot(30, 30))
    den.set_option(hgrms.HGRMS_OPT_PASSES, 1 if max_k < 9 else 0)
    den.set_option(hgrms.HGRMS_OPT_LIST_CAP, cap)
    try:
        ts = [torch_cuda.from_numpy(im.copy()).cuda() for im in imgs]
        ks = den.denoise_batch(ts, 10, beta, max_k)
    finally:
        den.set_option(hgrms.HGRMS_OPT_PASSES, 0)
        den.set_option(hgrms.HGRMS_OPT_LIST_CAP, 0)
    for i, (im, t, k) in enumerate(zip(imgs, ts, ks)):
        ref, k_ref, c_ref = oracle_mod.denoise(im, 10, beta, max_k)
        assert k == k_ref and (k < max_k) == c_ref, (i, k, k_ref)
        assert np.array_equal(t.cpu().numpy(), ref), i


@pytest.mark.gpu
@pytest.mark.parametrize("alpha,beta", [(0, 1), (1, 1), (2, 1), (0, 2), (1, 2), (2, 2), (0, 3), (1, 3), (0, 5)])
def test_dense_lists(oracle_mod, den, torch_cuda, alpha, beta):
    """Lists of more than 1/32 and 1/8 of the pixels, with and without
    overflow, down to short ones: one image and a batch, from one fused pass on."""
    from paper_1306_5390_gb300 import hgrms
    clean = synth.noisy_image(403, 517, 0.0, 81)[1].astype(np.int64)
    rng = np.random.default_rng(82)
    img = np.clip(clean + rng.integers(-8, 9, clean.shape), 0, 255).astype(np.uint8)
    u = rng.random(img.shape)
    img[u < 0.3], img[u > 0.7] = 0, 255
    imgs = [img, np.ascontiguousarray(img[:150, :301]), np.ascontiguousarray(img[::-1])]
    refs = [oracle_mod.denoise(im, alpha, beta, 27) for im in imgs]
    first, n = oracle_mod.one_pass(img, alpha, beta)
    assert n > img.size // 8 and n > 4096
    for cap in (0, 1 << 20):
        den.set_option(hgrms.HGRMS_OPT_PASSES, 1)
        den.set_option(hgrms.HGRMS_OPT_LIST_CAP, cap)
        try:
            t = torch_cuda.from_numpy(img.copy()).cuda()
            k, conv = den.denoise(t, alpha, beta, 27), den.converged()
            ts = [torch_cuda.from_numpy(im.copy()).cuda() for im in imgs]
            ks = den.denoise_batch(ts, alpha, beta, 27)
        finally:
            den.set_option(hgrms.HGRMS_OPT_PASSES, 0)
            den.set_option(hgrms.HGRMS_OPT_LIST_CAP, 0)
        assert (k, conv) == refs[0][1:] and np.array_equal(t.cpu().numpy(), refs[0][0])
        for t, k, ref in zip(ts, ks, refs):
            assert k == ref[1] and np.array_equal(t.cpu().numpy(), ref[0])


# Random images whose lists never get empty, by alpha: cycles of 3, 4 and 6
# passes, each of one to three listed pixels: (seed, rows, columns).
CYCLES = {2: [(506, 11, 8), (612, 12, 6), (777, 14, 11), (792, 13, 11), (804, 9, 14)],
          3: [(45, 15, 11), (219, 6, 12), (785, 13, 9), (843, 15, 15)]}


@pytest.mark.gpu
@pytest.mark.parametrize("more", [0, 1, 2, 3, 1023, 1024, 1025, 3000])
@pytest.mark.parametrize("alpha", sorted(CYCLES))
def test_short_lists_that_outlive_a_round_of_one_cta(oracle_mod, den, torch_cuda, alpha, more):
    """One CTA runs at most 1024 passes before the others hear of them, and at
    once starts the next round when the list is still short: calls that end
    with, and a few passes after, the first, second and third round (the
    fused launch runs 8 passes), one image and all of them, against the
    oracle."""
    max_k = 8 + 1024 + more
    imgs = [synth.random_image(r, c, seed) for seed, r, c in CYCLES[alpha]]
    refs = [oracle_mod.denoise(im, alpha, 1, max_k) for im in imgs]
    for im, ref in zip(imgs, refs):
        assert ref[1] == max_k and not ref[2]
        assert not np.array_equal(ref[0], oracle_mod.denoise(im, alpha, 1, max_k - 2)[0])  # a list to the end
    for im, ref in zip(imgs, refs):
        for _ in range(5):
            t = torch_cuda.from_numpy(im.copy()).cuda()
            assert den.denoise(t, alpha, 1, max_k) == max_k and not den.converged()
            assert np.array_equal(t.cpu().numpy(), ref[0])
    for _ in range(5):
        ts = [torch_cuda.from_numpy(im.copy()).cuda() for im in imgs]
        assert den.denoise_batch(ts, alpha, 1, max_k) == [max_k] * len(imgs) and not den.converged()
        for t, ref in zip(ts, refs):
            assert np.array_equal(t.cpu().numpy(), ref[0])


# Images whose lists cross the line to one CTA's passes and back: (beta, alpha,
# rows, columns, density, seed, how often they come back).
CROSSING = [(1, 2, 108, 57, 0.105, 229, 1), (3, 1, 114, 113, 0.304, 51, 1), (5, 0, 88, 33, 0.516, 97, 2),
            (5, 1, 109, 74, 0.640, 223, 2)]


@pytest.mark.gpu
@pytest.mark.parametrize("beta,alpha,rows,cols,density,seed,back", CROSSING)
def test_lists_go_back_from_one_cta_to_the_grid(oracle_mod, den, torch_cuda, beta, alpha, rows, cols, density, seed, back):
    """Lists that get longer than one CTA takes after passes that it ran, once
    and twice: the image alone, in batches beside images that do not change and
    beside a copy of itself, calls that end around the crossings."""
    from paper_1306_5390_gb300 import hgrms
    img = synth.noisy_image(rows, cols, density, seed)[1]
    still = np.full((90, 140), 100, np.uint8)
    first, _ = oracle_mod.one_pass(img, alpha, beta)
    line = 112 if beta == 1 else 2048 // (2 * beta + 1) ** 2
    sizes = []
    list_passes(oracle_mod, first, img, 1, alpha, beta, 60, 6, sizes=sizes)
    short = [n <= line for n in sizes]
    at = [i for i in range(len(short) - 1) if short[i] and not short[i + 1]]
    assert len(at) >= back
    den.set_option(hgrms.HGRMS_OPT_PASSES, 1)
    try:
        for max_k in sorted({60, 1 + at[0], 2 + at[0], 3 + at[0], 4 + at[-1]}):
            ref, k_ref, c_ref = oracle_mod.denoise(img, alpha, beta, max_k)
            t = torch_cuda.from_numpy(img.copy()).cuda()
            assert den.denoise(t, alpha, beta, max_k) == k_ref and den.converged() == c_ref
            assert np.array_equal(t.cpu().numpy(), ref)
            for batch in ([still, img, still], [still] * 40 + [img], [img, img]):
                ts = [torch_cuda.from_numpy(im.copy()).cuda() for im in batch]
                ks = den.denoise_batch(ts, alpha, beta, max_k)
                for im, t, k in zip(batch, ts, ks):
                    assert k == (0 if im is still else k_ref)
                    assert np.array_equal(t.cpu().numpy(), still if im is still else ref)
    finally:
        den.set_option(hgrms.HGRMS_OPT_PASSES, 0)


@pytest.mark.gpu
@pytest.mark.parametrize("cols", [225, 239, 240, 241, 255, 257, 480])
@pytest.mark.parametrize("beta", [1, 2, 3])
def test_change_set_of_a_dense_last_pass(oracle_mod, den, torch_cuda, beta, cols):
    """One fused pass that leaves more changes per tile than the passes' own
    lists hold, at widths around the ends of tiles and bitmap words; then list
    passes."""
    from paper_1306_5390_gb300 import hgrms
    img = synth.random_image(131, cols, 40 + cols)
    assert oracle_mod.one_pass(img, 2, beta)[1] > 2 * 1024
    ref, k_ref, c_ref = oracle_mod.denoise(img, 2, beta, 12)
    den.set_option(hgrms.HGRMS_OPT_PASSES, 1)
    den.set_option(hgrms.HGRMS_OPT_LIST_CAP, 1 << 20)
    try:
        t = torch_cuda.from_numpy(img.copy()).cuda()
        k = den.denoise(t, 2, beta, 12)
    finally:
        den.set_option(hgrms.HGRMS_OPT_PASSES, 0)
        den.set_option(hgrms.HGRMS_OPT_LIST_CAP, 0)
    assert (k, den.converged()) == (k_ref, c_ref)
    assert np.array_equal(t.cpu().numpy(), ref)


@pytest.mark.gpu
@pytest.mark.parametrize("alpha", [0, 1, 2])
def test_relaunch_rule_of_large_calls(oracle_mod, den, torch_cuda, alpha):
    """Calls of 4 Mi pixels: alpha 0 and 1 run further fused launches, others list passes only."""
    img = synth.noisy_image(2051, 2049, 0.3, 74)[1]
    t = torch_cuda.from_numpy(img.copy()).cuda()
    k = den.denoise(t, alpha, 1, 18)
    ref, k_ref, c_ref = oracle_mod.denoise(img, alpha, 1, 18)
    assert den.stats()["launches"] == (4 if alpha <= 1 else 2)
    assert (k, den.converged()) == (k_ref, c_ref)
    assert np.array_equal(t.cpu().numpy(), ref)
