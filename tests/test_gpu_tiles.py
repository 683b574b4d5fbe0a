"""Edges of the tiled kernels and of the rules that choose between them,
against the FP64 oracle: the transpose tiles (32 x 32 and 16 x 16 pixels, the
small-image form up to 64^2), the image layouts (32 x 32 tiles with a border of
two elements), the view table and its order (one CTA of 256 views, sorting
above 256 views, no sort above 4096), the interleaved derivative modes and the
fan-beam transpose with its source near the image.

Normwise relative tolerances as in the other parity tests: float32 1e-5,
float64 1e-12.
"""
import numpy as np
import pytest

import oracle
from paper_2605_06336_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {torch.float32: 1e-5, torch.float64: 1e-12}


def dev(a, dtype=torch.float64):
    return torch.tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def host(t):
    return t.detach().double().cpu().numpy()


def rel(a, b):
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


def _setup(N, B, vpf, K, dtype, seed, D=None):
    from paper_2605_06336_gb300 import ct
    rng = np.random.default_rng(seed)
    V = sum(vpf)
    theta = rng.uniform(-2 * np.pi, 2 * np.pi, V)  # every quadrant, negative angles
    delta = rng.normal(0, 0.7, V)
    X = rng.uniform(size=(K, len(vpf) * N * N))
    Y = rng.standard_normal((K, V * B))
    op = ct.CTOperator(N, B, V, vpf, max_batch=K, dtype=dtype, source_distance=D)
    return op, oracle.Geometry(N, B, V, vpf, fan_D=D), theta, delta, X, Y, rng


# N, bins (None: the default), views per frame, batch
TRANSPOSE = [
    (2, None, [3], 1), (16, None, [5], 2), (33, 21, [7], 4), (63, None, [9, 0, 4], 3), (64, None, [30], 1),
    (64, 91, [12, 5], 8),                      # up to 64^2: the small-image form and its limit of tiles
    (65, None, [11], 1), (96, 97, [6, 0, 13], 5), (97, None, [64], 2), (128, 33, [10], 7), (160, None, [9], 8),
    (65, 400, [130], 4),                       # detector wider than the image
    (65, None, [40], 1), (65, None, [60], 4),  # 4 and 6 CTAs a tile
    (65, None, [1100], 4), (65, 30, [1100], 8),  # more than the 128 views a CTA stages at a time
]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("case", TRANSPOSE, ids=lambda c: f"N{c[0]}_B{c[1]}_F{len(c[2])}_K{c[3]}")
def test_transpose_tiles(case, dtype):
    N, B, vpf, K = case
    B = B or synth.n_bins(N)
    op, g, theta, delta, _, Y, _ = _setup(N, B, vpf, K, dtype, 7 * N + K)
    ref = oracle.adjoint(g, theta, Y, delta)
    th, dl, Yg = dev(theta), dev(delta), dev(Y, dtype)
    assert rel(host(op.adjoint(Yg, th, dl)), ref) <= TOL[dtype]
    base = op.tuning
    for kb in (1, 2, 4, 8):
        for split in (1, 2, 4):
            t = list(base)
            t[3], t[4] = kb, split
            op.tuning = t
            assert rel(host(op.adjoint(Yg, th, dl)), ref) <= TOL[dtype], (kb, split)


@pytest.mark.parametrize("K", [1, 2, 8])
def test_transpose_keeps_a_non_finite_sample_to_its_pixels(K):
    """An infinite sample reaches the pixels whose interpolation cell holds it, of its own image alone."""
    N, V = 70, 5
    B = synth.n_bins(N)
    op, g, theta, delta, _, Y, _ = _setup(N, B, [V], K, torch.float32, K)
    v, b, k = 2, B // 2, K - 1
    clean = Y.copy()
    clean[k, v * B + b] = 0.0
    near = np.zeros((3, V * B))
    for i in range(3):
        near[i, v * B + b - 1 + i] = 1.0
    w = oracle.adjoint(g, theta, near, delta)
    ref = oracle.adjoint(g, theta, clean, delta)
    Y[k, v * B + b] = np.inf
    got = host(op.adjoint(dev(Y, torch.float32), dev(theta), dev(delta)))
    for i in range(K):
        if i != k:
            assert rel(got[i], ref[i]) <= 1e-5
    assert not np.isfinite(got[k][w[1] > 1e-4]).any()
    far = (w == 0).all(0)
    assert far.sum() > N * N // 2
    assert np.abs(got[k][far] - ref[k][far]).max() <= 1e-4


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("K", [1, 2, 8])
@pytest.mark.parametrize("N", [40, 70])
def test_transpose_of_views_shifted_off_the_detector(N, K, dtype):
    """Offsets beyond 32-bit bin numbers, and beyond 64-bit fixed point: such a view adds nothing."""
    far = [2.0 ** 31 + 3, -(2.0 ** 32) + 5.5, 2.0 ** 32 - 9.25, 3e9, 1e12, -1e12, 1e300, -1e300]
    V = len(far) + 4
    op, g, theta, delta, _, Y, _ = _setup(N, synth.n_bins(N), [V], K, dtype, 3 * N + K)
    Y = Y.reshape(K, V, g.B)
    zeroed = Y.copy()
    zeroed[:, :len(far)] = 0.0
    ref = oracle.adjoint(g, theta, zeroed.reshape(K, -1), delta)
    delta[:len(far)] = far
    got = host(op.adjoint(dev(Y.reshape(K, -1), dtype), dev(theta), dev(delta)))
    assert rel(got, ref) <= TOL[dtype]


# N, views, laid-out batch, repeated batches: other numbers of tiles, groups cut, groups left out
REPEAT = [(256, 180, 16, [1, 8, 11, 15]), (130, 90, 9, [3, 8, 9]), (64, 30, 40, [2, 8, 33]), (97, 40, 7, [1, 4, 6])]


@pytest.mark.parametrize("fan", [False, True])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("case", REPEAT, ids=lambda c: f"N{c[0]}_K{c[2]}")
def test_repeated_transpose_of_fewer_sinograms_gives_the_same_bits(case, dtype, fan):
    from paper_2605_06336_gb300 import ct
    N, V, K, fewer = case
    rng = np.random.default_rng(N)
    op = ct.CTOperator(N, synth.n_bins(N), V, max_batch=K, dtype=dtype, source_distance=2.0 * N if fan else None)
    Y = dev(rng.standard_normal((K, op.m)), dtype)
    whole = op.adjoint(Y, dev(rng.uniform(0, np.pi, V))).clone()
    for k in fewer:
        X = torch.zeros_like(whole)
        ct.ct_adjoint_repeat(op.h, X, k)
        assert torch.equal(X[:k], whole[:k]), k
        assert not X[k:].any(), k


# N, views, batch: the order of the views (counted, sorted, none) and the CTAs of the view table
VIEWS = [(16, 255, 1), (16, 256, 2), (16, 257, 1), (8, 512, 1), (8, 513, 4), (8, 1200, 1), (8, 2049, 4), (8, 4096, 1), (8, 4096, 5), (8, 4097, 2)]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("case", VIEWS, ids=lambda c: f"N{c[0]}_V{c[1]}_K{c[2]}")
def test_view_table_sizes(case, dtype):
    """Forward with one set of angles, then a part of them changed; then a transpose that brings new angles."""
    N, V, K = case
    op, g, theta, delta, X, Y, rng = _setup(N, synth.n_bins(N), [V - 3, 0, 3], K, dtype, V + K)
    Xg, dl = dev(X, dtype), dev(delta)
    for _ in range(2):
        assert rel(host(op.forward(Xg, dev(theta), dl)), oracle.forward(g, theta, X, delta)) <= TOL[dtype]
        theta = theta + np.where(rng.uniform(size=V) < 0.01, 0.3, 0.0)
        theta[V - 1] -= 0.2
    theta = theta + 0.1
    assert rel(host(op.adjoint(dev(Y, dtype), dev(theta), dl)), oracle.adjoint(g, theta, Y, delta)) <= TOL[dtype]
    assert rel(host(op.forward(Xg, dev(theta), dl)), oracle.forward(g, theta, X, delta)) <= TOL[dtype]


# N around the 32-element tiles of the layouts (N + 4 elements a row), frames, batch (groups of 4, 2 and 1)
LAYOUTS = [(2, 1, 1), (27, 1, 2), (28, 2, 7), (29, 1, 4), (31, 3, 3), (32, 1, 6), (33, 1, 5), (60, 2, 1), (61, 1, 8)]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("case", LAYOUTS, ids=lambda c: f"N{c[0]}_F{c[1]}_K{c[2]}")
def test_image_layouts(case, dtype):
    N, F, K = case
    vpf = [6] * F
    op, g, theta, delta, X, _, rng = _setup(N, synth.n_bins(N), vpf, K, dtype, N * K)
    th, dl, Xg = dev(theta), dev(delta), dev(X, dtype)
    ref = oracle.forward(g, theta, X, delta)
    y = op.forward(Xg, th, dl).clone()
    assert rel(host(y), ref) <= TOL[dtype]
    if dtype == torch.float32 and K >= 2:  # interleaved groups and pairs give the same bits
        kb = 8 if K >= 8 else 4
        dth, R = dev(rng.standard_normal(g.V)), dev(rng.standard_normal((K, g.m)), dtype)
        out = []
        for inter in (0, 1):
            op.tuning = [kb, 1, 1, 1, 1, 1, 1, 0, 0, 0, 4, inter]
            out.append([op.forward(Xg, th, dl), op.jac_batch(Xg, th, dth, dl), op.jacT_batch(Xg, th, R, dl)])
        assert all(torch.equal(p, q) for p, q in zip(*out))


@pytest.mark.parametrize("max_batch", [2, 3, 7, 8])
@pytest.mark.parametrize("der_kb", [1, 4])
def test_products_of_fewer_images_after_an_interleaved_call(max_batch, der_kb):
    """Any order of products that pass no images after a call that laid out a batch interleaved: one image, some
    and all of them, then the whole batch again -- the bits that passing the images to another handle gives."""
    from paper_2605_06336_gb300 import ct
    N, vpf, K = 37, [7, 5], max_batch
    V, B = sum(vpf), synth.n_bins(37)
    rng = np.random.default_rng(max_batch)
    ops = [ct.CTOperator(N, B, V, vpf, max_batch=K, dtype=torch.float32) for _ in range(2)]
    for op in ops:
        op.tuning = [4, 2, 2, 4, 1, 4, 1, 0, 0, 0, der_kb, 1]
    op, other = ops
    th, dth, dl = dev(rng.uniform(-3, 3, V)), dev(rng.standard_normal(V)), dev(rng.normal(0, 0.5, V))
    R = dev(rng.standard_normal((K, op.m)), torch.float32)
    X0 = [dev(rng.uniform(size=(K, op.n)), torch.float32) for _ in range(2)]

    def fwd(o, X, k):
        return o.forward(X, th, dl, batch=k) if X is None else o.forward(X[:k], th, dl)

    def jac1(o, X, k):
        return o.jac(None if X is None else X[0], th, dth, dl)

    def jacT(o, X, k):
        g = torch.zeros(k, V, dtype=torch.float64, device="cuda")
        ct.ct_jacT_batch(o.h, th, dl, None if X is None else X[:k].contiguous(), R, g, None, k)
        return g

    def gn(o, X, k):
        out = [torch.zeros(k, V, dtype=torch.float64, device="cuda") for _ in range(3)]
        ct.ct_gn_terms_batch(o.h, th, dl, None if X is None else X[:k].contiguous(), R, None, *out, k)
        return torch.stack(out)

    calls = [(f, k) for f in (fwd, jac1, jacT, gn) for k in {1, 2, (K + 1) // 2, K}]
    for trial in range(12):
        X = X0[trial % 2]
        first = (fwd, jacT)[trial % 2 if der_kb == 4 else 0]
        first(op, X, K)
        for q in rng.permutation(len(calls))[:8]:
            f, k = calls[q]
            assert torch.equal(f(op, None, k), f(other, X, k)), (trial, f.__name__, k)
    for op in ops:
        op.close()


def test_one_changed_value_of_a_handles_own_tuning_is_taken():
    """Handles that start on interleaved images: their values with any one of the forward's changed are valid."""
    from paper_2605_06336_gb300 import ct
    N, V, K = 40, 9, 8
    B = synth.n_bins(N)
    rng = np.random.default_rng(0)
    op = ct.CTOperator(N, B, V, max_batch=K, dtype=torch.float32)
    theta, X = rng.uniform(-3, 3, V), rng.uniform(size=(K, N * N))
    ref = oracle.forward(oracle.Geometry(N, B, V), theta, X)
    own = op.tuning
    assert own[0] >= 4 and own[7] == 0 and own[11] == 1
    for change, layout in (({0: 1}, 0), ({0: 2}, 0), ({0: 8}, 1), ({2: 8, 7: 8}, 0), ({2: 4, 7: 4, 1: 1}, 0), ({}, 1)):
        t = list(own)
        for i, v in change.items():
            t[i] = v
        op.tuning = t
        assert op.tuning == t[:11] + [layout]
        assert rel(host(op.forward(dev(X, torch.float32), dev(theta))), ref) <= TOL[torch.float32]
    op.close()


def test_interleaved_images_take_no_memory_of_their_own():
    """A handle that starts on interleaved images allocates what the pair images, the sinograms and the
    partials take (in 2 MB pieces), and selecting the layout allocates nothing."""
    from paper_2605_06336_gb300 import ct
    N, V, K = 1024, 60, 8
    B = synth.n_bins(N)

    def used():
        torch.cuda.synchronize()
        free, total = torch.cuda.mem_get_info()
        return total - free
    ct.CTOperator(64, 91, 8, max_batch=K).close()  # the context and the kernels are loaded
    made, more = [], []
    for _ in range(4):  # (the smallest of a few: another process may use the device meanwhile)
        before = used()
        op = ct.CTOperator(N, B, V, max_batch=K, dtype=torch.float32)
        made.append(used() - before)
        assert op.tuning[11] == 1
        op.tuning = [4, 2, 2, 4, 1, 4, 1, 0, 0, 0, 1, 1]
        more.append(used() - before - made[-1])
        op.close()
    pairs, sino, partials = 2 * (K + 1) * N * (N + 4) * 8, K * V * (B + 5) * 8, 32 * K * V * ((B + 31) // 32)
    assert min(made) <= pairs + sino + partials + 24 * 2 ** 20
    assert min(more) <= 0


# the source as near as the geometry takes it (0.75 max(N, B) + 2): wide ray windows at the far side
FAN = [(33, [9], 1), (48, [5, 0, 6], 3), (65, [12], 8)]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("case", FAN, ids=lambda c: f"N{c[0]}_F{len(c[1])}_K{c[2]}")
def test_fan_source_near_the_image(case, dtype):
    N, vpf, K = case
    B = synth.n_bins(N)
    D = 0.75 * max(N, B) + 2.5
    op, g, theta, delta, X, Y, _ = _setup(N, B, vpf, K, dtype, N + K, D)
    th, dl = dev(theta), dev(delta)
    fwd, adj = oracle.forward(g, theta, X, delta), oracle.adjoint(g, theta, Y, delta)
    for tuned in (False, True):
        if tuned:  # fresh angles after autotune: its own trial angles must not stay behind
            op.autotune()
        assert rel(host(op.forward(dev(X, dtype), th, dl)), fwd) <= TOL[dtype]
        assert rel(host(op.adjoint(dev(Y, dtype), th, dl)), adj) <= TOL[dtype]
