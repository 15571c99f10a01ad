"""GPU parity of the comparison layers (EvoNorm-S0, range batch-norm) against the double-precision oracle,
through the C ABI.  fp32 elementwise work with double sums: 1e-5 relative + 1e-6 absolute, the absolute term
scaled by the tensor's largest magnitude for sums of signed terms."""
import numpy as np
import pytest
import torch

import oracle
from paper_2111_09389_b200 import api

pytestmark = pytest.mark.gpu

RTOL, ATOL = 1e-5, 1e-6


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def close(got, want, scale=1.0):
    got = got.cpu().numpy().astype(np.float64) if isinstance(got, torch.Tensor) else got
    want = np.asarray(want, np.float64)
    err = np.abs(got - want)
    ok = err <= ATOL * max(1.0, scale) + RTOL * np.abs(want)
    assert ok.all(), f"{(~ok).sum()} of {ok.size} outside tolerance, worst {err.max():.3e}"


def ws_bytes(n):
    return torch.empty(max(int(n), 256), dtype=torch.uint8, device="cuda")


def _inputs(case, seed):
    nodes, B, H, W, C = case
    rng = np.random.default_rng(seed)
    x = (1.5 * rng.standard_normal((nodes, B, H, W, C)) + 0.3).astype(np.float32)
    pad = 5
    P = rng.uniform(0.5, 1.5, (nodes, 3 * C + pad)).astype(np.float32)
    P[:, 2 * C:3 * C] -= 1.0
    dy = rng.standard_normal(x.shape).astype(np.float32)
    return x, P, dy


EVO_CASES = [((4, 8, 16, 16, 16), 4), ((2, 3, 32, 32, 16), 2), ((2, 2, 8, 8, 64), 8), ((1, 3, 5, 7, 6), 3),
             ((1, 2, 4, 4, 12), 1), ((2, 2, 32, 32, 64), 8), ((1, 2, 2, 2, 512), 64), ((1, 1, 1, 1, 8), 2),
             ((1, 2, 9, 9, 24), 3),
             # samples split over a cluster of 2, 4 or 8 CTAs (ragged last share)
             ((1, 2, 31, 33, 64), 16), ((2, 2, 40, 40, 64), 8), ((1, 3, 64, 64, 32), 4), ((1, 1, 96, 96, 64), 8),
             ((1, 1, 160, 160, 64), 8)]


@pytest.mark.parametrize("case,groups", EVO_CASES)
def test_evonorm_s0_fwd_bwd(case, groups):
    nodes, B, H, W, C = case
    x, P, dy = _inputs(case, seed=C + groups)
    eps = 1e-5
    v, g, b = P[:, :C], P[:, C:2 * C], P[:, 2 * C:3 * C]
    y_ref, mu_ref, var_ref = oracle.evonorm_s0_fwd(x, v, g, b, groups, eps)
    xd, Pd = dev(x), dev(P)
    stride = P.shape[1]
    f = lambda *s: torch.empty(*s, dtype=torch.float32, device="cuda")
    y, gmean, gvar = f(*x.shape), f(nodes, B, groups), f(nodes, B, groups)
    api.lpdt_evonorm_s0_fwd(nodes, B, H, W, C, groups, eps, xd, Pd, Pd[:, C:], Pd[:, 2 * C:], stride, y, gmean, gvar)
    close(gmean, mu_ref); close(gvar, var_ref)
    close(y, y_ref, scale=float(np.abs(y_ref).max()))
    # backward from the statistics the forward stored (both sides read the same fp32 values)
    mu32, var32 = gmean.cpu().numpy(), gvar.cpu().numpy()
    dx_ref, dv_ref, dg_ref, db_ref = oracle.evonorm_s0_bwd(dy, x, v, g, mu32, var32, groups, eps)
    G = torch.zeros(nodes, stride, dtype=torch.float32, device="cuda")
    dx = f(*x.shape)
    ws = ws_bytes(api.lpdt_evonorm_s0_bwd_workspace_size(nodes, B, C))
    api.lpdt_evonorm_s0_bwd(nodes, B, H, W, C, groups, eps, dev(dy), xd, Pd, Pd[:, C:], stride, gmean, gvar, dx, G,
                            G[:, C:], G[:, 2 * C:], stride, ws)
    close(dx, dx_ref, scale=float(np.abs(dx_ref).max()))
    Gh = G.cpu().numpy()
    close(Gh[:, :C], dv_ref, scale=float(np.abs(dv_ref).max()))
    close(Gh[:, C:2 * C], dg_ref, scale=float(np.abs(dg_ref).max()))
    close(Gh[:, 2 * C:3 * C], db_ref, scale=float(np.abs(db_ref).max()))
    assert not Gh[:, 3 * C:].any()


# Widths whose channel columns divide no warp: held by a cluster of 2, 4 or 8 CTAs (ragged last share) in either direction, by
# none of them in the backward pass, and by none at all.
@pytest.mark.parametrize("case,groups", [((1, 3, 15, 15, 96), 12), ((2, 2, 33, 31, 48), 6), ((2, 2, 40, 40, 96), 12), ((1, 2, 28, 28, 512), 64),
                                         ((1, 2, 16, 16, 256), 32), ((1, 1, 64, 64, 48), 4), ((1, 1, 96, 96, 48), 6)])
def test_evonorm_s0_widths_beyond_a_warp(case, groups):
    test_evonorm_s0_fwd_bwd(case, groups)


# samples held in shared memory by one to eight CTAs (ragged last share) because the batch is less than a wave, and just beyond one
@pytest.mark.parametrize("case,groups", [((3, 2, 8, 8, 128), 16), ((1, 2, 33, 31, 128), 16), ((2, 2, 17, 19, 64), 16), ((1, 3, 1, 1, 128), 32),
                                         ((4, 37, 5, 5, 128), 16), ((3, 99, 3, 3, 128), 16)])
def test_evonorm_s0_held_samples(case, groups):
    test_evonorm_s0_fwd_bwd(case, groups)


@pytest.mark.parametrize("case", [(1, 3, 56, 56, 64), (2, 2, 96, 96, 16), (2, 5, 32, 32, 64), (1, 4, 33, 31, 128), (3, 2, 7, 9, 4)])
def test_evonorm_s0_gradient_sums_lose_nothing(case):
    """With v = 0, gamma = 1 and x and dy on grids every term of a parameter gradient is exact in fp32, with no bit to spare for
    sums of them; in double these are exact too, and what remains is the rounding of 1/D and of the result, half an ulp (2^-24)
    each."""
    nodes, B, H, W, C = case
    groups, eps = C // 4, 1e-5
    rng = np.random.default_rng(C + H)
    x = rng.integers(-32, 33, (nodes, B, H, W, C)).astype(np.float32) / 16
    f = lambda *s: torch.empty(*s, dtype=torch.float32, device="cuda")
    v, one = torch.zeros(nodes, C, device="cuda"), torch.ones(nodes, C, device="cuda")
    xd, y, dx, gmean, gvar = dev(x), f(*x.shape), f(*x.shape), f(nodes, B, groups), f(nodes, B, groups)
    api.lpdt_evonorm_s0_fwd(nodes, B, H, W, C, groups, eps, xd, v, one, v, C, y, gmean, gvar)
    D = np.sqrt(gvar.cpu().numpy().astype(np.float64) + np.float64(np.float32(eps))).repeat(4, -1)      # [nodes][B][C]
    ws = ws_bytes(api.lpdt_evonorm_s0_bwd_workspace_size(nodes, B, C))
    for power, bits in ((0, 24), (1, 19), (2, 14)):        # of x in the terms, and of dy: 5 bits less for each x
        dy = rng.integers(-2 ** (bits - 1), 2 ** (bits - 1), x.shape).astype(np.float32) * np.float32(2.0 ** (2 - bits))
        out = f(3, nodes, C)
        api.lpdt_evonorm_s0_bwd(nodes, B, H, W, C, groups, eps, dev(dy), xd, v, one, C, gmean, gvar, dx, out[2], out[1], out[0], C, ws)
        parts = (dy.astype(np.float64) * (x.astype(np.float64) / 2) ** power).sum((2, 3))               # sigmoid(0) = 1/2
        if power:
            parts /= D
        want = parts.sum(1)
        # (1/D is rounded once per sample: that half ulp is of the samples' parts)
        bar = 1.001 * 2.0 ** -24 * (np.abs(want) + (np.abs(parts).sum(1) if power else 0))
        err = np.abs(out[power].cpu().numpy() - want)
        assert (err <= bar).all(), (power, (err / np.maximum(bar, 1e-30)).max())


RBN_CASES = [(4, 8, 16, 16, 16), (2, 3, 32, 32, 16), (2, 2, 8, 8, 64), (1, 3, 5, 7, 6), (1, 2, 1, 1, 12),
             (2, 32, 8, 8, 64), (1, 2, 2, 2, 512), (3, 40, 9, 7, 24)]


@pytest.mark.parametrize("case", RBN_CASES)
@pytest.mark.parametrize("ties", [False, True])
def test_range_bn_fwd_bwd(case, ties):
    nodes, B, H, W, C = case
    x, P, dy = _inputs(case, seed=C + B)
    if ties:
        x = (np.round(x * 2) / 2).astype(np.float32)      # coarse grid: the extrema repeat, zeros of both signs occur
        x[x == 0] *= -1.0
    eps = 1e-5
    g, b = P[:, :C], P[:, C:2 * C]
    y_ref, mu_ref, mn_ref, mx_ref, amn_ref, amx_ref = oracle.range_bn_fwd(x, g, b, eps)
    xd, Pd = dev(x), dev(P)
    stride = P.shape[1]
    f = lambda *s: torch.empty(*s, dtype=torch.float32, device="cuda")
    i = lambda *s: torch.empty(*s, dtype=torch.int32, device="cuda")
    y, cmean, cmin, cmax, amin_, amax_ = f(*x.shape), f(nodes, C), f(nodes, C), f(nodes, C), i(nodes, C), i(nodes, C)
    ws = ws_bytes(api.lpdt_range_bn_workspace_size(nodes, C))
    api.lpdt_range_bn_fwd(nodes, B, H, W, C, eps, xd, Pd, Pd[:, C:], stride, y, cmean, cmin, cmax, amin_, amax_, ws)
    assert np.array_equal(cmin.cpu().numpy(), mn_ref) and np.array_equal(cmax.cpu().numpy(), mx_ref)
    assert np.array_equal(amin_.cpu().numpy(), amn_ref) and np.array_equal(amax_.cpu().numpy(), amx_ref)
    close(cmean, mu_ref)
    close(y, y_ref, scale=float(np.abs(y_ref).max()))
    mu32 = cmean.cpu().numpy()
    dx_ref, dg_ref, db_ref = oracle.range_bn_bwd(dy, x, g, mu32, mn_ref, mx_ref, amn_ref, amx_ref, eps)
    G = torch.zeros(nodes, stride, dtype=torch.float32, device="cuda")
    dx = f(*x.shape)
    api.lpdt_range_bn_bwd(nodes, B, H, W, C, eps, dev(dy), xd, Pd, stride, cmean, cmin, cmax, amin_, amax_, dx, G,
                          G[:, C:], stride, ws)
    close(dx, dx_ref, scale=float(np.abs(dx_ref).max()))
    Gh = G.cpu().numpy()
    close(Gh[:, :C], dg_ref, scale=float(np.abs(dg_ref).max()))
    close(Gh[:, C:2 * C], db_ref, scale=float(np.abs(db_ref).max()))
    assert not Gh[:, 2 * C:].any()


def test_norm_layer_errors():
    t = torch.zeros(64, device="cuda"); ti = torch.zeros(64, dtype=torch.int32, device="cuda")
    with pytest.raises(api.LpdtError) as e:      # batch of one: the constant C(b) is infinite
        api.lpdt_range_bn_fwd(1, 1, 2, 2, 4, 1e-5, t, t, t, 4, t, t, t, t, ti, ti, ws_bytes(4096))
    assert e.value.code == 1
    with pytest.raises(api.LpdtError) as e:      # workspace too small
        api.lpdt_range_bn_fwd(1, 2, 2, 2, 4, 1e-5, t, t, t, 4, t, t, t, t, ti, ti, None)
    assert e.value.code == 3
    with pytest.raises(api.LpdtError) as e:      # groups must divide C
        api.lpdt_evonorm_s0_fwd(1, 1, 2, 2, 6, 4, 1e-5, t, t, t, t, 6, t, t, t)
    assert e.value.code == 1


def test_evonorm_s0_two_pass_kernels():
    """The kernels of one CTA per sample serve what neither clusters nor shared memory take; the cases are re-run on them in a
    child process."""
    import os, subprocess, sys
    if os.environ.get("LPDT_CHILD") == "1":
        pytest.skip("already inside a child run")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    child_env = dict(os.environ, LPDT_CHILD="1", LPDT_EVONORM_TWO_PASS="1")
    r = subprocess.run([sys.executable, "-m", "pytest", os.path.join(root, "tests", "test_gpu_norms.py"), "-m", "gpu",
                        "-q", "-x", "-k", "test_evonorm_s0_fwd_bwd"], env=child_env, cwd=root,
                       capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and " passed" in r.stdout, r.stdout[-3000:] + r.stderr[-2000:]
