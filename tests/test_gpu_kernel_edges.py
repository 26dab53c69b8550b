"""The kernels' dispatch at the edges of its rules, where a tile, a warp or a
launch is nearly empty: digit-slice FP64 stages, two-step FP32 stages, ring
FFTs of few bins, rings without weight, and explicit inverses of small levels.

Tolerances: FP64 transforms of lmax <= 200 round at about lmax 2^-53 (2e-14)
in the oracle's one-step recurrence, 1e-12 leaves a factor 50; FP32 stages
have 1e-5 as elsewhere.  Two forms of the same FP32 level solve differ by
rounding times the condition of a tile's factor, 2e-4 as for the sweeps
against the oracle."""
import numpy as np
import pytest
import torch

from gpu_util import cuda_device, rel_l2
from oracle import geometry, sht
from paper_1308_5299_gb300 import binding, synthetic

pytestmark = pytest.mark.gpu

TOL = {torch.float64: 1e-12, torch.float32: 1e-5}


@pytest.fixture(scope="module")
def dev():
    return cuda_device()


def transforms(dev, grid, lmax, dtype):
    """Relative errors of synthesis and adjoint against the oracle."""
    kw = {"nside": grid} if isinstance(grid, int) else {"gl": grid}
    g = geometry.healpix_grid(grid) if isinstance(grid, int) else geometry.gl_grid(*grid)
    plan = binding.Plan(lmax, **kw)
    a = synthetic.random_alm(lmax, seed=11)
    y = synthetic.random_map(g["npix"], seed=12)
    cdtype = torch.complex128 if dtype == torch.float64 else torch.complex64
    m = torch.empty(g["npix"], dtype=dtype, device=dev)
    plan.sht_synth(torch.from_numpy(a).to(cdtype).to(dev), m)
    b = torch.empty(sht.n_lm(lmax), dtype=cdtype, device=dev)
    plan.sht_adjoint(torch.from_numpy(y).to(dtype).to(dev), b)
    return rel_l2(m.cpu().numpy(), sht.synth(a, lmax, g)), rel_l2(b.cpu().numpy(), sht.adjoint(y, lmax, g))


# 64 pairs and lmax 64 are the smallest of the digit slices, 63 of either goes
# the other way; 128 and 129 pairs fill a tile and begin the next; odd counts
# have a ring on the equator; ring lengths of few bins fold rows many times,
# with (2 lmax > 3 M) and without the row in shared memory
@pytest.mark.parametrize("grid,lmax", [
    (32, 63), (32, 64), (32, 191), ((125, 160), 70), ((127, 160), 64), ((128, 160), 65), ((255, 160), 79),
    ((257, 160), 80), ((258, 162), 127), ((20, 4), 40), ((20, 6), 40), ((20, 34), 60), ((130, 10), 100),
])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_transforms_at_the_edges(dev, grid, lmax, dtype):
    for e in transforms(dev, grid, lmax, dtype):
        assert e < TOL[dtype]


@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 5, 9])
def test_digit_slices_of_several_right_hand_sides(dev, nrhs):
    """Columns of one launch are independent: each equals its own call."""
    lmax = 95
    cl = 1.0 / np.arange(1.0, lmax + 2.0) ** 2
    bl = np.exp(-0.5 * np.arange(lmax + 1) ** 2 * 1e-4)
    ninv = np.abs(synthetic.random_map(12 * 32 * 32, seed=4)) + 0.1
    plan = binding.Plan(lmax, nside=32, cl=cl, bl=bl, ninv=torch.from_numpy(ninv).to(dev))
    x = torch.from_numpy(np.stack([synthetic.random_alm(lmax, seed=20 + j) * 10.0 ** (j - 4) for j in range(nrhs)])).to(dev)
    y = torch.empty_like(x)
    plan.apply_A(x, y)
    for j in range(nrhs):
        one = torch.empty_like(x[j])
        plan.apply_A(x[j].contiguous(), one)
        assert rel_l2(y[j].cpu().numpy(), one.cpu().numpy()) < 1e-13


@pytest.mark.parametrize("bad", [float("inf"), float("nan")])
def test_digit_slices_pass_on_what_is_not_finite(dev, bad):
    lmax, g = 95, geometry.healpix_grid(32)
    plan = binding.Plan(lmax, nside=32)
    a = torch.from_numpy(synthetic.random_alm(lmax, seed=1)).to(dev)
    a[5] = bad  # m = 0
    m = torch.empty(g["npix"], dtype=torch.float64, device=dev)
    plan.sht_synth(a, m)
    assert not torch.isfinite(m).any()
    y = torch.from_numpy(synthetic.random_map(g["npix"], seed=2)).to(dev)
    y[g["npix"] // 2] = bad
    b = torch.empty(sht.n_lm(lmax), dtype=torch.complex128, device=dev)
    plan.sht_adjoint(y, b)
    assert not torch.isfinite(b.real).any()


# rings without weight: none, one, both caps, all but one, all; every other
# ring (pairs half masked); grids on either side of the digit slices
@pytest.mark.parametrize("nside,lmax", [(8, 23), (32, 95), (64, 191)])
@pytest.mark.parametrize("mask", ["none", "one", "caps", "north", "most", "all", "every other"])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_rings_without_weight_against_the_full_transforms(dev, nside, lmax, mask, dtype):
    g = geometry.healpix_grid(nside)
    nring = 4 * nside - 1
    z = np.arange(nring)
    off = {"none": z < 0, "one": z == nside, "caps": np.minimum(z, nring - 1 - z) < nside,
           "north": z < nring // 2, "most": z != nring - 3, "all": z >= 0, "every other": z % 2 == 0}[mask]
    n = np.where(np.minimum(z, nring - 1 - z) < nside, 4 * (np.minimum(z, nring - 1 - z) + 1), 4 * nside)
    assert n.sum() == g["npix"]
    ninv = np.abs(synthetic.random_map(g["npix"], seed=8)) + 0.1
    ninv[np.repeat(off, n)] = 0.0
    l = np.arange(lmax + 1)
    cl, bl = 1.0 / (l + 1.0) ** 2, np.exp(-1e-4 * l * (l + 1.0))
    plan = binding.Plan(lmax, nside=nside, cl=cl, bl=bl, ninv=torch.from_numpy(ninv).to(dev))
    cdtype = torch.complex128 if dtype == torch.float64 else torch.complex64
    x = torch.from_numpy(synthetic.random_alm(lmax, seed=9)).to(cdtype).to(dev)
    y = torch.empty_like(x)
    plan.apply_A(x, y)
    ell = np.concatenate([np.arange(m, lmax + 1) for m in range(lmax + 1)])
    b = torch.from_numpy(bl[ell]).to(dev)
    p = torch.empty(g["npix"], dtype=torch.float64, device=dev)
    plan.sht_synth(x.to(torch.complex128) * b, p)
    t = torch.empty_like(x, dtype=torch.complex128)
    plan.sht_adjoint(p * torch.from_numpy(ninv).to(dev), t)
    full = x.to(torch.complex128) / torch.from_numpy(cl[ell]).to(dev) + b * t
    assert rel_l2(y.cpu().numpy(), full.cpu().numpy()) < TOL[dtype]


def test_explicit_inverse_of_small_levels_against_the_sweeps(dev):
    """Levels up to 48 tiles multiply by the inverse of the sweeps' factor."""
    cfg, cl, bl, ninv = synthetic.problem_inputs("nside32_lmax95")
    kw = dict(nside=cfg["nside"], cl=cl, bl=bl, ninv=torch.from_numpy(ninv).to(dev), levels="default")
    sweeps = binding.Plan(cfg["lmax"], smoother_sweep="per_colour", **kw)
    ridges = [sweeps.level(h)["ridge"] for h in range(1, sweeps.nlevels() + 1)]
    auto = binding.Plan(cfg["lmax"], ridge_alpha=ridges, **kw)
    for h in range(1, sweeps.nlevels() + 1):
        L = auto.level(h)["lmax_h"]
        r = torch.from_numpy(synthetic.random_alm(L, seed=40 + h)).to(dev)
        a, b = torch.empty_like(r), torch.empty_like(r)
        auto.smooth(h, r, a)
        sweeps.smooth(h, r, b)
        assert rel_l2(a.cpu().numpy(), b.cpu().numpy()) < 2e-4, h


@pytest.fixture(scope="module")
def levels256(dev):
    cfg, cl, bl, ninv = synthetic.problem_inputs("nside256_lmax767")
    return binding.Plan(cfg["lmax"], nside=cfg["nside"], cl=cl, bl=bl, ninv=torch.from_numpy(ninv).to(dev),
                        levels="default")


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("nrhs", [1, 2, 16])
def test_pixel_smoother_in_place(dev, levels256, nrhs, dtype):
    """map_out may be map_in on every level, also where each output depends
    on the whole input: the same numbers as with a buffer of its own."""
    plan = levels256
    for h in range(1, plan.nlevels() + 1):
        npix = 12 * plan.level(h)["nside_h"] ** 2
        m = torch.from_numpy(synthetic.random_map(nrhs * npix, seed=60 + h)).to(dtype).to(dev).reshape(nrhs, npix)
        out = torch.empty_like(m)
        plan.pixel_smoother(h, m, out)
        for _ in range(5):
            a = m.clone()
            plan.pixel_smoother(h, a, a)
            assert torch.equal(a, out), h


@pytest.mark.parametrize("grid,lmax", [(64, 384), (512, 1023), ((901, 1802), 900), ((258, 520), 257)])
def test_fp32_ring_by_ring(dev, grid, lmax):
    """Every ring of an FP32 synthesis, and the FP32 adjoint of single rings
    next to the equator, against FP64: the sums of about lmax / 2 terms round
    as a random walk, sqrt(lmax) 2^-24, and a rounding of the argument shifts
    the phase of P~_l by l z 2^-24; twice their sum is allowed."""
    if isinstance(grid, int):
        z, n = (np.asarray(v) for v in synthetic.healpix_ring_table(grid)[:2])
        plan = binding.Plan(lmax, nside=grid)
    else:
        z, n = np.polynomial.legendre.leggauss(grid[0])[0], np.full(grid[0], grid[1])
        plan = binding.Plan(lmax, gl=grid)
    tol = 2.0**-23 * (np.sqrt(lmax) + 2.0 * lmax * np.abs(z))
    ring = np.repeat(np.arange(len(n)), n)
    a = torch.from_numpy(synthetic.random_alm(lmax, seed=13)).to(dev).to(torch.complex64)
    m32 = torch.empty(len(ring), dtype=torch.float32, device=dev)
    m64 = torch.empty(len(ring), dtype=torch.float64, device=dev)
    plan.sht_synth(a, m32)
    plan.sht_synth(a.to(torch.complex128), m64)
    ref = m64.cpu().numpy()
    err = np.sqrt(np.bincount(ring, (m32.cpu().numpy() - ref) ** 2) / np.bincount(ring, ref**2))
    assert (err < tol).all(), (err / tol).max()
    near = np.argsort(np.abs(z), kind="stable")
    for k in (0, 1, 3, 7, 15, 31):
        i = near[k]
        y = torch.zeros(len(ring), dtype=torch.float32, device=dev)
        y[torch.from_numpy(ring == i).to(dev)] = torch.from_numpy(synthetic.random_map(n[i], seed=80 + k)).to(dev).float()
        b32 = torch.empty(sht.n_lm(lmax), dtype=torch.complex64, device=dev)
        b64 = torch.empty(sht.n_lm(lmax), dtype=torch.complex128, device=dev)
        plan.sht_adjoint(y, b32)
        plan.sht_adjoint(y.double(), b64)
        assert rel_l2(b32.cpu().numpy().astype(np.complex128), b64.cpu().numpy()) < tol[i], k


@pytest.mark.parametrize("nside,lmax", [(32, 95), (64, 191), (256, 700)])
def test_fp64_small_parts_beside_large_ones(dev, nside, lmax):
    """One m at a time, the rings of a synthesis fall off by many orders
    towards the poles; and where one ring of a map is 1e10 times brighter, the
    rows of high m that do not reach it are small beside the others.  Such
    parts keep their own precision down to what the terms below 2^-60, which
    are left out, can give (twice 2^-60 over their size): 2^-54 of the largest
    would be 30 times that."""
    g = geometry.healpix_grid(nside)
    n = np.asarray(synthetic.healpix_ring_table(nside)[1])
    ring = np.repeat(np.arange(len(n)), n)
    plan = binding.Plan(lmax, nside=nside)
    o = torch.empty(g["npix"], dtype=torch.float64, device=dev)
    ms = np.concatenate([np.full(lmax + 1 - m, m) for m in range(lmax + 1)])

    def check(err, ref, part, least):
        e, r = (np.sqrt(np.bincount(part, np.abs(v) ** 2)) for v in (err, ref))
        keep = r > least * r.max()
        assert (e <= 2.0**-59 / least * r)[keep].all(), (e[keep] / r[keep]).max()

    for m in (lmax // 3, lmax // 2, 3 * lmax // 4, lmax - 3):
        a = synthetic.random_alm(lmax, seed=90 + m) * (ms == m)
        plan.sht_synth(torch.from_numpy(a).to(dev), o)
        ref = sht.synth(a, lmax, g)
        check(o.cpu().numpy() - ref, ref, ring, 1e-9)
    b = torch.empty(sht.n_lm(lmax), dtype=torch.complex128, device=dev)
    for k in (nside // 4, nside):
        y = synthetic.random_map(g["npix"], seed=95) * np.where(ring == k, 1e10, 1.0)
        plan.sht_adjoint(torch.from_numpy(y).to(dev), b)
        ref = sht.adjoint(y, lmax, g)
        check(b.cpu().numpy() - ref, ref, ms, 3e-10)


@pytest.mark.parametrize("mt", [1, 2])
@pytest.mark.parametrize("rp", [2, 4, 8])
@pytest.mark.parametrize("grid,lmax", [(8, 23), (16, 47), (16, 64), ((125, 130), 63), ((300, 130), 48)])
def test_fp64_shapes_below_the_digit_slices(dev, grid, lmax, rp, mt):
    """Every ring-block shape of the plain FP64 kernels on the grids that run
    on them: fewer than 64 ring pairs, or lmax below 64."""
    g = geometry.healpix_grid(grid) if isinstance(grid, int) else geometry.gl_grid(*grid)
    for stage in ("synthesis", "adjoint"):
        binding.tune_set(g["nring"], g["npix"], lmax, "f64", stage, rp, m_tile=mt)
    for e in transforms(dev, grid, lmax, torch.float64):
        assert e < TOL[torch.float64]


def test_autotuner_times_what_runs(dev):
    """FP64 stages on digit slices have one form: one time under every choice;
    smaller grids time every choice."""
    for nside, lmax, forms in ((32, 70, 1), (16, 50, 6)):
        plan = binding.Plan(lmax, nside=nside)
        rows = [t for t in plan.autotune() if (t["nring"], t["lmax"], t["precision"]) == (4 * nside - 1, lmax, "f64")]
        assert len(rows) == 2
        for t in rows:
            ms = list(t["ms"].values()) + list(t["ms_m_tile2"].values())
            assert len(ms) == 6 and all(v > 0 for v in ms)
            if forms == 1:
                assert len(set(ms)) == 1
            else:
                assert len(set(ms)) > 1


def test_two_threads_with_plans_of_different_sizes(dev):
    """Two host threads, a plan and a stream each: launches that take much and
    little shared memory of the same kernels at the same time."""
    import threading

    def work(gl, lmax, dtype, errors):
        try:
            s = torch.cuda.Stream()
            plan = binding.Plan(lmax, gl=gl, stream=s)
            cdtype = torch.complex128 if dtype == torch.float64 else torch.complex64
            a = torch.from_numpy(synthetic.random_alm(lmax, seed=3)).to(dev).to(cdtype)
            m = torch.from_numpy(synthetic.random_map(gl[0] * gl[1], seed=4)).to(dev).to(dtype)
            b, o = torch.empty_like(a), torch.empty_like(m)
            torch.cuda.synchronize()
            for _ in range(2000):
                plan.sht_synth(a, o)
                plan.sht_adjoint(m, b)
            s.synchronize()
        except Exception as e:
            errors.append(e)

    # ring FFTs of 64 and 16 KB in FP64; fused adjoints of 51 and 20 KB in FP32
    for dtype, big, small in ((torch.float64, ((33, 3000), 40), ((33, 82), 40)),
                              (torch.float32, ((255, 1802), 900), ((33, 82), 40))):
        errors = []
        t = [threading.Thread(target=work, args=(gl, lmax, dtype, errors)) for gl, lmax in (big, small)]
        for x in t:
            x.start()
        for x in t:
            x.join()
        assert not errors, errors


@pytest.mark.parametrize("preset", ["nside32_lmax95", "nside512_lmax1023"])
def test_explicit_inverses_are_symmetric_and_positive(dev, preset):
    """M of the levels of at most 48 tiles, column by column: symmetric to the
    bit, and positive definite, as the factor's L^-T L^-1 is."""
    cfg, cl, bl, ninv = synthetic.problem_inputs(preset)
    plan = binding.Plan(cfg["lmax"], nside=cfg["nside"], cl=cl, bl=bl, ninv=torch.from_numpy(ninv).to(dev),
                        levels="default", ridge_bisections=8)
    seen = 0
    for h in range(1, plan.nlevels() + 1):
        n = 12 * plan.level(h)["nside_h"] ** 2
        if n > 48 * 64:
            continue
        eye, m = torch.eye(n, dtype=torch.float32, device=dev), torch.empty((n, n), dtype=torch.float32, device=dev)
        for i in range(n):
            plan.pixel_smoother(h, eye[i], m[i])
        assert torch.equal(m, m.T), h
        w = torch.linalg.eigvalsh(m.double())
        assert w[0] > 0, (h, w[0], w[-1])
        seen += 1
    assert seen
