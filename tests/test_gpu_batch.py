"""Batched CG over lattices of uneven sizes through the C ABI: every lattice's solution is judged by
the oracle's true FP64 residual and compared with the single-lattice CG solution."""
import numpy as np
import pytest

import hisq_inputs as hin
import oracle

pytestmark = pytest.mark.gpu

SMALL_MIX = [((8, 8, 8, 8), 0.1, 0.3), ((4, 6, 8, 10), 0.02, 0.25), ((8, 10, 12, 14), 0.05, 0.35),
             ((16, 16, 16, 16), 0.01, 0.3), ((8, 8, 8, 8), 0.007, 0.4)]


def build(hisq, mix, seed0=500):
    batch = hisq.Batch([m[0] for m in mix])
    folded, bs = [], []
    for l, (L, mass, eps) in enumerate(mix):
        fat, lng = hin.gen_links(L, seed0 + l, eps, 0.1)
        batch.load(l, fat, lng)
        folded.append(oracle.fold_links(L, fat.reshape(-1, 4, 3, 3), lng.reshape(-1, 4, 3, 3)))
        bs.append(hin.gen_source(seed0 + 100 + l, oracle.volume(L) // 2, 1)[0])
    b = np.concatenate([v.reshape(-1) for v in bs]).reshape(-1, 3)
    return batch, folded, bs, b


@pytest.mark.parametrize("inner", [0, 1])
def test_batch_small_mix(hisq, inner):
    import torch
    batch, folded, bs, b = build(hisq, SMALL_MIX)
    masses = [m[1] for m in SMALL_MIX]
    x = torch.zeros(b.shape, dtype=torch.complex128, device="cuda")
    rc, st = batch.cg(x, torch.from_numpy(b).cuda(), masses, 1e-10, 5000, inner_prec=inner)
    assert rc == 0 and st["converged"] == 1
    xs = x.cpu().numpy()
    for l, (L, mass, eps) in enumerate(SMALL_MIX):
        o0, o1 = batch.offsets[l] // 3, batch.offsets[l + 1] // 3
        r = oracle.true_residual(L, folded[l][0], folded[l][1], mass, bs[l], xs[o0:o1])
        assert r <= 1e-10, (l, r)
        assert abs(r - st["lattice_residual"][l]) < 1e-11
        x_ref, _ = oracle.cg(L, folded[l][0], folded[l][1], mass, bs[l], tol=1e-12)
        assert np.linalg.norm(xs[o0:o1] - x_ref) / np.linalg.norm(x_ref) < 1e-7
    # lighter masses need more iterations; every lattice counted its own
    its = st["lattice_iters"]
    assert its[4] > its[0]
    assert st["kernel_launches"] > 0


def test_batch_matches_single_lattice_cg(hisq):
    import torch
    mix = SMALL_MIX[:3]
    batch, folded, bs, b = build(hisq, mix, seed0=700)
    x = torch.zeros(b.shape, dtype=torch.complex128, device="cuda")
    batch.cg(x, torch.from_numpy(b).cuda(), [m[1] for m in mix], 1e-10, 5000, inner_prec=1)
    for l, (L, mass, eps) in enumerate(mix):
        fat, lng = hin.gen_links(L, 700 + l, eps, 0.1)
        lat = hisq.Lattice(L, precs=(0, 1)).load(fat, lng)
        xl = torch.zeros((1, lat.half, 3), dtype=torch.complex128, device="cuda")
        lat.cg(xl, torch.from_numpy(bs[l]).reshape(1, -1, 3).cuda(), mass, 1e-10, 5000, inner_prec=1)
        o0, o1 = batch.offsets[l] // 3, batch.offsets[l + 1] // 3
        d = (x[o0:o1] - xl[0]).norm() / xl.norm()
        assert float(d) < 1e-8


def test_batch_host_buffers(hisq):
    mix = SMALL_MIX[:2]
    batch, folded, bs, b = build(hisq, mix, seed0=900)
    x = np.zeros_like(b)
    rc, st = batch.cg(x, b, [m[1] for m in mix], 1e-10, 5000, inner_prec=1)
    for l, (L, mass, eps) in enumerate(mix):
        o0, o1 = batch.offsets[l] // 3, batch.offsets[l + 1] // 3
        assert oracle.true_residual(L, folded[l][0], folded[l][1], mass, bs[l], x[o0:o1]) <= 1e-10


def test_batch_64_uneven_lattices(hisq):
    """The uneven-batch workload: 64 lattices (32 x 16^4, 19 x 24^3x8, 13 x 32^3x8), per-lattice eps and
    mass, FP32/FP64 mixed CG to 1e-10. Sampled lattices are checked with the oracle; all report <= 1e-10."""
    import torch
    mix = hin.lattice_mix_64()
    batch = hisq.Batch([m["dims"] for m in mix])
    bs = []
    for l, m in enumerate(mix):
        fat, lng = hin.gen_links(m["dims"], m["gauge_seed"], m["eps"], 0.1)
        batch.load(l, fat, lng)
        bs.append(hin.gen_source(m["source_seed"], oracle.volume(m["dims"]) // 2, 1)[0])
    b = np.concatenate([v.reshape(-1) for v in bs]).reshape(-1, 3)
    x = torch.zeros(b.shape, dtype=torch.complex128, device="cuda")
    rc, st = batch.cg(x, torch.from_numpy(b).cuda(), [m["mass"] for m in mix], 1e-10, 5000, inner_prec=1)
    assert rc == 0 and st["converged"] == 1
    assert max(st["lattice_residual"]) <= 1e-10
    xs = x.cpu().numpy()
    for l in (0, 31, 32, 50, 51, 63):
        m = mix[l]
        L = m["dims"]
        fat, lng = hin.gen_links(L, m["gauge_seed"], m["eps"], 0.1)
        ff, lf = oracle.fold_links(L, fat.reshape(-1, 4, 3, 3), lng.reshape(-1, 4, 3, 3))
        o0, o1 = batch.offsets[l] // 3, batch.offsets[l + 1] // 3
        assert oracle.true_residual(L, ff, lf, m["mass"], bs[l], xs[o0:o1]) <= 1e-10


def test_batch_errors(hisq):
    with pytest.raises(hisq.HisqError) as e:
        hisq.hisq_batch_create([(8, 8, 8, 7)])
    assert e.value.code == hisq.HISQ_EINVAL
    batch = hisq.Batch([(4, 6, 8, 10), (8, 8, 8, 8)])
    x = np.zeros((batch.offsets[-1] // 3, 3), np.complex128)
    with pytest.raises(hisq.HisqError) as e:
        batch.cg(x, x.copy(), [0.1, 0.1], 1e-10, 100)  # no links
    assert e.value.code == hisq.HISQ_ENOLINKS


def residuals(batch, mix, folded, masses, bs, x):
    xs = x.cpu().numpy()
    return [oracle.true_residual(m[0], *folded[l], masses[l], bs[l], xs[batch.offsets[l] // 3:batch.offsets[l + 1] // 3])
            for l, m in enumerate(mix)]


@pytest.mark.parametrize("inner", [0, 1])
def test_batch_initial_guesses(hisq, inner):
    """Guesses that are not zero, for some lattices or all (the FP64 operator at the start, which a zero guess skips),
    the solution itself (no iterations), and one with a NaN (refused)."""
    import torch
    batch, folded, bs, b = build(hisq, SMALL_MIX, seed0=1100)
    masses = [m[1] for m in SMALL_MIX]
    bd = torch.from_numpy(b).cuda()
    guess = torch.from_numpy(hin.gen_source(1150, len(b), 1)[0]).cuda()
    for part in ((1, 3), (0, 1, 2, 3, 4)):
        x = torch.zeros_like(bd)
        for l in part:
            x[batch.offsets[l] // 3:batch.offsets[l + 1] // 3] = guess[batch.offsets[l] // 3:batch.offsets[l + 1] // 3]
        rc, st = batch.cg(x, bd, masses, 1e-10, 5000, inner_prec=inner)
        assert rc == 0 and st["converged"] == 1
        r = residuals(batch, SMALL_MIX, folded, masses, bs, x)
        assert max(r) <= 1e-10, (part, r)
        assert max(abs(a - c) for a, c in zip(r, st["lattice_residual"])) < 1e-11
    x0 = x.clone()
    rc, st = batch.cg(x, bd, masses, 1e-10, 5000, inner_prec=inner)
    assert rc == 0 and max(st["lattice_iters"]) == 0 and torch.equal(x, x0)
    x[7, 1] = float("nan")
    with pytest.raises(hisq.HisqError) as e:
        batch.cg(x, bd, masses, 1e-10, 5000, inner_prec=inner)
    assert e.value.code == hisq.HISQ_ENONFINITE


@pytest.mark.parametrize("inner", [0, 1])
def test_batch_solves_one_after_the_other(hisq, inner):
    """The iteration graph that a batch keeps: other masses, sources, solution buffers (FP64 accumulates in the
    caller's), periods and links of one lattice, each solve judged by the oracle; and the first one again, bit for bit."""
    import torch
    batch, folded, bs, b = build(hisq, SMALL_MIX, seed0=1200)
    masses = [m[1] for m in SMALL_MIX]
    b2 = np.concatenate([hin.gen_source(1260 + l, len(v), 1)[0] for l, v in enumerate(bs)])
    bs2 = [b2[batch.offsets[l] // 3:batch.offsets[l + 1] // 3] for l in range(len(bs))]
    keep = []  # every x stays allocated, so each solve has a buffer of its own

    def solve(src, srcs, ms, fold, **opts):
        x = torch.zeros(src.shape, dtype=torch.complex128, device="cuda")
        keep.append(x)
        rc, st = batch.cg(x, torch.from_numpy(src).cuda(), ms, 1e-10, 5000, inner_prec=inner, **opts)
        assert rc == 0 and st["converged"] == 1
        assert max(residuals(batch, SMALL_MIX, fold, ms, srcs, x)) <= 1e-10
        return x

    first = solve(b, bs, masses, folded)
    solve(b2, bs2, masses, folded)
    solve(b2, bs2, [0.3 * m for m in masses[::-1]], folded)
    solve(b, bs, masses, folded, reliable_period=17)
    L = SMALL_MIX[2][0]
    fat, lng = hin.gen_links(L, 1299, 0.3, 0.1)
    batch.load(2, fat, lng)
    other = list(folded)
    other[2] = oracle.fold_links(L, fat.reshape(-1, 4, 3, 3), lng.reshape(-1, 4, 3, 3))
    solve(b, bs, masses, other)
    batch.load(2, *hin.gen_links(L, 1202, SMALL_MIX[2][2], 0.1))
    assert torch.equal(solve(b, bs, masses, folded), first)


def test_batch_shapes_of_no_workload(hisq):
    """Extents that share no tile size: 12^4, 20^3x10, 28^3x6 and the smallest, light and heavy masses mixed, so that
    lattices leave the iteration at different times."""
    import torch
    mix = [((12, 12, 12, 12), 0.01, 0.3), ((20, 20, 20, 10), 0.1, 0.35), ((28, 28, 28, 6), 0.03, 0.25),
           ((4, 4, 4, 4), 0.2, 0.3), ((4, 10, 6, 26), 0.005, 0.4)]
    batch, folded, bs, b = build(hisq, mix, seed0=1300)
    masses = [m[1] for m in mix]
    for inner in (1, 0):
        x = torch.zeros(b.shape, dtype=torch.complex128, device="cuda")
        rc, st = batch.cg(x, torch.from_numpy(b).cuda(), masses, 1e-10, 5000, inner_prec=inner)
        assert rc == 0 and st["converged"] == 1
        assert max(residuals(batch, mix, folded, masses, bs, x)) <= 1e-10


@pytest.mark.parametrize("inner", [0, 1])
def test_batch_every_form_and_tile(hisq, inner):
    """Each tile the tuner may choose, and FP32's form in fewer registers, forced: lattices of fewer sites than a tile,
    of a ragged number of tiles, and one of many, each solve judged by the oracle. The forms add in different orders:
    iteration counts may differ by a step or two."""
    import torch
    mix = [((4, 4, 4, 4), 0.2, 0.3), ((6, 6, 10, 14), 0.05, 0.3), ((16, 16, 16, 16), 0.05, 0.3)]
    batch, folded, bs, b = build(hisq, mix, seed0=1400)
    masses = [m[1] for m in mix]
    its = []
    for form, tile in [(0, t) for t in range(64, 257, 32)] + ([(1, 128)] if inner == 1 else []):
        hisq.hisq_selftest_batch_form(batch.h, form, tile)
        x = torch.zeros(b.shape, dtype=torch.complex128, device="cuda")
        rc, st = batch.cg(x, torch.from_numpy(b).cuda(), masses, 1e-10, 5000, inner_prec=inner)
        assert rc == 0 and st["converged"] == 1
        assert max(residuals(batch, mix, folded, masses, bs, x)) <= 1e-10, (form, tile)
        its.append(st["lattice_iters"])
    for l in range(len(mix)):
        assert max(i[l] for i in its) - min(i[l] for i in its) <= 2, its
    for form, tile in ((0, 32), (0, 100), (1, 64), (2, 128)):
        with pytest.raises(hisq.HisqError) as e:
            hisq.hisq_selftest_batch_form(batch.h, form, tile)
        assert e.value.code == hisq.HISQ_EINVAL
