"""The PTC network on the GPU (weights rounded to BF16, FP32 arithmetic) against the FP64 oracle: forward
output, loss and weight gradients; flexible CG with the network as preconditioner judged by the oracle's true
residual. Tolerances with weights that BF16 rounds: forward <= 1e-2, gradients <= 2e-2 (relative)."""
import numpy as np
import pytest

import hisq_inputs as hin
import oracle
import oracle.ptc as optc

pytestmark = pytest.mark.gpu

L = (8, 10, 12, 14)


@pytest.fixture(scope="module")
def setup(hisq):
    fat, lng = hin.gen_links(L, 4242, 0.35, 0.1)
    lat = hisq.Lattice(L, precs=(0, 1)).load(fat, lng)
    ff, lf = oracle.fold_links(L, fat.reshape(-1, 4, 3, 3), lng.reshape(-1, 4, 3, 3))
    net = hisq.Ptc(lat)
    return lat, net, ff, lf


def rel(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def test_ptc_forward_parity(setup):
    import torch
    lat, net, ff, lf = setup
    W1, W2 = optc.init_weights(11)
    net.set_weights(W1, W2)
    r = hin.gen_source(12, lat.half, 2)
    rd = torch.from_numpy(r).to(torch.complex64).cuda()
    z = torch.empty_like(rd)
    net.apply(z, rd, 2)
    zg = z.cpu().numpy().astype(np.complex128)
    w1, w2 = W1.astype(np.complex64).astype(np.complex128), W2.astype(np.complex64).astype(np.complex128)
    for v in range(2):
        ref, _ = optc.network_forward(L, ff, w1, w2, r[v])
        assert rel(zg[v], ref) <= 1e-2, rel(zg[v], ref)


def test_ptc_apply_programmatic_launch_bitwise(setup, hisq):
    """The network's two passes as programmatic dependent launches give the bits of plain launches, also
    when applications are chained (each one's input is the previous one's output)."""
    import torch
    lat, net, ff, lf = setup
    W1, W2 = optc.init_weights(17)
    net.set_weights(W1, W2)
    r = torch.from_numpy(hin.gen_source(18, lat.half, 1)).to(torch.complex64).cuda()
    outs = {}
    for pdl in (1, 0):
        hisq.hisq_set_pdl(lat.ctx, pdl)
        zs = [r]
        for _ in range(3):
            z = torch.empty_like(r)
            net.apply(z, zs[-1], 1)
            zs.append(z)
        torch.cuda.synchronize()
        outs[pdl] = [t.clone() for t in zs[1:]]
    hisq.hisq_set_pdl(lat.ctx, 1)
    for a, b in zip(outs[1], outs[0]):
        assert torch.equal(a, b)


def test_ptc_identity_network(setup):
    """W1 = W2 = identity hop on channel 0 only: N(r) = r (up to BF16 rounding of r)."""
    import torch
    lat, net, ff, lf = setup
    W1 = np.zeros((8, 1, 9), np.complex128)
    W2 = np.zeros((1, 8, 9), np.complex128)
    W1[0, 0, 0] = 1.0
    W2[0, 0, 0] = 1.0
    net.set_weights(W1, W2)
    r = hin.gen_source(13, lat.half, 1)
    rd = torch.from_numpy(r).to(torch.complex64).cuda()
    z = torch.empty_like(rd)
    net.apply(z, rd, 1)
    assert rel(z.cpu().numpy()[0].astype(np.complex128), r[0]) <= 5e-3


def test_ptc_gradient_parity(setup):
    import torch
    lat, net, ff, lf = setup
    W1, W2 = optc.init_weights(21)
    net.set_weights(W1, W2)
    bs = hin.gen_source(30, lat.half, 3)
    xs = hin.gen_source(40, lat.half, 3)
    bd = torch.from_numpy(bs).to(torch.complex64).cuda()
    xd = torch.from_numpy(xs).to(torch.complex64).cuda()
    loss, g1, g2 = net.train_step(bd, xd, 3, 0.0)
    w1, w2 = W1.astype(np.complex64).astype(np.complex128), W2.astype(np.complex64).astype(np.complex128)
    rloss, r1, r2 = optc.loss_and_grads(L, ff, w1, w2, list(bs), list(xs))
    assert abs(loss - rloss) <= 1e-2 * abs(rloss)
    assert rel(g1.astype(np.complex128), r1) <= 2e-2, rel(g1, r1)
    assert rel(g2.astype(np.complex128), r2) <= 2e-2, rel(g2, r2)
    # weights unchanged with lr = 0
    a, b = net.get_weights()
    assert np.allclose(a, W1.astype(np.complex64)) and np.allclose(b, W2.astype(np.complex64))


def test_ptc_training_reduces_loss(setup):
    import torch
    lat, net, ff, lf = setup
    W1, W2 = optc.init_weights(31, scale=0.05)
    net.set_weights(W1, W2)
    mass = 0.05
    bs = hin.gen_source(50, lat.half, 8)
    xs = np.stack([oracle.cg(L, ff, lf, mass, bs[i], tol=1e-8)[0] for i in range(8)])
    bd = torch.from_numpy(bs).to(torch.complex64).cuda()
    xd = torch.from_numpy(xs).to(torch.complex64).cuda()
    first = net.train_step(bd, xd, 8, 0.02)[0]
    for _ in range(60):
        last = net.train_step(bd, xd, 8, 0.02)[0]
    assert last < 0.8 * first, (first, last)


@pytest.mark.parametrize("weights", ["identity", "trained"])
def test_fcg_true_residual(setup, weights):
    import torch
    lat, net, ff, lf = setup
    mass = 0.05
    if weights == "identity":
        W1 = np.zeros((8, 1, 9), np.complex128)
        W2 = np.zeros((1, 8, 9), np.complex128)
        W1[0, 0, 0] = 1.0
        W2[0, 0, 0] = 1.0
        net.set_weights(W1, W2)
    else:
        # the tied network N = B^dag B is Hermitian positive semi-definite
        W1, W2 = optc.init_weights(41, scale=0.05)
        W1[0, 0, 0] = 1.0
        net.set_tied(True)
        net.set_weights(W1, optc.tie(W1))
        bs = hin.gen_source(70, lat.half, 8)
        xs = np.stack([oracle.cg(L, ff, lf, mass, bs[i], tol=1e-8)[0] for i in range(8)])
        bd = torch.from_numpy(bs).to(torch.complex64).cuda()
        xd = torch.from_numpy(xs).to(torch.complex64).cuda()
        for _ in range(40):
            net.train_step(bd, xd, 8, 0.01)
    b = hin.gen_source(60, lat.half, 1)
    x = torch.zeros((1, lat.half, 3), dtype=torch.complex128, device="cuda")
    rc, st = net.fcg(x, torch.from_numpy(b).cuda(), mass, 1e-10, 3000)
    assert rc == 0 and st["converged"] == 1
    r = oracle.true_residual(L, ff, lf, mass, b[0], x.cpu().numpy()[0])
    assert r <= 1e-10
    assert abs(r - st["true_rel_residual"]) < 1e-11
    net.set_tied(False)
    if weights == "identity":
        # identity preconditioner: FCG takes about as many iterations as CG
        xc = torch.zeros_like(x)
        _, sc = lat.cg(xc, torch.from_numpy(b).cuda(), mass, 1e-10, 3000, inner_prec=1)
        assert abs(st["iters"] - sc["iters"]) <= 0.15 * sc["iters"] + 5


def test_ptc_tied_gradient_parity(setup):
    import torch
    lat, net, ff, lf = setup
    W1, _ = optc.init_weights(51)
    net.set_tied(True)
    net.set_weights(W1, optc.tie(W1))
    bs = hin.gen_source(52, lat.half, 2)
    xs = hin.gen_source(53, lat.half, 2)
    bd = torch.from_numpy(bs).to(torch.complex64).cuda()
    xd = torch.from_numpy(xs).to(torch.complex64).cuda()
    loss, g1, _ = net.train_step(bd, xd, 2, 0.0)
    a, b = net.get_weights()
    net.set_tied(False)
    w1 = W1.astype(np.complex64).astype(np.complex128)
    assert np.allclose(b, optc.tie(w1).astype(np.complex64))  # layer 2 follows layer 1
    rloss, G = optc.loss_and_grads_tied(L, ff, w1, list(bs), list(xs))
    assert abs(loss - rloss) <= 1e-2 * abs(rloss)
    assert rel(g1.astype(np.complex128), G) <= 2e-2, rel(g1, G)


def test_trained_network_gains_over_the_method_without_it(hisq):
    """The learned preconditioner's gain, measured: the tied network is trained on the GPU on 3 seeded
    gauge fields x 128 (Gaussian source, solution) pairs at 16^3x8, m = 0.001 (the solutions from the
    library's mixed CG to 1e-10), then flexible CG with it solves a held-out field's source to a true
    residual of 1e-10 (judged by the oracle). It must take at least 9% fewer iterations than both the
    method without a trained network -- flexible CG with the identity network, and the plain
    mixed-precision CG -- on that field. The bar is conservative: the 32^3x8 workload with 512 pairs saves
    26% (87 against 117 iterations) and this recipe measured 90 against 120 on two held-out fields."""
    import torch
    L, mass, npair, bp = (16, 16, 16, 8), 0.001, 128, 16

    def field(seed):
        fat, lng = hin.gen_links(L, seed, 0.35, 0.1)
        return hisq.Lattice(L, precs=(0, 1)).load(fat, lng), fat, lng

    train = [field(7000 + i)[0] for i in range(3)]
    half = train[0].half
    pairs = []
    for i, lat in enumerate(train):
        b = torch.from_numpy(hin.gen_source(7100 + i, half, npair)).cuda()
        x = torch.zeros_like(b)
        torch.cuda.synchronize()
        for k in range(0, npair, 16):
            rc, _ = lat.cg(x[k:k + 16], b[k:k + 16], mass, 1e-10, 20000, nrhs=16, inner_prec=1)
            assert rc == 0
        pairs.append((b.to(torch.complex64), x.to(torch.complex64)))
    W1, _ = optc.init_weights(7000, scale=0.05)
    W1[0, 0, 0] = 1.0
    net = hisq.Ptc(train[0])
    net.set_tied(True)
    net.set_weights(W1, optc.tie(W1))
    losses = []
    for ep in range(12):
        for k in range(0, npair, bp):
            for i, lat in enumerate(train):
                net.bind(lat)
                b, x = pairs[i]
                losses.append(net.train_step(b[k:k + bp].contiguous(), x[k:k + bp].contiguous(), bp, 0.02)[0])
    assert np.mean(losses[-24:]) < 0.5 * np.mean(losses[:24])
    Wt = net.get_weights()

    lat, fat, lng = field(7200)
    ff, lf = oracle.fold_links(L, fat.reshape(-1, 4, 3, 3), lng.reshape(-1, 4, 3, 3))
    b = hin.gen_source(7300, half, 1)
    bd = torch.from_numpy(b).cuda()
    net.bind(lat)
    x = torch.zeros_like(bd)
    rc, st = net.fcg(x, bd, mass, 1e-10, 20000)
    assert rc == 0 and oracle.true_residual(L, ff, lf, mass, b[0], x.cpu().numpy()[0]) <= 1e-10
    trained = st["iters"]
    I1 = np.zeros((8, 1, 9), np.complex128)
    I1[0, 0, 0] = 1.0
    net.set_weights(I1, optc.tie(I1))
    x.zero_()
    rc, st = net.fcg(x, bd, mass, 1e-10, 20000)
    assert rc == 0
    identity = st["iters"]
    x.zero_()
    rc, st = lat.cg(x, bd, mass, 1e-10, 20000, inner_prec=1)
    assert rc == 0
    mixed = st["iters"]
    net.set_tied(False)
    assert trained <= 0.91 * min(identity, mixed), (trained, identity, mixed)


@pytest.mark.parametrize("npairs", [1, 2, 3, 7, 17])
@pytest.mark.parametrize("dims", [(6, 6, 6, 6), (4, 4, 4, 4), (4, 6, 8, 10)])
def test_ptc_gradient_groups_and_tiles(hisq, dims, npairs):
    """Loss and gradients of every grouping of the pairs (4, 2 and 1 per link read, chunks of 16) on lattices whose
    sites fill the last tile of 32 or not (6^4: 648 = 20 * 32 + 8), with inputs far from unit scale. FP32
    arithmetic on BF16-exact weights: transports and 8-term sums round by a few 2^-24, so 1e-5 leaves a factor
    of more than ten for the cancellation in N(b) - x."""
    import torch
    fat, lng = hin.gen_links(dims, 77, 0.35, 0.1)
    lat = hisq.Lattice(dims, precs=(0, 1)).load(fat, lng)
    ff, _ = oracle.fold_links(dims, fat.reshape(-1, 4, 3, 3), lng.reshape(-1, 4, 3, 3))
    net = hisq.Ptc(lat)
    W = [torch.view_as_complex(torch.view_as_real(torch.from_numpy(w.astype(np.complex64))).to(torch.bfloat16).float())
         .numpy() for w in optc.init_weights(78)]
    net.set_weights(*W)
    b = (3e6 * hin.gen_source(79, lat.half, npairs)).astype(np.complex64)
    x = (3e6 * hin.gen_source(80, lat.half, npairs)).astype(np.complex64)
    loss, g1, g2 = net.train_step(torch.from_numpy(b).cuda(), torch.from_numpy(x).cuda(), npairs, 0.0)
    rl, r1, r2 = optc.loss_and_grads(dims, ff, *(w.astype(np.complex128) for w in W), list(b.astype(np.complex128)),
                                     list(x.astype(np.complex128)))
    assert abs(loss - rl) <= 1e-5 * rl
    assert rel(g1, r1) <= 1e-5 and rel(g2, r2) <= 1e-5, (rel(g1, r1), rel(g2, r2))


def test_ptc_loss_sums_over_many_tiles_per_block(hisq):
    """|d|^2 and |x|^2 over the 40 or 41 tiles a block has at 32^3x24, every term exact in FP32: the identity network
    and b = x + 1, x = 3497/2048 everywhere, so that the loss is 1 / x^2. Rounded once, to FP32: 2^-24, with a factor
    of two. Plain FP32 running sums are off by 5.7e-7."""
    import torch
    L, xi = (32, 32, 32, 24), 3497 / 2048
    lat = hisq.Lattice(L, precs=(0, 1))
    links = torch.zeros((int(np.prod(L)), 4, 3, 3), dtype=torch.complex128, device="cuda")
    lat.load(links, links)
    net = hisq.Ptc(lat)
    w1, w2 = np.zeros((8, 1, 9), np.complex64), np.zeros((1, 8, 9), np.complex64)
    w1[0, 0, 0] = w2[0, 0, 0] = 1
    net.set_weights(w1, w2)
    for npairs in (1, 2, 4):
        x = torch.full((npairs, lat.half, 3), xi, dtype=torch.complex64, device="cuda")
        loss, g1, g2 = net.train_step(x + 1, x, npairs, 0.0)
        assert abs(loss * xi * xi - 1) <= 2.0 ** -23, npairs
        # dL/dconj W[0][0] = sum conj(b) d / |x|^2, the same for both layers
        for g in (g1[0, 0, 0], g2[0, 0, 0]):
            assert abs(g * xi * xi / (xi + 1) - 1) <= 2.0 ** -23, npairs


@pytest.mark.parametrize("scale", [1e-18, 1e-6, 1e16])
def test_ptc_gradients_over_many_tiles_and_scales(hisq, scale):
    """Gradients over 28 tiles per block, at the ends of the inputs' range: against the same step with the inputs at
    unit scale (the loss and gradients do not depend on a common factor of b and x), and loss and gradients together
    by the network's linearity: with d = N(b) - x and N linear in each layer, Re <W1, G1> = Re <W2, G2> =
    Re <N(b), d> / |x|^2, formed here in FP64. FP32 terms round by a few 2^-24 and a thread's FP32 sums have some 170
    terms; 1e-5 as for the small lattices."""
    import torch
    L = (32, 32, 32, 16)
    torch.manual_seed(3)
    U = 0.6 * torch.randn(int(np.prod(L)), 4, 3, 3, dtype=torch.complex128, device="cuda")  # any matrices will do
    lat = hisq.Lattice(L, precs=(0, 1)).load(U, U)
    net = hisq.Ptc(lat)
    W = [torch.view_as_complex(torch.view_as_real(torch.from_numpy(w.astype(np.complex64))).to(torch.bfloat16).float())
         .numpy() for w in optc.init_weights(81)]
    net.set_weights(*W)
    b = torch.randn(4, lat.half, 3, dtype=torch.complex64, device="cuda")
    x = torch.randn(4, lat.half, 3, dtype=torch.complex64, device="cuda")
    loss1, a1, a2 = net.train_step(b, x, 4, 0.0)
    z = torch.empty_like(b)
    net.apply(z, b, 4)
    z, t = z.to(torch.complex128), x.to(torch.complex128)
    nx = t.abs().square().sum((1, 2))
    zd = float(((z.conj() * (z - t)).real.sum((1, 2)) / nx).mean())
    for w, g in zip(W, (a1, a2)):
        # the apply rounds its activation to FP16: 2^-11 per entry, averaged over the sites
        assert abs(float((w.conj() * g).real.sum()) - zd) <= 1e-4 * abs(zd)
    loss, g1, g2 = net.train_step(b * scale, x * scale, 4, 0.0)
    assert abs(loss - loss1) <= 1e-5 * loss1
    assert rel(g1, a1) <= 1e-5 and rel(g2, a2) <= 1e-5


def test_fcg_solves_one_after_the_other(hisq):
    """The iteration graph that a context keeps for the flexible CG: other masses, sources, solution buffers, periods,
    weights, a second network, links loaded anew and compressed long links, each solve judged by the oracle; and the
    first solve again, bit for bit."""
    import torch
    naik = -1.0 / 24.0
    fat, lng = hin.gen_links(L, 901, 0.35, 0.1)
    fat2, lng2 = hin.gen_links(L, 902, 0.3, 0.1)
    lat = hisq.Lattice(L, precs=(0, 1)).load(fat, lng)
    fold = [oracle.fold_links(L, f.reshape(-1, 4, 3, 3), l.reshape(-1, 4, 3, 3)) for f, l in ((fat, lng), (fat2, lng2))]
    Wa = optc.init_weights(91, scale=0.02)[0]
    Wb = optc.init_weights(92, scale=0.03)[0]
    Wa[0, 0, 0] = Wb[0, 0, 0] = 1.0

    def network(W):
        n = hisq.Ptc(lat)
        n.set_tied(True)
        n.set_weights(W, optc.tie(W))
        return n

    net, keep = network(Wa), []
    src = hin.gen_source(903, lat.half, 2)

    def solve(n, b, mass, links, **opts):
        x = torch.zeros((1, lat.half, 3), dtype=torch.complex128, device="cuda")
        keep.append(x)
        rc, st = n.fcg(x, torch.from_numpy(b[None]).cuda(), mass, 1e-10, 3000, **opts)
        assert rc == 0 and st["converged"] == 1
        assert oracle.true_residual(L, *fold[links], mass, b, x.cpu().numpy()[0]) <= 1e-10
        return x

    first = solve(net, src[0], 0.05, 0)
    solve(net, src[1], 0.05, 0)
    solve(net, src[0], 0.2, 0)
    solve(net, src[0], 0.05, 0, reliable_period=9)
    net.set_weights(Wb, optc.tie(Wb))
    solve(net, src[0], 0.05, 0)
    second = network(Wa)
    assert torch.equal(solve(second, src[0], 0.05, 0), first)
    lat.load(fat2, lng2)
    solve(second, src[0], 0.05, 1)
    lat.compress_long(naik).load(fat, lng)
    solve(second, src[0], 0.05, 0)
    lat.compress_long(0.0).load(fat, lng)
    net.set_weights(Wa, optc.tie(Wa))
    assert torch.equal(solve(net, src[0], 0.05, 0), first)
