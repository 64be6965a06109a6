"""GPU kernels at the sizes where their tiling, splitting or dispatch changes,
against the oracle or a plain reference of the same operation."""
import numpy as np
import pytest

import paper_1204_2280_gb300 as B
from oracle import mlp as OM

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 4097, 40000])
def test_training_gradient_tiles(n):
    """Gradient and loss of n rows (32-row tiles, up to 304 blocks that loop
    over them) against the FP64 oracle on the same BF16-rounded values.  An
    activation within FP32 rounding of a BF16 tie may round the other way
    (2^-8 of one activation), so the gradient is held to 2^-6 of its norm and
    the loss to 2^-8."""
    rng = np.random.default_rng(n)
    X = rng.normal(size=(n, B.MLP_IN)).astype(np.float32)
    Y = (rng.normal(size=(n, B.MLP_OUT)) * 5e-3).astype(np.float32)
    net = B.MLP(3)
    norm = np.concatenate([np.zeros(B.MLP_IN), np.ones(B.MLP_IN), [5e-3]]).astype(np.float32)
    net.set_params(None, norm)
    P, _ = net.get_params()
    g, loss = net.grad(X, Y)
    loss_ref, g_ref = OM.loss_grad(P, norm, X, Y)
    assert np.linalg.norm(g - g_ref) <= 2.0 ** -6 * np.linalg.norm(g_ref)
    assert abs(loss - loss_ref) <= 2.0 ** -8 * loss_ref


@pytest.mark.parametrize("n", [1, 127, 129, 152 * 128 + 1])
def test_normalisation_blocks(n):
    """Mean, standard deviation and target RMS over one to all blocks: FP64
    sums, so FP32 results within one rounding of numpy's (the standard
    deviation within sqrt of the FP64 cancellation, far below 1e-6 here)."""
    rng = np.random.default_rng(n)
    X = (rng.normal(size=(n, B.MLP_IN)) + 2.0).astype(np.float32)
    Y = rng.normal(size=(n, B.MLP_OUT)).astype(np.float32)
    net = B.MLP(0)
    for _ in range(2):                       # the arrival count starts over
        net.fit_norm(X, Y)
        _, norm = net.get_params()
        x, y = X.astype(np.float64), Y.astype(np.float64)
        ref = np.concatenate([x.mean(0), np.maximum(x.std(0), 1e-6), [np.sqrt((y * y).mean())]])
        assert np.abs(norm - ref).max() <= 1e-6 * np.abs(ref).max()


def _stable(keys):
    return np.argsort(keys, kind="stable")


@pytest.mark.parametrize("n", [1, 2, 4607, 4608, 4609, 9216, 9217, 13825, 65536])
def test_merge_sort_tiles(n):
    """The static sort at the edges of its 4608-key tiles and runs, with few
    distinct keys (long runs of equal ones), reversed keys and random ones:
    equal to numpy's stable sort."""
    import torch
    rng = np.random.default_rng(n)
    for keys in (rng.integers(0, 3, n), np.arange(n)[::-1].copy(), rng.integers(0, 2 ** 62, n) * 2 + 1,
                 np.full(n, 2 ** 63 - 1)):
        k = torch.from_numpy(keys.astype(np.int64)).cuda()
        out, perm = torch.empty_like(k), torch.empty(n, dtype=torch.int32, device="cuda")
        B.bonsai_sort_keys_static(k, out, perm)
        ref = _stable(keys)
        assert np.array_equal(perm.cpu().numpy(), ref)
        assert np.array_equal(out.cpu().numpy(), keys[ref])


@pytest.mark.parametrize("n", [1, 4608, 4609, 9217, 36865, (1 << 20) - 1, 1 << 20, (1 << 20) + 1, 3000001,
                               (1 << 22) - 1, 1 << 22, (1 << 22) + 1])
def test_build_order_across_sorts(n):
    """Keys, permutation and moved bodies of a build on both sides of the
    tile, run and sort choices, with duplicate positions, against the
    oracle's keys and a stable sort; a rebuild from the sorted state keeps
    the order."""
    import oracle
    rng = np.random.default_rng(n)
    pos = rng.normal(size=(n, 3)).astype(np.float32)
    pos[n // 2:n // 2 + n // 8] = pos[0]
    mass = rng.uniform(0.5, 1.5, n).astype(np.float32)
    mn, S = oracle.domain(pos)
    k = oracle.keys(pos, mn, S)
    ref = _stable(k)
    with B.Bonsai(B.Config(ncrit=32)) as bz:
        bz.set_bodies(pos, mass, pos)
        for _ in range(2):
            bz.build()
            kk, pp = B.bonsai_get_keys(bz.ctx)
            assert np.array_equal(kk, k[ref]) and np.array_equal(pp, ref)
            x, v = np.zeros((n, 3), np.float32), np.zeros((n, 3), np.float32)
            B.bonsai_get_bodies(bz.ctx, x, v)
            assert np.array_equal(x, pos) and np.array_equal(v, pos)
        bz.sync()


def test_build_order_when_the_sort_changes():
    """One context whose loads cross the sort choice (2^22 bodies) both ways,
    and that builds several systems in between: the radix sort's counts are
    its own each time."""
    import oracle
    sizes = [(1 << 22) + 1, 70001, (1 << 22) + 3, 4608, 5000]
    rng = np.random.default_rng(3)
    pos = rng.normal(size=(max(sizes), 3)).astype(np.float32)
    mass = np.ones(max(sizes), np.float32)
    with B.Bonsai(B.Config(ncrit=32)) as bz:
        for n in sizes:
            p = pos[-n:]
            bz.set_bodies(p, mass[:n]).build()
            k = oracle.keys(p, *oracle.domain(p))
            ref = _stable(k)
            kk, pp = B.bonsai_get_keys(bz.ctx)
            assert np.array_equal(kk, k[ref]) and np.array_equal(pp, ref)
            if n < 100000:
                half = n // 3
                bz.set_bodies(p, mass[:n]).set_systems([0, half, n]).build()
                kk, pp = B.bonsai_get_keys(bz.ctx)
                for lo, hi in ((0, half), (half, n)):
                    k = oracle.keys(p[lo:hi], *oracle.domain(p[lo:hi]))
                    ref = _stable(k)
                    assert np.array_equal(kk[lo:hi], k[ref]) and np.array_equal(pp[lo:hi], lo + ref)
        bz.sync()


@pytest.mark.parametrize("n,ncrit", [(1, 32), (7, 32), (9, 64), (63, 64), (65, 32), (129, 64), (200, 16), (700, 64)])
def test_sph_candidate_rings(n, ncrit):
    """Neighbour counts and densities where the candidates end inside, at and
    past the 64-source ring: every body a neighbour of every other, and about
    half of them.  Counts are decided in FP32 as the oracle decides them;
    densities are sums of up to n FP32 terms in chains of at most 64 with
    compensated adds: within 2e-5."""
    import oracle
    rng = np.random.default_rng(n)
    pos = rng.normal(size=(n, 3)).astype(np.float32)
    mass = rng.uniform(0.5, 1.5, n).astype(np.float32)
    for h in (np.full(n, 50.0, np.float32), rng.uniform(1.0, 2.5, n).astype(np.float32)):
        rho, cnt = np.zeros(n, np.float32), np.zeros(n, np.int32)
        with B.Bonsai(B.Config(ncrit=ncrit)) as bz:
            bz.set_bodies(pos, mass).build()
            B.bonsai_sph_density(bz.ctx, h, rho, cnt)
            bz.sync()
        ref = oracle.sph_density(pos, mass, h)
        assert np.array_equal(cnt, ref[1]) and np.abs(rho / ref[0] - 1.0).max() <= 2e-5


@pytest.mark.parametrize("n", [1, 33, 700])
@pytest.mark.parametrize("scale,h", [(1.0, 1e19), (1.0, np.inf), (1e17, 2e17)])
def test_sph_counts_bodies_only(n, scale, h):
    """Neighbour counts where no finite place is out of reach (h^2 near and
    past the largest float: every body is a neighbour) and for bodies about
    1e18 from the origin: the oracle's, whatever the last ring of candidates
    holds past its end."""
    import oracle
    rng = np.random.default_rng(n)
    pos = (rng.normal(size=(n, 3)) * scale + (1e18 if scale > 1.0 else 0.0)).astype(np.float32)
    mass, hs = np.ones(n, np.float32), np.full(n, h, np.float32)
    rho, cnt = np.zeros(n, np.float32), np.zeros(n, np.int32)
    with B.Bonsai(B.Config(ncrit=32)) as bz:
        bz.set_bodies(pos, mass).build()
        B.bonsai_sph_density(bz.ctx, hs, rho, cnt)
        bz.sync()
    assert np.array_equal(cnt, oracle.sph_density(pos, mass, hs)[1])


@pytest.mark.parametrize("n", [(1 << 18) - 1, 1 << 18, (1 << 18) + 1, 300001])
def test_caller_order_outputs(n):
    """Positions, velocities, forces and potentials in caller order on both
    sides of the gather's size rule, each output alone and together, device
    and host: loaded values come back bit for bit, forces equal the sorted
    ones through the permutation."""
    import torch
    rng = np.random.default_rng(n)
    pos, vel = (rng.normal(size=(n, 3)).astype(np.float32) for _ in range(2))
    mass = np.full(n, 1.0 / n, np.float32)
    with B.Bonsai(B.Config(ncrit=32, group_pack=1)) as bz:
        bz.set_bodies(pos, mass, vel).build().multipoles()
        x, v = (torch.zeros(n, 3, device="cuda") for _ in range(2))
        B.bonsai_get_bodies(bz.ctx, x, v)
        assert np.array_equal(x.cpu().numpy(), pos) and np.array_equal(v.cpu().numpy(), vel)
        v.zero_()
        B.bonsai_get_bodies(bz.ctx, None, v)
        assert np.array_equal(v.cpu().numpy(), vel)
        hx = np.zeros((n, 3), np.float32)
        B.bonsai_get_bodies(bz.ctx, hx, None)
        assert np.array_equal(hx, pos)
        acc, pot = torch.zeros(n, 3, device="cuda"), torch.zeros(n, device="cuda")
        bz.forces(1.0, 0.01, acc, pot)
        both = acc.cpu().numpy(), pot.cpu().numpy()
        alone = np.zeros((n, 3), np.float32), np.zeros(n, np.float32)
        bz.forces(1.0, 0.01, alone[0], None)
        bz.forces(1.0, 0.01, None, alone[1])
        bz.sync()
        assert np.array_equal(both[0], alone[0]) and np.array_equal(both[1], alone[1])
    # the scatter's route: potentials alone; a rotated order of the same bodies
    perm = np.roll(np.arange(n), 12345)
    with B.Bonsai(B.Config(ncrit=32, group_pack=1)) as bz:
        a2, p2 = torch.zeros(n, 3, device="cuda"), torch.zeros(n, device="cuda")
        bz.set_bodies(pos[perm], mass, vel[perm]).build().multipoles().forces(1.0, 0.01, a2, p2)
        bz.sync()
        assert np.array_equal(a2.cpu().numpy(), both[0][perm]) and np.array_equal(p2.cpu().numpy(), both[1][perm])


@pytest.mark.parametrize("n", [1, (1 << 18) - 1, (1 << 18) + 1])
def test_outputs_before_the_first_build(n):
    """Loaded bodies read back without a build, alone and together."""
    rng = np.random.default_rng(n)
    pos, vel = (rng.normal(size=(n, 3)).astype(np.float32) for _ in range(2))
    with B.Bonsai(B.Config(ncrit=32)) as bz:
        bz.set_bodies(pos, np.ones(n, np.float32), vel)
        for want in ((True, True), (True, False), (False, True)):
            x, v = (np.zeros((n, 3), np.float32) if w else None for w in want)
            B.bonsai_get_bodies(bz.ctx, x, v)
            assert (x is None or np.array_equal(x, pos)) and (v is None or np.array_equal(v, vel))
        bz.sync()


@pytest.mark.parametrize("n", [1, 16, 31, 33, 127, 129, 5000])
def test_network_rows(n):
    """Inference of 32-row warp tiles against the FP64 oracle on the same
    BF16-rounded weights: within 1e-2 of the output scale (BF16 ties)."""
    rng = np.random.default_rng(n)
    X = rng.normal(size=(n, B.MLP_IN)).astype(np.float32)
    net = B.MLP(11)
    P, norm = net.get_params()
    y = net.predict(X)
    ref, _ = OM.forward(P, norm, X)
    assert np.abs(y - ref).max() <= 1e-2 * np.abs(ref).max()


@pytest.mark.parametrize("n", [1, 2, 3, 101, 513, 4095, 4097, 30001])
def test_judge_sizes(n):
    """The judge at sizes around its target blocks and source splits: p99
    against numpy's percentile of the oracle's direct sum, 1e-4 relative (the
    FP32 error of both sums, 1e-7, against errors of at least 1e-3 of it)."""
    import oracle
    rng = np.random.default_rng(n)
    pos = rng.normal(size=(n, 3)).astype(np.float32)
    mass = np.full(n, 1.0 / n, np.float32)
    acc = np.zeros((n, 3), np.float32)
    with B.Bonsai(B.Config(ncrit=64)) as bz:
        bz.set_bodies(pos, mass).build().multipoles()
        bz.forces(1.1, 0.05, acc)
        p = B.bonsai_judge(bz.ctx, 0.05)
        _, perm = B.bonsai_get_keys(bz.ctx)
        bz.sync()
    t = min(n, 4096)
    ids = perm[(np.arange(t, dtype=np.int64) * n) // t].astype(np.int64)
    a, _ = oracle.direct(pos, mass, 0.05, ids)
    norm = np.linalg.norm(a, axis=1)
    e = np.where(norm > 0, np.linalg.norm(acc[ids] - a, axis=1) / np.maximum(norm, 1e-300), 0.0)
    ref = np.percentile(e, 99)
    assert abs(p - ref) <= 1e-4 * ref + 1e-6


@pytest.mark.parametrize("sizes", [(30001, 5000, 20000, 3000, 4500), (9000, 4096, 9000, 4095)])
def test_judge_other_bodies(sizes):
    """One context judged with one set of bodies and then with smaller and
    larger ones: each judgement samples the bodies of its own set (p99 against
    the oracle's direct sum at them, as above)."""
    import oracle
    with B.Bonsai(B.Config(ncrit=64)) as bz:
        for n in sizes:
            rng = np.random.default_rng(n)
            pos, mass = rng.normal(size=(n, 3)).astype(np.float32), np.full(n, 1.0 / n, np.float32)
            acc = np.zeros((n, 3), np.float32)
            bz.set_bodies(pos, mass).build().multipoles().forces(1.1, 0.05, acc)
            p = B.bonsai_judge(bz.ctx, 0.05)
            t = min(n, 4096)
            ids = B.bonsai_get_keys(bz.ctx)[1][(np.arange(t, dtype=np.int64) * n) // t].astype(np.int64)
            a, _ = oracle.direct(pos, mass, 0.05, ids)
            ref = np.percentile(np.linalg.norm(acc[ids] - a, axis=1) / np.linalg.norm(a, axis=1), 99)
            assert abs(p - ref) <= 1e-4 * ref + 1e-6
        bz.sync()


def test_own_judgement_leaves_the_learned_one():
    """bonsai_judge between learned evaluations: their last judgement (p99 and
    fallback) stays readable and in force until the next judged one."""
    n = 3000
    rng = np.random.default_rng(4)
    pos, mass = rng.normal(size=(n, 3)).astype(np.float32), np.full(n, 1.0 / n, np.float32)
    fine, a = np.zeros((n, 3), np.float32), np.zeros((n, 3), np.float32)
    net = B.MLP(1)
    with B.Bonsai(B.Config(ncrit=64)) as bz:
        bz.set_bodies(pos, mass).build().multipoles().forces(0.5, 0.01, fine)
        B.bonsai_set_learned(bz.ctx, net, 1.0, 0.5, 0.0)         # every judged evaluation falls back
        B.bonsai_set_judge_interval(bz.ctx, 3)
        B.bonsai_forces_learned(bz.ctx, 0.01, a)
        last = B.bonsai_get_judge(bz.ctx)
        assert last[1] and np.array_equal(a, fine)
        assert B.bonsai_judge(bz.ctx, 0.01) < last[0]            # of the fine forces, not of the network's
        assert B.bonsai_get_judge(bz.ctx) == last
        B.bonsai_forces_learned(bz.ctx, 0.01, a)                 # not judged: the decision holds
        assert B.bonsai_get_judge(bz.ctx) == last and np.array_equal(a, fine)
        bz.sync()


@pytest.mark.parametrize("n", [1, 300, 5000])
def test_nan_correction_falls_back(n):
    """A network whose outputs are NaN is rejected by the judge at every finite
    budget: the forces are the fine walk's, bit for bit."""
    rng = np.random.default_rng(n)
    pos, mass = rng.normal(size=(n, 3)).astype(np.float32), np.full(n, 1.0 / n, np.float32)
    net = B.MLP(0)
    P, norm = net.get_params()
    P[-B.MLP_OUT:] = np.nan                              # the output layer's biases
    net.set_params(P, norm)
    fine, a = np.zeros((n, 3), np.float32), np.zeros((n, 3), np.float32)
    with B.Bonsai(B.Config(ncrit=64)) as bz:
        bz.set_bodies(pos, mass).build().multipoles().forces(0.5, 0.01, fine)
        for budget in (1.0, 1e30):
            B.bonsai_set_learned(bz.ctx, net, 1.0, 0.5, budget)
            B.bonsai_forces_learned(bz.ctx, 0.01, a)
            assert B.bonsai_get_judge(bz.ctx) == (np.inf, True) and np.array_equal(a, fine)
        bz.sync()


@pytest.mark.parametrize("n", [1, 255, 257, 5000, 1216 * 256 + 1])
def test_domain_of_loaded_bodies(n):
    """The domain box that loading leaves for the first build (block boxes,
    last block adds up), against the oracle, also after other bodies, for two
    systems, after a rebuild, and with walks repeated without multipoles
    between them."""
    import oracle
    rng = np.random.default_rng(n)
    acc = [np.zeros((n, 3), np.float32) for _ in range(3)]
    with B.Bonsai(B.Config(ncrit=32)) as bz:
        for scale in (1.0, 1e-3, 50.0):
            pos = (rng.normal(size=(n, 3)) * scale + scale).astype(np.float32)
            mass = np.full(n, 1.0 / n, np.float32)
            bz.set_bodies(pos, mass).build()
            mn, S = oracle.domain(pos)
            for _ in range(2):
                m, s = B.bonsai_get_domain(bz.ctx)
                assert np.array_equal(m, mn) and s == S
                bz.build()
        bz.multipoles().forces(0.75, 0.1, acc[0])
        tot = B.bonsai_get_counts(bz.ctx)[2]
        bz.forces(0.75, 0.1, acc[1])                 # no multipoles between: the queues start over
        assert B.bonsai_get_counts(bz.ctx)[2] == tot
        bz.multipoles()
        assert B.bonsai_get_counts(bz.ctx)[2] == tot  # the last walk's totals stay readable
        bz.forces(0.75, 0.1, acc[2])
        assert B.bonsai_get_counts(bz.ctx)[2] == tot
        assert np.array_equal(acc[0], acc[1]) and np.array_equal(acc[0], acc[2])
        if n > 1:
            bz.set_bodies(pos, mass).set_systems([0, n // 2, n]).build()
            m, s = B.bonsai_get_domains(bz.ctx, 2)
            for k, (lo, hi) in enumerate(((0, n // 2), (n // 2, n))):
                mn, S = oracle.domain(pos[lo:hi])
                assert np.array_equal(m[k], mn) and s[k] == S
        bz.sync()


@pytest.mark.parametrize("call,when", [("forces", "before forces"), ("sph", "before forces"), ("all", "before forces"),
                                       ("learned", "before build"), ("learned", "before forces"),
                                       ("multipoles", "after forces")])
def test_replays_between_calls(call, when):
    """A graph of the context's calls that its caller captured, replayed
    between direct calls: it uses the walk's queues and the domain box, and the
    direct calls that follow (another opening angle) give what they give
    without it, with their own interaction totals."""
    import torch
    n = 20000
    rng = np.random.default_rng(8)
    pos = torch.from_numpy(rng.normal(size=(n, 3)).astype(np.float32)).cuda()
    mass, h = torch.full((n,), 1.0 / n, device="cuda"), torch.full((n,), 0.2, device="cuda")
    ref, acc, out = (torch.zeros(n, 3, device="cuda") for _ in range(3))
    rho, cnt = torch.zeros(n, device="cuda"), torch.zeros(n, dtype=torch.int32, device="cuda")
    with B.Bonsai(B.Config(ncrit=32)) as bz:
        bz.set_bodies(pos, mass).build().multipoles().forces(0.5, 0.01, ref)
        tot = B.bonsai_get_counts(bz.ctx)[2]
        bz.sync()
    s, net = torch.cuda.Stream(), B.MLP(0)
    with B.Bonsai(B.Config(ncrit=32), s.cuda_stream) as bz:
        B.bonsai_set_learned(bz.ctx, net, 1.0, 0.9, 1e30)
        run = dict(forces=lambda: bz.forces(0.9, 0.01, acc), multipoles=bz.multipoles,
                   sph=lambda: B.bonsai_sph_density(bz.ctx, h, rho, cnt),
                   learned=lambda: B.bonsai_forces_learned(bz.ctx, 0.01, acc),
                   all=lambda: bz.build().multipoles().forces(0.9, 0.01, acc))[call]
        for _ in range(2):
            bz.set_bodies(pos, mass).build().multipoles()
            run()                                        # direct: sets up what a capture may not
        bz.set_bodies(pos, mass).build().multipoles().sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s, capture_error_mode="thread_local"):
            run()

        def replay(now):
            if now == when:
                with torch.cuda.stream(s):
                    g.replay()

        for _ in range(3):                               # direct launches, captured and replayed ones
            out.zero_()
            torch.cuda.synchronize()
            bz.set_bodies(pos, mass)
            replay("before build")
            bz.build().multipoles()
            replay("before forces")
            bz.forces(0.5, 0.01, out)
            replay("after forces")
            assert B.bonsai_get_counts(bz.ctx)[2] == tot
            bz.sync()
            assert torch.equal(out, ref)


@pytest.mark.parametrize("ncrit,pack,n", [(64, 0, 1), (64, 0, 33), (64, 0, 65), (33, 0, 500), (64, 1, 3000),
                                          (64, 0, 12000), (48, 1, 20000), (64, 1, (1 << 18) - 3), (32, 1, 17),
                                          (32, 0, 500), (32, 1, 24), (32, 1, 9000), (24, 1, 30000), (32, 1, 65536),
                                          (64, 1, 19999), (64, 1, 20000)])
def test_walk_in_parts(ncrit, pack, n):
    """Groups of 33..64 bodies walked in two parts (up to 2^18 bodies) and of
    17..24 in three (up to 2^16), against block time steps' walk, which has
    two or three bodies per lane: a one-level
    cycle moves every body as the step does, bit for bit, with the same
    interaction counts.  Identical positions, oversize leaves and single
    bodies included; and the forces of a system alone against those beside
    a system large enough for that walk."""
    import torch
    from gpu_common import edge_bodies
    b = edge_bodies(n, 5) if n > 200 else None
    rng = np.random.default_rng(n)
    pos = b.pos if b else rng.normal(size=(n, 3)).astype(np.float32)
    mass = b.mass if b else np.full(n, 1.0 / n, np.float32)
    mass = mass.astype(np.float32)
    out = []
    for block in (False, True):
        with B.Bonsai(B.Config(ncrit=ncrit, group_pack=pack)) as bz:
            bz.set_bodies(pos, mass).build().multipoles().forces(0.9, 0.01)
            if block:
                bz.block_cycle(1.0 / 64, 0, 0.2)
            else:
                bz.step(1.0 / 64)
            x, v = np.zeros((n, 3), np.float32), np.zeros((n, 3), np.float32)
            B.bonsai_get_bodies(bz.ctx, x, v)
            bz.sync()
            out.append((x, v, B.bonsai_get_counts(bz.ctx)))
    (x0, v0, c0), (x1, v1, c1) = out
    assert np.array_equal(x0, x1) and np.array_equal(v0, v1)
    assert np.array_equal(c0[0], c1[0]) and np.array_equal(c0[1], c1[1]) and c0[2] == c1[2]
    # the forces themselves: alone, and beside a larger system
    m = 1 << 18
    pos2 = np.concatenate([pos, rng.normal(size=(m, 3)).astype(np.float32)])
    mass2 = np.concatenate([mass, np.full(m, 1.0 / m, np.float32)])
    res = []
    for p, q, off in ((pos, mass, None), (pos2, mass2, [0, n, n + m])):
        with B.Bonsai(B.Config(ncrit=ncrit, group_pack=pack)) as bz:
            acc, pot = torch.zeros(len(q), 3, device="cuda"), torch.zeros(len(q), device="cuda")
            bz.set_bodies(p, q)
            if off:
                bz.set_systems(off)
            bz.build().multipoles().forces(0.9, 0.01, acc, pot)
            bz.sync()
            res.append((acc[:n].cpu().numpy(), pot[:n].cpu().numpy()))
    assert np.array_equal(res[0][0], res[1][0]) and np.array_equal(res[0][1], res[1][1])


@pytest.mark.parametrize("sizes", [[1], [17], [130], [20000], [30] * 256, [100] * 256, [1, 17, 9000, 16, 600, 2] * 3,
                                   [17] * 255 + [40000], [1500] * 120, [4000] * 200, [17] * 2 + [600000, 500000]], ids=lambda s: f"{len(s)}x{s[0]}..{s[-1]}")
def test_root_moments(sizes):
    """The roots that a warp combines (none, one or many to a warp) against
    FP64 sums over each system's bodies: sums of at most a hundred FP32 terms
    per level of the few levels, errors mostly cancelling, so within 128
    roundings of the mass, of the extent and of mass times extent^2; and
    every system's root bit for bit that of the system alone."""
    rng = np.random.default_rng(len(sizes) + sizes[-1])
    off = np.concatenate([[0], np.cumsum(sizes)])
    pos = (rng.normal(size=(off[-1], 3)) + 3.0).astype(np.float32)
    mass = rng.uniform(0.5, 1.5, off[-1]).astype(np.float32)
    mass[off[:-1][::3]] = 0.0                            # a system of one massless body too
    with B.Bonsai(B.Config()) as bz:
        bz.set_bodies(pos, mass).set_systems(off).build().multipoles()
        mono, quad = B.bonsai_get_moments(bz.ctx)
        bz.sync()
    for k in list(range(0, len(sizes), max(1, len(sizes) // 8))) + [len(sizes) - 1]:
        p, m = pos[off[k]:off[k + 1]].astype(np.float64), mass[off[k]:off[k + 1]].astype(np.float64)
        if m.sum() > 0:
            tol, M, com = 128 * 2.0 ** -24, m.sum(), (m[:, None] * p).sum(0) / m.sum()
            y, size = p - com, np.abs(p).max()
            q = np.einsum("i,ij,ik->jk", m, y, y) * 3 - np.eye(3) * (m * (y * y).sum(1)).sum()
            assert abs(mono[k, 3] - M) <= tol * M
            assert np.abs(mono[k, :3] - com).max() <= tol * size
            assert np.abs(quad[k] - q[[0, 1, 2, 0, 0, 1], [0, 1, 2, 1, 2, 2]]).max() <= tol * M * size ** 2
        with B.Bonsai(B.Config()) as bz:
            bz.set_bodies(pos[off[k]:off[k + 1]], mass[off[k]:off[k + 1]]).build().multipoles()
            m1, q1 = B.bonsai_get_moments(bz.ctx)
        assert np.array_equal(mono[k], m1[0]) and np.array_equal(quad[k], q1[0])


@pytest.mark.parametrize("n", [1, 1023, 1024, 1025, 4097, (1 << 18) - 1, (1 << 18) + 1])
def test_build_blocks(n):
    """Trees at the edges of the build's blocks (1,024 bodies up to 2^18, whose
    counts pass 3 adds up, then 4,096), with runs of identical positions across block borders: cells, links,
    levels and groups equal the oracle's, also for two systems and for few
    bodies in a context that held many."""
    import oracle
    rng = np.random.default_rng(n)
    pos = rng.normal(size=(n, 3)).astype(np.float32)
    if n > 4000:
        pos[rng.permutation(n)[:3000]] = pos[0]           # longer than a small block
    few = rng.normal(size=(600, 3)).astype(np.float32)
    half = n // 2

    def alone(bz, p):
        bz.set_bodies(p, np.ones(len(p), np.float32)).build()
        key, _ = B.bonsai_get_keys(bz.ctx)
        ref, t = oracle.build_tree(key, 8), B.bonsai_get_tree(bz.ctx)
        for name in ("body_begin", "body_count", "child_begin", "nchild", "level"):
            assert np.array_equal(t[name], getattr(ref, name)), name
        groups, got = oracle.groups(ref, 16), B.bonsai_get_groups(bz.ctx)
        assert np.array_equal(got[0], groups[0]) and np.array_equal(got[1], groups[1])
        return ref.ncells, groups

    with B.Bonsai(B.Config(nleaf=8, ncrit=16)) as bz:
        alone(bz, pos)
        alone(bz, few)
        if n > 1:
            (c0, g0), (c1, g1) = alone(bz, pos[:half]), alone(bz, pos[half:])
            bz.set_bodies(pos, np.ones(n, np.float32)).set_systems([0, half, n]).build()
            assert B.bonsai_get_sizes(bz.ctx)[1] == c0 + c1
            got = B.bonsai_get_groups(bz.ctx)
            assert np.array_equal(got[0], np.concatenate([g0[0], half + g1[0]]))
            assert np.array_equal(got[1], np.concatenate([g0[1], g1[1]]))
        bz.sync()
