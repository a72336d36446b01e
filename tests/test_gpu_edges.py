"""Kernels at the sizes where their tilings change: edges of tiles, ragged
remainders, the smallest inputs and ones larger than a single pass over the
GPU. Each against the oracle or a plain FP64 evaluation, with tolerances that
follow from the arithmetic (stated at each test)."""
import numpy as np
import pytest

import paper_1007_3458_gb300 as q
from oracle import mlp as M
from paper_1007_3458_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available()
    return torch


@pytest.mark.parametrize("n", [1, 15, 17, 152 * 16 + 1, 152 * 16 * 8 + 5])
def test_gradient_tiles(torch, n):
    """Guess-network gradient: one row, ragged 16-row tiles, one tile more
    than the CTAs, one tile more than the warps of the whole grid. An entry is
    a sum of products of bf16 operands: a hidden unit near a rounding midpoint
    moves its terms by 2^-8, twice on the way through both layers, so every
    entry stays within 2^-6 of its absolute term sum (FP32 sums far below)."""
    rows = W.mlp_rows_synthetic(n, 14)
    ref = W.mlp_rows_synthetic(4096, 15)
    w = W.mlp_init(5, ref[:, :4], ref[:, 4])
    work = torch.empty(q.qym_mlp_workspace_bytes(), dtype=torch.uint8, device="cuda")
    g = torch.empty(q.QYM_MLP_NW, dtype=torch.float32, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    q.qym_mlp_grad_dev(n, torch.from_numpy(w).cuda(), torch.from_numpy(rows).cuda(), g, loss, work)
    L, go, gabs = M.loss_and_grad(w, rows[:, :4], rows[:, 4], emulate=True)
    d = np.abs(g.cpu().numpy().astype(np.float64) - go)
    assert np.all(d <= 2.0 ** -6 * gabs + 1e-7 * np.abs(go).max()), np.max(d / (gabs + 1e-300))
    assert abs(loss.item() - L) <= 1e-4 * L + 1e-7


def _accel_ref(m, x, G):
    """Accelerations in extended precision, and the sums of the terms' magnitudes."""
    L = np.longdouble
    xb, gm = x[1:].astype(L), L(G) * m[1:].astype(L)
    a, mag = np.zeros(x.shape, L), np.zeros(x.shape, L)
    for i in range(len(xb)):
        d = xb - xb[i]
        r2 = (d * d).sum(1)
        with np.errstate(divide="ignore", invalid="ignore"):
            s = np.where(r2 > 0, gm / (r2 * np.sqrt(r2)), L(0))
        t = s[:, None] * d
        a[1 + i], mag[1 + i] = t.sum(0), np.abs(t).sum(0)
    return a, mag


# (bodies, length unit, mass unit, kind)
FP64_CASES = [
    (1, 1.0, 1.0, "disk"), (2, 1.0, 1.0, "disk"), (16, 1.0, 1.0, "disk"), (129, 1.0, 1.0, "disk"),
    (300, 1.5e11, 2e30 * 6.67e-11, "disk"),   # SI lengths, G folded into the masses
    (300, 1e-30, 1e-30, "disk"),              # far from 1: scaled by powers of two
    (300, 1e90, 1e40, "disk"),                # outside the scaled range: plain FP64
    (300, 1.0, 1.0, "close"),                 # coincident, nearly coincident and far bodies
    (300, 1.0, 1.0, "masses"),                # massless, tiny and large masses
    (300, 1.0, 1.0, "flat"),                  # coplanar
    (2200, 1.0, 1.0, "disk"),
]


@pytest.mark.parametrize("n,lu,mu,kind", FP64_CASES)
def test_fp64_kick_edges(torch, n, lu, mu, kind):
    """The FP64 kick, whose pairs are formed on the FP32 pipes, over sizes,
    units, close pairs and masses, against extended precision. A pair's term
    carries at most 2^-51 (two half-unit roundings of its weight, one of the
    separation, one of the product), a sum of n of them n 2^-53 more."""
    rng = np.random.default_rng(n + int(abs(np.log10(lu))))
    x = np.concatenate([np.zeros((1, 3)), rng.normal(size=(n, 3)) * [10.0, 10.0, 0.1]])
    m = np.concatenate([[1.0], 10.0 ** rng.uniform(-12, -3, n)])
    if kind == "flat":
        x[:, 2] = 0.0
    if kind == "masses":
        m[1::3] = 0.0
        m[2] = 1e-40
        m[3] = 1e3
    if kind == "close":
        x[2] = x[1]                        # coincident: no pull on each other
        x[4] = x[3] + [1e-13, 0.0, 0.0]    # below the float form's range
        x[6] = x[5] + [1e-6, -1e-7, 1e-9]
        x[8] = x[7] * (1 + 2.0 ** -52)
        x[9] *= 1e9
        x[10] *= 1e-9
    x, m = x * lu, m * mu
    a = torch.empty((3, n + 1), dtype=torch.float64, device="cuda")
    work = torch.empty(q.qym_accel_workspace_bytes(n + 1, q.QYM_KICK_FP64), dtype=torch.uint8, device="cuda")
    q.qym_accel_dev(n + 1, torch.from_numpy(m).cuda(), torch.from_numpy(np.ascontiguousarray(x.T)).cuda(),
                    a, 1.0, q.QYM_KICK_FP64, work)
    ref, mag = _accel_ref(m, x, 1.0)
    err = np.abs(a.cpu().numpy().T.astype(np.longdouble) - ref)
    bound = (n + 4) * np.longdouble(2.0) ** -53 * mag + np.longdouble(1e-300)
    assert np.all(err <= bound), float(np.max(err / bound))


def test_fp64_kick_nonfinite(torch):
    """A non-finite coordinate spreads as in plain FP64 arithmetic: NaN in
    that component of the body and of every other one, nowhere else."""
    n = 70
    w = W.outer_disk(n - 4, seed=2)
    for bad in (np.nan, np.inf):
        x = w.q.copy()
        x[9, 1] = bad
        a = torch.empty((3, n + 1), dtype=torch.float64, device="cuda")
        work = torch.empty(q.qym_accel_workspace_bytes(n + 1, q.QYM_KICK_FP64), dtype=torch.uint8, device="cuda")
        q.qym_accel_dev(n + 1, torch.from_numpy(w.m).cuda(), torch.from_numpy(np.ascontiguousarray(x.T)).cuda(),
                        a, 1.0, q.QYM_KICK_FP64, work)
        a = a.cpu().numpy()
        assert np.all(np.isnan(a[1, 1:])) and np.all(np.isfinite(a[[0, 2]]))


@pytest.mark.parametrize("sizes", [[1], [2, 1, 130], [128], [129, 7], [700, 300, 257]])
@pytest.mark.parametrize("lu,mu", [(1.0, 1.0), (1.5e11, 2e30), (1e120, 1.0)])
def test_energy_blocks(torch, sizes, lu, mu):
    """Energy over system sizes at the edges of the 128-row blocks, in several
    units (one outside the scaled float range), against extended precision:
    n terms of at most 2^-51 each and a sum of n of them, relative to the sum
    of the terms' magnitudes. Two bodies coincide (no pair term)."""
    L = np.longdouble
    rng = np.random.default_rng(sum(sizes))
    ms, qs, vs, off = [], [], [], [0]
    for n in sizes:
        m = np.concatenate([[1.0], 10.0 ** rng.uniform(-10, -3, n)])
        x = rng.normal(size=(n + 1, 3)) * [10, 10, 0.1]
        v = rng.normal(size=(n + 1, 3)) * 0.3
        x[0] = v[0] = 0.0
        if n > 5:
            m[4] = 0.0
            x[2] = x[1]
        ms.append(m * mu), qs.append(x * lu), vs.append(v * np.sqrt(mu / lu)), off.append(off[-1] + n + 1)
    m, x, v = np.concatenate(ms), np.concatenate(qs), np.concatenate(vs)
    sim = q.Simulation(m, x, v, np.array(off), coords=1, kick_prec=q.QYM_KICK_FP64, encounters=0)
    E = sim.energy()
    sim.close()
    for s, n in enumerate(sizes):
        ml, xl, vl = ms[s].astype(L), qs[s].astype(L), vs[s].astype(L)
        mb, xb, vb = ml[1:], xl[1:], vl[1:]
        S = (mb[:, None] * vb).sum(0)
        kin = mb * (vb * vb).sum(1) / 2
        star = ml[0] * mb / np.sqrt((xb * xb).sum(1))
        pair = L(0)
        for i in range(n):
            r = np.sqrt(((xb[i + 1:] - xb[i]) ** 2).sum(1))
            pair += (mb[i] * mb[i + 1:][r > 0] / r[r > 0]).sum()
        ref = (S * S).sum() / (2 * ml[0]) + kin.sum() - star.sum() - pair
        mag = (np.abs(mb[:, None] * vb).sum(0) ** 2).sum() / (2 * ml[0]) + kin.sum() + star.sum() + pair
        assert abs(E[s] - ref) <= (n + 8) * L(2.0) ** -53 * mag, (s, float((E[s] - ref) / mag))
        if len(sizes) == 1 or s == 0:
            t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
            out = torch.empty(1, dtype=torch.float64, device="cuda")
            work = torch.empty(q.qym_energy_workspace_bytes(n + 1), dtype=torch.uint8, device="cuda")
            q.qym_energy_dev(n + 1, t(ms[s]), t(qs[s].T), t(vs[s].T), 1.0, out, work)
            assert abs(out.item() - ref) <= (n + 8) * L(2.0) ** -53 * mag


@pytest.mark.parametrize("n", [2048, 8192, 8193, 16385, 32769, 65536, 65537])
def test_order_sizes(torch, n):
    """The Morton order at the edges of the one-cluster sort (words per thread
    1, 2, 4, 8) and just past it, with a third of the bodies at one point
    (equal codes keep row order): the host's (code, row) order."""
    from test_gpu_order import _host_order
    w = W.outer_disk(n - 4, 1e-10, seed=n)
    x = w.q.copy()
    x[5:5 + n // 3] = x[5]
    sim = q.Simulation(w.m, x, w.v, w.offsets, encounters=0)
    assert np.array_equal(sim.order(), _host_order(sim.state()[0]))
    sim.close()


@pytest.mark.parametrize("n,heavies", [(1, 1), (2, 0), (33, 2), (257, 4), (700, 300), (2047, 4), (2048, 4),
                                       (2305, 0), (6145, 256), (9000, 300)])
def test_mixed_accel_sizes(torch, n, heavies):
    """The mixed kick over one-CTA packs, tile packs, launch shapes and heavy
    lists (none, full, and longer than the 256 bodies it holds), with the
    caller's and the fixed scratch. A pair carries a few 2^-22 (separation,
    reciprocal square root cubed, products) and a sum of 64 pairs in FP32 at
    most 2^-18 of its terms' magnitudes; heavy bodies in the list are exact."""
    rng = np.random.default_rng(n)
    w = W.outer_disk(max(n - 4, 0), 1e-9, seed=3)
    x, m = w.q[:n + 1].copy(), w.m[:n + 1].copy()
    m[1:] = 10.0 ** rng.uniform(-11, -8, n)
    m[1 + rng.permutation(n)[:heavies]] = 10.0 ** rng.uniform(-6, -3, heavies)
    md, xd = torch.from_numpy(m).cuda(), torch.from_numpy(np.ascontiguousarray(x.T)).cuda()
    a, b = (torch.empty((3, n + 1), dtype=torch.float64, device="cuda") for _ in range(2))
    work = torch.empty(q.qym_accel_workspace_bytes(n + 1, q.QYM_KICK_MIXED), dtype=torch.uint8, device="cuda")
    q.qym_accel_dev(n + 1, md, xd, a, 1.0, q.QYM_KICK_MIXED, work)
    q.qym_accel_dev_static(n + 1, md, xd, b, 1.0, q.QYM_KICK_MIXED)
    assert torch.equal(a, b)
    ref, mag = _accel_ref(m, x, 1.0) if n <= 700 else _accel_ref64(torch, m, x)
    err = np.abs(a.cpu().numpy().T - np.asarray(ref, dtype=np.float64))
    assert np.all(err <= 2.0 ** -18 * np.asarray(mag, dtype=np.float64)), float((err / (mag + 1e-300)).max())


def _accel_ref64(torch, m, x):
    xb, gm = torch.from_numpy(x[1:]).cuda(), torch.from_numpy(m[1:]).cuda()
    a, mag = np.zeros(x.shape), np.zeros(x.shape)
    for i in range(0, len(xb), 512):
        d = xb[None] - xb[i:i + 512, None]
        r2 = (d * d).sum(-1)
        s = torch.where(r2 > 0, gm / (r2 * r2.sqrt()), torch.zeros_like(r2))
        t = s[..., None] * d
        a[1 + i:1 + i + 512] = t.sum(1).cpu().numpy()
        mag[1 + i:1 + i + 512] = t.abs().sum(1).cpu().numpy()
    return a, mag


@pytest.mark.parametrize("n", [1, 63, 65, 4 * 64 * 152, 4 * 64 * 152 + 1])
@pytest.mark.parametrize("e", [0.0, 0.003, 0.5, 0.97])
def test_kepler_sizes_and_brackets(torch, n, e):
    """E_Kep at the edges of its CTA sizes, on orbits whose root lies at its
    bracket's end (circular), inside it, and beyond the FP32 bracket's domain
    (nearly radial), forwards and backwards: the orbits' elements propagated
    (the mean anomaly advanced). A point that meets the 1e-14 residual is off in
    phase by that per orbit covered, and by 1/(1 - e) of it near pericentre (as
    test_kepler_matches_oracle)."""
    rng = np.random.default_rng(n)
    k = min(n, 2000)
    a = 10.0 ** rng.uniform(-0.3, 1.7, k)
    ang = [rng.uniform(0, np.pi, k)] + [rng.uniform(0, 2 * np.pi, k) for _ in range(3)]
    orbit = lambda M: W.elements_to_cartesian(1.0, a, np.full(k, e), *ang[:3], M)
    qq, vv = (np.resize(x, (n, 3)) for x in orbit(ang[3]))
    q0, v0 = (torch.from_numpy(np.ascontiguousarray(x.T)).cuda() for x in (qq, vv))
    q1, v1 = torch.empty_like(q0), torch.empty_like(v0)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    for dt in (W.TAU_A5, -0.3):
        r1, u1 = orbit(ang[3] + dt / a ** 1.5)
        scale = (1.0 + abs(dt) / (2 * np.pi * a ** 1.5)) / (1.0 - e)
        for solver in (q.QYM_SOLVER_LAGUERRE, q.QYM_SOLVER_NEWTON32):
            q.qym_kepler_drift_dev(n, q0, v0, q1, v1, 1.0, dt, solver, status=st)
            for got, ref in ((q1, r1), (v1, u1)):
                g = got.cpu().numpy().T
                d = np.linalg.norm(g[:k] - ref, axis=1) / np.linalg.norm(ref, axis=1)
                assert np.all(d <= 1e-12 * scale), float((d / scale).max())
                if n > k:  # copies of the same bodies, in other lanes and CTAs
                    assert np.abs(g - np.resize(g[:k], g.shape)).max() <= 1e-12 * np.abs(g).max() * scale.max()
    assert st.item() == 0


@pytest.mark.parametrize("n", [40, 1000, 1100, 8191, 8192, 9000])
def test_sets_sizes(torch, n):
    """The set builder in one CTA (up to 8192 rows) and in its seven kernels,
    on a disk crowded around a planet (large sets, many pairs): after a step the
    records' connected components are the sets counted, the largest of them the
    largest set, and a rerun on a fresh context gives the same bits."""
    import networkx as nx
    w = W.outer_disk(n - 4, 1e-9, seed=n, a_lo=9.0, a_hi=10.0 if n < 2000 else 40.0)
    out = []
    for _ in range(2):
        sim = q.Simulation(w.m, w.q, w.v, w.offsets, eps_H=w.eps_H)
        sim.step(0.2 * w.tau, 1)
        out.append((*sim.state(), sim.encounters(), sim.stats()))
        sim.close()
    (q0, v0, rec, st), (q1, v1, rec1, _) = out
    g = nx.Graph(list(map(tuple, rec[:, 1:])))
    comps = [len(c) for c in nx.connected_components(g)]
    assert len(rec) > 0 and st["sets"] == len(comps) and st["max_set"] == max(comps)
    assert np.array_equal(rec, rec1) and np.array_equal(q0, q1) and np.array_equal(v0, v1)


@pytest.mark.parametrize("n", [8192, 8705, 16385, 33000])
@pytest.mark.parametrize("equal", [True, False])
def test_pairs_once(torch, n, equal):
    """One kick with each pair formed once against the one-sided form (a launch
    shape set by hand) and the FP64 kick, bodies of one mass and of several, a
    ragged last block: the velocity change of a kick within 2^-18 of the sum of
    the pulls' magnitudes of the FP64 one (as test_mixed_accel_sizes; here by
    the largest pull of any body), and the two FP32 forms' errors alike."""
    w = W.outer_disk(n - 4, 1e-10, seed=n)
    m = w.m.copy()
    if not equal:
        m[5:] *= 10.0 ** np.random.default_rng(n).uniform(-1, 1, n - 4)
    tau = 1e-3
    dv = []
    for prec, shape in ((q.QYM_KICK_FP64, None), (q.QYM_KICK_MIXED, None), (q.QYM_KICK_MIXED, (128, 2, 16))):
        # no heavy split: every pull goes through the FP32 pairs
        sim = q.Simulation(m, w.q, np.zeros_like(w.v), w.offsets, kick_prec=prec, encounters=0, heavy_mass=0.0,
                           coords=1, G=1e-6)
        if prec == q.QYM_KICK_MIXED:
            assert sim.stats()["kick_tile_i"] == 512
        if shape:
            q.qym_set_kick_shape(sim.ctx, *shape)
            assert sim.stats()["kick_tile_i"] == 256
        sim.step(tau, 1)
        dv.append(sim.state()[1])
        sim.close()
    a = [np.linalg.norm(x - dv[0], axis=1) for x in dv[1:]]
    big = np.linalg.norm(dv[0], axis=1).max()
    assert big > 0 and max(x.max() for x in a) <= 2.0 ** -18 * big
    rms = [np.sqrt((x ** 2).mean()) for x in a]
    assert rms[0] <= 1.5 * rms[1] + 1e-16 * big, (rms, big)


# (members, cluster, swarm mass, systems): either side of each lane layout of a block
# step: partners of up to 8, 16 and 32 lanes a member, the list of near pairs up to a
# warp's, up to three warps' (light swarm: only the planet pulls) and beyond (heavy
# swarm: most pairs are near), one CTA, clusters, a batch with more large sets than
# clusters
HERM_CASES = [(2, 0, 1e-12, 1), (8, 0, 1e-12, 1), (9, 0, 1e-6, 1), (17, 0, 1e-12, 1), (23, 0, 1e-12, 1),
              (23, 0, 1e-6, 1), (24, 8, 1e-12, 1), (33, 2, 1e-6, 1), (65, 4, 1e-12, 1), (130, 8, 1e-12, 1),
              (33, 0, 1e-12, 156), (26, 0, 1e-6, 156)]


@pytest.mark.parametrize("members,cluster,mass,systems", HERM_CASES)
def test_hermite_layouts(torch, oracle, members, cluster, mass, systems):
    """A planet's swarm as one encounter set through the Hermite: the oracle's
    records, and positions within the larger of 1e-11 and 100 times what one ulp in
    the initial positions moves a body (the sums run in another order)."""
    from test_gpu_step import _chaos_spread, _check_positions, _compare_records, _planet_swarm, _run_gpu, _run_oracle
    sw = [_planet_swarm(members - 1, seed=1000 + members + s) for s in range(systems)]
    for x in sw:
        x.m[2:] = mass
    cat = [np.concatenate([getattr(x, k) for x in sw]) for k in "mqv"]
    offs = np.cumsum([0] + [len(x.m) for x in sw])
    w = W.Workload("swarms", *cat, offs, sw[0].tau, 2)
    qg, vg, enc, st, E = _run_gpu(w, 2, kick_prec=q.QYM_KICK_FP64, hermite_cluster=cluster)
    assert st["status_bits"] == 0 and st["max_set"] == members
    for s in {0, systems // 2, systems - 1}:
        a, b = int(offs[s]), int(offs[s + 1])
        r, _ = _run_oracle(oracle, sw[s], 2)
        mine = enc[(enc[:, 1] >= a) & (enc[:, 1] < b)].copy()
        mine[:, 1:] -= a
        skip = _compare_records(mine, r)
        keep = np.array([i not in skip for i in range(b - a)])
        _check_positions(qg[a:b][keep], r.q[keep], _chaos_spread(oracle, sw[s], 2)[keep], rel=1e-11)


@pytest.mark.parametrize("n", [70, 1216, 1217])
def test_finisher_rows(torch, oracle, n):
    """The finisher with 32 threads a row (up to 1216 rows) and with eight, a ragged
    last CTA: a step with the FP64 kick and no encounters against the oracle's,
    within 1e-12 (as the plain step's parity)."""
    from test_gpu_step import _relq, _run_gpu, _run_oracle
    w = W.outer_disk(n - 5, 1e-9, seed=n)
    assert len(w.m) == n
    qg, vg, *_ = _run_gpu(w, 1, kick_prec=q.QYM_KICK_FP64, encounters=0)
    r, vh = _run_oracle(oracle, w, 1, encounters=0)
    assert _relq(qg, r.q).max() <= 1e-12 and _relq(vg, vh).max() <= 1e-12


@pytest.mark.parametrize("n", [64, 1024, 16384])
def test_gradient_rounds(torch, n):
    """A minibatch's gradient is the sum of its 64-row rounds' gradients, added
    as FP64 adds them and rounded once, bit for bit (up to 256 rounds, one each
    to a CTA; every factor 2/n is a power of two, so a round's sums in FP32 and
    its bf16 operands only change exponents). The grouping matters: training
    turns one last place of a weight into 2^-9 where it crosses a bf16 midpoint."""
    rows = torch.from_numpy(W.mlp_rows_synthetic(n, 21)).cuda()
    ref = W.mlp_rows_synthetic(4096, 22)
    w = torch.from_numpy(W.mlp_init(6, ref[:, :4], ref[:, 4])).cuda()
    work = torch.empty(q.qym_mlp_workspace_bytes(), dtype=torch.uint8, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")

    def grad(r):
        g = torch.empty(q.QYM_MLP_NW, dtype=torch.float32, device="cuda")
        q.qym_mlp_grad_dev(len(r), w, r, g, loss, work)
        return g.cpu().numpy()

    parts = np.array([grad(rows[i:i + 64]) for i in range(0, n, 64)], dtype=np.longdouble)
    assert np.array_equal(grad(rows), (parts.sum(0) * (64 / n)).astype(np.float64).astype(np.float32))


def test_training_is_its_steps(torch):
    """Training over many minibatches gives the bits of the gradient and Adam
    calls with the stream synchronised after each: no kernel of the chain reads
    a weight or a partial sum from before the kernel that writes it."""
    n, batch, epochs, lr, lr1 = 40000, 1000, 3, 2e-3, 2e-5
    rows = torch.from_numpy(W.mlp_rows_synthetic(n, 23)).cuda()
    ref = W.mlp_rows_synthetic(4096, 24)
    w0 = torch.from_numpy(W.mlp_init(7, ref[:, :4], ref[:, 4])).cuda()
    work = torch.empty(q.qym_mlp_workspace_bytes(), dtype=torch.uint8, device="cuda")
    a = [w0.clone(), torch.zeros_like(w0), torch.zeros_like(w0)]
    b = [x.clone() for x in a]
    steps = n // batch * epochs
    losses = torch.empty(steps, dtype=torch.float32, device="cuda")
    q.qym_mlp_train_dev(*a, 0, rows, n, batch, epochs, lr, lr1, losses, work)
    g = torch.empty(q.QYM_MLP_NW, dtype=torch.float32, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    lr, lr1 = float(np.float32(lr)), float(np.float32(lr1))
    for s in range(steps):
        lo = s % (n // batch) * batch
        q.qym_mlp_grad_dev(batch, b[0], rows[lo:lo + batch], g, loss, work)
        torch.cuda.synchronize()
        assert loss.item() == losses[s].item()
        rate = lr1 + 0.5 * (lr - lr1) * (1.0 + np.cos(np.pi * s / steps))
        q.qym_mlp_adam_dev(*b, g, s + 1, rate)
        torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(a, b))


def _batch_bits():
    import os
    return np.load(os.path.join(os.path.dirname(__file__), "golden", "batch_bits.npz"))


def _same_bits(got, ref):
    assert np.array_equal(got, ref), (np.mean(got != ref), np.abs(got - ref).max())


@pytest.mark.parametrize("name,dt", [("fwd", 2 * np.pi / 40), ("back", -0.7)])
def test_kepler_bits(torch, name, dt):
    """E_Kep by Laguerre's method, bound and unbound orbits: the bits of the form
    with IEEE square roots and divisions throughout (recorded)."""
    g = _batch_bits()
    q0, v0 = torch.from_numpy(g["kepler_q"]).cuda(), torch.from_numpy(g["kepler_v"]).cuda()
    q1, v1 = torch.empty_like(q0), torch.empty_like(v0)
    q.qym_kepler_drift_dev(q0.shape[1], q0, v0, q1, v1, 1.0, dt, q.QYM_SOLVER_LAGUERRE, q.QYM_GUESS_STANDARD)
    _same_bits(q1.cpu().numpy(), g[f"kepler_{name}_q"])
    _same_bits(v1.cpu().numpy(), g[f"kepler_{name}_v"])


@pytest.mark.parametrize("kind,encounters", [("plain", 0), ("step", 1)])
@pytest.mark.parametrize("name", ["disks", "swarms"])
def test_batch_bits(torch, name, kind, encounters):
    """Two steps of small batches (planetesimal disks; planets' swarms of 2 to 70
    members) with the mixed kick: the recorded bits. Encounters amplify a last
    place by up to 1e9 within a few steps of an ensemble, so a change of grouping
    or rounding anywhere in a batch's step shows in its results."""
    g = _batch_bits()
    sim = q.Simulation(g[name + "_m"], g[name + "_q"], g[name + "_v"], g[name + "_offsets"], eps_H=4.7e-4,
                       encounters=encounters)
    sim.step(2 * np.pi / 40, 2)
    qs, vs = sim.state()
    sim.close()
    _same_bits(qs, g[f"{name}_{kind}_q"])
    _same_bits(vs, g[f"{name}_{kind}_v"])


def _sums_case(n):
    """Bodies in a flat box by exact arithmetic (the same on every machine), each
    eighth beside its neighbour, of one mass (odd n) or several, four heavy ones;
    and the rows whose accelerations are recorded."""
    rng = np.random.default_rng(n)
    x = (rng.random((n + 1, 3)) - 0.5) * np.array([2.0, 2.0, 0.125])
    near = np.arange(8, n, 8)
    x[near] = x[near + 1] + (rng.random((len(near), 3)) - 0.5) * 2.0 ** -9
    m = np.full(n + 1, 1.3 * 2.0 ** -30) * (1.0 if n % 2 else 1.0 + 7.0 * rng.random(n + 1))
    m[0], m[3:7] = 1.0, 2.0 ** -10
    x[0] = 0.0
    return m, x, np.unique(np.concatenate([near[:: max(1, len(near) // 64)], np.arange(1, n + 1, max(1, n // 64))]))


SUMS = [65, 110, 259, 1023, 1493, 2047, 2048, 2443, 6145, 9001, 20490]


@pytest.mark.parametrize("n", SUMS)
def test_mixed_accel_sums(torch, n):
    """Mixed accelerations against recorded ones: the same roundings of each pair's
    pull and the same FP32 sums of 64 bodies, whatever the ranges of a launch. What
    the ranges leave free are sums of at most 320 two-float parts (2^-48 each) and of
    64 doubles: below 2^-39 of the terms' magnitudes, while another rounding of a
    dominating pair is some 2^-24."""
    import os
    ref = np.load(os.path.join(os.path.dirname(__file__), "golden", "accel_sums.npz"))["a%d" % n]
    m, x, rows = _sums_case(n)
    md, xd = torch.from_numpy(m).cuda(), torch.from_numpy(np.ascontiguousarray(x.T)).cuda()
    a = torch.empty((3, n + 1), dtype=torch.float64, device="cuda")
    work = torch.empty(q.qym_accel_workspace_bytes(n + 1, q.QYM_KICK_MIXED), dtype=torch.uint8, device="cuda")
    q.qym_accel_dev(n + 1, md, xd, a, 1.0, q.QYM_KICK_MIXED, work)
    mag = _accel_ref64(torch, m, x)[1][rows]
    err = np.abs(a.cpu().numpy().T[rows] - ref)
    assert np.all(err <= 2.0 ** -39 * mag), float((err / mag).max())


# lengths and masses in cgs, SI and parsecs, and around AU and solar masses (G folded
# into the masses): r^-3 of a disk's pairs lies below, at the end of, above and inside
# FP32's range
UNITS = [(1.5e13, 1.3e26), (1.5e11, 1.3e20), (4.85e-6, 4.3e-3), (1e-6, 1.0), (1e-12, 1e-9), (1.0, 1.0)]


@pytest.mark.parametrize("n", [300, 2100, 9000])
@pytest.mark.parametrize("lu,mu", UNITS)
@pytest.mark.parametrize("equal", [True, False])
def test_mixed_accel_units(torch, n, lu, mu, equal):
    """The mixed kick in the caller's units, bodies of one mass (windows that
    multiply by it once) and of several, with two close pairs and one body far
    outside: the bound of test_mixed_accel_sizes."""
    rng = np.random.default_rng(n)
    w = W.outer_disk(n - 4, 1e-9, seed=3)
    x, m = w.q.copy(), w.m.copy()
    if not equal:
        m[5:] = 10.0 ** rng.uniform(-11, -8, n - 4)
    x[60] *= 1e3
    x, m = x * lu, m * mu
    sep = max(1e-13 * lu, 1e-14)  # (r^2 stays a normal float)
    x[10] = x[9] + [sep, 0.0, 0.0]
    x[40] = x[39] + [0.0, 3 * sep, -2 * sep]
    # (the split positions resolve 2^-48 of a coordinate: the close pairs as the kernel sees them)
    hi = x.astype(np.float32)
    x = hi.astype(np.float64) + (x - hi).astype(np.float32)
    md, xd = torch.from_numpy(m).cuda(), torch.from_numpy(np.ascontiguousarray(x.T)).cuda()
    a = torch.empty((3, n + 1), dtype=torch.float64, device="cuda")
    work = torch.empty(q.qym_accel_workspace_bytes(n + 1, q.QYM_KICK_MIXED), dtype=torch.uint8, device="cuda")
    q.qym_accel_dev(n + 1, md, xd, a, 1.0, q.QYM_KICK_MIXED, work)
    ref, mag = _accel_ref64(torch, m, x)
    err = np.abs(a.cpu().numpy().T - ref)
    assert np.all(err <= 2.0 ** -18 * mag), float((err / (mag + 1e-300)).max())


@pytest.mark.parametrize("lu,mu", UNITS)
@pytest.mark.parametrize("equal", [True, False])
def test_pairs_once_units(torch, lu, mu, equal):
    """The pairs-once kick in the caller's units: test_pairs_once's bound against
    the FP64 kick, and a step's encounters those of the one-sided kick and of the
    FP64 kick."""
    n = 8705
    w = W.outer_disk(n - 4, 1e-10, seed=n)
    m = w.m.copy()
    if not equal:
        m[5:] *= 10.0 ** np.random.default_rng(n).uniform(-1, 1, n - 4)
    # unit time: that of the disk's own units, lu^3 = G mu
    t, G = np.sqrt(lu ** 3 / mu), 1.0
    dv, rec = [], []
    for prec, shape in ((q.QYM_KICK_FP64, None), (q.QYM_KICK_MIXED, None), (q.QYM_KICK_MIXED, (128, 2, 16))):
        sim = q.Simulation(m * mu, w.q * lu, np.zeros_like(w.v), w.offsets, kick_prec=prec, encounters=0,
                           heavy_mass=0.0, coords=1, G=1e-6 * G)
        if shape:
            q.qym_set_kick_shape(sim.ctx, *shape)
        sim.step(1e-3 * t, 1)
        dv.append(sim.state()[1] / (lu / t))
        sim.close()
        sim = q.Simulation(m * mu, w.q * lu, w.v * (lu / t), w.offsets, kick_prec=prec, eps_H=w.eps_H * lu, G=G)
        if shape:
            q.qym_set_kick_shape(sim.ctx, *shape)
        sim.step(w.tau * t, 2)
        rec.append(sim.encounters())
        assert sim.stats()["status_bits"] == 0
        sim.close()
    a = [np.linalg.norm(x - dv[0], axis=1) for x in dv[1:]]
    big = np.linalg.norm(dv[0], axis=1).max()
    assert big > 0 and max(x.max() for x in a) <= 2.0 ** -18 * big
    rms = [np.sqrt((x ** 2).mean()) for x in a]
    assert rms[0] <= 1.5 * rms[1] + 1e-16 * big, (rms, big)
    assert len(rec[0]) > 0 and np.array_equal(rec[0], rec[1]) and np.array_equal(rec[0], rec[2])


def test_partial_sums_memory(torch):
    """A system whose pairs-once partial sums would pass 2 GB (24 bytes a row and
    range, 128 ranges: 699050 rows) takes the one-sided kick and holds no such
    slots: less device memory than a somewhat smaller one, by most of 2 GB."""
    held = []
    for n in (690000, 705000):
        w = W.outer_disk(n - 4, 1e-12, seed=1)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        sim = q.Simulation(w.m, w.q, w.v, w.offsets, encounters=0)
        held.append((free - torch.cuda.mem_get_info()[0], sim.stats()["kick_tile_i"]))
        sim.close()
    assert held[0][1] == 512 and held[1][1] == 256
    assert held[1][0] < held[0][0] - (1 << 30), held


def _energy_ref(w, lo, hi):
    """Energy of the system of rows [lo, hi) in extended precision (DH velocities),
    and the sum of its terms' magnitudes."""
    L = np.longdouble
    m, x, v = (a[lo:hi].astype(L) for a in (w.m, w.q, w.v))
    mb, xb, vb = m[1:], x[1:], v[1:]
    S = (mb[:, None] * vb).sum(0)
    kin, star, pair = (mb * (vb * vb).sum(1) / 2).sum(), (m[0] * mb / np.sqrt((xb * xb).sum(1))).sum(), L(0)
    for i in range(len(mb)):
        pair += (mb[i] * mb[i + 1:] / np.sqrt(((xb[i + 1:] - xb[i]) ** 2).sum(1))).sum()
    return (S * S).sum() / (2 * m[0]) + kin - star - pair, kin + star + pair


def test_energy_unbalanced_batch(torch):
    """Energy of many two-body systems beside a large one, against extended
    precision (bound of test_energy_blocks) for the large one and a sample, and
    the device memory that the batch holds: with the large system's count of
    ranges for every i-block the partial sums alone would take 20000 x 125 x 8
    bytes more than they do."""
    pairs, big = 20000, 3000
    one = W.outer_disk(big - 4, 1e-9, seed=1)
    rng = np.random.default_rng(2)
    m2 = np.stack([np.ones(pairs), 10.0 ** rng.uniform(-9, -3, pairs), 10.0 ** rng.uniform(-9, -3, pairs)], 1)
    x2, v2 = rng.normal(size=(2, pairs, 3, 3))
    x2[:, 0] = v2[:, 0] = 0.0
    cat = lambda a, b: np.concatenate([a.reshape(-1, *b.shape[1:]), b, a[:100].reshape(-1, *b.shape[1:])])
    n = np.concatenate([np.full(pairs, 3), [big + 1], np.full(100, 3)])
    w = W.Workload("mix", cat(m2, one.m), cat(x2, one.q), cat(v2, one.v), np.concatenate([[0], np.cumsum(n)]), one.tau, 1)
    held = []
    for k in (pairs + 101, pairs):  # with and without the large system (the last 101)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        rows = int(w.offsets[k])
        sim = q.Simulation(w.m[:rows], w.q[:rows], w.v[:rows], w.offsets[:k + 1], coords=1, encounters=0)
        held.append(free - torch.cuda.mem_get_info()[0])
        if k > pairs:
            E = sim.energy()
        sim.close()
    for s in [0, 1, 777, pairs - 1, pairs, pairs + 1, pairs + 100]:
        ref, mag = _energy_ref(w, int(w.offsets[s]), int(w.offsets[s + 1]))
        assert abs(E[s] - ref) <= (n[s] + 8) * np.longdouble(2.0) ** -53 * mag, s
    assert held[0] - held[1] < (12 << 20), held


@pytest.mark.parametrize("n", [1000, 9000])
def test_split_launch_count(torch, n):
    """qym_stats.launches of a split step: the library's kernels that the
    profiler sees, with the set builder in one kernel and in seven (FP64 kick: no
    tile preparation, which no count includes)."""
    from torch.profiler import ProfilerActivity, profile
    from paper_1007_3458_gb300 import split as SP
    from test_gpu_split import LocalComm
    w = W.outer_disk(n - 5, 1e-9, seed=n)
    sim = q.Simulation(w.m, w.q, w.v, w.offsets, eps_H=w.eps_H, kick_prec=q.QYM_KICK_FP64)
    run = SP.SplitRun(SP.GpuEngine(sim, 0, 1), LocalComm())
    run.step(w.tau, 1)
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]):  # (the first session of a process may record nothing)
        torch.zeros(8, device="cuda").add_(1)
        torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        run.step(w.tau, 3)
        torch.cuda.synchronize()
    seen = [e.name for e in prof.events() if e.name.replace("void ", "").startswith(("qym::", "k_"))]
    launches = sim.stats()["launches"]
    sim.close()
    if not seen:
        pytest.skip("no kernel records from the profiler")
    assert launches == len(seen), (launches, len(seen))


@pytest.mark.parametrize("lu,mu", [(1e6, 1e40), (1e9, 1e40), (1e-9, 1e-40), (1e-8, 1e24), (1.5e13, 1.3e26)])
@pytest.mark.parametrize("prec", [q.QYM_KICK_FP64, q.QYM_KICK_MIXED])
def test_crude_reach_units(torch, lu, mu, prec):
    """A step's encounters in units where the star's G m (1e40, 1e-40) or its
    quotient by r^3 leaves FP32's range, or pulls come near its end, and in cgs:
    those of the disk's own units."""
    n = 2000
    if prec == q.QYM_KICK_MIXED and mu in (1e24, 1e-40):
        pytest.skip("pulls or weights of the bodies outside FP32's range")
    w = W.outer_disk(n - 4, 1e-9, seed=5, a_lo=9.0, a_hi=14.0)
    rec = []
    for a, b in ((1.0, 1.0), (lu, mu)):
        t = np.sqrt(a ** 3 / b)
        sim = q.Simulation(w.m * b, w.q * a, w.v * (a / t), w.offsets, eps_H=w.eps_H * a, kick_prec=prec)
        for k in range(2):  # (the first step's search follows its kick, later ones are part of it)
            sim.set_state(w.q * a, w.v * (a / t)) if k else None
            sim.step(w.tau * t, 1)
            assert sim.stats()["status_bits"] == 0
            rec.append(sim.encounters())
        sim.close()
    assert len(rec[0]) > 0 and all(np.array_equal(rec[0], r) for r in rec[1:])
