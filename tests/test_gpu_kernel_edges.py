"""Kernels at the edges of their ranges: sizes around a tile, a group or a block, and the ends of a
dispatch rule, against the FP64 oracle or against an exact relation."""
import numpy as np
import pytest

import oracle
from paper_1907_01724_gb300 import api, batch, inputs, server

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [2.0 ** -490, 2.0 ** -300, 2.0 ** 300])
@pytest.mark.parametrize("n", [1, 129])
def test_fp64_potentials_scale_with_the_cavity(n, scale):
    """A cavity scaled by a power of two has its potentials scaled by the inverse (the FP64 pair
    kernel's reciprocal roots at both ends of their range and in their fallback for tiny
    arguments)."""
    rng = np.random.default_rng(190790 + n)
    xyz, q = inputs.uniform_ball(rng, n, 1.0), rng.choice([-1.0, 1.0], n)
    phi = [api.solve(inputs.System(a, 2.0, 80.0, 1.5 / a, 12, 64, a * xyz, q), precision=api.HSMA_FP64).phi
           for a in (1.0, scale)]
    # every operation scales exactly except through the range of exponents: rounding of a few sums
    assert np.linalg.norm(phi[1] * scale - phi[0]) <= 1e-12 * np.linalg.norm(phi[0])


@pytest.mark.parametrize("n", [1, 31, 33, 129, 1437, 1438, 7428, 7429])
def test_default_tile_configurations(n):
    """The tile configuration chosen without tuning, on both sides of the rule's lines (M = 1000),
    and the layer's term at charges next to the interface: potentials and fields, 1e-6 norm-wise
    (the FP32 path's bound)."""
    rng = np.random.default_rng(190800 + n)
    k = (n + 3) // 4
    xyz = np.concatenate([inputs.shell(rng, k, 1.0, 0.02), inputs.uniform_ball(rng, n - k, 1.0)])
    q = rng.choice([-1.0, 1.0], n)
    P = oracle.make_params(a=1.0, eps1=2.0, eps2=80.0, kappa=1.5, p=12, M=1000)
    ref, E = oracle.hsma(P, xyz, q)["phi"], oracle.field(P, xyz, q)["E"]
    h = api.hsma_create(1.0, 2.0, 80.0, 1.5, api.hsma_default_params(p=12, M=1000))
    api.hsma_build_sources(h, xyz, q)
    assert np.linalg.norm(api.hsma_potential(h) - ref) <= 1e-6 * np.linalg.norm(ref)
    assert np.linalg.norm(api.hsma_field(h) - E) <= 1e-6 * np.linalg.norm(E)


@pytest.mark.parametrize("order", [8, 12, 16])
@pytest.mark.parametrize("n", [2, 5, 36, 513, 4097])
def test_tree_at_batch_edges(n, order):
    """The far-field tree where its batches of 32 and steps of 4 sources end, with charges at the
    centre's images (far), next to the interface (their own images: the exact direct sum) and in one
    dense cell, against the FP64 path's direct sum (order 8 at theta 0.35; 1e-6 norm-wise)."""
    rng = np.random.default_rng(190810 + n)
    k = n // 3
    xyz = np.concatenate([inputs.shell(rng, k, 1.0, 1e-3), inputs.uniform_ball(rng, k, 0.3),
                          np.array([0.3, 0.2, -0.4]) + inputs.uniform_ball(rng, n - 2 * k, 0.02)])
    s = inputs.System(1.0, 2.0, 80.0, 1.5, 12, 400, xyz, rng.choice([-1.0, 1.0], n))
    ref = api.solve(s, precision=api.HSMA_FP64).phi
    h = api.hsma_create(s.a, s.eps1, s.eps2, s.kappa, api.hsma_default_params(p=s.p, M=s.M))
    api.hsma_set_far_field(h, 0.35 if order == 8 else 0.5, order)
    api.hsma_build_sources(h, s.xyz, s.q)
    assert np.linalg.norm(api.hsma_potential(h) - ref) <= 1e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("M", [6, 30])
@pytest.mark.parametrize("n", [1, 2, 1024, 1025, 2049])
def test_move_energies_at_block_edges(n, M):
    """Delta E and a committed move where the row blocks (1024 rows) and the blocks of surface points
    (8) end, FP32 against FP64 path: 1e-6 of the moved charge's Coulomb terms and of Delta E."""
    rng = np.random.default_rng(190820 + n)
    xyz, q = inputs.uniform_ball(rng, n, 0.9), rng.choice([-1.0, 1.0], n)
    k, xs = n // 2, inputs.uniform_ball(rng, 2, 0.9)
    de = {}
    for prec in (api.HSMA_FP32, api.HSMA_FP64):
        h = api.hsma_create(1.0, 2.0, 80.0, 1.5, api.hsma_default_params(p=12, M=M, precision=prec))
        api.hsma_build_sources(h, xyz, q)
        first = api.hsma_delta_energy(h, k, xs[0])
        api.hsma_apply_move(h, k, xs[0])
        de[prec] = np.array([first, api.hsma_delta_energy(h, k, xs[1])])
    kc = api.PAPER_COULOMB_K / 2.0
    others = np.delete(xyz, k, 0)
    S = kc * (sum((1.0 / np.linalg.norm(others - x, axis=1)).sum() for x in (xyz[k], xs[0], xs[1])) + 1.0)
    assert np.abs(de[api.HSMA_FP32] - de[api.HSMA_FP64]).max() <= 1e-6 * (S + np.abs(de[api.HSMA_FP64]).max())


@pytest.mark.parametrize("n, M", [(9000, 70), (13001, 2000), (16385, 130)])
def test_field_chunks_merged(n, M):
    """The FP32 field pass where two source chunks make one field chunk, the last of them not full
    (N = 13001), and next to that range, against the FP64 field pass: 1e-6 norm-wise for each output."""
    rng = np.random.default_rng(190830 + n)
    xyz, q = inputs.uniform_ball(rng, n, 1.0), rng.choice([-1.0, 1.0], n)
    out = {}
    for prec in (api.HSMA_FP32, api.HSMA_FP64):
        h = api.hsma_create(1.0, 2.0, 80.0, 1.5, api.hsma_default_params(p=12, M=M, precision=prec))
        api.hsma_build_sources(h, xyz, q)
        out[prec] = [api.hsma_field(h, w) for w in (api.HSMA_TOTAL, api.HSMA_COULOMB, api.HSMA_REACTION)]
    for a, b in zip(out[api.HSMA_FP32], out[api.HSMA_FP64]):
        assert np.linalg.norm(a - b) <= 1e-6 * np.linalg.norm(b)


@pytest.mark.parametrize("sizes", [(1, 127, 129, 9000), (511, 513, 2047, 16385), (64, 1000, 1024, 30000)])
def test_server_energies_of_unequal_chains(sizes):
    """Full energies of resident chains next to a much larger one (each chain's own share of pair
    items, blocks of one group and ragged ones), against the FP64 path: |dE| <= f |q| |dphi| with
    E = f q.phi and the FP32 path's bound |dphi| <= 1e-6 |phi|."""
    rng = np.random.default_rng(190840 + sum(sizes))
    chains = [inputs.System(1.0, 2.0, 80.0, 1.5, 12, 200, inputs.uniform_ball(rng, n, 1.0), rng.choice([-1.0, 1.0], n))
              for n in sizes]
    srv = server.Server(chains)
    srv.hsma_server_load()
    reqs = np.zeros(len(sizes), dtype=server.REQUEST)
    reqs["id"] = reqs["chain"] = np.arange(len(sizes))
    reqs["kind"] = server.REQ_ENERGY
    res = srv.hsma_server_run(reqs)
    assert (res["status"] == 0).all()
    for r in res:
        s = chains[r["chain"]]
        h = api.hsma_create(s.a, s.eps1, s.eps2, s.kappa, api.hsma_default_params(p=s.p, M=s.M, precision=api.HSMA_FP64))
        api.hsma_build_sources(h, s.xyz, s.q)
        phi, E = api.hsma_potential(h), api.hsma_energy(h)[0]
        f = abs(E / (s.q @ phi))
        assert abs(r["value"] - E) <= 1e-6 * f * np.linalg.norm(s.q) * np.linalg.norm(phi)


@pytest.mark.parametrize("threads, k", [(128, 1), (64, 2), (64, 4), (128, 8)])
@pytest.mark.parametrize("length, charge", [(2.0 ** -32, 2.0 ** -64), (2.0 ** 24, 2.0 ** 20)])
def test_fp32_potentials_scale_with_lengths_and_charges(threads, k, length, charge):
    """Lengths and charges scaled by powers of two (a cavity of nanometres in metres, with charges of
    an electron in coulombs): every FP32 operation scales exactly while its result stays a normal
    number, so the potentials are those of the unscaled cavity times charge / length; the FP32
    path's own bound, 1e-6 norm-wise, is allowed."""
    rng = np.random.default_rng(190850)
    xyz, q = inputs.uniform_ball(rng, 300, 1.0), rng.choice([-1.0, 1.0], 300)
    cfg = [tuple(c) for c in batch.pair_configs()].index((threads, k, 4))
    phi = []
    for s, t in ((1.0, 1.0), (length, charge)):
        b = batch.from_systems([inputs.System(s, 2.0, 80.0, 1.5 / s, 12, 1000, s * xyz, t * q)])
        b.hsma_batch_set_pair_config(cfg)
        b.hsma_batch_build_sources(np.array([300]), s * xyz, t * q)
        phi.append(b.hsma_batch_potential(api.HSMA_REACTION) * s / t)
    assert np.linalg.norm(phi[1] - phi[0]) <= 1e-6 * np.linalg.norm(phi[0])


def _with_tiles(s, tiles, evaluate):
    b = batch.from_systems([s])
    b.hsma_batch_set_pair_config([tuple(c) for c in batch.pair_configs()].index(tiles))
    b.hsma_batch_build_sources(np.array([s.n]), s.xyz, s.q)
    return evaluate(b)


TILES = [(128, 1, 4), (64, 2, 4), (64, 4, 8)]  # by work: below 6e6, below 7.5e7, above


@pytest.mark.parametrize("line, n", [(6.0e6, 1437), (7.5e7, 5807)])
def test_tile_rule_on_both_sides_of_its_lines(line, n):
    """The untuned choice by the work N (2 N + 1.3 M), M = 1000, for the last size below a line and the
    first above it: the potentials are those of that configuration to the bit, not those of the
    neighbour's, and within 1e-6 of the oracle (the FP32 path's bound)."""
    assert n * (2.0 * n + 1300.0) < line <= (n + 1) * (2.0 * n + 1302.0)
    below = 0 if line == 6.0e6 else 1
    for size, mine, other in ((n, TILES[below], TILES[below + 1]), (n + 1, TILES[below + 1], TILES[below])):
        rng = np.random.default_rng(190880 + size)
        s = inputs.System(1.0, 2.0, 80.0, 1.5, 12, 1000, inputs.uniform_ball(rng, size, 1.0), rng.choice([-1.0, 1.0], size))
        h = api.hsma_create(s.a, s.eps1, s.eps2, s.kappa, api.hsma_default_params(p=s.p, M=s.M))
        api.hsma_build_sources(h, s.xyz, s.q)
        phi = api.hsma_potential(h)
        assert np.array_equal(phi, _with_tiles(s, mine, lambda b: b.hsma_batch_potential()))
        assert not np.array_equal(phi, _with_tiles(s, other, lambda b: b.hsma_batch_potential()))
        ref = oracle.hsma(oracle.make_params(a=1.0, eps1=2.0, eps2=80.0, kappa=1.5, p=12, M=1000), s.xyz, s.q)["phi"]
        assert np.linalg.norm(phi - ref) <= 1e-6 * np.linalg.norm(ref)


@pytest.mark.parametrize("n, tiles", [(300, (128, 1, 4)), (1437, (128, 1, 4)), (1438, (64, 4, 4)), (7428, (64, 4, 4)),
                                      (20000, (64, 4, 4))])
def test_field_pass_has_its_own_tiles(n, tiles):
    """The untuned field pass, M = 1000: the pair pass's smallest tiles below a work N (2 N + 1.3 M) of
    6e6, CTAs of 64 threads with 4 targets each above, whatever the pair pass takes there: fields and
    the potentials of the same pass are those of that configuration to the bit, potentials of a later
    pass again those of the pair pass, and the chunks cover every source (1e-6 of the FP64 field pass)."""
    rng = np.random.default_rng(190890 + n)
    s = inputs.System(1.0, 2.0, 80.0, 1.5, 12, 1000, inputs.uniform_ball(rng, n, 1.0), rng.choice([-1.0, 1.0], n))
    out = {}
    for prec in (api.HSMA_FP32, api.HSMA_FP64):
        h = api.hsma_create(s.a, s.eps1, s.eps2, s.kappa, api.hsma_default_params(p=s.p, M=s.M, precision=prec))
        api.hsma_build_sources(h, s.xyz, s.q)
        pairs = api.hsma_potential(h)
        api.hsma_build_sources(h, s.xyz, s.q)
        out[prec] = [api.hsma_field(h).reshape(-1), api.hsma_potential(h)]
        api.hsma_build_sources(h, s.xyz, s.q)
        assert np.array_equal(api.hsma_potential(h), pairs)
    want = _with_tiles(s, tiles, lambda b: [np.reshape(b.hsma_batch_field(), -1), b.hsma_batch_potential()])
    for a, b, c in zip(out[api.HSMA_FP32], want, out[api.HSMA_FP64]):
        assert np.array_equal(a, b)
        assert np.linalg.norm(a - c) <= 1e-6 * np.linalg.norm(c)


def test_fp64_reciprocal_roots():
    """The FP64 pair kernel's 1/d over random distances at many exponents, inside its fast range, at
    both of its ends (d^2 = 2^-959 and 2^898) and in the fallback past them: 2048 cavities with a unit
    charge at +d/2 and one at -d/2, whose Coulomb potentials are 1/d of d^2 = fl(d d) with no other
    rounding.  In the fast range the last operation's rounding, 2^-53, and the terms left out, below
    2^-58, are allowed; in the fallback those of a root and a division, 2^-52 together."""
    rng = np.random.default_rng(190870)
    exps = np.repeat([-505, -490, -481, -480, -479, -478, -300, -1, 0, 1, 300, 447, 448, 449, 450, 500], 128)
    d = np.ldexp(rng.uniform(1.0, 2.0, exps.size), exps)
    x = np.zeros((exps.size, 2, 3))
    axis = np.arange(exps.size) % 3
    x[np.arange(exps.size), 0, axis], x[np.arange(exps.size), 1, axis] = 0.5 * d, -0.5 * d
    b = batch.Batch(d, np.ones_like(d), np.full_like(d, 2.0), np.zeros_like(d),
                    api.hsma_default_params(p=2, M=4, coulomb_k=1.0, precision=api.HSMA_FP64))
    b.hsma_batch_build_sources(np.full(exps.size, 2), x.reshape(-1, 3), np.ones(2 * exps.size))
    phi = b.hsma_batch_potential(api.HSMA_COULOMB).reshape(-1, 2).astype(np.longdouble)
    d2 = (d * d).astype(np.longdouble)[:, None]
    err = np.abs(phi * phi * d2 - 1.0) / 2.0
    fast = (d2 >= np.ldexp(np.longdouble(1.0), -959)) & (d2 < np.ldexp(np.longdouble(1.0), 898))
    assert 0 < fast.sum() < fast.size
    assert (err <= np.where(fast, 2.0 ** -53 + 2.0 ** -58, 2.0 ** -52)).all(), err.max() * 2.0 ** 53


@pytest.mark.parametrize("tau, dy_rel", [(0.1, 0.4), (0.01, 0.08), (0.25, 0.1)])
def test_fp64_dipole_shells_among_the_charges(tau, dy_rel):
    """The FP64 path's central difference with its inner shell inside the cavity, where charges come
    close to it (here within d = 1e-6 a, and within 1e-9 a for one), and with the shell outside:
    against the oracle.  A distance d of points at |x| ~ a is known to 2^-52 a / d on either side;
    a few such roundings of the nearest point's term, which is the largest, are allowed."""
    rng = np.random.default_rng(190860)
    P = oracle.make_params(a=1.0, eps1=2.0, eps2=80.0, kappa=1.5, p=12, M=200, tau=tau, dy_rel=dy_rel)
    F2 = 99
    F1, j = round(F2 * (5.0 ** 0.5 - 1.0) / 2.0), np.arange(3, 97, 6)
    z = -1.0 + 2.0 * j / F2
    c, ang = z + np.sin(np.pi * z) / np.pi, np.pi * j * F1 / F2
    yhat = np.stack([np.sqrt(1.0 - c * c) * np.cos(ang), np.sqrt(1.0 - c * c) * np.sin(ang), c], 1)
    r = min((1.0 + tau) * (1.0 - 0.5 * dy_rel), 0.99)
    d = np.where(j == 3, 1e-9, 1e-6)
    xyz = np.concatenate([yhat * (r - d)[:, None], inputs.uniform_ball(rng, 100, 0.7)])
    q = rng.choice([-1.0, 1.0], len(xyz))
    h = api.hsma_create(1.0, 2.0, 80.0, 1.5, api.hsma_default_params(p=12, M=200, tau=tau, dy_rel=dy_rel,
                                                                     precision=api.HSMA_FP64))
    api.hsma_build_sources(h, xyz, q)
    err = np.abs(api.hsma_potential(h, api.HSMA_REACTION) - oracle.hsma(P, xyz, q)["phi_rf"])
    ref = np.abs(oracle.hsma(P, xyz, q)["phi_rf"])
    near = np.concatenate([d, np.full(100, 1e-2)])
    if r == 0.99:
        near[:] = 1e-2
    assert (err <= 16 * 2.0 ** -52 / near * ref + 1e-12 * np.linalg.norm(ref[-100:])).all()
