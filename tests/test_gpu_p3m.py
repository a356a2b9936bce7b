"""GPU P3M electrostatics (pdq_p3m_*) against the reference P3M of oracle/p3m.py
and against the exact periodic sum, through the C ABI.

The GPU and the reference take the same steps on the same mesh, so their sums
agree to rounding (atomics and FFT ordering: 1e-9 of the RMS sum); both sit
within the method's accuracy (RMS 1e-3 for a cloud with charges of both
signs) of the exact sum over the z images.
The P3M step is checked against the oracle stepping with the reference sums.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle  # noqa: E402
from oracle import p3m as ref  # noqa: E402

ST3 = [0.1, 1.0, 10.0]
GRID = dict(n_r=33, n_th=16, n_z=32)
M, NZ, AH = 32, 64, 0.5


@pytest.fixture(scope="module")
def pdq():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_04979_gb300 import build
    build.build()
    import paper_2205_04979_gb300.pdq as p
    return p


@pytest.fixture(scope="module")
def setup(pdq):
    f = pdq.Field(pdq.field_desc(**GRID), 0)
    of = oracle.field_desc(**GRID)
    grid = oracle.field_grid(of, oracle.field_modes(of, 0))
    h = 2 * 180.0 / M
    alpha = AH / h
    plan = pdq.P3M(f, M=M, Nz=NZ, alpha=alpha, r_cut=3.3 / alpha, n_img=100, max_particles=2000)
    d = ref.Desc(180.0, 720.0, M, NZ, alpha, 3.3 / alpha, n_img=100)
    return f, of, grid, plan, d, ref.influence(d)


def _cloud(counts, seed):
    rng = np.random.default_rng(seed)
    n = int(np.sum(counts))
    cls = rng.integers(0, 3, n).astype(np.int32)
    dplus = oracle.class_table(ST3)[cls, 1]
    r = (180.0 - 0.5 * dplus) * np.sqrt(rng.uniform(size=n))
    th = rng.uniform(0, 2 * np.pi, n)
    x, y, z = r * np.cos(th), r * np.sin(th), rng.uniform(0, 720.0, n)
    q = 0.05 * oracle.class_table(ST3)[cls, 4] * np.where(rng.uniform(size=n) < 0.3, -1.0, 1.0)
    v = rng.normal(0, 0.5, (n, 3))
    ids = np.concatenate([np.arange(c) for c in counts]).astype(np.int32)
    return x, y, z, q, v, cls, ids


def _state(pdq, precision, counts, arr, alive=None):
    x, y, z, q, v, cls, ids = arr
    n = len(x)
    alive = np.ones(n) if alive is None else alive
    st = pdq.State(precision, counts, ST3)
    pos, vel, xy = st.current()
    pos.copy_(torch.tensor(np.stack([x, y, z, q * alive], 1)).to(pos.dtype))
    vel.copy_(torch.tensor(np.concatenate([v, alive[:, None]], 1)).to(vel.dtype))
    if xy is not None:
        xy.copy_(torch.tensor(np.stack([x, y], 1)))
    st.tag.copy_(torch.tensor(np.stack([ids, cls], 1), dtype=torch.int32))
    return st


def _ref_sums(d, Gh, counts, x, y, z, q, alive=None):
    off = np.r_[0, np.cumsum(counts)]
    out = np.zeros((len(x), 3))
    dc = oracle.class_table(ST3)[:, 1].max()
    for s in range(len(counts)):
        sl = slice(off[s], off[s + 1])
        out[sl] = ref.coulomb_sums(d, x[sl], y[sl], z[sl], q[sl], dc, Gh, None if alive is None else alive[sl])
    return out


def _rms(a):
    return np.sqrt(np.mean(np.sum(a * a, 1)))


def test_p3m_sums_match_reference_fp64(pdq, setup):
    f, of, grid, plan, d, Gh = setup
    counts = [700, 333]
    arr = _cloud(counts, 1)
    alive = (np.random.default_rng(2).uniform(size=len(arr[0])) > 0.1).astype(np.float64)
    st = _state(pdq, 0, counts, arr, alive)
    got = plan.coulomb(pdq.phys_default(), st).cpu().numpy()
    x, y, z, q = arr[:4]
    want = _ref_sums(d, Gh, counts, x, y, z, q, alive > 0.5)
    assert np.max(np.abs(got - want)) <= 1e-9 * _rms(want)
    assert np.all(got[alive < 0.5] == 0)


def test_p3m_sums_accuracy_against_exact(pdq, setup):
    f, of, grid, plan, d, Gh = setup
    counts = [900]
    arr = _cloud(counts, 3)
    st = _state(pdq, 0, counts, arr)
    got = plan.coulomb(pdq.phys_default(), st).cpu().numpy()
    x, y, z, q = arr[:4]
    dc = oracle.class_table(ST3)[:, 1].max()
    exact = oracle.coulomb_periodic(x, y, z, q, 720.0, dc, n_img=1000)
    # charges of both signs partly cancel, so the relative error is above the 1.4e-4 of a
    # like-signed cloud; it is the reference's own error on this cloud
    want = _ref_sums(d, Gh, counts, x, y, z, q)
    assert _rms(got - exact) < 1e-3 * _rms(exact)
    assert _rms(got - exact) <= 1.001 * _rms(want - exact)


def test_p3m_sums_mixed_state(pdq, setup):
    f, of, grid, plan, d, Gh = setup
    counts = [513]
    arr = _cloud(counts, 4)
    st = _state(pdq, 1, counts, arr)
    got = plan.coulomb(pdq.phys_default(), st).cpu().numpy()
    x, y, z, q = arr[:4]
    z32, q32 = z.astype(np.float32).astype(np.float64), q.astype(np.float32).astype(np.float64)
    want = _ref_sums(d, Gh, counts, x, y, z32, q32)
    assert np.max(np.abs(got - want)) <= 1e-9 * _rms(want)


def _two_particle_errors(pdq, plan, d, Gh, a, b):
    """Error of the GPU's sums relative to the larger one, per sample of two particles a[k], b[k]."""
    n = len(a)
    X = np.stack([a, b], 1).reshape(-1, 3)
    x, y, z = X[:, 0].copy(), X[:, 1].copy(), np.mod(X[:, 2], d.L)
    q = np.tile([0.7, 0.4], n)
    st = _state(pdq, 0, [2] * n, (x, y, z, q, np.zeros((2 * n, 3)), np.full(2 * n, 2, np.int32),
                                  np.tile([0, 1], n).astype(np.int32)))
    got = plan.coulomb(pdq.phys_default(), st).cpu().numpy()
    want = _ref_sums(d, Gh, [2] * n, x, y, z, q)
    return np.abs(got - want).reshape(n, 6).max(1) / np.abs(want).reshape(n, 6).max(1)


def test_p3m_short_range_pairs_in_double(pdq, setup):
    # pairs alone in a sample from alpha r = 0.18 (below it the reference's own closed form cancels) to near r_cut.
    # Bar: a pair and its table 2^-52, the transforms over 2^18 nodes 18 2^-53 of a mesh field that is up to ~100
    # times the pair's force near r_cut (self-fields that cancel): 4e-13
    f, of, grid, plan, d, Gh = setup
    rng = np.random.default_rng(5)
    r = np.geomspace(0.18 / plan.alpha, 0.95 * plan.r_cut, 24)
    u = rng.standard_normal((24, 3))
    a = np.stack([rng.uniform(-60, 60, 24), rng.uniform(-60, 60, 24), rng.uniform(0, 720, 24)], 1)
    assert np.max(_two_particle_errors(pdq, plan, d, Gh, a, a + u * (r / np.linalg.norm(u, axis=1))[:, None])) <= 4e-13


def test_p3m_pairs_just_inside_the_cut_of_a_long_pipe(pdq):
    # a pipe whose coordinates lie on a grid of g = 8192 2^-23 in FP32: pairs 2e-4 inside r_cut whose coordinates all
    # round away from each other, by 0.98 g each, still count.  A lost pair changes the sum by K_S(r_cut) r_cut^2 =
    # 0.07 of the pair's force at alpha r_cut = 1.9; bar as above
    L, M, Nz, g = 8000.0, 16, 512, 8192.0 * 2.0 ** -23
    desc = pdq.field_desc(n_r=17, n_th=8, n_z=16)
    desc.l_plus = L
    f = pdq.Field(desc, 0)
    alpha = AH / (2 * 180.0 / M)
    side = (round(1.9 / alpha / np.sqrt(3) / g) + 0.02) * g
    rc = np.sqrt(3) * side + 2e-4
    plan = pdq.P3M(f, M=M, Nz=Nz, alpha=alpha, r_cut=rc, n_img=20, max_particles=2)
    d = ref.Desc(180.0, L, M, Nz, alpha, rc, n_img=20)
    m = np.random.default_rng(6).uniform([0, 0, 100], [60, 60, 7900], (16, 3))
    a = (np.round(m / g) + 0.51) * g
    assert np.max(_two_particle_errors(pdq, plan, d, ref.influence(d), a, a - side)) <= 1e-9


@pytest.mark.parametrize("seam", [False, True])
@pytest.mark.parametrize("at", ["contact", "table", "cut"])
def test_p3m_short_range_pairs_at_their_edges(pdq, setup, at, seam):
    # pairs alone in a sample: at and around the clamp d_c (a coincident pair too), on the edges of the
    # long-range table's intervals, and just inside and outside r_cut; along x and across the period.
    # Bar as above: the float-float pair (2^-46) and the table (2e-15) sit far below it, the mesh part
    # differs by the ordering of the transforms
    f, of, grid, plan, d, Gh = setup
    dc = oracle.class_table(ST3)[:, 1].max()
    r = {"contact": dc * np.array([0.0, 1e-3, 0.5, 1 - 1e-12, 1.0, 1 + 1e-12, 1.5]),
         "table": plan.r_cut * np.sqrt(np.array([1, 2, 511, 1023]) / 1024.0 * (1 + 1e-15)),
         "cut": plan.r_cut * np.array([1 - 1e-3, 1 - 1e-10, 1 + 1e-10, 1 + 1e-3])}[at]
    n = len(r)
    x, y, z = np.zeros(2 * n), np.full(2 * n, 17.25), np.full(2 * n, 0.03125)
    if seam:      # the second particle a distance r below z = 0, wrapped
        z[1::2] = np.mod(z[1::2] - r, 720.0)
    else:
        x[0::2], x[1::2] = 100.0, 100.0 - r
    q = np.tile([0.7, -0.4], n)
    ids = np.tile([0, 1], n).astype(np.int32)
    st = _state(pdq, 0, [2] * n, (x, y, z, q, np.zeros((2 * n, 3)), np.full(2 * n, 2, np.int32), ids))
    got = plan.coulomb(pdq.phys_default(), st).cpu().numpy()
    want = _ref_sums(d, Gh, [2] * n, x, y, z, q)
    assert np.all(np.isfinite(got))
    scale = np.maximum(np.abs(want).reshape(n, 6).max(1), _rms(want) * 1e-3).repeat(2)[:, None]
    assert np.max(np.abs(got - want) / scale) <= 1e-9


@pytest.mark.parametrize("block", [64, 256])
def test_p3m_step_matches_oracle(pdq, setup, block):
    # the P3M step = the oracle's step with the reference P3M sums of each step's start state
    f, of, grid, plan, d, Gh = setup
    counts = [600, 257]
    arr = _cloud(counts, 5)
    x, y, z, q, v, cls, ids = arr
    st = _state(pdq, 0, counts, arr)
    prm = np.array([[0.05, 0.5, 0.5], [0.1, 0.2, 0.3]])
    cfg = pdq.step_cfg(0.1, block=block, window_start=0)
    tally = pdq.Tally(2, 3)
    steps = 4
    pdq.step_particles_p3m(f, pdq.phys_default(), st, pdq.params_tensor(prm), cfg, steps, tally, plan,
                           pdq.workspace(st, cfg))
    assert pdq.check_state(st) == 0
    ost = oracle.State(len(x))
    ost.x, ost.y, ost.z, ost.q, ost.cls, ost.id = x.copy(), y.copy(), z.copy(), q.copy(), cls.copy(), ids.copy()
    ost.vx, ost.vy, ost.vz = v[:, 0].copy(), v[:, 1].copy(), v[:, 2].copy()
    off = np.r_[0, np.cumsum(counts)]
    tallies = (np.zeros((2, 3), np.int64), np.zeros((2, 3), np.int64))
    for k in range(steps):
        ext = _ref_sums(d, Gh, counts, ost.x, ost.y, ost.z, ost.q, ost.alive == 1)
        oracle.run_ext(of, grid, oracle.cfg(0.1, window_start=0), ST3, off, prm, ost, ext, step0=k, tallies=tallies)
    gx = st.positions64().cpu().numpy()
    gv = st.current()[1].double().cpu().numpy()
    tag = st.tag.cpu().numpy()
    gidx = off[np.repeat(np.arange(2), counts)] + tag[:, 0]
    live = gv[:, 3] > 0.5
    assert np.array_equal(live, ost.alive[gidx] == 1)
    rx = np.stack([ost.x, ost.y, ost.z], 1)[gidx]
    rv = np.stack([ost.vx, ost.vy, ost.vz], 1)[gidx]
    assert np.max(np.abs(gx[live] - rx[live]) / (1 + np.abs(rx[live]))) < 1e-11
    assert np.max(np.abs(gv[live, :3] - rv[live]) / (1 + np.abs(rv[live]))) < 1e-10
    assert np.array_equal(tally.n_alive.cpu().numpy(), tallies[1])


def test_p3m_step_takes_a_workspace_without_partial_sums(pdq, setup):
    # 2,000 FP64 particles at 32 threads: given sums need no partial sums of the tile pairs, so a workspace with the
    # 17 chunks that a one-sided pair sum of this size is cut into (items, order, tags, counters, sums) is enough
    f, of, grid, plan, d, Gh = setup
    counts = [1200, 800]
    arr = _cloud(counts, 8)
    prm = pdq.params_tensor(np.array([[0.05, 0.5, 0.5], [0.1, 0.2, 0.3]]))
    cfg = pdq.step_cfg(0.1, block=32, window_start=0)

    def a256(v):
        return (v + 255) // 256 * 256
    tiles, chunks = 2000 // 32 + 2 + 1, 17
    small = a256(8 * tiles * chunks) + a256(4 * 2) + a256(8 * 2000) + a256(4 * tiles) + a256(24 * chunks * 2000)
    out = []
    for ws in (None, torch.empty(small, dtype=torch.uint8, device="cuda")):
        st = _state(pdq, 0, counts, arr)
        ws = pdq.workspace(st, cfg) if ws is None else ws
        pdq.step_particles_p3m(f, pdq.phys_default(), st, prm, cfg, 1, pdq.Tally(2, 3), plan, ws)
        out.append(st.current()[0].clone())
    assert torch.allclose(out[0], out[1], rtol=1e-12, atol=1e-12)
