"""V-cycle kernels on both sides of the rule that lets them load ahead of their wait: one
batch of every direction (large launches, plain kernels) and one direction to a batch
(small launches, loads ahead) solve the same problem."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1910_11463_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pair():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__ as g
    g.build()
    from paper_1910_11463_gb300 import pair as P
    return P


# every solve ends at ||b - A psi|| <= inner_tol ||b||, so two of them differ by a small
# multiple of inner_tol however their sums are ordered
@pytest.mark.parametrize("mesh,n", [("hex", 20), ("tet", 12)])
@pytest.mark.parametrize("precision,inner_tol,tol", [(0, 1e-12, 1e-10), (1, 1e-10, 1e-8), (2, 1e-10, 1e-8)])
def test_batch_size_does_not_change_the_flux(pair, mesh, n, precision, inner_tol, tol):
    prob = I.small_hex(n, order=4, seed=3) if mesh == "hex" else I.small_tet(n, order=4, seed=3)
    air = pair.default_air_params(precision=precision, distance=1 if mesh == "hex" else 2, theta=0.5, phi_A=0.05)
    out = []
    for concurrent, batch in ((1, 0), (1, 1)):
        si = pair.default_si_params(max_iters=3, fixed_iters=1, inner_tol=inner_tol, concurrent=concurrent, batch=batch)
        phi, _, info = pair.si_solve_problem(prob, air=air, si=si)
        assert info["batches"] == (1 if batch == 0 else prob.M)
        out.append(phi.cpu().numpy())
    assert np.linalg.norm(out[0] - out[1]) <= tol * np.linalg.norm(out[0])


# the coarsest sweeps as a dense product against plain sweeps: segments of one row, of
# a row block and its neighbours, the largest, and one past it (which keeps the sweeps); the
# two differ by at most about n eps ||B|| / ||x|| sqrt(n) (n = 128: 3e-13, in FP32 1e-4)
@pytest.mark.parametrize("n", [1, 3, 31, 32, 33, 97, 128, 129])
@pytest.mark.parametrize("sweeps", [0, 1, 7])
def test_coarsest_product_equals_sweeps(pair, n, sweeps):
    g = np.random.default_rng(n)
    A = np.eye(n) + np.tril(g.uniform(-1, 1, (n, n)) * (g.random((n, n)) < 0.2), -1) / np.sqrt(n)
    A[np.arange(n), np.arange(n)] += 0.5 * g.random(n)
    ci = [np.nonzero(r)[0] for r in A]
    rp = np.concatenate([[0], np.cumsum([len(c) for c in ci])]).astype(np.int32)
    col = np.concatenate(ci).astype(np.int32)
    val = np.concatenate([A[i, c] for i, c in enumerate(ci)])
    b = g.standard_normal(n)
    want = np.zeros(n)
    for _ in range(sweeps):
        want = want + (b - A @ want) / np.diag(A)
    for precision, tol in ((0, 1e-12), (1, 1e-4)):
        dev = [torch.as_tensor(a, device="cuda") for a in (rp, col, val)]
        h = pair.Hierarchy([tuple(dev)] * 2, pair.default_air_params(precision=precision, max_coarse=1000,
                                                                      coarse_sweeps=sweeps))
        x = h.vcycle(torch.as_tensor(np.tile(b, 2), device="cuda"), torch.zeros(2 * n, dtype=torch.float64, device="cuda"))
        x = x.cpu().numpy()
        assert np.array_equal(x[:n], x[n:])
        assert np.linalg.norm(x[:n] - want) <= tol * max(np.linalg.norm(want), 1e-300)


# the first F sweep through P columns: offsets that fit 16 bits and ones that do not, rows
# without a coarse neighbour, one to three F sweeps; FP64 cycles of a few dozen additions a
# row agree to 1e-12
@pytest.mark.parametrize("n,far,f_sweeps", [(300, False, 1), (3000, False, 2), (3000, False, 3), (150_000, True, 2),
                                            (150_000, True, 1)])
def test_first_sweep_through_p_columns(pair, n, far, f_sweeps):
    from oracle import oracle as O
    g = np.random.default_rng(n + f_sweeps)
    k = 3
    off = g.integers(0, n, (n, k)) if far else np.clip(np.arange(n)[:, None] + g.integers(-20, 21, (n, k)), 0, n - 1)
    off[::9] = np.arange(n)[::9, None]   # rows that depend on nothing
    rows = np.repeat(np.arange(n), k)
    cols = off.ravel()
    keep = cols != rows
    key = np.unique(rows[keep].astype(np.int64) * n + cols[keep])
    key = np.unique(np.concatenate([key, np.arange(n, dtype=np.int64) * (n + 1)]))
    r, c = key // n, (key % n).astype(np.int32)
    v = np.where(r == c, 1.0, g.uniform(-0.3, 0.3, key.size))
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]).astype(np.int32)
    kw = dict(theta=0.5, max_coarse=50, max_levels=4, f_sweeps=f_sweeps)
    b, x0 = g.random(n), g.random(n)
    h = pair.Hierarchy([tuple(torch.as_tensor(a, device="cuda") for a in (rp, c, v))],
                       pair.default_air_params(precision=0, **kw))
    x = h.vcycle(torch.as_tensor(b, device="cuda"), torch.as_tensor(x0, device="cuda").clone()).cpu().numpy()
    H = O.Hierarchy(rp, c, v, O.default_params(**kw))
    assert H.nlev >= 2
    xo = H.vcycle(b, x0.copy())
    assert np.linalg.norm(x - xo) <= 1e-12 * np.linalg.norm(xo)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("precision,n", [(0, 33), (0, 100), (1, 100)])
def test_nonfinite_right_hand_side_reaches_the_rows_the_sweeps_reach(pair, precision, n, bad):
    """One infinity or NaN in the right-hand side of a coarsest level: the rows that the
    sweeps couple to it, and no others, are not finite afterwards."""
    from oracle import oracle as O
    g = np.random.default_rng(n)
    A = np.eye(n) + np.tril(g.uniform(-0.5, 0.5, (n, n)) * (g.random((n, n)) < 0.05), -1)
    ci = [np.nonzero(r)[0] for r in A]
    rp = np.concatenate([[0], np.cumsum([len(c) for c in ci])]).astype(np.int32)
    col = np.concatenate(ci).astype(np.int32)
    val = np.concatenate([A[i, c] for i, c in enumerate(ci)])
    b = g.uniform(1.0, 2.0, n)
    b[n // 4] = bad
    kw = dict(max_coarse=1000, coarse_sweeps=4)
    h = pair.Hierarchy([tuple(torch.as_tensor(a, device="cuda") for a in (rp, col, val))],
                       pair.default_air_params(precision=precision, **kw))
    x = h.vcycle(torch.as_tensor(b, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda")).cpu().numpy()
    xo = O.Hierarchy(rp, col, val, O.default_params(**kw)).vcycle(b, np.zeros(n))
    ok = np.isfinite(xo)
    assert 0 < ok.sum() < n and np.array_equal(np.isfinite(x), ok)
    assert np.allclose(x[ok], xo[ok], rtol=1e-12 if precision == 0 else 2e-5, atol=0)   # (condition below 13)


_MANY = """
import numpy as np, torch
from paper_1910_11463_gb300 import pair
count, n, sweeps = 6000, 100, 3
g = np.random.default_rng(0)
rp = np.concatenate([[0], 1 + 2 * np.arange(n)]).astype(np.int32)
col = np.concatenate([[0]] + [[i - 1, i] for i in range(1, n)]).astype(np.int32)
val = np.concatenate([[1.0]] + [[g.uniform(-0.5, 0.5), 1.0] for i in range(1, n)])
dev = tuple(torch.as_tensor(a, device="cuda") for a in (rp, col, val))
prm = pair.default_air_params(precision=0, coarse_sweeps=sweeps)
b = torch.as_tensor(np.tile(g.standard_normal(n), count), device="cuda")
x = torch.zeros_like(b)
small = pair.Hierarchy([dev] * 2, prm).vcycle(b[:2 * n].clone(), torch.zeros(2 * n, dtype=torch.float64, device="cuda"))
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
h = pair.Hierarchy([dev] * count, prm)
h.vcycle(b, x)
torch.cuda.synchronize()
print((free - torch.cuda.mem_get_info()[0]) / 2 ** 20)
x = x.view(count, n)
assert torch.equal(x, x[:1].expand(count, n))
assert torch.allclose(x[0], small[:n], rtol=1e-13, atol=1e-13)
"""


def test_coarsest_products_are_bounded_in_memory(pair):
    """6000 matrices of 100 rows: their products would take 590 MB, the operators, vectors
    and the setup's scratch take less than 200."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _MANY], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert float(r.stdout.split()[-1]) < 400.0


# the traffic counters of the SELL levels, from the exported hierarchies: 16-bit columns
# everywhere (n = 5), and a level 0 whose columns take 32 bits and P columns 16 (n = 38)
@pytest.mark.parametrize("n,f_sweeps", [(5, 1), (5, 3), (38, 2)])
def test_relaxation_traffic_counters(pair, n, f_sweeps):
    prob = I.small_tet(n, order=2, seed=4)
    air = pair.default_air_params(precision=0, theta=0.5, f_sweeps=f_sweeps, max_levels=3, max_coarse=20, coarse_sweeps=1)
    si = pair.default_si_params(max_iters=1, fixed_iters=1, inner_cycles=1, concurrent=1, timing=1)
    _, _, info = pair.si_solve_problem(prob, air=air, si=si)
    assert info["batches"] == 1 and info["n_relax0"] == 1
    mesh = pair.TetMesh(prob.verts, prob.tets, prob.nbr)
    st = torch.as_tensor(prob.sigma_t, device="cuda")
    levels = [[], []]   # per level and direction: rows, entries and widths
    nx, big = 0, False   # rows of the coarsest level; a segment of it past 40 KB: grid-wide sweeps
    for m in range(prob.M):
        h = pair.Hierarchy([pair.dg_assemble_tet(mesh, prob.omega[m], st)], air)
        assert h.nlevels() == 3
        X = h.level(0, 2)
        nx += X.n
        big |= X.nnz * 12 + X.n * 32 + (X.n + 1) * 4 > 40 * 1024
        for l in (0, 1):
            L = h.level(0, l)
            F = L.cf == 0
            lens = np.diff(L.rowptr)
            rows = np.repeat(np.arange(L.n), lens)
            near = np.abs(L.col - rows) <= 32767
            pc, fe = L.pmap[L.col], F[rows]
            org = L.pmap.copy()   # a row's origin: its own P column, else its first entry's
            p = np.nonzero(fe & (pc >= 0) & (org[rows] < 0))[0][::-1]
            org[rows[p]] = pc[p]   # (of repeated rows the last assignment, the first entry, stays)
            pnear = (pc < 0) | (np.abs(pc - org[rows]) <= 32767)
            levels[l].append((F.sum(), (~F).sum(), lens[F].sum(), lens[~F].sum(), near[fe].all(), near[~fe].all(),
                              pnear[fe].all()))
    want = []
    for l in (0, 1):
        a = np.array(levels[l], dtype=np.int64)
        nF, nC, eF, eC = a[:, :4].sum(0)
        cF, cC, cP = (2 if ok else 4 for ok in a[:, 4:].all(0))
        if n == 38 and l == 0:
            assert (cF, cP) == (4, 2)
        b = nF * (12 + 32) + eF * (cP + 8) + nC * (4 + 24) + (f_sweeps - 1) * (nF * (8 + 32) + eF * (cF + 8))
        b += (nF * 16 + nC * (8 + 24 + 16) if l == 0 else nF * 8 + nC * (8 + 32)) + eC * (cC + 8)
        want.append(b)
    if big:
        want[1] += nx * (4 + 24)   # the one coarsest sweep: position, b and dinv read, value written
    for got, w in zip((info["gb_relax0"], info["gb_relaxc"]), want):
        assert abs(got * 1e9 - w) <= 1e-9 * w


# the same in FP32 cycles: the first sweep's gathers, C rows and second target with 16-bit
# and 32-bit P columns; a cycle's values pass through about 40 roundings of sums of at most
# a few dozen terms, 6e-8 each against values of the size of x
@pytest.mark.parametrize("n,far,f_sweeps", [(300, False, 1), (3000, False, 2), (3000, False, 3), (150_000, True, 2)])
def test_first_sweep_through_p_columns_fp32(pair, n, far, f_sweeps):
    from oracle import oracle as O
    g = np.random.default_rng(n + f_sweeps)
    k = 3
    off = g.integers(0, n, (n, k)) if far else np.clip(np.arange(n)[:, None] + g.integers(-20, 21, (n, k)), 0, n - 1)
    off[::9] = np.arange(n)[::9, None]   # rows that depend on nothing
    r, c = np.repeat(np.arange(n), k), off.ravel()
    key = np.unique(np.concatenate([r.astype(np.int64) * n + c, np.arange(n, dtype=np.int64) * (n + 1)]))
    r, c = key // n, (key % n).astype(np.int32)
    v = np.where(r == c, 1.0, g.uniform(-0.3, 0.3, key.size))
    rp = np.concatenate([[0], np.cumsum(np.bincount(r, minlength=n))]).astype(np.int32)
    kw = dict(theta=0.5, max_coarse=50, max_levels=4, f_sweeps=f_sweeps)
    b, x0 = g.random(n), g.random(n)
    h = pair.Hierarchy([tuple(torch.as_tensor(a, device="cuda") for a in (rp, c, v))],
                       pair.default_air_params(precision=1, **kw))
    x = h.vcycle(torch.as_tensor(b, device="cuda"), torch.as_tensor(x0, device="cuda").clone()).cpu().numpy()
    H = O.Hierarchy(rp, c, v, O.default_params(**kw))
    assert H.nlev >= 2
    xo = H.vcycle(b, x0.copy())
    assert np.linalg.norm(x - xo) <= 40 * 6e-8 * np.linalg.norm(xo)
