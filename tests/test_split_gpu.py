"""GPU parity of node splitting (tn_split_node, Sec. III.B "Node Splitting",
Appendix A) against the FP64 oracle on the same float32 inputs.

What is unique is compared: the singular values (kept and dropped), the kept
count (the truncation rule applied to the GPU's own values must give the
GPU's count exactly, and the oracle's count where no limit sits near a partial
sum), and the truncated product U S V^T when the kept and dropped values are
separated. Singular vectors are unique only up to sign, so they are checked
for what must hold instead: orthonormal columns of U and rows of V^T (for
non-zero values) and sqrt(S) carried on both sides by split_node.

Tolerances (float32 one-sided Jacobi, column norms in float64): singular
values within 5e-5 of the largest one; products within 5e-5 of |A|_F;
orthonormality within 1e-4.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tn():
    from paper_1905_01330_gb300 import build, tn as tnmod
    build.build()
    tnmod.load()
    return tnmod


def planted(m, n, s, seed):
    rng = np.random.default_rng(seed)
    r = len(s)
    q1, _ = np.linalg.qr(rng.standard_normal((m, r)))
    q2, _ = np.linalg.qr(rng.standard_normal((n, r)))
    return ((q1 * np.asarray(s)[None, :]) @ q2.T).astype(np.float32)


def check(tn, A, left, right, max_sv=None, max_err=None, At=None, expect_k=None):
    """A: float32 numpy array (the node's values); At: the device tensor (a view) if not A itself."""
    At = torch.from_numpy(A).cuda() if At is None else At
    info = {}
    us, svh, drop = tn.split_node(At, left, right, max_sv, max_err, info=info)
    u, s, vh, drop2 = tn.split_node(At, left, right, max_sv, max_err, full_svd=True)
    torch.cuda.synchronize()
    assert info["sweeps"] > 0
    mat, ldims, rdims = oracle.matrix_view(A.astype(np.float64), left, right)
    U, S, Vt, _, _ = oracle.svd(A.astype(np.float64), left, right)
    r = len(S)
    k = us.shape[-1]
    assert list(us.shape) == ldims + [k] and list(svh.shape) == [k] + rdims
    assert list(u.shape) == ldims + [k] and list(vh.shape) == [k] + rdims
    assert s.shape == (k,) and drop.shape == (r - k,) and drop2.shape == (r - k,)
    sg = np.concatenate([s.cpu().numpy(), drop2.cpu().numpy()]).astype(np.float64)
    assert np.array_equal(drop.cpu().numpy(), drop2.cpu().numpy())
    smax = max(S[0], 1e-30)
    assert np.all(np.diff(sg) <= 0)
    assert np.abs(sg - S).max() <= 5e-5 * smax, np.abs(sg - S).max() / smax
    # the kept count: the rule on the GPU's own values, and the oracle's count
    assert k == oracle.truncation_count([float(v) for v in s.cpu().numpy()] + [float(v) for v in drop2.cpu().numpy()],
                                        max_sv, max_err)
    k_or = oracle.truncation_count(S, max_sv, max_err)
    assert k == (k_or if expect_k is None else expect_k)
    if k == 0:
        return
    # truncated product against the oracle's, when the cut separates the values
    nrm = max(np.linalg.norm(mat), 1e-30)
    rec = us.reshape(-1, k).double().cpu().numpy() @ svh.reshape(k, -1).double().cpu().numpy()
    rec_or = (U[:, :k] * S[:k]) @ Vt[:k]
    if k == r or S[k - 1] - S[k] > 1e-3 * smax:
        assert np.linalg.norm(rec - rec_or) <= 5e-5 * nrm
    rec_full = u.reshape(-1, k).double().cpu().numpy() @ np.diag(s.double().cpu().numpy()) @ \
        vh.reshape(k, -1).double().cpu().numpy()
    assert np.linalg.norm(rec_full - rec) <= 5e-5 * nrm
    # orthonormal factors for the non-zero values; sqrt(S) on both sides
    nz = s.cpu().numpy() > 1e-3 * smax
    Ug = u.reshape(-1, k).double().cpu().numpy()[:, nz]
    Vg = vh.reshape(k, -1).double().cpu().numpy()[nz]
    assert np.abs(Ug.T @ Ug - np.eye(Ug.shape[1])).max() <= 1e-4
    assert np.abs(Vg @ Vg.T - np.eye(Vg.shape[0])).max() <= 1e-4
    root = np.sqrt(s.double().cpu().numpy())
    assert np.allclose(np.linalg.norm(us.reshape(-1, k).double().cpu().numpy(), axis=0)[nz], root[nz], rtol=1e-4)
    assert np.allclose(np.linalg.norm(svh.reshape(k, -1).double().cpu().numpy(), axis=1)[nz], root[nz], rtol=1e-4)


def rand(seed, shape):
    return np.random.default_rng(seed).standard_normal(shape).astype(np.float32)


def test_paper_shapes(tn):
    A = rand(1, (2, 3, 4, 5, 6))
    check(tn, A, [0, 1, 2], [3, 4])                     # (2,3,4,24) and (24,5,6)


@pytest.mark.parametrize("shape,left,right", [
    ((50, 20), [0], [1]),              # M > N: W is the matrix view
    ((20, 50), [0], [1]),              # M < N: W is its transpose
    ((64, 64), [1], [0]),              # square, legs swapped
    ((6, 5, 8), [2, 0], [1]),          # left legs out of order
    ((3, 4, 5, 2), [3, 1], [0, 2]),
    ((1, 50), [0], [1]), ((50, 1), [0], [1]),           # one singular value
    ((33, 7, 3), [0], [1, 2]),         # odd r: a dummy slot in every round
])
def test_random_nodes(tn, shape, left, right):
    check(tn, rand(2, shape), left, right)


@pytest.mark.parametrize("shape", [(256, 256), (512, 512), (700, 650)])
def test_two_site_sizes(tn, shape):
    """Square and near-square nodes of the sizes a two-site split of an MPS
    sweep meets (chi = 128, 256): hundreds of rounds per sweep."""
    check(tn, rand(9, shape), [0], [1])


def test_strided_view(tn):
    base = rand(3, (8, 6, 10))
    At = torch.from_numpy(base).cuda().permute(2, 0, 1)[:, ::2]   # (10, 4, 6), non-contiguous
    A = np.ascontiguousarray(base.transpose(2, 0, 1)[:, ::2])
    check(tn, A, [1, 0], [2], At=At)


def test_rank_deficient(tn):
    rng = np.random.default_rng(4)
    A = np.multiply.outer(rng.standard_normal(30), rng.standard_normal(40)).astype(np.float32)
    check(tn, A, [0], [1])
    check(tn, A, [0], [1], max_err=1e-3, expect_k=1)    # the zeros (and rounding noise) dropped


def test_truncation(tn):
    s = np.linspace(4.0, 0.02, 200)
    A = planted(300, 200, s, 5)
    check(tn, A, [0], [1], max_sv=5)
    # limit halfway between two partial sums of the tail: no rounding decides k
    tail = np.cumsum(s[::-1])
    check(tn, A, [0], [1], max_err=0.5 * (tail[59] + tail[60]))
    check(tn, A, [0], [1], max_sv=100, max_err=0.5 * (tail[59] + tail[60]))


def test_paper_truncation_example(tn):
    """Appendix A: a (1000, 1000) node with max_singular_values=5 keeps 5 and
    drops 995 (largest size in this suite)."""
    A = planted(1000, 1000, 0.99 ** np.arange(1000), 6)
    us, svh, drop = tn.split_node(torch.from_numpy(A).cuda(), [0], [1], max_singular_values=5)
    assert tuple(us.shape) == (1000, 5) and tuple(svh.shape) == (5, 1000) and tuple(drop.shape) == (995,)
    check(tn, A, [0], [1], max_sv=5)


def test_empty_node(tn):
    At = torch.empty((0, 5), device="cuda")
    us, svh, drop = tn.split_node(At, [0], [1])
    assert tuple(us.shape) == (0, 0) and tuple(svh.shape) == (0, 5) and drop.numel() == 0


def test_legs_must_partition(tn):
    At = torch.zeros((2, 3, 4), device="cuda")
    with pytest.raises(tn.TnError):
        tn.split_node(At, [0], [1])


@pytest.mark.parametrize("shape,scale", [((16, 16), 1.0), ((17, 40), 1.0), ((33, 33), 1e15), ((47, 300), 1.0),
                                         ((48, 257), 1e-15), ((700, 20), 1.0), ((2100, 35), 1.0), ((5, 600), 1.0),
                                         ((1, 9), 1.0)])
def test_block_edges(tn, shape, scale):
    # blocks of 16 columns (one, an odd count, a ragged last one), rows past a
    # staged chunk (256) and shared out over a cluster, norms whose squares
    # come near the ends of the exponent range; tolerances as above
    A = (rand(31, shape) * np.float32(scale)).astype(np.float32)
    check(tn, A, [0], [1])


def node_kinds():
    """Nodes whose columns (of the matrix, or what rotations leave of them) have
    norms far apart, or whose squares leave the exponent range: low rank, few
    non-zero rows, zero-padded bonds, blocks beside tiny entries, graded columns."""
    out = []
    for scale in (1.0, 1e-8, 1e-12, 1e-13, 1e-15, 1e-18, 1e18):
        for rank in (1, 4):
            out.append(("rank", (32, 32), rank, scale))
    out += [("rank", (256, 256), 3, 1e-13), ("rank", (40, 600), 2, 1e-14)]
    for size in (4, 16):
        for tiny in (1e-12, 1e-19, 1e-20, 1e-22):
            out.append(("block", (32, 32), size, tiny))
    for rows in (1, 2, 3, 4, 6, 8):
        out += [("rows", (32, 16), rows, 1.0), ("rows", (48, 40), rows, 1e-10)]
    for z in (1, 2, 3, 4):
        out.append(("bond", (8, 2, 2, 8), z, 1.0))
    for last in (1e-12, 1e-22, 1e-30):
        out.append(("graded", (40, 40), 0, last))
    out += [("ones", shape, 0, scale) for shape in ((100, 20), (48, 50), (100, 50)) for scale in (1e8, 1e25, 1e32)]
    out += [("full", (32, 32), 0, scale) for scale in (1e-18, 1e-20, 1e-25, 1e18, 1e25)]
    return out


@pytest.mark.parametrize("kind,shape,count,size", node_kinds())
@pytest.mark.parametrize("seed", [0, 1, 2])
def test_norms_far_apart(tn, kind, shape, count, size, seed):
    # singular values and products as above, and the sweeps end by themselves
    rng = np.random.default_rng(1000 * seed + count)
    A = rng.standard_normal(shape)
    if kind == "rank":
        A = rng.standard_normal((shape[0], count)) @ rng.standard_normal((count, shape[1])) * size
    elif kind == "block":
        A[count:] *= size
        A[:count, count:] *= size
    elif kind == "rows":
        A[count:] = 0.0
        A *= size
    elif kind == "bond":
        A[count:] = 0.0
    elif kind == "ones":  # null columns of rounding noise far below a large value
        A = np.full(shape, size)
    elif kind == "graded":
        A *= np.logspace(0, np.log10(size), shape[1])
    else:
        A *= size
    legs = ([0, 1], [2, 3]) if len(shape) == 4 else ([0], [1])
    check(tn, A.astype(np.float32), *legs)


@pytest.mark.parametrize("shape", [(9215, 3), (9216, 1), (9217, 3), (10000, 4), (20001, 5), (9300, 8), (12001, 9),
                                   (30000, 16), (9216, 17), (100003, 32), (9999, 33), (2, 20000), (17, 9999), (1, 300000)])
def test_tall_nodes(tn, shape):
    # rows shared out over the grid from 9216 on, stored 4, 8, 16 or 32 columns
    # wide, ragged last parts and chunks, either side the long one; and the
    # norms' row parts (4096); tolerances as above
    check(tn, rand(51, shape), [0], [1])


@pytest.mark.parametrize("count,rank,scale", [(4, 1, 1.0), (7, 2, 1e-13), (16, 3, 1e15), (31, 4, 1.0), (12, 12, 1e-20)])
def test_tall_nodes_of_low_rank(tn, count, rank, scale):
    rng = np.random.default_rng(60 + count)
    A = rng.standard_normal((11000, rank)) @ rng.standard_normal((rank, count)) * scale
    check(tn, A.astype(np.float32), [0], [1])


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("shape", [(40, 24), (24, 40), (300, 65), (11000, 5), (3, 20000)])
def test_an_infinite_or_nan_entry_stays_in_its_column(tn, shape, value):
    # the column (of the shorter side) that holds it has no finite value: first
    # among the values if infinite, last if NaN; the others' are theirs
    A = rand(71, shape)
    short = int(shape[0] >= shape[1])
    at = (shape[0] // 2, shape[1] // 3)
    A[at] = value
    info = {}
    _, s, _, d = tn.split_node(torch.from_numpy(A).cuda(), [0], [1], full_svd=True, info=info)
    got = s.cpu().numpy().astype(np.float64)
    assert info["sweeps"] > 0 and len(got) == min(shape) and d.numel() == 0
    rest = np.linalg.svd(np.delete(A.astype(np.float64), at[short], axis=short), compute_uv=False)
    odd, others = (got[-1], got[:-1]) if np.isnan(value) else (got[0], got[1:])
    assert np.isnan(odd) if np.isnan(value) else odd == np.inf
    assert np.abs(others - rest).max() <= 5e-5 * rest[0]
