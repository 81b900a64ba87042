"""GPU parity: fe_spmm against the oracle's plain-definition SpMM (Section 3.3).

Tolerances (the SpMM accuracy requirement of 1e-6 relative, read per entry against A|X|, the condition
number of a sum): FP64 |Y - Y*| <= 1e-13 (A|X|), FP32 <= 1e-6 (A|X|) with Y* the FP64 sum of
the same FP32 inputs.  A 1 = degree must be exact in either precision.  Inputs of one sign
(where rounding errors of a plain in-order sum do not cancel) are checked against the FP32
kernel's stated worst case, 9 * 2^-24 (A|X|).
"""
import numpy as np
import pytest

import graphgen
import paper_1602_01421_gb300 as fe
from tests.gpu_util import assert_spmm_close, to_dev, torch

pytestmark = pytest.mark.gpu

TOL = {"f32": 1e-6, "f64": 1e-13}
# the FP32 kernel's worst case per entry (compensated lane sums, <= 5 tree levels, one rounding
# of a split hub row's FP64 sum), in units of A|X|
F32_BOUND = 9 * 2.0 ** -24
# all-equal entries: a plain in-order FP32 sum of 127 (69) copies of this value is off by 1.47e-6
# (1.05e-6) of the exact sum (found by scanning 20000 values in [1, 2) with numpy float32 sums)
ADVERSARIAL_C = np.float32(1.9397392272949219)


def one_signed_block(kind, n, b, seed):
    """U[0,1), U[1,2) or the constant ADVERSARIAL_C, FP32, n x b."""
    if kind == "const":
        return np.full((n, b), ADVERSARIAL_C, dtype=np.float32)
    lo = 0.0 if kind == "u01" else 1.0
    return (lo + graphgen.uniform_block(n, b, seed=seed)).astype(np.float32)


def plain_sum_error(g, X, rows):
    """Largest |in-order FP32 sum - exact| / A|X| over `rows` (what a kernel summing each row
    in order, uncompensated, would get) -- shows that an input can catch such a kernel."""
    worst = 0.0
    for i in rows:
        cols = g.colidx[g.rowptr[i]:g.rowptr[i + 1]]
        if len(cols) == 0:
            continue
        s = np.zeros(X.shape[1], dtype=np.float32)
        for c in cols:
            s = (s + X[c]).astype(np.float32)
        exact = X[cols].astype(np.float64).sum(0)
        worst = max(worst, float((np.abs(s - exact) / np.abs(X[cols]).astype(np.float64).sum(0)).max()))
    return worst
NP = {"f32": np.float32, "f64": np.float64}

GRAPHS = {
    "rmat12": lambda: graphgen.rmat(12, seed=3),
    "rmat14": lambda: graphgen.rmat(14, seed=1),
    "rmat13-noperm": lambda: graphgen.rmat(13, seed=2, permute=False),
    "star9000": lambda: graphgen.star(9000),              # one hub split into 3 chunks
    "complete70": lambda: graphgen.complete(70),          # all rows in one slice bucket (deg 69)
    "complete128": lambda: graphgen.complete(128),        # slice rows of degree 127
    "complete300": lambda: graphgen.complete(300),        # all rows warp tasks (deg 299)
    "cycle1001": lambda: graphgen.cycle(1001),            # all rows tail (deg 2), ragged slice
    "er3000": lambda: graphgen.erdos_renyi(3000, 12.0, seed=5),
    "union-isolated": lambda: graphgen.disjoint_union(graphgen.star(5000), graphgen.path(33),
                                                      graphgen.from_edges(77, [], [], "iso77")),
}


@pytest.fixture(scope="module")
def graphs():
    return {k: v() for k, v in GRAPHS.items()}


@pytest.mark.parametrize("name", list(GRAPHS))
@pytest.mark.parametrize("b", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_spmm_parity(graphs, name, b, prec):
    g = graphs[name]
    X = graphgen.normal_block(g.n, b, seed=100 + b, dtype=NP[prec])
    with fe.Csr.from_graph(g) as h:
        Y = fe.spmm(h, to_dev(X)).cpu().numpy()
    assert_spmm_close(g, X, Y, TOL[prec])


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("knobs", [dict(tail_max=1, hub_min=8, hub_chunk=8),
                                   dict(tail_max=32, hub_min=40, hub_chunk=64),
                                   dict(tail_max=4, hub_min=64, hub_chunk=4096),
                                   dict(tail_max=128, hub_min=200, hub_chunk=100)])
def test_spmm_parity_all_paths_small(prec, knobs):
    """Tiny thresholds push most rows through the hub split and the partial reduce, with plain
    and with packed column indices."""
    g = graphgen.rmat(13, seed=9)
    for fmt in ("plain", "packed"):
        for b in (1, 4, 16):
            X = graphgen.normal_block(g.n, b, seed=b, dtype=NP[prec])
            with fe.Csr.from_graph(g, index_format=fmt, **knobs) as h:
                info = h.info()
                Y = fe.spmm(h, to_dev(X)).cpu().numpy()
            assert info["rows_hub"] > 0
            assert_spmm_close(g, X, Y, TOL[prec])


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("tail_max", [64, 128])
def test_spmm_parity_wide_tail(graphs, prec, tail_max):
    """Rows up to degree 64 / 128 in the thread-per-row slices (exact-degree buckets)."""
    for name in ("rmat14", "complete70", "er3000"):
        g = graphs[name]
        for b in (1, 4, 8, 16):
            X = graphgen.normal_block(g.n, b, seed=b + 7, dtype=NP[prec])
            with fe.Csr.from_graph(g, tail_max=tail_max) as h:
                info = h.info()
                Y = fe.spmm(h, to_dev(X)).cpu().numpy()
            deg = g.degrees()
            assert info["rows_tail"] == ((deg >= 1) & (deg <= tail_max)).sum()
            assert_spmm_close(g, X, Y, TOL[prec])


@pytest.mark.parametrize("prec,b", [("f32", 8), ("f32", 16), ("f64", 4), ("f64", 8), ("f64", 16)])
def test_spmm_parity_16_byte_aligned_blocks(graphs, prec, b):
    """X and Y 16-byte but not 32-byte aligned: the 16-byte gather path (32-byte rows are
    otherwise gathered with one 256-bit load per lane)."""
    t = torch()
    g = graphs["rmat14"]
    dt = t.float32 if prec == "f32" else t.float64
    shift = 16 // (4 if prec == "f32" else 8)
    X = graphgen.normal_block(g.n, b, seed=3, dtype=NP[prec])
    xbuf = t.zeros(g.n * b + 64, dtype=dt, device="cuda")
    ybuf = t.zeros(g.n * b + 64, dtype=dt, device="cuda")
    assert xbuf.data_ptr() % 32 == 0
    xv = xbuf[shift:shift + g.n * b].view(g.n, b)
    yv = ybuf[shift:shift + g.n * b].view(g.n, b)
    assert xv.data_ptr() % 32 == 16
    xv.copy_(to_dev(X))
    with fe.Csr.from_graph(g, tail_max=64) as h:
        fe.spmm(h, xv, yv)
        Y16 = yv.cpu().numpy()
        Y32 = fe.spmm(h, to_dev(X)).cpu().numpy()
    assert_spmm_close(g, X, Y16, TOL[prec])
    assert_spmm_close(g, X, Y32, TOL[prec])


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("name", ["rmat14", "rmat13-noperm", "star9000", "complete300", "er3000",
                                  "union-isolated"])
def test_spmm_parity_packed_index(graphs, prec, name):
    """Task rows' columns as bit-packed gaps (index_format packed): same results as the oracle,
    fewer index bytes than the plain plan."""
    g = graphs[name]
    with fe.Csr.from_graph(g, index_format="packed") as h, fe.Csr.from_graph(g, tail_max=16) as hp:
        info, info_plain = h.info(), hp.info()
        assert info["index_format"] == 2 and info_plain["index_format"] == 1
        assert info["tail_max"] == 16
        if info["rows_mid"] + info["rows_hub"] > 0:
            assert info["index_bytes"] < info_plain["index_bytes"]
        for b in (1, 2, 4, 8, 16):
            X = graphgen.normal_block(g.n, b, seed=b + 30, dtype=NP[prec])
            Y = fe.spmm(h, to_dev(X)).cpu().numpy()
            assert_spmm_close(g, X, Y, TOL[prec])
            # same column order and task split as the plain plan: identical results
            assert np.array_equal(Y, fe.spmm(hp, to_dev(X)).cpu().numpy())


@pytest.mark.parametrize("fmt", ["plain", "packed"])
def test_spmm_unsorted_rows_and_duplicates(fmt):
    """CSR rows in arbitrary order with repeated entries (A_ij = multiplicity); the packed
    plan sorts each row before taking gaps (gap 0 for a repeat)."""
    g = graphgen.rmat(12, seed=4)
    rng = np.random.default_rng(3)
    rows, cols = [], []
    for i in range(g.n):
        c = list(g.colidx[g.rowptr[i]:g.rowptr[i + 1]])
        c += [int(x) for x in rng.choice(c, size=min(len(c), 3), replace=False)] if c else []
        rng.shuffle(c)
        rows.append(len(c))
        cols.extend(c)
    rowptr = np.concatenate([[0], np.cumsum(rows)]).astype(np.int64)
    colidx = np.array(cols, dtype=np.int32)
    gu = graphgen.CSR(g.n, rowptr, colidx, "unsorted-dup")
    for prec in ("f32", "f64"):
        for b in (1, 4, 16):
            X = graphgen.normal_block(g.n, b, seed=b, dtype=NP[prec])
            with fe.Csr(rowptr, colidx, index_format=fmt, tail_max=8, hub_min=64, hub_chunk=48) as h:
                Y = fe.spmm(h, to_dev(X)).cpu().numpy()
            assert_spmm_close(gu, X, Y, TOL[prec])


@pytest.mark.parametrize("kind", ["u01", "u12", "const"])
@pytest.mark.parametrize("fmt", ["plain", "packed"])
@pytest.mark.parametrize("b", [1, 4, 16])
def test_spmm_f32_one_signed_inputs(graphs, kind, fmt, b):
    """FP32 with inputs of one sign (the rounding errors of a plain in-order sum then add up
    instead of cancelling): every entry within the stated worst case 9 * 2^-24 (A|X|), on
    graphs whose rows reach every path (slices up to degree 128, warp tasks, split hubs)."""
    for name in ("rmat14", "complete70", "complete128", "complete300", "star9000", "er3000"):
        g = graphs[name]
        X = one_signed_block(kind, g.n, b, seed=11 + b)
        with fe.Csr.from_graph(g, index_format=fmt) as h:
            Y = fe.spmm(h, to_dev(X)).cpu().numpy()
        ratio = assert_spmm_close(g, X, Y, F32_BOUND)
        assert ratio <= F32_BOUND
    if kind == "const" and fmt == "plain" and b == 1:
        # the constant input catches an uncompensated kernel: plain in-order sums of the
        # degree-69 and degree-127 rows of K70 and K128 miss the 1e-6 contract
        for name in ("complete70", "complete128"):
            g = graphs[name]
            assert plain_sum_error(g, one_signed_block("const", g.n, 1, 0), range(4)) > TOL["f32"]


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_ones_give_degrees_exactly(graphs, prec):
    t = torch()
    for name in ("rmat14", "star9000", "union-isolated"):
        g = graphs[name]
        with fe.Csr.from_graph(g) as h:
            for b in (1, 4, 16):
                X = t.ones((g.n, b), dtype=t.float32 if prec == "f32" else t.float64, device="cuda")
                Y = fe.spmm(h, X).cpu().numpy()
                assert np.array_equal(Y, np.repeat(g.degrees()[:, None], b, 1).astype(Y.dtype))


def test_empty_matrix_and_single_vertex():
    t = torch()
    for n in (1, 37):
        g = graphgen.from_edges(n, [], [], "empty")
        with fe.Csr.from_graph(g) as h:
            X = t.randn((n, 4), dtype=t.float64, device="cuda")
            Y = t.full_like(X, 7.0)
            fe.spmm(h, X, Y)
            assert t.count_nonzero(Y).item() == 0


def test_handle_info_bins(graphs):
    g = graphs["rmat14"]
    with fe.Csr.from_graph(g) as h:
        i = h.info()
    deg = g.degrees()
    assert i["n"] == g.n and i["nnz"] == g.nnz and i["max_degree"] == deg.max()
    assert i["rows_empty"] == (deg == 0).sum()
    assert i["rows_tail"] == ((deg >= 1) & (deg <= 128)).sum()
    assert i["rows_mid"] == ((deg > 128) & (deg <= 4096)).sum()
    assert i["rows_empty"] + i["rows_tail"] + i["rows_mid"] + i["rows_hub"] == g.n


def test_spmm_rejects_bad_arguments(graphs):
    t = torch()
    g = graphs["cycle1001"]
    with fe.Csr.from_graph(g) as h:
        X = t.zeros((g.n, 3), dtype=t.float64, device="cuda")
        with pytest.raises(fe.FeError):
            fe.spmm(h, X)                                  # b = 3 unsupported
        X = t.zeros((g.n, 4), dtype=t.float64, device="cuda")
        with pytest.raises(fe.FeError):
            fe.spmm(h, X, X)                               # in place
        big = t.zeros((2 * g.n * 4 + 2,), dtype=t.float64, device="cuda")
        lib = fe.load()                                    # misaligned (8-byte offset)
        rc = lib.fe_spmm(h.handle, big[1:].data_ptr(), big[g.n * 4 + 1:].data_ptr(), 4, 1)
        assert rc == -1 and b"aligned" in lib.fe_last_error()


@pytest.mark.slow
@pytest.mark.parametrize("prec,b", [("f32", 4), ("f64", 4), ("f32", 16), ("f64", 1)])
def test_spmm_full_size_sampled_rows(prec, b):
    """R-MAT scale 22 (the benchmark graph), in the benchmark's launch configuration; checked
    on 20000 random rows plus every hub row and the 2000 highest-degree rows."""
    g = graphgen.rmat(22, seed=1)
    X = graphgen.normal_block(g.n, b, seed=7, dtype=NP[prec])
    with fe.Csr.from_graph(g) as h:
        Y = fe.spmm(h, to_dev(X)).cpu().numpy()
    deg = g.degrees()
    rng = np.random.default_rng(0)
    rows = np.unique(np.concatenate([rng.integers(0, g.n, 20000), np.argsort(-deg)[:2000],
                                     np.nonzero(deg > 4096)[0]]))
    assert_spmm_close(g, X, Y, TOL[prec], rows=rows)
    # ones: exact degrees everywhere
    t = torch()
    with fe.Csr.from_graph(g) as h:
        ones = t.ones((g.n, b), dtype=t.float32 if prec == "f32" else t.float64, device="cuda")
        Yd = fe.spmm(h, ones)[:, 0].cpu().numpy()
    assert np.array_equal(Yd, deg.astype(Yd.dtype))


@pytest.mark.slow
@pytest.mark.parametrize("fmt", ["plain", "packed"])
@pytest.mark.parametrize("kind", ["u12", "const"])
def test_spmm_f32_one_signed_full_size(fmt, kind):
    """R-MAT scale 22, FP32 b in {1, 4, 16}, inputs of one sign: every row of degree 64..128
    (the longest thread-per-row sums of the default plan; warp tasks in the packed plan), every
    hub row and the 2000 highest-degree rows, within 9 * 2^-24 (A|X|)."""
    g = graphgen.rmat(22, seed=1)
    deg = g.degrees()
    rows = np.unique(np.concatenate([np.nonzero((deg >= 64) & (deg <= 128))[0],
                                     np.argsort(-deg)[:2000], np.nonzero(deg > 4096)[0]]))
    with fe.Csr.from_graph(g, index_format=fmt) as h:
        for b in (1, 4, 16):
            X = one_signed_block(kind, g.n, b, seed=5 + b)
            Y = fe.spmm(h, to_dev(X)).cpu().numpy()
            assert assert_spmm_close(g, X, Y, F32_BOUND, rows=rows) <= F32_BOUND


@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_spmm_l2_window_same_results(graphs, prec):
    """An L2 access-policy window on X (l2_persist) changes only cache policy: identical results."""
    g = graphs["rmat14"]
    for b in (1, 4, 16):
        X = to_dev(graphgen.normal_block(g.n, b, seed=b, dtype=NP[prec]))
        with fe.Csr.from_graph(g) as h, fe.Csr.from_graph(g, l2_persist=True) as hl:
            assert np.array_equal(fe.spmm(h, X).cpu().numpy(), fe.spmm(hl, X).cpu().numpy())


def _f64_bound(deg, b, fmt):
    """The interface's FP64 bound for a row: (m + 9) 2^-53 of A|X|, m the longest run that a lane adds --
    in the slices (degree up to 128, packed 16) the row's steps over the lanes that share it, in multiples
    of 4; else the entries of a task of at most 4096 over the lanes that gather whole X rows."""
    if deg <= (128 if fmt == "plain" else 16):
        pieces = 1 if deg <= 32 else 2 if deg <= 64 else 4
        m = min(deg, (-(-deg // pieces) + 3) // 4 * 4)
    else:
        m = -(-min(deg, 4096) // (32 // max(1, b // 2)))
    return (m + 9) * 2.0 ** -53


@pytest.mark.parametrize("ncols", [9000, (1 << 19) + 3])
@pytest.mark.parametrize("fmt", ["plain", "packed"])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_spmm_shared_rows(prec, fmt, ncols):
    """Rows at the edges of the sharing rules: 32 | 33 and 64 | 65 steps of a slice (one, two and
    four lanes a row), 128 | 129, tasks of 1024 | 1025 and 2048 | 2049 entries (one, two and four
    warps where the matrix has few columns), hub chunks of 4096 with a ragged last one and hubs with
    more than 64 partials per lane.  Bounds: those of the interface, 9 * 2^-24 and _f64_bound of
    A|X|, the exact sums in extended precision."""
    r = np.random.default_rng(ncols)
    degs = [0, 1, 3, 4, 31, 32, 33, 35, 63, 64, 65, 66, 97, 127, 128, 129, 1023, 1024, 1025, 1057, 2047, 2048,
            2049, 2177, 4095, 4096, 4097, 5000, 8192, 8999] * 2
    cols = [np.sort(r.choice(ncols, d, replace=False)).astype(np.int32) for d in degs]
    big = np.sort(r.integers(0, ncols, 700000)).astype(np.int32)   # repeated columns
    cols.append(big)
    rowptr = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int64)
    colidx = np.concatenate(cols)
    with fe.Csr(rowptr, colidx, ncols=ncols, index_format=fmt) as h:
        for b in (1, 2, 4, 8, 16):
            X = r.standard_normal((ncols, b)).astype(NP[prec])
            Y = fe.spmm(h, to_dev(X)).cpu().numpy()
            for i, c in enumerate(cols):
                ref = X[c].astype(np.longdouble).sum(0)
                mag = np.abs(X[c]).astype(np.longdouble).sum(0)
                bound = (9 * 2.0 ** -24 if prec == "f32" else _f64_bound(len(c), b, fmt)) * mag
                assert np.all(np.abs(Y[i] - ref) <= bound), (len(c), b)


@pytest.mark.parametrize("fmt", ["plain", "packed"])
@pytest.mark.parametrize("b", [2, 4, 8, 16])
def test_spmm_f64_exponents(b, fmt):
    """The aligned integer sums of FP64 blocks: columns whose entries span all exponents (2^-1000 to
    2^1000, rising and falling along a row, so that the common exponent rises at any point), columns
    of equal sign, zeros of both signs among values, sums that cancel.  Bound of the interface
    (_f64_bound of A|X|, the sums in extended precision)."""
    r = np.random.default_rng(b)
    n = 3000
    degs = [1, 4, 11, 12, 13, 16, 31, 32, 33, 64, 65, 100, 128, 129, 200, 1025, 2049, 2600]
    cols = [np.sort(r.choice(n, d, replace=False)).astype(np.int32) for d in degs]
    rowptr = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int64)
    with fe.Csr(rowptr, np.concatenate(cols), ncols=n, index_format=fmt) as h:
        for kind in range(6):
            v = r.standard_normal((n, b))
            if kind == 0:
                v = np.ldexp(v, r.integers(-1000, 1000, (n, b)))
            elif kind == 1:
                v = np.ldexp(v, np.arange(n)[:, None] // 3 - 500)       # rises along a row
            elif kind == 2:
                v = np.ldexp(v, 500 - np.arange(n)[:, None] // 3)       # falls along a row
            elif kind == 3:
                v = np.abs(v) + 1.0
            elif kind == 4:
                v = np.where(r.random((n, b)) < 0.7, np.where(r.random((n, b)) < 0.5, 0.0, -0.0), v)
            else:
                v = np.round(v * 2.0 ** 20) * 2.0 ** 30 + np.round(r.standard_normal((n, b)) * 8)  # 53 bits
            Y = fe.spmm(h, to_dev(v)).cpu().numpy()
            for i, c in enumerate(cols):
                ref = v[c].astype(np.longdouble).sum(0)
                mag = np.abs(v[c]).astype(np.longdouble).sum(0)
                assert np.all(np.abs(Y[i] - ref) <= _f64_bound(len(c), b, fmt) * mag), (kind, len(c))


@pytest.mark.parametrize("b", [2, 4, 16])
def test_spmm_f64_special_values(b):
    """Infinities, NaN, subnormals, zeros and values near overflow give what FP64 adds give: the
    integer sums hand such rows back.  One special value per row of otherwise ordinary ones."""
    n = 2500
    r = np.random.default_rng(b)
    degs = [12, 40, 128, 130, 1100, 2100, 2499]
    cols = [np.arange(d, dtype=np.int32) for d in degs]
    rowptr = np.concatenate([[0], np.cumsum(degs)]).astype(np.int64)
    with fe.Csr(rowptr, np.concatenate(cols), ncols=n) as h:
        for special in (np.inf, -np.inf, np.nan, 1.7e308, -1.7e308):
            v = r.standard_normal((n, b))
            v[5, 0] = special
            Y = fe.spmm(h, to_dev(v)).cpu().numpy()
            for i, d in enumerate(degs):
                want = v[:d].sum(0)
                assert np.array_equal(np.isnan(Y[i]), np.isnan(want))
                ok = ~np.isnan(want)
                assert np.allclose(Y[i][ok], want[ok], rtol=1e-12, atol=1e-12)
        v = np.zeros((n, b))
        assert np.all(fe.spmm(h, to_dev(v)).cpu().numpy() == 0.0)
        assert np.all(fe.spmm(h, to_dev(-v)).cpu().numpy() == 0.0)
        v = r.integers(-1000, 1000, (n, b)) * 5e-324                    # subnormals: exact sums
        Y = fe.spmm(h, to_dev(v)).cpu().numpy()
        for i, d in enumerate(degs):
            assert np.array_equal(Y[i], v[:d].sum(0))
        v = r.standard_normal((n, b)) * 1e-290
        Y = fe.spmm(h, to_dev(v)).cpu().numpy()
        for i, d in enumerate(degs):
            assert np.all(np.abs(Y[i] - v[:d].sum(0)) <= 518 * 2.0 ** -53 * np.abs(v[:d]).sum(0) * 2)


@pytest.mark.parametrize("fmt", ["plain", "packed"])
@pytest.mark.parametrize("b", [1, 2, 4, 8, 16])
def test_spmm_f64_integers_exact(b, fmt):
    """Whole numbers of both signs whose sums fit 53 bits come out exact, as FP64 adds give them: +-1,
    small ones, 40-bit ones, sums that cancel, zeros of both signs, the same scaled by a power of
    two.  Rows in the slices (12 is the first degree with integer sums), tasks on one to four warps and
    split hub rows."""
    r = np.random.default_rng(100 + b)
    n = 9000
    degs = [2, 11, 12, 13, 15, 16, 31, 32, 33, 48, 64, 65, 100, 127, 128, 129, 200, 1025, 2049, 4097, 8999] * 3
    cols = [np.sort(r.choice(n, d, replace=False)).astype(np.int32) for d in degs]
    rowptr = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int64)
    sign = np.where(r.random((n, b)) < 0.5, -1.0, 1.0)
    alternate = np.where(np.arange(n)[:, None] % 2 == 0, 1.0, -1.0) * np.ones((1, b))
    blocks = [sign, alternate, r.integers(-9, 10, (n, b)).astype(float),
              r.integers(-2 ** 40, 2 ** 40, (n, b)).astype(float),
              np.where(r.random((n, b)) < 0.5, -0.0, sign), sign * 2.0 ** -300, sign * 3.0 * 2.0 ** 400]
    with fe.Csr(rowptr, np.concatenate(cols), ncols=n, index_format=fmt) as h:
        for k, X in enumerate(blocks):
            Y = fe.spmm(h, to_dev(X)).cpu().numpy()
            want = np.array([[float(v) for v in X[c].astype(np.longdouble).sum(0)] for c in cols])
            assert np.array_equal(Y, want), k


@pytest.mark.parametrize("tail_max", [8, 63, 64, 128])
def test_spmm_f64_b2_split(tail_max):
    """FP64 b = 2 on both sides of the rule that chooses plain adds or integer sums by the plan's
    tail_max: both index formats of one split agree bit for bit, and either is within the interface's
    bound (518 * 2^-53 of A|X|, the sums in extended precision)."""
    r = np.random.default_rng(tail_max)
    n = 6000
    degs = [1, 7, 8, 9, 12, 30, 63, 64, 65, 127, 128, 129, 500, 1025, 2049, 5000] * 3
    cols = [np.sort(r.choice(n, d, replace=False)).astype(np.int32) for d in degs]
    rowptr = np.concatenate([[0], np.cumsum([len(c) for c in cols])]).astype(np.int64)
    X = r.standard_normal((n, 2))
    Y = []
    for fmt in ("plain", "packed"):
        with fe.Csr(rowptr, np.concatenate(cols), ncols=n, index_format=fmt, tail_max=tail_max) as h:
            Y.append(fe.spmm(h, to_dev(X)).cpu().numpy())
    assert np.array_equal(Y[0], Y[1])
    for i, c in enumerate(cols):
        ref, mag = X[c].astype(np.longdouble).sum(0), np.abs(X[c]).astype(np.longdouble).sum(0)
        assert np.all(np.abs(Y[0][i] - ref) <= 518 * 2.0 ** -53 * mag)


@pytest.mark.parametrize("fmt", ["plain", "packed"])
@pytest.mark.parametrize("b", [1, 2, 4, 8])
def test_spmm_f64_hub_chunks(b, fmt):
    """A hub row of many small chunks, 64 for every lane that adds them: their sum is compensated and adds
    no more than its rounding, whatever their number.  The interface's bound, (m + 9) 2^-53 of A|X| with
    at most m = 64 / (32 / max(1, b / 2)) entries a lane in a chunk of 64, on a constant whose chunk sums round
    the same way in every addition (plain adds of 64 of them are 16 units off)."""
    c, ncols, chunks = float.fromhex("0x1.f1e4b2c84ce60p+0"), 4096, 64 * (32 // b)
    m = 64 // (32 // max(1, b // 2))
    deg = 64 * chunks
    cols = np.sort(np.arange(deg) % ncols).astype(np.int32)
    rowptr = np.array([0, deg, deg + 3], dtype=np.int64)
    X = np.full((ncols, b), c)
    with fe.Csr(rowptr, np.concatenate([cols, np.arange(3, dtype=np.int32)]), ncols=ncols, hub_min=128, hub_chunk=64,
                index_format=fmt) as h:
        assert h.info()["hub_chunks"] == chunks
        Y = fe.spmm(h, to_dev(X)).cpu().numpy()
    want = deg * np.longdouble(c)
    assert np.all(np.abs(Y[0] - want) <= (m + 9) * 2.0 ** -53 * want)
    assert np.all(np.abs(Y[1] - 3 * np.longdouble(c)) <= 3 * 2.0 ** -53 * 3 * c)


@pytest.mark.parametrize("fmt", ["plain", "packed"])
@pytest.mark.parametrize("deg,W", [(9, 0), (40, 0), (64, 0), (65, 0), (127, 0), (700, 1), (1500, 2), (5000, 4),
                                   (20 * 3000 + 17, 4)])
def test_spmm_f32_rounds_once(deg, W, fmt):
    """FP32 sums of one column, bit for bit as the summation restated on the CPU gives them: slice rows of
    one, two and four lanes (W = 0), a warp's lanes compensated and added by a tree, the warps that share a
    task and a hub row's chunks of 3000 in FP64, rounded to FP32 once."""
    from tests.test_spmm_f32_summation import hub_sum, shared_task_sum, slice_row_sum, task_sum
    ncols, chunk = 70000, 3000
    r = np.random.default_rng(deg)
    cols = np.sort(r.choice(ncols, deg, replace=False)).astype(np.int32)
    rowptr = np.array([0, deg], dtype=np.int64)
    with fe.Csr(rowptr, cols, ncols=ncols, tail_max=128, hub_min=10000, hub_chunk=chunk, index_format=fmt) as h:
        for X in (r.random(ncols) + 1.0, r.standard_normal(ncols)):
            X = X.astype(np.float32)
            Y = fe.spmm(h, to_dev(X[:, None])).cpu().numpy()
            want = (hub_sum(X[cols], chunk, 32, 1, W) if deg > 10000 else slice_row_sum(X[cols]) if W == 0 else
                    np.float32(shared_task_sum(X[cols], 32, W) if W > 1 else task_sum(X[cols], 32)))
            assert Y[0, 0] == want


def test_spmm_f32_no_error_growth_from_sharing():
    """A row that lanes or warps share is as accurate as one lane's compensated sum: over 300 rows each of
    degree 40 (two lanes), 100 (four) and 3000 (four warps) of values in [1, 2) the error stays within
    half a unit in the last place of the sum, what one rounding makes, and 2^-40 of it for the rest."""
    ncols = 9000
    r = np.random.default_rng(3)
    degs = [40] * 300 + [100] * 300 + [3000] * 300
    cols = [np.sort(r.choice(ncols, d, replace=False)).astype(np.int32) for d in degs]
    rowptr = np.concatenate([[0], np.cumsum(degs)]).astype(np.int64)
    X = (r.random((ncols, 4)) + 1.0).astype(np.float32)
    with fe.Csr(rowptr, np.concatenate(cols), ncols=ncols) as h:
        Y = fe.spmm(h, to_dev(X)).cpu().numpy().astype(np.float64)
    for i, c in enumerate(cols):
        ref = X[c].astype(np.float64).sum(0)
        half_ulp = np.spacing(ref.astype(np.float32)).astype(np.float64) / 2
        assert np.all(np.abs(Y[i] - ref) <= half_ulp + 2.0 ** -40 * ref), degs[i]
