"""CPU pins of the tables the kernels read (pg_kernel_tables_export).

The same bytes that are uploaded: digit tables with their biases per contraction
kind, the latency form's matrices and the chain's coefficients, all in Montgomery
form and with the chain scaled by seventh roots.  The tests redo with Python
integers what the kernels compute from them -- operand bytes times decoded fp16
digits plus the kind's bias block, as fp32 bit patterns, then the byte permutes
and adds of tc_combine -- and require the plain products, from the exported plain
matrices, with the scaling worked out here.  Every sum has to stay in the window
[2^23, 2^24) for any bytes.  Whole permutations through both forms equal the
oracle's, for both parameter sets.
"""
import numpy as np
import pytest

import oracle
import pg_synth

pg = pytest.importorskip("paper_2506_09505_gb300")

P = 0xFFFFFFFF00000001
R = (1 << 64) % P
RINV = pow(R, -1, P)
T, RF, RP, SPLIT, UA = 12, 8, 22, 11, 10
KIND_UA, KIND_UB, KIND_W = 8, 9, 10
HALF = [("m", 96 * 96), ("pre", 96 * 96), ("b_bias", 12 * 2 * 64), ("a_bias", 10 * 64), ("a_zcap", 4 * 64),
        ("vpa", 80 * 96), ("vpb", 96 * 96), ("bs", 96 * 96), ("w1", 96 * 96), ("w2", 96 * 96)]
WORDS = [("rc0", 1), ("add", RF), ("wm", T), ("wpre", T), ("ua", T), ("ub", T), ("ua_add", 1), ("ub_add", 1),
         ("x_add", 1), ("ba", RP), ("bb", RP), ("w", RP)]


@pytest.fixture(params=[None, "pg12_small"])
def tab(request):
    pg.load(build_if_missing=True)
    pg.params_select(request.param)
    try:
        raw = pg.kernel_tables_export()
        out, off = {"params": request.param}, 0
        for name, n in HALF:
            out[name] = np.frombuffer(raw, np.uint16, n, off)
            off += 2 * n
        for name, rows in WORDS:
            out[name] = [[int(v) for v in row] for row in np.frombuffer(raw, np.uint64, 16 * rows, off).reshape(rows, 16)]
            off += 128 * rows
        out["beta"] = [[int(v) for v in row] for row in np.frombuffer(raw, np.uint64, RP * RP, off).reshape(RP, RP)]
        assert off + 8 * RP * RP == len(raw)
        out["opt"] = {k: np.array(v, dtype=object) for k, v in pg.params_export_optimized().items()}
        out["chain"] = [np.array(v, dtype=object) for v in pg.params_export_chain()]
        yield out
    finally:
        pg.params_select(None)


def scaled(t):
    """The matrices and constants as the kernels need them, from the plain exports."""
    op, (vp, beta, w) = t["opt"], t["chain"]
    r6, seventh = pow(R, 6, P), pow(7, -1, P - 1)
    lam, kap = [0] * RP + [1], [0] * RP
    for q in reversed(range(RP)):
        kap[q] = lam[q + 1] * int(beta[q][q]) % P
        lam[q] = pow(kap[q] * r6 % P, seventh, P)
    kinv = [pow(k, -1, P) for k in kap]
    s = {"m": [[int(v) * r6 % P for v in row] for row in op["mds"]],
         "pre": [[int(v) * r6 * (lam[0] if i == 0 else 1) % P for v in row] for i, row in enumerate(op["pre"])],
         "u": [[int(v) * r6 * lam[q + 1] % P for v in vp[q]] for q in range(RP)],
         "beta": [[int(beta[q][r]) * lam[q + 1] * kinv[r] % P if r <= q else 0 for r in range(RP)] for q in range(RP)],
         "w": [[int(w[i][r]) * kinv[r] % P for r in range(RP)] for i in range(T)]}
    rc = [[int(v) % P for v in row] for row in op["full_rc"]]
    s["rc0"], s["x_add"] = rc[0], rc[4]
    s["add"] = [rc[r + 1] if r not in (3, 7) else [0] * T for r in range(RF)]
    s["add"][3] = [int(op["part_rc"][0]) * lam[0] % P] + [0] * (T - 1)
    s["u_add"] = [int(op["part_rc"][q + 1]) * lam[q + 1] % P for q in range(RP - 1)] + [0]
    return s


def decode(half, n):
    """digits[i][b][j][a] of a table of n output and 12 input words."""
    v = half.view(np.float16).astype(np.float64).reshape(n, T, 8, 8)  # row group, chunk, row, byte column
    assert (v == np.rint(v)).all() and v.min() >= -128 and v.max() <= 127
    return np.rint(v).astype(np.int64).transpose(0, 2, 1, 3)


def magic(t, kind, n):
    """[i][b]: what the bias block of a kind adds, in units of 2^-24."""
    a = t["a_bias"].view(np.float16).astype(np.float64).reshape(10, 8, 8)
    first, step = (1 + kind, 8 - kind) if kind < 8 else (0, kind - 7)
    row = np.concatenate([a[first], a[first + step]], axis=1)  # 8 rows x 16 columns
    assert (row == row[0]).all()
    b = t["b_bias"].view(np.float16).astype(np.float64).reshape(T, 2, 8, 8)
    out = np.einsum("c,ibc->ib", row[0], np.concatenate([b[:, 0], b[:, 1]], axis=2)) * 2.0 ** 24
    assert (out == np.rint(out)).all()
    return np.rint(out).astype(np.int64)[:n]


def bytes_of(words):
    return np.array([[(int(v) >> (8 * a)) & 0xFF for a in range(8)] for v in words], dtype=np.int64)


def perm(a, b, sel):
    src = [(a >> (8 * k)) & 0xFF for k in range(4)] + [(b >> (8 * k)) & 0xFF for k in range(4)]
    return sum(src[(sel >> (4 * k)) & 7] << (8 * k) for k in range(4))


def combine(w):
    """tc_bytes_sum on eight column words, mod p."""
    a = perm(w[0], w[3], 0x4210) | perm(w[3], w[6], 0x5421) << 32 | (w[6] >> 16) << 64
    b = perm(w[1], w[1], 0x2103) | perm(w[4], w[7], 0x4210) << 32 | (w[7] >> 8) << 64
    c = perm(w[2], w[2], 0x1033) | perm(w[2], w[5], 0x6542) << 32
    total = a + b + c
    assert total >> 64 < 1 << 31  # fold_small's range
    return total % P


def contract(digs, mags, operands):
    """A contraction of the kernels: the tables' digits on the operands' bytes, one accumulator."""
    z = sum(np.einsum("ibja,ja->ib", d, bytes_of(x)) for d, x in zip(digs, operands)) + mags
    assert z.min() >= 1 << 23 and z.max() < 1 << 24
    return [combine([0x3F000000 + int(v) - (1 << 23) for v in row]) for row in z]


def window(digs, mags):
    low = mags - 255 * sum(np.clip(-d, 0, None).sum(axis=(2, 3)) for d in digs)
    high = mags + 255 * sum(np.clip(d, 0, None).sum(axis=(2, 3)) for d in digs)
    assert low.min() >= 1 << 23 and high.max() < 1 << 24


def plain(mat, x, add):
    return [(sum(m * int(v) for m, v in zip(row, x)) + a) % P for row, a in zip(mat, add)]


def contractions(t):
    """(digit tables, matrices, kind, constants) of every contraction the kernels run."""
    s = scaled(t)
    half = lambda name, n=T: decode(t[name], n)  # noqa: E731
    for r in range(RF):
        if r != 3:
            yield [half("m")], [s["m"]], r, s["add"][r]
    yield [half("pre")], [s["pre"]], 3, s["add"][3]
    yield [half("vpa", UA)], [s["u"][:UA]], KIND_UA, s["u_add"][:UA]
    bs = [[s["beta"][UA + i][r] if UA + i < RP - 1 and r < SPLIT else 0 for r in range(T)] for i in range(T)]
    yield [half("vpb"), half("bs")], [s["u"][UA:], bs], KIND_UB, s["u_add"][UA:]
    w1 = [row[:SPLIT] + [0] for row in s["w"]]
    w2 = [row[SPLIT:] + [0] for row in s["w"]]
    yield [half("w1"), half("w2")], [w1, w2], KIND_W, s["x_add"]


def test_every_contraction_gives_the_scaled_products_and_constants(tab):
    edge = [[(1 << 64) - 1] * T, [0] * T, [P - 1] * T]
    for digs, mats, kind, add in contractions(tab):
        mags = magic(tab, kind, len(add))
        window(digs, mags)
        window(digs[:1], mags)  # a first table alone, before the second accumulates
        for k in range(6):
            xs = [edge[k] if k < 3 else [int(v) for v in pg_synth.words(0x8A00 + 16 * k + j, T, bound=None)]
                  for j in range(len(digs))]
            want = [sum(v) % P for v in zip(plain(mats[0], xs[0], add), *(plain(m, x, [0] * T) for m, x in zip(mats[1:], xs[1:])))]
            assert contract(digs, mags, xs) == want


def test_latency_tables_and_chain_are_the_scaled_matrices(tab):
    s = scaled(tab)
    pad = lambda row: list(row) + [0] * (16 - len(row))  # noqa: E731
    assert tab["rc0"] == [pad(s["rc0"])] and tab["x_add"] == [pad(s["x_add"])]
    assert tab["add"] == [pad(row) for row in s["add"]]
    for name, mat in (("wm", s["m"]), ("wpre", s["pre"])):
        assert tab[name] == [pad([mat[i][j] * R % P for i in range(T)]) for j in range(T)]
    assert tab["ua"] == [[s["u"][q][j] * R % P for q in range(16)] for j in range(T)]
    assert tab["ub"] == [pad([s["u"][q][j] * R % P for q in range(16, RP)]) for j in range(T)]
    assert tab["ua_add"] == [s["u_add"][:16]]
    assert tab["ub_add"] == [pad(s["u_add"][16:RP - 1] + [s["x_add"][0]])]
    assert tab["ba"] == [[s["beta"][q][r] * R % P if r < q else 0 for q in range(16)] for r in range(RP)]
    assert tab["bb"] == [pad([s["beta"][q][r] * R % P if r < q else 0 for q in range(16, RP)]) for r in range(RP)]
    assert tab["w"] == [pad([s["w"][i][r] * R % P for i in range(T)]) for r in range(RP)]
    for q in range(RP):
        assert s["beta"][q][q] == 1
        assert tab["beta"][q] == [v * R % P for v in s["beta"][q]]


def f(x):
    return pow(x, 7, P) * pow(RINV, 6, P) % P


def test_zero_capacity_bytes_are_the_constant_sbox_outputs(tab):
    for j in range(8, T):
        rows = tab["a_zcap"].reshape(4, 8, 8)[j - 8]
        assert (rows == rows[0]).all() and rows.max() < 256
        assert sum(int(v) << (8 * a) for a, v in enumerate(rows[0])) == f(scaled(tab)["rc0"][j])


def tensor_form(t, x):
    """tc_permute and tc_partial on one state."""
    dense = {r: ([decode(t["m" if r != 3 else "pre"], T)], magic(t, r, T)) for r in range(RF)}
    vpa, vpb, bs, w1, w2 = (decode(t[n], k) for n, k in (("vpa", UA), ("vpb", T), ("bs", T), ("w1", T), ("w2", T)))
    ua_m, ub_m, w_m = (magic(t, k, n) for k, n in ((KIND_UA, UA), (KIND_UB, T), (KIND_W, T)))

    def half(c, q0, u):
        s = []
        for q in range(SPLIT):
            s.append(f(c))
            if q < SPLIT - 1:
                c = (u[q] + sum(s[r] * t["beta"][q0 + q][q0 + r] for r in range(q)) * RINV + s[q]) % P
        return s
    x = [(int(v) + c) % P for v, c in zip(x, t["rc0"][0])]
    for r in range(RF):
        y = [f(v) for v in x]
        x = contract(*dense[r], [y])
        if r != 3:
            continue
        u = contract([vpa], ua_m, [y])
        s1 = half(x[0], 0, u)
        stale = [y[11]]  # input word 11 of the later operands
        u2 = contract([vpb, bs], ub_m, [y, s1 + stale])
        s2 = half(u2[0], SPLIT, u2[1:])
        ws = contract([w1, w2], w_m, [s1 + stale, s2 + stale])
        x = [(a + b) % P for a, b in zip([u2[RP - 1 - UA]] + x[1:], ws)]
    return x


def latency_form(t, x):
    """permute_wide on one state."""
    dot = lambda y, mat, e: sum(v * row[e] for v, row in zip(y, mat)) * RINV  # noqa: E731
    x = [(int(v) + c) % P for v, c in zip(x, t["rc0"][0])]
    for r in range(RF):
        y = [f(v) for v in x]
        x = [(dot(y, t["wm" if r != 3 else "wpre"], e) + t["add"][r][e]) % P for e in range(T)]
        if r != 3:
            continue
        row = [(dot(y, t["ua"], q) + t["ua_add"][0][q]) % P if q < 16 else
               (dot(y, t["ub"], q - 16) + t["ub_add"][0][q - 16]) % P for q in range(RP)]
        c, s = x[0], []
        for q in range(RP):
            s.append(f(c))
            for k in range(q + 1, RP):
                row[k] = (row[k] + s[q] * (t["ba"][q][k] if k < 16 else t["bb"][q][k - 16]) * RINV) % P
            c = (row[q] + s[q]) % P
        x = [c] + [(x[e] + t["x_add"][0][e] + dot(s, t["w"], e)) % P for e in range(1, T)]
    return x


def test_both_forms_of_the_permutation_equal_the_oracle(tab):
    rc, mds = (oracle.params() if tab["params"] is None else oracle.params_small())[:2]
    st = pg_synth.matrix(0x8B00, 6, T)
    st[0], st[1] = 0, np.uint64((1 << 64) - 1)
    want = oracle.permute(st, rc=rc, mds=mds)
    for k in range(st.shape[0]):
        assert tensor_form(tab, st[k]) == [int(v) for v in want[k]]
        assert latency_form(tab, st[k]) == [int(v) for v in want[k]]
