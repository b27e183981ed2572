"""The products of a Newton-Schulz run as the library plans them
(malt_ns_plan), carried out on the CPU in the kernel's arithmetic: 16-bit
stored matrices, fp32 products, symmetric products mirrored from their upper
triangle.

The grouped form (wide frames, 3 to 8 iterations, 4 to 8 where the frames are not
preconditioned: Muon) must compute the oracle's
iteration and be no further from fp64 than the iterated bf16 form that it
replaces: as a whole frame, and row by row and column by column, so that rows
and columns far smaller than the rest keep their relative accuracy too.
Frames, runs and coefficients outside its rule keep the iterated form."""
import numpy as np
import pytest

import oracle.malt_ref as ref
from paper_2608_05088_gb300 import build
from tests.bf16_ns_model import newton_schulz_bf16


@pytest.fixture(scope="module")
def malt():
    build.build()
    import paper_2608_05088_gb300.malt as m
    return m


def _mirror(x):
    u = np.triu(x)
    return u + np.triu(u, 1).T


def run_plan(ops, Mt, rounded=True):
    """O of the frame Mt (wide) by the listed operations."""
    f32 = np.float32

    def store(x, f16):
        if not rounded:
            return x
        with np.errstate(over="ignore"):
            return x.astype(np.float16).astype(f32) if f16 else ref.round_to_bf16(x).astype(f32)

    k = float(f32(1.0) / (f32(np.linalg.norm(Mt)) + f32(1e-7)))
    dt = f32 if rounded else np.float64
    bufs = {4: (store(Mt.astype(dt), False), 0)}
    for o in ops:
        a, fa = bufs[o.a]
        b, fb = bufs[o.b]
        assert fa == o.in_f16 and fb == o.in_f16           # operands hold the type they are read as
        assert o.out not in (o.a, o.b, o.e)                 # tiles are read while others are written
        x = a @ (b.T if o.kind == 0 else b)
        x = (o.gamma * k ** o.kx) * x
        if o.e >= 0:
            assert bufs[o.e][1] == o.in_f16
            x = x + o.beta * bufs[o.e][0] + o.alpha * np.eye(x.shape[0])
        if o.kind != 2:
            x = _mirror(x)
        bufs[o.out] = (store(x.astype(dt), o.out_f16), o.out_f16)
    return bufs[6][0].astype(np.float64)


def _rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def frames(p, q):
    rng = np.random.default_rng(7)
    U = np.linalg.qr(rng.standard_normal((p, p)))[0]
    V = np.linalg.qr(rng.standard_normal((q, p)))[0].T
    i = np.arange(p)
    for name, s in (("flat", np.ones(p)), ("geometric 1e2", 10 ** (-2 * i / p)), ("1/i", 1 / (1 + i))):
        yield name, (U * s) @ V
    X = rng.standard_normal((p, q))
    yield "half the rows 1e-6", X * np.where(i < p // 2, 1.0, 1e-6)[:, None]
    yield "sparse", X * (rng.random((p, q)) < 0.02)
    yield "large norm", X * 1e6
    for sig in (0.0, 1.5, 3.0):
        G = X * np.exp(sig * rng.standard_normal(p))[:, None] * np.exp(sig * rng.standard_normal(q))[None, :]
        L, R = ((G * G).sum(1) * 0.01 + 1e-8) ** -0.125, ((G * G).sum(0) * 0.01 + 1e-8) ** -0.125
        yield f"log-normal {sig}", L[:, None] * G * R[None, :]


def is_grouped(ops):
    return any(o.in_f16 for o in ops)


GROUPED = [(k, False) for k in range(3, 9)] + [(k, True) for k in range(4, 9)]


@pytest.mark.parametrize("k,muon", GROUPED)
def test_grouped_form(malt, k, muon):
    hp = malt.hparams(ns_steps=k)
    for p, q in ((64, 512), (128, 256)):
        ops = malt.malt_ns_plan(p, q, 1000, hp, muon)
        assert is_grouped(ops)
        for name, Mt in frames(p, q):
            Mt = Mt.astype(np.float32).astype(np.float64)
            want = ref.newton_schulz(Mt, k, tuple(float(np.float32(c)) for c in ref.DEFAULT_NS_COEFFS))
            # without rounding it is the oracle's polynomial (k is fp32, so 1e-6 on it)
            assert _rel(run_plan(ops, Mt, rounded=False), want) < 1e-4, (p, q, name)
            err, old = _rel(run_plan(ops, Mt), want), _rel(newton_schulz_bf16(Mt, k), want)
            # fp32 summation order moves either by a few percent of itself
            assert err < 1.1 * old, (p, q, name, err, old)


def graded_frames(p, q, muon, k):
    """Rows or columns far smaller than the rest, down to where the form's range ends,
    and scales of sigma 3, preconditioned or (Muon) as they are."""
    rng = np.random.default_rng(11)
    X, i, j = rng.standard_normal((p, q)), np.arange(p), np.arange(q)
    for e in (4, 6) if k == 3 else (4, 6, 8):
        yield f"half the rows 1e-{e}", X * np.where(i < p // 2, 1.0, 10.0 ** -e)[:, None]
    for e in (6, 10, 14) if muon else (6, 7) if k == 3 else (6, 8):
        yield f"half the columns 1e-{e}", X * np.where(j < q // 2, 1.0, 10.0 ** -e)[None, :]
    B = X * ((i < p // 2)[:, None] == (j < q // 2)[None, :])
    yield "two blocks, one 1e-6", B * np.where(i < p // 2, 1.0, 1e-6)[:, None]
    yield "all 1e-12 (below ns_eps)", X * 1e-12
    G = X * np.exp(3.0 * rng.standard_normal(p))[:, None] * np.exp(3.0 * rng.standard_normal(q))[None, :]
    if muon:
        yield "sigma 3", G
    else:
        L, R = ((G * G).sum(1) * 0.01 + 1e-8) ** -0.125, ((G * G).sum(0) * 0.01 + 1e-8) ** -0.125
        yield "sigma 3, preconditioned", L[:, None] * G * R[None, :]


@pytest.mark.parametrize("k,muon", GROUPED)
def test_grouped_form_by_rows_and_columns(malt, k, muon):
    hp = malt.hparams(ns_steps=k)
    for p, q in ((128, 512), (256, 1024)):
        ops = malt.malt_ns_plan(p, q, 1000, hp, muon)
        assert is_grouped(ops)
        for name, Mt in graded_frames(p, q, muon, k):
            Mt = Mt.astype(np.float32).astype(np.float64)
            want = ref.newton_schulz(Mt, k, tuple(float(np.float32(c)) for c in ref.DEFAULT_NS_COEFFS))
            new, old = run_plan(ops, Mt) - want, newton_schulz_bf16(Mt, k) - want
            for axis in (0, 1):
                size = np.linalg.norm(want, axis=axis)
                e_new, e_old = (np.linalg.norm(d, axis=axis) / size for d in (new, old))
                # The median and the root mean square of many slices are steady; the
                # worst slice of either form is one draw of p or q (it varies by up to
                # 1.5 between seeds), and a slice that lost its range is off by 1.
                assert np.median(e_new) < 1.1 * np.median(e_old), (p, q, name, axis)
                assert np.sqrt(np.mean(e_new ** 2)) < 1.1 * np.sqrt(np.mean(e_old ** 2)), (p, q, name, axis)
                assert e_new.max() < 2.0 * e_old.max(), (p, q, name, axis, e_new.max(), e_old.max())


def test_values_stay_in_range(malt):
    """No stored value of a grouped run reaches fp16's largest, for the frames whose
    iterates are largest (constant singular values at the maximum of the polynomial)
    and for the coefficients with the widest bounds that the rule admits."""
    rng = np.random.default_rng(5)
    p, q = 64, 128
    U = np.linalg.qr(rng.standard_normal((p, p)))[0]
    V = np.linalg.qr(rng.standard_normal((q, p)))[0].T
    for co in (ref.DEFAULT_NS_COEFFS, (1.5, -0.5, 0.0), (4.0848, -6.8946, 2.9270), (4.5, -2.88, 0.3686)):
        for k in range(3, 9):
            for muon in (False, True):
                ops = malt.malt_ns_plan(p, q, 1000, malt.hparams(ns_steps=k, ns_coeffs=co), muon)
                if not is_grouped(ops):
                    continue
                for r in (1, 2, 3, 4, 8, 20, p):
                    s = np.where(np.arange(p) < r, 1.0, 1e-3)
                    # rank r: singular values 1 / sqrt(r); a single entry; a single row
                    for Mt in ((U * s) @ V, np.eye(p, q) * s[:, None], np.where(np.arange(p) < r, 1.0, 0.0)[:, None]
                               * np.ones((1, q))):
                        out = run_plan(ops, Mt.astype(np.float32).astype(np.float64))
                        assert np.all(np.isfinite(out)), (co, k, muon, r)


def test_rule(malt):
    hp = malt.hparams
    default = hp()
    for shape, n in (((1280, 5120), 1), ((5120, 1280), 1), ((1280, 3840), 36), ((768, 1536), 32), ((2048, 4096), 1),
                     ((256, 4096), 1), ((8, 16), 10000)):
        assert is_grouped(malt.malt_ns_plan(*shape, n, default)), shape
    for shape, n in (((1024, 2040), 100), ((4096, 4096), 1), ((256, 512), 1), ((512, 1024), 32), ((768, 768), 12)):
        assert not is_grouped(malt.malt_ns_plan(*shape, n, default)), shape
    for k, muon in ((1, False), (2, False), (3, True), (9, False), (64, True)):
        ops = malt.malt_ns_plan(256, 1024, 500, hp(ns_steps=k), muon)
        assert not is_grouped(ops) and len(ops) == 3 * k
    # the classical cubic is in range; growing or strongly amplifying runs are not
    assert is_grouped(malt.malt_ns_plan(256, 1024, 500, hp(ns_coeffs=(1.5, -0.5, 0.0))))
    for co in ((10.0, -4.0, 1.0), (4.2, -5.0, 2.0), (2.0, 1.0, 1.0), (float("nan"), 0.0, 0.0),
               (3.4445, -4.775, 1e30)):
        assert not is_grouped(malt.malt_ns_plan(256, 1024, 500, hp(ns_coeffs=co, ns_steps=8))), co


def test_iterated_form_is_unchanged(malt):
    """Square frames: the bf16 model's operations (fp32 sums in another order)."""
    Mt = np.random.default_rng(3).standard_normal((96, 96))
    want = ref.newton_schulz(Mt)
    err, old = _rel(run_plan(malt.malt_ns_plan(96, 96, 1, malt.hparams()), Mt), want), _rel(newton_schulz_bf16(Mt), want)
    assert 0.8 * old < err < 1.25 * old, (err, old)


def test_plan_of_any_number_of_matrices(malt):
    """The plan depends on the set's size through its number of tiles only, and takes
    no memory in it: a set larger than any memory is answered, not aborted on."""
    hp = malt.hparams()
    for shape in ((8, 16), (1280, 5120), (300, 77)):
        for muon in (False, True):
            big = malt.malt_ns_plan(*shape, 2 ** 31 - 1, hp, muon)
            assert is_grouped(big) == (max(shape) >= 2 * min(shape))
            assert len(malt.malt_ns_plan(*shape, 100000, hp, muon)) == len(big)
