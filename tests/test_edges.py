"""Edges of the kernels' ranges, on the GPU through the C ABI: K ranges around the
engine's drain points and its split over K with every digit at its largest, column
tiles that are trimmed, the register blocks of the densities' pair kernel beyond one
group, and contexts of several threads and streams sharing the memory pool."""
import threading
from fractions import Fraction

import numpy as np
import pytest

import oracle
from cc3_inputs import make_inputs, make_trial_vectors
from split_tol import split_close, split_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import paper_2007_01088_gb300 as g
    return g


# 16 K per step: a tile of 1, 2, 3 steps; level 3 due (12), its limit (16, 17),
# level 2's (20, 21), level 1's (24, 28, 29), level 0's (48, 56, 57), the W build of
# nv = 250 (36); one and two parts of a tile split over K (800, 801)
@pytest.mark.parametrize("steps", [1, 2, 3, 12, 16, 17, 20, 21, 24, 28, 29, 36, 48, 56, 57, 130,
                                   800, 801])
@pytest.mark.parametrize("slices", [6, 7, 5, 4, 3])
def test_engine_sums_at_drain_points(g, steps, slices):
    """Every slice digit 127: each accumulator takes the largest sums it can, so a
    drain that comes too late loses low bits of all elements at once."""
    K = 16 * steps
    T = sum(127 * 256**p for p in range(slices))
    T -= 3 if slices == 7 else 0  # 53 of 55 bits: the last digit is 124
    x = float(T) * 2.0 ** -(7 + 8 * (slices - 1))
    A = np.full((130, K), x)
    B = np.full((24, K), x)
    B[1::2] *= -1.0
    B[2::3, ::2] *= -1.0
    sums = B.sum(axis=1) / x  # small integers
    ref = np.array([float(Fraction(x) * Fraction(x) * round(s)) for s in sums])
    C = g.cc3_debug_split_gemm(A, B, slices)
    # In units of the largest digit product (2^14): products below the last level are
    # slices - 1 pairs of digits of 2^-8s per k; the shared accumulator (levels from 4
    # on) holds 5 2^-32 per k so far, and each of its products of a step (5, 11 or 18)
    # adds to it in up to two parts (8 of its 16 k each), each of which drops at most
    # 2^-23 of that: 22 2^-23 5 2^-32 16 (1 + 2 + ... + steps) for 6 slices.
    left_out = (slices - 1) * 2.0 ** (-8 * slices) * 1.01 * K
    shared = sum(L + 1 for L in range(4, slices))
    rounded = 2 * shared * 5 * 16 * 2.0**-56 * steps * (steps + 1)
    assert np.abs(C - ref[None, :]).max() <= left_out + rounded + 2.0**-52 * K


@pytest.mark.parametrize("slices,left_out", [(6, 2.0**-44), (7, 0.0)])
def test_engine_keeps_the_last_levels_of_small_elements(g, slices, left_out):
    """Elements of digits -1, 0, 1 in the second to fourth slice, next to a large one
    that sets the scale: products of the levels 2 to 6, whose sums the accumulators hold
    exactly, down to 2^-48 of a digit product's unit (2^-14 here)."""
    rng = np.random.default_rng(slices)

    def operand(rows):
        d = rng.integers(-1, 2, size=(rows, 16, 3))
        x = (d * 2.0 ** (-8.0 * np.arange(1, 4))).sum(-1)
        x[0, 0] = 127.0
        return x / 128

    A, B = operand(130), operand(40)
    C = g.cc3_debug_split_gemm(A, B, slices)
    err = np.abs(C - A @ B.T)[1:, 1:].max() * 2.0**14
    # 6 slices leave out the 16 products of level 6; the sums are read to 2^-47
    assert err <= left_out + (2.0**-34 if slices == 6 else 2.0**-48), err


def test_engine_overflow_is_infinite(g):
    A = np.full((3, 16), 1e200)
    assert np.all(g.cc3_debug_split_gemm(A, np.full((2, 16), -1e200), 6) == -np.inf)
    C = g.cc3_debug_split_gemm(A, np.full((2, 16), 1e100), 6)
    assert np.abs(C / 1.6e301 - 1.0).max() <= 1e-13


@pytest.mark.parametrize("N", [16, 81, 97, 112, 177, 200, 250])
def test_engine_trimmed_column_tiles(g, N):
    rng = np.random.default_rng(N)
    A, B = rng.normal(size=(129, 80)), rng.normal(size=(N, 80))
    C = g.cc3_debug_split_gemm(A, B, 6)
    scale = np.abs(A).max() * np.abs(B).max() * 80
    assert np.abs(C - A @ B.T).max() <= 1e-13 * scale


# rows and K blocks of the slicing kernels that end inside a block, and batches of
# unequal size (no = 9: 156 triples)
@pytest.mark.parametrize("no,nv", [(9, 7), (8, 24), (7, 25), (2, 100)])
def test_residual_at_slicing_edges(g, no, nv):
    inp = make_inputs(no, nv, seed=3 * no + nv)
    ref = oracle.omega_inputs(inp)
    o1, o2, _ = g.Context(inp).omega(g.CC3_SPLIT_BF16)
    assert split_close(o1, ref["omega1"]), split_err(o1, ref["omega1"])
    assert split_close(o2, ref["omega2"]), split_err(o2, ref["omega2"])


@pytest.mark.parametrize("slices", [3, 4, 5, 7])
def test_residual_with_other_slice_counts(g, slices):
    # odd counts leave the last pair of slices half filled; each slice less costs 8 bits
    # of the 1e-10 that six are held to; the seventh takes these sums to the floor of the
    # double-float steps (1.4e-13 of Omega1; 5e-13 with six slices)
    inp = make_inputs(4, 19, seed=11)
    ref = oracle.omega_inputs(inp)
    ctx = g.Context(inp)
    g.cc3_ctx_set_slices(ctx.ctx, slices)
    got = ctx.omega(g.CC3_SPLIT_BF16)
    tol = 2.5e-13 if slices == 7 else 1e-10 * 256.0 ** (6 - slices)
    for x, k in zip(got, ("omega1", "omega2")):
        err, scale = split_err(x, ref[k])
        assert err <= tol * scale, (err, scale)


# permutations stacked along M in the vvov contraction: rows of 8, 64 and one past,
# 128 and both sides; singles columns of q in one and in two groups of eight (no > 8),
# the second of which ends on (nv = 80) and past (88) a column tile
@pytest.mark.parametrize("no,nv", [(17, 5), (9, 31), (9, 64), (3, 65), (9, 80), (9, 88), (2, 127),
                                   (2, 128), (3, 129)])
def test_contractions_of_stacked_permutations(g, no, nv):
    inp = make_inputs(no, nv, seed=no + 2 * nv)
    ref = oracle.omega_inputs(inp)
    ctx = g.Context(inp)
    o1, o2, _ = ctx.omega(g.CC3_SPLIT_BF16)
    assert split_close(o1, ref["omega1"]), split_err(o1, ref["omega1"])
    assert split_close(o2, ref["omega2"]), split_err(o2, ref["omega2"])
    if no * nv > 500:
        return
    R1, R2 = make_trial_vectors(no, nv, 2, seed=9)
    ref = oracle.jacobian(inp, R1, R2, [0.2, -0.1])
    got = ctx.jacobian(R1, R2, [0.2, -0.1], g.CC3_SPLIT_BF16)
    for x, k in zip(got, ("rho1", "rho2")):
        assert split_close(x, ref[k]), split_err(x, ref[k])
    ref = oracle.left_jacobian(inp, R1, R2, [0.2, -0.1])
    got = ctx.left_jacobian(R1, R2, [0.2, -0.1], g.CC3_SPLIT_BF16)
    for x, k in zip(got, ("sigma1", "sigma2")):
        assert split_close(x, ref[k]), split_err(x, ref[k])


def test_densities_beyond_one_group_of_blocks(g):
    # 66 occupied orbitals: 17 x 17 blocks of 4 x 4 products, two groups of 256
    no, nv = 66, 3
    inp = make_inputs(no, nv, seed=5)
    L1, L2 = make_trial_vectors(no, nv, 1, seed=6)
    ref = oracle.density_inputs(inp, 0.2, L1[0], L2[0])
    d = g.Context(inp).density(L1[0], L2[0], 0.2, prec=g.CC3_SPLIT_BF16)
    for x, y in zip(d, (ref["Doo"], ref["Dov"], ref["Dvv"])):
        assert split_close(x, y), split_err(x, y)


def test_doo_sums_of_many_terms(g):
    """2286 products of one sign in each thread's sums (one block per pair): their pairs
    of FP32 values take 128 terms at most before they join the total."""
    no, nv = 9, 40
    trip = [(i, j, k) for i in range(no) for j in range(i + 1) for k in range(j + 1)]
    idx = {t: n for n, t in enumerate(trip)}
    rng = np.random.default_rng(3)
    orders = ((0, 1, 2), (1, 0, 2), (2, 1, 0), (0, 2, 1), (1, 2, 0), (2, 0, 1))

    def pairs():
        x = np.abs(rng.normal(size=(len(trip), nv, nv, nv)))
        hi = x.astype(np.float32)
        return np.stack([hi, (x - hi).astype(np.float32)], -1)

    def view(x, *pqr):
        s = tuple(sorted(pqr, reverse=True))
        m = next(m for m in orders if tuple(s[u] for u in m) == pqr)
        y = x[idx[s]].astype(np.float64).sum(-1)  # 48 bits: exact
        return y.transpose(m).reshape(-1)

    tau, lt = pairs(), pairs()
    ref = np.zeros((no, no))
    for i in range(no):
        for j in range(i + 1):
            T = [view(tau, i, j, k) for k in range(no)]
            for k in range(no):
                if not i == j == k:
                    L = view(lt, i, j, k) * (1.0 if i == j else 2.0)
                    for l in range(no):
                        ref[l, k] -= 0.5 * float(np.sum(L * T[l], dtype=np.longdouble))
    got = g.cc3_debug_doo_pairs(tau, lt, blocks_per_pair=1)
    # A pair's low part, some 2^-24 of its sum S, is rounded to 2^-24 of itself in each of
    # 128 additions: about 2^-48 0.3 sqrt(128 / 3) S at random, over the root of the 500
    # pairs of an element 3e-16 of it; the same again for the products' own cross terms.
    # Pairs that take all 2286 terms are off by 3.3e-15.
    assert (np.abs(got - ref) / np.abs(ref)).max() <= 1.2e-15


# FP64 tiles of one to four row and column groups, ending one past, on and one before a multiple
# of 16, short sums (K = no) and launches split over K (left: 3 tiles, K = 3 n nv)
@pytest.mark.parametrize("no,nv", [(3, 15), (3, 16), (2, 17), (2, 40), (2, 65)])
def test_fp64_left_at_tile_edges(g, no, nv):
    inp = make_inputs(no, nv, seed=no + nv)
    L1, L2 = make_trial_vectors(no, nv, 2, seed=7)
    ref = oracle.left_jacobian(inp, L1, L2, [0.2, -0.1])
    s1, s2 = g.Context(inp).left_jacobian(L1, L2, [0.2, -0.1], g.CC3_FP64)
    for x, y in ((s1, ref["sigma1"]), (s2, ref["sigma2"])):
        assert np.abs(x - y).max() <= 1e-11 * np.abs(y).max()


def test_densities_of_several_sizes_at_once(g):
    """The D_oo kernel takes 8 KB of shared memory for 4 occupied orbitals, 57 KB for 28."""
    probs = []
    for no, nv in ((4, 8), (28, 3)):
        inp = make_inputs(no, nv, seed=no)
        L1, L2 = make_trial_vectors(no, nv, 1, seed=no)
        ref = oracle.density_inputs(inp, 0.2, L1[0], L2[0])
        probs.append((inp, L1[0], L2[0], [ref[k] for k in ("Doo", "Dov", "Dvv")]))
    bad = []

    def work(p):
        inp, L1, L2, ref = probs[p]
        c = g.Context(inp)
        for _ in range(40):
            try:
                d = c.density(L1, L2, 0.2, prec=g.CC3_SPLIT_BF16)
                if not all(split_close(x, y) for x, y in zip(d, ref)):
                    bad.append(p)
            except g.CC3Error as e:
                bad.append(str(e))

    threads = [threading.Thread(target=work, args=(p,)) for p in (0, 0, 1, 1)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad


def test_contexts_of_several_threads_share_the_pool(g):
    """Contexts made, used and destroyed by four threads on streams of their own give
    the results they give alone: no block of the pool serves two of them at a time."""
    import torch
    probs = [make_inputs(4, 20 + 7 * t, seed=t) for t in range(4)]
    alone = []
    for p in probs:
        c = g.Context(p)
        alone.append(c.omega(g.CC3_SPLIT_BF16))
        c.close()
    bad = []

    def work(t):
        st = torch.cuda.Stream()
        for _ in range(6):
            c = g.Context(probs[t], stream=st)
            for _ in range(2):
                got = c.omega(g.CC3_SPLIT_BF16)
                for x, y in zip(got, alone[t]):
                    # atomics add in another order
                    if not np.abs(x - y).max() <= 1e-13 * np.abs(y).max():
                        bad.append(t)
            c.close()

    threads = [threading.Thread(target=work, args=(t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad
