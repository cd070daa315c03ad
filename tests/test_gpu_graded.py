"""States whose boundary tensors span many binades inside one row or column: the
digit products (program choice bit 3) have to be as good as the multiply-add
pipes (bit 3 cleared) there too."""
import numpy as np
import pytest

import oracle
from paper_1908_08553_gb300 import inputs, tn

pytestmark = pytest.mark.gpu
E = tn.TN_WORK_ENERGY
NO_PLANES = 15 & ~8


@pytest.fixture(scope="module")
def ctx():
    import torch
    torch.cuda.init()
    c = tn.tn_ctx_create(0, 0)
    yield c
    tn.tn_ctx_destroy(c)


def _full(ctx, L, W, D, A, knobs, prec):
    """log2 of the norm as (mantissa, exponent), then <X>, <ZZ>, <Z>."""
    tn.tn_autotune_set(L, W, D, prec, E, knobs)
    lat = tn.tn_create_lattice(ctx, L, W, D)
    try:
        tn.tn_set_site_tensors(lat, A)
        r, sx, zz, sz, _ = tn.tn_energy_full(lat, 1.0, 3.04, prec, tn.TN_SCHED_AUTO, L, W)
        return (r.norm.mant, r.norm.exp2), sx, zz, sz
    finally:
        tn.tn_destroy_lattice(lat)
        tn.tn_autotune_clear()


def _off(norm, ref):
    return abs(norm[0] / ref[0] * 2.0 ** (norm[1] - ref[1]) - 1.0)


def seam_ising(L, W, beta):
    """Classical Ising model as a PEPS (the norm is its partition function): legs carry
    spins, all couplings +1 but -1 on the lower half's middle column of bonds, so the
    two halves prefer different configurations on the cut between them.  All entries
    are non-negative: sums of products lose nothing to cancellation."""
    w = np.exp(0.5 * beta * np.array([[1.0, -1.0], [-1.0, 1.0]]))
    one = np.ones((1, 2))
    sites = []
    for r in range(L):
        for c in range(W):
            u, l, dn, rt = inputs.site_dims(L, W, 2, r, c)
            up = w if u > 1 else one
            anti = r >= L // 2 and c == W // 2
            left = (1.0 / w if anti else w) if l > 1 else one
            A = np.zeros((2, u, l, dn, rt))
            for p in range(2):
                A[p, :, :, p if dn > 1 else 0, p if rt > 1 else 0] = np.outer(up[:, p], left[:, p])
            sites.append(A.ravel())
    return np.concatenate(sites)


# The products' operands are non-negative, so every sum keeps its relative accuracy: in
# FP64 three ring products and 64 absorptions of at most 256 + 16 roundings each stay
# below (3 * 256 + 64 * 16) 2^-53 = 2e-13 if all of them pull one way.
@pytest.mark.parametrize("beta", [1.5, 2.0])
def test_frustrated_seam_fp64(ctx, beta):
    L = W = 8
    A = seam_ising(L, W, beta)
    ref = oracle.norm(L, W, 2, A)
    obs = oracle.observables(L, W, 2, A, with_z=True)
    for knobs in (NO_PLANES, 15):
        norm, sx, zz, sz = _full(ctx, L, W, 2, A, knobs, tn.TN_FP64)
        assert _off(norm, ref) <= 1e-12, knobs
        for x, y in ((sx, obs.sx), (zz, obs.szsz), (sz, obs.sz)):
            assert np.max(np.abs(x - y)) <= 1e-12, knobs


# FP32: a product's roundings add up to sqrt(1024) 2^-24 = 2e-6 of a sum of non-negative
# terms, a digit product's to at most 2e-6; three of them and 100 absorptions of 4e-7
# (0.24e-6 sqrt(100)) give 1.2e-5 at most.
@pytest.mark.parametrize("beta", [0.75, 1.0])
def test_frustrated_seam_fp32(ctx, beta):
    L = W = 10
    A = seam_ising(L, W, beta)
    ref, _, zz64, _ = _full(ctx, L, W, 2, A, NO_PLANES, tn.TN_FP64)
    for knobs in (NO_PLANES, 15):
        norm, _, zz, _ = _full(ctx, L, W, 2, A, knobs, tn.TN_FP32)
        assert _off(norm, ref) <= 1.2e-5, knobs
        assert np.max(np.abs(zz - zz64)) <= 1.2e-5, knobs


def parity_state(L, W, eps, seed, D=2):
    """Random state that conserves the parity of its legs up to entries of size eps:
    nearly block-diagonal boundary tensors, and <X> (odd) of the order of eps."""
    sites = []
    for t in inputs.split_sites(inputs.random_lattice(L, W, D, seed), L, W, D):
        odd = np.indices(t.shape).sum(0) % 2 == 1
        sites.append(np.where(odd, eps * t, t).ravel())
    return np.concatenate(sites)


# <X> is a sum of terms eps times those of the norm, so it keeps a relative accuracy
# of its own; the pipe's error is the yardstick (a handful of roundings either way),
# with 2^-20 of the largest <X> for the products' own.
@pytest.mark.parametrize("L,W,prec,ulp", [(8, 8, tn.TN_FP64, 2.0 ** -46), (10, 10, tn.TN_FP32, 2.0 ** -17)])
@pytest.mark.parametrize("eps", [2.0 ** -10, 2.0 ** -20])
def test_nearly_block_diagonal(ctx, L, W, prec, ulp, eps):
    A = parity_state(L, W, eps, 4100)
    ref = (oracle.observables(L, W, 2, A).sx if prec == tn.TN_FP64
           else _full(ctx, L, W, 2, A, NO_PLANES, tn.TN_FP64)[1])
    pipe, dig = (_full(ctx, L, W, 2, A, k, prec)[1] for k in (NO_PLANES, 15))
    bound = 4 * np.max(np.abs(pipe - ref)) + ulp * np.max(np.abs(ref))
    assert np.max(np.abs(dig - ref)) <= bound


# exactly conserved parity: half of every boundary tensor is structurally zero
def test_conserved_parity(ctx):
    L, W = 8, 8
    A = parity_state(L, W, 0.0, 4200)
    obs = oracle.observables(L, W, 2, A, with_z=True)
    _, sx, zz, sz = _full(ctx, L, W, 2, A, 15, tn.TN_FP64)
    assert np.all(sx == 0.0)
    for x, y in ((zz, obs.szsz), (sz, obs.sz)):
        assert np.max(np.abs(x - y)) <= 1e-12


# D = 3: absorptions of 81 and 9 legs from digits; <X> against the oracle's as above
@pytest.mark.parametrize("eps", [2.0 ** -10, 2.0 ** -18, 2.0 ** -26])
def test_nearly_block_diagonal_d3(ctx, eps):
    L, W = 4, 5
    A = parity_state(L, W, eps, 4300, 3)
    ref = oracle.observables(L, W, 3, A).sx
    pipe, dig = (_full(ctx, L, W, 3, A, k, tn.TN_FP64)[1] for k in (NO_PLANES, 15))
    assert np.max(np.abs(dig - ref)) <= 4 * np.max(np.abs(pipe - ref)) + 2.0 ** -46 * np.max(np.abs(ref))


# one end of every bond padded: leg index D - 1 has zeros on the right / lower site and
# entries 2^g above the others on the left / upper one.  The state is the one of bond
# dimension D - 1; the inputs' largest entries meet empty rows of the site matrices.
# 4 x 5 sites of at most 81 roundings a step: sqrt(20 * 81) 2^-53 = 4.5e-15 on a sum,
# 10 times that on the ratios.
@pytest.mark.parametrize("D", [2, 3])
@pytest.mark.parametrize("g", [6, 9, 30])
def test_bonds_padded_at_one_end(ctx, D, g):
    L, W = 4, 5
    sites = [np.array(t) for t in inputs.split_sites(inputs.random_lattice(L, W, D, 4400 + D), L, W, D)]
    for t in sites:
        for axis in (1, 2):
            if t.shape[axis] > 1:
                np.moveaxis(t, axis, 0)[D - 1] = 0.0
        for axis in (3, 4):
            if t.shape[axis] > 1:
                np.moveaxis(t, axis, 0)[D - 1] *= 2.0 ** g
    A = inputs.join_sites(sites)
    small = inputs.join_sites([t[:, :max(1, t.shape[1] - (t.shape[1] > 1)), :max(1, t.shape[2] - (t.shape[2] > 1)),
                                 :max(1, t.shape[3] - (t.shape[3] > 1)), :max(1, t.shape[4] - (t.shape[4] > 1))]
                               for t in sites])
    obs = oracle.observables(L, W, D - 1, small, with_z=True)
    _, sx, zz, sz = _full(ctx, L, W, D, A, 15, tn.TN_FP64)
    for x, y in ((sx, obs.sx), (zz, obs.szsz), (sz, obs.sz)):
        assert np.max(np.abs(x - y)) <= 5e-14


# an output of a product may lie as far below its operands' largest entries as FP32
# reaches: in the upper half, column 2's sites carry one sector along the cut, 0 with
# weight 1 or 1 with a small one, column 3's sector 2 with weight 1 or 1 with a small
# one; only sector 1 crosses, so that half's ring product is 2^-112 of its operands'
# largest entries, in rows and columns of its own.  FP32 keeps 2^-24 of each of the
# norm's 729 x 729 products of random sign: 2e-5 of a norm 1/300 of its terms' size at
# worst.
def test_fp32_products_of_small_rows_and_columns(ctx):
    L = W = 6
    D, f = 3, 2.0 ** -9.3
    sites = [np.array(t) for t in inputs.split_sites(inputs.random_lattice(L, W, D, 4500), L, W, D)]
    for r in range(L // 2):
        for c, legs, weight in ((2, (1, 3, 4), (1.0, f, 0.0)), (3, (1, 3, 2), (0.0, f, 1.0))):
            t = sites[r * W + c]
            idx = np.indices(t.shape)
            cut = idx[legs[2]]
            same = [idx[leg] == cut for leg in legs[:2] if t.shape[leg] > 1]
            sites[r * W + c] = t * np.array(weight)[cut] * np.logical_and.reduce(same)
    A = inputs.join_sites(sites)
    ref = oracle.norm(L, W, D, A)
    for knobs in (NO_PLANES, 15):
        norm, _, _, _ = _full(ctx, L, W, D, A, knobs, tn.TN_FP32)
        assert _off(norm, ref) <= 2e-5, knobs


# outputs left to the pipe in a large launch (8 of its 16 x 16 tiles a block) and in a
# small one (one a block): the same sums in the same order, so the same bits.  256^3 and
# 729^3 products (ragged last tiles of a row); the batches' launches have more than
# 49,152 tiles, those of one lattice fewer.
@pytest.mark.parametrize("L,W,D,n", [(8, 8, 2, 128), (6, 6, 3, 24)])
def test_batches_of_graded_states_equal_alone(ctx, L, W, D, n):
    kinds = [parity_state(L, W, 2.0 ** -20, 4600, D), inputs.random_lattice(L, W, D, 4601),
             parity_state(L, W, 2.0 ** -12, 4602, D)]
    if D == 2:
        kinds.append(seam_ising(L, W, 1.5))
    b, rows = tn.tn_batch_create(ctx, [L] * n, [W] * n, [D] * n, tn.TN_FP64), []
    try:
        tn.tn_batch_set_tensors(b, np.concatenate([kinds[k % len(kinds)] for k in range(n)]))
        tn.tn_batch_run(b, 1.0, np.full(n, 3.04))
        got = tn.tn_batch_results_host(b).reshape(n, -1)
    finally:
        tn.tn_batch_destroy(b)
    for A in kinds:
        b1 = tn.tn_batch_create(ctx, [L], [W], [D], tn.TN_FP64)
        try:
            tn.tn_batch_set_tensors(b1, A)
            tn.tn_batch_run(b1, 1.0, np.full(1, 3.04))
            rows.append(tn.tn_batch_results_host(b1).copy())
        finally:
            tn.tn_batch_destroy(b1)
    for k in range(n):
        assert np.array_equal(got[k], rows[k % len(kinds)]), k
