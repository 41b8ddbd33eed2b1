"""Parity of the summation variants (Section 6: GRAPE-style 64-bit fixed-point
sums; FP32 sums in index order and smallest force first) with the oracle.

Every variant evaluates its single-precision pair terms with IEEE
round-to-nearest operations in a fixed order, so the GPU must reproduce the
oracle bit for bit: forces on every block size, kernel split and ragged tail,
and (fixed point) whole block-step trajectories.
"""
import numpy as np
import pytest

import oracle
from synth import plummer, salpeter_masses, sample_active
from nbtest import nb  # noqa: F401

pytestmark = pytest.mark.gpu

EPS = 1.0 / 256
MODES = {"fixed": (1, oracle.SUM_FIXED), "fp32": (2, oracle.SUM_FP32),
         "sorted": (3, oracle.SUM_FP32_SORTED)}


def _gpu_force(nb, m, x, v, eps, idx, summation, split=0, no_force=False):
    o = nb.nb_default_opts(summation=summation, split_j=split,
                           flags=nb.NB_INIT_NO_FORCE if no_force else 0)
    ctx = nb.nb_init(m, x, v, eps, o)
    try:
        return nb.nb_force(ctx, idx)
    finally:
        nb.nb_free(ctx)


def _assert_same(got, ref, label):
    for name, g, r in zip(("acc", "jerk", "pot"), got, ref):
        bad = np.nonzero(~((g == r) | (np.isnan(g) & np.isnan(r))).reshape(len(g), -1).all(axis=1))[0]
        assert bad.size == 0, "%s %s differs at %d particles, first %d: %r vs %r" % (
            label, name, bad.size, bad[0], g[bad[0]], r[bad[0]])


@pytest.mark.parametrize("mode", sorted(MODES))
@pytest.mark.parametrize("n", [2, 3, 130, 1031, 4099])
def test_full_sweep_bit_exact(nb, mode, n):
    m, x, v = plummer(n, 200 + n)
    idx = np.arange(n, dtype=np.int32)
    if mode == "sorted" and n > 1100:
        idx = sample_active(n, 300, 5)
    got = _gpu_force(nb, m, x, v, EPS, idx, MODES[mode][0])
    ref = oracle.force_summed(m, x, v, EPS, idx, mode=MODES[mode][1], nthreads=8)
    _assert_same(got, ref, "%s n=%d" % (mode, n))


@pytest.mark.parametrize("split", [0, 1, 3, 17])
@pytest.mark.parametrize("na", [1, 7, 33, 128, 129, 255, 256, 257, 1000, 3001])
def test_fixed_block_sizes_and_splits_bit_exact(nb, na, split):
    n = 3001
    m, x, v = plummer(n, 7)
    idx = sample_active(n, na, 11 + na)
    got = _gpu_force(nb, m, x, v, EPS, idx, nb.NB_SUM_FIXED, split=split)
    ref = oracle.force_summed(m, x, v, EPS, idx, mode=oracle.SUM_FIXED, nthreads=8)
    _assert_same(got, ref, "na=%d split=%d" % (na, split))


@pytest.mark.parametrize("mode", ["fp32", "sorted"])
@pytest.mark.parametrize("na", [1, 5, 129, 700])
def test_fp32_block_sizes_bit_exact(nb, mode, na):
    n = 2053
    m, x, v = plummer(n, 17)
    idx = sample_active(n, na, 3 + na)
    got = _gpu_force(nb, m, x, v, EPS, idx, MODES[mode][0])
    ref = oracle.force_summed(m, x, v, EPS, idx, mode=MODES[mode][1], nthreads=8)
    _assert_same(got, ref, "%s na=%d" % (mode, na))


@pytest.mark.parametrize("mode", sorted(MODES))
def test_unequal_masses_far_from_origin_bit_exact(nb, mode):
    n = 1500
    m, x, v = plummer(n, 23, masses=salpeter_masses(n, 23))
    x = x + np.array([100.0, -50.0, 25.0])
    idx = sample_active(n, 200, 9)
    got = _gpu_force(nb, m, x, v, EPS, idx, MODES[mode][0])
    ref = oracle.force_summed(m, x, v, EPS, idx, mode=MODES[mode][1], nthreads=8)
    _assert_same(got, ref, mode)


def test_fixed_is_independent_of_particle_order(nb):
    n = 2500
    m, x, v = plummer(n, 31)
    perm = np.random.default_rng(4).permutation(n)
    idx = np.arange(n, dtype=np.int32)
    a0, k0, p0 = _gpu_force(nb, m, x, v, EPS, idx, nb.NB_SUM_FIXED)
    a1, k1, p1 = _gpu_force(nb, m[perm], x[perm], v[perm], EPS, idx, nb.NB_SUM_FIXED, split=5)
    assert np.array_equal(a1, a0[perm]) and np.array_equal(k1, k0[perm])
    assert np.array_equal(p1, p0[perm])


@pytest.mark.parametrize("mode", ["fp32", "sorted"])
def test_fp32_unsoftened_coincident_pair_is_skipped(nb, mode):
    m, x, v = plummer(300, 3)
    x[7] = x[3]                     # distinct particles at one point, eps = 0
    idx = np.array([3, 7, 100], dtype=np.int32)
    got = _gpu_force(nb, m, x, v, 0.0, idx, MODES[mode][0])
    ref = oracle.force_summed(m, x, v, 0.0, idx, mode=MODES[mode][1])
    assert np.all(np.isfinite(got[0]))
    _assert_same(got, ref, mode)


def test_fixed_rejects_unrepresentable_units(nb):
    # masses of 1e30 with eps = 1e-10 put the jerk unit below 2^-126: the
    # kernel reports it and the start-up sweep fails cleanly
    m, x, v = plummer(64, 2)
    with pytest.raises(nb.NbError) as ei:
        nb.nb_init(m * 1e30, x, v * 1e10, 1e-10, nb.nb_default_opts(summation=nb.NB_SUM_FIXED))
    assert ei.value.code == nb.NB_EINVAL


def test_fixed_force_dev_matches_host_call(nb):
    import torch
    n = 1200
    m, x, v = plummer(n, 5)
    idx = sample_active(n, 150, 2)
    ctx = nb.Context(m, x, v, EPS, summation=nb.NB_SUM_FIXED)
    try:
        host = ctx.nb_force(idx)
        d_idx = torch.tensor(idx, device="cuda")
        acc = torch.empty((len(idx), 3), dtype=torch.float64, device="cuda")
        jerk = torch.empty_like(acc)
        pot = torch.empty(len(idx), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        ctx.nb_force_dev(d_idx.data_ptr(), len(idx), acc.data_ptr(), jerk.data_ptr(), pot.data_ptr())
        nb.nb_get_state(ctx.ctx)    # synchronises the context's stream
        assert np.array_equal(acc.cpu().numpy(), host[0])
        assert np.array_equal(jerk.cpu().numpy(), host[1])
        assert np.array_equal(pot.cpu().numpy(), host[2])
    finally:
        ctx.nb_free()


# ---------------------------------------------------------------------------
# trajectories: with fixed-point sums the whole block-step integration is
# reproducible, so the device-driven steps must equal the oracle bit for bit


def _assert_state_equal(st, orc, label):
    for key, ref in (("x", orc.x), ("v", orc.v), ("a", orc.a), ("k", orc.k), ("t", orc.t),
                     ("level", orc.lev)):
        assert np.array_equal(st[key], ref), "%s: %s differs at %d particles" % (
            label, key, int(np.sum(np.any((st[key] != ref).reshape(len(ref), -1), axis=1))))


def test_fixed_block_steps_bit_exact(nb):
    n = 1024
    m, x, v = plummer(n, 1)
    orc = oracle.Integrator(m, x, v, EPS, summation=oracle.SUM_FIXED, nthreads=8)
    ctx = nb.Context(m, x, v, EPS, summation=nb.NB_SUM_FIXED)
    try:
        _assert_state_equal(ctx.nb_get_state(), orc, "start")
        for s in range(64):
            t, na = ctx.nb_step()
            tn, act = orc.step()
            assert t == tn / oracle.TICKS_PER_UNIT and na == len(act), s
            _assert_state_equal(ctx.nb_get_state(), orc, "step %d" % s)
    finally:
        ctx.nb_free()


def test_fixed_graph_run_bit_exact(nb):
    n = 1500
    m, x, v = plummer(n, 4, masses=salpeter_masses(n, 4))
    orc = oracle.Integrator(m, x, v, EPS, summation=oracle.SUM_FIXED, nthreads=8)
    ctx = nb.Context(m, x, v, EPS, summation=nb.NB_SUM_FIXED)
    try:
        steps, _ = ctx.nb_run(1.0 / 32)
        osteps, _, _ = orc.run(1.0 / 32)
        assert steps == osteps
        _assert_state_equal(ctx.nb_get_state(), orc, "t=1/32")
    finally:
        ctx.nb_free()


# ---------------------------------------------------------------------------
# the full-size system: sampled particles computed one by one by the oracle


@pytest.mark.parametrize("mode", sorted(MODES))
def test_million_body_sampled_bit_exact(nb, mode):
    n = 1 << 20
    m, x, v = plummer(n, 3, exact_virial_max=0)
    eps = 1.0 / 1024
    na = 16 if mode == "sorted" else 64
    idx = sample_active(n, na, 3 + na)
    got = _gpu_force(nb, m, x, v, eps, idx, MODES[mode][0], no_force=True)
    ref = oracle.force_summed(m, x, v, eps, idx, mode=MODES[mode][1], nthreads=oracle.max_threads())
    _assert_same(got, ref, "%s n=2^20" % mode)


@pytest.mark.parametrize("na", [300, 456, 600, 1216, 1217, 2432, 2433])
def test_fp32_particles_per_cta_bit_exact(nb, na):
    # on 152 SMs: 2, 3, 4, 8, 9 and 16 particles per CTA (every tile length),
    # then two rounds; 2500 bodies end inside a tile of each length.  The sums
    # have a fixed order, so the tolerance is zero.
    n = 2500
    m, x, v = plummer(n, 31)
    idx = sample_active(n, na, 5 + na)
    got = _gpu_force(nb, m, x, v, EPS, idx, nb.NB_SUM_FP32)
    ref = oracle.force_summed(m, x, v, EPS, idx, mode=oracle.SUM_FP32, nthreads=8)
    _assert_same(got, ref, "fp32 na=%d" % na)


@pytest.mark.parametrize("mode", ["fp32", "sorted"])
def test_block_size_read_on_the_device(nb, mode):
    # a device-driven block step equals predict, force and correct from the host
    m, x, v = plummer(700, 37)
    a = nb.Context(m, x, v, EPS, summation=MODES[mode][0])
    b = nb.Context(m, x, v, EPS, summation=MODES[mode][0])
    try:
        for _ in range(3):
            t, na = a.nb_step()
            idx, _ = a.nb_get_active()
            assert len(idx) == na
            b.nb_predict(t)
            b.nb_force(idx)
            b.nb_correct(idx, t)
            sa, sb = a.nb_get_state(), b.nb_get_state()
            for key in sa:
                assert np.array_equal(sa[key], sb[key]), key
    finally:
        a.nb_free()
        b.nb_free()


@pytest.mark.parametrize("mode", sorted(MODES))
@pytest.mark.parametrize("case", ["below_a_power_of_four", "tiny", "tiny_light", "huge"])
def test_square_root_exceptions_bit_exact(nb, mode, case):
    # r^2 where the short 1/sqrt gives way to the intrinsics: single-precision
    # values just below a power of four, below 2^-87 and above 2^126
    if (mode, case) == ("fixed", "tiny"):
        pytest.skip("m / r^3 is above the single-precision range: no fixed-point term")
    n = 400
    rng = np.random.RandomState(3)
    m = np.full(n, 1.0 / n)
    v = rng.normal(size=(n, 3))
    if case == "below_a_power_of_four":
        eps = 0.5   # r^2 = x^2 + 1/4 around 1, from consecutive single-precision x
        x = np.zeros((n, 3))
        d = np.float32(np.sqrt(0.75)).view(np.int32) + np.arange(-200, 199)
        x[1:, 0] = d.astype(np.int32).view(np.float32)
        r2 = (x[1:, 0].astype(np.float32) ** 2 + np.float32(0.25)).astype(np.float32).view(np.uint32)
        assert np.any((r2 & 0xffffff) - 0x7ffffa < 6)
        idx = np.array([0], dtype=np.int32)
    elif case in ("tiny", "tiny_light"):
        eps = 1e-14
        if case == "tiny_light":
            m = np.full(n, 1e-9)
        x = rng.normal(size=(n, 3)) * 1e-14
        idx = np.arange(n, dtype=np.int32)
    else:
        eps = 1.0 / 256
        x = rng.normal(size=(n, 3)) * 7e18
        idx = np.arange(n, dtype=np.int32)
    got = _gpu_force(nb, m, x, v, eps, idx, MODES[mode][0], no_force=True)
    ref = oracle.force_summed(m, x, v, eps, idx, mode=MODES[mode][1], nthreads=8)
    _assert_same(got, ref, "%s %s" % (mode, case))


@pytest.mark.parametrize("n", [255, 256, 257, 2047, 2049, 4096, 4097, 9000])
def test_sorted_chunks_bit_exact(nb, n):
    # sizes around a row, a chunk and a tile; the sums have a fixed order
    m, x, v = plummer(n, 41)
    idx = sample_active(n, 12, n)
    got = _gpu_force(nb, m, x, v, EPS, idx, nb.NB_SUM_FP32_SORTED, no_force=True)
    ref = oracle.force_summed(m, x, v, EPS, idx, mode=oracle.SUM_FP32_SORTED, nthreads=8)
    _assert_same(got, ref, "sorted n=%d" % n)


@pytest.mark.parametrize("case", ["lattice", "one_bin", "wide", "massless"])
def test_sorted_key_distributions_bit_exact(nb, case):
    # many equal keys, one bin above a chunk's size (both sorted in the
    # scratch), keys over most of the single-precision range, and zero keys
    rng = np.random.RandomState(8)
    n = 5000
    m = np.full(n, 1.0 / n)
    v = rng.normal(size=(n, 3))
    if case == "lattice":
        x = np.stack(np.meshgrid(*[np.arange(18.0)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n] / 4
    elif case == "one_bin":
        u = rng.normal(size=(n, 3))
        x = u / np.linalg.norm(u, axis=1)[:, None] * (1 + 1e-3 * rng.uniform(size=(n, 1)))
        x[0] = 0.0
    else:
        x = rng.normal(size=(n, 3)) * 10.0 ** rng.uniform(-3, 8, (n, 1))
        if case == "massless":
            m[rng.permutation(n)[:3000]] = 0.0
    idx = np.array([0, 1, 77, n - 1], dtype=np.int32)
    got = _gpu_force(nb, m, x, v, EPS, idx, nb.NB_SUM_FP32_SORTED, no_force=True)
    ref = oracle.force_summed(m, x, v, EPS, idx, mode=oracle.SUM_FP32_SORTED, nthreads=8)
    _assert_same(got, ref, "sorted %s" % case)


@pytest.mark.parametrize("n", [300, 3000, 9000])
@pytest.mark.parametrize("share", ["one", "half", "all"])
def test_sorted_masses_of_negative_zero_bit_exact(nb, n, share):
    # -0.0 is a mass of zero: its key has to fall into a bin, and its terms
    # change no sum.  Sizes of one and of several chunks.
    m, x, v = plummer(n, 43)
    where = np.random.RandomState(4).permutation(n)[:{"one": 1, "half": n // 2, "all": n}[share]]
    m = m.copy()
    m[where] = -0.0
    idx = np.unique(np.concatenate([where[:3], sample_active(n, 9, n)])).astype(np.int32)
    got = _gpu_force(nb, m, x, v, EPS, idx, nb.NB_SUM_FP32_SORTED, no_force=True)
    ref = oracle.force_summed(m, x, v, EPS, idx, mode=oracle.SUM_FP32_SORTED, nthreads=8)
    _assert_same(got, ref, "sorted n=%d" % n)
    pos = np.where(m == 0.0, 0.0, m)
    same = _gpu_force(nb, pos, x, v, EPS, idx, nb.NB_SUM_FP32_SORTED, no_force=True)
    _assert_same(got, same, "masses of +0.0, n=%d" % n)


@pytest.mark.parametrize("n", [64, 3000])
def test_fixed_masses_of_negative_zero_bit_exact(nb, n):
    # the units follow the largest mass; -0.0 is not it.  Force, persistent
    # run and graph run.
    m, x, v = plummer(n, 47)
    m = m.copy()
    m[1::3] = -0.0
    idx = sample_active(n, 20, n)
    got = _gpu_force(nb, m, x, v, EPS, idx, nb.NB_SUM_FIXED)
    ref = oracle.force_summed(m, x, v, EPS, idx, mode=oracle.SUM_FIXED, nthreads=8)
    _assert_same(got, ref, "fixed n=%d" % n)
    for flags in (0, nb.NB_RUN_GRAPH):
        orc = oracle.Integrator(m, x, v, EPS, summation=oracle.SUM_FIXED, nthreads=8)
        ctx = nb.Context(m, x, v, EPS, summation=nb.NB_SUM_FIXED, flags=flags)
        try:
            assert ctx.nb_run(1.0, 12)[0] == 12
            for _ in range(12):
                orc.step()
            _assert_state_equal(ctx.nb_get_state(), orc, "flags=%d" % flags)
        finally:
            ctx.nb_free()


@pytest.mark.parametrize("size", [127, 128, 129, 140, 500, 1000])
def test_sorted_equal_keys_in_a_chunk_bit_exact(nb, size):
    # clumps of `size` coincident particles: equal keys that differ in their jerk,
    # so that the order by index shows, around the largest bucket that is ranked
    # by comparisons, in short and in full chunks
    rng = np.random.RandomState(size)
    c = rng.normal(size=(max(2, 6000 // size), 3))
    x = np.repeat(c, size, axis=0)[rng.permutation(len(c) * size)]
    n = len(x)
    m = np.full(n, 1.0 / n)
    v = rng.normal(size=(n, 3))
    idx = sample_active(n, 6, size)
    for k in (n, 3 * size):       # the first particles alone: one short chunk
        few = idx[idx < k] if (idx < k).any() else np.array([0], dtype=np.int32)
        got = _gpu_force(nb, m[:k], x[:k], v[:k], EPS, few, nb.NB_SUM_FP32_SORTED, no_force=True)
        ref = oracle.force_summed(m[:k], x[:k], v[:k], EPS, few, mode=oracle.SUM_FP32_SORTED, nthreads=8)
        _assert_same(got, ref, "n=%d" % k)
def test_sorted_scratch_size(nb):
    # 8 n bytes for each of at most four CTAs an SM, beside what every context holds
    import torch
    n = 65536
    m, x, v = plummer(n, 3, exact_virial_max=0)
    held = []
    for summation in (nb.NB_SUM_FP32, nb.NB_SUM_FP32_SORTED):
        nb.Context(m, x, v, EPS, summation=summation, flags=nb.NB_INIT_NO_FORCE).nb_free()   # first use of the module
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        ctx = nb.Context(m, x, v, EPS, summation=summation, flags=nb.NB_INIT_NO_FORCE)
        held.append(free - torch.cuda.mem_get_info()[0])
        ctx.nb_free()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert held[1] - held[0] <= 4 * sms * 8 * n + (8 << 20)   # and the allocator's granules


def test_sorted_in_the_scratch_bit_exact(nb):
    # more keys in a bin than a chunk takes, several tiles of the scratch sort, and
    # more active particles than CTAs
    rng = np.random.RandomState(9)
    n = 20000
    m = np.full(n, 1.0 / n)
    v = rng.normal(size=(n, 3))
    x = rng.normal(size=(4, 3))[rng.randint(0, 4, n)]          # four points, keys equal in index order
    x[:5] = rng.normal(size=(5, 3))
    idx = sample_active(n, 700, 2)
    got = _gpu_force(nb, m, x, v, EPS, idx, nb.NB_SUM_FP32_SORTED, no_force=True)
    few = np.concatenate([idx[:6], idx[-6:]])
    ref = oracle.force_summed(m, x, v, EPS, few, mode=oracle.SUM_FP32_SORTED, nthreads=8)
    _assert_same([np.concatenate([g[:6], g[-6:]]) for g in got], ref, "scratch")


@pytest.mark.parametrize("case", ["far_out", "far_out_close_pair", "wide_and_crowded"])
def test_sorted_overfull_bins_bit_exact(nb, case):
    # overfull bins of 1/32 octave: one distance for nearly all (finer bins over a
    # range of one bin), the same beside a close neighbour (a range of many bins),
    # and equal keys beside keys over more octaves than finer bins can take
    rng = np.random.RandomState(12)
    n = 9000
    m = np.full(n, 1.0 / n)
    x, v = rng.normal(size=(n, 3)) * 1e-3, rng.normal(size=(n, 3))
    x[0] = [10.0, 0.0, 0.0]
    if case == "far_out_close_pair":
        x[1] = x[0] + [1e-3, 0.0, 0.0]
        x[2] = [0.0, 1e3, 0.0]
    elif case == "wide_and_crowded":
        x[3:4000] = [1.0, 2.0, 3.0]
        x[4000:] *= 10.0 ** rng.uniform(-3, 16, (n - 4000, 1))
        m[4000:] *= 10.0 ** rng.uniform(-8, 0, n - 4000)
    idx = np.array([0, 1, 2, 5000], dtype=np.int32)
    got = _gpu_force(nb, m, x, v, EPS, idx, nb.NB_SUM_FP32_SORTED, no_force=True)
    ref = oracle.force_summed(m, x, v, EPS, idx, mode=oracle.SUM_FP32_SORTED, nthreads=8)
    _assert_same(got, ref, "sorted %s" % case)
