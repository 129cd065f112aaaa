"""GPU parity: the CUDA path (through the C ABI) against the complex128 oracle.

Every result is held to its plain relative error |a - a_ref| / |a_ref| (tests/parity.py):
complex128 1e-12 (against the state vector / oracle), complex64 1e-5, split-TF32 1e-5 and
split-BF16 1e-4 -- the bounds the workload definition states for single-amplitude results.
"""
import math

import numpy as np
import pytest

from oracle import contract as oc
from oracle import costs as ocost
from oracle import greedy as og
from oracle import statevector as sv
from paper_2507_20667_gb300 import inputs as tni
from parity import TOL, amplitude_bitstring, check, check_observable

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tnsa():
    from paper_2507_20667_gb300 import tnsa as mod
    return mod


@pytest.fixture(scope="module")
def ctx(tnsa):
    return tnsa.tn_ctx_create(0)


def oracle_amp(net):
    steps = og.greedy_steps(list(ocost.leaf_legs(net)), ocost.edge_dims(net))
    return oc.contract_scalar(net, steps)


def gpu_amp(tnsa, ctx, net, plan=None, prec="c64", k=1, **kw):
    h = tnsa.tn_build(net)
    if plan is None:
        plan = tnsa.tn_plan_create(h, k=k, **kw)
    m, e, info = tnsa.tn_contract(ctx, h, plan, prec)
    return tnsa.amplitude(m, e), info


@pytest.mark.parametrize("prec", ["c128", "c64", "tf32", "bf16"])
def test_cfg1_all_precisions(tnsa, ctx, prec):
    circ, _ = tni.cfg1()
    x, ref, _ = amplitude_bitstring(lambda y: sv.amplitude(circ, y), 10, 1001, tni.random_bitstring)
    net = tni.amplitude_tn(circ, x)
    assert abs(oracle_amp(net) - ref) < 1e-13 * abs(ref)
    got, info = gpu_amp(tnsa, ctx, net, prec=prec)
    check(got, ref, TOL[prec])
    assert info["launches"] >= 1


@pytest.mark.parametrize("prec", ["c128", "c64"])
def test_closed_forms(tnsa, ctx, prec):
    n = 9
    g = tni.ghz(n)
    for bits, want in (([0] * n, 1 / math.sqrt(2)), ([1] * n, 1 / math.sqrt(2))):
        got, _ = gpu_amp(tnsa, ctx, tni.amplitude_tn(g, bits), prec=prec)
        check(got, want, TOL[prec], "GHZ")
    # an exactly zero amplitude has no relative error: its error is bounded on the scale 2^(-1/2)
    # of the nonzero ones
    got, _ = gpu_amp(tnsa, ctx, tni.amplitude_tn(g, [0, 1] + [0] * (n - 2)), prec=prec)
    assert abs(got) <= TOL[prec] / math.sqrt(2)
    circ = tni.brickwork_1d(8, 6, seed=31)
    for net in (tni.inverse_tn(circ), tni.norm_tn(circ)):
        got, _ = gpu_amp(tnsa, ctx, net, prec=prec, k=2, iterations=20,
                         position=net.qubit)
        check(got, 1.0, TOL[prec], "<0|C^-1 C|0> or <psi|psi>")
    zz = sv.zz_expectation(circ, 2, 6)
    got, _ = gpu_amp(tnsa, ctx, tni.zz_tn(circ, 2, 6), prec=prec)
    check_observable(got, zz, TOL[prec], 1.0, "<Z2 Z6>")


@pytest.mark.parametrize("k", [1, 2, 3, 4, 6])
def test_partition_and_order_invariance(tnsa, ctx, k):
    """The amplitude does not depend on the tree or the partitioning (Section 2.3)."""
    circ = tni.brickwork_1d(12, 10, seed=40)
    x, ref, _ = amplitude_bitstring(lambda y: sv.amplitude(circ, y), 12, 41, tni.random_bitstring)
    net = tni.amplitude_tn(circ, x)
    pos = net.qubit if k > 1 else None
    for mode in ("directed", "naive"):
        got, _ = gpu_amp(tnsa, ctx, net, prec="c128", k=k, mode=mode, iterations=30, seed=k,
                         position=pos)
        check(got, ref, TOL["c128"], mode)
        got, _ = gpu_amp(tnsa, ctx, net, prec="c64", k=k, mode=mode, iterations=30, seed=k,
                         position=pos)
        check(got, ref, TOL["c64"], mode)


@pytest.mark.parametrize("seed", range(6))
def test_random_networks_mixed_dims(tnsa, ctx, seed):
    """Non-power-of-two dimensions exercise the general (div/mod) index maps."""
    net = tni.random_network(14, 10, (1, 2, 3, 5, 6), seed=seed)
    ref = oracle_amp(net)
    for prec in ("c128", "c64"):
        got, _ = gpu_amp(tnsa, ctx, net, prec=prec)
        check(got, ref, TOL[prec], prec)


def test_random_tree_import(tnsa, ctx):
    """Arbitrary imported trees, with larger intermediates and the tiled kernel class."""
    net = tni.random_network(10, 12, (2, 3, 4), seed=77)
    ref = oracle_amp(net)
    rng = np.random.default_rng(5)
    n = net.n_tensors
    for trial in range(3):
        alive, steps, nxt = list(range(n)), [], n
        while len(alive) > 1:
            i, j = sorted(rng.choice(len(alive), 2, replace=False))
            a, b = alive[i], alive[j]
            steps.append((min(a, b), max(a, b)))
            alive = [t for t in alive if t not in (a, b)] + [nxt]
            nxt += 1
        h = tnsa.tn_build(net)
        plan = tnsa.tn_plan_import(h, steps)
        for prec in ("c128", "c64"):
            m, e, info = tnsa.tn_contract(ctx, h, plan, prec)
            check(tnsa.amplitude(m, e), ref, TOL[prec], f"tree {trial} {prec}")


@pytest.mark.parametrize("prec", ["c128", "c64", "tf32", "bf16"])
def test_cfg3_oracle_instance(tnsa, ctx, prec):
    """2D grid 4x5, depth 8, k = 8 partitions: against the 2^20 state vector."""
    circ, _ = tni.cfg3(small=True)
    x, ref, _ = amplitude_bitstring(lambda y: sv.amplitude(circ, y), 20, 1003, tni.random_bitstring)
    net = tni.amplitude_tn(circ, x)
    got, info = gpu_amp(tnsa, ctx, net, prec=prec, k=8, iterations=200, steps_per_temp=8, seed=7,
                        position=net.qubit)
    check(got, ref, TOL[prec])
    if prec in ("tf32", "bf16"):   # the dense fan-in steps run on the tensor cores
        assert info["n_tc"] > 0


def test_cfg2_full_size(tnsa, ctx):
    """24-qubit brickwork, depth 14, k = 4 SA partitions, complex64; the oracle contracts the
    same network along its own Greedy tree."""
    circ, _ = tni.cfg2()
    x, ref, _ = amplitude_bitstring(lambda y: oracle_amp(tni.amplitude_tn(circ, y)), 24, 1002,
                                    tni.random_bitstring)
    net = tni.amplitude_tn(circ, x)
    h = tnsa.tn_build(net)
    plan = tnsa.tn_plan_create(h, k=4, iterations=2000, steps_per_temp=8, seed=7,
                               position=net.qubit)
    for prec in ("c64", "c128"):
        m, e, info = tnsa.tn_contract(ctx, h, plan, prec)
        check(tnsa.amplitude(m, e), ref, TOL[prec], prec)


def test_new_bitstring_reuploads_leaves(tnsa, ctx):
    circ, x = tni.cfg1()
    net = tni.amplitude_tn(circ, x)
    h = tnsa.tn_build(net)
    plan = tnsa.tn_plan_create(h, k=1)
    y = 1 - np.asarray(x)
    n = circ.n_qubits
    for q in range(n):  # bra tensors are the last n tensors
        v = np.zeros(2, np.complex128)
        v[y[q]] = 1
        tnsa.tn_net_set_tensor(h, net.n_tensors - n + q, v)
    m, e, _ = tnsa.tn_contract(ctx, h, plan, "c128")
    check(tnsa.amplitude(m, e), sv.amplitude(circ, y), TOL["c128"])


def test_degenerate_networks(tnsa, ctx):
    class Net:
        pass
    # a single scalar tensor
    s = Net()
    s.degrees = np.array([0], np.int32)
    s.dims = np.zeros(0, np.int64)
    s.data = np.array([0.25, -0.5])
    s.edges = np.zeros((0, 4), np.int32)
    h = tnsa.tn_build(s)
    plan = tnsa.tn_plan_create(h, k=1)
    for prec in ("c128", "c64"):
        m, e, _ = tnsa.tn_contract(ctx, h, plan, prec)
        assert tnsa.amplitude(m, e) == complex(0.25, -0.5)
    # two disconnected closed components: the outer product of their amplitudes
    c1, c2 = tni.brickwork_1d(4, 3, seed=1), tni.brickwork_1d(5, 3, seed=2)
    n1 = tni.amplitude_tn(c1, [0, 1, 1, 0])
    n2 = tni.amplitude_tn(c2, [1, 1, 0, 0, 1])
    both = Net()
    both.tensors = n1.tensors + n2.tensors
    both.degrees = np.concatenate([n1.degrees, n2.degrees])
    both.dims = np.concatenate([n1.dims, n2.dims])
    both.data = np.concatenate([n1.data, n2.data])
    e2 = n2.edges.copy()
    e2[:, 0] += n1.n_tensors
    e2[:, 2] += n1.n_tensors
    both.edges = np.concatenate([n1.edges, e2])
    want = sv.amplitude(c1, [0, 1, 1, 0]) * sv.amplitude(c2, [1, 1, 0, 0, 1])
    h = tnsa.tn_build(both)
    for k in (1, 2, 3):
        plan = tnsa.tn_plan_create(h, k=k, iterations=10)
        m, e, _ = tnsa.tn_contract(ctx, h, plan, "c128")
        check(tnsa.amplitude(m, e), want, TOL["c128"], f"k={k}")
    # an open network is refused by the scalar entry point
    o = tni.random_network(5, 2, (2,), seed=1, n_open=1)
    h = tnsa.tn_build(o)
    plan = tnsa.tn_plan_create(h, k=1)
    with pytest.raises(tnsa.TnError) as ei:
        tnsa.tn_contract(ctx, h, plan, "c64")
    assert ei.value.status == tnsa.TN_EUNSUPPORTED


def test_budget_rejection(tnsa):
    ctx = tnsa.tn_ctx_create(0, hbm_budget_bytes=1024)
    net = tni.amplitude_tn(*tni.cfg1())
    h = tnsa.tn_build(net)
    plan = tnsa.tn_plan_create(h, k=1)
    with pytest.raises(tnsa.TnError) as ei:
        tnsa.tn_contract(ctx, h, plan, "c64")
    assert ei.value.status == tnsa.TN_EBUDGET


@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("shift", [-8, 8])
def test_power_of_two_scaling_is_load_bearing(tnsa, ctx, prec, shift):
    """Every leaf of cfg1 multiplied by 2^shift: the value is 2^(146 shift) times the amplitude,
    far outside the range of FP32 and of FP64 (2^-1168 or 2^1168), so only the per-step
    power-of-two scaling keeps the intermediates representable.  Scaling by powers of two is
    exact, so the mantissa is bit-identical to the unscaled run and the exponent moves by exactly
    146 shift; the unscaled value agrees with the oracle."""
    circ, x = tni.cfg1()
    net = tni.amplitude_tn(circ, x)
    h = tnsa.tn_build(net)
    plan = tnsa.tn_plan_create(h, k=1)
    m0, e0, _ = tnsa.tn_contract(ctx, h, plan, prec)
    check(tnsa.amplitude(m0, e0), sv.amplitude(circ, x), TOL[prec])

    class Scaled:
        pass
    s = Scaled()
    s.degrees, s.dims, s.edges = net.degrees, net.dims, net.edges
    s.data = np.ldexp(np.asarray(net.data, np.float64), shift)
    hs = tnsa.tn_build(s)
    m1, e1, _ = tnsa.tn_contract(ctx, hs, tnsa.tn_plan_create(hs, k=1), prec)
    assert e1 - e0 == shift * net.n_tensors
    assert np.array([m1]).view(np.uint64).tolist() == np.array([m0]).view(np.uint64).tolist()


def test_rows_steps_with_odd_width(tnsa, ctx):
    """Mixed-dimension networks (dims 3 and 5) with every step global: the row kernel of the
    dataflow kernel runs steps of odd width N, where the paired 16-byte loads of B have a
    one-entry tail; compared with the oracle."""
    found = 0
    for seed in range(40):
        net = tni.random_network(12, 6, (3, 5), seed=seed)
        h = tnsa.tn_build(net)
        plan = tnsa.tn_plan_create(h, k=1)
        steps = tnsa.tn_plan_compile_steps(h, plan, "c64", 0)
        odd = [s for s in steps if s[0] == 0 and s[2] % 2 == 1 and s[2] > 1]
        if not odd:
            continue
        found += 1
        ref = oracle_amp(net)
        c = tnsa.tn_ctx_create(0)
        tnsa.tn_ctx_set_local_budget(c, 0)
        for prec in ("c64", "c128"):
            m, e, _ = tnsa.tn_contract(c, h, plan, prec)
            check(tnsa.amplitude(m, e), ref, TOL[prec], f"seed {seed} {prec}")
        if found == 4:
            break
    assert found >= 1


def _split_row_steps(geo):
    """Steps of a 256-thread block program that the narrow row kernel runs with 2 or 4 threads per
    row: not small enough for one warp (M N > 256 or M N K > 4096), N and K <= 16, and so few rows
    (R = 32 / NT per thread, NT = N rounded up to 4, 8 or 16) that at least half the threads would
    hold none.  Both operand orders are considered, since the program may swap A and B."""
    hits = []
    for kind, M, N, K, *_ in geo:
        for m, n in ((M, N), (N, M)):
            if n > 16 or K > 16 or not (m * n > 256 or m * n * K > 4096):
                continue
            nt = 4 if n <= 4 else 8 if n <= 8 else 16
            if 2 * -(-m // (32 // nt)) <= 256:
                hits.append((int(m), int(n), int(K)))
    return hits


def test_block_row_steps_shared_between_threads(tnsa, ctx):
    """Mixed-dimension networks (dims 3 and 5) that run entirely as subtree programs: their
    block-wide row steps with few rows share each row between 2 or 4 threads, and odd widths leave
    part of the last thread's columns empty.  Compared with the oracle in complex64 and
    complex128."""
    found = 0
    for seed in range(40):
        net = tni.random_network(12, 6, (3, 5), seed=seed)
        h = tnsa.tn_build(net)
        plan = tnsa.tn_plan_create(h, k=1)
        hits = [s for s in _split_row_steps(tnsa.tn_plan_compile_steps(h, plan, "c64", 0)) if s[1] % 2]
        progs = tnsa.tn_plan_compile_steps(h, plan, "c64", 64 * 1024)
        if not hits or not all(p[0] == 5 for p in progs):
            continue
        found += 1
        ref = oracle_amp(net)
        for prec in ("c64", "c128"):
            m, e, _ = tnsa.tn_contract(ctx, h, plan, prec)
            check(tnsa.amplitude(m, e), ref, TOL[prec], f"seed {seed} {prec} {hits}")
        if found == 6:
            break
    assert found >= 3


@pytest.mark.parametrize("prec", ["c64", "c128"])
def test_large_leaves_max_abs_across_slices(tnsa, ctx, prec):
    """Two vectors of 50000 entries (leaves above 64 entries are converted by blocks per slice of
    the leaf, whose max-abs values merge into one): their entries are about 2^60, except one near
    the end of each at 0.75 * 2^127, just below the largest entry the boundary accepts.  Scaled by
    the max-abs of the small entries alone, the product of the two large ones would overflow
    complex64; the true max-abs of the whole leaf keeps it finite, and a max-abs of 2^126 or more
    still gives a normal scale factor (the scale exponent stops at 126).  The dot product is
    compared with numpy on the stored values."""
    L = 50000
    rng = np.random.default_rng(11)
    big, small = 127, 60

    def vec():
        v = (rng.standard_normal(L) + 1j * rng.standard_normal(L)) * 2.0 ** small
        v[L - 7] = (0.75 + 0.5j) * 2.0 ** big
        return v

    class Dot:
        pass
    net = Dot()
    u, v = vec(), vec()
    net.degrees = np.array([1, 1], np.int32)
    net.dims = np.array([L, L], np.int64)
    net.edges = np.array([[0, 0, 1, 0]], np.int32)
    net.data = np.concatenate([u, v]).view(np.float64)
    h = tnsa.tn_build(net)
    plan = tnsa.tn_plan_import(h, [(0, 1)])
    m, e, _ = tnsa.tn_contract(ctx, h, plan, prec)
    m = complex(m)
    assert np.isfinite(m.real) and np.isfinite(m.imag)
    st = np.complex64 if prec == "c64" else np.complex128
    us, vs = u.astype(st).astype(np.complex128), v.astype(st).astype(np.complex128)

    def down(z):   # exact scaling by 2^-big, so that the products stay inside the float64 range
        return np.ldexp(z.real, -big) + 1j * np.ldexp(z.imag, -big)
    ref = np.dot(down(us), down(vs))
    got = complex(np.ldexp(m.real, int(e) - 2 * big), np.ldexp(m.imag, int(e) - 2 * big))
    check(got, ref, TOL[prec], f"{prec} dot of {L} entries")


# small steps: (free legs of A, shared legs, free legs of B) -- one pass or several, shared indices split
# over lanes or not, tabulated index maps (up to 256 outputs) or decoded ones, dims that are no powers of two
@pytest.mark.parametrize("legs", [((2,), (2,), ()), ((2, 2), (2,), (2, 2)), ((2,) * 3, (2,) * 4, (2,)),
                                  ((2,) * 4, (2,) * 3, (2,) * 4), ((2,) * 4, (2,) * 4, (2,) * 4), ((), (2,) * 6, (2,)),
                                  ((2,) * 5, (2,), ()), ((4, 8), (2, 4), (4,)), ((3,), (3,), (2,)), ((5,), (3, 2), (3,)),
                                  ((3, 7), (2,), (5,)), ((2, 8), (1,), (2, 4))])
@pytest.mark.parametrize("precision", ["c64", "c128"])
def test_small_step_shapes(tnsa, legs, precision):
    fa, sh, fb = legs
    rng = np.random.default_rng(len(fa) * 100 + len(sh) * 10 + len(fb))
    names = iter("abcdefghijklmnopqrstuvwxyz")
    la, ls, lb = [[next(names) for _ in x] for x in legs]
    dim = dict(zip(la + ls + lb, fa + sh + fb))
    # the legs of each operand in an order of their own
    axes = [list(rng.permutation(x)) for x in (la + ls, ls + lb, la + lb)]
    tensors = [rng.standard_normal([dim[i] for i in x]) + 1j * rng.standard_normal([dim[i] for i in x]) for x in axes]
    where = {}
    for t, x in enumerate(axes):
        for i, name in enumerate(x):
            where.setdefault(name, []).extend((t, i))
    net = tni.Network([np.ascontiguousarray(t) for t in tensors], np.array(list(where.values()), np.int32).reshape(-1, 4),
                         np.zeros(3, np.int32), ["t"] * 3)
    h = tnsa.tn_build(net)
    plan = tnsa.tn_plan_import(h, [(0, 1), (3, 2)])
    m, e, _ = tnsa.tn_contract(tnsa.tn_ctx_create(0), h, plan, precision)
    spec = ",".join("".join(x) for x in axes) + "->"
    ref, scale = np.einsum(spec, *tensors), np.einsum(spec, *(np.abs(t) for t in tensors))
    # each factor is rounded once, so are the step's outputs and the closing products
    assert abs(m * 2.0 ** e - ref) <= 8 * (2.0 ** -24 if precision == "c64" else 2.0 ** -53 * sum(map(len, axes))) * scale


@pytest.mark.parametrize("length", [32, 33, 70])
def test_warp_program_with_many_leaves(tnsa, length):
    """A closed chain of 2 x 2 matrices: one warp program with more staging pieces than lanes."""
    rng = np.random.default_rng(length)
    mats = [np.linalg.qr(rng.standard_normal((2, 2)) + 1j * rng.standard_normal((2, 2)))[0] for _ in range(length)]
    edges = [(i, 1, (i + 1) % length, 0) for i in range(length)]
    net = tni.Network(mats, np.array(edges, np.int32), np.zeros(length, np.int32), ["t"] * length)
    h = tnsa.tn_build(net)
    steps = [(0, 1)] + [(length + i - 2, i) for i in range(2, length)]
    m, e, _ = tnsa.tn_contract(tnsa.tn_ctx_create(0), h, tnsa.tn_plan_import(h, steps), "c64")
    # unitary factors: every rounding adds at most 2^-24 of the norm of a 2 x 2 block, twice per factor
    assert abs(m * 2.0 ** e - np.trace(np.linalg.multi_dot(mats))) <= 4 * length * 2.0 ** -24


# closing dots on the dataflow path: lengths around the burst and tile sizes, both operands contiguous (with
# and without 16-byte alignment: a first pair of `shift` entries moves the others) or one of them transposed
@pytest.mark.parametrize("dims", [(1,), (7,), (511,), (4097,), (8191,), (8193,), (100001,), (130, 200), (64, 257, 3)])
@pytest.mark.parametrize("shift", [2, 3])
@pytest.mark.parametrize("transposed", [False, True])
@pytest.mark.parametrize("precision", ["c64", "c128"])
def test_long_dots(tnsa, dims, shift, transposed, precision):
    if transposed and len(dims) == 1:
        pytest.skip("one leg has one order")
    rng = np.random.default_rng(len(dims) * 10 + shift)

    def normal(*shape):
        return rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    a, b = normal(*dims), normal(*(dims[::-1] if transposed else dims))
    p, q = normal(shift), normal(shift)
    n = len(dims)
    edges = [(0, 0, 1, 0)] + [(2, i, 3, n - 1 - i if transposed else i) for i in range(n)]
    net = tni.Network([p, q, a, b], np.array(edges, np.int32), np.zeros(4, np.int32), ["t"] * 4)
    h = tnsa.tn_build(net)
    plan = tnsa.tn_plan_import(h, [(2, 3), (0, 1), (4, 5)])
    c = tnsa.tn_ctx_create(0)
    tnsa.tn_ctx_set_local_budget(c, 0)
    m, e, _ = tnsa.tn_contract(c, h, plan, precision)
    bt = b.transpose() if transposed else b
    ref, scale = (a * bt).sum() * (p * q).sum(), np.abs(a * bt).sum() * np.abs(p * q).sum()
    # complex64: leaves, products, sums of 8 products and the two stored dots are rounded (16 roundings at
    # most on the way of a term); complex128: 8 products and then a sum per burst
    eps = 16 * 2.0 ** -24 if precision == "c64" else (64 + math.prod(dims) / 2048) * 2.0 ** -53
    assert abs(m * 2.0 ** e - ref) <= 2 * eps * scale


# steps staged whole through shared memory, alone and as a chain of two: every thread tile, its largest row
# counts, widths and shared indices that are no powers of two, entries past one fetch ahead, and sizes past
# the limits (which run as other steps); factors near the ends of the FP32 range move the scales to A
@pytest.mark.parametrize("shape", [(512, 16, 16), (1024, 8, 8), (2048, 4, 4), (256, 32, 32), (128, 64, 32), (144, 64, 64),
                                   (512, 2, 4), (2048, 1, 4), (300, 5, 7), (100, 20, 33), (511, 17, 3), (2047, 3, 2),
                                   (9, 63, 64), (129, 64, 32), (513, 16, 16), (140, 60, 65), (2, 40, 50)])
@pytest.mark.parametrize("tail", [0, 8])
@pytest.mark.parametrize("magnitude", [1.0, 2.0 ** 100])
def test_staged_step_shapes(tnsa, shape, tail, magnitude):
    M, N, K = shape
    rng = np.random.default_rng(M * 64 + N)

    def normal(*s):
        return rng.standard_normal(s) + 1j * rng.standard_normal(s)
    x, y, b = normal(M, 2) * magnitude, normal(2, K), normal(K, N) / magnitude
    f, d = (normal(N, tail), normal(M, tail)) if tail else (None, normal(M, N))
    tensors = [x, y, b] + ([f] if tail else []) + [d]
    last = len(tensors) - 1
    edges = [(0, 1, 1, 0), (1, 1, 2, 0), (0, 0, last, 0)]
    edges += [(2, 1, 3, 0), (3, 1, 4, 1)] if tail else [(2, 1, 3, 1)]
    net = tni.Network(tensors, np.array(edges, np.int32), np.zeros(len(tensors), np.int32), ["t"] * len(tensors))
    h = tnsa.tn_build(net)
    n = len(tensors)
    plan = tnsa.tn_plan_import(h, [(0, 1)] + [(n + i, 2 + i) for i in range(n - 2)])
    c = tnsa.tn_ctx_create(0)
    out = []
    for chains in (1, 0):
        tnsa.tn_ctx_set_config(c, local_budget=0, rows_chains=chains)
        m, e, _ = tnsa.tn_contract(c, h, plan, "c64")
        out.append(m * 2.0 ** e)
    assert out[0] == out[1]

    def value(*t):
        r = t[0] @ t[1] @ t[2]
        return ((r @ t[3] if tail else r) * t[-1]).sum()
    # one rounding per leaf and stored step, two per term of a sum of K (or N, 2) complex products, 16 in the dot
    eps = (2 * (K + 2 + (N if tail else 0)) + 24) * 2.0 ** -24
    assert abs(out[0] - value(*tensors)) <= eps * value(*(np.abs(t) for t in tensors))


# register-tiled steps: sizes around the tiles (64 x 64, 128 x 32, 16 x 16 with the shared index split, 32 x 32 in
# complex128), both contiguities of each operand, entries so large or small that the scales move to the operands
@pytest.mark.parametrize("shape", [(64, 64, 65), (65, 63, 129), (200, 70, 300), (129, 33, 70), (300, 31, 100), (8, 8, 512),
                                   (17, 5, 300), (64, 16, 256), (15, 16, 1000), (2048, 33, 3), (1024, 4, 65)])
@pytest.mark.parametrize("transposed", [(0, 0), (1, 0), (0, 1)])
@pytest.mark.parametrize("precision,magnitude", [("c64", 1.0), ("c64", 2.0 ** 60), ("c64", 2.0 ** -60), ("c128", 1.0)])
def test_register_tiled_step_shapes(tnsa, shape, transposed, precision, magnitude):
    M, N, K = shape
    rng = np.random.default_rng(M + N + K)

    def normal(*s):
        return (rng.standard_normal(s) + 1j * rng.standard_normal(s)) / math.sqrt(2)
    a, b, c = normal(M, K) * magnitude, normal(K, N), normal(N, M)
    ta, tb = transposed
    edges = [(0, 0 if ta else 1, 1, 1 if tb else 0), (1, 0 if tb else 1, 2, 0), (2, 1, 0, 1 if ta else 0)]
    net = tni.Network([a.T.copy() if ta else a, b.T.copy() if tb else b, c], np.array(edges, np.int32),
                      np.zeros(3, np.int32), ["t"] * 3)
    h = tnsa.tn_build(net)
    ctx = tnsa.tn_ctx_create(0)
    tnsa.tn_ctx_set_config(ctx, local_budget=0)
    m, e, _ = tnsa.tn_contract(ctx, h, tnsa.tn_plan_import(h, [(0, 1), (3, 2)]), precision)
    ref = np.einsum("ij,ji->", a @ b, c)
    scale = np.einsum("ij,ji->", np.abs(a) @ np.abs(b), np.abs(c))
    # two roundings per term of the complex sum over K, the leaves, the stored step and 16 in the closing dot
    assert abs(m * 2.0 ** e - ref) <= (2 * K + 24) * (2.0 ** -24 if precision == "c64" else 2.0 ** -53 * 4) * scale


# chains of `length` staged steps: from four on the ring of three step heads wraps around, past 32 the chain is cut
@pytest.mark.parametrize("length", [3, 4, 5, 9, 40])
@pytest.mark.parametrize("shape", [(512, 4), (512, 16), (256, 32)])
def test_long_chains_of_staged_steps(tnsa, length, shape):
    """Every step of a chain completes its own counter (a wrong one would leave a consumer waiting or let it
    start early): many jobs, statuses, and the bits of the same steps run one by one."""
    M, K = shape
    rng = np.random.default_rng(length * 100 + K)

    def normal(*s):
        return rng.standard_normal(s) + 1j * rng.standard_normal(s)
    nets = []
    for _ in range(4):
        mats = [np.linalg.qr(normal(K, K))[0] for _ in range(length)]
        edges = [(0, 1, 1, 0)] + [(i, 1, i + 1, 0) for i in range(1, length + 2)] + [(length + 2, 1, 0, 0)]
        nets.append(tni.Network([normal(M, 2), normal(2, K)] + mats + [normal(K, M)], np.array(edges, np.int32),
                                np.zeros(length + 3, np.int32), ["t"] * (length + 3)))
    hs = [tnsa.tn_build(n) for n in nets]
    plan = tnsa.tn_plan_import(hs[0], [(0, 1)] + [(length + 3 + i, 2 + i) for i in range(length + 1)])
    assert tnsa.tn_plan_compile_stats(hs[0], plan, "c64", 0)["n_chained"] == length - (length + 31) // 32
    out = []
    for chains in (1, 0):
        c = tnsa.tn_ctx_create(0)
        tnsa.tn_ctx_set_config(c, local_budget=0, rows_chains=chains)
        b = tnsa.tn_batch_create(c, hs * 100, [plan] * 400, "c64")
        tnsa.tn_batch_run(b)
        m, e, st = tnsa.tn_batch_results(b)
        assert (st == 0).all()
        out.append((m, e))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    for i, n in enumerate(nets):
        # a step rounds its B and its output once and sums K complex products: its error is at most 2 (K + 2) 2^-24
        # of |A| |B|, whose norm is at most sqrt(K) times that of A (B is unitary); the dot adds 16 roundings
        t = n.tensors
        bound = (length * 2 * (K + 2) * math.sqrt(K) + 32) * 2.0 ** -24 * math.prod(map(np.linalg.norm, (t[0], t[1], t[-1])))
        got = out[0][0][i::4] * np.exp2(out[0][1][i::4].astype(float))
        assert (np.abs(got - np.trace(np.linalg.multi_dot(t))) <= bound).all()


# staged steps whose B lies behind A in shared memory (it does not fit the scratch area), M K no multiple of 16, an A
# whose exponent is not 0, and a B near the ends of the FP32 range: A is then scaled where it lies
@pytest.mark.parametrize("shape", [(101, 50, 45), (77, 33, 44), (126, 64, 45)])
@pytest.mark.parametrize("magnitude", [1.0, 2.0 ** 100, 2.0 ** -100])
def test_staged_step_scales_only_its_own_operand(tnsa, shape, magnitude):
    M, N, K = shape
    rng = np.random.default_rng(M + N + K)

    def normal(*s):
        return rng.standard_normal(s) + 1j * rng.standard_normal(s)

    def exponent(t):
        return int(np.frexp(max(np.abs(t.real).max(), np.abs(t.imag).max()))[1])
    x, y, b, d = normal(M, 16), normal(16, K), normal(K, N) * magnitude, normal(M, N)
    assert exponent((x * 2.0 ** -exponent(x)) @ (y * 2.0 ** -exponent(y))) != 0
    net = tni.Network([x, y, b, d], np.array([(0, 1, 1, 0), (1, 1, 2, 0), (0, 0, 3, 0), (2, 1, 3, 1)], np.int32),
                      np.zeros(4, np.int32), ["t"] * 4)
    h = tnsa.tn_build(net)
    c = tnsa.tn_ctx_create(0)
    tnsa.tn_ctx_set_config(c, local_budget=0)
    m, e, _ = tnsa.tn_contract(c, h, tnsa.tn_plan_import(h, [(0, 1), (4, 2), (5, 3)]), "c64")
    ref, scale = ((x @ y @ b) * d).sum(), ((np.abs(x) @ np.abs(y) @ np.abs(b)) * np.abs(d)).sum()
    # one rounding per leaf and stored step, two per term of the sums over 16 and K, 16 in the dot
    assert abs(m * 2.0 ** e - ref) <= (2 * (K + 16) + 24) * 2.0 ** -24 * scale


def _one_output_far_below(precision, exps, shape, depth):
    """Leaves a (M x K) and b (K x N) with max-abs exponents `exps`, row 1 of a and column 2 of b 2^-depth lower,
    and a closing tensor that takes the output (1, 2) alone: that output, 2^-(2 depth) of the others, has to keep
    its own relative accuracy.  Also its value over 2^(exps - 2 depth) and the bound of its error."""
    M, N, K = shape
    rng = np.random.default_rng(sum(shape))
    a, b = (rng.uniform(0.5, 1, s) + 1j * rng.uniform(0.5, 1, s) for s in ((M, K), (K, N)))
    ref, terms = a[1] @ b[:, 2], np.abs(a[1]) @ np.abs(b[:, 2])
    a[1] *= 2.0 ** -depth
    b[:, 2] *= 2.0 ** -depth
    d = np.zeros((N, M), np.complex128)
    d[2, 1] = 1.0
    net = tni.Network([a * 2.0 ** exps[0], b * 2.0 ** exps[1], d], np.array([(0, 1, 1, 0), (1, 1, 2, 0), (2, 1, 0, 0)], np.int32),
                      np.zeros(3, np.int32), ["t"] * 3)
    # two roundings per term of the complex sum over K, the leaves, the stored step and 16 in the closing dot
    return net, [(0, 1), (3, 2)], ref, (2 * K + 24) * (2.0 ** -24 if precision == "c64" else 2.0 ** -53 * 4) * terms


def _check_far_below(tnsa, net, steps, ref, bound, precision, exp, budget=0):
    h = tnsa.tn_build(net)
    c = tnsa.tn_ctx_create(0)
    tnsa.tn_ctx_set_config(c, local_budget=budget)
    m, e, _ = tnsa.tn_contract(c, h, tnsa.tn_plan_import(h, steps), precision)
    got = complex(math.ldexp(m.real, int(e) - exp), math.ldexp(m.imag, int(e) - exp))
    assert abs(got - ref) <= bound


# register-tiled steps (64 x 64, 128 x 32, 16 x 16 with a long shared index, 32 x 32 complex128): exponents around
# those up to which the scales are applied to the sums, of one sign and of both
@pytest.mark.parametrize("shape", [(70, 65, 100), (129, 31, 70), (17, 5, 300)])
@pytest.mark.parametrize("precision,exps,depth", [
    ("c64", (0, 0), 33), ("c64", (-39, -38), 33), ("c64", (-20, -20), 50), ("c64", (39, 38), 50), ("c64", (39, -39), 50),
    ("c64", (-39, 12), 50), ("c64", (-40, -40), 33), ("c64", (-60, -60), 33), ("c128", (-119, -118), 400),
    ("c128", (100, -119), 400)])
def test_register_tiled_steps_keep_small_outputs(tnsa, shape, precision, exps, depth):
    net, steps, ref, bound = _one_output_far_below(precision, exps, shape, depth)
    _check_far_below(tnsa, net, steps, ref, bound, precision, sum(exps) - 2 * depth)


# small steps on their own and in programs: exponents of either sign, operands with entries far below the largest
@pytest.mark.parametrize("shape", [(16, 16, 16), (20, 6, 30), (3, 5, 7)])
@pytest.mark.parametrize("exps", [(0, 0), (100, 0), (59, -30), (0, 100), (-59, 40), (-80, 19), (70, 50)])
@pytest.mark.parametrize("budget", [0, -1])
def test_small_steps_keep_small_outputs(tnsa, shape, exps, budget):
    net, steps, ref, bound = _one_output_far_below("c64", exps, shape, 40)
    _check_far_below(tnsa, net, steps, ref, bound, "c64", sum(exps) - 80, budget)


# staged steps whose A comes from a long sum (exponent 12), B with a column 2^-125 below its largest entry
@pytest.mark.parametrize("shape", [(16, 12, 16), (200, 16, 16), (256, 32, 32), (128, 64, 40), (101, 50, 45), (511, 17, 3)])
def test_staged_steps_keep_small_outputs(tnsa, shape):
    M, N, K = shape
    rng = np.random.default_rng(M + N)
    x, y = np.ones((M, 4096), np.complex128), np.ones((4096, 1)) * rng.integers(4, 8, K) / 8 + 0j   # exact sums
    b = rng.uniform(0.5, 1, (K, N)) + 0j
    ref = (x[1] @ y @ b[:, 2]).real
    b[:, 2] *= 2.0 ** -125
    d = np.zeros((M, N), np.complex128)
    d[1, 2] = 1.0
    net = tni.Network([x, y, b, d], np.array([(0, 1, 1, 0), (1, 1, 2, 0), (0, 0, 3, 0), (2, 1, 3, 1)], np.int32),
                      np.zeros(4, np.int32), ["t"] * 4)
    # two roundings per term of the sum over K, the leaves, the stored steps and 16 in the closing dot
    _check_far_below(tnsa, net, [(0, 1), (4, 2), (5, 3)], ref, (2 * K + 24) * 2.0 ** -24 * ref, "c64", -125)


# few outputs with a long shared index, more of them than eight 16 x 16 tiles: 32 x 32 tiles, the index split four ways
@pytest.mark.parametrize("shape", [(64, 64, 256), (33, 33, 257), (128, 32, 300), (63, 65, 1001), (49, 48, 512), (17, 240, 260)])
@pytest.mark.parametrize("transposed", [(0, 0), (1, 0), (0, 1)])
@pytest.mark.parametrize("magnitude", [1.0, 2.0 ** 60, 2.0 ** -30])
def test_long_shared_index_in_wider_tiles(tnsa, shape, transposed, magnitude):
    M, N, K = shape
    rng = np.random.default_rng(M + N + K)

    def normal(*s):
        return (rng.standard_normal(s) + 1j * rng.standard_normal(s)) / math.sqrt(2)
    a, b, c = normal(M, K) * magnitude, normal(K, N), normal(N, M)
    ta, tb = transposed
    edges = [(0, 0 if ta else 1, 1, 1 if tb else 0), (1, 0 if tb else 1, 2, 0), (2, 1, 0, 1 if ta else 0)]
    net = tni.Network([a.T.copy() if ta else a, b.T.copy() if tb else b, c], np.array(edges, np.int32),
                      np.zeros(3, np.int32), ["t"] * 3)
    h = tnsa.tn_build(net)
    ctx = tnsa.tn_ctx_create(0)
    tnsa.tn_ctx_set_config(ctx, local_budget=0)
    m, e, _ = tnsa.tn_contract(ctx, h, tnsa.tn_plan_import(h, [(0, 1), (3, 2)]), "c64")
    ref = np.einsum("ij,ji->", a @ b, c)
    scale = np.einsum("ij,ji->", np.abs(a) @ np.abs(b), np.abs(c))
    # two roundings per term of the complex sum over K, the leaves, the stored step and 16 in the closing dot
    assert abs(m * 2.0 ** e - ref) <= (2 * K + 24) * 2.0 ** -24 * scale
