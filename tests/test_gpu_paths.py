"""GPU kernels at the sizes where their variants change (edges of tiles,
remainders, smallest and largest of a rule's range), against the oracle."""
import numpy as np
import pytest

import oracle
from paper_2405_14060_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
if torch.cuda.is_available():
    from paper_2405_14060_gb300 import tn


def _two_tables(nvars, card, seed):
    """Two factors over the same variables: the last contraction sums them all."""
    rng = np.random.default_rng(seed)
    scope = np.arange(nvars, dtype=np.int32)
    t = [rng.random(card ** nvars) + 1e-3 for _ in range(2)]
    return synth.Model(np.full(nvars, card, np.int32), [scope, scope], t)


# summed spaces: two and eight entries (registers), scanned (27, 511 and one
# label of 100), block sums (512 and 2187 entries, a ragged last block)
@pytest.mark.parametrize("nvars,card", [(1, 2), (3, 2), (3, 3), (1, 100), (9, 2), (7, 3)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_sampling_summed_spaces(nvars, card, prec):
    m = _two_tables(nvars, card, nvars)
    M = tn.Model.from_synth(m)
    n = 100000
    s = M.sample(n, seed=11, prec=prec)
    idx = np.zeros(n, np.int64)
    for v in range(nvars):
        idx = idx * card + s[:, v]
    joint = m.tables[0] * m.tables[1]
    expc = joint / joint.sum() * n
    emp = np.bincount(idx, minlength=len(joint))
    keep = expc >= 5
    chi2 = np.sum((emp[keep] - expc[keep]) ** 2 / expc[keep])
    dof = int(keep.sum()) - 1
    assert chi2 < dof + 6 * np.sqrt(2 * dof)
    for k in (1, 33, 129):      # counter-based: a longer run starts with a shorter one's rows
        np.testing.assert_array_equal(M.sample(k, seed=11, prec=prec), s[:k])


# values of a sample in shared memory with 128, 64 and 32 threads a block, and
# beyond its size in the output rows
@pytest.mark.parametrize("nvars", [7, 900, 2000, 3300])
def test_sampling_many_variables(nvars):
    m = synth.tree_ising(nvars, 5, 0.7)
    M = tn.Model.from_synth(m)
    n = 4001
    s = M.sample(n, seed=3)
    # closed form: the spins of an edge agree with probability e^J / (e^J + e^-J)
    spin = 2 * s.astype(np.int64) - 1
    for (i, j), t in list(zip(m.scopes, m.tables))[:50]:
        want = (t[0] - t[1]) / (t[0] + t[1])
        assert abs(np.mean(spin[:, i] * spin[:, j]) - want) < 6 / np.sqrt(n)
    np.testing.assert_array_equal(M.sample(130, seed=3), s[:130])


@pytest.mark.parametrize("mk", [lambda: synth.chain_model(40, [5, 2, 3, 4] * 10, 3),
                                lambda: synth.bayes_net(60, 4),
                                lambda: synth.grid_ising(5, 6),
                                lambda: _two_tables(4, 5, 9)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_backtrack_levels(mk, prec):
    m = mk()
    M = tn.Model.from_synth(m)
    for method in (0, 1):
        M.set_order(*M.optimize_order(method, 2, 1))
        x, lp = M.map(prec=prec)
        xo, lpo = oracle.ve_map(m)
        np.testing.assert_array_equal(x, xo)
        assert abs(lp - lpo) < (1e-9 if prec == "fp64" else 1e-4)


# micro subtrees: batches whose items share a warp or not (2 to 48 entries an
# item, powers of two and not), summed spaces shared by lanes, cards that give
# tables with and without power-of-two sizes, tensors too large to be staged
@pytest.mark.parametrize("batch", [1, 3, 32, 100])
@pytest.mark.parametrize("mk", [lambda: synth.random_markov(12, 14, 3, 2, cards=(2, 3)),
                                lambda: synth.bayes_net(30, 8, cards=(2, 4)),
                                lambda: synth.chain_model(12, [37] * 12, 4),
                                lambda: synth.grid_ising(6, 9)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_micro_subtrees(mk, batch, prec):
    m = mk()
    ev = synth.evidence_batch(m, batch, 0.2, 17)
    M = tn.Model.from_synth(m)
    lz, mg = M.mar(ev, prec=prec)
    tol = 1e-10 if prec == "fp64" else 1e-4
    for b in sorted({0, batch // 2, batch - 1}):
        lo, mo = oracle.ve_mar(m, ev[b])
        # the stated log Z (relative) and marginal tolerances of each precision
        assert abs(lz[b] - lo) <= tol * max(1.0, abs(lo))
        assert np.max(np.abs(mg[b] - np.concatenate(mo))) <= tol


# direct form of the FP64 batched GEMM: one row or column, rows and columns
# around the strip sizes (32 rows, 1 / 2 / 4 columns), lanes sharing a summed
# space, splits over blocks with a ragged last one, either side fastest in the
# output, a group label, GEMM-sized groups
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (1, 5, 9), (3, 2, 4097), (20, 30, 9000), (31, 4, 8),
                                   (33, 7, 17), (64, 65, 66), (130, 3, 700), (257, 129, 64)])
@pytest.mark.parametrize("spec", ["mk,kn->mn", "km,nk->nm", "gmk,kgn->mgn"])
def test_direct_fp64(m, n, k, spec):
    (a, b), c = spec.split("->")[0].split(","), spec.split("->")[1]
    letters = "gkmn"
    size = dict(g=3, k=k, m=m, n=n)
    rng = np.random.default_rng(m * n + k)
    A = rng.random([size[l] for l in a])
    B = rng.random([size[l] for l in b])
    ref = np.einsum(spec, A, B)
    C = torch.full([size[l] for l in c], float("nan"), dtype=torch.float64, device="cuda")
    tn.contract_dev([size[l] for l in letters], [letters.index(l) for l in a], torch.tensor(A).cuda(),
                    [letters.index(l) for l in b], torch.tensor(B).cuda(),
                    [letters.index(l) for l in c], C)
    # positive terms: every order of summation is within k ulp
    np.testing.assert_allclose(C.cpu().numpy(), ref, rtol=k * 2.3e-16 + 1e-15, atol=0)


# FP32 batched GEMM: rows and columns around every tile (8, 16, 32, 64, 128
# columns), last K steps of at most half (8, 24, 37) and more (13, 16), copies of
# 4, 2 and 1 floats, summed fastest in one, both or no operand, quads / pairs /
# single floats of C side by side, a group label inside C's sectors
@pytest.mark.parametrize("m,n,k", [(1, 1, 3), (100, 8, 24), (300, 7, 37), (2048, 8, 13), (257, 16, 8),
                                   (640, 33, 16), (130, 66, 100), (3000, 130, 7), (16384, 128, 20)])
@pytest.mark.parametrize("spec", ["mk,kn->mn", "km,kn->nm", "mk,nk->nm", "gkm,kgn->gnm",
                                  "mgk,kgn->nmg", "kmg,gnk->mng", "mhk,kn->nmh"])
def test_bgemm_fp32_tiles(m, n, k, spec):
    (a, b), c = spec.split("->")[0].split(","), spec.split("->")[1]
    letters = "ghkmn"
    size = dict(g=2, h=2, k=k, m=m, n=n)
    rng = np.random.default_rng(m + n * k)
    A = rng.random([size[l] for l in a]).astype(np.float32)
    B = rng.random([size[l] for l in b]).astype(np.float32)
    ref = np.einsum(spec, A.astype(np.float64), B.astype(np.float64))
    C = torch.full([size[l] for l in c], float("nan"), dtype=torch.float32, device="cuda")
    tn.contract_dev([size[l] for l in letters], [letters.index(l) for l in a], torch.tensor(A).cuda(),
                    [letters.index(l) for l in b], torch.tensor(B).cuda(),
                    [letters.index(l) for l in c], C, prec="fp32")
    # positive terms: every order of summation is within k + 1 roundings
    np.testing.assert_allclose(C.cpu().numpy(), ref, rtol=(k + 1) * 6e-8, atol=0)


# FP32 GEMM: one tile of every shape and several, ragged rows, columns and
# summed space, operands already in GEMM form, split long summed spaces
@pytest.mark.parametrize("m,n,k", [(64, 64, 64), (65, 70, 77), (193, 129, 96), (1000, 900, 130),
                                   (2500, 2000, 64), (100, 130, 3000)])
@pytest.mark.parametrize("spec", ["mk,nk->mn", "km,kn->nm", "gmk,gkn->gmn"])
def test_gemm_fp32_tiles(m, n, k, spec):
    (a, b), c = spec.split("->")[0].split(","), spec.split("->")[1]
    letters = "gkmn"
    size = dict(g=2, k=k, m=m, n=n)
    rng = np.random.default_rng(m + n * k)
    A = rng.random([size[l] for l in a]).astype(np.float32)
    B = rng.random([size[l] for l in b]).astype(np.float32)
    ref = torch.einsum(spec, torch.tensor(A).cuda().double(), torch.tensor(B).cuda().double())
    C = torch.full([size[l] for l in c], float("nan"), dtype=torch.float32, device="cuda")
    tn.contract_dev([size[l] for l in letters], [letters.index(l) for l in a], torch.tensor(A).cuda(),
                    [letters.index(l) for l in b], torch.tensor(B).cuda(),
                    [letters.index(l) for l in c], C, prec="fp32")
    err = ((C.double() - ref).abs() / ref).max().item()
    assert err <= (k + 1) * 6e-8


# tensor-core GEMM: rows and columns around its 128 x 256 (long summed space:
# 256 x 256) tiles and the 32-column chunks of the epilogue, row lengths that
# allow 16-byte stores or not, short (persistent) and long summed spaces
@pytest.mark.parametrize("m,n,k", [(64, 64, 64), (127, 257, 100), (129, 290, 64), (300, 770, 96),
                                   (1000, 260, 72), (200, 300, 2300), (520, 515, 4500)])
@pytest.mark.parametrize("prec", ["tf32", "bf16"])
@pytest.mark.parametrize("spec", ["mk,nk->mn", "gmk,gkn->gmn"])
def test_tc_gemm_edges(m, n, k, prec, spec):
    (a, b), c = spec.split("->")[0].split(","), spec.split("->")[1]
    letters = "gkmn"
    size = dict(g=2, k=k, m=m, n=n)
    rng = np.random.default_rng(m + n * k)
    A = torch.tensor(rng.random([size[l] for l in a]), dtype=torch.float32, device="cuda")
    B = torch.tensor(rng.random([size[l] for l in b]), dtype=torch.float32, device="cuda")
    ref = torch.einsum(spec, A.double(), B.double())
    C = torch.full([size[l] for l in c], float("nan"), dtype=torch.float32, device="cuda")
    tn.contract_dev([size[l] for l in letters], [letters.index(l) for l in a], A,
                    [letters.index(l) for l in b], B, [letters.index(l) for l in c], C, prec=prec)
    # two roundings of each product's inputs (2^-11 TF32 truncated to 2^-10, 2^-9 BF16)
    err = ((C.double() - ref).abs() / ref).max().item()
    assert err <= (2 * 2.0 ** -10 if prec == "tf32" else 2 * 2.0 ** -8)


# domains of one value in the backtrack (no record maximises them): inside larger
# factors, alone, eliminated before and after their neighbours, observed and
# queried; the last model's records do not fit shared memory
def _size1_model(card, scopes, seed):
    rng = np.random.default_rng(seed)
    card = np.array(card, np.int32)
    return synth.Model(card, [np.array(s, np.int32) for s in scopes],
                       [rng.random(int(np.prod(card[s]))) + 0.1 for s in scopes])


SIZE1 = [([1, 2], [[0, 1], [1]]),
         ([1, 2, 1, 3], [[0, 1], [1, 2, 3], [3, 0], [2]]),
         ([2, 1, 1, 4, 1], [[1, 0, 2, 3], [3, 1], [0, 2], [2, 1], [4]]),
         ([1, 1], [[0, 1]])]


@pytest.mark.parametrize("card,scopes", SIZE1)
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_backtrack_size1_domains(card, scopes, prec):
    m = _size1_model(card, scopes, len(card))
    M = tn.Model.from_synth(m)
    tol = 1e-9 if prec == "fp64" else 1e-4
    ev = np.full(m.nvars, -1, np.int32)
    for observed in ([], [card.index(1)]):
        ev[observed] = 0
        xb, lb = oracle.brute_map(m, ev)
        for method in range(4):
            M.set_order(*M.optimize_order(method, 2, 1))
            x, lp = M.map(ev, prec=prec)
            np.testing.assert_array_equal(x, xb)
            assert abs(lp - lb) < tol
    if m.nvars < 3:
        return
    for query in ([0, 3], [1, 2], [0, 1, 2], [3, 2]):
        xb, lb = oracle.brute_mmap(m, query)
        x, lp = M.mmap(query, prec=prec)
        np.testing.assert_array_equal(x, xb)
        assert abs(lp - lb) < tol


def test_backtrack_size1_domains_large():
    m = synth.chain_model(5000, [2, 1, 3, 2] * 1250, 7)
    x, lp = tn.Model.from_synth(m).map()
    best, back = np.log(m.tables[0]), []     # Viterbi along the chain
    for one, s, t in zip(m.tables[1:], m.scopes[m.nvars:], m.tables[m.nvars:]):
        w = best[:, None] + np.log(t.reshape(m.card[s])) + np.log(one)
        back.append(w.argmax(0))
        best = w.max(0)
    xo = [int(best.argmax())]
    for b in reversed(back):
        xo.append(int(b[xo[-1]]))
    np.testing.assert_array_equal(x, xo[::-1])
    assert abs(lp - best.max()) < 1e-9 * abs(best.max())


# tables with negative zeros are those with zeros: draws of up to 2, up to 8 and
# more entries
@pytest.mark.parametrize("card", [2, 3, 8, 9, 120])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_negative_zero_sampling(card, prec):
    t = np.linspace(1.0, 2.0, card)
    t[0] = t[card // 2 + 1:] = -0.0
    M = tn.Model.from_arrays([card], [[0]], [t])
    s = M.sample(20000, seed=5, prec=prec)[:, 0].astype(np.int64)
    pos = tn.Model.from_arrays([card], [[0]], [np.abs(t)])
    np.testing.assert_array_equal(s, pos.sample(20000, seed=5, prec=prec)[:, 0])
    emp = np.bincount(s, minlength=card) / 20000
    assert np.all(np.abs(emp - np.abs(t) / t.sum()) < 5 * np.sqrt(0.25 / 20000))


# scratch kept between single contractions stays within the stated bound (1.3 GiB
# of operand workspaces here)
def test_scratch_kept_is_bounded():
    for n in (128, 13312):       # (the first loads the kernels)
        A, B, C = (torch.zeros(n, n, device="cuda") for _ in range(3))
        torch.cuda.empty_cache()
        free = torch.cuda.mem_get_info()[0]
        tn.contract_dev([n, n, n], [2, 0], A, [2, 1], B, [0, 1], C, prec="tf32")
    assert free - torch.cuda.mem_get_info()[0] <= 1 << 30


# the memory that single contractions leave with the library serves other
# allocations of the process: a model whose tables would not fit beside it (153 MB
# of tables, 134 MB free, 472 MB kept)
def test_scratch_kept_is_given_back_to_models():
    n = 7680
    A, B, C = (torch.zeros(n, n, device="cuda") for _ in range(3))
    rng = np.random.default_rng(0)
    size = [3] * 14 + [2, 2]
    m = synth.Model(np.array(size, np.int32), [np.arange(16, dtype=np.int32)],
                    [rng.random(int(np.prod(size)))])
    M = tn.Model.from_synth(m)
    small = tn.Model.from_synth(synth.grid_ising(3, 1))
    small.pr(prec="fp32")        # the kernels are loaded
    tn.contract_dev([n, n, n], [2, 0], A, [2, 1], B, [0, 1], C, prec="tf32")
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    fill = torch.empty(free - (128 << 20), dtype=torch.uint8, device="cuda")
    try:
        lz = M.pr(prec="fp32")[0]
    finally:
        del fill
        torch.cuda.empty_cache()
    want = np.log(m.tables[0].sum())
    assert abs(lz - want) <= 1e-4 * abs(want)


# operands of more than 2^31 entries with groups too small for a GEMM: rows at both
# ends, summed fastest and not
@pytest.mark.parametrize("spec", ["mk,kn->mn", "km,kn->nm"])
def test_skinny_beyond_32bit_offsets(spec):
    size = dict(k=136, m=(1 << 24) + 3, n=3)
    (a, b), c = spec.split("->")[0].split(","), spec.split("->")[1]
    letters = "kmn"
    gen = torch.Generator(device="cuda").manual_seed(4)
    A, B = (torch.rand([size[l] for l in s], generator=gen, device="cuda") for s in (a, b))
    C = torch.full([size[l] for l in c], float("nan"), device="cuda")
    tn.contract_dev([size[l] for l in letters], [letters.index(l) for l in a], A,
                    [letters.index(l) for l in b], B, [letters.index(l) for l in c], C, prec="fp32")
    assert A.numel() > 1 << 31
    for first in (0, size["m"] // 2, size["m"] - 5000):
        x, y = A.narrow(a.index("m"), first, 5000), C.narrow(c.index("m"), first, 5000)
        ref = torch.einsum(spec, x.double(), B.double())
        # positive terms: every order of summation is within k + 1 roundings
        assert ((y.double() - ref).abs() / ref).max().item() <= (size["k"] + 1) * 6e-8
    del A, B, C, x, y
    torch.cuda.empty_cache()


def _contract(spec, size, A, B, C, prec):
    (a, b), c = spec.split("->")[0].split(","), spec.split("->")[1]
    letters = sorted(size)
    tn.contract_dev([size[l] for l in letters], [letters.index(l) for l in a], A,
                    [letters.index(l) for l in b], B, [letters.index(l) for l in c], C, prec=prec)


# 256 x 256 tiles (more than 64 summed slabs, and half the rounds of 128 x 256
# tiles): a last row tile with rows in its first half only and in both, a ragged
# last 32-column chunk, row lengths with and without 16-byte stores, a K tail.
# Whole numbers up to 3: products, and sums below 2^24, are exact
@pytest.mark.parametrize("prec,k", [("tf32", 2100), ("bf16", 4150)])
@pytest.mark.parametrize("m,n,g", [(3172, 2317, 1), (3272, 2348, 1), (3172, 1101, 2)])
def test_tc_gemm_wide_tiles(prec, k, m, n, g):
    spec = "mk,nk->mn" if g == 1 else "gmk,gkn->gmn"
    (a, b), c = spec.split("->")[0].split(","), spec.split("->")[1]
    size = dict(k=k, m=m, n=n) if g == 1 else dict(g=g, k=k, m=m, n=n)
    gen = torch.Generator(device="cuda").manual_seed(m + n)
    A, B = (torch.randint(0, 4, [size[l] for l in s], generator=gen, device="cuda").float()
            for s in (a, b))
    C = torch.full([size[l] for l in c], float("nan"), device="cuda")
    _contract(spec, size, A, B, C, prec)
    assert torch.equal(C.double(), torch.einsum(spec, A.double(), B.double()))


# operands and results that start off 16-byte boundaries (views into a buffer):
# copies and stores fall back to the widest their addresses allow
@pytest.mark.parametrize("oa,ob,oc", [(1, 0, 0), (0, 1, 0), (0, 0, 1), (2, 2, 2), (3, 1, 2)])
@pytest.mark.parametrize("spec,size", [
    ("mk,nk->mn", dict(k=96, m=400, n=260)),            # GEMM form, in place when aligned
    ("km,kn->nm", dict(k=96, m=400, n=260)),            # both operands and the result reordered
    ("gmk,gkn->gmn", dict(g=2, k=72, m=130, n=1100)),
    ("km,kn->nm", dict(k=24, m=2048, n=40)),            # batched GEMM: copies and stores of quads
    ("mgk,kgn->ngm", dict(g=4, k=20, m=1000, n=64)),
    ("mk,kn->mn", dict(k=12, m=3000, n=72))])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "tf32", "bf16"])
def test_contract_unaligned_pointers(spec, size, oa, ob, oc, prec):
    (a, b), c = spec.split("->")[0].split(","), spec.split("->")[1]
    dt = torch.float64 if prec == "fp64" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(7)

    def view(s, off):
        shape = [size[l] for l in s]
        n = int(np.prod(shape))
        return torch.randint(0, 4, [n + off], generator=gen, device="cuda").to(dt)[off:].view(shape)
    A, B, C = view(a, oa), view(b, ob), view(c, oc)
    _contract(spec, size, A, B, C, prec)
    # whole numbers: exact in every precision and order
    assert torch.equal(C.double(), torch.einsum(spec, A.double(), B.double()))


# FP64 GEMM form past the direct kernel's limits: 2^26 table entries (operands in
# place) and 2^31 entries (prepared)
@pytest.mark.parametrize("m", [(1 << 25) - 64, (1 << 25) + 3])
def test_fp64_gemm_past_direct_limits(m):
    k = n = 64
    gen = torch.Generator(device="cuda").manual_seed(2)
    A, B = (torch.rand(s, generator=gen, device="cuda", dtype=torch.float64)
            for s in ((m, k), (n, k)))
    C = torch.full((m, n), float("nan"), dtype=torch.float64, device="cuda")
    _contract("mk,nk->mn", dict(k=k, m=m, n=n), A, B, C, "fp64")
    for first in (0, m // 2, m - 5000):
        ref = A[first:first + 5000] @ B.T
        err = ((C[first:first + 5000] - ref).abs() / ref).max().item()
        assert err <= k * 2.3e-16 + 1e-15      # positive terms, as above
    del A, B, C, ref
    torch.cuda.empty_cache()
