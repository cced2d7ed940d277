"""Block substitutions at the edges of their variants: record sizes, slices and
groups that are full, partial or empty, rows longer than the records, wide and
one-row wavefronts, vectors in shared and in global memory.

The handle is built from random triangular factors (no coupling, no
correction), so one application is U^-1 L^-1 r per block, compared with plain
FP64 substitutions.  The off-diagonal row sums are at most 1/2 and the
diagonals in [1, 2]: each triangular inverse has infinity norm at most 2, a row of
m entries is summed with a relative error of at most (m + 3) eps, and so two
solves stay within 8 (m + 3) eps of the largest component; with m <= 40 that
is 4e-14 in FP64 and 2.1e-5 in FP32 (FP32 factors and right-hand side: 4 eps
more).
"""
import numpy as np
import pytest
import scipy.sparse as sp

import gemslr_inputs as gi
from oracle.ilu import lu_solve

pytestmark = pytest.mark.gpu

# name: (rows of every block, most entries per row, band, chain: every row needs the one before)
CASES = {
    "one_row": ([1, 2, 3], 2, 4, False),
    "two_entries": ([33, 257, 130], 2, 60, False),
    "six_entries": ([31, 200, 700], 6, 90, False),
    "ten_entries": ([64, 1000, 5000], 10, 300, False),
    "near_ten": ([97, 600], 10, 12, True),            # many entries from the slice just before
    "sixteen_entries": ([500, 129], 16, 400, False),
    "seventeen_entries": ([500, 40], 17, 100, False),
    "forty_entries": ([400, 350], 40, 200, False),
    "chain": ([300, 45], 3, 5, True),                 # one row per wavefront
    "long_chain": ([300, 45], 24, 40, True),          # the same with rows longer than a record
    "no_lower": ([200, 70], 0, 50, False),
    "wide": ([6000, 5000], 3, 6000, False),           # wavefronts of hundreds of rows
    "global_vector": ([46000, 300], 2, 9000, False),  # beyond shared memory in every precision
}


def _triangles(rng, n, most, band, chain, cplx):
    """Strictly lower L and upper U (diagonal included) with the stated patterns."""
    val = (lambda k: rng.uniform(-1, 1, k) + 1j * rng.uniform(-1, 1, k)) if cplx else (lambda k: rng.uniform(-1, 1, k))
    out = []
    for up in (False, True):
        ptr, ind, dat = [0], [], []
        for i in range(n):
            room = min(band, n - 1 - i if up else i)
            k = min(int(rng.integers(0, most + 1)), room)
            off = set(rng.choice(room, size=k, replace=False) + 1) if k else set()
            if chain and room and most:
                off = set(list(off)[: most - 1]) | {1}
            cols = sorted(i + o if up else i - o for o in off)
            v = val(len(cols))
            v = v * (0.5 / max(np.abs(v).sum(), 0.5)) if len(cols) else v
            if up:
                d = rng.uniform(1, 2)
                cols, v = [i] + cols, np.concatenate([[d], v * d])
            ind += cols
            dat.append(v)
            ptr.append(len(ind))
        dat = np.concatenate(dat) if ind else np.zeros(0)
        out.append(sp.csr_matrix((dat, np.array(ind, dtype=np.int32), ptr), shape=(n, n)))
    return out


def _system(name, cplx):
    """(random generator, blocks, sizes, matrix, partition, factors) of one case."""
    sizes, most, band, chain = CASES[name]
    rng = np.random.default_rng(len(name) + most)
    blocks = [_triangles(rng, n, most, band, chain, cplx) for n in sizes]
    d, tail = sum(sizes), 5
    n = d + tail
    eye = sp.identity(tail, format="csr", dtype=complex if cplx else float)
    zero = sp.csr_matrix((tail, tail), dtype=complex if cplx else float)
    fac = dict(levels=[dict(s=0, e=d, L=sp.block_diag([b[0] for b in blocks], format="csr"),
                            U=sp.block_diag([b[1] for b in blocks], format="csr"),
                            E=sp.csr_matrix((tail, d)), F=sp.csr_matrix((d, tail)),
                            W=np.zeros((tail, 0)), H=np.zeros((0, 0)))], last=dict(L=zero, U=eye))
    A = gi.CSR(n, np.arange(n + 1), np.arange(n), np.ones(n))
    part = dict(perm=np.arange(n, dtype=np.int32), level_ptr=np.array([0, d, n], dtype=np.int64),
                nblk=np.array([len(sizes), 1], dtype=np.int32),
                block_ptr=np.concatenate([np.cumsum([0] + sizes), [0, tail]]).astype(np.int64))
    return rng, blocks, sizes, A, part, fac


def _solved(blocks, sizes, r):
    ref = r.copy()
    o = 0
    for (L, U), m in zip(blocks, sizes):
        ref[o:o + m] = lu_solve(L, U, r[o:o + m])
        o += m
    return ref


@pytest.mark.parametrize("kind", ["fp64", "mixed", "complex"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_substitutions_against_plain_solves(name, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_03224_gb300 import Gemslr
    cplx = kind == "complex"
    rng, blocks, sizes, A, part, fac = _system(name, cplx)
    G = Gemslr.from_factors(A, part, fac, precision="mixed" if kind == "mixed" else "fp64")
    r = rng.uniform(-1, 1, A.n) + (1j * rng.uniform(-1, 1, A.n) if cplx else 0)
    z = G.apply(torch.from_numpy(r).cuda()).cpu().numpy()
    ref = _solved(blocks, sizes, r)
    tol = 3e-5 if kind == "mixed" else 1e-13
    assert np.max(np.abs(z - ref)) <= tol * np.max(np.abs(ref)), np.max(np.abs(z - ref))


# The batched substitutions (FP32): one right-hand side, a partial group and a full
# one; blocks of one row up to several thousand; systems whose rows are too long
# for the stored records.
@pytest.mark.parametrize("nrhs", [1, 5, 8])
@pytest.mark.parametrize("name", sorted(set(CASES) - {"global_vector"}))
def test_batched_substitutions_against_plain_solves(name, nrhs):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_03224_gb300 import GemslrBatch
    sy = [_system(name, False), _system("two_entries", False)]
    B = GemslrBatch.from_factors([s[3] for s in sy], [s[4] for s in sy], [s[5] for s in sy])
    rng = np.random.default_rng(nrhs)
    r = [rng.uniform(-1, 1, (nrhs, s[3].n)) for s in sy]
    z = B.apply(torch.from_numpy(np.concatenate([a.ravel() for a in r])).cuda(), nrhs).cpu().numpy()
    o = 0
    for (_, blocks, sizes, A, _, _), rs in zip(sy, r):
        for q in range(nrhs):
            got, ref = z[o:o + A.n], _solved(blocks, sizes, rs[q])
            o += A.n
            assert np.max(np.abs(got - ref)) <= 3e-5 * np.max(np.abs(ref)), (q, np.max(np.abs(got - ref)))


@pytest.mark.parametrize("name", ["chain", "long_chain", "forty_entries"])
def test_partial_slices_give_the_same_bits_every_time(name):
    """A slice of fewer rows than lanes: the lanes without a row of their own must
    not touch x.  Such a lane storing late shows in some applications only."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_03224_gb300 import Gemslr
    rng, blocks, sizes, A, part, fac = _system(name, False)
    G = Gemslr.from_factors(A, part, fac, precision="mixed")
    r = rng.uniform(-1, 1, A.n)
    rd = torch.from_numpy(r).cuda()
    z = G.apply(rd)
    for _ in range(100):
        assert torch.equal(G.apply(rd), z)
    ref = _solved(blocks, sizes, r)
    assert np.max(np.abs(z.cpu().numpy() - ref)) <= 3e-5 * np.max(np.abs(ref))


# Batched levels that are not streamed (a block beyond shared memory even for four
# right-hand sides, with and without rows longer than a record): the right-hand sides
# split over CTAs while these run in one wave, else vectors in global memory.
CASES.update(large_block=([13000, 4000], 7, 900, False), large_block_long_rows=([13000, 4000], 20, 60, False))


@pytest.mark.parametrize("nsys,per_cta", [(3, 2), (24, 0)])
@pytest.mark.parametrize("name", ["large_block", "large_block_long_rows"])
def test_batched_large_blocks_against_plain_solves(name, nsys, per_cta):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_03224_gb300 import GemslrBatch
    rng, blocks, sizes, A, part, fac = _system(name, False)
    B = GemslrBatch.from_factors([A] * nsys, [part] * nsys, [fac] * nsys)
    assert B.stats()["rhs_per_cta"] == per_cta
    r = rng.uniform(-1, 1, (nsys, 8, A.n))
    z = B.apply(torch.from_numpy(r.ravel()).cuda(), 8).cpu().numpy().reshape(r.shape)
    for s, q in ((0, 0), (0, 7), (1, 3), (nsys - 1, 0), (nsys - 1, 7)):
        ref = _solved(blocks, sizes, r[s, q])
        assert np.max(np.abs(z[s, q] - ref)) <= 3e-5 * np.max(np.abs(ref)), (s, q)


# One row longer than a record must not change a whole level's schedule.  The variant
# for such levels adds a test to the work on a slice, and for the slice of that row
# one more read and gather (about 60 of 200 cycles): half as long again is the bound,
# where one warp walking the level alone took two to three times as long.
def test_one_long_row_costs_little():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_03224_gb300 import Gemslr
    CASES["long_row"] = ([3000, 3000], 16, 300, False)
    _, blocks, sizes, A, part, fac = _system("long_row", False)
    times = []
    for longer in (False, True):
        if longer:
            L = fac["levels"][0]["L"].tolil()
            free = sorted(set(range(2000, 2990)) - set(L.rows[2990]))
            for c in free[:: len(free) // 17][: 17 - len(L.rows[2990])]:
                L[2990, c] = 1e-3
            fac["levels"][0]["L"] = L.tocsr()
            assert np.diff(fac["levels"][0]["L"].indptr).max() == 17
        G = Gemslr.from_factors(A, part, fac, precision="mixed")
        r = torch.rand(A.n, dtype=torch.float64, device="cuda")
        best = float("inf")
        for _ in range(8):
            start, end = torch.cuda.Event(True), torch.cuda.Event(True)
            start.record()
            for _ in range(20):
                G.apply(r)
            end.record()
            end.synchronize()
            best = min(best, start.elapsed_time(end))
        times.append(best)
    assert times[1] <= 1.5 * times[0], times


# Rests so long that few rows, or one, fill a group's item.  The bound of the module's
# note for m = 300: 8 (m + 3) eps = 1.45e-4.
@pytest.mark.parametrize("rows,chain", [(900, False), (900, True)])
def test_rows_of_hundreds_of_entries(rows, chain):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_03224_gb300 import Gemslr
    CASES["hundreds"] = ([rows, 350], 300, 800, chain)
    rng, blocks, sizes, A, part, fac = _system("hundreds", False)
    G = Gemslr.from_factors(A, part, fac, precision="mixed")
    r = rng.uniform(-1, 1, A.n)
    z = G.apply(torch.from_numpy(r).cuda()).cpu().numpy()
    ref = _solved(blocks, sizes, r)
    assert np.max(np.abs(z - ref)) <= 1.6e-4 * np.max(np.abs(ref)), np.max(np.abs(z - ref))


# Streamed batched levels whose blocks hold four right-hand sides at a time, beside
# blocks that hold all eight.  The levels that are not streamed would take four here
# only in one wave (152 CTAs), and these blocks are more than that: so four is the
# streamed split.
@pytest.mark.parametrize("nrhs", [1, 5, 8])
@pytest.mark.parametrize("most", [3, 10, 16])
def test_batched_streams_of_four_right_hand_sides(most, nrhs):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_03224_gb300 import GemslrBatch
    CASES["four"] = ([9000, 8500, 300], most, 500, False)
    _, blocks, sizes, A, part, fac = _system("four", False)
    nsys = 40
    B = GemslrBatch.from_factors([A] * nsys, [part] * nsys, [fac] * nsys)
    assert B.stats()["rhs_per_cta"] == 4
    rng = np.random.default_rng(nrhs)
    r = rng.uniform(-1, 1, (nsys, nrhs, A.n))
    z = B.apply(torch.from_numpy(r.ravel()).cuda(), nrhs).cpu().numpy().reshape(r.shape)
    for s, q in {(0, 0), (17, nrhs // 2), (nsys - 1, nrhs - 1)}:
        ref = _solved(blocks, sizes, r[s, q])
        assert np.max(np.abs(z[s, q] - ref)) <= 3e-5 * np.max(np.abs(ref)), (s, q)


# More blocks than SMs (152): CTAs share an SM, in FP32 with the four walking warps
# only; every record size, and blocks of one row among them.
@pytest.mark.parametrize("kind", ["fp64", "mixed", "complex"])
@pytest.mark.parametrize("most", [1, 6, 10, 16, 20])
def test_more_blocks_than_sms_against_plain_solves(most, kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_03224_gb300 import Gemslr
    cplx = kind == "complex"
    CASES["many"] = ([61, 1, 40, 90] * 80, most, 30, False)
    rng, blocks, sizes, A, part, fac = _system("many", cplx)
    G = Gemslr.from_factors(A, part, fac, precision="mixed" if kind == "mixed" else "fp64")
    r = rng.uniform(-1, 1, A.n) + (1j * rng.uniform(-1, 1, A.n) if cplx else 0)
    z = G.apply(torch.from_numpy(r).cuda()).cpu().numpy()
    ref = _solved(blocks, sizes, r)
    tol = 3e-5 if kind == "mixed" else 1e-13
    assert np.max(np.abs(z - ref)) <= tol * np.max(np.abs(ref)), np.max(np.abs(z - ref))
