"""GPU parity of the local / global averages (Algorithm 1, Sec. 3.1): the CUDA
kernels, called through the C ABI, must be bit-identical to the oracle's
fixed-order tree on the same inputs."""
import numpy as np
import pytest
import torch

import oracle
from paper_1903_05133_gb300 import hier_avg as ha
from paper_1903_05133_gb300.inputs import replica_matrix

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda(lib):
    assert torch.cuda.is_available(), "GPU tests need CUDA"


def _bits(a: np.ndarray) -> np.ndarray:
    return np.ascontiguousarray(a, dtype=np.float32).view(np.uint32)


def _gpu(w_host: np.ndarray, op, S=None, ld=None, offset=0):
    P, D = w_host.shape
    ld = D if ld is None else ld
    big = torch.full((P, ld + offset + 8), float("nan"), dtype=torch.float32, device="cuda")
    view = big[:, offset:offset + D]
    view.copy_(torch.from_numpy(w_host))
    if op == "local":
        ha.local_average_buffer(view, S)
    elif op == "global":
        ha.global_average_buffer(view)
    else:
        ha.local_global_average_buffer(view, S)
    torch.cuda.synchronize()
    out = big.cpu().numpy()
    # nothing outside the [P, D] window may change
    assert np.all(np.isnan(out[:, :offset])) and np.all(np.isnan(out[:, offset + D:]))
    return out[:, offset:offset + D]


def _oracle(w_host, op, S=None):
    w = w_host.copy()
    if op == "local":
        oracle.local_average(w, S)
    elif op == "global":
        oracle.global_average(w)
    else:
        oracle.local_average(w, S)
        oracle.global_average(w)
    return w


CASES = [(4, 2, 1000), (4, 2, 8), (8, 4, 4099), (6, 3, 1001), (16, 4, 4096), (128, 32, 10000),
         (128, 2, 33333), (16, 16, 777), (5, 5, 64), (7, 1, 100), (12, 4, 4099), (64, 8, 65536),
         (32, 8, 12345), (1, 1, 17), (3, 1, 5), (128, 128, 2048), (24, 6, 3000)]


@pytest.mark.parametrize("P,S,D", CASES)
@pytest.mark.parametrize("op", ["local", "global", "local_global"])
def test_bitexact(P, S, D, op):
    w = replica_matrix(P, D, seed=P * 1000 + S).numpy()
    got = _gpu(w, op, S)
    want = _oracle(w, op, S)
    assert np.array_equal(_bits(got), _bits(want))


@pytest.mark.parametrize("offset,ld_extra", [(1, 3), (0, 5), (2, 0), (4, 60)])
def test_strided_and_misaligned(offset, ld_extra):
    # unaligned base and odd leading dimensions take the scalar path for part or all
    P, S, D = 8, 4, 1037
    w = replica_matrix(P, D, seed=77).numpy()
    for op in ("local", "global", "local_global"):
        got = _gpu(w, op, S, ld=D + ld_extra, offset=offset)
        assert np.array_equal(_bits(got), _bits(_oracle(w, op, S)))


# The generic kernels at the edges of their dispatch: rows of 1 to 4 columns past a quad, a
# CTA or the four-columns-per-thread limit (152 x 2048 columns), aligned rows with a partial
# last quad, unaligned rows; group sizes around 16 (blocks of 16 rows) and 256 (the register
# variants), none of them powers of two, and clusters whose copies end inside a block of the
# global tree.
@pytest.mark.parametrize("P,S,D,offset,ld_extra", [
    (6, 3, 5, 0, 3), (6, 3, 1025, 0, 3), (12, 6, 1023, 1, 0), (15, 5, 1022, 0, 2), (17, 17, 1021, 0, 7),
    (30, 15, 770, 0, 6), (34, 17, 258, 3, 0), (48, 16, 515, 0, 1), (96, 3, 259, 0, 1), (100, 20, 301, 2, 1),
    (250, 25, 130, 0, 2), (255, 51, 67, 0, 0), (256, 64, 37, 1, 0), (300, 100, 33, 0, 3), (514, 257, 9, 0, 0),
    (4100, 4100, 6, 0, 2), (3, 3, 311297, 0, 0), (4, 2, 311299, 1, 0), (6, 2, 155649, 0, 0)])
def test_generic_kernels(P, S, D, offset, ld_extra):
    w = replica_matrix(P, D, seed=P + D).numpy()
    for op in ("local", "global", "local_global"):
        got = _gpu(w, op, S, ld=D + ld_extra, offset=offset)
        assert np.array_equal(_bits(got), _bits(_oracle(w, op, S))), op


# The fused average over many clusters: small ones (a looped counter) and clusters of 16 rows
# and more, under and from 256 and 4096 rows on, the last columns of rows on both sides of the
# four-columns-per-thread limit, aligned and not.  The oracle checks a sample of the columns.
@pytest.mark.parametrize("P,S,D,ld", [
    (24, 3, 40001, 40001), (250, 2, 1003, 1024), (48, 3, 311299, 311300), (255, 17, 1001, 1001),
    (256, 2, 311300, 311300), (300, 3, 311299, 311299), (258, 43, 311299, 311299), (512, 16, 515, 516),
    (1023, 3, 130, 131), (4095, 5, 33, 36), (4096, 2, 130, 130), (5000, 2500, 67, 67)])
def test_local_global_of_many_clusters(P, S, D, ld):
    torch.manual_seed(P + D)
    w = torch.randn(P, ld, device="cuda")[:, :D]
    cols = torch.cat([torch.randint(0, D, (64,), device="cuda"), torch.arange(D - 8, D, device="cuda")])
    src = w[:, cols].cpu().numpy()
    ha.local_global_average_buffer(w, S)
    assert np.array_equal(_bits(w[:, cols].cpu().numpy()), _bits(_oracle(src, "local_global", S)))


# Aligned rows of odd length, group sizes that are powers of two: the columns after the last quad
# are a CTA of their own in the same launch.  One, two and three such columns; rows of less than
# a quad (the generic kernels) and of one; a column's rows split between two threads (up to
# 622592 quads in all groups together) and not.
@pytest.mark.parametrize("P,S,D,ld_extra", [
    (4, 2, 3, 1), (8, 2, 5, 3), (8, 4, 1037, 3), (4, 4, 1022, 2), (128, 32, 515, 1), (32, 2, 131, 1),
    (64, 16, 1025, 3), (8, 2, 622602, 2), (2, 2, 2490375, 1)])
def test_power_of_two_groups_of_odd_rows(P, S, D, ld_extra):
    w = replica_matrix(P, D, seed=P + D).numpy()
    for op in ("local", "global", "local_global"):
        got = _gpu(w, op, S, ld=D + ld_extra)
        assert np.array_equal(_bits(got), _bits(_oracle(w, op, S))), op


def test_edge_values():
    P, S, D = 8, 2, 64
    rng = np.random.default_rng(5)
    w = rng.standard_normal((P, D)).astype(np.float32)
    w[:, 0] = -0.0
    w[::2, 1] = 0.0
    w[:, 2] = np.float32(1e-45) * np.arange(1, P + 1)            # subnormals
    w[:, 3] = np.float32(1e-40)
    w[0, 4] = np.inf
    w[:, 5] = np.float32(3e38)                                     # sums overflow to inf
    w[:, 6] = np.float32([1, 2 ** 24, 1, -2 ** 24, 3, 5, 7, 11])   # order-sensitive
    w[:, 7] = np.float32(1.17549435e-38)                           # smallest normal
    for op in ("local", "global", "local_global"):
        got = _gpu(w, op, S)
        want = _oracle(w, op, S)
        assert np.array_equal(_bits(got), _bits(want)), op


def test_invariants_after_average():
    P, S, D = 16, 4, 5000
    w = replica_matrix(P, D, seed=3).numpy()
    got = _gpu(w, "local", S)
    for g in range(P // S):
        blk = _bits(got[g * S:(g + 1) * S])
        assert np.all(blk == blk[0])
    got = _gpu(w, "local_global", S)
    assert np.all(_bits(got) == _bits(got[0]))


@pytest.mark.parametrize("D", [1_000_000, 64_000_000])
def test_sweep_size_sampled(D):
    # The averaging sweep at its full size (P = 128): every column is independent,
    # so the oracle checks a random sample of columns one by one.
    P = 128
    torch.manual_seed(0)
    w = torch.randn(P, D, device="cuda", dtype=torch.float32)
    cols = torch.randint(0, D, (512,), device="cuda")
    cols = torch.cat([cols, torch.tensor([0, D - 1], device="cuda")])
    for op, S in (("local", 2), ("local", 32), ("local_global", 8), ("global", None)):
        src = w[:, cols].cpu().numpy()
        work = w.clone()
        if op == "local":
            ha.local_average_buffer(work, S)
        elif op == "global":
            ha.global_average_buffer(work)
        else:
            ha.local_global_average_buffer(work, S)
        torch.cuda.synchronize()
        got = work[:, cols].cpu().numpy()
        del work
        assert np.array_equal(_bits(got), _bits(_oracle(src, op, S))), (op, S)
