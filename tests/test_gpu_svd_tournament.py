"""The FP32 tournament of the large sectors on clusters of 16 and of 8 CTAs (the
second where the device has none of 16), called on its own: for sizes around a
block, around its register blocking (384 rows) and with ranks below the columns.
Two Newton-Schulz steps make V orthogonal, as the stages after it need (up to 15
sweeps of n rotations, each off by up to 2^-23 in the same direction, 9e-4 at
n = 513, and 3/4 of the square twice: 1e-12), and the largest overlap that B V is
left with on 8 CTAs, which does the same rotations in another order, is of the
size of that on 16 (a factor of 4)."""
import ctypes as C

import numpy as np
import pytest

from internal_calls import launcher, struct

pytestmark = pytest.mark.gpu


def _rotations(B, rank, csize):
    """V after the tournament and two Newton-Schulz steps; row j: column j."""
    import torch
    ca = len(B)
    nn = ca * ca
    Job, launch = struct("SvdJob"), launcher("launch_jacobi32_stream")
    job = Job(r=ca, c=ca, rows_a=ca, cols_a=ca, j_off=0, b_off=nn, x_off=2 * nn, perm_off=0)
    work = torch.zeros(3 * nn + 8, device="cuda", dtype=torch.float64)
    iwork = torch.zeros(ca + 4, device="cuda", dtype=torch.int32)
    iwork[ca] = rank
    jobs = torch.tensor(np.frombuffer(bytes(job), dtype=np.uint8).copy(), device="cuda")
    order = torch.zeros(1, device="cuda", dtype=torch.int32)
    work[:nn] = torch.eye(ca, device="cuda", dtype=torch.float64).reshape(-1)
    work[nn:2 * nn] = torch.tensor(B.reshape(-1), device="cuda")
    s = launch(C.c_void_p(jobs.data_ptr()), C.c_void_p(order.data_ptr()), 1, ca, csize, C.c_void_p(work.data_ptr()),
               C.c_void_p(iwork.data_ptr()), C.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert s == 0
    torch.cuda.synchronize()
    V = work[:nn].view(ca, ca).cpu().numpy()
    for _ in range(2):
        V = 1.5 * V - 0.5 * (V @ V.T) @ V
    return V


@pytest.mark.parametrize("ca,rank", [(2, 2), (33, 33), (160, 150), (384, 384), (385, 1), (513, 512)])
def test_clusters_of_8_do_as_those_of_16(ca, rank):
    rng = np.random.default_rng(ca)
    B = np.zeros((ca, ca))  # row j: column j
    B[:rank] = rng.standard_normal((rank, ca)) * 10.0 ** -rng.uniform(0, 3, (rank, 1))
    left = []
    for csize in (16, 8):
        V = _rotations(B, rank, csize)
        assert np.max(np.abs(V @ V.T - np.eye(ca))) < 1e-12
        X = (V @ B)[:rank]
        X /= np.linalg.norm(X, axis=1, keepdims=True)
        left.append(np.max(np.abs(X @ X.T - np.eye(rank))))
    assert left[1] < 4 * left[0] + 1e-6, left
