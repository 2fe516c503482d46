"""The check at the end of the SVD refinement, its kernels called on their own.

Not-a-numbers: the library refuses a non-finite wavefunction before the SVD, so
this is the second line of defence.  A sector with a non-finite column, or with an
overlap that is not a number, counts as unfinished (flag behind the job's
permutation not 0: the final Jacobi sweeps it), and a non-finite column is handed
on as it came; a sector of orthonormal columns is finished."""
import ctypes as C
import re

import numpy as np
import pytest

from internal_calls import HEADER, launcher, struct

pytestmark = pytest.mark.gpu

PARTS = re.search(r"enum SvdRefine \{(.*?)\}", HEADER, re.S).group(1).replace(" ", "").split(",")
CA = 80  # two rows of tiles and a ragged third


def _sector():
    """One sector of CA columns, norms 1 .. 0.1: job, arrays, call(part)."""
    import torch
    nn = CA * CA
    Job, refine = struct("SvdJob"), launcher("launch_svd_refine")
    job = Job(r=CA, c=CA, rows_a=CA, cols_a=CA, a_off=0, j_off=nn, b_off=2 * nn, x_off=3 * nn, tau_off=4 * nn,
              w_off=4 * nn + CA, t_off=5 * nn + CA, perm_off=0, sv_off=0)
    work = torch.zeros(8 * nn + CA, device="cuda", dtype=torch.float64)
    iwork = torch.zeros(CA + 4, device="cuda", dtype=torch.int32)
    iwork[CA] = CA  # rank
    sv = torch.zeros(CA, device="cuda", dtype=torch.float64)
    jobs = torch.tensor(np.frombuffer(bytes(job), dtype=np.uint8).copy(), device="cuda")
    order = torch.zeros(1, device="cuda", dtype=torch.int32)
    X = torch.tensor(np.linalg.qr(np.random.default_rng(3).standard_normal((CA, CA)))[0], device="cuda")
    X = X * torch.linspace(1.0, 0.1, CA, device="cuda", dtype=torch.float64)[:, None]  # row j: column j of X
    area = lambda off: work[off:off + nn].view(CA, CA)
    area(job.j_off).copy_(torch.eye(CA))

    def part(name, stage=0):
        s = refine(PARTS.index(name), stage, C.c_void_p(jobs.data_ptr()), C.c_void_p(order.data_ptr()), 1, CA,
                   C.c_void_p(work.data_ptr()), C.c_void_p(iwork.data_ptr()), C.c_void_p(sv.data_ptr()),
                   C.c_void_p(torch.cuda.current_stream().cuda_stream))
        assert s == 0
        torch.cuda.synchronize()

    return job, X, area, iwork, part


@pytest.mark.parametrize("what", ["finite", "column", "overlap"])
def test_not_a_number_is_unfinished(what):
    import torch
    job, X, area, iwork, part = _sector()
    if what == "column":
        X[70, 5] = float("nan")
    area(job.b_off).copy_(X)
    part("REF_SCALE")
    area(job.x_off).copy_(area(job.b_off) @ area(job.b_off).T)
    if what == "overlap":
        area(job.x_off)[70, 3] = float("nan")
    part("REF_CHECK")
    assert (iwork[CA + 3].item() != 0) == (what != "finite")
    if what != "overlap":
        got = area(job.b_off)
        assert torch.equal(torch.isnan(got), torch.isnan(X))
        assert (got - X).abs().nan_to_num().max().item() < 1e-15


@pytest.mark.parametrize("norm2,overlap,finished", [(1.0, 0.9, True), (1.0, 1.1, False), (4.0, 3.9, True), (4.0, 4.1, False),
                                                    (0.25, 0.24, True), (0.25, 0.26, False)])
def test_overlaps_count_against_the_norms(norm2, overlap, finished):
    """The threshold sqrt(columns) 2^-52 is of g / (|x_i| |x_j|), whatever the
    corrections made of the norms."""
    import torch
    job, X, area, iwork, part = _sector()
    area(job.b_off).copy_(X)
    part("REF_SCALE")
    G = norm2 * torch.eye(CA, device="cuda", dtype=torch.float64)
    G[70, 3] = G[3, 70] = overlap * CA**0.5 * 2.0**-52
    area(job.x_off).copy_(G)
    part("REF_CHECK")
    assert (iwork[CA + 3].item() == 0) == finished
