"""The C-ABI library loads (no GPU needed) and exports every symbol that
include/lsq.h declares; host-only entry points answer without a device."""
import ctypes as C
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def liblsq():
    from paper_2603_16644_gb300 import _build

    path = _build.build()
    return C.CDLL(path)


def declared_symbols():
    txt = open(os.path.join(ROOT, "include", "lsq.h")).read()
    txt = re.sub(r"/\*.*?\*/", "", txt, flags=re.S)
    return sorted(set(re.findall(r"\b(lsq_[a-z0-9_]+)\s*\(", txt)))


def test_header_declares_the_boundary():
    syms = declared_symbols()
    for need in ["lsq_sketch", "lsq_precond_qr", "lsq_condest", "lsq_pne_solve", "lsq_hpne_solve",
                 "lsq_workspace_size", "lsq_trsm_gram", "lsq_factor_solve", "lsq_pne_solve_host"]:
        assert need in syms


def test_every_declared_symbol_is_exported(liblsq):
    missing = [s for s in declared_symbols() if not hasattr(liblsq, s)]
    assert not missing, missing


def test_host_only_calls(liblsq):
    liblsq.lsq_precision_from_kappa0.restype = C.c_int32
    liblsq.lsq_precision_from_kappa0.argtypes = [C.c_double]
    f = liblsq.lsq_precision_from_kappa0
    assert [f(1.0), f(2.5), f(3.5), f(6.0), f(8.0), f(9.0), f(float("inf")), f(float("nan"))] == [0, 1, 2, 3, 3, 4, 4, 4]
    liblsq.lsq_status_string.restype = C.c_char_p
    assert liblsq.lsq_status_string(0) == b"LSQ_OK"
    assert liblsq.lsq_version() >= 100
    # test-only wait bound of the triangular solves: host state only
    liblsq.lsq_test_set_solve_wait_ns.restype = C.c_int64
    liblsq.lsq_test_set_solve_wait_ns.argtypes = [C.c_int64]
    s = liblsq.lsq_test_set_solve_wait_ns
    assert s(0) == -1 and s(-5) == -1
    old = s(1000)
    assert old == 2_000_000_000
    assert s(old) == 1000


def test_binding_matches_oracle_precision_table(liblsq):
    import oracle as O
    import paper_2603_16644_gb300 as lsq

    for k in [-1.0, 0.0, 1.99, 2.0, 2.99, 3.0, 3.99, 4.0, 7.5, 8.0, 8.0000001, 12.0, float("inf")]:
        assert lsq.precision_from_kappa0(k) == O.precision_from_kappa0(k)


def test_calls_fail_loudly_without_cuda_tensors(liblsq):
    import torch

    import paper_2603_16644_gb300 as lsq

    A = torch.zeros((10, 3), dtype=torch.float64)
    with pytest.raises(lsq.LsqError):
        lsq.pne(A, torch.zeros(10, dtype=torch.float64))


@pytest.mark.parametrize("s,n", [(96, 48), (600, 300), (2000, 1000), (8192, 4096)])
def test_sketch_accumulation_chain_is_bounded(liblsq, s, n):
    """One accumulator of an FP32 Gaussian sketch sums at most 96 K blocks of
    64 products, whatever the rows (64 splits reach that at 131072 rows)."""
    f = liblsq.lsq_test_sketch_chain
    f.restype = C.c_int64
    f.argtypes = [C.c_int64, C.c_int64, C.c_int64, C.c_int32]
    assert f(s, n, 16383, 152) == 0 and f(s, n, 0, 152) == -1
    for m in [16384, 16385, 50001, 131072, 131073, 200000, 262144, 262145, 1000000, 3000017]:
        assert 0 < f(s, n, m, 152) <= 96 * 64, m


def test_lu_panel_cluster_follows_the_device(liblsq):
    """The LU panel's cluster never exceeds what the device schedules, leaves a
    CTA at most 512 rows, and gives way to the one-CTA kernel beyond."""
    f = liblsq.lsq_test_lu_cluster
    f.restype = C.c_int32
    f.argtypes = [C.c_int64, C.c_int32]
    for cap in (16, 8, 0):
        for rows in [1, 63, 64, 65, 128, 129, 512, 513, 1024, 1025, 4096, 4097, 8192, 8193, 100000]:
            cl = f(rows, cap)
            assert 0 <= cl <= cap
            if cl:
                assert cl * 512 >= rows and (cl == cap or cl * 64 >= rows)
            else:
                assert cap * 512 < rows
    assert [f(r, 16) for r in (64, 65, 1024, 8192, 8193)] == [1, 2, 16, 16, 0]
    assert [f(r, 8) for r in (512, 513, 4096, 4097)] == [8, 8, 8, 0]
