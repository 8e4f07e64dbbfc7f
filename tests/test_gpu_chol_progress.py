"""The one-launch factorisation with few CTAs resident, and when a wait runs out.  The kernel is launched directly: with
one CTA and with two, the column chain's CTA told to leave its SM to the chain, it must finish; with its first ticket
withheld (the chain's, so that no column is ever factored) every group must give up within its limit, report the wait
site 8 and leave the device usable.  Sigma_ij = 0.9^|i - j|, whose factor is known: L_ij = 0.9^(i - j) sqrt(0.19), the
first column without the root.  Bound: (N + 1) u per entry of L L', with the same factor of 4 as at the tile edges."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2008_07437_gb300 import build

pytestmark = pytest.mark.gpu

SRC = r"""
#include "chol64.cu"
thread_local Profiler *t_prof = nullptr;
KScope::KScope(int, cudaStream_t, double, double) {}
KScope::~KScope() {}
// host: N + 1 rows, N columns, in and out; status: DevStatus
extern "C" int run(double *host, int N, int ctas, int withhold, long long limit, int *status) {
    const long long ld = (N + 1 + 31) / 32 * 32;
    double *A;
    int *sync;
    DevStatus *st;
    if (cudaMalloc(&A, sizeof(double) * ld * N) || cudaMalloc(&sync, sizeof(int) * GEO_CHOL_SYNC_INTS) ||
        cudaMalloc(&st, sizeof(DevStatus)))
        return 1;
    cudaMemset(sync, 0, sizeof(int) * GEO_CHOL_SYNC_INTS);
    cudaMemset(st, 0, sizeof(DevStatus));
    cudaMemcpy2D(A, sizeof(double) * ld, host, sizeof(double) * (N + 1), sizeof(double) * (N + 1), N, cudaMemcpyHostToDevice);
    const int T = (N + DT - 1) / DT, E = 1;
    DfArgs a{A, ld, 0, N, A + N, ld, 1, T, E, 1, nullptr, 0, sync, T * (T + E) - T * (T - 1) / 2, 1, 1, 0, 0, st, limit};
    if (withhold) cudaMemset(sync, 1, 1);   // the ticket counter starts at 1: nobody runs the chain
    constexpr size_t smem = sizeof(DfSmem) * DF_GROUPS;
    if (cudaFuncSetAttribute(k_chol_df<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) return 2;
    k_chol_df<false><<<ctas, DF_THREADS, smem>>>(a);
    DevStatus h;
    if (cudaGetLastError() || cudaDeviceSynchronize() || cudaMemcpy(&h, st, sizeof h, cudaMemcpyDeviceToHost)) return 3;
    status[0] = h.info;
    status[1] = h.timeout;
    cudaMemcpy2D(host, sizeof(double) * (N + 1), A, sizeof(double) * ld, sizeof(double) * (N + 1), N, cudaMemcpyDeviceToHost);
    cudaFree(A);
    cudaFree(sync);
    cudaFree(st);
    return cudaGetLastError() != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    d = tmp_path_factory.mktemp("df")
    (d / "df.cu").write_text(SRC)
    subprocess.run([build.NVCC, "-shared", "-o", str(d / "df.so"), str(d / "df.cu")] + build._flags(False), check=True)
    lib = ctypes.CDLL(str(d / "df.so"))

    def f(N, ctas, withhold=0, limit=4_000_000_000):
        S = 0.9 ** np.abs(np.arange(N)[:, None] - np.arange(N)[None, :])
        A = np.vstack([S, np.ones((1, N))]).T.copy()       # column-major (N + 1) x N, the last row z' = 1'
        status = (ctypes.c_int * 2)()
        rc = lib.run(A.ctypes.data_as(ctypes.c_void_p), N, ctas, withhold, ctypes.c_longlong(limit), status)
        assert rc == 0
        return S, np.tril(A.T[:N]), A.T[N], list(status)

    return f


def _check(S, L, y, status):
    N = len(S)
    assert status == [0, 0]
    g = 4 * (N + 1) * 2.0 ** -53
    assert np.all(np.abs(L @ L.T - S) <= g)
    assert np.all(np.abs(L @ y - 1.0) <= g * (np.abs(L) @ np.abs(y)))


@pytest.mark.parametrize("ctas", [1, 2, 9])
@pytest.mark.parametrize("N", [33, 64, 100, 1000])
def test_finishes_with_few_ctas(run, N, ctas):
    _check(*run(N, ctas))


def test_a_withheld_ticket_ends_in_a_report(run):
    status = run(400, 9, withhold=1, limit=2_000_000)[3]   # about 1 ms
    assert status == [0, 8]
    _check(*run(400, 9))
