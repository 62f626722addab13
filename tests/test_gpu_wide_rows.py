"""FP64 row products (the Cholesky-QR update of complex128 and the Ritz rotation)
of blocks wider than a row and a matrix row fit in shared memory together, up to
the most states whose row fits by itself (14,528), called below the C ABI: a
Gram matrix of that size is factored in minutes.  Sums of S products in FP64: 1e-12
of the largest value; a complex64 block is rounded once: 2^-24."""
import ctypes as C

import pytest
import torch

from paper_1501_05654_gb300 import rsg

pytestmark = pytest.mark.gpu


def _call(name, x, M):
    f = getattr(rsg.load(), name)
    f.restype, f.argtypes = C.c_int, [C.c_void_p, C.c_int64, C.c_int, C.c_int, C.c_void_p, C.c_void_p]
    torch.cuda.synchronize()
    assert f(x.data_ptr(), x.shape[0], x.shape[1], M.shape[0], M.data_ptr(), torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()


@pytest.mark.parametrize("S", [130, 7264, 7265, 14528])
@pytest.mark.parametrize("tri,dtype", [(True, torch.complex128), (False, torch.complex128), (False, torch.complex64)])
def test_wide_rows(S, tri, dtype):
    g = torch.Generator(device="cuda").manual_seed(S)
    x = torch.randn((3, S + 2), dtype=torch.complex128, device="cuda", generator=g).to(dtype)
    M = torch.zeros((S, S), dtype=torch.complex128, device="cuda")
    # bands that reach the corners: a full matrix is 3.4 GB
    i = torch.arange(S, device="cuda")
    for d in (0, 1, 2, 31, 64, S // 2, S - 1):
        v = torch.randn(S - d, dtype=torch.complex128, device="cuda", generator=g)
        M[i[d:], i[:S - d]] = v
        if not tri and d:
            M[i[:S - d], i[d:]] = v.flip(0)
    y = x[:, :S].to(torch.complex128)
    want = y @ (M.conj().T if tri else M)
    pad = x[:, S:].clone()
    kind = "d" if dtype == torch.complex128 else "f"
    _call(f"_ZN3rsg16launch_tri_applyI{kind}EE9cudaErrorPvliiPKdP11CUstream_st" if tri else
          f"_ZN3rsg13launch_rotateI{kind}EE9cudaErrorPvliiPKdP11CUstream_st", x, M)
    assert torch.equal(x[:, S:], pad)
    err = ((x[:, :S].to(torch.complex128) - want).abs().max() / want.abs().max()).item()
    assert err < (1e-12 if dtype == torch.complex128 else 2.0 ** -24), err
