"""Every number of warps of the split float32 inverse (k_gj_split), forced one after the other: the same
inverses to the last bit, of packed and of whole blocks, some of them coupled (those go through the list,
longer than the CTAs that share it at B = 15).  Bound: ||X^ - X|| <= 4 kappa_2 B u32 ||X||, as the other
inverse tests."""
import ctypes

import numpy as np
import pytest

from tests.cuda_helper import compile_cuda

pytestmark = pytest.mark.gpu

SOURCE = r'''
#include "gj.cu"
// Inverts E blocks in place; out: the elements' flags.  -1: not a variant of this size.
extern "C" int unit(int B, int v, int E, float* blk, int packed, int* flag) {
    using namespace emg;
    if (!gj_split_ok(B, v)) return -1;
    float* d = nullptr;
    int* w = nullptr;
    const size_t nb = (size_t)E * B * B * 4, nw = (size_t)(4 * E + 4) * 4;
    if (cudaMalloc((void**)&d, nb) != cudaSuccess || cudaMalloc((void**)&w, nw) != cudaSuccess) return 1;
    cudaMemcpy(d, blk, nb, cudaMemcpyHostToDevice);
    cudaMemset(w, 0, nw);
    const GjWork k = gj_work(w, E);
    cudaMemcpy(k.asm_flag, flag, (size_t)E * 4, cudaMemcpyHostToDevice);
    cudaError_t e = gj_split_dispatch(B, v, (unsigned)E, d, w, packed != 0, 0);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    cudaMemcpy(blk, d, nb, cudaMemcpyDeviceToHost);
    cudaMemcpy(flag, k.flag, (size_t)E * 4, cudaMemcpyDeviceToHost);
    cudaFree(d);
    cudaFree(w);
    return (int)e;
}
'''


@pytest.fixture(scope="module")
def unit(tmp_path_factory):
    return compile_cuda(SOURCE, str(tmp_path_factory.mktemp("variants")), link_library=True).unit


def order(N):
    """Block rows of the packed order: variables 0, 1, 2, 4, then 3."""
    return np.concatenate([np.arange(3 * N), np.arange(4 * N, 5 * N), np.arange(3 * N, 4 * N)])


@pytest.mark.parametrize("N,E", [(3, 1400), (6, 40), (10, 21), (15, 9)])
@pytest.mark.parametrize("packed", [False, True])
def test_all_warps_give_the_same_inverses(unit, N, E, packed):
    B, B4 = 5 * N, 4 * N
    rng = np.random.default_rng(N)
    P = rng.uniform(-0.5, 0.5, (E, B, B)).astype(np.float32)
    w = np.arange(B) // N == 3
    coupled = np.arange(E) % 8 != 7 if N == 3 else np.arange(E) % 3 == 0   # N = 3: 1225 on the list
    P[np.ix_(~coupled, w, ~w)] = 0.0
    P[np.ix_(~coupled, ~w, w)] = 0.0
    o = order(N)

    def at(e):
        return (e * B * B + 3) // 4 * 4

    blk = P.reshape(-1).copy()
    if packed:
        for e in np.nonzero(~coupled)[0]:
            Q = P[e][np.ix_(o, o)]
            blk[at(e):at(e) + 17 * N * N] = np.concatenate([Q[:B4, :B4].ravel(), Q[B4:, B4:].ravel()])
    results = []
    for v in range(4):
        b, f = blk.copy(), (~coupled).astype(np.int32)
        st = unit(B, v, E, ctypes.c_void_p(b.ctypes.data), int(packed), ctypes.c_void_p(f.ctypes.data))
        if st == -1:
            continue
        assert st == 0
        np.testing.assert_array_equal(f != 0, ~coupled)
        X = np.zeros((E, B, B), dtype=np.float32)
        for e in range(E):
            if coupled[e]:
                X[e] = b[e * B * B:(e + 1) * B * B].reshape(B, B).T
            else:
                q = b[at(e):at(e) + 17 * N * N]
                Y = np.zeros((B, B), dtype=np.float32)
                Y[:B4, :B4] = q[:B4 * B4].reshape(B4, B4).T
                Y[B4:, B4:] = q[B4 * B4:].reshape(N, N).T
                X[e][np.ix_(o, o)] = Y
        results.append(X)
    assert len(results) >= 2
    for X in results[1:]:
        np.testing.assert_array_equal(X, results[0])
    Xo = np.linalg.inv(P.astype(np.float64))
    err = np.linalg.norm(results[0] - Xo, ord=2, axis=(1, 2)) / np.linalg.norm(Xo, ord=2, axis=(1, 2))
    assert (err <= 4 * np.linalg.cond(P.astype(np.float64)) * B * 2.0 ** -24).all()
