"""The order in which the fp32-scale product kernel walks a parent's products, and the sums it carries from one to the next
(csrc/fmm_walk.h, plain C++, compiled here): the carried sums decode to the same C, no block gets to see a product that it is
not fed by, and the running sums cost no more rounding error than the stated factor."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2609_26077_b200 import build as B, realizations as P

CXX = shutil.which("g++") or shutil.which("c++")
pytestmark = pytest.mark.skipif(CXX is None, reason="no C++ compiler")
DENSE = [f"orbit_{k:02d}" for k in range(1, 15)]
NAMES = ["strassen", "winograd", "phi_optimal", "strassen_rb", "winograd_rb"] + P.PERTURBATIONS + DENSE


@pytest.fixture(scope="module")
def walk(tmp_path_factory):
    tmp = tmp_path_factory.mktemp("walk")
    src, so = tmp / "walk.cpp", tmp / "walk.so"
    src.write_text('#include "fmm_walk.h"\n'
                   'typedef const float (*Rows)[4];\n'
                   'extern "C" void walk(int R, const float* U, const float* V, const float* W, int* order, float* carry)\n'
                   '{ fmm_choose_walk(R, (Rows)U, (Rows)V, (Rows)W, order, carry); }\n'
                   'extern "C" float emitted(float w, float c, float n) { return fmm_emitted_weight(w, c, n); }\n')
    subprocess.check_call([CXX, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", B.CSRC, str(src), "-o", str(so)])
    lib = C.CDLL(str(so))
    lib.emitted.restype = C.c_float
    lib.emitted.argtypes = [C.c_float] * 3

    def run(U, V, W):
        U, V, W = (np.ascontiguousarray(x, dtype=np.float32) for x in (U, V, W))
        R = len(W)
        order, carry = np.zeros(R, np.int32), np.zeros(R, np.float32)
        lib.walk(C.c_int(R), U.ctypes.data_as(C.c_void_p), V.ctypes.data_as(C.c_void_p), W.ctypes.data_as(C.c_void_p), order.ctypes.data_as(C.c_void_p), carry.ctypes.data_as(C.c_void_p))
        weights = np.array([[lib.emitted(W[r][q], carry[s + 1], W[order[s + 1]][q]) if s + 1 < R else W[r][q] for q in range(4)]
                            for s, r in enumerate(order)], dtype=np.float32)
        return W, order, carry, weights

    return run


def sizes(U, V):
    """Variances of the products of operands with independent elements."""
    return (U.astype(np.float64) ** 2).sum(1) * (V.astype(np.float64) ** 2).sum(1)


def growth(size, W, order, carry):
    """Rounding error of C against separate sums, for independent products M_r of variance size[r]: the running sum holds
    v_t = size_t + c_t^2 v_{t-1}; adding M_t to it in many small steps rounds at sizes from c_t^2 v_{t-1} up to v_t, in the
    mean size_t / 2 + c_t^2 v_{t-1} against size_t / 2; and an error of S_t reaches C_q with the factor W_t[q], like M_t itself."""
    v, fresh, extra = 0.0, 0.0, 0.0
    for r, c in zip(order, carry):
        w2 = float((W[r].astype(np.float64) ** 2).sum())
        fresh += w2 * size[r]
        extra += 2.0 * w2 * c * c * v
        v = size[r] + c * c * v
    return float(np.sqrt(1.0 + extra / fresh))


@pytest.mark.parametrize("name", NAMES + ["cubic8"])
def test_carried_sums_decode_to_the_same_result(walk, name):
    W, order, carry, weights = walk(*P.get(name))
    R = len(W)
    assert sorted(order) == list(range(R)) and carry[0] == 0.0
    sums = np.zeros((R, R))                               # S_t in terms of the products
    for t, r in enumerate(order):
        sums[t] = carry[t] * (sums[t - 1] if t else 0.0)
        sums[t, r] += 1.0
    got = sums.T @ weights.astype(np.float64)
    assert np.abs(got - W).max() <= 4e-7 * np.abs(W).max()


@pytest.mark.parametrize("name,updates", [("strassen", 10), ("winograd", 7), ("phi_optimal", 12), ("cubic8", 4)] + [(n, 17) for n in DENSE])
def test_updates_of_c(walk, name, updates):
    assert np.count_nonzero(walk(*P.get(name))[3]) == updates


@pytest.mark.parametrize("name", NAMES + ["cubic8"])
def test_running_sums_round_little_more_than_separate_ones(walk, name):
    W, order, carry, _ = walk(*P.get(name))
    # one ulp of the coefficients above 1
    assert np.abs(carry).max() <= 1.0 + 2e-6
    # three sums in a row carried with 1 make it 1.57 for the Winograd form and 1.64 for some of the perturbed realizations
    assert growth(sizes(*P.get(name)[:2]), W, order, carry) <= 1.65


def test_no_block_sees_a_product_that_does_not_feed_it(walk):
    rng = np.random.default_rng(5)
    tables = [P.get(n) for n in NAMES]
    # small integers with many zeros: proportional parts of rows whose supports differ
    tables += [rng.integers(-1, 2, (3, 7, 4)).astype(np.float32) for _ in range(200)]
    for table in tables:
        W, order, carry, weights = walk(*table)
        fed = np.zeros(4, bool)                           # blocks that every product in the running sum feeds
        for t, r in enumerate(order):
            fed = (fed & (W[r] != 0)) if carry[t] != 0 else (W[r] != 0)
            # what goes out now and what is carried on reaches only blocks that all of the sum's products feed
            assert not ((weights[t] != 0) & ~fed).any()
            if t + 1 < len(order) and carry[t + 1] != 0:
                assert not ((W[order[t + 1]] != 0) & ~fed).any()


@pytest.mark.parametrize("name", ["winograd", "phi_optimal", "orbit_10", "orbit_12"])
def test_fp32_sums_against_exact_ones(walk, name):
    # the promotion loop restated: 128 K blocks per product, fp32 accumulators, one rounding per block and element
    W, order, carry, weights = walk(*P.get(name))
    rng = np.random.default_rng(11)
    size = sizes(*P.get(name)[:2])
    M = (rng.standard_normal((len(W), 128, 4096)) * np.sqrt(size)[:, None, None]).astype(np.float32)
    exact = np.einsum("rq,rkx->qx", W.astype(np.float64), M.astype(np.float64))

    def error(use_carry):
        out, acc = np.zeros((4, M.shape[2]), np.float32), np.zeros(M.shape[2], np.float32)
        for t, r in enumerate(order):
            acc = acc * carry[t] if use_carry and t else np.zeros_like(acc)
            for k in range(M.shape[1]):
                acc = acc + M[r, k]
            for q in range(4):
                w = (weights[t] if use_carry else W[r])[q]
                if w != 0:
                    out[q] = out[q] + w * acc
        return np.linalg.norm(out - exact)

    # the model's bound and the scatter of 4 x 4096 elements' rounding errors
    assert error(True) <= 1.05 * growth(size, W, order, carry) * error(False)
    assert error(True) <= 1.7 * error(False)
