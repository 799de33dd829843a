"""The FP64 inverse and products of the prefactorisation by themselves (a small
program around csrc/k_dense64.cu), against results that are exact in FP64:
I + v v^T with powers of two in v, whose inverse I - v v^T / (1 + v^T v) has
representable entries; products of integers, and of full 53-bit values with
signed permutations.

Tolerances, u = 2^-53: an inverse is a chain of n / 64 block steps that round
every entry once or twice, errors growing by the condition number at most:
|X - X*| <= (2 n / 64 + 16) kappa u max |X*|.  The pivot blocks' double-float
sweep alone (2^-46 kappa) does not meet it.  Integers below 2^49 and single
53-bit values come out exactly."""
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
U = 2.0 ** -53

HARNESS = r"""
#include <cstdio>
#include <vector>
#include "k_dense64.cu"
namespace pdg { void set_error(const std::string& m) { std::fprintf(stderr, "%s\n", m.c_str()); } }
using namespace pdg;
static std::vector<double> get(size_t n) {
    std::vector<double> v(n);
    if (std::fread(v.data(), 8, n, stdin) != n) std::exit(2);
    return v;
}
int main(int argc, char** argv) {   // inv n batch | gemm ta tb M N K batch: matrices in and out by stdin and stdout
    auto arg = [&](int k) { return k < argc ? std::atoi(argv[k]) : 0; };
    cudaStream_t s;
    PDG_CUDA(cudaStreamCreate(&s));
    DBuf<double> a, b, c;
    DBuf<int> err;
    err.alloc(1);
    PDG_CUDA(cudaMemsetAsync(err.p, 0, 4, s));
    std::vector<double> out;
    if (std::string(argv[1]) == "inv") {
        const int n = arg(2), batch = arg(3);
        const size_t nn = (size_t)n * n;
        const std::vector<double> A = get(nn * batch);
        upload(a, A, s);
        c.alloc(nn * batch);
        dense_spd_inverse(a.p, n, n, nn, c.p, n, nn, batch, err.p, s);
        out.resize(nn * batch);
    } else {
        const int ta = arg(2), tb = arg(3), M = arg(4), N = arg(5), K = arg(6), batch = arg(7);
        const std::vector<double> A = get((size_t)M * K * batch), B = get((size_t)K * N * batch);
        upload(a, A, s);
        upload(b, B, s);
        c.alloc((size_t)M * N * batch);
        dense_gemm(ta, tb, M, N, K, -1.0, a.p, ta ? M : K, (int64_t)M * K, b.p, tb ? K : N, (int64_t)K * N, 0.0, c.p, N,
                   (int64_t)M * N, batch, s);
        out.resize((size_t)M * N * batch);
    }
    int e = 0;
    PDG_CUDA(cudaMemcpyAsync(out.data(), c.p, 8 * out.size(), cudaMemcpyDeviceToHost, s));
    PDG_CUDA(cudaMemcpyAsync(&e, err.p, 4, cudaMemcpyDeviceToHost, s));
    PDG_CUDA(cudaStreamSynchronize(s));
    std::fwrite(out.data(), 8, out.size(), stdout);
    std::fwrite(&e, 4, 1, stdout);
}
"""


@pytest.fixture(scope="module")
def dense(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2405_12484_gb300 import build
    d = tmp_path_factory.mktemp("dense64")
    (d / "t.cu").write_text(HARNESS)
    subprocess.run([build._nvcc(), build.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC,
                    str(d / "t.cu"), "-o", str(d / "t")], check=True, capture_output=True)

    def call(args, *mats):
        r = subprocess.run([str(d / "t"), *map(str, args)], input=b"".join(np.ascontiguousarray(m).tobytes() for m in mats),
                           capture_output=True, timeout=120)
        assert r.returncode == 0, r.stderr
        return np.frombuffer(r.stdout[:-4]), int(np.frombuffer(r.stdout[-4:], np.int32)[0])
    return call


def _rank_one(rng, n, kind):
    """(A, exact inverse, condition number)"""
    v = np.zeros(n)
    if kind == "mild":      # v^T v = 1 or 3
        m = 4 ** int(np.log2(n) // 2) if n < 192 else 3 * 4 ** int(np.log2(n / 3) // 2)
        v[:m] = 1.0 / np.sqrt(m if n < 192 else m / 3)
    else:                   # three entries of each of 1, 2 .. 512: 1 + v^T v = 2^20
        v[:30] = np.repeat(2.0 ** np.arange(10), 3)
    v = (v * rng.choice([-1.0, 1.0], n))[rng.permutation(n)]
    k = 1.0 + v @ v
    return np.eye(n) + np.outer(v, v), np.eye(n) - np.outer(v, v) / k, k


@pytest.mark.parametrize("kind", ["mild", "steep"])
@pytest.mark.parametrize("n,batch", [(64, 1), (64, 350), (128, 3), (192, 2), (768, 1), (1024, 5), (2048, 1)])
def test_inverse_of_rank_one_updates(dense, n, batch, kind):
    """One pivot to 32; a batch of 350 is more than one slice of the digits' scratch (255 at n = 64)."""
    rng = np.random.default_rng(n + batch)
    A, X, k = zip(*(_rank_one(rng, n, kind) for _ in range(batch)))
    got, err = dense(("inv", n, batch), np.stack(A))
    assert err == 0
    got = got.reshape(batch, n, n)
    for z in range(batch):
        assert np.abs(got[z] - X[z]).max() <= (2 * n / 64 + 16) * k[z] * U * np.abs(X[z]).max()


@pytest.mark.parametrize("n,bad", [(64, 0), (64, 63), (192, 64), (192, 191), (1024, 700)])
def test_a_pivot_that_is_not_positive_is_reported(dense, n, bad):
    A, _, _ = _rank_one(np.random.default_rng(n), n, "mild")
    A[bad, bad] = -1.0
    assert dense(("inv", n, 1), A)[1] != 0


@pytest.mark.parametrize("M,N,K,batch", [(1, 1, 1, 1), (64, 64, 64, 1), (65, 63, 129, 3), (200, 8, 300, 2), (8, 40, 2048, 2),
                                         (520, 2048, 2048, 1)])
def test_products_of_integers_are_exact(dense, M, N, K, batch):
    """The last size is cut into row slices (its digits exceed the scratch)."""
    rng = np.random.default_rng(M + K)
    A, B = (rng.integers(-2 ** 19, 2 ** 19, s).astype(np.float64) for s in ((batch, M, K), (batch, K, N)))
    want = -np.matmul(A.astype(np.int64), B.astype(np.int64)) if M * N * K < 10 ** 8 else -np.matmul(A, B)
    for ta in (0, 1):
        for tb in (0, 1):
            got, _ = dense(("gemm", ta, tb, M, N, K, batch), A.transpose(0, 2, 1) if ta else A, B.transpose(0, 2, 1) if tb else B)
            assert np.array_equal(got.reshape(batch, M, N), want.astype(np.float64))


def test_products_keep_all_53_bits(dense):
    rng = np.random.default_rng(7)
    n = 150
    A = rng.uniform(0.125, 1.0, (n, n)) * rng.choice([-1.0, 1.0], (n, n)) * 2.0 ** rng.integers(-200, 200, (n, 1))
    P = np.zeros((n, n))
    P[np.arange(n), rng.permutation(n)] = rng.choice([-1.0, 1.0], n)
    got, _ = dense(("gemm", 0, 0, n, n, n, 1), A, P)
    assert np.array_equal(got.reshape(n, n), -(A @ P))
