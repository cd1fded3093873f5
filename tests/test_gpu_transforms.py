"""The FP64 path's transform kernels sequence by sequence: the rows of one block do not share their accuracy.

The kernel is compiled into a small program with the library's own sources, since the C ABI has no entry for
a transform alone."""
import glob
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_1812_01178_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "k_poisson.cu"
#include <cstdio>
#include <cstdlib>
// rows of n pairs of doubles from a file -> their transform (sign; Fourier or cosine) in another, R rows a block
int main(int argc, char** argv) {
  const int n = atoi(argv[3]), R = atoi(argv[4]), rows = atoi(argv[5]), sign = atoi(argv[6]), cosine = atoi(argv[7]);
  const size_t bytes = (size_t)rows * n * sizeof(double2);
  std::vector<char> h(bytes);
  FILE* f = fopen(argv[1], "rb");
  if (!f || fread(h.data(), 1, bytes, f) != bytes) return 2;
  fclose(f);
  std::vector<FxTw> tw(4 * (size_t)n);
  fx_twiddles(n, tw.data());
  fx_dct_twiddles(n, tw.data() + 3 * n);
  double2* d;
  FxTw* t;
  if (cudaMalloc(&d, bytes) != cudaSuccess || cudaMalloc(&t, tw.size() * sizeof(FxTw)) != cudaSuccess) return 3;
  cudaMemcpy(d, h.data(), bytes, cudaMemcpyHostToDevice);
  cudaMemcpy(t, tw.data(), tw.size() * sizeof(FxTw), cudaMemcpyHostToDevice);
  if (poisson_set_attributes() != cudaSuccess) return 4;
  const size_t smem = (size_t)2 * R * (n + 1) * sizeof(double2);
  const unsigned blocks = (rows + R - 1) / R;
  if (cosine && sign < 0)
    dctx_fwd_kernel<<<blocks, 256, smem>>>(d, t, t + 3 * n, rows, n, fft_plan(n), R);
  else if (cosine)
    dctx_inv_kernel<<<blocks, 256, smem>>>(d, t, t + 3 * n, rows, n, fft_plan(n), R);
  else if (sign < 0)
    single_kernel<FftxK<-1>><<<blocks, 256, smem>>>(FftxK<-1>::Args{d, t, rows, n, fft_plan(n), R});
  else
    single_kernel<FftxK<1>><<<blocks, 256, smem>>>(FftxK<1>::Args{d, t, rows, n, fft_plan(n), R});
  if (cudaGetLastError() != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) return 5;
  cudaMemcpy(h.data(), d, bytes, cudaMemcpyDeviceToHost);
  f = fopen(argv[2], "wb");
  return f && fwrite(h.data(), 1, bytes, f) == bytes && fclose(f) == 0 ? 0 : 6;
}
"""


@pytest.fixture(scope="module")
def transform(tmp_path_factory):
    d = tmp_path_factory.mktemp("transform")
    (d / "main.cu").write_text(SOURCE)
    objs = [o for o in glob.glob(os.path.join(build.OUT, "*.o")) if os.path.basename(o) != "k_poisson.o"]
    subprocess.run([build._nvcc(), *build.NVCC_FLAGS, "-I", build.CSRC, str(d / "main.cu"), *objs, "-lcudart", "-o",
                    str(d / "main")], check=True, capture_output=True)

    def run(x, R, sign, cosine=0):
        x = np.ascontiguousarray(x, dtype=np.complex128)
        x.tofile(d / "in")
        subprocess.run([str(d / "main"), str(d / "in"), str(d / "out"), str(x.shape[1]), str(R), str(x.shape[0]),
                        str(sign), str(cosine)], check=True, timeout=120)
        return np.fromfile(d / "out", dtype=np.complex128).reshape(x.shape)

    return run


def _dft(x, sign):
    """Row transforms in extended precision (a matrix of exact roots, summed by halves)."""
    n = x.shape[1]
    k = np.arange(n)
    pi = np.longdouble("3.14159265358979323846264338327950288")
    root = 2 * pi * k.astype(np.longdouble) / n
    c, s = np.cos(root), sign * np.sin(root)
    out = np.empty(x.shape + (2,), dtype=np.longdouble)
    a, b = x.real.astype(np.longdouble), x.imag.astype(np.longdouble)
    for m in range(n):
        q = (m * k) % n
        out[:, m, 0] = a @ c[q] - b @ s[q]
        out[:, m, 1] = a @ s[q] + b @ c[q]
    return out


def _rows(n, rng):
    """Sequences whose sums grow by n beside some that hardly grow."""
    i = np.arange(n)
    noise = lambda: rng.standard_normal(n) + 1j * rng.standard_normal(n)
    pulse = np.where((i >= 5) & (i < 8), noise(), 0)
    return [np.full(n, 1.37 + 0.4j), pulse, noise() / (1.0 + i) ** 2, noise(), np.exp(2j * np.pi * 3 * i / n),
            1e-6 * pulse, 1e4 * np.full(n, 1 - 1j), 1e-3 * noise() / (1.0 + i) ** 2]


# R as the library takes them in x (512: 3, 216 and 144: 8 and 12, 64: 16) or as many pairs as in z (1024: 2, 256: 4)
@pytest.mark.parametrize("n, R", [(8, 16), (24, 16), (32, 8), (64, 16), (144, 12), (216, 8), (256, 4), (512, 3), (1024, 2)])
@pytest.mark.parametrize("sign", [-1, 1])
def test_error_of_each_sequence(transform, n, R, sign):
    """The relative error of every sequence (2-norm) stays below 1.2e-16, as for one transformed alone: the
    rounding of its results to FP64, 2^-53 / sqrt(3) = 6.4e-17 at most, and, for its largest element up to
    sqrt(1024) times the mean one, 32 2^-62 times four bits of shifts and roundings.  FP64 butterflies
    leave 1.4e-16 to 4e-16."""
    rng = np.random.default_rng(n)
    rows = _rows(n, rng)
    x = np.array([rows[q] for q in rng.permutation(np.arange(4 * R) % len(rows))])
    got, ref = transform(x, R, sign), _dft(x, sign)
    err = np.hypot(got.real - ref[..., 0], got.imag - ref[..., 1])
    rel = np.sqrt((err ** 2).sum(1) / (ref ** 2).sum((1, 2)))
    assert rel.max() <= 1.2e-16, [(float(r), int(q)) for r, q in zip(rel, range(len(x))) if r > 1.2e-16][:8]


@pytest.mark.parametrize("cosine", [0, 1])
@pytest.mark.parametrize("n, R", [(24, 16), (64, 16), (216, 8), (256, 4), (512, 3)])
@pytest.mark.parametrize("sign", [-1, 1])
def test_sequences_outside_the_range_leave_the_others(transform, n, R, sign, cosine):
    """An infinity, a NaN or values near an end of the binary64 range in some sequences: the others come out
    the same, bit for bit, those scaled by a power of two as FP64 arithmetic leaves them.  (In FP64 throughout,
    those would be the scaled results bit for bit: that they differ shows that the others were not.)"""
    rng = np.random.default_rng(n)
    rows = 4 * R + 1
    x = rng.standard_normal((rows, n)) + 1j * rng.standard_normal((rows, n))
    clean = transform(x, R, sign, cosine)
    odd = np.arange(rows) % 3 == 1
    kind = np.arange(rows) // 3 % 4
    y = x.copy()
    y[odd & (kind == 0), 1] = np.inf
    y[odd & (kind == 1), n // 2] = complex(0.0, np.nan)
    y[odd & (kind == 2)] *= 2.0 ** -960
    y[odd & (kind == 3)] *= 2.0 ** 930
    got = transform(y, R, sign, cosine)
    assert (got[~odd] == clean[~odd]).all()
    assert not np.isfinite(got[odd & (kind < 2)]).all(1).any()
    for k, e in ((2, 960), (3, -930)):
        a, b = got[odd & (kind == k)] * 2.0 ** e, clean[odd & (kind == k)]
        # 3 log2(n) roundings at most, either way
        assert (a != b).any()
        assert (np.abs(a - b).max(1) <= 6 * np.log2(n) * 2.0 ** -53 * np.abs(b).max(1)).all()
