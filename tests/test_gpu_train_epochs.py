"""Training over several epochs: each epoch takes its own shuffle of the samples.
Six epochs twice are bit for bit the same, and so is one epoch over a training set
that lists the samples of all six in the order they were drawn (the shuffle of the
longer set undone beforehand)."""
import shutil
import subprocess

import numpy as np
import pytest

from oracle import mlp as M

pytestmark = pytest.mark.gpu

SHUFFLE = """
#include <algorithm>
#include <cstdint>
#include <random>
extern "C" void shuffles(uint64_t seed, int64_t n, int epochs, int64_t* out) {
  std::mt19937_64 rng(seed);
  for (int64_t i = 0; i < n; ++i) out[i] = i;
  for (int e = 0; e < epochs; ++e) {
    if (e) std::copy(out + (e - 1) * n, out + e * n, out + e * n);
    std::shuffle(out + e * n, out + (e + 1) * n, rng);
  }
}
"""


@pytest.mark.parametrize("n,batch", [(60000, 3000), (1 << 20, 1 << 17)])
def test_epochs_are_their_own_shuffles(n, batch, tmp_path):
    import ctypes
    import torch
    from paper_1806_02343_gb300.binding import mlp_train
    epochs, seed, nin = 6, 5, 16
    src, so = tmp_path / "shuffle.cpp", tmp_path / "libshuffle.so"
    src.write_text(SHUFFLE)
    subprocess.run([shutil.which("g++") or "c++", "-O1", "-shared", "-fPIC", "-o", str(so), str(src)], check=True)
    lib = ctypes.CDLL(str(so))

    def shuffles(count, e):
        out = np.zeros(count * e, np.int64)
        lib.shuffles(ctypes.c_uint64(seed), ctypes.c_int64(count), e, out.ctypes.data_as(ctypes.c_void_p))
        return out

    r = np.random.default_rng(1)
    X = torch.as_tensor(r.normal(size=(n, nin)).astype(np.float32), device="cuda")
    y = (X[:, 0] > 0.5).to(torch.uint8)
    order = shuffles(n, epochs)              # the samples of all epochs, in the order they are drawn
    long = np.empty(n * epochs, np.int64)
    long[shuffles(n * epochs, 1)] = order    # its own shuffle gives that order back
    pick = torch.as_tensor(long, device="cuda")
    outs = []
    for data, labels, count in ((X, y, epochs), (X, y, epochs), (X[pick], y[pick], 1)):
        th = torch.as_tensor(M.init_params(nin, seed=2), dtype=torch.float32, device="cuda")
        mlp_train(data, labels, th, nin, epochs=count, batch=batch, lr=1e-3, seed=seed)
        outs.append(th)
    assert torch.equal(outs[0], outs[1]) and torch.equal(outs[0], outs[2])
