"""Host side of the launch code, on a stand-in for the CUDA runtime
(fake_cudart.cpp): kernels do nothing, copies and launch limits behave as the
runtime documents them. No GPU."""
import os
import shutil
import subprocess
import sys

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_1806_02343_gb300 import build
    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    subprocess.run([shutil.which("g++") or "c++", "-O1", "-shared", "-fPIC", "-o", so,
                    os.path.join(ROOT, "tests", "fake_cudart.cpp")], check=True)
    return so


def _run(fake, code, **env):
    pre = "import ctypes, os, sys\nimport numpy as np\nfrom paper_1806_02343_gb300 import binding as Bd\n" \
          "lib, vp = Bd.lib(), ctypes.c_void_p\n"
    r = subprocess.run([sys.executable, "-c", pre + code], cwd=ROOT, capture_output=True, text=True, timeout=300,
                       env=dict(os.environ, PYTHONPATH=ROOT, LD_PRELOAD=fake, **env))
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout


TRAIN = """
def train(n=96, nin=6, epochs=6, batch=32):
    X, y, th = (np.zeros(s, t) for s, t in (((n, nin), np.float32), (n, np.uint8), (64 * nin + 64 * 64 + 193, np.float32)))
    p = lambda a: vp(a.ctypes.data)
    return lib.dg_mhd_mlp_train(p(X), nin, p(y), n, nin, p(th), epochs, batch, 1e-3, 1.0, 5, None, None)
"""


def test_training_reads_every_epochs_own_shuffle(fake, tmp_path):
    """The copy of a shuffle from pageable memory may run as late as its place in the stream: the permutations the
    epochs train on do not depend on when."""
    seen = []
    for defer in "01":
        log = str(tmp_path / f"copies{defer}")
        _run(fake, TRAIN + "assert train() == 0\n", FAKE_DEFER=defer, FAKE_LOG=log)
        seen.append(np.fromfile(log, np.int64).reshape(6, 96))
    assert all(np.array_equal(np.sort(p), np.arange(96)) for p in seen[0])
    assert len({p.tobytes() for p in seen[0]}) == 6
    assert np.array_equal(*seen)


CONTEXTS = """
fake = ctypes.CDLL(os.environ["LD_PRELOAD"])
def rhs(divb, degree, **prm):
    m, p, h = Bd.mesh_desc(3, (6, 5, 4)), Bd.default_params(c_h_fixed=1.0, **prm), vp()
    assert lib.dg_mhd_init(ctypes.byref(m), degree, Bd.DG_DIVB_GLM if divb == "glm" else Bd.DG_DIVB_POWELL, 5 / 3,
                           ctypes.byref(p), ctypes.byref(h)) == 0
    r, k, c, s = (ctypes.c_int64() for _ in range(4))
    lib.dg_mhd_state_layout(h, *(ctypes.byref(x) for x in (r, k, c, s)))
    buf = [np.zeros(r.value * s.value) for _ in range(4)]
    w, out, wm, om = (vp(b.ctypes.data) for b in buf)
    e = lib.dg_mhd_rhs(h, w, wm, out, om, None)
    if not e and prm.get("precision"):
        nin = 8 * [1, 4, 10, 20][degree] + 30
        th = np.zeros(64 * nin + 64 * 64 + 193, np.float32)
        e = lib.dg_mhd_mlp_set_weights(h, vp(th.ctypes.data), nin, 0.5) or lib.dg_mhd_mlp_infer(h, w, wm, out, None, None)
    lib.dg_mhd_destroy(h)
    return e
bad = []
for device in (0, 1):
    fake.fake_device(device)
    if train():
        bad.append((device, "train"))
    for prec in (Bd.DG_PREC_FP64, Bd.DG_PREC_FP32MIX):
        for divb, degree, gen in [("glm", d, 0) for d in (1, 2, 3)] + [("powell", d, 0) for d in (1, 2)] + [("glm", 2, 2)]:
            if rhs(divb, degree, precision=prec, generic_kernels=gen):
                bad.append((device, divb, degree, prec, gen))
print(bad)
assert not bad, bad
"""


def test_launches_work_on_every_device(fake):
    """A kernel's shared-memory limit is set on the device that a call runs on, not once per process."""
    _run(fake, TRAIN + CONTEXTS)


GRADIENT = """
n, nin = 1 << 21, 110
X, y, th = np.zeros((n, nin), np.float32), np.zeros(n, np.uint8), np.zeros(64 * nin + 64 * 64 + 193, np.float32)
grad, p = np.zeros_like(th), lambda a: vp(a.ctypes.data)
assert lib.dg_mhd_mlp_loss_grad(p(X), nin, p(y), n, nin, p(th), 1.0, p(grad), None, None) == 0
assert train(n=n, nin=nin, epochs=1, batch=n) == 0
"""


def test_gradients_of_many_samples_fit_beside_them(fake):
    """Two million samples (0.9 GB of inputs) with 2.2 GB left on the device: four activation rows of each fit."""
    _run(fake, TRAIN + GRADIENT, FAKE_MEMORY=str(2200 << 20))
