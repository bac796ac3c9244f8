"""Contexts on two devices of one process, without a GPU: the library's calls go
to a stand-in for the CUDA runtime that keeps kernels' shared memory limits per
device.  Every build of every size must be one the runtime would launch, on the
second device as on the first.
"""
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CHILD = """
import ctypes as C, sys
sys.path.insert(0, {root!r})
import paper_0909_0541_gb300 as nb
fake = C.CDLL({fake!r})
for device in (0, 1):
    for n in (1000, 2000, 4096, 5000, 100000):
        cfg, h = nb.nb_config(), C.c_void_p()
        nb._lib.nb_config_default(C.byref(cfg), n)
        cfg.device, cfg.max_systems = device, 70000 if n == 100000 else 2
        rc = [nb._lib.nb_create(C.byref(h), C.byref(cfg)), nb._lib.nb_build_tree(h, 4096, 4096, n)]
        for systems in (2, 70000 if n == 100000 else 1):
            rc.append(nb._lib.nb_build_tree_batched(h, 4096, 4096, 4096, systems, n))
        nb._lib.nb_destroy(h)
        print(device, n, rc, C.c_int.in_dll(fake, "fake_refused").value)
print("launches", C.c_int.in_dll(fake, "fake_launches").value > 200)
"""


def test_builds_on_a_second_device(tmp_path):
    import paper_0909_0541_gb300  # noqa: F401  (builds the library)
    fake = str(tmp_path / "fake_cudart.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-o", fake,
                    os.path.join(HERE, "fake_cudart.c")], check=True)
    r = subprocess.run([sys.executable, "-c", CHILD.format(root=os.path.dirname(HERE), fake=fake)],
                       env=dict(os.environ, LD_PRELOAD=fake, CUDA_VISIBLE_DEVICES=""),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    lines = r.stdout.strip().splitlines()
    assert lines[-1] == "launches True"
    for line in lines[:-1]:
        assert line.endswith("[0, 0, 0, 0] 0"), r.stdout
    assert len(lines) == 11
