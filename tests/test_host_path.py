"""The native host path of the calls (csrc/stb_bind.cpp) on a machine without a GPU: what torch throws inside it reaches Python."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

NO_DEVICE = """
import sys
sys.path.insert(0, sys.argv[1])
import torch
import paper_2408_01803_b200 as stb
buf, status = torch.zeros(4096, dtype=torch.uint8), torch.zeros(1, dtype=torch.int32)
layer = stb.PackedLayer(32, 128, 4, buf, status)
x, y = torch.zeros(1, 128, dtype=torch.float16), torch.zeros(1, 32)
steps = stb.make_steps([(layer, x, y)])
calls = [lambda: stb.layer_stack(None, dev_status=status, marshalled=steps),
         lambda: stb.layer_stack_resident(None, buf, dev_status=status, marshalled=steps),
         lambda: stb.layer_stack([(layer, x, y)]),
         lambda: stb.gemv(layer, x), lambda: stb.gemm_f16(layer, x), lambda: stb.gemm(layer, x.bfloat16())]
for call in calls:
    try:
        call()
    except (RuntimeError, AssertionError) as e:
        print("raised", type(e).__name__)
"""


def test_calls_without_a_device_raise():
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="")
    r = subprocess.run([sys.executable, "-c", NO_DEVICE, ROOT], capture_output=True, text=True, timeout=600, env=env)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.count("raised") == 6, r.stdout


def test_without_the_native_module_the_python_forms_take_every_call(monkeypatch, tmp_path):
    import pytest
    import paper_2408_01803_b200 as stb
    broken = tmp_path / "broken.so"
    broken.write_bytes(b"not a shared object")
    for path in (tmp_path / "missing.so", broken):
        monkeypatch.setattr(stb, "BIND_PATH", str(path))
        monkeypatch.setattr(stb, "_bind", None)
        with pytest.warns(UserWarning, match="native host path"):
            forms = stb._fast()
        for name in ("gemv", "gemm", "gemm_f16", "layer_stack", "layer_stack_resident"):
            assert getattr(forms, name) is getattr(stb, "_%s_py" % name)
        assert stb._fast() is forms


def test_the_native_module_is_rebuilt_for_another_torch(monkeypatch, tmp_path):
    from paper_2408_01803_b200 import build
    import pytest
    if not os.path.exists(build.BIND):
        pytest.skip("not built")
    ran = []

    def run(cmd, **kw):
        ran.append(cmd)
        if cmd[0] == "g++":
            open(cmd[cmd.index("-o") + 1], "w").close()
        return subprocess.CompletedProcess(cmd, 0, "1\n", "")

    monkeypatch.setattr(build.subprocess, "run", run)
    monkeypatch.setattr(build, "BIND", str(tmp_path / "b.so"))
    monkeypatch.setattr(build, "BIND_FOR", str(tmp_path / "b.for"))
    monkeypatch.setattr(build, "OBJ", str(tmp_path))
    build.build_bind()
    compiled = sum(c[0] == "g++" for c in ran)
    build.build_bind()                                      # nothing changed
    assert compiled == 1 and sum(c[0] == "g++" for c in ran) == 1
    monkeypatch.setattr(build, "_bind_target", lambda d: "another torch")
    build.build_bind()
    assert sum(c[0] == "g++" for c in ran) == 2
