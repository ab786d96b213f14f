"""The call module's behaviour at its edges, on a host without a GPU: each case runs in a child process, since what is tested
would otherwise take the test process down."""
import os
import subprocess
import sys
import textwrap

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _child(code):
    r = subprocess.run([sys.executable, "-c", textwrap.dedent(code)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout


def test_exceptions_of_the_tensor_library_become_python_exceptions():
    """Tensors whose storage or layout cannot be asked for raise; an exception that left the C++ code would end the process."""
    out = _child("""
        import torch
        from torch._subclasses.fake_tensor import FakeTensorMode
        from paper_2605_13915_b200 import binding
        calls = binding._calls()
        with FakeTensorMode():
            t = lambda *s, dtype=torch.int8: torch.empty(*s, dtype=dtype, device="cuda")
            x, w, s, y = t(16, 64, dtype=torch.bfloat16), t(32, 64), t(32, dtype=torch.float32), t(16, 32, dtype=torch.bfloat16)
            ws = t(4096, dtype=torch.uint8)
            q = t(1, 4, 64, dtype=torch.bfloat16)
            k, ks, cu = t(8, 1, 64), t(8, 1, dtype=torch.float32), t(2, dtype=torch.int32)
            w3, s2 = t(1, 32, 64), t(1, 32, dtype=torch.float32)
            for name, args in (("gemm_w8a16", (x, w, s, ws, y, None, 0)), ("gemm_w4a16", (x, w, s, 1, ws, y)),
                               ("grouped_gemm_w8a16", (x, w3, s2, [16], ws, y)),
                               ("grouped_gemm_w4a16", (x, t(1, 32, 32), s2, [16], 1, ws, y)),
                               ("attn_decode_int8kv", (q, k, k, ks, ks, cu, 8, 0.1, 64, ws, q, None)),
                               ("attn_decode_int8kv_spec", (q[None], k, k, ks, ks, cu, 8, 0.1, 64, ws, q[None], None)),
                               ("attn_decode_int8kv_paged", (q, k, k, ks, ks, cu[None], cu, 8, 8, 0.1, 64, ws, q, None))):
                try:
                    getattr(calls, name)(*args)
                except RuntimeError as e:
                    print("raised", name)
        """)
    assert out.count("raised") == 7
