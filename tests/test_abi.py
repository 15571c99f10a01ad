"""The C-ABI library loads without a GPU and exports every symbol the header declares."""
import os
import re

from paper_2111_09389_b200 import _lib

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def declared_symbols():
    text = open(os.path.join(ROOT, "include", "lpdt.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(lpdt_[a-z0-9_]+)\s*\(", text)))


def test_header_symbols_are_exported_and_bound():
    lib = _lib.lib()
    names = declared_symbols()
    assert len(names) >= 20
    for n in names:
        assert hasattr(lib, n), n
        assert n in _lib.SIGNATURES, f"{n} has no ctypes signature"
    assert set(_lib.SIGNATURES) == set(names)


def test_version_and_status_strings():
    lib = _lib.lib()
    assert b"sm_100a" in lib.lpdt_version()
    assert lib.lpdt_status_string(0) == b"ok"
    assert lib.lpdt_status_string(3) == b"workspace missing or too small"


def test_binding_names_match_the_abi():
    from paper_2111_09389_b200 import api
    for n in declared_symbols():
        if n == "lpdt_status_string":
            continue
        assert hasattr(api, n), n


def test_recorded_calls_are_checked():
    """lpdt_run_calls: unknown items, items that do not fit, streams out of range and failing calls are errors."""
    import ctypes as C
    from paper_2111_09389_b200 import api
    code = lambda *w: (C.c_uint64 * len(w))(*[v & 0xFFFFFFFFFFFFFFFF for v in w])
    sgd = api.lpdt_call_id("lpdt_sgd_update")              # n, x, g, lr, out
    assert sgd >= 0 and api.lpdt_call_id("lpdt_version") == -1 and api.lpdt_call_id("no such call") == -1
    empty = [sgd, 0, 0, 0, 0, 0, 0]                        # no parameters: nothing to launch
    assert api.lpdt_run_calls(code(*empty, *empty), [0]) == (0, 1)
    assert api.lpdt_run_calls(code(*empty, sgd, 0, -1, 0, 0, 0, 0), [0]) == (1, 1)        # the second call refuses n < 0
    for bad in ([77, 0], [-1, 0], [sgd, 1, 0, 0, 0, 0, 0], empty[:-1], [api.CALL_WAIT, 0, 0], [api.CALL_WAIT, 0, 1, 1],
                [api.CALL_WAIT, 0, 0, 0]):
        assert api.lpdt_run_calls(code(*bad), [0])[0] == 1, bad


def test_zero_point_backward_weight_asks_for_what_it_writes():
    """Raw sums and the two tables of tap sums, besides the contraction's own workspace: nothing that grows with the image."""
    from paper_2111_09389_b200 import api
    up = lambda n: (n + 255) // 256 * 256
    for nodes, H, cin, cout, R in ((1, 8, 64, 32, 3), (3, 56, 64, 32, 3), (2, 20, 48, 80, 1), (2, 9, 7, 10, 3)):
        d = api.conv_desc(nodes, 4, H, H, cin, cout, R, R, 1, R // 2)
        own = up(4 * nodes * R * R * cin * cout) + up(4 * nodes * R * R * cout) + up(4 * nodes * R * R * cin)
        assert api.lpdt_qconv_bwd_weight_affine_workspace_size(d) == own + api.lpdt_qconv_workspace_size(d, 2)


def test_which_weight_gradients_take_one_launch():
    """Many output tiles and a short pixel loop: no sums in memory.  Few tiles, padded channels, no work: sums, or nothing."""
    from paper_2111_09389_b200 import api
    direct = lambda *d: api.lpdt_qconv_bwd_weight_direct(api.conv_desc(*d))
    assert direct(8, 32, 2, 2, 512, 512) == 1 and direct(8, 32, 8, 8, 256, 256) == 1
    assert direct(16, 32, 32, 32, 16, 16) == 0
    assert direct(8, 32, 32, 32, 3, 64) == 0 and direct(0, 32, 2, 2, 512, 512) == 0 and direct(8, 0, 2, 2, 512, 512) == 0
    assert direct(8, 4, 16, 16, 512, 512, 9, 9, 1, 4) == 0 and direct(8, 32, 4, 4, 512, 512, 1, 1, 3, 0) == 0      # CUDA cores only
    import os, subprocess, sys
    out = subprocess.run([sys.executable, "-c", "from paper_2111_09389_b200 import api\n"
                          "print(api.lpdt_qconv_bwd_weight_direct(api.conv_desc(8, 32, 2, 2, 512, 512)))"],
                         env=dict(os.environ, LPDT_DISABLE_TC="1"), capture_output=True, text=True, timeout=300,
                         cwd=os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
    assert out.stdout.split() == ["0"], out.stderr
