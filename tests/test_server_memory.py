"""The server's memory estimate."""
import pytest

from paper_2506_04489_gb300 import serve

CODE = {"fp64": 0, "fp32": 1, "mixed": 2, "df32": 3}


@pytest.mark.parametrize("precision", list(CODE))
def test_sizes_that_no_plan_takes_have_an_estimate(precision):
    from paper_2506_04489_gb300 import build
    build.build()
    from paper_2506_04489_gb300 import _native as N
    cfg = N.ServerConfig(-1.0, 1.0, 1e9, 2, 4, 2, 2, 2 * 128 ** 3, 256 ** 3)
    for n in (1, 1025, 1100, 2000):
        assert N.lib.sp_server_entry_bytes(cfg, n, CODE[precision]) == serve.entry_bytes(n, precision, 2) > 0
