"""Host-side checks that need no GPU: the library loads, exports every symbol the
header declares, and validates configurations before touching the device."""
import ctypes as C
import os
import re

import pytest

from paper_2503_05330_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    build.build()
    return binding.lib()


def test_every_declared_symbol_is_exported(lib):
    header = open(os.path.join(ROOT, "include", "sdms.h")).read()
    declared = set(re.findall(r"\b(sdms_[a-z_]+)\s*\(", header))
    assert declared == set(binding.EXPORTS)
    for name in declared:
        assert hasattr(lib, name), name


def test_workspace_bytes_and_config_validation(lib):
    cfg = binding.make_config(1, 16, 1024, 128256, 4, 8)
    n = binding.sdms_workspace_bytes(cfg)
    # path store (tokens + probabilities) plus k_max tables of 2*N*L 32-byte buckets
    assert n >= 2 * 16 * 1024 * 4 + 4 * 2 * 16 * 1024 * 32
    assert n % 256 == 0
    assert binding.sdms_workspace_bytes(binding.make_config(1, 16, 1024, 128256, 4, 8, index_max_n=2)) < n - 2 * 2 * 16 * 1024 * 32 + 4096
    assert binding.sdms_workspace_bytes(binding.make_config(1, 16, 1024, 128256, 4, 8, epsilon=1, wide_table_bytes=-1)) <= n - 4 * 2 * 16 * 1024 * 32   # no index
    # (with a table area: at most the 32 MiB of the hand-over to the wide pass)
    assert 0 < binding.sdms_workspace_bytes(binding.make_config(1, 16, 1024, 128256, 4, 8, epsilon=1)) <= n + (32 << 20)
    bigger = binding.make_config(1, 16, 1024, 128256, 4, 8, B=8, Ke=4)
    assert binding.sdms_workspace_bytes(bigger) > n
    bad = [dict(G=0), dict(N=0), dict(N=2000), dict(L=1), dict(V=0), dict(k_max=0), dict(k_max=17), dict(D=0),
           dict(D=33), dict(max_append=0), dict(max_append=10), dict(B=33), dict(B=4, Ke=0), dict(search_mode=3), dict(search_mode=2, pool_mode=1),
           dict(alpha=1.5), dict(alpha=-0.1), dict(match_capacity=-1), dict(epsilon=2), dict(epsilon=-1), dict(pool_mode=3), dict(pool_mode=-1),
           dict(max_matches_per_path=-1), dict(max_beams=9), dict(max_beams=-1), dict(max_beams=2, pool_mode=1), dict(index_max_n=4), dict(index_max_n=-1)]
    base = dict(G=1, N=4, L=64, V=100, k_max=3, D=4)
    for change in bad:
        kw = dict(base, **change)
        with pytest.raises(binding.SdmsError) as e:
            binding.sdms_workspace_bytes(binding.make_config(**kw))
        assert e.value.code == binding.ERR_INVALID_ARG, change
    cfg = binding.make_config(**base)
    cfg.struct_size = 8
    with pytest.raises(binding.SdmsError):
        binding.sdms_workspace_bytes(cfg)
    # fuzzy matching on small and on large prompts
    assert binding.sdms_workspace_bytes(binding.make_config(1, 256, 8192, 1000, 2, 4, epsilon=1)) > 0
    assert binding.sdms_workspace_bytes(binding.make_config(1, 16, 1024, 1000, 2, 4, epsilon=1)) > 0
    # positions must fit in int32
    with pytest.raises(binding.SdmsError):
        binding.sdms_workspace_bytes(binding.make_config(4096, 1024, 8192, 100, 2, 4))


def test_create_rejects_bad_arguments_without_touching_the_device(lib):
    cfg = binding.make_config(1, 4, 64, 100, 3, 4)
    h = C.c_void_p()
    assert lib.sdms_create(C.byref(cfg), None, 1 << 30, C.byref(h)) == binding.ERR_INVALID_ARG
    assert lib.sdms_create(C.byref(cfg), C.c_void_p(4096 + 8), 1 << 30, C.byref(h)) == binding.ERR_INVALID_ARG
    assert lib.sdms_create(C.byref(cfg), C.c_void_p(4096), 16, C.byref(h)) == binding.ERR_WORKSPACE_TOO_SMALL
    assert lib.sdms_create(C.byref(cfg), C.c_void_p(4096), 1 << 30, None) == binding.ERR_INVALID_ARG
    assert h.value is None
    assert lib.sdms_destroy(None) == binding.ERR_INVALID_ARG
    assert lib.sdms_append(None, None, None, None, 1, None) == binding.ERR_INVALID_ARG
    assert lib.sdms_strerror(binding.ERR_WORKSPACE_TOO_SMALL) == b"workspace too small"
    assert lib.sdms_kernel_name(2) == b"scan"


def test_kernels_that_follow_a_step_do_not_read_path_state_as_read_only():
    # they are resident while it commits (launch_overlapped): no load through the non-coherent path
    csrc = os.path.join(ROOT, "paper_2503_05330_b200", "csrc")
    for name in ("dag.cu", "dag_wide.cu", "beams.cu", "wide_dev.cuh", "beam_dev.cuh"):
        with open(os.path.join(csrc, name)) as f:
            text = f.read()
        assert "__ldg" not in text and "ld.global.nc" not in text, name


def test_inputs_that_another_call_may_still_write_are_not_declared_read_only():
    with open(os.path.join(ROOT, "paper_2503_05330_b200", "csrc", "append.cu")) as f:
        text = f.read()
    for kernel in ("append_kernel", "append_plan_kernel", "accept_kernel", "trim_shift_kernel"):
        params = re.search(kernel + r"\(Dev s,([^)]*)\) \{", text).group(1)
        assert "__restrict__" not in params, kernel


def test_the_default_table_area_follows_the_configuration(lib):
    # 16 bytes per layer and match: every 64th position of a prompt for each of its paths (tolerance 1: 16th), at least eight queries of 14336, at most 320 MiB
    def area(G, N, L, D, **kw):
        with_it, without = (binding.sdms_workspace_bytes(binding.make_config(G, N, L, 1000, 2, D, wide_table_bytes=w, **kw)) for w in (0, -1))
        return with_it - without

    for G, N, L, D, kw, matches in ((32, 16, 4096, 12, {}, 32 * 16 * 16 * 4096 // 64), (1, 64, 2048, 8, {}, 64 * 64 * 2048 // 64),
                                    (1, 16, 4096, 12, {}, 8 * 14336), (8, 32, 1024, 8, dict(epsilon=1), 256 * 32 * 1024 // 16)):
        lists = area(G, N, L, D, **kw) - 16 * D * matches
        assert 0 <= lists < 1 << 15                                  # (the pass's list of queries)
    assert area(2, 256, 512, 32) > 320 << 20 > area(2, 256, 512, 32) - (1 << 15)
    assert area(1, 16, 1024, 8) == 0                                 # no hand-over, no area
