"""The C-ABI library builds, loads and exports every function include/moehub.h declares; the host-side
argument checks answer without a GPU.  No compute call is made here."""
import ctypes
import os
import re

import pytest

import __graft_entry__ as entry
from paper_2605_05888_b200 import binding as B

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    entry.build()
    return B.lib()


def declared_functions():
    text = open(os.path.join(ROOT, "include", "moehub.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(moe_[a-z_0-9]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    names = declared_functions()
    assert len(names) >= 14
    for n in names:
        assert hasattr(lib, n), f"{n} declared in moehub.h but not exported"
    assert sorted(B.EXPORTS) == names, "binding.EXPORTS and the header disagree"


def header_config_fields():
    """(name, ctypes type) of every field of moe_config_t, parsed from the header."""
    text = open(os.path.join(ROOT, "include", "moehub.h")).read()
    body = re.search(r"typedef struct \{(.*?)\} moe_config_t;", text, flags=re.S).group(1)
    body = re.sub(r"/\*.*?\*/", "", body, flags=re.S)
    ctype = {"int32_t": ctypes.c_int32, "int64_t": ctypes.c_int64, "uint64_t": ctypes.c_uint64}
    fields = []
    for decl in body.split(";"):
        decl = decl.strip()
        if not decl:
            continue
        ty, names = decl.split(None, 1)
        for name in names.split(","):
            name = name.strip()
            m = re.fullmatch(r"(\w+)\[(\d+)\]", name)
            fields.append((m.group(1), ctype[ty] * int(m.group(2))) if m else (name, ctype[ty]))
    return fields


def test_config_struct_matches_header():
    """Same fields, same order, same types: the binding's ctypes structure mirrors the C struct."""
    want = header_config_fields()
    got = [(n, t) for n, t in B.MoeConfig._fields_]
    assert [n for n, _ in got] == [n for n, _ in want]
    for (n, t_got), (_, t_want) in zip(got, want):
        assert ctypes.sizeof(t_got) == ctypes.sizeof(t_want), n

    class Mirror(ctypes.Structure):
        _fields_ = want
    assert ctypes.sizeof(B.MoeConfig) == ctypes.sizeof(Mirror)
    for n, _ in want:
        assert getattr(B.MoeConfig, n).offset == getattr(Mirror, n).offset, n


def test_host_side_checks_without_gpu(lib):
    ok = B.make_config(4096, 4096, 8, 8, 2, 14336, B.DTYPE_BF16)
    assert B.moe_pool_tiles(ok) == 4096 * 2 // 128 + 8
    assert B.moe_workspace_bytes(ok) > 2 * 72 * 128 * 4096 * 2
    static = B.make_config(300, 128, 8, 2, 2, 64, B.DTYPE_BF16, dispatch_mode=B.DISPATCH_ATOMIC_STATIC)
    assert B.moe_pool_tiles(static) == 8 * 3            # capacity defaults to T rounded up to 128
    for bad, code in [(B.make_config(16, 100, 8, 2, 2, 64, B.DTYPE_BF16), -2),      # H*2 not multiple of 16
                      (B.make_config(16, 128, 8, 3, 2, 64, B.DTYPE_BF16), -1),      # E % R
                      (B.make_config(16, 128, 8, 2, 9, 64, B.DTYPE_BF16), -1),      # K > E
                      (B.make_config(16, 128, 512, 2, 2, 64, B.DTYPE_BF16), -3),    # E > 256
                      (B.make_config(16, 128, 8, 2, 2, 64, 7), -1)]:                # dtype
        with pytest.raises(B.MoeError) as ei:
            B.moe_workspace_bytes(bad)
        assert ei.value.code == code
    assert B.strerror(0) == "ok" and "overflow" in B.strerror(-5)
    h = ctypes.c_void_p()
    assert lib.moe_plan_create(ctypes.byref(ok), None, 0, ctypes.byref(h)) == -1   # null workspace
    assert lib.moe_route(None, None, None, None, None, None, None) == -1


def test_workspace_holds_the_wide_router_logits_only_where_a_kernel_reads_them(lib):
    """[T, 256] fp32 (and 256 squared norms) for the tensor-core filter; nothing for routers of many tokens without it."""
    T, H, E = 2048, 256, 256

    def need(dtype, route_filter=0, tokens=T):
        return B.moe_workspace_bytes(B.make_config(tokens, H, E, 1, 8, 0, dtype, identity_experts=1, route_filter=route_filter))

    plain = need(B.DTYPE_BF16, -1)
    assert need(B.DTYPE_BF16) == plain + T * 1024 + 1024
    rows = B.moe_pool_tiles(B.make_config(T, H, E, 1, 8, 0, B.DTYPE_FP32, identity_experts=1)) * 128
    assert need(B.DTYPE_FP32) == plain + 2 * H * (rows + 4 * T)      # fp32 rows and staging buffers, no logits
    # a batch that the chain kernel takes keeps its logits, whatever route_filter says
    assert need(B.DTYPE_BF16, 0, 512) == need(B.DTYPE_BF16, -1, 512)


def test_fp32_workspace_holds_the_operands_parts_only_where_tensor_cores_read_them(lib):
    def need(T, H, E, K, F, kernel, mode=B.DISPATCH_ATOMIC_PAGED, **kw):
        return B.moe_workspace_bytes(B.make_config(T, H, E, 1, K, F, B.DTYPE_FP32, dispatch_mode=mode, ffn_kernel=kernel, **kw))

    paged = (8192, 4096, 8, 2, 14336)
    rows = (8192 * 2 // 128 + 8) * 128
    assert need(*paged, 0) == need(*paged, 1) + rows * (6 * 4096 + 2 * 14336) + -(-rows // 16 // 256) * 256
    static = (4096, 4096, 64, 2, 2048)                # a region of every expert for every token: 32 times the rows there are
    assert need(*static, 0, B.DISPATCH_ATOMIC_STATIC) == need(*static, 1, B.DISPATCH_ATOMIC_STATIC) < 11.1e9
    assert need(*static, 0, B.DISPATCH_ATOMIC_STATIC, capacity_rows=256) > need(*static, 1, B.DISPATCH_ATOMIC_STATIC, capacity_rows=256)
    assert need(*static, 0, B.DISPATCH_ATOMIC_STATIC, capacity_rows=384) == need(*static, 1, B.DISPATCH_ATOMIC_STATIC, capacity_rows=384)
    assert need(16, 256, 8, 2, 256, 0) == need(16, 256, 8, 2, 256, 1)      # (little work: FMAs)
    for E, H, F, least in ((8, 380, 400, 40e6), (4, 384, 400, 24e6), (17, 512, 400, 90e6), (8, 4, 900, 1)):     # (little work)
        rows = max(int(-(-least // (H * F))), 16 * E)
        assert need(rows, H, E, 1, F, 0) > need(rows, H, E, 1, F, 1), (E, H)
        if least > 1:
            assert need(rows - 1, H, E, 1, F, 0) == need(rows - 1, H, E, 1, F, 1), (E, H)
    for E, H, rows_per_expert in ((8, 512, 8), (16, 512, 8), (17, 512, 16), (64, 256, 16), (65, 384, 16), (65, 380, 32), (256, 256, 32)):
        at, below = rows_per_expert * E, rows_per_expert * E - 1           # (few rows per expert: FMAs, the more experts the longer)
        assert need(at, H, E, 1, 1024, 0) > need(at, H, E, 1, 1024, 1), (E, H)
        assert need(below, H, E, 1, 1024, 0) == need(below, H, E, 1, 1024, 1), (E, H)


def test_wide_router_hands_over_to_the_filter_where_the_chains_get_slower(lib):
    """256 experts and long rows: from 865 tokens on the filter (its squared norms are in the workspace); shorter rows: 1025.
    (H 8200, and 2400 with 256 experts, are where the form that fetches its candidates' rows one by one never applies.)"""
    def norms(tokens, H, E=256):
        a, b = (B.moe_workspace_bytes(B.make_config(tokens, H, E, 1, 8, 0, B.DTYPE_BF16, identity_experts=1, route_filter=f)) for f in (0, -1))
        return a - b - (tokens * 1024 if tokens > 1024 else 0)

    assert [norms(t, 8200) for t in (864, 865, 1024, 1025)] == [0, 1024, 1024, 1024]
    assert [norms(t, 2400) for t in (864, 865, 1024, 1025)] == [0, 0, 0, 1024]
    assert [norms(t, 8200, 192) for t in (865, 1024, 1025)] == [0, 0, 1024]


def test_router_that_fetches_its_candidates_holds_one_set_of_logits_per_slice(lib):
    """From T*E*H = 3.2e8 on (beyond 592 tokens twice that), up to 1184 tokens and H 8192: [slices, T, 256] fp32 and the squared
    norms; outside, what the chains (one set of logits) or the filter (one set and the norms) need."""
    def extra(tokens, H, E):
        a, b = (B.moe_workspace_bytes(B.make_config(tokens, H, E, 1, 4, 0, B.DTYPE_BF16, identity_experts=1, route_filter=f)) for f in (0, -1))
        return a - b + (tokens * 1024 if tokens <= 1024 else 0)      # (-1: the chains' logits up to 1024 tokens)

    def slices(tokens, H, E):      # as many CTAs of 128 tokens x 128 experts as SMs, at most 16 slices, of 4 steps of 64 columns at least
        tiles, steps = -(-tokens // 128) * -(-E // 128), -(-H // 64)
        return -(-steps // -(-steps // max(1, min(148 // tiles, steps // 4, 16))))

    for tokens, H, E in ((175, 7168, 256), (592, 2112, 256), (593, 4224, 256), (864, 7168, 256), (1025, 7168, 256), (1184, 7168, 256), (300, 8192, 160),
                         (1000, 8192, 80)):
        assert extra(tokens, H, E) == slices(tokens, H, E) * tokens * 1024 + 1024, (tokens, H, E)
    for tokens, H, E in ((174, 7168, 256), (592, 2104, 256), (593, 4208, 256), (300, 8200, 160), (1000, 8192, 64)):      # the chains
        assert extra(tokens, H, E) == tokens * 1024, (tokens, H, E)
    for tokens, H, E in ((1185, 7168, 256), (865, 8200, 256), (1184, 2048, 256)):                                        # the filter over all rows
        assert extra(tokens, H, E) == tokens * 1024 + 1024, (tokens, H, E)
