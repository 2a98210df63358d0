"""Host-side checks of the C-ABI library that need no GPU: it loads, exports every symbol the
header declares, sizes workspaces, and rejects bad arguments before touching the device."""
import ctypes
import os
import re

import pytest

from paper_2406_17542_b200 import binding as B
from paper_2406_17542_b200 import build as cdq_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    if not os.path.exists(B.LIB_PATH):
        cdq_build.build()
    return B.load()


def _declared_symbols():
    text = open(os.path.join(ROOT, "include", "cdq.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    return sorted(set(re.findall(r"\b(cdq_[a-z0-9_]+)\s*\(", text)))


def test_every_declared_symbol_is_exported(lib):
    names = _declared_symbols()
    assert set(names) == set(B.EXPORTS)
    for name in names:
        assert getattr(lib, name) is not None


def test_version_and_status_strings(lib):
    assert lib.cdq_version() >= 100
    seen = {lib.cdq_status_string(s) for s in range(7)}
    assert len(seen) == 7 and b"ok" in seen


def test_workspace_sizes(lib):
    g = B.Grid(bits=3)
    cd = B.workspace_bytes(B.CALL_CD_SOLVE, 0, 2048, 16384, g)
    ll = B.workspace_bytes(B.CALL_LAYER_LOSS, 0, 2048, 16384, g)
    assert cd % 256 == 0 and ll % 256 == 0
    # residual (fp64) + gradient (fp64) + transposed codes
    assert cd >= 2048 * 16384 * (8 + 8 + 1)
    assert ll >= 2048 * 16384 * 8 and ll < cd
    assert B.workspace_bytes(B.CALL_HESSIAN, 1024, 256, 0, None, "verify") >= 256 * 256 * 8
    owc = B.workspace_bytes(B.CALL_INIT_RTN, 0, 4096, 4096, B.Grid(2, 128, 20, 0.5, 1.0))
    mm = B.workspace_bytes(B.CALL_INIT_RTN, 0, 4096, 4096, B.Grid(2, 128))
    assert owc > mm > 0
    assert B.workspace_bytes(B.CALL_INIT_RTN, 0, 100, 8, B.Grid(2, 7)) == 0   # 100 % 7 != 0
    # pairs: the table of all steps' pairs (16 bytes per pair and step) on top of the descent's workspace
    b0 = B.workspace_bytes(B.CALL_BCD_SOLVE, 0, 2048, 16384, g)
    b256 = B.workspace_bytes(B.CALL_BCD_SOLVE, 256, 2048, 16384, g)
    assert b0 == cd and b256 - b0 >= 256 * 1024 * 16 and b256 - b0 < 256 * 1024 * 16 + 4096
    assert B.workspace_bytes(B.CALL_BCD_SOLVE, 256, 2048, 16384, g, "verify") == B.workspace_bytes(B.CALL_CD_SOLVE, 0, 2048, 16384, g, "verify")
    owc_cd = B.workspace_bytes(B.CALL_INIT_OWC_CD, 0, 4096, 4096, B.Grid(2, 128, 20, 0.5, 1.0))
    assert owc_cd > 2 * 20 * 4096 * 8


def test_padded_rows_of_odd_layers_cost_workspace_only_where_nothing_else_lies_idle(lib):
    """The descent's copy of H with rows on 16-byte boundaries (4 bytes per entry) takes the place of the residual or of the
    slices of H; only narrow layers, which have neither, get room for it, and calls that never build it get none."""
    need = lambda which, d_in, d_out, g=0, n=0, mode="fast": B.workspace_bytes(which, n, d_in, d_out, B.Grid(3, g), mode)
    for d_in, d_out in [(8193, 150), (18431, 256), (1350, 677), (301, 200), (255, 255), (129, 70)]:
        up = (d_in + 3) // 4 * 4
        assert need(B.CALL_CD_SOLVE, d_in, d_out) <= need(B.CALL_CD_SOLVE, up, d_out)
    assert need(B.CALL_CD_SOLVE, 8193, 3) >= 4 * 8193 * 8196
    # the fixed-order kernel: rows past the fast kernels' range, groups that are not a multiple of four, the verification mode
    for d_in, d_out, g, mode in [(20001, 8, 0, "fast"), (8190, 8, 10, "fast"), (8193, 8, 0, "verify")]:
        assert need(B.CALL_CD_SOLVE, d_in, d_out, g, mode=mode) < 4 * d_in * d_in
    # pairs with 4 d_in steps need more for their table than the copy would take
    assert need(B.CALL_BCD_SOLVE, 1026, 8, n=4104) < need(B.CALL_BCD_SOLVE, 1028, 8, n=4104) + 4096


def test_small_groups_keep_the_tables_of_the_general_owc_cd_kernel(lib):
    """The kernel on codes takes a fraction of the general kernel's tables (16 bytes per strength and coordinate for each of up to 296
    columns); on small groups it is the slower one."""
    tables = lambda d_in, d_out, nk: 16 * nk * d_in * min(d_out, 296)
    ws = lambda d_in, d_out, g, nk: B.workspace_bytes(B.CALL_INIT_OWC_CD, 0, d_in, d_out, B.Grid(2, g, nk, 0.5, 1.0))
    for d_in, d_out, g, nk in [(2048, 512, 16, 20), (256, 2000, 2, 4), (256, 2000, 1, 2), (768, 300, 24, 32), (4096, 512, 32, 20)]:
        assert ws(d_in, d_out, g, nk) >= tables(d_in, d_out, nk)
    for d_in, d_out, g, nk in [(4096, 1024, 128, 20), (1920, 512, 64, 32)]:
        assert ws(d_in, d_out, g, nk) - ws(d_in, d_out, g, 2) < tables(d_in, d_out, nk) / 2


def test_workspaces_hold_what_their_call_uses(lib):
    """Losses take no matrix of products beside the residual, and descents none of the slices that only losses use: E and G in fp64, codes, and
    one byte per digit of H (rows of d_in rounded up to 128) and of the residual, with one percent for what goes by rows or columns."""
    for d_in, d_out, g, clips in [(4096, 4096, 128, 20), (3072, 130, 0, 4), (14336, 592, 0, 2), (18432, 1184, 128, 20), (19000, 140, 0, 8)]:
        kp = (d_in + 127) // 128 * 128
        need = lambda which, n_clip=1: B.workspace_bytes(which, 0, d_in, d_out, B.Grid(3, g, n_clip, 0.5, 1.0))
        E, small = 8 * d_in * d_out, 16 * (d_in // 128 + 3) * d_out + 64 * (d_in + d_out) + 8192
        loss = E + 6 * d_in * kp + 5 * d_out * kp + small
        assert need(B.CALL_LAYER_LOSS) <= 1.01 * loss
        assert need(B.CALL_CD_SOLVE) <= 1.01 * (loss + 9 * d_out * ((d_in + 3) // 4 * 4))
        assert need(B.CALL_LAYER_LOSS) <= need(B.CALL_CD_SOLVE)
        width = max(d_out + 128, d_out * max(1, min(clips, 2 ** 30 // E) if clips >= 4 else 1))   # columns of one product of the search
        assert need(B.CALL_INIT_RTN, clips) - need(B.CALL_INIT_RTN) <= 1.01 * (
            8 * d_in * width + 4 * d_in * kp + 4 * width * kp + 16 * (d_in // 128 + 3) * width + 40 * clips * d_out + small)


def test_hessians_without_k_splits_take_no_partial_tiles(lib):
    need = lambda n, d_in: B.workspace_bytes(B.CALL_HESSIAN, n, d_in, 0, None)
    for n, d_in in [(4096, 8192), (1000, 4100), (16384, 18432)]:
        assert need(n, d_in) <= 8 * (d_in // 128 + 2) ** 2
    assert need(16448, 18432) >= 4 * 18432 * 18432 // 2    # more rows than one accumulator takes: the chunks of a tile are summed there


def test_bad_arguments_are_rejected_before_any_launch(lib):
    gd = B.Grid(bits=3).c()
    dummy = ctypes.c_void_p(256)  # never dereferenced: validation fails first
    null = None
    st = lib.cdq_hessian(null, 0, 16, 8, 8, 0.0, 0, dummy, 0, null, 0, null)
    assert st == 1
    st = lib.cdq_hessian(dummy, 0, 16, 8, 4, 0.0, 0, dummy, 0, null, 0, null)   # ldx < d_in
    assert st == 2
    st = lib.cdq_hessian(dummy, 7, 16, 8, 8, 0.0, 0, dummy, 0, null, 0, null)   # bad dtype
    assert st == 1
    bad_bits = B.Grid(bits=9).c()
    st = lib.cdq_init_rtn(dummy, 0, 8, 8, 8, null, ctypes.byref(bad_bits), dummy, dummy, dummy, null, 0, null, 0, null)
    assert st == 1
    bad_group = B.Grid(bits=3, group_size=3).c()
    st = lib.cdq_init_rtn(dummy, 0, 8, 8, 8, null, ctypes.byref(bad_group), dummy, dummy, dummy, null, 0, null, 0, null)
    assert st == 2
    owc_no_h = B.Grid(bits=3, n_clip=4, clip_lo=0.5, clip_hi=1.0).c()
    st = lib.cdq_init_rtn(dummy, 0, 8, 8, 8, null, ctypes.byref(owc_no_h), dummy, dummy, dummy, null, 0, null, 0, null)
    assert st == 1
    # workspace missing / too small / misaligned
    st = lib.cdq_cd_solve(dummy, dummy, 0, 8, 8, 8, ctypes.byref(gd), dummy, dummy, dummy, 1, 0, None, null, 0, null)
    assert st == 4
    st = lib.cdq_cd_solve(dummy, dummy, 0, 8, 8, 8, ctypes.byref(gd), dummy, dummy, dummy, 1, 0, None,
                          ctypes.c_void_p(257), 1 << 30, null)
    assert st == 4
    st = lib.cdq_layer_loss(dummy, dummy, 0, 8, 8, 4, ctypes.byref(gd), dummy, dummy, dummy, None, null, 0, null, 0, null)
    assert st == 2   # ldw < d_out
    st = lib.cdq_cd_solve(dummy, dummy, 0, 8, 8, 8, ctypes.byref(gd), dummy, dummy, dummy, -1, 0, None, null, 0, null)
    assert st == 1
    # pairs: block sizes, odd d_in, too many steps for the table, regulariser arguments
    bcd = lambda d_in, block, steps: lib.cdq_bcd_solve(dummy, dummy, 0, d_in, 8, 8, ctypes.byref(gd), dummy, dummy, dummy,
                                                       block, steps, 0, 0, None, null, 0, null)
    assert bcd(8, 0, 4) == 1
    assert bcd(9, 2, 4) == 2
    assert bcd(8, 3, 4) == 2          # 8 % 3 != 0
    assert bcd(9, 3, 4) == 3          # blocks of three are not built
    assert bcd(8, 2, 70000) == 3
    assert bcd(8, 2, 4) == 4          # valid arguments: the workspace is what is missing
    assert lib.cdq_hessian_add_lambda(null, 8, 0.1, null) == 1
    assert lib.cdq_hessian_add_lambda(dummy, 0, 0.1, null) == 2
    assert lib.cdq_hessian_add_lambda(dummy, 8, -1.0, null) == 1


def test_misaligned_hessian_is_rejected_before_any_launch(lib):
    """H is read with 16-byte vector loads and bulk copies: a pointer 4 bytes off (a view into a larger
    tensor, say) must be refused by every entry point that takes H, not faulted on."""
    gd = B.Grid(bits=3).c()
    owc = B.Grid(bits=3, n_clip=4, clip_lo=0.5, clip_hi=1.0).c()
    dummy, off4, null = ctypes.c_void_p(256), ctypes.c_void_p(260), None
    big = 1 << 30
    assert lib.cdq_hessian(dummy, 0, 16, 8, 8, 0.0, 0, off4, 0, dummy, big, null) == 1
    assert lib.cdq_init_rtn(dummy, 0, 8, 8, 8, off4, ctypes.byref(owc), dummy, dummy, dummy, null, 0, dummy, big, null) == 1
    assert lib.cdq_init_owc_cd(dummy, 0, 8, 8, 8, off4, ctypes.byref(owc), 0, dummy, dummy, dummy, null, None, 0,
                               dummy, big, null) == 1
    assert lib.cdq_cd_solve(off4, dummy, 0, 8, 8, 8, ctypes.byref(gd), dummy, dummy, dummy, 1, 0, None, dummy, big, null) == 1
    assert lib.cdq_cd_solve_steps(off4, dummy, 0, 8, 8, 8, ctypes.byref(gd), dummy, dummy, dummy, 4, 0, None, dummy, big,
                                  null) == 1
    assert lib.cdq_bcd_solve(off4, dummy, 0, 8, 8, 8, ctypes.byref(gd), dummy, dummy, dummy, 2, 4, 0, 0, None, dummy, big,
                             null) == 1
    assert lib.cdq_layer_loss(off4, dummy, 0, 8, 8, 8, ctypes.byref(gd), dummy, dummy, dummy, None, null, 0, dummy, big,
                              null) == 1
    assert lib.cdq_layer_loss_static(off4, dummy, 0, 8, 8, 8, ctypes.byref(gd), dummy, dummy, dummy, None, null, null) == 1
    # the diagnostics entry points check their ranges before touching the device
    assert lib.cdq_debug_expire_wait(0, null) == 1
    assert lib.cdq_debug_set_device_status(7) == 1
    assert lib.cdq_kernel_launches() == 0   # nothing above reached a launch


def test_missing_library_fails_loudly(monkeypatch, tmp_path):
    monkeypatch.setattr(B, "_lib", None)
    monkeypatch.setattr(B, "LIB_PATH", str(tmp_path / "nope.so"))
    with pytest.raises(ImportError):
        B.load()
