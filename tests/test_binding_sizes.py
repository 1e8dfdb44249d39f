"""The binding refuses tensors that hold less than a call reads or writes, before anything is launched: the C ABI takes
plain pointers.  Flags and sizes are looked at first, so most of this needs no GPU."""
import pytest
import torch

from paper_2609_35465_b200 import build as tbuild


@pytest.fixture(scope="module")
def tt():
    tbuild.build()
    from paper_2609_35465_b200 import tetra
    return tetra


def u8(n, device="cpu"):
    return torch.zeros(n, dtype=torch.uint8, device=device)


def test_decode_packed_wants_the_whole_matrix(tt):
    packed = u8(tt.tetra_codes_bytes(16, 3) - 1)
    with pytest.raises(tt.TetraError, match="packed.*needs 288"):
        tt.tetra_decode_packed(packed, None, 16, 3)


@pytest.mark.parametrize("call", ["gemv", "gemv_tail", "noalloc", "batched", "list", "grouped_run", "encode", "pack"])
def test_every_call_wants_the_whole_table(tt, call):
    f, h = torch.zeros(8, dtype=torch.float32), torch.zeros(24, dtype=torch.float16)
    table = u8(tt.tetra_table_bytes() - 1)
    with pytest.raises(tt.TetraError, match="table.*needs"):
        if call == "gemv":
            tt.tetra_gemv(u8(48), f, table, h, f, 8, 24)
        elif call == "gemv_tail":
            tt.tetra_gemv_tail(u8(48), f, table, h, f, 8, 24)
        elif call == "noalloc":
            tt.tetra_gemv_noalloc(u8(48), f, table, h, f, 8, 24)
        elif call == "batched":
            tt.tetra_gemv_batched(u8(48), f, table, h, f, 8, 24, 1, None, u8(1 << 16))
        elif call == "list":
            tt.tetra_gemv_list((tt.Problem * 1)(), table)
        elif call == "grouped_run":
            tt.tetra_gemv_grouped_run(u8(4096), table)
        elif call == "encode":
            tt.tetra_encode_blocks(torch.zeros((0, 24)), table)
        else:
            tt.tetra_pack_codes(u8(48), table, 8, 1)


@pytest.mark.gpu
def test_packed_output_and_sources(tt):
    table = tt.tetra_build_table()
    codes, n = u8(16 * 3 * 6, "cuda").reshape(16, 3, 6), tt.tetra_codes_bytes(16, 3)
    for out in (u8(2 * n, "cuda")[::2], u8(n)):  # every second byte; memory the device cannot reach
        with pytest.raises(tt.TetraError, match="out: tensor is n"):
            tt.tetra_pack_codes(codes, table, 16, 3, out)
    with pytest.raises(AssertionError):
        tt.tetra_pack_codes(codes, table, 16, 3, u8(n - 1, "cuda"))
    packed = tt.tetra_pack_codes(codes, table, 16, 3, u8(n + 16, "cuda"))
    y, mg = tt.tetra_decode_packed(packed, table, 16, 3)
    with pytest.raises(tt.TetraError, match="not contiguous"):
        tt.tetra_decode_packed(u8(2 * n, "cuda")[::2], table, 16, 3)
    with pytest.raises(tt.TetraError, match="needs"):
        tt.tetra_decode_packed(packed[:n - 16], table, 16, 3)
    torch.cuda.synchronize()
    assert not y.any() and not mg.any()  # the all-zero word is the origin


@pytest.mark.gpu
def test_batched_workspace_is_counted_in_bytes(tt):
    table = tt.tetra_build_table()
    need = tt.tetra_batched_workspace_bytes(8, 24)
    rs, x = torch.ones(8, device="cuda"), torch.ones((2, 24), dtype=torch.float16, device="cuda")
    y = torch.empty((2, 8), device="cuda")
    for n, fits in ((need // 4, True), (need // 4 - 1, False)):
        ws = torch.empty(n, dtype=torch.float32, device="cuda")
        if fits:
            tt.tetra_gemv_batched(u8(48, "cuda"), rs, table, x, y, 8, 24, 2, None, ws)
        else:
            with pytest.raises(tt.TetraError, match="too small"):
                tt.tetra_gemv_batched(u8(48, "cuda"), rs, table, x, y, 8, 24, 2, None, ws)
    torch.cuda.synchronize()
    assert not y.any()


class Undecided:
    def __bool__(self):
        raise ValueError("neither")


def test_a_flag_without_a_truth_value_is_an_error(tt):
    with pytest.raises(ValueError, match="neither"):
        tt.tetra_decode_packed(u8(48), None, 8, 1, Undecided())
    with pytest.raises(ValueError, match="neither"):
        tt.tetra_encode_blocks(torch.zeros((0, 24)), None, None, Undecided())


def short(t):
    """All of a tensor but its last element."""
    return t.reshape(-1)[:-1]


# The calls that go through ctypes: comparison arms, host activations, plans, 4-bit lists.  Sources are cut by one element in
# turn; nothing here reaches the library.
@pytest.mark.parametrize("name", ["table", "codes", "row_scales", "x", "y", "tail"])
def test_paper_design_sizes(tt, name, monkeypatch):
    monkeypatch.setattr(torch.Tensor, "is_pinned", lambda self: True)
    t = dict(table=u8(tt.tetra_table_bytes()), codes=u8(3 * 14 + 12), row_scales=torch.zeros(4), tail=torch.zeros((4, 2), dtype=torch.float16),
             x=torch.zeros(50, dtype=torch.float16), y=torch.zeros(4))
    t[name] = short(t[name])
    with pytest.raises(tt.TetraError, match="%s: .*needs" % name):
        tt.tetra_gemv_paper_design(t["codes"], 14, t["row_scales"], t["table"], t["x"], t["y"], 4, 50, 1, t["tail"])


@pytest.mark.parametrize("name", ["table", "codes", "row_scales", "x", "y", "x_host", "y_host"])
def test_hostio_sizes(tt, name, monkeypatch):
    monkeypatch.setattr(torch.Tensor, "is_pinned", lambda self: True)
    h, f = torch.zeros((2, 48), dtype=torch.float16), torch.zeros((2, 8))
    t = dict(table=u8(tt.tetra_table_bytes()), codes=u8(96), row_scales=torch.zeros(8), x=h, y=f, x_host=h, y_host=f)
    t[name] = short(t[name])
    with pytest.raises(tt.TetraError, match="%s: .*needs" % name):
        tt.tetra_gemv_hostio(t["codes"], t["row_scales"], t["table"], t["x_host"], t["y_host"], t["x"], t["y"], 8, 48, 2)


@pytest.mark.parametrize("name", ["table", "x_host", "y_host"])
def test_grouped_hostio_sizes(tt, name, monkeypatch):
    monkeypatch.setattr(torch.Tensor, "is_pinned", lambda self: True)
    t = dict(table=u8(tt.tetra_table_bytes()), x_host=torch.zeros(24, dtype=torch.float16), y_host=torch.zeros(8))
    x_dev, y_dev = t["x_host"].clone(), t["y_host"].clone()
    t[name] = short(t[name])
    with pytest.raises(tt.TetraError, match="%s: .*needs" % name):
        tt.tetra_gemv_grouped_hostio(u8(4096), t["table"], t["x_host"], x_dev, t["y_host"], y_dev)


@pytest.mark.parametrize("name", ["packed", "x", "y"])
def test_q4_problem_sizes(tt, name, monkeypatch):
    monkeypatch.setattr(torch.Tensor, "is_pinned", lambda self: True)
    for K, G in ((192, 64), (256, 128)):
        it = dict(packed=u8(tt.tetra_q4_packed_bytes(40, K, G)), x=torch.zeros(K, dtype=torch.float16), y=torch.zeros(40), N=40, K=K)
        tt.make_q4_problems([it])
        it[name] = short(it[name])
        with pytest.raises(tt.TetraError, match="%s: .*needs" % name):
            tt.make_q4_problems([it])


def test_a_plan_wants_a_workspace_on_the_device(tt):
    with pytest.raises(tt.TetraError, match="workspace.*neither"):
        tt.tetra_gemv_grouped_plan((tt.Problem * 1)(), u8(4096))
