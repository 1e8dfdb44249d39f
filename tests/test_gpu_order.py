"""A product right behind the packing of its matrix, nothing between the two: it must multiply the new codes.  The packed
buffer holds another valid matrix before (every word is legal), so a read that comes too early is only a wrong number;
the same calls with a synchronisation between them give the bits to expect."""
import pytest
import torch

from paper_2609_35465_b200 import synth

pytestmark = pytest.mark.gpu
REPEATS = 5


@pytest.fixture(scope="module")
def tt():
    from paper_2609_35465_b200 import tetra
    return tetra


def random_bytes(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randint(0, 256, shape, dtype=torch.uint8, device="cuda", generator=g)


def halves(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(*shape, device="cuda", generator=g).to(torch.float16)


def captured(step):
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        step()
    return graph.replay


def queued(step):
    def go():
        torch.cuda._sleep(2_000_000)  # about a millisecond: the calls below are enqueued before the first one starts
        step()
    return go


def check(pack, products, outputs):
    """pack(which) packs matrix 0 or 1; products: calls that read the packed buffer and write `outputs`."""
    for product in products:
        for o in outputs:
            o.zero_()
        pack(0)
        torch.cuda.synchronize()
        product()
        torch.cuda.synchronize()
        want = [o.clone() for o in outputs]
        pack(1)
        torch.cuda.synchronize()
        product()
        torch.cuda.synchronize()
        assert not all(torch.equal(o, w) for o, w in zip(outputs, want))  # the two matrices tell themselves apart

        def step():
            pack(0)
            product()
        for go in (captured(step), queued(step)):
            for _ in range(REPEATS):
                pack(1)
                for o in outputs:
                    o.zero_()
                torch.cuda.synchronize()
                go()
                torch.cuda.synchronize()
                assert all(torch.equal(o, w) for o, w in zip(outputs, want))


# One row group, a matrix that leaves most SMs free, and one whose packing takes every SM several times over.
@pytest.mark.parametrize("N,K", [(8, 240), (64, 2304), (12288, 4080)])
@pytest.mark.parametrize("entry", ["gemv", "gemv_tail", "list", "grouped", "batched_1", "batched_3", "batched_7", "decode_gemv"])
def test_product_behind_packing(tt, N, K, entry):
    B = K // 24
    table = tt.tetra_build_table(synth.DEFAULT_GAIN)
    codes = [random_bytes(91 + i, N, B, 6) for i in range(2)]
    packed = torch.empty(tt.tetra_codes_bytes(N, B), dtype=torch.uint8, device="cuda")
    V = int(entry[8:]) if entry.startswith("batched") else 1
    rs, x = torch.rand(N, device="cuda"), halves(93, V, K)
    y = torch.zeros((V, N), dtype=torch.float32, device="cuda")
    item = dict(codes=packed, row_scales=rs, x=x[0], tail=None, y=y[0], N=N, K=K)
    problems = tt.make_problems([item])
    outputs = [y]
    if entry == "grouped":
        ws = torch.empty(tt.tetra_grouped_workspace_bytes(problems), dtype=torch.uint8, device="cuda")
        tt.tetra_gemv_grouped_plan(problems, ws)
    if entry.startswith("batched"):
        ws = torch.empty(tt.tetra_batched_workspace_bytes(N, K), dtype=torch.uint8, device="cuda")
    if entry == "decode_gemv":  # a kernel that releases its dependents early stands between the two
        coords = torch.zeros((N, B, 24), dtype=torch.int8, device="cuda")
        outputs.append(coords)

    def product():
        if entry == "gemv":
            tt.tetra_gemv(packed, rs, table, x, y, N, K)
        elif entry == "gemv_tail":
            tt.tetra_gemv_tail(packed, rs, table, x, y, N, K)
        elif entry == "list":
            tt.tetra_gemv_list(problems, table)
        elif entry == "grouped":
            tt.tetra_gemv_grouped_run(ws, table)
        elif entry == "decode_gemv":
            assert tt.lib().tetra_decode_packed(tt._ptr(packed), tt._ptr(table), tt._ptr(coords), None, N, B, tt._stream()) == 0
            tt.tetra_gemv(packed, rs, table, x, y, N, K)
        else:
            tt.tetra_gemv_batched(packed, rs, table, x, y, N, K, V, None, ws)

    check(lambda i: tt.tetra_pack_codes(codes[i], table, N, B, packed), [product], outputs)


@pytest.mark.parametrize("N,K,G", [(32, 256, 64), (1024, 4096, 128), (12288, 4096, 128), (30000, 4096, 64)])
def test_q4_product_behind_packing(tt, N, K, G):
    nbytes = tt.tetra_q4_packed_bytes(N, K, G)
    packed = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    source = [(random_bytes(95 + i, N, K // 2), halves(97 + i, N, K // G).abs(), halves(99 + i, N, K // G)) for i in range(2)]
    x = halves(94, 3, K)
    y = torch.zeros((3, N), dtype=torch.float32, device="cuda")
    ids = torch.randint(0, N, (33,), dtype=torch.int32, device="cuda")
    rows = torch.zeros((33, K), dtype=torch.float16, device="cuda")
    plan = tt.tetra_q4_list_plan(tt.make_q4_problems([dict(packed=packed, x=x[0], y=y[0], N=N, K=K)]), G)

    def pack(i):
        q, scale, offset = source[i]
        p = tt._ptr
        assert tt.lib().tetra_q4_pack(p(q), p(scale), p(offset), p(packed), nbytes, N, K, G, tt._stream()) == 0

    def behind_rows():  # a kernel that releases its dependents early stands between the two
        tt.tetra_q4_rows(packed, ids, rows, N, K, G)
        tt.tetra_q4_gemv(packed, x, y, N, K, G, 3)

    check(pack, [lambda: tt.tetra_q4_gemv(packed, x, y, N, K, G, 3), lambda: tt.tetra_q4_gemv(packed, x, y, N, K, G, 1),
                 lambda: tt.tetra_q4_list_run(plan, G), lambda: tt.tetra_q4_rows(packed, ids, rows, N, K, G), behind_rows],
          [y, rows])
