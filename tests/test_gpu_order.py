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


# Writes n 16-byte pieces to `to`, but lets the next kernel of the stream start first and waits for about 50 us (a bounded number of
# turns) before it does.
LATE_COPY = """
extern "C" __global__ void late_copy(const uint4* from, uint4* to, int n) {
    asm volatile("griddepcontrol.launch_dependents;");
    const long long begin = clock64();
    for (int turn = 0; turn < 1000000 && clock64() - begin < 100000; ++turn) {}
    for (int i = threadIdx.x; i < n; i += blockDim.x) to[i] = from[i];
}
"""


@pytest.mark.parametrize("shapes", [[(64, 24 * 40)], [(4096, 24 * 42 + 5), (17, 24 * 33 + 5), (3001, 24 * 32)]])
def test_run_behind_a_kernel_that_writes_the_plan_late(tt, shapes):
    """Nothing of a plan is read before the kernel that writes it is complete.  The plan that lies there before is of the same shapes,
    with other matrices, inputs and outputs, all of them valid: a word read too early is only a wrong number.  (That the run's second
    kernel, which reads the plan ahead of its own wait, is let go only behind the first one's does not show in a run: it finds no
    registers beside the first.  test_launch_order_source.py reads it from the source.)"""
    table = tt.tetra_build_table(synth.DEFAULT_GAIN)
    late_copy = torch.cuda._compile_kernel(LATE_COPY, "late_copy")
    held, plans, outputs, want = [], [], [], []
    for which in range(2):
        items = []
        for i, (N, K) in enumerate(shapes):
            seed = 1000 * which + 10 * i
            packed = tt.tetra_pack_codes(random_bytes(seed, N, K // 24, 6), table, N, K // 24)
            items.append(dict(codes=packed, row_scales=torch.rand(N, device="cuda"), x=halves(seed + 1, K), N=N, K=K,
                              tail=halves(seed + 2, N, K % 24) if K % 24 else None, y=torch.zeros(N, device="cuda")))
        problems = tt.make_problems(items)
        ws = torch.zeros(-(-tt.tetra_grouped_workspace_bytes(problems) // 16) * 16, dtype=torch.uint8, device="cuda")
        tt.tetra_gemv_grouped_plan(problems, ws)
        held.append(items)
        plans.append(ws)
        outputs.append([it["y"] for it in items])
    for ws, ys in zip(plans, outputs):
        other = ws.clone()
        tt.tetra_gemv_grouped_run(other, table)
        torch.cuda.synchronize()
        want.append([y.clone() for y in ys])
    shared = plans[0].clone()
    for turn in range(1, 9):
        which = turn % 2
        for ys in outputs:
            for y in ys:
                y.fill_(-1.0)
        torch.cuda.synchronize()
        late_copy(grid=(1, 1, 1), block=(1024, 1, 1), args=[plans[which], shared, plans[which].numel() // 16])
        tt.tetra_gemv_grouped_run(shared, table)
        torch.cuda.synchronize()
        assert all(torch.equal(y, w) for y, w in zip(outputs[which], want[which])), turn
        assert all(bool((y == -1.0).all()) for y in outputs[1 - which]), turn
