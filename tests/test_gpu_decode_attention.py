"""Split-KV attention of a few new rows per sequence (dmtd_attention_decode) where its key shares, pieces and tiles
end, against softmax(Q K^T / sqrt(d)) V in fp64."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dmtd():
    import paper_2510_11958_b200 as pkg
    pkg.load_library()
    return pkg


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("B,R,nq,nkv,n_keys", [
    (1, 1, 8, 2, 1),            # one key
    (1, 1, 8, 2, 16),           # one warp's tile
    (1, 3, 8, 2, 65),           # one key in the second unit, 12 query rows
    (1, 1, 32, 8, 1000),        # fewer units than blocks
    (2, 4, 8, 2, 129),          # 16 query rows
    (3, 5, 8, 2, 200),          # two row blocks
    (1, 1, 16, 1, 4097),        # one item, many pieces
    (5, 2, 32, 8, 777),         # shares that cross item boundaries
    (40, 1, 32, 8, 333),        # more items than blocks
    (37, 3, 8, 8, 70),          # one query head per kv head
    (150, 1, 8, 2, 515),
])
def test_attention_decode_pieces(dmtd, dtype, B, R, nq, nkv, n_keys):
    D, G, pos0 = 128, nq // nkv, n_keys - R
    g = torch.Generator(device="cuda").manual_seed(11)
    q = torch.randn(B, R, nq, D, generator=g, device="cuda") * 2
    k, v = (torch.randn(B, nkv, n_keys + 3, D, generator=g, device="cuda").to(dtype) for _ in range(2))
    k[:, :, n_keys:] = float("nan")                          # nothing behind the last key may be used
    v[:, :, n_keys:] = float("nan")
    out = dmtd.attention_decode(q, k, v, pos0)
    kd, vd = (x[:, :, :n_keys].double().repeat_interleave(G, 1) for x in (k, v))
    s = torch.einsum("brhd,bhkd->bhrk", q.double(), kd) / D ** 0.5
    hidden = torch.arange(n_keys, device="cuda")[None] > (pos0 + torch.arange(R, device="cuda"))[:, None]
    p = torch.softmax(s.masked_fill(hidden, float("-inf")), -1)
    ref = torch.einsum("bhrk,bhkd->brhd", p, vd)
    # the query is rounded once (relative 2^-9 or 2^-12, which moves a score of size |s| by as much) and the
    # probabilities once; |s| stays below 12 here
    u = 2.0 ** -9 if dtype == torch.bfloat16 else 2.0 ** -12
    err = (out.double() - ref).abs().max().item()
    assert err <= 4 * u * max(1.0, ref.abs().max().item()), err


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("R,n_keys", [(1, 1000), (4, 1000), (1, 8000), (4, 2052)])
def test_largest_probability_of_a_tile_is_not_rounded(dmtd, dtype, R, n_keys):
    """Every 16 keys one that counts, with a value of its own: its weight carries no 16-bit rounding, whatever number of
    tiles a warp walks."""
    nq, nkv, D, pos0 = 32, 8, 128, n_keys - R
    g = torch.Generator(device="cuda").manual_seed(13)
    q = torch.zeros(1, R, nq, D, device="cuda")              # exact in 16 bits once it is scaled by 1 / sqrt(D)
    q[..., 0] = torch.tensor([1.0, -1.0, 0.5, -0.75], device="cuda").repeat(nkv)
    q[..., 1] = 1.0
    k, v = (torch.zeros(1, nkv, n_keys, D, device="cuda") for _ in range(2))
    tiles = n_keys // 16
    k[..., 1] = -40.0                                        # exp(-40): below the bound
    k[:, :, :tiles * 16:16, 1] = 0.0
    k[:, :, :tiles * 16:16, 0] = torch.randint(-96, 97, (1, nkv, tiles), generator=g, device="cuda") / 64.0
    t = torch.arange(tiles, device="cuda")
    v[:, :, t * 16, t % D] = 1.0
    out = dmtd.attention_decode(q * D ** 0.5, k.to(dtype), v.to(dtype), pos0)
    s = torch.einsum("brhd,bhkd->bhrk", q.double(), k.double().repeat_interleave(nq // nkv, 1))
    hidden = torch.arange(n_keys, device="cuda")[None] > (pos0 + torch.arange(R, device="cuda"))[:, None]
    p = torch.softmax(s.masked_fill(hidden, float("-inf")), -1)
    ref = torch.einsum("bhrk,bhkd->brhd", p, v.double().repeat_interleave(nq // nkv, 1))
    seen = ref > 1e-12
    # fp32: exponentials of at most 4 to 2^-21 or two, a factor of as much per tile of a warp's chain (8000 keys: 16)
    assert ((out.double() - ref).abs() / ref)[seen].max() <= 2e-5


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
@pytest.mark.parametrize("R,n_keys", [(1, 40), (3, 1000)])
def test_results_off_a_16_byte_boundary(dmtd, dtype, R, n_keys):
    """q and out are float arrays of the caller: views into larger buffers begin at any float."""
    B, nq, nkv, D, pos0 = 2, 8, 2, 128, n_keys - R
    g = torch.Generator(device="cuda").manual_seed(14)
    k, v = (torch.randn(B, nkv, n_keys, D, generator=g, device="cuda").to(dtype) for _ in range(2))
    n = B * R * nq * D
    q_room = torch.randn(n + 8, generator=g, device="cuda")
    want = dmtd.attention_decode(q_room[:n].reshape(B, R, nq, D), k, v, pos0)
    dll, code = dmtd.load_library(), {torch.float16: 2, torch.bfloat16: 1}[dtype]
    scratch = torch.empty(dll.dmtd_attention_scratch_bytes(B, R, nq, D, n_keys), dtype=torch.uint8, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream
    u = 2.0 ** -9 if dtype == torch.bfloat16 else 2.0 ** -12            # the probabilities' rounding, on both sides
    for off in (1, 2, 3):
        q = torch.empty(n + 8, device="cuda")[off:off + n].view(B, R, nq, D).copy_(q_room[:n].view(B, R, nq, D))
        room = torch.full((2, n + 8), 7.0, device="cuda")
        dmtd.attention_decode_static(q, k, v, pos0, room[0, off:off + n].view(B, R, nq, D))
        out = room[1, off:off + n]
        assert dll.dmtd_attention_decode(q.data_ptr(), k.data_ptr(), v.data_ptr(), code, B, R, nq, nkv, D, n_keys, pos0,
                                         scratch.data_ptr(), scratch.numel(), out.data_ptr(), stream) == 0
        for row in room:
            assert (row[off:off + n].view_as(want) - want).abs().max() <= 4 * u * max(1.0, want.abs().max().item())
            assert (row[:off] == 7.0).all() and (row[off + n:] == 7.0).all()


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16, torch.float32])
@pytest.mark.parametrize("B,R,nq,nkv,n_keys", [
    (1, 1, 4, 2, 1),            # one key
    (1, 4, 16, 4, 2300),        # 16 query rows, 36 slices x 4 heads: 144 blocks
    (1, 4, 16, 4, 2400),        # 152 blocks: more than one to an SM
    (2, 1, 16, 2, 4100),        # 8 query rows, slices of 64 keys, two blocks to an SM and a few more
    (3, 300, 8, 8, 310),        # many row blocks, the last of 12 rows
    (2, 40, 16, 1, 129),        # 16 query heads per kv head
])
def test_attention_head_dim_64(dmtd, dtype, B, R, nq, nkv, n_keys):
    D, G, pos0 = 64, nq // nkv, n_keys - R
    g = torch.Generator(device="cuda").manual_seed(12)
    q = torch.randn(B, R, nq, D, generator=g, device="cuda") * 2
    k, v = (torch.randn(B, nkv, n_keys + 3, D, generator=g, device="cuda").to(dtype) for _ in range(2))
    k[:, :, n_keys:] = float("nan")                          # nothing behind the last key may be used
    v[:, :, n_keys:] = float("nan")
    out = dmtd.attention_decode(q, k, v, pos0)
    for b in range(B):
        kd, vd = (x[b, :, :n_keys].double().repeat_interleave(G, 0) for x in (k, v))
        s = torch.einsum("rhd,hkd->hrk", q[b].double(), kd) / D ** 0.5
        hidden = torch.arange(n_keys, device="cuda")[None] > (pos0 + torch.arange(R, device="cuda"))[:, None]
        ref = torch.einsum("hrk,hkd->rhd", torch.softmax(s.masked_fill(hidden, float("-inf")), -1), vd)
        # fp32 throughout: scores of size below 16 to 2^-20, the exponential's two units in the last place
        assert (out[b].double() - ref).abs().max() <= 2e-5 * max(1.0, ref.abs().max().item())
