"""The work that is measured: sorts as a program that uses this package calls them.

Every pass puts fresh input into the program's working buffers (the sorts work
in place) and sorts it through a public entry point, with the workspace and
the alternate buffers that such a program keeps.  Sizes are those of the
package's own benchmark and tests (2^20, 2^26 and 2^27 elements, 20,000
segments, the lengths around the one-CTA and one-cluster forms) and ragged
ones between them.
"""
import torch

from paper_1511_03404_gb300 import rs

# name -> (storage dtype, key kind, bytes)
KEYS = {
    "u32": (torch.int32, rs.RS_KEY_UNSIGNED, 4),
    "i32": (torch.int32, rs.RS_KEY_SIGNED, 4),
    "f32": (torch.float32, rs.RS_KEY_FLOAT, 4),
    "u64": (torch.int64, rs.RS_KEY_UNSIGNED, 8),
    "i64": (torch.int64, rs.RS_KEY_SIGNED, 8),
    "f64": (torch.float64, rs.RS_KEY_FLOAT, 8),
}


def listed():
    return [
        # the smallest call: ranking a few thousand scores, best first; latency and launches
        dict(name="keys_f32_desc_3k", kind="sort", key="f32", pairs=False, n=3000,
             dist="gaussian", descending=True),
        # a small pair sort, as one step of a larger program
        dict(name="pairs_u32_50k", kind="sort", key="u32", pairs=True, n=50000, dist="uniform"),
        # time stamps with row numbers, a few hundred thousand of them
        dict(name="pairs_i64_300k", kind="sort", key="i64", pairs=True, n=300007,
             dist="gaussian"),
        # the benchmark's array that stays in the L2: launches and latency beside the passes
        dict(name="keys_u32_1m", kind="sort", key="u32", pairs=False, n=1 << 20, dist="uniform"),
        # particles by cell number: 20 of the 32 key bits, an odd pass count, a ragged length
        dict(name="pairs_u32_20bit_10m", kind="sort", key="u32", pairs=True, n=10000019,
             dist="uniform", end=20),
        # the headline: 2^26 pairs of 32-bit key and value
        dict(name="pairs_u32_2p26", kind="sort", key="u32", pairs=True, n=1 << 26,
             dist="uniform"),
        # the largest: 2^27 64-bit keys
        dict(name="keys_u64_2p27", kind="sort", key="u64", pairs=False, n=1 << 27,
             dist="uniform"),
        # 64-bit floats with row numbers, ragged length
        dict(name="pairs_f64_30m", kind="sort", key="f64", pairs=True, n=30000001,
             dist="gaussian"),
        # the batched workload: 20,000 segments, lengths log-uniform over six decades
        dict(name="seg_pairs_u32_20k", kind="segmented", key="u32", pairs=True, n=1 << 26,
             segments=20000, lengths="log"),
        # many short rows (posting lists, candidate lists), keys only
        dict(name="seg_keys_u32_rows", kind="segmented", key="u32", pairs=False, n=15000000,
             segments=10000, lengths="even"),
        # comparison keys the digit passes do not take: 128 bits with a 64-bit payload
        dict(name="merge_u128_4m", kind="merge", n=4000037),
        # from pinned host memory and back in one call
        dict(name="host_pairs_u32_4m", kind="host", key="u32", pairs=True, n=4000003,
             dist="uniform"),
    ]


def _log_n(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random())) | rng.randrange(2)


def draw(rng):
    kind = rng.choice(["sort"] * 5 + ["segmented"] * 2 + ["merge", "host"])
    if kind == "merge":
        return dict(kind=kind, n=_log_n(rng, 1 << 18, 1 << 23))
    if kind == "segmented":
        segments = _log_n(rng, 100, 20000)
        return dict(kind=kind, key=rng.choice(["u32", "u64"]), pairs=rng.random() < 0.5,
                    n=max(_log_n(rng, 1 << 20, 1 << 26), 2 * segments), segments=segments,
                    lengths=rng.choice(["log", "even"]))
    key = rng.choice(sorted(KEYS))
    c = dict(kind=kind, key=key, pairs=rng.random() < 0.5,
             n=_log_n(rng, 1 << 20, 1 << 23) if kind == "host" else _log_n(rng, 1000, 1 << 26),
             dist=rng.choice(["uniform", "uniform", "gaussian", "low16", "sorted"]))
    if kind == "sort":
        c["descending"] = rng.random() < 0.25
        if key in ("u32", "u64") and rng.random() < 0.25:
            c["end"] = rng.randrange(9, 8 * KEYS[key][2])
    return c


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _keys(name, n, dist, g):
    dtype, _, nb = KEYS[name]
    if dtype.is_floating_point:
        if dist == "gaussian":
            k = torch.randn(n, generator=g, device="cuda", dtype=dtype)
        elif dist == "low16":
            k = torch.randint(0, 1 << 16, (n,), generator=g, device="cuda").to(dtype)
        else:
            k = torch.rand(n, generator=g, device="cuda", dtype=dtype)
        return torch.sort(k)[0] if dist == "sorted" else k
    bits = 8 * nb

    def raw():
        return torch.randint(-(1 << (bits - 1)), (1 << (bits - 1)) - 1, (n,), generator=g,
                             device="cuda", dtype=dtype)

    if dist == "gaussian":  # the mean of four draws
        k = raw() // 4
        for _ in range(3):
            k += raw() // 4
        return k
    if dist == "low16":
        return raw() & 0xFFFF
    k = raw()
    return torch.sort(k)[0] if dist == "sorted" else k


def _offsets(case, g):
    """n_seg + 1 segment bounds; the lengths follow the case's law and add up to n."""
    s, n = case["segments"], case["n"]
    u = torch.rand(s, generator=g, device="cuda", dtype=torch.float64)
    ln = torch.exp2(20.0 * u) if case["lengths"] == "log" else 1.0 + 2999.0 * u
    end = torch.floor(torch.cumsum(ln, 0) * (n / float(ln.sum()))).to(torch.int64).clamp_(0, n)
    end[-1] = n
    return torch.cat([torch.zeros(1, dtype=torch.int64, device="cuda"), end])


def _end(case):
    return case.get("end") or 8 * KEYS[case["key"]][2]


def _index(n, nb):
    return torch.arange(n, device="cuda", dtype=torch.int32 if nb == 4 else torch.int64)


def prepare(case, seed):
    g, n = _gen(seed), case["n"]
    st = {"case": dict(case)}
    if case["kind"] == "merge":
        # 128-bit keys as two little-endian words; many share the upper one
        lo = torch.randint(-(1 << 63), (1 << 63) - 1, (n,), generator=g, device="cuda")
        hi = torch.randint(0, 1 << 12, (n,), generator=g, device="cuda")
        st["src"] = torch.stack([lo, hi], 1).contiguous()
        st["vsrc"] = _index(n, 8)
        err, need = rs.rs_merge_workspace_bytes(16, 8, n)
        rs.check(err, "rs_merge_workspace_bytes")
        st["ws"] = torch.empty(max(need, 256), dtype=torch.uint8, device="cuda")
        st["buf"] = [torch.empty_like(st["src"]) for _ in range(2)]
        st["vbuf"] = [torch.empty_like(st["vsrc"]) for _ in range(2)]
        return st
    _, _, nb = KEYS[case["key"]]
    vb = nb if case["pairs"] else 0
    st["src"] = _keys(case["key"], n, case.get("dist", "uniform"), g)
    st["vsrc"] = _index(n, nb) if vb else None
    st["buf"] = torch.empty_like(st["src"])
    st["vbuf"] = torch.empty_like(st["vsrc"]) if vb else None
    if case["kind"] == "segmented":
        st["off"] = _offsets(case, g)
        err, need = rs.rs_segmented_workspace_bytes_typed(nb, vb, n, case["segments"])
        rs.check(err, "rs_segmented_workspace_bytes_typed")
        st["ws"] = torch.empty(max(need, 256), dtype=torch.uint8, device="cuda")
        return st
    st["ws"] = rs.workspace(nb, vb, n, 0, _end(case))
    st["alt"] = (torch.empty_like(st["buf"]), torch.empty_like(st["vbuf"]) if vb else None)
    if case["kind"] == "host":
        st["src"] = st["src"].cpu().pin_memory()
        st["vsrc"] = st["vsrc"].cpu().pin_memory() if vb else None
        st["out"] = torch.empty_like(st["src"]).pin_memory()
        st["vout"] = torch.empty_like(st["vsrc"]).pin_memory() if vb else None
    return st


def _ptr(t):
    return None if t is None else t.data_ptr()


def run(st):
    case, ws = st["case"], st["ws"]
    kind, n = case["kind"], case["n"]
    stream = torch.cuda.current_stream().cuda_stream
    if kind == "host":
        _, key_kind, nb = KEYS[case["key"]]
        err, _ = rs.rs_sort_host(nb, nb if case["pairs"] else 0, _ptr(st["src"]),
                                 _ptr(st["vsrc"]), _ptr(st["out"]), _ptr(st["vout"]), n, 0,
                                 8 * nb, _ptr(st["buf"]), _ptr(st["vbuf"]), _ptr(st["alt"][0]),
                                 _ptr(st["alt"][1]), _ptr(ws), ws.numel(), stream,
                                 key_kind=key_kind)
        rs.check(err, "rs_sort_host")
        return [st["out"], st["vout"]] if case["pairs"] else st["out"]
    if kind == "merge":
        k, v = st["buf"], st["vbuf"]
        k[0].copy_(st["src"])
        v[0].copy_(st["vsrc"])
        err, alt = rs.rs_merge_sort(16, 8, _ptr(k[0]), _ptr(v[0]), _ptr(k[1]), _ptr(v[1]), n,
                                    _ptr(ws), ws.numel(), stream)
        rs.check(err, "rs_merge_sort")
        return [k[alt], v[alt]]
    keys, vals = st["buf"], st["vbuf"]
    keys.copy_(st["src"])
    if vals is not None:
        vals.copy_(st["vsrc"])
    if kind == "segmented":
        rs.segmented_sort(keys, st["off"], vals, ws=ws)
    else:
        rs.sort(keys, vals, 0, _end(case), ws=ws, alt=st["alt"],
                descending=case.get("descending", False), key_kind=KEYS[case["key"]][1])
    return keys if vals is None else [keys, vals]


def work(case):
    nb = 24 if case["kind"] == "merge" else KEYS[case["key"]][2] * (2 if case["pairs"] else 1)
    return {"bytes": 2 * case["n"] * nb, "flops": 0}


def tolerance(case):
    return "exact"  # keys and values are moved, never computed


def _order(bits, kind, descending):
    """Signed integers that ascend in the order of the keys whose bit patterns these are."""
    top = torch.iinfo(bits.dtype).min
    if kind == rs.RS_KEY_UNSIGNED:
        bits = bits ^ top
    elif kind == rs.RS_KEY_FLOAT:
        bits = torch.where(bits < 0, ~(bits ^ top), bits)
    return ~bits if descending else bits


def exact(case, seed):
    g, n = _gen(seed), case["n"]
    if case["kind"] == "merge":
        lo = torch.randint(-(1 << 63), (1 << 63) - 1, (n,), generator=g, device="cuda")
        hi = torch.randint(0, 1 << 12, (n,), generator=g, device="cuda")
        at = torch.sort(_order(lo, rs.RS_KEY_UNSIGNED, False), stable=True)[1]
        at = at[torch.sort(hi[at], stable=True)[1]]
        return [torch.stack([lo[at], hi[at]], 1), at]
    _, kind, nb = KEYS[case["key"]]
    k = _keys(case["key"], n, case.get("dist", "uniform"), g)
    bits = k.view(torch.int32 if nb == 4 else torch.int64)
    if case["kind"] == "segmented":
        off = _offsets(case, g)
        at = torch.sort(_order(bits, rs.RS_KEY_UNSIGNED, False), stable=True)[1]
        seg = torch.searchsorted(off[1:].contiguous(), at, right=True)
        at = at[torch.sort(seg, stable=True)[1]]
    else:
        o = _order(bits, kind, case.get("descending", False))
        if _end(case) < 8 * nb:  # the sorted bits alone, still unsigned
            o = o & ((1 << _end(case)) - 1)
        at = torch.sort(o, stable=True)[1]
    out = k[at].double() if k.dtype.is_floating_point else k[at]
    if case["kind"] == "host":
        out, at = out.cpu(), at.cpu()
    return [out, at.to(torch.int32 if nb == 4 else torch.int64)] if case["pairs"] else out
