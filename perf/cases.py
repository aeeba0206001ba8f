"""The work that programs have this library do, as timed cases.

Each case is one call (or one submit-and-drain of the server) through the
public entry points of ``paper_1902_05234_gb300.aesgb``, at the sizes of this
repository's own workloads: the files of the paper's tables (1,202 to 1,190,402
bytes), the single-buffer sweep (1 MiB to 1 GiB), the batch of 4,096 messages of
16 B to 16 MiB with mixed keys and directions, the served request stream of 64 B
to 4 MiB over 1,024 resident keys, the chained and counter modes, the
constant-time cipher and ECB on page-locked host buffers.  Launch
configurations are the library's defaults (no tuning run), as a program gets
them that calls the library without further set-up.

A case is a dict:
  kind      ecb, ctr, cbc, cfb (decryption), ct (constant-time ECB), host (ECB
            on page-locked host memory), batch (aes_ecb_batch), serve (aes_srv_*)
  keybits   128, 192 or 256 (batch and serve: drawn per key from the three)
  dir       0 encrypt, 1 decrypt (ecb, ct, host; batch and serve draw it)
  blocks    16-byte blocks in the buffer (single-buffer kinds)
  inplace   ecb: output over the input
  staged    host: through a device staging buffer instead of directly
  messages, lo, hi, keys   batch and serve: number of messages, range of their
            log-uniform lengths in bytes, number of distinct keys

Inputs are uniform random bytes: the kernels' work does not depend on the data.
Outputs are bytes and have to be exact.
"""
import ctypes
import math

import numpy as np
import torch

from paper_1902_05234_gb300 import aesgb

SERVE_BUDGET = 4 << 30  # bytes in flight, as the served workload sets it
SERVE_SLOTS = 4
STAGING_BYTES = 96 << 20


def listed():
    return [
        # one short message under one key: the paper's 4,652-byte file in whole
        # blocks; call latency is all there is
        {"name": "ecb enc 128, 4.5 KiB", "kind": "ecb", "keybits": 128, "dir": 0, "blocks": 290, "inplace": False},
        # a mid-size buffer decrypted in place, a ragged 16 MiB
        {"name": "ecb dec 256 in place, 16 MiB+", "kind": "ecb", "keybits": 256, "dir": 1, "blocks": 1048583,
         "inplace": True},
        # bulk encryption: the headline size
        {"name": "ecb enc 128, 1 GiB", "kind": "ecb", "keybits": 128, "dir": 0, "blocks": 1 << 26, "inplace": False},
        # the paper's largest file under CTR, about 1 MiB
        {"name": "ctr 128, 1.1 MiB", "kind": "ctr", "keybits": 128, "dir": 0, "blocks": 74400},
        # bulk CTR
        {"name": "ctr 256, 256 MiB", "kind": "ctr", "keybits": 256, "dir": 0, "blocks": 1 << 24},
        # a chained mode's parallel direction on a mid-size, ragged buffer
        {"name": "cbc dec 192, 4 MiB+", "kind": "cbc", "keybits": 192, "dir": 1, "blocks": 262147},
        # data that starts and ends in host memory
        {"name": "host enc 128, 64 MiB", "kind": "host", "keybits": 128, "dir": 0, "blocks": 1 << 22,
         "staged": False},
        # many messages of very different sizes, a key, a key size and a
        # direction each, in one launch
        {"name": "batch 4096 x 16 B..16 MiB", "kind": "batch", "messages": 4096, "lo": 16, "hi": 16 << 20,
         "keys": 4096},
        # many short records (packets, rows, pages) over a set of session keys
        {"name": "batch 20000 x 16 B..16 KiB", "kind": "batch", "messages": 20000, "lo": 16, "hi": 16 << 10,
         "keys": 1024},
        # a burst of requests through the server
        {"name": "serve 2000 x 64 B..4 MiB", "kind": "serve", "messages": 2000, "lo": 64, "hi": 4 << 20,
         "keys": 1024},
        # the table-free cipher on an ordinary and on a bulk buffer
        {"name": "ct enc 128, 1 MiB", "kind": "ct", "keybits": 128, "dir": 0, "blocks": 1 << 16},
        {"name": "ct dec 256, 256 MiB", "kind": "ct", "keybits": 256, "dir": 1, "blocks": 1 << 24},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["ecb", "ecb", "ctr", "cbc", "cfb", "ct", "host", "batch", "batch", "serve"])
    if kind in ("batch", "serve"):
        # messages from 16 B up, fewer of them where they may be long, so that
        # the whole stays below the largest listed batch
        hi = _log_int(rng, 256, 16 << 20 if kind == "batch" else 4 << 20) // 16 * 16
        most = min(30000 if kind == "batch" else 4000, (2 << 30) // hi * 4)
        return {"kind": kind, "messages": _log_int(rng, 1 if kind == "serve" else 4, most),
                "lo": 16 if kind == "batch" else 64, "hi": hi, "keys": rng.choice([1, 64, 1024])}
    c = {"kind": kind, "keybits": rng.choice([128, 192, 256]),
         "dir": {"ctr": 0, "cbc": 1, "cfb": 1}.get(kind, rng.randrange(2))}
    c["blocks"] = _log_int(rng, 1, {"ct": 1 << 24, "host": 1 << 22}.get(kind, 1 << 26))
    if kind == "ecb":
        c["inplace"] = rng.random() < 0.5
    if kind == "host":
        c["staged"] = rng.random() < 0.5
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _bytes_on_gpu(n, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))
    # whole words are drawn: four bytes at a time
    words = torch.randint(-(1 << 31), 1 << 31, ((n + 3) // 4,), generator=g, device="cuda", dtype=torch.int32)
    return words.view(torch.uint8)[:n]


def _small(case, seed):
    """Host-side random parts of a case: keys, the counter block / IV, and for
    batch and serve the messages' lengths, keys and directions.  The lengths are
    the same set for every seed, in an order of the seed's own, so that a case
    is always the same number of bytes."""
    r = np.random.Generator(np.random.PCG64([int(seed), 190205234]))
    s = {}
    if case["kind"] in ("batch", "serve"):
        n = case["messages"]
        lengths = np.random.Generator(np.random.PCG64([n, case["lo"], case["hi"]]))
        u = lengths.uniform(math.log(case["lo"]), math.log(case["hi"]), n)
        s["blocks"] = r.permutation(np.maximum(1, np.floor(np.exp(u) / 16)).astype(np.int64))
        s["dirs"] = r.integers(0, 2, n)
        s["keybits"] = r.choice(np.array([128, 192, 256]), case["keys"])
        s["keys"] = [r.integers(0, 256, int(kb) // 8, dtype=np.uint8) for kb in s["keybits"]]
        s["key_ids"] = np.arange(n) if case["keys"] == n else r.integers(0, case["keys"], n)
    else:
        s["key"] = r.integers(0, 256, case["keybits"] // 8, dtype=np.uint8)
        s["iv"] = r.integers(0, 256, 16, dtype=np.uint8)
    return s


class _Server:
    """A server handle that ends with the state that holds it."""

    def __init__(self, keys):
        self.handle = aesgb.aes_srv_create(SERVE_BUDGET, max(1, len(keys)), 4096, SERVE_SLOTS)
        for i, k in enumerate(keys):
            aesgb.aes_srv_put_key(self.handle, i, 8 * k.size, k.tobytes())

    def __del__(self):
        if self.handle:
            aesgb.aes_srv_destroy(self.handle)
            self.handle = None


def prepare(case, seed):
    kind, small = case["kind"], _small(case, seed)
    st = {"kind": kind, "case": case}
    if kind in ("batch", "serve"):
        offs = np.zeros(case["messages"] + 1, np.int64)
        np.cumsum(16 * small["blocks"], out=offs[1:])
        st["in"] = _bytes_on_gpu(int(offs[-1]), seed)
        st["out"] = torch.empty_like(st["in"])
        ins = st["in"].data_ptr() + offs[:-1].astype(np.uint64)
        outs = st["out"].data_ptr() + offs[:-1].astype(np.uint64)
        if kind == "serve":
            st["srv"] = _Server(small["keys"])
            st["req"] = (small["key_ids"].astype(np.int32), small["dirs"].astype(np.int32), ins, outs,
                         (16 * small["blocks"]).astype(np.uint64))
            return st
        # expanded keys on the device: encryption schedules, then decryption ones
        nk = case["keys"]
        rks = np.zeros((2, nk, 64), np.uint32)
        nrs = np.zeros(nk, np.int64)
        for i, k in enumerate(small["keys"]):
            rks[0, i, :60], rks[1, i, :60], nrs[i] = aesgb.aes_expand_key(8 * k.size, k)
        st["rk"] = torch.from_numpy(rks.view(np.uint8).reshape(-1)).cuda()
        rk = st["rk"].data_ptr() + 256 * (small["dirs"] * nk + small["key_ids"]).astype(np.uint64)
        table = aesgb.pack_descs(rk, ins, outs, small["blocks"], nrs[small["key_ids"]], small["dirs"])
        st["desc"] = torch.from_numpy(table.view(np.uint8)).cuda()
        return st
    n = 16 * case["blocks"]
    enc, dec, st["nr"] = aesgb.aes_expand_key(case["keybits"], small["key"])
    # CBC decrypts with the inverse cipher; CTR and CFB run the forward one
    st["rk"] = dec if kind == "cbc" or (kind in ("ecb", "ct", "host") and case["dir"] == 1) else enc
    st["iv"] = small["iv"]
    data = _bytes_on_gpu(n, seed)
    if kind == "host":
        st["in"] = torch.empty(n, dtype=torch.uint8, pin_memory=True)
        st["in"].copy_(data)
        st["out"] = torch.empty(n, dtype=torch.uint8, pin_memory=True)
        if case["staged"]:
            st["staging"] = torch.empty(STAGING_BYTES, dtype=torch.uint8, device="cuda")
    else:
        st["in"] = data
        st["out"] = data if case.get("inplace") else torch.empty_like(data)
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(st):
    kind, case = st["kind"], st["case"]
    if kind == "batch":
        aesgb.aes_ecb_batch(st["desc"], case["messages"])
        return st["out"]
    if kind == "serve":
        srv = st["srv"].handle
        code, tickets = aesgb.aes_srv_submit_many(srv, *st["req"])
        if code < 0:
            raise aesgb.AesError(code, "submit")
        aesgb.aes_srv_drain(srv, 60000)
        status, _, _ = aesgb.aes_srv_results(srv, tickets, release=True)
        return {"out": st["out"], "status": status}
    rk, nr, x, y, n = st["rk"], st["nr"], st["in"], st["out"], case["blocks"]
    if kind == "ecb":
        (aesgb.aes_ecb_encrypt if case["dir"] == 0 else aesgb.aes_ecb_decrypt)(rk, nr, x, y, n)
    elif kind == "ctr":
        aesgb.aes_ctr_crypt(rk, nr, st["iv"], x, y, n)
    elif kind == "cbc":
        aesgb.aes_cbc_decrypt(rk, nr, st["iv"], x, y, n)
    elif kind == "cfb":
        aesgb.aes_cfb_decrypt(rk, nr, st["iv"], x, y, n)
    elif kind == "ct":
        aesgb.aes_ecb_crypt_ct(case["dir"], rk, nr, x, y, n)
    elif case["staged"]:
        aesgb.aes_ecb_host(case["dir"], rk, nr, x, y, n, st["staging"], STAGING_BYTES)
    else:
        aesgb.aes_ecb_host_direct(case["dir"], rk, nr, x, y, n)
    return y


def work(case):
    """Bytes: input read once, output written once (and a batch's descriptors
    and schedules).  No floating-point operations: the cipher is table lookups
    and logic, 16 lookups per block and round."""
    if case["kind"] in ("batch", "serve"):
        lo, hi = case["lo"] / 16, case["hi"] / 16
        mean = max(1.0, (hi - lo) / math.log(hi / lo)) if hi > lo else hi  # of a log-uniform length
        return {"bytes": case["messages"] * (32.0 * mean + ctypes.sizeof(aesgb.aes_desc)) + 240.0 * case["keys"],
                "flops": 0}
    return {"bytes": 32.0 * case["blocks"], "flops": 0}


def tolerance(case):
    return "exact"


# ---------------------------------------------------------------------------
# the same results in plain torch, from the definitions of FIPS-197 and
# SP 800-38A
# ---------------------------------------------------------------------------
def _gf_mul(a, b):
    p = 0
    while b:
        p ^= a if b & 1 else 0
        a = (a << 1) ^ (0x11B if a & 0x80 else 0)
        b >>= 1
    return p


def _sbox():
    inv = [0] * 256
    for a in range(1, 256):
        inv[a] = next(b for b in range(1, 256) if _gf_mul(a, b) == 1) if not inv[a] else inv[a]
        inv[inv[a]] = a
    s = []
    for x in inv:
        y = 0x63
        for k in range(5):
            y ^= ((x << k) | (x >> (8 - k))) & 0xFF
        s.append(y)
    return s


def _expand(key, sbox):
    """Round keys of the encryption schedule, [Nr + 1, 16]."""
    nk = len(key) // 4
    nr = nk + 6
    w = [list(key[4 * i:4 * i + 4]) for i in range(nk)]
    rcon = 1
    for i in range(nk, 4 * (nr + 1)):
        t = list(w[i - 1])
        if i % nk == 0:
            t = [sbox[v] for v in t[1:] + t[:1]]
            t[0] ^= rcon
            rcon = _gf_mul(rcon, 2)
        elif nk > 6 and i % nk == 4:
            t = [sbox[v] for v in t]
        w.append([a ^ b for a, b in zip(w[i - nk], t)])
    return np.array(w, np.uint8).reshape(nr + 1, 16)


class _Plain:
    def __init__(self, device="cuda"):
        self.sbox = _sbox()
        self.device = device
        t = lambda v: torch.tensor(v, dtype=torch.uint8, device=device)  # noqa: E731
        self.s = t(self.sbox)
        self.si = t([self.sbox.index(x) for x in range(256)])
        self.mul = {k: t([_gf_mul(x, k) for x in range(256)]) for k in (2, 3, 9, 11, 13, 14)}
        rows = torch.arange(16, device=device)
        r, c = rows % 4, rows // 4
        self.shift = r + 4 * ((c + r) % 4)       # byte that ShiftRows brings to each place
        self.unshift = r + 4 * ((c - r) % 4)

    def _mix(self, x, coef):
        v = x.view(-1, 4, 4).long()              # [block, column, row]
        out = torch.zeros_like(x).view(-1, 4, 4)
        for k, f in enumerate(coef):             # row r takes coef[k] times row r + k
            y = v.roll(-k, 2)
            out ^= y.to(torch.uint8) if f == 1 else self.mul[f][y]
        return out.view(-1, 16)

    def cipher(self, x, keys, which, decrypt):
        """x: [n, 16]; keys: [number of keys, Nr + 1, 16]; which: key of each block."""
        k = (lambda i: keys[0, i]) if which is None else (lambda i: keys[which, i])
        nr = keys.shape[1] - 1
        if not decrypt:
            x = x ^ k(0)
            for i in range(1, nr + 1):
                x = self.s[x.long()][:, self.shift]
                if i < nr:
                    x = self._mix(x, (2, 3, 1, 1))
                x = x ^ k(i)
            return x
        x = x ^ k(nr)
        for i in range(nr - 1, -1, -1):
            x = self.si[x[:, self.unshift].long()] ^ k(i)
            if i:
                x = self._mix(x, (14, 11, 13, 9))
        return x

    def run(self, x, keys, which, decrypt, out):
        step = 1 << 20
        for a in range(0, x.shape[0], step):
            out[a:a + step] = self.cipher(x[a:a + step], keys, None if which is None else which[a:a + step], decrypt)


def exact(case, seed):
    p, small, kind = _Plain(), _small(case, seed), case["kind"]
    dev = p.device
    if kind in ("batch", "serve"):
        n = int(small["blocks"].sum())
        x = _bytes_on_gpu(16 * n, seed).view(-1, 16)
        out = torch.empty_like(x)
        blocks = torch.from_numpy(small["blocks"]).to(dev)
        msg = torch.repeat_interleave(torch.arange(len(blocks), device=dev, dtype=torch.int32), blocks)
        bits = small["keybits"][small["key_ids"]]
        for kb in (128, 192, 256):
            mine = [i for i, k in enumerate(small["keys"]) if 8 * k.size == kb]
            if not mine:
                continue
            keys = torch.from_numpy(np.stack([_expand([int(v) for v in small["keys"][i]], p.sbox) for i in mine])).to(dev)
            place = np.zeros(len(small["keys"]), np.int64)
            place[mine] = np.arange(len(mine))
            of_msg = torch.from_numpy(place[small["key_ids"]]).to(dev)
            for d in (0, 1):
                take = torch.from_numpy((bits == kb) & (small["dirs"] == d)).to(dev)
                at = torch.nonzero(take[msg.long()]).flatten() if n < (1 << 27) else None
                step = 1 << 20
                if at is not None:
                    for a in range(0, at.numel(), step):
                        i = at[a:a + step]
                        out[i] = p.cipher(x[i], keys, of_msg[msg[i].long()], d == 1)
                    continue
                for a in range(0, n, 8 * step):  # large batches: the selection itself in pieces
                    m = msg[a:a + 8 * step].long()
                    at = a + torch.nonzero(take[m]).flatten()
                    for b in range(0, at.numel(), step):
                        i = at[b:b + step]
                        out[i] = p.cipher(x[i], keys, of_msg[msg[i].long()], d == 1)
        out = out.view(-1)
        return {"out": out, "status": np.zeros(case["messages"], np.int32)} if kind == "serve" else out
    keys = torch.from_numpy(_expand([int(v) for v in small["key"]], p.sbox)[None]).to(dev)
    x = _bytes_on_gpu(16 * case["blocks"], seed).view(-1, 16)
    out = torch.empty_like(x)
    if kind in ("ecb", "ct", "host"):
        p.run(x, keys, None, case["dir"] == 1, out)
        return out.view(-1).cpu() if kind == "host" else out.view(-1)
    iv = torch.from_numpy(small["iv"]).to(dev)
    if kind == "ctr":
        first = int.from_bytes(small["iv"].tobytes(), "big")
        hi, lo = first >> 64, first & ((1 << 64) - 1)
        # 64-bit halves as signed words, bytes taken by shifts; at most one carry
        # into the upper half
        left = (1 << 64) - lo                    # blocks until the lower half wraps
        signed = lambda v: v - (1 << 64) if v >> 63 else v  # noqa: E731
        step = 1 << 20
        for a in range(0, case["blocks"], step):
            m = min(step, case["blocks"] - a)
            i = torch.arange(a, a + m, device=dev)
            low = i + torch.tensor(signed(lo), device=dev)  # wraps modulo 2^64
            high = torch.full_like(i, signed(hi))
            if left < a + m:
                high = torch.where(i >= left, torch.full_like(i, signed((hi + 1) & ((1 << 64) - 1))), high)
            ctr = torch.stack([(v >> s) & 0xFF for v in (high, low) for s in range(56, -1, -8)], 1).to(torch.uint8)
            out[a:a + m] = x[a:a + m] ^ p.cipher(ctr, keys, None, False)
        return out.view(-1)
    prev = torch.cat([iv[None], x[:-1]])
    if kind == "cbc":
        p.run(x, keys, None, True, out)
        out ^= prev
    else:
        p.run(prev, keys, None, False, out)
        out ^= x
    return out.view(-1)
