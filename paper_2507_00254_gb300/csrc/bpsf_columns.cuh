// The column path of the persistent kernel; included by bpsf_persistent.cuh,
// whose slots, boxes and manager it shares.
#pragma once

namespace bpsf {

// ---------------------------------------------------------------------------
// Column path (flooding, exact-degree codes): one column per lane.
//
// A team has a lane for every column of the code, so a lane keeps everything
// but the messages in registers for the whole launch: its column's message
// addresses, checks, channel LLR and flip words, and its row's syndrome signs.
// Shared memory then carries the messages (16 bytes per edge-update and slot)
// and the residual syndrome, one word per row with a bit per slot.  An
// iteration is short, so few runs are in flight and a failed shot's chain of
// iterations ends early.
//
// A lane serves all V slots of its column in the V phase, and half of the
// slots of a row in the C phase (a team has twice as many columns as rows, so
// both phases fill its warps).  The decision on an iteration is made beside
// the next C phase; the C phase of a finished run is wasted, and the run that
// takes its slot starts at a V phase, with the C2V messages that every run's
// first C phase gives: +-c2v0, by the check's syndrome bit.
//
// The last warp of the team is its service warp.  A service step comes after
// an iteration that ended a run, and every fourth iteration while a slot is
// empty or trials may be stopped: the service warp looks at the boxes and
// writes what it saw (service word: bits 0..7 slots to stop, 8..15 inbox holds
// an item, 16..23 outbox free, 31 leave), which the warps read after a
// barrier; every warp packs its columns' decisions of the finished slots;
// after a barrier the service warp publishes them while every warp installs
// its rows' and columns' part of the new items; a third barrier ends it.
// ---------------------------------------------------------------------------
template <int FB, int V>
__device__ __forceinline__ unsigned flip_field(typename FlipPack<FB, V>::U w, int c) {
    return ((unsigned)w >> (8 * FB * c)) & ((1u << (8 * FB)) - 1u);
}
template <>
__device__ __forceinline__ unsigned flip_field<2, 4>(uint2 w, int c) {
    return ((c < 2 ? w.x : w.y) >> (16 * (c & 1))) & 0xffffu;
}
template <int FB, int V>
__device__ __forceinline__ void flip_clear(typename FlipPack<FB, V>::U &w, int c) {
    w = (typename FlipPack<FB, V>::U)((unsigned)w & ~(((1u << (8 * FB)) - 1u) << (8 * FB * c)));
}
template <>
__device__ __forceinline__ void flip_clear<2, 4>(uint2 &w, int c) {
    unsigned &h = c < 2 ? w.x : w.y;
    h &= ~(0xffffu << (16 * (c & 1)));
}

// The first of the running slots' caps (lanes c < V hold slot c's in SlotState::limit).
__device__ __forceinline__ int first_cap(const SlotState *st, unsigned run, int lane) {
    return __reduce_min_sync(FULLMASK, ((run >> lane) & 1u) ? st[lane].limit : 0x7fffffff);
}

// sd, to: the block's copies in shared memory; tb: the team's offset there.
// LONG: codes with more columns than a team has lanes, of at most DC ones per
// row and DV per column.  Lanes loop over columns and rows, whose tables and
// flip words are in shared memory, and the syndrome bits of 32 / V rows share a
// word (bit j*V + c, as in the team path): fewer words to look at, and few
// decisions change.
template <int DC, int DV, int DVS, int V, bool LONG, bool DEBUG, int FB>
__device__ __forceinline__ void column_loop(const StreamDev &sd, const TeamOffsets &to, BlockHdr *hdr,
                                            const LayoutMem &L, const int tb, const int W, const int tid_,
                                            const int bar_id) {
    typedef typename VecF<V>::T VT;
    typedef FlipPack<FB, V> FP;
    constexpr int lgS = V == 4 ? 2 : V - 1;
    constexpr unsigned full = (1u << V) - 1u;
    constexpr int CV = V > 1 ? V / 2 : 1;  // slots per lane in the C phase
    constexpr int CG = V / CV;             // lanes per row there
    typedef typename VecF<CV>::T CT;
    const CodeDev &cd = sd.code;
    extern __shared__ __align__(16) unsigned char smem[];
    const int tid = tid_, nth_ = 32 * W, nth = nth_, lane = tid & 31;
    const bool sw = (tid >> 5) == W - 1;  // service warp
    const int M = keep(cd.M), N = keep(cd.N);
    const int nw = LONG ? keep(((M << lgS) + 31) >> 5) : M;  // residual words
    const int o_mism = keep(tb + to.mism), o_m = keep(tb + to.m), o_flips = keep(tb + to.flips);
    const int o_syn = keep(tb + to.syn);
    const int mstride = keep(cd.Mp * (int)sizeof(VT));
    // !LONG: the lane's row part (seeds) and column: message and residual word
    // (byte offsets in shared memory), channel LLR, flip words.
    float seed[CV];
#pragma unroll
    for (int c = 0; c < CV; ++c) seed[c] = 0.f;
    int mcol[DV], res[DV];
    float lc = 0.f;
    typename FP::U fw = typename FP::U();
    if (!LONG) {
        const int i = tid < N ? tid : 0;
#pragma unroll
        for (int d = 0; d < DV; ++d) {
            mcol[d] = o_m + (int)cd.vpos[i * DVS + d] * (int)sizeof(VT);
            res[d] = o_mism + 4 * (int)cd.vchk[i * DVS + d];
        }
        lc = cd.lch[i];
    }
    typename FP::D on = FP::on(0u);  // the running slots' decision bits
    const bool adaptive = keep(!(cd.alpha > 0.f));
    const bool first_rule = keep(cd.select == 1);
    // Damping of the row slots' last iteration.  Adaptive: 1 - 2^-t, and the next
    // is half of 1 + that, rounded once (both are exact up to t = 24, and 1 after).
    float al[CV];
#pragma unroll
    for (int c = 0; c < CV; ++c) al[c] = cd.alpha;
    // Slot masks (the same in every warp): running; and in one word finished, not
    // yet packed (bits 0..7), of these the converged (8..15), initial runs (16..23).
    unsigned run = 0u, rest = 0u;
    int tt = 0;                 // team iterations so far
    int next_cap = 0x7fffffff;  // the first of the running slots' caps
    if (sw && lane == 0) {
        TeamCtl *ctl = reinterpret_cast<TeamCtl *>(smem + tb + to.ctl);
        ctl->idle_since = 0;
        ctl->idle_ns = kIdleMinNs;
        ctl->idle_looks = 0;
        ctl->flushed = 0;
    }
    for (;;) {
        if (run != 0u) {
            // C phase; the decision on the previous iteration is made beside it.
            uint4 w4 = make_uint4(0u, 0u, 0u, 0u);
            if (!LONG && 4 * lane < nw) w4 = *reinterpret_cast<const uint4 *>(smem + o_mism + 16 * lane);
            if (adaptive) {
#pragma unroll
                for (int c = 0; c < CV; ++c) al[c] = __fmaf_rn(al[c], 0.5f, 0.5f);
            }
            auto row_part = [&](int task) {
                const int deg = LONG ? (int)L.row_deg[task / CG] : DC;
                unsigned char *row = smem + o_m + task * (int)sizeof(CT);
                float x[DC][CV], sd_[CV];
#pragma unroll
                for (int k = 0; k < DC; ++k) {
                    if (!LONG || k < deg) {
                        vload<CV>(x[k], reinterpret_cast<const CT *>(row + k * mstride));
                    } else {
#pragma unroll
                        for (int c = 0; c < CV; ++c) x[k][c] = __int_as_float(0x7f800000);
                    }
                }
#pragma unroll
                for (int c = 0; c < CV; ++c) sd_[c] = seed[c];
                if (LONG) {
                    const int b = task * CV;  // the part's first syndrome bit
                    row_seed<CV, true>(sd_, *reinterpret_cast<const uint32_t *>(smem + o_syn + (b >> 5) * 4) >> (b & 31));
                }
#pragma unroll
                for (int k = 0; k < DC; ++k) vmul<CV>(x[k], x[k], al);
                row_outputs<DC, CV>(x, sd_);
#pragma unroll
                for (int k = 0; k < DC; ++k)
                    if (!LONG || k < deg) vstore<CV>(reinterpret_cast<CT *>(row + k * mstride), x[k]);
            };
            if constexpr (LONG) {
#pragma unroll 1
                for (int task = tid; task < CG * M; task += nth) row_part(task);
                if (4 * lane < nw) w4 = *reinterpret_cast<const uint4 *>(smem + o_mism + 16 * lane);
            } else if (tid < CG * M) {
                row_part(tid);
            }
            unsigned acc = (w4.x | w4.y) | (w4.z | w4.w);
            for (int j = 4 * lane + 128; j < nw; j += 128) {
                w4 = *reinterpret_cast<const uint4 *>(smem + o_mism + 4 * j);
                acc |= (w4.x | w4.y) | (w4.z | w4.w);
            }
            if (LONG) {
#pragma unroll
                for (int sh = 16; sh >= V; sh >>= 1) acc |= acc >> sh;
            }
            const unsigned nconv = __reduce_or_sync(FULLMASK, acc) & full;
            if ((run & ~nconv) || tt >= next_cap) {
                SlotState *st = reinterpret_cast<SlotState *>(smem + tb + to.state);
                const bool mine = (run >> lane) & 1u;
                const unsigned done = run & (~nconv | __ballot_sync(FULLMASK, mine && tt >= st[lane].limit));
                if (sw && ((done >> lane) & 1u)) {
                    st[lane].iter = tt - st[lane].start;
                    st[lane].outcome = ((nconv >> lane) & 1u) ? 2 : 1;
                }
                rest = (rest & ~(done << 8)) | ((done & ~nconv) << 8) | done;
                run &= ~done;
                on = FP::on(run);
                next_cap = first_cap(st, run, lane);
            }
        }
        if (run == 0u || (rest & full) || ((tt & 3) == 0 && (run != full || first_rule))) {
            // Service step.  (Its index arithmetic is kept from moving out of the loop,
            // where it would hold registers all the time.)
            const int tid = keep(tid_), nth = keep(nth_), lane = tid & 31;
            const TeamMem T = team_mem(smem + tb, to);
            unsigned pend = rest & full, pconv = (rest >> 8) & full, initm = rest >> 16;
            if (sw) {
                const bool in = lane < V && *vflag(&T.ibf[lane < V ? lane : 0]) != 0;
                const bool out = lane < V && *vflag(&T.ob[lane < V ? lane : 0].full) == 0;
                unsigned e = (__ballot_sync(FULLMASK, in) << 8) | (__ballot_sync(FULLMASK, out) << 16);
                if (first_rule) {
                    bool cancel = false;
                    if (((run & ~initm) >> lane) & 1u)
                        cancel = *reinterpret_cast<volatile long long *>(&T.st[lane].cancel) ==
                                 T.st[lane].shot * (long long)cd.n_trials + T.st[lane].kidx + 1;
                    e |= __ballot_sync(FULLMASK, cancel);
                }
                if (run == 0u) {
                    if (!((pend & (e >> 16)) | (full & ~pend & (e >> 8)))) {
                        if (hdr->exit) {
                            e = 0x80000000u;
                        } else {
                            // Never wait forever: give up only if the manager has made
                            // no pass for twice the bound on any of its own waits.
                            const unsigned long long now = globaltimer_ns();
                            const unsigned beat = hdr->heartbeat;
                            unsigned long long since_ns = T.ctl->idle_since;
                            if (since_ns == 0 || beat != T.ctl->last_beat) since_ns = now;
                            if (now - since_ns > 2 * hdr->wait_ns) e = 0x80000000u;
                            unsigned ns = T.ctl->idle_ns;
                            const unsigned looks = T.ctl->idle_looks + 1;
                            __nanosleep(ns);
                            if (looks > kIdleLooks) ns = ns < kIdleMaxNs ? 2 * ns : kIdleMaxNs;
                            __syncwarp();
                            if (lane == 0) {
                                T.ctl->idle_since = since_ns;
                                T.ctl->last_beat = beat;
                                T.ctl->idle_ns = ns;
                                T.ctl->idle_looks = looks;
                            }
                        }
                    } else if (lane == 0) {
                        T.ctl->idle_since = 0;
                        T.ctl->idle_ns = kIdleMinNs;
                        T.ctl->idle_looks = 0;
                    }
                }
                if (lane == 0) T.ctl->run_mask = e;
            }
            team_sync(W, bar_id);  // also: every warp is through its C phase
            const unsigned ev = T.ctl->run_mask;
            if (ev >> 31) break;
            const unsigned stop = run & ev & full;  // trials asked to stop
            if (stop) {
                if (sw && ((stop >> lane) & 1u)) {
                    T.st[lane].iter = tt - T.st[lane].start;
                    T.st[lane].outcome = 3;
                }
                pconv &= ~stop;
                pend |= stop;
                run &= ~stop;
                next_cap = first_cap(T.st, run, lane);
            }
            const unsigned pk = pend & (ev >> 16);
            const unsigned inst = (full & ~run & ~(pend & ~pk)) & (ev >> 8);
            if (pk) {
                // Pack: a warp's k-th columns are one word of a finished slot's decision.
#pragma unroll 1
                for (unsigned m = pk; m; m &= m - 1u) {
                    const int c = __ffs(m) - 1;
                    const bool counts = ((initm & ~pconv) >> c) & 1u;
                    // A long code's converged initial run: its decision goes out at once (the
                    // manager's one lane would write 81 words).
                    uint32_t *words = T.ebits + c * cd.Wn;
                    if (LONG && ((initm & pconv) >> c & 1u)) words = sd.job.corr + row_of(sd, T.st[c].shot) * sd.job.corr_stride;
#pragma unroll 2
                    for (int i0 = tid - lane; i0 < N; i0 += nth) {
                        const int i = i0 + lane;
                        unsigned f = 0u;
                        if (!LONG)
                            f = flip_field<FB, V>(fw, c);
                        else if (i < N)
                            f = (unsigned)flipw<FB>(T)[(i << lgS) + c];
                        const unsigned word = __ballot_sync(FULLMASK, i < N && flip_dec<FB>(f) != 0u);
                        if (lane == 0) words[i >> 5] = word;
                        if (!LONG && i < N && counts) flipw<FB>(T)[(i << lgS) + c] = (typename FlipW<FB>::W)f;
                        if (DEBUG && sd.dbg.flips && i < N && ((initm >> c) & 1u))
                            sd.dbg.flips[T.st[c].shot * N + i] = (uint16_t)flip_count<FB>(f);
                    }
                }
                team_sync(W, bar_id);
                if (sw) {
                    // The work counters first: the manager adds them up once every
                    // slot of the block reads empty.
                    if (lane == 0) {
                        for (unsigned m = pk; m; m &= m - 1u) T.ctl->iters += T.st[__ffs(m) - 1].iter;
                        T.ctl->cap += (unsigned long long)(tt - T.ctl->flushed) * (unsigned)V;
                        T.ctl->flushed = tt;
                    }
#pragma unroll 1
                    for (unsigned m = pk; m; m &= m - 1u) {
                        const int c = __ffs(m) - 1;
                        const SlotState *ss = &T.st[c];
                        if (((initm >> c) & 1u) && ss->outcome == 2 && cd.w > 0)
                            publish_failure<DEBUG, FB, !LONG>(sd, T, lgS, c, lane, hdr->wait_ns);
                        if (lane == 0) {
                            OutBox *ob = &T.ob[c];
                            ob->kind = ss->kind;
                            ob->kidx = ss->kidx;
                            ob->rec = ss->rec;
                            ob->outcome = ss->outcome;
                            ob->iter = ss->iter;
                            ob->shot = ss->shot;
                            // The outbox flag before the slot reads EMPTY (the manager's
                            // exit test reads the state first, then the outbox flag).
                            __threadfence_block();
                            *vflag(&ob->full) = 1;
                            __threadfence_block();
                            *vstate(&T.st[c]) = kSlotEmpty;
                        }
                        __syncwarp();
                    }
                }
                // A failed run's record is made from the syndrome and flip words that an
                // install rewrites (!LONG: its words are the service warp's own).
                if (LONG && (pk & initm & ~pconv)) team_sync(W, bar_id);
                pend &= ~pk;
            }
            if (inst) {
                __threadfence_block();  // the inbox items are visible
                unsigned live = 0u;
                unsigned mis = !LONG && tid < M ? T.mism[tid] : 0u;
#pragma unroll 1
                for (unsigned m = inst; m; m &= m - 1u) {
                    const int c = __ffs(m) - 1;
                    const QEntry *e = reinterpret_cast<const QEntry *>(T.ib + c * T.ibstride);
                    const uint32_t *src = reinterpret_cast<const uint32_t *>(T.ib + c * T.ibstride + sizeof(QEntry));
                    const int kind = e->kind;
                    if (kind == 0) continue;
                    live |= 1u << c;
                    initm = kind == 1 ? initm | (1u << c) : initm & ~(1u << c);
                    if (!LONG) {
                        if (tid < M) mis = (mis & ~(1u << c)) | (((src[tid >> 5] >> (tid & 31)) & 1u) << c);
                        if (tid < CG * M && c / CV == tid % CG) {
                            // The stored C2V messages carry the opposite sign.
                            const int j = tid / CG;
                            const unsigned b = (src[j >> 5] >> (j & 31)) & 1u;
                            const float v = __uint_as_float((b ? 0u : 0x80000000u) | 0x71800000u);
                            const bool last = CV == 1 || (c & 1);  // selects: an index would put the array in memory
                            seed[0] = CV > 1 && last ? seed[0] : v;
                            seed[CV - 1] = last ? v : seed[CV - 1];
                        }
                        flip_clear<FB, V>(fw, c);
                    } else {
                        // Word w: rows w * 32/V .., slot c at bits c, c + V, ...
                        constexpr int per = 32 / V;
                        for (int w = tid; w < nw; w += nth) {
                            const unsigned b = src[(w * per) >> 5] >> ((w * per) & 31);
                            unsigned keep_ = 0u, put = 0u;
#pragma unroll
                            for (int j = 0; j < per; ++j) {
                                keep_ |= 1u << (j * V);
                                put |= (w * per + j < M ? (b >> j) & 1u : 0u) << (j * V);
                            }
                            T.mism[w] = (T.mism[w] & ~(keep_ << c)) | (put << c);
                            T.syn[w] = (T.syn[w] & ~(keep_ << c)) | (put << c);
                        }
                        for (int i = tid; i < N; i += nth) flipw<FB>(T)[(i << lgS) + c] = 0;
                    }
                    if (c / CV == tid % CG) {
                        const bool last = CV == 1 || (c & 1);
                        al[0] = !adaptive || (CV > 1 && last) ? al[0] : 0.5f;
                        al[CV - 1] = adaptive && last ? 0.5f : al[CV - 1];
                    }
                    // The rows' first C2V messages, by their syndrome bits.
                    const bool same = cd.uniform != 0;
                    const float first = fminf(__fmul_rn(adaptive ? 0.5f : cd.alpha, cd.lch0), kMagClamp);
                    for (int j = tid; j < M; j += nth) {
                        const unsigned flip = ((src[j >> 5] >> (j & 31)) & 1u) ? 0u : 0x80000000u;
                        const int dj = LONG ? (int)L.row_deg[j] : DC;
                        float *msg = reinterpret_cast<float *>(smem + o_m) + j * V + c;
#pragma unroll
                        for (int k = 0; k < DC; ++k)
                            if (!LONG || k < dj)
                                msg[k * (mstride >> 2)] =
                                    __uint_as_float(__float_as_uint(same ? first : __ldg(cd.c2v0 + k * cd.Mp + j)) ^ flip);
                    }
                    if (sw) {
                        for (int w = lane; !LONG && w < cd.Ws; w += 32) T.syn[c * cd.Ws + w] = src[w];
                        if (lane == 0) {
                            SlotState *ss = &T.st[c];
                            ss->kind = kind;
                            ss->kidx = e->kidx;
                            ss->rec = e->rec;
                            ss->shot = e->shot;
                            ss->cancel = 0;
                            ss->start = tt;
                            ss->limit = tt + (kind == 1 ? cd.max_iter : cd.short_iter);
                        }
                    }
                }
                if (!LONG && tid < M) T.mism[tid] = mis;
                team_sync(W, bar_id);
                if (sw && lane == 0) {
                    // RUNNING before the inbox reads empty: the manager's exit test
                    // reads the inbox flag first, then the state.
#pragma unroll
                    for (int c = 0; c < V; ++c)
                        if ((live >> c) & 1u) *vstate(&T.st[c]) = kSlotRunning;
                    __threadfence_block();
#pragma unroll
                    for (int c = 0; c < V; ++c)
                        if ((inst >> c) & 1u) *vflag(&T.ibf[c]) = 0;
                }
                __syncwarp();
                run |= live;
                next_cap = first_cap(T.st, run, lane);
            }
            rest = pend | (pconv << 8) | (initm << 16);
            on = FP::on(run);
            if (run == 0u) {
                if (!inst) team_sync(W, bar_id);  // every warp has read the word that the next look rewrites
                continue;
            }
        } else {
            team_sync(W, bar_id);
        }
        // V phase.  mp: the messages' places, -1 where the column has no such edge.
        auto column = [&](int i, const int (&mp)[DV], float l, typename FP::U &f) {
            float r[DV][V], pre[V], nl[V];
#pragma unroll
            for (int d = 0; d < DV; ++d) {
                if (!LONG || mp[d] >= 0) {
                    vload<V>(r[d], reinterpret_cast<const VT *>(smem + mp[d]));
                } else {
#pragma unroll
                    for (int c = 0; c < V; ++c) r[d][c] = 0.f;
                }
            }
#pragma unroll
            for (int c = 0; c < V; ++c) pre[c] = l;
#pragma unroll
            for (int d = 0; d < DV; ++d) {
                float acc[V];
#pragma unroll
                for (int c = 0; c < V; ++c) acc[c] = pre[c];
#pragma unroll
                for (int d2 = d + 1; d2 < DV; ++d2) vsub<V>(acc, acc, r[d2]);
                if (d + 1 < DV)
                    vsub<V>(pre, pre, r[d]);
                else
                    vnegdiff<V>(nl, pre, r[d]);  // -l_out
                if (!LONG || mp[d] >= 0) vstore<V>(reinterpret_cast<VT *>(smem + mp[d]), acc);
            }
            if (DEBUG && sd.dbg.lout) {
                const SlotState *st = reinterpret_cast<const SlotState *>(smem + tb + to.state);
#pragma unroll
                for (int c = 0; c < V; ++c)
                    if (((run & (rest >> 16)) >> c) & 1u) sd.dbg.lout[st[c].shot * N + i] = __fsub_rn(0.f, nl[c]);
            }
            const typename FP::U f0 = f;
            const typename FP::D dd = FP::diff(nl, f0, on);
            if (FP::any(dd)) {
                f = FP::bump(f0, dd);
                const unsigned bm = FP::slots(dd);
#pragma unroll
                for (int d = 0; d < DV; ++d) {
                    if (!LONG) {
                        atomicXor(reinterpret_cast<uint32_t *>(smem + res[d]), bm);
                    } else if (mp[d] >= 0) {
                        const int b = (int)__ldg(cd.vchk + i * DVS + d) << lgS;
                        atomicXor(reinterpret_cast<uint32_t *>(smem + o_mism) + (b >> 5), bm << (b & 31));
                    }
                }
            }
        };
        if constexpr (!LONG) {
            if (tid < N) column(tid, mcol, lc, fw);
        } else {
            typename FP::U *fl = reinterpret_cast<typename FP::U *>(smem + o_flips);
#pragma unroll 1
            for (int i = tid; i < N; i += nth) {
                static_assert(!LONG || DVS == 4, "a column's places are one 64-bit word");
                const uint2 raw = *reinterpret_cast<const uint2 *>(L.vpos + i * DVS);
                const unsigned p[4] = {raw.x & 0xffffu, raw.x >> 16, raw.y & 0xffffu, raw.y >> 16};
                int mp[DV];
#pragma unroll
                for (int d = 0; d < DV; ++d) mp[d] = p[d & 3] == 0xffffu ? -1 : o_m + (int)p[d & 3] * (int)sizeof(VT);
                column(i, mp, L.lch[i], fl[i]);
            }
        }
        ++tt;
        team_sync(W, bar_id);
    }
}

}  // namespace bpsf
