// mlp_exchange.h -- who sends what to whom in the network's forward and
// backward pass (net_kernel in mlp.cu), and the proof that no piece meets an
// earlier one.  Plain C++, so that a host compiler checks it too.
//
// A cluster's CTAs hold two operand buffers each.  In an exchange every
// sender writes its units into its own buffer and copies them to the same
// place in the buffer of every receiver; a receiver waits until all pieces
// have arrived (one phase of the buffer's mbarrier), takes the product from
// the buffer and goes on.  The copies are asynchronous and not ordered among
// themselves, and a phase of the mbarrier counts whatever bytes arrive, so a
// CTA may send only when it knows, through the pieces it has itself waited
// for, that
//   (a) each receiver has finished its previous product from that buffer: the
//       phase is complete, no earlier piece is under way and none is read;
//   (b) its own earlier pieces from that buffer have arrived everywhere, as
//       it writes over the memory that they are copied from.
// ordered() follows what each CTA knows from exchange to exchange.
#pragma once

namespace iblb {

struct Exchange {
    int buffer;
    int senders, receivers;      // CTAs 0 .. senders - 1 send, 0 .. receivers - 1 receive
    int units;                   // K columns per sender: sender c's are units * c ..
};

constexpr int EX_CTAS = 8;       // CTAs per cluster: CTA c owns units 32c .. 32c + 31 of a hidden layer
constexpr int EX_OUT = 4;        // the output layer's 64 units on four of them

// The third hidden layer goes to the output layer's CTAs alone.  Sent to all
// eight, nothing would tell the others' senders that it had arrived there:
// only CTAs 0 .. 3 answer it (with dy), and the next use of that buffer could
// overtake it.
constexpr Exchange EX_H1{0, EX_CTAS, EX_CTAS, 32}, EX_H2{1, EX_CTAS, EX_CTAS, 32}, EX_H3{0, EX_CTAS, EX_OUT, 32};
constexpr Exchange EX_DY{1, EX_OUT, EX_CTAS, 16}, EX_D3{0, EX_CTAS, EX_CTAS, 32}, EX_D2{1, EX_CTAS, EX_CTAS, 32};
constexpr Exchange EX_FORWARD[] = {EX_H1, EX_H2, EX_H3};
constexpr Exchange EX_TRAINING[] = {EX_H1, EX_H2, EX_H3, EX_DY, EX_D3, EX_D2};

template <int N>
constexpr bool ordered(const Exchange (&x)[N])
{
    // known[i][r]: the last exchange that CTA i knows CTA r to have finished
    int known[EX_CTAS][EX_CTAS] = {}, told[EX_CTAS][EX_CTAS] = {};
    for (int i = 0; i < EX_CTAS; ++i)
        for (int r = 0; r < EX_CTAS; ++r)
            known[i][r] = -1;
    for (int k = 0; k < N; ++k) {
        for (int i = 0; i < x[k].senders; ++i)
            for (int e = 0; e < k; ++e) {
                if (x[e].buffer != x[k].buffer)
                    continue;
                for (int r = 0; r < x[e].receivers; ++r) {
                    const bool writes_there = r < x[k].receivers || r == i;              // (a)
                    const bool copied_from_here = i < x[e].senders;                      // (b)
                    if ((writes_there || copied_from_here) && known[i][r] < e)
                        return false;
                }
            }
        for (int i = 0; i < EX_CTAS; ++i)
            for (int r = 0; r < EX_CTAS; ++r)
                told[i][r] = known[i][r];                  // what travels with the pieces
        for (int i = 0; i < x[k].receivers; ++i) {
            for (int s = 0; s < x[k].senders; ++s)
                for (int r = 0; r < EX_CTAS; ++r)
                    if (told[s][r] > known[i][r])
                        known[i][r] = told[s][r];
            known[i][i] = k;
        }
    }
    return true;
}
static_assert(ordered(EX_FORWARD) && ordered(EX_TRAINING), "a piece could meet an earlier one");

}  // namespace iblb
